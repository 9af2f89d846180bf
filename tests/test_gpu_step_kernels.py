"""Edges of the kernels of the inner step, against the oracle."""
import pytest
import torch

from paper_2602_04396_b200 import lordo, synth
from tests import harness as hz
from tests.harness import RunSpec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(8, 8, 8), (72, 64, 8), (136, 72, 64), (1000, 64, 16), (520, 600, 72)])
@pytest.mark.parametrize("side", [0, 1])
def test_fp32_products_in_ranges_of_k(shape, side):
    """The fp32 products with their contraction in one CTA or dealt out over a cluster (few tiles, long
    contraction), ranges without a slice and a ragged last slice among them. The ranges meet in fp64, so the
    bound of the other check-mode tests (1e-3, a few fp32 ulps per step in fact) is held to 2e-5."""
    m, n, r = shape
    if side:
        m, n = n, m
    wl = synth.Workload("t", ((m, n, r),), K=2, H=2, rounds=1, grad="gauss", clip_rho=30.0, sides=(side,))
    spec = RunSpec(wl, variant=1, form=2, lr=0.01, omega=0.9, eps=0.05, refresh=False)
    opt, orc = hz.run_gpu(spec), hz.run_oracle(spec)
    st = hz.compare_states(opt, orc)
    assert opt.poll_status() == 0
    assert max(st["W"], st["E"], st["u"], st["v"]) < 2e-5, st
    opt.close()


@pytest.mark.parametrize("mats,K", [(((1001, 1336, 72), (527, 392, 136), (200, 136, 24)), 3), (((2200, 264, 72), (72, 4040, 24), (96, 1536, 8)), 1)])
@pytest.mark.parametrize("side", [0, 1])
def test_fp32_products_of_many_tiles(side, mats, K):
    """More tiles than the device holds at once, worked on by threads of eight rows: ragged in every direction, a tile with 8 of 64 rows, a
    contraction that ends within a slice, with one product and with two. Then a few tiles of a long contraction among many of a
    short one, in clusters of eight CTAs of which most have no slice of the short ones. Bound as above."""
    if side:
        mats = tuple((n, (m + 7) // 8 * 8, r) for m, n, r in mats)
    wl = synth.Workload("t", mats, K=K, H=2, rounds=1, grad="gauss", clip_rho=30.0, sides=(side,) * 3)
    spec = RunSpec(wl, variant=1, form=2, lr=0.01, omega=0.9, eps=0.05, refresh=False)
    opt, orc = hz.run_gpu(spec), hz.run_oracle(spec)
    st = hz.compare_states(opt, orc)
    assert opt.poll_status() == 0
    assert max(st["W"], st["E"], st["u"], st["v"]) < 2e-5, st
    opt.close()


@pytest.mark.parametrize("mats", [((72, 64, 8),), ((2056, 136, 24), (136, 2088, 64)), ((4104, 136, 24),), ((1544, 264, 72), (520, 1032, 264))])
@pytest.mark.parametrize("side", [0, 1])
def test_strips_in_pieces(mats, side):
    """The update's strips whole, in two pieces and in many (one matrix with few columns and many rows), shorter
    than the shortest piece, of very different lengths in one list, with one sweep and with two (r > 256)."""
    mats = tuple((n, m, r) if side else (m, n, r) for m, n, r in mats)
    wl = synth.Workload("t", mats, K=2, H=2, rounds=1, grad="gauss", clip_rho=30.0, w_dtype="bf16", g_dtype="bf16", e_dtype="bf16",
                        sides=(side,) * len(mats))
    spec = RunSpec(wl, variant=0, form=2, lr=0.01, omega=0.9, check_mode=0, eps=0.05, refresh=False)
    opt, orc = hz.run_gpu(spec), hz.run_oracle(spec)
    st = hz.compare_states(opt, orc)
    assert opt.poll_status() == 0
    tol = 8 * 2.0 ** -9  # bf16 operands, as for the other fast-mode tests
    assert st["u"] < tol and st["v"] < 2 * tol and st["E"] < 2 * tol, st
    for i in range(len(mats)):
        d = hz.bf16_ulp_distance(hz._np_state(opt.W[i]), orc.W[i])
        assert (d <= 1).mean() > 0.99 and d.max() <= 8, ((d <= 1).mean(), d.max())
    opt.close()


@pytest.mark.parametrize("dt", ["f32", "bf16"])
@pytest.mark.parametrize("mats,K", [(((8, 8, 8),), 1), (((256, 256, 16),), 2), (((200, 136, 24), (8, 2056, 8), (264, 520, 40)), 5),
                                    (((24, 24, 8),) * 300, 3), (((2048, 2056, 8),), 3)])
@pytest.mark.parametrize("scope", [0, 1])
def test_clip_coefficients_in_one_launch(dt, mats, K, scope):
    """One chunk and many per (matrix, worker), a ragged last chunk, more matrices than threads; three launches in
    a row (the counters return to zero). Sums of squares: fp32 over at most 128 values, then fp64: 1e-5 relative."""
    gdt = synth.torch_dtype(dt)
    opt = lordo.Lordo(mats, K, 8, [torch.zeros(m, n, dtype=gdt) for m, n, _ in mats], g_dtype=gdt, e_dtype=gdt, clip_rho=2.0, clip_scope=scope)
    gen = torch.Generator(device="cuda")
    for step in range(3):
        G = []
        for i, (m, n, _) in enumerate(mats):
            gen.manual_seed(100 * step + i)
            G.append(torch.empty(K, m, n, device="cuda").normal_(generator=gen).to(gdt))
        opt.inner_step(G, 0.01, 0.9, 0.9, 2)
        sq = torch.stack([g.double().square().sum((1, 2)) for g in G])
        ref = (2.0 / ((sq if scope else sq.sum(0, keepdim=True).expand_as(sq)).sqrt() + 1e-6)).clamp(max=1.0)
        assert ((opt.clip_coefficients().double() - ref).abs() / ref).max().item() < 1e-5
    assert opt.poll_status() == 0
    opt.close()


@pytest.mark.parametrize("m,n,r", [(2048, 136, 16), (1096, 264, 240), (528, 1032, 144), (1032, 264, 256), (600, 72, 40), (72, 64, 8)])
@pytest.mark.parametrize("form", [1, 2])
def test_fp32_storage_strips_dealt_out(m, n, r, form):
    """fp32 storage: the projection with a strip's rows over one, two and four CTAs, ranks that do not divide evenly
    among them, more CTAs than chunks of 16 ranks; the update's strips whole and in pieces."""
    wl = synth.Workload("t", ((m, n, r),), K=2, H=3, rounds=1, grad="gauss", clip_rho=30.0)
    spec = RunSpec(wl, variant=0, form=form, lr=0.01, omega=0.9, check_mode=0, eps=0.05, refresh=False)
    opt, orc = hz.run_gpu(spec), hz.run_oracle(spec)
    st = hz.compare_states(opt, orc)
    assert opt.poll_status() == 0
    tol = 8 * 2.0 ** -9  # bf16 operands, as for the other fast-mode tests
    assert st["u"] < tol and st["v"] < 2 * tol and st["E"] < tol and st["W"] < tol * 3 * 0.01 / 0.02, st
    opt.close()


@pytest.mark.parametrize("mats", [((9, 8, 8),), ((33, 136, 8), (1001, 264, 40)), ((265, 392, 256), (40, 2056, 24)), ((2053, 520, 72),) * 5])
@pytest.mark.parametrize("ef", [True, False])
def test_fp32_storage_update_tiles(mats, ef):
    """The update's tiles of 32 rows x 128 columns in fp32: fewer rows than a tile or than the eight that are stored at a
    time, a last row alone, fewer columns than a strip, strips of different lengths in one list, more strips than SMs."""
    wl = synth.Workload("t", mats, K=2 if len(mats) < 5 else 8, H=2, rounds=1, grad="gauss", clip_rho=30.0)
    spec = RunSpec(wl, variant=1, form=2, lr=0.01, omega=0.9, check_mode=0, eps=0.05, refresh=False, error_feedback=ef)
    opt, orc = hz.run_gpu(spec), hz.run_oracle(spec)
    st = hz.compare_states(opt, orc)
    assert opt.poll_status() == 0
    tol = 8 * 2.0 ** -9  # bf16 operands, as for the other fast-mode tests
    assert st["u"] < tol and st["v"] < 2 * tol and st["W"] < tol * 2 * 0.01 / 0.02, st
    assert not ef or st["E"] < tol, st
    opt.close()


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("count", [1, 33])
def test_gradients_in_other_buffers_every_step(dt, count):
    """The table of pointers and the tensor maps behind it, copied as one into either slot in turn: the same bits as
    with every step's gradients copied into the buffers of the first."""
    mats = [(72, 136, 16)] * count
    gen = torch.Generator(device="cuda").manual_seed(3)
    G = [[torch.randn(2, m, n, device="cuda", generator=gen).to(dt) for m, n, _ in mats] for _ in range(4)]
    kw = dict(check_mode=0, clip_rho=1.0, seed=1, g_dtype=dt, e_dtype=dt)
    a, b = (lordo.Lordo(mats, 2, 8, [torch.zeros(m, n, dtype=dt) for m, n, _ in mats], **kw) for _ in range(2))
    fixed = [g.clone() for g in G[0]]
    for g in G:
        a.inner_step(g, 0.01, 0.9, 0.9, 1)
        for x, y in zip(fixed, g):
            x.copy_(y)
        b.inner_step(fixed, 0.01, 0.9, 0.9, 1)
    assert a.poll_status() == 0 and b.poll_status() == 0
    for x, y in zip(a.W + a.E + a.u + a.v, b.W + b.E + b.u + b.v):
        assert torch.equal(x, y)
    a.close()
    b.close()
