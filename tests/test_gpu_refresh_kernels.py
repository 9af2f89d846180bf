"""Edges of the kernels of the tensor-core refresh, against the oracle on the CUDA path's own state."""
import ctypes as C
import subprocess

import pytest
import torch

from paper_2602_04396_b200 import build as lbuild
from paper_2602_04396_b200 import lordo, synth
from tests import harness as hz
from tests.harness import RunSpec

pytestmark = pytest.mark.gpu

ANGLE_TOL, ORTH_TOL, ROT_TOL = 1e-3, 1e-5, 16 * 2.0 ** -16  # as for the other refresh tests


def _refresh(m, n, r, K=1, variant=1, grad="gauss", q=0, **kw):
    wl = synth.Workload(f"t{m}x{n}r{r}", ((m, n, r),), K=K, H=1, rounds=2, grad=grad, clip_rho=30.0, power_iters=q,
                        w_dtype="bf16", g_dtype="bf16", e_dtype="bf16", **kw)
    opt, _, worst = hz.run_lockstep_refresh(RunSpec(wl, variant=variant, form=1, lr=0.01, check_mode=0, eps=0.05), rounded_signal=True)
    assert opt.poll_status() == 0
    opt.close()
    return worst


@pytest.mark.parametrize("shape", [(64, 72, 8), (1096, 264, 8), (2056, 520, 264), (600, 4104, 40), (1544, 768, 512)])
def test_gram_in_ranges_of_k(shape):
    """Gram matrices in one range of k, in many, with a ragged last step and at both tile counts (r up to 256
    and above). Gaussian noise as the signal: the sketch has exact operands, only the QR is left to differ."""
    w = _refresh(*shape)
    assert w["P_angle"] < ANGLE_TOL and w["P_orth"] < ORTH_TOL, w
    assert w["rot_u"] < ROT_TOL and w["rot_v"] < 2 * ROT_TOL, w


@pytest.mark.parametrize("shape,q", [((70000, 64, 8), 0), ((64, 70000, 8), 1), ((90048, 72, 40), 0)])
def test_gram_of_a_vocabulary_sized_matrix(shape, q):
    """More rows (or, with an iteration, columns) than 32 ranges of 64 steps hold; Rot above 64 ranges of 64 steps. Signal of
    rank r plus 0.5 % noise, so that the iteration's span is well conditioned; tolerances as above."""
    kw = dict(grad="lowrank", signal_rank=shape[2], noise=0.005) if q else {}
    w = _refresh(*shape, q=q, **kw)
    assert w["P_orth"] < ORTH_TOL and w["rot_u"] < ROT_TOL and w["rot_v"] < 2 * ROT_TOL, w
    assert w["P_angle_bf16rhs"] < ANGLE_TOL, w


@pytest.mark.parametrize("r,count", [(8, 1), (32, 1), (40, 3), (256, 2), (264, 40), (504, 1), (296, 80), (512, 75), (136, 3), (512, 16), (192, 148), (256, 60)])
def test_cholesky_panels_and_clusters(r, count):
    """The factorisation behind P_0 = Q of a 2r x r integer matrix, against a QR in fp64: one panel, whole and
    ragged panels, clusters of eight CTAs (few matrices) down to one (many), more blocks per CTA than it sums at
    once (r = 192, 296, 512 in one CTA), one to four blocks for four units (test_plan_host.py holds the counts). The condition of such a matrix
    is about 6 (the ratio of the edges of its singular values): CholeskyQR2 in fp32 is off by a small multiple of 6^2 2^-24 = 2e-6."""
    mats = [(2 * r, r, r)] * count
    opt = lordo.Lordo(mats, 1, 1, [torch.zeros(2 * r, r)] * count, check_mode=0, seed=5)
    assert opt.poll_status() == 0
    for i in {0, count // 2, count - 1}:
        q, t = torch.linalg.qr(lordo.fill_random(5, 1, i, 0, 0, 2 * r, r).double())
        q = q * torch.sign(torch.diagonal(t))
        assert ((opt.P[i].double() - q).norm() / q.norm()).item() < 1e-5
    opt.close()


RECIP = """
#include "lordo_recip.cuh"
__global__ void kernel(const double* d, double* out, int n) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  double r0, e;
  lordo::recip_parts(d[i], r0, e);
  out[i] = fma(r0, e, r0);
  out[n + i] = lordo::recip_sqrt(d[i]);
  out[2 * n + i] = 1.0 / d[i];
  out[3 * n + i] = 1.0 / sqrt(d[i]);
}
extern "C" int run(const double* d, double* out, int n) {
  kernel<<<(n + 255) / 256, 256>>>(d, out, n);
  return (int)cudaDeviceSynchronize();
}
"""


def test_reciprocals_of_the_pivots(tmp_path):
    """lordo_recip.cuh against CUDA's division and square root: both sides are within 2^-52 of the exact value (the
    header's bound; half an ulp for the division, an ulp for the root and the division behind it), so they differ by 2^-51 at
    most. Every exponent that a pivot of an fp32 Gram matrix can have, powers of two and their neighbours, and pivots at
    the two floors."""
    src, so = tmp_path / "recip.cu", tmp_path / "recip.so"
    src.write_text(RECIP)
    subprocess.run(["/usr/local/cuda/bin/nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "-I", lbuild.CSRC, "-o", str(so), str(src)], check=True)
    gen = torch.Generator().manual_seed(1)
    exps = torch.arange(-190, 130, dtype=torch.float64)
    mant = torch.cat([1 + torch.rand(4000, generator=gen, dtype=torch.float64), torch.tensor([1.0, 1 + 2.0 ** -52, 2 - 2.0 ** -52, 1.5])])
    d = (2.0 ** exps[:, None] * mant).flatten()
    diag = torch.rand(4000, generator=gen) * 1e3
    d = torch.cat([d, (3e-5 * diag).double(), (1e-12 * diag).double().clamp_min(1e-30), torch.ones(1, dtype=torch.float64)]).cuda()
    out = torch.empty(4, d.numel(), device="cuda", dtype=torch.float64)
    assert C.CDLL(str(so)).run(C.c_void_p(d.data_ptr()), C.c_void_p(out.data_ptr()), d.numel()) == 0
    for mine, cuda in ((out[0], out[2]), (out[1], out[3])):
        assert ((mine - cuda).abs() / cuda).max().item() <= 2.0 ** -51


@pytest.mark.parametrize("mats,K", [(((72, 64, 8),), 1), (((136, 264, 40), (264, 392, 136)), 3), (((520, 648, 256), (600, 1032, 264)), 2),
                                    (((1032, 1544, 512),), 2), (((64, 40, 8), (64, 2056, 24)), 2), (((392, 1288, 264),), 16)])
@pytest.mark.parametrize("variant,side", [(0, 0), (1, 0), (1, 1)])
def test_rotation_in_place(mats, K, variant, side):
    """Rotated moments against the oracle's rotation lines on the bases of the CUDA path: ranks below one stage of
    32, ragged stages, above and below 256 in one launch (pairs that share a strip and pairs that do not), an odd
    number of strips, several shared strips one after the other in a pair (176 strips), one basis and one per worker."""
    mats = tuple((n, m, r) if side else (m, n, r) for m, n, r in mats)
    wl = synth.Workload("t", mats, K=K, H=2, rounds=2, grad="gauss", clip_rho=30.0, w_dtype="bf16", g_dtype="bf16", e_dtype="bf16",
                        sides=(side,) * len(mats))
    opt, _, w = hz.run_lockstep_refresh(RunSpec(wl, variant=variant, form=1, lr=0.01, check_mode=0, eps=0.05), rounded_signal=True)
    assert opt.poll_status() == 0
    opt.close()
    assert w["rot_u"] < ROT_TOL and w["rot_v"] < 2 * ROT_TOL, w


@pytest.mark.parametrize("shape", [(136, 72, 16), (520, 1032, 40), (648, 776, 264)])
@pytest.mark.parametrize("q,warm,side", [(1, False, 0), (2, False, 1), (1, True, 0), (2, True, 1)])
def test_signal_kept_for_later_products(shape, q, warm, side):
    """Local rule with several products per refresh: c G + E is formed once, by a product of either orientation,
    with ragged edges in both directions. Signal of rank r plus 0.5 % noise, as in the tests of the subspace angle."""
    m, n, r = shape
    if side:
        m, n = n, m
    wl = synth.Workload("t", ((m, n, r),), K=2, H=2, rounds=2, grad="lowrank", signal_rank=r, noise=0.005, clip_rho=30.0, power_iters=q,
                        w_dtype="bf16", g_dtype="bf16", e_dtype="bf16", sides=(side,))
    spec = RunSpec(wl, variant=1, form=1, lr=0.01, check_mode=0, eps=0.05, warm_start=warm)
    opt, _, w = hz.run_lockstep_refresh(spec, rounded_signal=True)
    assert opt.poll_status() == 0
    opt.close()
    assert w["P_orth"] < ORTH_TOL and w["rot_u"] < ROT_TOL and w["rot_v"] < 2 * ROT_TOL, w
    assert w["P_angle_bf16rhs"] < (5e-3 if warm else ANGLE_TOL), w  # warm: from the first columns of the identity
