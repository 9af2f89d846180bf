"""Rules by which the host layer deals work out (csrc/lordo_plan.h, compiled here on its own)."""
import ctypes as C
import os
import subprocess

import pytest

from paper_2602_04396_b200 import build as lbuild
from paper_2602_04396_b200 import lordo

WRAPPER = """
#include "lordo_plan.h"
extern "C" int deal(int n, const int* len, int workers, int split, int f32, int busy, int* seg, int* start, int* starts) {
  std::vector<lordo::WorkItem> items;
  for (int i = 0; i < n; ++i) items.push_back({i, i, len[i], (double)len[i]});
  std::vector<lordo::TcSeg> list;
  std::vector<int> st;
  lordo::deal_out(items, workers, split != 0, split ? lordo::kPieceHead : 0, f32 ? lordo::kMinPiece32 : lordo::kMinPiece, busy, list, st);
  if ((int)list.size() > n + workers || (int)st.size() > workers + 1) return -1;
  for (size_t i = 0; i < list.size(); ++i) { seg[3 * i] = list[i].prob; seg[3 * i + 1] = list[i].t0; seg[3 * i + 2] = list[i].t1; }
  for (size_t i = 0; i < st.size(); ++i) start[i] = st[i];
  *starts = (int)st.size();
  return (int)list.size();
}
extern "C" int split(int n, const int* slices, const int* tiles, int carry, int sms) {
  std::vector<lordo::ProductRun> runs;
  for (int i = 0; i < n; ++i) runs.push_back({slices[i], tiles[i]});
  const lordo::ProductSplit s = carry ? lordo::split_by_time(runs, sms) : lordo::split_by_turns(runs, sms);
  return 10 * s.rows + s.ctas;
}
extern "C" int factor(int panels, int matrices, const int* fits) { return lordo::factor_ctas(panels, matrices, fits); }
extern "C" int ranges(long long tiles, long long steps, long long most, long long pairs) { return lordo::k_ranges(tiles, steps, most, pairs); }
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, so = str(d / "plan.cpp"), str(d / "plan.so")
    with open(src, "w") as f:
        f.write(WRAPPER)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", lbuild.CSRC, "-o", so, src], check=True)
    lib = C.CDLL(so)
    lib.ranges.argtypes = [C.c_longlong] * 4
    lib.deal.argtypes = [C.c_int, C.c_void_p, C.c_int, C.c_int, C.c_int, C.c_int, C.c_void_p, C.c_void_p, C.c_void_p]
    return lib


MIN_PIECE, HEAD = 8, 4


# strips (count, 64-row steps); on 148 SMs: are strips cut, and the longest worker over the mean. One long strip, few long ones, two halves
# each, most of the SMs busy with whole strips, one turn and a bit, several turns, too short to cut, ragged
@pytest.mark.parametrize("strips,cut,most", [([(1, 2004)], True, 1.1), ([(6, 500)], True, 1.1), ([(1, 172)], True, 1.4), ([(74, 32)], True, 1.01),
                                             ([(40, 64)], True, 1.1), ([(100, 64)], True, 1.25), ([(120, 64)], False, 1.25), ([(128, 64)], False, 1.2),
                                             ([(156, 64)], True, 1.15), ([(64, 63)], True, 1.2), ([(2432, 32), (256, 88)], False, 1.05),
                                             ([(1, 7)], False, 1.0), ([(1, 15)], False, 1.0), ([(149, 9)], False, 2.0), ([(576, 12), (48, 48)], False, 1.1),
                                             ([(33, 16), (48, 9), (72, 8), (27, 11), (51, 3)], False, 1.25)])
@pytest.mark.parametrize("sms", [148, 40])
@pytest.mark.parametrize("split", [1, 0])
def test_strips_dealt_out(plan, strips, cut, most, sms, split):
    """Every step of every strip once, no piece below the shortest, at most strips + workers pieces (the room that the table has), and
    on 148 SMs the longest worker at most `most` times the mean, heads of pieces counted."""
    lens = [ln for count, ln in strips for _ in range(count)]
    workers = min(sms, max(len(lens), sum(lens) // MIN_PIECE))
    seg, start, starts = (C.c_int * (3 * (len(lens) + workers)))(), (C.c_int * (workers + 1))(), C.c_int()
    pieces = plan.deal(len(lens), (C.c_int * len(lens))(*lens), workers, split, 0, sms * 7 // 9, seg, start, C.byref(starts))
    assert 0 < pieces <= len(lens) + workers
    got = [(seg[3 * i], seg[3 * i + 1], seg[3 * i + 2]) for i in range(pieces)]
    at = [0] * len(lens)
    for prob, t0, t1 in sorted(got):
        assert t0 == at[prob] and t1 - t0 >= min(MIN_PIECE, lens[prob])
        at[prob] = t1
    assert at == lens and (split or pieces == len(lens))
    starts = list(start)[:starts.value]
    assert starts[0] == 0 and starts[-1] == pieces and starts == sorted(starts)
    if split and sms == 148:
        loads = [sum(t1 - t0 + HEAD for _, t0, t1 in got[a:b]) for a, b in zip(starts, starts[1:])]
        assert max(loads) <= most * sum(loads) / workers and (pieces > len(lens)) == cut


# fp32 storage: strips (count, 32-row steps), and the workers and the longest worker's steps at most on 148 SMs
@pytest.mark.parametrize("strips,workers,longest", [([(1, 34)], 17, 3), ([(10, 15)], 75, 3), ([(4, 44)], 88, 3), ([(1, 3)], 1, 3), ([(28, 4)], 56, 2),
                                                    ([(64, 64)], 148, 32), ([(149, 3)], 148, 6)])
def test_strips_of_fp32_storage_dealt_out(plan, strips, workers, longest):
    """Every step of every strip once, in pieces of two steps or more: few short strips reach as many SMs as their rows allow."""
    lens = [ln for count, ln in strips for _ in range(count)]
    most = min(148, max(len(lens), sum(lens) // 2))
    seg, start, starts = (C.c_int * (3 * (len(lens) + most)))(), (C.c_int * (most + 1))(), C.c_int()
    pieces = plan.deal(len(lens), (C.c_int * len(lens))(*lens), most, 1, 1, 148 * 7 // 9, seg, start, C.byref(starts))
    got = [(seg[3 * i], seg[3 * i + 1], seg[3 * i + 2]) for i in range(pieces)]
    at = [0] * len(lens)
    for prob, t0, t1 in sorted(got):
        assert t0 == at[prob] and t1 - t0 >= 2
        at[prob] = t1
    assert at == lens
    starts = list(start)[:starts.value]
    loads = [sum(t1 - t0 for _, t0, t1 in got[a:b]) for a, b in zip(starts, starts[1:])]
    assert len(loads) >= 0.8 * workers and max(loads) <= longest, loads


@pytest.mark.parametrize("rows", [8, 64, 520, 4096, 65536, 65600, 70000, 87424, 128256, 151936, 1 << 20])
@pytest.mark.parametrize("pairs_of_planes,most", [(2, 32), (3, 64)])  # Gram matrices, Rot
@pytest.mark.parametrize("tiles", [1, 2, 14, 64, 1000])
def test_a_range_of_k_has_at_most_64_steps(plan, rows, pairs_of_planes, most, tiles):
    """The bound up to which the truncating fp32 accumulation of a range is left alone, at vocabulary sizes as well."""
    steps = pairs_of_planes * ((rows + 63) // 64)
    ns = plan.ranges(tiles, steps, most, 74)
    longest = max(steps * (x + 1) // ns - steps * x // ns for x in range(ns))
    assert 1 <= longest <= 64
    assert ns <= max(most, (steps + 63) // 64)


@pytest.mark.parametrize("kw", [dict(), dict(variant=lordo.LOCAL, power_iters=1), dict(sides=(1, 0)), dict(oversample=8, power_iters=1), dict(time_buffer=1),
                                dict(check_mode=0), dict(w_dtype=lordo.BF16, g_dtype=lordo.BF16, e_dtype=lordo.BF16, check_mode=0)])
def test_every_product_is_one_that_its_kernel_takes(kw):
    """The plans of every kind of run at the least multiples of n, r (and m, projected from the right) that are accepted: extents and
    strides of the fp32 products' operands are multiples of four, the second product's operand lies as the first's. A plan
    that breaks this is refused."""
    m = 1000 if "sides" in kw else 1001
    cfg, _keep = lordo.make_config([(m, 72, 8), (129, 1336, 24)], 3, 2, **kw)
    assert lordo.query_workspace(cfg) > 0


def test_workspace_holds_the_ranges_of_tall_matrices():
    """The partial Gram matrices are sized by the same rule: more rows never need fewer of them."""
    def size(m, **kw):
        cfg, _keep = lordo.make_config([(m, 256, 256)], 1, 1, w_dtype=lordo.BF16, g_dtype=lordo.BF16, e_dtype=lordo.BF16, check_mode=0, **kw)
        return lordo.query_workspace(cfg)
    for m in (65536, 87360, 128256):
        assert size(m) < size(m + 64)


def test_workspace_of_the_kept_signal():
    """Local rule with iterations: the signal c G + E kept in bf16 lies where the new and the old basis are put after it, and nothing that
    only the fp32 path uses is set aside: at large ranks the workspace stays below 4.88 and 39.04 GB, what it took before the
    signal was kept; at small ones the signal's own 2 bytes per weight-replica are all that it adds."""
    def size(mats, K, q, ef=True):
        cfg, _keep = lordo.make_config(mats, K, 1, w_dtype=lordo.BF16, g_dtype=lordo.BF16, e_dtype=lordo.BF16, check_mode=0, variant=lordo.LOCAL,
                                       power_iters=q, error_feedback=ef)
        return lordo.query_workspace(cfg)
    big = (4096, 11008, 512)
    assert size([big], 16, 2) <= 4.88e9 and size([big] * 8, 16, 2) <= 39.04e9
    for m, n, r, K in ((2048, 2048, 64, 8), (7504, 3888, 168, 2), (200, 1112, 8, 1), (2048, 2048, 256, 8)):
        assert size([(m, n, r)], K, 1) - size([(m, n, r)], K, 1, ef=False) <= 2 * K * m * n


# launches of the fp32 products, (slices of k, tiles) in the order of the tiles, and what each split of them took, us: contractions of one
# length with few and with many tiles, and long ones among short ones
@pytest.mark.parametrize("runs,took", [
    ([(16, 8)], {41: 16.9, 42: 13.1, 44: 9.0, 48: 8.9, 81: 21.2, 82: 16.9, 84: 10.9, 88: 9.0}),
    ([(250, 64)], {41: 205.6, 42: 107.4, 44: 78.7, 48: 86.8, 81: 283.3, 82: 148.2, 84: 94.0, 88: 105.2}),
    ([(71, 264)], {41: 92.0, 42: 97.6, 44: 111.4, 48: 147.7, 81: 106.4, 82: 109.8, 84: 106.2, 88: 132.5}),
    ([(9, 3168)], {41: 196.3, 42: 273.7, 44: 527.8, 48: 1166.9, 81: 173.0, 82: 236.8, 84: 421.8, 88: 929.8}),
    ([(22, 9), (342, 18), (232, 2), (4, 62), (6, 95), (68, 3)], {41: 295.8, 42: 153.2, 44: 87.1, 48: 77.0, 81: 406.2, 82: 209.6, 84: 112.4, 88: 71.1}),
    ([(216, 1), (29, 177), (36, 12), (15, 2)], {41: 193.5, 42: 102.1, 44: 61.9, 48: 82.2, 81: 258.8, 82: 138.0, 84: 78.6, 88: 69.0}),
    ([(52, 57), (69, 184), (58, 156), (4, 1), (368, 3)], {41: 381.2, 42: 252.2, 44: 213.8, 48: 244.5, 81: 453.9, 82: 290.0, 84: 216.2, 88: 230.6}),
])
def test_fp32_products_split_by_time(plan, runs, took):
    """The split that the rule chooses took at most a tenth longer than the best."""
    n = len(runs)
    chosen = plan.split(n, (C.c_int * n)(*[s for s, _ in runs]), (C.c_int * n)(*[t for _, t in runs]), 1, 148)
    assert took[chosen] <= 1.1 * min(took.values()), chosen


@pytest.mark.parametrize("carry", [0, 1])
@pytest.mark.parametrize("sms", [148, 20])
def test_fp32_products_split_of_any_launch(plan, carry, sms):
    """A count that the longest contraction has two slices for, also at one slice, one tile and more tiles than are timed."""
    for runs in ([(1, 1)], [(1, 100000)], [(3, 7)], [(4, 1), (1, 1)], [(2, 50000), (400, 1), (3, 50000)], [(8, 3), (9, 3000000)]):
        n = len(runs)
        got = plan.split(n, (C.c_int * n)(*[s for s, _ in runs]), (C.c_int * n)(*[t for _, t in runs]), carry, sms)
        rows, ctas = got // 10, got % 10
        assert rows in ((4, 8) if carry else (4,)) and ctas in (1, 2, 4, 8) and (ctas == 1 or max(s for s, _ in runs) >= 2 * ctas)


# the cases of the factorisation's GPU test: CTAs per matrix on a B200 and row blocks of a CTA at most (up to four have a unit each, of which
# those left over help; with more, some blocks wait for a second batch, or with more than eight beside the diagonal's a third)
@pytest.mark.parametrize("r,count,ctas,blocks", [(8, 1, 1, 1), (32, 1, 1, 1), (40, 3, 1, 2), (256, 2, 4, 2), (264, 40, 3, 3), (504, 1, 8, 2), (296, 80, 1, 10),
                                                 (512, 75, 1, 16), (136, 3, 3, 2), (512, 16, 6, 3), (192, 148, 1, 6), (256, 60, 2, 4)])
def test_ctas_of_the_factorisation(plan, r, count, ctas, blocks):
    fits = (C.c_int * 9)(0, 148, 74, 45, 33, 26, 22, 15, 15)  # clusters of 0 to 8 CTAs that a B200 holds
    panels = (r + 31) // 32
    assert plan.factor(panels, count, fits) == ctas and (panels + ctas - 1) // ctas == blocks
