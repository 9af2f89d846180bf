"""Rules by which the host layer deals work out (csrc/lordo_plan.h, compiled here on its own)."""
import ctypes as C
import os
import subprocess

import pytest

from paper_2602_04396_b200 import build as lbuild
from paper_2602_04396_b200 import lordo

WRAPPER = """
#include "lordo_plan.h"
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
    return lib


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
