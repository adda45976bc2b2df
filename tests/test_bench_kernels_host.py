"""Host-side accounting of bench.py (no GPU): the field kernel that it names follows the library's rules, and
the launches of a batched step the batch's work lists."""
import os
import re

import bench
from paper_2111_13072_gb300.inputs import Workload

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _kernel(n, **kw):
    kw = dict(dict(l_max=12, T_e_eV=2.0, n_e_m3=1e15, precision=1), **kw)
    return bench.field_kernel(Workload("w", N=n, **kw), n).split()[0]


def test_field_kernel_rule_matches_the_library():
    csrc = os.path.join(ROOT, "paper_2111_13072_gb300", "csrc")
    dev = open(os.path.join(csrc, "imrp_device.cuh")).read()
    assert "kPairMinN = int64_t(1) << 19;" in dev and bench.PAIR_MIN_N == 1 << 19
    assert re.search(r"kPairMinL = (\d+);", dev).group(1) == str(bench.PAIR_MIN_L)
    assert re.search(r"kImgInTileMaxN = (\d+);", dev).group(1) == str(bench.IMG_IN_TILE_MAX_N)
    assert "elem_size == 8 && (n + 1023) / 1024 < 100" in open(os.path.join(csrc, "imrp_internal.h")).read()
    assert (bench.FP64_SMALL_MOMENTS_MAX_N + 1023) // 1024 < 100 <= (bench.FP64_SMALL_MOMENTS_MAX_N + 1024) // 1024
    # (n, FP32 and FP64 with all m; the same with m = 0 alone)
    assert _kernel(1024) == "k_field_small" and _kernel(1025) == "k_field"
    assert _kernel((1 << 19) - 1) == "k_field" and _kernel(1 << 19) == "k_field_pair"
    assert _kernel(1 << 19, l_max=8) == "k_field"
    assert _kernel(1 << 19, m0_only=1) == "k_field" and _kernel(1000, m0_only=1) == "k_field_small"
    assert _kernel(1000, precision=0) == _kernel(1 << 20, precision=0) == "k_field_team"
    assert _kernel(1000, precision=0, m0_only=1) == _kernel(1 << 20, precision=0, m0_only=1) == "k_field"


def test_batched_launches():
    def ws(*cs):
        return [Workload("w", N=n, l_max=L, T_e_eV=2.0, n_e_m3=1e15, precision=p) for p, L, n in cs]
    assert bench.batched_launches(ws((1, 8, 10000), (1, 8, 900000))) == 2
    assert bench.batched_launches(ws((1, 12, 10000), (1, 12, 900000))) == 3  # k_field_batch and k_field_pair_batch
    assert bench.batched_launches(ws((1, 12, 900000), (1, 12, 800000))) == 2
    assert bench.batched_launches(ws((1, 12, 10000), (1, 16, 900000))) == 4
    assert bench.batched_launches(ws((0, 8, 10000), (0, 8, 20000))) == 2
    assert bench.batched_launches(ws((0, 8, 10000), (0, 8, 200000))) == 3  # both shapes of the moments
