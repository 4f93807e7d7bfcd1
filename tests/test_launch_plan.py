"""How kernel 1's launches are divided, for devices other than the one at hand: the plan is plain C++, compiled here.

Cluster sizes above 8 are not portable: a device (or a partition of one) may be unable to launch them, and then a plan must not
ask for one.  Whatever the plan, its shared memory stays within the limit that is set once per layer.
"""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_27003_b200", "csrc")
SHIM = """
#include "quantize_plan.h"
extern "C" void plan(int M, int G, int r, int sms, const int* fitting, int wide, int image, int* out) {
  const w4a4::QuantizePlan p = w4a4::quantize_plan(M, G, r, sms, fitting, wide, static_cast<size_t>(image));
  out[0] = p.steps, out[1] = p.warps, out[2] = p.splits;
  out[3] = static_cast<int>(w4a4::quantize_smem_bytes(r, p.steps, p.warps, p.splits));
  out[4] = static_cast<int>(w4a4::quantize_smem_bytes(r, p.steps, w4a4::kQuantWarps, w4a4::kMaxKSplits));
  out[5] = w4a4::quantize_rows(p.steps, p.warps), out[6] = p.spare;
}
"""
FULL = [0, 0, 74, 45, 33, 26, 22, 15, 15]   # clusters of 2 .. 8 that fit a whole B200, one CTA to an SM
ROWS = [1, 7, 8, 9, 63, 64, 65, 200, 448, 449, 700, 896, 897, 1024, 1025, 1560, 2048, 4352, 4353, 9300, 32760, 75600]
GROUPS = [1, 2, 3, 4, 8, 9, 16, 31, 32, 33, 80, 216, 256]


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, lib = d / "plan.cpp", d / "plan.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, "-o", str(lib), str(src)], check=True)
    fn = ctypes.CDLL(str(lib)).plan

    def call(M, G, r, sms=148, fitting=FULL, wide=7, int4=True, image=1 << 22):
        out = (ctypes.c_int * 7)()
        fn(M, G, r, sms, (ctypes.c_int * 9)(*fitting), wide, image if int4 else 0, out)
        return dict(zip(("steps", "warps", "splits", "smem", "limit", "rows", "spare"), out))
    return call


@pytest.mark.parametrize("fitting,wide,most", [
    (FULL, 7, 16),
    (FULL, 0, 8),                                    # no GPC offers 16 SMs
    ([0, 0, 8, 4, 4, 0, 0, 0, 0], 0, 4),             # a partition with GPCs of four or five SMs
    ([0] * 9, 0, 1),                                 # no clusters at all
])
def test_a_plan_asks_for_no_cluster_that_the_device_cannot_launch(plan, fitting, wide, most):
    for M in ROWS:
        for G in GROUPS:
            for r in (16, 32, 64, 96):
                for int4 in (False, True):
                    p = plan(M, G, r, fitting=fitting, wide=wide, int4=int4)
                    assert 1 <= p["splits"] <= most and p["splits"] <= max(1, G // 2), (M, G, r, int4, p)
                    assert p["splits"] == 1 or (wide if p["splits"] > 8 else fitting[p["splits"]]) > 0, (M, G, r, int4, p)


def test_every_plan_stays_within_the_limits_set_at_pack_time(plan):
    for M in ROWS:
        for G in GROUPS:
            for r in (0, 16, 32, 64, 96):
                for int4 in (False, True):
                    p = plan(M, G, r, int4=int4)
                    assert p["steps"] in (2, 4) and 1 <= p["warps"] <= p["warps"] + p["spare"] <= 8 and 1 <= p["splits"] <= max(1, G), (M, G, r, int4, p)
                    assert p["smem"] <= p["limit"] <= 232448, (M, G, r, int4, p)
                    assert p["rows"] <= 128


@pytest.mark.parametrize("M", [6000, 9600, 12000, 14000])
@pytest.mark.parametrize("int4", [False, True])
def test_the_middle_of_the_range_fills_the_machine(plan, M, int4):
    # A warp's chain takes about eight warps' issue time, so fewer than that per SM leave it waiting; two CTAs fit.
    p = plan(M, 216, 16, int4=int4)
    assert -(-M // p["rows"]) * p["splits"] * p["warps"] >= 8 * 148, p


@pytest.mark.parametrize("r", [16, 32, 64, 96])
def test_the_model_keeps_the_plan_of_full_launches(plan, r):
    # 293 CTAs of seven warps, two to an SM, in one wave.
    for int4 in (False, True):
        p = plan(32760, 80, r, int4=int4)
        assert (p["steps"], p["warps"], p["splits"]) == (4, 7, 1), p


@pytest.mark.parametrize("G", [8, 16, 80, 216])
def test_few_rows_leave_enough_warps_for_the_weight_expansion(plan, G):
    # The CTAs that expand weights have the plan's warps: with one or two each, a large layer's expansion took twice its time.
    for M in (1, 8, 16, 64, 130, 300, 448):
        p = plan(M, G, 16, image=5120 * 5120)
        assert 6 <= p["warps"] + p["spare"] <= 8 and (M <= 256 or p["splits"] <= 8)
        assert plan(M, G, 16, image=1024 * 1024)["spare"] == 0


@pytest.mark.parametrize("M", [2000, 6000, 12000, 20000])
def test_without_a_low_rank_branch_every_sm_gets_several_ctas(plan, M):
    p = plan(M, 216, 0)
    assert -(-M // p["rows"]) * p["splits"] >= 4 * 148, p
