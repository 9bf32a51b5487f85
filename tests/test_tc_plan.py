"""The planner of the tcgen05 kernel (csrc/tc_plan.h), compiled by itself and asked on the host: every plan is one that the
kernel can run, and on layers whose candidates were all timed on a B200 it picks one of the fastest."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DENSE4, SPARSE4, DENSE8, DEFERRED4, ZERO4 = range(5)
RESIDENT = [0, 148, 74, 45, 33, 26, 22, 15, 15]  # clusters of that size that a B200 holds at once

SHIM = """
#include "tc_plan.h"
extern "C" void plan(int format, int M, int kb, int N, int sms, int most, long long* out) {
  const marlin_b200::TcPlan p = marlin_b200::plan_tc(format, M, kb, N, sms, most);
  out[0] = p.nt; out[1] = p.whole; out[2] = p.split; out[3] = p.cluster; out[4] = p.workers; out[5] = p.ncols;
}
extern "C" int slab_rows(int format, int M, int nt) { return marlin_b200::tc_slab_rows(format, M, nt); }
"""


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "shim.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2408_11743_b200", "csrc"),
                    str(d / "shim.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.fixture(scope="module")
def plan(shim):
    def ask(fmt, M, K, N, sms=148, most=160):
        out = (ctypes.c_longlong * 6)()
        shim.plan(fmt, M, K // 128, N, sms, most, out)
        return dict(zip(("nt", "whole", "split", "cluster", "workers", "ncols"), out))
    return ask


@pytest.mark.parametrize("fmt", [DENSE4, SPARSE4, DENSE8, DEFERRED4, ZERO4])
@pytest.mark.parametrize("env", [{}, {"MARLIN_B200_TC_SPLIT": "0"}, {"MARLIN_B200_TC_SPLIT": "3"}, {"MARLIN_B200_TC_CLUSTER": "0"},
                                 {"MARLIN_B200_TC_TILE": "256"}])
def test_every_plan_can_run(plan, monkeypatch, fmt, env):
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    rng = random.Random(fmt)
    for _ in range(400):
        M = rng.choice([1, 16, 17, 32, 33, 64, 65, 128, 129, 1000, 4096, rng.randint(1, 5000)])
        K, N = 128 * rng.randint(1, 256), (64 if fmt in (DENSE4, DEFERRED4) else 256) * rng.randint(1, 112)
        sms = rng.choice([148, 148, 132, 7, 1])
        p = plan(fmt, M, K, N, sms)
        mpad = 32 if M <= 32 else 64 if M <= 64 else 128
        kb, slabs = K // 128, -(-M // mpad)
        assert p["nt"] == 1 if fmt == DEFERRED4 else p["nt"] in (1, 2)
        assert p["ncols"] == -(-N // (128 * p["nt"])) * slabs
        assert 1 <= p["workers"] <= min(sms, 160, p["ncols"] * kb)
        if p["split"]:
            assert p["split"] <= kb and p["workers"] == p["split"] * p["ncols"] and p["split"] % p["cluster"] == 0
            assert p["cluster"] == 1 or p["workers"] <= RESIDENT[p["cluster"]] * p["cluster"]
        else:
            assert p["cluster"] == 0
        if p["whole"]:
            assert not p["split"] and p["ncols"] >= p["workers"]


# (format, rows, K, N): candidates within 5 % of the fastest as (128-column tiles, form), the form a number of k-ranges, "whole"
# tiles or "even" stripes.  Behind them the times of what the constants from a dozen shapes had picked and of the best, in us.
# (Timed when the constants were fitted.  On the kernel as it is now the picks are within 2 % of the fastest but for zero points at 200 and 22 rows, 6 and
# 10 % above other stripes, and 2:4 at one row of 4096 x 22016, 8 % above one k-range per tile.)
@pytest.mark.parametrize("fmt,M,K,N,good", [
    (SPARSE4, 200, 1536, 24576, {(1, "whole")}),           # 22.1 / 15.7
    (SPARSE4, 64, 4096, 22016, {(2, 1)}),                  # 17.4 / 12.7
    (DENSE4, 512, 17408, 1536, {(1, 3)}),                  # 38.0 / 29.7
    (DENSE4, 48, 28672, 8192, {(2, 4)}),                   # 44.6 / 36.7
    (DENSE4, 48, 4096, 12288, {(1, 1), (2, 2)}),           # 15.2 / 12.7
    (DENSE4, 48, 5120, 13824, {(1, 1), (2, 2)}),           # 17.6 / 15.1
    (DENSE4, 129, 8192, 8192, {(1, 1)}),                   # 36.5 / 31.0
    (DENSE4, 17, 1024, 4096, {(1, 1), (1, 2)}),            # 5.4 / 4.6
    (DENSE4, 160, 4096, 4096, {(1, 2)}),                   # 13.6 / 11.8
    (DENSE8, 64, 4096, 12288, {(1, 1)}),                   # 16.5 / 13.2
    (DENSE8, 1, 17408, 1536, {(1, 8)}),                    # 12.2 / 9.8
    (DENSE8, 32, 2048, 8192, {(1, 1), (1, 2)}),            # 8.1 / 7.0
    (DENSE8, 2048, 2048, 1280, {(1, "whole"), (2, 1)}),    # 18.6 / 16.5
    (DENSE8, 2300, 8192, 8192, {(2, "whole")}),            # 352 / 310
    (SPARSE4, 384, 1024, 4096, {(1, 1)}),                  # 7.8 / 6.4
    (SPARSE4, 128, 4096, 4096, {(1, 4), (1, 3)}),          # 10.1 / 9.1
    (DEFERRED4, 160, 1024, 14400, {(1, "whole")}),         # 17.7 / 15.8
    (DEFERRED4, 24, 4096, 2752, {(1, 4)}),                 # 7.0 in 22 clusters of six / 6.8
    (DENSE4, 2, 4096, 5632, {(2, 4)}),                     # 8.5 / 8.0, likewise
    (DEFERRED4, 24, 4096, 1344, {(1, 6)}),                 # half as many clusters of six: 5.7, 6.2 with four
    (ZERO4, 200, 5120, 13824, {(1, "whole")}),             # 42.3 / 38.8 with the k-blocks of DENSE4
    (SPARSE4, 1, 4096, 22016, {(2, "even")}),              # 14.7 / 12.5 with the k-blocks of more rows
    (SPARSE4, 1, 2048, 8192, {(2, 2)}),                    # 6.2 / 5.6
    (ZERO4, 22, 4096, 22016, {(2, "even")}),               # 19.5 / 18.1
    (ZERO4, 777, 11008, 4096, {(1, "whole"), (1, "even")}),  # 86.8 / 80.7
])
def test_picks_among_the_fastest_of_the_timed_candidates(plan, fmt, M, K, N, good):
    p = plan(fmt, M, K, N)
    assert (p["nt"], p["split"] or ("whole" if p["whole"] else "even")) in good


@pytest.mark.parametrize("fmt", [DENSE4, SPARSE4, DENSE8, DEFERRED4, ZERO4])
def test_slabs_cover_every_batch(shim, fmt):
    for M in list(range(1, 3000)) + [4095, 4096, 4097, 65535, 70000]:
        mpad = 32 if M <= 32 else 64 if M <= 64 else 128
        slabs = -(-M // mpad)
        for nt in (1, 2):
            rows = shim.slab_rows(fmt, M, nt)
            assert rows % 16 == 0 and rows <= mpad  # the MMA's N; the instance's stages and accumulators
            assert (slabs - 1) * rows < M <= slabs * rows  # all rows, no empty slab
            # the heights that the issuers have loops for; the planner counts on one height for both tile widths where there are several slabs
            assert rows in ({16, 32} if mpad == 32 else {64} if mpad == 64 else {80, 96, 112, 128})
            assert rows == mpad or (fmt != DEFERRED4 and (mpad == 128 or (M <= 16 and nt == 2)))
        assert slabs == 1 or shim.slab_rows(fmt, M, 1) == shim.slab_rows(fmt, M, 2)
