"""The planner of the warp-level kernel (csrc/dense_plan.h), compiled by itself: the partition that a launch takes, worker by worker
with the kernel's own formulas."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = """
#include "dense_plan.h"
extern "C" void plan(int mb, int sparse, int kb, int N, int most, int teams_too, int* out) {
  const marlin_b200::DensePartition p = marlin_b200::plan_dense(mb, sparse != 0, kb, N, most, teams_too != 0);
  out[0] = p.nw; out[1] = p.ncols; out[2] = p.split; out[3] = p.teams; out[4] = p.workers; out[5] = p.cw;
}
extern "C" unsigned first_tile(unsigned t, unsigned tiles, unsigned extra) { return marlin_b200::team_first_tile(t, tiles, extra); }
"""
SHAPES = [(4096, 4096), (8192, 8192), (4096, 12288), (4096, 22016), (11008, 4096), (8192, 57344), (28672, 8192), (28672, 1024),
          (128, 64), (256, 192), (256, 64 * 149), (384, 128 * 150), (1280, 64 * 222), (1152, 128 * 172), (2048, 1024), (1024, 1024)]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "shim.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2408_11743_b200", "csrc"),
                    str(d / "shim.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


def _plan(lib, mb, sparse, K, N, sms, teams_too=True):
    out = (ctypes.c_int * 6)()
    lib.plan(mb, int(sparse), K // 128, N, sms, int(teams_too), out)
    return dict(zip(("nw", "ncols", "split", "teams", "workers", "cw"), out))


def _bounds(lib, p, kb):
    """First unit of every worker, and the end, as the kernel computes them."""
    U, P, S = p["ncols"] * kb, p["workers"], p["split"]
    if not S:
        return [w * U // P for w in range(P + 1)]
    tiles, extra = divmod(p["ncols"], p["teams"])
    b = []
    for w in range(P):
        team, rank = divmod(w, S)
        c0 = lib.first_tile(team, tiles, extra)
        units = (lib.first_tile(team + 1, tiles, extra) - c0) * kb
        b.append(c0 * kb + rank * units // S)
    assert lib.first_tile(p["teams"], tiles, extra) == p["ncols"]
    return b + [U]


@pytest.mark.parametrize("K,N", SHAPES)
@pytest.mark.parametrize("mb", [1, 2])
@pytest.mark.parametrize("sms", [148, 132, 7])
@pytest.mark.parametrize("nw", [None, "1", "2"])
def test_the_launched_partition_covers_every_unit_once(lib, monkeypatch, K, N, mb, sms, nw):
    if nw:
        monkeypatch.setenv("MARLIN_B200_NW", nw)
    kb = K // 128
    for sparse in (False, True):
        p = _plan(lib, mb, sparse, K, N, sms)
        assert p["nw"] in (1, 2, 4) and p["ncols"] * 64 * p["nw"] == N and 1 <= p["workers"] <= min(sms, p["ncols"] * kb)
        assert p["cw"] == 8 or (p["cw"] == 12 and mb == 1 and not sparse and p["nw"] == 2)
        if p["split"]:
            assert p["workers"] == p["split"] * p["teams"] and 1 <= p["teams"] <= p["ncols"]
            assert p["teams"] == p["ncols"] or p["split"] <= 2  # several tiles: whole ones, or pairs of CTAs
        b = _bounds(lib, p, kb)
        assert b[0] == 0 and b[-1] == p["ncols"] * kb and all(x < y for x, y in zip(b, b[1:]))
        if p["split"]:
            for w in range(p["workers"]):
                # a tile that is cut stays inside one team, and whoever has its beginning has it as the last of his tiles: the
                # exchange buffer of a CTA receives the partial tiles of that one alone
                if w % p["split"] == 0:
                    assert b[w] % kb == 0
                first, last = b[w] // kb, (b[w + 1] - 1) // kb
                for tile in range(first, last):
                    assert b[w + 1] >= (tile + 1) * kb


@pytest.mark.parametrize("K,N,split,teams", [
    (4096, 22016, 2, 58),   # pairs with two or three 128-column tiles: 13.2 us, 14.0 in even stripes on 148 SMs
    (8192, 1024, 4, 16),    # 64 CTAs let the next launch start beside them: 4.1 us, 5.5 with nine k-ranges
    (4096, 12288, 1, 96),   # whole tiles: 8.4 us, 9.2 with three k-ranges of 256 columns
])
def test_teams_where_they_were_measured_faster(lib, K, N, split, teams):
    p = _plan(lib, 1, False, K, N, 148)
    assert (p["split"], p["teams"]) == (split, teams)


@pytest.mark.parametrize("K,N", SHAPES)
def test_plan_stripes_reports_the_base_form(lib, K, N):
    from paper_2408_11743_b200 import build
    build.build()
    import paper_2408_11743_b200 as m
    for M in (1, 16):
        n_tile, workers, _ = m.plan_stripes(M, K, N, 148)
        p = _plan(lib, 1 if M <= 8 else 2, False, K, N, 148, teams_too=False)
        assert (n_tile, workers) == (64 * p["nw"], p["workers"])
