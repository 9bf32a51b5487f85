"""GPU parity of the tcgen05 kernel (gemm_tc.cuh) where its variants meet: column tiles of 128 and 256, the edges of the
row paddings, narrow last tiles, deferred scales above 64 rows, both conversions, one and several clusters per tile.

Bound: |C - C_ref| <= 5e-3 * (|C_ref| + rms(C_ref)) per element, the bound of the layer.
"""
import numpy as np
import pytest

from paper_2408_11743_b200 import inputs
from gpu_util import DenseLayer, SparseLayer, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def marlin():
    import torch
    assert torch.cuda.is_available()
    import paper_2408_11743_b200 as m
    m.lib()
    return m


def _check(oracle_lib, C, C_ref):
    bad, worst, rms = oracle_lib.check_tolerance(C, C_ref)
    assert bad == 0, f"{bad} elements out of tolerance, worst ratio {worst:.3f}, rms {rms:.3f}"


# rows at the edges of the paddings (32, 64, 128, slabs); N of whole tiles, of a narrow last one, of 64 columns alone
@pytest.mark.parametrize("tile", ["128", "256"])
@pytest.mark.parametrize("M,K,N,G", [(17, 128, 256, 128), (32, 384, 512, 128), (33, 512, 320, -1), (64, 1024, 256, 128),
                                     (65, 640, 64, -1), (128, 2048, 768, 128), (129, 512, 1024, -1), (300, 256, 448, -1)])
def test_both_tile_widths_match_the_oracle_and_are_reproducible(marlin, oracle_lib, monkeypatch, tile, M, K, N, G):
    monkeypatch.setenv("MARLIN_B200_TC_TILE", tile)
    case = inputs.make_dense(M, K, N, G, seed=M + K + N)
    layer = DenseLayer(marlin, case.q_kpacked, case.S, case.G, max_M=M)
    C = layer(case.A)
    _check(oracle_lib, C, oracle_lib.gemm(case.A, case.q_kpacked, case.S, case.G))
    assert np.array_equal(layer(case.A).view(np.uint16), C.view(np.uint16))  # partial tiles are added in a fixed order


# deferred scales: N a multiple of 64 but not of 256
@pytest.mark.parametrize("M", [17, 33, 64, 65, 128, 129, 300])
@pytest.mark.parametrize("K,N,G", [(256, 64, 128), (1152, 448, 384), (2048, 1344, 128)])
def test_deferred_scales_at_every_row_padding(marlin, oracle_lib, M, K, N, G):
    case = inputs.make_dense(M, K, N, G, seed=M + K + N)
    C = DenseLayer(marlin, case.q_kpacked, case.S, G, max_M=M)(case.A)
    _check(oracle_lib, C, oracle_lib.gemm(case.A, case.q_kpacked, case.S, G))


# few column tiles and a long K: several clusters share a tile, their shares meet in the workspace
@pytest.mark.parametrize("M,K,N,G", [(20, 16384, 256, 128), (128, 16384, 512, 128), (48, 8192, 192, 128), (100, 12288, 320, -1)])
def test_several_clusters_per_tile(marlin, oracle_lib, M, K, N, G):
    case = inputs.make_dense(M, K, N, G, seed=M + N)
    layer = DenseLayer(marlin, case.q_kpacked, case.S, case.G, max_M=M)
    C = layer(case.A)
    _check(oracle_lib, C, oracle_lib.gemm(case.A, case.q_kpacked, case.S, case.G))
    assert np.array_equal(layer(case.A).view(np.uint16), C.view(np.uint16))


# the conversion with one fma per pair holds for scales up to 0.0624; larger, negative and zero ones among them
@pytest.mark.parametrize("sparse", [False, True])
@pytest.mark.parametrize("G", [128, 64, 32])
def test_scales_on_both_sides_of_the_short_conversion(marlin, oracle_lib, sparse, G):
    M, K, N = 40, 1024, 512
    case = (inputs.make_sparse24 if sparse else inputs.make_dense)(M, K, N, G, seed=G)
    rng = np.random.default_rng(G)
    S = case.S.copy()
    S[:, : N // 2] *= rng.choice(np.array([1, -1, 3, 40, 0], np.float16), size=(S.shape[0], N // 2))
    S[0, :4] = [0.0624, 0.0625, 0.06238, -0.0625]  # the last fp16 values on either side
    case.S = S
    if sparse:
        _check(oracle_lib, SparseLayer(marlin, case, M)(case.A),
               oracle_lib.gemm_sparse24(case.A, case.qc_kpacked, case.idx, S, G))
    else:
        _check(oracle_lib, DenseLayer(marlin, case.q_kpacked, S, G, max_M=M)(case.A), oracle_lib.gemm(case.A, case.q_kpacked, S, G))


# one scale per column on a large layer: the rows at which the two kernels change over, on either side of the size rule
@pytest.mark.parametrize("M", [8, 9, 16, 17])
@pytest.mark.parametrize("K,N", [(8192, 8192), (8192, 8256), (3072, 22016)])
def test_large_layers_with_one_scale_per_column_change_kernels_at_nine_rows(marlin, oracle_lib, M, K, N):
    case = inputs.make_dense(M, K, N, -1, seed=5 + M + N)
    layer = DenseLayer(marlin, case.q_kpacked, case.S, case.G, max_M=M)
    C = layer(case.A)
    bad, worst, rms = oracle_lib.check_tolerance(C, oracle_lib.gemm(case.A, case.q_kpacked, case.S, case.G))
    assert bad == 0, (bad, worst, rms)


# Finished tiles go to C through buffers of several blocks of eight rows: rows at the edges of a block, of a buffer (64) and of a
# slab, one tile per CTA and several, whole and narrow last tiles.  C lies in a larger buffer whose surroundings must survive.
@pytest.mark.parametrize("M,K,N,G,split", [
    (17, 256, 256, 128, "1"), (31, 256, 320, 128, "1"), (33, 256, 512, -1, "1"), (63, 384, 320, -1, "1"), (65, 256, 512, 128, "1"),
    (72, 256, 576, 128, "1"), (121, 512, 256, 64, "1"), (127, 256, 1344, 256, "1"), (137, 256, 768, 128, "1"),
    (250, 128, 320, 128, "1"), (300, 256, 12800, 128, None), (130, 128, 22016, -1, None), (200, 256, 10304, 128, None)])
@pytest.mark.parametrize("tile", ["128", "256"])
def test_every_row_of_c_and_nothing_else_is_written(marlin, oracle_lib, monkeypatch, tile, M, K, N, G, split):
    import torch
    monkeypatch.setenv("MARLIN_B200_TC_TILE", tile)
    if split:
        monkeypatch.setenv("MARLIN_B200_TC_SPLIT", split)
    rng = np.random.default_rng(M + N)
    Gn = K if G == -1 else G
    Q = rng.integers(0, 16, size=(K, N), dtype=np.uint8)
    A = rng.integers(-3, 4, size=(M, K)).astype(np.float16)
    S = np.ldexp(1.0, rng.integers(-4, 1, size=(K // Gn, N))).astype(np.float16)
    q = inputs.kpack(Q)
    layer = DenseLayer(marlin, q, S, G, max_M=M)
    guard = 64 * N
    big = torch.full((2 * guard + M * N,), float("nan"), dtype=torch.float16, device="cuda")
    out = big[guard:guard + M * N].view(M, N)
    marlin.gemm(to_dev(A), layer.w, layer.s, K, N, G, layer.ws, out=out)
    torch.cuda.synchronize()
    assert marlin.read_status(layer.ws) == 0
    want = (A.astype(np.float64) @ ((Q.astype(np.float64) - 8) * np.repeat(S.astype(np.float64), Gn, axis=0))).astype(np.float16)
    assert np.array_equal(to_host(out), want)  # integers times powers of two: every partial sum is exact
    assert bool(big[:guard].isnan().all()) and bool(big[guard + M * N:].isnan().all())


# the fused activation on the way out: H against silu(g) * u of the g and u that the same layer gives without it.  Bound: one
# rounding to fp16 (2^-11) and the fp32 exponential and division (below 2^-18 for |g| < 88): 2^-10.9 of |H|, and half of the smallest fp16.
@pytest.mark.parametrize("M,I,G", [(17, 128, 128), (40, 160, 128), (72, 672, 128), (121, 128, 64), (129, 256, -1), (250, 160, -1),
                                   (300, 6400, 128)])
def test_fused_activation_on_the_way_out(marlin, M, I, G):
    import torch
    K, N = 256, 2 * I
    case = inputs.make_dense(M, K, N, G, seed=M + I)
    layer = DenseLayer(marlin, case.q_kpacked, case.S, G, max_M=M)
    A = to_dev(case.A)
    C = to_host(marlin.gemm(A, layer.w, layer.s, K, N, G, layer.ws)).astype(np.float64).reshape(M, I // 8, 2, 8)
    guard = 64 * I
    big = torch.full((2 * guard + M * I,), float("nan"), dtype=torch.float16, device="cuda")
    H = big[guard:guard + M * I].view(M, I)
    marlin.gemm_swiglu(A, layer.w, layer.s, K, N, G, layer.ws, out=H)
    torch.cuda.synchronize()
    g, u = C[:, :, 0].reshape(M, I), C[:, :, 1].reshape(M, I)
    want = g / (1 + np.exp(-g)) * u
    err = np.abs(to_host(H).astype(np.float64) - want)
    assert np.all(err <= 2.0 ** -10.9 * np.abs(want) + 2.0 ** -25 + 1e-9)
    assert bool(big[:guard].isnan().all()) and bool(big[guard + M * I:].isnan().all())


# One scale per column: every CTA scales its exact integer sums, each product rounded to fp32, and the parts are added in worker order, each
# sum rounded; a product that entered a sum unrounded would show in about one result of 2^13.  k-ranges without clusters and stripes
# (a CTA adds onto its own part or goes through a slot, by who comes last), one cluster per tile, two.
@pytest.mark.parametrize("tile", ["128", "256"])
@pytest.mark.parametrize("split,cluster", [(3, 0), (0, 0), (3, 3), (4, 4), (4, 2)])
def test_scaled_parts_are_rounded_and_added_in_worker_order(marlin, monkeypatch, tile, split, cluster):
    import torch
    for k, v in (("TILE", tile), ("SPLIT", split), ("CLUSTER", cluster)):
        monkeypatch.setenv("MARLIN_B200_TC_" + k, str(v))
    M, K, N = 128, 3072, 4096
    rng = np.random.default_rng(split + cluster)
    Q = rng.integers(0, 16, size=(K, N), dtype=np.uint8)
    A = to_dev(rng.integers(-3, 4, size=(M, K)).astype(np.float16))
    S = (rng.random((1, N)) * 0.015 + 0.005).astype(np.float16)
    layer = DenseLayer(marlin, inputs.kpack(Q), S, -1, max_M=M)
    W, s = to_dev(Q).double() - 8, to_dev(S).float()
    KB, TN = K // 128, int(tile)
    tiles = N // TN
    workers = split * tiles if split else min(KB * tiles, torch.cuda.get_device_properties(0).multi_processor_count)
    cuts = {t * KB + r * KB // split for t in range(tiles) for r in range(split)} if split else {w * KB * tiles // workers for w in range(workers)}
    want = torch.empty(M, N, dtype=torch.float16, device="cuda")
    for t in range(tiles):
        col = slice(t * TN, (t + 1) * TN)
        edges = sorted({t * KB, (t + 1) * KB} | {c for c in cuts if t * KB < c < (t + 1) * KB})
        parts = []
        for u0, u1 in zip(edges, edges[1:]):
            k = slice((u0 - t * KB) * 128, (u1 - t * KB) * 128)
            parts.append((A[:, k].double() @ W[k, col]).float() * s[:, col])
        per = cluster if cluster > 1 else len(parts)
        shares = []
        for c in range(0, len(parts), per):
            shares.append(parts[c])
            for part in parts[c + 1:c + per]:
                shares[-1] = shares[-1] + part
        total = shares[0]
        for share in shares[1:]:
            total = total + share
        want[:, col] = total.half()
    for _ in range(20):
        C = marlin.gemm(A, layer.w, layer.s, K, N, K, layer.ws)
        torch.cuda.synchronize()
        assert marlin.read_status(layer.ws) == 0
        assert torch.equal(C, want), int((C != want).sum())


# Every format at the edges of slabs, units of eight rows and instances, in clusters of every size, stripes and k-ranges without
# clusters.  Small integers times powers of two: every partial sum is exact, in any order.
@pytest.mark.parametrize("tile", ["128", "256"])
@pytest.mark.parametrize("fmt", ["column", "group", "zp", "sub", "w8", "w8-column", "sparse24", "sparse24-sub", "swiglu"])
def test_every_format_at_every_height_and_cluster_size(marlin, monkeypatch, fmt, tile):
    import torch
    monkeypatch.setenv("MARLIN_B200_TC_TILE", tile)
    K, N = 1024, 512
    G = K if "column" in fmt else 64 if "sub" in fmt else 128
    rng = np.random.default_rng(len(fmt))
    s = np.ldexp(1.0, rng.integers(-6, -2, size=(K // G, N))).astype(np.float16)
    S = np.repeat(s.astype(np.float64), G, axis=0)
    ws = marlin.new_workspace(400, K, N)
    if "w8" in fmt:
        Q = rng.integers(0, 256, size=(K, N), dtype=np.uint8)
        W = (Q - 128.0) * S
        layer = marlin.Layer(*marlin.pack_w8(to_dev(Q), to_dev(s), G), K, N, G, ws, w8=True)
    elif "sparse24" in fmt:
        case = inputs.make_sparse24(1, K, N, G, seed=3)
        codes = np.stack([(case.qc_kpacked >> np.uint32(4 * j)) & 15 for j in range(8)], axis=1).reshape(K // 2, N)
        W = np.zeros((K, N))
        np.put_along_axis(W.reshape(K // 4, 4, N), case.idx.reshape(K // 4, 2, N).astype(np.int64), codes.reshape(K // 4, 2, N) - 8.0, axis=1)
        W *= S
        w, meta, sp = marlin.pack_sparse24(to_dev(case.qc_kpacked), to_dev(case.idx), to_dev(s), G)
        layer = marlin.Layer(w, sp, K, N, G, ws, meta_packed=meta)
    else:
        Q = rng.integers(0, 16, size=(K, N), dtype=np.uint8)
        Z = rng.integers(0, 16, size=(K // G, N), dtype=np.uint8) if fmt == "zp" else np.full((K // G, N), 8, np.uint8)
        W = (Q - np.repeat(Z.astype(np.float64), G, axis=0)) * S
        packed = marlin.pack(to_dev(inputs.kpack(Q)), to_dev(s), G)
        z = {"z_packed": marlin.pack_zeros(to_dev(Z), K, N, G)} if fmt == "zp" else {}
        layer = marlin.Layer(*packed, K, N, G, ws, **z)
    W = torch.from_numpy(W).cuda()
    first = 17 if fmt in ("column", "group", "zp", "swiglu") else 1  # (below that the warp-level kernel)
    for M in [m for m in (1, 8, 9, 15, 16, 17, 24, 25, 32, 33, 40, 48, 49, 64, 65, 72, 80, 81, 97, 112, 113, 128, 130, 161, 225, 300) if m >= first]:
        A = to_dev(rng.integers(-2, 3, size=(M, K)).astype(np.float16))
        want = (A.double() @ W).half()
        for split, cluster in [(2, 8), (3, 8), (4, 8), (5, 8), (6, 8), (7, 8), (8, 8), (4, 2), (6, 3), (6, 2), (8, 4), (3, 0), (0, 0), (1, 8)]:
            monkeypatch.setenv("MARLIN_B200_TC_SPLIT", str(split))
            monkeypatch.setenv("MARLIN_B200_TC_CLUSTER", str(cluster))
            if fmt == "swiglu":
                H = marlin.gemm_swiglu(A, *packed, K, N, G, ws)
                c = want.double().view(M, N // 16, 2, 8)
                g, u = c[:, :, 0].reshape(M, N // 2), c[:, :, 1].reshape(M, N // 2)
                h = g / (1 + torch.exp(-g)) * u  # the bound of test_fused_activation_on_the_way_out
                assert bool(((H.double() - h).abs() <= 2.0 ** -10.9 * h.abs() + 2.0 ** -25 + 1e-9).all()), (M, split, cluster)
            else:
                assert torch.equal(layer(A), want), (M, split, cluster)
    torch.cuda.synchronize()
    assert marlin.read_status(ws) == 0
    assert bool((ws[256:] == 0).all())
