"""GPU parity of the tcgen05 kernel with deferred scales (gemm_tc.cuh, kDeferred: an accumulator per k-block, which the draining warps
scale and add up in fp32) through the C ABI: layers with group scales whose N is a multiple of 64 but not of 256, from 17 rows.

Run in the partition that the planner picks, in even stripes (tiles shared by CTAs, segments that end in the middle of a stripe)
and without clusters (partial tiles meet in the workspace); pipelines longer than the rings, every row padding, narrow last
tiles, zero points and the fused activation.

Bound: |C - C_ref| <= 5e-3 * (|C_ref| + rms(C_ref)) per element; integer-valued closed forms bit for bit.
"""
import numpy as np
import pytest

from paper_2408_11743_b200 import inputs
from gpu_util import DenseLayer, to_dev, to_host

pytestmark = pytest.mark.gpu

MODES = [{}, {"MARLIN_B200_TC_SPLIT": "0"}, {"MARLIN_B200_TC_CLUSTER": "0"}]


@pytest.fixture(scope="module")
def marlin():
    import torch
    assert torch.cuda.is_available()
    import paper_2408_11743_b200 as m
    m.lib()
    return m


@pytest.fixture(params=range(len(MODES)), ids=["planned", "even", "no_clusters"])
def mode(request, monkeypatch):
    for k, v in MODES[request.param].items():
        monkeypatch.setenv(k, v)


SHAPES = [(17, 256, 192, 128), (24, 1152, 384, 384), (32, 2048, 1088, 128), (33, 1024, 576, 128), (64, 4096, 4160, 128),
          (65, 2048, 64, 256), (100, 1024, 640, 512), (128, 8192, 320, 128), (150, 512, 384, 128), (300, 3072, 1344, 128),
          (20, 28672, 1088, 128)]


@pytest.mark.parametrize("M,K,N,G", SHAPES)
def test_tcd_kernel_matches_oracle_and_is_reproducible(marlin, oracle_lib, mode, M, K, N, G):
    case = inputs.make_dense(M, K, N, G, seed=3000 + M + K + N)
    layer = DenseLayer(marlin, case.q_kpacked, case.S, G, max_M=M)
    C = layer(case.A)
    bad, worst, rms = oracle_lib.check_tolerance(C, oracle_lib.gemm(case.A, case.q_kpacked, case.S, case.G))
    assert bad == 0, f"{bad} elements out of tolerance, worst ratio {worst:.3f}, rms {rms:.3f}"
    # partial tiles are added in a fixed order: the same bits on every call
    for _ in range(3):
        assert np.array_equal(layer(case.A).view(np.uint16), C.view(np.uint16))
    assert np.all(to_host(layer.ws[256:8192]) == 0)  # arrival counters left clean


@pytest.mark.parametrize("zero_points", [False, True])
@pytest.mark.parametrize("M,K,N,G", [(17, 4096, 320, 128), (32, 8192, 192, 128), (33, 1024, 1344, 256), (64, 2048, 576, 128),
                                     (128, 2048, 320, 256), (129, 1024, 192, 128), (300, 1024, 1344, 128)])
def test_tcd_integer_closed_form_is_bit_exact(marlin, mode, zero_points, M, K, N, G):
    # scales powers of two, activations small integers: every product and partial sum is exact in fp32, in any order
    import torch
    rng = np.random.default_rng(M + K)
    Q = rng.integers(0, 16, size=(K, N), dtype=np.uint8)
    A = rng.integers(-3, 4, size=(M, K)).astype(np.float16)
    S = np.ldexp(1.0, rng.integers(-4, 1, size=(K // G, N))).astype(np.float16)
    Z = rng.integers(0, 16, size=(K // G, N), dtype=np.uint8) if zero_points else np.full((K // G, N), 8, np.uint8)
    layer = DenseLayer(marlin, inputs.kpack(Q), S, G, max_M=M)
    if zero_points:
        z = marlin.pack_zeros(to_dev(Z), K, N, G)
        C = to_host(marlin.gemm_zp(to_dev(A), layer.w, layer.s, z, K, N, G, layer.ws))
        torch.cuda.synchronize()
        assert marlin.read_status(layer.ws) == 0
    else:
        C = layer(A)
    W = (Q.astype(np.float64) - np.repeat(Z, G, axis=0)) * np.repeat(S.astype(np.float64), G, axis=0)
    assert np.array_equal(C, (A.astype(np.float64) @ W).astype(np.float16))


@pytest.mark.parametrize("M", [17, 32, 64, 128, 300])
def test_tcd_one_hot_rows_probe_every_k_position(marlin, mode, M):
    K, N, G = 512, 320, 128
    rng = np.random.default_rng(50 + M)
    Q = rng.integers(0, 16, size=(K, N), dtype=np.uint8)
    expo = rng.integers(-5, 2, size=(K // G, N))
    S = np.ldexp(1.0, expo).astype(np.float16)
    layer = DenseLayer(marlin, inputs.kpack(Q), S, G, max_M=M)
    W = (Q.astype(np.float64) - 8) * np.ldexp(1.0, np.repeat(expo, G, axis=0))
    for k0 in range(0, K, M):
        ks = (k0 + np.arange(M)) % K
        A = np.zeros((M, K), dtype=np.float16)
        A[np.arange(M), ks] = 1.0
        assert np.array_equal(layer(A).astype(np.float64), W[ks]), f"rows from {k0}"


def test_default_routing_uses_it_for_n_multiple_of_128_only(marlin, oracle_lib):
    # N = 384 (no whole 256-column tiles) at 40 rows: one launch of this kernel
    case = inputs.make_dense(40, 2048, 384, 128, seed=8)
    C = DenseLayer(marlin, case.q_kpacked, case.S, 128, max_M=40)(case.A)
    bad, worst, _ = oracle_lib.check_tolerance(C, oracle_lib.gemm(case.A, case.q_kpacked, case.S, 128))
    assert bad == 0, worst


# g = gate, u = up of the same layer without the fused activation: one more rounding to fp16 and the fp32 exponential and division
@pytest.mark.parametrize("M,I", [(17, 160), (64, 672), (128, 96)])
def test_tcd_fused_activation(marlin, mode, M, I):
    K, N = 1024, 2 * I
    case = inputs.make_dense(M, K, N, 128, seed=M + I)
    layer = DenseLayer(marlin, case.q_kpacked, case.S, 128, max_M=M)
    C = layer(case.A).astype(np.float64).reshape(M, I // 8, 2, 8)
    g, u = C[:, :, 0].reshape(M, I), C[:, :, 1].reshape(M, I)
    H = to_host(marlin.gemm_swiglu(to_dev(case.A), layer.w, layer.s, K, N, 128, layer.ws)).astype(np.float64)
    want = g / (1 + np.exp(-g)) * u
    assert np.all(np.abs(H - want) <= 2.0 ** -10.9 * np.abs(want) + 2.0 ** -24)


@pytest.mark.parametrize("M,K,N", [(17, 4096, 2752), (64, 2048, 4160), (128, 4096, 1344), (200, 1024, 5504)])
def test_tcd_long_stream_of_overlapping_launches_is_stable(marlin, mode, M, K, N):
    import torch
    case0 = inputs.make_dense(M, K, N, 128, seed=5)
    case1 = inputs.make_dense(M, K, N, 128, seed=6)
    layer = DenseLayer(marlin, case0.q_kpacked, case0.S, 128, max_M=M)
    A = [to_dev(case0.A), to_dev(case1.A)]
    want = []
    for a in A:
        want.append(to_host(marlin.gemm(a, layer.w, layer.s, K, N, 128, layer.ws)).copy())
        torch.cuda.synchronize()
    C = [torch.empty((M, N), dtype=torch.float16, device="cuda") for _ in range(2)]
    for rep in range(3):
        for c in C:
            c.fill_(float("nan"))
        for i in range(120):
            marlin.gemm(A[i % 2], layer.w, layer.s, K, N, 128, layer.ws, out=C[i % 2])
        torch.cuda.synchronize()
        assert marlin.read_status(layer.ws) == 0
        for i in range(2):
            assert np.array_equal(to_host(C[i]).view(np.uint16), want[i].view(np.uint16)), f"repetition {rep}, buffer {i}"
