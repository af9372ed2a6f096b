"""GPU parity of the two-SM grouped GEMM at the sizes where its tiling can go wrong: batches one row either side of a
half tile and of a whole token tile, an odd number of 128-channel tiles, K below and just above a k-block, rows that are
consecutive in X (read as boxes), scattered (gathered) and mixed, and the split by k-blocks against whole tiles.

Tolerance: that of the routed product (bf16 output, fp32 sums), max relative error 1e-2, mean absolute error 2e-3.
"""
import numpy as np
import pytest

import oracle
import moqe_workloads as wl

pytestmark = pytest.mark.gpu

FORMATS = [(8, 0, True), (4, 128, False), (3, 64, False), (2, 32, True), (4, 0, False)]


def _ids(kind, M, E):
    g = np.random.default_rng(M * 31 + E)
    if kind == "scattered":
        return g.integers(0, E, size=M).astype(np.int32)
    if kind == "runs":                                       # long runs: whole boxes are consecutive rows of X
        return np.sort(g.integers(0, E, size=M)).astype(np.int32)
    return np.repeat(g.integers(0, E, size=(M + 44) // 45), 45)[:M].astype(np.int32)   # short runs: boxes straddle them


def _run(X, ids, gpu, path):
    import torch
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import dev, bf16_to_torch, torch_to_bits
    Y = torch.full((X.shape[0], gpu[0].N), float("nan"), dtype=torch.bfloat16, device=dev())
    moqe.moqe_routed_qgemm(bf16_to_torch(X), torch.from_numpy(ids).to(dev()), gpu, Y=Y, path=path)
    assert moqe.moqe_async_status() == moqe.OK
    return torch_to_bits(Y)


@pytest.mark.parametrize("kind", ["scattered", "runs", "short runs"])
@pytest.mark.parametrize("M,N,K", [(1, 8, 32), (127, 128, 64), (129, 136, 192), (257, 384, 1088), (640, 264, 640)])
def test_pair_kernel_edges(M, N, K, kind):
    from gpu_helpers import build_experts, assert_close
    specs = [f for f in FORMATS if f[1] == 0 or K % f[1] == 0]
    W = wl.weights_f32(f"pair/{N}/{K}", N, K)
    X = wl.activations_bf16(f"pair/{M}/{K}", M, K)
    gpu, What, _ = build_experts(W, specs)
    ids = _ids(kind, M, len(specs))
    ref = oracle.routed_gemm(X, ids, What)
    for path in (2, 3, 4):                                   # split by k-blocks; whole tiles of 128 and of 256 tokens
        assert_close(_run(X, ids, gpu, path), ref, f"path {path} {kind} M{M} N{N} K{K}")


def test_pair_kernel_split_is_deterministic_and_clears_its_counters():
    """One token tile of one expert, 40 k-blocks deep: every cluster holds a part of it; the parts are added in a fixed
    order (same bits every time) and the arrival counters come back to zero (calls on a sorted batch, whose workspace is
    cleared once, still complete)."""
    import torch
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import build_experts, assert_close, bf16_to_torch, dev, torch_to_bits
    M, N, K = 200, 256, 5120
    W = wl.weights_f32("pair/split", N, K)
    X = wl.activations_bf16("pair/split/X", M, K)
    gpu, What, _ = build_experts(W, [(4, 128, False)])
    ids = np.zeros(M, np.int32)
    first = _run(X, ids, gpu, 2)
    assert_close(first, oracle.routed_gemm(X, ids, What), "split")
    for _ in range(3):
        assert np.array_equal(_run(X, ids, gpu, 2), first)
    _, perm, offsets = moqe.moqe_permute(None, torch.from_numpy(ids).to(dev()), 1)
    ws = moqe.alloc_workspace(moqe.moqe_routed_qgemm_workspace(M, N, K, 1))
    ws.fill_(0xFF)
    moqe.moqe_routed_qgemm_workspace_clear(ws, M, N, K, 1)
    for _ in range(4):
        Y = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device=dev())
        moqe.moqe_routed_qgemm_sorted(bf16_to_torch(X), perm, offsets, gpu, Y, ws, path=2)
        assert moqe.moqe_async_status() == moqe.OK
        assert np.array_equal(torch_to_bits(Y), first)


@pytest.mark.parametrize("M,N,K", [(192, 19200, 64), (192, 19200, 128), (96, 9600, 640), (48, 6000, 1152)])
def test_steps_of_one_k_block(M, N, K):
    """64-token tiles take two k-blocks a step; here every step, or the last of every piece, has one, and a cluster has several
    tiles or pieces in a row: the dequant group without a k-block must not run ahead of the other.  Same bits every time."""
    from gpu_helpers import build_experts, assert_close
    W = wl.weights_f32(f"pair/{N}/{K}", N, K)
    X = wl.activations_bf16(f"pair/{M}/{K}", M, K)
    gpu, What, _ = build_experts(W, [(4, 64, False), (8, 0, True), (3, 0, False)])
    ids = (np.arange(M) % 3).astype(np.int32)
    first = _run(X, ids, gpu, 2)
    assert_close(first, oracle.routed_gemm(X, ids, What), f"odd steps M{M} N{N} K{K}")
    for _ in range(30):
        assert np.array_equal(_run(X, ids, gpu, 2), first)


@pytest.mark.parametrize("M,N,K,specs", [(300, 6016, 1408, FORMATS), (700, 6016, 1408, FORMATS), (700, 6000, 1024, [(4, 128, False)]), (300, 9600, 640, [(4, 32, False), (8, 64, True)]),
                                         (700, 6400, 384, [(8, 32, True)])])
def test_wide_tiles_split(M, N, K, specs):
    """Layers wide enough for the automatic choice to keep tiles of 128 and 256 tokens, and tiles left over that are split by k-blocks
    (the last shape: one tile, whose cost is that of three units); an odd number of 128-channel tiles among them."""
    from gpu_helpers import build_experts, assert_close
    W = wl.weights_f32(f"pair/{N}/{K}", N, K)
    X = wl.activations_bf16(f"pair/{M}/{K}", M, K)
    specs = [f for f in specs if f[1] == 0 or K % f[1] == 0]
    gpu, What, _ = build_experts(W, specs)
    ids = _ids("short runs", M, len(specs))
    first = _run(X, ids, gpu, 2)
    assert_close(first, oracle.routed_gemm(X, ids, What), f"wide M{M} N{N} K{K}")
    for _ in range(3):
        assert np.array_equal(_run(X, ids, gpu, 2), first)


@pytest.mark.parametrize("M,N,K", [(40, 384, 8192), (33, 128, 2048), (64, 256, 640)])
def test_few_deep_tiles(M, N, K):
    """One to three tiles over all clusters, from many units to a share down to fewer than one cluster's four."""
    from gpu_helpers import build_experts, assert_close
    W = wl.weights_f32(f"pair/{N}/{K}", N, K)
    X = wl.activations_bf16(f"pair/{M}/{K}", M, K)
    gpu, What, _ = build_experts(W, [(8, 0, True), (4, 128, False), (3, 64, False)])
    for used in (1, 2, 3):
        ids = (np.arange(M) % used).astype(np.int32)
        assert_close(_run(X, ids, gpu, 2), oracle.routed_gemm(X, ids, What), f"deep M{M} N{N} K{K} {used}")
