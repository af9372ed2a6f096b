"""Grouped GEMM: token rows that come in boxes, that are gathered, or both in one tile; a routing that differs from the one whose
offset table is still in the workspace; the hand-over of packed tiles."""
import numpy as np
import pytest
import torch

import oracle
import moqe_workloads as wl

pytestmark = pytest.mark.gpu


def _rows(M):
    return np.unique(np.concatenate([np.linspace(0, M - 1, 40).astype(int), [0, M - 1]]))


def _channels(N):
    """The ends of every tile of 128 channels, and some in between."""
    return np.unique(np.concatenate([np.arange(0, N, 128), np.minimum(np.arange(127, N + 127, 128), N - 1), np.arange(0, N, 61)]))


def _ids(M, runs, E):
    ids, e, i = np.zeros(M, np.int32), 0, 0
    while i < M:
        n = runs[e % len(runs)]
        ids[i:i + n] = e % E
        i, e = i + n, e + 1
    return ids


def _check(M, N, K, ids, specs, path, what):
    """Every row of a product that starts from NaN, at _channels(N)."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_close, bf16_to_torch, build_experts, dev, torch_to_bits
    W, X = wl.weights_f32(f"tcrows/{N}/{K}", N, K), wl.activations_bf16(f"tcrows/{M}/{K}", M, K)
    experts, What, _ = build_experts(W, specs)
    Y = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device=dev())
    moqe.moqe_routed_qgemm(bf16_to_torch(X), torch.from_numpy(ids).to(dev()), experts, Y=Y, path=path)
    assert moqe.moqe_async_status() == moqe.OK and not bool(Y.isnan().any())
    c = _channels(N)
    assert_close(torch_to_bits(Y)[:, c], oracle.routed_gemm(X, ids, [w[c] for w in What]), what)


TILES = {2: "64 tokens", 3: "128 tokens", 4: "256 tokens"}     # (2: the automatic choice, which takes 64 where there are so few channels)


@pytest.mark.parametrize("path", TILES)
@pytest.mark.parametrize("specs", [((8, 0, True), (4, 128, False), (3, 64, False)), ((4, 32, False), (2, 128, True))])
@pytest.mark.parametrize("M", [70, 150, 300, 500, 780])
@pytest.mark.parametrize("runs", [(1,), (8, 9), (100, 31, 5), (4000,)])
def test_runs_of_rows(M, runs, specs, path):
    """Runs of one row are gathered, runs that cover a half tile come in one box (of 9 rows and more), others leave pieces that are
    gathered as a whole; tiles of 64, 128 and 256 tokens."""
    _check(M, 200, 384, _ids(M, runs, len(specs)), specs, path, f"runs {runs}, {TILES[path]}")


@pytest.mark.parametrize("specs", [((8, 0, True), (4, 128, False), (3, 64, False)), ((4, 0, False), (2, 32, True))])
@pytest.mark.parametrize("M", [150, 200, 440, 900])
@pytest.mark.parametrize("runs", [(1,), (100, 31, 5), (300, 1, 2), (4000,)])
def test_several_pieces_to_a_cluster(M, runs, specs):
    """24 pairs of channel tiles and 9 k-blocks: two and more pieces to each of 74 clusters (the automatic choice keeps 64, 128 and 256
    tokens for these batches), some in boxes and some gathered, whole tiles and parts; the ring of four token stages wraps."""
    _check(M, 6008, 1152, _ids(M, runs, len(specs)), specs, 2, f"runs {runs}")


@pytest.mark.parametrize("M", [200, 900])
def test_several_pieces_with_ragged_k(M):
    _check(M, 6008, 1160, _ids(M, (300, 1, 40), 2), ((8, 0, True), (3, 0, False)), 2, "ragged k")


@pytest.mark.parametrize("K", [72, 136, 328])
@pytest.mark.parametrize("run", [1, 64])
def test_ragged_k(K, run):
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_close, bf16_to_torch, build_experts, dev, torch_to_bits
    M, N = 200, 136
    W, X = wl.weights_f32(f"tcrows/{N}/{K}", N, K), wl.activations_bf16(f"tcrows/{M}/{K}", M, K)
    experts, What, _ = build_experts(W, ((8, 0, True), (4, 0, False)))
    ids = (np.arange(M) // run % 2).astype(np.int32)
    Y = moqe.moqe_routed_qgemm(bf16_to_torch(X), torch.from_numpy(ids).to(dev()), experts, path=moqe.PATH_TCGEN05)
    assert moqe.moqe_async_status() == moqe.OK
    r = _rows(M)
    assert_close(torch_to_bits(Y)[r], oracle.routed_gemm(X[r], ids[r], What), f"K {K}")


@pytest.mark.parametrize("N,K", [(520, 512), (4104, 1152)])
def test_routing_changes_from_call_to_call(N, K):
    """The schedule is worked out ahead from the table that the call before left behind: other counts, experts without rows, and
    a smaller batch (whose table holds offsets beyond it).  520 channels: tiles of 64 tokens; 4104: of 64, 128 and 256, several pieces to
    a cluster."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_close, bf16_to_torch, build_experts, dev, torch_to_bits
    E = 3
    W = wl.weights_f32(f"tcrows/{N}/{K}", N, K)
    experts, What, _ = build_experts(W, ((8, 0, True), (4, 128, False), (3, 128, False)))
    g = np.random.default_rng(7)
    calls = []
    for M, p in ((900, (1, 0, 0)), (900, (0, 0.5, 0.5)), (400, (0, 0, 1)), (900, (0.1, 0.8, 0.1)), (130, (0.4, 0.3, 0.3)), (880, (0.3, 0.3, 0.4))):
        ids = g.choice(E, size=M, p=p).astype(np.int32)
        X = wl.activations_bf16(f"tcrows/{M}/{K}", M, K)
        calls.append((M, ids, X, bf16_to_torch(X), torch.from_numpy(ids).to(dev()), torch.full((M, N), float("nan"), dtype=torch.bfloat16, device=dev())))
    ws = moqe.alloc_workspace(max(moqe.moqe_routed_qgemm_workspace(c[0], N, K, E) for c in calls))
    for _ in range(3):
        for c in calls:
            moqe.moqe_routed_qgemm(c[3], c[4], experts, Y=c[5], workspace=ws, path=moqe.PATH_TCGEN05)
    assert moqe.moqe_async_status() == moqe.OK
    c = _channels(N)
    for M, ids, X, _, _, Y in calls:
        assert not bool(Y.isnan().any())
        assert_close(torch_to_bits(Y)[:, c], oracle.routed_gemm(X, ids, [w[c] for w in What]), f"{M} rows")


@pytest.mark.parametrize("spec", [(8, 0, True), (4, 128, False), (3, 64, False)])
def test_repeats_bit_for_bit(spec):
    """8192 rows x 11008 x 4096: every packed stage is refilled hundreds of times.  A stage handed back before its codes have been
    read shows as single channels that differ from run to run."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import dev
    M, N, K = 8192, 11008, 4096
    g = torch.Generator("cuda")
    g.manual_seed(1)
    e = [moqe.moqe_quantize_rtn(torch.randn((N, K), device=dev(), generator=g) * 0.02, *spec)]
    X = torch.randn((M, K), device=dev(), generator=g, dtype=torch.bfloat16)
    order = moqe.moqe_permute(None, torch.zeros(M, dtype=torch.int32, device=dev()), 1)[1:]
    ws = moqe.alloc_workspace(moqe.moqe_routed_qgemm_workspace(M, N, K, 1))
    moqe.moqe_routed_qgemm_workspace_clear(ws, M, N, K, 1)
    Y = [torch.empty((M, N), dtype=torch.bfloat16, device=dev()) for _ in range(4)]
    first = None
    for _ in range(6):
        for y in Y:
            moqe.moqe_routed_qgemm_sorted(X, *order, e, y, ws)
        first = Y[0].clone() if first is None else first
        assert all(torch.equal(y, first) for y in Y)
    assert moqe.moqe_async_status() == moqe.OK


@pytest.mark.parametrize("K,group,want", [(512, 64, "qgemm_tc_kernel"), (504, 0, "qgemm_dense_kernel"), (512, 32, "qgemm_dense_kernel")])
def test_many_rows_of_512_k(K, group, want):
    """31000 rows: 512 k without groups of 32 go to the grouped GEMM, 504 k and groups of 32 to the dense-weights one."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_close, bf16_to_torch, build_experts, dev, torch_to_bits
    M, N = 31000, 256
    W, X = wl.weights_f32(f"tcrows/{N}/{K}", N, K), wl.activations_bf16(f"tcrows/{M}/{K}", M, K)
    experts, What, _ = build_experts(W, ((8, 0, True), (4, group, False)))
    ids = (np.arange(M) // 196 % 2).astype(np.int32)
    assert moqe.moqe_routed_qgemm_kernel(M, experts) == want
    Y = moqe.moqe_routed_qgemm(bf16_to_torch(X), torch.from_numpy(ids).to(dev()), experts)
    assert moqe.moqe_async_status() == moqe.OK
    r = _rows(M)
    assert_close(torch_to_bits(Y)[r], oracle.routed_gemm(X[r], ids[r], What), f"K {K}")
