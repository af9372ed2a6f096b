"""Calls on a sorted batch that follow one another on ONE workspace, cleared once: whichever kernel the one before took, and
whatever it left in the workspace, the arrival counters of the next are zero.  Outputs are filled with NaN first and compared bit for
bit with what the same call gives on a workspace of its own."""
import itertools

import numpy as np
import pytest
import torch

import oracle
import moqe_workloads as wl

pytestmark = pytest.mark.gpu


class Layer:
    """A layer's experts (`specs`: bits, group, symmetric), input and, for some rows, the oracle's output."""

    def __init__(self, M, N, K, specs, ids):
        from gpu_helpers import bf16_to_torch, build_experts
        W = wl.weights_f32(f"shared/{N}/{K}", N, K)
        X = wl.activations_bf16(f"shared/{M}/{K}", M, K)
        self.shape, self.X = (M, N, K, len(specs)), bf16_to_torch(X)
        self.experts, What, _ = build_experts(W, specs)
        self.rows = np.unique(np.linspace(0, M - 1, 24).astype(int))
        self.ref = oracle.routed_gemm(X[self.rows], ids[self.rows], What)

    def size(self):
        import paper_2508_09204_b200 as moqe
        return moqe.moqe_routed_qgemm_workspace(*self.shape)

    def run(self, order, ws, path):
        import paper_2508_09204_b200 as moqe
        from gpu_helpers import dev, torch_to_bits
        Y = torch.full(self.shape[:2], float("nan"), dtype=torch.bfloat16, device=dev())
        moqe.moqe_routed_qgemm_sorted(self.X, *order, self.experts, Y, ws, path=path)
        assert moqe.moqe_async_status() == moqe.OK
        return torch_to_bits(Y)


def _workspace(layers):
    import paper_2508_09204_b200 as moqe
    ws = moqe.alloc_workspace(max(l.size() for l in layers))
    ws.fill_(0xFF)
    moqe.moqe_routed_qgemm_workspace_clear(ws, *layers[0].shape)
    return ws


def _check(M, E, ids, calls):
    """Every ordered pair of `calls` (layer, path) on one workspace."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_close, dev
    order = moqe.moqe_permute(None, torch.from_numpy(ids).to(dev()), E)[1:]
    layers = [l for l, _ in calls]
    alone = []
    for l, path in calls:
        alone.append(l.run(order, _workspace([l]), path))
        assert_close(alone[-1][l.rows], l.ref, f"path {path}")
    ws = _workspace(layers)
    for i, j in itertools.product(range(len(calls)), repeat=2):
        for k in (i, j):
            got = calls[k][0].run(order, ws, calls[k][1])
            assert np.array_equal(got, alone[k]), f"{calls[k][0].shape} path {calls[k][1]} (pair {i}, {j}): {(got != alone[k]).sum()} of {got.size} outputs"


@pytest.mark.parametrize("M,N,K,paths", [(16, 384, 2048, (0, 1, 2, 5)), (40, 512, 3584, (0, 1, 2, 3)), (60, 2400, 1152, (1, 2)), (300, 1000, 1024, (2, 4, 6))])
def test_every_kernel_after_every_other(M, N, K, paths):
    ids = np.random.default_rng(M).integers(0, 3, size=M).astype(np.int32)
    wide = Layer(M, N, K, [(8, 0, True), (4, 128, False), (3, 128, False)], ids)
    fine = Layer(M, N, K, [(8, 0, True), (4, 32, False), (3, 64, False)], ids)
    _check(M, 3, ids, [(wide, p) for p in paths] + [(fine, p) for p in paths if p != 5])


@pytest.mark.parametrize("M,N,K,specs,paths", [(21000, 256, 1024, ((4, 32, False), (4, 64, False)), (0, 0)),     # the automatic choice: dense weights, grouped
                                               (4800, 1024, 1024, ((4, 32, False), (4, 32, False)), (6, 2)),
                                               (40, 512, 3584, ((4, 64, False), (4, 128, False)), (0, 0))])     # ... streaming, grouped
def test_formats_of_the_same_shape(M, N, K, specs, paths):
    ids = np.zeros(M, np.int32)
    _check(M, 1, ids, [(Layer(M, N, K, [s], ids), p) for s, p in zip(specs, paths)])


def test_layers_of_different_shapes_above_64_rows():
    M = 300
    ids = (np.arange(M) % 2).astype(np.int32)
    specs = [(8, 0, True), (4, 32, False)]
    _check(M, 2, ids, [(Layer(M, 64, 256, specs, ids), 6), (Layer(M, 2304, 4096, specs, ids), 0), (Layer(M, 264, 640, specs, ids), 2)])
