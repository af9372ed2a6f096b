"""Decode batches whose work split falls on segment boundaries (as many segments as CTAs, a few CTAs to a segment, several
segments to a CTA) and their neighbours whose split does not, with one to four experts in use and formats of unequal cost."""
import numpy as np
import pytest
import torch

import oracle
import moqe_workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(1, 256, 1152), (3, 4096, 512), (4, 9472, 256), (16, 9728, 384), (12, 12288, 256), (20, 18944, 128), (8, 264, 4096)])
def test_split_at_segment_ends(M, N, K):
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_close, bf16_to_torch, build_experts, dev, torch_to_bits
    W = wl.weights_f32(f"align/{N}/{K}", N, K)
    X = wl.activations_bf16(f"align/{M}/{K}", M, K)
    gpu, What, _ = build_experts(W, [(8, 0, True), (4, 128, False), (3, 128, False), (3, 64, False)])
    for used in ((0,), (0, 1, 2), (0, 1, 2, 3)):
        ids = np.array([used[i % len(used)] for i in range(M)], np.int32)
        ref = oracle.routed_gemm(X, ids, What)
        for _ in range(2):                                       # twice: the arrival counters come back to zero
            Y = moqe.moqe_routed_qgemm(bf16_to_torch(X), torch.from_numpy(ids).to(dev()), gpu)
            assert moqe.moqe_async_status() == moqe.OK
            assert_close(torch_to_bits(Y), ref, f"aligned M{M} N{N} K{K} {used}")
        # without the narrow groups: the other instantiation
        if 3 not in used:
            Y = moqe.moqe_routed_qgemm(bf16_to_torch(X), torch.from_numpy(ids).to(dev()), gpu[:3])
            assert_close(torch_to_bits(Y), ref, f"aligned M{M} N{N} K{K} {used}")


@pytest.mark.parametrize("M,N,K", [(8, 2304, 256), (5, 512, 2048), (24, 2048, 512), (4, 9472, 128), (4, 9728, 128)])
def test_one_super_tile_to_a_cta(M, N, K):
    """Fewer super-tiles than CTAs, as many and a few more, of formats whose costs are far apart: each piece of a segment is a
    single super-tile, and the formats' costs are left out of the split."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_close, bf16_to_torch, build_experts, dev, torch_to_bits
    W = wl.weights_f32(f"one/{N}/{K}", N, K)
    X = wl.activations_bf16(f"one/{M}/{K}", M, K)
    gpu, What, _ = build_experts(W, [(4, 0, False), (8, 32, True), (3, 64, False), (2, 32, True)])
    for experts in (range(4), range(1, 3), range(3, 4)):
        ids = np.array([experts[i % len(experts)] for i in range(M)], np.int32)
        ref = oracle.routed_gemm(X, ids, What)
        for _ in range(2):
            Y = moqe.moqe_routed_qgemm(bf16_to_torch(X), torch.from_numpy(ids).to(dev()), gpu)
            assert moqe.moqe_async_status() == moqe.OK
            assert_close(torch_to_bits(Y), ref, f"M{M} N{N} K{K} {experts}")
