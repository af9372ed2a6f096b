"""Batches of at most 32 rows on experts with groups of 32 and 64 k, beside wider formats: the edges of a token block (8, 16
rows of one expert), a last k-block that is only partly there, a ragged last channel tile, pieces split over many CTAs."""
import numpy as np
import pytest
import torch

import oracle
import moqe_workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("one", [False, True])
@pytest.mark.parametrize("M,N,K", [(1, 128, 64), (8, 200, 320), (9, 1000, 192), (16, 264, 1088), (17, 384, 640), (32, 128, 4096)])
def test_fine_groups(M, N, K, one):
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_close, bf16_to_torch, build_experts, dev, torch_to_bits
    specs = [(b, g, sym) for b in (8, 4, 3, 2) for g, sym in ((32, True), (32, False), (64, True), (64, False))] + [(8, 0, True), (3, 0, False)]
    if K % 128 == 0:
        specs.append((4, 128, False))
    W = wl.weights_f32(f"fine/{N}/{K}", N, K)
    X = wl.activations_bf16(f"fine/{M}/{K}", M, K)
    gpu, What, _ = build_experts(W, specs)
    turns = range(len(specs)) if one else range(2)               # every expert alone with all rows / spread over the experts
    for i in turns:
        ids = np.full(M, i, np.int32) if one else ((np.arange(M) * 5 + i) % len(specs)).astype(np.int32)
        before = moqe.moqe_launch_count()
        Y = moqe.moqe_routed_qgemm(bf16_to_torch(X), torch.from_numpy(ids).to(dev()), gpu)
        assert moqe.moqe_launch_count() > before and moqe.moqe_async_status() == moqe.OK
        assert_close(torch_to_bits(Y), oracle.routed_gemm(X, ids, What), f"fine M{M} N{N} K{K} {i}")


def test_fine_groups_take_the_whole_bf16_range():
    """Rows of 2^100, 2^-100 and ordinary size: the kernel multiplies fp16 tokens, so a row tile is divided by a power of two
    first (batches with such experts took any bf16 value before this kernel did them)."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_close, bf16_to_torch, build_experts, dev, torch_to_bits
    M, N, K = 24, 256, 2432
    W = wl.weights_f32("fine/range", N, K)
    gpu, What, _ = build_experts(W, [(3, 64, False), (4, 128, False), (8, 0, True)])
    for e in (100, -100, 0):
        X = torch.from_numpy(wl.activations_bf16("fine/range/X", M, K).view(np.int16)).view(torch.bfloat16)
        X = torch_to_bits(X * 2.0 ** e)
        ids = (np.arange(M) % 3).astype(np.int32)
        Y = moqe.moqe_routed_qgemm(bf16_to_torch(X), torch.from_numpy(ids).to(dev()), gpu)
        # (both sides are scaled back by the exact power of two before they are compared)
        back = lambda bits: torch_to_bits(torch.from_numpy(np.ascontiguousarray(bits).view(np.int16)).view(torch.bfloat16) * 2.0 ** -e)
        assert_close(back(torch_to_bits(Y)), back(oracle.routed_gemm(X, ids, What)), f"rows of 2^{e}")
    assert moqe.moqe_async_status() == moqe.OK


@pytest.mark.parametrize("bits,group,sym", [(8, 64, True), (8, 0, False), (4, 32, False), (4, 64, True), (4, 128, False), (3, 64, False), (3, 0, True),
                                            (2, 32, True), (2, 0, False)])
def test_sums_are_as_exact_as_the_streaming_kernels(bits, group, sym):
    """Codes enter the MMA with an offset that is taken out of the fp32 sums again, and the sums' error goes with its size.
    What shows of it is how many outputs are not the bf16 number nearest to the sum in 64 bits: no more than the streaming
    kernel has, which takes the same batches (plus three standard deviations of the two counts)."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import bf16_to_torch, dev
    M, N, K = 32, 2048, 3968
    W = torch.from_numpy(wl.weights_f32("fine/exact", N, K)).to(dev())
    X = bf16_to_torch(wl.activations_bf16("fine/exact/X", M, K))
    experts = [moqe.moqe_quantize_rtn(W, bits, group, sym), moqe.moqe_quantize_rtn(W, 4, 64, False)]
    ids = torch.zeros(M, dtype=torch.int32, device=dev())
    c, s, z = (t.double() for t in moqe.moqe_expert_export(experts[0]))
    What = ((c.view(N, s.shape[1], -1) - z[:, :, None]) * s[:, :, None]).view(N, K)
    nearest = (X.double() @ What.T).to(torch.bfloat16)
    off = [int((moqe.moqe_routed_qgemm(X, ids, experts, path=path) != nearest).sum()) for path in (moqe.PATH_AUTO, moqe.PATH_STREAM)]
    assert moqe.moqe_async_status() == moqe.OK
    assert off[0] <= off[1] + 3 * (off[0] + off[1]) ** 0.5, off
