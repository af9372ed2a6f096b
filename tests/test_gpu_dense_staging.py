"""The dense-weights GEMM with a last channel chunk narrower than the others: each half of an output row is staged in
shared memory and leaves by an asynchronous copy of its own, so the second half of the narrow chunk must not be staged
where the first half of the wide one is still being read (zeros used to appear in columns 32..39 of single rows)."""
import numpy as np
import pytest
import torch

import oracle
import moqe_workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(392, 264, 200), (2048, 320, 64), (1024, 520, 128)])
def test_narrow_last_chunk_many_times(M, N, K):
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_close, bf16_to_torch, build_experts, dev, torch_to_bits
    W = wl.weights_f32(f"dn/narrow/{N}", N, K)
    X = wl.activations_bf16(f"dn/narrow/{M}", M, K, relu=True)
    gpu, What, _ = build_experts(W, [(8, 0, True), (4, 0, False)])
    ids = np.repeat(np.arange((M + 195) // 196) % 2, 196)[:M].astype(np.int32)
    ref = oracle.routed_gemm(X, ids, What)
    Xd, idd = bf16_to_torch(X), torch.from_numpy(ids).to(dev())
    for _ in range(25):
        Y = moqe.moqe_routed_qgemm(Xd, idd, gpu, path=moqe.PATH_DENSE)
        assert_close(torch_to_bits(Y), ref, f"dense M{M} N{N} K{K}")


@pytest.mark.parametrize("N,K", [(320, 64), (576, 128), (1024, 64), (64, 64)])
def test_output_boxes_are_free_before_they_are_filled(N, K):
    """Three and more tiles to a CTA, of rows that are stored by box, scattered ones and both, with one, two and no boxes to a warp in the
    last channel chunk; every element against the grouped GEMM."""
    import torch
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_close, bf16_to_torch, build_experts, dev, torch_to_bits
    M = 70000
    g = np.random.default_rng(N)
    ids = np.concatenate([np.repeat(g.integers(0, 3, 140), 250), g.integers(0, 3, 15000), np.repeat(g.integers(0, 3, 200), 100)]).astype(np.int32)
    assert ids.size == M
    gpu, _, _ = build_experts(wl.weights_f32(f"boxes/{N}/{K}", N, K), [(8, 0, True), (4, 0, False), (4, 32, False)])
    X, row_ids = bf16_to_torch(wl.activations_bf16(f"boxes/{K}", M, K)), torch.from_numpy(ids).to(dev())
    out = []
    for path in (moqe.PATH_TCGEN05, moqe.PATH_DENSE, moqe.PATH_DENSE):
        Y = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device=dev())
        moqe.moqe_routed_qgemm(X, row_ids, gpu, Y=Y, path=path)
        assert moqe.moqe_async_status() == moqe.OK
        out.append(torch_to_bits(Y))
    assert_close(out[1], out[0], f"boxes N{N} K{K}")
    assert np.array_equal(out[1], out[2])
