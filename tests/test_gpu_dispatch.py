"""The automatic choice either side of its lines: the kernel that the library names, the same bits as that kernel asked for
explicitly, and another kernel's result within the tolerance of the routed product."""
import numpy as np
import pytest
import torch

import moqe_workloads as wl

pytestmark = pytest.mark.gpu

STREAM, GROUPED, DECODE, DENSE = 1, 2, 5, 6
NAMES = {STREAM: "qgemm_stream_kernel", GROUPED: "qgemm_tc_kernel", DECODE: "qgemm_decode_kernel", DENSE: "qgemm_dense_kernel"}
PC, G64, G32 = [(8, 0, True), (4, 0, False)], [(8, 0, True), (4, 64, False)], [(4, 0, False), (4, 32, False)]


@pytest.mark.parametrize("M,N,K,specs,want,other", [
    (32, 264, 640, PC, DECODE, STREAM), (33, 264, 640, PC, GROUPED, STREAM),
    (48, 264, 640, G64, STREAM, GROUPED), (49, 264, 640, G64, GROUPED, STREAM),
    (128, 256, 256, PC, GROUPED, STREAM), (129, 256, 256, PC, DENSE, GROUPED), (129, 264, 256, PC, GROUPED, STREAM),
    (11999, 256, 1024, G32, GROUPED, DENSE), (12000, 256, 1024, G32, DENSE, GROUPED), (12000, 520, 256, G32, GROUPED, DENSE),
    (29999, 520, 256, PC, GROUPED, DENSE), (30000, 520, 256, PC, DENSE, GROUPED), (30000, 1032, 64, PC, GROUPED, STREAM)])
def test_automatic_choice(M, N, K, specs, want, other):
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_close, bf16_to_torch, build_experts, dev, torch_to_bits
    gpu, _, _ = build_experts(wl.weights_f32(f"choice/{N}/{K}", N, K), specs)
    X = bf16_to_torch(wl.activations_bf16(f"choice/{M}/{K}", M, K))
    ids = torch.arange(M, device=dev(), dtype=torch.int32) // 64 % len(specs)
    assert moqe.moqe_routed_qgemm_kernel(M, gpu) == NAMES[want]
    out = []
    for path in (moqe.PATH_AUTO, want, other):
        Y = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device=dev())
        moqe.moqe_routed_qgemm(X, ids, gpu, Y=Y, path=path)
        assert moqe.moqe_async_status() == moqe.OK
        out.append(torch_to_bits(Y))
    assert np.array_equal(out[0], out[1])
    assert_close(out[2], out[0], f"M{M} N{N} K{K}")


@pytest.mark.parametrize("M,N,K,specs,want,other", [
    (30000, 264, 512, PC, DENSE, GROUPED), (30000, 320, 568, PC, DENSE, GROUPED), (30000, 328, 512, PC, GROUPED, DENSE), (30000, 264, 576, PC, GROUPED, DENSE),
    (30000, 256, 512, PC, GROUPED, DENSE), (29999, 264, 512, PC, GROUPED, DENSE), (30000, 264, 512, G64, GROUPED, DENSE)])
def test_padded_channels_of_512_k(M, N, K, specs, want, other):
    """Per-channel experts of 512 k whose second pair of channel tiles is mostly padding."""
    test_automatic_choice(M, N, K, specs, want, other)
