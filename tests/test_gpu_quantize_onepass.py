"""Expert construction in one kernel: bit-exact codes, scales and zero-points where its rounding shortcut has to fall back
to the division (weights exactly halfway between two codes), at padded sizes, and in memory that an earlier, destroyed
expert has used (nothing of it may be left in the padding, which the products read)."""
import numpy as np
import pytest
import torch

import oracle
import moqe_workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,group,sym", [(8, 0, True), (4, 0, False), (3, 32, True), (2, 64, False), (4, 128, False), (8, 64, False)])
@pytest.mark.parametrize("N,K", [(8, 64), (136, 192), (264, 1088), (16, 8192)])
def test_halfway_weights_and_reused_memory(N, K, bits, group, sym):
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_close, assert_expert_matches, bf16_to_torch, dev, torch_to_bits
    if group and K % group:
        pytest.skip("the group does not divide K")
    g = np.random.default_rng(bits * 1000 + group + N)
    # multiples of half a step of a power-of-two grid; the extremes pin the grid's scale
    top = 2 ** (bits - 1) - 1
    W = (g.integers(-2 * top, 2 * top + 1, size=(N, K)) * 0.5).astype(np.float32)
    per = group or K
    W[:, ::per], W[:, 1::per] = top, (-top if sym else -(2 ** bits - 1 - top))
    W *= np.float32(2.0 ** -7)
    big = moqe.moqe_quantize_rtn(torch.full((2 * N + 128, 2 * K), 3.0, device=dev()), 8, 0, False)
    big.close()
    e = moqe.moqe_quantize_rtn(torch.from_numpy(W).to(dev()), bits, group, sym)
    c, s, z = oracle.quantize_rtn(W, bits, group, sym)
    assert_expert_matches(e, (c, s, z))
    M = 136
    X = wl.activations_bf16(f"onepass/{K}", M, K)
    ids = np.zeros(M, np.int32)
    Y = moqe.moqe_routed_qgemm(bf16_to_torch(X), torch.from_numpy(ids).to(dev()), [e], path=moqe.PATH_TCGEN05)
    assert moqe.moqe_async_status() == moqe.OK
    assert_close(torch_to_bits(Y), oracle.routed_gemm(X, ids, [oracle.dequantize(c, s, z, group)]), "product")


@pytest.mark.parametrize("bits,group,sym", [(4, 128, False), (3, 64, False), (8, 32, True), (2, 32, False)])
@pytest.mark.parametrize("N,K", [(8, 128), (2368, 1536), (2360, 1664), (1192, 8192)])
def test_blobs_to_a_warp(N, K, bits, group, sym):
    """8 blobs of 16 channels x 128 k for 1776 warps (148 SMs); one each; for some two; two or three, so that stages are filled
    again.  The channels' sizes go from scales that underflow in fp16 to large ones."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_expert_matches, dev
    W = wl.weights_f32(f"blobs/{N}/{K}", N, K) * np.exp2(np.arange(N) % 43 - 30).astype(np.float32)[:, None]
    e = moqe.moqe_quantize_rtn(torch.from_numpy(W).to(dev()), bits, group, sym)
    assert_expert_matches(e, oracle.quantize_rtn(W, bits, group, sym))


@pytest.mark.parametrize("bits,sym", [(8, True), (4, False), (3, False), (2, True)])
@pytest.mark.parametrize("N,K", [(2296, 1088), (2368, 64), (2056, 1088), (2376, 5128), (2296, 5120), (2048, 1152), (264, 1024), (264, 1032)])
def test_per_channel_by_one_kernel_and_by_two(N, K, bits, sym):
    """144 and 148 strips of 16 rows are for one kernel on 148 SMs, up to K = 5120; 136 and 152 strips, and longer rows, for two;
    up to K = 1024 all are for one.  Without padding (2048 x 1152) nothing is cleared first.  The memory is that of a larger expert before."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_close, assert_expert_matches, bf16_to_torch, dev, torch_to_bits
    W = wl.weights_f32(f"pc/{N}/{K}", N, K)
    moqe.moqe_quantize_rtn(torch.full((2 * N + 128, 2 * K), 3.0, device=dev()), 8, 0, False).close()
    e = moqe.moqe_quantize_rtn(torch.from_numpy(W).to(dev()), bits, 0, sym)
    canon = oracle.quantize_rtn(W, bits, 0, sym)
    assert_expert_matches(e, canon)
    X = wl.activations_bf16(f"pc/{K}", 40, K)
    ids = np.zeros(40, np.int32)
    Y = moqe.moqe_routed_qgemm(bf16_to_torch(X), torch.from_numpy(ids).to(dev()), [e], path=moqe.PATH_TCGEN05)
    assert moqe.moqe_async_status() == moqe.OK
    assert_close(torch_to_bits(Y), oracle.routed_gemm(X, ids, [oracle.dequantize(*canon, 0)]), "product")


def test_rows_longer_than_a_grid_has_blocks():
    """More than 65535 eights of k-blocks to a row."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import dev
    N, K = 8, 65536 * 1024 + 128
    W = torch.zeros((N, K), device=dev())
    W[:, ::2] = 1.0
    W[:, -128:] *= 2.0
    codes, scales, zeros = moqe.moqe_expert_export(moqe.moqe_quantize_rtn(W, 8, 128, False))
    assert bool((codes[:, ::2] == 255).all()) and not bool(codes[:, 1::2].any()) and not bool(zeros.any())
    s = torch.tensor([1.0 / 255], dtype=torch.float32).half().to(dev())
    assert bool((scales[:, :-1] == s).all()) and bool((scales[:, -1] == torch.tensor(2.0 / 255).half().to(dev())).all())
