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


def _grid(W, bits, group, sym):
    """Codes, scales and zero-points as the header states them, in fp32 and clamped before they become whole numbers."""
    N, K = W.shape
    w, L, qmax = W.reshape(N, -1, group or K), np.float32(2 ** bits - 1), np.float32(2 ** (bits - 1) - 1)
    lo, hi = w.min(2, keepdims=True, initial=0), w.max(2, keepdims=True, initial=0)
    with np.errstate(all="ignore"):
        s16 = (np.maximum(-lo, hi) / qmax if sym else (hi - lo) / L).astype(np.float16)
        s16 = np.where((s16 > 0) & np.isfinite(s16), s16, np.float16(1))
        s = s16.astype(np.float32)
        q = np.rint(w / s)
        z = np.full_like(s, 2 ** (bits - 1)) if sym else np.clip(np.rint(-lo / s), 0, L) + np.float32(0)
        c = np.clip(q, -qmax, qmax) + z if sym else np.clip(q + z, 0, L)
    return c.reshape(N, K).astype(np.uint8), s16[..., 0].view(np.uint16), z[..., 0].astype(np.float16).view(np.uint16)


@pytest.mark.parametrize("bits,group,sym", [(8, 0, True), (4, 0, False), (3, 32, True), (2, 64, True), (4, 128, True), (4, 128, False), (8, 256, True), (3, 256, False)])
@pytest.mark.parametrize("N,K", [(16, 512), (16, 6144)])
def test_weights_beyond_every_scale(N, K, bits, group, sym):
    """Scale 1 where fp16 has none for the group, and quotients beyond 2^31: codes at the ends of the range, by one kernel (groups up to
    128 k, short rows) and by two."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_expert_matches, dev
    W = wl.weights_f32(f"beyond/{N}/{K}", N, K)
    assert all(np.array_equal(a, b) for a, b in zip(_grid(W, bits, group, sym), oracle.quantize_rtn(W, bits, group, sym)))
    W[1::2, ::7], W[1::2, 3::11], W[5::4, 5::13] = 3e9, -3e9, 3e38
    e = moqe.moqe_quantize_rtn(torch.from_numpy(W).to(dev()), bits, group, sym)
    assert_expert_matches(e, _grid(W, bits, group, sym))


@pytest.mark.parametrize("bits,group,sym", [(8, 0, True), (4, 0, False), (3, 32, True), (2, 64, False), (4, 128, True), (4, 128, False), (4, 256, False)])
@pytest.mark.parametrize("N,K", [(16, 512), (16, 6144)])
def test_weights_that_are_no_numbers(N, K, bits, group, sym):
    """They have the zero-point's code and leave scales and the other codes alone, by one kernel and by two."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_expert_matches, dev
    W = wl.weights_f32(f"nan/{N}/{K}", N, K)
    gone = np.zeros((N, K), bool)
    gone[1::2, ::5] = gone[1::2, 17:41] = gone[4] = True
    W[gone] = 0.0                                                  # (the code of 0 is the zero-point)
    canon = oracle.quantize_rtn(W, bits, group, sym)
    W[gone] = np.nan
    assert_expert_matches(moqe.moqe_quantize_rtn(torch.from_numpy(W).to(dev()), bits, group, sym), canon)


@pytest.mark.parametrize("bits,group,sym", [(4, 128, False), (3, 64, False), (8, 32, True), (2, 32, False)])
@pytest.mark.parametrize("N,K", [(8, 128), (2304, 1536), (2368, 1536), (2360, 1664), (1192, 8192), (2936, 6400)])
def test_blobs_to_a_warp(N, K, bits, group, sym):
    """Blobs of 16 channels x 128 k, N padded to 128, for the 12 warps of each of 148 SMs: 8; 1728, at most one each; 1824 and 1976, for
    some two; 5120, two or three; 9200, five or six, so that both stages are filled twice again and their barriers' parity comes
    round.  The channels' sizes go from scales that underflow in fp16 to large ones."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import assert_expert_matches, dev
    W = wl.weights_f32(f"blobs/{N}/{K}", N, K) * np.exp2(np.arange(N) % 43 - 30).astype(np.float32)[:, None]
    e = moqe.moqe_quantize_rtn(torch.from_numpy(W).to(dev()), bits, group, sym)
    assert_expert_matches(e, oracle.quantize_rtn(W, bits, group, sym))


@pytest.mark.parametrize("bits,sym", [(8, True), (4, False), (3, False), (2, True)])
@pytest.mark.parametrize("N,K", [(2296, 1088), (2368, 64), (2056, 1088), (2376, 5128), (2296, 5120), (2048, 1152), (264, 1024), (264, 1032), (9464, 3848), (9464, 3840)])
def test_per_channel_by_one_kernel_and_by_two(N, K, bits, sym):
    """144 and 148 strips of 16 rows are for one kernel on 148 SMs, up to K = 5120; 136 and 152 strips, and longer rows, for two;
    up to K = 1024 all are for one.  Without padding (2048 x 1152) nothing is cleared first.  Four strips to an SM go two at a time from
    3848 k on, three at a time before.  The memory is that of a larger expert before."""
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
