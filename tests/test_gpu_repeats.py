"""The decode and the streaming kernel hand a stage back to the bulk copies once its codes and scales have been used: repeated
products are the same bit for bit.  (A stage handed back while they are being read shows as channels that differ from run to run.)"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path,M,specs", [("PATH_DECODE", 16, ((8, 0, True), (4, 128, False), (3, 128, False))), ("PATH_AUTO", 24, ((8, 0, False), (4, 32, True), (3, 64, False))),
                                          ("PATH_DECODE", 32, ((2, 128, False), (4, 0, True))), ("PATH_STREAM", 40, ((8, 0, True), (4, 64, False), (3, 32, True))),
                                          ("PATH_STREAM", 9, ((2, 0, False), (4, 128, True)))])
def test_repeats_bit_for_bit(path, M, specs):
    """7168 x 4096: every stage of the ring is filled again some dozens of times in a CTA."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import dev
    N, K, E = 7168, 4096, len(specs)
    g = torch.Generator("cuda")
    g.manual_seed(M)
    W = torch.randn((N, K), device=dev(), generator=g) * 0.02
    experts = [moqe.moqe_quantize_rtn(W, *s) for s in specs]
    want = "qgemm_stream_kernel" if path == "PATH_STREAM" else "qgemm_decode_kernel"
    assert moqe.moqe_routed_qgemm_kernel(M, experts, getattr(moqe, path)) == want
    X = torch.randn((M, K), device=dev(), generator=g, dtype=torch.bfloat16)
    order = moqe.moqe_permute(None, (torch.arange(M, device=dev()) % E).to(torch.int32), E)[1:]
    ws = moqe.alloc_workspace(moqe.moqe_routed_qgemm_workspace(M, N, K, E))
    moqe.moqe_routed_qgemm_workspace_clear(ws, M, N, K, E)
    Y = torch.empty((32, M, N), dtype=torch.bfloat16, device=dev())
    first = None
    for _ in range(8):
        for y in Y:
            moqe.moqe_routed_qgemm_sorted(X, *order, experts, y, ws, getattr(moqe, path))
        first = Y[0].clone() if first is None else first
        assert bool((Y == first).all())
    assert moqe.moqe_async_status() == moqe.OK
