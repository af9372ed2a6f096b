"""Grouped GEMM: the hand-over of packed tiles."""
import pytest
import torch

pytestmark = pytest.mark.gpu


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
