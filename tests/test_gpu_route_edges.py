"""The routing chain where its kernels change shape: the two-kernel sort up to 2048 blocks of 1024 rows (fewer with many
experts) and the three-kernel one beyond (33 buckets, invalid ids among them), rows expanded four at a time, samples of the router's hidden layer taken
four to a warp.  All of it is integer work or fp32 sums, compared as the other tests of these calls do."""
import numpy as np
import pytest
import torch

import oracle
import moqe_workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,E", [(1025, 32), (2048, 1), (2 * 1024 * 1024, 4), (2 * 1024 * 1024 + 1, 4), (2 * 1024 * 1024 + 1, 32)])
def test_sort_with_invalid_ids(M, E):
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import dev
    ids = np.random.default_rng(M + E).integers(-1, E + 1, size=M).astype(np.int32)
    bucket = np.where((ids < 0) | (ids >= E), E, ids)
    _, perm, offsets = moqe.moqe_permute(None, torch.from_numpy(ids).to(dev()), E)
    counts = np.bincount(bucket, minlength=E + 1)
    assert np.array_equal(offsets.cpu().numpy(), np.concatenate([[0], np.cumsum(counts[:E])]))
    assert np.array_equal(perm.cpu().numpy(), np.argsort(bucket, kind="stable"))
    assert moqe.moqe_async_status() == moqe.ERR_EXPERT_ID


@pytest.mark.parametrize("rows", [(1,), (3, 0, 0, 2), (5, 1020, 0, 1), (1, 1, 1, 1, 1, 1, 4093)])
def test_expand_rows(rows):
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import dev
    off = np.concatenate([[0], np.cumsum(rows)]).astype(np.int32)
    ids = np.arange(len(rows), dtype=np.int32)[::-1].copy()
    got = moqe.moqe_expand_ids(torch.from_numpy(ids).to(dev()), torch.from_numpy(off).to(dev()), int(off[-1]))
    assert np.array_equal(got.cpu().numpy(), np.repeat(ids, rows))


@pytest.mark.parametrize("S,H,D", [(1, 8, 1), (7, 264, 9), (8, 128, 8), (9, 136, 17), (17, 512, 7)])
def test_router_sample_groups(S, H, D):
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import dev, bf16_to_torch
    n = 1 + (np.arange(S) * 37) % 70
    off = np.concatenate([[0], np.cumsum(n)]).astype(np.int32)
    X = wl.activations_bf16(f"route/groups/{S}", int(off[-1]), H)
    W1 = wl.normal_f32(f"route/groups/w1/{S}", (D, H), 1.0 / np.sqrt(H))
    W2 = wl.normal_f32(f"route/groups/w2/{S}", (3, D), 1.0 / np.sqrt(D))
    ref, _ = oracle.router_mlp(X, off, W1, W2)
    lg, ids = moqe.moqe_router_mlp(bf16_to_torch(X), torch.from_numpy(off).to(dev()), torch.from_numpy(W1).to(dev()),
                                   torch.from_numpy(W2).to(dev()))
    # fp32 sums of at most 70 + 512 terms of size ~1: 1e-6 relative, a hundredth of the bound
    assert np.all(np.abs(lg.cpu().numpy().astype(np.float64) - ref) <= 1e-4 * (1.0 + np.abs(ref)))
    assert np.array_equal(ids.cpu().numpy(), oracle.route(lg.cpu().numpy()))


@pytest.mark.parametrize("M", [2 ** 31 - 1, 2 ** 31 - 300])
def test_expand_ids_at_the_largest_row_counts(M):
    """The last thread's four rows reach past row 2^31 - 1, which no 32-bit row offset marks as the end."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import dev
    off = torch.tensor([0, 5, 5, 2 ** 30, M], dtype=torch.int32, device=dev())
    ids = torch.tensor([3, 9, 1, 2], dtype=torch.int32, device=dev())
    rows = moqe.moqe_expand_ids(ids, off, M)
    assert moqe.moqe_async_status() == moqe.OK
    for lo, hi, want in ((0, 5, 3), (5, 2 ** 30, 1), (2 ** 30, M, 2)):
        assert int(rows[lo:hi].min()) == want and int(rows[lo:hi].max()) == want


def test_a_refused_launch_leaves_no_error_for_the_next_call():
    """Launches into a capture that has become invalid are refused by the runtime on the host; calls after that are not."""
    import ctypes
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import dev
    rt = ctypes.CDLL("libcudart.so.12")
    L, side = moqe.lib(), torch.cuda.Stream()
    st = ctypes.c_void_p(side.cuda_stream)
    logits = torch.zeros((4, 3), device=dev())
    ids = torch.zeros(4, dtype=torch.int32, device=dev())
    off = torch.arange(5, dtype=torch.int32, device=dev())
    rows, perm = torch.empty_like(ids), torch.empty_like(ids)
    Y = torch.zeros((4, 8), dtype=torch.bfloat16, device=dev())
    order = torch.arange(4, dtype=torch.int32, device=dev())
    torch.cuda.synchronize()
    calls = [lambda: L.moqe_route(logits.data_ptr(), 4, 3, ids.data_ptr(), st),
             lambda: L.moqe_expand_ids(ids.data_ptr(), off.data_ptr(), 4, 4, rows.data_ptr(), st),
             lambda: L.moqe_permute(None, ids.data_ptr(), 4, 0, 3, None, perm.data_ptr(), off.data_ptr(), None, 0, st)]
    for call in calls:
        assert rt.cudaStreamBeginCapture(st, 2) == 0            # (relaxed)
        assert rt.cudaStreamSynchronize(st) != 0                # not allowed in a capture: it is invalid from here on
        refused = call()
        graph = ctypes.c_void_p()
        assert rt.cudaStreamEndCapture(st, ctypes.byref(graph)) != 0
        rt.cudaGetLastError()
        assert refused == moqe.ERR_CUDA
        assert moqe.lib().moqe_unpermute(Y.data_ptr(), order.data_ptr(), 4, 8, Y.data_ptr(), torch.cuda.current_stream().cuda_stream) == moqe.OK
    torch.cuda.synchronize()


@pytest.mark.parametrize("blocks,E", [(1348, 32), (1349, 32), (2048, 13), (2048, 14)])
def test_sort_either_side_of_the_fused_scan(blocks, E):
    """nblk^2 (E + 1) up to 60 million totals: two kernels, above: three."""
    import paper_2508_09204_b200 as moqe
    from gpu_helpers import dev
    ids = torch.randint(-1, E + 1, (blocks * 1024 - 5,), device=dev(), dtype=torch.int32, generator=torch.Generator(dev()).manual_seed(blocks))
    before = moqe.moqe_launch_count()
    _, perm, offsets = moqe.moqe_permute(None, ids, E)
    assert moqe.moqe_launch_count() - before == (2 if blocks * blocks * (E + 1) <= 60_000_000 else 3)
    moqe.moqe_async_status()                                   # (invalid ids were latched)
    bucket = torch.where((ids < 0) | (ids >= E), E, ids)
    assert torch.equal(perm, torch.argsort(bucket, stable=True).to(torch.int32))
    ends = torch.bincount(bucket, minlength=E + 1).cumsum(0)[:E]
    assert torch.equal(offsets, torch.cat([ends.new_zeros(1), ends]).to(torch.int32))
