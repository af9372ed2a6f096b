"""Where experts' device memory comes from and goes to: giving it back waits for the device and disturbs nobody's capture."""
import ctypes
import os
import subprocess
import sys
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu

THREAD_LOCAL, RELAXED = 1, 2                    # cudaStreamCaptureMode


def _runtime():
    return ctypes.CDLL("libcudart.so.12")


class _Capture:
    """A capture on a stream of its own; `graph` afterwards, `valid` whether it came to one."""

    def __init__(self, mode):
        self.mode, self.stream, self.graph = mode, torch.cuda.Stream(), ctypes.c_void_p()
        self.handle = ctypes.c_void_p(self.stream.cuda_stream)

    def __enter__(self):
        torch.cuda.synchronize()
        assert _runtime().cudaStreamBeginCapture(self.handle, self.mode) == 0
        return self

    def __exit__(self, *exc):
        self.valid = _runtime().cudaStreamEndCapture(self.handle, ctypes.byref(self.graph)) == 0
        _runtime().cudaGetLastError()


def _elsewhere(call):
    got = []

    def run():
        torch.cuda.set_device(0)
        got.append(call())
    t = threading.Thread(target=run)
    t.start()
    t.join()
    return got[0]


def _expert(N=512, K=512):
    import paper_2508_09204_b200 as moqe
    W = torch.randn((N, K), device="cuda", generator=torch.Generator("cuda").manual_seed(N + K))
    return W, moqe.moqe_quantize_rtn(W, 4, 128, False)


def test_destroy_waits_for_every_stream():
    import paper_2508_09204_b200 as moqe
    side = torch.cuda.Stream()
    _, e = _expert()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)           # some 10 ms
    assert not side.query()
    e.close()
    assert side.query()
    assert moqe.moqe_async_status() == moqe.OK


@pytest.mark.parametrize("mode,same_thread", [(THREAD_LOCAL, False), (RELAXED, False), (RELAXED, True)])
def test_destroy_beside_a_capture(mode, same_thread):
    import paper_2508_09204_b200 as moqe
    _, e = _expert()
    handle, e.handle = e.handle, None
    with _Capture(mode) as c:
        destroy = lambda: moqe.lib().moqe_expert_destroy(handle)
        status = destroy() if same_thread else _elsewhere(destroy)
    assert status == moqe.OK and c.valid


@pytest.mark.parametrize("what", ["quantize", "prefetch"])
@pytest.mark.parametrize("mode,same_thread", [(THREAD_LOCAL, False), (RELAXED, True)])
def test_building_in_a_capture(mode, same_thread, what):
    """The expert's memory exists at once, and the graph fills it when it runs."""
    import paper_2508_09204_b200 as moqe
    W, e = _expert()
    host = moqe.moqe_expert_offload(e)
    out = ctypes.c_void_p()
    with _Capture(mode) as c:
        if what == "quantize":
            build = lambda: moqe.lib().moqe_quantize_rtn(W.data_ptr(), *W.shape, 4, 128, 0, c.handle, ctypes.byref(out))
        else:
            build = lambda: moqe.lib().moqe_expert_prefetch(host.handle, c.handle, ctypes.byref(out))
        status = build() if same_thread else _elsewhere(build)
    assert status == moqe.OK and c.valid
    run = ctypes.c_void_p()
    assert _runtime().cudaGraphInstantiate(ctypes.byref(run), c.graph, ctypes.c_ulonglong(0)) == 0
    assert _runtime().cudaGraphLaunch(run, c.handle) == 0
    torch.cuda.synchronize()
    built = moqe.Expert(out.value)
    for a, b in zip(moqe.moqe_expert_export(built), moqe.moqe_expert_export(e)):
        assert torch.equal(a, b)
    torch.cuda.synchronize()
    _runtime().cudaGraphExecDestroy(run)
    _runtime().cudaGraphDestroy(c.graph)
    built.close()


_FIRST_BUILD = """
import ctypes, sys, threading, torch
import paper_2508_09204_b200 as moqe
mode, captured = int(sys.argv[1]), sys.argv[2] == "captured"
rt = ctypes.CDLL("libcudart.so.12")
W = torch.randn((512, 512), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
side, blocking, graph, out = torch.cuda.Stream(), ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
assert rt.cudaStreamCreate(ctypes.byref(blocking)) == 0
torch.cuda.synchronize()
assert rt.cudaStreamBeginCapture(blocking, mode) == 0
got = []
def build():
    torch.cuda.set_device(0)
    got.append(moqe.lib().moqe_quantize_rtn(W.data_ptr(), 512, 512, 4, 128, 0, blocking if captured else side.cuda_stream, ctypes.byref(out)))
t = threading.Thread(target=build)
t.start()
t.join()
assert rt.cudaStreamEndCapture(blocking, ctypes.byref(graph)) == 0, "the capture is invalid"
assert got == [moqe.OK], got
if captured:
    run = ctypes.c_void_p()
    assert rt.cudaGraphInstantiate(ctypes.byref(run), graph, ctypes.c_ulonglong(0)) == 0 and rt.cudaGraphLaunch(run, blocking) == 0
torch.cuda.synchronize()
a, b = moqe.moqe_expert_export(moqe.Expert(out.value)), moqe.moqe_expert_export(moqe.moqe_quantize_rtn(W, 4, 128, False))
assert all(torch.equal(x, y) for x, y in zip(a, b)) and moqe.moqe_async_status() == moqe.OK
"""


@pytest.mark.parametrize("mode,where", [(THREAD_LOCAL, "beside"), (RELAXED, "beside"), (THREAD_LOCAL, "captured")])
def test_the_first_build_of_a_process(mode, where):
    """A build by groups, the first thing a process has the library do, while a blocking stream is being captured by another thread: it
    leaves the capture alone, and its status word exists in the captured stream too."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _FIRST_BUILD, str(mode), where], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr


def test_trim_gives_freed_memory_back():
    import paper_2508_09204_b200 as moqe
    W = torch.randn((8192, 4096), device="cuda")
    free = lambda: (torch.cuda.empty_cache(), torch.cuda.mem_get_info()[0])[1]         # (without what torch keeps)
    moqe.moqe_expert_pool_trim()
    before = free()
    experts = [moqe.moqe_quantize_rtn(W, 8, 0, True) for _ in range(12)]
    bytes_each = experts[0].alloc_bytes
    assert before - free() >= 12 * bytes_each
    for e in experts[1:]:
        e.close()
    assert free() < before - 12 * bytes_each + (1 << 20)          # kept for the next expert
    moqe.moqe_expert_pool_trim(6 * bytes_each)
    assert before - 7 * bytes_each <= free() <= before - bytes_each
    moqe.moqe_expert_pool_trim()
    assert before - 3 * bytes_each <= free() <= before - bytes_each  # (the living one, in the pool's own granularity)
    assert torch.equal(moqe.moqe_expert_export(experts[0])[0], moqe.moqe_expert_export(moqe.moqe_quantize_rtn(W, 8, 0, True))[0])
    experts[0].close()
    moqe.moqe_expert_pool_trim()
    assert free() == before
