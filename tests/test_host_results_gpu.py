"""Results that kernels write to the calling thread's page-locked buffer: calls of several threads on streams of their own, calls whose
results do not fit it, and calls after the context has ended."""
import math
import os
import subprocess
import sys
import threading
import time

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu


def test_threads_have_results_of_their_own():
    import torch
    from paper_2505_03803_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(3)
    mats = [torch.randn((256, 512), generator=g, device="cuda").half() * (0.01 + i) for i in range(6)]
    want = [B.rwkvq_proxy_segments(w, 16, 128, 4, 3.0, math.inf) for w in mats]
    ws = [torch.empty(B.rwkvq_proxy_workspace_bytes(1), dtype=torch.uint8, device="cuda") for _ in mats]
    whole = [B.rwkvq_proxy_select([w], 4, 3.0, math.inf, k) for w, k in zip(mats, ws)]
    torch.cuda.synchronize()
    wrong = []

    def work(i):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            for _ in range(40):
                got = B.rwkvq_proxy_segments(mats[i], 16, 128, 4, 3.0, math.inf)
                one = B.rwkvq_proxy_select([mats[i]], 4, 3.0, math.inf, ws[i])
                if not all(np.array_equal(a, b) for a, b in zip(got, want[i])) or not all(np.array_equal(a, b) for a, b in zip(one, whole[i])):
                    wrong.append(i)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(mats))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


@pytest.mark.parametrize("rows", [2730, 2731, 43690, 43691])
def test_results_up_to_and_beyond_the_buffer(rows):
    """24 bytes a tile: 64 KB and 1 MB hold 2730 and 43 690."""
    import torch
    from oracle import rwkvq_oracle as orc
    from paper_2505_03803_b200 import binding as B
    w = torch.randn((rows, 8), generator=torch.Generator(device="cuda").manual_seed(rows), device="cuda").half()
    pc, pf, _ = B.rwkvq_proxy_segments(w, 1, 8, 4, 3.0, math.inf)
    pick = np.array([0, 1, rows // 2, rows - 2, rows - 1])
    rpc, rpf = orc.proxy_segments(w[torch.from_numpy(pick).cuda()].double().cpu().numpy(), 1, 8, K=4)
    assert np.allclose(pc[pick], rpc, rtol=1e-9, atol=1e-9) and np.allclose(pf[pick], rpf, rtol=1e-8, atol=1e-8)


@pytest.mark.parametrize("what", ["segments", "whole"])
def test_a_call_that_fails_has_ended_its_work(what):
    """An error that an earlier call of the program left behind is reported after the kernels are enqueued: they have ended when the call returns, and the
    thread's next call, on another stream, gets the buffer to itself."""
    import ctypes as C

    import torch
    from paper_2505_03803_b200 import binding as B
    w = torch.randn((256, 512), generator=torch.Generator(device="cuda").manual_seed(8), device="cuda").half()
    ws = torch.empty(max(B.rwkvq_proxy_workspace_bytes(1), B.lib().rwkvq_proxy_segments_workspace_bytes(256, 512, 16, 128)), dtype=torch.uint8, device="cuda")

    def call(stream):      # without torch, whose allocator would report the error
        pc, pf, phi = np.zeros(64), np.zeros(64), np.zeros(64, np.int32)
        if what == "segments":
            status = B.lib().rwkvq_proxy_segments(w.data_ptr(), B.RWKVQ_F16, 256, 512, 16, 128, 4, 3.0, math.inf, pc.ctypes.data, pf.ctypes.data,
                                                  phi.ctypes.data, ws.data_ptr(), ws.nbytes, stream.cuda_stream)
        else:
            mat, oc, ic, dbl = (C.c_void_p * 1)(w.data_ptr()), (C.c_int * 1)(256), (C.c_int * 1)(512), C.POINTER(C.c_double)
            status = B.lib().rwkvq_proxy_select(mat, oc, ic, 1, 4, 3.0, math.inf, pc.ctypes.data_as(dbl), pf.ctypes.data_as(dbl),
                                                phi.ctypes.data_as(C.POINTER(C.c_int)), ws.data_ptr(), ws.nbytes, stream.cuda_stream)
        return status, pc, pf, phi

    busy, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    want = call(other)
    assert want[0] == 0
    rt, p = C.CDLL("libcudart.so.12"), C.c_void_p()
    with torch.cuda.stream(busy):
        torch.cuda._sleep(100_000_000)
    assert rt.cudaMalloc(C.byref(p), C.c_size_t(1 << 60)) != 0
    status = call(busy)[0]
    idle = busy.query()
    assert status == 6 and idle
    assert all(np.array_equal(a, b) for a, b in zip(call(other), want))


def test_a_thread_may_end_while_another_captures():
    import torch
    from paper_2505_03803_b200 import binding as B
    w = torch.randn((256, 512), device="cuda").half()
    called, end = threading.Event(), threading.Event()

    def work():
        B.rwkvq_proxy_segments(w, 16, 128, 4, 3.0, math.inf)
        called.set()
        end.wait(60)

    t = threading.Thread(target=work)
    t.start()
    assert called.wait(60)
    x, graph = torch.zeros(64, device="cuda"), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        end.set()
        t.join()
        time.sleep(0.2)             # the system's thread ends a little after the interpreter's
        x += 1
    graph.replay()
    torch.cuda.synchronize()
    assert float(x.sum()) == 64


@pytest.mark.parametrize("what", ["calls", "thread"])
def test_results_after_a_device_reset(what):
    r = subprocess.run([sys.executable, "-m", "tests.test_host_results_gpu", what], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.split()[-1] == "same", r.stdout + r.stderr


if __name__ == "__main__":
    import ctypes as C

    from paper_2505_03803_b200 import binding as B
    from tests.test_context_reset_gpu import _Cuda
    cu, out = _Cuda(), []
    w16 = np.random.default_rng(1).standard_normal((64, 256)).astype(np.float16)

    def call():
        w, n = cu.put(w16), int(B.lib().rwkvq_proxy_segments_workspace_bytes(64, 256, 1, 256))
        pc, pf, phi = np.empty(64), np.empty(64), np.empty(64, np.int32)
        cu.ok(B.lib().rwkvq_proxy_segments(w, B.RWKVQ_F16, 64, 256, 1, 256, 4, 3.0, math.inf, pc.ctypes.data, pf.ctypes.data, phi.ctypes.data, cu.zeros(n), n, None))
        out.append((pc, pf, phi))

    if sys.argv[1] == "calls":
        for _ in range(3):
            call()
            cu.ok(cu.rt.cudaDeviceReset())
        assert all(np.array_equal(a, b) for o in out[1:] for a, b in zip(out[0], o)) and np.isfinite(out[0][0]).all()
    else:
        # a thread ends in a later context than its buffer's: what lies at the buffer's address by then stays
        called, end = threading.Event(), threading.Event()
        t = threading.Thread(target=lambda: (call(), called.set(), end.wait(60)))
        t.start()
        assert called.wait(60)
        cu.ok(cu.rt.cudaDeviceReset())
        later = []
        for _ in range(4):
            p = C.c_void_p()
            cu.ok(cu.rt.cudaMallocHost(C.byref(p), 64 << 10))
            later.append(p)
        end.set()
        t.join()
        time.sleep(0.2)
        for p in later:
            cu.ok(cu.rt.cudaFreeHost(p))
    print("same")
