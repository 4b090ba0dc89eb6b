"""The library after cudaDeviceReset: what it keeps between calls (the opt-in to more shared memory, addresses of its own device
variables, the streams of host-buffer steps) ends with the context, and the calls work in the next one as in the first.
Runs in a process of its own, without torch, whose context can be ended."""
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.gpu
def test_calls_work_again_after_a_device_reset():
    r = subprocess.run([sys.executable, "-m", "tests.test_context_reset_gpu"], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.split()[-1] == "same", r.stdout + r.stderr


class _Cuda:
    def __init__(self):
        import ctypes as C
        self.C, self.rt = C, C.CDLL("libcudart.so.12")
        for name in ("cudaMalloc", "cudaMallocHost"):
            getattr(self.rt, name).argtypes = [C.POINTER(C.c_void_p), C.c_size_t]
        self.rt.cudaMemcpy.argtypes = [C.c_void_p, C.c_void_p, C.c_size_t, C.c_int]

    def ok(self, status):
        assert status == 0, status

    def zeros(self, n, host=False):
        p = self.C.c_void_p()
        self.ok((self.rt.cudaMallocHost if host else self.rt.cudaMalloc)(self.C.byref(p), n))
        self.ok(self.rt.cudaMemcpy(p, np.zeros(n, np.uint8).ctypes.data, n, 4))
        return p.value

    def put(self, a, host=False):
        a = np.ascontiguousarray(a)
        p = self.zeros(a.nbytes, host)
        self.ok(self.rt.cudaMemcpy(p, a.ctypes.data, a.nbytes, 4))
        return p

    def get(self, p, shape, dtype):
        self.ok(self.rt.cudaDeviceSynchronize())
        a = np.empty(shape, dtype)
        self.ok(self.rt.cudaMemcpy(a.ctypes.data, p, a.nbytes, 4))
        return a


def _every_path(cu, B, inputs):
    """Results of one call of each kind that keeps something of the context."""
    C, L, out = cu.C, B.lib(), []
    rng = np.random.default_rng(5)
    # products: more than 48 KB of shared memory, and the library's own scratch array (splits through global memory)
    for oc, ic, bits, static in ((256, 1024, 8, False), (256, 6400, 6, True)):
        blob = B.rwkvq_pack(None, oc, ic, B.RWKVQ_VQ, bits, codes=inputs.random_vq_codes(oc + ic, oc, ic, bits))
        W, x, y = cu.put(blob.image()), cu.put(rng.standard_normal((1, ic)).astype(np.float16)), cu.zeros(4 * oc)
        n = int(L.rwkvq_gemv_workspace_bytes(blob.desc, 1))
        cu.ok(L.rwkvq_gemv_static(blob.desc, W, None, None, x, None, 1, y, 0, None) if static else
              L.rwkvq_gemv(blob.desc, W, None, None, x, None, 1, y, 0, cu.zeros(max(256, n)), max(256, n), None))
        out.append(cu.get(y, oc, np.float32))
    # a prompt
    M = 20
    X, Y, n = cu.put((rng.standard_normal((M, ic)).astype(np.float32).view(np.uint32) >> 16).astype(np.uint16)), cu.zeros(4 * M * oc), int(L.rwkvq_prefill_workspace_bytes(blob.desc, M, 0))
    cu.ok(L.rwkvq_gemm_prefill(blob.desc, W, None, None, X, None, M, Y, 0, cu.zeros(n), n, None))
    out.append(cu.get(Y, (M, oc), np.float32))
    # a matrix and a vector quantized on the device
    for oc, ic in ((256, 256), (1, 4096)):
        d = B.rwkvq_desc_for(oc, ic, B.RWKVQ_VQ, 6)
        image, w = cu.zeros(int(d.image_bytes)), cu.put(rng.standard_normal((oc, ic)).astype(np.float16))
        cfg = B.QuantCfg(method=B.RWKVQ_VQ, bits=6, group=128, vec_dim=2, tile=256, kmeans_iters=3, seed=1, codes_in=None)
        cu.ok(L.rwkvq_quantize_dev(w, oc, ic, C.byref(cfg), None, image, int(d.image_bytes), None, cu.zeros(256), 256, None))
        out.append(cu.get(image, int(d.image_bytes), np.uint8))
    # a step of four products, one behind the other, from and to host buffers of 0.6 MB in all (overlapped copies)
    oc = ic = 512
    b, k, blob = 8, 8, B.rwkvq_pack(None, oc, ic, B.RWKVQ_SQ, 3, codes=inputs.random_sq_codes(3, oc, ic))
    W, gap = cu.put(blob.image()), 65536
    x = np.zeros((k, gap // 2), np.float16)
    x[:, :b * ic] = rng.standard_normal((k, b * ic))
    act, act_h, y, y_h = cu.zeros(k * gap), cu.put(x, host=True), cu.zeros(k * 4 * b * oc), cu.zeros(k * 4 * b * oc, host=True)
    ops = (B.GemvOp * k)()
    for i, o in enumerate(ops):
        o.W_desc, o.W_image_dev, o.x_fp16_dev, o.y_dev, o.stage, o.y_dtype = blob.desc, W, act + i * gap, y + i * 4 * b * oc, i, 0
    n = int(L.rwkvq_step_plan_bytes(ops, k, b))
    plan = cu.zeros(n)
    cu.ok(L.rwkvq_step_plan(ops, k, b, plan, n, None))
    run = lambda: cu.ok(L.rwkvq_step_run_host(plan, n, act_h, act, k * gap, y, y_h, k * 4 * b * oc, None))
    run()
    out.append(cu.get(y_h, (k, b, oc), np.float32).round(3))
    # waits that run out are reported through the status word, once
    cu.ok(L.rwkvq_step_set_wait(plan, 2000, 1))
    cu.ok(L.rwkvq_step_run(plan, n, None))
    assert [L.rwkvq_device_status(None), L.rwkvq_device_status(None)] == [8, 0]
    cu.ok(L.rwkvq_step_set_wait(plan, 0, 0))
    run()
    out.append(cu.get(y_h, (k, b, oc), np.float32).round(3))
    cu.ok(L.rwkvq_step_plan_release(plan))
    assert L.rwkvq_device_status(None) == 0
    return out


if __name__ == "__main__":
    from paper_2505_03803_b200 import binding, inputs as inp
    cuda = _Cuda()
    first = _every_path(cuda, binding, inp)
    for _ in range(2):
        cuda.ok(cuda.rt.cudaDeviceReset())
        for a, b in zip(first, _every_path(cuda, binding, inp)):
            if a.dtype == np.uint8:
                assert np.array_equal(a, b)
            else:      # a step adds partial sums in the order they come
                assert np.abs(a).max() > 1.0 and np.allclose(a, b, rtol=1e-4, atol=2e-3)
    print("same")
