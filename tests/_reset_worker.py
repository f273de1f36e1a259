"""Child process: aggregates, resets the device (which ends this process' own
context) and aggregates again, without torch."""
import ctypes
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import oracle  # noqa: E402
import paper_2108_02416_gb300 as ap  # noqa: E402

cuda = ctypes.CDLL("libcudart.so.13", mode=ctypes.RTLD_GLOBAL)


def ok(code):
    if code:
        raise RuntimeError(f"CUDA error {code}")


def on_device(x):
    p = ctypes.c_void_p()
    ok(cuda.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(x.nbytes)))
    ok(cuda.cudaMemcpy(p, x.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(x.nbytes), 1))
    return p


def aggregate(K, r, d, mode):
    a = ap.aspis_assign(K, r)
    rng = np.random.default_rng(d)
    host = rng.standard_normal((a.f, r, d), dtype=np.float32)
    host[:, :, 5] = 2.0
    sel = rng.integers(0, r, a.f).astype(np.int8)
    copies, dsel = on_device(host), on_device(sel)
    det, out = on_device(np.zeros(ap.DETECTION_BYTES, np.uint8)), on_device(np.zeros(d, np.float32))
    code = ap.lib.aspis_aggregate(copies, d, d, a.ref, dsel, det, mode, out, None)
    if code:
        raise RuntimeError(f"aspis_aggregate K={K} r={r} d={d}: {ap.status_str(code)}")
    got = np.zeros(d, np.float32)
    ok(cuda.cudaMemcpy(got.ctypes.data_as(ctypes.c_void_p), out, ctypes.c_size_t(got.nbytes), 2))
    want = oracle.aggregate(host, sel, mode, 0, d)
    if mode == 0:
        assert np.array_equal(got.view(np.uint32), want.view(np.uint32)), (K, r, d)
    else:
        assert np.abs(got - want).max() < 1e-5, (K, r, d)
    return a


kept = []                       # (assignments of a context that is gone are not freed)
for _ in range(2):
    for case in ((7, 3, 300, 0), (15, 3, 300, 0), (15, 3, 20_000, 0), (18, 3, 20_000, 0), (20, 3, 20_000, 0),
                 (22, 3, 500, 0), (15, 3, 20_000, 1)):
        kept.append(aggregate(*case))
    ok(cuda.cudaDeviceReset())
print("done", flush=True)
os._exit(0)
