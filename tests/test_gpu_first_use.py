"""The first use of a pass that reads tables from device memory: they are uploaded in the
order of the call's own stream (not of the default stream, which non-blocking streams are
not ordered after) and complete when the pass runs.

A process of its own, without torch, whose kernels are loaded at the start: the default
stream is held for a second by a host function while the first dense or parametric call
runs on a non-blocking stream."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import ctypes as C, glob, sys, time
import numpy as np
import paper_1307_3519_gb300 as k
kind = sys.argv[1]
rt = C.CDLL(sorted(glob.glob("/usr/local/cuda/lib64/libcudart.so*"))[0])
def cu(e):
    assert e == 0, e
def dev(nbytes):
    p = C.c_void_p()
    cu(rt.cudaMalloc(C.byref(p), C.c_size_t(nbytes)))
    return p
def up(a):
    p = dev(a.nbytes)
    cu(rt.cudaMemcpy(p, C.c_void_p(a.ctypes.data), C.c_size_t(a.nbytes), 1))
    return p
def down(p, n):
    a = np.empty(n)
    cu(rt.cudaMemcpy(C.c_void_p(a.ctypes.data), p, C.c_size_t(a.nbytes), 2))
    return a
T, S, N, cap, big = 300, 4000, 102, 100_000, 3_000_000
rng = np.random.default_rng(5)
geno, expr = up(rng.integers(0, 3, (S, N)).astype(np.int8)), up(rng.standard_normal((T, N)).astype(np.float32))
lib = k.load_library()
h, rs, n, stream, event = C.c_void_p(), C.c_void_p(), C.c_int64(), C.c_void_p(), C.c_void_p()
cu(lib.krux_create(C.byref(h), 0))
cu(rt.cudaStreamCreateWithFlags(C.byref(stream), 1))
cu(rt.cudaEventCreate(C.byref(event)))
hits, H, p = dev(big * 16), dev(big * 8), dev(big * 8)
dense = dev(T * S * 8), dev(T * S * 8)
o = k.Opts()
o.pthresh, o.hit_capacity, o.snp_end = 1e-3, big, S
cu(lib.krux_rank(h, expr, T, N, N, C.byref(rs), stream))
cu(lib.krux_scan(h, rs, geno, S, N, C.byref(o), hits, H, p, C.byref(n), stream))  # sizes the buffers
def call():
    o.hit_capacity = cap
    if kind == "anova":
        cu(lib.krux_scan_parametric(h, expr, T, N, N, geno, S, N, 0, C.byref(o), hits, H, p, C.byref(n), stream))
        return
    o.dense_H, o.dense_p = dense[0].value, dense[1].value
    cu(lib.krux_scan(h, rs, geno, S, N, C.byref(o), hits, H, p, C.byref(n), stream))
def result():
    if kind == "anova":
        return np.sort(down(H, n.value)), np.sort(down(p, n.value))
    return down(dense[0], T * S), down(dense[1], T * S)
cu(rt.cudaDeviceSynchronize())
hold = C.CFUNCTYPE(None, C.c_void_p)(lambda _: time.sleep(1.0))
cu(rt.cudaLaunchHostFunc(None, hold, None))
cu(rt.cudaEventRecord(event, None))
call()
still = rt.cudaEventQuery(event) != 0
cu(rt.cudaDeviceSynchronize())
first = result()
call()
again = result()
assert n.value > 0 and all(np.array_equal(a, b) for a, b in zip(first, again))
assert still, "the first call waited for the default stream"
print("FIRST_USE_OK")
"""


@pytest.mark.parametrize("kind", ["dense", "anova"])
def test_tables_are_uploaded_on_the_calls_stream(kind):
    from paper_1307_3519_gb300 import build
    build.build()
    env = dict(os.environ, CUDA_MODULE_LOADING="EAGER")
    r = subprocess.run([sys.executable, "-c", CODE, kind], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=120)
    assert "FIRST_USE_OK" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]
