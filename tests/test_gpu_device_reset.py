"""A process that resets its device and starts over (cudaDeviceReset ends its own CUDA context and what belongs to it): contexts and
workspace-free calls made afterwards give what they gave before.  In a child process, since torch's own state would not survive."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes as C, sys
import numpy as np
from paper_2601_17261_b200 import binding as B

L = B.lib()
rt = C.CDLL("libcudart.so.12")
rt.cudaMalloc.argtypes = [C.POINTER(C.c_void_p), C.c_size_t]
rt.cudaMemcpy.argtypes = [C.c_void_p, C.c_void_p, C.c_size_t, C.c_int]


def ok(status):
    assert status == 0, status


def alloc(n):
    p = C.c_void_p()
    ok(rt.cudaMalloc(C.byref(p), n))
    return p.value


def upload(a):
    a = np.ascontiguousarray(a)
    p = alloc(a.nbytes)
    ok(rt.cudaMemcpy(p, a.ctypes.data, a.nbytes, 1))
    return p


def download(p, shape, dtype):
    out = np.empty(shape, dtype)
    ok(rt.cudaMemcpy(out.ctypes.data, p, out.nbytes, 2))      # waits for the legacy stream, which all calls here use
    return out


def bf16(a):
    return (a.view(np.uint32) >> 16).astype(np.uint16)


def iteration():
    # ranks and widths whose kernels need more shared memory than a launch gets unasked: sweeps, fused step, panel QR, passes
    out = []
    rng = np.random.default_rng(3)
    for r, d_in, kind in ((16, 4096, "bf16"), (24, 1024, "bf16"), (40, 1024, "f32"), (64, 512, "bf16")):
        m, d_out = 600, 256
        X, W = rng.standard_normal((m, d_in), np.float32), rng.standard_normal((d_out, d_in), np.float32)
        if kind == "bf16":
            X, W = bf16(X), bf16(W)
        dt = B.AGZO_BF16 if kind == "bf16" else B.AGZO_F32
        V, Wd = upload(np.zeros((r, d_in), np.float32)), upload(W)
        layer = B.agzo_layer(Wd, d_in, None, 0, upload(X), d_in, V, d_in, dt, dt, d_out, d_in, m, r, 1, 0)
        arr = B.layer_array([layer])
        size = C.c_size_t()
        ok(L.agzo_workspace_bytes(arr, 1, C.byref(size)))
        ctx = C.c_void_p()
        ok(L.agzo_create(C.byref(ctx), 0, alloc(size.value), size.value))
        ok(L.agzo_set_option(ctx, b"extract_fused", 2))
        ok(L.agzo_extract_subspace(ctx, arr, 1, 5, 2, None))
        ok(L.agzo_perturb(ctx, arr, 1, 5, 1e-2, None))
        ok(L.agzo_poll(ctx, None))
        out += [download(V, (r, d_in), np.float32), download(Wd, W.shape, W.dtype)]
        ok(L.agzo_destroy(ctx))
    return out


def workspace_free():
    out = []
    for r, d_in in ((8, 1024), (16, 2048), (40, 256)):
        X = np.random.default_rng(r).standard_normal((512, d_in), np.float32)
        V = upload(np.zeros((r, d_in), np.float32))
        ok(L.agzo_extract_subspace_static(upload(X), d_in, B.AGZO_F32, 512, d_in, r, 2, 9, 1, V, d_in, None, None))
        out.append(download(V, (r, d_in), np.float32))
    return out


run = {"context": iteration, "static": workspace_free}[sys.argv[1]]
first = run()
for _ in range(2):
    ok(rt.cudaDeviceReset())
    again = run()
    assert all(np.array_equal(a, b) and np.isfinite(a.astype(np.float32)).all() and a.any() for a, b in zip(first, again))
print("same")
"""


@pytest.mark.parametrize("what", ["context", "static"])
def test_after_a_device_reset(what):
    p = subprocess.run([sys.executable, "-c", CHILD, what], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert p.returncode == 0 and p.stdout.strip() == "same", p.stdout + p.stderr
