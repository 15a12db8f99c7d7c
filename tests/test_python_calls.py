"""agzo_perturb_dense by the compiled entry and by ctypes: the same arguments reach the library."""
import ctypes as C
import sysconfig
import types

import numpy as np
import pytest
import torch

from paper_2601_17261_b200 import binding as B


def test_arguments_are_checked_as_before():
    fn = B._perturb_dense()
    assert fn is not B.lib().agzo_perturb_dense          # built with the library
    assert fn(0, 0, 4, 0, 1, 2, 0.5, 0, 0) == B.AGZO_ERR_STATE
    assert fn(0, 0, 4, 0, -1, 1 << 40, 1, 0, 0) == B.AGZO_ERR_STATE     # integers are taken modulo their width
    with pytest.raises(TypeError):
        fn(0, 0, 4, 0, 1.5, 2, 0.5, 0, 0)
    with pytest.raises(TypeError):
        fn(0, 0, 4, 0, 1, 2, 0.5, 0)
    with pytest.raises(ValueError):
        B.agzo_perturb_dense(None, torch.zeros(4, 4).t()[:2], 1, 2, 0.5)


def test_what_ctypes_takes_and_refuses(monkeypatch):
    ctx, w = types.SimpleNamespace(handle=None), torch.zeros(8)
    monkeypatch.setattr(B, "_raw_stream", lambda device: 0)
    monkeypatch.setattr(B, "_current_device", lambda: 0)
    for seed, layer, scale in ((C.c_uint64(5), C.c_uint32(1), C.c_float(0.5)), (True, 1, np.float32(0.5)), (1 << 70, -1, 1),
                               (np.int64(5), np.int32(1), 0.5)):
        with pytest.raises(B.AgzoError) as e:            # they reach the library, which has no context here
            B.agzo_perturb_dense(ctx, w, seed, layer, scale)
        assert e.value.status == B.AGZO_ERR_STATE
    for seed, layer, scale in ((1.5, 1, 0.5), (1, 1.0, 0.5), (1, 1, "x"), (None, 1, 0.5)):
        with pytest.raises(C.ArgumentError):
            B.agzo_perturb_dense(ctx, w, seed, layer, scale)


def test_only_the_interpreter_it_was_built_for_loads_the_entry(monkeypatch):
    loaded = B._perturb_dense()
    assert loaded.__self__.__file__.endswith("_agzo_calls" + sysconfig.get_config_var("EXT_SUFFIX"))
    monkeypatch.setattr(B, "_dense_call", None)
    monkeypatch.setattr(sysconfig, "get_config_var", lambda name: ".cpython-399-x86_64-linux-gnu.so")
    assert B._perturb_dense() is B.lib().agzo_perturb_dense


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("n,skip", [(0, 0), (1, 0), (1027, 0), (1027, 1)])
@pytest.mark.parametrize("scaled", [False, True])
def test_same_result_as_ctypes(dtype, n, skip, scaled):
    dev = "cuda:0"
    ctx = B.Context(0, 4096)
    a = torch.full((n + skip,), 0.5, dtype=dtype, device=dev)[skip:]
    b = a.clone() if skip == 0 else torch.full((n + skip,), 0.5, dtype=dtype, device=dev)[skip:]
    g = torch.tensor([0.75], device=dev) if scaled else None
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    B.agzo_perturb_dense(ctx, a, (1 << 63) + 5, 7, 1e-2, g, stream=s)
    code = {torch.bfloat16: B.AGZO_BF16, torch.float32: B.AGZO_F32}[dtype]
    assert B.lib().agzo_perturb_dense(ctx.handle, b.data_ptr(), n, code, (1 << 63) + 5, 7, 1e-2,
                                      g.data_ptr() if scaled else None, C.c_void_p(s.cuda_stream)) == B.AGZO_OK
    torch.cuda.synchronize()
    assert torch.equal(a, b)
    assert n == 0 or not torch.equal(a, torch.full_like(a, 0.5))
    with pytest.raises(TypeError):
        B.agzo_perturb_dense(ctx, torch.zeros(4, dtype=torch.float16, device=dev), 1, 2, 0.5)
    B.agzo_destroy(ctx)
    with pytest.raises(B.AgzoError):
        B.agzo_perturb_dense(ctx, a, 1, 2, 0.5)
