"""Nothing starts beside the last kernel of a call, or beside the one before a callback: a caller's kernel that is launched with
programmatic stream serialisation and reads before its own wait (GEMMs that fetch their weights early do) finds what the call
wrote.  Every call that leaves something on the device, by each of its last kernels."""
import pytest
import torch

from paper_2601_17261_b200 import binding as B
from paper_2601_17261_b200 import workloads as WL

from gpu_helpers import DEV, Ctx, to_dev

pytestmark = pytest.mark.gpu
ROUNDS = 8


def busy():
    """Half a millisecond of work in front, so that the calls and the reader queue up behind it and meet on the device."""
    torch.cuda._sleep(1_000_000)


def early(ctx, out):
    """What a kernel queued behind the last call reads of `out` before it waits."""
    dst = torch.empty_like(out)
    return lambda: (B.agzo_debug_early_copy(ctx, out, dst), dst)[1]


def compare(got, out):
    torch.cuda.synchronize()
    assert torch.equal(got, out)


# (weights, r, d_out, d_in): tensor-core pass with R regenerated and staged, tiles of the CUDA-core pass that start early (one per
# CTA) and that do not, by rank class, element by element
@pytest.mark.parametrize("kind,r,d_out,d_in", [("bf16", 8, 4096, 4096), ("bf16", 24, 2048, 4096), ("bf16", 8, 512, 256), ("bf16", 2, 256, 2048),
                                               ("bf16", 4, 8192, 4096), ("f32", 8, 256, 256), ("f32", 40, 512, 1024), ("pair", 8, 1024, 1024),
                                               ("f32", 4, 700, 1001)])
def test_weights_behind_a_pass(kind, r, d_out, d_in):
    W, _ = to_dev(WL.gaussian_weights(d_out, d_in, 0.02, seed=1, bf16=kind == "bf16"), kind == "bf16")
    W16 = W.to(torch.bfloat16) if kind == "pair" else None
    out = W if W16 is None else W16
    V = torch.randn(r, d_in, device=DEV)
    g = torch.full((1,), 0.5, device=DEV)
    layers = [B.make_layer(W=W, W16=W16, V=V, r=r, layer_id=0)]
    with Ctx(layers) as ctx:
        look = early(ctx, out)
        torch.cuda.synchronize()
        for seed in range(ROUNDS):
            busy()
            B.agzo_perturb(ctx, layers, seed, 0.5)
            compare(look(), out)
            busy()
            B.agzo_restore_update(ctx, layers, seed, 0.5, 0.1, 0, g)
            compare(look(), out)


@pytest.mark.parametrize("n", [1024, 1 << 24, 1027 * 8 + 4])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_vector_behind_the_dense_direction(n, dtype):
    w = torch.zeros(n, dtype=dtype, device=DEV)
    ctx = B.Context(0, 4096)
    look = early(ctx, w if w.nbytes % 16 == 0 else w[:n // 8 * 8])
    for seed in range(ROUNDS):
        busy()
        for _ in range(3):                       # a kernel still at work in front of the last one
            B.agzo_perturb_dense(ctx, w, seed, 3, 1.0)
        got = look()
        compare(got, w[:got.numel()])
    B.agzo_destroy(ctx)


def test_scalar_and_basis():
    losses = torch.tensor([[float(i + 1), 0.0] for i in range(ROUNDS)], dtype=torch.float64, device=DEV)
    g = torch.zeros(4, device=DEV)
    V = torch.zeros(16, 4096, device=DEV)
    layers = [B.make_layer(V=V, r=16, layer_id=0, d_in=4096)]
    with Ctx(layers) as ctx:
        look_g, look_v = early(ctx, g), early(ctx, V)
        torch.cuda.synchronize()
        for i in range(ROUNDS):
            busy()
            B.agzo_ghat(ctx, losses[i, 0:1], losses[i, 1:2], 1e-3, 0, g)
            compare(look_g(), g)
            busy()
            B.agzo_fill_gaussian_basis(ctx, layers, i)
            compare(look_v(), V)


@pytest.mark.parametrize("r,m,d_in,bf16", [(4, 512, 256, False), (8, 613, 1024, True), (16, 2048, 4096, True), (24, 613, 1024, True),
                                           (64, 1024, 4096, True)])
@pytest.mark.parametrize("resident", [0, 2])
def test_basis_behind_an_extraction(r, m, d_in, bf16, resident):
    X, _ = to_dev(WL.planted_activations(m, d_in, 16, seed=m, bf16=bf16), bf16)
    V = torch.zeros(r, d_in, device=DEV)
    layers = [B.make_layer(X=X, V=V, r=r, layer_id=0)]
    with Ctx(layers) as ctx:
        B.agzo_set_option(ctx, "extract_resident", resident)
        look = early(ctx, V)
        torch.cuda.synchronize()
        for seed in range(ROUNDS):
            busy()
            B.agzo_extract_subspace(ctx, layers, seed, 1)
            compare(look(), V)
        if d_in <= 1024 and r <= 8:
            route = B.STATIC_RESIDENT if resident else B.STATIC_CHAIN
            for flag in (None, torch.zeros(1, dtype=torch.int32, device=DEV)):
                for seed in range(ROUNDS):
                    busy()
                    B.agzo_debug_extract_static(X, V, r, 1, seed, 1, route, flag)
                    compare(look(), V)


def test_panels_before_the_all_reduce():
    m, d_in, r = 4096, 4096, 32
    X, _ = to_dev(WL.planted_activations(m, d_in, 16, seed=m, bf16=True), True)
    V = torch.zeros(r, d_in, device=DEV)
    layers = [B.make_layer(X=X, V=V, r=r, layer_id=0)]
    dst, seen = torch.empty(r * d_in, device=DEV), []
    with Ctx(layers) as ctx:
        def reduce(buf, stream):
            B.agzo_debug_early_copy(ctx, buf, dst, stream=stream)
            torch.cuda.synchronize()
            seen.append(torch.equal(dst, buf))
        B.agzo_set_allreduce(ctx, reduce, 0)
        for seed in range(ROUNDS):
            busy()
            B.agzo_extract_subspace(ctx, layers, seed, 1)
        assert B.agzo_poll(ctx) == B.AGZO_OK
    assert seen == [True] * (2 * ROUNDS)
