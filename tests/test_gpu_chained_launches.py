"""Kernels that may start while their predecessor runs out: whole iterations issued back to back give bit for bit what
they give when the device is idle before every call (whatever a kernel read too early would differ)."""
import numpy as np
import pytest
import torch

from oracle import agzo_oracle as O
from paper_2601_17261_b200 import binding as B
from paper_2601_17261_b200 import workloads as WL

from gpu_helpers import DEV, projector_distance, to_dev, to_host

pytestmark = pytest.mark.gpu


def build(shapes, m, r, bf16):
    out = []
    for i, (d_in, d_out) in enumerate(shapes):
        X, _ = to_dev(WL.planted_activations(m, d_in, min(16, d_in), seed=i, bf16=bf16), bf16)
        W, _ = to_dev(WL.gaussian_weights(d_out, d_in, 0.02, seed=i, bf16=bf16), bf16)
        V = torch.zeros(r, d_in, device=DEV)
        out.append((X, W, V, B.make_layer(X=X, W=W, V=V, r=r, layer_id=i)))
    return out


def iterate(sets, sync, resident, streams=(None,)):
    ctxs = [B.agzo_create([t[3] for t in s], 0) for s in sets]
    for ctx in ctxs:
        B.agzo_set_option(ctx, "extract_resident", resident)
    losses = torch.tensor([1.0, 0.999], dtype=torch.float64, device=DEV)
    ghats = [torch.zeros(1, device=DEV) for _ in sets]
    torch.cuda.synchronize()
    wait = torch.cuda.synchronize if sync else (lambda: None)
    for seed in range(4):
        for j, (s, ctx) in enumerate(zip(sets, ctxs)):
            st = streams[j % len(streams)]
            L = [t[3] for t in s]
            B.agzo_extract_subspace(ctx, L, seed, 2, stream=st); wait()
            B.agzo_perturb(ctx, L, seed, 1e-2, stream=st); wait()
            B.agzo_perturb(ctx, L, seed, -2e-2, stream=st); wait()
            B.agzo_ghat(ctx, losses[0:1], losses[1:2], 1e-2, 0, ghats[j], stream=st); wait()
            B.agzo_restore_update(ctx, L, seed, 1e-2, 1e-1, 0, ghats[j], stream=st); wait()
            B.agzo_perturb_dense(ctx, s[0][1], seed, 7, 1e-3, stream=st); wait()
    torch.cuda.synchronize()
    for ctx in ctxs:
        assert B.agzo_poll(ctx) == B.AGZO_OK
        B.agzo_destroy(ctx)
    return [t[k].clone() for s in sets for t in s for k in (1, 2)]


@pytest.mark.parametrize("n_streams", [1, 2])
@pytest.mark.parametrize("r,bf16,resident", [(3, False, 0), (4, True, 0), (8, True, 0), (24, True, 0), (40, True, 0), (3, False, 2), (8, True, 2)])
def test_back_to_back_equals_one_by_one(r, bf16, resident, n_streams):
    shapes = [[(256, 64)], [(1024, 300), (512, 96)], [(1160, 40)] * 3]
    streams = [torch.cuda.Stream() for _ in range(n_streams)]
    a = iterate([build(s, 600, r, bf16) for s in shapes], sync=True, resident=resident)
    b = iterate([build(s, 600, r, bf16) for s in shapes], sync=False, resident=resident, streams=streams)
    for x, y in zip(a, b):
        assert torch.equal(x, y)


@pytest.mark.parametrize("route", [B.STATIC_CHAIN, B.STATIC_RESIDENT])
def test_workspace_free_calls_back_to_back(route):
    Xs = [to_dev(WL.planted_activations(m, d, 8, seed=m, bf16=False), False)[0] for m, d in ((300, 200), (1000, 512), (64, 128))]
    got = []
    for sync in (True, False):
        Vs = [torch.zeros(8, X.shape[1], device=DEV) for X in Xs for _ in range(2)]
        for i, V in enumerate(Vs):
            B.agzo_debug_extract_static(Xs[i // 2], V, 8, 2, i, i, route)
            if sync:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        got.append(Vs)
    for x, y in zip(*got):
        assert torch.equal(x, y)


def test_layer_lists_alternate_without_waiting():
    # lists on both sides of every way their tables are uploaded (in a kernel's parameters of three sizes, from pinned memory)
    X, _ = to_dev(WL.planted_activations(70, 64, 8, seed=1, bf16=True), True)
    counts = (3, 4, 11, 12, 36, 37, 60)
    got = []
    for sync in (True, False):
        Ws = [to_dev(WL.gaussian_weights(24, 64, 0.02, seed=i, bf16=True), True)[0] for i in range(sum(counts))]
        Vs = [torch.zeros(4, 64, device=DEV) for _ in Ws]
        layers = [B.make_layer(X=X, W=W, V=V, r=4, layer_id=i) for i, (W, V) in enumerate(zip(Ws, Vs))]
        ctx = B.agzo_create(layers, 0)
        B.agzo_set_option(ctx, "extract_resident", 0)            # the kernels that read the tables
        torch.cuda.synchronize()
        for seed in range(3):
            at = 0
            for n in counts:
                B.agzo_extract_subspace(ctx, layers[at:at + n], seed, 1)
                if sync:
                    torch.cuda.synchronize()
                B.agzo_perturb(ctx, layers[at:at + n], seed, 1e-2)
                if sync:
                    torch.cuda.synchronize()
                at += n
        assert B.agzo_poll(ctx) == B.AGZO_OK
        B.agzo_destroy(ctx)
        got.append(Ws + Vs)
    for x, y in zip(*got):
        assert torch.equal(x, y)


@pytest.mark.parametrize("fused", [1, 2])
@pytest.mark.parametrize("r", [5, 8, 24])              # 5: the group of three runs fused as one layer of 15 ranks
def test_layer_lists_with_descriptors_alternate_without_waiting(r, fused):
    # lists of equal and of different length whose activations, weights and shapes all differ, on the tensor-core kernels: every
    # call finds new TMA descriptors and records at the addresses of the previous call's, which its kernels fetch first of all
    lists = [[(1024, 300)], [(512, 136), (512, 264)], [(1160, 200)], [(264, 128)] * 3, [(2048, 96), (640, 520)], [(768, 1000)]]
    got = []
    for sync in (True, False):
        made, layers = [], []
        for k, shapes in enumerate(lists):
            m = 300 + 64 * k
            Xs = {d: to_dev(WL.planted_activations(m, d, 16, seed=k, bf16=True), True)[0] for d, _ in shapes}     # equal widths share
            one = []
            for d_in, d_out in shapes:
                W, _ = to_dev(WL.gaussian_weights(d_out, d_in, 0.02, seed=len(made), bf16=True), True)
                V = torch.zeros(r, d_in, device=DEV)
                one.append(B.make_layer(X=Xs[d_in], W=W, V=V, r=r, layer_id=len(made)))
                made.append((W, V, Xs[d_in]))
            layers.append(one)
        ctx = B.Context(0, max(B.agzo_workspace_bytes(one) for one in layers))
        B.agzo_set_option(ctx, "extract_path", 2)
        B.agzo_set_option(ctx, "extract_fused", fused)
        torch.cuda.synchronize()
        for seed in range(4):
            for one in layers:
                B.agzo_extract_subspace(ctx, one, seed, 1)
                if sync:
                    torch.cuda.synchronize()
            for one in layers:                       # the first kernel of each call is the pass itself
                B.agzo_perturb(ctx, one, seed, 1e-2)
                if sync:
                    torch.cuda.synchronize()
        assert B.agzo_poll(ctx) == B.AGZO_OK
        B.agzo_destroy(ctx)
        got.append([t for W, V, _ in made for t in (W, V)])
    for x, y in zip(*got):
        assert torch.equal(x, y)


@pytest.mark.parametrize("r,bf16", [(4, False), (5, True), (8, True), (40, True)])
@pytest.mark.parametrize("m,d_in", [(256, 128), (300, 200), (513, 520), (600, 1160), (2100, 264)])
def test_activations_written_just_before_the_call(m, d_in, r, bf16):
    # the products ask for their first tiles of X before they wait for the kernel before them: from one tile in all to
    # more than any ring holds, in buffers that every call finds rewritten by the work queued right before it
    src = [to_dev(WL.planted_activations(m, d_in, 16, seed=i, bf16=bf16), bf16)[0] for i in range(4)]
    got = []
    for sync in (True, False):
        X = torch.zeros_like(src[0])
        Vs = [torch.zeros(r, d_in, device=DEV) for _ in src]
        ctx = B.agzo_create([B.make_layer(X=X, V=Vs[0], r=r, layer_id=3)], 0)
        B.agzo_set_option(ctx, "extract_path", 3 if bf16 else 1)
        torch.cuda.synchronize()
        for s, V in zip(src, Vs):
            X.copy_(s)
            B.agzo_extract_subspace(ctx, [B.make_layer(X=X, V=V, r=r, layer_id=3)], 6, 2)
            if sync:
                torch.cuda.synchronize()
        assert B.agzo_poll(ctx) == B.AGZO_OK
        B.agzo_destroy(ctx)
        got.append(Vs)
    for x, y in zip(*got):
        assert torch.equal(x, y)
    for i in (0, 3):
        Vg = to_host(got[1][i])
        assert np.abs(Vg.astype(np.float64) @ Vg.T - np.eye(r)).max() <= 1e-5
        assert projector_distance(Vg, O.extract_subspace(to_host(src[i]), r, 2, 6, 3)) <= 1e-3
