"""The products in bf16 parts on the tensor cores, at the edges of their steps of 64 and blocks of 128: columns and tokens around them,
rows that allow accesses of eight columns, of four and of one, ranks around the panels of 8, 16 and 24 and beyond one unit, several
layers on one X and more units than the short list of a launch holds, clusters of which some CTAs have no columns.

Tolerance: that of the CUDA-core products (fp32 sums over at most 1300 terms), which these replace: 1e-5 orthonormality and 1e-4
projector distance."""
import numpy as np
import pytest
import torch

from oracle import agzo_oracle as O
from paper_2601_17261_b200 import binding as B
from paper_2601_17261_b200 import workloads as WL

from gpu_helpers import DEV, Ctx, projector_distance, to_dev, to_host

pytestmark = pytest.mark.gpu


def check(X, V, r, K, seed, layer, tol=1e-4):
    Vg = to_host(V)
    assert np.abs(Vg.astype(np.float64) @ Vg.T - np.eye(r)).max() <= 1e-5
    assert projector_distance(Vg, O.extract_subspace(X, r, K, seed, layer)) <= tol


def options(ctx):
    B.agzo_set_option(ctx, "extract_resident", 0)
    B.agzo_set_option(ctx, "extract_split", 2)


@pytest.mark.parametrize("r", [1, 8, 9, 17, 25])
@pytest.mark.parametrize("m,d_in", [(40, 40), (64, 64), (127, 129), (129, 132), (257, 200), (640, 516), (1300, 1032)])
@pytest.mark.parametrize("bf16,extra", [(False, 0), (False, 3), (True, 1), (True, 4)])
def test_split_products(r, m, d_in, bf16, extra):
    X = WL.planted_activations(m, d_in, min(32, d_in // 2), seed=m + d_in, bf16=bf16)
    Xd, _ = to_dev(X, bf16, pitch=d_in + extra if extra else None)
    V = torch.zeros(r, d_in, device=DEV)
    layers = [B.make_layer(X=Xd, V=V, r=r, layer_id=3)]
    with Ctx(layers) as ctx:
        options(ctx)
        B.agzo_extract_subspace(ctx, layers, 9, 2)
        assert B.agzo_poll(ctx) == B.AGZO_OK
    check(X, V, r, 2, 9, 3)


@pytest.mark.parametrize("ranks", [(8, 8, 8), (3, 5, 1, 2, 6), (64,), (20, 20)])
def test_split_products_of_layers_on_one_input(ranks):
    m, d_in = 700, 300
    X = WL.planted_activations(m, d_in, 96, seed=5, bf16=False)
    Xd, _ = to_dev(X, False)
    V = [torch.zeros(r, d_in, device=DEV) for r in ranks]
    layers = [B.make_layer(X=Xd, V=v, r=r, layer_id=i) for i, (v, r) in enumerate(zip(V, ranks))]
    with Ctx(layers) as ctx:
        options(ctx)
        B.agzo_extract_subspace(ctx, layers, 4, 1)
        assert B.agzo_poll(ctx) == B.AGZO_OK
    for i, (v, r) in enumerate(zip(V, ranks)):
        check(X, v, r, 1, 4, i, 1e-3 if r == 64 else 1e-4)


def test_split_products_of_many_layers():
    shapes = [(300 + 17 * i, 96 + 36 * (i % 5), 1 + i % 9) for i in range(23)]      # of any order of widths
    data, layers = [], []
    for i, (m, d, r) in enumerate(shapes):
        X = WL.planted_activations(m, d, 16, seed=i, bf16=False)
        Xd, V = to_dev(X, False)[0], torch.zeros(r, d, device=DEV)
        data.append((X, Xd, V, r))
        layers.append(B.make_layer(X=Xd, V=V, r=r, layer_id=i))
    with Ctx(layers) as ctx:
        options(ctx)
        B.agzo_extract_subspace(ctx, layers, 8, 1)
        assert B.agzo_poll(ctx) == B.AGZO_OK
    for i, (X, _, V, r) in enumerate(data):
        check(X, V, r, 1, 8, i)


def test_small_fp32_inputs_keep_their_bits_without_a_power_step():
    # K = 0 of inputs whose third bf16 part would not exist stays with the fp32 products
    m, d_in, r = 300, 256, 4
    X = (WL.planted_activations(m, d_in, 16, seed=2, bf16=False).astype(np.float32) * np.float32(2.0 ** -118)).astype(np.float32)
    Xd, V = to_dev(X, False)[0], torch.zeros(r, d_in, device=DEV)
    layers = [B.make_layer(X=Xd, V=V, r=r, layer_id=0)]
    with Ctx(layers) as ctx:
        options(ctx)
        B.agzo_extract_subspace(ctx, layers, 9, 0)
        assert B.agzo_poll(ctx) == B.AGZO_OK
    Vo = O.extract_subspace(X.astype(np.float64) * 2.0 ** 118, r, 0, 9, 0)
    assert projector_distance(to_host(V), Vo) <= 1e-6


@pytest.mark.parametrize("specs,K", [([(5000, 700, 24, False)] * 2, 0), ([(12000, 512, 16, False)], 0), ([(3000, 516, 9, False), (2000, 1001, 5, True)], 2)])
def test_what_stays_with_the_cuda_cores_is_cut_for_them(specs, K):
    # fp32 without a power step, and a wave of both types: the same bits as where there are no products in parts, so the same token slabs
    X = [torch.randn(m, d, device=DEV).to(torch.bfloat16 if bf16 else torch.float32) for m, d, _, bf16 in specs]
    V = [[torch.zeros(r, d, device=DEV) for _, d, r, _ in specs] for _ in range(3)]
    for split in range(3):
        layers = [B.make_layer(X=x, V=v, r=s[2], layer_id=i) for i, (x, v, s) in enumerate(zip(X, V[split], specs))]
        with Ctx(layers) as ctx:
            B.agzo_set_option(ctx, "extract_resident", 0)
            B.agzo_set_option(ctx, "extract_split", split)
            B.agzo_extract_subspace(ctx, layers, 9, K)
            assert B.agzo_poll(ctx) == B.AGZO_OK
    for split in (1, 2):
        assert all(torch.equal(a, b) for a, b in zip(V[0], V[split])), split
