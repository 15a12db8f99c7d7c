"""The products in bf16 parts on the tensor cores, at the edges of their steps of 64 and blocks of 128: columns and tokens around them,
rows that allow accesses of four columns and of one, ranks around the panels of 8, 16 and 24 and beyond one unit, several
layers on one X and more units than the short list of a launch holds, clusters of which some CTAs have no columns and clusters with
several items; their precision, and that they are what ran.

Tolerance: that of the CUDA-core products (fp32 sums over at most 1300 terms), which these replace: 1e-5 orthonormality and 1e-4
projector distance.  Where three parts are to be told from two: 2e-6.  On these inputs, emulated on the CPU with sums in fp32 and an accumulator
that truncates, three parts are at most 8e-7 from the oracle and two at least 3.8e-6."""
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


def ran_in_parts(ctx, layers, K=2):
    # a barrier of these kernels that expects more than comes: only where they run does the extraction then end with a wait that ran out
    found = []
    for kind in (B.KC_XT_T, B.KC_X_Q):
        B.agzo_set_option(ctx, "debug_missing_class", kind)
        B.agzo_extract_subspace(ctx, layers, 9, K)
        found.append(B.agzo_poll(ctx) == B.AGZO_ERR_TIMEOUT)
    B.agzo_set_option(ctx, "debug_missing_class", 0)
    return found


def extract_in_parts(specs, K):
    """specs: (m, d_in, r, bf16, extra columns of the pitch); V of each layer, after the oracle's bounds for three parts"""
    data, layers = [], []
    for i, (m, d, r, bf16, extra) in enumerate(specs):
        X = WL.planted_activations(m, d, min(32, d // 2), seed=m + d, bf16=bf16)
        Xd, V = to_dev(X, bf16, pitch=d + extra if extra else None)[0], torch.zeros(r, d, device=DEV)
        data.append((X, Xd, V))
        layers.append(B.make_layer(X=Xd, V=V, r=r, layer_id=3))
    with Ctx(layers) as ctx:
        options(ctx)
        assert ran_in_parts(ctx, layers, K) == [True, True]
        B.agzo_extract_subspace(ctx, layers, 9, K)
        assert B.agzo_poll(ctx) == B.AGZO_OK
    for (X, _, V), s in zip(data, specs):
        check(X, V, s[2], K, 9, 3, 2e-6)


@pytest.mark.parametrize("r", [1, 8, 17, 25])
@pytest.mark.parametrize("m,d_in", [(40, 40), (129, 132), (1300, 1032)])
@pytest.mark.parametrize("bf16,extra", [(False, 0), (False, 3), (True, 1)])
def test_products_in_parts_have_fp32_precision(r, m, d_in, bf16, extra):
    extract_in_parts([(m, d_in, r, bf16, extra)], 2)


# T = X Q on 148 SMs by clusters of four, whose CTAs have most to do 18 steps of 64 columns (one CTA an item 64, pairs 34): the unit of 4096 columns in
# one cluster, the 40 items of the other unit in the other 31, so nine of them have two; 64 columns leave three CTAs of four without any
@pytest.mark.parametrize("d_in", [64, 256])
@pytest.mark.parametrize("bf16", [False, True])
def test_clusters_with_empty_shares_and_several_items(d_in, bf16):
    extra = 1 if bf16 else 0
    extract_in_parts([(128, 4096, 4, bf16, extra), (5120, d_in, 4, bf16, extra)], 1)


def test_products_in_parts_where_they_pay_and_without_workspace():
    # two uses whose products are the faster ones in parts, in the automatic choice; the call without workspace takes the same route: the bits
    # of the context's call in parts, which the CUDA-core kernels do not give
    for m, d_in, bf16 in ((5000, 1001, True), (8000, 1024, False)):
        r = 8
        X = torch.randn(m, d_in, device=DEV).to(torch.bfloat16 if bf16 else torch.float32)
        V = torch.zeros(3, r, d_in, device=DEV)
        for split in (0, 1):
            layers = [B.make_layer(X=X, V=V[split], r=r, layer_id=3)]
            with Ctx(layers) as ctx:
                B.agzo_set_option(ctx, "extract_resident", 0)
                B.agzo_set_option(ctx, "extract_split", split)
                assert ran_in_parts(ctx, layers) == [split == 1] * 2
                B.agzo_extract_subspace(ctx, layers, 9, 2)
                assert B.agzo_poll(ctx) == B.AGZO_OK
        B.agzo_debug_extract_static(X, V[2], r, 2, 9, 3, B.STATIC_CHAIN)
        assert torch.equal(V[2], V[1]) and not torch.equal(V[2], V[0])


@pytest.mark.parametrize("m,d_in,r", [(7858, 828, 3), (9315, 584, 4), (9258, 1992, 5), (3965, 1388, 5)])
def test_the_cuda_cores_keep_single_fp32_layers_of_low_rank(m, d_in, r):
    # inputs that L2 holds: 6 to 24 % slower in parts, which the estimates favour by up to 15 %
    X, V = torch.randn(m, d_in, device=DEV), torch.zeros(2, r, d_in, device=DEV)
    layers = [B.make_layer(X=X, V=V[0], r=r, layer_id=3)]
    with Ctx(layers) as ctx:
        B.agzo_set_option(ctx, "extract_resident", 0)
        assert ran_in_parts(ctx, layers) == [False, False]
        B.agzo_extract_subspace(ctx, layers, 9, 2)
        assert B.agzo_poll(ctx) == B.AGZO_OK
    B.agzo_debug_extract_static(X, V[1], r, 2, 9, 3, B.STATIC_CHAIN)
    assert torch.equal(V[0], V[1])


def test_larger_fp32_sets_run_in_parts():
    # two 0.6B-shaped blocks, 229 MB: by estimate 4 % faster in parts, measured 17 %
    layers, keep = [], []
    for _ in range(2):
        for d_in, ranks in ((1024, (8, 8, 8)), (2048, (8,)), (1024, (8, 8)), (3072, (8,))):
            X = torch.randn(4000, d_in, device=DEV)
            keep.append((X, [torch.zeros(r, d_in, device=DEV) for r in ranks]))
            layers += [B.make_layer(X=X, V=v, r=8, layer_id=len(layers) + i) for i, v in enumerate(keep[-1][1])]
    with Ctx(layers) as ctx:
        assert ran_in_parts(ctx, layers) == [True, True]
