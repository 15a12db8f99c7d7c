"""Layers that read one X as one operand panel: ranks that fill the panel's rows of eight and that leave padding, sums on
both sides of the fused power step's 16 ranks and of the sweeps' 128, with neighbours of their own input around them.

Tolerances are the suite's for extraction (1e-5 orthonormality, 1e-3 projector distance)."""
import numpy as np
import pytest
import torch

from oracle import agzo_oracle as O
from paper_2601_17261_b200 import binding as B
from paper_2601_17261_b200 import workloads as WL

from gpu_helpers import DEV, Ctx, projector_distance, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fused", [0, 1, 2])
@pytest.mark.parametrize("ranks", [(1, 1, 1), (4, 4, 4), (8, 8), (5, 11), (3, 2, 11), (5, 8, 4), (16, 16), (64, 63, 1), (64, 64, 1), (40, 60, 7, 30)])
@pytest.mark.parametrize("m,d_in", [(300, 264), (1153, 1032)])
def test_groups(fused, ranks, m, d_in):
    X = WL.planted_activations(m, d_in, 16, seed=m, bf16=True)
    Z = WL.planted_activations(m, d_in, 16, seed=m + 1, bf16=True)
    Xd, Zd = to_dev(X, True)[0], to_dev(Z, True)[0]
    rs = [7, *ranks, 6]
    src = [(Z, Zd), *[(X, Xd)] * len(ranks), (Z, Zd)]
    Vs = [torch.zeros(r, d_in, device=DEV) for r in rs]
    layers = [B.make_layer(X=x[1], V=V, r=r, layer_id=i) for i, (x, V, r) in enumerate(zip(src, Vs, rs))]
    with Ctx(layers) as ctx:
        B.agzo_set_option(ctx, "extract_path", 2)
        B.agzo_set_option(ctx, "extract_fused", fused)
        served = B.agzo_query_fused(ctx, layers)
        if fused == 2:
            assert [c > 0 for c in served[1:-1]] == [sum(ranks) <= 16 or r <= 16 for r in ranks]
        for K in (0, 2):
            B.agzo_extract_subspace(ctx, layers, 9, K)
            assert B.agzo_poll(ctx) == B.AGZO_OK
            for i, r in enumerate(rs):
                Vg = to_host(Vs[i])
                assert np.abs(Vg.astype(np.float64) @ Vg.T - np.eye(r)).max() <= 1e-5, (K, i)
                assert projector_distance(Vg, O.extract_subspace(src[i][0], r, K, 9, i)) <= 1e-3, (K, i)


@pytest.mark.parametrize("r", [1, 8, 24, 48, 64])
@pytest.mark.parametrize("m,d_in", [(256, 128), (300, 520), (613, 1024), (1300, 1480), (4000, 264)])
def test_columns_split_over_a_cluster(r, m, d_in):
    # few token tiles: T = X Q splits the columns over 2, 4 or 8 CTAs, with steps left over
    X = WL.planted_activations(m, d_in, 16, seed=m, bf16=True)
    Xd = to_dev(X, True)[0]
    V = torch.zeros(r, d_in, device=DEV)
    layers = [B.make_layer(X=Xd, V=V, r=r, layer_id=2)]
    with Ctx(layers) as ctx:
        B.agzo_set_option(ctx, "extract_path", 3)
        B.agzo_extract_subspace(ctx, layers, 4, 2)
        assert B.agzo_poll(ctx) == B.AGZO_OK
    Vg = to_host(V)
    assert np.abs(Vg.astype(np.float64) @ Vg.T - np.eye(r)).max() <= 1e-5
    assert projector_distance(Vg, O.extract_subspace(X, r, 2, 4, 2)) <= 1e-3


@pytest.mark.parametrize("ranks", [(48,), (24, 24), (64, 64)])
def test_two_blocks_per_cta(ranks):
    # enough tiles for two blocks of 128 rows per CTA; ragged tokens and columns leave half-empty pairs
    shapes = [(8300, 1160)] * 6 + [(8300, 904)] * 6
    Xs = {s: WL.planted_activations(*s, 16, seed=s[1], bf16=True) for s in set(shapes)}
    Xd = [to_dev(Xs[s], True)[0] for s in shapes]
    Vs, layers = [], []
    for i, s in enumerate(shapes):
        for r in ranks:
            Vs.append((s, r, torch.zeros(r, s[1], device=DEV)))
            layers.append(B.make_layer(X=Xd[i], V=Vs[-1][2], r=r, layer_id=len(layers)))
    with Ctx(layers) as ctx:
        B.agzo_extract_subspace(ctx, layers, 4, 1)
        assert B.agzo_poll(ctx) == B.AGZO_OK
    for i in (0, len(Vs) - 1):
        s, r, V = Vs[i]
        Vg = to_host(V)
        assert np.abs(Vg.astype(np.float64) @ Vg.T - np.eye(r)).max() <= 1e-5
        assert projector_distance(Vg, O.extract_subspace(Xs[s], r, 1, 4, i)) <= 1e-3


@pytest.mark.parametrize("r", [8, 16])
@pytest.mark.parametrize("widths", [(1024, 2048), (3072, 1024, 2048, 1024), (8192, 1024, 4096)])
def test_power_step_of_several_cluster_sizes(widths, r):
    # one launch per cluster size, running into one another; twice, with and without the device idle between the calls
    m = 1500
    Xs = [WL.planted_activations(m, d, 16, seed=i, bf16=True) for i, d in enumerate(widths)]
    Xd = [to_dev(X, True)[0] for X in Xs]
    runs = []
    for sync in (True, False):
        Vs = [[torch.zeros(r, d, device=DEV) for d in widths] for _ in range(3)]
        sets = [[B.make_layer(X=x, V=v, r=r, layer_id=i) for i, (x, v) in enumerate(zip(Xd, V))] for V in Vs]
        with Ctx(sets[0]) as ctx:
            B.agzo_set_option(ctx, "extract_fused", 2)
            assert len({c for c in B.agzo_query_fused(ctx, sets[0]) if c > 0}) >= 2
            for k, layers in enumerate(sets):
                B.agzo_extract_subspace(ctx, layers, k, 3)
                if sync:
                    torch.cuda.synchronize()
            assert B.agzo_poll(ctx) == B.AGZO_OK
        runs.append(Vs)
    for a, b in zip(runs[0], runs[1]):
        for x, y in zip(a, b):
            assert torch.equal(x, y)
    for i, d in enumerate(widths):
        Vg = to_host(runs[1][2][i])
        assert np.abs(Vg.astype(np.float64) @ Vg.T - np.eye(r)).max() <= 1e-5, i
        assert projector_distance(Vg, O.extract_subspace(Xs[i], r, 3, 2, i)) <= 1e-3, i
