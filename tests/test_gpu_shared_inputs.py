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
