"""The Gaussian generator over four million consecutive elements of a stream: uniforms down to the ends of their range (logarithms of
numbers next to 1, angles next to every quadrant boundary).

Tolerance: 2e-6 max(1, |g|), the bound every stream in the suite is held to; on top of it the root mean square of the
difference stays below 2e-7, a few units in the last place of fp32 at the size of a normal."""
import numpy as np
import pytest
import torch

from oracle import agzo_oracle as O
from paper_2601_17261_b200 import binding as B
from paper_2601_17261_b200 import workloads as WL

from gpu_helpers import DEV, Ctx, projector_distance, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed,layer", [(1, 0), (1 << 40, 77)])
def test_normals(seed, layer):
    n, r = 1 << 22, 4
    ctx = B.Context(0, 4096)
    got = B.agzo_debug_gaussian(ctx, seed, layer, 0, 0, n).cpu().numpy().astype(np.float64)
    want = O.gen_G(seed, layer, n // r, r).astype(np.float64).reshape(-1)
    d = np.abs(got - want)
    assert (d <= 2e-6 * np.maximum(1.0, np.abs(want))).all()
    assert np.sqrt(np.mean(d * d)) <= 2e-7
    assert np.isfinite(got).all()
    B.agzo_destroy(ctx)


@pytest.mark.parametrize("m", [301, 75777])
@pytest.mark.parametrize("r", [3, 61, 64])
def test_first_product_with_the_test_matrix(m, r):
    # K = 0 is qr(X^T Omega): one token a thread for the short batch, two (and an odd last token) for the long one
    d_in = 128
    X = WL.planted_activations(m, d_in, 16, seed=m, bf16=True)
    Xd = to_dev(X, True)[0]
    V = torch.zeros(r, d_in, device=DEV)
    layers = [B.make_layer(X=Xd, V=V, r=r, layer_id=4)]
    with Ctx(layers) as ctx:
        B.agzo_set_option(ctx, "extract_path", 2)
        B.agzo_extract_subspace(ctx, layers, 9, 0)
        assert B.agzo_poll(ctx) == B.AGZO_OK
    Vg = to_host(V)
    assert np.abs(Vg.astype(np.float64) @ Vg.T - np.eye(r)).max() <= 1e-5
    assert projector_distance(Vg, O.extract_subspace(X, r, 0, 9, 4)) <= 1e-3
