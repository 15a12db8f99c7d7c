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


def test_parts_of_a_normal():
    """Every argument that the generator can get, against float64: the logarithm within 1.4 x 2^-24 relative, the root of what the
    logarithm gave within 1.01 x 2^-24 relative (one rounding and the step's own error), sine and cosine within 2^-24."""
    ctx, chunk, ulp = B.Context(0, 4096), 1 << 22, 2.0 ** -24
    for first in range(0, 1 << 24, chunk):
        y, s, sn, cs = B.agzo_debug_normal_parts(ctx, first, chunk).cpu().numpy().T
        k = np.arange(first, first + chunk, dtype=np.float64)
        want = -2.0 * np.log1p((k + 1.0 - 2.0 ** 24) * ulp)              # exact argument, accurate next to 1
        assert (np.abs(y - want) <= 1.4 * ulp * want).all()
        last = k == (1 << 24) - 1                                        # u = 1: y = 0, and a root that is no more than 1e-10
        assert (np.abs(s - np.sqrt(y.astype(np.float64))) <= np.where(last, 1e-10, 1.01 * ulp * s)).all()
        # quarter turns are exact: reduce by them in integers before the float64 functions
        turn, rest = np.divmod(np.arange(first, first + chunk) + (1 << 21), 1 << 22)
        x = 2.0 * np.pi * ulp * (rest - (1 << 21))
        quads = np.stack([np.sin(x), np.cos(x), -np.sin(x), -np.cos(x)])
        i = np.arange(chunk)
        assert (np.abs(sn - quads[turn % 4, i]) <= ulp).all()
        assert (np.abs(cs - quads[(turn + 1) % 4, i]) <= ulp).all()
    for first, n in ((0, (1 << 24) + 1), (1 << 24, 1), ((1 << 24) + 1, 0)):
        with pytest.raises(B.AgzoError):
            B.agzo_debug_normal_parts(ctx, first, n)
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


def test_dense_direction_beyond_one_launch():
    """A launch of the dense pass holds 2^34 elements; the ones after it belong to blocks whose numbers have another upper word."""
    n = (1 << 34) + 4096 + 5
    if torch.cuda.mem_get_info()[0] < 2 * n + (4 << 30):
        pytest.skip("needs 36 GB")
    w = torch.zeros(n, dtype=torch.bfloat16, device=DEV)
    ctx = B.Context(0, 4096)
    B.agzo_perturb_dense(ctx, w, 77, 3, 1.0)
    for first in (0, (1 << 34) - 2048, 1 << 34):
        k = min(4096 + 5, n - first)
        want = B.agzo_debug_gaussian(ctx, 77, 3, 2, first, k).to(torch.bfloat16)
        assert torch.equal(w[first:first + k], want)
    B.agzo_destroy(ctx)
    del w
    torch.cuda.empty_cache()
