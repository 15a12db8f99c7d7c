"""Tensor-core in-place pass with several work items per CTA: the operand made from V is rebuilt between them (read 16 bytes
at a time where V's rows allow it, an element at a time elsewhere), items of every height, panels and row blocks cut off by
the layer's edges, and lists so short that the items are made smaller.

Tolerances are those of the pass's other tests (share of results on the neighbouring bf16 value from the split operands)."""
import numpy as np
import pytest
import torch

from oracle import agzo_oracle as O
from paper_2601_17261_b200 import binding as B
from paper_2601_17261_b200 import workloads as WL

from gpu_helpers import DEV, Ctx, assert_weights_match, cancellation_floor, tc_mismatch_bound, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [5, 16, 24, 40, 64])
@pytest.mark.parametrize("n,d_out,d_in,pad", [(1, 130, 264, 0), (7, 2100, 1288, 0), (7, 2100, 1288, 2)])
def test_items_that_rebuild_the_operand(n, d_out, d_in, pad, r):
    seed, c = 11, -2e-3
    W0 = WL.gaussian_weights(d_out, d_in, 0.02, seed=r, bf16=True)
    rng = np.random.default_rng(r)
    Vh = np.linalg.qr(rng.standard_normal((d_in, r)))[0].T.astype(np.float32).copy()
    Ws = [to_dev(W0, True)[0] for _ in range(n)]
    V = torch.full((r, d_in + pad), 5.0, device=DEV)[:, :d_in]
    V.copy_(torch.from_numpy(Vh))
    layers = [B.make_layer(W=W, V=V, r=r, layer_id=i) for i, W in enumerate(Ws)]
    with Ctx(layers, extra=1 << 22) as ctx:
        B.agzo_set_option(ctx, "rmw_path", 2)
        B.agzo_perturb(ctx, layers, seed, c)
        assert B.agzo_poll(ctx) == B.AGZO_OK
    for i in sorted({0, n // 2, n - 1}):
        want = O.apply_direction(W0, Vh, seed, i, np.float32(c), "bf16")
        assert_weights_match(to_host(Ws[i]), want, "bf16", frac=tc_mismatch_bound(want, c, seed, i, Vh),
                             floor=cancellation_floor(W0, c, seed, i, Vh, rel=2.0 ** -16))


@pytest.mark.parametrize("r", [12, 40])
def test_last_layers_of_a_few_rounds_have_shorter_items(r):
    # about one and a half rounds of items over the SMs: the last layers' are cut shorter, with remainders in both directions
    n, d_out, d_in, seed, c = 9, 1300, 1096, 13, 1e-3
    W0 = WL.gaussian_weights(d_out, d_in, 0.02, seed=r, bf16=True)
    Vh = np.linalg.qr(np.random.default_rng(r).standard_normal((d_in, r)))[0].T.astype(np.float32).copy()
    Ws, V = [to_dev(W0, True)[0] for _ in range(n)], to_dev(Vh, False)[0]
    layers = [B.make_layer(W=W, V=V, r=r, layer_id=i) for i, W in enumerate(Ws)]
    with Ctx(layers, extra=1 << 24) as ctx:
        B.agzo_perturb(ctx, layers, seed, c)
        assert B.agzo_poll(ctx) == B.AGZO_OK
    for i in (0, n - 2, n - 1):
        want = O.apply_direction(W0, Vh, seed, i, np.float32(c), "bf16")
        assert_weights_match(to_host(Ws[i]), want, "bf16", frac=tc_mismatch_bound(want, c, seed, i, Vh),
                             floor=cancellation_floor(W0, c, seed, i, Vh, rel=2.0 ** -16))
