"""qr(Y) at the edges of its dispatch: ranks around the tiles of eight, the change of form above rank 32, slices that
stay in shared memory and slices that do not, every cluster size (layers per launch), panels without 16-byte rows.

Tolerances: orthonormality 1e-5 (Q is rounded to fp32: r entries of 2^-24 relative error each, with the Gram matrix and
the factor in double); projectors 1e-3 as everywhere (the fp32 product before the factorisation)."""
import numpy as np
import pytest
import torch

from oracle import agzo_oracle as O
from paper_2601_17261_b200 import binding as B
from paper_2601_17261_b200 import workloads as WL

from gpu_helpers import DEV, Ctx, projector_distance, to_dev, to_host

pytestmark = pytest.mark.gpu


def check(m, dims, r, K, bf16, n_layers=1):
    Xs = [WL.planted_activations(m, d, min(16, d), seed=7 + d, bf16=bf16) for d in dims]
    devs = [to_dev(X, bf16)[0] for X in Xs]
    pick = [i % len(dims) for i in range(n_layers)]
    Vs = [torch.full((r, dims[p]), 7.0, device=DEV) for p in pick]
    layers = [B.make_layer(X=devs[p], V=V, r=r, layer_id=i) for i, (p, V) in enumerate(zip(pick, Vs))]
    with Ctx(layers) as ctx:
        B.agzo_set_option(ctx, "extract_resident", 0)            # the kernel of this file, whatever would be faster
        B.agzo_extract_subspace(ctx, layers, 5, K)
        assert B.agzo_poll(ctx) == B.AGZO_OK
    for i in sorted({0, n_layers // 2, n_layers - 1}):
        Vg = to_host(Vs[i])
        assert np.abs(Vg.astype(np.float64) @ Vg.T - np.eye(r)).max() <= 1e-5, i
        assert projector_distance(Vg, O.extract_subspace(Xs[pick[i]], r, K, 5, i)) <= 1e-3, i


@pytest.mark.parametrize("r", [1, 7, 8, 9, 16, 17, 32, 33, 40, 41, 64])
@pytest.mark.parametrize("d_in", [67, 130, 1160])
def test_ranks_and_columns(r, d_in):
    check(300, [d_in], r, 1, bf16=False)


@pytest.mark.parametrize("r,dims", [(16, [12288]), (16, [12416]), (32, [4096]), (8, [24704])])
def test_slices_in_and_out_of_shared_memory(r, dims):
    check(256, dims, r, 1, bf16=True)


# Shares of S sent or read: sixteen CTAs with the widest slices that leave room for the shares, and the next ones; two to eight CTAs
# (8, 9: layers per launch; 200, 300: chunks of columns), one of them without columns of its own
@pytest.mark.parametrize("r,dims,n_layers", [(16, [18432], 1), (16, [20480], 1), (8, [2176], 8), (8, [2176], 9), (4, [300], 1), (12, [200], 9),
                                             (16, [1160, 140], 12)])
def test_shares_sent_and_read(r, dims, n_layers):
    check(300, dims, r, 2, True, n_layers)


@pytest.mark.parametrize("n_layers", [40, 41, 80, 81])
def test_layers_per_launch(n_layers):
    check(256, [1032, 128, 3080], 12, 1, bf16=True, n_layers=n_layers)


@pytest.mark.parametrize("r", [3, 4, 8, 13, 24, 40, 64])
@pytest.mark.parametrize("power", [-12, -5, 7, 12])
@pytest.mark.parametrize("resident", [0, 2])                     # whose factorisation is the same code
def test_scaled_inputs_give_the_same_basis(r, power, resident):
    # every step scales exactly by powers of two (S by 4^n, its roots by 2^n, with two exponents of each parity), so V is
    # the same bit for bit; the roots see mantissas over the whole of [1, 4)
    X = WL.planted_activations(300, 264, 16, seed=r, bf16=True)
    got = []
    for scale in (1.0, 2.0 ** power):
        Xd = to_dev(X * np.float32(scale), True)[0]
        V = torch.zeros(r, 264, device=DEV)
        layers = [B.make_layer(X=Xd, V=V, r=r, layer_id=2)]
        with Ctx(layers) as ctx:
            B.agzo_set_option(ctx, "extract_resident", resident)
            B.agzo_extract_subspace(ctx, layers, 5, 1)
            assert B.agzo_poll(ctx) == B.AGZO_OK
        got.append(V)
    assert torch.equal(got[0], got[1])
    assert projector_distance(to_host(got[0]), O.extract_subspace(X, r, 1, 5, 2)) <= 1e-3
