"""The CUDA-core products X^T T and X Q at the edges of their tiles: columns around 128 and 512, tokens around the staging
and slab sizes, every rank class, fp32 and bf16 activations with and without vector-aligned rows.

Tolerance: fp32 sums over at most 1300 terms, 1e-5 orthonormality and 1e-4 projector distance (the fp32 rounding of the
products, about 1300 x 2^-24, against the spectrum's gap; the suite allows 1e-3 everywhere)."""
import numpy as np
import pytest
import torch

from oracle import agzo_oracle as O
from paper_2601_17261_b200 import binding as B
from paper_2601_17261_b200 import workloads as WL

from gpu_helpers import DEV, Ctx, projector_distance, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [1, 4, 5, 8, 9, 17])
@pytest.mark.parametrize("m,d_in", [(33, 17), (64, 127), (65, 128), (129, 516), (257, 130), (1300, 1032)])
@pytest.mark.parametrize("bf16,extra", [(False, 0), (False, 3), (True, 0), (True, 4), (True, 5)])
def test_cuda_core_extraction(r, m, d_in, bf16, extra):
    X = WL.planted_activations(m, d_in, min(16, d_in // 2), seed=m + d_in, bf16=bf16)
    Xd, _ = to_dev(X, bf16, pitch=d_in + extra if extra else None)
    V, V2, V3 = (torch.zeros(r, d_in, device=DEV) for _ in range(3))
    layers = [B.make_layer(X=Xd, V=V, r=r, layer_id=3)]
    with Ctx(layers) as ctx:
        B.agzo_set_option(ctx, "extract_path", 1)
        B.agzo_extract_subspace(ctx, layers, 9, 2)
        assert B.agzo_poll(ctx) == B.AGZO_OK
    Vo = O.extract_subspace(X, r, 2, 9, 3)
    B.agzo_debug_extract_static(Xd, V2, r, 2, 9, 3, B.STATIC_CHAIN)
    B.agzo_extract_subspace_static(Xd, V3, r, 2, 9, 3)           # by the faster kernels, these or the resident one
    for Vg in (to_host(V), to_host(V2), to_host(V3)):
        assert np.abs(Vg.astype(np.float64) @ Vg.T - np.eye(r)).max() <= 1e-5
        assert projector_distance(Vg, Vo) <= 1e-4


@pytest.mark.parametrize("m,d_in,r,bf16", [(528, 1376, 16, False), (194, 1568, 24, True), (447, 4538, 32, True), (1020, 2720, 5, False),
                                           (2016, 1500, 40, False), (243, 6272, 2, True)])
def test_a_workspace_with_room_for_slabs_of_256_tokens_is_enough(m, d_in, r, bf16):
    # more and shorter slabs are taken where the workspace has room for them; what must fit is slabs of at least 256 tokens
    up = lambda x: (x + 255) // 256 * 256
    slabs = -(-m // max(256, -(-(-(-m // 32)) // 32) * 32))
    need = up(4 * m * r) + up(4 * slabs * r * d_in) + up(4 * r * d_in) + up(8 * -(-d_in // 128) * r * r) + up(8 * r * r)
    X = WL.planted_activations(m, d_in, 16, seed=m, bf16=bf16)
    Xd = to_dev(X, bf16)[0]
    V = torch.zeros(r, d_in, device=DEV)
    layers = [B.make_layer(X=Xd, V=V, r=r, layer_id=1)]
    tables = 2048                                          # header, record, prefixes and descriptors of one layer, alignment
    assert tables + need < B.agzo_workspace_bytes(layers)
    ctx = B.Context(0, tables + need)
    B.agzo_set_option(ctx, "extract_path", 1)
    B.agzo_extract_subspace(ctx, layers, 7, 2)
    assert B.agzo_poll(ctx) == B.AGZO_OK
    B.agzo_destroy(ctx)
    Vg = to_host(V)
    assert np.abs(Vg.astype(np.float64) @ Vg.T - np.eye(r)).max() <= 1e-5
    assert projector_distance(Vg, O.extract_subspace(X, r, 2, 7, 1)) <= 1e-3
