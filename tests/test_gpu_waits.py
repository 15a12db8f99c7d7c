"""An extraction during which a bounded wait runs out leaves V = 0 and the status word says so; the next one is as ever.

The wait that runs out is the library's debug kernel, put between the extraction's own kernels by the all-reduce callback (the sum over
one rank: nothing to add), or one of a kernel's own, whose barrier expects more than comes."""
import pytest
import torch

from paper_2601_17261_b200 import binding as B
from paper_2601_17261_b200 import workloads as WL

from gpu_helpers import DEV, Ctx, to_dev

pytestmark = pytest.mark.gpu


# the panel QR up to rank 16 (shares sent), up to 32 (read from the peers), above (three launches); behind the tensor-core sweeps and fused
# power steps, the products in parts and the CUDA-core products; d_in = 200 leaves CTAs of a cluster without columns
@pytest.mark.parametrize("r,d_in,bf16,split", [(8, 1024, True, 1), (20, 512, True, 1), (40, 512, True, 1), (6, 200, False, 2), (12, 300, False, 0)])
def test_a_wait_that_ran_out_leaves_no_basis(r, d_in, bf16, split):
    m, K = 600, 2
    X = to_dev(WL.planted_activations(m, d_in, 64, seed=r, bf16=bf16), bf16)[0]
    V, V1 = torch.zeros(r, d_in + 8, device=DEV)[:, :d_in], torch.zeros(3, d_in, device=DEV)
    layers = [B.make_layer(X=X, V=V, r=r, layer_id=1), B.make_layer(X=X, V=V1, r=3, layer_id=2)]
    with Ctx(layers) as ctx:
        at, call = [-1], [0]

        def between(buf, stream):
            if call[0] == at[0]:
                B.agzo_debug_wait_timeout(ctx, stream)
            call[0] += 1

        def extract(when):
            at[0], call[0] = when, 0
            V.fill_(7.0)
            V1.fill_(7.0)
            B.agzo_extract_subspace(ctx, layers, 9, K)
            return V.clone(), V1.clone(), B.agzo_poll(ctx)

        B.agzo_set_option(ctx, "extract_split", split)
        B.agzo_set_allreduce(ctx, between)
        want, want1, status = extract(-1)
        assert status == B.AGZO_OK and call[0] == K + 1
        for when in (0, K):                       # before a power step, and before the round that stores V
            got, got1, status = extract(when)
            assert status == B.AGZO_ERR_TIMEOUT and not got.any() and not got1.any()
        got, got1, status = extract(-1)
        assert status == B.AGZO_OK and torch.equal(got, want) and torch.equal(got1, want1)
        # one that ran out before the call began is reported, and is none of the call's
        B.agzo_debug_wait_timeout(ctx)
        got, got1, status = extract(-1)
        assert status == B.AGZO_ERR_TIMEOUT and torch.equal(got, want) and torch.equal(got1, want1)


# clusters of 16 CTAs of the panel QR, and of two with ragged columns; products in parts without clusters, with clusters of four for T = X Q, and
# with several items per cluster
@pytest.mark.parametrize("kind,m,d_in,ranks,bf16", [
    (B.KC_PANEL_QR, 700, 2048, (8,), True), (B.KC_PANEL_QR, 700, 200, (16, 3), False), (B.KC_XT_T, 1300, 516, (8, 20), False),
    (B.KC_X_Q, 16384, 512, (8,), False), (B.KC_X_Q, 4000, 1024, (8,), False), (B.KC_X_Q, 5000, 1001, (8,), True), (B.KC_X_Q, 4600, 1024, (16,), False)])
def test_a_wait_of_a_kernel_runs_out(kind, m, d_in, ranks, bf16):
    X = torch.randn(m, d_in, device=DEV).to(torch.bfloat16 if bf16 else torch.float32)
    V = [torch.zeros(r, d_in, device=DEV) for r in ranks]
    layers = [B.make_layer(X=X, V=v, r=r, layer_id=i) for i, (v, r) in enumerate(zip(V, ranks))]
    with Ctx(layers) as ctx:
        B.agzo_set_option(ctx, "extract_resident", 0)
        B.agzo_set_option(ctx, "extract_split", 2)

        def extract(missing):
            B.agzo_set_option(ctx, "debug_missing_class", missing)
            for v in V:
                v.fill_(7.0)
            B.agzo_extract_subspace(ctx, layers, 9, 2)
            return B.agzo_poll(ctx), [v.clone() for v in V]

        status, want = extract(0)
        assert status == B.AGZO_OK
        for _ in range(3):
            status, got = extract(kind)
            assert status == B.AGZO_ERR_TIMEOUT and not any(v.any() for v in got)
            status, got = extract(0)
            assert status == B.AGZO_OK and all(torch.equal(a, b) for a, b in zip(got, want))
