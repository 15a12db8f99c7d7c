"""A power step of several cluster sizes is several launches that run into one another: the first publishes, under the step's
number, that the operand panel is there, the others read the panel only once they have seen that number, and the extraction's last
round takes the number back.  The word lies in the status record at the start of the workspace (one per scratch region, after
four others); the all-reduce callback, called between the rounds on the caller's stream, is where it can be looked at."""
import numpy as np
import pytest
import torch

from oracle import agzo_oracle as O
from paper_2601_17261_b200 import binding as B
from paper_2601_17261_b200 import workloads as WL

from gpu_helpers import DEV, Ctx, projector_distance, to_dev, to_host

pytestmark = pytest.mark.gpu
K = 3


def panel_ready(ctx):
    return ctx.workspace[:24].view(torch.int32)[4:6].tolist()


@pytest.mark.parametrize("last_r", [4, 40])         # 40: the round's factorisation is three launches, the layer takes the sweeps
@pytest.mark.parametrize("d_ins", [(512,), (512, 1024), (512, 1024, 2048)])
def test_the_first_launch_of_a_step_publishes_the_panel(d_ins, last_r):
    specs = [(700 + 130 * i, d, 8) for i, d in enumerate(d_ins)] + [(640, 4608, last_r)]
    Xs = [WL.planted_activations(m, d, 16, seed=30 + i, bf16=True) for i, (m, d, _) in enumerate(specs)]
    devs = [(to_dev(X, True)[0], torch.zeros(r, d, device=DEV)) for X, (m, d, r) in zip(Xs, specs)]
    layers = [B.make_layer(X=X, V=V, r=V.shape[0], layer_id=i) for i, (X, V) in enumerate(devs)]
    seen = []

    def look(buf, stream):
        torch.cuda.synchronize()
        seen.append(panel_ready(ctx))

    with Ctx(layers) as ctx:
        B.agzo_set_option(ctx, "extract_path", 2)
        B.agzo_set_option(ctx, "extract_fused", 2)
        sizes = {c for c in B.agzo_query_fused(ctx, layers) if c}
        assert len(sizes) >= len(d_ins)
        B.agzo_set_allreduce(ctx, look, 0)
        for _ in range(2):
            B.agzo_extract_subspace(ctx, layers, 5, K)
            torch.cuda.synchronize()
            seen.append(panel_ready(ctx))
            assert B.agzo_poll(ctx) == B.AGZO_OK
    several = len(sizes) > 1
    assert seen == [[s if several else 0, 0] for s in (0, 1, 2, 3, 0, 0, 4, 5, 6, 0)]
    for i, (X, (_, V)) in enumerate(zip(Xs, devs)):
        Vg = to_host(V)
        assert np.abs(Vg.astype(np.float64) @ Vg.T - np.eye(V.shape[0])).max() <= 1e-5
        assert projector_distance(Vg, O.extract_subspace(X, V.shape[0], K, 5, i)) <= 1e-3
