"""An iteration captured into a CUDA graph (its layer list has been used before, so its tables are in place) gives on every replay
bit for bit what the calls give one by one: chained launches, helper streams and power steps of several launches among them."""
import pytest
import torch

from paper_2601_17261_b200 import binding as B
from paper_2601_17261_b200 import workloads as WL

from gpu_helpers import DEV, Ctx, to_dev

pytestmark = pytest.mark.gpu


def calls(ctx, layers, K, losses, g, vec):
    B.agzo_extract_subspace(ctx, layers, 5, K)
    B.agzo_perturb(ctx, layers, 5, 1e-2)
    B.agzo_perturb(ctx, layers, 5, -2e-2)
    B.agzo_ghat(ctx, losses[0:1], losses[1:2], 1e-2, 0, g)
    B.agzo_restore_update(ctx, layers, 5, 1e-2, 1e-1, 0, g)
    B.agzo_perturb_dense(ctx, vec, 5, 9, 1e-3, g)


@pytest.mark.parametrize("K", [1, 2])
@pytest.mark.parametrize("wave_bytes", [1, 1 << 40])            # a layer per wave on two helper streams; one wave
@pytest.mark.parametrize("r,bf16", [(4, False), (8, True), (24, True), (40, True)])
def test_replays(r, bf16, wave_bytes, K):
    shapes = [(512, 64), (1024, 300), (2048, 96), (1160, 40)]
    Xs = [to_dev(WL.planted_activations(600, d, 16, seed=i, bf16=bf16), bf16)[0] for i, (d, _) in enumerate(shapes)]
    W0 = [to_dev(WL.gaussian_weights(o, d, 0.02, seed=i, bf16=bf16), bf16)[0] for i, (d, o) in enumerate(shapes)]
    Ws, Vs = [w.clone() for w in W0], [torch.zeros(r, d, device=DEV) for d, _ in shapes]
    layers = [B.make_layer(X=X, W=W, V=V, r=r, layer_id=i) for i, (X, W, V) in enumerate(zip(Xs, Ws, Vs))]
    losses, g = torch.tensor([1.0, 0.999], dtype=torch.float64, device=DEV), torch.zeros(1, device=DEV)
    vec = torch.zeros(1000, device=DEV)
    state = [*Ws, *Vs, g, vec]

    def reset():
        torch.cuda.synchronize()
        for w, w0 in zip(Ws, W0):
            w.copy_(w0)
        for t in (*Vs, g, vec):
            t.zero_()
        torch.cuda.synchronize()

    s = torch.cuda.Stream()
    with Ctx(layers) as ctx:
        B.agzo_set_option(ctx, "wave_bytes", wave_bytes)
        B.agzo_set_option(ctx, "extract_fused", 2)
        with torch.cuda.stream(s):
            calls(ctx, layers, K, losses, g, vec)
        reset()
        with torch.cuda.stream(s):
            calls(ctx, layers, K, losses, g, vec)
        torch.cuda.synchronize()
        want = [t.clone() for t in state]
        reset()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            calls(ctx, layers, K, losses, g, vec)
        for _ in range(3):
            reset()
            graph.replay()
            torch.cuda.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(state, want))
        graph.replay()                           # back to back
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(Vs, want[len(Ws):]))
        assert B.agzo_poll(ctx) == B.AGZO_OK
        del graph


def two_lists(m=300, r=8):
    Xs = [to_dev(WL.planted_activations(m, d, 16, seed=d, bf16=True), True)[0] for d in (512, 264)]
    Vs = [torch.zeros(r, X.shape[1], device=DEV) for X in Xs]
    return Xs, Vs, [[B.make_layer(X=X, V=V, r=r, layer_id=i)] for i, (X, V) in enumerate(zip(Xs, Vs))]


def test_tables_uploaded_inside_a_capture_are_not_in_place_outside():
    # a list without weights that only the resident kernel has served has no tables: captured on the other kernels, its upload is a
    # node of the graph, so a call before the first replay brings its own
    _, Vs, (one, _) = two_lists()
    s = torch.cuda.Stream()
    with Ctx(one) as ctx:
        B.agzo_set_option(ctx, "extract_resident", 0)
        with torch.cuda.stream(s):
            B.agzo_extract_subspace(ctx, one, 5, 2)
        torch.cuda.synchronize()
        want = Vs[0].clone()
    with Ctx(one) as ctx:
        B.agzo_set_option(ctx, "extract_resident", 2)
        with torch.cuda.stream(s):
            B.agzo_extract_subspace(ctx, one, 5, 1)
        B.agzo_set_option(ctx, "extract_resident", 0)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            B.agzo_extract_subspace(ctx, one, 5, 2)
        B.agzo_read_counters(ctx)
        for replay in (False, True, True):
            Vs[0].zero_()
            if replay:
                graph.replay()
            else:
                B.agzo_extract_subspace(ctx, one, 5, 2)
                n = B.agzo_read_counters(ctx)[2]
            torch.cuda.synchronize()
            assert torch.equal(Vs[0], want)
        B.agzo_extract_subspace(ctx, one, 5, 2)                  # now they are: a launch less
        assert B.agzo_read_counters(ctx)[2] == n - 1
        assert B.agzo_poll(ctx) == B.AGZO_OK
        del graph


def test_a_list_used_again_is_in_place_for_its_graph():
    # another list's tables took the place of the captured one's; using that one again, by whichever kernels, brings them back
    _, Vs, (one, other) = two_lists()
    s = torch.cuda.Stream()
    ctx = B.Context(0, max(B.agzo_workspace_bytes(L) for L in (one, other)))
    B.agzo_set_option(ctx, "extract_resident", 0)
    with torch.cuda.stream(s):
        B.agzo_extract_subspace(ctx, one, 5, 2)
    torch.cuda.synchronize()
    want = Vs[0].clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        B.agzo_extract_subspace(ctx, one, 5, 2)
    with torch.cuda.stream(s):
        B.agzo_extract_subspace(ctx, other, 5, 2)
        B.agzo_set_option(ctx, "extract_resident", 2)
        B.agzo_extract_subspace(ctx, one, 5, 1)
    torch.cuda.synchronize()
    for V in Vs:
        V.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(Vs[0], want) and not Vs[1].any()
    assert B.agzo_poll(ctx) == B.AGZO_OK
    del graph
    B.agzo_destroy(ctx)


def test_a_list_without_tables_is_captured_beside_an_upload_on_another_stream():
    _, Vs, (one, other) = two_lists()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    ctx = B.Context(0, max(B.agzo_workspace_bytes(L) for L in (one, other)))
    B.agzo_set_option(ctx, "extract_resident", 0)
    with torch.cuda.stream(a):
        B.agzo_extract_subspace(ctx, other, 5, 2)                # uploads its tables on this stream
    torch.cuda.synchronize()
    B.agzo_set_option(ctx, "extract_resident", 2)
    with torch.cuda.stream(b):
        B.agzo_extract_subspace(ctx, one, 5, 2)
    torch.cuda.synchronize()
    want = Vs[0].clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=b):
        B.agzo_extract_subspace(ctx, one, 5, 2)
    Vs[0].zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(Vs[0], want)
    assert B.agzo_poll(ctx) == B.AGZO_OK
    del graph
    B.agzo_destroy(ctx)
