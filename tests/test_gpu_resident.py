"""Extraction by one kernel that keeps X in shared memory: blocks of 128 x 128 full, ragged and nearly empty, units on one CTA, one cluster
and several, columns of Y summed whole and in pieces, groups on one X, the forms of X that are read element by element, and the
launches in a row that share its counters.

Against the oracle at the suite's tolerances for extraction (1e-5 orthonormality, 1e-3 projector distance), and against the kernels
of the other paths on the same inputs: operands in three bf16 parts carry 24 bits, as fp32 does, so that both sides are within a
few 2^-24 sqrt(K + 1) of the exact basis times the spread of the spectrum (at most 5 in these inputs): 1e-5; operands in two
parts leave up to 2^-17 of an element, 2^-17 / sqrt(3) rms and of either sign, in each of 2 K + 1 products on both sides: times the
spread 7e-5 for K = 2, and 1e-4 (a product without one of its parts leaves 2^-9)."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import agzo_oracle as O
from paper_2601_17261_b200 import binding as B
from paper_2601_17261_b200 import workloads as WL

from gpu_helpers import DEV, Ctx, projector_distance, to_dev, to_host

pytestmark = pytest.mark.gpu


def launches(ctx, layers, seed, K):
    B.agzo_read_counters(ctx)
    B.agzo_extract_subspace(ctx, layers, seed, K)
    return B.agzo_read_counters(ctx)[2]


def check(units, K, seed=6, served=True, pieces=None):
    """units: (m, d_in, ranks of the layers on that X, bf16, pitch); pieces: which of them add Y up in pieces of its columns"""
    Xs, Vs, layers, held = [], [], [], []
    for n, (m, d, ranks, bf16, pitch) in enumerate(units):
        X = WL.planted_activations(m, d, min(16, d, m), seed=m + n, bf16=bf16)
        Xd = to_dev(X, bf16, pitch=pitch)[0]
        held.append(Xd)
        for r in ranks:
            Vb = torch.full((r + 2, d + 5), 7.0, device=DEV)
            Xs.append((X, r))
            Vs.append((Vb, Vb[1:1 + r, :d]))
            layers.append(B.make_layer(X=Xd, V=Vs[-1][1], r=r, layer_id=len(layers)))
    three = any(not b or d % 8 or d < 128 or m < 256 or (p or 0) % 8 for m, d, _, b, p in units)
    with Ctx(layers) as ctx:
        B.agzo_set_option(ctx, "extract_resident", 2)
        how = B.agzo_query_resident(ctx, layers, K)
        assert (len(how) == len(units)) == served and (pieces is None or [u["sub"] > 0 for u in how] == pieces), how
        n = launches(ctx, layers, seed, K)
        assert (n == 1) == served, n
        assert B.agzo_poll(ctx) == B.AGZO_OK
        first = [V.clone() for _, V in Vs]
        launches(ctx, layers, seed + 1, K)
        launches(ctx, layers, seed, K)
        assert all(torch.equal(a, V) for a, (_, V) in zip(first, Vs))
        B.agzo_set_option(ctx, "extract_resident", 0)
        assert launches(ctx, layers, seed, K) > 1
        assert B.agzo_poll(ctx) == B.AGZO_OK
    for i, ((X, r), a, (Vb, V)) in enumerate(zip(Xs, first, Vs)):
        got = to_host(a)
        assert np.abs(got.astype(np.float64) @ got.T - np.eye(r)).max() <= 1e-5, i
        assert projector_distance(got, O.extract_subspace(X, r, K, seed, i)) <= 1e-3, i
        assert float((a - V).norm() / V.norm()) <= (1e-5 if three else 1e-4), i
        edge = Vb.clone()
        edge[1:1 + r, :X.shape[1]] = 7.0
        assert bool((edge == 7.0).all()), i


@pytest.mark.parametrize("K", [0, 2])
@pytest.mark.parametrize("m,d_in,r,bf16,pitch", [
    (16, 16, 16, False, None), (64, 64, 4, True, None), (128, 128, 1, False, None), (129, 130, 3, False, 131), (127, 257, 8, True, 259),
    (300, 520, 16, True, 528), (512, 256, 4, False, None), (613, 1024, 8, True, None), (1000, 1000, 5, True, None), (1111, 515, 9, False, 516),
    (4096, 256, 16, False, None), (2100, 2048, 16, True, None), (4096, 2048, 16, True, None), (700, 4096, 12, True, None)])
def test_one_layer(m, d_in, r, bf16, pitch, K):
    check([(m, d_in, (r,), bf16, pitch)], K)


@pytest.mark.parametrize("ranks", [(8, 8, 8), (1, 1), (4, 4, 4), (5, 11), (16, 9), (3, 2, 11, 7), (1, 1, 1, 1, 1)])
@pytest.mark.parametrize("m,d_in,bf16", [(300, 264, True), (613, 1024, True), (257, 130, False)])
def test_layers_on_one_x(ranks, m, d_in, bf16):
    check([(m, d_in, ranks, bf16, None)], 2, served=sum(ranks) <= 24 and len(ranks) <= 4)


@pytest.mark.parametrize("units", [
    [(300, 256, (8, 8), True, None), (300, 512, (4,), True, None), (300, 264, (16, 2, 1), True, None)],
    [(512, 200 + 40 * i, (4,), False, None) for i in range(8)],
    [(613, 1024, (8, 8, 8), True, None), (613, 2048, (8,), True, None), (130, 128, (2,), True, None)]])
def test_units_side_by_side(units):
    check(units, 2)


# columns of Y added up in pieces that meet once more: groups of layers on one X with rows of padding between them, the last piece
# ragged or empty, element by element and in three parts, beside a unit that adds up whole columns
@pytest.mark.parametrize("units,pieces", [
    ([(8000, 1024, (12, 12), True, None)], [True]), ([(8000, 1000, (3, 5, 9), True, None)], [True]), ([(4000, 500, (5, 6, 8), False, None)], [True]),
    ([(8000, 250, (4, 4, 4), False, None)], [True]), ([(8000, 253, (2, 7), True, None)], [True]), ([(4096, 256, (8, 8), False, None)], [True]),
    ([(2000, 2048, (8, 8, 8), True, None)], None), ([(4000, 512, (9, 12), True, None), (300, 256, (4,), True, None)], None)])      # by the device's clusters
def test_columns_in_pieces(units, pieces):
    check(units, 2, pieces=pieces)


# What the CTAs of a cluster exchange, sent or read: clusters of two, four and eight side by side, one to three blocks of tokens, shares of
# all 512 elements, units without an exchange beside others, and both sides of where it is sent (six clusters; 1024 pieces of T)
@pytest.mark.parametrize("units", [
    [(128, 256, (4,), True, None)], [(320, 280, (8,), True, None), (1974, 128, (8,), True, None)], [(300, 264, (9, 9, 1, 1), True, None)],
    [(384, 512, (16,), False, None)], [(44, 136, (6,), True, None)], [(250, 1000, (9, 9, 1, 1), False, None)],
    [(613, 1024, (8, 8, 8), True, None), (613, 2048, (8,), True, None)], [(640, 1024, (16,), True, None)], [(1000, 1024, (16,), True, None)],
    [(2500, 1024, (8,), True, None)], [(2500, 1024, (16,), True, None)], [(2385, 1125, (4, 7), True, None), (127, 872, (7, 4), True, None)]])
@pytest.mark.parametrize("K", [1, 3])
def test_exchange_within_a_cluster(units, K):
    check(units, K)


def test_a_refused_launch_leaves_the_call_to_the_other_kernels():
    X = to_dev(WL.planted_activations(300, 256, 16, seed=1, bf16=True), True)[0]
    V = torch.zeros(4, 256, device=DEV)
    layers = [B.make_layer(X=X, V=V, r=4, layer_id=0)]
    with Ctx(layers) as ctx:
        B.agzo_set_option(ctx, "extract_resident", 0)
        n = launches(ctx, layers, 5, 2)
        want = V.clone()
        B.agzo_set_option(ctx, "extract_resident", 2)
        assert launches(ctx, layers, 5, 2) == 1
        B.agzo_set_option(ctx, "debug_refuse_resident", 1)
        V.zero_()
        assert launches(ctx, layers, 5, 2) == n - 1              # the same kernels; the tables are in place
        assert torch.equal(V, want)
        assert B.agzo_poll(ctx) == B.AGZO_OK


def test_static_entry_and_what_it_reports():
    for m, d_in, r, bf16 in [(700, 256, 4, False), (300, 130, 16, True), (1500, 520, 8, True)]:
        X = WL.planted_activations(m, d_in, 16, seed=m, bf16=bf16)
        Xd = to_dev(X, bf16)[0]
        V, flag = torch.zeros(r, d_in, device=DEV), torch.full((1,), -1, dtype=torch.int32, device=DEV)
        B.agzo_debug_extract_static(Xd, V, r, 2, 3, 7, B.STATIC_RESIDENT, flag)
        assert flag.item() == 0
        other, both = torch.zeros_like(V), torch.zeros_like(V)
        B.agzo_extract_subspace_static(Xd, both, r, 2, 3, 7)     # one of the two, bit for bit
        B.agzo_debug_extract_static(Xd, other, r, 2, 3, 7, B.STATIC_CHAIN)
        assert not torch.equal(V, other) and (torch.equal(both, V) or torch.equal(both, other))
        assert float((V - other).norm() / V.norm()) <= 1e-5
        assert projector_distance(to_host(V), O.extract_subspace(X, r, 2, 3, 7)) <= 1e-3
        Xd[:, 2:] = 0                                          # rank two
        B.agzo_debug_extract_static(Xd, V, r, 2, 3, 7, B.STATIC_RESIDENT, flag)
        assert flag.item() == 1 and int((V.norm(dim=1) == 0).sum()) == r - 2


def test_dependent_columns_and_a_small_workspace():
    m, d_in, r = 400, 384, 8
    X = torch.zeros(m, d_in, dtype=torch.bfloat16, device=DEV)
    X[:, :3] = torch.randn(m, 3, device=DEV)
    V = torch.zeros(r, d_in, device=DEV)
    layers = [B.make_layer(X=X, V=V, r=r, layer_id=0)]
    with Ctx(layers) as ctx:
        B.agzo_set_option(ctx, "extract_resident", 2)
        assert launches(ctx, layers, 1, 2) == 1
        assert B.agzo_poll(ctx) == B.AGZO_WARN_RANK_DEFICIENT
        assert B.agzo_poll(ctx) == B.AGZO_OK
        assert int((V.norm(dim=1) == 0).sum()) == r - 3
    # a workspace without room for it: the other kernels, or their refusal
    Y = torch.randn(2048, 256, device=DEV)
    W = torch.zeros(4, 256, device=DEV)
    layers = [B.make_layer(X=Y, V=W, r=4, layer_id=0)]
    size = 4096 + 2048 * 16 + 3 * 4096
    small = B.Context(0, size)
    B.agzo_destroy(small)                                        # the same on the inside of a larger buffer
    around = torch.full((size + 2 * (1 << 20),), 0x5a, dtype=torch.uint8, device=DEV)
    small.handle = C.c_void_p()
    assert B.lib().agzo_create(C.byref(small.handle), 0, around.data_ptr() + (1 << 20), size) == B.AGZO_OK
    B.agzo_set_option(small, "extract_resident", 2)
    assert launches(small, layers, 1, 1) > 1 and B.agzo_query_resident(small, layers, 1) == []
    a = W.clone()
    assert bool((around[:1 << 20] == 0x5a).all()) and bool((around[-(1 << 20):] == 0x5a).all())
    with Ctx(layers) as ctx:
        B.agzo_set_option(ctx, "extract_resident", 2)
        assert launches(ctx, layers, 1, 1) == 1
    assert float((a - W).norm() / W.norm()) <= 1e-5
    B.agzo_destroy(small)


def test_a_graph_of_it_replays():
    X = to_dev(WL.planted_activations(900, 640, 16, seed=1, bf16=True), True)[0]
    V = torch.zeros(8, 640, device=DEV)
    layers = [B.make_layer(X=X, V=V, r=8, layer_id=0)]
    s = torch.cuda.Stream()
    with Ctx(layers) as ctx:
        B.agzo_set_option(ctx, "extract_resident", 2)
        with torch.cuda.stream(s):
            assert launches(ctx, layers, 5, 2) == 1
        torch.cuda.synchronize()
        want = V.clone()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            B.agzo_extract_subspace(ctx, layers, 5, 2)
        for _ in range(3):
            V.zero_()
            graph.replay()
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(V, want)
        del graph


def test_static_entry_reports_a_wait_that_ran_out():
    # 128 blocks that meet eight times, one of which comes to the first meeting 0.1 ms later than the others wait
    X = to_dev(WL.planted_activations(4096, 2048, 16, seed=3, bf16=True), True)[0]
    want, V = torch.zeros(16, 2048, device=DEV), torch.zeros(16, 2048, device=DEV)
    flag = torch.full((1,), -1, dtype=torch.int32, device=DEV)
    B.agzo_debug_extract_static(X, want, 16, 3, 5, 1, B.STATIC_RESIDENT, flag)
    assert flag.item() == 0 and want.any()
    for _ in range(3):
        V.fill_(7.0)
        B.agzo_debug_extract_static(X, V, 16, 3, 5, 1, B.STATIC_RESIDENT, flag, wait_ns=0)
        assert flag.item() == 2 and not V.any()
        B.agzo_extract_subspace_static(X, V, 16, 3, 5, 1, flag)         # the next call is whole again
        assert flag.item() == 0 and torch.equal(V, want)


def test_a_wait_that_ran_out_where_a_cluster_sends():
    # 96 blocks, twelve clusters of eight that send one another their sums; the rest as above
    X = to_dev(WL.planted_activations(1500, 1024, 16, seed=3, bf16=True), True)[0]
    want, V = torch.zeros(8, 1024, device=DEV), torch.zeros(8, 1024, device=DEV)
    flag = torch.full((1,), -1, dtype=torch.int32, device=DEV)
    B.agzo_debug_extract_static(X, want, 8, 3, 5, 1, B.STATIC_RESIDENT, flag)
    assert flag.item() == 0 and want.any()
    for _ in range(3):
        V.fill_(7.0)
        B.agzo_debug_extract_static(X, V, 8, 3, 5, 1, B.STATIC_RESIDENT, flag, wait_ns=0)
        assert flag.item() == 2 and not V.any()
        B.agzo_debug_extract_static(X, V, 8, 3, 5, 1, B.STATIC_RESIDENT, flag)
        assert flag.item() == 0 and torch.equal(V, want)


@pytest.mark.parametrize("d_in", [128, 130])
def test_tiny_fp32_inputs_keep_their_bits(d_in):
    # scaled by a power of two that leaves every element a normal fp32 number: without a power step nothing underflows, so V is that of
    # the unscaled inputs to fp32 rounding of sums of 300 terms (300 x 2^-24 = 2e-5 at worst, 1e-6 with rounding errors of random sign)
    X = to_dev(WL.planted_activations(300, d_in, 16, seed=2, bf16=False), False)[0]
    X = torch.where(X.abs() < 2.0 ** -6, torch.zeros_like(X), X)
    tiny = X * 2.0 ** -118
    assert torch.equal(tiny * 2.0 ** 118, X)
    V, T = torch.zeros(8, d_in, device=DEV), torch.zeros(8, d_in, device=DEV)
    one, two = [[B.make_layer(X=A, V=A2, r=8, layer_id=1)] for A, A2 in ((X, V), (tiny, T))]
    with Ctx(one) as ctx:
        B.agzo_extract_subspace(ctx, one, 5, 0)
        B.agzo_extract_subspace(ctx, two, 5, 0)
        assert B.agzo_poll(ctx) == B.AGZO_OK
    assert float((T - V).norm() / V.norm()) <= 1e-6
    B.agzo_extract_subspace_static(tiny, T, 8, 0, 5, 1)
    assert float((T - V).norm() / V.norm()) <= 1e-6


def test_kernel_classes_are_timed():
    # asking for the time of a kernel of the chain has the chain run, asking for the resident kernel's or for a pass's does not
    X = to_dev(WL.planted_activations(300, 256, 16, seed=1, bf16=True), True)[0]
    V = torch.zeros(4, 256, device=DEV)
    layers = [B.make_layer(X=X, V=V, r=4, layer_id=0)]
    with Ctx(layers) as ctx:
        B.agzo_extract_subspace(ctx, layers, 5, 2)
        B.agzo_read_counters(ctx)
        for kind, timed, all_of_them in ((B.KC_RESIDENT, 1, 1), (B.KC_RMW, 0, 1), (B.KC_PANEL_QR, 3, None), (B.KC_TC_XT_T, 3, None), (0, 0, 1)):
            B.agzo_set_option(ctx, "time_kernel_class", kind)
            B.agzo_extract_subspace(ctx, layers, 5, 2)
            ms, n, total = B.agzo_read_counters(ctx)
            assert n == timed and (ms > 0) == (timed > 0), kind
            assert total == 1 if all_of_them else total > 3, kind


@pytest.mark.parametrize("resident", [0, 1, 2])
def test_a_workspace_that_the_other_kernels_refuse_is_refused(resident):
    X, V = torch.randn(2048, 256, device=DEV), torch.full((4, 256), 7.0, device=DEV)
    layers = [B.make_layer(X=X, V=V, r=4, layer_id=0)]
    ctx = B.Context(0, 16384)                                    # tables fit, T does not
    B.agzo_set_option(ctx, "extract_resident", resident)
    for _ in range(2):
        with pytest.raises(B.AgzoError) as e:
            B.agzo_extract_subspace(ctx, layers, 1, 3)
        assert e.value.status == B.AGZO_ERR_WORKSPACE
    torch.cuda.synchronize()
    assert bool((V == 7.0).all())
    B.agzo_destroy(ctx)


def test_the_default_takes_the_faster_kernels():
    # lists that either side serves at least 20 % faster (measured on this chip): 300 x 256 29 against 43 us, 4000 x 1024 fp32 and
    # element by element far more; few tokens on wide layers 45 against 32, and fp32 without a power step stays where its bits are
    for units, K, resident in [([(300, 256, (4,), True)], 3, True), ([(1000, 1003, (8,), True)], 3, True), ([(300, 256, (4,), True)], 1, True),
                               ([(130, 3072, (8, 8, 8), True)], 1, False), ([(130, 2048, (4, 4, 4), True)], 1, False),
                               ([(300, 130, (4,), False)], 0, False), ([(300, 130, (4,), False)], 3, True), ([(16384, 1024, (8,), True)], 3, False)]:
        layers, keep = [], []
        for m, d, ranks, bf16 in units:
            X = torch.randn(m, d, device=DEV).to(torch.bfloat16 if bf16 else torch.float32)
            for r in ranks:
                keep += [X, torch.zeros(r, d, device=DEV)]
                layers.append(B.make_layer(X=X, V=keep[-1], r=r, layer_id=len(layers)))
        with Ctx(layers) as ctx:
            assert (launches(ctx, layers, 1, K) == 1) == resident, (units, K)
            assert B.agzo_poll(ctx) == B.AGZO_OK
