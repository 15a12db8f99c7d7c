"""Planning on the host, which every new list of layers pays for (a program whose activations are new in every step: each step)."""
import ctypes as C
import time

import pytest

from paper_2601_17261_b200 import binding as B

from test_tile_rows import BLOCK_0P6B, BLOCK_8B, layers_of


@pytest.mark.parametrize("shapes", [BLOCK_0P6B * 4, BLOCK_0P6B * 8, BLOCK_8B])
def test_shorter_items_are_found_quickly(shapes):
    # bf16 lists whose items make a few rounds over the SMs get some of them shorter; fp32 ones of the same shapes have no items.
    # Three to four times as long; going through the items one by one for every try took 12 to 70 times.
    def best(layers):
        arr, out, lib = B.layer_array(layers), C.c_size_t(0), B.lib()
        times = []
        for _ in range(40):
            t = time.perf_counter()
            for _ in range(5):
                assert lib.agzo_workspace_bytes(arr, len(layers), C.byref(out)) == B.AGZO_OK
            times.append(time.perf_counter() - t)
        return min(times)
    assert best(layers_of(shapes, 8, f32=False)) < 7 * best(layers_of(shapes, 8))


@pytest.mark.gpu
def test_two_kinds_of_token_slabs_are_planned_as_quickly_as_one():
    # where products run in parts every layer has two slab counts; 64 layers of as many tokens: 31 and 30 us, with each count tried out for each
    # layer several times 101 and 65
    import torch
    X, V = torch.zeros(4000, 256, device="cuda"), torch.zeros(2, 64, 8, 256, device="cuda")
    lists = [[B.make_layer(X=X, V=V[k, i], r=8, layer_id=i) for i in range(64)] for k in range(2)]
    ctx = B.agzo_create(lists[0])
    B.agzo_set_option(ctx, "share_inputs", 0)

    def best(split):
        B.agzo_set_option(ctx, "extract_split", split)
        times = []
        for k in range(60):                    # alternate lists: each is new to the plan
            t = time.perf_counter()
            B.agzo_query_fused(ctx, lists[k & 1])
            times.append(time.perf_counter() - t)
            torch.cuda.synchronize()
        return min(times)
    best(0)
    assert best(2) < 1.3 * best(0)
    B.agzo_destroy(ctx)
