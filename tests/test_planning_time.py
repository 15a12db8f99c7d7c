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
