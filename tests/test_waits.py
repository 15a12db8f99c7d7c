"""Bounded waits in the kernels' sources.  A wait that runs out does so for each lane by itself, since lanes read the clock and the
barrier one after another; where a warp goes on together (votes, shuffles, tcgen05.ld), the answer has to be the warp's."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_17261_b200", "csrc")


def test_warps_of_the_products_in_parts_wait_together():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "agzo_extract_split.cu")).read())
    waits = re.findall(r"\bmbar_wait\w*(?=\()", src)
    assert len(waits) >= 7 and set(waits) == {"mbar_wait_warp", "mbar_wait_cluster_warp"}


def test_whichever_lane_waited_in_vain_tells_the_cluster():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "agzo_extract_resident.cu")).read())
    body = re.search(r"void product_failed\([^)]*\)\s*\{(.*?)\n\}", src, re.S).group(1)
    assert "st_cluster_u32" in body and not re.search(r"threadIdx|lane", body)
