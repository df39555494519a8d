"""The one-warp Cholesky orders its lanes' accesses to the diagonal tile.

In warp_chol.cuh every lane of the warp loads the whole diagonal tile, factors
it in registers and stores it: nothing but a __syncwarp between the loads and
the stores keeps a lane that falls behind from loading factored values (lanes of
a warp need not run in lockstep).  No run can show such a race reliably, so the
order is checked in the source: in warp_cholesky, after the last load from the
tile and before the first store to it.
"""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1705_04159_gb300", "csrc",
                   "warp_chol.cuh")


def test_lanes_meet_between_the_loads_and_the_stores_of_the_diagonal_tile():
    with open(SRC) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    body = text[text.index("bool warp_cholesky("):]
    body = body[:body.index("\n}\n")]
    tile = body[body.index("float* D ="):]  # the diagonal tile of block column J
    loads = [m.end() for m in re.finditer(r"\bld8\(D\b", tile)]
    stores = [m.start() for m in re.finditer(r"reinterpret_cast<float4\*>\(D\b|\bst8\(D\b", tile)]
    assert loads and stores and loads[-1] < stores[0]
    assert "__syncwarp()" in tile[loads[-1]:stores[0]]
    # and the block column is complete before the next one reads it
    assert "__syncwarp()" in tile[tile.index("warp_panel<"):]
