"""Threads per block of the Newton stage (fp_opts.points_per_block, any
multiple of 32): blocks that small calls shrink stay whole warps, and no size
changes a result.  Tile orders and an order with one thread per pair, both
forms, few pairs (one to a few blocks per SM, where blocks are shrunk) and
many."""
import numpy as np
import pytest

import synth
from gpu_util import gpu_find

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("N", [2, 4, 7, 9])
def test_every_block_size_gives_the_same_bits(N, prec):
    mesh, q = synth.deformed_cube(ne=6, N=N, P_uniform=9000, P_face=600)
    for P in (1, 150, 460, 800, q.P):
        pts = np.ascontiguousarray(q.pts[:, :P])
        base = gpu_find(mesh, pts, prec=prec)
        for block in (32, 96, 128, 160, 192, 224):
            g = gpu_find(mesh, pts, prec=prec, points_per_block=block)
            for k in ("code", "sub", "elem", "rst", "dist2"):
                np.testing.assert_array_equal(g[k], base[k], err_msg=f"{block} threads, {P} points, {k}")
