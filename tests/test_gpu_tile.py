"""The tensor-core Newton kernels at the sizes where a tile can go wrong:
elements with 1 to 33 points (a warp holds up to 32 pairs in two 16-row
tiles), points on faces, edges and corners, elements bent through a quarter
turn (no affine start), orders from the smallest to the largest that have
them."""
import types

import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_parity, gpu_find, oracle_find

pytestmark = pytest.mark.gpu

COUNTS = [1, 32, 7, 8, 9, 15, 16, 17, 31, 33, 2, 48]


def quarter_turns(N):
    """A ring of 4 x 2 x 2 elements of a quarter turn each, and one straight
    block of 2 x 2 x 2 sheared elements beside it."""
    z, _ = oracle.gll(N)
    t = 0.5 * (np.asarray(z) + 1.0)
    el = []
    for kz in range(2):
        for kr in range(2):
            for ka in range(4):
                Z, R, A = np.meshgrid(kz + t, 1.0 + 0.6 * (kr + t), 0.5 * np.pi * (ka + t), indexing="ij")
                el.append([R * np.cos(A), R * np.sin(A) + 0.05 * np.sin(3 * Z) * R, Z])
    for kz in range(2):
        for ky in range(2):
            for kx in range(2):
                Z, Y, X = np.meshgrid(kz + t, ky + t, kx + t, indexing="ij")
                el.append([4.0 + X + 0.2 * Y + 0.03 * np.sin(2 * X * Z), Y + 0.04 * np.sin(3 * X), Z + 0.1 * X])
    c = np.array(el).reshape(len(el), 3, (N + 1) ** 3).transpose(1, 0, 2)
    return types.SimpleNamespace(coords=np.ascontiguousarray(c), N=N, sub=np.zeros(len(el), np.int32), dist=None)


def points(mesh):
    rng = np.random.default_rng(mesh.N)
    pts = []
    for e in range(mesh.coords.shape[1]):
        r = rng.uniform(-1, 1, (3, COUNTS[e % len(COUNTS)]))
        r[rng.integers(0, 3), ::5] = rng.choice([-1.0, 1.0])
        if r.shape[1] > 30:
            r[:, 3] = [1.0, -1.0, 0.25]
            r[:, 4] = [-1.0, 1.0, 1.0]
        pts.append(oracle.map_points(mesh.coords, mesh.N, e, r)[0])
    out = np.array([[9.0, 0.0], [0.0, 9.0], [0.5, 0.5]])
    p = np.concatenate(pts + [out], axis=1)
    return np.ascontiguousarray(p[:, rng.permutation(p.shape[1])])


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("N", [3, 4, 5, 6, 7, 8, 9])
def test_tile_edges(N, prec):
    mesh = quarter_turns(N)
    pts = points(mesh)
    g = gpu_find(mesh, pts, prec=prec)
    r = oracle_find(mesh, pts)
    assert (r["code"] == oracle.NOT_FOUND).sum() == 2
    assert_parity(g, r, prec)
    # many more pairs (the two-launch sequence, other tiles): the same bits
    import paper_1811_04891_gb300 as fg
    k = 70000 // pts.shape[1] + 1
    many = fg.fp_find(g["handle"], torch.from_numpy(np.tile(pts, k)).cuda())
    for name, a in zip(["code", "sub", "elem", "rst", "dist2"], many):
        a = a.cpu().numpy()
        np.testing.assert_array_equal(a.reshape(a.shape[:-1] + (k, -1)), np.stack([g[name]] * k, axis=-2), err_msg=name)
