"""Starts of the quadrilateral Newton solves: elements bent through a quarter
turn (nearest node) beside sheared ones (affine start and FP32 steps), points
inside, on edges and corners, near them and outside."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_parity

pytestmark = pytest.mark.gpu


def rings(N):
    t = 0.5 * (np.asarray(oracle.gll(N)[0]) + 1.0)
    el = []
    for kr in range(2):
        for ka in range(4):
            R, A = np.meshgrid(1.0 + 0.6 * (kr + t), 0.5 * np.pi * (ka + t), indexing="ij")
            el.append([R * np.cos(A), R * np.sin(A)])
    for ky in range(3):
        for kx in range(3):
            Y, X = np.meshgrid(ky + t, kx + t, indexing="ij")
            el.append([4.0 + X + 0.3 * Y + 0.05 * np.sin(2 * X), Y + 0.05 * np.sin(3 * X) - 0.2 * X])
    c = np.array(el).reshape(len(el), 2, (N + 1) ** 2).transpose(1, 0, 2)
    return np.ascontiguousarray(c)


@pytest.mark.parametrize("N", [1, 2, 7, 11, 15])
def test_2d_starts(N):
    import paper_1811_04891_gb300 as fg
    coords = rings(N)
    E = coords.shape[1]
    rng = np.random.default_rng(N)
    pts = []
    for e in range(E):
        r = rng.uniform(-1, 1, (2, 40))
        r[0, :6] = [-1.0, 1.0, 1.0, 0.3, -1.0, 0.999999]
        r[1, :6] = [-1.0, 1.0, 0.2, -1.0, 0.5, -0.4]
        pts.append(oracle.map_points(coords, N, e, r)[0])
    pts = np.ascontiguousarray(np.concatenate(pts + [np.array([[0.0, 30.0], [0.1, 30.0]])], axis=1))
    sub = np.zeros(E, np.int32)
    h = fg.fp_setup_2d(torch.from_numpy(coords).cuda(), N, torch.from_numpy(sub).cuda(), None, opts=fg.default_opts())
    out = [x.cpu().numpy() for x in fg.fp_find(h, torch.from_numpy(pts).cuda())]
    ref = oracle.find(coords, N, sub, pts)
    assert (ref["code"] == oracle.NOT_FOUND).sum() == 2
    assert_parity(dict(zip(["code", "sub", "elem", "rst", "dist2"], out)), ref, 0)
