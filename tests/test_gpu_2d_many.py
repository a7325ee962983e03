"""Quadrilateral solves of a large call (FP32 starts, the rest listed and solved
by a second launch) and of a small one (every solve from the nearest node, one
launch): both against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from gpu_kernels import kernel_names
from gpu_util import assert_parity
from test_gpu_2d_start import rings

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 2, 7, 11, 15])
def test_few_and_many(N):
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
    ref = oracle.find(coords, N, sub, pts)
    for k, listed in ((1, False), (70, True)):
        many = torch.from_numpy(np.ascontiguousarray(np.tile(pts, k))).cuda()
        out, names = kernel_names(lambda: fg.fp_find(h, many))
        out = [x.cpu().numpy() for x in out]
        assert any("k_newton2" in v for v in names) and any("k_newton2_listed" in v for v in names) == listed
        tiled = {key: np.tile(ref[key], k) for key in ("code", "sub", "elem", "rst", "dist2")}
        assert_parity(dict(zip(["code", "sub", "elem", "rst", "dist2"], out)), tiled, 0)
