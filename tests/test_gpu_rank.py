"""Ownership where 1 to 5 subdomains cover every point: one D^k per winner, up
to more of them than a block lists."""
import types

import numpy as np
import pytest

import oracle
from gpu_util import assert_parity, gpu_find, oracle_find

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nsub", [1, 2, 3, 4, 5])
def test_owner_among_covering_subdomains(nsub, prec):
    N = 4
    t = 0.5 * (np.asarray(oracle.gll(N)[0]) + 1.0)
    el, dist, sub = [], [], []
    for s in range(nsub):
        for kx in range(2):
            Z, Y, X = np.meshgrid(t, t, kx + t, indexing="ij")
            el.append([X + 0.02 * (s + 1) * np.sin(3 * Y) * X * (2 - X), Y, Z])
            # a plane per subdomain: each one is the largest somewhere
            dist.append(1.0 + 0.1 * np.cos(2.0 * s) * (X - 1) + 0.1 * np.sin(2.0 * s) * (2 * Y - 1) + 0.02 * s * Z)
            sub.append(s)
    E, n3 = len(el), (N + 1) ** 3
    mesh = types.SimpleNamespace(coords=np.ascontiguousarray(np.array(el).reshape(E, 3, n3).transpose(1, 0, 2)), N=N,
                                 sub=np.array(sub, np.int32), dist=np.ascontiguousarray(np.array(dist).reshape(E, n3)))
    rng = np.random.default_rng(nsub)
    pts = rng.uniform(0.05, 0.95, (3, 700)) * np.array([[2.0], [1.0], [1.0]])
    pts[0, ::13] = 1.0                                  # on the face between a subdomain's two elements
    g, r = gpu_find(mesh, pts, prec=prec), oracle_find(mesh, pts)
    assert set(np.unique(r["sub"])) == set(range(nsub))
    assert_parity(g, r, prec)
