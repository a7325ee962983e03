"""Elements of a boundary layer: a column of elements 0.1 wide and 0.1 / ratio
thin on the plane z = 0, bent in every direction.  Each coordinate has to keep
its own relative accuracy: r along the thin direction is as accurate as along
the wide ones, and the mixed form's FP32 steps still reach the solution."""
import types

import numpy as np
import pytest

import oracle
from gpu_util import assert_parity, gpu_find, oracle_find

pytestmark = pytest.mark.gpu


def layer(N, ratio):
    z, _ = oracle.gll(N)
    t = 0.5 * np.asarray(z)
    el = []
    for k in range(4):
        Z, Y, X = np.meshgrid(k + 0.5 + t, t, t, indexing="ij")
        el.append([0.1 * (X + 0.04 * np.sin(2 * Y)), 0.1 * (Y + 0.04 * np.sin(3 * X)),
                   0.1 / ratio * Z * (1 + 0.05 * np.sin(2 * X) * np.cos(1.7 * Y))])
    c = np.array(el).reshape(4, 3, (N + 1) ** 3).transpose(1, 0, 2)
    mesh = types.SimpleNamespace(coords=np.ascontiguousarray(c), N=N, sub=np.zeros(4, np.int32), dist=None)
    rng = np.random.default_rng(N)
    pts = [oracle.map_points(mesh.coords, N, e, rng.uniform(-0.999, 0.999, (3, 500)))[0] for e in range(4)]
    return mesh, np.ascontiguousarray(np.concatenate(pts, axis=1)[:, rng.permutation(2000)])


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("N,ratio", [(3, 1000), (4, 100), (4, 1000), (7, 1), (7, 100), (7, 1000), (9, 1000)])
def test_layer_parity(N, ratio, prec):
    # FP64 form: solves end at steps of at most 2 eps |x*| ||J^-1|| = 4.4e-16 * 0.06 * 2e4 = 5e-13
    # at ratio 1000, the oracle's at 1e-13: within the 1e-12 of every parity test
    mesh, pts = layer(N, ratio)
    g = gpu_find(mesh, pts, prec=prec)
    r = oracle_find(mesh, pts)
    assert (r["code"] == oracle.INSIDE).all()
    assert_parity(g, r, prec)


@pytest.mark.parametrize("N,ratio", [(4, 1000), (7, 1000), (7, 10000), (9, 10000)])
def test_layer_needs_no_fallback(N, ratio):
    mesh, pts = layer(N, ratio)
    g = gpu_find(mesh, pts, prec=1, paths=True)
    assert (g["code"] == 0).all()
    assert g["paths"]["fallback"] == 0 and g["paths"]["fp32_not_converged"] == 0, g["paths"]
