"""How accurate the element map of the tensor-core kernels is, against residuals
in extended precision at the r that a find returns.  Bent elements around the
origin, where FP64 sum factorisation resolves the map to about 3e-16 of half an
element's width and sums of float pairs (with a double-float basis) to 1e-14."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def bent_box(N):
    t = np.asarray(oracle.gll(N)[0])
    el = []
    for e in range(8):
        Z, Y, X = np.meshgrid(*(t + (1 if e >> a & 1 else -1) for a in (2, 1, 0)), indexing="ij")
        el.append([X + 0.05 * np.sin(Y) * np.cos(0.5 * Z), Y + 0.06 * np.sin(0.7 * X), Z + 0.05 * np.sin(0.8 * X + 0.3 * Y)])
    return np.ascontiguousarray(np.array(el).reshape(8, 3, (N + 1) ** 3).transpose(1, 0, 2))


def basis(N, r):
    """h_i(r) in extended precision on the FP64 nodes."""
    xi = np.asarray(oracle.gll(N)[0]).astype(np.longdouble)
    h = []
    for i in range(N + 1):
        others = [m for m in range(N + 1) if m != i]
        h.append(np.prod([r - xi[m] for m in others], axis=0) / np.prod([xi[i] - xi[m] for m in others]))
    return h


def residuals(coords, N, elem, r, x):
    """x^e(r) - x in extended precision, [3][P]."""
    h = [basis(N, r[a].astype(np.longdouble)) for a in range(3)]
    out = []
    for a in range(3):
        X = coords[a][elem].astype(np.longdouble).reshape(-1, N + 1, N + 1, N + 1)
        v = sum(X[..., i] * h[0][i][:, None, None] for i in range(N + 1))
        v = sum(v[:, :, j] * h[1][j][:, None] for j in range(N + 1))
        v = sum(v[:, k] * h[2][k] for k in range(N + 1))
        out.append(v - x[a].astype(np.longdouble))
    return np.array(out).astype(float)


def find(N, prec, per):
    import paper_1811_04891_gb300 as fg
    coords = bent_box(N)
    rng = np.random.default_rng(N)
    pts = np.concatenate([oracle.map_points(coords, N, e, rng.uniform(-0.99, 0.99, (3, per)))[0] for e in range(8)], axis=1)
    h = fg.fp_setup(torch.from_numpy(coords).cuda(), N, opts=fg.default_opts(precision=prec))
    code, _, elem, rst, dist2 = (x.cpu().numpy() for x in fg.fp_find(h, torch.from_numpy(np.ascontiguousarray(pts)).cuda()))
    assert (code == 0).all()
    np.testing.assert_array_equal(elem, np.repeat(np.arange(8), per))
    return dist2, residuals(coords, N, elem, rst, pts)


@pytest.mark.parametrize("N", [3, 5, 7, 8, 9])
def test_fp64_form_resolves_fp64(N):
    """Half an element is 1 wide.  The map's error in a coordinate, computed
    with 6 digits and in FP64 by sum factorisation, is 2e-16 to 3e-16 rms, in
    the residual's length at most sqrt(3) of it; 1e-15 leaves a factor of two.
    Node and basis digits cut at 2^-50 give 4e-15."""
    dist2, f = find(N, 0, 60)
    err = np.sqrt(dist2) - np.sqrt((f ** 2).sum(0))
    assert np.sqrt(np.mean(err ** 2)) <= 1e-15
    assert np.abs(err).max() <= 5e-15


@pytest.mark.parametrize("N,rms", [(6, 1.07e-14), (8, 1.40e-14), (9, 1.40e-14)])
def test_mixed_form_resolves_float_pairs(N, rms):
    """Points whose last step was taken (their residual is that of the linear
    model, 0): what is left is the error of the compensated residual that the
    step came from, and 1e-4 of a step of at most 5e-11.  rms: that error by
    sums of float pairs, simulated operation by operation for these elements;
    the digits with orders 0 to 5 stay 1 to 5 % below it, without order 5
    they are 1.8 times as far off.  A quarter is allowed for the sample."""
    dist2, f = find(N, 1, 200)
    taken = dist2 == 0.0
    assert taken.sum() >= 50
    assert np.sqrt(np.mean(f[:, taken] ** 2)) <= 1.25 * rms
