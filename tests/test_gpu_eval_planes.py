"""Evaluation by planes (few points) against the oracle, and bit for bit
against the one-thread form that the same points take among many: every
number of lanes per point (2, 4, 8, 16), one field to more than a group's
lanes, point counts around a warp's, points that were not found."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("N,F,P", [(1, 3, 1), (2, 1, 31), (3, 5, 33), (4, 9, 7), (7, 1, 129), (7, 4, 1000), (8, 2, 63),
                                   (9, 17, 5), (12, 3, 65), (15, 2, 32)])
def test_planes(N, F, P, prec):
    import paper_1811_04891_gb300 as fg
    coords = synth.box_mesh((2, 2, 2), N, amp_frac=0.1)
    rng = np.random.default_rng(N)
    E, n3 = coords.shape[1], (N + 1) ** 3
    fields = rng.standard_normal((F, E, n3))
    many = 70000
    e = rng.integers(0, E, many).astype(np.int32)
    r = rng.uniform(-1, 1, (3, many))
    code = np.zeros(many, np.int32)
    code[3::11] = oracle.NOT_FOUND
    e[code == oracle.NOT_FOUND] = -1
    h = fg.fp_setup(torch.from_numpy(np.ascontiguousarray(coords)).cuda(), N, opts=fg.default_opts(precision=prec))
    fd = torch.from_numpy(fields).cuda()
    posted = fg.Fields(h, fd) if prec else None

    def ev(m):
        a = [torch.from_numpy(np.ascontiguousarray(x[..., :m])).cuda() for x in (code, e, r)]
        return (fg.fp_eval_df(h, posted, *a) if prec else fg.fp_eval(h, *a, fd)).cpu().numpy()

    few, all_ = ev(P), ev(many)
    np.testing.assert_array_equal(few, all_[:, :P])
    ref = oracle.evaluate(N, code[:P], e[:P], np.ascontiguousarray(r[:, :P]), fields)
    assert np.array_equal(np.isnan(few), np.isnan(ref))
    # sums of n^3 products, weights with sum of magnitudes below 5^3 for N <= 15; 2^-44 covers 2^-48 a term
    ok = ~np.isnan(ref)
    assert np.abs(few - ref)[ok].max(initial=0.0) <= (2.0 ** -44 if prec else 2.0 ** -46) * 125 * np.abs(fields).max()
    # the fused call: the find's own (e, r) evaluated by planes and one thread per pair
    pts = np.concatenate([oracle.map_points(coords, N, k, rng.uniform(-1, 1, (3, 5)))[0] for k in range(E)], axis=1)
    kw = {"fields": None, "posted": posted} if prec else {"fields": fd, "posted": None}
    one = fg.fp_find_eval(h, torch.from_numpy(np.ascontiguousarray(pts)).cuda(), **kw)[-1].cpu().numpy()
    k = 25000 // pts.shape[1] + 1
    rep = fg.fp_find_eval(h, torch.from_numpy(np.tile(pts, k)).cuda(), **kw)[-1].cpu().numpy()
    np.testing.assert_array_equal(rep.reshape(F, k, -1), np.repeat(one[:, None], k, axis=1))
