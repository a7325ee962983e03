"""Which kernel an evaluation runs (the forms give the same bits): staging in
shared memory whenever it is asked for, planes only where they are the faster
form, and every form of a fused evaluation against the separate one."""
import numpy as np
import pytest
import torch

import synth
from gpu_kernels import kernel_names

pytestmark = pytest.mark.gpu


def setup(N, F, P, prec):
    import paper_1811_04891_gb300 as fg
    mesh, q = synth.deformed_cube(ne=4, N=N, P_uniform=P, P_face=0)
    h = fg.fp_setup(torch.from_numpy(mesh.coords).cuda(), N, opts=fg.default_opts(precision=prec))
    fields = torch.from_numpy(np.random.default_rng(N).standard_normal((F, mesh.E, (N + 1) ** 3))).cuda()
    posted = fg.Fields(h, fields) if prec else None
    return fg, h, torch.from_numpy(np.ascontiguousarray(q.pts)).cuda(), {"fields": None if prec else fields, "posted": posted}


def has(names, kernel):
    return any(kernel in n for n in names)


@pytest.mark.parametrize("N,F,P", [(7, 4, 1500), (7, 5, 24000), (3, 2, 500)])
def test_staging_is_done_when_asked_for(N, F, P):
    fg, h, pts, kw = setup(N, F, P, 1)
    plain, names = kernel_names(lambda: fg.fp_find_eval(h, pts, **kw))
    assert not has(names, "k_eval_pairs_staged")
    fg.fp_set_eval_staging(h, True)
    staged, names = kernel_names(lambda: fg.fp_find_eval(h, pts, **kw))
    assert has(names, "k_eval_pairs_staged")
    for a, b in zip(plain, staged):
        assert torch.equal(a, b)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("N,F,P,planes", [(7, 2, 5000, True), (7, 12, 15000, None), (9, 2, 5000, True), (9, 3, 5000, False),
                                          (12, 6, 2000, None), (5, 3, 20000, True), (5, 3, 30000, False), (7, 3, 45000, False)])
def test_fused_forms(N, F, P, planes, prec):
    fg, h, pts, kw = setup(N, F, P, prec)
    out, names = kernel_names(lambda: fg.fp_find_eval(h, pts, **kw))
    if planes is None:
        planes = prec == 0
    assert has(names, "k_eval_pairs_planes") == planes
    sep = fg.fp_eval_df(h, kw["posted"], out[0], out[2], out[3]) if prec else fg.fp_eval(h, out[0], out[2], out[3], kw["fields"])
    np.testing.assert_array_equal(out[5].cpu().numpy(), sep.cpu().numpy())


@pytest.mark.parametrize("F,P,planes", [(1, 10000, True), (1, 10001, False), (3, 3000, True), (4, 1000, False)])
def test_posted_points(F, P, planes):
    fg, h, pts, kw = setup(7, F, P, 1)
    out = fg.fp_find(h, pts)
    q = fg.Points(h, P)
    q.set(out[0], out[2], out[3])
    v, names = kernel_names(lambda: q.eval(kw["posted"]))
    assert has(names, "k_eval_planes") == planes and has(names, "k_eval_points_df") != planes
    np.testing.assert_array_equal(v.cpu().numpy(), fg.fp_eval_df(h, kw["posted"], out[0], out[2], out[3]).cpu().numpy())
