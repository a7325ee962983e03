"""Which kernel an evaluation runs (the forms give the same bits): staging in
shared memory whenever it is asked for."""
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
