"""Meshes without stored node digits (fp_set_node_digits): every kind of find
gives the bits it gives with them, the memory is given back, and a server
whose budget leaves no room for them still starts."""
import numpy as np
import pytest
import torch

import synth
from test_gpu_tile import points, quarter_turns

pytestmark = pytest.mark.gpu


def tensors(mesh):
    return torch.from_numpy(np.ascontiguousarray(mesh.coords)).cuda(), torch.from_numpy(mesh.sub).cuda()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("N", [3, 4, 5, 6, 7, 8, 9])
def test_same_bits_without_digits(N, prec):
    import paper_1811_04891_gb300 as fg
    mesh = quarter_turns(N)
    # one thin direction, so that the coordinates' scales differ
    mesh.coords[2] *= 1e-3
    coords, sub = tensors(mesh)
    h = fg.fp_setup(coords, N, sub, opts=fg.default_opts(precision=prec))
    pts = points(mesh)
    k = 70000 // pts.shape[1] + 1
    few, many = (torch.from_numpy(np.ascontiguousarray(p)).cuda() for p in (pts, np.tile(pts, k)))
    ws = fg.Workspace(h, many.shape[1], 4 * many.shape[1])

    def all_finds():
        fg.fp_update_coords(h, coords)
        out = [fg.fp_find(h, few), fg.fp_find(h, many), fg.fp_find_static(h, few), fg.fp_find_ws(h, ws, many)]
        b = fg.Batch([h, h], [few.shape[1]] * 2)
        outs = b.outputs()
        b.run(torch.cat([few, few], dim=1).contiguous(), outs)
        out.append(outs[:5])
        torch.cuda.synchronize()
        return [[x.clone() for x in o] for o in out]

    stored = all_finds()
    held = fg.fp_memory(h)["resident"]
    fg.fp_set_node_digits(h, False)
    less = held - fg.fp_memory(h)["resident"]
    tile = N in (4, 6, 7, 8, 9) or prec == 0
    assert less >= 8 * coords.numel() if tile else less == 0
    fly = all_finds()
    fg.fp_set_node_digits(h, True)
    assert fg.fp_memory(h)["resident"] == held
    again = all_finds()
    for a, b, c in zip(stored, fly, again):
        for x, y, z in zip(a, b, c):
            assert torch.equal(x, y) and torch.equal(x, z)


def test_server_without_room_for_digits():
    import paper_1811_04891_gb300 as fg
    from paper_1811_04891_gb300 import serve
    mesh, q = synth.deformed_cube(ne=6, P_uniform=9000, P_face=900)
    coords, sub = tensors(mesh)
    fields = torch.from_numpy(q.fields).cuda()
    out = []
    for tight in (False, True):
        h = fg.fp_setup(coords, mesh.N, sub, opts=fg.default_opts(precision=1))
        roomy = serve.Server(h, fields, chunk_points=4096, streams=1)
        digits = fg.fp_memory(h)["resident"]
        fg.fp_set_node_digits(h, False)
        digits -= fg.fp_memory(h)["resident"]
        fg.fp_set_node_digits(h, True)
        budget = fg.fp_memory(h)["resident"] - digits / 2 + 1.1 * roomy.bytes_for(4096)
        srv = serve.Server(h, fields, budget_bytes=budget, chunk_points=4096, streams=1) if tight else roomy
        done, _ = serve.run_stream(srv, [serve.Request(0, 0.0, q.pts, np.full(q.P, -1, np.int32))])
        assert len(done) == 1 and (fg.fp_memory(h)["resident"] <= budget - roomy.bytes_for(4096)) == tight
        out.append(done[0])
        srv.close()
    for name in ("code", "elem", "rst", "values"):
        np.testing.assert_array_equal(getattr(out[0], name), getattr(out[1], name))
    with pytest.raises(ValueError):
        serve.Server(h, fields, budget_bytes=1e5, chunk_points=4096, streams=1)
