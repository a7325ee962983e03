"""Timed cases of the point-location / interpolation library: what its users
have it do, through the public entry points, over the range of sizes, orders,
forms and call styles it serves.

Meshes are deformed boxes (hexahedra and quadrilaterals) and a box overlapped
by an annular cylinder.  Query points are made by mapping random reference
coordinates of random elements, so their exact location is known, in random
order (a point cloud is not sorted by element), with a share of
  - points on and within 1e-9 of element faces (interface nodes),
  - points just outside the mesh, found on the border: meshes whose surfaces
    do not match to the last digit.  `tol_border` is 1e-3 (mixed form 1e-4)
    for that reason, and dist2 is then a measured distance rather than a
    rounding residue.  The mixed form computes it from residuals rounded to
    FP32, so a program that stores it keeps 32 bits,
  - points outside the mesh.
"""
import math

import numpy as np
import torch

import paper_1811_04891_gb300 as fg
from paper_1811_04891_gb300.schwarz import InterfaceExchange

FP64, MIXED = 0, 1
TOL_BORDER = {FP64: 1e-3, MIXED: 1e-4}


def _dev():
    return torch.device("cuda")


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # one time step's probes of a small block: latency and launches count
        {"name": "small_mixed", "kind": "find_eval", "form": MIXED, "ne": 4, "N": 7, "P": 10000, "F": 1},
        # a solver that owns its device memory asks for a few points per rank (allocation-free call)
        {"name": "static_fp64", "kind": "static", "form": FP64, "ne": 6, "N": 6, "P": 1501, "F": 0},
        # overset interface exchange: tagged interface nodes and untagged points of an overlap, owner rule
        {"name": "overlap_mixed", "kind": "overlap", "form": MIXED, "N": 7, "nb": 8, "naz": 32, "nrad": 4, "nax": 8,
         "P": 40001, "F": 4},
        # one time step of a receiving subdomain: boundary data predicted, then re-interpolated and flux-corrected
        {"name": "schwarz_mixed", "kind": "schwarz", "form": MIXED, "N": 7, "nb": 8, "naz": 32, "nrad": 4, "nax": 8,
         "P": 0, "F": 4},
        # post-processing / tracer cloud of a large mesh, posted fields
        {"name": "cloud_mixed", "kind": "find_eval", "form": MIXED, "ne": 32, "N": 7, "P": 10100000, "F": 5},
        # tracer cloud in FP64, fields as the solver holds them
        {"name": "cloud_fp64", "kind": "find_eval", "form": FP64, "ne": 20, "N": 7, "P": 2000003, "F": 3},
        # high order, few points per element
        {"name": "sparse_mixed", "kind": "find_eval", "form": MIXED, "ne": 16, "N": 9, "P": 16411, "F": 3},
        # independent problems of several orders in one captured launch sequence
        {"name": "batch_mixed", "kind": "batch", "form": MIXED, "inst": 24, "P": 1200000, "E": 24000, "F": 1},
        # a mesh that moves every step: rebuild, warm-started search, interpolation
        {"name": "moving_mixed", "kind": "moving", "form": MIXED, "ne": 16, "N": 7, "P": 400009, "F": 4},
        # particles in host memory, streamed through the device
        {"name": "host_mixed", "kind": "host", "form": MIXED, "ne": 16, "N": 7, "P": 3000017, "F": 2},
        # fields of a new time step at points that stay where they are (FP64 fields, many of them)
        {"name": "eval_fp64", "kind": "eval", "form": FP64, "ne": 12, "N": 8, "P": 500009, "F": 6},
        # two-dimensional overset meshes
        {"name": "planar_fp64", "kind": "planar", "form": FP64, "ne": 128, "N": 7, "P": 1500001, "F": 3},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["find_eval", "find_eval", "find_eval", "overlap", "schwarz", "eval", "batch", "moving", "host",
                       "planar", "static"])
    form = FP64 if kind == "planar" else rng.choice([FP64, MIXED])
    cap = 1500000 if form == FP64 else 6000000
    if kind in ("overlap", "schwarz"):
        N = rng.choice([4, 5, 6, 7, 9])
        return {"kind": kind, "form": form, "N": N, "nb": rng.randint(4, 12), "naz": rng.choice([16, 32, 48]),
                "nrad": rng.randint(2, 4), "nax": rng.randint(3, 10),
                "P": _log(rng, 2000, cap // 4) if kind == "overlap" else 0, "F": rng.randint(3, 5)}
    if kind == "batch":
        P = _log(rng, 30000, cap // 2)
        return {"kind": kind, "form": form, "inst": rng.randint(3, 32), "P": P, "E": _log(rng, 1000, 30000), "F": 1}
    if kind == "planar":
        N = rng.randint(3, 12)
        return {"kind": kind, "form": form, "ne": _log(rng, 8, 160), "N": N, "P": _log(rng, 1000, 2000000),
                "F": rng.randint(1, 4)}
    if kind == "static":
        return {"kind": kind, "form": form, "ne": rng.randint(2, 12), "N": rng.randint(2, 9),
                "P": _log(rng, 100, 16000), "F": 0}
    N = rng.choice([2, 3, 4, 5, 5, 6, 7, 7, 7, 8, 9, 9, 10, 12])
    most = int(cap * min(1.0, (8.0 / (N + 1)) ** 4))
    ne = _log(rng, 3, max(4, int(26 * min(1.0, 8.0 / (N + 1)))))
    lo = 200000 if kind == "host" else 1000
    return {"kind": kind, "form": form, "ne": ne, "N": N, "P": _log(rng, lo, max(most // (1 if kind != "host" else 2),
                                                                                2 * lo)), "F": rng.randint(1, 6)}


# ---------------------------------------------------------------------------
# reference grid, interpolation and meshes in plain torch, 64 bits
# ---------------------------------------------------------------------------
def _gll(N):
    x = np.concatenate([[-1.0], np.sort(np.polynomial.legendre.Legendre.basis(N).deriv().roots().real), [1.0]])
    return 0.5 * (x - x[::-1])


def _basis(N, r):
    """[len(r)][N+1] Lagrange values on the Gauss-Lobatto-Legendre points."""
    xi = _gll(N)
    cols = []
    for i in range(N + 1):
        h = torch.ones_like(r)
        for m in range(N + 1):
            if m != i:
                h = h * ((r - float(xi[m])) * (1.0 / float(xi[i] - xi[m])))
        cols.append(h)
    return torch.stack(cols, 1)


def _interp(N, nodal, e, r):
    """nodal [A][E][n^d] at (e, r [d][P]) -> [A][P]."""
    n, d, P = N + 1, r.shape[0], e.numel()
    out = torch.empty((nodal.shape[0], P), dtype=torch.float64, device=r.device)
    step = max(1, (1 << 27) // n ** d)
    for p in range(0, P, step):
        h = [_basis(N, r[a, p:p + step]) for a in range(d)]
        c = h[0].shape[0]
        for a in range(nodal.shape[0]):
            v = nodal[a][e[p:p + step]].reshape(c, n ** (d - 1), n)
            v = torch.bmm(v, h[0].unsqueeze(2)).reshape(c, n ** (d - 2), n)
            v = torch.bmm(v, h[1].unsqueeze(2)).reshape(c, -1)
            out[a, p:p + step] = (v * h[2]).sum(1) if d == 3 else v[:, 0]
    return out


def _axis(m, a, b, xi):
    g = a + (b - a) * (torch.arange(m, dtype=torch.float64, device=_dev())[:, None] + 0.5 * (xi[None, :] + 1.0)) / m
    ends = a + (b - a) * (torch.arange(m + 1, dtype=torch.float64, device=_dev()) / m)
    g[:, 0], g[:, -1] = ends[:-1], ends[1:]
    return g


def _box(shape, N, lo, hi, amp):
    """Deformed box: coords [d][E][n^d], elements and nodes with the first
    direction fastest.  Nodes inside the box move by one scalar in every
    coordinate; the outer faces stay plane."""
    d, n = len(shape), N + 1
    xi = torch.from_numpy(_gll(N)).to(_dev())
    X = []
    for a in range(d):
        view = [1] * (2 * d)
        view[d - 1 - a], view[2 * d - 1 - a] = shape[a], n
        X.append(_axis(shape[a], lo[a], hi[a], xi).reshape(view).expand([*shape[::-1], *([n] * d)]).reshape(-1))
    C = torch.stack(X)
    if amp:
        u = [(X[a] - lo[a]) / (hi[a] - lo[a]) for a in range(d)]
        bump = torch.ones_like(u[0])
        for a in range(d):
            bump = bump * torch.sin(2 * math.pi * u[a])
        C = C + amp * min((hi[a] - lo[a]) / shape[a] for a in range(d)) * bump
    return C.reshape(d, math.prod(shape), n ** d).contiguous()


def _annulus(c, N):
    """Annular cylinder 0.15 <= rho <= 0.35, 0 <= z <= 1 around (1, 0.5):
    r radial, s azimuthal, t axial.  coords and distance to its boundary."""
    n = N + 1
    xi = torch.from_numpy(_gll(N)).to(_dev())
    shp = (c["nax"], c["naz"], c["nrad"], n, n, n)
    rho = _axis(c["nrad"], 0.15, 0.35, xi).reshape(1, 1, -1, 1, 1, n).expand(shp).reshape(-1, n ** 3)
    th = _axis(c["naz"], 0.0, 2 * math.pi, xi)
    th[-1, -1] = 0.0
    th = th.reshape(1, -1, 1, 1, n, 1).expand(shp).reshape(-1, n ** 3)
    z = _axis(c["nax"], 0.0, 1.0, xi).reshape(-1, 1, 1, n, 1, 1).expand(shp).reshape(-1, n ** 3)
    X = torch.stack([1.0 + rho * torch.cos(th), 0.5 + rho * torch.sin(th), z]).contiguous()
    return X, torch.minimum(torch.minimum(rho - 0.15, 0.35 - rho), torch.minimum(z, 1 - z)).clamp_min(0.0)


def _fields(coords, F, g):
    """F smooth fields, sine products of random wave numbers and phases."""
    out = []
    for _ in range(F):
        a = torch.rand(3, generator=g, device=_dev(), dtype=torch.float64) * 2 * math.pi + math.pi
        b = torch.rand(3, generator=g, device=_dev(), dtype=torch.float64) * 2 * math.pi
        v = torch.ones_like(coords[0])
        for q in range(coords.shape[0]):
            v = v * torch.sin(a[q] * coords[q] + b[q])
        out.append(v)
    return torch.stack(out).contiguous()


def _gen(seed):
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed))
    return g


def _cloud(coords, N, shape, lo, hi, P, g, tol):
    """P query points of a box mesh with their exact answers: points, element,
    r, squared distance (0 inside, inf not found) and code."""
    d, E = len(shape), math.prod(shape)
    e = torch.randint(0, E, (P,), generator=g, device=_dev())
    r = 2 * torch.rand((d, P), generator=g, device=_dev(), dtype=torch.float64) - 1
    n_face, n_bord, n_out = P // 100, P // 100, P // 200
    delta = torch.zeros(P, dtype=torch.float64, device=_dev())
    code = torch.zeros(P, dtype=torch.int32, device=_dev())
    idx = torch.arange(P, device=_dev())
    # on the face towards the next element (this one has the lower id), half of them up to 1e-9 inside it
    q = idx[:n_face]
    ax = q % d
    off = torch.where((q // d) % 2 == 0, 0.0, 10.0 ** (-11 + 2 * torch.rand(n_face, generator=g, device=_dev(),
                                                                          dtype=torch.float64)))
    r[ax, q] = 1.0 - 2.0 * off
    # just outside an outer face, up to 0.8 of the border tolerance: an element of the last layer, moved out
    q = idx[n_face:n_face + n_bord]
    ax = q % d
    he = math.sqrt(sum(((hi[a] - lo[a]) / shape[a]) ** 2 for a in range(d)))
    stride = [math.prod(shape[:a]) for a in range(d)]
    for a in range(d):
        w = q[ax == a]
        pos = (e[w] // stride[a]) % shape[a]
        e[w] = e[w] + (shape[a] - 1 - pos) * stride[a]
        r[a, w] = 1.0
        delta[w] = he * tol * (0.3 + 0.5 * torch.rand(w.numel(), generator=g, device=_dev(), dtype=torch.float64))
    code[q] = 1
    x = _interp(N, coords, e, r)
    for a in range(d):
        w = q[ax == a]
        x[a, w] = hi[a] + delta[w]
    q = idx[n_face + n_bord:n_face + n_bord + n_out]
    x[:, q] = hi[0] + 1.0 + torch.rand((d, q.numel()), generator=g, device=_dev(), dtype=torch.float64)
    code[q] = 2
    e[q] = -1
    r[:, q] = 0.0
    d2 = delta * delta
    d2[q] = math.inf
    perm = torch.randperm(P, generator=g, device=_dev())
    return x[:, perm].contiguous(), e[perm], r[:, perm].contiguous(), d2[perm], code[perm]


def _opts(case):
    return fg.default_opts(precision=case["form"], tol_border=TOL_BORDER[case["form"]])


# ---------------------------------------------------------------------------
# what a user's program has in hand
# ---------------------------------------------------------------------------
def _box_inputs(case, seed):
    g = _gen(seed)
    d = 2 if case["kind"] == "planar" else 3
    shape, lo, hi = (case["ne"],) * d, (0.0,) * d, (1.0,) * d
    coords = _box(shape, case["N"], lo, hi, 0.1)
    F = max(case["F"], 1)
    fields = _fields(coords, F, g)
    where = coords
    if case["kind"] == "moving":
        where = _box(shape, case["N"], lo, hi, 0.08)
    pts, e, r, d2, code = _cloud(where, case["N"], shape, lo, hi, case["P"], g,
                                  TOL_BORDER[case["form"]])
    return {"coords": coords, "where": where, "fields": fields, "pts": pts, "e": e, "r": r, "d2": d2, "code": code}


def _overlap_inputs(case, seed):
    """Box (session 0) overlapped by an annular cylinder (session 1): a third
    of the queries are cylinder points tagged 1 (found in the box), a third
    tagged 0 (found in the cylinder), the rest untagged (the owner rule).
    One in a hundred lies just above both meshes (the border)."""
    g = _gen(seed)
    N, P, nb = case["N"], case["P"], case["nb"]
    shape, lo, hi = (2 * nb, nb, nb), (0.0, 0.0, 0.0), (2.0, 1.0, 1.0)
    cb = _box(shape, N, lo, hi, 0.0)
    db = torch.minimum(torch.minimum(torch.minimum(cb[0], 2 - cb[0]), torch.minimum(cb[1], 1 - cb[1])),
                       torch.minimum(cb[2], 1 - cb[2])).clamp_min(0.0)
    cc, dc = _annulus(case, N)
    Eb, Ec = cb.shape[1], cc.shape[1]
    coords, dist = torch.cat([cb, cc], 1).contiguous(), torch.cat([db, dc]).contiguous()
    sub = torch.cat([torch.zeros(Eb, dtype=torch.int32), torch.ones(Ec, dtype=torch.int32)]).to(_dev())
    e = Eb + torch.randint(0, Ec, (P,), generator=g, device=_dev())
    r = (2 * torch.rand((3, P), generator=g, device=_dev(), dtype=torch.float64) - 1) * 0.999
    top = torch.arange(P, device=_dev()) % 100 == 7
    last = case["naz"] * case["nrad"] * (case["nax"] - 1)
    e[top] = Eb + last + (e[top] - Eb) % (case["naz"] * case["nrad"])
    r[2, top] = 1.0
    x = _interp(N, coords, e, r)
    delta = torch.zeros_like(x[0])
    delta[top] = 1e-5 * (0.4 + 0.4 * torch.rand(int(top.sum()), generator=g, device=_dev(), dtype=torch.float64))
    x[2, top] = 1.0 + delta[top]
    tag = (torch.arange(P, device=_dev()) % 3 - 1).to(torch.int32)
    tag = tag[torch.randperm(P, generator=g, device=_dev())].contiguous()
    return {"coords": coords, "dist": dist, "sub": sub, "pts": x.contiguous(), "tag": tag, "e": e, "r": r,
            "top": top, "d2": delta * delta, "fields": _fields(coords, case["F"], g), "shape": shape, "hi": hi,
            "Eb": Eb, "g": g}


def _in_box(s, x):
    """Element and r in the (undeformed) box of the overlap, in closed form."""
    e, r = torch.zeros(x.shape[1], dtype=torch.int64, device=x.device), torch.empty_like(x)
    stride = 1
    for a in range(3):
        m = s["shape"][a]
        u = (x[a] / (s["hi"][a] / m)).clamp(0.0, float(m))
        k = u.floor().clamp(0, m - 1)
        e += k.long() * stride
        r[a] = 2 * (u - k) - 1
        stride *= m
    return e, r


def _faces(case, s):
    """Marks of the cylinder's faces [E][6]: 2 = radial faces (interpolated
    data), 1 = end faces (prescribed data); and the prescribed velocity."""
    Ec = s["coords"].shape[1] - s["Eb"]
    el = torch.arange(Ec, device=_dev())
    er, ez = el % case["nrad"], el // (case["nrad"] * case["naz"])
    kind = torch.zeros((s["coords"].shape[1], 6), dtype=torch.int8, device=_dev())
    kind[s["Eb"]:, 0] = (er == 0).to(torch.int8) * 2
    kind[s["Eb"]:, 1] = (er == case["nrad"] - 1).to(torch.int8) * 2
    kind[s["Eb"]:, 4] = (ez == 0).to(torch.int8)
    kind[s["Eb"]:, 5] = (ez == case["nax"] - 1).to(torch.int8)
    M = int((kind != 0).sum()) * (case["N"] + 1) ** 2
    return kind, torch.rand((3, M), generator=s["g"], device=_dev(), dtype=torch.float64) - 0.5


def _batch_inputs(case, seed):
    """Instances of orders 5, 7 and 9 whose sizes spread over a factor of
    sixteen around the mean."""
    g, R = _gen(seed), np.random.default_rng(1)
    k = case["inst"]
    wp, we = (np.exp(R.uniform(-1.4, 1.4, k)) for _ in range(2))
    out = []
    for i in range(k):
        N = (5, 7, 9)[i % 3]
        ne = max(2, int(round((case["E"] * we[i] / we.sum()) ** (1 / 3))))
        P = max(50, int(case["P"] * wp[i] / wp.sum()))
        lo, hi = (0.0,) * 3, (1.0,) * 3
        coords = _box((ne,) * 3, N, lo, hi, 0.05)
        fields = _fields(coords, 1, g)
        out.append((N, coords, fields, *_cloud(coords, N, (ne,) * 3, lo, hi, P, g, TOL_BORDER[case["form"]])))
    return out


def prepare(case, seed):
    kind, mixed = case["kind"], case["form"] == MIXED
    if kind == "batch":
        inst = _batch_inputs(case, seed)
        hs = [fg.fp_setup(c, N, opts=_opts(case)) for N, c, *_ in inst]
        b = fg.Batch(hs, [v[3].shape[1] for v in inst], fields=[v[2] for v in inst])
        pts = torch.cat([v[3] for v in inst], 1).contiguous()
        outs = b.outputs()
        b.capture(pts, outs)
        return {"kind": kind, "mixed": mixed, "b": b, "pts": pts, "outs": outs}
    if kind == "overlap":
        s = _overlap_inputs(case, seed)
        h = fg.fp_setup(s["coords"], case["N"], s["sub"], s["dist"], opts=_opts(case))
        fg.fp_reserve(h, case["P"])
        return {"kind": kind, "mixed": mixed, "h": h, "pts": s["pts"], "tag": s["tag"],
                **_posted(h, s["fields"], mixed)}
    if kind == "schwarz":
        s = _overlap_inputs(dict(case, P=300), seed)
        h = fg.fp_setup(s["coords"], case["N"], s["sub"], s["dist"], opts=_opts(case))
        marks, u_pres = _faces(case, s)
        posted = fg.Fields(h, s["fields"]) if mixed else None
        ex = InterfaceExchange(h, fg.BFaces(h, marks), 1, s["fields"], posted, order=2)
        ex.u_pres.copy_(u_pres)
        return {"kind": kind, "ex": ex}
    s = _box_inputs(case, seed)
    if kind == "planar":
        h = fg.fp_setup_2d(s["coords"], case["N"], opts=_opts(case))
    else:
        h = fg.fp_setup(s["coords"], case["N"], opts=_opts(case))
    st = {"kind": kind, "mixed": mixed, "h": h, "pts": s["pts"]}
    if kind == "static":
        return st
    st.update(_posted(h, s["fields"], mixed))
    if kind == "host":
        # a program keeps its pinned buffers
        P, F = case["P"], case["F"]
        st["pts"] = s["pts"].cpu().pin_memory()
        st["out"] = tuple(torch.empty(P, dtype=torch.int32).pin_memory() for _ in range(3)) + (
            torch.empty((3, P), dtype=torch.float64).pin_memory(), torch.empty(P, dtype=torch.float64).pin_memory())
        st["values"] = torch.empty((F, P), dtype=torch.float64).pin_memory()
        return st
    fg.fp_reserve(h, case["P"])
    if kind == "eval":
        st.update(code=s["code"], elem=s["e"].to(torch.int32), rst=s["r"])
    if kind == "moving":
        # where the points were on the mesh of the last step
        st["last"] = fg.fp_find(h, s["pts"])
        st["where"] = s["where"]
    return st


def _posted(h, fields, mixed):
    return {"fields": None, "posted": fg.Fields(h, fields)} if mixed else {"fields": fields, "posted": None}


def _stored(out, s):
    """What is kept of a find: dist2 in the precision it has."""
    return (*out[:4], out[4].float(), *out[5:]) if s["mixed"] else out


def run(s):
    kind = s["kind"]
    if kind == "batch":
        s["b"].launch()
        return _stored(s["outs"], s)
    if kind == "schwarz":
        ex = s["ex"]
        return ex.step(kappa=4), ex.gamma, ex.flux
    h = s["h"]
    if kind == "static":
        return _stored(fg.fp_find_static(h, s["pts"]), s)
    if kind == "overlap":
        return _stored(fg.fp_find_eval(h, s["pts"], s["tag"], fields=s["fields"], posted=s["posted"]), s)
    if kind == "host":
        return _stored(fg.fp_find_eval_host(h, s["pts"], fields=s["fields"], posted=s["posted"], out=s["out"],
                                            values=s["values"]), s)
    if kind == "eval":
        if s["posted"] is not None:
            return fg.fp_eval_df(h, s["posted"], s["code"], s["elem"], s["rst"])
        return fg.fp_eval(h, s["code"], s["elem"], s["rst"], s["fields"])
    if kind == "moving":
        fg.fp_update_coords(h, s["where"])
        return _stored(fg.fp_find_warm(h, s["pts"], warm=(s["last"][2], s["last"][3]), fields=s["fields"],
                                       posted=s["posted"]), s)
    return _stored(fg.fp_find_eval(h, s["pts"], fields=s["fields"], posted=s["posted"]), s)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _find_work(E, N, P, F, d, coords=1):
    """Two Newton evaluations of the element map with its Jacobian, one of the
    map alone, and F interpolations per point, sum-factorised; points, tags of
    the mesh that is touched, fields and results moved once."""
    n = N + 1
    nodes = n ** d
    touched = min(E, P) * nodes * 8
    full = 2 * sum(n ** k for k in range(1, d + 1))
    jac = d * 2 * (2 * n ** d + (3 if d == 3 else 0) * n ** 2 + d * n)
    return {"bytes": touched * (d * coords + F) + P * (8 * d + 12 + 8 * d + 8 + 8 * F),
            "flops": P * (2 * jac + (d + F) * full)}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = {"bytes": 0, "flops": 0}
        for N in (5, 7, 9):
            v = _find_work(case["E"] // 3, N, case["P"] // 3, 1, 3)
            w = {k: w[k] + v[k] for k in w}
        return w
    N, P, F, n = case["N"], case["P"], case["F"], case["N"] + 1
    if kind == "schwarz":
        # four interpolations at the interface nodes, each followed by the flux correction of all face nodes
        Mi, M = (2 * case["naz"] * case["nax"] * n * n, 2 * case["naz"] * (case["nax"] + case["nrad"]) * n * n)
        E = min(2 * case["nb"] ** 3, Mi)
        return {"bytes": 4 * (E * F * n ** 3 * 8 + Mi * (28 + 8 * F) + M * 8 * 10),
                "flops": 4 * (Mi * F * 2 * (n + n * n + n ** 3) + M * 14)}
    if kind == "overlap":
        return _find_work(2 * case["nb"] ** 3 + case["naz"] * case["nrad"] * case["nax"], N, P, F, 3)
    d = 2 if kind == "planar" else 3
    E = case["ne"] ** d
    if kind == "eval":
        full = 2 * (n + n * n + n ** 3)
        return {"bytes": min(E, P) * F * n ** 3 * 8 + P * (8 + 24 + 8 * F), "flops": P * F * full}
    return _find_work(E, N, P, F, d, coords=2 if kind == "moving" else 1)


# ---------------------------------------------------------------------------
# the answers in 64 bits
# ---------------------------------------------------------------------------
def _values(N, fields, e, r, code):
    v = _interp(N, fields, e.clamp_min(0), r)
    v[:, code == 2] = math.nan
    return v


def _schwarz(case, seed):
    """u + gamma n on the interface nodes, gamma = -(int u.n) / (interface
    area), by quadrature on the face nodes (faces in element order, a face's
    first reference direction fastest)."""
    s = _overlap_inputs(dict(case, P=300), seed)
    kind, u = _faces(case, s)
    N, n = case["N"], case["N"] + 1
    xi = _gll(N)
    V = np.polynomial.legendre.legvander(xi, N)
    w = torch.from_numpy(2.0 / (N * n * V[:, N] ** 2)).to(_dev())
    D = np.array([[0.0 if a == i else V[a, N] / (V[i, N] * (xi[a] - xi[i])) for i in range(n)] for a in range(n)])
    D = torch.from_numpy(D - np.diag(D.sum(1))).to(_dev())
    e, f = torch.nonzero(kind, as_tuple=True)
    X = s["coords"][:, e].reshape(3, -1, n, n, n)
    X = torch.stack([X[:, :, :, :, 0], X[:, :, :, :, N], X[:, :, 0], X[:, :, N]], 0)
    at = torch.tensor([0, 1, 0, 0, 2, 3], device=_dev())[f]
    X = X[at, :, torch.arange(len(e), device=_dev())].permute(1, 0, 2, 3)
    t1, t2 = torch.einsum("xfbi,ai->xfba", X, D), torch.einsum("xfja,bj->xfba", X, D)
    nv = torch.linalg.cross(t1, t2, dim=0) * torch.where(f % 2 == 1, 1.0, -1.0)[None, :, None, None]
    area = nv.norm(dim=0)
    nv, dA = (nv / area).reshape(3, -1), (area * w[None, :, None] * w[None, None, :]).reshape(-1)
    iface = (kind[e, f] == 2)[:, None].expand(-1, n * n).reshape(-1)
    x = X.reshape(3, -1)
    u[:, iface] = _interp(N, s["fields"][:3], *_in_box(s, x[:, iface]))
    flux = ((u * nv).sum(0) * dA).sum()
    gamma = -flux / dA[iface].sum()
    u[:, iface] += gamma * nv[:, iface]
    return u, gamma.reshape(1), flux.reshape(1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        rst, d2, val = [], [], []
        for N, _, fields, _, e, r, dd, code in _batch_inputs(case, seed):
            rst.append(r)
            d2.append(dd)
            val.append(_values(N, fields, e, r, code))
        return None, None, None, torch.cat(rst, 1), torch.cat(d2), torch.cat(val, 1)
    if kind == "overlap":
        s = _overlap_inputs(case, seed)
        N = case["N"]
        eb, rb = _in_box(s, s["pts"])
        in_box = s["tag"] == 1
        free = s["tag"] < 0
        db = _interp(N, s["dist"][None], eb, rb)[0]
        dc = _interp(N, s["dist"][None], s["e"], s["r"])[0]
        in_box = in_box | (free & (s["top"] | (db >= dc)))
        e = torch.where(in_box, eb, s["e"])
        r = torch.where(in_box[None], rb, s["r"])
        return None, None, None, r, s["d2"], _interp(N, s["fields"], e, r)
    if kind == "schwarz":
        return _schwarz(case, seed)
    s = _box_inputs(case, seed)
    if kind == "static":
        return None, None, None, s["r"], s["d2"]
    val = _values(case["N"], s["fields"], s["e"], s["r"], s["code"])
    if kind == "eval":
        return val
    return None, None, None, s["r"], s["d2"], val
