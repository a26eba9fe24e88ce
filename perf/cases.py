"""Cases that time the library the way its users call it.

Each case is one call (or the usual short sequence of calls) of the public Python API on
seeded synthetic meshes: a pair compared once (build B, then the bracket of h(A, B)), a kept
reference B that a new A is measured against, the two-sided distance, many pairs in one batched
call, nearest-triangle queries, and host arrays in, bracket out.  Meshes are made on the GPU in
double and stored as the case says.  ``shape`` selects

  torus    A: a regular grid with normal noise; B: its own grid with 0.3-cell parameter jitter
  sphere   the same on a latitude-longitude sphere (its pole rows are zero-area triangles)
  soup     A: a superquadric plus ``extra`` loose triangles up to 0.1 off it; B: another
           triangulation of the superquadric
  slivers  A: thin triangles tiling a sphere in latitude bands; B: a superquadric inside it
"""
import math
import random

import numpy as np
import torch

import paper_2406_10357_gb300 as hd

DEV = "cuda"


def listed():
    return [
        # two tiny meshes compared once with the default options (a unit test, a CAD part check)
        dict(name="tiny_pair_fp64", call="pair", shape="sphere", a0=16, a1=10, b0=16, b1=10, extra=0, noise=0.01,
             tol=1e-4, rel=False, mixed=False, double=True),
        # a remeshing check: the noisy original against an independent triangulation
        dict(name="torus_pair_mixed", call="pair", shape="torus", a0=400, a1=250, b0=224, b1=112, extra=0, noise=1e-3,
             tol=1e-5, rel=True, mixed=True, double=False),
        # the same with the default precision
        dict(name="torus_pair_fp64", call="pair", shape="torus", a0=400, a1=250, b0=224, b1=112, extra=0, noise=1e-3,
             tol=1e-5, rel=True, mixed=False, double=False),
        # the largest: two million triangles a side, with loose pieces
        dict(name="soup_pair_mixed", call="pair", shape="soup", a0=975, a1=975, b0=1000, b1=1000, extra=100_000,
             noise=0.0, tol=1e-6, rel=True, mixed=True, double=False),
        # thin triangles against a large reference whose BVH is kept
        dict(name="slivers_kept_mixed", call="kept", shape="slivers", a0=100_000, a1=1, b0=1000, b1=500, extra=0,
             noise=1e-4, tol=1e-6, rel=True, mixed=True, double=False),
        # the symmetric distance of two scans of odd sizes, double vertices, default precision
        dict(name="scan_sym_fp64", call="sym", shape="torus", a0=113, a1=31, b0=149, b1=41, extra=0, noise=2e-3,
             tol=1e-4, rel=True, mixed=False, double=True),
        # a data set's pairs in one batched call
        dict(name="batch_mixed", call="batch", pairs=128, lo=1000, hi=200_000, sizes=5000, tol=1e-4, rel=True,
             mixed=True, double=False),
        # a few dozen small parts in one batched call, default precision
        dict(name="batch_small_fp64", call="batch", pairs=32, lo=300, hi=3000, sizes=5000, tol=1e-4, rel=True,
             mixed=False, double=False),
        # a scan's points against a kept model
        dict(name="nearest_scan_mixed", call="nearest", shape="torus", b0=224, b1=112, points=500_000, where="surface",
             noise=0.01, mixed=True, double=False, noalloc=False),
        # distances sampled through a volume (a distance field), default precision, double points
        dict(name="nearest_volume_fp64", call="nearest", shape="torus", b0=224, b1=112, points=40_001, where="volume",
             noise=0.0, mixed=False, double=True, noalloc=False),
        # one small request of an allocation-free loop
        dict(name="nearest_noalloc_mixed", call="nearest", shape="torus", b0=224, b1=112, points=1000, where="surface",
             noise=0.01, mixed=True, double=False, noalloc=True),
        # a service call: host arrays in, bracket out
        dict(name="host_pair_mixed", call="host", shape="torus", a0=141, a1=71, b0=141, b1=71, extra=0, noise=1e-3,
             tol=1e-4, rel=True, mixed=True, double=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi, ratio):
    """Grid sizes (first, second) of about n = 2 * first * second faces, n log-uniform in [lo, hi]."""
    n = _log(rng, lo, hi)
    second = max(5, int(round(math.sqrt(n / (2 * ratio)))))
    return max(5, n // (2 * second)), second


def draw(rng):
    call = rng.choice(["pair", "pair", "kept", "sym", "batch", "nearest", "nearest", "host"])
    mixed, double = rng.random() < 0.6, rng.random() < 0.3
    if call == "batch":
        if mixed:
            return dict(call=call, pairs=_log(rng, 3, 100), lo=1000, hi=_log(rng, 5000, 200_000),
                        sizes=rng.randrange(1 << 20), tol=1e-4, rel=True, mixed=True, double=False)
        return dict(call=call, pairs=_log(rng, 3, 32), lo=300, hi=_log(rng, 1000, 3000), sizes=rng.randrange(1 << 20),
                    tol=1e-4, rel=True, mixed=False, double=double)
    if call == "nearest":
        b0, b1 = _grid(rng, 1000, 50_000, 2)
        noalloc, where = rng.random() < 0.3, rng.choice(["surface", "volume"])
        n = _log(rng, 100, 65_536 if noalloc else 40_000 if where == "volume" else 500_000)
        return dict(call=call, shape=rng.choice(["torus", "sphere"]), b0=b0, b1=b1, points=n, where=where,
                    noise=10 ** rng.uniform(-3, -2), mixed=mixed, double=double, noalloc=noalloc)
    if call == "pair":
        shape = rng.choice(["torus", "sphere", "soup"])
    elif call == "kept":
        shape = rng.choice(["torus", "slivers"])
    else:
        shape = rng.choice(["torus", "sphere"])
    if shape == "slivers":
        a0, a1 = _log(rng, 1000, 60_000), 1
        b0, b1 = _grid(rng, 10_000, 600_000, 2)
        return dict(call=call, shape=shape, a0=a0, a1=a1, b0=b0, b1=b1, extra=0, noise=1e-4, tol=1e-6, rel=True,
                    mixed=True, double=False)
    if shape == "soup":
        a0, a1 = _grid(rng, 2000, 1_800_000 if mixed else 400_000, 1)
        b0, b1 = _grid(rng, 2000, 1_800_000 if mixed else 400_000, 1)
        return dict(call=call, shape=shape, a0=a0, a1=a1, b0=b0, b1=b1, extra=a0 * a1 // 10 + 4, noise=0.0, tol=1e-6,
                    rel=True, mixed=mixed, double=False)
    # near-identical pairs: B at least a fifth as fine as A, so that the split counts stay those
    # of a remeshing check
    hi = 20_000 if call in ("host", "sym") else 200_000
    a0, a1 = _grid(rng, 320, hi, 2)
    n = 2 * a0 * a1
    b0, b1 = _grid(rng, max(320, n // 5), max(640, min(n, 50_000)), 2)
    return dict(call=call, shape=shape, a0=a0, a1=a1, b0=b0, b1=b1, extra=0, noise=10 ** rng.uniform(-3, -2),
                tol=10 ** rng.uniform(-5, -4), rel=True, mixed=mixed, double=double)


# ----------------------------------------------------------------------------- meshes


def _gen(seed, part):
    return torch.Generator(device=DEV).manual_seed(seed * 64 + part)


def _normal(g, *shape):
    return torch.randn(*shape, dtype=torch.float64, device=DEV, generator=g)


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, dtype=torch.float64, device=DEV, generator=g)


def _faces(nu, nv, wrap_u):
    """Two triangles per cell of an nu x nv vertex grid, vertex (i, j) -> i * nv + j, wrapping in j."""
    i = torch.arange(nu if wrap_u else nu - 1, device=DEV)[:, None]
    j = torch.arange(nv, device=DEV)[None, :]
    i1, j1 = (i + 1) % nu, (j + 1) % nv
    v00, v10, v11, v01 = i * nv + j, i1 * nv + j, i1 * nv + j1, i * nv + j1
    return torch.stack([torch.stack([v00, v10, v11], -1), torch.stack([v00, v11, v01], -1)], 2).reshape(-1, 3).int()


def _torus(nu, nv, jitter=0.0, g=None):
    i = torch.arange(nu, dtype=torch.float64, device=DEV)[:, None].expand(nu, nv)
    j = torch.arange(nv, dtype=torch.float64, device=DEV)[None, :].expand(nu, nv)
    if jitter:
        i, j = i + _uniform(g, -jitter, jitter, nu, nv), j + _uniform(g, -jitter, jitter, nu, nv)
    u, v = (i * (2 * math.pi / nu)).reshape(-1), (j * (2 * math.pi / nv)).reshape(-1)
    n = torch.stack([v.cos() * u.cos(), v.cos() * u.sin(), v.sin()], 1)
    ring = torch.stack([u.cos(), u.sin(), torch.zeros_like(u)], 1)
    return ring + 0.3 * n, _faces(nu, nv, True), n


def _spow(x, e):
    return x.sign() * x.abs() ** e


def _superquadric(n_lon, n_lat, e1, e2, scale, jitter=0.0, g=None):
    """Rows from pole to pole, n_lon vertices each (the pole rows coincide: zero-area triangles)."""
    j = torch.arange(n_lat + 1, dtype=torch.float64, device=DEV)[:, None].expand(n_lat + 1, n_lon).clone()
    i = torch.arange(n_lon, dtype=torch.float64, device=DEV)[None, :].expand(n_lat + 1, n_lon)
    if jitter:
        j[1:-1] += _uniform(g, -jitter, jitter, n_lat - 1, n_lon)
        i = i + _uniform(g, -jitter, jitter, n_lat + 1, n_lon)
    eta, om = -math.pi / 2 + j * (math.pi / n_lat), -math.pi + i * (2 * math.pi / n_lon)
    ce = torch.where(eta.cos().abs() < 1e-15, torch.zeros_like(eta), eta.cos())
    p = torch.stack([_spow(ce, e1) * _spow(om.cos(), e2), _spow(ce, e1) * _spow(om.sin(), e2), _spow(eta.sin(), e1)], -1)
    return scale * p.reshape(-1, 3), _faces(n_lat + 1, n_lon, False)


def _loose(n, edge, g):
    """n separate triangles of that edge length, pushed off the superquadric by up to 0.1."""
    e1, e2 = 0.8, 1.2
    eta, om = _uniform(g, -math.pi / 2 + 0.05, math.pi / 2 - 0.05, n), _uniform(g, -math.pi, math.pi, n)
    ce = eta.cos()
    p = torch.stack([_spow(ce, e1) * _spow(om.cos(), e2), _spow(ce, e1) * _spow(om.sin(), e2), _spow(eta.sin(), e1)], 1)
    a = p.abs().clamp_min(1e-12)
    f = (2 / e1) * (a[:, 0] ** (2 / e2) + a[:, 1] ** (2 / e2)) ** (e2 / e1 - 1)
    m = torch.stack([f * a[:, 0] ** (2 / e2 - 1), f * a[:, 1] ** (2 / e2 - 1), (2 / e1) * a[:, 2] ** (2 / e1 - 1)], 1)
    m = torch.nn.functional.normalize(m * p.sign(), dim=1)
    c = p + m * _uniform(g, -0.1, 0.1, n, 1)
    x = torch.nn.functional.normalize(_normal(g, n, 3), dim=1)
    y = _normal(g, n, 3)
    y = torch.nn.functional.normalize(y - (y * x).sum(1, keepdim=True) * x, dim=1)
    ang = torch.tensor([0.0, 2 * math.pi / 3, 4 * math.pi / 3], dtype=torch.float64, device=DEV)[None, :, None]
    v = c[:, None] + edge / math.sqrt(3.0) * (ang.cos() * x[:, None] + ang.sin() * y[:, None])
    return v.reshape(-1, 3), torch.arange(3 * n, device=DEV, dtype=torch.int32).reshape(n, 3)


def _slivers(n, noise, g, rng):
    """About n thin triangles tiling the unit sphere in latitude bands, aspect ratio of a band
    log-uniform in [10, 1e4]; bands share no vertices."""
    area, theta, bands = 4 * math.pi / n, 0.0, []
    while theta < math.pi - 1e-12:
        a = 10 ** rng.uniform(1, 4)
        h = math.sqrt(2 * area / a)
        t1 = min(theta + h, math.pi)
        bands.append((theta, t1, max(3, round(2 * math.pi * math.sin(0.5 * (theta + t1)) / (a * h))), rng.uniform(0, 2 * math.pi)))
        theta = t1
    t0, t1, nc, ph = (torch.tensor(x, dtype=torch.float64, device=DEV) for x in zip(*bands))
    nc = nc.long()
    start = torch.cumsum(nc, 0) - nc
    b = torch.repeat_interleave(torch.arange(len(nc), device=DEV), nc)
    k = torch.arange(len(b), device=DEV) - start[b]
    k1 = (k + 1) % nc[b]
    phi = ph[b] + 2 * math.pi * k / nc[b]
    ring = [torch.stack([t[b].sin() * phi.cos(), t[b].sin() * phi.sin(), t[b].cos()], 1) for t in (t0, t1)]
    total = len(b)
    a0, a1 = start[b] + k, start[b] + k1
    f = torch.stack([torch.stack([a0, a1, a1 + total], 1), torch.stack([a0, a1 + total, a0 + total], 1)], 1)
    v = torch.cat(ring)
    return v + noise * _normal(g, *v.shape), f.reshape(-1, 3).int()


def _mesh_a(case, seed):
    g = _gen(seed, 1)
    if case["shape"] == "torus":
        v, f, n = _torus(case["a0"], case["a1"])
        return v + n * case["noise"] * _normal(g, len(v), 1), f
    if case["shape"] == "sphere":
        v, f = _superquadric(case["a0"], case["a1"], 1.0, 1.0, 1.0)
        return v * (1 + case["noise"] * _normal(g, len(v), 1)), f
    if case["shape"] == "slivers":
        return _slivers(case["a0"], case["noise"], g, random.Random(seed))
    v, f = _superquadric(case["a0"], case["a1"], 0.8, 1.2, 1.0)
    edge = float((v[f[:, 1].long()] - v[f[:, 0].long()]).norm(dim=1).mean())
    w, e = _loose(case["extra"], edge, g)
    return torch.cat([v, w]), torch.cat([f, e + len(v)])


def _mesh_b(case, seed):
    g = _gen(seed, 2)
    if case["shape"] == "torus":
        return _torus(case["b0"], case["b1"], 0.3, g)[:2]
    if case["shape"] == "sphere":
        return _superquadric(case["b0"], case["b1"], 1.0, 1.0, 1.0, 0.3, g)
    if case["shape"] == "slivers":
        return _superquadric(case["b0"], case["b1"], 0.8, 1.2, 0.999)
    return _superquadric(case["b0"], case["b1"], 0.8, 1.2, 1.0, 0.3, g)


def _stored(v, case):
    return v.contiguous() if case["double"] else v.float().contiguous()


def _batch_sizes(case):
    """Per pair: shape, A's and B's grids, whether B is A perturbed, and the noise."""
    rng = random.Random(case["sizes"])
    out = []
    for _ in range(case["pairs"]):
        na, nb = (_log(rng, case["lo"], case["hi"]) for _ in range(2))
        shape, perturbed, sigma = rng.randrange(3), rng.random() < 0.5, 10 ** rng.uniform(-5, -2)
        grids = []
        for n in (na, nb):
            if shape == 1:
                m = max(4, round(math.sqrt(n / 8)))
                grids.append((4 * m, m))
            else:
                m = max(3, round(math.sqrt(n / 4)))
                grids.append((2 * m, m))
        out.append((shape, grids[0], grids[0] if perturbed else grids[1], perturbed, sigma))
    return out


def _batch_mesh(shape, grid, jitter, g):
    if shape == 1:
        return _torus(grid[0], grid[1], jitter, g)[:2]
    return _superquadric(grid[0], grid[1], *((1.0, 1.0) if shape == 0 else (0.8, 1.2)), 1.0, jitter, g)


def _batch_pair(case, seed, k, spec):
    shape, ga, gb, perturbed, sigma = spec
    g = _gen(seed, 3 + k % 60)
    va, fa = _batch_mesh(shape, ga, 0.0, g)
    if perturbed:
        centre = va * torch.tensor([1.0, 1.0, 0.0], dtype=torch.float64, device=DEV)
        out = va - torch.nn.functional.normalize(centre, dim=1) if shape == 1 else va
        vb, fb = va + torch.nn.functional.normalize(out, dim=1) * sigma * _normal(g, len(va), 1), fa.clone()
    else:
        vb, fb = _batch_mesh(shape, gb, 0.3, g)
    return _stored(va, case), fa, _stored(vb, case), fb


def _points(case, seed):
    g = _gen(seed, 4)
    n = case["points"]
    if case["where"] == "volume":
        half = torch.tensor([1.5, 1.5, 0.5] if case["shape"] == "torus" else [1.5, 1.5, 1.5], dtype=torch.float64, device=DEV)
        p = _uniform(g, -1.0, 1.0, n, 3) * half
    else:
        u, v = _uniform(g, 0, 2 * math.pi, n), _uniform(g, 0, 2 * math.pi, n)
        if case["shape"] == "torus":
            m = torch.stack([v.cos() * u.cos(), v.cos() * u.sin(), v.sin()], 1)
            p = torch.stack([u.cos(), u.sin(), torch.zeros_like(u)], 1) + 0.3 * m
        else:
            m = torch.nn.functional.normalize(_normal(g, n, 3), dim=1)
            p = m
        p = p + m * case["noise"] * _normal(g, n, 1)
    return _stored(p, case)


# ----------------------------------------------------------------------------- the cases


def _options(case, **kw):
    return hd.hd_options_default(tol_mode=hd.HD_TOL_REL if case["rel"] else hd.HD_TOL_ABS,
                                 precision=hd.HD_MIXED if case["mixed"] else hd.HD_FP64, **kw)


def prepare(case, seed):
    call = case["call"]
    if call == "batch":
        pairs = [_batch_pair(case, seed, k, s) for k, s in enumerate(_batch_sizes(case))]
        return dict(case=case, A=[p[:2] for p in pairs], bvh=[hd.hd_build_B(*p[2:]) for p in pairs], opt=_options(case))
    if call == "nearest":
        vb, fb = _mesh_b(case, seed)
        s = dict(case=case, bvh=hd.hd_build_B(_stored(vb, case), fb), P=_points(case, seed), out=None)
        if case["noalloc"]:
            n = case["points"]
            s["out"] = (torch.empty(n, dtype=torch.float64, device=DEV), torch.empty(n, dtype=torch.int32, device=DEV),
                        torch.empty((n, 3), dtype=torch.float64, device=DEV), torch.empty(n, dtype=torch.float64, device=DEV))
        return s
    (va, fa), (vb, fb) = _mesh_a(case, seed), _mesh_b(case, seed)
    s = dict(case=case, VA=_stored(va, case), FA=fa, VB=_stored(vb, case), FB=fb, opt=_options(case))
    if call == "kept":
        s["bvh"] = hd.hd_build_B(s["VB"], s["FB"], s["opt"])
    if call == "host":  # NumPy arrays in, B's build queued ahead of the comparison
        s.update({k: s[k].cpu().numpy() for k in ("VA", "FA", "VB", "FB")})
        s["opt"] = _options(case, flags=hd.HD_FLAG_ASYNC_BUILD)
    return s


def _bracket(r):
    """What the method computes.  The statistics beside it count how the work was done."""
    return dict(lower=r["lower"], upper=r["upper"], status=r["status"], eps=r["stats"]["eps_abs"], dA=r["stats"]["dA"])


def _brackets(rs, case):
    """The same of many pairs, an array each; brackets in the type of the bounds that make them."""
    rs, kind = [_bracket(r) for r in rs], np.float32 if case["mixed"] else np.float64
    return {k: np.array([r[k] for r in rs], dtype=np.int32 if k == "status" else kind if k in ("lower", "upper") else np.float64)
            for k in rs[0]}


def run(s):
    case = s["case"]
    call = case["call"]
    if call == "batch":
        return _brackets(hd.hd_hausdorff_batched(s["bvh"], s["A"], case["tol"], s["opt"]), case)
    if call == "nearest":
        prec = hd.HD_MIXED if case["mixed"] else hd.HD_FP64
        if case["noalloc"]:
            return hd.hd_nearest_noalloc(s["bvh"], s["P"], prec, out=s["out"])
        return hd.hd_nearest(s["bvh"], s["P"], prec)
    if call == "kept":
        return _bracket(hd.hd_hausdorff(s["bvh"], s["VA"], s["FA"], case["tol"], s["opt"]))
    bvh = hd.hd_build_B(s["VB"], s["FB"], s["opt"])
    if call == "sym":
        bvh_a = hd.hd_build_B(s["VA"], s["FA"], s["opt"])
        rs = hd.hd_hausdorff_sym(bvh, s["VA"], s["FA"], bvh_a, s["VB"], s["FB"], case["tol"], s["opt"])
        return [_bracket(r) for r in rs]
    return _bracket(hd.hd_hausdorff(bvh, s["VA"], s["FA"], case["tol"], s["opt"]))


def _faces_of(case):
    """(vertices, faces) of A and of B as the case makes them."""
    if case["shape"] == "torus":
        grids = [(case[k + "0"] * case[k + "1"], 2 * case[k + "0"] * case[k + "1"]) for k in ("a", "b") if k + "0" in case]
    else:
        grids = [(case[k + "0"] * (case[k + "1"] + 1), 2 * case[k + "0"] * case[k + "1"]) for k in ("a", "b") if k + "0" in case]
    if case["shape"] == "slivers":
        grids[0] = (2 * case["a0"], case["a0"])
    if case["shape"] == "soup":
        grids[0] = (grids[0][0] + 3 * case["extra"], grids[0][1] + case["extra"])
    return grids


def work(case):
    """Each mesh (or BVH triangle, or point) read once, each result written once; per vertex or
    point of A one point-triangle distance (80 operations), per face of A one bound (100), both
    ways for the two-sided distance."""
    call, real = case["call"], 8 if case["double"] else 4
    if call == "batch":
        sizes = [(ga[0] * ga[1], 2 * ga[0] * ga[1], 2 * gb[0] * gb[1]) for _, ga, gb, _, _ in _batch_sizes(case)]
        return {"bytes": sum(3 * real * v + 12 * f + 9 * real * t + 16 for v, f, t in sizes),
                "flops": sum(80 * v + 100 * f for v, f, _ in sizes)}
    if call == "nearest":
        (_, t), n = _faces_of(case)[0], case["points"]
        return {"bytes": n * (3 * real + 44) + 9 * real * t, "flops": 80 * n}
    (va, fa), (vb, fb) = _faces_of(case)
    both = call == "sym"
    return {"bytes": 3 * real * (va + vb) + 12 * (fa + fb) + 16,
            "flops": 80 * (va + both * vb) + 100 * (fa + both * fb)}


# ----------------------------------------------------------------------------- 64-bit values


def _closest(p, a, b, c):
    """Closest points of triangles (a, b, c) to p, all (..., 3) in double: the foot on the plane
    where it lies inside, else the nearest of the three edges' feet."""
    def edge(x, y):
        e = y - x
        ee = (e * e).sum(-1, keepdim=True)
        t = torch.where(ee > 0, ((p - x) * e).sum(-1, keepdim=True) / ee.clamp_min(1e-300), torch.zeros_like(ee))
        return x + t.clamp(0, 1) * e

    q, d = None, None
    for x, y in ((a, b), (b, c), (c, a)):
        r = edge(x, y)
        e = ((p - r) ** 2).sum(-1, keepdim=True)
        q, d = (r, e) if q is None else (torch.where(e < d, r, q), torch.minimum(e, d))
    ab, ac, ap = b - a, c - a, p - a
    d00, d01, d11 = ((x * y).sum(-1, keepdim=True) for x, y in ((ab, ab), (ab, ac), (ac, ac)))
    d20, d21 = ((ap * x).sum(-1, keepdim=True) for x in (ab, ac))
    den = d00 * d11 - d01 * d01
    good = den > 1e-14 * d00 * d11
    den = torch.where(good, den, torch.ones_like(den))
    v, w = (d11 * d20 - d01 * d21) / den, (d00 * d21 - d01 * d20) / den
    r = a + v * ab + w * ac
    e = ((p - r) ** 2).sum(-1, keepdim=True)
    inside = good & (v >= 0) & (w >= 0) & (v + w <= 1) & (e < d)
    return torch.where(inside, r, q), torch.where(inside, e, d).squeeze(-1)


def _nearest64(P, V, F):
    """Distance and closest point of each row of P: the triangles whose centroid is among the
    nearest, and where those cannot be shown to hold the nearest one, all of them."""
    T = V.double()[F.long()]
    cen = T.mean(1)
    rad = float((T - cen[:, None]).norm(dim=-1).max())
    k = min(len(T), 96)
    dist, foot = torch.empty(len(P), dtype=torch.float64, device=DEV), torch.empty(len(P), 3, dtype=torch.float64, device=DEV)
    for at in range(0, len(P), 8192):
        p = P[at:at + 8192].double()
        near, idx = torch.cdist(p.float(), cen.float(), compute_mode="use_mm_for_euclid_dist").topk(k, largest=False)
        t = T[idx]
        q, e = _closest(p[:, None], t[:, :, 0], t[:, :, 1], t[:, :, 2])
        e, i = e.min(1)
        q = q[torch.arange(len(p), device=DEV), i]
        if k < len(T):
            open_ = torch.nonzero(near[:, -1].double() - 2e-3 - rad < e.sqrt()).squeeze(1)
            for sub in open_.split(max(1, 40_000_000 // len(T))):
                qs, es = _closest(p[sub][:, None], T[None, :, 0], T[None, :, 1], T[None, :, 2])
                e[sub], i = es.min(1)
                q[sub] = qs[torch.arange(len(sub), device=DEV), i]
        dist[at:at + 8192], foot[at:at + 8192] = e.sqrt(), q
    return dist, foot


def _diagonal(V, F):
    v = torch.as_tensor(V).to(DEV).double()[torch.as_tensor(F).to(DEV).long().reshape(-1)]
    return float((v.amax(0) - v.amin(0)).norm())


def exact(case, seed):
    """The distances, closest points, tolerances and diagonals.  A bracket has no one value: any
    [lower, upper] around h within the tolerance is a result, so its ends are None; so is the
    index of a nearest triangle, which ties leave open."""
    call = case["call"]
    if call == "nearest":
        vb, fb = _mesh_b(case, seed)
        P = _points(case, seed)
        if len(P) * len(fb) > 3e10:
            return None
        dist, foot = _nearest64(P, _stored(vb, case), fb)
        return dist, None, foot, dist.clone()

    def one(V, F, eps=None):
        dA = _diagonal(V, F)
        return dict(lower=None, upper=None, status=None, eps=eps or (case["tol"] * dA if case["rel"] else case["tol"]), dA=dA)

    if call == "batch":
        rs = [one(*_batch_pair(case, seed, k, s)[:2]) for k, s in enumerate(_batch_sizes(case))]
        return dict(lower=None, upper=None, status=None, eps=np.array([r["eps"] for r in rs]), dA=np.array([r["dA"] for r in rs]))
    va, fa = _mesh_a(case, seed)
    ab = one(_stored(va, case), fa)
    if call != "sym":
        return ab
    vb, fb = _mesh_b(case, seed)
    return [ab, ab, one(_stored(vb, case), fb, ab["eps"])]
