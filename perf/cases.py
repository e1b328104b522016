"""The performance cases of the geometry library: what a user's program has it do, through the
public Python calls, over the range of sizes, solids, precisions and outputs that are in use.

A case is a dict of plain values.  ``form`` names the call:

  query      ``gv.query`` of one basket against one solid, device arrays
  host       ``gv.query_host`` of one basket in pinned host memory through a ``gv.Pipeline``
  batch      ``gv.Batch.run``: many baskets of mixed sizes, each against its own solid
  locate     ``gv.Geometry.locate``
  nav        ``gv.Geometry.step``: one navigation step
  transport  ``gv.Geometry.transport``: the transport loop

``solid`` is one of the library's benchmark solids (``*_bench``) or a kind, whose parameters
(1-100 mm) come from ``solid_seed``.  Tracks: half drawn inside the solid, half uniform in a world
box of twice its extent, a tenth moved to within 1e-8 mm of a surface; isotropic directions.
"""
import math
import random

import numpy as np
import torch

import paper_1512_06637_gb300 as gv

TWO_PI = 2.0 * math.pi
DEG = math.pi / 180.0
AXES = ("x", "y", "z", "dx", "dy", "dz")
OUTPUTS = {
    "all": ("inside", "dist_in", "dist_out", "safety_in", "safety_out"),
    "dist_out": ("dist_out",),
    "dist_in": ("dist_in",),
    "inside": ("inside",),
    "safety": ("inside", "safety_in", "safety_out"),
    "outside": ("inside", "dist_in", "safety_in"),
}
HALF_TOL = 0.5e-9  # half width of the surface band (mm)
MERGE = 1e-12      # crossings closer than this are one


def listed():
    return [
        # The smallest call: a basket of 1024 against a box (the latency row of the benchmark).
        {"name": "box_1k_fp32", "form": "query", "solid": "box_bench", "solid_seed": 0, "n": 1024,
         "precision": "fp32_refine", "want": "all"},
        # The paper's experiment (DistanceToOut of a tube) at a middle basket size that fills no
        # power of two, in the default precision.
        {"name": "tube_out_50k_fp64", "form": "query", "solid": "tube_bench", "solid_seed": 0, "n": 50021,
         "precision": "fp64", "want": "dist_out"},
        # An ordinary large basket of a planar solid in the mixed precision.
        {"name": "trap_3m_fp32", "form": "query", "solid": "trap", "solid_seed": 5, "n": 3000017,
         "precision": "fp32_refine", "want": "all"},
        # The headline form's largest solid call: 2^24 tracks against the 8-plane polycone.
        {"name": "polycone_16m_fp32", "form": "query", "solid": "polycone_bench", "solid_seed": 0, "n": 1 << 24,
         "precision": "fp32_refine", "want": "all"},
        # The benchmark's binary64 cone basket (the default precision).
        {"name": "cone_1m_fp64", "form": "query", "solid": "cone_bench", "solid_seed": 0, "n": 1 << 20,
         "precision": "fp64", "want": "all"},
        # A large polycone basket in the default precision.
        {"name": "polycone_4m_fp64", "form": "query", "solid": "polycone_bench", "solid_seed": 0, "n": 4000037,
         "precision": "fp64", "want": "all"},
        # A boolean solid (a box minus a tube), the benchmark's basket size.
        {"name": "subtraction_1m_fp64", "form": "query", "solid": "subtraction_bench", "solid_seed": 0,
         "n": 1 << 20, "precision": "fp64", "want": "all"},
        # Baskets in pinned host memory: copies in, the pass, copies out.
        {"name": "host_tube_4m_fp32", "form": "host", "solid": "tube_bench", "solid_seed": 0, "n": 4100003,
         "precision": "fp32_refine", "want": "all"},
        # The scheduler's form: 4096 baskets of 16 to 4096 tracks over 64 solids of the six kinds.
        {"name": "batch_4096_fp32", "form": "batch", "solid_seed": 4, "solids": 64, "baskets": 4096, "lo": 16,
         "hi": 4096, "precision": "fp32_refine"},
        # One navigation step in the nested detector (world, 10 tube shells, 320 box cells).
        {"name": "nav_nested_4m_fp32", "form": "nav", "geometry": "nested", "shells": 10, "n": 1 << 22,
         "precision": "fp32_refine", "safety": True},
        # One navigation step, with safety, in a volume with 1728 daughters of every kind.
        {"name": "nav_crowded_256k_fp64", "form": "nav", "geometry": "crowded", "lattice": 12, "n": 1 << 18,
         "precision": "fp64", "safety": True},
        # The transport loop in the nested detector, default precision.
        {"name": "transport_1m_fp64", "form": "transport", "geometry": "nested", "shells": 10, "n": 1 << 20,
         "kmax": 32, "precision": "fp64"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: mostly single-solid baskets of 16 to 12 M tracks, of any kind, either
    precision and any set of outputs; else one of the other forms over its range of sizes."""
    form = rng.choice(["query"] * 6 + ["boolean", "host", "batch", "nav", "crowded", "locate", "transport"])
    precision = rng.choice(["fp64", "fp32_refine"])
    if form in ("query", "host"):
        kind = rng.choice(["box", "trd", "trap", "tube", "cone", "polycone"])
        heavy = kind == "polycone" and precision == "fp64"
        hi = 4_000_000 if heavy or form == "host" else 12_000_000
        return {"form": form, "solid": kind, "solid_seed": rng.randrange(1000),
                "n": _log_int(rng, 16 if form == "query" else 20_000, hi), "precision": precision,
                "want": rng.choice(["all", "all", "all", "dist_out", "dist_in", "inside", "safety", "outside"])}
    if form == "boolean":
        return {"form": "query", "solid": rng.choice(["union", "subtraction", "intersection"]),
                "solid_seed": rng.randrange(1000), "n": _log_int(rng, 100, 2_000_000), "precision": "fp64",
                "want": rng.choice(["all", "all", "dist_out", "dist_in", "safety"])}
    if form == "batch":
        return {"form": "batch", "solid_seed": rng.randrange(1000), "solids": rng.randrange(1, 100),
                "baskets": _log_int(rng, 8, 4096), "lo": rng.randrange(1, 65), "hi": rng.randrange(128, 4097),
                "precision": precision}
    if form == "nav":
        return {"form": "nav", "geometry": "nested", "shells": rng.randrange(2, 11), "n": _log_int(rng, 100, 4_000_000),
                "precision": precision, "safety": rng.random() < 0.7}
    if form == "crowded":
        return {"form": "nav", "geometry": "crowded", "lattice": rng.randrange(3, 11), "n": _log_int(rng, 100, 100_000),
                "precision": precision, "safety": rng.random() < 0.5}
    if form == "locate":
        if rng.random() < 0.5:
            return {"form": "locate", "geometry": "nested", "shells": rng.randrange(2, 11), "n": _log_int(rng, 100, 8_000_000)}
        return {"form": "locate", "geometry": "crowded", "lattice": rng.randrange(3, 11), "n": _log_int(rng, 100, 2_000_000)}
    return {"form": "transport", "geometry": "nested", "shells": rng.randrange(2, 11), "n": _log_int(rng, 100, 1_000_000),
            "kmax": rng.randrange(4, 33), "precision": precision}


# ---------------------------------------------------------------- solids

def _random_primitive(kind, r, lo=1.0, hi=100.0):
    u = lambda a=lo, b=hi: r.uniform(a, b)  # noqa: E731
    if kind == "box":
        return {"kind": "box", "params": (u(), u(), u())}
    if kind == "trd":
        return {"kind": "trd", "params": (u(), u(), u(), u(), u())}
    if kind == "trap":  # the +dz face is k times the -dz face: planar side faces
        dz, dy, dxa, dxb = u(), u(lo, hi / 1.5), u(lo, hi / 1.5), u(lo, hi / 1.5)
        k, th, ph, al = r.uniform(0.5, 1.5), r.uniform(0, 15) * DEG, r.uniform(0, 15) * DEG, r.uniform(-15, 15) * DEG
        return {"kind": "trap", "params": ((dz, th, ph, dy, dxa, dxb, al, k * dy, k * dxa, k * dxb, al),)}
    sphi, dphi = 0.0, TWO_PI
    if r.randrange(3):
        sphi, dphi = r.uniform(0, 360) * DEG, r.uniform(30, 330) * DEG
    if kind == "tube":
        rmax = u(lo + 1.0)
        return {"kind": "tube", "params": (r.uniform(0, rmax - 0.5) if r.randrange(4) else 0.0, rmax, u(), sphi, dphi)}
    if kind == "cone":
        a, b = u(lo + 1.0), u(lo + 1.0)
        return {"kind": "cone", "params": (r.uniform(0, a - 0.5) if r.randrange(3) else 0.0, a,
                                           r.uniform(0, b - 0.5) if r.randrange(3) else 0.0, b, u(), sphi, dphi)}
    nz, span = r.randrange(2, 9), u(max(lo, 10.0))
    z = sorted(r.uniform(-span, span) for _ in range(nz))
    z = [v + 0.5 * i for i, v in enumerate(z)]
    rmin = [r.uniform(0, 0.5 * hi) * (r.random() < 0.7) for _ in range(nz)]
    return {"kind": "polycone", "params": (tuple(z), tuple(rmin), tuple(v + r.uniform(lo, 0.5 * hi) for v in rmin), sphi, dphi)}


def _rotation(r):
    q, t = np.linalg.qr(np.array([[r.gauss(0, 1) for _ in range(3)] for _ in range(3)]))
    q = q * np.sign(np.diag(t))
    if np.linalg.det(q) < 0:
        q[:, 0] = -q[:, 0]
    return q


def _random_boolean(r, op, lo, hi):
    kinds = ("box", "trd", "trap", "tube", "cone", "polycone")
    a = _random_primitive(r.choice(kinds), r, lo, hi)
    c = _random_primitive(r.choice(kinds), r, lo, 0.7 * hi)
    R = _rotation(r)
    t = np.array([r.uniform(-0.3, 0.3) for _ in range(3)]) * _half(a)
    return {"kind": "boolean", "params": (op, a, c, R.tolist(), t.tolist())}


def _polycone_bench():
    g = np.random.Generator(np.random.PCG64(1512_06637 + 1002))
    z = -50.0 + np.sort(g.uniform(0.0, 86.0, 8)) + 2.0 * np.arange(8)
    rmin = g.uniform(1.0, 40.0, 8)
    rmax = np.minimum(50.0, rmin + g.uniform(2.0, 30.0, 8))
    return {"kind": "polycone", "params": (tuple(z.tolist()), tuple(rmin.tolist()), tuple(rmax.tolist()), 0.0, TWO_PI)}


def _spec(kind, seed):
    if kind == "box_bench":
        return {"kind": "box", "params": (10.0, 20.0, 30.0)}
    if kind == "tube_bench":
        return {"kind": "tube", "params": (5.0, 20.0, 30.0, 0.0, 270.0 * DEG)}
    if kind == "cone_bench":
        return {"kind": "cone", "params": (0.0, 10.0, 5.0, 25.0, 40.0, 0.0, TWO_PI)}
    if kind == "polycone_bench":
        return _polycone_bench()
    if kind == "subtraction_bench":
        return {"kind": "boolean", "params": ("subtraction", {"kind": "box", "params": (10.0, 20.0, 30.0)},
                                              {"kind": "tube", "params": (5.0, 20.0, 30.0, 0.0, 270.0 * DEG)},
                                              [[1.0, 0, 0], [0, 1.0, 0], [0, 0, 1.0]], [3.0, -4.0, 5.0])}
    r = random.Random("%s %d" % (kind, seed))
    if kind in ("union", "subtraction", "intersection"):
        return _random_boolean(r, kind, 5.0, 60.0)
    return _random_primitive(kind, r)


def _trap_params(spec):
    k, p = spec["kind"], spec["params"]
    if k == "box":
        return (p[2], 0, 0, p[1], p[0], p[0], 0, p[1], p[0], p[0], 0)
    if k == "trd":
        return (p[4], 0, 0, p[2], p[0], p[0], 0, p[3], p[1], p[1], 0)
    return p[0]


def _vertices(spec):
    dz, th, ph, dy1, dx1, dx2, a1, dy2, dx3, dx4, a2 = _trap_params(spec)
    out = []
    for zf, dy, dxa, dxb, al in ((-dz, dy1, dx1, dx2, a1), (dz, dy2, dx3, dx4, a2)):
        cx, cy = zf * math.tan(th) * math.cos(ph), zf * math.tan(th) * math.sin(ph)
        sh = dy * math.tan(al)
        out += [(cx - sh - dxa, cy - dy, zf), (cx - sh + dxa, cy - dy, zf),
                (cx + sh - dxb, cy + dy, zf), (cx + sh + dxb, cy + dy, zf)]
    return np.array(out, dtype=np.float64)


def _profile(spec):
    k, p = spec["kind"], spec["params"]
    if k == "tube":
        return [-p[2], p[2]], [p[0], p[0]], [p[1], p[1]], p[3], p[4]
    if k == "cone":
        return [-p[4], p[4]], [p[0], p[2]], [p[1], p[3]], p[5], p[6]
    return [list(v) if i < 3 else v for i, v in enumerate(p)]


PLANAR = ("box", "trd", "trap")


def _half(spec):
    """Half extents of a box around the origin that holds the solid."""
    if spec["kind"] == "boolean":
        _, a, c, R, t = spec["params"]
        corners = np.array([[i, j, k] for i in (-1, 1) for j in (-1, 1) for k in (-1, 1)]) * _half(c)
        return np.maximum(_half(a), np.abs(corners @ np.array(R).T + np.array(t)).max(axis=0))
    if spec["kind"] in PLANAR:
        return np.abs(_vertices(spec)).max(axis=0)
    z, _, rmax, _, _ = _profile(spec)
    return np.array([max(rmax), max(rmax), max(abs(z[0]), abs(z[-1]))])


# ---------------------------------------------------------------- inputs

def _rand(g, *shape):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)


def _isotropic(g, n):
    d = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64)
    return d / d.norm(dim=1, keepdim=True)


def _points(spec, n, g, surface):
    """n points drawn from the solid's parametric interior, or on its faces."""
    if spec["kind"] == "boolean":
        _, a, c, R, t = spec["params"]
        R, t = (torch.tensor(v, device="cuda", dtype=torch.float64) for v in (R, t))
        m = n // 2
        return torch.cat([_points(a, m, g, surface), _points(c, n - m, g, surface) @ R.T + t])
    face = torch.randint(0, 6, (n,), generator=g, device="cuda") if surface else None
    if spec["kind"] in PLANAR:
        v = torch.tensor(_vertices(spec), device="cuda")
        w = _rand(g, 3, n)
        if surface:
            for i in range(3):
                w[i] = torch.where(face == 2 * i, 0.0, torch.where(face == 2 * i + 1, 1.0, w[i]))
        out = torch.zeros((n, 3), device="cuda", dtype=torch.float64)
        for j in range(2):
            for i in range(2):
                for k in range(2):
                    b = (w[2] if j else 1 - w[2]) * (w[1] if i else 1 - w[1]) * (w[0] if k else 1 - w[0])
                    out += b[:, None] * v[4 * j + 2 * i + k]
        return out
    z, rmin, rmax, sphi, dphi = _profile(spec)
    zt, lo, hi = (torch.tensor(v, device="cuda", dtype=torch.float64) for v in (z, rmin, rmax))
    wz, wr, wp = _rand(g, 3, n)
    if surface:
        wz = torch.where(face == 0, 0.0, torch.where(face == 1, 1.0, wz))
        wr = torch.where(face == 2, 0.0, torch.where(face == 3, 1.0, wr))
        if dphi < TWO_PI:
            wp = torch.where(face == 4, 0.0, torch.where(face == 5, 1.0, wp))
    zz = zt[0] + wz * (zt[-1] - zt[0])
    k = (torch.searchsorted(zt, zz, right=True) - 1).clamp(0, len(z) - 2)
    f = (zz - zt[k]) / (zt[k + 1] - zt[k])
    r0, r1 = lo[k] + f * (lo[k + 1] - lo[k]), hi[k] + f * (hi[k + 1] - hi[k])
    r = torch.where(wr == 1.0, r1, (r0 * r0 + wr * (r1 * r1 - r0 * r0)).sqrt())
    p = sphi + wp * min(dphi, TWO_PI)
    return torch.stack([r * p.cos(), r * p.sin(), zz], 1)


def _soa(p, d):
    return dict(zip(AXES, [c.contiguous() for c in (*p.T, *d.T)]))


def _tracks(spec, n, g):
    half = torch.tensor(_half(spec) * 2.0 + 1.0, device="cuda", dtype=torch.float64)
    p = (2 * _rand(g, n, 3) - 1) * half
    pick = _rand(g, n)
    inside = pick < 0.45
    near = (pick >= 0.45) & (pick < 0.55)
    p[inside] = _points(spec, int(inside.sum()), g, False)
    m = int(near.sum())
    p[near] = _points(spec, m, g, True) + _isotropic(g, m) * (1e-8 * _rand(g, m, 1))
    return _soa(p, _isotropic(g, n))


def _baskets(case):
    r = random.Random("baskets %d %d" % (case["solid_seed"], case["baskets"]))
    kinds = ("box", "trd", "trap", "tube", "cone", "polycone")
    solids = [_random_primitive(kinds[i % 6], r) for i in range(case["solids"])]
    sizes = [max(case["lo"], min(case["hi"], int(math.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]))))))
             for _ in range(case["baskets"])]
    return solids, np.array(sizes), np.array([r.randrange(case["solids"]) for _ in sizes])


def _nested(shells):
    """World box, tube shells, 32 box cells in each shell."""
    eye = np.eye(3)
    solids = [{"kind": "box", "params": (250.0, 250.0, 550.0)}, {"kind": "box", "params": (4.5, 4.5, 112.5)}]
    nodes = [{"solid": 0, "parent": -1, "R": eye, "t": np.zeros(3)}]
    for k in range(shells):
        rmin = 10.0 + 19.0 * k
        solids.append({"kind": "tube", "params": (rmin, rmin + 18.0, 500.0, 0.0, TWO_PI)})
        nodes.append({"solid": 2 + k, "parent": 0, "R": eye, "t": np.zeros(3)})
    for k in range(shells):
        for zc in (-375.0, -125.0, 125.0, 375.0):
            for j in range(8):
                c, s = math.cos((22.5 + 45.0 * j) * DEG), math.sin((22.5 + 45.0 * j) * DEG)
                rm = 19.0 + 19.0 * k
                nodes.append({"solid": 1, "parent": 1 + k, "R": np.array([[c, -s, 0.0], [s, c, 0.0], [0.0, 0.0, 1.0]]),
                              "t": np.array([rm * c, rm * s, zc])})
    return solids, nodes, np.array([250.0, 250.0, 550.0])


def _crowded(lattice):
    """A world box holding lattice^3 randomly rotated solids at a 100 mm pitch, every eighth
    solid a boolean, one of the daughters a box with 27 daughters of its own."""
    r = random.Random("crowded %d" % lattice)
    kinds = ("box", "trd", "trap", "tube", "cone", "polycone")
    half = 50.0 * lattice
    table, small = [], []
    while len(table) < 40:
        k = len(table)
        s = (_random_boolean(r, r.choice(["union", "subtraction", "intersection"]), 5.0, 18.0) if k % 8 == 7
             else _random_primitive(kinds[k % 6], r, 4.0, 26.0))
        if np.linalg.norm(_half(s)) < 45.0:
            table.append(s)
    while len(small) < 12:
        s = _random_primitive(kinds[len(small) % 6], r, 0.8, 5.2)
        if np.linalg.norm(_half(s)) < 9.0:
            small.append(s)
    solids = [{"kind": "box", "params": (half, half, half)}] + table + small + [{"kind": "box", "params": (28.0, 28.0, 28.0)}]
    nodes = [{"solid": 0, "parent": -1, "R": np.eye(3), "t": np.zeros(3)}]
    c0 = -50.0 * (lattice - 1)
    for q in range(lattice ** 3):
        t = np.array([c0 + 100.0 * (q // lattice ** 2), c0 + 100.0 * (q // lattice % lattice), c0 + 100.0 * (q % lattice)])
        if q == 0:
            nodes.append({"solid": len(solids) - 1, "parent": 0, "R": _rotation(r), "t": t})
        else:
            nodes.append({"solid": 1 + r.randrange(40), "parent": 0, "R": _rotation(r),
                          "t": t + np.array([r.uniform(-5, 5) for _ in range(3)])})
    for q in range(27):
        nodes.append({"solid": 41 + r.randrange(12), "parent": 1, "R": _rotation(r),
                      "t": 18.0 * np.array([q // 9 - 1.0, q // 3 % 3 - 1.0, q % 3 - 1.0])})
    return solids, nodes, np.array([half, half, half])


def _tables(case):
    return _nested(case["shells"]) if case["geometry"] == "nested" else _crowded(case["lattice"])


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    n, form = case.get("n"), case["form"]
    if form in ("query", "host"):
        spec = _spec(case["solid"], case["solid_seed"])
        tr = _tracks(spec, n, g)
        want = OUTPUTS[case["want"]]
        if form == "host":
            pin = {k: torch.empty(n, dtype=torch.float64, pin_memory=True).copy_(v) for k, v in tr.items()}
            out = {k: torch.zeros(n, dtype=torch.int8 if k == "inside" else torch.float64, pin_memory=True) for k in want}
            return {"case": case, "solid": gv.Solid.from_spec(spec), "tracks": pin, "out": out,
                    "pipeline": gv.Pipeline(chunk_tracks=1 << 20, slots=3)}
        return {"case": case, "solid": gv.Solid.from_spec(spec), "tracks": tr,
                "out": gv.alloc_results(n, tr["x"].device, want),
                "workspace": gv.Workspace(n) if case["precision"] == "fp32_refine" else None}
    if form == "batch":
        solids, sizes, ids = _baskets(case)
        total, offs = int(sizes.sum()), np.concatenate([[0], np.cumsum(sizes)[:-1]])
        owner = torch.tensor(np.repeat(ids, sizes), device="cuda")
        tr = {k: torch.empty(total, dtype=torch.float64, device="cuda") for k in AXES}
        for s, spec in enumerate(solids):
            at = (owner == s).nonzero(as_tuple=True)[0]
            for k, v in _tracks(spec, at.numel(), g).items():
                tr[k][at] = v
        return {"case": case, "tracks": tr, "out": gv.alloc_results(total, tr["x"].device),
                "batch": gv.Batch([gv.Solid.from_spec(s) for s in solids], offs, sizes, ids)}
    solids, nodes, half = _tables(case)
    geom = gv.Geometry(solids, nodes)
    p = (2 * _rand(g, n, 3) - 1) * torch.tensor(half, device="cuda")
    st = {"case": case, "geometry": geom, "tracks": _soa(p, _isotropic(g, n))}
    if form == "locate":
        st["out"] = torch.empty(n, dtype=torch.int32, device="cuda")
        return st
    st["node"] = geom.locate(st["tracks"])
    if form == "nav":
        st["out"] = {"step": torch.empty(n, dtype=torch.float64, device="cuda"),
                     "next": torch.empty(n, dtype=torch.int32, device="cuda")}
        if case["safety"]:
            st["out"]["safety"] = torch.empty(n, dtype=torch.float64, device="cuda")
        st["workspace"] = gv.Workspace(n) if case["precision"] == "fp32_refine" else None
        return st
    # transport: vacuum world, a light material in the shells, a dense one in the cells
    st["material"] = torch.tensor([0 if d["parent"] < 0 else 1 if d["parent"] == 0 else 2 for d in nodes],
                                  dtype=torch.int32, device="cuda")
    st["sigma_n"] = torch.tensor([[0.0, 0.0], [0.01, 0.002], [0.05, 0.02]], dtype=torch.float64, device="cuda")
    st["xi"] = 1.0 - _rand(g, n, case["kmax"], 4)
    return st


def run(state):
    case = state["case"]
    form = case["form"]
    if form == "query":
        return gv.query(state["solid"], state["tracks"], precision=case["precision"], out=state["out"],
                        workspace=state["workspace"])
    if form == "host":
        out = gv.query_host(state["solid"], state["tracks"], state["out"], state["pipeline"], precision=case["precision"])
        state["pipeline"].join()
        return out
    if form == "batch":
        return state["batch"].run(state["tracks"], state["out"], precision=case["precision"])
    if form == "locate":
        return state["geometry"].locate(state["tracks"], out=state["out"])
    if form == "nav":
        return state["geometry"].step(state["tracks"], state["node"], precision=case["precision"], out=state["out"],
                                      workspace=state["workspace"], safety=case["safety"])
    return state["geometry"].transport(state["tracks"], state["node"], state["material"], state["sigma_n"], state["xi"],
                                       case["kmax"], precision=case["precision"])


def work(case):
    """Bytes: every input read once, every output written once.  Operations: the decision
    quantities of the solid's surfaces and one crossing of one surface per distance, a few
    surfaces per track; for the forms over a geometry, of the volume the track is in, the one it
    goes to and its nearest (transport: ten steps)."""
    form = case["form"]
    if form in ("query", "host"):
        want = OUTPUTS[case["want"]]
        dirs = "dist_in" in want or "dist_out" in want
        b = 24 + 24 * dirs + sum(1 if k == "inside" else 8 for k in want)
        return {"bytes": float(b * case["n"]), "flops": float((20 + 20 * dirs) * case["n"])}
    if form == "batch":
        n = float(_baskets(case)[1].sum())
        return {"bytes": 81 * n, "flops": 40 * n}
    n = float(case["n"])
    if form == "locate":
        return {"bytes": 28 * n, "flops": 60 * n}
    if form == "nav":
        return {"bytes": (52 + 12 + 8 * case["safety"]) * n, "flops": 150 * n}
    steps = min(10.0, case["kmax"])
    return {"bytes": (52 + 42 + 32 * steps) * n, "flops": 200 * steps * n}


# ------------------------------------------------- the same in plain 64-bit torch
#
# A solid as a list of constraints whose largest value s is negative inside.  A distance is found
# by taking every crossing of every constraint surface along the ray, sorting them and testing
# the middle of each gap.

def _build(spec):
    kind = spec["kind"]
    if kind == "boolean":
        op, a, c, R, t = spec["params"]
        return {"bool": op, "a": _build(a), "c": _build(c), "R": np.array(R, float), "t": np.array(t, float)}
    if kind == "box":
        return {"box": [float(v) for v in spec["params"]]}
    if kind in PLANAR:
        v = _vertices(spec)
        mid, planes = v.mean(axis=0), []
        for q in ((0, 4, 5, 1), (2, 3, 7, 6), (0, 2, 6, 4), (1, 5, 7, 3)):
            A, B, C, D = v[list(q)]
            m = np.cross(C - A, D - B)
            m = m / np.linalg.norm(m)
            if m @ (mid - A) > 0:
                m = -m
            planes.append((*m, float(np.mean(v[list(q)] @ m))))
        return {"planes": planes, "dz": float(_trap_params(spec)[0])}
    z, rmin, rmax, sphi, dphi = _profile(spec)
    line = lambda r, k: ((r[k + 1] - r[k]) / (z[k + 1] - z[k]), r[k] - (r[k + 1] - r[k]) / (z[k + 1] - z[k]) * z[k])  # noqa: E731
    last = len(z) - 1
    return {"z": [float(v) for v in z], "out": [line(rmax, k) for k in range(last)],
            "in": [line(rmin, k) if rmin[k] > 0 or rmin[k + 1] > 0 else None for k in range(last)],
            "phi": None if dphi >= TWO_PI else
            ((math.sin(sphi), -math.cos(sphi)), (-math.sin(sphi + dphi), math.cos(sphi + dphi)), dphi > math.pi)}


def _section(S, z):
    zt = torch.tensor(S["z"], device=z.device, dtype=torch.float64)
    return (torch.searchsorted(zt, z.contiguous(), right=True) - 1).clamp(0, len(S["z"]) - 2)


def _walls(S, k):
    """Coefficients (a, b, cosine) of the outer and inner walls of section k, per track."""
    dev = k.device
    def col(lines):  # noqa: E306
        a, b = (torch.tensor([0.0 if q is None else q[j] for q in lines], device=dev, dtype=torch.float64)[k] for j in (0, 1))
        return a, b, 1.0 / (1.0 + a * a).sqrt()
    has = torch.tensor([q is not None for q in S["in"]], device=dev)[k]
    return col(S["out"]), col(S["in"]), has


def _phi_pair(S, x, y):
    return [n[0] * x + n[1] * y for n in S["phi"][:2]]


def _s(S, x, y, z, closed=None):
    """The decision quantity at points; closed: of a polycone's section as a piece of its own."""
    if "box" in S:
        D = S["box"]
        return torch.maximum(torch.maximum(x.abs() - D[0], y.abs() - D[1]), z.abs() - D[2])
    if "planes" in S:
        v = z.abs() - S["dz"]
        for p in S["planes"]:
            v = torch.maximum(v, p[0] * x + p[1] * y + p[2] * z - p[3])
        return v
    r = (x * x + y * y).sqrt()
    k = _section(S, z) if closed is None else torch.full_like(z, closed, dtype=torch.int64)
    (oa, ob, oc), (ia, ib, ic), has = _walls(S, k)
    zt = torch.tensor(S["z"], device=z.device, dtype=torch.float64)
    lo, hi = (zt[0], zt[-1]) if closed is None else (zt[closed], zt[closed + 1])
    v = torch.maximum(torch.maximum((r - (oa * z + ob)) * oc, lo - z), z - hi)
    v = torch.maximum(v, torch.where(has, ((ia * z + ib) - r) * ic, -math.inf))
    if S["phi"]:
        f = _phi_pair(S, x, y)
        v = torch.maximum(v, torch.minimum(*f) if S["phi"][2] else torch.maximum(*f))
    return v


def _frame(B, q):
    """Tracks in the second component's frame."""
    M, t = B["R"], B["t"]
    p = [q[i] - t[i] for i in range(3)]
    rot = lambda v: [M[0, i] * v[0] + M[1, i] * v[1] + M[2, i] * v[2] for i in range(3)]  # noqa: E731
    return rot(p) + (rot(q[3:]) if len(q) > 3 else [])


def _s_any(S, q):
    if "bool" not in S:
        return _s(S, *q[:3])
    a, c = _s(S["a"], *q[:3]), _s(S["c"], *_frame(S, q[:3]))
    return {"union": torch.minimum, "intersection": torch.maximum}.get(S["bool"], lambda p, r: torch.maximum(p, -r))(a, c)


def _code(s):
    return torch.where(s < -HALF_TOL, 0, torch.where(s > HALF_TOL, 2, 1))


def _safeties(S, q):
    """(code, SafetyToIn, SafetyToOut)."""
    s = _s_any(S, q)
    code = _code(s)
    v_in, v_out = s, -s
    if "bool" in S:
        ca, ia, oa = _safeties(S["a"], q)
        cc, ic, oc = _safeties(S["c"], _frame(S, q[:3]))
        none = torch.full_like(s, -math.inf)
        if S["bool"] == "union":
            v_in = torch.minimum(ia, ic)
            v_out = torch.maximum(torch.where(ca == 0, oa, none), torch.where(cc == 0, oc, none))
        elif S["bool"] == "intersection":
            v_out = torch.minimum(oa, oc)
            v_in = torch.maximum(torch.where(ca == 2, ia, none), torch.where(cc == 2, ic, none))
        else:
            v_out = torch.minimum(oa, ic)
            v_in = torch.maximum(torch.where(ca == 2, ia, none), torch.where(cc == 0, oc, none))
    elif "z" in S and len(S["z"]) > 2:
        pieces = torch.stack([_s(S, *q[:3], closed=k) for k in range(len(S["z"]) - 1)])
        v_in = pieces.min(dim=0).values
        v_out = -pieces.gather(0, _section(S, q[2])[None])[0]
    return code, torch.where(code == 0, -1.0, torch.where(code == 1, 0.0, v_in)), \
        torch.where(code == 2, -1.0, torch.where(code == 1, 0.0, v_out))


def _crossings(S, q):
    x, y, z, u, v, w = q
    if "bool" in S:
        return _crossings(S["a"], q) + _crossings(S["c"], _frame(S, q))
    if "box" in S:
        return [(e * S["box"][i] - q[i]) / q[3 + i] for i in range(3) for e in (-1.0, 1.0)]
    if "planes" in S:
        return [-(p[0] * x + p[1] * y + p[2] * z - p[3]) / (p[0] * u + p[1] * v + p[2] * w) for p in S["planes"]] + \
            [(e * S["dz"] - z) / w for e in (-1.0, 1.0)]
    out = [(e - z) / w for e in S["z"]]
    if S["phi"]:
        out += [-a / b for a, b in zip(_phi_pair(S, x, y), _phi_pair(S, u, v))]
    r2, rad, a0 = x * x + y * y, x * u + y * v, u * u + v * v
    r = r2.sqrt()
    for k in range(len(S["z"]) - 1):
        for wall in (S["out"][k], S["in"][k]):
            if wall is None:
                continue
            P, D = wall[0] * z + wall[1], wall[0] * w
            A, B, C = a0 - D * D, rad - P * D, (r - P) * (r + P)
            disc = B * B - A * C
            h = -(B + torch.where(B >= 0, 1.0, -1.0) * disc.clamp(min=0).sqrt())
            for t in (h / A, C / h):
                out.append(torch.where((disc > 0) & (P + t * D >= 0), t, math.nan))
    return out


def _starts(S, q, grows=False):
    """Surface start: does every constraint within the band shrink along the ray (grows: does
    one of them grow)?"""
    x, y, z, u, v, w = q
    if "box" in S:
        g = [(q[i].abs() - S["box"][i], torch.where(q[i] < 0, -q[3 + i], q[3 + i])) for i in range(3)]
    elif "planes" in S:
        g = [(p[0] * x + p[1] * y + p[2] * z - p[3], p[0] * u + p[1] * v + p[2] * w) for p in S["planes"]]
        g.append((z.abs() - S["dz"], torch.where(z < 0, -w, w)))
    else:
        r = (x * x + y * y).sqrt()
        rd = (x * u + y * v) / r
        (oa, ob, oc), (ia, ib, ic), has = _walls(S, _section(S, z))
        g = [((r - (oa * z + ob)) * oc, (rd - oa * w) * oc),
             (torch.where(has, ((ia * z + ib) - r) * ic, -math.inf), (ia * w - rd) * ic),
             (S["z"][0] - z, -w), (z - S["z"][-1], w)]
        if S["phi"]:
            f, d = _phi_pair(S, x, y), _phi_pair(S, u, v)
            if S["phi"][2]:
                g.append((torch.minimum(*f), torch.where(f[0] <= f[1], d[0], d[1])))
            else:
                g += list(zip(f, d))
    res = torch.full_like(x, not grows, dtype=torch.bool)
    for val, der in g:
        near = val >= -HALF_TOL
        res = (res | (near & (der > 0))) if grows else (res & ~(near & (der >= 0)))
    return res


def _entering(S, q):
    if "bool" not in S:
        return _starts(S, q)
    qc = _frame(S, q)
    na, nc = (_s(S["a"], *q[:3]).abs() <= HALF_TOL), (_s(S["c"], *qc[:3]).abs() <= HALF_TOL)
    ea, ec = _starts(S["a"], q), _starts(S["c"], qc, grows=S["bool"] == "subtraction")
    return (na & ea) | (nc & ec) if S["bool"] == "union" else (~na | ea) & (~nc | ec)


def _distances(S, q, code):
    """(DistanceToIn, DistanceToOut)."""
    t = torch.stack(_crossings(S, q))
    t = torch.where(t > 0, t, math.inf)  # NaN and crossings behind the start: none
    t = t.sort(dim=0).values
    edge = torch.cat([torch.zeros_like(t[:1]), t])
    fin = torch.isfinite(t)
    ahead = torch.where(fin, t, torch.nan_to_num(edge[:-1], posinf=0.0) + 1.0)
    m = 0.5 * (torch.nan_to_num(edge[:-1], posinf=0.0) + ahead)
    m = torch.cat([m, torch.where(fin[-1:], t[-1:] + 1.0, 0.0)])
    m = torch.where(torch.isfinite(edge), m, 1e9)  # past the last crossing: outside
    inside = _s_any(S, [(a + m * b) for a, b in zip(q[:3], q[3:])]) <= 0
    inside &= torch.isfinite(edge)
    short = torch.cat([(t - edge[:-1]) <= MERGE, torch.zeros_like(fin[:1])])
    for i in range(1, len(inside)):  # a gap shorter than the merge distance vanishes
        inside[i] = torch.where(short[i], inside[i - 1], inside[i])
    d_in, d_out = torch.full_like(t[0], math.inf), torch.full_like(t[0], math.inf)
    for i in range(len(t) - 1, -1, -1):
        d_in = torch.where(inside[i + 1] & ~inside[i], t[i], d_in)
        d_out = torch.where(inside[i] & ~inside[i + 1], t[i], d_out)
    ent = _entering(S, q)
    d_out = torch.where(torch.isfinite(d_out), d_out, torch.where(code == 1, 0.0, d_out))
    d_in = torch.where(code == 0, -1.0, torch.where((code == 1) & ent, 0.0, d_in))
    d_out = torch.where(code == 2, -1.0, torch.where((code == 1) & ~ent, 0.0, d_out))
    return d_in, d_out


def _answers(spec, tr, want, chunk=1 << 18):
    S, n = _build(spec), tr["x"].numel()
    out = {k: torch.empty(n, dtype=torch.float64, device="cuda") for k in want if k != "inside"}
    for i in range(0, n, chunk):
        q = [tr[k][i:i + chunk] for k in AXES]
        code, s_in, s_out = _safeties(S, q)
        vals = {"safety_in": s_in, "safety_out": s_out}
        if "dist_in" in want or "dist_out" in want:
            vals["dist_in"], vals["dist_out"] = _distances(S, q, code)
        for k in out:
            out[k][i:i + chunk] = vals[k]
    return dict(out, inside=None) if "inside" in want else out


def exact(case, seed):
    form = case["form"]
    if form in ("locate", "transport") or case.get("geometry") == "crowded":
        return None  # whole numbers only; or too long in plain torch
    st = prepare(case, seed)
    if form in ("query", "host"):
        tr = {k: v.cuda() for k, v in st["tracks"].items()}
        return _answers(_spec(case["solid"], case["solid_seed"]), tr, OUTPUTS[case["want"]])
    if form == "batch":
        solids, sizes, ids = _baskets(case)
        owner = torch.tensor(np.repeat(ids, sizes), device="cuda")
        out = {k: torch.empty(owner.numel(), dtype=torch.float64, device="cuda") for k in OUTPUTS["all"] if k != "inside"}
        for s, spec in enumerate(solids):
            at = (owner == s).nonzero(as_tuple=True)[0]
            if at.numel():
                for k, v in _answers(spec, {a: st["tracks"][a][at] for a in AXES}, OUTPUTS["all"]).items():
                    if v is not None:
                        out[k][at] = v
        return dict(out, inside=None)
    solids, nodes, _ = _tables(case)
    place = []
    for d in nodes:  # global placements
        R, t = np.asarray(d["R"], float), np.asarray(d["t"], float)
        place.append((R, t) if d["parent"] < 0 else (place[d["parent"]][0] @ R, place[d["parent"]][0] @ t + place[d["parent"]][1]))
    tr, node = st["tracks"], st["node"]
    step = torch.full_like(tr["x"], -1.0)
    safe = torch.full_like(tr["x"], -1.0)
    for v in range(len(nodes)):
        every = (node == v).nonzero(as_tuple=True)[0]
        for at in every.split(1 << 19):
            q = [tr[k][at] for k in AXES]
            best, near = None, None
            for c in [v] + [i for i, d in enumerate(nodes) if d["parent"] == v]:
                S = _build(solids[nodes[c]["solid"]])
                loc = _frame({"R": place[c][0], "t": place[c][1]}, q)
                code, s_in, s_out = _safeties(S, loc)
                d_in, d_out = _distances(S, loc, code)
                d, s = (d_out, s_out) if c == v else (d_in, s_in)
                d, s = torch.where(d < 0, math.inf, d), torch.where(s < 0, math.inf, s)
                best = d if best is None else torch.minimum(best, d)
                near = s if near is None else torch.minimum(near, s)
            step[at] = torch.where(torch.isfinite(best), best, -1.0)
            safe[at] = torch.where(torch.isfinite(near), near, -1.0)
    return {"step": step, "next": None, "safety": safe if case["safety"] else None}
