"""The navigation step's plain binary32 look at a placed daughter, compiled for the host, against the
whole binary64 evaluation in the daughter's frame: a miss is one, the bounds hold the entry, a point
called outside is, and the safety lies within the margin.  Boxes and tubes of 0.1 to 1000 mm at random
placements up to 1000 mm away; points far off, near and on the surface; rays toward the daughter, at
random, along axes and nearly along them."""
import ctypes

import numpy as np
import pytest

import cpu_baseline
import workloads as W


def _look(tag, half, rmin, R, t, tr):
    n = len(tr["x"])
    cols = [np.ascontiguousarray(tr[k]) for k in ("x", "y", "z", "dx", "dy", "dz")]
    out = np.zeros((n, 7), np.float32)
    p = lambda a: ctypes.c_void_p(np.ascontiguousarray(a, np.float64).ctypes.data)  # noqa: E731
    keep = [np.ascontiguousarray(a, np.float64) for a in (half, R, t)]
    cpu_baseline.load_ranked().gvcpu_plain_look(
        ctypes.c_int(tag), p(keep[0]), ctypes.c_double(rmin), p(keep[1]), p(keep[2]), ctypes.c_int64(n),
        (ctypes.c_void_p * 6)(*[c.ctypes.data for c in cols]), ctypes.c_void_p(out.ctypes.data))
    return out.astype(np.float64)


@pytest.mark.parametrize("seed", range(24))
def test_plain_look_bounds(seed):
    g = np.random.default_rng(100 + seed)
    size = 10.0 ** g.uniform(-1, 3)
    kind = ("box", "tube", "trd")[seed % 3]
    if kind == "box":
        spec, rmin = {"kind": "box", "params": tuple(size * g.uniform(0.05, 1, 3))}, 0.0
    elif kind == "tube":
        rmax = size * g.uniform(0.1, 1)
        rmin = rmax * g.uniform(0.1, 0.98) if g.random() < 0.7 else 0.0
        spec = {"kind": "tube", "params": (rmin, rmax, size * g.uniform(0.05, 1), 0.0, W.TWO_PI)}
    else:
        spec, rmin = {"kind": "trd", "params": tuple(size * g.uniform(0.1, 1, 5))}, 0.0
    R = W.random_rotation(g) if g.random() < 0.7 else np.eye(3)
    t = g.uniform(-1, 1, 3) * 10.0 ** g.uniform(0, 3)
    n = 30_000
    half = W.bounding_half(spec)
    loc = g.uniform(-1, 1, (n, 3)) * half * 10.0 ** g.uniform(0, 2.5, (n, 1))
    m = n // 4
    loc[:m] = W._sample_surface(spec, m, g) + W.isotropic(m, g) * 10.0 ** g.uniform(-10, 0, (m, 1)) * size
    d = W.isotropic(n, g)
    aim = g.uniform(-1.1, 1.1, (n, 3)) * half - loc
    d = np.where(g.random((n, 1)) < 0.6, aim / np.linalg.norm(aim, axis=1, keepdims=True), d)
    ax = np.zeros((n, 3))
    ax[np.arange(n), g.integers(0, 3, n)] = 1.0
    along = g.random((n, 1)) < 0.1
    tilt = ax + W.isotropic(n, g) * 10.0 ** g.uniform(-12, -1, (n, 1)) * (g.random((n, 1)) < 0.7)
    d = np.where(along, tilt / np.linalg.norm(tilt, axis=1, keepdims=True), d)
    world = W.soa(loc @ R.T + t, d @ R.T)
    # the frame change of the library, in its order
    v = np.stack([world["x"] - t[0], world["y"] - t[1], world["z"] - t[2]])
    e = np.stack([world["dx"], world["dy"], world["dz"]])
    back = lambda a: [(R[0, i] * a[0] + R[1, i] * a[1]) + R[2, i] * a[2] for i in range(3)]  # noqa: E731
    tr = W.soa(np.stack(back(v), 1), np.stack(back(e), 1))
    whole = cpu_baseline.Solid(spec).query(**tr, threads=4)
    miss, lo, by, miss2, outside, saf, margin = _look({"box": 0, "tube": 1, "trd": 2}[kind], half, rmin, R, t, world).T
    din = whole["dist_in"]
    hit = np.isfinite(din) & (din >= 0)
    assert not (hit & (miss == 1)).any() and not (hit & (miss2 == 1)).any()
    assert (lo[hit] <= din[hit]).all(), (lo[hit] - din[hit]).max()
    sure = by < 1e36
    assert (whole["inside"][sure] == 2).all()
    assert np.isfinite(din[sure]).all() and (din[sure] <= by[sure]).all()
    assert (whole["inside"][outside == 1] == 2).all()
    if kind != "trd":
        s = np.where(whole["inside"] == 2, whole["safety_in"], np.where(whole["inside"] == 0, -whole["safety_out"], 0.0))
        assert (np.abs(saf - s) <= margin).all()
    # the look is worth something: most misses are seen, most entries bounded from both sides
    far = margin < 1e-3 * size
    if far.all():
        assert (miss == 1).sum() > 0.5 * (~np.isfinite(din)).sum()
