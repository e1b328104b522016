"""The ranked evaluation of booleans (bool_rank.cuh) has the bits of the whole one, compiled for the
host: every operation, random pairs of all primitive kinds and placements, sets of outputs, and components
with faces on one another."""
import ctypes

import numpy as np
import pytest

import cpu_baseline
import workloads as W

OPS = ("union", "subtraction", "intersection")


def _both(spec, tr, want):
    op, a, c, R, t = spec["params"]
    sa, sc = cpu_baseline.Solid(a), cpu_baseline.Solid(c)
    n = len(tr["x"])
    cols = [np.ascontiguousarray(tr[k]) for k in ("x", "y", "z", "dx", "dy", "dz")]
    Rv, tv = np.ascontiguousarray(R, np.float64).reshape(9), np.ascontiguousarray(t, np.float64)
    whole, got, ranked = np.zeros((n, 5)), np.zeros((n, 5)), np.zeros(n, np.int8)
    p = lambda x: ctypes.c_void_p(x.ctypes.data)  # noqa: E731
    cpu_baseline.load_ranked().gvcpu_bool(OPS.index(op), sa._buf, sc._buf, p(Rv), p(tv), ctypes.c_int64(n),
                                          (ctypes.c_void_p * 6)(*[x.ctypes.data for x in cols]), ctypes.c_uint(want),
                                          p(whole), p(got), p(ranked))
    return whole, got, ranked == 1


def _check(spec, tr, want, least):
    whole, got, sure = _both(spec, tr, want)
    assert sure.mean() >= least, sure.mean()
    for bit, col in ((1, 0), (2, 1), (4, 2), (8, 3), (16, 4)):
        if want & bit:
            same = (whole[sure, col] == got[sure, col]) | (np.isnan(whole[sure, col]) & np.isnan(got[sure, col]))
            assert same.all(), (bit, int((~same).sum()), whole[sure][~same][:2], got[sure][~same][:2])


@pytest.mark.parametrize("seed", range(60))
def test_ranked_boolean_bits(seed):
    g = np.random.default_rng(300 + seed)
    spec = W.boolean_random(g, op=OPS[seed % 3])
    tr = W.tracks_for_solid(spec, 8009, seed=400 + seed)
    form = all(s["kind"] != "polycone" or len(s["params"][0]) == 2 for s in spec["params"][1:3])
    for want in (31, 25, 4, 3):
        # a tenth of the tracks is on a component's surface, of which about a tenth within the band
        _check(spec, tr, want, 0.9 if form else 0.0)


@pytest.mark.parametrize("op", OPS)
def test_ranked_boolean_shared_faces(op):
    """Unrotated components with common planes and axes: many crossings coincide."""
    tube = {"kind": "tube", "params": (5.0, 10.0, 30.0, 0.0, W.TWO_PI)}
    for a, c, t in (({"kind": "box", "params": (10.0, 20.0, 30.0)}, {"kind": "box", "params": (10.0, 10.0, 30.0)}, (0, 10, 0)),
                    ({"kind": "box", "params": (10.0, 20.0, 30.0)}, tube, (0, 0, 0)), (tube, tube, (0, 0, 30)), (tube, tube, (0, 0, 0))):
        spec = {"kind": "boolean", "params": (op, a, c, np.eye(3), np.array(t, float))}
        _check(spec, W.tracks_for_solid(spec, 8009, seed=77), 31, 0.0)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 257, 152 * 2 * 256 + 91])
@pytest.mark.parametrize("op", OPS)
def test_query_boolean_bits_of_the_whole_evaluation(op, n):
    import torch

    import paper_1512_06637_gb300 as gv
    names = ("inside", "dist_in", "dist_out", "safety_in", "safety_out")
    for seed in range(4):
        spec = W.boolean_random(np.random.default_rng(500 + seed), op=op)
        tr = W.tracks_for_solid(spec, n, seed=600 + seed, near_frac=0.1 if n > 1 else 0.0)
        whole = _both(spec, tr, 31)[0]
        dev = {k: torch.from_numpy(v).cuda() for k, v in tr.items()}
        solid = gv.Solid.from_spec(spec)
        for keys in (names, ("dist_in",), ("inside", "safety_out")):
            got = gv.query(solid, dev, precision="fp64", want=keys)
            for k in keys:
                assert (got[k].cpu().numpy() == whole[:, names.index(k)]).all(), (seed, k)
