"""The ranked binary64 evaluation (a certified binary32 ranking decides which constraint and which
crossing give the results; binary64 evaluates those) has the bits of the whole evaluation.  On the
CPU: the same sources compiled for the host, over every kind, set of outputs, grazing rays and
degenerate solids.  On the GPU: the query call against the closed-form CPU loop at the edges of
rows and tiles."""
import ctypes

import numpy as np
import pytest

import cpu_baseline
import workloads as W

OUT = ("inside", "dist_in", "dist_out", "safety_in", "safety_out")
NAMED = {"box": W.BOX_M1, "trd": W.TRD_M3, "tube": W.TUBE_M2, "cone": W.CONE_M2, "polycone": W.polycone_m3()}
TABLE = W.solid_table(18, seed=21)


def _ranked(spec, tr, want, given):
    solid = cpu_baseline.Solid(spec)
    n = len(tr["x"])
    cols = [np.ascontiguousarray(tr[k]) for k in ("x", "y", "z", "dx", "dy", "dz")]
    ranked = np.zeros(n, np.int8)
    out = {k: np.zeros(n, np.int8 if k == "inside" else np.float64) for k in OUT}
    p = lambda a: ctypes.c_void_p(a.ctypes.data)  # noqa: E731
    cpu_baseline.load_ranked().gvcpu_query_ranked(
        solid._buf, ctypes.c_int64(n), (ctypes.c_void_p * 6)(*[c.ctypes.data for c in cols]), ctypes.c_uint(want),
        ctypes.c_int(given), p(ranked), *[p(out[k]) for k in OUT])
    return ranked == 1, out


def _same_bits(spec, tr, want, least):
    """Ranked with the code from binary32, and with the code given from binary64 (which leaves fewer
    tracks uncertain)."""
    whole = cpu_baseline.Solid(spec).query(**tr, threads=4)
    before = 0.0
    for given in (0, 1):
        sure, got = _ranked(spec, tr, want, given)
        assert sure.mean() >= max(least, before), sure.mean()
        before = sure.mean()
        for bit, k in enumerate(OUT):
            if want >> bit & 1:
                assert (got[k][sure] == whole[k][sure]).all(), (given, k, int((got[k][sure] != whole[k][sure]).sum()))


@pytest.mark.parametrize("i", range(len(TABLE)))
@pytest.mark.parametrize("want", [31, 1, 25, 4, 27, 29])
def test_ranked_random_solids(i, want):
    # a tenth of the tracks lies within 1e-8 mm of a surface; the inside code is not certain within
    # about 1e-11 mm of the band's edges, which with a few dozen ulps of margin is below 1%
    _same_bits(TABLE[i], W.tracks_for_solid(TABLE[i], 20011, seed=900 + i), want, 0.99)


@pytest.mark.parametrize("fam", W.GRAZING_FAMILIES)
def test_ranked_grazing(fam):
    spec, tr, _ = W.grazing_tracks(fam, 4000, 950 + W.GRAZING_FAMILIES.index(fam))
    _same_bits(spec, tr, 31, 0.0)


@pytest.mark.parametrize("i", range(len(W.degenerate_table())))
def test_ranked_degenerate(i):
    spec = W.degenerate_table()[i]
    _same_bits(spec, W.tracks_for_solid(spec, 20011, seed=970 + i), 31, 0.0)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 255, 257, 70_001, 152 * 3 * 1024 + 33])
@pytest.mark.parametrize("name", list(NAMED))
def test_query_fp64_bits_of_the_whole_evaluation(name, n):
    import torch

    import paper_1512_06637_gb300 as gv
    spec = NAMED[name]
    tr = W.tracks_for_solid(spec, n, seed=1000 + len(name))
    want = cpu_baseline.Solid(spec).query(**tr, threads=8)
    dev = {k: torch.from_numpy(v).cuda() for k, v in tr.items()}
    solid = gv.Solid.from_spec(spec)
    for keys in (OUT, ("dist_in",), ("inside", "safety_in")):
        got = gv.query(solid, dev, precision="fp64", want=keys)
        for k in keys:
            assert (got[k].cpu().numpy() == want[k]).all(), k


@pytest.mark.gpu
def test_polycone_fp64_two_launches_and_in_place():
    """A large polycone basket ranks in a launch of its own that leaves its verdicts in a distance
    result; a call whose result arrays are its inputs takes the one-launch pass.  Same bits."""
    import torch

    import paper_1512_06637_gb300 as gv
    n = (1 << 19) + 77
    spec = NAMED["polycone"]
    tr = W.tracks_for_solid(spec, n, seed=1100)
    want = cpu_baseline.Solid(spec).query(**tr, threads=8)
    solid = gv.Solid.from_spec(spec)
    dev = {k: torch.from_numpy(v).cuda() for k, v in tr.items()}
    for keys in (OUT, ("dist_in",), ("dist_out", "inside")):
        got = gv.query(solid, dev, precision="fp64", want=keys)
        for k in keys:
            assert (got[k].cpu().numpy() == want[k]).all(), k
    for k, col in (("dist_out", "x"), ("dist_in", "dz")):
        cols = {c: v.clone() for c, v in dev.items()}
        gv.query(solid, cols, precision="fp64", out={k: cols[col]})
        assert (cols[col].cpu().numpy() == want[k]).all(), k
