"""The transport loop's tie flag between daughters without a binary32 form.  Two boolean daughters
share a face that the ray crosses 5e-10 mm after it has entered the first one, with the two entries on
either side of a binary32 rounding boundary: neighbouring floats lie 3.8e-6 mm apart there, the
binary64 distances within the tie margin 1e-9 (1 + d)."""
import numpy as np
import pytest

import oracle
from tests.helpers import to_device

pytestmark = pytest.mark.gpu

HALF = 2.5e-10  # the entries lie this far from the rounding boundary (mm)


def abutting_booleans():
    """Two unions of boxes over x in [0, 20], one with y in [-20, 0], one with y in [0, 20]."""
    eye = np.eye(3)
    box = {"kind": "box", "params": (10.0, 10.0, 10.0)}
    core = {"kind": "box", "params": (5.0, 5.0, 5.0)}
    union = {"kind": "boolean", "params": ("union", box, core, eye, np.zeros(3))}
    solids = [{"kind": "box", "params": (200.0, 200.0, 200.0)}, union]
    nodes = [{"solid": 0, "parent": -1, "R": eye, "t": np.zeros(3)}]
    nodes += [{"solid": 1, "parent": 0, "R": eye, "t": np.array([10.0, y, 0.0])} for y in (-10.0, 10.0)]
    return {"solids": solids, "nodes": nodes}


def straddling_tracks(n):
    """Rays with direction (0.48, 0.6, 0.64) that enter x = 0 at T - HALF and y = 0 at T + HALF, T half way
    between two binary32 numbers in [32, 64)."""
    k = np.random.default_rng(12).integers(0, 1 << 22, n)
    T = 32.0 + (2 * k + 1) * 2.0 ** -19
    o = np.zeros(n)
    return {"x": -0.48 * (T - HALF), "y": -0.6 * (T + HALF), "z": np.linspace(-4.0, 4.0, n) - 0.64 * T,
            "dx": o + 0.48, "dy": o + 0.6, "dz": o + 0.64}


@pytest.mark.parametrize("n", [1, 1025])
def test_tie_across_a_float_boundary(n):
    import torch

    import paper_1512_06637_gb300 as gv
    geo, tr = abutting_booleans(), straddling_tracks(n)
    node0, mat, sig, xi = np.zeros(n, np.int32), np.zeros(3, np.int32), np.zeros((1, 2)), np.full((n, 1, 4), 0.5)
    want = oracle.Geometry(geo["solids"], geo["nodes"]).transport(
        *[tr[k] for k in ("x", "y", "z", "dx", "dy", "dz")], node0, mat, sig, xi, 1)
    assert (want["tie"] == 1).all()
    out = gv.Geometry(geo["solids"], geo["nodes"]).transport(
        to_device(tr, torch), torch.from_numpy(node0).cuda(), torch.from_numpy(mat).cuda(), torch.from_numpy(sig).cuda(),
        torch.from_numpy(xi).cuda(), 1)
    got = {k: v.cpu().numpy() for k, v in out.items()}
    assert (got["tie"] == 1).all(), int((got["tie"] == 0).sum())
    # the two sides form the distances with different operations: a few units in the last place of 64
    assert np.abs(got["path"] - want["path"]).max() <= 1e-12
