"""The scanned navigation step: daughters pass a plain binary32 look before their certified
evaluation.  Checked against the oracle at the edges of rows and tiles, over many daughters (several
masks of 32) with voxel grids off, at points as far from three and more daughters, and for rays
along faces; step and safety within the step's tolerances, ``next`` exactly."""
import numpy as np
import pytest

import oracle
import workloads as W
from tests.helpers import to_device
from tests.test_gpu_nav import check_nav

pytestmark = pytest.mark.gpu


def lattice_geometry():
    """216 rotated primitives (no booleans) in a box, on a 100 mm pitch."""
    geo = W.crowded_geometry(6, seed=3)
    kinds = [s["kind"] for s in geo["solids"]]
    for nd in geo["nodes"]:
        if kinds[nd["solid"]] == "boolean":
            nd["solid"] = kinds.index("tube")
    return geo


def symmetric_tracks(n):
    """Points of the nested detector's shells midway between four cells."""
    g = np.random.default_rng(5)
    k, j, iz = g.integers(0, 10, n), g.integers(0, 8, n), g.integers(0, 3, n)
    r, ph = 19.0 + 19.0 * k, np.pi / 4 * j
    pts = np.stack([r * np.cos(ph), r * np.sin(ph), np.array([-250.0, 0.0, 250.0])[iz]], 1)
    return W.soa(pts, W.isotropic(n, g))


def axis_tracks(geo, n):
    tr = W.nested_tracks(n, 77)
    g = np.random.default_rng(6)
    ax = g.integers(0, 3, n)
    for i, c in enumerate(("dx", "dy", "dz")):
        tr[c] = np.where(ax == i, np.where(g.random(n) < 0.5, -1.0, 1.0), 0.0)
    return tr


CASES = [("lattice", 1), ("lattice", 255), ("lattice", 20_003), ("nested", 257), ("nested", 304 * 1024 + 1025),
         ("symmetric", 5001), ("axis", 20_011)]


@pytest.mark.parametrize("precision", ["fp64", "fp32_refine"])
@pytest.mark.parametrize("which,n", CASES)
def test_scan_matches_oracle(which, n, precision):
    import torch

    import paper_1512_06637_gb300 as gv
    geo = lattice_geometry() if which == "lattice" else W.nested_geometry()
    G, O = gv.Geometry(geo["solids"], geo["nodes"]), oracle.Geometry(geo["solids"], geo["nodes"])
    if which == "lattice":
        G.set_voxels(False)
        tr = W.crowded_tracks(geo, n, 8, surf_frac=0.2 if n > 1 else 0.0)
    else:
        tr = {"nested": lambda: W.nested_tracks(n, 9), "symmetric": lambda: symmetric_tracks(n),
              "axis": lambda: axis_tracks(geo, n)}[which]()
    node = O.locate(tr["x"], tr["y"], tr["z"])
    dev, dnode = to_device(tr, torch), torch.from_numpy(node).cuda()
    want = O.nav_step(*[tr[k] for k in ("x", "y", "z", "dx", "dy", "dz")], node)
    for safety in (True, False):
        out = G.step(dev, dnode, precision=precision, workspace=gv.Workspace(n), safety=safety)
        got = {k: v.cpu().numpy() for k, v in out.items()}
        if not safety:
            got["safety"] = want["safety"]
        check_nav(got, want, "fp64" if precision == "fp64" else "fp32", f"{which}-{precision}-{safety}")


@pytest.mark.parametrize("n", [1, 31, 20_003])
def test_grid_walk_matches_oracle(n):
    """The binary32 step along a grid of 216 daughters, the ones the ray certainly misses left out."""
    import torch

    import paper_1512_06637_gb300 as gv
    geo = lattice_geometry()
    G, O = gv.Geometry(geo["solids"], geo["nodes"]), oracle.Geometry(geo["solids"], geo["nodes"])
    for name, tr in (("crowded", W.crowded_tracks(geo, n, 18, surf_frac=0.2 if n > 1 else 0.0)), ("axis", axis_tracks(geo, n))):
        node = O.locate(tr["x"], tr["y"], tr["z"])
        want = O.nav_step(*[tr[k] for k in ("x", "y", "z", "dx", "dy", "dz")], node)
        out = G.step(to_device(tr, torch), torch.from_numpy(node).cuda(), precision="fp32_refine",
                     workspace=gv.Workspace(n), safety=False)
        got = {k: v.cpu().numpy() for k, v in out.items()}
        check_nav(dict(got, safety=want["safety"]), want, "fp32", f"{name}-{n}")
