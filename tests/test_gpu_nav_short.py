"""Short binary32 navigation baskets (8 lanes per track, tracks left over evaluated whole one per
thread) against the oracle on both sides of the limit, with and without booleans among the daughters,
and tracks whose node does not exist."""
import numpy as np
import pytest

import oracle
import workloads as W
from tests.helpers import to_device
from tests.test_gpu_nav import check_nav
from tests.test_gpu_nav_scan import axis_tracks, symmetric_tracks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 8192, 8193])
@pytest.mark.parametrize("which", ["nested", "symmetric", "axis", "crowded"])
def test_short_baskets_match_oracle(which, n):
    import torch

    import paper_1512_06637_gb300 as gv
    geo = W.crowded_geometry(4) if which == "crowded" else W.nested_geometry()
    G, O = gv.Geometry(geo["solids"], geo["nodes"]), oracle.Geometry(geo["solids"], geo["nodes"])
    tr = {"nested": lambda: W.nested_tracks(n, 19), "symmetric": lambda: symmetric_tracks(n), "axis": lambda: axis_tracks(geo, n),
          "crowded": lambda: W.crowded_tracks(geo, n, 20, surf_frac=0.3 if n > 1 else 0.0)}[which]()
    node = O.locate(tr["x"], tr["y"], tr["z"])
    dev, dnode = to_device(tr, torch), torch.from_numpy(node).cuda()
    want = O.nav_step(*[tr[k] for k in ("x", "y", "z", "dx", "dy", "dz")], node)
    for safety in (True, False):
        out = G.step(dev, dnode, precision="fp32_refine", workspace=gv.Workspace(n), safety=safety)
        got = {k: v.cpu().numpy() for k, v in out.items()}
        if not safety:
            got["safety"] = want["safety"]
        check_nav(got, want, "fp32", f"{which}-{n}-{safety}")


def test_short_basket_unknown_nodes():
    import torch

    import paper_1512_06637_gb300 as gv
    geo = W.nested_geometry()
    n = 257
    node = np.full(n, -1, np.int32)
    node[::2] = len(geo["nodes"])
    out = gv.Geometry(geo["solids"], geo["nodes"]).step(to_device(W.nested_tracks(n, 21), torch), torch.from_numpy(node).cuda(),
                                                        precision="fp32_refine", workspace=gv.Workspace(n))
    for k in ("step", "safety", "next"):
        assert (out[k].cpu().numpy() == -1).all(), k
