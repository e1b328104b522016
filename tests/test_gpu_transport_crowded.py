"""The transport loop among more than 128 daughters of every kind, booleans among them, against the
oracle's loop (the nested detector of the other transport tests holds boxes and full tubes): the walk
along the grid and its resumption, candidates without a binary32 form, tracks evaluated whole, starts on
surfaces; and the same with the grids off."""
import numpy as np
import pytest

import oracle
import workloads as W
from tests.helpers import to_device
from tests.test_gpu_transport import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,n,surf", [(6, 6007, 0.0), (6, 6007, 0.3), (8, 2003, 0.1)])
def test_crowded_transport_matches_oracle(lattice, n, surf):
    import torch

    import paper_1512_06637_gb300 as gv
    geo, kmax = W.crowded_geometry(lattice), 24
    tr = W.crowded_tracks(geo, n, seed=50 + lattice, surf_frac=surf)
    m, xi = W.crowded_materials(geo), W.transport_xi(n, kmax, seed=51)
    O, G = oracle.Geometry(geo["solids"], geo["nodes"]), gv.Geometry(geo["solids"], geo["nodes"])
    assert G.voxel_count >= 1
    node0 = O.locate(tr["x"], tr["y"], tr["z"])
    want = O.transport(*[tr[k] for k in ("x", "y", "z", "dx", "dy", "dz")], node0, m["node_material"], m["sigma_n"], xi, kmax)
    args = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (node0, m["node_material"], np.asarray(m["sigma_n"], np.float64), xi)]
    for grids in (True, False):
        G.set_voxels(grids)
        out = G.transport(to_device(tr, torch), *args, kmax)
        check({k: v.cpu().numpy() for k, v in out.items()}, want)
        tie = out["tie"].cpu().numpy()
        assert (tie != want["tie"]).mean() < 0.01, (grids, (tie != want["tie"]).sum())
