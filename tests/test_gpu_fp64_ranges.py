"""Binary64 queries at every kernel of their dispatch against the whole evaluation on the CPU, bit for bit:
the ranked kernels (one track per thread, rows of 256, tiles of 1024 and 2048) and, for solids finer than
binary32 resolves, index order and tiles of 1024 and 2048 in order of work class.  Baskets repeat a short
set of tracks, so that the reference stays short."""
import numpy as np
import pytest

import cpu_baseline
import workloads as W

pytestmark = pytest.mark.gpu
OUT = ("inside", "dist_in", "dist_out", "safety_in", "safety_out")
SETS = (OUT, ("dist_out",), ("inside", "safety_in", "safety_out"), ("inside",))
SMS = 152
NAMED = {"box": W.BOX_M1, "trd": W.TRD_M3, "tube": W.TUBE_M2, "cone": W.CONE_M2, "polycone": W.polycone_m3()}
FINE = {"box": {"kind": "box", "params": (500.0, 0.005, 400.0)},
        "trd": {"kind": "trd", "params": (300.0, 280.0, 200.0, 220.0, 0.003)},
        "tube": {"kind": "tube", "params": (20.0 - 1e-6, 20.0, 30.0, 0.0, W.TWO_PI)},
        "polycone": {"kind": "polycone", "params": ((-30.0, 0.0, 2e-4, 25.0), (5.0, 5.0, 6.0, 0.0), (20.0, 30.0, 30.0, 25.0), 0.3, 4.0)}}


def _check(spec, n, seed):
    import torch

    import paper_1512_06637_gb300 as gv
    tr = W.tracks_for_solid(spec, 40_013, seed=seed, near_frac=0.2)
    want = cpu_baseline.Solid(spec).query(**tr, threads=8)
    pick = torch.from_numpy(np.random.default_rng(n).integers(0, 40_013, n)).cuda()
    dev = {k: torch.from_numpy(v).cuda()[pick] for k, v in tr.items()}
    ref = {k: torch.from_numpy(np.ascontiguousarray(want[k])).cuda()[pick] for k in OUT}
    solid = gv.Solid.from_spec(spec)
    for keys in SETS:
        got = gv.query(solid, dev, precision="fp64", want=keys)
        for k in keys:
            assert torch.equal(got[k], ref[k]), (keys, k, int((got[k] != ref[k]).sum()))


@pytest.mark.parametrize("name,n", [("tube", SMS * 1024 - 1), ("tube", SMS * 1024 + 33), ("cone", SMS * 1024 + 33)] +
                         [(k, m) for k in NAMED for m in (SMS * 3 * 1024 + 91, SMS * 3 * 4 * 2048 + 5)])
def test_ranked_kernels(name, n):
    _check(NAMED[name], n, 1200 + len(name))


@pytest.mark.parametrize("n", [SMS * 2048 - 1, SMS * 2048 + 7, SMS * 2 * 4 * 2048 + 5])
@pytest.mark.parametrize("name", list(FINE))
def test_fine_featured_kernels(name, n):
    _check(FINE[name], n, 1300 + len(name))
