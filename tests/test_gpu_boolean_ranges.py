"""Boolean queries at the limits of their dispatch (evaluated whole, ranked in rows of 256 or tiles of 1024
per block, in equal parts or in turn) give the bits of the same tracks in short baskets, which are
evaluated whole; random tracks and starts on the components' surfaces."""
import numpy as np
import pytest

import workloads as W
from tests.helpers import QUERIES, to_device

pytestmark = pytest.mark.gpu
SPECS = {"subtraction": W.boolean_random(np.random.default_rng(500), op="subtraction"),
         "union": W.boolean_random(np.random.default_rng(501), op="union"),
         "intersection": W.boolean_random(np.random.default_rng(511), op="intersection")}
SMS = 152


@pytest.mark.parametrize("n", [SMS * 256, SMS * 256 + 1, SMS * 512 + 1, SMS * 1024 + 1, SMS * 2048 - 1, SMS * 2048, SMS * 6144 - 31,
                               SMS * 6144 + 91])
@pytest.mark.parametrize("op", list(SPECS))
def test_boolean_dispatch_keeps_the_bits(op, n):
    import torch

    import paper_1512_06637_gb300 as gv
    spec = SPECS[op]
    tr = W.tracks_for_solid(spec, 40_013, seed=700 + len(op), near_frac=0.4)
    pick = np.random.default_rng(n).integers(0, 40_013, n)  # repeated tracks: the reference stays short
    solid = gv.Solid.from_spec(spec)
    ref, half = {}, 20_007
    for at in (0, half):
        part = gv.query(solid, to_device({k: v[at:at + half] for k, v in tr.items()}, torch), precision="fp64")
        for k, v in part.items():
            ref.setdefault(k, []).append(v)
    index = torch.from_numpy(pick).cuda()
    ref = {k: torch.cat(v)[index] for k, v in ref.items()}
    dev = {k: v[index].contiguous() for k, v in to_device(tr, torch).items()}
    for keys in (QUERIES, ("dist_out",), ("inside", "safety_in", "safety_out"), ("inside",)):
        got = gv.query(solid, dev, precision="fp64", want=keys)
        for k in keys:
            assert torch.equal(got[k], ref[k]), (keys, k)
