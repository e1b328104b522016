"""The binary32 pass for planar solids: a call for some of the outputs (codes and safeties take an
instance without distances, large box baskets another refinement) gives the bits of the same call on the
same tracks in short baskets, which take the one-launch pass, at the edges of the dispatch.  (Which
tracks are refined depends on the outputs asked for, so other output sets may differ in the last bits.)"""
import pytest

import workloads as W
from tests.helpers import QUERIES, to_device

pytestmark = pytest.mark.gpu

SOLIDS = {"box": W.BOX_M1, "trd": W.TRD_M3, "trap": next(s for s in W.solid_table(18, seed=21) if s["kind"] == "trap")}
SETS = (("inside",), ("inside", "safety_in", "safety_out"), ("safety_out",), ("dist_in",), ("inside", "dist_out"))


@pytest.mark.parametrize("name,n", [("box", 65537), ("box", 1 << 22), ("box", (1 << 22) + 5), ("trd", 65537), ("trd", 300_007),
                                    ("trap", 65537), ("trap", 300_007)])
def test_output_sets_have_the_bits_of_short_baskets(name, n):
    import torch

    import paper_1512_06637_gb300 as gv
    dev = to_device(W.tracks_for_solid(SOLIDS[name], n, seed=31), torch)
    solid, ws = gv.Solid.from_spec(SOLIDS[name]), gv.Workspace(n)
    for keys in (QUERIES,) + SETS:
        got = gv.query(solid, dev, precision="fp32_refine", workspace=ws, want=keys)
        ref = gv.alloc_results(n, "cuda", keys)
        for at in range(0, n, 65536):
            part = slice(at, min(at + 65536, n))
            gv.query(solid, {k: v[part] for k, v in dev.items()}, precision="fp32_refine", workspace=ws,
                     out={k: v[part] for k, v in ref.items()})
        for k in keys:
            assert torch.equal(got[k], ref[k]), (keys, k)
