"""Batches with booleans and fine-featured solids (evaluated whole by a kernel of their own) among solids
that rank: the bits of the single-solid binary64 call for every basket, in both precisions for the solids
evaluated in binary64, with baskets at the edges of tiles and parts and the largest tile length."""
import numpy as np
import pytest

import workloads as W
from tests.helpers import QUERIES, to_device

pytestmark = pytest.mark.gpu
FINE = {"kind": "tube", "params": (20.0 - 1e-6, 20.0, 30.0, 0.0, W.TWO_PI)}
SPECS = [W.boolean_random(np.random.default_rng(500), op="subtraction"), FINE, W.CONE_M2,
         W.boolean_random(np.random.default_rng(505), op="union"), W.BOX_M1]
SIZES = [1, 255, 257, 2047, 2049, 5003, 31, 512, 8193, 1024]


@pytest.mark.parametrize("precision", ["fp64", "fp32_refine"])
@pytest.mark.parametrize("ids", [[0, 1, 2, 3, 4, 0, 1, 2, 3, 4], [0, 3, 1, 0, 3, 1, 0, 3, 1, 0], [2, 4] * 5])
@pytest.mark.parametrize("config", [None, (512, 16)])
def test_batch_has_the_bits_of_single_calls(ids, precision, config):
    import torch

    import paper_1512_06637_gb300 as gv
    offs = np.concatenate([[0], np.cumsum(SIZES)[:-1]])
    parts = [W.tracks_for_solid(SPECS[s], n, seed=40 + i, near_frac=0.2 if n > 1 else 0.0) for i, (s, n) in enumerate(zip(ids, SIZES))]
    tr = to_device({k: np.concatenate([p[k] for p in parts]) for k in parts[0]}, torch)
    solids = [gv.Solid.from_spec(s) for s in SPECS]
    batch = gv.Batch(solids, offs, np.array(SIZES), np.array(ids))
    if config:
        batch.set_config(*config)
    n = sum(SIZES)
    for keys in (QUERIES, ("inside", "safety_in")):
        out = gv.alloc_results(n, "cuda", keys)
        batch.run(tr, out, precision=precision)
        for s, size, at in zip(ids, SIZES, offs):
            if precision != "fp64" and s in (2, 4):
                continue
            part = slice(int(at), int(at + size))
            want = gv.query(solids[s], {k: v[part] for k, v in tr.items()}, precision="fp64", want=keys)
            for k in keys:
                assert torch.equal(out[k][part], want[k]), (s, size, k)
