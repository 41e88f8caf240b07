"""Batches whose work list holds k segments of a grid's columns.

Few deep grids: the list then has more items than (grid, tile) pairs, and the
results equal, bit for bit, those of the single-grid kernel.
"""
import pytest
import torch

import paper_2301_13016_gb300 as pwlib
from paper_2301_13016_gb300 import inputs
from gpu_util import NAN

pytestmark = pytest.mark.gpu


# 17 levels: the least depth that can be cut in two; grids of one tile and several
@pytest.mark.parametrize("shapes", [[(64, 16, 17)], [(64, 16, 16), (100, 40, 100)], [(4, 5, 3), (260, 33, 128), (64, 64, 61)]],
                         ids=["one", "two", "three"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_segments_give_the_single_grids_bits(dtype, shapes):
    grids = [pwlib.Grid(*s, dtype=dtype) for s in shapes]
    coeffs = [inputs.make_coeffs(s[2], anelastic=True) for s in shapes]
    dev = [[g.from_dense(f) for f in inputs.random_fields(*s, seeds=(q, q + 10, q + 20))]
           for q, (g, s) in enumerate(zip(grids, shapes))]
    out = [[g.alloc(fill=NAN) for _ in range(3)] for g in grids]
    b = pwlib.Batch(grids, coeffs)
    tiles = sum(-(-nx // 64) * -(-ny // 16) for nx, ny, _ in shapes)
    assert b.info()["items"] > tiles
    b.tendencies(*[[d[q] for d in dev] for q in range(3)], *[[o[q] for o in out] for q in range(3)])
    b.sync()
    for g, c, d, o in zip(grids, coeffs, dev, out):
        ref = [g.alloc(fill=NAN) for _ in range(3)]
        h = pwlib.PW(g, c)
        h.tendencies(*d, *ref)
        h.sync()
        for x, y in zip(o, ref):
            assert torch.equal(x.view(torch.int16), y.view(torch.int16)) if dtype == "bf16" else torch.equal(
                x.nan_to_num(7.0), y.nan_to_num(7.0))
