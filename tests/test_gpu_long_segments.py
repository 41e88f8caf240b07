"""k segments longer than the coefficient table a CTA holds (64 levels for the
scalar forms, 128 for x pairs), on every tile of the automatic choice.

One segment gives, bit for bit, the result of many short ones, at depths just
below, at and above the table's refills; ragged widths too (a segment count
alone fixes no shape), each of whose tiles is reached at one of the widths."""
import pytest
import torch

import paper_2301_13016_gb300 as pwlib
from paper_2301_13016_gb300 import inputs
from gpu_util import NAN

pytestmark = pytest.mark.gpu

# dtype, call, width -> lanes x rows x cells, form
TILES = {
    ("f32", "tendencies", 127): (32, 4, 4, 1), ("f32", "tendencies", 191): (16, 8, 4, 1),
    ("f32", "tendencies", 95): (8, 16, 4, 1), ("f32", "tendencies", 128): (32, 4, 4, 1),
    ("f32", "step", 127): (32, 4, 4, 1), ("f32", "step", 191): (16, 8, 4, 1), ("f32", "step", 95): (8, 16, 4, 1),
    ("f32", "step", 128): (32, 4, 4, 1), ("f32", "tendencies", 64): (16, 4, 4, 1), ("f32", "step", 60): (16, 4, 4, 1),
    ("bf16", "tendencies", 127): (16, 8, 8, 3), ("bf16", "tendencies", 191): (8, 16, 8, 3),
    ("bf16", "tendencies", 128): (16, 8, 8, 3), ("bf16", "step", 127): (32, 4, 4, 3),
    ("bf16", "step", 191): (16, 8, 4, 3), ("bf16", "step", 128): (16, 8, 8, 3),
}


@pytest.mark.parametrize("nz", [64, 65, 66, 127, 128, 129, 130])
@pytest.mark.parametrize("dtype,call,nx", list(TILES))
def test_one_segment_equals_many(dtype, call, nx, nz):
    # above the ragged rule's least size; narrower tiles are for grids of several waves of CTAs
    ny = 705 if nx in (95, 191) else -(-(1 << 19) // (nx * nz)) + 5 if nx > 64 else 9
    g = pwlib.Grid(nx, ny, nz, dtype=dtype)
    q = [g.from_dense(x) for x in inputs.random_fields(nx, ny, nz, device="cuda")]
    out = []
    for nseg in (1, nz // 2):
        h = pwlib.PW(g, inputs.make_coeffs(nz, anelastic=True))
        h.set_tma_config(nseg=nseg)
        cfg = h.tma_config(step=call == "step")
        assert cfg["nseg"] == nseg and cfg["stages"] == 4
        if nseg == 1:
            assert (cfg["lanes_x"], cfg["ty"], cfg["cells"], cfg["rows"]) == TILES[dtype, call, nx]
        res = [g.alloc(fill=NAN) for _ in range(3)]
        h.step_to(*q, *res, 0.25) if call == "step" else h.tendencies(*q, *res)
        h.sync()
        assert h.last_kernel == 2
        out.append([g.view(t)[1:-1, 1:-1, 1:-1] for t in res])
    for a, b in zip(*out):
        assert torch.isfinite(a.float()).all() and torch.equal(a, b)
