"""Fused steps of few CTAs run an instance of their own.

It gives the bits of the instance larger grids take (forced here by fixing the
shape), halo images included, on both sides of the rule's limits: 2^17 cells and
64 columns for 16 lanes per row; 2^18 cells, and above that one wave of CTAs (608 on
152 SMs), for 32."""
import pytest
import torch

import paper_2301_13016_gb300 as pwlib
from paper_2301_13016_gb300 import inputs
from gpu_util import NAN

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,shape", [("f32", s) for s in (
    (4, 1, 3), (60, 1, 12), (60, 5, 3), (52, 52, 43), (60, 84, 26), (60, 85, 26), (64, 30, 20),     # 131040, 132600 cells
    (68, 1, 3), (68, 9, 12), (120, 64, 17), (132, 7, 70), (256, 32, 32), (256, 33, 32), (592, 89, 38), (256, 256, 64))] + [
    ("bf16", (60, 5, 7)), ("bf16", (32, 69, 25)), ("f16", (60, 84, 26))])
def test_few_cells_give_the_same_bits(dtype, shape):
    nx, ny, nz = shape
    g = pwlib.Grid(nx, ny, nz, dtype=dtype)
    c = inputs.make_coeffs(nz, anelastic=True)
    q = [g.from_dense(x, scale=0.125) for x in inputs.random_fields(nx, ny, nz)]
    out = []
    for fixed in (False, True):
        h = pwlib.PW(g, c)
        if fixed:
            h.set_tma_config(ty=4, stages=4, lanes_x=32 if nx > 64 else 16, cells=4, rows=1)
        res = [g.alloc(fill=NAN) for _ in range(3)]
        h.step_to(*q, *res, 0.25, scale=(0.125,) * 3)
        h.sync()
        assert h.last_kernel == 2
        out.append([g.view(t)[1:-1].cpu() for t in res])
    for a, b in zip(*out):
        assert torch.isfinite(a.float()).all()
        assert torch.equal(a.view(torch.int16 if dtype != "f32" else torch.int32),
                           b.view(torch.int16 if dtype != "f32" else torch.int32))
