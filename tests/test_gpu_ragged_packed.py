"""Narrow widths that are no multiple of 4 on the k-march's packed rows.

A 64-column tile leaves up to half of its lanes beyond the end of such a row;
packed rows cover the width in vectors of 4.  Source terms and one step equal,
bit for bit, those of a grid widened to a multiple of 4 that holds the same
values (the same operations per cell).  Heights sit at the edges of a CTA's
rows, depths at those of the coefficient table (64 levels) in one k segment.
"""
import pytest
import torch

import paper_2301_13016_gb300 as pwlib
from paper_2301_13016_gb300 import inputs
from gpu_util import NAN

pytestmark = pytest.mark.gpu


def _pair(nx, ny, nz, dtype, halo, call, nseg=0):
    """(widened, narrow) results of one call on the same values, levels 1..nz
    with the one-cell halo; the narrow handle and grid."""
    c = inputs.make_coeffs(nz, anelastic=True)
    wide = 4 * ((nx + 1) // 4 + 1)                  # holds column nx + 1
    f = inputs.random_fields(wide, ny, nz)
    scale = (2.0 ** -8,) * 3 + (64.0,) * 3 if dtype == "f16" else None
    out = []
    for n in (wide, nx):
        g = pwlib.Grid(n, ny, nz, halo=halo, dtype=dtype)
        h = pwlib.PW(g, c)
        if n == nx and nseg:
            h.set_tma_config(nseg=nseg)
        dev = [g.from_dense(x[:, :, :n + 2], scale=s) for x, s in zip(f, scale or (1.0,) * 3)]
        res = [g.alloc(fill=NAN) for _ in range(3)]
        if call == "step":
            h.step_to(*dev, *res, 0.25, scale=scale and scale[:3])
        else:
            h.tendencies(*dev, *res, scale=scale)
        h.sync()
        assert h.last_kernel == 2
        out.append([g.view(t)[:, halo - 1:halo + ny + 1, halo - 1:halo + n + 1].cpu() for t in res])
    return out[0], out[1], h, g


@pytest.mark.parametrize("call", ["tendencies", "step"])
@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("nx,over", [(33, 0), (33, 1), (35, -1), (47, 1), (62, -1), (65, 1), (79, 0), (95, 1)])
def test_packed_rows_equal_widened_grid_bitwise(nx, over, dtype, call):
    if nx > 80 and dtype == "f32":
        pytest.skip("tiles from here on")
    vec = -(-nx // 4)
    rows = 128 // vec if dtype == "f32" or vec > 10 else 13 if vec == 9 else 12
    nz = 66
    ny = rows * -(-(1 << 19) // (nx * nz * rows)) + rows + over      # above the rule's least size
    wide, got, h, g = _pair(nx, ny, nz, dtype, 1, call)
    cfg = h.tma_config(step=call == "step")
    assert (cfg["lanes_x"], cfg["ty"], cfg["cells"]) == (vec, rows, 4)
    assert 4 * 128 <= 1.25 * nx * rows              # threads without a cell: at most a fifth
    for a, b in zip(wide, got):
        assert torch.equal(a[1:-1, 1:-1, 1:nx + 1], b[1:-1, 1:-1, 1:nx + 1])
        if call == "step":                          # periodic images all round
            v = b[1:-1]
            assert torch.equal(v[:, :, 0], v[:, :, nx]) and torch.equal(v[:, :, nx + 1], v[:, :, 1])
            assert torch.equal(v[:, 0], v[:, ny]) and torch.equal(v[:, ny + 1], v[:, 1])
        else:                                       # the halo is not written
            assert torch.isnan(b[:, :, 0]).all() and torch.isnan(b[:, :, nx + 1]).all()
            assert torch.isnan(b[:, 0]).all() and torch.isnan(b[:, -1]).all()


@pytest.mark.parametrize("call", ["tendencies", "step"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("nx,nz", [(41, 64), (41, 65), (41, 130), (62, 66)])
def test_packed_rows_in_one_segment(nx, nz, dtype, call):
    ny = -(-(1 << 19) // (nx * nz)) + 3
    wide, got, h, _ = _pair(nx, ny, nz, dtype, 2, call, nseg=1)
    assert h.tma_config(step=call == "step")["nseg"] == 1
    for a, b in zip(wide, got):
        assert torch.equal(a[1:-1, 1:-1, 1:nx + 1], b[1:-1, 1:-1, 1:nx + 1])


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("nx", [97, 127, 130, 133, 191])
def test_tiled_steps_equal_widened_grid_bitwise(nx, dtype):
    """Wider ones, on tiles: every cell of a row's tail, and the images."""
    ny, nz = 169 if nx < 127 else 129, 130          # above the least size of FP32 steps on tiles
    wide, got, _, _ = _pair(nx, ny, nz, dtype, 1, "step")
    for a, b in zip(wide, got):
        assert torch.equal(a[1:-1, 1:-1, 1:nx + 1], b[1:-1, 1:-1, 1:nx + 1])
        v = b[1:-1]
        assert torch.equal(v[:, :, 0], v[:, :, nx]) and torch.equal(v[:, :, nx + 1], v[:, :, 1])
        assert torch.equal(v[:, 0], v[:, ny]) and torch.equal(v[:, ny + 1], v[:, 1])
