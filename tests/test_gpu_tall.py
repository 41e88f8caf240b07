"""Grids taller than a launch has tiles of rows for (65535 along y).

The generic kernels take any height; a width or mode that the k-march took over
from them must still run there."""
import pytest
import torch

import paper_2301_13016_gb300 as pwlib
from paper_2301_13016_gb300 import inputs

pytestmark = pytest.mark.gpu


def _random(g, n, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn(g.alloc_elems, generator=gen, device="cuda") for _ in range(n)]


def _rows(g, t, y0):
    return g.view(t)[1:-1, y0:y0 + 7, 1:-1].cpu()


@pytest.mark.parametrize("call", ["tendencies", "step"])
def test_ragged_width_beyond_the_tallest_tile_grid(call):
    """127 columns: tiles of 4 rows.  The last rows equal those of a low grid on
    the generic kernel that holds the same values."""
    ny, low, nz = 4 * 65535 + 1, 9, 3
    c = inputs.make_coeffs(nz)
    g = pwlib.Grid(127, ny, nz)
    gl = pwlib.Grid(127, low, nz)
    q = _random(g, 3, 1)
    ql = [gl.alloc() for _ in range(3)]
    for a, b in zip(q, ql):
        gl.view(b).copy_(g.view(a)[:, ny - low:])
    out = []
    for grid, f in ((g, q), (gl, ql)):
        h = pwlib.PW(grid, c)
        res = [grid.alloc() for _ in range(3)]
        h.step_to(*f, *res, 0.25) if call == "step" else h.tendencies(*f, *res)
        h.sync()
        assert h.last_kernel == 1
        out.append([_rows(grid, t, grid.ny - 7) for t in res])
    for a, b in zip(*out):
        assert torch.equal(a, b)


def test_open_adjoint_beyond_the_tallest_tile_grid():
    ny, nz = 8 * 65535 - 1, 3                       # rows 0..ny+1 in tiles of 8
    g = pwlib.Grid(5, ny, nz)
    f = _random(g, 6, 2)
    h = pwlib.PW(g, inputs.make_coeffs(nz))
    out = [torch.full((g.alloc_elems,), 7.0, device="cuda") for _ in range(3)]
    h.adjoint(*f, *out)
    h.sync()
    assert h.last_kernel == 1
    for t in out:
        v = g.view(t)[1:-1]
        assert not (v[:, 0] == 7.0).any() and not (v[:, -1] == 7.0).any() and torch.isfinite(v).all()
