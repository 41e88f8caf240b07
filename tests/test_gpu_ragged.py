"""Widths that are no multiple of 4 on the k-march (its row tails).

The widths sit at the edges of a thread's vector (4 or 8 cells) and of a tile
(64 or 128 columns).  The source terms must equal, bit for bit, those of a
grid widened to a multiple of 4 that holds the same values (the same
operations per cell); the fused step is held to the oracle with the bounds of
the aligned widths, and its halo to the exact periodic images.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2301_13016_gb300 as pwlib
from paper_2301_13016_gb300 import inputs
from gpu_util import NAN, interior

pytestmark = pytest.mark.gpu

WIDTHS = [33, 34, 61, 63, 65, 66, 67, 127, 129, 133, 135, 257]   # with 129 x 128 rows and levels: above the rule's least size


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("nx", WIDTHS)
def test_ragged_tendencies_equal_widened_grid_bitwise(nx, dtype):
    ny, nz = 129, 128
    c = inputs.make_coeffs(nz, anelastic=True)
    wide = 4 * (nx // 4 + 1)
    if wide == nx + 1:
        wide += 4                                   # the widened grid needs column nx+1 inside
    f = inputs.random_fields(wide, ny, nz)
    gw, g = pwlib.Grid(wide, ny, nz, dtype=dtype), pwlib.Grid(nx, ny, nz, dtype=dtype)
    scale = (2.0 ** -8,) * 3 + (64.0,) * 3 if dtype == "f16" else None
    ins = scale[:3] if scale else (1.0,) * 3
    out = []
    for grid, n in ((gw, wide), (g, nx)):
        h = pwlib.PW(grid, c)
        dev = [grid.from_dense(x[:, :, :n + 2], scale=s) for x, s in zip(f, ins)]
        res = [grid.alloc(fill=NAN) for _ in range(3)]
        h.tendencies(*dev, *res, scale=scale)
        h.sync()
        assert h.last_kernel == 2
        out.append([grid.view(t)[:, :, :n + 2].cpu() for t in res])
    for a, b in zip(*out):
        assert torch.equal(a[1:-1, 1:-1, 1:nx + 1], b[1:-1, 1:-1, 1:nx + 1])
        assert torch.isnan(b[:, :, 0]).all() and torch.isnan(b[:, :, nx + 1]).all()   # halo columns not written
        assert torch.isnan(b[:, 0]).all() and torch.isnan(b[:, -1]).all()


@pytest.mark.parametrize("dtype,tol", [("f32", 3e-5), ("bf16", 3 * 2.0 ** -8), ("f16", 3 * 2.0 ** -11)])
@pytest.mark.parametrize("halo", [1, 2])
@pytest.mark.parametrize("nx", [33, 66, 127, 135])
def test_ragged_steps_match_oracle(nx, halo, dtype, tol):
    """Three fused steps: one unit roundoff of the state per step for 16-bit
    storage (1.5 would be the stated bound), 1e-5 per step for FP32."""
    ny, nz = 129, 125
    c = inputs.make_coeffs(nz)
    f = inputs.smooth_fields(nx, ny, nz)
    g = pwlib.Grid(nx, ny, nz, halo=halo, dtype=dtype)
    h = pwlib.PW(g, c)
    scale = (2.0 ** -8,) * 3 if dtype == "f16" else None
    ins = scale or (1.0,) * 3
    q = [g.from_dense(x, scale=s) for x, s in zip(f, ins)]
    tmp = [g.alloc(fill=NAN) for _ in range(3)]
    q0 = [g.to_dense(t, s).numpy() for t, s in zip(q, ins)]
    h.step(*q, *tmp, 1.0, 3, scale=scale)
    h.sync()
    assert h.last_kernel == 2
    ref = oracle.step(*q0, c, 1.0, 3)
    for t, r, s in zip(q, ref, ins):
        got = g.to_dense(t, s).numpy()
        assert np.abs(interior(got) - interior(r)).max() <= 1.5 * tol * np.abs(interior(r)).max()
        assert np.array_equal(got[1:-1], oracle.fill_halo_periodic(got)[1:-1])
        v = g.view(t)[1:-1].cpu()
        for d in range(1, halo + 1):                # halos of any depth hold the images
            assert torch.equal(v[:, :, halo - d], v[:, :, halo - d + nx])
            assert torch.equal(v[:, :, halo + nx + d - 1], v[:, :, halo + d - 1])


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("shape", [(160, 824, 41), (184, 1280, 21), (320, 512, 21), (1056, 300, 24), (164, 824, 41)])
def test_automatic_shapes_give_the_first_shapes_bits(shape, dtype):
    """Grids large enough for the choice among tile widths: source terms and a
    step equal, bit for bit, those of the first shape in one k segment."""
    nx, ny, nz = shape
    c = inputs.make_coeffs(nz, anelastic=True)
    g = pwlib.Grid(nx, ny, nz, dtype=dtype)
    f = inputs.random_fields(nx, ny, nz)
    dev = [g.from_dense(x) for x in f]
    out = []
    for fixed in (False, True):
        h = pwlib.PW(g, c)
        for call in (0, 1):
            if fixed:
                cells = 4 if dtype == "f32" or (call and nx % 8) else 8
                h.set_tma_config(ty=4 if cells == 4 else 8, stages=4, nseg=1, lanes_x=32 if cells == 4 else 16,
                                 cells=cells, rows=1 if dtype == "f32" else 3)
            res = [g.alloc(fill=NAN) for _ in range(3)]
            h.step_to(*dev, *res, 0.25) if call else h.tendencies(*dev, *res)
            h.sync()
            assert h.last_kernel == 2
            out.append([g.view(t)[1:-1].cpu() for t in res])
    for a, b in zip(out[0] + out[1], out[2] + out[3]):
        assert torch.equal(a.view(torch.int16 if dtype == "bf16" else torch.int32),
                           b.view(torch.int16 if dtype == "bf16" else torch.int32))


def test_ragged_refusals_unchanged():
    """pw_set_kernel(2), two steps per pass and a fixed launch shape still treat
    such a width as not eligible for the k-march."""
    c = inputs.make_coeffs(64)
    g = pwlib.Grid(65, 129, 64, halo=2)
    h = pwlib.PW(g, c)
    q = [g.alloc() for _ in range(6)]
    h.set_kernel(2)
    for call in (lambda: h.tendencies(*q), lambda: h.step(*q, 1.0, 1), lambda: h.step_to(*q, 1.0)):
        with pytest.raises(pwlib.PwError) as e:
            call()
        assert e.value.status == pwlib.PW_ERR_UNSUPPORTED
    h.set_kernel(0)
    h.set_step_blocking(2)
    with pytest.raises(pwlib.PwError) as e:
        h.step(*q, 1.0, 2)
    assert e.value.status == pwlib.PW_ERR_UNSUPPORTED
    h.set_step_blocking(0)
    for cfg, kernel in ((dict(lanes_x=16), 1), ({}, 2)):
        h.set_tma_config(**cfg)
        h.tendencies(*q)
        h.sync()
        assert h.last_kernel == kernel
