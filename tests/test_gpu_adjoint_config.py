"""The adjoint's launch shape as callers read, keep and restore it, and its long
k segments (126 levels; 64 where levels may be redone)."""
import numpy as np
import pytest
import torch

import paper_2301_13016_gb300 as pwlib
from paper_2301_13016_gb300 import inputs
from gpu_util import NAN

pytestmark = pytest.mark.gpu
PER = pwlib.PW_ADJ_PERIODIC


def _fields(g, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return [g.from_dense(inputs.wrap_halo_(torch.randn((g.nz + 2, g.ny + 2, g.nx + 2), generator=gen, device="cuda")))
            for _ in range(6)]


def _run(h, f, flags):
    out = [h.grid.alloc(fill=7.0) for _ in range(3)]
    h.adjoint(*f, *out, alpha=0.7, flags=flags)
    h.sync()
    return [h.grid.view(t).cpu().numpy() for t in out], h.last_kernel


def _close(a, b, tol=3e-6):   # as in test_gpu_adjoint_march.py: a few roundings of the largest partial sums
    for x, y in zip(a, b):
        assert np.array_equal(np.isnan(x), np.isnan(y)) and np.array_equal(np.isinf(x), np.isinf(y))
        m = np.isfinite(y)
        assert np.abs(x[m] - y[m]).max() <= tol * np.abs(y[m]).max()


@pytest.mark.parametrize("shape", [(64, 8, 4), (64, 64, 64), (65, 64, 64), (128, 40, 130)])
def test_config_read_back_can_be_set(shape):
    """From 2^18 cells up the automatic shape is (4, 8, 3); set again it gives
    the same kernels in both modes."""
    g = pwlib.Grid(*shape)
    h = pwlib.PW(g, inputs.make_coeffs(g.nz, anelastic=True))
    f = _fields(g, 1)
    before = [_run(h, f, flags) for flags in (0, PER)]
    cfg = h.adjoint_config()
    h.set_adjoint_config(**cfg)
    assert h.adjoint_config() == cfg
    if g.cells >= 1 << 18:
        assert (cfg["cells"], cfg["ty"], cfg["stages"]) == (4, 8, 3)
        for flags, (ref, kernel) in zip((0, PER), before):
            got, k = _run(h, f, flags)
            assert k == kernel == 2
            _close(got, ref)


@pytest.mark.parametrize("nx", [61, 64])
@pytest.mark.parametrize("nz", [64, 65, 126, 127])
def test_one_segment_and_values_that_are_not_finite(nx, nz):
    """nseg alone fixes no shape; a segment holds at most 64 levels where levels
    are redone, else 126; the top and bottom levels are among the redone."""
    g = pwlib.Grid(nx, 70, nz)
    h = pwlib.PW(g, inputs.make_coeffs(nz, anelastic=True))
    h.set_adjoint_config(nseg=1)
    assert h.adjoint_config()["nseg"] == -(-nz // (126 if nx % 4 == 0 else 64))
    hg = pwlib.PW(g, inputs.make_coeffs(nz, anelastic=True))
    hg.set_kernel(1)
    f = _fields(g, 2)
    for flags in (0, PER):
        got, k = _run(h, f, flags)
        assert k == 2
        _close(got, _run(hg, f, flags)[0])
    for k in (1, 2, 33, min(nz, 64), nz - 1, nz):     # (the top level of a first segment among them)
        for q, t in enumerate(f[:3]):
            g.view(t)[k, 20 + q, 9:30] = float("inf")
            g.view(f[3 + q])[k - 1:k + 2, 17:27, 15:40] = 0.0
    for flags in ((0, PER) if nx % 4 else (0,)):      # (aligned periodic: zero sensitivities are not skipped)
        march, k = _run(h, f, flags)
        assert k == 2
        _close(march, _run(hg, f, flags)[0])
