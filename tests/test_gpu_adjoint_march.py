"""The k-march adjoint against the generic gather kernel.

Both evaluate the same terms in FP32 in different orders, so they may differ by
a few roundings of the largest partial sums: 64 terms of at most 8 roundings
each bound the difference by 512 u ~ 3e-5 of the terms' sizes; random terms
stay near sqrt(64) u, held to 3e-6 of the largest entry here.  Both modes are
also held to the oracle elsewhere (tests/test_gpu_adjoint.py).
"""
import numpy as np
import pytest
import torch

import paper_2301_13016_gb300 as pwlib
from paper_2301_13016_gb300 import inputs
from gpu_util import NAN

pytestmark = pytest.mark.gpu
INF = float("inf")


def _fields(g, seed, n=6, wrap=False):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for _ in range(n):
        x = torch.randn((g.nz + 2, g.ny + 2, g.nx + 2), generator=gen, device="cuda")
        out.append(g.from_dense(inputs.wrap_halo_(x) if wrap else x))
    return out


def _both(g, fields, flags, base=None, shapes=True):
    """(march, generic) results, levels 1..nz with the one-cell halo."""
    res = []
    for kernel in (0, 1):
        h = pwlib.PW(g, inputs.make_coeffs(g.nz, anelastic=True))
        h.set_kernel(kernel)
        out = [b.clone() for b in base] if base else [g.alloc(fill=7.0) for _ in range(3)]
        h.adjoint(*fields, *out, alpha=0.7, flags=flags)
        h.sync()
        assert h.last_kernel == (1 if kernel else 2)
        res.append([g.view(t).cpu().numpy() for t in out])
    return res


def _close(a, b, tol=3e-6):
    for x, y in zip(a, b):
        assert np.array_equal(np.isnan(x), np.isnan(y)) and np.array_equal(np.isinf(x), np.isinf(y))
        m = np.isfinite(y)
        assert np.abs(x[m] - y[m]).max() <= tol * np.abs(y[m]).max()


# widths at the edges of vectors and of 64- and 128-column tiles (which start at
# column -3), rows at the edges of 8- and 16-row tiles (which start at row 0)
OPEN = [(5, 4, 3), (33, 7, 5), (57, 14, 9), (59, 15, 70), (60, 30, 17), (123, 6, 12), (124, 9, 64), (125, 31, 65),
        (252, 40, 6), (389, 21, 20)]


@pytest.mark.parametrize("halo", [1, 2])
@pytest.mark.parametrize("shape", OPEN, ids=[f"{a}x{b}x{c}" for a, b, c in OPEN])
def test_open_mode_matches_generic(shape, halo):
    if halo > min(shape[:2]):
        pytest.skip("halo deeper than the grid")
    g = pwlib.Grid(*shape, halo=halo)
    f = _fields(g, 1)
    base = _fields(g, 2, 3)
    _close(*_both(g, f, 0))
    _close(*_both(g, f, pwlib.PW_ADJ_ADD_LAMBDA))
    _close(*_both(g, f, pwlib.PW_ADJ_ACCUMULATE, base))


@pytest.mark.parametrize("shape", [(512, 24, 24), (256, 33, 40), (64, 100, 44), (60, 130, 70), (388, 43, 131)])
def test_periodic_automatic_shapes_match_generic(shape):
    """Above the size from which the automatic shapes are taken."""
    g = pwlib.Grid(*shape)
    f = _fields(g, 3, wrap=True)
    base = _fields(g, 4, 3)
    _close(*_both(g, f, pwlib.PW_ADJ_PERIODIC))
    _close(*_both(g, f, pwlib.PW_ADJ_PERIODIC | pwlib.PW_ADJ_ADD_LAMBDA))
    _close(*_both(g, f, pwlib.PW_ADJ_PERIODIC | pwlib.PW_ADJ_ACCUMULATE, base))


# widths that are no multiple of 4: the march writes all but the outermost ring of
# cells; the sensitivities' halos (here NaN) are neither read nor written
@pytest.mark.parametrize("shape", [(33, 200, 40), (61, 70, 65), (126, 63, 34), (127, 64, 40), (193, 15, 100)])
def test_periodic_any_width_matches_generic(shape):
    g = pwlib.Grid(*shape)
    f = _fields(g, 3, wrap=True)
    for t in f[3:]:
        v = g.view(t)
        v[:, 0] = v[:, -1] = NAN
        v[:, :, 0] = v[:, :, -1] = NAN
    lam = [t.clone() for t in f[3:]]
    base = _fields(g, 4, 3)
    _close(*_both(g, f, pwlib.PW_ADJ_PERIODIC))
    _close(*_both(g, f, pwlib.PW_ADJ_PERIODIC | pwlib.PW_ADJ_ADD_LAMBDA))
    _close(*_both(g, f, pwlib.PW_ADJ_PERIODIC | pwlib.PW_ADJ_ACCUMULATE, base))
    for a, b in zip(f[3:], lam):
        assert torch.equal(a.nan_to_num(5.0), b.nan_to_num(5.0))
    v = g.view(f[1])                                # values that are not finite under zero sensitivities
    v[3:9, 5:11, 7:30] = INF
    for t in f[3:]:
        g.view(t)[2:11, 4:13, 6:32] = 0.0
    march, generic = _both(g, f, pwlib.PW_ADJ_PERIODIC)
    _close(march, generic)
    assert all(np.isfinite(x).all() for x in march)


@pytest.mark.parametrize("bad", [NAN, INF, -INF])
@pytest.mark.parametrize("flags", [0, pwlib.PW_ADJ_ADD_LAMBDA, pwlib.PW_ADJ_ACCUMULATE])
def test_open_mode_skips_zero_sensitivities(bad, flags):
    """Values that are not finite count only where a sensitivity is not 0, in
    the interior, the halo, its corners, at the surface, the lid and the
    padding around the field."""
    g = pwlib.Grid(125, 21, 12, halo=2)
    f = _fields(g, 5)
    base = _fields(g, 6, 3)
    gen = torch.Generator().manual_seed(7)
    for q in range(3):
        keep = g.view(f[q]).clone()
        f[q].fill_(bad)                          # row padding, z halos, outer halo
        g.view(f[q])[1:-1, 1:-1, 1:-1] = keep[1:-1, 1:-1, 1:-1]
        v = g.view(f[q])
        v[1:-1, 1, 1] = v[1:-1, -2, -2] = bad    # two corners of the one-cell halo
        for _ in range(40):
            k, j, i = (int(torch.randint(1, n + 1, (1,), generator=gen)) for n in (g.nz, g.ny, g.nx))
            v[k, j + 1, i + 1] = bad
        v[1, 5, 9:40] = bad
        v[g.nz, 7, 50:90] = bad
    for q in range(3, 6):                        # half of the sensitivities are 0
        v = g.view(f[q])
        m = torch.rand(v.shape, generator=torch.Generator(device="cuda").manual_seed(8 + q), device="cuda") < 0.5
        v[m] = 0.0
    march, generic = _both(g, f, flags, base if flags == pwlib.PW_ADJ_ACCUMULATE else None)
    cut = (slice(1, -1),) * 3                    # the one-cell halo of a halo of 2
    _close([x[cut] for x in march], [y[cut] for y in generic])


def test_open_mode_routes():
    """A fixed shape, pw_set_kernel(1) and a misaligned output keep the gather kernel."""
    g = pwlib.Grid(61, 20, 9)
    f = _fields(g, 9)
    h = pwlib.PW(g, inputs.make_coeffs(9))
    out = [g.alloc() for _ in range(3)]
    h.set_adjoint_config(2, 4, 4)
    h.adjoint(*f, *out)
    assert h.last_kernel == 1
    h.set_adjoint_config()
    h.adjoint(*f, *out)
    assert h.last_kernel == 2
    ref = [t.clone() for t in out]
    odd = [torch.zeros(g.alloc_elems + 1, device="cuda")[1:] for _ in range(3)]
    h.adjoint(*f, *odd)
    h.sync()
    assert h.last_kernel == 1
    for a, b in zip(odd, ref):
        assert torch.allclose(g.view(a), g.view(b), rtol=0, atol=3e-6 * float(b.abs().max()))
