"""pw_keep_interior: interiors copied bit for bit, zeros in every other element."""
import pytest
import torch

import paper_2301_13016_gb300 as pwlib
from paper_2301_13016_gb300 import inputs
from gpu_util import NAN

pytestmark = pytest.mark.gpu


def _grids():
    return [pwlib.Grid(5, 3, 3), pwlib.Grid(130, 7, 5), pwlib.Grid(33, 9, 4, halo=3), pwlib.Grid(64, 6, 5, dtype="bf16"),
            pwlib.Grid(17, 5, 4, pitch_j=23, pitch_k=23 * 7 + 11, origin=2)]   # rows of odd length, a gap between levels


@pytest.mark.parametrize("n", range(5))
@pytest.mark.parametrize("in_place", [False, True])
def test_keep_interior(n, in_place):
    g = _grids()[n]
    h = pwlib.PW(g, inputs.make_coeffs(g.nz))
    src = [torch.randn(g.alloc_elems, device="cuda").to(g.torch_dtype) for _ in range(3)]
    want = []
    for q, s in enumerate(src):
        w = torch.zeros_like(s)
        if q != 1 or in_place:
            cut = (slice(1, -1), slice(g.halo, g.halo + g.ny), slice(g.halo, g.halo + g.nx))
            g.view(w)[cut] = g.view(s)[cut]
        want.append(w)
    dst = src if in_place else [g.alloc(fill=NAN) for _ in range(3)]
    h.keep_interior(src if in_place else [src[0], None, src[2]], dst)
    h.sync()
    for a, b in zip(dst, want):
        assert torch.equal(a, b)


def test_keep_interior_misaligned_buffers():
    g = pwlib.Grid(30, 6, 4)
    h = pwlib.PW(g, inputs.make_coeffs(4))
    src = [torch.randn(g.alloc_elems + 1, device="cuda")[1:] for _ in range(3)]
    dst = [g.alloc(fill=NAN) for _ in range(3)]
    h.keep_interior(src, dst)
    h.sync()
    for s, d in zip(src, dst):
        want = torch.zeros_like(d)
        g.view(want)[1:-1, 1:-1, 1:-1] = g.view(s)[1:-1, 1:-1, 1:-1]
        assert torch.equal(d, want)


def test_keep_interior_refusals():
    g = pwlib.Grid(8, 4, 3)
    h = pwlib.PW(g, inputs.make_coeffs(3))
    t = [g.alloc() for _ in range(4)]
    for src, dst in ((t[:3], [t[0], t[0], t[2]]), ([t[1], t[0], t[2]], t[:3])):
        with pytest.raises(pwlib.PwError) as e:
            h.keep_interior(src, dst)
        assert e.value.status == pwlib.PW_ERR_ARG
