"""Tuning a grid whose width is no multiple of 4 keeps it on the k-march, which
such widths take with the automatic shape only."""
import json

import pytest

import paper_2301_13016_gb300 as pwlib
from paper_2301_13016_gb300 import autotune, inputs

pytestmark = pytest.mark.gpu
FIXED = dict(lanes_x=32, ty=4, stages=4, nseg=0, cells=4, rows=1)


@pytest.mark.parametrize("shape,kernel", [((65, 130, 64), 2), ((65, 20, 16), 1)], ids=["k-march", "generic"])
def test_tuned_ragged_grid_keeps_its_kernel(tmp_path, shape, kernel):
    g = pwlib.Grid(*shape)
    f = [g.alloc() for _ in range(6)]
    path = str(tmp_path / "tune.json")
    h = pwlib.PW(g, inputs.make_coeffs(g.nz))
    cfg, times = autotune.tune_grid(h, f, cache_path=path, reps=2)
    assert cfg in autotune.GRID_CANDIDATES and times
    h.tendencies(*f)
    assert h.last_kernel == kernel
    if kernel == 2:                                  # candidates without one that keeps the k-march
        assert autotune.tune_grid(h, f, candidates=[FIXED], cache_path=str(tmp_path / "u.json"))[0] == autotune.AUTOMATIC
    h2 = pwlib.PW(g, inputs.make_coeffs(g.nz))       # the cached choice, applied as it is
    with open(path) as fh:
        data = json.load(fh)
    assert autotune.tune_grid(h2, f, cache_path=path) == (cfg, times)
    for entry in data.values():                      # a fixed shape cached earlier
        entry["config"] = FIXED
    with open(path, "w") as fh:
        json.dump(data, fh)
    autotune.tune_grid(h2, f, cache_path=path, reps=2)
    h2.tendencies(*f)
    h2.sync()
    assert h2.last_kernel == kernel
