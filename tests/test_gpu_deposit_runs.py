"""The FP32 2D deposit's ways of adding particles (runs of a cell in registers, rows of 32 consecutive cells
summed across the lanes, particles on their own) against the oracle: uneven runs, runs longer than
a warp's cut, rows that wrap, short runs, steps back by more than half a cell, skipped particles."""
import numpy as np
import pytest

from gpu_util import hyb_module, need_gpu, rel_err, to_np, torch

pytestmark = pytest.mark.gpu


def _case(kind, n1, n2, rng):
    cells = n1 * n2
    if kind == "even":                       # 8 in every cell: 32 consecutive cells a warp
        k = np.repeat(np.arange(cells), 8)
    elif kind == "one":                      # one in every cell
        k = np.arange(cells)
    elif kind == "poisson":
        k = np.repeat(np.arange(cells), rng.poisson(5.0, cells))
    elif kind == "heap":                     # hundreds in a few cells, at the corners
        k = np.repeat([0, n1 - 1, cells - n1, cells - 1], [700, 33, 1, 259])
    else:                                    # no order
        k = rng.integers(0, cells, 5000)
    return np.stack([k % n1, k // n1], axis=1).astype(np.int32)


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("kind", ["even", "one", "poisson", "heap", "random"])
@pytest.mark.parametrize("n1,n2", [(8, 3), (64, 37), (32, 5)])
def test_runs_match_oracle(n1, n2, kind, order):
    need_gpu()
    hyb = hyb_module()
    import oracle as orc
    orc.build()
    rng = np.random.default_rng(n1 + 10 * n2 + order)
    cell = _case(kind, n1, n2, rng)
    n = len(cell)
    f = np.float32
    off0 = rng.uniform(0, 1, (n, 2)).astype(f)
    off0[off0 >= 1] = 0
    off1 = (off0 + rng.uniform(-0.95, 0.95, (n, 2))).astype(f)
    v3, q = rng.uniform(-1, 1, n).astype(f), rng.uniform(-1, 1, n).astype(f)
    g = hyb.Grid(hyb.make_desc(n1=n1, n2=n2, dx1=0.2, dx2=0.25, dt=0.08, precision=32))
    z = [[torch.zeros(n2, n1, device="cuda") for _ in range(3)] for _ in range(3)]
    g.bind(*z)
    dev = [torch.from_numpy(a).cuda() for a in (cell, off0, off1, v3, q)]
    g.deposit(*dev, order)
    g.check()
    go = orc.grid(n1=n1, n2=n2, dx1=0.2, dx2=0.25, dt=0.08)
    d = [a.astype(np.float64) for a in (off0, off1, v3, q)]
    Jo = orc.deposit(go, cell, *d, order)
    for a, b in zip(z[2], Jo):
        assert rel_err(to_np(a), b) < 1e-5
    # every tenth particle broken: skipped and flagged, the others as before
    bad = np.arange(0, n, 10)
    off0[bad[::2]] = np.nan
    cell[bad[1::2], 0] = n1
    g.deposit(torch.from_numpy(cell).cuda(), torch.from_numpy(off0).cuda(), *dev[2:], order)
    with pytest.raises(hyb.HybError):
        g.check()
    ok = np.setdiff1d(np.arange(n), bad)
    Jo = orc.deposit(go, np.ascontiguousarray(cell[ok]), *[np.ascontiguousarray(a[ok]) for a in d], order)
    for a, b in zip(z[2], Jo):
        assert rel_err(to_np(a), b) < 1e-5
    g.close()
