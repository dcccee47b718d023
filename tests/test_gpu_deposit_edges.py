"""FP32 2D deposits at the edges of the run kernel's conditions."""
import numpy as np
import pytest

from gpu_util import hyb_module, need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("ordered", [True, False])
@pytest.mark.parametrize("q_bad", [float("inf"), 3e38])
def test_no_v3_leaves_j3_at_zero_whatever_the_charge(order, ordered, q_bad):
    """Without v3 there is no out-of-plane current, whether particles share cells (runs) or are scattered: j3 stays
    0 and j1, j2 of the particles away from the infinite (or overflowing) charge stay finite."""
    need_gpu()
    hyb = hyb_module()
    n1, n2, ppc = 64, 64, 16
    g = hyb.Grid(hyb.make_desc(dims=2, n1=n1, n2=n2, dx1=0.2, dx2=0.2, dt=0.08, precision=32, filt_kc=0.0, filt_w=0.0))
    z = [[torch.full((n2, n1), 7.0, device="cuda") for _ in range(3)] for _ in range(3)]
    g.bind(*z)
    i = torch.arange(n1 * n2, dtype=torch.int32)
    cell = torch.stack([i % n1, i // n1], 1).repeat_interleave(ppc, 0)
    gen = torch.Generator().manual_seed(5)
    off = torch.rand(cell.shape, generator=gen)
    new = off + 0.3 * (torch.rand(cell.shape, generator=gen) - 0.5)
    q = torch.ones(len(cell))
    q[ppc * (n1 * 32 + 32)] = q_bad                       # a particle of cell (32, 32)
    if not ordered:
        mix = torch.randperm(len(cell), generator=gen)
        cell, off, new, q = cell[mix], off[mix], new[mix], q[mix]
    cell, off, new, q = [t.contiguous().cuda() for t in (cell, off, new, q)]
    g.deposit(cell, off, new, None, q, order)
    g.check()
    J1, J2, J3 = [t.cpu().numpy() for t in z[2]]
    assert np.all(J3 == 0.0)
    far = np.ones((n2, n1), bool)
    far[28:37, 28:37] = False                             # the cell's window
    assert np.isfinite(J1[far]).all() and np.isfinite(J2[far]).all() and np.abs(J1[far]).max() > 0
    g.close()
