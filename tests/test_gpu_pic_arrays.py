"""The arrays a PIC step works on: what the captured step of a longer call holds after a rebind, and what the call
asks of its arguments."""
import numpy as np
import pytest

from paper_1502_01376_gb300 import workloads as wl

from gpu_util import hyb_module, need_gpu, rel_err, torch

pytestmark = pytest.mark.gpu


def _run(hyb, path, swap, fresh):
    """Two calls of six steps (the last five of each replayed), the arrays `swap` rebound to copies in between; the
    arrays bound first stay allocated and are filled with a marker.  fresh: another Pic for the second call."""
    w = wl.Workload("pic_arrays", 2, 512, 16, dx1=0.2, dx2=0.2, dt=0.08, precision=32, filt_kc=0.5, filt_w=0.2,
                    shape_order=2, seed=31, kind="plasma", ppc=2, gamma=1.5, u_th=0.5, field_amp=0.05)
    E, B = [[torch.from_numpy(a).to("cuda", torch.float32) for a in f] for f in wl.band_limited_fields(w)]
    F = {"E": E, "B": B, "J": [torch.zeros(w.shape, device="cuda") for _ in range(3)]}
    g = hyb.Grid(hyb.desc_from_workload(w, path=path))
    g.bind(F["E"], F["B"], F["J"])
    cell, off, u, qm, q = wl.pic_plasma_torch(w, "cuda")
    new, v3 = torch.empty_like(off), torch.empty_like(qm)
    pic = hyb.Pic(g)
    pic.step(cell, off, u, qm, q, new, v3, order=2, nsteps=6)
    torch.cuda.synchronize()
    old = []
    for name, c in swap:
        old.append(F[name][c])
        F[name][c] = F[name][c].clone()
        old[-1].fill_(3.0)
    g.bind(F["E"], F["B"], F["J"])
    if fresh:
        pic.close()
        pic = hyb.Pic(g)
    pic.step(cell, off, u, qm, q, new, v3, order=2, nsteps=6)
    g.check()
    out = [t.cpu().numpy() for t in F["E"] + F["B"] + F["J"] + [off, u]], [bool((t == 3.0).all()) for t in old]
    pic.close()
    g.close()
    return out


@pytest.mark.parametrize("path", [1, 2])
@pytest.mark.parametrize("swap", [[("B", 1)], [("B", 2)], [("J", 1)], [("J", 2)], [("B", 1), ("J", 2)]])
def test_replayed_step_follows_a_rebind(path, swap):
    """A Pic whose grid is rebound with some of its arrays replaced goes on in the new arrays, as a new Pic does, and
    leaves the old ones alone."""
    need_gpu()
    hyb = hyb_module()
    a, untouched = _run(hyb, path, swap, False)
    assert all(untouched)
    b, _ = _run(hyb, path, swap, True)
    for x, y in zip(a, b):
        assert rel_err(x, y) < 1e-4                          # FP32, atomic sums in another order, twelve steps
