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


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("which", ["cell", "off", "off_new"])
@pytest.mark.parametrize("nsteps", [1, 6])
def test_particle_pairs_must_be_aligned(prec, which, nsteps):
    """2D arrays that start in the middle of a particle's pair are refused on the host, as hyb_push refuses them,
    and nothing is touched."""
    need_gpu()
    hyb = hyb_module()
    dt = torch.float64 if prec == 64 else torch.float32
    n = 100
    g = hyb.Grid(hyb.make_desc(dims=2, n1=32, n2=16, dx1=0.2, dx2=0.2, dt=0.08, precision=prec, filt_kc=0.0, filt_w=0.0))
    F = [[torch.zeros((16, 32), device="cuda", dtype=dt) for _ in range(3)] for _ in range(3)]
    g.bind(*F)
    pic = hyb.Pic(g)

    def pairs(name, fill, t):
        flat = torch.full((2 * n + 1,), fill, device="cuda", dtype=t)
        return (flat[1:] if name == which else flat[:-1]).view(n, 2)
    cell, off, new = pairs("cell", 3, torch.int32), pairs("off", 0.25, dt), pairs("off_new", 9.0, dt)
    u = torch.ones((n, 3), device="cuda", dtype=dt)
    one, v3 = torch.ones(n, device="cuda", dtype=dt), torch.empty(n, device="cuda", dtype=dt)
    with pytest.raises(hyb.HybError) as e:
        pic.step(cell, off, u, one, one, new, v3, order=2, nsteps=nsteps)
    assert e.value.status == hyb.HYB_EALIGN
    torch.cuda.synchronize()
    assert bool((cell == 3).all() and (off == 0.25).all() and (new == 9.0).all() and (u == 1).all())
    assert all(bool((t == 0).all()) for f in F for t in f)
    pic.close()
    g.close()
