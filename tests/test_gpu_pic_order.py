"""PIC steps of enough particles to be listed cell by cell: particles in cell order, shuffled, and shuffled with
some the push rejects, on one step against the oracle's composition (as in test_gpu_pic.py), and the
calls that change how many particles there are."""
import numpy as np
import pytest

from paper_1502_01376_gb300 import workloads as wl

from gpu_util import hyb_module, need_gpu, rel_err, torch
from test_gpu_pic import _oracle_pic

pytestmark = pytest.mark.gpu


def _setup(hyb, prec, resident, n1=64, n2=45, ppc=12):
    w = wl.Workload("pic_order", 2, n1, n2, dx1=0.2, dx2=0.2, dt=0.08, precision=prec, filt_kc=0.5, filt_w=0.2,
                    shape_order=2, seed=31, kind="plasma", ppc=ppc, gamma=1.5, u_th=0.5, field_amp=0.05)
    tdt, real = (torch.float64, np.float64) if prec == 64 else (torch.float32, np.float32)
    F = [[a.astype(real).astype(np.float64) for a in f] for f in wl.band_limited_fields(w)]
    g = hyb.Grid(hyb.desc_from_workload(w))
    E, B = [[torch.from_numpy(a).to("cuda", tdt) for a in f] for f in F]
    g.bind(E, B, [torch.zeros(w.shape, dtype=tdt, device="cuda") for _ in range(3)])
    if resident:
        g.set_resident(True)
    return w, g, F, E, B


@pytest.mark.parametrize("prec,resident,shuffle,bad", [(64, False, True, 0), (64, True, True, 0), (64, False, False, 0),
                                                       (32, False, True, 0), (32, True, False, 0), (32, False, True, 7)])
def test_listed_particles_match_oracle(prec, resident, shuffle, bad, orc):
    need_gpu()
    hyb = hyb_module()
    w, g, F, E, B = _setup(hyb, prec, resident)
    p = wl.pic_plasma_torch(w, "cuda")
    assert p[4].numel() >= 65536
    if shuffle:
        order = torch.randperm(p[4].numel(), generator=torch.Generator().manual_seed(3)).cuda()
        p = [t[order].contiguous() for t in p]
    cell, off, u, qm, q = p
    if bad:
        cell[::bad, 1] = w.n2                              # out of range: left alone and flagged
        before = [t[::bad].clone() for t in (cell, off, u)]
    ins = [t.cpu().numpy() for t in p]
    pic = hyb.Pic(g)
    pic.step(cell, off, u, qm, q, torch.empty_like(off), torch.empty_like(qm), order=2, nsteps=1)
    keep = np.ones(len(ins[4]), bool)
    if bad:
        with pytest.raises(hyb.HybError):
            g.check()
        for t, b in zip((cell, off, u), before):
            assert torch.equal(t[::bad], b)
        keep[::bad] = False
    else:
        g.check()
    go = orc.grid(n1=w.n1, n2=w.n2, dx1=w.dx1, dx2=w.dx2, dt=w.dt, filt_kc=w.filt_kc, filt_w=w.filt_w)
    a = [np.ascontiguousarray(x[keep]) for x in ins]
    Eo, Bo, co, oo, uo = _oracle_pic(orc, go, F[0], F[1], a[0], a[1], *[x.astype(np.float64) for x in a[2:]], 2, w.dt,
                                     np.array([w.dx1, w.dx2]), 1)
    tol = 1e-12 if prec == 64 else 1e-5
    for x, y in zip(E + B, Eo + Bo):
        assert rel_err(x.cpu().numpy(), y) < tol
    assert np.array_equal(cell.cpu().numpy()[keep], co)
    assert np.max(np.abs(off.cpu().numpy().astype(np.float64)[keep] - oo)) < tol
    assert np.max(np.abs(u.cpu().numpy().astype(np.float64)[keep] - uo)) < tol * np.max(np.abs(uo))
    pic.close()
    g.close()


def test_particle_sets_of_several_sizes():
    """One Pic with sets that grow and shrink (the list is kept and outgrown), in one step and in several (the
    captured step): as separate Pics give."""
    need_gpu()
    hyb = hyb_module()
    sizes = [70000, 66000, 69120, 140000, 1000]
    out = []
    for shared in (True, False):
        w, g, F, E, B = _setup(hyb, 64, False)
        pic = hyb.Pic(g)
        gen = torch.Generator(device="cuda").manual_seed(9)
        for n in sizes:
            cell = torch.stack([torch.randint(0, k, (n,), generator=gen, device="cuda", dtype=torch.int32) for k in (64, 45)], 1).contiguous()
            off = torch.rand(n, 2, generator=gen, device="cuda", dtype=torch.float64)
            u = torch.randn(n, 3, generator=gen, device="cuda", dtype=torch.float64)
            qm = torch.ones(n, device="cuda", dtype=torch.float64)
            if not shared:
                pic.close()
                pic = hyb.Pic(g)
            pic.step(cell, off, u, qm, qm * 1e-4, torch.empty_like(off), torch.empty_like(qm), order=2, nsteps=1 if n != 66000 else 6)
            g.check()
            out.append([t.cpu().numpy() for t in (cell, off, u, E[0], E[1], B[2])])
        pic.close()
        g.close()
    for a, b in zip(out[:len(sizes)], out[len(sizes):]):
        assert np.array_equal(a[0], b[0])
        for x, y in zip(a[1:], b[1:]):
            assert rel_err(x, y) < 1e-9                     # atomic sums in another order, over up to ten steps


@pytest.mark.parametrize("n1,n2,n", [(64, 45, 66000), (64, 45, 64 * 45 * 32), (64, 45, 64 * 45 * 32 + 1), (1024, 1024, 70000), (2048, 1024, 70000)])
def test_list_beside_the_scratch_and_beyond(n1, n2, n):
    """Sets that fit the list made with the Pic, fill it, and outgrow it, and a grid without one: the order in which
    shuffled particles are stored makes no difference."""
    need_gpu()
    hyb = hyb_module()
    out = []
    for shuffle in (False, True):
        w, g, F, E, B = _setup(hyb, 64, False, n1=n1, n2=n2, ppc=1)
        gen = torch.Generator(device="cuda").manual_seed(4)
        cell = torch.stack([torch.randint(0, k, (n,), generator=gen, device="cuda", dtype=torch.int32) for k in (n1, n2)], 1).contiguous()
        off = torch.rand(n, 2, generator=gen, device="cuda", dtype=torch.float64)
        u = torch.randn(n, 3, generator=gen, device="cuda", dtype=torch.float64)
        if not shuffle:
            key = torch.argsort(cell[:, 1].long() * n1 + cell[:, 0], stable=True)
            cell, off, u = [t[key].contiguous() for t in (cell, off, u)]
        qm = torch.ones(n, device="cuda", dtype=torch.float64)
        pic = hyb.Pic(g)
        pic.step(cell, off, u, qm, qm * 1e-4, torch.empty_like(off), torch.empty_like(qm), order=2, nsteps=1)
        g.check()
        out.append([t.cpu().numpy() for t in E + B])
        pic.close()
        g.close()
    for x, y in zip(*out):
        assert rel_err(x, y) < 1e-9                         # atomic sums in another order


@pytest.mark.parametrize("prec,order,ppc", [(64, 2, 23), (32, 2, 23), (64, 3, 18), (32, 3, 18), (32, 1, 46)])
def test_listed_particles_from_the_rule_on(prec, order, ppc, orc):
    """Shuffled particles, just enough of them to be listed at each shape order, on one step against the oracle's composition."""
    need_gpu()
    hyb = hyb_module()
    w, g, F, E, B = _setup(hyb, prec, False, ppc=ppc)
    p = wl.pic_plasma_torch(w, "cuda")
    assert p[4].numel() >= {1: 1 << 18, 2: 1 << 17, 3: 3 << 15}[order]
    mix = torch.randperm(p[4].numel(), generator=torch.Generator().manual_seed(3)).cuda()
    cell, off, u, qm, q = p = [t[mix].contiguous() for t in p]
    a = [t.cpu().numpy() for t in p]
    pic = hyb.Pic(g)
    pic.step(cell, off, u, qm, q, torch.empty_like(off), torch.empty_like(qm), order=order, nsteps=1)
    g.check()
    go = orc.grid(n1=w.n1, n2=w.n2, dx1=w.dx1, dx2=w.dx2, dt=w.dt, filt_kc=w.filt_kc, filt_w=w.filt_w)
    Eo, Bo, co, oo, uo = _oracle_pic(orc, go, F[0], F[1], a[0], a[1].astype(np.float64), *[x.astype(np.float64) for x in a[2:]], order, w.dt,
                                     np.array([w.dx1, w.dx2]), 1)
    tol = 1e-12 if prec == 64 else 1e-5
    for x, y in zip(E + B, Eo + Bo):
        assert rel_err(x.cpu().numpy(), y) < tol
    assert np.array_equal(cell.cpu().numpy(), co)
    pic.close()
    g.close()
