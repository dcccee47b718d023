"""PIC steps whose particles are listed cell by cell, each with the library's word that they were (hyb_pic_listed):
against the oracle's composition, with k1-resident fields, with particles the push rejects, over sets that
grow and shrink, on lists beside the scratch and allocated, replayed and captured."""
import numpy as np
import pytest

from paper_1502_01376_gb300 import workloads as wl

from gpu_util import hyb_module, need_gpu, rel_err, torch
from test_gpu_pic import _oracle_pic

pytestmark = pytest.mark.gpu


def _setup(hyb, prec, resident, n1=64, n2=45, ppc=23):
    w = wl.Workload("pic_listed", 2, n1, n2, dx1=0.2, dx2=0.2, dt=0.08, precision=prec, filt_kc=0.5, filt_w=0.2,
                    shape_order=2, seed=31, kind="plasma", ppc=ppc, gamma=1.5, u_th=0.5, field_amp=0.05)
    tdt, real = (torch.float64, np.float64) if prec == 64 else (torch.float32, np.float32)
    F = [[a.astype(real).astype(np.float64) for a in f] for f in wl.band_limited_fields(w)]
    g = hyb.Grid(hyb.desc_from_workload(w))
    E, B = [[torch.from_numpy(a).to("cuda", tdt) for a in f] for f in F]
    g.bind(E, B, [torch.zeros(w.shape, dtype=tdt, device="cuda") for _ in range(3)])
    if resident:
        g.set_resident(True)
    return w, g, F, E, B


@pytest.mark.parametrize("resident", [False, True])
@pytest.mark.parametrize("prec,order,ppc,shuffle,bad,listed", [
    (32, 2, 23, True, 0, 1), (32, 2, 23, True, 7, 1), (32, 2, 23, False, 0, 0), (32, 2, 23, False, 7, 0), (32, 3, 18, True, 0, 1),
    (32, 1, 92, True, 7, 1), (32, 2, 22, True, 0, -1), (32, 3, 17, True, 0, -1), (32, 1, 91, True, 0, -1), (64, 2, 23, True, 7, -1)])
def test_listed_steps_match_the_oracle(prec, order, ppc, shuffle, bad, listed, resident, orc):
    """One step.  bad: every bad-th particle has a cell out of range, is left alone and flagged."""
    need_gpu()
    hyb = hyb_module()
    w, g, F, E, B = _setup(hyb, prec, resident, ppc=ppc)
    p = wl.pic_plasma_torch(w, "cuda")
    if shuffle:
        mix = torch.randperm(p[4].numel(), generator=torch.Generator().manual_seed(3)).cuda()
        p = [t[mix].contiguous() for t in p]
    cell, off, u, qm, q = p
    if bad:
        cell[::bad, 1] = w.n2
        before = [t[::bad].clone() for t in (cell, off, u)]
    ins = [t.cpu().numpy() for t in p]
    pic = hyb.Pic(g)
    pic.step(cell, off, u, qm, q, torch.empty_like(off), torch.empty_like(qm), order=order, nsteps=1)
    assert pic.listed() == listed
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
    Eo, Bo, co, oo, uo = _oracle_pic(orc, go, F[0], F[1], a[0], *[x.astype(np.float64) for x in a[1:]], order, w.dt,
                                     np.array([w.dx1, w.dx2]), 1)
    tol = 1e-12 if prec == 64 else 1e-5
    for x, y in zip(E + B, Eo + Bo):
        assert rel_err(x.cpu().numpy(), y) < tol
    assert np.array_equal(cell.cpu().numpy()[keep], co)
    assert np.max(np.abs(off.cpu().numpy().astype(np.float64)[keep] - oo)) < tol
    assert np.max(np.abs(u.cpu().numpy().astype(np.float64)[keep] - uo)) < tol * np.max(np.abs(uo))
    pic.close()
    g.close()


def _random_set(n, n1, n2, gen, ordered=False):
    cell = torch.stack([torch.randint(0, k, (n,), generator=gen, device="cuda", dtype=torch.int32) for k in (n1, n2)], 1)
    off, u = torch.rand(n, 2, generator=gen, device="cuda") * 0.999, torch.randn(n, 3, generator=gen, device="cuda")
    if ordered:
        key = torch.argsort(cell[:, 1].long() * n1 + cell[:, 0], stable=True)
        cell, off, u = cell[key], off[key], u[key]
    qm = torch.ones(n, device="cuda")
    return cell.contiguous(), off.contiguous(), u.contiguous(), qm, qm * 1e-4


def _same_places(a, b, n1, n2):
    """Cells and offsets of two runs, as positions on the periodic grid (a last bit may put a particle on the other side of
    an edge)."""
    d = a[0].astype(np.float64) + a[1] - b[0] - b[1]
    ext = np.array([n1, n2])
    return np.max(np.abs((d + ext / 2) % ext - ext / 2)) < 1e-4


@pytest.mark.parametrize("resident", [False, True])
def test_sets_that_grow_and_shrink(resident):
    """One Pic with sets that outgrow its list and fall below the rule, in one step and in several (the captured step, a
    second time after the list has moved): as separate Pics give."""
    need_gpu()
    hyb = hyb_module()
    n1, n2 = 64, 45
    calls = [(140000, 1), (132000, 6), (131072, 1), (300000, 1), (132000, 6), (1000, 6), (299000, 5), (131071, 1)]
    out = []
    for shared in (True, False):
        w, g, F, E, B = _setup(hyb, 32, resident)
        pic = hyb.Pic(g)
        gen = torch.Generator(device="cuda").manual_seed(9)
        for n, steps in calls:
            p = _random_set(n, n1, n2, gen)
            if not shared:
                pic.close()
                pic = hyb.Pic(g)
            pic.step(*p, torch.empty_like(p[1]), torch.empty_like(p[3]), order=2, nsteps=steps)
            assert pic.listed() == (1 if n >= 1 << 17 else -1)
            g.check()
            out.append([t.cpu().numpy() for t in (*p[:3], E[0], E[1], B[2])])
        pic.close()
        g.close()
    for a, b in zip(out[:len(calls)], out[len(calls):]):
        assert _same_places(a, b, n1, n2)
        for x, y in zip(a[2:], b[2:]):
            assert rel_err(x, y) < 1e-4                         # FP32, atomic sums in another order, over up to 27 steps


@pytest.mark.parametrize("n1,n2,n", [(64, 80, 135000), (64, 80, 64 * 80 * 32), (64, 80, 64 * 80 * 32 + 1), (1024, 1025, 140000)])
def test_lists_beside_the_scratch_and_beyond(n1, n2, n):
    """Sets that fit the list made with the Pic, fill it, and outgrow it, and a grid without one: the order in which
    particles are stored makes no difference."""
    need_gpu()
    hyb = hyb_module()
    out = []
    for ordered in (False, True):
        w, g, F, E, B = _setup(hyb, 32, False, n1=n1, n2=n2, ppc=1)
        p = _random_set(n, n1, n2, torch.Generator(device="cuda").manual_seed(4), ordered)
        pic = hyb.Pic(g)
        pic.step(*p, torch.empty_like(p[1]), torch.empty_like(p[3]), order=2, nsteps=1)
        assert pic.listed() == (0 if ordered and n > n1 * n2 else 1)      # (a tenth of a particle per cell is no order)
        g.check()
        out.append([t.cpu().numpy() for t in E + B])
        pic.close()
        g.close()
    for x, y in zip(*out):
        assert rel_err(x, y) < 1e-5                                   # atomic sums in another order


def test_a_step_captured_by_the_caller():
    """A listed step in the caller's own graph, replayed, as plain steps give."""
    need_gpu()
    hyb = hyb_module()
    out = []
    for captured in (True, False):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            w, g, F, E, B = _setup(hyb, 32, False, n1=64, n2=80)
            p = _random_set(150000, 64, 80, torch.Generator(device="cuda").manual_seed(4))
            new, v3 = torch.empty_like(p[1]), torch.empty_like(p[3])
            pic = hyb.Pic(g)
            pic.step(*p, new, v3, order=2, nsteps=1)
            s.synchronize()
            if captured:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=s):
                    pic.step(*p, new, v3, order=2, nsteps=1)
                for _ in range(3):
                    graph.replay()
            else:
                for _ in range(3):
                    pic.step(*p, new, v3, order=2, nsteps=1)
            assert pic.listed() == 1
            g.check()
            out.append([t.cpu().numpy() for t in (*p[:3], *E, *B)])
            if captured:
                del graph
            pic.close()
            g.close()
    assert _same_places(out[0], out[1], 64, 80)
    for x, y in zip(out[0][2:], out[1][2:]):
        assert rel_err(x, y) < 1e-4


@pytest.mark.parametrize("n1,n2", [(64, 56), (32, 96)])
def test_a_captured_first_step_is_listed_on_small_grids(n1, n2):
    """The list for up to 32 particles per cell comes with the Pic: a first step that the caller captures, when nothing
    can be allocated, lists order-3 sets from 98304 particles on, on grids from 3072 cells on."""
    need_gpu()
    hyb = hyb_module()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        w, g, F, E, B = _setup(hyb, 32, False, n1=n1, n2=n2, ppc=1)
        p = _random_set(98304, n1, n2, torch.Generator(device="cuda").manual_seed(4))
        new, v3 = torch.empty_like(p[1]), torch.empty_like(p[3])
        pic = hyb.Pic(g)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            pic.step(*p, new, v3, order=3, nsteps=1)
        graph.replay()
        assert pic.listed() == 1
        g.check()
        del graph
        pic.close()
        g.close()
