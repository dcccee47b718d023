"""What the performance of this framework is measured on: the calls its users make, through
the public binding, over the sizes they use.

listed() names twelve calls, draw() gives more of the same ranges, prepare() makes what a
program holds before the call (fields, particles, the grid handle), run() is the call, work()
what it cannot do without, and exact() the same result in 64-bit torch, written from the
equations and without the library.
"""
import math

import numpy as np
import torch

from paper_1502_01376_gb300 import hyb

DEV = "cuda"
GAMMA, DENSITY = 50.0, 100.0        # the drifting plasma of Table 1
FILT_KC, FILT_W = 0.5, 0.2
MLP_IN = 6


def listed():
    return [
        # the vacuum-beam check a user runs first: a beam's current and one step, FP64; latency only
        dict(name="beam_2d_128x64_f64", kind="beam", n1=128, n2=64, order=1, np=4096, bits=64),
        # the production 2D field step: the drifting-plasma grid
        dict(name="advance_2d_4096x1024_f32", kind="advance", dims=2, n1=4096, n2=1024, n3=1, bits=32, resident=False),
        # an ordinary 2D grid with a row count that fits no tile
        dict(name="advance_2d_1024x777_f32", kind="advance", dims=2, n1=1024, n2=777, n3=1, bits=32, resident=False),
        # the boosted-frame wakefield grid of the paper's Table 2: the longest rows
        dict(name="advance_2d_8192x512_f32", kind="advance", dims=2, n1=8192, n2=512, n3=1, bits=32, resident=False),
        # the 3D drifting plasma: the largest grid
        dict(name="advance_3d_1024x256x256_f32", kind="advance", dims=3, n1=1024, n2=256, n3=256, bits=32, resident=False),
        # one azimuthal mode of a quasi-3D run
        dict(name="quasi3d_2048x512_m1_f32", kind="quasi3d", n1=2048, n2=512, m=1, bits=32),
        # a parameter scan: sixteen uneven 2D grids and three azimuthal modes advanced together
        dict(name="batch_16x2d_3xq3d_f32", kind="batch", grids=16, modes=3, nz=2048, nr=512, sizes=3),
        # the particle push of the drifting plasma, 8 + 8 particles per cell in cell order
        dict(name="push_2d_67M_f32", kind="push", dims=2, n1=4096, n2=1024, n3=1, ppc=8, order=2, bits=32),
        # its charge-conserving deposit
        dict(name="deposit_2d_67M_f32", kind="deposit", dims=2, n1=4096, n2=1024, n3=1, ppc=8, order=2, u_th=1e-4, bits=32),
        # one step of the particle-in-cell loop on the Table 1 box
        dict(name="pic_2d_256x256_f32", kind="pic", n1=256, n2=256, ppc=8, order=2, u_th=1.0, bits=32, resident=False),
        # training the growth-rate surrogate: sixteen Adam steps on minibatches, then the weights are read
        dict(name="mlp_train_6x256x4_b8192", kind="mlp_train", width=256, depth=4, batch=8192, steps=16),
        # the root solver's scan of candidate settings over a (k1, k2) grid
        dict(name="nci_scan_32256", kind="nci", rows=32256, order=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["beam", "advance", "advance", "advance", "advance", "quasi3d", "batch", "push", "deposit", "pic",
                       "mlp_train", "mlp_forward", "nci"])
    if kind == "beam":
        return dict(kind=kind, n1=rng.choice([64, 128, 256]), n2=_log(rng, 16, 200), order=rng.choice([1, 2, 3]),
                    np=_log(rng, 500, 20000), bits=64)
    if kind == "advance":
        if rng.random() < 0.6:
            bits = rng.choice([32, 32, 32, 64])
            n1 = rng.choice([64, 128, 256, 512, 1024, 2048, 4096, 8192])
            n2 = _log(rng, 16, max(32, min(4000, (1 << (22 if bits == 32 else 20)) // n1)))
            return dict(kind=kind, dims=2, n1=n1, n2=n2, n3=1, bits=bits, resident=rng.random() < 0.2)
        return dict(kind=kind, dims=3, n1=rng.choice([32, 64, 128, 256, 512, 1024]), n2=_log(rng, 8, 160),
                    n3=_log(rng, 8, 160), bits=rng.choice([32, 32, 32, 64]), resident=rng.random() < 0.3)
    if kind == "quasi3d":
        return dict(kind=kind, n1=rng.choice([256, 512, 1024, 2048, 2048]), n2=_log(rng, 40, 800), m=rng.choice([0, 1, 2, 3]),
                    bits=rng.choice([32, 32, 32, 64]))
    if kind == "batch":
        return dict(kind=kind, grids=rng.randint(2, 16), modes=rng.randint(0, 3), nz=2048, nr=_log(rng, 100, 512),
                    sizes=rng.randint(10, 10000))
    if kind in ("push", "deposit"):
        c = dict(kind=kind, dims=rng.choice([2, 2, 3]), order=rng.choice([1, 2, 2, 3]), bits=rng.choice([32, 32, 32, 64]))
        c["ppc"] = rng.choice([1, 2, 4, 8, 8, 13])
        if c["dims"] == 2:
            c.update(n1=rng.choice([128, 256, 1024, 4096]), n2=_log(rng, 30, 900), n3=1)
        else:
            c.update(n1=rng.choice([32, 64, 128]), n2=_log(rng, 10, 60), n3=_log(rng, 10, 60))
        if kind == "deposit":
            c["u_th"] = math.exp(rng.uniform(math.log(1e-4), 0.0))
        return c
    if kind == "pic":
        return dict(kind=kind, n1=rng.choice([64, 128, 256, 512]), n2=_log(rng, 40, 500), ppc=rng.choice([2, 4, 8]),
                    order=rng.choice([1, 2, 3]), u_th=rng.uniform(0.5, 2.0), bits=rng.choice([32, 32, 64]),
                    resident=rng.random() < 0.5)
    if kind == "mlp_train":
        return dict(kind=kind, width=rng.choice([64, 128, 256, 256]), depth=rng.choice([2, 3, 4]), batch=_log(rng, 1000, 10000),
                    steps=16)
    if kind == "mlp_forward":
        return dict(kind=kind, width=rng.choice([64, 128, 256, 256]), depth=rng.choice([2, 3, 4]), batch=_log(rng, 500, 130000))
    return dict(kind="nci", rows=_log(rng, 500, 32000), order=rng.choice([1, 2, 2, 3]))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _real(bits):
    return torch.float32 if bits == 32 else torch.float64


def _band_limited(shape, gen, amp, dtype):
    """A real random field with no content above half of the Nyquist wavenumber, of rms amp."""
    axes = [torch.fft.fftfreq(n, device=DEV) * 2 for n in shape[:-1]] + [torch.fft.rfftfreq(shape[-1], device=DEV) * 2]
    k2 = sum(a.reshape([-1 if i == d else 1 for i in range(len(shape))]) ** 2 for d, a in enumerate(axes))
    spec = torch.randn(k2.shape, generator=gen, device=DEV) + 1j * torch.randn(k2.shape, generator=gen, device=DEV)
    spec *= k2 < 0.25
    f = torch.fft.irfftn(spec, s=shape)
    f *= amp / f.square().mean().sqrt().clamp_min(1e-30)
    return f.to(dtype).contiguous()


def _fields(shape, gen, dtype, amp=1e-3, current=None):
    E = [_band_limited(shape, gen, amp, dtype) for _ in range(3)]
    B = [_band_limited(shape, gen, amp, dtype) for _ in range(3)]
    J = [_band_limited(shape, gen, amp if current is None else current, dtype) for _ in range(3)]
    return E, B, J


def _dt(dims):
    return 0.1 if dims == 2 else 0.08


def _grid_kw(c):
    """dx, dt and options of a case's 2D or 3D grid."""
    kw = dict(dims=c.get("dims", 2), n1=c["n1"], n2=c["n2"], n3=c.get("n3", 1), dx1=0.2, dx2=0.2, dx3=0.2,
              dt=_dt(c.get("dims", 2)), precision=c["bits"], filt_kc=FILT_KC, filt_w=FILT_W)
    if c["kind"] == "beam":
        kw.update(dx1=0.1, dx2=0.1, dx3=0.1, dt=0.05, filt_kc=0.0, filt_w=0.0)
    if c["kind"] == "pic":
        kw.update(dt=0.08)
    return kw


def _shape(c):
    return (c["n3"], c["n2"], c["n1"]) if c.get("dims", 2) == 3 else (c["n2"], c["n1"])


def _plasma(c, gen, kw):
    """Both species of the drifting plasma in cell order, ppc of each per cell at independent random
    positions: cell, offset, u = gamma v, q/m, macro-particle charge."""
    d, ppc, dtype = c.get("dims", 2), c["ppc"], _real(c["bits"])
    cells = c["n1"] * c["n2"] * c.get("n3", 1)
    i = torch.arange(cells, device=DEV, dtype=torch.int32)
    ax = [i % c["n1"], (i // c["n1"]) % c["n2"], i // (c["n1"] * c["n2"])][:d]
    cell = torch.stack(ax, 1).repeat_interleave(ppc, 0).repeat(2, 1).contiguous()
    n = cell.shape[0]
    off = torch.rand((n, d), generator=gen, device=DEV, dtype=dtype)
    u = torch.randn((n, 3), generator=gen, device=DEV, dtype=dtype) * c.get("u_th", 1e-4)
    u[:, 0] += math.sqrt(GAMMA ** 2 - 1.0)
    sign = torch.cat([torch.full((n // 2,), s, device=DEV, dtype=dtype) for s in (-1.0, 1.0)])
    q = sign * (DENSITY / (4 * math.pi) * kw["dx1"] * kw["dx2"] * (kw["dx3"] if d == 3 else 1.0) / ppc)
    return cell, off, u, sign, q


def _move(off, u, kw):
    """The next offsets and the third velocity component of a ballistic step."""
    gi = torch.rsqrt(1 + u.double().square().sum(1, keepdim=True))
    v = u.double() * gi
    s = torch.tensor([kw["dt"] / kw["dx1"], kw["dt"] / kw["dx2"], kw["dt"] / kw["dx3"]][: off.shape[1]], device=DEV, dtype=torch.float64)
    return (off.double() + v[:, : off.shape[1]] * s).to(off.dtype).contiguous(), v[:, 2].to(off.dtype).contiguous()


def _beam(c, gen, kw):
    n = c["np"]
    ext = torch.tensor([c["n1"], c["n2"]], device=DEV, dtype=torch.float64)
    x = torch.rand((n, 2), generator=gen, device=DEV, dtype=torch.float64) * ext
    cell = torch.minimum(x.floor(), ext - 1)
    off = (x - cell).clamp(0, 1 - 1e-12)
    off_new = off.clone()
    off_new[:, 0] += 0.99 * kw["dt"] / kw["dx1"]
    return (cell.to(torch.int32).contiguous(), off, off_new, torch.zeros(n, device=DEV, dtype=torch.float64),
            torch.full((n,), -0.01, device=DEV, dtype=torch.float64))


def _batch_grids(c):
    """(make_desc arguments) of a batch's grids: 2D rows and heights of the scan, then the modes."""
    r = np.random.default_rng(c["sizes"])
    out = [dict(dims=2, n1=int(r.choice([512, 1024, 2048, 4096])), n2=int(r.choice([128, 256, 512, 1024])), dx1=0.2, dx2=0.2,
                dt=0.08, precision=32, filt_kc=FILT_KC, filt_w=FILT_W) for _ in range(c["grids"])]
    return out + [_q3d_kw(dict(n1=c["nz"], n2=c["nr"], m=m, bits=32)) for m in range(c["modes"])]


def _q3d_kw(c):
    m = c["m"]
    dt = min(0.08, 0.9 * 2 / math.sqrt(math.pi ** 2 / 0.2 ** 2 + (4 * m * m + 6) / 0.2 ** 2))
    return dict(dims=20, n1=c["n1"], n2=c["n2"], dx1=0.2, dx2=0.2, dt=dt, precision=c["bits"], filt_kc=FILT_KC,
                filt_w=FILT_W, azimuthal_m=m)


def _q3d_fields(c, gen):
    """Complex mode amplitudes E, B, J, each smooth in z (band-limited) and random in r."""
    t = torch.complex64 if c["bits"] == 32 else torch.complex128
    def one():
        k = torch.fft.fftfreq(c["n1"], device=DEV).abs() * 2
        s = torch.randn((c["n2"], c["n1"]), generator=gen, device=DEV) + 1j * torch.randn((c["n2"], c["n1"]), generator=gen, device=DEV)
        f = torch.fft.ifft(s * (k < 0.5), dim=1)
        return (f * (1e-3 / f.abs().square().mean().sqrt())).to(t).contiguous()
    return [[one() for _ in range(3)] for _ in range(3)]


def _batch_fields(c, gen):
    """Per grid one [9, n2, n1] array: E, B, J."""
    out = []
    for kw in _batch_grids(c):
        if kw["dims"] == 2:
            out.append(torch.stack(sum(_fields((kw["n2"], kw["n1"]), gen, torch.float32), [])))
        else:
            out.append(torch.stack(sum(_q3d_fields(dict(n1=kw["n1"], n2=kw["n2"], bits=32), gen), [])))
    return out


def _nci_rows(c, gen):
    """Rows of the root solver (dt, dx1, dx2, gamma, n/n_p, kc, w, k1, k2) below the Courant limit."""
    n, dx1 = c["rows"], 0.2
    u = lambda lo, hi: lo + (hi - lo) * torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)  # noqa: E731
    dx2 = dx1 * u(0.5, 2.0)
    limit = 2.0 / torch.sqrt(math.pi ** 2 / dx1 ** 2 + 4.0 / dx2 ** 2)
    dt = torch.minimum(dx1 * u(0.1, 0.9), limit * 0.999)
    one = torch.ones_like(dt)
    return torch.stack([dt, dx1 * one, dx2, u(5.0, 100.0), DENSITY * one, u(0.3, 1.0), FILT_W * one,
                        u(0.01, 1.0) * (math.pi / dx1), u(0.01, 1.0) * math.pi / dx2], 1).contiguous()


def _mlp_params(c, seed):
    r = np.random.default_rng(seed)
    dims = [MLP_IN] + [c["width"]] * c["depth"] + [1]
    parts = []
    for fi, fo in zip(dims[:-1], dims[1:]):
        lim = math.sqrt(6.0 / (fi + fo))
        parts += [r.uniform(-lim, lim, fo * fi), r.uniform(-0.05, 0.05, fo)]
    return np.concatenate(parts).astype(np.float32)


def _mlp_data(c, gen, n):
    """Features in [-1, 1] and a growth-rate-like target: zero over much of the domain, smooth bumps elsewhere."""
    x = 2 * torch.rand((n, MLP_IN), generator=gen, device=DEV) - 1
    t = torch.relu(torch.sin(3 * x[:, 4]) * torch.cos(2 * x[:, 5]) + 0.3 * x[:, 0] - 0.4 * x[:, 3] * x[:, 2])
    return x.contiguous(), t.contiguous()


def _inputs(c, seed):
    g, kind = _gen(seed), c["kind"]
    if kind == "beam":
        kw = _grid_kw(c)
        return kw, _fields(_shape(c), g, torch.float64), _beam(c, g, kw)
    if kind == "advance":
        return _grid_kw(c), _fields(_shape(c), g, _real(c["bits"]))
    if kind == "quasi3d":
        return _q3d_kw(c), _q3d_fields(c, g)
    if kind == "batch":
        return _batch_grids(c), _batch_fields(c, g)
    if kind == "push":
        kw = _grid_kw(c)
        f = _fields(_shape(c), g, _real(c["bits"]))
        cell, off, u, qm, q = _plasma(c, g, kw)
        return kw, f, (cell, _move(off, u, kw)[0], u, qm)      # offsets as the step before left them
    if kind == "deposit":
        kw = _grid_kw(c)
        cell, off, u, qm, q = _plasma(c, g, kw)
        off_new, v3 = _move(off, u, kw)
        return kw, (cell, off, off_new, v3, q)
    if kind == "pic":
        kw = _grid_kw(c)
        return kw, _fields(_shape(c), g, _real(c["bits"]), amp=0.1), _plasma(c, g, kw)
    if kind == "mlp_train":
        x, t = _mlp_data(c, g, c["batch"] * c["steps"])
        return _mlp_params(c, seed), x.view(c["steps"], c["batch"], MLP_IN), t.view(c["steps"], c["batch"])
    if kind == "mlp_forward":
        return _mlp_params(c, seed), _mlp_data(c, g, c["batch"])[0]
    return _nci_rows(c, g)


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"kind": kind, "case": c}
    got = _inputs(c, seed)
    if kind in ("beam", "advance", "quasi3d", "push", "pic"):
        kw, (E, B, J) = got[0], got[1]
    if kind == "beam":
        s.update(grid=hyb.Grid(hyb.make_desc(**kw)).bind(E, B, J), E=E, B=B, J=J, p=got[2])
    elif kind in ("advance", "quasi3d"):
        g = hyb.Grid(hyb.make_desc(**kw)).bind(E, B, J)
        if c.get("resident"):
            g.set_resident(True)
        s.update(grid=g, E=E, B=B)
    elif kind == "batch":
        kws, arrs = got
        b = hyb.Batch([hyb.make_desc(**kw) for kw in kws])
        for i, a in enumerate(arrs):
            b.bind(i, [a[0], a[1], a[2]], [a[3], a[4], a[5]], [a[6], a[7], a[8]])
        b.tune(5)
        s.update(batch=b, arrs=arrs)
    elif kind == "push":
        cell, off, u, qm = got[2]
        s.update(grid=hyb.Grid(hyb.make_desc(**kw)).bind(E, B, J), p=(cell, off, u, qm), off_new=torch.empty_like(off),
                 v3=torch.empty_like(qm) if c["dims"] == 2 else None)
    elif kind == "deposit":
        kw, p = got
        f = [[torch.zeros(_shape(c), device=DEV, dtype=_real(c["bits"])) for _ in range(3)] for _ in range(3)]
        s.update(grid=hyb.Grid(hyb.make_desc(**kw)).bind(*f), J=f[2], p=p)
    elif kind == "pic":
        cell, off, u, qm, q = got[2]
        g = hyb.Grid(hyb.make_desc(**kw)).bind(E, B, J)
        if c["resident"]:
            g.set_resident(True)
        s.update(grid=g, pic=hyb.Pic(g), E=E, B=B, J=J, p=(cell, off, u, qm, q), off_new=torch.empty_like(off),
                 v3=torch.empty_like(qm))
    elif kind in ("mlp_train", "mlp_forward"):
        s.update(mlp=hyb.MLP(MLP_IN, c["width"], c["depth"], params=got[0]), x=got[1])
        if kind == "mlp_train":
            s.update(t=got[2], loss=torch.zeros(c["steps"], device=DEV))
    else:
        s.update(rows=got)
    return s


def run(state):
    s, c = state, state["case"]
    kind = s["kind"]
    if kind == "beam":
        cell, off, off_new, v3, q = s["p"]
        s["grid"].deposit(cell, off, off_new, v3, q, c["order"])
        s["grid"].advance(1)
        return {"E": s["E"], "B": s["B"], "J": s["J"]}
    if kind in ("advance", "quasi3d"):
        s["grid"].advance(1)
        return {"E": s["E"], "B": s["B"]}
    if kind == "batch":
        s["batch"].advance(1)
        return [a[:6] for a in s["arrs"]]
    if kind == "push":
        cell, off, u, qm = s["p"]
        s["grid"].push(cell, off, u, qm, s["off_new"], s["v3"], order=c["order"])
        return {"cell": cell, "off": off, "u": u, "off_new": s["off_new"], "v3": s["v3"]}
    if kind == "deposit":
        cell, off, off_new, v3, q = s["p"]
        s["grid"].deposit(cell, off, off_new, v3 if c["dims"] == 2 else None, q, c["order"])
        return {"J": s["J"]}
    if kind == "pic":
        cell, off, u, qm, q = s["p"]
        s["pic"].step(cell, off, u, qm, q, s["off_new"], s["v3"], order=c["order"], nsteps=1)
        return {"E": s["E"], "B": s["B"], "J": s["J"], "cell": cell, "off": off, "u": u, "v3": s["v3"]}
    if kind == "mlp_train":
        for k in range(c["steps"]):
            s["mlp"].train_step(s["x"][k], s["t"][k], 1e-3, s["loss"][k:k + 1])
        return {"params": s["mlp"].get_params(), "loss": s["loss"]}
    if kind == "mlp_forward":
        return {"y": s["mlp"].forward(s["x"])}
    return {"growth": hyb.nci_growth(s["rows"], order=c["order"])}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    c, kind = case, case["kind"]
    w = c.get("bits", 32) // 8
    step = lambda n1, cells: cells * (15 * 2.5 * math.log2(n1) + 36)  # noqa: E731  15 real row transforms, the updates
    if kind == "nci":
        # counting the zeros of a disk and Newton to them: some hundred evaluations of the relation
        return {"bytes": c["rows"] * (12 + 3) * 8.0, "flops": c["rows"] * 3 * 3.0e4}
    if kind in ("mlp_train", "mlp_forward"):
        dims = [MLP_IN] + [c["width"]] * c["depth"] + [1]
        p = sum((a + 1) * b for a, b in zip(dims[:-1], dims[1:]))
        if kind == "mlp_forward":
            return {"bytes": c["batch"] * 4.0 * (MLP_IN + 1) + 4.0 * p, "flops": 2.0 * p * c["batch"]}
        return {"bytes": c["steps"] * (c["batch"] * 4.0 * (MLP_IN + 1) + 24.0 * p), "flops": 6.0 * p * c["batch"] * c["steps"]}
    if kind == "batch":
        b = f = 0.0
        for kw in _batch_grids(c):
            cells, q = kw["n1"] * kw["n2"], 2 if kw["dims"] == 20 else 1
            b += 60.0 * q * cells
            f += q * step(kw["n1"], cells)
        return {"bytes": b, "flops": f}
    cells = c["n1"] * c["n2"] * c.get("n3", 1)
    if kind == "quasi3d":
        return {"bytes": 30.0 * w * cells, "flops": 2 * step(c["n1"], cells)}
    if kind == "advance":
        return {"bytes": 15.0 * w * cells, "flops": step(c["n1"], cells)}
    d = c.get("dims", 2)
    n = c["np"] if kind == "beam" else 2 * c["ppc"] * cells
    pts = (c["order"] + 1) ** d
    dep_b = n * (4.0 * d + w * (2 * d + (2 if d == 2 else 1))) + 3.0 * w * cells
    dep_f = n * 3.0 * 4 * (c["order"] + 2) ** d
    push_b = n * (8.0 * d + w * (3 * d + 7 + (1 if d == 2 else 0))) + 6.0 * w * cells
    push_f = n * (12.0 * pts + 150)
    if kind == "push":
        return {"bytes": push_b, "flops": push_f}
    if kind == "deposit":
        return {"bytes": dep_b, "flops": dep_f}
    if kind == "beam":
        return {"bytes": dep_b + 12.0 * w * cells, "flops": dep_f + step(c["n1"], cells)}
    # one particle-in-cell step: each particle and each field value read and written once
    return {"bytes": n * (16.0 + w * (2 * 2 + 2 * 3 + 2 + 1)) + 15.0 * w * cells,
            "flops": dep_f + push_f + step(c["n1"], cells)}


# ------------------------------------------------------------------ the same results in 64 bits
def _tables(kw, k):
    """sigma+, sigma-, the j1 correction and the current filter at the wavenumbers k (float64)."""
    ph = 0.5 * k * kw["dx1"]
    sp, sm = 1j * k * torch.exp(1j * ph), 1j * k * torch.exp(-1j * ph)
    corr = torch.where(k == 0, torch.ones_like(k), torch.sin(ph) / torch.where(k == 0, torch.ones_like(k), ph))
    F = torch.ones_like(k)
    if 0 < kw["filt_kc"] < 1:
        kn, a = math.pi / kw["dx1"], k.abs()
        lo, hi = (kw["filt_kc"] - 0.5 * kw["filt_w"]) * kn, (kw["filt_kc"] + 0.5 * kw["filt_w"]) * kn
        F = torch.where(a <= lo, F, torch.where(a >= hi, torch.zeros_like(k), torch.cos(0.5 * math.pi * (a - lo) / (hi - lo)) ** 2))
    return sp, sm, corr, F


def _x_step(kw, E, B, J=None, faraday_only=False):
    """One hybrid step in 64 bits: E^{n+1}, B^{n+1/2} (or B^{n+1/2} alone)."""
    n1, dt, d3 = kw["n1"], kw["dt"], kw["dims"] == 3
    k = 2 * math.pi * torch.arange(n1 // 2 + 1, device=DEV, dtype=torch.float64) / (n1 * kw["dx1"])
    sp, sm, corr, F = _tables(kw, k)
    E = [torch.fft.rfft(f.double()) for f in E]
    B = [torch.fft.rfft(f.double()) for f in B]
    up = lambda f, ax, dx: (torch.roll(f, -1, ax) - f) * (dt / dx)  # noqa: E731
    dn = lambda f, ax, dx: (f - torch.roll(f, 1, ax)) * (dt / dx)  # noqa: E731
    B[0] -= up(E[2], -2, kw["dx2"])
    B[1] += dt * sp * E[2]
    B[2] -= dt * sp * E[1] - up(E[0], -2, kw["dx2"])
    if d3:
        B[0] += up(E[1], 0, kw["dx3"])
        B[1] -= up(E[0], 0, kw["dx3"])
    inv = lambda f: torch.fft.irfft(f, n=n1)  # noqa: E731
    if faraday_only:
        return [inv(f) for f in B]
    a = 4 * math.pi * dt
    E[0] += dn(B[2], -2, kw["dx2"]) - (a * F * corr) * torch.fft.rfft(J[0].double())
    E[1] -= dt * sm * B[2] + (a * F) * torch.fft.rfft(J[1].double())
    E[2] += dt * sm * B[1] - dn(B[0], -2, kw["dx2"]) - (a * F) * torch.fft.rfft(J[2].double())
    if d3:
        E[0] -= dn(B[1], 0, kw["dx3"])
        E[1] += dn(B[0], 0, kw["dx3"])
    return [inv(f) for f in E], [inv(f) for f in B]


def _x_q3d(kw, E, B, J):
    nz, nr, dt, dr, m = kw["n1"], kw["n2"], kw["dt"], kw["dx2"], kw["azimuthal_m"]
    kap = torch.fft.fftfreq(nz, 1.0 / nz, device=DEV, dtype=torch.float64)
    kap[nz // 2] = nz // 2
    sp, sm, corr, F = _tables(kw, 2 * math.pi * kap / (nz * kw["dx1"]))
    Ez, Er, Ep, Bz, Br, Bp, Jz, Jr, Jp = (torch.fft.fft(f.to(torch.complex128), dim=1) for f in E + B + J)
    j = torch.arange(nr, device=DEV, dtype=torch.float64)[:, None]
    r, rh = j * dr, (j + 0.5) * dr
    rs = torch.where(r > 0, r, torch.ones_like(r))
    zero = torch.zeros((1, nz), device=DEV, dtype=torch.complex128)
    above = lambda f: torch.cat([f[1:], zero])  # noqa: E731  0 at the wall
    below = lambda f: torch.cat([zero, f[:-1]])  # noqa: E731
    cr = torch.where(r > 0, 1j * m / rs, torch.zeros_like(rs) * 1j) * Ez - sp * Ep
    if m == 1:
        cr[0] = 1j * m * Ez[1] / dr - sp * Ep[0]
    Bz = Bz - dt * (((r + dr) * above(Ep) - r * Ep) / (rh * dr) - 1j * m / rh * Er)
    Bp = Bp - dt * (sp * Er - (above(Ez) - Ez) / dr)
    Br = Br - dt * cr
    if m != 1:
        Br[0] = 0
    cz = (rh * Bp - (rh - dr) * below(Bp)) / (rs * dr) - 1j * m / rs * Br
    cp = sm * Br - (Bz - below(Bz)) / dr
    cz[0] = 4 * Bp[0] / dr if m == 0 else 0
    cp[0] = sm * Br[0] - 2 * Bz[0] / dr if m == 1 else 0
    a = 4 * math.pi * dt
    Er = Er + dt * (1j * m / rh * Bz - sm * Bp) - a * F * Jr
    Ep = Ep + dt * cp - a * F * Jp
    Ez = Ez + dt * cz - a * F * corr * Jz
    if m != 0:
        Ez[0] = 0
    if m != 1:
        Ep[0] = 0
    inv = lambda f: torch.fft.ifft(f, dim=1)  # noqa: E731
    return [inv(f) for f in (Ez, Er, Ep)], [inv(f) for f in (Bz, Br, Bp)]


def _shape_fn(order, d):
    a = d.abs()
    if order == 1:
        return (1 - a).clamp_min(0)
    if order == 2:
        return torch.where(a <= 0.5, 0.75 - a * a, 0.5 * (1.5 - a).clamp_min(0) ** 2)
    return torch.where(a <= 1, (4 - 6 * a * a + 3 * a ** 3) / 6, (2 - a).clamp_min(0) ** 3 / 6)


def _chunks(n, size=1 << 21):
    return [slice(i, min(n, i + size)) for i in range(0, n, size)]


def _x_gather(c, kw, fields, cell, off, order):
    """The six fields at the particles: [n, 6]."""
    d, ext = cell.shape[1], [c["n1"], c["n2"], c.get("n3", 1)]
    stag = [(1, 0, 0), (0, 1, 0), (0, 0, d - 2), (0, 1, d - 2), (1, 0, d - 2), (1, 1, 0)]
    flat = [f.double().reshape(-1) for f in fields]
    W, I = {}, {}
    for a in range(d):
        for h in (0, 1):
            p = off[:, a] - 0.5 * h
            i0 = p.floor() - 1
            W[a, h] = [_shape_fn(order, p - i0 - k) for k in range(4)]
            I[a, h] = [(cell[:, a].long() + i0.long() + k) % ext[a] for k in range(4)]
    out = torch.zeros((cell.shape[0], 6), device=DEV, dtype=torch.float64)
    for f, s in enumerate(stag):
        for k in range(4 if d == 3 else 1):
            for j in range(4):
                row = I[1, s[1]][j] if d == 2 else I[2, s[2]][k] * ext[1] + I[1, s[1]][j]
                w = W[1, s[1]][j] if d == 2 else W[1, s[1]][j] * W[2, s[2]][k]
                for i in range(4):
                    out[:, f] += flat[f][row * ext[0] + I[0, s[0]][i]] * (W[0, s[0]][i] * w)
    return out


def _x_push(c, kw, fields, cell, off, u, qm, order):
    d = cell.shape[1]
    ext = torch.tensor([c["n1"], c["n2"], c.get("n3", 1)][:d], device=DEV, dtype=torch.int32)
    s = torch.tensor([kw["dt"] / kw["dx1"], kw["dt"] / kw["dx2"], kw["dt"] / kw["dx3"]][:d], device=DEV, dtype=torch.float64)
    out = []
    for q in _chunks(cell.shape[0]):
        o, ce = off[q].double(), cell[q]
        f = o.floor()
        ce, o = torch.remainder(ce + f.to(torch.int32), ext), o - f
        F = _x_gather(c, kw, fields, ce, o, order)
        h = (qm[q].double() * (0.5 * kw["dt"]))[:, None]
        um = u[q].double() + h * F[:, :3]
        t = h * F[:, 3:] * torch.rsqrt(1 + um.square().sum(1, keepdim=True))
        up = um + torch.linalg.cross(um, t)
        un = um + torch.linalg.cross(up, 2 * t / (1 + t.square().sum(1, keepdim=True))) + h * F[:, :3]
        v = un * torch.rsqrt(1 + un.square().sum(1, keepdim=True))
        out.append((ce, o, un, o + v[:, :d] * s, v[:, 2]))
    return [torch.cat(x) for x in zip(*out)]


def _x_deposit(c, kw, cell, off, off_new, v3, q, order):
    d, ext, dt = cell.shape[1], [c["n1"], c["n2"], c.get("n3", 1)], kw["dt"]
    J = [torch.zeros(c["n1"] * c["n2"] * c.get("n3", 1), device=DEV, dtype=torch.float64) for _ in range(3)]
    W = order + 2
    for sl in _chunks(cell.shape[0], 1 << 22 if d == 2 else 1 << 19):
        S0, dS, I = [], [], []
        for a in range(d):
            x0, x1 = off[sl, a].double(), off_new[sl, a].double()
            g = (torch.minimum(x0, x1) - 0.5 * (order + 1)).floor() + 1
            s0 = [_shape_fn(order, x0 - g - w) for w in range(W)]
            S0.append(s0)
            dS.append([_shape_fn(order, x1 - g - w) - s0[w] for w in range(W)])
            I.append([(cell[sl, a].long() + g.long() + w) % ext[a] for w in range(W)])
        qq = q[sl].double()
        if d == 2:
            scale = [-qq / (dt * kw["dx2"]), -qq / (dt * kw["dx1"]), qq * v3[sl].double() / (kw["dx1"] * kw["dx2"])]
            for j in range(W):
                acc = torch.zeros_like(qq)
                for i in range(W):
                    acc = acc + dS[0][i] * (S0[1][j] + 0.5 * dS[1][j])
                    J[0].index_add_(0, I[1][j] * ext[0] + I[0][i], scale[0] * acc)
                    w3 = S0[0][i] * S0[1][j] + 0.5 * (dS[0][i] * S0[1][j] + S0[0][i] * dS[1][j]) + dS[0][i] * dS[1][j] / 3
                    J[2].index_add_(0, I[1][j] * ext[0] + I[0][i], scale[2] * w3)
            for i in range(W):
                acc = torch.zeros_like(qq)
                for j in range(W):
                    acc = acc + dS[1][j] * (S0[0][i] + 0.5 * dS[0][i])
                    J[1].index_add_(0, I[1][j] * ext[0] + I[0][i], scale[1] * acc)
            continue
        dx = [kw["dx1"], kw["dx2"], kw["dx3"]]
        for a in range(3):
            b, e = (a + 1) % 3, (a + 2) % 3
            scale = -qq / (dt * dx[b] * dx[e])
            for v in range(W):
                for w in range(W):
                    t = S0[b][v] * S0[e][w] + 0.5 * (dS[b][v] * S0[e][w] + S0[b][v] * dS[e][w]) + dS[b][v] * dS[e][w] / 3
                    acc = torch.zeros_like(qq)
                    for i in range(W):
                        acc = acc + dS[a][i] * t
                        at = {a: I[a][i], b: I[b][v], e: I[e][w]}
                        J[a].index_add_(0, (at[2] * ext[1] + at[1]) * ext[0] + at[0], scale * acc)
    return [j.reshape(_shape(c)) for j in J]


def _x_mlp(c, p, x, want_grad=None):
    """The network in 64 bits; p a flat float64 parameter vector."""
    dims, o = [MLP_IN] + [c["width"]] * c["depth"] + [1], 0
    h = x.double()
    for l, (fi, fo) in enumerate(zip(dims[:-1], dims[1:])):
        h = h @ p[o:o + fo * fi].view(fo, fi).T + p[o + fo * fi:o + fo * fi + fo]
        o += fo * fi + fo
        if l < c["depth"]:
            h = torch.tanh(h)
    return h[:, 0]


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "nci":
        return None                      # complete root sets: only a root finder gives them
    got = _inputs(c, seed)
    if kind == "beam":
        kw, (E, B, J), p = got
        J = _x_deposit(c, kw, *p, c["order"])
        E, B = _x_step(kw, E, B, J)
        return {"E": E, "B": B, "J": J}
    if kind == "advance":
        E, B = _x_step(got[0], *got[1])
        return {"E": E, "B": B}
    if kind == "quasi3d":
        E, B = _x_q3d(got[0], *got[1])
        return {"E": E, "B": B}
    if kind == "batch":
        out = []
        for kw, a in zip(*got):
            f = [list(a[3 * i:3 * i + 3]) for i in range(3)]
            E, B = _x_step(kw, *f) if kw["dims"] == 2 else _x_q3d(kw, *f)
            out.append(torch.stack(E + B))
        return out
    if kind == "push":
        kw, (E, B, J), p = got
        r = _x_push(c, kw, E + B, *p, c["order"])
        return dict(zip(("cell", "off", "u", "off_new", "v3"), r[:4] + [r[4] if c["dims"] == 2 else None]))
    if kind == "deposit":
        return {"J": _x_deposit(c, got[0], *got[1], c["order"])}
    if kind == "pic":
        kw, (E, B, J), (cell, off, u, qm, q) = got
        Bn = [(a.double() + b) / 2 for a, b in zip(B, _x_step(kw, E, B, faraday_only=True))]
        cell, o, u, on, v3 = _x_push(c, kw, E + Bn, cell, off, u, qm, c["order"])
        J = _x_deposit(c, kw, cell, o, on, v3, q, c["order"])
        E, B = _x_step(kw, E, B, J)
        return {"E": E, "B": B, "J": J, "cell": cell, "off": on, "u": u, "v3": v3}
    p = torch.from_numpy(got[0]).to(DEV).double()
    if kind == "mlp_forward":
        return {"y": _x_mlp(c, p, got[1])}
    m, v, losses = torch.zeros_like(p), torch.zeros_like(p), []
    for k in range(c["steps"]):
        p.requires_grad_(True)
        loss = (_x_mlp(c, p, got[1][k]) - got[2][k].double()).square().mean()
        g, = torch.autograd.grad(loss, p)
        losses.append(loss.detach())
        with torch.no_grad():
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            p = p - 1e-3 * (m / (1 - 0.9 ** (k + 1))) / ((v / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
    return {"params": p.detach().cpu().numpy(), "loss": torch.stack(losses)}
