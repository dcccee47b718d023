"""The register-resident row transforms through the advance: every row length they take, 2D and 3D, row counts that
fill no block, from two rows, both sides of the FP64 size rule, the three FP32 forms of a step (by row length and cells), k1-resident and not, against the oracle (the
tolerances of the other parity tests)."""
import numpy as np
import pytest

from paper_1502_01376_gb300 import workloads as wl

from gpu_util import hyb_module, need_gpu, orc_grid, rel_err, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("resident", [False, True])
@pytest.mark.parametrize("prec,n1,n2,n3", [(32, 128, 2, 1), (32, 128, 37, 1), (32, 256, 9, 1), (32, 512, 3, 1), (32, 2048, 5, 1),
                                           (32, 4096, 3, 1), (32, 8192, 2, 1), (32, 8192, 41, 1), (32, 128, 7, 5), (32, 512, 3, 4),
                                           (64, 64, 2, 1), (64, 64, 33, 1), (64, 128, 17, 1), (64, 256, 5, 1), (64, 256, 256, 1),
                                           (64, 256, 257, 1), (64, 128, 6, 3), (64, 512, 7, 1),
                                           (32, 1024, 5, 1), (32, 1024, 4, 3), (32, 128, 16411, 1), (32, 256, 111, 75), (32, 512, 4099, 1),
                                           (32, 1024, 2053, 1), (32, 1024, 29, 67), (32, 2048, 1031, 1), (32, 4096, 523, 1), (32, 8192, 311, 1),
                                           (32, 128, 257, 257), (32, 1024, 8209, 1), (32, 4096, 67, 31),
                                           (32, 1024, 511, 1), (32, 1024, 513, 1), (32, 8192, 1031, 1)])
def test_row_transforms_in_the_advance(prec, n1, n2, n3, resident, orc):
    need_gpu()
    hyb = hyb_module()
    dims = 3 if n3 > 1 else 2
    w = wl.Workload("rf", dims, n1, n2, n3, dx1=0.2, dx2=0.25, dx3=0.3, dt=0.06, precision=prec, filt_kc=0.6, filt_w=0.2)
    rng = np.random.default_rng(n1 + n2)
    real, tdt = (np.float32, torch.float32) if prec == 32 else (np.float64, torch.float64)
    F = [(rng.standard_normal(w.shape) * 1e-3).astype(real).astype(np.float64) for _ in range(9)]
    D = [torch.from_numpy(a).to("cuda", tdt) for a in F]
    g = hyb.Grid(hyb.desc_from_workload(w, path=1)).bind(D[:3], D[3:6], D[6:])
    if resident:
        g.set_resident(True)
    g.advance(3)
    g.check()
    orc.step(orc_grid(orc, w), F[:3], F[3:6], F[6:], nsteps=3)
    for a, b in zip(D[:6], F[:6]):
        assert rel_err(a.cpu().numpy(), b) < (1e-5 if prec == 32 else 1e-12)
    g.close()


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("n1,n2", [(64, 5), (128, 3), (256, 300), (8192, 3)])
def test_standalone_corrections_agree(n1, n2, prec):
    """hyb_correct_current with the grid's tables and the allocation-free entry point with its own."""
    need_gpu()
    hyb = hyb_module()
    tdt = torch.float32 if prec == 32 else torch.float64
    desc = hyb.make_desc(n1=n1, n2=n2, dx1=0.2, dx2=0.2, dt=0.1, precision=prec, path=1)
    D = [torch.randn(n2, n1, device="cuda", dtype=tdt) for _ in range(9)]
    other = D[6].clone()
    g = hyb.Grid(desc).bind(D[:3], D[3:6], D[6:])
    g.correct_current()
    hyb.hyb_correct_current_noalloc(desc, int(other.data_ptr()), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert rel_err(D[6].cpu().numpy(), other.cpu().numpy()) < (1e-6 if prec == 32 else 1e-14)
    g.close()
