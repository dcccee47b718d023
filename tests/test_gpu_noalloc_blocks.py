"""hyb_correct_current_noalloc: its row blocks hold as many rows as the working array has room for, and every table that a
transform reads is there at each row length."""
import pytest

from gpu_util import hyb_module, need_gpu, rel_err, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("n1", [8, 32, 64, 128, 256, 512, 1024, 2048, 4096, 8192])
@pytest.mark.parametrize("n2", [2, 37, 300])
def test_agrees_with_the_grid_at_every_row_length(n1, n2, prec):
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


def test_500_long_rows_take_four_blocks():
    """FP64 rows of 8192: 125 of them fit a block, so 500 take as long as 496 (a block more took 1.24 times as long)."""
    need_gpu()
    hyb = hyb_module()
    t = {}
    for n2 in (496, 500):
        j = torch.randn(n2, 8192, device="cuda", dtype=torch.float64)
        desc = hyb.make_desc(n1=8192, n2=n2, dx1=0.2, dx2=0.2, dt=0.08, precision=64, path=1)
        best = 1e9
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(4):
                hyb.hyb_correct_current_noalloc(desc, int(j.data_ptr()), torch.cuda.current_stream().cuda_stream)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        t[n2] = best
    assert t[500] < 1.1 * t[496], t
