"""The root solver's division of work: a call gives a warp up to 32 (sample, alias) pairs, fewer on
small calls.  A pair's roots do not depend on the pairs beside it, and settings whose disk is wide
against 1/h (the trigonometric calls instead of the series) still match the oracle."""
import numpy as np
import pytest

from gpu_util import hyb_module, need_gpu, torch
from test_gpu_nci import ALIASES, _samples

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 11, 2701, 13003])
def test_roots_do_not_depend_on_the_group(n):
    need_gpu()
    hyb = hyb_module()
    S = torch.from_numpy(_samples(n, 77, bump_every=7)).cuda()
    R, C, G, _ = hyb.nci_roots(S, aliases=ALIASES, order=2)      # groups of 1, 1, 6 and 32 pairs
    for lo in (0, n // 3, max(0, n - 5)):
        r, c, g, _ = hyb.nci_roots(S[lo:lo + 5], aliases=ALIASES, order=2)
        assert torch.equal(c, C[lo:lo + 5]) and torch.equal(g, G[lo:lo + 5])
        assert torch.equal(torch.view_as_real(r), torch.view_as_real(R[lo:lo + 5]))


def test_wide_disk_matches_oracle():
    """rho h between 0.4 and 1.1: points of the circle beyond the series' range."""
    need_gpu()
    hyb = hyb_module()
    from oracle import nci
    rows = [[dt, 1.0, 1.0, gam, 100.0, 0.0, 0.2, 1.1, 0.7, 0, 0, 0]
            for dt, gam in ((0.3, 5.0), (0.45, 3.0), (0.5, 2.0), (0.5, 1.5))]
    S = np.array(rows)
    R, C, G, err = hyb.nci_roots(torch.from_numpy(S).cuda(), aliases=ALIASES, order=2)
    assert err == 0
    R, C = R.cpu().numpy(), C.cpu().numpy()
    for i, (dt, dx1, dx2, gam, wp2, kc, fw, k1, k2, kl, ku, km) in enumerate(rows):
        P = nci.NciParams(dt=dt, dx1=dx1, dx2=dx2, gamma=gam, wp2=wp2, order=2, filt_kc=kc, filt_w=fw,
                          kmod_l=kl, kmod_u=ku, kmod_max=km)
        for a, (mu, nu) in enumerate(ALIASES):
            ro, rg = nci.roots(P, k1, k2, mu, nu), list(R[i, a, :C[i, a]])
            c, rho = nci.resonance(P, nci.symbols(P, k1, k2, mu, nu)), nci.region_radius(P)
            if any(abs(abs(w - c) - rho) < 1e-6 * rho for w in ro + rg):
                continue
            assert len(rg) == len(ro), (i, a, ro, rg)
            for w in ro:
                assert min(abs(w - u) for u in rg) < 1e-7 * max(1.0, abs(w)), (i, a, w, rg)
