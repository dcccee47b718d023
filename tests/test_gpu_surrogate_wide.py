"""Networks wider than 64 (the chained kernel): forward, loss, gradients and the Adam step at the edges of its
tiles: widths around a 128-row tile, batches around its 64 rows, one and many layers, few and many inputs.
Tolerances as for the narrow networks: the oracle rounds to BF16 at the same points, and a value that falls on the other
side of a rounding moves one operand by 2^-8 of itself."""
import numpy as np
import pytest

from oracle import mlp as omlp

from gpu_util import hyb_module, need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in,width,depth,B", [(6, 65, 2, 64), (6, 128, 1, 63), (3, 144, 3, 65), (40, 100, 2, 1), (256, 256, 2, 200),
                                                (1, 250, 5, 1000), (6, 256, 4, 8200), (17, 129, 16, 129)])
def test_wide_networks_match_oracle(n_in, width, depth, B):
    need_gpu()
    hyb = hyb_module()
    rng = np.random.default_rng(width + B)
    p = hyb.mlp_init_params(n_in, width, depth, seed=width)
    p[-1:] = 0.1
    net = hyb.MLP(n_in, width, depth, params=p)
    x = rng.uniform(-1, 1, (B, n_in)).astype(np.float32)
    t = rng.uniform(0, 2, B).astype(np.float32)
    xg, tg = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    y = net.forward(xg).cpu().numpy()
    P = p.astype(np.float64)
    yo = omlp.forward(P, x, n_in, width, depth)[0]
    assert np.linalg.norm(y - yo) / np.linalg.norm(yo) < 2e-3
    g, loss = net.gradients(xg, tg)
    go, lo = omlp.gradients(P, x, t, n_in, width, depth)
    assert abs(loss - lo) / lo < 2e-3
    assert np.linalg.norm(g - go) / np.linalg.norm(go) < 5e-3
    net.train_step(xg, tg, 1e-2)
    assert np.max(np.abs(net.get_params() - (p - 1e-2 * g / (np.abs(g) + 1e-8)))) < 1e-5
    y2 = net.forward(xg).cpu().numpy()                       # the updated weights are the ones that run
    yo2 = omlp.forward(net.get_params().astype(np.float64), x, n_in, width, depth)[0]
    assert np.linalg.norm(y2 - yo2) / np.linalg.norm(yo2) < 2e-3
    net.close()


def test_wide_training_is_repeatable():
    need_gpu()
    hyb = hyb_module()
    rng = np.random.default_rng(1)
    p = hyb.mlp_init_params(6, 200, 3, seed=1)
    nets = [hyb.MLP(6, 200, 3, params=p) for _ in range(2)]
    for B in (1000, 70, 3000):                               # the buffers grow and are used in part
        x = torch.from_numpy(rng.uniform(-1, 1, (B, 6)).astype(np.float32)).cuda()
        t = torch.from_numpy(rng.uniform(0, 2, B).astype(np.float32)).cuda()
        for net in nets:
            net.train_step(x, t, 1e-3)
    assert np.array_equal(nets[0].get_params(), nets[1].get_params())
    for n in nets:
        n.close()
