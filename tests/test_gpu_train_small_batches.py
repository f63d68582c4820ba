"""GPU: training with batches that leave blocks of the cluster without samples (8
blocks below 32 samples, 16 from there on, in units of 4 samples): many steps in one
launch give the bits of single steps, and the gradients of the float64 reference."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from synth.band import mlp_init

import paper_2205_07610_gb300 as ga

pytestmark = pytest.mark.gpu

SIZES = (1, 5, 16, 17, 29, 32, 33, 36, 48, 64, 65, 100, 257, 260, 300)


def _problem(n, seed):
    rng = np.random.default_rng(seed)
    x = rng.uniform(0, 1, size=(n, 32)).astype(np.float32)
    t = rng.uniform(0, 12, size=n).astype(np.float32)
    return mlp_init(seed), x, t


@pytest.mark.parametrize("n", SIZES)
def test_many_steps_equal_single_steps(n):
    steps = 40
    p, x, t = _problem(500, 200 + n)
    X, T = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    idx = torch.from_numpy(np.random.default_rng(n).integers(0, 500, size=(steps, n)).astype(np.int32)).cuda()
    runs = []
    for cut in ([steps], [1] * steps):
        master = torch.from_numpy(p.copy()).cuda()
        am, av = torch.zeros_like(master), torch.zeros_like(master)
        wb = ga.mlp_cast(master)
        losses, k = [], 0
        for s in cut:
            losses.append(ga.mlp_train(master, wb, am, av, X, T, idx[k:k + s].contiguous(), step0=k, lr=1e-3))
            k += s
        runs.append([a.cpu().numpy() for a in (master, am, av, wb, torch.cat(losses))])
    for a, b in zip(*runs):
        np.testing.assert_array_equal(a, b)
    assert np.isfinite(runs[0][4]).all()


@pytest.mark.parametrize("n", SIZES)
def test_gradient_parity(n):
    p, x, t = _problem(n, 300 + n)
    wb = ga.mlp_cast(torch.from_numpy(p).cuda())
    p64 = (wb.cpu().numpy().view(np.uint16).astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    loss, g = ga.mlp_loss_grad(wb, torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
    L, gref = omlp.loss_grad(p64, x.astype(np.float64), t.astype(np.float64))
    # float32 sums of n terms: (n + 160) roundings of 2^-24 of the largest terms
    tol = (n + 160) * 2.0 ** -24
    assert abs(float(loss.item()) - L) <= 4 * tol * max(1.0, L)
    scale = np.abs(t).max() * max(1.0, np.abs(p64).max()) * 8
    assert np.max(np.abs(g.cpu().numpy() - gref)) <= 4 * tol * scale + 1e-6
