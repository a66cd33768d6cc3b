"""Closure training data and training at the edges of their tiles: filter widths that do and do not
divide a block's threads, rows that end inside a block's group of coarse cells, batches that run as
one cluster per epoch (at most 16 tiles of 128 samples) and larger ones (a block per tile).
"""
import numpy as np
import pytest

import oracle as O
import workloads as W
from oracle import closure as C
from paper_2410_09739_gb300 import fpclbm as F

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,coarse", [(1, (5, 4, 3)), (2, (3, 3, 2)), (3, (7, 2, 2)), (4, (66, 2, 1)), (5, (53, 1, 1)),
                                      (70, (1, 1, 1))])
@pytest.mark.parametrize("prec,steps", [("fp64", 2), ("fp32", 3)])
def test_sample_edges(r, coarse, prec, steps):
    """Like test_sample_matches_oracle_filter: float32 on output, 1e-5 of each column's scale; the
    labels divide by the strain, so only their bound (a rate change in (-2, 0]) and, where the
    strain is not near zero, their value are checked."""
    nx, ny, nz = (r * c for c in coarse)
    with F.Lattice(nx, ny, nz, prec) as lat:
        lat.set_params(0.6)
        lat.set_force(1e-5, -2e-5, 1e-5)
        lat.init_fields(*W.random_fields(nx, ny, nz, 3, u_amp=0.05))
        lat.step(steps)
        f = lat.get_populations()
        nc = coarse[0] * coarse[1] * coarse[2]
        X, T = np.empty((nc, 9), np.float32), np.empty(nc, np.float32)
        F.fpclbm_closure_sample(lat.h, r, 0.55, X, T)
    Xr, Tr = C.sample(*O.moments(f, (1e-5, -2e-5, 1e-5)), r, 0.55, False)
    for k in range(9):
        assert np.max(np.abs(X[:, k] - Xr[:, k])) <= 1e-5 * np.max(np.abs(Xr)) , k
    assert np.all((T <= 0) & (T > -2))
    if min(coarse) > 1:
        assert np.max(np.abs(T - Tr)) <= 1e-4 * (np.max(np.abs(Tr)) + 1e-30)


def data(n):
    rng = np.random.default_rng(n)
    X = rng.normal(scale=0.05, size=(n, 9)).astype(np.float32)
    t = (0.1 * np.tanh(20 * X[:, 0] * X[:, 7]) + 0.01 * rng.normal(size=n)).astype(np.float32)
    return torch.from_numpy(X).cuda(), torch.from_numpy(t).cuda()


@pytest.mark.parametrize("n", [2, 127, 128, 129, 1000, 4500])
def test_batch_tilings_agree_on_the_loss(n):
    """A learning rate that leaves every fp32 weight unchanged: an epoch's loss is that of the initial
    network whatever the batch, in multiples of the tile so that the tiles are the same (fp64 sums)."""
    X, t = data(n)
    losses = [F.fpclbm_closure_train(X, t, n, 2, b, 1e-30, seed=3)[1] for b in (128, 384, 1024, 2048, 4096)]
    for l in losses[1:]:
        assert np.allclose(l, losses[0], rtol=1e-12, atol=0)


@pytest.mark.parametrize("batch", [100, 128, 700, 1024, 1100, 2048, 2100])
def test_training_repeats_bit_for_bit(batch):
    X, t = data(4500)
    w, l = F.fpclbm_closure_train(X, t, 4500, 20, batch, 3e-3, seed=1)
    w2, l2 = F.fpclbm_closure_train(X, t, 4500, 20, batch, 3e-3, seed=1)
    assert np.array_equal(w, w2) and np.array_equal(l, l2)
    assert np.all(np.isfinite(l)) and l[-1] < l[0]
