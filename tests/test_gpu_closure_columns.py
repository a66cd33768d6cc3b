"""Closure training data column by column, every storage type, periodic boxes and channels: rows that
end inside a block's group of coarse cells and rows that several blocks share.

The features leave in float32 (one rounding of each value, 2^-24) and come from fields that agree with
fp64 sums to 1e-12 (as in test_gpu_fields.py), differenced over two coarse cells: 2^-23 of the column's
own scale and 1e-11 absolute.  The labels divide by the strain; 1e-5 of their scale, as in
test_gpu_closure.py.
"""
import numpy as np
import pytest

import oracle as O
import workloads as W
from oracle import closure as C
from paper_2410_09739_gb300 import fpclbm as F

pytestmark = pytest.mark.gpu

FORCE = (1e-5, -2e-5, 1e-5)


@pytest.mark.parametrize("r,coarse", [(2, (129, 2, 2)), (3, (7, 2, 2)), (4, (66, 2, 2)), (5, (53, 3, 2)), (40, (3, 2, 2)),
                                      # short rows, blocks of one warp and of eight
                                      (1, (2, 5, 4)), (2, (2, 40, 40)), (3, (5, 9, 50)), (2, (8, 72, 72)), (1, (3, 210, 130))])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("walls", [0, 1])
def test_every_column(r, coarse, prec, walls):
    nx, ny, nz = (r * c for c in coarse)
    nc = coarse[0] * coarse[1] * coarse[2]
    X, T = np.empty((nc, 9), np.float32), np.empty(nc, np.float32)
    with F.Lattice(nx, ny, nz, prec, walls) as lat:
        lat.set_params(0.6)
        lat.set_force(*FORCE)
        lat.init_fields(*W.random_fields(nx, ny, nz, 3, u_amp=0.05))
        lat.step(3)
        f = lat.get_populations()
        F.fpclbm_closure_sample(lat.h, r, 0.55, X, T)
    Xr, Tr = C.sample(*O.moments(f, FORCE), r, 0.55, bool(walls))
    for k in range(9):
        assert np.max(np.abs(X[:, k] - Xr[:, k])) <= 2.0 ** -23 * np.max(np.abs(Xr[:, k])) + 1e-11, k
    assert np.max(np.abs(T - Tr)) <= 1e-5 * np.max(np.abs(Tr))
