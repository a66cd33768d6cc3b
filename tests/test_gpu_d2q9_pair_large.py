"""The 2D step with two cells per thread from 2^17 cells on (2^18 for odd rows): even and odd rows, odd cell
counts, rows of two cells and two rows, periodic and closed boxes, against the oracle, with the bounds of
test_gpu_d2q9_pair.py (fp32 1e-6 absolute per step; 16-bit storage one rounding of the deviation more).
"""
import numpy as np
import pytest

from oracle import oracle2d as O2
from paper_2410_09739_gb300 import fpclbm as F

pytestmark = pytest.mark.gpu

UNIT = {"fp32": 0.0, "fp16": 2.0 ** -11, "bf16": 2.0 ** -8}
FORCE, LID = (2e-4, -1e-4), 0.05


@pytest.mark.parametrize("prec", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("shape", [(512, 256), (513, 512), (515, 511), (65536, 2), (2, 65537)])  # nx, ny
@pytest.mark.parametrize("box", [False, True])
@pytest.mark.parametrize("force,mode", [(False, 0), (True, 0), (False, 1)])
def test_one_step_of_each_parity(prec, shape, box, force, mode):
    nx, ny = shape
    rng = np.random.default_rng(nx)
    f0 = O2.init_equilibrium(1 + 0.02 * rng.uniform(-1, 1, (ny, nx)), *(0.05 * rng.uniform(-1, 1, (2, ny, nx))))
    rest = O2.init_equilibrium(np.ones((1, 1)), np.zeros((1, 1)), np.zeros((1, 1)))
    with F.Lattice2D(nx, ny, prec) as lat:
        lat.set_params(0.6, 1.2, 0.3, mode)
        lat.set_force(*(FORCE if force else (0.0, 0.0)))
        if box:
            lat.set_boundary(F.FPCLBM_BC_BOX, LID)
        lat.set_populations(f0 * (1 + 0.02 * rng.uniform(-1, 1, f0.shape)))
        for _ in range(2):
            before = lat.get_populations()
            lat.step(1)
            ref = O2.run(before, 1, F=FORCE if force else (0.0, 0.0), omega=O2.rates(0.6, 1.2, 0.3), mode=mode,
                         bc=2 if box else 0, uw=LID if box else 0.0)
            u = UNIT[prec]
            assert np.all(np.abs(lat.get_populations() - ref) <= u * np.abs(ref - rest) + 1e-6 * (1 + u) + 2.0 ** -25)
