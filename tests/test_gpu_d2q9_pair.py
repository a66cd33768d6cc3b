"""The 2D step with two cells per thread (boxes of at least 65,536 cells): even and odd rows, odd cell
counts, periodic and closed boxes, against the oracle.  FP32: 1e-6 absolute per step; 16-bit storage:
the oracle starts from the stored populations, so one step differs by one rounding of the deviation
plus the fp32 term (bounds of test_gpu_parity.py).
"""
import numpy as np
import pytest

from oracle import oracle2d as O2
from paper_2410_09739_gb300 import fpclbm as F

pytestmark = pytest.mark.gpu

SHAPES = [(256, 256), (257, 256), (259, 255), (32768, 2), (2, 32769)]  # nx, ny


def start(nx, ny, seed):
    rng = np.random.default_rng(seed)
    f = O2.init_equilibrium(1 + 0.02 * rng.uniform(-1, 1, (ny, nx)), *(0.05 * rng.uniform(-1, 1, (2, ny, nx))))
    return f * (1 + 0.02 * rng.uniform(-1, 1, f.shape))


def advance(nx, ny, prec, f0, n, box, force, mode):
    with F.Lattice2D(nx, ny, prec) as lat:
        lat.set_params(0.6, 1.2, 0.3, mode)
        lat.set_force(*((2e-4, -1e-4) if force else (0.0, 0.0)))
        if box:
            lat.set_boundary(F.FPCLBM_BC_BOX, 0.05)
        lat.set_populations(f0)
        fq = lat.get_populations()
        lat.step(n)
        got = lat.get_populations()
    ref = O2.run(fq, n, F=(2e-4, -1e-4) if force else (0.0, 0.0), omega=O2.rates(0.6, 1.2, 0.3), mode=mode,
                 bc=2 if box else 0, uw=0.05 if box else 0.0)
    return got, ref


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("box", [False, True])
@pytest.mark.parametrize("force,mode", [(False, 0), (True, 0), (False, 1)])
def test_fp32_matches_oracle(shape, box, force, mode):
    f0 = start(*shape, 3)
    for n in (1, 2, 5):
        got, ref = advance(*shape, "fp32", f0, n, box, force, mode)
        assert np.max(np.abs(got - ref)) <= 1e-6 * n, n


@pytest.mark.parametrize("prec,unit", [("fp16", 2.0 ** -11), ("bf16", 2.0 ** -8)])
@pytest.mark.parametrize("shape", SHAPES[:3])
@pytest.mark.parametrize("box", [False, True])
def test_16_bit_storage_is_one_rounding_off(prec, unit, shape, box):
    got, ref = advance(*shape, prec, start(*shape, 4), 1, box, True, 0)
    w = np.array([1 / 6, 2 / 3, 1 / 6])
    ex, ey = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1]), np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])
    dev = np.abs(ref - (w[ex + 1] * w[ey + 1])[:, None, None])
    assert np.all(np.abs(got - ref) <= unit * dev + 1e-6)
