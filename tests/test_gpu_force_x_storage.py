"""A body force along x with unit rates (the channels' collision) in 16-bit and fp32 storage: every
kernel variant, both parities, on the boundary kinds whose paired kernels differ (registers, pairing of
the odd step): periodic, resting walls, a moving wall, the symmetry plane; rows of odd and even length,
odd cell counts.

One step at a time from the stored state, against one step of the oracle from the same state: the
difference of a population is the fp32 collision's (1e-6 absolute, as in test_gpu_parity.py) and one
rounding of its deviation to the storage type (unit roundoff u, 2^-25 absolute below fp16's normal
numbers).  The variants that take neighbouring cells store the same bits.
"""
import numpy as np
import pytest

import oracle as O
import workloads as W
from paper_2410_09739_gb300 import fpclbm as F

pytestmark = pytest.mark.gpu

UNIT = {"fp32": 2.0 ** -24, "fp16": 2.0 ** -11, "bf16": 2.0 ** -8}
FX, LID = 3e-4, 0.05
REST = O.equilibrium(1.0, [0, 0, 0])[:, None, None, None]


@pytest.mark.parametrize("prec", ["bf16", "fp16", "fp32"])
@pytest.mark.parametrize("shape", [(2, 3, 3), (17, 9, 5), (6, 5, 3), (16, 9, 5), (34, 8, 3)])
@pytest.mark.parametrize("bc,lid", [(0, 0.0), (1, 0.0), (1, LID), (3, 0.0)])
@pytest.mark.parametrize("mode", [0, 1])
def test_one_step_of_each_parity(monkeypatch, prec, shape, bc, lid, mode):
    f0 = O.init_equilibrium(*W.random_fields(*shape, 13 + bc + mode, u_amp=0.05))
    f0 = f0 * (1.0 + 0.02 * np.random.default_rng(shape[0]).uniform(-1, 1, f0.shape))
    staged = not lid and bc < 2 and (shape[0] * (4 if prec == "fp32" else 2)) % 16 == 0
    after = {}
    for variant in (0, 2, 3) if staged else (0, 2):
        monkeypatch.setenv("FPCLBM_LAUNCH", "128:2:%d" % variant)
        with F.Lattice(*shape, prec, bc) as lat:
            lat.set_params(0.7, 0.0, mode)
            lat.set_force(FX)
            if lid:
                lat.set_wall_velocity(lid)
            lat.set_populations(f0)
            for parity in (0, 1):
                before = lat.get_populations()
                lat.step(1)
                assert lat.launch()["variant"] == variant
                got = lat.get_populations()
                ref = O.run(before, 1, bc=bc, F=(FX, 0, 0), omega=O.rates(0.7), mode=mode, uw=(lid, 0.0, 0.0))
                bound = UNIT[prec] * np.abs(ref - REST) + 1e-6 * (1 + UNIT[prec]) + 2.0 ** -25
                assert np.all(np.abs(got - ref) <= bound), (variant, parity)
            after[variant] = got
    if staged:
        assert np.array_equal(after[2], after[3])
