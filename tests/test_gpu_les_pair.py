"""The Smagorinsky mode with unit rates of orders 3-6: two cells per thread and one, even and odd rows
(the neighbouring-cell odd step needs even nx; the symmetry plane of the half channel moves links in
x), with and without a force along x, against the oracle.  FP32: 1e-6 absolute per step as in
test_gpu_parity.py.
"""
import numpy as np
import pytest

import oracle as O
import workloads as W
from paper_2410_09739_gb300 import fpclbm as F

pytestmark = pytest.mark.gpu

LES = (0.17, 0.01, 26.0)


def advance(shape, prec, bc, fx, n, f0, smag=True):
    with F.Lattice(*shape, prec, bc) as lat:
        lat.set_params(0.52, 0.0, F.FPCLBM_DIFF_FP_SMAGORINSKY if smag else F.FPCLBM_DIFF_FP)
        if smag:
            lat.set_smagorinsky(*LES)
        lat.set_force(fx)
        lat.set_populations(f0)
        fq = lat.get_populations()
        lat.step(n)
        return fq, lat.get_populations(), lat.launch()


def start(shape, seed):
    f = O.init_equilibrium(*W.random_fields(*shape, seed, u_amp=0.05))
    return f * (1.0 + 0.02 * np.random.default_rng(seed).uniform(-1, 1, f.shape))


@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 2), (6, 5, 4), (7, 6, 5), (34, 8, 3)])
@pytest.mark.parametrize("bc", [0, 1, 3])
@pytest.mark.parametrize("fx", [0.0, 3e-4])
@pytest.mark.parametrize("launch", ["128:2:2", "128:1:0"])
def test_fp32_matches_oracle(monkeypatch, shape, bc, fx, launch):
    monkeypatch.setenv("FPCLBM_LAUNCH", launch)
    f0 = start(shape, 5 + bc)
    for n in (1, 4):
        fq, got, lau = advance(shape, "fp32", bc, fx, n, f0)
        ref = O.run(fq, n, bc=bc, F=(fx, 0, 0), omega=O.rates(0.52), les=LES)
        assert np.max(np.abs(got - ref)) <= 1e-6 * n
        assert lau["mode"] == 3 and lau["variant"] == int(launch[-1])


@pytest.mark.parametrize("bc", [0, 1, 3])
@pytest.mark.parametrize("fx", [0.0, 3e-3])
def test_fp64_matches_oracle(bc, fx):
    shape = (7, 6, 5)
    fq, got, _ = advance(shape, "fp64", bc, fx, 3, start(shape, 9))
    ref = O.run(fq, 3, bc=bc, F=(fx, 0, 0), omega=O.rates(0.52), les=LES)
    assert np.max(np.abs(got - ref)) <= 3e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("prec", ["fp16", "bf16"])
def test_half_channel_plain_pair_even_rows(monkeypatch, prec):
    """The neighbouring-cell odd step through the symmetry plane with 16-bit storage: equal to the
    cells c, c + N/2 pairing of the same arithmetic (which a box with odd nx would take), here
    checked against the oracle within one rounding of the stored deviations per step."""
    monkeypatch.setenv("FPCLBM_LAUNCH", "128:2:2")
    shape = (10, 6, 5)
    fq, got, _ = advance(shape, prec, 3, 0.0, 2, start(shape, 3), smag=False)
    ref = O.run(fq, 2, bc=3, omega=O.rates(0.52))
    dev = np.max(np.abs(ref - O.equilibrium(1.0, [0, 0, 0])[:, None, None, None]))
    assert np.max(np.abs(got - ref)) <= 2 * {"fp16": 2.0 ** -11, "bf16": 2.0 ** -8}[prec] * dev * 2 + 2e-6
