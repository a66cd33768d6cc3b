"""Unit rates of orders 3-6 with a body force along x (the channels): the collision that forms only
the moments this force's sources read, on every boundary kind and kernel variant, against the oracle
(general sources).  Bounds as in test_gpu_parity.py: 1e-12 relative per FP64 step, 1e-6 absolute per
FP32 step.
"""
import numpy as np
import pytest

import oracle as O
import workloads as W
from paper_2410_09739_gb300 import fpclbm as F

pytestmark = pytest.mark.gpu


def start(shape, seed, near=True):
    nx, ny, nz = shape
    if not near:
        return W.random_populations(nx * ny * nz, seed).reshape(27, nz, ny, nx)
    f = O.init_equilibrium(*W.random_fields(nx, ny, nz, seed, u_amp=0.05))
    return f * (1.0 + 0.02 * np.random.default_rng(seed).uniform(-1, 1, f.shape))


@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 3, 3), (17, 9, 5)])
@pytest.mark.parametrize("bc", [0, 1, 2, 3])
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("fx", [2e-3, -3e-2])
def test_one_step_fp64(shape, bc, mode, fx):
    """Random populations far from equilibrium and random shear and bulk rates."""
    nx, ny, nz = shape
    seed = 40 + nx + 3 * bc + mode
    f0 = start(shape, seed, near=False)
    om = np.ones(27)
    om[4:10] = np.random.default_rng(seed).uniform(0.4, 1.8, 6)
    with F.Lattice(nx, ny, nz, "fp64", bc) as lat:
        lat.set_params(1.0, 0.0, mode)
        lat.set_rates(om)
        lat.set_force(fx)
        lat.set_populations(f0)
        lat.step(1)
        got = lat.get_populations()
    ref = O.step(f0, bc=bc, F=(fx, 0, 0), omega=om, mode=mode)
    assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("launch,shape", [("128:2:0", (17, 9, 5)), ("128:2:2", (17, 9, 5)), ("128:2:2", (16, 9, 5)),
                                          ("128:2:3", (16, 9, 6)), ("128:2:1", (17, 9, 5))])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("mode", [0, 1])
def test_variants_fp32(monkeypatch, launch, shape, bc, mode):
    monkeypatch.setenv("FPCLBM_LAUNCH", launch)
    nx, ny, nz = shape
    f0 = start(shape, 7 + bc + mode)
    with F.Lattice(nx, ny, nz, "fp32", bc) as lat:
        lat.set_params(0.7, 0.0, mode)
        lat.set_force(3e-4)
        lat.set_populations(f0)
        fq = lat.get_populations()
        lat.step(5)
        got = lat.get_populations()
    ref = O.run(fq, 5, bc=bc, F=(3e-4, 0, 0), omega=O.rates(0.7), mode=mode)
    assert np.max(np.abs(got - ref)) <= 5e-6


def test_ensemble_equals_single_box():
    with F.Lattice.ensemble([(6, 5, 4), (7, 6, 5)], [0.7, 0.9], "fp32") as ens:
        ens.set_force(3e-4)
        f = [start(s, 11) for s in ((6, 5, 4), (7, 6, 5))]
        ens.set_populations(np.concatenate([a.reshape(27, -1) for a in f], axis=1))
        ens.step(5)
        got = ens.get_populations()
    at = 0
    for s, tau, f0 in zip(((6, 5, 4), (7, 6, 5)), (0.7, 0.9), f):
        n = s[0] * s[1] * s[2]
        ref = O.run(f0, 5, F=(3e-4, 0, 0), omega=O.rates(tau))
        assert np.max(np.abs(got[:, at:at + n] - ref.reshape(27, -1))) <= 5e-6
        at += n


@pytest.mark.parametrize("variant", ["128:2:2", "128:2:0", "128:1:0"])
def test_learned_closure_with_force_x(monkeypatch, variant):
    """Zero network weights leave the rates unchanged: the learned mode equals the plain one."""
    monkeypatch.setenv("FPCLBM_LAUNCH", variant)
    shape = (16, 9, 5)
    f0 = start(shape, 21)
    with F.Lattice(*shape, "fp32", 1) as lat:
        lat.set_closure(np.zeros(4865, np.uint16))
        lat.set_params(0.7, 0.0, F.FPCLBM_DIFF_FP_LEARNED)
        lat.set_force(3e-4)
        lat.set_populations(f0)
        fq = lat.get_populations()
        lat.step(3)
        got = lat.get_populations()
    ref = O.run(fq, 3, bc=1, F=(3e-4, 0, 0), omega=O.rates(0.7))
    assert np.max(np.abs(got - ref)) <= 3e-6
