"""Field kernels on fp32 and 16-bit storage (equilibrium from rho, u; rho, u from populations), whose
arithmetic runs on pairs of fp32 values instead of fp64: small and rest velocities, where the
deviations are far below the weights, and cells outside the pairs' range, which take the fp64 form.
"""
import numpy as np
import pytest

import oracle as O
import workloads as W
from oracle import oracle2d as O2
from paper_2410_09739_gb300 import fpclbm as F

pytestmark = pytest.mark.gpu

W1 = np.array([1 / 6, 2 / 3, 1 / 6])
UNIT = {"fp32": 2.0 ** -24, "fp16": 2.0 ** -11, "bf16": 2.0 ** -8}


def _deviations2d(lat, shape):
    """The stored deviations of a 2D box: populations minus the rest weights (exact to ~1e-16)."""
    ex = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])
    ey = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])
    w = W1[ex + 1] * W1[ey + 1]
    return lat.get_populations() - w[:, None, None], w


@pytest.mark.parametrize("prec", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("amp", [0.1, 1e-4, 0.0])
def test_init_2d_is_the_rounded_equilibrium(prec, amp):
    """One rounding to the stored type (fp16: plus half its smallest subnormal), plus 4e-16 for the
    fp64 populations that both sides pass through (weights up to 4/9: two roundings of 2^-53)."""
    nx, ny = 37, 19
    rng = np.random.default_rng(3)
    rho = 1.0 + 0.5 * amp * rng.uniform(-1, 1, (ny, nx))
    ux, uy = amp * rng.uniform(-1, 1, (2, ny, nx))
    with F.Lattice2D(nx, ny, prec) as lat:
        lat.init_fields(rho, ux, uy)
        got, w = _deviations2d(lat, (ny, nx))
    want = O2.init_equilibrium(rho, ux, uy) - w[:, None, None]
    slack = 4e-15 + (2.0 ** -25 if prec == "fp16" else 0.0)
    err = np.abs(got - want) - 1.001 * UNIT[prec] * np.abs(want)
    assert np.max(err) <= slack, float(np.max(err))


@pytest.mark.parametrize("prec", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("steps", [0, 3])
@pytest.mark.parametrize("box", [False, True])
def test_moments_2d_are_fp64_sums(prec, steps, box):
    nx, ny = 21, 11
    rng = np.random.default_rng(4)
    with F.Lattice2D(nx, ny, prec) as lat:
        lat.set_params(0.7)
        lat.set_force(1e-4, -2e-4)
        if box:
            lat.set_boundary(F.FPCLBM_BC_BOX, 0.05)
        lat.init_fields(1 + 0.02 * rng.uniform(-1, 1, (ny, nx)), *(0.08 * rng.uniform(-1, 1, (2, ny, nx))))
        if steps:
            lat.step(steps)
        got = lat.moments()
        f = lat.get_populations()
    for x, y in zip(got, O2.moments(f, (1e-4, -2e-4))):
        assert np.max(np.abs(x - y)) <= 2e-15  # nine fp64 terms of up to 4/9 on the oracle's side


@pytest.mark.parametrize("scale", [1e-3, 1e-7, 0.0])
def test_init_3d_fp32_small_velocities(scale):
    nx, ny, nz = 19, 5, 3
    rho, ux, uy, uz = W.random_fields(nx, ny, nz, seed=8, u_amp=scale, rho_amp=scale)
    with F.Lattice(nx, ny, nz, "fp32") as lat:
        lat.init_fields(rho, ux, uy, uz)
        raw, _ = lat.get_state()
    got = raw.view(np.float32).reshape(27, -1)[:, :nx * ny * nz].astype(np.float64)
    # the expanded form in fp64: no cancellation against the weights
    d = [[0.5 * (v * v - v), -v * v, 0.5 * (v * v + v)] for v in (ux.ravel(), uy.ravel(), uz.ravel())]
    for s in range(27):
        ix, iy, iz = s % 3, (s // 3) % 3, s // 9
        A, B, C = W1[ix], W1[iy], W1[iz]
        a, b, c = d[0][ix], d[1][iy], d[2][iz]
        t = [(rho.ravel() - 1) * ((A + a) * (B + b) * (C + c)), a * (B + b) * (C + c), A * b * (C + c), A * B * c]
        want = t[0] + t[1] + t[2] + t[3]
        big = sum(np.abs(x) for x in t)  # the terms may cancel: 2^-40 of them bounds the pairs' own error
        assert np.all(np.abs(got[s] - want) <= 2.0 ** -24 * np.abs(want) + 2.0 ** -40 * big + 2.0 ** -149)


def test_extreme_cells_take_the_fp64_form():
    """Cells whose density or velocity lies beyond the pairs' range, or is not finite: finite where
    the fp64 form is (one fp32 rounding, plus 2^-50 of the largest term for its own rounding), the
    same non-finite slots otherwise; ordinary neighbours are untouched."""
    rho = np.array([1.0, 2000.0, 1.0, np.inf, 1.0, 1.0, 1.0, np.nan])
    ux = np.array([0.1, 0.1, 3000.0, 0.1, np.inf, 0.1, 0.1, 0.1])
    uy = np.array([0.1, -0.2, 0.1, 0.1, 0.1, -5e4, 0.1, 0.1])
    uz = np.full(8, 0.05)
    with F.Lattice(8, 1, 1, "fp32") as lat:
        lat.init_fields(rho, ux, uy, uz)
        raw, _ = lat.get_state()
    got = raw.view(np.float32).reshape(27, -1)[:, :8].astype(np.float64)
    ordinary = np.zeros(8, bool)
    ordinary[[0, 1, 2, 5, 6]] = True
    with np.errstate(all="ignore"):
        ph = [[W1[0] + 0.5 * (v * v - v), W1[1] - v * v, W1[2] + 0.5 * (v * v + v)] for v in (ux, uy, uz)]
        f = np.array([rho * ph[0][s % 3] * ph[1][(s // 3) % 3] * ph[2][s // 9] -
                      W1[s % 3] * W1[(s // 3) % 3] * W1[s // 9] for s in range(27)])
    assert np.all(np.isfinite(got[:, ordinary]))
    scale = np.max(np.abs(f[:, ordinary]), axis=0)
    assert np.all(np.abs(got[:, ordinary] - f[:, ordinary]) <= 2.0 ** -24 * np.abs(f[:, ordinary]) + 2.0 ** -45 * scale)
    assert not np.any(np.isfinite(got[:, [3, 4, 7]]).all(axis=0))


def test_ensemble_fields_on_the_device_equal_single_boxes():
    """Fields in and out of an ensemble in one launch each, boxes of odd sizes (odd offsets in the
    concatenated arrays, ragged tiles): the same populations and moments as single boxes."""
    torch = pytest.importorskip("torch")
    dims = [(7, 5, 3), (16, 9, 2), (1, 1, 1), (31, 3, 3), (40, 7, 5)]
    taus = [0.6, 0.7, 0.8, 0.9, 1.0]
    flds = [W.random_fields(*d, seed=20 + i) for i, d in enumerate(dims)]
    flat = [torch.from_numpy(np.concatenate([f[q].ravel() for f in flds])).cuda() for q in range(4)]
    for steps in (0, 3):
        with F.Lattice.ensemble(dims, taus, "fp32") as ens:
            ens.set_force(1e-4, 0.0, -1e-4)
            F.fpclbm_init_fields(ens.h, *flat, on_device=1)
            ens.step(steps)
            out = [torch.full((ens.ncells,), np.nan, dtype=torch.float64, device="cuda") for _ in range(4)]
            F.fpclbm_moments(ens.h, *out, on_device=1)
            only = torch.full((ens.ncells,), np.nan, dtype=torch.float64, device="cuda")
            from ctypes import c_void_p
            assert F.load().fpclbm_moments(ens.h, None, None, c_void_p(only.data_ptr()), None, 1) == 0
            f = ens.get_populations()
        assert torch.equal(only, out[2])
        at = 0
        for d, tau, fl in zip(dims, taus, flds):
            n = d[0] * d[1] * d[2]
            with F.Lattice(*d, "fp32") as one:
                one.set_params(tau)
                one.set_force(1e-4, 0.0, -1e-4)
                one.init_fields(*fl)
                g = one.get_populations().reshape(27, -1)
                if steps == 0:
                    assert np.array_equal(f[:, at:at + n], g)
                one.set_populations(f[:, at:at + n])
                ref = one.moments()
            for a, b in zip(out, ref):
                assert np.max(np.abs(a[at:at + n].cpu().numpy() - b.ravel())) <= 1e-7
            at += n
