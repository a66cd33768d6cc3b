"""Field kernels at the edges of their arithmetic: 16-bit storage in 2D rounded once from the exact
equilibrium; infinite, huge and vanishing densities, which the sums of fp32 pairs leave to fp64.
"""
import numpy as np
import pytest

import oracle as O
from paper_2410_09739_gb300 import fpclbm as F

pytestmark = pytest.mark.gpu

W1 = np.array([1 / 6, 2 / 3, 1 / 6])
EX2, EY2 = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1]), np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])
W2 = (W1[EX2 + 1] * W1[EY2 + 1])[:, None, None]
BITS = {"fp16": 11, "bf16": 8}
LOWEST = {"fp16": -24, "bf16": -133}  # exponent of the smallest subnormal


def rounded(x, prec):
    """x (fp64) to the storage type, half to even, and where x lies within 2^-30 of a spacing of a tie."""
    _, e = np.frexp(x)
    unit = np.exp2(np.maximum(e - BITS[prec], LOWEST[prec]).astype(np.float64))
    q = x / unit
    return np.rint(q) * unit, np.abs(np.abs(q - np.floor(q)) - 0.5) < 2.0 ** -30


@pytest.mark.parametrize("prec", ["fp16", "bf16"])
@pytest.mark.parametrize("amp", [0.1, 1e-3])
def test_init_2d_16_bit_rounds_once(prec, amp):
    """512 x 512 cells x 9: one in 2^13 (fp16) or 2^16 (bf16) values lies so near a tie that rounding
    to fp32 first would move it there."""
    n = 512
    rng = np.random.default_rng(11)
    rho = 1.0 + 0.3 * amp * rng.uniform(-1, 1, (n, n))
    ux, uy = amp * rng.uniform(-1, 1, (2, n, n))
    with F.Lattice2D(n, n, prec) as lat:
        lat.init_fields(rho, ux, uy)
        got, _ = rounded(lat.get_populations() - W2, prec)  # the weights leave errors of 1e-16: far below a spacing
    d = [[0.5 * (v * v - v), -v * v, 0.5 * (v * v + v)] for v in (ux, uy)]
    for a in range(9):
        A, B, p, q = W1[EX2[a] + 1], W1[EY2[a] + 1], d[0][EX2[a] + 1], d[1][EY2[a] + 1]
        want, tie = rounded((rho - 1) * ((A + p) * (B + q)) + (p * (B + q) + A * q), prec)
        assert np.array_equal(got[a][~tie], want[~tie]), a
        assert np.mean(tie) < 1e-6


def same(a, b, rtol):
    """Equal up to rtol, and infinite or NaN in the same places."""
    with np.errstate(invalid="ignore"):
        near = np.abs(a - b) <= rtol * np.abs(b)
    return np.all((np.isnan(a) & np.isnan(b)) | (a == b) | near)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("box", [False, True])
@pytest.mark.parametrize("force", [False, True])
def test_moments_2d_of_extreme_cells(prec, box, force):
    """Infinite, NaN, huge and cancelling populations and a density of exactly zero: what fp64 sums and
    divisions give; ordinary neighbours to the bound of test_moments_2d_are_fp64_sums."""
    big = 2.0 ** 127
    w = W2[:, 0, 0]
    f = np.tile(W2, (1, 3, 4))
    f[0, 0, 0] = np.inf
    f[1, 0, 1] = -np.inf
    f[5, 0, 2] = np.inf
    f[6, 0, 2] = -np.inf
    f[2, 0, 3] = np.nan
    f[1, 1, 0] = f[2, 1, 0] = big            # the sum leaves fp32
    f[1, 1, 1], f[3, 1, 1], f[5, 1, 1] = big, big, -big
    f[0, 1, 2] = w[0] - 1.25                # density 0, momentum (0.25, 0)
    f[1, 1, 2] = w[1] + 0.25
    f[0, 1, 3] = w[0] - 1.0                 # density 0 at rest
    f[3, 2, 0] += 0.125
    f[:, 2, 1] *= 1.0 + 2.0 ** -6
    F0 = (2.0 ** -8, -2.0 ** -9) if force else (0.0, 0.0)
    with F.Lattice2D(4, 3, prec) as lat:
        lat.set_params(0.7)
        lat.set_force(*F0)
        if box:
            lat.set_boundary(F.FPCLBM_BC_BOX, 0.0)
        lat.set_populations(f)
        got = lat.moments()
        g = lat.get_populations() - W2       # the stored deviations
    with np.errstate(all="ignore"):
        rho = 1.0 + g.sum(0)
        # a product with a zero component is NaN for an infinite population, as in the fp64 kernel
        j = [(e[:, None, None] * g).sum(0) + 0.5 * Fk for e, Fk in zip((EX2, EY2), F0)]
        ref = [rho, j[0] / rho, j[1] / rho]
    # densities of exactly zero: the stored deviations -1 - 0.25 + 0.25 have no rounding error
    ref[0][1, 2:4] = 0.0
    with np.errstate(all="ignore"):
        ref[1][1, 2], ref[2][1, 2] = (0.25 + 0.5 * F0[0]) / np.float64(0.0), 0.5 * F0[1] / np.float64(0.0)
        ref[1][1, 3], ref[2][1, 3] = (0.5 * np.array(F0)) / np.float64(0.0)
    for x, y in zip(got, ref):
        assert same(x[:2], y[:2], 1e-14), (x, y)
        assert np.max(np.abs(x[2] - y[2])) <= 2e-15


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("r", [2, 3])
def test_sample_of_extreme_cells(prec, r):
    """Coarse cells that hold one infinite population (density infinite, velocity NaN), two huge ones
    whose sum leaves fp32, and a density of exactly zero moving along +x, as fp64 gives them; coarse
    cells with no such cell next to them stay finite."""
    n, big = 8 * r, 2.0 ** 127
    f = O.init_equilibrium(np.ones((n, n, n)), *(0.02 * np.random.default_rng(5).uniform(-1, 1, (3, n, n, n))))
    e = O.velocity_set()
    w = W1[e[:, 0] + 1] * W1[e[:, 1] + 1] * W1[e[:, 2] + 1]
    at = {tuple(int(c) for c in v): a for a, v in enumerate(e)}
    rest, east = at[(0, 0, 0)], at[(1, 0, 0)]
    f[rest, 0, 0, 0] = np.inf
    f[rest, 0, 0, 3 * r] = f[east, 0, 0, 3 * r] = big
    f[:, 0, 4 * r, 0] = w
    f[rest, 0, 4 * r, 0] -= 1.25
    f[east, 0, 4 * r, 0] += 0.25
    with F.Lattice(n, n, n, prec) as lat:
        lat.set_params(0.6)
        lat.set_populations(f)
        X, T = np.empty((512, 9), np.float32), np.empty(512, np.float32)
        F.fpclbm_closure_sample(lat.h, r, 0.55, X, T)
    X = X.reshape(8, 8, 8, 9)
    assert np.all(np.isinf(X[0, 0, 0, :6])) and np.all(np.isnan(X[0, 0, 0, 6:]))
    # density 2^128 + 1, momentum 2^127 along x: velocity 1/2 there, a mean of 1 / (2 r^3) and noise
    assert np.all(np.isinf(X[0, 0, 3, :6]) | (np.abs(X[0, 0, 3, :6]) > 1e30))
    assert abs(X[0, 0, 3, 6] - 0.5 / r ** 3) < 0.02 and np.all(np.abs(X[0, 0, 3, 7:]) < 0.02)
    assert X[0, 4, 0, 6] == np.inf
    assert np.all(np.isfinite(X[2:7]))
