"""Field kernels at the edges of their arithmetic: 16-bit storage in 2D rounded once from the exact
equilibrium.
"""
import numpy as np
import pytest

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
