"""The odd step of neighbouring cells with a force along x in 16-bit storage runs five blocks per SM where
the populations do not stay in L2, four otherwise: the same arithmetic, so a large box made of copies of
a small one along x and z holds the small one's populations bit for bit.
"""
import numpy as np
import pytest

import workloads as W
from paper_2410_09739_gb300 import fpclbm as F

pytestmark = pytest.mark.gpu


def advance(fields, shape, prec, bc, mode):
    with F.Lattice(*shape, prec, bc) as lat:
        lat.set_params(0.6, 0.0, mode)
        lat.set_force(3e-4)
        lat.init_fields(*(a.reshape(-1) for a in fields))
        lat.step(3)
        assert lat.launch()["variant"] == 2
        raw = lat.get_state()[0]
    nx, ny, nz = shape
    return raw.view(np.uint16).reshape(27, -1)[:, :nx * ny * nz].reshape(27, nz, ny, nx)


@pytest.mark.parametrize("prec", ["fp16", "bf16"])
@pytest.mark.parametrize("bc", [0, 1, 3])
@pytest.mark.parametrize("mode", [0, 1])
def test_large_box_of_copies(monkeypatch, prec, bc, mode):
    monkeypatch.setenv("FPCLBM_LAUNCH", "128:2:2")
    nx, ny, nz, cx, cz = 34, 24, 13, 15, 16  # 2,545,920 cells: 137 MB
    small = [a.reshape(nz, ny, nx) for a in W.random_fields(nx, ny, nz, 5, u_amp=0.05)]
    one = advance(small, (nx, ny, nz), prec, bc, mode)
    many = advance([np.tile(a, (cz, 1, cx)) for a in small], (nx * cx, ny, nz * cz), prec, bc, mode)
    assert np.array_equal(many, np.tile(one, (1, cz, 1, cx)))
