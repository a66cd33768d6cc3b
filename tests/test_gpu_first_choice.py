"""The variant of boxes too small to tune: one cell per thread until the step is longer than its latency,
later for odd rows and for the closed box, in the Smagorinsky mode as in the others.
"""
import pytest

import workloads as W
from paper_2410_09739_gb300 import fpclbm as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc,diffusion,shape,variant", [
    (0, 0, (40, 40, 40), 0), (0, 0, (64, 32, 32), 2), (1, 1, (45, 37, 53), 0), (1, 1, (65, 64, 64), 2),
    (2, 0, (44, 46, 45), 0), (2, 0, (48, 64, 32), 2), (2, 1, (45, 46, 64), 0), (2, 1, (65, 64, 64), 2),
    (1, 3, (8, 8, 8), 0), (3, 3, (40, 40, 40), 0), (3, 3, (64, 32, 32), 2), (0, 3, (45, 37, 53), 0), (1, 3, (65, 64, 64), 2),
])
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_variant(monkeypatch, prec, bc, diffusion, shape, variant):
    monkeypatch.delenv("FPCLBM_LAUNCH", raising=False)
    monkeypatch.delenv("FPCLBM_TUNE_CACHE", raising=False)
    with F.Lattice(*shape, prec, bc) as lat:
        lat.set_params(0.6, 0.0, diffusion)
        if bc == 2:
            lat.set_wall_velocity(0.01)
        if diffusion == 3:
            lat.set_smagorinsky(0.1, 0.005, 26.0)
            lat.set_force(1e-5)
        lat.init_fields(*W.random_fields(*shape, 1, u_amp=0.02))
        lat.step(2)
        assert lat.launch()["variant"] == variant
