"""The variant of boxes too small to tune: one cell per thread until the step is longer than its latency,
later for odd rows and for the closed box, in the Smagorinsky mode as in the others; in the learned mode,
whose pairs evaluate the network twice, up to 2^19 cells in 16-bit storage.
"""
import numpy as np
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


@pytest.mark.parametrize("prec,shape,variant,minb", [
    ("fp32", (17, 15, 16), 0, 1), ("bf16", (32, 33, 32), 0, 1), ("fp32", (40, 41, 40), 0, 2), ("bf16", (80, 80, 80), 0, 2),
    ("fp16", (64, 64, 128), 2, 2), ("fp32", (100, 100, 100), 0, 2),
])
@pytest.mark.parametrize("bc", [0, 1])
def test_learned_variant(monkeypatch, prec, shape, variant, minb, bc):
    monkeypatch.delenv("FPCLBM_LAUNCH", raising=False)
    monkeypatch.delenv("FPCLBM_TUNE_CACHE", raising=False)
    with F.Lattice(*shape, prec, bc) as lat:
        lat.set_closure(np.zeros(4865, np.uint16))
        lat.set_params(0.6, 0.0, 2)
        lat.init_fields(*W.random_fields(*shape, 1, u_amp=0.02))
        lat.step(2)
        got = lat.launch()
        assert got["variant"] == variant and got["minb"] == minb
