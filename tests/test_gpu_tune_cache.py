"""The tuner's choices are kept by box class, in the process and in the file FPCLBM_TUNE_CACHE names.  A
row-staged choice (variant 3) holds for rows that bulk copies can move and whose tiles fit in shared
memory: boxes of the same cell count and other rows must tune for themselves, and step as before.

The files are written by hand (the tuner may not choose variant 3 by itself): the entries of both boxes
are replaced by a row-staged one for rows of at most 256 cells with three input stages.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# steps boxes of the given shapes one after the other; prints variant, block and stages of each, and
# whether the first one's state equals that of the paired variant, bit for bit
CODE = """
import os, sys
import numpy as np
import workloads as W
from paper_2410_09739_gb300 import fpclbm as F
prec, shapes = sys.argv[1], [tuple(map(int, s.split('x'))) for s in sys.argv[2:]]
for shape in shapes:
    f, states = W.random_fields(*shape, 1, u_amp=0.02), []
    for forced in (None, "128:2:2"):
        os.environ.pop("FPCLBM_LAUNCH", None)
        if forced: os.environ["FPCLBM_LAUNCH"] = forced
        with F.Lattice(*shape, prec) as lat:
            lat.set_params(0.7)
            lat.init_fields(*f)
            lat.step(2)
            if not forced: took = lat.launch()
            states.append(lat.get_state()[0].copy())
    print(took["variant"], took["block"], int(np.array_equal(*states)))
"""


def steps(cache, prec, *shapes):
    env = {k: v for k, v in os.environ.items() if k != "FPCLBM_LAUNCH"}
    r = subprocess.run([sys.executable, "-c", CODE, prec, *shapes], cwd=ROOT, capture_output=True, text=True,
                       env={**env, "FPCLBM_TUNE_CACHE": str(cache), "PYTHONPATH": ROOT})
    assert r.returncode == 0, r.stderr
    return [tuple(map(int, line.split())) for line in r.stdout.splitlines()]


@pytest.mark.parametrize("prec,staged,other", [
    ("fp32", "256x64x72", "512x64x36"),   # three stages of tiles of 512 fp32 cells: 276 KB
    ("bf16", "128x128x72", "130x126x72"),  # rows of 260 bytes
    ("bf16", "128x128x72", "129x128x72"),
])
def test_staged_choice_of_other_rows(tmp_path, prec, staged, other):
    cache = tmp_path / "choices"
    steps(cache, prec, staged, other)
    keys = [line.split()[0] for line in cache.read_text().splitlines()]
    assert len(keys) == 2  # a box class each
    # the entry of the staged box alone, then of both
    first = min(keys, key=len)
    for those in ([first], keys):
        cache.write_text("".join("%s 160 2 3 3\n" % k for k in those))
        (variant, block, _), (v2, _, equal2) = steps(cache, prec, staged, other)
        assert (variant, block) == (3, 160)
        assert v2 != 3 or prec == "fp32"  # rows of 512 fp32 cells can be staged, with two stages
        assert v2 != 3 or equal2


def test_staged_choice_reports_its_own_block(tmp_path):
    cache = tmp_path / "choices"
    steps(cache, "bf16", "384x64x48")
    key, = [line.split()[0] for line in cache.read_text().splitlines()]
    cache.write_text("%s 160 2 2 3\n" % key)
    assert steps(cache, "bf16", "384x64x48") == [(3, 224, 1)]
