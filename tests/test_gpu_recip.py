"""The short reciprocal of the density (recip_newton, csrc/pair.cuh) against CUDA's correctly rounded
one for every fp32 argument that is not subnormal and whose reciprocal is not: all bits, infinities,
zeros and NaN included; in the packed form finite arguments from 0 to 1e30, the densities of a run
that has not diverged.  And what rests on it: with general rates the
row-staged kernel (CUDA's reciprocal) and the paired one (the short one) store the same bits at
densities next to 1, where a reciprocal lies next to the middle of two fp32 values.
"""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2410_09739_gb300 import build as B
from paper_2410_09739_gb300 import fpclbm as F

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "pair.cuh"
// out[0]: arguments whose bits differ, out[1], out[2]: the bits of one such argument and result
__global__ void check(unsigned* out)
{
    for (unsigned long long i = blockIdx.x * blockDim.x + threadIdx.x; i < (1ull << 32); i += gridDim.x * blockDim.x) {
        const unsigned b = (unsigned)i, e = (b >> 23) & 255u;
        const bool zero = (b & 0x7fffffffu) == 0u, finite = e < 255u;
        if ((e == 0u && !zero) || (finite && (b & 0x7fffffffu) > 0x7e800000u)) continue;  // subnormal, or above 2^126
        const float a = __uint_as_float(b), want = __frcp_rn(a);
        const float one = fpc::recip_newton(a);
        const fpc::f2 two = fpc::recip_newton(fpc::f2(a, 1.f)), other = fpc::recip_newton(fpc::f2(1.f, a));
        const float got[3] = {one, two.v.x, other.v.y};
        const bool flagged = finite && !zero && !(a > 0.f && a < 1e30f);
        for (int k = 0; k < (flagged ? 1 : 3); ++k)
            if (__float_as_uint(got[k]) != __float_as_uint(want) && !(isnan(got[k]) && isnan(want))) {
                atomicAdd(out, 1u);
                out[1] = b;
                out[2] = __float_as_uint(got[k]);
            }
        if (two.v.y != 1.f || other.v.x != 1.f) atomicAdd(out, 1u);
    }
}
extern "C" int run(unsigned* host)
{
    unsigned* d;
    if (cudaMalloc(&d, 12) != cudaSuccess || cudaMemset(d, 0, 12) != cudaSuccess) return 1;
    check<<<152 * 8, 256>>>(d);
    const int e = cudaMemcpy(host, d, 12, cudaMemcpyDeviceToHost) != cudaSuccess;
    cudaFree(d);
    return e;
}
"""


def test_every_argument(tmp_path):
    src, lib = tmp_path / "recip.cu", tmp_path / "recip.so"
    src.write_text(SOURCE)
    subprocess.run([B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-Xcompiler", "-fvisibility=default", "-shared", str(src), "-o",
                    str(lib)], check=True, capture_output=True)
    out = np.zeros(3, np.uint32)
    assert ctypes.CDLL(str(lib)).run(out.ctypes.data_as(ctypes.c_void_p)) == 0
    assert out[0] == 0, [hex(v) for v in out]


@pytest.mark.parametrize("prec", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("bc", [0, 1])
def test_staged_equals_paired_next_to_density_one(monkeypatch, prec, bc):
    """Densities 1 - k 2^-24, k = -8 .. 8, moving, as the state that an odd step reads."""
    nx, ny, nz = 64, 16, 8
    rng = np.random.default_rng(3)
    rho = 1.0 - rng.integers(-8, 9, (nz, ny, nx)) * 2.0 ** -24
    u = 0.05 * rng.uniform(-1, 1, (3, nz, ny, nx))
    states = []
    for variant in ("128:2:3", "128:2:2"):
        monkeypatch.setenv("FPCLBM_LAUNCH", variant)
        with F.Lattice(nx, ny, nz, prec, bc) as lat:
            lat.set_params(0.6, 0.3)
            lat.init_fields(rho, *u)
            raw, _ = lat.get_state()
            got = []
            for at in (0, 1):
                lat.set_state(raw, at)
                lat.step(1)
                got.append(lat.get_state()[0].copy())
            assert lat.launch()["variant"] == int(variant[-1])
            states.append(got)
    for a, b in zip(*states):
        assert np.array_equal(a, b)
