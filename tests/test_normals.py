"""The normals of the sparse part-step (psgld_normals.cuh), at every value
that their uniforms take: compiled for the host, where each operation rounds
as on the device, and held to FP64 by the accuracy of the same formula
through logf, sqrtf and sincospif: relative error of a normal at most 2.1e-7,
4.6e-8 rms.  On the GPU, through a chain without data whose step is the noise
itself, against the oracle's FP64 normals of the same Philox words."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from paper_1506_01418_gb300 import psgld as P

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_01418_gb300", "csrc")
MAX, RMS = 2.1e-7, 4.6e-8

MAIN = r"""
#include "psgld_normals.cuh"
// Relative errors of both normals of u0 = (m + 1/2) 2^-23, u1 = (n + 1/2) 2^-23
// as either pair of a call: the largest, and the sum of squares.
static void one(uint32_t m, uint32_t n, double *worst, double *sum)
{
    const double r = sqrt(-2.0 * log((m + 0.5) / 8388608.0));
    const double turn = (n + 0.5) / 8388608.0;
    const int quarter = (int)(4.0 * turn + 0.5);                 // nearest; the rest is exact
    const double a = 2.0 * M_PI * (turn - 0.25 * quarter), s = sin(a), c = cos(a);
    const double cs[4] = {c, -s, -c, s}, sn[4] = {s, c, -s, -c};
    const double want[2] = {r * cs[quarter & 3], r * sn[quarter & 3]};
    const uint32_t low = (m * 2654435761u) >> 23;                // bits below the uniform's do not count
    const uint4 w = {m << 9 | low, n << 9 | (low ^ 511u), m << 9, n << 9 | 511u};
    const float4 z = psgld::dev::normals4(w);
    const double got[4] = {z.x, z.y, z.z, z.w};
    for (int k = 0; k < 4; ++k) {
        const double e = fabs(got[k] - want[k & 1]) / fabs(want[k & 1]);
        if (!(e <= *worst)) *worst = e;
        *sum += e * e;
    }
}
// every m, each with another n (or, swapped, every n, each with another m)
extern "C" void sweep(uint32_t mul, uint32_t add, int swap, double *worst, double *sum)
{
    for (uint32_t k = 0; k < 8388608u; ++k) {
        const uint32_t o = (k * mul + add) & 8388607u;
        if (swap) one(o, k, worst, sum);
        else one(k, o, worst, sum);
    }
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    gxx, nvcc = shutil.which("g++"), shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if gxx is None or not os.path.exists(os.path.join(inc, "vector_types.h")):
        pytest.skip("no host compiler or CUDA headers")
    d = tmp_path_factory.mktemp("normals")
    (d / "main.cpp").write_text(MAIN)
    # -ffp-contract=off: a product and a sum of the header stay two operations
    subprocess.run([gxx, "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, "-I", inc,
                    str(d / "main.cpp"), "-o", str(d / "main.so")], check=True)
    return C.CDLL(str(d / "main.so"))


# every u0, each with another u1; every u1 (all quarter turns' edges), each
# with another u0; every u1 with one u0: the smallest, the largest, one half
@pytest.mark.parametrize("mul,add,swap", [(2654435761, 12345, 0), (40503, 77, 1), (0, 0, 1), (0, 8388607, 1),
                                          (0, 4194304, 1), (0, 5931641, 1), (0, 5931642, 1)])
def test_normals_at_every_uniform(host, mul, add, swap):
    worst, total = C.c_double(0.0), C.c_double(0.0)
    host.sweep(C.c_uint32(mul), C.c_uint32(add), swap, C.byref(worst), C.byref(total))
    rms = (total.value / (4 * 2 ** 23)) ** 0.5
    print(f"largest {worst.value:.3e} rms {rms:.3e}")
    assert worst.value <= MAX
    if mul:   # one u0 alone shares its radius's error among all its normals
        assert rms <= RMS


@pytest.mark.gpu
@pytest.mark.parametrize("I,K", [(36000, 50), (400000, 8), (150000, 16)])   # by rows, by rows, by units
def test_noise_of_a_step_matches_fp64(I, K):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    J, seed, empty = 2000, 77, np.zeros(0, np.int32)
    ch = P.PSGLD(I, J, K, 1, 0.0, 1.0, prior_kind=P.PSGLD_PRIOR_GAUSSIAN, seed=seed, eps=0.5)
    ch.set_data_coo(empty, empty, np.zeros(0, np.float32))
    ch.set_factors(np.zeros((I, K), np.float32), np.zeros((J, K), np.float32))
    ch.part_step(1)                       # x = 0 + 0.5 (0 + 0) + sqrt(2 0.5) z
    got = [x.cpu().numpy().astype(np.float64) for x in ch.get_factors()]
    ch.close()
    for mat, z in enumerate(got):
        want = oracle.noise_matrix(seed, 1, mat, z.shape[0], K)
        e = np.abs(z - want) / np.abs(want)
        assert e.max() <= MAX and np.sqrt(np.mean(e * e)) <= RMS
