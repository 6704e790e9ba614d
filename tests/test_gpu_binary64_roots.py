"""The binary64 reciprocal and roots of the equation of state (lbpc_device.cuh): third-order steps from the hardware's
approximations, against the exact values over their range, and the special values of psi.

The bounds follow from the steps. The approximations see and give the upper 32 bits of a binary64 number (20 of the
significand), so they are off by two truncations of 2^-20 and their own error: |e| <= 2^-18 for the reciprocal's
residual 1 - x r and for the root's 1 - x y^2, which the test checks first. What a step leaves is e^3 <= 2^-54 for the
reciprocal and 5/16 e^3 <= 2^-55.6 for the roots, where an ulp is 2^-53 or more. With the last operation's rounding
(half an ulp) the reciprocal is within 1 ulp. The roots also carry half the rounding of s = x y: a quarter of an ulp of
sqrt(x), which has the size of s, up to half an ulp of 1/sqrt(x): 1 and 1.25 ulp."""

import math
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <stdio.h>
#include <vector>
#include "lbpc_device.cuh"
using namespace lbpc;
__global__ void k(const double* x, int n, double* out) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  double r, y, ir, rt;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x[i]));
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x[i]));
  roots_of(x[i], ir, rt);
  double* o = out + 6 * (long long)i;
  o[0] = r, o[1] = y, o[2] = inverse_of(x[i]), o[3] = rt, o[4] = ir, o[5] = psi_of(x[i]);
}
int main(int argc, char** argv) {
  FILE* f = fopen(argv[1], "rb");
  fseek(f, 0, SEEK_END);
  const int n = (int)(ftell(f) / 8);
  rewind(f);
  std::vector<double> x(n), o(6 * (size_t)n);
  if (fread(x.data(), 8, n, f) != (size_t)n) return 1;
  fclose(f);
  double *dx, *d;
  if (cudaMalloc(&dx, 8 * n) || cudaMalloc(&d, 48 * n)) return 2;
  cudaMemcpy(dx, x.data(), 8 * n, cudaMemcpyHostToDevice);
  k<<<(n + 255) / 256, 256>>>(dx, n, d);
  if (cudaMemcpy(o.data(), d, 48 * n, cudaMemcpyDeviceToHost)) return 3;
  f = fopen(argv[2], "wb");
  fwrite(o.data(), 8, 6 * (size_t)n, f);
  fclose(f);
  return 0;
}
"""


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = tmp_path_factory.mktemp("roots")
    (d / "t.cu").write_text(PROGRAM)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-I",
                    os.path.join(ROOT, "paper_1709_04400_gb300", "csrc"), "-o", str(d / "t"), str(d / "t.cu")], check=True)

    def run(x):
        np.asarray(x, dtype=np.float64).tofile(d / "in")
        subprocess.run([str(d / "t"), str(d / "in"), str(d / "out")], check=True, timeout=60)
        return np.fromfile(d / "out", dtype=np.float64).reshape(-1, 6)

    return run


def _arguments():
    """Exponents from 2^-1000 to 2^1000, odd and even, with significands at the ends, with all low 32 bits set (which
    the approximations do not see), and random."""
    rng = np.random.RandomState(5)
    exps = np.concatenate([np.arange(-6, 7), rng.randint(-1000, 1000, 400)])
    low = (1 << 32) - 1
    out = []
    for e in exps:
        bits = [0, 1, low, (1 << 52) - 1, ((1 << 20) - 2) << 32, (((1 << 20) - 2) << 32) | low]
        bits += [(int(b) << 32) | low for b in rng.randint(0, 1 << 20, 8)]
        bits += [int(b) for b in rng.randint(0, 1 << 52, 16)]
        out += [math.ldexp(1.0 + b / 2.0**52, int(e)) for b in bits]
    return out


def test_within_their_bounds(evaluate):
    x = _arguments()
    worst = [0.0] * 5
    for v, (r, y, inv, root, inv_root, psi) in zip(x, evaluate(x).tolist()):
        X, I, S, Q = Fraction(v), Fraction(inv), Fraction(root), Fraction(inv_root)
        err = (abs(1 - X * Fraction(r)), abs(1 - X * Fraction(y) ** 2),  # residuals of the approximations
               abs(I - 1 / X) / Fraction(math.ulp(inv)),
               # to first order in the error, whose square is below 2^-100
               abs(S * S - X) / (2 * S) / Fraction(math.ulp(root)),
               abs(1 - X * Q * Q) / 2 * Q / Fraction(math.ulp(inv_root)))
        worst = [max(a, float(b)) for a, b in zip(worst, err)]
        assert psi == root
    print("residuals 2^%.2f, 2^%.2f; ulp: 1/x %.3f, sqrt %.3f, 1/sqrt %.3f" % (*map(math.log2, worst[:2]), *worst[2:]))
    assert max(worst[:2]) <= 2.0**-18
    assert worst[2] <= 1.0 and worst[3] <= 1.0 and worst[4] <= 1.25


def test_special_values_of_psi(evaluate):
    """psi = sqrt(max(psi^2, 0)), a NaN and a subnormal number counting as 0."""
    tiny = np.finfo(np.float64).tiny
    x = [0.0, -0.0, -1.0, -tiny, -math.inf, math.nan, -math.nan, 5e-324, tiny * (1 - 2.0**-52), math.inf]
    assert evaluate(x)[:, 5].tolist() == [0.0] * 9 + [math.inf]
    x = [tiny, tiny * (1 + 2.0**-52), 4 * tiny, float(np.finfo(np.float64).max)]
    for v, psi in zip(x, evaluate(x)[:, 5].tolist()):
        assert abs(psi - math.sqrt(v)) <= math.ulp(psi)
