"""The integer division and square root of the FP64 kernels (fp64_int.cuh) against
the built-in IEEE operations, bit for bit: random operands of ordinary and of
all exponents, quotients and roots next to a rounding boundary, exact ones,
significands next to 1 and 2, and the exponents at the ends of the fast path, in
both signs.  The routines without branches say where they do not apply; in the
ordinary range they must."""
from __future__ import annotations

import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_10983_gb300 import build  # noqa: E402

SOURCE = r"""
#include "fp64_int.cuh"
using namespace pic;
__device__ bool differ(double a, double b) {
  if (a != a && b != b) return false;
  return __double_as_longlong(a) != __double_as_longlong(b);
}
// out: wrong results of div_rn, sqrt_rn, div2_try, div_sqrt_try (quotients, root); then how often the last two apply
__global__ void check_kernel(const double* A, const double* B, const double* C, long long n, unsigned long long* out) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double a = A[i], b = B[i], c = C[i];
    if (differ(div_rn(a, b), a / b)) atomicAdd(out, 1ull);
    if (differ(sqrt_rn(a), sqrt(a))) atomicAdd(out + 1, 1ull);
    double q, qt, qu, g;
    if (div2_try(a, b, q)) {
      atomicAdd(out + 5, 1ull);
      // 2 a / b rounded once; where 2 a overflows, the quotient doubled (exact)
      const double r = isinf(2.0 * a) ? 2.0 * (a / b) : (2.0 * a) / b;
      if (differ(q, r)) atomicAdd(out + 2, 1ull);
    }
    if (div_sqrt_try<true>(b, c, a, qt, qu, g)) {
      atomicAdd(out + 6, 1ull);
      const double r = sqrt(a);
      if (differ(qt, b / r) || differ(qu, c / r)) atomicAdd(out + 3, 1ull);
      if (differ(g, r)) atomicAdd(out + 4, 1ull);
    }
  }
}
extern "C" int check(const double* a, const double* b, const double* c, long long n, unsigned long long* out) {
  check_kernel<<<1216, 256>>>(a, b, c, n, out);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    d = tmp_path_factory.mktemp("fp64_int")
    src, so = d / "check.cu", d / "check.so"
    src.write_text(SOURCE)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, "-shared", "-o", str(so), str(src), *build.GENCODE, "-O3", "-std=c++17", "-fmad=false",
                    "-Xcompiler", "-fPIC", "-cudart", "shared", "-I", build.CSRC, "-I", build.INCLUDE], check=True)
    lib = ctypes.CDLL(os.fspath(so))

    def run(a, b, c):
        a, b, c = (torch.as_tensor(v, dtype=torch.float64, device="cuda").contiguous() for v in (a, b, c))
        out = torch.zeros(7, dtype=torch.int64, device="cuda")
        P = ctypes.c_void_p
        assert lib.check(P(a.data_ptr()), P(b.data_ptr()), P(c.data_ptr()), ctypes.c_longlong(a.numel()),
                         P(out.data_ptr())) == 0
        out = out.tolist()
        assert out[:5] == [0] * 5, out
        return out[5], out[6]
    return run


def _bits(n, gen, lo, hi, signs=True):
    """Random significands, exponent fields in [lo, hi]."""
    m = torch.randint(0, 1 << 52, (n,), device="cuda", generator=gen)
    e = torch.randint(lo, hi + 1, (n,), device="cuda", generator=gen)
    s = torch.randint(0, 2, (n,), device="cuda", generator=gen) if signs else torch.zeros_like(e)
    return (m + (e << 52) + (s << 63)).view(torch.float64)


@pytest.mark.parametrize("seed", range(3))
def test_ordinary_operands(check, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = 1 << 23
    a, b, c = _bits(n, gen, 983, 1063, signs=False), _bits(n, gen, 983, 1063), _bits(n, gen, 983, 1063)
    assert check(a, b, c) == (n, n)


def test_all_exponents(check):
    gen = torch.Generator(device="cuda").manual_seed(9)
    n = 1 << 23
    check(_bits(n, gen, 0, 2047), _bits(n, gen, 0, 2047), _bits(n, gen, 0, 2047))


def test_near_a_rounding_boundary(check):
    """a / b and sqrt(a) within a 53-bit rounding of a number half-way between two
    53-bit ones, and exact squares and products."""
    rng = np.random.Generator(np.random.PCG64(1))
    a, b = [], []
    for _ in range(60000):
        half = (int(rng.integers(1 << 52, 1 << 53)) << 1) | 1  # 54 bits, odd
        d = int(rng.integers(1 << 52, 1 << 53))
        p = half * d
        shift = p.bit_length() - 53
        for q in (p >> shift, (p >> shift) + 1):
            a.append(float(q))
            b.append(float(d))
        r = half * half
        shift = (r.bit_length() - 53 + 1) & ~1  # an even power of two keeps the root's significand
        for q in (r >> shift, (r >> shift) + 1):
            if q.bit_length() <= 53:
                a.append(float(q))
                b.append(float(d))
        u, v = (int(t) for t in rng.integers(1 << 25, 1 << 26, 2))
        a += [float(u * u), float(u * v)]
        b += [float(u), float(v)]
    a, b = np.array(a), np.array(b)
    assert check(a, b, -b) == (a.size, a.size)
    assert check(a * 2.0, b, -a) == (a.size, a.size)  # the other parity of the exponent


def test_significands_and_exponents_at_the_ends(check):
    ulp = np.uint64(1)
    one, two = np.uint64(0), np.uint64(0xfffffffffffff)
    sig = np.array([one, one + ulp, one + ulp + ulp, two, two - ulp, np.uint64(1) << np.uint64(51)], dtype=np.uint64)
    exp = np.array([0, 1, 2, 3, 54, 55, 1021, 1022, 1023, 1024, 1025, 1992, 1993, 2044, 2045, 2046, 2047],
                   dtype=np.uint64)
    sgn = np.array([0, 1], dtype=np.uint64)
    v = (sig[:, None, None] | (exp[None, :, None] << np.uint64(52)) | (sgn[None, None, :] << np.uint64(63))).reshape(-1)
    v = v.view(np.float64)
    a, b = (t.reshape(-1) for t in np.meshgrid(v, v))
    check(a.copy(), b.copy(), b[::-1].copy())
