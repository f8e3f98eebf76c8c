"""The device's own scalar arithmetic against CUDA's: conversions between FP32
and FP64 on the integer pipe are bitwise the instructions' for every float and
for doubles on, beside and between all floats (ties, the range's edges,
subnormals, infinities, NaN); the step scalars' division is within one unit in
the last place of CUDA's.  (Its reciprocal is good to 2^-40 after one Newton
step on an estimate of 2^-20, so the corrected quotient is within 2^-79 of the
exact one before its rounding: the same rounding, or the other neighbour of a
near tie.)  Operands outside its range take CUDA's division itself."""
import ctypes

import pytest

from tests.cuda_unit import compile_cuda

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
#define FTGCR_THREADS 512
#include "ftgcr_band.cuh"
using namespace ftgcr;
typedef unsigned long long u64;
// every float bit pattern: widen, and narrow at the offsets of the 29 low bits
__global__ void k_conversions(u64* bad) {
  const u64 total = 1ull << 32;
  for (u64 q = blockIdx.x * (u64)blockDim.x + threadIdx.x; q < total; q += (u64)gridDim.x * blockDim.x) {
    const float f = __uint_as_float((unsigned)q);
    const double d = (double)f;
    if (__double_as_longlong(widen(f)) != __double_as_longlong(d)) atomicAdd(bad, 1ull);
    const u64 low[7] = {0ull, 1ull, 0xfffffffull, 0x10000000ull, 0x10000001ull, 0x1fffffffull, q * 0x9E3779B97F4A7C15ull >> 35};
    for (int i = 0; i < 7; ++i) {
      const double x = __longlong_as_double(__double_as_longlong(d) | (long long)(low[i] & 0x1fffffffull));
      if (__float_as_uint(narrow(x)) != __float_as_uint((float)x)) atomicAdd(bad + 1, 1ull);
    }
    // any double
    const double r = __longlong_as_double((long long)((q + 1) * 0xBF58476D1CE4E5B9ull ^ (q << 31)));
    if (__float_as_uint(narrow(r)) != __float_as_uint((float)r)) atomicAdd(bad + 1, 1ull);
  }
}
__global__ void k_division(const double* a, const double* b, long long n, long long* worst, u64* differ) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double q = quick_div(a[i], b[i]), e = a[i] / b[i];
    if (isnan(q) && isnan(e)) continue;
    const long long d = llabs(__double_as_longlong(q) - __double_as_longlong(e));
    if (d) atomicAdd(differ, 1ull);
    atomicMax(worst, d);
  }
}
extern "C" int conversions(u64* bad) {
  k_conversions<<<1520, 256>>>(bad);
  return (int)cudaDeviceSynchronize();
}
extern "C" int division(const double* a, const double* b, long long n, long long* worst, u64* differ) {
  k_division<<<1520, 256>>>(a, b, n, worst, differ);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def unit(tmp_path_factory):
    return compile_cuda(SOURCE, tmp_path_factory.mktemp("arithmetic"))


def test_conversions_are_the_instructions(unit):
    bad = torch.zeros(2, dtype=torch.int64, device="cuda")
    assert unit.conversions(ctypes.c_void_p(bad.data_ptr())) == 0
    assert bad.tolist() == [0, 0]


def _divide(unit, a, b):
    worst, differ = (torch.zeros(1, dtype=torch.int64, device="cuda") for _ in range(2))
    p = [ctypes.c_void_p(t.data_ptr()) for t in (a, b, worst, differ)]
    assert unit.division(p[0], p[1], ctypes.c_longlong(a.numel()), p[2], p[3]) == 0
    return worst.item(), differ.item()


def test_division_is_within_one_unit_in_the_last_place(unit):
    g = torch.Generator(device="cuda").manual_seed(5)
    n = 1 << 24

    def operands(lo, hi):  # binary exponents, both signs
        e = torch.randint(lo, hi, (n,), generator=g, device="cuda")
        m = 1 + torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
        s = 1.0 - 2.0 * torch.randint(0, 2, (n,), generator=g, device="cuda").double()
        return torch.ldexp(s * m, e)

    for lo, hi in ((-40, 40), (-422, 424), (-425, -418), (418, 426)):  # the fast path's range ends at -422 and 423
        assert _divide(unit, operands(lo, hi), operands(lo, hi))[0] <= 1, (lo, hi)
    # quotients next to 1 and 2, where a unit in the last place changes size
    b = operands(-3, 3)
    for f in (1.0, 2.0):
        for d in (-1, 0, 1):
            a = torch.ldexp((b * f).view(torch.int64).add(d).view(torch.float64), torch.zeros_like(b))
            assert _divide(unit, a, b)[0] <= 1


def test_division_outside_its_range_is_cudas(unit):
    inf, nan, tiny, huge = float("inf"), float("nan"), 5e-324, 1.7e308
    v = [0.0, -0.0, inf, -inf, nan, tiny, -tiny, 2.3e-308, huge, -huge, 1e-200, 1e200]
    inside = [1.0, -3.0, 2.0 ** -423, 2.0 ** 424]
    pairs = [(a, b) for a in v for b in v + inside] + [(a, b) for a in inside for b in v]
    pairs = [(a, b) for a, b in pairs if not (a == 0.0 and b in inside)]  # zero over an ordinary number: below
    a, b = (torch.tensor(c, dtype=torch.float64, device="cuda") for c in zip(*pairs))
    assert _divide(unit, a, b) == (0, 0)
    z, o = torch.zeros(4, dtype=torch.float64, device="cuda"), torch.tensor(inside, dtype=torch.float64, device="cuda")
    q = _divide(unit, z, o.abs())
    assert q == (0, 0)
