"""The branch-free quotient, reciprocal and square root of the surrogate's Adam update, and the update with
its branch for values near the ends of the range, bit for bit against the IEEE operations (/ and sqrtf).

A kernel around csrc/surrogate_math.cuh, compiled here with the library's flags, counts the differences."""
import ctypes
import os
import subprocess

import pytest

from paper_2207_09431_gb300 import _build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "surrogate_math.cuh"
using namespace surr;
typedef unsigned long long u64;
__device__ unsigned next(u64 &s) {  // SplitMix64
  u64 z = (s += 0x9E3779B97F4A7C15ULL);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return (unsigned)((z ^ (z >> 31)) >> 16);
}
__device__ bool differ(float a, float b) { return !(a != a && b != b) && __float_as_int(a) != __float_as_int(b); }
// a float of either sign, exponent lo .. hi; one in four significands within 8 of 0 or of all ones
__device__ float draw(u64 &s, int lo, int hi) {
  const unsigned r = next(s), k = next(s);
  unsigned f = r & 0x7fffffu;
  if (k % 4 == 0) f = (k & 16) ? (r & 7u) : 0x7fffffu - (r & 7u);
  const unsigned e = (unsigned)(127 + lo + (int)(next(s) % (unsigned)(hi - lo + 1)));
  return __int_as_float((int)((r & 0x80000000u) | (e << 23) | f));
}
__global__ void all_reciprocals(u64 *bad) {  // every significand but the one with every bit set, exponents over the range
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (1 << 23) - 1) return;
  for (int e = -80; e < 80; e += 53) {
    const float b = ldexpf(__int_as_float(0x3f800000 + i), e);
    if (differ(reciprocal(b), 1.0f / b)) atomicAdd(bad, 1ull);
  }
}
__global__ void all_roots(u64 *bad) {  // two binades, at even exponents over the range
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  for (int e = -80; e < 80; e += 26) {
    const float x = ldexpf(__int_as_float(0x3f800000 + i), e);
    if (differ(square_root(x), sqrtf(x))) atomicAdd(bad, 1ull);
  }
  if (i == 0 && differ(square_root(0.0f), 0.0f)) atomicAdd(bad, 1ull);
}
__global__ void quotients(u64 *bad, int n) {
  u64 s = (u64)(blockIdx.x * blockDim.x + threadIdx.x) * 0x1234567ull + 7;
  for (int k = 0; k < n; ++k) {
    // dividends over the whole range that plain() accepts; divisors as the update has them, from eps = 1e-8 to the
    // root of its upper end, and bias corrections in [1e-4, 1]
    float a = draw(s, -80, 79), b = fabsf(draw(s, -27, 45)), c = fabsf(draw(s, -13, -1));
    if (k % 64 == 0) a = (k & 64) ? 0x1p-80f : -0x1p80f;
    if (k % 97 == 0) a = 0.0f;
    if ((__float_as_int(b) & 0x7fffff) != 0x7fffff && differ(quotient(a, b, reciprocal(b)), a / b)) atomicAdd(bad, 1ull);
    if (differ(quotient(a, c, 1.0f / c), a / c)) atomicAdd(bad, 1ull);
  }
}
template <int N>
__global__ void updates(u64 *bad, u64 *general, int n) {
  u64 s = (u64)(blockIdx.x * blockDim.x + threadIdx.x) * 0x7654321ull + 11;
  for (int k = 0; k < n; ++k) {
    float w[N], m[N], v[N], g[N], w0[N], m0[N], v0[N];
    const int kind = next(s) % 8, odd = next(s) % N;
    for (int i = 0; i < N; ++i) {
      w[i] = draw(s, -20, 5);
      m[i] = kind == 1 ? 0.0f : draw(s, -40, 10);
      v[i] = kind == 1 ? 0.0f : fabsf(draw(s, -60, 20));
      g[i] = kind == 2 ? 0.0f : draw(s, -30, 10);
    }
    // one parameter near and past the ends of the range, or not finite
    if (kind == 3) m[odd] = draw(s, -126, -70), g[odd] = draw(s, -126, -70);
    if (kind == 4) v[odd] = fabsf(draw(s, -126, -70)), g[odd] = draw(s, -63, -40);
    if (kind == 5) g[odd] = draw(s, 30, 127);
    if (kind == 6) v[odd] = fabsf(draw(s, 70, 127)), m[odd] = draw(s, 70, 127);
    if (kind == 7) (k & 1 ? g[odd] : m[odd]) = __int_as_float(k & 2 ? 0x7f800000 : 0x7fc00000);
    const float c1 = fabsf(draw(s, -4, -1)), c2 = fabsf(draw(s, -10, -1)), lr = 2e-3f, eps = 1e-8f;
    bool ok = true;
    for (int i = 0; i < N; ++i) {
      m0[i] = fmaf(1.f - 0.9f, g[i], __fmul_rn(0.9f, m[i]));
      v0[i] = fmaf(__fmul_rn(1.f - 0.999f, g[i]), g[i], __fmul_rn(0.999f, v[i]));
      w0[i] = __fsub_rn(w[i], __fdiv_rn(__fmul_rn(lr, __fdiv_rn(m0[i], c1)), __fadd_rn(__fsqrt_rn(__fdiv_rn(v0[i], c2)), eps)));
      ok = ok && plain(m0[i]) && plain(v0[i]);
    }
    adam(w, m, v, g, lr, 0.9f, 0.999f, c1, c2, 1.0f / c1, 1.0f / c2, eps);
    if (!ok) atomicAdd(general, 1ull);
    for (int i = 0; i < N; ++i)
      if (differ(w[i], w0[i]) || differ(m[i], m0[i]) || differ(v[i], v0[i])) atomicAdd(bad, 1ull);
  }
}
extern "C" int count(u64 *out) {  // differences: reciprocals, roots, quotients, updates of 4 and of 8; general branches
  u64 *d;
  if (cudaMalloc(&d, 8 * sizeof(u64)) != cudaSuccess) return 1;
  cudaMemset(d, 0, 8 * sizeof(u64));
  all_reciprocals<<<(1 << 23) / 256, 256>>>(d);
  all_roots<<<(1 << 24) / 256, 256>>>(d + 1);
  quotients<<<1216, 256>>>(d + 2, 2000);
  updates<4><<<608, 128>>>(d + 3, d + 5, 200);
  updates<8><<<608, 128>>>(d + 4, d + 5, 200);
  const cudaError_t e = cudaMemcpy(out, d, 8 * sizeof(u64), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
"""


def test_update_is_correctly_rounded(tmp_path):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    source, library = tmp_path / "math.cu", tmp_path / "math.so"
    source.write_text(SOURCE)
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", str(source), "-o", str(library)], check=True,
                   env={**os.environ, "TMPDIR": str(tmp_path)})
    out = (ctypes.c_ulonglong * 8)()
    assert ctypes.CDLL(str(library)).count(out) == 0
    reciprocals, roots, quotients, four, eight, general = list(out)[:6]
    assert (reciprocals, roots, quotients, four, eight) == (0, 0, 0, 0, 0)
    assert general > 1000  # the branch for values near the ends of the range was taken
