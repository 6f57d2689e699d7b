// Compares the fused AdamW epilogue's square root and quotient with the correctly rounded ones
// (compiled and called by test_gpu_arith.py).  bad[i] counts the operands of check i that differ.
#include <cuda_runtime.h>

#include "../paper_2406_14898_gb300/csrc/common.cuh"

namespace {

FL_DEV uint64_t mix(uint64_t z) {  // SplitMix64's finaliser (Steele, Lea & Flood 2014)
  z ^= z >> 30;
  z *= 0xBF58476D1CE4E5B9ull;
  z ^= z >> 27;
  z *= 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
FL_DEV bool same(float a, float b) { return a == b || (a != a && b != b); }
FL_DEV float pick(uint32_t h, int lo, int hi) {  // random sign and significand, exponent in [lo, hi]
  const uint32_t e = 127 + lo + (h >> 24) % (hi - lo + 1);
  return __uint_as_float((h & 0x80000000u) | (e << 23) | (h & 0x7fffffu));
}

// every significand and exponent parity, at the exponents 2 e; every subnormal
__global__ void sqrt_kernel(unsigned long long* bad) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;  // 2^24
  for (int e = -62; e <= 62; e += 4) {
    const float x = __uint_as_float((uint32_t(127 + 2 * e) << 23) + i);
    if (!same(sqrt_nr(x), __fsqrt_rn(x))) atomicAdd(bad + 0, 1ull);
  }
  const float x = __uint_as_float(i);  // subnormals and the smallest normal numbers
  if (!same(sqrt_nr(x), __fsqrt_rn(x))) atomicAdd(bad + 1, 1ull);
}
// the quotients nearest to a midpoint between two floats: for every odd 24-bit significand d and
// small odd r the q with (2 q + 1) d = r mod 2^25, and a = ((2 q + 1) d - r) / 2^25, at random scales
__global__ void div_hard_kernel(unsigned long long* bad) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;  // 2^22
  const uint32_t md = (1u << 23) | (2 * i + 1);
  uint32_t inv = md;
  for (int k = 0; k < 5; ++k) inv *= 2u - md * inv;  // modulo 2^32
  for (int r = -31; r <= 31; r += 2) {
    const uint32_t t = (uint32_t(r) * inv) & ((1u << 25) - 1);
    if (t < (1u << 24)) continue;
    const int64_t a = (int64_t(t) * md - r) >> 25;
    const uint32_t h = uint32_t(mix(uint64_t(i) * 64 + r + 32));
    const float fa = ldexpf(float(a), int(h % 70) - 80), fd = ldexpf(float(md), int((h >> 8) % 60) - 60);
    if (!same(div_nr(fa, fd), __fdiv_rn(fa, fd))) atomicAdd(bad + 2, 1ull);
  }
}
// random operands: |a| >= 2^-100 and a quotient in the normal range (3); else at most two ulps,
// or one step of 2^-149 (4): the residual may round to nothing there
__global__ void div_kernel(unsigned long long* bad) {
  const uint64_t n = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x;
  for (int k = 0; k < 64; ++k) {
    const uint64_t h = mix((n * 64 + k + 1) * 0x9E3779B97F4A7C15ull);
    float a = pick(uint32_t(h), -126, 126);
    const float d = fabsf(pick(uint32_t(h >> 32), -126, 124));
    if (k % 8 == 0) a = __uint_as_float(__float_as_uint(a) & 0x807fffffu);  // subnormal
    const float want = __fdiv_rn(a, d), got = div_nr(a, d), m = fabsf(want);
    if (fabsf(a) >= 0x1p-100f && m >= 0x1p-126f) {
      // (next to overflow the uncorrected quotient may be infinite already)
      if (!same(got, want) && !(m > 0x1.fffffcp127f)) atomicAdd(bad + 3, 1ull);
    } else if (!(fabsf(got - want) <= fmaxf(m * 0x1p-22f, 0x1p-149f))) {
      atomicAdd(bad + 4, 1ull);
    }
  }
}
__global__ void special_kernel(unsigned long long* bad) {
  const float inf = INFINITY, nan = nanf("");
  const float as[] = {0.f, -0.f, 1.f, -3.f, 0x1p-149f, 0x1p-130f, 0x1p126f, -inf, inf, nan, 3.4e38f, 1e-45f};
  const float ds[] = {0.f, 0x1p-126f, 0x1.000002p-126f, 0x1p-100f, 0x1.fffffep-101f, 1e-8f, 1.f, 0x1p125f, inf, nan};
  for (float a : as)
    for (float d : ds) {
      const float want = __fdiv_rn(a, d);
      const float got = div_nr(a, d);
      if (fabsf(a) >= 0x1p-100f || a == 0.f || a != a ? !same(got, want) && fabsf(want) >= 0x1p-126f
                                                      : !same(got, want) && !(fabsf(got - want) <= fabsf(want) * 0x1p-22f))
        atomicAdd(bad + 5, 1ull);
    }
  const float xs[] = {0.f, 0x1p-149f, 0x1p-126f, 0x1p-100f, 0x1.fffffep-101f, 0x1.000002p-100f, 3.4e38f, inf, nan, -1.f};
  for (float x : xs)
    if (!same(sqrt_nr(x), __fsqrt_rn(x))) atomicAdd(bad + 6, 1ull);
}

}  // namespace

extern "C" int arith_check(unsigned long long* bad_host, int n) {
  unsigned long long* bad = nullptr;
  cudaError_t e = cudaMalloc(&bad, n * sizeof *bad);
  if (e != cudaSuccess) return (int)e;
  cudaMemset(bad, 0, n * sizeof *bad);
  sqrt_kernel<<<(1 << 24) / 256, 256>>>(bad);
  div_hard_kernel<<<(1 << 22) / 256, 256>>>(bad);
  div_kernel<<<(1 << 22) / 256, 256>>>(bad);
  special_kernel<<<1, 1>>>(bad);
  e = cudaMemcpy(bad_host, bad, n * sizeof *bad, cudaMemcpyDeviceToHost);
  cudaFree(bad);
  return (int)e;
}
