// FP64 numbers as sums of 8-bit digits for exact products on the tensor cores (the scheme of
// Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication", 2012).
//
// The numbers of one group (a column over 256 rows, or a row) share a power of two 2^e above
// their largest magnitude.  x becomes the whole number X = x 2^(55-e), |X| < 2^55, rounded to
// nearest (exact for every x within a factor of 4 of the group's binade), and X seven balanced
// digits, X = sum_k d_k 256^(6-k), -128 <= d_k <= 128.  A digit is exact in FP16, a product of two
// digits is a whole number of at most 2^14, and a sum of up to 2^10 such products is exact in the
// tensor core's FP32 accumulator, whatever the order.  Products with i + j <= 7 are kept: what is
// left out is below 2^-58 of the groups' largest product per term.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace lobpcg {
namespace slices {

constexpr int kSlices = 7;
constexpr int kDiags = 8;  // accumulators: i + j = 0 .. 7
// Groups whose biased exponent lies outside [kExpMin, kExpMax] (infinities and NaN among them)
// take the general kernels; all-zero groups use kExpOne.
constexpr int kExpMin = 1023 - 400, kExpMax = 1023 + 400, kExpOne = 1023;

// |x|'s high word for a maximum over a group; a subnormal with an empty high word counts as 1.
__device__ __forceinline__ uint32_t exp_key(double x) {
  const uint32_t hw = (uint32_t)__double2hiint(x) & 0x7fffffffu;
  return max(hw, (uint32_t)__double2loint(x) != 0u ? 1u : 0u);
}
// Biased exponent E of a group from the maximum of its keys (2^(E-1023) <= max < 2^(E-1022)), or
// -1 when the group is outside the range of the digits.
__device__ __forceinline__ int group_exp(uint32_t key) {
  if (key == 0u) return kExpOne;
  const int e = (int)(key >> 20);
  return e < kExpMin || e > kExpMax ? -1 : e;
}

// X + 0x0080808080808080 with 0x64 in the top byte: byte 6-k of the result is d_k + 128
// (a leading digit of 128 carries into the top byte).
__device__ __forceinline__ uint64_t digits(double x, int E) {
  const uint32_t hw = (uint32_t)__double2hiint(x), lw = (uint32_t)__double2loint(x);
  const uint32_t k = (uint32_t)(E - (int)((hw >> 20) & 0x7ffu));  // >= 0
  const uint64_t m = (uint64_t)((hw & 0xfffffu) | 0x100000u) << 32 | lw;
  uint64_t t;  // 2 |X|, cut; shr clamps, so zeros and subnormals shift out (E >= kExpMin)
  asm("shr.u64 %0, %1, %2;" : "=l"(t) : "l"(m << 3), "r"(k));
  const uint64_t neg = (uint64_t)(int64_t)((int32_t)hw >> 31);
  // X + bias = (t + 1 + 2 bias) / 2, or (-t + 2 bias) / 2 with -t = ~t + 1: rounding, sign and bias in one
  // addition
  return ((t ^ neg) + 0xc901010101010101ull) >> 1;
}

// (1024 + byte) - 1152 = byte - 128 in both halves, exact.
__device__ __forceinline__ uint32_t unbias(uint32_t r) {
  __half2 h = *reinterpret_cast<__half2*>(&r);
  h = __hsub2(h, __half2half2(__ushort_as_half(0x6480)));
  return *reinterpret_cast<uint32_t*>(&h);
}

// d[k]: the digits k of two numbers (a in the low half) as FP16.  A byte permute gathers two
// neighbouring digits of both numbers, a second one per digit sets 0x64 above each (1024 + byte).
__device__ __forceinline__ void digit_pairs(uint64_t a, uint64_t b, uint32_t (&d)[kSlices]) {
  constexpr uint32_t c = 0x64646464u;
  const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
  // bytes 7 and 6 are 0x64 (0x65 where the leading digit is 128) and the digit already
  d[0] = unbias(__byte_perm(ah, bh, 0x7632));
  uint32_t q = __byte_perm(ah, bh, 0x5410);  // bytes 4, 5 of a, then of b
  d[1] = unbias(__byte_perm(q, c, 0x4341));
  d[2] = unbias(__byte_perm(q, c, 0x4240));
  q = __byte_perm(al, bl, 0x7632);  // bytes 2, 3
  d[3] = unbias(__byte_perm(q, c, 0x4341));
  d[4] = unbias(__byte_perm(q, c, 0x4240));
  q = __byte_perm(al, bl, 0x5410);  // bytes 0, 1
  d[5] = unbias(__byte_perm(q, c, 0x4341));
  d[6] = unbias(__byte_perm(q, c, 0x4240));
}

// The digits of eight numbers, 16 bytes per digit, `step` bytes apart at o.
__device__ __forceinline__ void put_digits(const uint64_t (&w)[8], unsigned char* o, uint32_t step) {
  uint32_t d[4][kSlices];
#pragma unroll
  for (int i = 0; i < 4; ++i) digit_pairs(w[2 * i], w[2 * i + 1], d[i]);
#pragma unroll
  for (int k = 0; k < kSlices; ++k)
    *reinterpret_cast<uint4*>(o + k * step) = make_uint4(d[0][k], d[1][k], d[2][k], d[3][k]);
}

// sum_t v_t 256^(7-t) of eight whole FP32 numbers |v_t| <= 2^24, times 2^s, rounded to FP64 with
// integer operations only (an FP64 instruction takes 64 times the issue slots of an integer one) and
// without branches, so that the joins of several elements overlap.
__device__ __forceinline__ double join(const float (&v)[kDiags], int s) {
  auto i = [&](int t) { return __float2int_rn(v[t]); };
  int64_t hi = (int64_t)i(0) * (1 << 24) + ((int64_t)i(1) * (1 << 16) + ((int64_t)i(2) * (1 << 8) + i(3)));
  const int64_t lo = (int64_t)i(4) * (1 << 24) + ((int64_t)i(5) * (1 << 16) + ((int64_t)i(6) * (1 << 8) + i(7)));
  hi += lo >> 32;  // the sum is hi 2^32 + (low word of lo)
  const uint32_t neg = (uint32_t)(hi >> 63);
  // magnitude in three words: complement, plus one where negative
  uint32_t w0 = (uint32_t)lo ^ neg;
  uint64_t h = (uint64_t)hi ^ ((uint64_t)neg << 32 | neg);
  w0 -= neg;
  h += (neg & 1u) & (w0 == 0u ? 1u : 0u);
  uint32_t w2 = (uint32_t)(h >> 32), w1 = (uint32_t)h;
  int e = 1022 + 95 + s;  // biased exponent of the top bit of w2, less one for the implicit bit
  if (w2 == 0u) w2 = w1, w1 = w0, w0 = 0u, e -= 32;
  if (w2 == 0u) w2 = w1, w1 = w0, w0 = 0u, e -= 32;
  const int n = __clz((int)w2);
  const uint32_t m1 = __funnelshift_l(w1, w2, n), m0 = __funnelshift_l(w0, w1, n);
  const uint64_t m = (uint64_t)m1 << 32 | m0;
  const uint64_t bits = ((uint64_t)((uint32_t)(e - n) + (neg << 11)) << 52) + (m >> 11) + ((m0 >> 10) & 1u);
  return __longlong_as_double(w2 ? (long long)bits : 0ll);
}

}  // namespace slices
}  // namespace lobpcg
