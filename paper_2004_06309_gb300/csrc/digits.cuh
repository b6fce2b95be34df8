// Products of complex128 values on the tensor cores, by splitting the operands into digits whose
// products and sums are exact (Ozaki, Ogita, Oishi, Rump, Numer. Algorithms 59, 2012).
//
// A double x of a group whose largest exponent field is E becomes the integer
// D = x 2^(1084 - E), |D| < 2^62 (its lower bits are cut off), written as eight balanced base-256
// digits in [-128, 127] with 128 added to each (so a byte of the 64-bit word is a digit).
// mma.sync m16n8k16 multiplies digits as f16 and adds in f32: a product is at most 2^14, and while at
// most 2^10 of them meet in one accumulator (8 digit pairs x 128 columns), every sum is below 2^24
// and exact.
//
// Error: D keeps all 53 bits of a value down to 2^-9 of its group's largest, and fewer below; with the
// digit pairs left out a sum of n products is within about 2^-59 sqrt(n) of the product of the two
// groups' largest entries.  FP64 sums are within 2^-53 of the sum of the terms' magnitudes.  So the
// digits are the better ones while the terms reach 2^-6 of that product, as they do for matrices scaled to
// a diagonal of order one (launch_scaling) and vectors of like entries; the sweeps go back to the FP64
// units for sums far below it (sweeps64.cu, kGuardBits).
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace hz {

constexpr int kBias = 1084;               // D = x 2^(kBias - E)
constexpr uint64_t kDigitBias = 0x8080808080808080ull;
constexpr uint32_t kZeroWord = 0x80808080u;

__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// digits (with 128 added to each) of x, with x < 2^(E - 1022) for the largest exponent field E
// of its group; sh = 1 + E - max(exponent field of x, 1)
__device__ __forceinline__ uint64_t to_digits(double x, int sh) {
  const int hi = __double2hiint(x);
  const uint32_t top = (uint32_t(hi) & 0xfffffu) | (((hi >> 20) & 0x7ff) ? 0x100000u : 0u);
  const uint64_t m = ((uint64_t(top) << 32) | uint32_t(__double2loint(x))) << 10;
  const uint64_t d = m >> min(sh, 63);
  return (hi < 0 ? ~d + 1 : d) + kDigitBias;
}

// 2^e s for a result s of a digit product sum
__device__ __forceinline__ double scale2(double s, int e) {
  if (e >= -1000 && e <= 1000) return s * __hiloint2double((e + 1023) << 20, 0);
  return scalbn(s, e);
}

__device__ __forceinline__ uint32_t h2sub(uint32_t a) {      // half2 (1024 + b) -> b - 128
  const __half2 c = __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));
  __half2 v = *reinterpret_cast<__half2*>(&a);
  v = __hsub2(v, c);
  return *reinterpret_cast<uint32_t*>(&v);
}

// the four digits of two 32-bit digit words as half2 (x's digit, y's digit), most significant first
__device__ __forceinline__ void word_digits(uint32_t x, uint32_t y, uint32_t* out) {
  const uint32_t p = __byte_perm(x, y, 0x5140), q = __byte_perm(x, y, 0x7362);
  out[0] = h2sub(__byte_perm(q, 0x64646464u, 0x4342));
  out[1] = h2sub(__byte_perm(q, 0x64646464u, 0x4140));
  out[2] = h2sub(__byte_perm(p, 0x64646464u, 0x4342));
  out[3] = h2sub(__byte_perm(p, 0x64646464u, 0x4140));
}

__device__ __forceinline__ void mma16816(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
               "{%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint4 zero_entry() { return make_uint4(kZeroWord, kZeroWord, kZeroWord, kZeroWord); }

// One 16 x 16 step of A (entries raw[q], q = 0..7: row half q & 1, k order 2t, 2t+1, 2t+8, 2t+9 =
// q >> 1) times eight real columns, the real and imaginary parts of four complex ones.  The digit
// pairs (i, j) with i + j = d add up in accumulator d (cr: Re A, ci: Im A); pairs beyond d = 7 are
// below 2^-59 (rms, 64 columns) of the largest product and left out.  72 MMAs for 256 entries x 4
// columns: 0.14 SM-clocks per complex product, against 2 on the FP64 units.  b: digit j of the
// column pair at b[j * S2], the pairs eight further on in k at 4 * pstride.
__device__ __forceinline__ void step_multi(const uint4* raw, const uint32_t* bd, int S2, int pstride, float (*cr)[4],
                                           float (*ci)[4]) {
  uint32_t b[8][2];
#pragma unroll
  for (int j = 0; j < 8; j++) {
    b[j][0] = bd[j * S2];
    b[j][1] = bd[4 * pstride + j * S2];
  }
#pragma unroll
  for (int w = 0; w < 2; w++) {
#pragma unroll
    for (int part = 0; part < 2; part++) {
      uint32_t a[4][4];
#pragma unroll
      for (int h = 0; h < 2; h++)
#pragma unroll
        for (int kp = 0; kp < 2; kp++) {
          const uint4 x = raw[(2 * kp) * 2 + h], y = raw[(2 * kp + 1) * 2 + h];
          uint32_t o[4];
          if (part == 0) word_digits(w == 0 ? x.y : x.x, w == 0 ? y.y : y.x, o);
          else word_digits(w == 0 ? x.w : x.z, w == 0 ? y.w : y.z, o);
#pragma unroll
          for (int d = 0; d < 4; d++) a[d][2 * kp + h] = o[d];
        }
#pragma unroll
      for (int d = 0; d < 4; d++)
#pragma unroll
        for (int j = 0; j < 8 - (4 * w + d); j++) mma16816(part ? ci[4 * w + d + j] : cr[4 * w + d + j], a[d], b[j][0], b[j][1]);
    }
  }
}

// (hi + lo 2^-32) 2^e, rounded once, for |hi|, |lo| < 2^62.  In integer arithmetic: each of the two
// conversions, the FMA and the scaling holds its scheduler for 64 clocks on the FP64 units.  Same bits;
// factorisation of 54,925 dofs in FP64 35.9 -> 33.0 ms.
__device__ __forceinline__ double scaled_sum(int64_t hi, int64_t lo, int e) {
  const int64_t top = hi + (lo >> 32);                   // V = top 2^32 + low
  const uint32_t low = uint32_t(lo);
  const bool neg = top < 0;
  const uint64_t at = neg ? (low ? ~uint64_t(top) : 0 - uint64_t(top)) : uint64_t(top);
  const uint32_t al = neg ? 0u - low : low;              // |V| = at 2^32 + al
  const int s = __clzll(int64_t(at));
  const int be = 1022 + 63 - s + e;                      // biased exponent less one
  if ((at | al) == 0) return 0.0;
  if (at == 0 || be < 1 || be > 2044)                    // below 1 / 2^32 units, subnormal or overflowing: rare
    return scale2(fma(double(lo), 0x1p-32, double(hi)), e);
  const uint64_t w = (uint64_t(al) << 32) >> (64 - s);   // the bits of al that move up, s >= 1
  const uint32_t lost = s < 32 ? al << s : 0u;
  const uint64_t M = (at << s) | w;                      // leading one at bit 63
  const uint32_t rem = (uint32_t(M) & 0x7ffu) | uint32_t(lost != 0);
  const uint64_t mant = M >> 11;
  // to nearest, ties to even; below bit 0 of M only whether anything was lost matters
  const bool up = rem > 0x400u || (rem == 0x400u && (mant & 1));
  const uint64_t bits = (uint64_t(uint32_t(be)) << 52) + mant + uint64_t(up);
  return __longlong_as_double(int64_t(bits | (neg ? 1ull << 63 : 0ull)));
}

// the value of the eight digit-weight sums t, times 2^e
__device__ __forceinline__ double digit_value(const int* t, int e) {
  const int64_t hi = ((int64_t(t[0]) * 256 + t[1]) * 256 + t[2]) * 256 + t[3];
  const int64_t lo = ((int64_t(t[4]) * 256 + t[5]) * 256 + t[6]) * 256 + t[7];
  return scaled_sum(hi, lo, e);
}

// adds the accumulators of one flush to the FP64 sums: acc[h] (row half h) += this lane's
// right-hand side; ea, eb: the exponents of the two rows plus that of the column
__device__ __forceinline__ void flush_multi(float (*cr)[4], float (*ci)[4], double2* acc, int ea, int eb) {
#pragma unroll
  for (int h = 0; h < 2; h++) {
    int tr[8], ti[8];
#pragma unroll
    for (int d = 0; d < 8; d++) {
      tr[d] = __float2int_rn(cr[d][2 * h]) - __float2int_rn(ci[d][2 * h + 1]);
      ti[d] = __float2int_rn(cr[d][2 * h + 1]) + __float2int_rn(ci[d][2 * h]);
    }
    const int sc = 88 + (h ? eb : ea);
    acc[h].x += digit_value(tr, sc);
    acc[h].y += digit_value(ti, sc);
  }
#pragma unroll
  for (int d = 0; d < 8; d++)
#pragma unroll
    for (int q = 0; q < 4; q++) cr[d][q] = ci[d][q] = 0.f;
}

}  // namespace hz
