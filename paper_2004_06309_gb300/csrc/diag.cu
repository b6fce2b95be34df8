// Pivot blocks of the multifrontal factorisation: F11 = L D L^T (complex symmetric, no
// pivoting) and T = L^{-1}, in place in shared memory, one CTA per supernode.
//
// Left-looking by 16-column blocks.  With the rows above J done, step J
//   * subtracts W(I, q) L(J, q)^T, q < J, from the blocks of column J (W = L D) and forms
//     S(J') = sum_q L(J, q) T(q, J') for every J' < J: one product with L's block row J, nbk
//     tiles of 16 rows whatever J is;
//   * factors the 16 x 16 block and inverts its unit lower factor in the same 16 pivots;
//   * W(I, J) = A(I, J) L(J, J)^{-T} and T(J, J') = -L(J, J)^{-1} S(J'), a product with T(J, J) in
//     complex128, by substitution in complex64.  T's row J overwrites W's, which is not needed
//     any more.
// The unblocked loop (a barrier pair per column and per row of the inverse) took 1.36 ms per
// level in complex128 (width 112) and 0.61 ms in complex64 (width 128).  A complex128 product is
// 4 FP64 instructions of 64 clocks per scheduler, whatever its active lanes, so the block
// products run in digits on mma.sync (digits.cuh) and only the 16 x 16 blocks on the FP64
// units.  The next pivot's chain (diagonal entry, reciprocal, column) runs in its own warp beside the
// update, its two parts in different lanes of the same instructions; one after the other a pivot took 2,500
// clocks.  0.27 ms per level in complex128 and 0.12 ms in complex64 on the same models.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "dev.h"
#include "digits.cuh"
#include "dmath.cuh"

namespace hz {

namespace {

constexpr int kMaxNbk = 8;                          // 16-column blocks (complex64: width 128)

template <typename V> struct DiagLayout;
template <> struct DiagLayout<double2> {
  static constexpr int pitch = 17;                   // entries per block column (conflict-free rows and columns)
  static constexpr int pstride = 16 * 16 + 8;        // words per k pair of the digit operand: 8 digits x 32 columns
  static __host__ __device__ size_t operand_bytes(int nbk) { return size_t(8 * (nbk > 1 ? nbk - 1 : 1)) * pstride * 4; }
};
template <> struct DiagLayout<float2> {
  static constexpr int pitch = 18;                   // 16-byte aligned columns
  static __host__ __device__ size_t operand_bytes(int nbk) { return size_t(16 * nbk) * 16 * 8; }
};

template <typename V> size_t diag_bytes(int nbk) {
  constexpr int blk = 16 * DiagLayout<V>::pitch;
  return (size_t(nbk * (nbk + 1) / 2) + size_t(nbk)) * blk * sizeof(V) + DiagLayout<V>::operand_bytes(nbk);
}

__device__ __forceinline__ int blk_index(int I, int J) { return I * (I + 1) / 2 + J; }

// digits of a complex value in units of exponent E
__device__ __forceinline__ uint4 entry_digits(double2 v, int E) {
  const uint64_t a = to_digits(v.x, 1 + E - max(exp_field(v.x), 1));
  const uint64_t b = to_digits(v.y, 1 + E - max(exp_field(v.y), 1));
  return make_uint4(uint32_t(a), uint32_t(a >> 32), uint32_t(b), uint32_t(b >> 32));
}
__device__ __forceinline__ int entry_exp(double2 v) { return max(exp_field(v.x), exp_field(v.y)); }

// writes the digits of two consecutive k entries of complex column n as the B operand
__device__ __forceinline__ void put_operand_pair(uint32_t* dst, int n, uint4 x, uint4 y) {
  uint32_t o[4];
#pragma unroll
  for (int part = 0; part < 2; part++) {
    word_digits(part ? x.w : x.y, part ? y.w : y.y, o);
#pragma unroll
    for (int d = 0; d < 4; d++) dst[d * 32 + 2 * n + part] = o[d];
    word_digits(part ? x.z : x.x, part ? y.z : y.x, o);
#pragma unroll
    for (int d = 0; d < 4; d++) dst[(4 + d) * 32 + 2 * n + part] = o[d];
  }
}

}  // namespace

template <typename V>
__global__ void __launch_bounds__(256, 1) k_diag_blk(const int32_t* lev_sn, const SnDev* sn, const int16_t* sig, V* fronts,
                                                     DevStatus* status, double tiny) {
  using L = DiagLayout<V>;
  constexpr int P = L::pitch, BLK = 16 * P;
  constexpr bool dbl = sizeof(V) == 16;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ V dinv[16 * kMaxNbk], dval[16 * kMaxNbk];
  __shared__ V wcol2[2][16], trow2[2][16], xdiag[2], lcol[16];   // [2]: by the pivot's parity
  __shared__ V ljj[dbl ? 1 : 256];                         // L(J, J), column-major
  __shared__ int aexp[16 * kMaxNbk], bexp[2][16];
  const SnDev S = sn[lev_sn[blockIdx.x]];
  const int k = S.k, m = S.m, nbk = (k + 15) / 16;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  V* A = reinterpret_cast<V*>(smem_raw);               // lower blocks, column-major
  V* Sb = A + (nbk * (nbk + 1) / 2) * BLK;             // S(J')^T: [column of J'][row of J]
  void* opnd = Sb + nbk * BLK;                         // L's block row J as the second factor
  V* F = fronts + S.frontoff;
  auto blk = [&](int I, int J) { return A + blk_index(I, J) * BLK; };
  // load the lower triangle; identity beyond k
  for (int c = wid; c < 16 * nbk; c += 8)
    for (int r = (c & ~15) + lane; r < 16 * nbk; r += 32) {
      V v = czero<V>();
      if (r < k && c < k) {
        if (r >= c) v = F[r + int64_t(c) * m];
      } else if (r == c) {
        v.x = 1;
      }
      blk(r >> 4, c >> 4)[(r & 15) + P * (c & 15)] = v;
    }
  __syncthreads();

  // vector v of tile a at step J, entry kk of block q: rows of W(a, q) for a >= J, columns of
  // T(q, a) for a < J
  auto avec = [&](int a, int J, int q, int r, int kk) -> V {
    if (a >= J) return blk(a, q)[r + P * kk];
    if (q > a) return blk(q, a)[kk + P * r];
    V v = blk(a, a)[kk + P * r];                       // unit lower: zeros stored above
    if (kk == r) {
      v = czero<V>();
      v.x = 1;
    }
    return v;
  };

  for (int J = 0; J < nbk; J++) {
    if (J > 0) {
      if constexpr (dbl) {
        uint32_t* bd = reinterpret_cast<uint32_t*>(opnd);
        // L(J, q) = W(J, q) D^{-1}: rows n = 0..15, this thread's k pair p of blocks q = qh, qh + 2, ..
        const int n = tid & 15, p = (tid >> 4) & 7, qh = tid >> 7;
        V l[kMaxNbk / 2][2];
        int e = 1;
        if (tid < 16) bexp[0][tid] = 1;
        if (tid < 16 * nbk) aexp[tid] = 1;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kMaxNbk / 2; u++) {
          const int q = qh + 2 * u;
          if (q < J) {
#pragma unroll
            for (int h = 0; h < 2; h++) {
              const int kk = 2 * p + h;
              l[u][h] = cmul(blk(J, q)[n + P * kk], dinv[16 * q + kk]);
              e = max(e, entry_exp(l[u][h]));
            }
          }
        }
        e = max(e, __shfl_xor_sync(0xffffffffu, e, 16));
        if (lane < 16) atomicMax(&bexp[0][n], e);
        // exponents of the first factor's vectors, two threads each
        if (tid < 32 * nbk) {
          const int v = tid >> 1, a = v >> 4, r = v & 15;
          int ev = 1;
          for (int q = a < J ? a : 0; q < J; q++)
#pragma unroll 4
            for (int kk = tid & 1; kk < 16; kk += 2) ev = max(ev, entry_exp(avec(a, J, q, r, kk)));
          atomicMax(&aexp[v], ev);
        }
        __syncthreads();
        // digits hold no infinity or NaN: report the matrix as one without usable pivots
        if (tid < 16 * nbk && (aexp[tid] == 0x7ff || (tid < 16 && bexp[0][tid] == 0x7ff)))
          atomicOr(&status->zero_pivot, 1u);
        {
          const int E = bexp[0][n];
#pragma unroll
          for (int u = 0; u < kMaxNbk / 2; u++) {
            const int q = qh + 2 * u;
            if (q < J)
              put_operand_pair(bd + (8 * q + p) * L::pstride, n, entry_digits(l[u][0], E), entry_digits(l[u][1], E));
          }
        }
        __syncthreads();
        const int g = lane >> 2, t = lane & 3;
        for (int job = wid; job < 2 * nbk; job += 8) {     // (tile, two of the four column groups)
          const int a = job >> 1, nh = job & 1;
          const int ea = aexp[16 * a + g], eb = aexp[16 * a + g + 8];
          float cr[2][8][4], ci[2][8][4];
#pragma unroll
          for (int u = 0; u < 2; u++)
#pragma unroll
            for (int d = 0; d < 8; d++)
#pragma unroll
              for (int x = 0; x < 4; x++) cr[u][d][x] = ci[u][d][x] = 0.f;
          for (int q = a < J ? a : 0; q < J; q++) {
            uint4 raw[8];
#pragma unroll
            for (int x = 0; x < 4; x++) {
              const int kk = 2 * t + (x & 1) + 8 * (x >> 1);
              raw[2 * x] = entry_digits(avec(a, J, q, g, kk), ea);
              raw[2 * x + 1] = entry_digits(avec(a, J, q, g + 8, kk), eb);
            }
#pragma unroll
            for (int u = 0; u < 2; u++)
              step_multi(raw, bd + (8 * q + t) * L::pstride + 8 * (2 * nh + u) + g, 32, L::pstride, cr[u], ci[u]);
          }
#pragma unroll
          for (int u = 0; u < 2; u++) {
            const int nn = 4 * (2 * nh + u) + t, en = bexp[0][nn] - 2 * kBias;
            double2 acc[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
            flush_multi(cr[u], ci[u], acc, ea + en, eb + en);
#pragma unroll
            for (int h = 0; h < 2; h++) {
              const int r = g + 8 * h;
              if (a >= J) {
                V* o = blk(a, J) + r + P * nn;
                *o = csub(*o, acc[h]);
              } else {
                Sb[a * BLK + nn + P * r] = acc[h];
              }
            }
          }
        }
      } else {
        V* Lb = reinterpret_cast<V*>(opnd);                // [kk][n]
        for (int e = tid; e < 256 * J; e += 256) {
          const int n = e & 15, kk = (e >> 4) & 15, q = e >> 8;
          Lb[(16 * q + kk) * 16 + n] = cmul(blk(J, q)[n + P * kk], dinv[16 * q + kk]);
        }
        __syncthreads();
        // the sums start from -A, as subtracting column by column did: summed from zero and subtracted
        // at the end, the error of the complex64 M^{-1} v was 5 % higher
        if (wid < nbk) {
          const int a = wid, r = lane & 15, h = lane >> 4;
          V acc[8];
#pragma unroll
          for (int x = 0; x < 8; x++) acc[x] = a >= J ? cneg(blk(a, J)[r + P * (8 * h + x)]) : czero<V>();
          for (int q = a < J ? a : 0; q < J; q++)
#pragma unroll 4
            for (int kk = 0; kk < 16; kk++) {
              const V av = avec(a, J, q, r, kk);
              const V* b = Lb + (16 * q + kk) * 16 + 8 * h;
#pragma unroll
              for (int x = 0; x < 8; x++) acc[x] = cmad(av, b[x], acc[x]);
            }
#pragma unroll
          for (int x = 0; x < 8; x++) {
            if (a >= J) blk(a, J)[r + P * (8 * h + x)] = cneg(acc[x]);
            else Sb[a * BLK + (8 * h + x) + P * r] = acc[x];
          }
        }
      }
      __syncthreads();
    }
    // 16 x 16 block.  Warps 2, 3, 6 and 7 hold its entries (row, c), two row pairs each: of the update
    // for c > pivot, of T from pivot c on.  Warp 0 does what the next pivot waits for beside them:
    // column of L, next diagonal entry, its reciprocal, real and imaginary parts in different lanes.
    {
      using R = decltype(V().x);
      const int c = lane & 15, uw = (wid & 2) ? (wid & 1) + 2 * (wid >> 2) : -1;
      const int part = lane >> 4;                          // warp 0: lanes (i = c, part)
      int row[2] = {0, 0};
      V y[2] = {czero<V>(), czero<V>()};
      if (uw >= 0) {
#pragma unroll
        for (int h = 0; h < 2; h++) {
          const int r = row[h] = 2 * (uw + 4 * h) + part;
          y[h] = blk(J, J)[r + P * c];
          if (c == 0) wcol2[0][r] = y[h];
          if (r == 1 && c == 1) xdiag[1] = y[h];
        }
      }
      if (tid == 0) {
        V one = czero<V>();
        one.x = 1;
        trow2[0][0] = one;
      }
      __syncthreads();
      V d = czero<V>(), di = czero<V>();
      auto reciprocal = [&]() {                            // warp 0: 1 / d
        const R q = d.x * d.x + d.y * d.y;
        const R v = (part ? -d.y : d.x) / q;
        di.x = __shfl_sync(0xffffffffu, v, 0);
        di.y = __shfl_sync(0xffffffffu, v, 16);
      };
      if (wid == 0) {
        d = wcol2[0][0];
        reciprocal();
      }
      for (int j = 0; j < 16; j++) {
        V *wcol = wcol2[j & 1], *trow = trow2[j & 1];
        if (wid == 0) {
          const V w = wcol[c];                             // w di, one part per lane
          const R v = xfma(w.x, part ? di.y : di.x, (part ? w.y : -w.y) * (part ? di.x : di.y));
          if (c > j) {
            reinterpret_cast<R*>(lcol + c)[part] = v;
            if constexpr (!dbl) reinterpret_cast<R*>(ljj + 16 * j + c)[part] = v;
          }
          if (lane == 0) {
            dval[16 * J + j] = d;
            dinv[16 * J + j] = di;
          }
        }
        __syncthreads();
        if (j == 15) break;
        if (uw >= 0) {
#pragma unroll
          for (int h = 0; h < 2; h++) {
            const int r = row[h];
            if (r <= j) continue;
            const bool t = c <= j;
            y[h] = cmsub(t ? lcol[r] : wcol[r], t ? trow[c] : lcol[c], c == j ? czero<V>() : y[h]);
            if (c == j + 1) wcol2[(j + 1) & 1][r] = y[h];
            if (r == j + 1 && c <= j + 1) {
              V v = y[h];
              if (c == j + 1) {
                v = czero<V>();
                v.x = 1;
              }
              trow2[(j + 1) & 1][c] = v;
            }
            if (r == j + 2 && c == j + 2) xdiag[j & 1] = y[h];
          }
        } else if (wid == 0) {
          const V w = wcol[j + 1], l = lcol[j + 1], x = xdiag[(j + 1) & 1];
          // one part per lane: x - w l
          R v = xfma(-w.x, part ? l.y : l.x, part ? x.y : x.x);
          v = xfma(part ? -w.y : w.y, part ? l.x : l.y, v);
          d.x = __shfl_sync(0xffffffffu, v, 0);
          d.y = __shfl_sync(0xffffffffu, v, 16);
          reciprocal();
        }
        __syncthreads();
      }
      if (uw >= 0) {
#pragma unroll
        for (int h = 0; h < 2; h++) blk(J, J)[row[h] + P * c] = row[h] > c ? y[h] : czero<V>();
      }
      __syncthreads();
    }
    // W(I, J) = A(I, J) T^T for I > J and T(J, J') = -T S(J') for J' < J
    if constexpr (dbl) {
      uint32_t* bd = reinterpret_cast<uint32_t*>(opnd);
      if (tid < 128) {                                     // T's rows n, k pair p
        const int n = tid & 15, p = tid >> 4;
        if (p == 0) {
          int e = 1;
#pragma unroll
          for (int kk = 0; kk < 16; kk++) e = max(e, entry_exp(blk(J, J)[n + P * kk]));
          bexp[1][n] = e;
        }
      }
      __syncthreads();
      if (tid < 128) {
        const int n = tid & 15, p = tid >> 4, E = bexp[1][n];
        put_operand_pair(bd + p * L::pstride, n, entry_digits(blk(J, J)[n + P * (2 * p)], E),
                         entry_digits(blk(J, J)[n + P * (2 * p + 1)], E));
      }
      __syncthreads();
      const int g = lane >> 2, t = lane & 3;
      if (wid < nbk && wid != J) {
        const int a = wid;
        V* src = a > J ? blk(a, J) : Sb + a * BLK;
        auto at = [&](int r, int kk) -> V& { return a > J ? src[r + P * kk] : src[kk + P * r]; };
        V va[4], vb[4];
        int ea = 1, eb = 1;
#pragma unroll
        for (int x = 0; x < 4; x++) {
          const int kk = 2 * t + (x & 1) + 8 * (x >> 1);
          va[x] = at(g, kk);
          vb[x] = at(g + 8, kk);
          ea = max(ea, entry_exp(va[x]));
          eb = max(eb, entry_exp(vb[x]));
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
          ea = max(ea, __shfl_xor_sync(0xffffffffu, ea, o));
          eb = max(eb, __shfl_xor_sync(0xffffffffu, eb, o));
        }
        uint4 raw[8];
#pragma unroll
        for (int x = 0; x < 4; x++) {
          raw[2 * x] = entry_digits(va[x], ea);
          raw[2 * x + 1] = entry_digits(vb[x], eb);
        }
#pragma unroll
        for (int u = 0; u < 4; u++) {
          float cr[8][4], ci[8][4];
#pragma unroll
          for (int d = 0; d < 8; d++)
#pragma unroll
            for (int x = 0; x < 4; x++) cr[d][x] = ci[d][x] = 0.f;
          step_multi(raw, bd + t * L::pstride + 8 * u + g, 32, L::pstride, cr, ci);
          const int nn = 4 * u + t, en = bexp[1][nn] - 2 * kBias;
          double2 acc[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
          flush_multi(cr, ci, acc, ea + en, eb + en);
#pragma unroll
          for (int h = 0; h < 2; h++) {
            const int r = g + 8 * h;
            const V w = cadd(at(r, nn), acc[h]);           // only this lane reads or writes (r, nn) from here on
            if (a > J) at(r, nn) = w;
            else blk(J, a)[nn + P * r] = cneg(w);
          }
        }
      }
    } else {
      // by substitution with L(J, J), one thread per vector
      if (tid < 16 * nbk && (tid >> 4) != J) {
        const int a = tid >> 4, r = tid & 15;
        V* src = a > J ? blk(a, J) + r : Sb + a * BLK + P * r;
        const int step = a > J ? P : 1;
        V w[16];
#pragma unroll
        for (int c = 0; c < 16; c++) w[c] = src[c * step];
#pragma unroll
        for (int c = 0; c < 15; c++)
#pragma unroll
          for (int i = c + 1; i < 16; i++) w[i] = cmsub(ljj[16 * c + i], w[c], w[i]);
        if (a > J) {
#pragma unroll
          for (int c = 0; c < 16; c++) src[c * step] = w[c];
        } else {
#pragma unroll
          for (int c = 0; c < 16; c++) blk(J, a)[c + P * r] = cneg(w[c]);
        }
      }
    }
    __syncthreads();
  }
  if (tid < k) {
    const V d = dval[tid];
    double mag = sqrt(double(d.x) * double(d.x) + double(d.y) * double(d.y));
    if constexpr (dbl) mag *= exp2i(2 * sig[S.first + tid]);
    atomicMin(reinterpret_cast<unsigned long long*>(&status->min_pivot),
              static_cast<unsigned long long>(__double_as_longlong(mag)));
    if (!(mag >= tiny)) atomicOr(&status->zero_pivot, 1u);
  }
  for (int c = wid; c < k; c += 8)
    for (int r = c + lane; r < k; r += 32)
      F[r + int64_t(c) * m] = r > c ? blk(r >> 4, c >> 4)[(r & 15) + P * (c & 15)] : dinv[c];
}

template <typename V>
static void launch_diag_t(int64_t nb, int maxk, const int32_t* lev_sn, const SnDev* sn, const int16_t* sig, V* fronts,
                          DevStatus* status, double tiny, cudaStream_t st) {
  static const bool attr = [] {
    cudaFuncSetAttribute(k_diag_blk<V>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
    return true;
  }();
  (void)attr;
  add_launches(1);
  k_diag_blk<V><<<unsigned(nb), 256, diag_bytes<V>((maxk + 15) / 16), st>>>(lev_sn, sn, sig, fronts, status, tiny);
}

void launch_diag(int precision, int64_t nb, int maxk, const int32_t* lev_sn, const SnDev* sn, const int16_t* sig,
                 void* fronts, DevStatus* status, double tiny, cudaStream_t st) {
  if (precision == 0) launch_diag_t(nb, maxk, lev_sn, sn, sig, (double2*)fronts, status, tiny, st);
  else launch_diag_t(nb, maxk, lev_sn, sn, sig, (float2*)fronts, status, tiny, st);
}

}  // namespace hz
