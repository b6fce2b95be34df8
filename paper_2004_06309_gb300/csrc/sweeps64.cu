// Triangular sweeps of the complex128 factors on the tensor cores (sm_103a).
//
// GB300 issues two FP64 FMAs per SM and clock, so a complex128 sweep on the FP64 units takes
// two SM-clocks per panel entry and right-hand side, three times what reading the entry
// costs.  Here the products run as exact integer products instead:
//   * after the factorisation every panel entry x (rows below the pivot) is rewritten in
//     place as two 64-bit integers D = x 2^(1084 - E), E the largest exponent field of the
//     entry's panel row, |D| < 2^62; each as eight balanced base-256 digits in [-128, 127],
//     stored with 128 added (so a byte is a digit).  The row's E - 1084 is kept beside the
//     panel.  Same bytes as the doubles; the diagonal keeps D^{-1} in FP64;
//   * the right-hand side of a task is written in digits too, with one exponent per task
//     and right-hand side;
//   * a digit product sum runs on mma.sync m16n8k16 (f16 in, f32 accumulators): a digit and
//     a product of digits are exact, and at most 8 digit pairs x 128 columns of products of
//     at most 2^14 meet in one accumulator: at most 2^24, so every sum is exact too.
//     Digit pairs (i, j) with i + j <= 7 are kept; what is dropped is below 2^-59 (rms) of
//     the largest product for 64 columns.
// The digits of one operand hold 62 bits below the largest entry of its group (a panel row; a task's
// right-hand side), against the 53 of a double below each entry, and the column sum is exact where the
// FP64 loop rounded at every step.  So a sum's error is relative to the product of the two groups'
// largest entries, not to its own terms; sums far below that product are done on the FP64 units
// (kGuardBits).  A right-hand side with an infinity or NaN gives NaN in every row of its tasks.
//
// Bound: reading the panels (16 bytes per entry: 0.69 SM-clocks at 6.8 TB/s), beside about
// 0.3 for unpacking digits (20 integer and half2 operations per entry) and 0.25 for the
// products of one right-hand side (32 MMAs of 2 clocks per 256 entries).
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "dev.h"
#include "digits.cuh"
#include "dmath.cuh"

namespace hz {

namespace {

constexpr int16_t kRowNonFinite = 0x7fff;
constexpr int kPairStride = 24;           // words per column pair of a digit vector (15 used; 24 t mod 32 differ)

__device__ __forceinline__ uint4 ld_panel(const uint4* p) { return __ldg(p); }
// Position of column pair p of a 16-column step in a digit vector: fragment register b0 reads
// pairs at positions 0-3, b1 at 4-7.  forward: pairs (2t, 2t + 1) and (2t + 8, 2t + 9) as they
// come; backward: lane t holds four consecutive rows, pairs 2t and 2t + 1.
__device__ __forceinline__ int pair_pos_bwd(int p) { return (p >> 1) + 4 * (p & 1); }

// One 16 x 16 step of the panel for one right-hand side: raw[q], q = 0..7, are the entries
// (row half q & 1, k index order 2t, 2t+1, 2t+8, 2t+9 = q >> 1).  c: Re x re, Im x im,
// Re x im and Im x re, whose eight columns are the digit weights (four chains of eight MMAs).
__device__ __forceinline__ void step_single(const uint4* raw, const uint32_t* bre, const uint32_t* bim, int off,
                                            float (*c)[4]) {
#pragma unroll
  for (int w = 0; w < 2; w++) {                      // high words: digits 0-3; low words: 4-7
    uint32_t ar[4][4], ai[4][4];                     // [digit][fragment register]
#pragma unroll
    for (int h = 0; h < 2; h++)                      // row half
#pragma unroll
      for (int kp = 0; kp < 2; kp++) {               // k pair
        const uint4 x = raw[(2 * kp) * 2 + h], y = raw[(2 * kp + 1) * 2 + h];
        uint32_t o[4];
        word_digits(w == 0 ? x.y : x.x, w == 0 ? y.y : y.x, o);
#pragma unroll
        for (int d = 0; d < 4; d++) ar[d][2 * kp + h] = o[d];
        word_digits(w == 0 ? x.w : x.z, w == 0 ? y.w : y.z, o);
#pragma unroll
        for (int d = 0; d < 4; d++) ai[d][2 * kp + h] = o[d];
      }
#pragma unroll
    for (int d = 0; d < 4; d++) {
      const int o = off - (4 * w + d);
      const uint32_t r0 = bre[o], r1 = bre[o + 4 * kPairStride], i0 = bim[o], i1 = bim[o + 4 * kPairStride];
      mma16816(c[0], ar[d], r0, r1);
      mma16816(c[1], ai[d], i0, i1);
      mma16816(c[2], ar[d], i0, i1);
      mma16816(c[3], ai[d], r0, r1);
    }
  }
}

// adds the accumulators to the sums of the real part (tot[0]) and the imaginary part (tot[1])
__device__ __forceinline__ void flush_single(float (*c)[4], int (*tot)[4]) {
#pragma unroll
  for (int q = 0; q < 4; q++) {
    tot[0][q] += __float2int_rn(c[0][q]) - __float2int_rn(c[1][q]);
    tot[1][q] += __float2int_rn(c[2][q]) + __float2int_rn(c[3][q]);
    c[0][q] = c[1][q] = c[2][q] = c[3][q] = 0.f;
  }
}

// The eight weighted digit sums of a row lie two per lane in a quad: lane t = 0 returns the upper
// four and t = 2 the lower four as one integer (digit weights 256^3 .. 1).
__device__ __forceinline__ int64_t quad_half(int hi, int lo) {
  const int64_t v = int64_t(hi) * 256 + lo;
  return v * 65536 + __shfl_xor_sync(0xffffffffu, v, 1);
}
// a + the pt-th parts of u[c0 .. c1), in order; the first two loads are issued together
__device__ __forceinline__ double add_updates_part(double a, const double* ud, uint32_t c0, uint32_t c1, int pt) {
  double v0 = 0.0, v1 = 0.0;
  if (c0 < c1) v0 = __ldcg(ud + 2 * int64_t(c0) + pt);
  if (c0 + 1 < c1) v1 = __ldcg(ud + 2 * int64_t(c0) + 2 + pt);
  a = (a + v0) + v1;
  for (uint32_t c = c0 + 2; c < c1; c++) a += __ldcg(ud + 2 * int64_t(c) + pt);
  return a;
}

// Writes the digits of the value pair (x, y) (already in units of the group's exponent) as the
// shifted-digit rows of a digit vector: word 7 + i is digit i, words 0-6 are zero.
__device__ __forceinline__ void put_pair(uint32_t* dst, uint64_t dx, uint64_t dy) {
#pragma unroll
  for (int i = 0; i < 7; i++) dst[i] = 0u;
  uint32_t o[4];
  word_digits(uint32_t(dx >> 32), uint32_t(dy >> 32), o);
#pragma unroll
  for (int i = 0; i < 4; i++) dst[7 + i] = o[i];
  word_digits(uint32_t(dx), uint32_t(dy), o);
#pragma unroll
  for (int i = 0; i < 4; i++) dst[11 + i] = o[i];
}

// A row's (column's) products are bounded by 2^(x - 960), x the exponent of its entries plus that of the
// right-hand side, and the digits miss each by about 2^-59 of this bound.  Where the sum and what it is
// added to both come out below 2^-kGuardBits of it, the large entries of one side meet small or zero
// ones of the other, and what is missed may matter beside what is left: the sum is done again on the
// FP64 units.  The panel itself is within 2^-62 of its row's largest entry either way; a zero is exact.
// One of 6 million sums comes below in M^{-1} of a random vector of 349,461 dofs, one of 5,000 in a solve
// for a point source, nearly all of them in its first application: M^{-1} v 4.48 -> 4.54 ms, six sources
// in four slots (9,801 dofs) 9.3 -> 9.7 ms.  With 10 bits, what is added to left out and columns of zeros
// not skipped, 1 of 24 columns came below: 6.1 and 17.0 ms.
constexpr int kGuardBits = 14;
__device__ __forceinline__ bool below_guard(int field, int x) { return field < x + 63 - kGuardBits; }

// a panel entry in units of 2^62 of its row
__device__ __forceinline__ double2 entry_value(uint4 w) {
  const int64_t x = int64_t(((uint64_t(w.y) << 32) | w.x) - kDigitBias), y = int64_t(((uint64_t(w.w) << 32) | w.z) - kDigitBias);
  return make_double2(double(x) * 0x1p-62, double(y) * 0x1p-62);
}
// sum over j < n of the entries of one panel row (p, columns ld apart) times b[j * stride], in units of
// the row; one warp, the sum in every lane
__device__ __noinline__ double2 row_dot(const uint4* p, int ld, int n, const double2* b, int stride) {
  double2 a = make_double2(0.0, 0.0);
  for (int j = threadIdx.x & 31; j < n; j += 32) a = cmad(entry_value(__ldg(p + int64_t(j) * ld)), b[j * stride], a);
  return warp_sum(a);
}

// sum over rows q0 <= q < n of one panel column (p) times v[q], with the rows' exponents; one warp
__device__ __noinline__ double2 column_dot(const uint4* p, int q0, int n, const double2* v, const int* vex) {
  double2 a = make_double2(0.0, 0.0);
  for (int q = q0 + (threadIdx.x & 31); q < n; q += 32) {
    const double2 x = v[q];
    const int e = vex[q] + 62;
    a = cmad(entry_value(__ldg(p + q)), make_double2(scale2(x.x, e), scale2(x.y, e)), a);
  }
  return warp_sum(a);
}

// largest value over the block (128 threads); syncs
__device__ __forceinline__ int block_max(int v, int* red) {
  v = __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  return max(max(red[0], red[1]), max(red[2], red[3]));
}

}  // namespace

// ---------------------------------------------------------------------------
// panels -> digits, in place; one task = RT rows of one solve supernode.  colnz (zeroed before): columns
// with an entry below the diagonal
// ---------------------------------------------------------------------------
template <int RT>
__global__ void __launch_bounds__(256) k_to_digits(const int2* tasks, const SnDev* sn, double2* panels,
                                                   int16_t* rexp, uint8_t* colnz) {
  constexpr int CG = 256 / RT;
  __shared__ int red[CG][RT];
  const int2 t = tasks[blockIdx.x];
  const SnDev S = sn[t.x];
  const int rr = threadIdx.x % RT, cg = threadIdx.x / RT, r = (t.y * gridDim.y + blockIdx.y) * RT + rr;
  const int jmax = r < S.m ? min(r, S.k) : 0;
  double2* P = panels + S.paneloff + r;
  int e = 1;
  for (int j = cg; j < jmax; j += CG) {
    const double2 v = P[int64_t(j) * S.ld];
    e = max(e, max(exp_field(v.x), exp_field(v.y)));
  }
  red[cg][rr] = e;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < CG; q++) e = max(e, red[q][rr]);
  for (int j = cg; j < jmax; j += CG) {
    const double2 v = P[int64_t(j) * S.ld];
    const uint64_t a = to_digits(v.x, 1 + e - max(exp_field(v.x), 1));
    const uint64_t b = to_digits(v.y, 1 + e - max(exp_field(v.y), 1));
    P[int64_t(j) * S.ld] = make_double2(__longlong_as_double(int64_t(a)), __longlong_as_double(int64_t(b)));
    if ((v.x != 0.0 || v.y != 0.0) && !__ldcg(colnz + S.first + j)) colnz[S.first + j] = 1;   // all write the same
  }
  if (cg == 0 && r < S.m) rexp[S.eoff + r] = e == 0x7ff ? kRowNonFinite : int16_t(e - kBias);
}

// ---------------------------------------------------------------------------
// one right-hand side
// ---------------------------------------------------------------------------
// Panel steps of a warp are copied into its own ring of kRing slots (4 KB each) by cp.async, the
// first ones before the right-hand side is gathered; each lane reads back only what it copied,
// so the ring needs no barrier.  Measured on the subdomain sweeps of the 349,461-dof survey
// model (9.8 GB, 16 subdomains): 5.82 ms on the FP64 units; with digits 4.7 ms with the panels
// in registers (one step ahead, two blocks of 256 threads per SM), 3.81 ms with this ring (four
// blocks of 128; five blocks 3.93, three slots 4.41).  About a third of a task's time is its
// 16-column steps; the rest is the chain task -> supernode -> right-hand side -> digits, which
// the other blocks of the SM cover only in part.
constexpr int kRing = 2;

// Forward, npass blocks of 16 MT rows of one supernode per task (rows < k: z = D^{-1} (T b1); rows
// >= k: u = children's updates - G b1); 4 warps = MT row tiles x 4 / MT groups of 16-column steps.
// The right-hand side is gathered and converted once per task; the ring runs through the blocks,
// and what a block's last step needs (children's updates of its rows, D^{-1}, row exponents) is
// loaded one block ahead.
template <int MT>
__global__ void __launch_bounds__(128, 4) k_fwd_dig(const int2* tasks, const SnDev* sn, const uint32_t* cptr,
                                                    const uint32_t* wpos, const double2* panels,
                                                    const int16_t* rexp, const double2* tin, double2* zout,
                                                    double2* u, int kpad, int npass) {
  pdl_trigger();
  constexpr int CG = 4 / MT, RT = 16 * MT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint4* ring = reinterpret_cast<uint4*>(smem_raw);                      // 4 warps x kRing x 8 x 32
  double* b1 = reinterpret_cast<double*>(ring + 4 * kRing * 256);        // kpad x 2
  uint32_t* bre = reinterpret_cast<uint32_t*>(b1 + 2 * kpad);            // kpad / 2 pairs x kPairStride
  uint32_t* bim = bre + (kpad / 2) * kPairStride;
  __shared__ int64_t sums[2][CG][RT][2][2];                              // [block parity][group][row][part][half]
  __shared__ int red[4];
  const int2 tk = tasks[blockIdx.x];
  const SnDev S = sn[tk.x];
  const int k = S.k, m = S.m, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int g = lane >> 2, t = lane & 3, mt = wid % MT, cg = wid / MT;
  const uint32_t* cp = cptr + S.rowoff + S.id;
  const int base = tk.y * RT * npass, np = min(npass, (m - base + RT - 1) / RT);
  const uint4* P = reinterpret_cast<const uint4*>(panels + S.paneloff);
  uint4* myring = ring + wid * (kRing * 256) + lane;
  auto nsteps = [&](int p) {                                             // 16-column steps of this warp's tile in block p
    const int row0 = base + p * RT + mt * 16;
    return row0 < m ? (min(row0 + 15, k) + 15) / 16 : 0;
  };
  int ip = 0, is = cg;                                                   // next step to copy: block, step
  auto issue = [&](int slot) {
    while (ip < np && is >= nsteps(ip)) {
      ip++;
      is = cg;
    }
    if (ip < np) {
      const int ra = base + ip * RT + mt * 16 + g, rb = ra + 8;
      const int ja = ra < m ? min(ra, k) : 0, jb = rb < m ? min(rb, k) : 0;
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const int j = 16 * is + 2 * t + (q & 1) + 8 * (q >> 1);
        const uint4* col = P + int64_t(j) * S.ld;
        if (j < ja) cp_async16(myring + slot * 256 + (2 * q) * 32, col + ra);
        if (j < jb) cp_async16(myring + slot * 256 + (2 * q + 1) * 32, col + rb);
      }
      is += CG;
    }
    cp_async_commit();
  };
#pragma unroll
  for (int q = 0; q < kRing; q++) issue(q);
  // this thread's result of a block: row tid / 2, part tid & 1; where its child contributions lie
  // and where its update goes
  const int pt = tid & 1;
  int re = 0;
  uint32_t h0 = 0, h1 = 0, uw = 0;
  double2 dinv = make_double2(0.0, 0.0);
  auto load_row = [&](int p) {
    const int r = base + p * RT + (tid >> 1);
    const bool mine = tid < 2 * RT && p < np && r < m, upd = mine && r >= k;
    re = mine ? rexp[S.eoff + r] : 0;
    if (mine && r < k) dinv = panels[S.paneloff + r + int64_t(r) * S.ld];
    h0 = upd ? cp[r] : 0u;
    h1 = upd ? cp[r + 1] : 0u;
    uw = upd ? wpos[S.rowoff + r] : 0u;
  };
  load_row(0);
  const uint32_t g0 = tid < 2 * k ? cp[tid >> 1] : 0u, g1 = tid < 2 * k ? cp[(tid >> 1) + 1] : 0u;
  const int q1 = tid + 128;
  const uint32_t g2 = q1 < 2 * k ? cp[q1 >> 1] : 0u, g3 = q1 < 2 * k ? cp[(q1 >> 1) + 1] : 0u;
  pdl_wait();
  const double *tind = reinterpret_cast<const double*>(tin + S.first), *ud = reinterpret_cast<const double*>(u + S.ubase);
  int e = 1;
  {
    // the first two rounds (64 columns each) have their row pointers and load together
    double a0 = 0.0, a1 = 0.0;
    if (tid < 2 * k) a0 = __ldcg(tind + tid);
    if (q1 < 2 * k) a1 = __ldcg(tind + q1);
    a0 = add_updates_part(a0, ud, g0, g1, pt);
    a1 = add_updates_part(a1, ud, g2, g3, pt);
    if (tid < 2 * k) b1[tid] = a0;
    if (q1 < 2 * k) b1[q1] = a1;
    e = max(e, max(exp_field(a0), exp_field(a1)));
  }
  for (int q = tid + 256; q < 2 * k; q += 128) {
    const double a = add_updates_part(__ldcg(tind + q), ud, cp[q >> 1], cp[(q >> 1) + 1], pt);
    b1[q] = a;
    e = max(e, exp_field(a));
  }
  const int E = block_max(e, red);                                       // publishes b1 too
  const int kp = (k + 15) / 16 * 16;
  for (int q = tid; q < kp; q += 128) {                                  // pair q / 2, part q & 1
    const int p = q >> 1, j = 2 * p;
    const double x = j < k ? b1[2 * j + (q & 1)] : 0.0, y = j + 1 < k ? b1[2 * j + 2 + (q & 1)] : 0.0;
    put_pair(((q & 1) ? bim : bre) + p * kPairStride, to_digits(x, 1 + E - max(exp_field(x), 1)),
             to_digits(y, 1 + E - max(exp_field(y), 1)));
  }
  __syncthreads();
  int it = 0;
  for (int p = 0; p < np; p++) {
    const int row0 = base + p * RT + mt * 16, ra = row0 + g, rb = ra + 8;
    const int ja = ra < m ? min(ra, k) : 0, jb = rb < m ? min(rb, k) : 0;
    const int nst = nsteps(p), nfull = row0 + 15 < m ? min(row0, k) / 16 : 0;   // steps without a masked entry
    const double b2 = add_updates_part(0.0, ud, h0, h1, pt);
    float c[4][4];
    int tot[2][4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      c[0][q] = c[1][q] = c[2][q] = c[3][q] = 0.f;
      tot[0][q] = tot[1][q] = 0;
    }
    int since = 0;
    for (int s = cg; s < nst; s += CG, it++) {
      cp_async_wait<kRing - 1>();
      const int slot = it % kRing;
      uint4 raw[8];
#pragma unroll
      for (int q = 0; q < 8; q++) raw[q] = myring[slot * 256 + q * 32];
      if (s >= nfull) {
#pragma unroll
        for (int q = 0; q < 4; q++) {
          const int j = 16 * s + 2 * t + (q & 1) + 8 * (q >> 1);
          if (j >= ja) raw[2 * q] = zero_entry();
          if (j >= jb) raw[2 * q + 1] = zero_entry();
        }
      }
      step_single(raw, bre, bim, (8 * s + t) * kPairStride + g + 7, c);
      issue(slot);                                                       // the slot's entries are in use above
      if ((++since & 7) == 0) flush_single(c, tot);                      // at most 128 columns per accumulator
    }
    flush_single(c, tot);
    const int64_t v0 = quad_half(tot[0][0], tot[0][1]), v1 = quad_half(tot[1][0], tot[1][1]);
    const int64_t v2 = quad_half(tot[0][2], tot[0][3]), v3 = quad_half(tot[1][2], tot[1][3]);
    int64_t(*sum)[RT][2][2] = sums[p & 1];
    if ((t & 1) == 0) {
      sum[cg][mt * 16 + g][0][t >> 1] = v0;
      sum[cg][mt * 16 + g][1][t >> 1] = v1;
      sum[cg][mt * 16 + g + 8][0][t >> 1] = v2;
      sum[cg][mt * 16 + g + 8][1][t >> 1] = v3;
    }
    __syncthreads();
    if (tid < 2 * RT) {                                                  // whole warps
      int64_t hi = 0, lo = 0;
#pragma unroll
      for (int q = 0; q < CG; q++) {
        hi += sum[q][tid >> 1][pt][0];
        lo += sum[q][tid >> 1][pt][1];
      }
      const int r = base + p * RT + (tid >> 1);
      double s = scaled_sum(hi, lo, 88 + re + E - kBias);
      const double to = r < k ? b1[2 * r + pt] : b2;
      const int f1 = max(exp_field(s), exp_field(to)), field = max(f1, __shfl_xor_sync(0xffffffffu, f1, 1));
      // r = 0 and rows of zeros have no sum
      const bool redo = r > 0 && r < m && re > 1 - kBias && below_guard(field, re + E);
      for (unsigned todo = __ballot_sync(0xffffffffu, redo); todo; todo &= todo - 1) {   // a row's two lanes are neighbours
        const int at = __ffs(todo) - 1, row = base + p * RT + ((tid & ~31) + at) / 2;
        todo &= todo - 1;
        const double2 d = row_dot(P + row, S.ld, min(row, k), reinterpret_cast<const double2*>(b1), 1);
        if (lane >> 1 == at >> 1) s = scale2(pt ? d.y : d.x, re + 62);
      }
      if (E == 0x7ff || re == kRowNonFinite) s = nan("");
      const double a = s + (r < k ? b1[2 * r + pt] : 0.0);
      const double o = __shfl_xor_sync(0xffffffffu, a, 1);               // the other part
      if (r < m) {
        // D^{-1} (a, o): real part dx a - dy o, imaginary part dx a + dy o (a, o swapped)
        if (r < k)
          reinterpret_cast<double*>(zout + S.first + r)[pt] = fma(dinv.x, a, pt ? dinv.y * o : -dinv.y * o);
        else
          reinterpret_cast<double*>(u + S.wbase + uw)[pt] = b2 - s;
      }
    }
    load_row(p + 1);
  }
}

// Backward, ncol blocks of 32 pivot columns x one row chunk per task: sums over the chunk's rows r > j
// of P[r][j] vec[r], vec = (z, -x[ancestor rows]), with each panel row's exponent folded into vec's,
// gathered and converted once per task.  4 warps = 2 column tiles x 2 groups of 16-row steps.  A
// supernode of one chunk is finished here, else by the last CTA of each column block (bwd_finish).
__global__ void __launch_bounds__(128, 4) k_bwd_dig(const int4* tasks, const SnDev* sn, const int32_t* rowlist,
                                                    const double2* panels, const int16_t* rexp,
                                                    const uint8_t* colnz, const double2* zin, double2* x,
                                                    double2* partial, int rows,
                                                    int rpad, int ncol, const int4* fins, unsigned int* counters) {
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint4* ring = reinterpret_cast<uint4*>(smem_raw);                      // 4 warps x kRing x 8 x 32
  double* vec = reinterpret_cast<double*>(ring + 4 * kRing * 256);       // rpad x 2
  uint32_t* vre = reinterpret_cast<uint32_t*>(vec + 2 * rpad);
  uint32_t* vim = vre + (rpad / 2) * kPairStride;
  int* vex = reinterpret_cast<int*>(vim + (rpad / 2) * kPairStride);     // rpad
  __shared__ int64_t sums[2][2][32][2][2];                               // [block parity][group][column][part][half]
  __shared__ int red[4];
  const int4 tk = tasks[blockIdx.x];
  const SnDev S = sn[tk.x];
  const int k = S.k, m = S.m, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int g = lane >> 2, t = lane & 3, ct = wid & 1, sl = wid >> 1;
  const int r0 = tk.z * rows, r1 = min(m, r0 + rows);
  const int nblk = min(ncol, (k - tk.y * 32 + 31) / 32);
  const uint4* P = reinterpret_cast<const uint4*>(panels + S.paneloff);
  const int nst = (r1 - r0 + 15) / 16;
  uint4* myring = ring + wid * (kRing * 256) + lane;
  // first step of this warp in block p: those whose rows all lie at or above the tile's first
  // column hold nothing
  auto first = [&](int p) {
    const int j0 = (tk.y + p) * 32 + ct * 16;
    const int f = j0 < k ? max(0, (j0 + 1 - r0) / 16) : nst;
    return f + ((sl - f) & 1);
  };
  int ip = 0, is = first(0);                                             // next step to copy: block, step
  auto issue = [&](int slot) {
    while (ip < nblk && is >= nst) {
      ip++;
      is = first(ip);
    }
    if (ip < nblk) {
      const int ja = (tk.y + ip) * 32 + ct * 16 + g, jb = ja + 8;
      const uint4 *Pa = P + int64_t(ja) * S.ld, *Pb = P + int64_t(jb) * S.ld;
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const int r = r0 + 16 * is + 4 * t + q;
        if (ja < k && r < r1 && r > ja) cp_async16(myring + slot * 256 + (2 * q) * 32, Pa + r);
        if (jb < k && r < r1 && r > jb) cp_async16(myring + slot * 256 + (2 * q + 1) * 32, Pb + r);
      }
      is += 2;
    }
    cp_async_commit();
  };
#pragma unroll
  for (int q = 0; q < kRing; q++) issue(q);
  const int32_t* rl = rowlist + S.rowoff;
  int e = -4000, bad = 0;
  pdl_wait();
  const int pt = tid & 1;
#pragma unroll 4
  for (int q = tid; q < 2 * (r1 - r0); q += 128) {
    const int r = r0 + (q >> 1);
    const double v = r < k ? __ldcg(reinterpret_cast<const double*>(zin + S.first + r) + pt)
                           : -__ldcg(reinterpret_cast<const double*>(x + rl[r]) + pt);
    const int re = rexp[S.eoff + r];
    vec[q] = v;
    if (pt == 0) vex[q >> 1] = re;
    const int ev = exp_field(v);
    bad |= (ev == 0x7ff) | (re == kRowNonFinite);
    e = max(e, max(ev, 1) + re);
  }
  const bool nonfinite = __syncthreads_or(bad) != 0;
  const int E = block_max(e, red);
  for (int q = tid; q < 16 * nst; q += 128) {
    const int p = q >> 1, r = 2 * p;
    double x0 = 0.0, x1 = 0.0;
    int e0 = 0, e1 = 0;
    if (r < r1 - r0) {
      x0 = vec[2 * r + pt];
      e0 = vex[r];
    }
    if (r + 1 < r1 - r0) {
      x1 = vec[2 * r + 2 + pt];
      e1 = vex[r + 1];
    }
    uint32_t* dst = (pt ? vim : vre) + ((p & ~7) + pair_pos_bwd(p & 7)) * kPairStride;
    put_pair(dst, to_digits(x0, 1 + E - max(exp_field(x0), 1) - e0), to_digits(x1, 1 + E - max(exp_field(x1), 1) - e1));
  }
  __syncthreads();
  const bool single = m <= rows;
  int it = 0;
  for (int p = 0; p < nblk; p++) {
    const int j0 = (tk.y + p) * 32 + ct * 16, ja = j0 + g, jb = ja + 8;
    const bool fullcols = j0 + 15 < k;
    const int j = (tk.y + p) * 32 + (tid >> 1);
    const double zj = single && tid < 64 && j < k ? __ldcg(reinterpret_cast<const double*>(zin + S.first + j) + pt) : 0.0;
    float c[4][4];
    int tot[2][4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      c[0][q] = c[1][q] = c[2][q] = c[3][q] = 0.f;
      tot[0][q] = tot[1][q] = 0;
    }
    int since = 0;
    for (int s = first(p); s < nst; s += 2, it++) {
      cp_async_wait<kRing - 1>();
      const int slot = it % kRing;
      uint4 raw[8];
#pragma unroll
      for (int q = 0; q < 8; q++) raw[q] = myring[slot * 256 + q * 32];
      const int rs = r0 + 16 * s;
      if (!fullcols || rs + 16 > r1 || rs <= j0 + 15) {
#pragma unroll
        for (int q = 0; q < 4; q++) {
          const int r = rs + 4 * t + q;
          if (ja >= k || r >= r1 || r <= ja) raw[2 * q] = zero_entry();
          if (jb >= k || r >= r1 || r <= jb) raw[2 * q + 1] = zero_entry();
        }
      }
      step_single(raw, vre, vim, (8 * s + t) * kPairStride + g + 7, c);
      issue(slot);
      if ((++since & 7) == 0) flush_single(c, tot);
    }
    flush_single(c, tot);
    const int64_t v0 = quad_half(tot[0][0], tot[0][1]), v1 = quad_half(tot[1][0], tot[1][1]);
    const int64_t v2 = quad_half(tot[0][2], tot[0][3]), v3 = quad_half(tot[1][2], tot[1][3]);
    int64_t(*sum)[32][2][2] = sums[p & 1];
    if ((t & 1) == 0) {
      sum[sl][ct * 16 + g][0][t >> 1] = v0;
      sum[sl][ct * 16 + g][1][t >> 1] = v1;
      sum[sl][ct * 16 + g + 8][0][t >> 1] = v2;
      sum[sl][ct * 16 + g + 8][1][t >> 1] = v3;
    }
    __syncthreads();
    if (tid < 64) {
      double s = scaled_sum(sum[0][tid >> 1][pt][0] + sum[1][tid >> 1][pt][0],
                            sum[0][tid >> 1][pt][1] + sum[1][tid >> 1][pt][1], 88 + E - kBias);
      bool redo = j < k && j + 1 < r1 && below_guard(exp_field(s), E) && colnz[S.first + j];
      if (redo) redo = below_guard(exp_field(__ldcg(reinterpret_cast<const double*>(zin + S.first + j) + pt)), E);
      const int both = __shfl_xor_sync(0xffffffffu, int(redo), 1);           // a column's two parts
      redo = redo && both;
      for (unsigned todo = __ballot_sync(0xffffffffu, redo); todo; todo &= todo - 1) {
        const int at = __ffs(todo) - 1, col = (tk.y + p) * 32 + ((tid & ~31) + at) / 2;
        todo &= todo - 1;
        const double2 d = column_dot(P + int64_t(col) * S.ld + r0, max(col + 1 - r0, 0), r1 - r0,
                                     reinterpret_cast<const double2*>(vec), vex);
        if (lane >> 1 == at >> 1) s = pt ? d.y : d.x;
      }
      if (nonfinite) s = nan("");
      if (!single)
        reinterpret_cast<double*>(partial)[(int64_t(fins[tk.w + p].z) + tk.z) * 64 + tid] = s;
      else if (j < k)
        reinterpret_cast<double*>(x + S.first + j)[pt] = zj + s;
    }
  }
  if (!single)
    for (int p = 0; p < nblk; p++) {
      bwd_finish<double2>(fins[tk.w + p], S, zin, partial, x, counters + tk.w + p);
      __syncthreads();                                                   // its shared ticket is used again
    }
}

// ---------------------------------------------------------------------------
// S right-hand sides (interleaved per row): step_multi, four right-hand sides per warp.  Panel
// digits are unpacked once per warp.
// ---------------------------------------------------------------------------
namespace {

// Digits of a block of kb values x S right-hand sides (src: row-major kb x S, rows >= cnt are
// zero) into bd[pair][digit][right-hand side][part]; the exponents of each right-hand side are
// already in ex.  rowe: row exponents folded in (backward), or null.
template <int S, bool BWD>
__device__ __forceinline__ void put_digits_multi(uint32_t* bd, int pstride, const double2* src, int cnt, int kb,
                                                 const int* ex, const int* rowe) {
  for (int q = threadIdx.x; q < (kb / 2) * S * 2; q += 256) {
    const int part = q & 1, i = (q >> 1) % S, p = (q >> 1) / S;
    const int r = 2 * p, E = ex[i];
    double x = 0.0, y = 0.0;
    int e0 = 0, e1 = 0;
    if (r < cnt) {
      const double2 v = src[r * S + i];
      x = part ? v.y : v.x;
      if (BWD) e0 = rowe[r];
    }
    if (r + 1 < cnt) {
      const double2 v = src[(r + 1) * S + i];
      y = part ? v.y : v.x;
      if (BWD) e1 = rowe[r + 1];
    }
    const uint64_t dx = to_digits(x, 1 + E - max(exp_field(x), 1) - e0);
    const uint64_t dy = to_digits(y, 1 + E - max(exp_field(y), 1) - e1);
    uint32_t* dst = bd + ((p & ~7) + (BWD ? pair_pos_bwd(p & 7) : (p & 7))) * pstride + 2 * i + part;
    uint32_t o[4];
    word_digits(uint32_t(dx >> 32), uint32_t(dy >> 32), o);
#pragma unroll
    for (int d = 0; d < 4; d++) dst[d * 2 * S] = o[d];
    word_digits(uint32_t(dx), uint32_t(dy), o);
#pragma unroll
    for (int d = 0; d < 4; d++) dst[(4 + d) * 2 * S] = o[d];
  }
}

// per right-hand side: largest exponent field (plus row exponent) of a block of values; 256
// threads = 256 / S rows at a time, right-hand side fastest
template <int S, bool BWD>
__device__ __forceinline__ void block_exponents(const double2* src, int cnt, int* ex, int* nonfin, const int* rowe) {
  const int i = threadIdx.x % S;
  int e = BWD ? -4000 : 1, bad = 0;
  for (int r = threadIdx.x / S; r < cnt; r += 256 / S) {
    const double2 v = src[r * S + i];
    const int ev = max(exp_field(v.x), exp_field(v.y));
    bad |= ev == 0x7ff;
    if (BWD) {
      bad |= rowe[r] == kRowNonFinite;
      e = max(e, max(ev, 1) + rowe[r]);
    } else {
      e = max(e, ev);
    }
  }
#pragma unroll
  for (int o = 16; o >= S; o >>= 1) {
    e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    bad |= __shfl_xor_sync(0xffffffffu, bad, o);
  }
  if ((threadIdx.x & 31) < S) {
    atomicMax(&ex[i], e);
    if (bad) atomicOr(&nonfin[i], 1);
  }
}

}  // namespace

// columns (forward) or rows (backward) whose digits are in shared memory at once, at most 128 per
// group of steps, so that no accumulator takes more.  Each such block costs three barriers, the
// conversion and a flush (20 FP64 instructions a warp), so it is as long as a supernode is wide.
template <int S> constexpr int kMultiKb = S == 4 ? 256 : 128;
template <int S> constexpr int kMultiPairStride = 16 * S + 8;     // words; 8 t mod 32 differ

// Forward: 16 MT rows x S right-hand sides per task; 8 warps = S / 4 groups of four
// right-hand sides x MT row tiles x KG groups of 16-column steps.
template <int S, int MT>
__global__ void __launch_bounds__(256) k_fwd_dig_multi(const int2* tasks, const SnDev* sn, const uint32_t* cptr,
                                                       const uint32_t* wpos, const double2* panels,
                                                       const int16_t* rexp, const double2* tin, double2* zout,
                                                       double2* u, int kpad) {
  constexpr int NT = S / 4, KG = 8 / (NT * MT), KB = kMultiKb<S>, PS = kMultiPairStride<S>, RT = 16 * MT;
  static_assert(NT * MT * KG == 8, "eight warps");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* b1 = reinterpret_cast<double2*>(smem_raw);                    // kpad x S
  double2* part = b1 + kpad * S;                                          // KG x RT x S
  uint32_t* bd = reinterpret_cast<uint32_t*>(part + KG * RT * S);        // KB / 2 x PS
  __shared__ int ex[2][S], exmax[S], nonfin[S];
  const int2 tk = tasks[blockIdx.x];
  const SnDev Sn = sn[tk.x];
  const int k = Sn.k, m = Sn.m, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int g = lane >> 2, t = lane & 3, nt = wid % NT, mt = (wid / NT) % MT, kg = wid / (NT * MT);
  const uint32_t* cp = cptr + Sn.rowoff + Sn.id;
  const int row0 = tk.y * RT + mt * 16, ra = row0 + g, rb = ra + 8;
  const int ja = ra < m ? min(ra, k) : 0, jb = rb < m ? min(rb, k) : 0;
  const int jend = min(min(tk.y * RT + RT - 1, m - 1), k);               // columns any row of the task needs
  const uint4* P = reinterpret_cast<const uint4*>(panels + Sn.paneloff);
  uint4 raw[8];
  auto load = [&](int s) {
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int j = 16 * s + 2 * t + (q & 1) + 8 * (q >> 1);
      const uint4* col = P + int64_t(j) * Sn.ld;
      raw[2 * q] = j < ja ? ld_panel(col + ra) : zero_entry();
      raw[2 * q + 1] = j < jb ? ld_panel(col + rb) : zero_entry();
    }
  };
  if (tid < S) {
    ex[0][tid] = 1;
    exmax[tid] = 1;
    nonfin[tid] = 0;
  }
  if (16 * kg < jend) load(kg);
  gather_rows<double2, S>(b1, tin + int64_t(Sn.first) * S, cp, u + Sn.ubase * S, k);
  UpdateRows<double2, S, RT> up;
  up.load(Sn, cp, wpos, u, tk.y * RT);
  float cr[8][4], ci[8][4];
#pragma unroll
  for (int d = 0; d < 8; d++)
#pragma unroll
    for (int q = 0; q < 4; q++) cr[d][q] = ci[d][q] = 0.f;
  double2 acc[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
  const int ea = ra < m ? rexp[Sn.eoff + ra] : 0, eb = rb < m ? rexp[Sn.eoff + rb] : 0;
  const int rhs = 4 * nt + t;                                             // this lane's right-hand side
  __syncthreads();
  for (int j0 = 0, blk = 0; j0 < jend; j0 += KB, blk++) {
    int* exb = ex[blk & 1];
    block_exponents<S, false>(b1 + j0 * S, min(KB, k - j0), exb, nonfin, nullptr);
    __syncthreads();
    put_digits_multi<S, false>(bd, PS, b1 + j0 * S, min(KB, k - j0), min(KB, (jend - j0 + 15) / 16 * 16), exb, nullptr);
    if (tid < S) {
      ex[(blk + 1) & 1][tid] = 1;
      exmax[tid] = max(exmax[tid], exb[tid]);
    }
    __syncthreads();
    for (int s = j0 / 16 + kg; s < (j0 + KB) / 16 && 16 * s < jend; s += KG) {
      step_multi(raw, bd + (8 * (s - j0 / 16) + t) * PS + 8 * nt + g, 2 * S, PS, cr, ci);
      if (16 * (s + KG) < jend) load(s + KG);
    }
    flush_multi(cr, ci, acc, ea + exb[rhs] - kBias, eb + exb[rhs] - kBias);
    __syncthreads();                                                      // bd and ex are reused
  }
  part[(kg * RT + mt * 16 + g) * S + rhs] = acc[0];
  part[(kg * RT + mt * 16 + g + 8) * S + rhs] = acc[1];
  __syncthreads();
#pragma unroll
  for (int n = 0; n < up.N; n++) {
    const int e = tid + 256 * n, i = e % S, r = tk.y * RT + e / S;
    const bool mine = e < RT * S && r < m;
    double2 s = make_double2(0.0, 0.0);
    int re = 0;
    if (mine) {
      s = part[e];
#pragma unroll
      for (int q = 1; q < KG; q++) s = cadd(s, part[q * RT * S + e]);
      re = rexp[Sn.eoff + r];
    }
    bool redo = mine && r > 0 && re > 1 - kBias && below_guard(max(exp_field(s.x), exp_field(s.y)), re + exmax[i]);
    if (redo) {
      const double2 to = r < k ? b1[r * S + i] : up.b2[n];
      redo = below_guard(max(exp_field(to.x), exp_field(to.y)), re + exmax[i]);
    }
    for (unsigned todo = __ballot_sync(0xffffffffu, redo); todo; todo &= todo - 1) {
      const int at = __ffs(todo) - 1, ea = e - lane + at, row = tk.y * RT + ea / S;
      const double2 d = row_dot(P + row, Sn.ld, min(row, k), b1 + ea % S, S);
      if (lane == at) s = make_double2(scale2(d.x, re + 62), scale2(d.y, re + 62));
    }
    if (!mine) continue;
    if (nonfin[i] || re == kRowNonFinite) s = make_double2(nan(""), nan(""));
    if (r < k)
      zout[int64_t(Sn.first + r) * S + i] = cmul(panels[Sn.paneloff + r + int64_t(r) * Sn.ld], cadd(b1[r * S + i], s));
    else
      u[(Sn.wbase + up.to[n]) * S + i] = csub(up.b2[n], s);
  }
}

// Backward: 32 pivot columns x S right-hand sides x one chunk of kMultiBwdRows rows per task.
template <int S>
__global__ void __launch_bounds__(256) k_bwd_dig_multi(const int4* tasks, const SnDev* sn, const int32_t* rowlist,
                                                       const double2* panels, const int16_t* rexp,
                                                       const uint8_t* colnz, const double2* zin, double2* x,
                                                       double2* partial,
                                                       const int4* fins, unsigned int* counters) {
  constexpr int NT = S / 4, KG = 4 / NT, KB = kMultiBwdRows, PS = kMultiPairStride<S>, ROWS = kMultiBwdRows;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* vec = reinterpret_cast<double2*>(smem_raw);                   // ROWS x S; then KG x 32 x S partial sums
  uint32_t* bd = reinterpret_cast<uint32_t*>(vec + ROWS * S);            // KB / 2 x PS
  __shared__ int ex[2][S], nonfin[S], vex[ROWS];
  __shared__ unsigned int ticket;
  const int4 tk = tasks[blockIdx.x];
  const SnDev Sn = sn[tk.x];
  const int k = Sn.k, m = Sn.m, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int g = lane >> 2, t = lane & 3, nt = wid % NT, ct = (wid / NT) & 1, kg = wid / (2 * NT);
  const int r0 = tk.z * ROWS, r1 = min(m, r0 + ROWS), cnt = r1 - r0;
  const int j0 = tk.y * 32 + ct * 16, ja = j0 + g, jb = ja + 8;
  const uint4* P = reinterpret_cast<const uint4*>(panels + Sn.paneloff);
  const uint4* Pa = P + int64_t(ja < k ? ja : 0) * Sn.ld;
  const uint4* Pb = P + int64_t(jb < k ? jb : 0) * Sn.ld;
  const int nst = (cnt + 15) / 16;
  uint4 raw[8];
  auto load = [&](int s) {
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int r = r0 + 16 * s + 4 * t + q;
      raw[2 * q] = (ja < k && r < r1 && r > ja) ? ld_panel(Pa + r) : zero_entry();
      raw[2 * q + 1] = (jb < k && r < r1 && r > jb) ? ld_panel(Pb + r) : zero_entry();
    }
  };
  if (tid < S) {
    ex[0][tid] = -4000;
    nonfin[tid] = 0;
  }
  if (kg < nst) load(kg);
  const int32_t* rl = rowlist + Sn.rowoff;
  for (int r = tid; r < cnt; r += 256) vex[r] = rexp[Sn.eoff + r0 + r];
  {
    constexpr int U = ROWS * S / 256 < 4 ? ROWS * S / 256 : 4;             // row indices of U values, then the values
    for (int e0 = tid; e0 < cnt * S; e0 += 256 * U) {
      int32_t at[U];
#pragma unroll
      for (int n = 0; n < U; n++) {
        const int r = r0 + (e0 + 256 * n) / S;
        at[n] = r < r1 && r >= k ? rl[r] : 0;
      }
#pragma unroll
      for (int n = 0; n < U; n++) {
        const int e = e0 + 256 * n, r = r0 + e / S, i = e % S;
        if (r < r1) vec[e] = r < k ? ldv(zin + int64_t(Sn.first + r) * S + i) : cneg(ldv(x + int64_t(at[n]) * S + i));
      }
    }
  }
  float cr[8][4], ci[8][4];
#pragma unroll
  for (int d = 0; d < 8; d++)
#pragma unroll
    for (int q = 0; q < 4; q++) cr[d][q] = ci[d][q] = 0.f;
  double2 acc[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
  const int rhs = 4 * nt + t;
  __syncthreads();
  for (int q0 = 0, blk = 0; q0 < cnt; q0 += KB, blk++) {
    int* exb = ex[blk & 1];
    const int nr = min(KB, cnt - q0);
    block_exponents<S, true>(vec + q0 * S, nr, exb, nonfin, vex + q0);
    __syncthreads();
    put_digits_multi<S, true>(bd, PS, vec + q0 * S, nr, (nr + 15) / 16 * 16, exb, vex + q0);
    if (tid < S) ex[(blk + 1) & 1][tid] = -4000;
    __syncthreads();
    for (int s = q0 / 16 + kg; s < (q0 + KB) / 16 && s < nst; s += KG) {
      step_multi(raw, bd + (8 * (s - q0 / 16) + t) * PS + 8 * nt + g, 2 * S, PS, cr, ci);
      if (s + KG < nst) load(s + KG);
    }
    flush_multi(cr, ci, acc, exb[rhs] - kBias, exb[rhs] - kBias);
    __syncthreads();
  }
  vec[(kg * 32 + ct * 16 + g) * S + rhs] = acc[0];
  vec[(kg * 32 + ct * 16 + g + 8) * S + rhs] = acc[1];
  __syncthreads();
  const bool single = m <= ROWS;
  double2* out = partial + int64_t(blockIdx.x) * 32 * S;
  for (int e = tid; e < 32 * S; e += 256) {
    double2 s = vec[e];
#pragma unroll
    for (int q = 1; q < KG; q++) s = cadd(s, vec[q * 32 * S + e]);
    const int j = tk.y * 32 + e / S;
    bool redo = j < k && j + 1 < r1 && below_guard(max(exp_field(s.x), exp_field(s.y)), ex[0][e % S]) &&
                colnz[Sn.first + j];
    if (redo) {
      const double2 to = ldv(zin + int64_t(Sn.first + j) * S + e % S);
      redo = below_guard(max(exp_field(to.x), exp_field(to.y)), ex[0][e % S]);
    }
    for (unsigned todo = __ballot_sync(0xffffffffu, redo); todo; todo &= todo - 1) {
      const int at = __ffs(todo) - 1, ea = e - lane + at, ia = ea % S, col = tk.y * 32 + ea / S;
      double2 d = make_double2(0.0, 0.0);                                  // vec holds sums now: from global memory
      for (int r = max(col + 1, r0) + lane; r < r1; r += 32) {
        const double2 v = r < k ? ldv(zin + int64_t(Sn.first + r) * S + ia) : cneg(ldv(x + int64_t(rl[r]) * S + ia));
        const int ev = vex[r - r0] + 62;
        d = cmad(entry_value(__ldg(P + int64_t(col) * Sn.ld + r)), make_double2(scale2(v.x, ev), scale2(v.y, ev)), d);
      }
      d = warp_sum(d);
      if (lane == at) s = d;
    }
    if (nonfin[e % S]) s = make_double2(nan(""), nan(""));
    if (!single)
      out[e] = s;
    else if (j < k)
      x[int64_t(Sn.first + j) * S + e % S] = cadd(ldv(zin + int64_t(Sn.first + j) * S + e % S), s);
  }
  if (single) return;
  // last CTA of the column block: partials in chunk order (no CTA waits on another)
  const int4 fin = fins[tk.w];
  __threadfence();
  __syncthreads();
  if (tid == 0) ticket = atomicAdd(counters + tk.w, 1u);
  __syncthreads();
  if (ticket != unsigned(fin.w) - 1) return;
  __threadfence();
  for (int e = tid; e < 32 * S; e += 256) {
    const int j = fin.y * 32 + e / S;
    if (j >= k) continue;
    double2 a = make_double2(0.0, 0.0);
    for (int ch = 0; ch < fin.w; ch++) a = cadd(a, ldv(partial + int64_t(fin.z + ch) * 32 * S + e));
    x[int64_t(Sn.first + j) * S + e % S] = cadd(ldv(zin + int64_t(Sn.first + j) * S + e % S), a);
  }
  if (tid == 0) counters[tk.w] = 0u;
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
namespace {

constexpr size_t kRingBytes = size_t(4) * kRing * 256 * 16;
size_t fwd_smem(int kpad) { return kRingBytes + size_t(kpad) * 16 + size_t(kpad) * kPairStride * 4; }
size_t bwd_smem(int rpad) { return kRingBytes + size_t(rpad) * 20 + size_t(rpad) * kPairStride * 4; }
template <int S, int MT> size_t fwd_multi_smem(int kpad) {
  constexpr int KG = 8 / (S / 4 * MT);
  return size_t(kpad) * S * 16 + size_t(KG) * 16 * MT * S * 16 + size_t(kMultiKb<S> / 2) * kMultiPairStride<S> * 4;
}
template <int S> size_t bwd_multi_smem() {
  return size_t(kMultiBwdRows) * S * 16 + size_t(kMultiBwdRows / 2) * kMultiPairStride<S> * 4;
}
template <typename K> void allow_smem(K kern) {
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
}
void set_attrs_dig() {
  static const bool done = [] {
    allow_smem(k_fwd_dig<1>);
    allow_smem(k_fwd_dig<4>);
    allow_smem(k_bwd_dig);
    allow_smem(k_fwd_dig_multi<4, 1>);
    allow_smem(k_fwd_dig_multi<4, 4>);
    allow_smem(k_fwd_dig_multi<8, 1>);
    allow_smem(k_fwd_dig_multi<8, 4>);
    allow_smem(k_fwd_dig_multi<16, 1>);
    allow_smem(k_fwd_dig_multi<16, 2>);
    allow_smem(k_bwd_dig_multi<4>);
    allow_smem(k_bwd_dig_multi<8>);
    allow_smem(k_bwd_dig_multi<16>);
    return true;
  }();
  (void)done;
}

}  // namespace

void launch_to_digits(const FactorDev& F, cudaStream_t st) {
  cudaMemsetAsync(F.colnz, 0, size_t(F.ntot), st);
  for (int l = 0; l < F.snlev; l++) {
    const int64_t b = F.h_fwd_ptr[l], e = F.h_fwd_ptr[l + 1];
    if (e == b) continue;
    add_launches(1);
    if (F.h_fwd_rt[l] == 16)
      k_to_digits<16><<<unsigned(e - b), 256, 0, st>>>(F.fwd_tasks + b, F.ssn, (double2*)F.panels, F.rexp,
                                                                F.colnz);
    else
      k_to_digits<64><<<dim3(unsigned(e - b), unsigned(F.h_fwd_rt[l] / 64)), 256, 0, st>>>(F.fwd_tasks + b, F.ssn,
                                                                                           (double2*)F.panels, F.rexp, F.colnz);
  }
}

void launch_solve_dig(const FactorDev& F, cudaStream_t st) {
  set_attrs_dig();
  const double2* P = (const double2*)F.panels;
  double2 *t = (double2*)F.t_loc, *z = (double2*)F.z_loc, *x = (double2*)F.x_loc, *u = (double2*)F.u_ws;
  const bool pdl = pdl_enabled();
  if (F.level_events) cudaEventRecord(F.level_events[0], st);
  for (int l = 0; l < F.snlev; l++) {
    const int64_t b = F.h_fwd_ptr[l], e = F.h_fwd_ptr[l + 1];
    if (e > b) {
      add_launches(1);
      const int kpad = F.h_lev_k[l];
      if (F.h_fwd_rt[l] == 16)
        launch_level(k_fwd_dig<1>, e - b, 128, fwd_smem(kpad), st, pdl, F.fwd_tasks + b, F.ssn, F.cptr, F.wpos, P,
                     F.rexp, t, z, u, kpad, 1);
      else
        launch_level(k_fwd_dig<4>, e - b, 128, fwd_smem(kpad), st, pdl, F.fwd_tasks + b, F.ssn, F.cptr, F.wpos, P,
                     F.rexp, t, z, u, kpad, F.h_fwd_rt[l] / 64);
    }
    if (F.level_events) cudaEventRecord(F.level_events[1 + l], st);
  }
  for (int l = F.snlev - 1; l >= 0; l--) {
    const int64_t b = F.h_bwd_ptr[l], e = F.h_bwd_ptr[l + 1];
    if (e > b) {
      add_launches(1);
      const int rows = F.h_bwd_rows[l], rpad = (std::min(rows, F.h_lev_m[l]) + 15) / 16 * 16;
      launch_level(k_bwd_dig, e - b, 128, bwd_smem(rpad), st, pdl, F.bwd_tasks + b, F.ssn, F.rowlist, P, F.rexp, F.colnz, z, x,
                   (double2*)F.bwd_partial, rows, rpad, F.h_bwd_cb[size_t(l)], F.bfin_tasks, F.bwd_counters);
    }
    if (F.level_events) cudaEventRecord(F.level_events[1 + F.snlev + (F.snlev - 1 - l)], st);
  }
}

template <int S, int MT>
static void fwd_multi_level(const FactorDev& F, int l, int64_t b, int64_t e, cudaStream_t st) {
  const int kpad = F.h_lev_k[l];
  k_fwd_dig_multi<S, MT><<<unsigned(e - b), 256, fwd_multi_smem<S, MT>(kpad), st>>>(
      F.mfwd_tasks + b, F.ssn, F.cptr, F.wpos, (const double2*)F.panels, F.rexp, (const double2*)F.mt_loc,
      (double2*)F.mz_loc, (double2*)F.mu_ws, kpad);
}

template <int S>
static void solve_dig_multi_t(const FactorDev& F, cudaStream_t st) {
  constexpr int MTW = S == 16 ? 2 : 4;
  for (int l = 0; l < F.snlev; l++) {
    const int64_t b = F.h_mfwd_ptr[l], e = F.h_mfwd_ptr[l + 1];
    if (e == b) continue;
    add_launches(1);
    if (F.h_mfwd_rt[l] == 16) fwd_multi_level<S, 1>(F, l, b, e, st);
    else fwd_multi_level<S, MTW>(F, l, b, e, st);
  }
  for (int l = F.snlev - 1; l >= 0; l--) {
    const int64_t b = F.h_mbwd_ptr[l], e = F.h_mbwd_ptr[l + 1];
    if (e == b) continue;
    add_launches(1);
    k_bwd_dig_multi<S><<<unsigned(e - b), 256, bwd_multi_smem<S>(), st>>>(
        F.mbwd_tasks + b, F.ssn, F.rowlist, (const double2*)F.panels, F.rexp, F.colnz, (const double2*)F.mz_loc,
        (double2*)F.mx_loc, (double2*)F.mbwd_partial, F.mbfin_tasks, F.mbwd_counters);
  }
}

void launch_solve_dig_multi(const FactorDev& F, int S, cudaStream_t st) {
  set_attrs_dig();
  if (S == 4) solve_dig_multi_t<4>(F, st);
  else if (S == 8) solve_dig_multi_t<8>(F, st);
  else solve_dig_multi_t<16>(F, st);
}

}  // namespace hz
