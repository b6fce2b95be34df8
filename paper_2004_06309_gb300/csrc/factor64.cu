// Complex128 products of the factorisation in digits on the tensor cores (digits.cuh): the
// off-diagonal panels (W = F21 T^T, L21 = W D^{-1}, G = L21 T), the Schur updates
// F22 -= W L21^T, and the products that merge solve supernodes.  On the FP64 units (2 FMAs per
// SM and clock) a complex product costs 2 SM-clocks; here 0.14, plus unpacking and the
// conversion of both operands (once per row block and column tile).
//
// A block's second factor, 16 complex columns, is expanded in shared memory as half2 digit
// planes; the first factor, 32 rows, is digit words.  8 warps = 2 row tiles x 4 groups of
// four columns.  At most 112 columns meet in an accumulator, fewer than the 128 that keep its
// sums exact.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "dev.h"
#include "digits.cuh"
#include "dmath.cuh"

namespace hz {

namespace {

constexpr int kPlane = 16 * 16 + 8;      // words per k pair: 8 digits x 32 real columns; 8 t mod 32 differ
constexpr int kRowPitch = 33;            // entries per column of a 32-row block: conflict-free fragments
constexpr int kMaxPairs = 4;             // k pairs per thread of an operand: 16 x 4 x 2 = 128 columns

__device__ __forceinline__ uint4 entry_digits(double2 v, int E) {
  const uint64_t a = to_digits(v.x, 1 + E - max(exp_field(v.x), 1));
  const uint64_t b = to_digits(v.y, 1 + E - max(exp_field(v.y), 1));
  return make_uint4(uint32_t(a), uint32_t(a >> 32), uint32_t(b), uint32_t(b >> 32));
}
__device__ __forceinline__ int entry_exp(double2 v) { return max(exp_field(v.x), exp_field(v.y)); }

// digits of the k pair (x, y) of complex column n
__device__ __forceinline__ void put_plane_pair(uint32_t* bd, int p, int n, uint4 x, uint4 y) {
  uint32_t* dst = bd + p * kPlane + 2 * n;
  uint32_t o[4];
#pragma unroll
  for (int part = 0; part < 2; part++) {
    word_digits(part ? x.w : x.y, part ? y.w : y.y, o);
#pragma unroll
    for (int d = 0; d < 4; d++) dst[d * 32 + part] = o[d];
    word_digits(part ? x.z : x.x, part ? y.z : y.x, o);
#pragma unroll
    for (int d = 0; d < 4; d++) dst[(4 + d) * 32 + part] = o[d];
  }
}

// The second factor held by a thread before its digits are written: column n = tid & 15, k pairs
// (tid >> 4) + 16 u.
struct Operand {
  double2 v[kMaxPairs][2];
  // get(n, kk): the entry, zero outside
  template <typename Get> __device__ __forceinline__ void load(int npairs, Get get) {
    const int n = threadIdx.x & 15, p0 = threadIdx.x >> 4;
#pragma unroll
    for (int u = 0; u < kMaxPairs; u++) {
      const int p = p0 + 16 * u;
      if (p < npairs) {
        v[u][0] = get(n, 2 * p);
        v[u][1] = get(n, 2 * p + 1);
      }
    }
  }
  // writes the planes of npairs k pairs and the columns' exponents; three barriers
  __device__ __forceinline__ void store(int npairs, uint32_t* bd, int* bexp) const {
    const int tid = threadIdx.x, n = tid & 15, p0 = tid >> 4;
    __syncthreads();                                   // the previous planes and exponents are used
    if (tid < 16) bexp[tid] = 1;
    int e = 1;
#pragma unroll
    for (int u = 0; u < kMaxPairs; u++)
      if (p0 + 16 * u < npairs) e = max(e, max(entry_exp(v[u][0]), entry_exp(v[u][1])));
    e = max(e, __shfl_xor_sync(0xffffffffu, e, 16));
    __syncthreads();
    if ((tid & 31) < 16) atomicMax(&bexp[n], e);
    __syncthreads();
    const int E = bexp[n];
#pragma unroll
    for (int u = 0; u < kMaxPairs; u++) {
      const int p = p0 + 16 * u;
      if (p < npairs) put_plane_pair(bd, p, n, entry_digits(v[u][0], E), entry_digits(v[u][1], E));
    }
    __syncthreads();
  }
};

// 32 rows x K of the first factor as digit words in shared memory ([kk][row], pitch kRowPitch) with
// the rows' exponents; get(row, kk) is called twice.  256 threads; ends with a barrier.
template <typename Get>
__device__ __forceinline__ void put_rows(uint4* A, int* aexp, int K16, Get get) {
  const int tid = threadIdx.x, row = tid & 31, c0 = tid >> 5;
  __syncthreads();
  if (tid < 32) aexp[tid] = 1;
  __syncthreads();
  int e = 1;
#pragma unroll 4
  for (int kk = c0; kk < K16; kk += 8) e = max(e, entry_exp(get(row, kk)));
  atomicMax(&aexp[row], e);
  __syncthreads();
  const int E = aexp[row];
#pragma unroll 4
  for (int kk = c0; kk < K16; kk += 8) A[kk * kRowPitch + row] = entry_digits(get(row, kk), E);
  __syncthreads();
}

__device__ __forceinline__ void zero_acc(float (*cr)[4], float (*ci)[4]) {
#pragma unroll
  for (int d = 0; d < 8; d++)
#pragma unroll
    for (int q = 0; q < 4; q++) cr[d][q] = ci[d][q] = 0.f;
}

// products of rows 16 mt.. of the digit words A with columns 4 nt.. of the planes, k steps [s0, s1)
__device__ __forceinline__ void tile_product(const uint4* A, const uint32_t* bd, int s0, int s1, int mt, int nt,
                                             float (*cr)[4], float (*ci)[4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  for (int s = s0; s < s1; s++) {
    uint4 raw[8];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const uint4* c = A + (16 * s + 2 * t + (q & 1) + 8 * (q >> 1)) * kRowPitch + 16 * mt + g;
      raw[2 * q] = c[0];
      raw[2 * q + 1] = c[8];
    }
    step_multi(raw, bd + (8 * s + t) * kPlane + 8 * nt + g, 32, kPlane, cr, ci);
  }
}

}  // namespace

// Off-diagonal panel of a supernode, 32 rows per task:
//   W = F21 T^T                 digits (and exponents) to the level scratch,
//   L21 = W D^{-1}              digits to the front's unused upper block F12 (row a of L21 in column
//                               k + a, contiguous),
//   G = L21 T                   over F21.
// Scratch of a supernode: W's digit words (r x k, column-major), then per row the exponents of W and L21.
__global__ void __launch_bounds__(256, 1) k_wg_dig(const int2* tasks, const SnDev* sn, const int64_t* scr_off,
                                                   double2* fronts, double2* scratch, DevStatus* status, int kpad) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint4* A = reinterpret_cast<uint4*>(smem_raw);                           // kpad x kRowPitch
  double2* Wf = reinterpret_cast<double2*>(A + kpad * kRowPitch);          // kpad x kRowPitch
  uint32_t* bd = reinterpret_cast<uint32_t*>(Wf + kpad * kRowPitch);       // kpad / 2 x kPlane
  __shared__ int aexp[32], bexp[16], lexp[32];
  __shared__ double2 dinv[128];
  const int2 tk = tasks[blockIdx.x];
  const SnDev S = sn[tk.x];
  const int k = S.k, m = S.m, r = m - k, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int g = lane >> 2, t = lane & 3, mt = wid & 1, nt = wid >> 1;
  double2* F = fronts + S.frontoff;
  const int R0 = tk.y * 32, nr = min(32, r - R0), K16 = (k + 15) / 16 * 16;
  double2* F21 = F + k + R0;
  const double2 z = make_double2(0.0, 0.0);
  Operand op;
  auto trow = [&](int j0) {                            // second factor of W: rows j of T, i < j
    op.load((min(j0 + 16, K16)) / 2, [&](int n, int i) {
      const int j = j0 + n;
      return (j < k && i < j) ? F[j + int64_t(i) * m] : z;
    });
  };
  auto tcol = [&](int j0) {                            // second factor of G: columns j of T, i > j, from i = j0
    op.load((K16 - j0) / 2, [&](int n, int i) {
      const int j = j0 + n;
      i += j0;
      return (j < k && i < k && i > j) ? F[i + int64_t(j) * m] : z;
    });
  };
  trow(0);
  for (int i = tid; i < k; i += 256) dinv[i] = F[i + int64_t(i) * m];
  put_rows(A, aexp, K16, [&](int row, int kk) { return (row < nr && kk < k) ? F21[row + int64_t(kk) * m] : z; });
  float cr[8][4], ci[8][4];
  for (int j0 = 0; j0 < k; j0 += 16) {
    op.store(min(j0 + 16, K16) / 2, bd, bexp);
    if (j0 + 16 < k) trow(j0 + 16);
    else tcol(0);
    const int j = j0 + 4 * nt + t;
    double2 acc[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const int row = 16 * mt + g + 8 * h;
      acc[h] = (row < nr && j < k) ? F21[row + int64_t(j) * m] : z;
    }
    zero_acc(cr, ci);
    tile_product(A, bd, 0, j0 / 16 + 1, mt, nt, cr, ci);
    const int en = bexp[4 * nt + t] - 2 * kBias;
    flush_multi(cr, ci, acc, aexp[16 * mt + g] + en, aexp[16 * mt + g + 8] + en);
    Wf[j * kRowPitch + 16 * mt + g] = acc[0];
    Wf[j * kRowPitch + 16 * mt + g + 8] = acc[1];
  }
  __syncthreads();
  // exponents of the rows of W and L21, then their digits; Wf becomes L21
  if (tid < 32) lexp[tid] = aexp[tid] = 1;
  __syncthreads();
  {
    const int row = tid & 31;
    int ew = 1, el = 1;
    for (int kk = tid >> 5; kk < k; kk += 8) {
      const double2 w = Wf[kk * kRowPitch + row];
      ew = max(ew, entry_exp(w));
      el = max(el, entry_exp(cmul(w, dinv[kk])));
    }
    atomicMax(&aexp[row], ew);
    atomicMax(&lexp[row], el);
    __syncthreads();
    const int EW = aexp[row], EL = lexp[row];
    // digits hold no infinity or NaN: report the matrix as one without usable pivots
    if (EW == 0x7ff || EL == 0x7ff) atomicOr(&status->zero_pivot, 1u);
    uint4* Wd = reinterpret_cast<uint4*>(scratch + scr_off[tk.x]);
    uint4* Ld = reinterpret_cast<uint4*>(F + int64_t(k) * m);
    for (int kk = tid >> 5; kk < K16; kk += 8) {
      const double2 w = kk < k ? Wf[kk * kRowPitch + row] : z;
      const double2 l = kk < k ? cmul(w, dinv[kk]) : z;
      const uint4 ld = entry_digits(l, EL);
      A[kk * kRowPitch + row] = ld;
      if (kk < k) {
        Wf[kk * kRowPitch + row] = l;
        if (row < nr) Wd[(R0 + row) + int64_t(kk) * r] = entry_digits(w, EW);
      }
    }
    __syncthreads();
    for (int e = tid; e < 32 * k; e += 256) {          // L21's rows, contiguous in F12
      const int i = e % k, a = e / k;
      if (a < nr) Ld[int64_t(R0 + a) * m + i] = A[i * kRowPitch + a];
    }
    if (tid < nr) reinterpret_cast<int2*>(Wd + int64_t(r) * k)[R0 + tid] = make_int2(aexp[tid], lexp[tid]);
  }
  for (int j0 = 0; j0 < k; j0 += 16) {
    op.store((K16 - j0) / 2, bd, bexp);
    if (j0 + 16 < k) tcol(j0 + 16);
    const int j = j0 + 4 * nt + t;
    double2 acc[2];
    acc[0] = Wf[j * kRowPitch + 16 * mt + g];
    acc[1] = Wf[j * kRowPitch + 16 * mt + g + 8];
    zero_acc(cr, ci);
    tile_product(A + j0 * kRowPitch, bd, 0, (K16 - j0) / 16, mt, nt, cr, ci);
    const int en = bexp[4 * nt + t] - 2 * kBias;
    flush_multi(cr, ci, acc, lexp[16 * mt + g] + en, lexp[16 * mt + g + 8] + en);
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const int row = 16 * mt + g + 8 * h;
      if (row < nr && j < k) F21[row + int64_t(j) * m] = acc[h];
    }
  }
}

// Schur update of the contribution block, lower triangle: 16 columns x up to kCbRows rows per task,
// F22[a][b] -= sum_i W[a][i] L21[b][i], from the digits k_wg_dig left.  L21's planes stay in shared
// memory while the task walks its rows; W's digit words are read by each warp from global memory
// (four warps share them through L1).
__global__ void __launch_bounds__(256, 1) k_cb_dig(const int4* tasks, const SnDev* sn, const int64_t* scr_off,
                                                   double2* fronts, const double2* scratch) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t* bd = reinterpret_cast<uint32_t*>(smem_raw);                    // kpad / 2 x kPlane
  const int4 tk = tasks[blockIdx.x];
  const SnDev S = sn[tk.x];
  const int k = S.k, m = S.m, r = m - k, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int g = lane >> 2, t = lane & 3, mt = wid & 1, nt = wid >> 1;
  const int nst = (k + 15) / 16;
  double2* F = fronts + S.frontoff;
  const uint4* Wd = reinterpret_cast<const uint4*>(scratch + scr_off[tk.x]);
  const int2* exps = reinterpret_cast<const int2*>(Wd + int64_t(r) * k);
  const uint4* Ld = reinterpret_cast<const uint4*>(F + int64_t(k) * m);
  const int b0 = tk.z * 16, a0 = tk.y * kCbRows, a1 = min(r, a0 + kCbRows);
  for (int e = tid; e < 8 * nst * 16; e += 256) {
    const int p = e % (8 * nst), n = e / (8 * nst), b = b0 + n;
    uint4 x = zero_entry(), y = x;
    if (b < r && 2 * p < k) x = Ld[int64_t(b) * m + 2 * p];
    if (b < r && 2 * p + 1 < k) y = Ld[int64_t(b) * m + 2 * p + 1];
    put_plane_pair(bd, p, n, x, y);
  }
  const int b = b0 + 4 * nt + t;
  const int eb = b < r ? exps[b].y : 1;
  __syncthreads();
  float cr[8][4], ci[8][4];
  for (int row0 = max(a0, b0 / 32 * 32) + 16 * mt; row0 < a1; row0 += 32) {
    if (row0 + 15 < b0) continue;
    const int ra = row0 + g, rb = ra + 8;
    const uint4 *Wa = Wd + ra, *Wb = Wd + rb;
    uint4 raw[8];
    auto load = [&](int s) {
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const int i = 16 * s + 2 * t + (q & 1) + 8 * (q >> 1);
        raw[2 * q] = (ra < a1 && i < k) ? __ldg(Wa + int64_t(i) * r) : zero_entry();
        raw[2 * q + 1] = (rb < a1 && i < k) ? __ldg(Wb + int64_t(i) * r) : zero_entry();
      }
    };
    load(0);
    const bool va = ra < a1 && b < r && ra >= b, vb = rb < a1 && b < r && rb >= b;
    double2* fa = F + (k + ra) + int64_t(k + b) * m;
    const double2 z = make_double2(0.0, 0.0);
    const double2 f0 = va ? fa[0] : z, f1 = vb ? fa[8] : z;
    const int ea = ra < a1 ? exps[ra].x : 1, ec = rb < a1 ? exps[rb].x : 1;
    zero_acc(cr, ci);
    for (int s = 0; s < nst; s++) {
      step_multi(raw, bd + (8 * s + t) * kPlane + 8 * nt + g, 32, kPlane, cr, ci);
      if (s + 1 < nst) load(s + 1);
    }
    double2 acc[2] = {z, z};
    flush_multi(cr, ci, acc, ea + eb - 2 * kBias, ec + eb - 2 * kBias);
    if (va) fa[0] = csub(f0, acc[0]);
    if (vb) fa[8] = csub(f1, acc[1]);
  }
}

// Merged solve supernodes (see kernels.cu): M[w + i, c] = (i >= ks ? M[w + i, c] : 0) -
// sum_q C(i, q) tmp[q, c] for i < ms, c < w, C = [T_s (unit diagonal); G_s]; 32 rows x 16 columns
// per block.
__global__ void __launch_bounds__(256, 1) k_merge_dig(double2* M, int ldm, int w, const double2* Ps, int lds, int ks,
                                                      int ms, const double2* tmp) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int K16 = (ks + 15) / 16 * 16;
  uint4* A = reinterpret_cast<uint4*>(smem_raw);                           // K16 x kRowPitch
  uint32_t* bd = reinterpret_cast<uint32_t*>(A + K16 * kRowPitch);         // K16 / 2 x kPlane
  __shared__ int aexp[32], bexp[16];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int g = lane >> 2, t = lane & 3, mt = wid & 1, nt = wid >> 1;
  const int i0 = blockIdx.x * 32, c0 = blockIdx.y * 16;
  const double2 z = make_double2(0.0, 0.0);
  Operand op;
  op.load(K16 / 2, [&](int n, int q) { return (c0 + n < w && q < ks) ? tmp[q + int64_t(ks) * (c0 + n)] : z; });
  put_rows(A, aexp, K16, [&](int row, int q) {
    const int i = i0 + row;
    if (i >= ms || q >= ks) return z;
    if (i >= ks || i > q) return Ps[i + int64_t(lds) * q];
    return i == q ? make_double2(1.0, 0.0) : z;
  });
  op.store(K16 / 2, bd, bexp);
  float cr[8][4], ci[8][4];
  zero_acc(cr, ci);
  tile_product(A, bd, 0, K16 / 16, mt, nt, cr, ci);
  const int c = c0 + 4 * nt + t, en = bexp[4 * nt + t] - 2 * kBias;
  double2 acc[2] = {z, z};
  flush_multi(cr, ci, acc, aexp[16 * mt + g] + en, aexp[16 * mt + g + 8] + en);
#pragma unroll
  for (int h = 0; h < 2; h++) {
    const int i = i0 + 16 * mt + g + 8 * h;
    if (i < ms && c < w) {
      double2* o = M + (w + i) + int64_t(ldm) * c;
      *o = csub(i >= ks ? *o : z, acc[h]);
    }
  }
}

namespace {
size_t rows_bytes(int K16) { return size_t(K16) * kRowPitch * 16; }
size_t plane_bytes(int K16) { return size_t(K16 / 2) * kPlane * 4; }
void set_attrs_factor64() {
  static const bool done = [] {
    cudaFuncSetAttribute(k_wg_dig, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    cudaFuncSetAttribute(k_cb_dig, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    cudaFuncSetAttribute(k_merge_dig, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    return true;
  }();
  (void)done;
}
}  // namespace

void launch_wg_dig(int64_t ntask, int maxk, const int2* tasks, const FactorDev& F, double2* fronts, double2* scratch,
                   DevStatus* status, cudaStream_t st) {
  set_attrs_factor64();
  const int K16 = (maxk + 15) / 16 * 16;
  add_launches(1);
  k_wg_dig<<<unsigned(ntask), 256, 2 * rows_bytes(K16) + plane_bytes(K16), st>>>(tasks, F.sn, F.scr_off, fronts,
                                                                                 scratch, status, K16);
}

void launch_cb_dig(int64_t ntask, int maxk, const int4* tasks, const FactorDev& F, double2* fronts,
                   const double2* scratch, cudaStream_t st) {
  set_attrs_factor64();
  add_launches(1);
  k_cb_dig<<<unsigned(ntask), 256, plane_bytes((maxk + 15) / 16 * 16), st>>>(tasks, F.sn, F.scr_off, fronts, scratch);
}

void launch_merge_dig(double2* M, int ldm, int w, const double2* Ps, int lds, int ks, int ms, const double2* tmp,
                      cudaStream_t st) {
  set_attrs_factor64();
  const int K16 = (ks + 15) / 16 * 16;
  add_launches(1);
  k_merge_dig<<<dim3(unsigned((ms + 31) / 32), unsigned((w + 15) / 16)), 256, rows_bytes(K16) + plane_bytes(K16), st>>>(
      M, ldm, w, Ps, lds, ks, ms, tmp);
}

}  // namespace hz
