// GMRES orthogonalisation: classical Gram-Schmidt passes (dots h = V^H w, updates w -= V h, and an
// update followed by the dots of the updated w), the squared norm of w, their fixed-order sums over
// the blocks, the Givens update of the Hessenberg column and the cycle-end triangular solve.  One
// launch serves a single vector or the S slots of a pseudo-block solve (grid.y = slot); a slot's
// arithmetic does not depend on the others.
//
// Bound: FP64 arithmetic (four FMAs per basis entry and pass, 2 per SM and clock: 59 us for 25
// columns of 349,461 rows) for long vectors; for short ones the chain of launches and of FP64
// instructions, each 64 clocks of a scheduler whatever its active lanes.  Hence: a warp's
// columns are summed over its lanes together (halving exchanges, 9 complex additions for 8 columns
// instead of 40); an update and the following dots share a launch; and for vectors of at most
// kFusedBlocks row chunks the last block of a pass adds the blocks' sums and, after the third
// pass, runs the Givens update, so an orthogonalisation takes three launches instead of eight.
// Measured (dots, update): 101, 80 us before, on 25 columns of 349,461 rows; 27, 8.6 us on 13
// columns of 2,197 rows with 6 us for each sum over blocks and 14 for Givens.
// A warp's loop is compiled for its own number of columns, and with at most four columns the warps
// share the rows.  With loops of 1, 2, 4 or 8 columns, unused ones skipped, CGS2 of 33 columns took
// 577 us at 349,461 rows and 3.45 ms at 2,368,333 (388 us and 2.22 ms so; 485 us and 2.51 ms with one
// launch per update and dot), of one column 105 and 422 us (69 and 166; 119 and 253).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "dev.h"
#include "dmath.cuh"

namespace hz {

namespace {

constexpr int kMaxCols = 64;
constexpr int kPartStride = kMaxCols + 1;
constexpr int kMinChunk = 64;
// the last block's own sum over this many blocks takes about as long as the launch it saves
constexpr int kFusedBlocks = 160;

// smallest power of two that holds NC values
template <int NC> constexpr int kPow2 = NC <= 1 ? 1 : (NC <= 2 ? 2 : (NC <= 4 ? 4 : 8));

// sums P (a power of two) complex values over a warp's lanes; the sum of value c ends in the lanes
// whose bits from 16 down spell c (most significant first)
template <int P> __device__ __forceinline__ double2 sum_columns(double2* v, int lane, int& c) {
  c = 0;
  int o = 16;
#pragma unroll
  for (int half = P / 2; half > 0; half >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < half; i++) {
      const double2 keep = up ? v[i + half] : v[i], give = up ? v[i] : v[i + half];
      v[i] = cadd(keep, shfl_xor(give, o));
    }
    c = 2 * c + (up ? 1 : 0);
  }
  double2 s = v[0];
  for (; o > 0; o >>= 1) s = cadd(s, shfl_xor(s, o));
  return s;
}

// acc[c] += the dots of column c (of C, every eighth one of the basis) over rows q0, q0 + step, .. < cnt
template <int C>
__device__ __forceinline__ void dot_rows(double2* acc, const double2* __restrict__ V, int64_t ld8, const double2* ws,
                                         int q0, int cnt, int step) {
  constexpr int U = C == 1 ? 8 : (C == 2 ? 4 : 2);
#pragma unroll U
  for (int q = q0; q < cnt; q += step) {
    const double2 x = ws[q];
#pragma unroll
    for (int c = 0; c < C; c++) acc[c] = cmadc(V[q + c * ld8], x, acc[c]);
  }
}
// the same for a warp that holds `mine` of at most C columns: a loop for each count.  Skipping columns
// inside one loop of C kept the FP64 units as busy as C of them
template <int C>
__device__ __forceinline__ void dot_rows_of(int mine, double2* acc, const double2* V, int64_t ld8, const double2* ws,
                                            int q0, int cnt, int step) {
  if (mine == C) dot_rows<C>(acc, V, ld8, ws, q0, cnt, step);
  else if constexpr (C > 1) dot_rows_of<C - 1>(mine, acc, V, ld8, ws, q0, cnt, step);
}

// Givens update of column j, one warp.  The chain over the earlier rotations is sequential; lanes 0-3
// hold the real and imaginary parts of its two results.  nrm2: |w|^2 after the passes.
__device__ void givens_update(const SlotGivens& p, int i, double nrm2) {
  const int lane = threadIdx.x & 31, j = p.j[i], m = p.m;
  double2* col = p.H + int64_t(i) * (m + 1) * m + int64_t(j) * (m + 1);
  double* cs = p.cs + int64_t(i) * m;
  double2 *sn = p.sn + int64_t(i) * m, *g = p.g + int64_t(i) * (m + 1);
  const double2 *h1 = p.h1 + int64_t(i) * kPartStride, *h2 = p.h2 + int64_t(i) * kPartStride;
  double* scal = p.scal + int64_t(i) * 8;
  // lane 0: hn = |w| after the passes, lane 1: before them
  double root = sqrt(lane == 0 ? nrm2 : h1[kMaxCols].x);
  const double hn = __shfl_sync(0xffffffffu, root, 0), w0 = __shfl_sync(0xffffffffu, root, 1);
  double2 hc[2];                                       // entries lane, lane + 32 of the column
#pragma unroll
  for (int q = 0; q < 2; q++) {
    const int r = lane + 32 * q;
    hc[q] = make_double2(0.0, 0.0);
    if (r <= j) hc[q] = cadd(h1[p.off + r], h2[p.off + r]);
    if (p.raw_h) {
      if (r <= j) p.raw_h[int64_t(j) * (m + 1) + r] = hc[q];
      if (r < p.off) p.raw_b[int64_t(j) * p.ldb + r] = cadd(h1[r], h2[r]);
    }
  }
  if (p.raw_h && lane == 0) p.raw_h[int64_t(j) * (m + 1) + j + 1] = make_double2(hn, 0.0);
  auto entry = [&](int r) {                            // r uniform
    return make_double2(__shfl_sync(0xffffffffu, r < 32 ? hc[0].x : hc[1].x, r & 31),
                        __shfl_sync(0xffffffffu, r < 32 ? hc[0].y : hc[1].y, r & 31));
  };
  double2 a = entry(0);
  for (int r = 0; r < j; r++) {
    const double2 b = entry(r + 1), s = sn[r];
    const double c = cs[r];
    // lanes 0, 1: c a + s b (the finished entry); 2, 3: c b - conj(s) a (carried on)
    const double x = lane == 0 ? a.x : (lane == 1 ? a.y : (lane == 2 ? b.x : b.y));
    const double y = lane == 0 ? b.x : (lane == 1 ? b.y : (lane == 2 ? -a.x : -a.y));
    const double z = lane == 0 ? -b.y : (lane == 1 ? b.x : (lane == 2 ? -a.y : a.x));
    const double v = fma(s.y, z, fma(s.x, y, c * x));
    if (lane < 2) reinterpret_cast<double*>(col + r)[lane] = v;
    a = make_double2(__shfl_sync(0xffffffffu, v, 2), __shfl_sync(0xffffffffu, v, 3));
  }
  const double a2 = a.x * a.x + a.y * a.y;
  root = sqrt(lane == 0 ? a2 : a2 + hn * hn);
  const double aa = __shfl_sync(0xffffffffu, root, 0), rho = __shfl_sync(0xffffffffu, root, 1);
  // lanes 0-4: c, the two parts of a / |a|, hn / rho, 1 / hn
  const double num = lane == 0 ? aa : (lane == 1 ? a.x : (lane == 2 ? a.y : (lane == 3 ? hn : 1.0)));
  const double den = lane == 0 || lane == 3 ? rho : (lane == 4 ? hn : aa);
  const double q = num / den;
  double c = __shfl_sync(0xffffffffu, q, 0);
  const double ux = __shfl_sync(0xffffffffu, q, 1), uy = __shfl_sync(0xffffffffu, q, 2);
  const double t = __shfl_sync(0xffffffffu, q, 3), invh = __shfl_sync(0xffffffffu, q, 4);
  double2 s = make_double2(ux * t, uy * t);
  if (aa == 0.0) {                                     // a = 0: c = 0, s = 1
    c = 0.0;
    s = make_double2(1.0, 0.0);
  }
  if (lane == 0) {
    cs[j] = c;
    sn[j] = s;
    col[j] = make_double2(fma(s.x, hn, c * a.x), fma(s.y, hn, c * a.y));
    col[j + 1] = make_double2(0.0, 0.0);
    const double2 gj = g[j];
    const double2 gn = cmul(make_double2(-s.x, s.y), gj);
    g[j + 1] = gn;
    g[j] = make_double2(c * gj.x, c * gj.y);
    scal[0] = sqrt(gn.x * gn.x + gn.y * gn.y) / scal[p.bn_off];
    scal[1] = invh;
    p.brk[i] = (hn <= 1e-14 * w0) ? 1 : 0;
  }
}

}  // namespace

int cgs_blocks() { return 152 * 4; }
static int64_t cgs_chunk(int64_t n) {
  const int64_t nb = cgs_blocks();
  return std::max<int64_t>(kMinChunk, ((n + nb - 1) / nb + 31) / 32 * 32);
}

enum { kAxpy = 1, kDots = 2 };

// One pass over a chunk of rows: the update (thread per row), then the dots (warp wid holds columns
// wid + 8 c, lanes over the rows kept in shared memory; with at most four columns the warps share
// the rows of each).  ticket != null: the slot's last block adds the blocks' sums into out (columns,
// and |w|^2 at 64) and runs the Givens update if asked.  NC: columns per warp of the widest slot.
template <int NC>
__global__ void __launch_bounds__(256) k_cgs(int64_t n, SlotCgs p, int mode, int64_t chunk, int sub, double2* partial,
                                             unsigned int* ticket, double2* out, SlotGivens gv, int givens) {
  const int i = blockIdx.y, nb = gridDim.x, ncols = p.ncols[i];
  if (ncols < 0) return;
  __shared__ double2 hs[kMaxCols];
  __shared__ double2 ws[256];
  __shared__ double2 gsum[8];
  __shared__ double red[8];
  __shared__ unsigned int order;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const double2* __restrict__ V = p.V[i];
  double2* w = p.w[i];
  const int64_t ld = p.ld;
  if (mode & kAxpy) {
    for (int j = tid; j < ncols; j += 256) hs[j] = p.h[i][j];
    __syncthreads();
  }
  const int64_t row0 = blockIdx.x * chunk, row1 = min(n, row0 + chunk);
  constexpr int P = kPow2<NC>;
  double2 acc[P];
#pragma unroll
  for (int c = 0; c < P; c++) acc[c] = make_double2(0.0, 0.0);
  // cw columns side by side in the warps, 8 / cw groups of warps over a column's rows
  const int cw = ncols > 4 ? 8 : (ncols > 2 ? 4 : (ncols > 1 ? 2 : 1)), col = wid & (cw - 1);
  const int q0 = lane + 32 * (wid / cw), step = 32 * (8 / cw), mine = col < ncols ? (ncols - col + 7) / 8 : 0;
  double nn = 0.0;
  for (int64_t base = row0; base < row1; base += sub) {
    const int cnt = int(min(int64_t(sub), row1 - base));
    const int64_t r = base + tid;
    double2 v = make_double2(0.0, 0.0);
    if (tid < cnt) {
      v = w[r];
      if (mode & kAxpy) {
        double2 a = make_double2(0.0, 0.0);
#pragma unroll 8
        for (int j = 0; j < ncols; j++) a = cmad(V[r + j * ld], hs[j], a);
        v = csub(v, a);
        w[r] = v;
      }
      nn = xfma(v.x, v.x, xfma(v.y, v.y, nn));
    }
    if (mode & kDots) {
      ws[tid] = v;
      __syncthreads();
      dot_rows_of<NC>(mine, acc, V + base + col * ld, 8 * ld, ws, q0, cnt, step);
      __syncthreads();
    }
  }
  double2* part = partial + (int64_t(i) * nb + blockIdx.x) * kPartStride;
  if (mode & kDots) {
    int c;
    const double2 s = sum_columns<P>(acc, lane, c);
    if (cw < 8) {
      if (lane == 0) gsum[wid] = s;
    } else if ((lane & (32 / P - 1)) == 0 && wid + 8 * c < ncols) {
      part[wid + 8 * c] = s;
    }
  }
  for (int o = 16; o > 0; o >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, o);
  if (lane == 0) red[wid] = nn;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int q = 0; q < 8; q++) s += red[q];
    part[kMaxCols] = make_double2(s, 0.0);
  }
  if ((mode & kDots) && cw < 8 && tid < ncols) {
    double2 s = gsum[tid];
    for (int q = tid + cw; q < 8; q += cw) s = cadd(s, gsum[q]);
    part[tid] = s;
  }
  if (!ticket) return;
  __threadfence();
  __syncthreads();
  if (tid == 0) order = atomicAdd(ticket + i, 1u);
  __syncthreads();
  if (order != unsigned(nb) - 1) return;
  __threadfence();
  const double2* all = partial + int64_t(i) * nb * kPartStride;
  double2* o = out + int64_t(i) * kPartStride;
  const int nsum = (mode & kDots) ? ncols : 0;
  for (int c = wid; c <= nsum; c += 8) {
    const int at = c < nsum ? c : kMaxCols;
    double2 s = make_double2(0.0, 0.0);
    for (int b = lane; b < nb; b += 32) s = cadd(s, ldv(all + int64_t(b) * kPartStride + at));
    s = warp_sum(s);
    if (lane == 0) {
      o[at] = s;
      if (at == kMaxCols) red[0] = s.x;
    }
  }
  if (tid == 0) ticket[i] = 0u;
  if (!givens) return;
  __syncthreads();
  if (wid == 0) givens_update(gv, i, red[0]);
}

// out[c] = sum over the blocks of their partial sums, one warp per column (and one for the norm)
__global__ void __launch_bounds__(256) k_cgs_sum(const double2* partial, int nb, SlotCgs p, int mode, double2* out) {
  const int i = blockIdx.y, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nsum = (mode & kDots) ? p.ncols[i] : 0;
  if (p.ncols[i] < 0 || int(blockIdx.x) > nsum) return;
  __shared__ double2 red[8];
  const int at = int(blockIdx.x) < nsum ? blockIdx.x : kMaxCols;
  const double2* all = partial + int64_t(i) * nb * kPartStride + at;
  double2 s = make_double2(0.0, 0.0);
#pragma unroll 4
  for (int b = threadIdx.x; b < nb; b += 256) s = cadd(s, ldv(all + int64_t(b) * kPartStride));
  s = warp_sum(s);
  if (lane == 0) red[wid] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < 8; q++) s = cadd(s, red[q]);
    out[int64_t(i) * kPartStride + at] = s;
  }
}

__global__ void k_givens(SlotGivens p) {
  const int i = blockIdx.x;
  if (p.j[i] < 0) return;
  givens_update(p, i, p.nrm[int64_t(i) * kPartStride + kMaxCols].x);
}

void launch_cgs_slots(int64_t n, int S, const SlotCgs& p, bool maxpy, bool dots, double2* partial,
                      unsigned int* ticket, double2* out, cudaStream_t st, const SlotGivens* givens) {
  const int64_t chunk = cgs_chunk(n);
  const int nb = int((n + chunk - 1) / chunk);
  const int nsub = int((chunk + 255) / 256), sub = int(((chunk + nsub - 1) / nsub + 31) / 32 * 32);
  const int mode = (maxpy ? kAxpy : 0) | (dots ? kDots : 0);
  int cols = 0;
  for (int i = 0; i < S; i++) cols = std::max(cols, p.ncols[i]);
  const bool fused = ticket && nb <= kFusedBlocks;
  unsigned int* tk = fused ? ticket : nullptr;
  const int gfused = fused && givens ? 1 : 0;
  SlotGivens gv{};
  if (givens) gv = *givens;
  const dim3 grid(unsigned(std::max(nb, 1)), unsigned(S));
  add_launches(1);
  const int nc = dots ? std::max((cols + 7) / 8, 1) : 1;
  auto pass = [&](auto* kern) { kern<<<grid, 256, 0, st>>>(n, p, mode, chunk, sub, partial, tk, out, gv, gfused); };
  switch (nc) {
    case 1: pass(k_cgs<1>); break;
    case 2: pass(k_cgs<2>); break;
    case 3: pass(k_cgs<3>); break;
    case 4: pass(k_cgs<4>); break;
    case 5: pass(k_cgs<5>); break;
    case 6: pass(k_cgs<6>); break;
    case 7: pass(k_cgs<7>); break;
    default: pass(k_cgs<8>); break;
  }
  if (fused) return;
  add_launches(1);
  k_cgs_sum<<<dim3(unsigned(dots ? cols + 1 : 1), unsigned(S)), 256, 0, st>>>(partial, int(grid.x), p, mode, out);
  if (givens) {
    add_launches(1);
    k_givens<<<S, 32, 0, st>>>(*givens);
  }
}

void launch_cgs(int64_t n, int ncols, const double2* V, int64_t ldv, const double2* h, double2* w, bool dots,
                double2* partial, unsigned int* ticket, double2* out, cudaStream_t st, const SlotGivens* givens) {
  SlotCgs p{};
  for (int i = 1; i < 16; i++) p.ncols[i] = -1;
  p.ld = ldv;
  p.V[0] = V;
  p.w[0] = w;
  p.h[0] = h;
  p.ncols[0] = ncols;
  launch_cgs_slots(n, 1, p, h != nullptr, dots || !h, partial, ticket, out, st, givens);
}

// y = R^{-1} g (upper triangular k x k of the rotated Hessenberg matrix, k <= 64), column by column:
// thread i owns row i
__global__ void __launch_bounds__(64) k_backsub(int k, const double2* H, int ldh, const double2* g, double2* y) {
  __shared__ double2 yi;
  const int i = threadIdx.x;
  double2 s = i < k ? g[i] : make_double2(0.0, 0.0);
  const double2 di = i < k ? cinv(H[i + int64_t(i) * ldh]) : make_double2(0.0, 0.0);
  double2 next = i < k ? H[i + int64_t(k - 1) * ldh] : make_double2(0.0, 0.0);
  for (int l = k - 1; l >= 0; l--) {
    const double2 h = next;
    if (l > 0 && i < l - 1) next = H[i + int64_t(l - 1) * ldh];
    if (i == l) {
      const double2 v = cmul(s, di);
      yi = v;
      y[i] = v;
    }
    __syncthreads();
    const double2 v = yi;
    if (i < l) s = cmsub(h, v, s);
    __syncthreads();
  }
}

void launch_update_x(int64_t n, int k, const double2* H, int ldh, const double2* g, double2* y, const double2* Zs,
                     int64_t ldz, double2* x, cudaStream_t st) {
  add_launches(1);
  k_backsub<<<1, 64, 0, st>>>(k, H, ldh, g, y);
  launch_gemv_add(n, k, y, Zs, ldz, x, st);
}

}  // namespace hz
