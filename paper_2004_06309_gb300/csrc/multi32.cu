// Complex64 triangular sweeps for S = 4, 8 or 16 right-hand sides (interleaved per row): every panel
// entry is read once for all of them.
//
// Bound: FP32 arithmetic (four FMAs per entry and right-hand side: 1.1 ms for the 76 GFLOP of one
// application on the 349,461-dof survey model with S = 16, against 0.7 ms to read the 4.95 GB of
// panels twice).  A thread owns a tile of 4 rows (forward) or 4 columns (backward) x 4 right-hand
// sides, 64 FMAs per 2 shared-memory and 2 panel loads of 16 bytes; with one row (or column) x S per
// thread the loads of the right-hand sides, and in the backward sweep 32 separate panel lines
// per load, held the two sweeps at 9.1 ms.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "dev.h"
#include "dmath.cuh"

namespace hz {

namespace {

constexpr int kVecPad = 2;                         // float2 per row: conflict-free reads of four row pairs
constexpr int kColPitch = kMultiBwdRows + 2;       // float2 per panel column in shared memory

__device__ __forceinline__ void mad4(float2 p, const float4* b, float2* acc) {
  const float4 u = b[0], v = b[1];
  acc[0] = cmad(p, make_float2(u.x, u.y), acc[0]);
  acc[1] = cmad(p, make_float2(u.z, u.w), acc[1]);
  acc[2] = cmad(p, make_float2(v.x, v.y), acc[2]);
  acc[3] = cmad(p, make_float2(v.z, v.w), acc[3]);
}

}  // namespace

// rows per forward task
template <int S> constexpr int kFwdRows32 = S == 4 ? 128 : 64;
// panel columns per ring slot: 32 KB
template <int S> constexpr int kFwdCols32 = S == 4 ? 32 : 64;

// Forward: z = D^{-1} (T b1) for pivot rows, u = children's updates - G b1 below.  The panel is copied
// to shared memory by cp.async, 64 columns per slot of a two-slot ring, both issued before the
// right-hand sides are gathered; a slot's columns are dealt to KG groups of threads whose sums are
// added in order.  A thread's rows are two pairs half a task apart (conflict-free 16-byte reads).
template <int S>
__global__ void __launch_bounds__(256, 2) k_fwd_multi32(const int2* tasks, const SnDev* sn, const uint32_t* cptr,
                                                        const uint32_t* wpos, const float2* panels,
                                                        const float2* tin, float2* zout, float2* u, int kpad) {
  constexpr int RT = kFwdRows32<S>, TG = RT * S / 16, KG = 256 / TG, CC = kFwdCols32<S>, SLOT = CC * RT;
  static_assert(KG * RT * S <= 2 * SLOT, "the partial sums reuse the ring");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* ring = reinterpret_cast<float2*>(smem_raw);                     // 2 x CC x RT; then KG x RT x S sums
  float2* b1 = ring + 2 * SLOT;                                            // kpad x S
  const int2 tk = tasks[blockIdx.x];
  const SnDev Sn = sn[tk.x];
  const int k = Sn.k, m = Sn.m, tid = threadIdx.x;
  const int tg = tid % TG, kg = tid / TG, rg = tg % (RT / 4), hg = tg / (RT / 4);
  const uint32_t* cp = cptr + Sn.rowoff + Sn.id;
  const int row0 = tk.y * RT;
  const int jend = min(min(row0 + RT, m) - 1, k);                          // columns any row of the task uses
  auto issue = [&](int c) {                                                // columns c CC .. of the panel into slot c & 1
    for (int e = tid; e < CC * (RT / 2); e += 256) {
      const int j = c * CC + e / (RT / 2), r = 2 * (e % (RT / 2));
      if (j < jend && row0 + r < m)                                        // ld % 4 == 0: pairs are whole
        cp_async16(ring + (c & 1) * SLOT + (e / (RT / 2)) * RT + r, panels + Sn.paneloff + int64_t(j) * Sn.ld + row0 + r);
    }
    cp_async_commit();
  };
  issue(0);
  issue(1);
  gather_rows<float2, S>(b1, tin + int64_t(Sn.first) * S, cp, u + Sn.ubase * S, k);
  UpdateRows<float2, S, RT> up;
  up.load(Sn, cp, wpos, u, row0);
  float2 acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) acc[a][b] = make_float2(0.f, 0.f);
  const int ra = 2 * rg, rb = ra + RT / 2;
  for (int c = 0; c * CC < jend; c++) {
    cp_async_wait<1>();
    __syncthreads();
    const float2* slot = ring + (c & 1) * SLOT;
    const int j1 = min(CC, jend - c * CC);
    const bool full = c * CC + j1 <= row0 && row0 + RT <= m;               // no masked entry in the slot
#pragma unroll 4
    for (int jj = kg; jj < j1; jj += KG) {
      float4 p = *reinterpret_cast<const float4*>(slot + jj * RT + ra);
      float4 q = *reinterpret_cast<const float4*>(slot + jj * RT + rb);
      const int j = c * CC + jj;
      if (!full) {
        const int va = row0 + ra, vb = row0 + rb;
        if (j >= va || va >= m) p.x = p.y = 0.f;
        if (j >= va + 1 || va + 1 >= m) p.z = p.w = 0.f;
        if (j >= vb || vb >= m) q.x = q.y = 0.f;
        if (j >= vb + 1 || vb + 1 >= m) q.z = q.w = 0.f;
      }
      const float4* b = reinterpret_cast<const float4*>(b1 + j * S + 4 * hg);
      mad4(make_float2(p.x, p.y), b, acc[0]);
      mad4(make_float2(p.z, p.w), b, acc[1]);
      mad4(make_float2(q.x, q.y), b, acc[2]);
      mad4(make_float2(q.z, q.w), b, acc[3]);
    }
    __syncthreads();                                                       // the slot is used
    issue(c + 2);
  }
  cp_async_wait<0>();
  __syncthreads();
  float2* part = ring;
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 4; b++)
      part[(kg * RT + (a < 2 ? ra + a : rb + a - 2)) * S + 4 * hg + b] = acc[a][b];
  __syncthreads();
#pragma unroll
  for (int n = 0; n < up.N; n++) {
    constexpr int LR = S / 2;
    const int e = tid + 256 * n, i = e % LR, r = row0 + e / LR;
    if (e >= RT * LR || r >= m) continue;
    const float4* p4 = reinterpret_cast<const float4*>(part);
    float4 s = p4[e];
#pragma unroll
    for (int q = 1; q < KG; q++) s = vadd(s, p4[q * RT * LR + e]);
    if (r < k) {
      const float2 d = panels[Sn.paneloff + r + int64_t(r) * Sn.ld];
      const float4 a = vadd(reinterpret_cast<const float4*>(b1)[r * LR + i], s);
      const float2 z0 = cmul(d, make_float2(a.x, a.y)), z1 = cmul(d, make_float2(a.z, a.w));
      reinterpret_cast<float4*>(zout)[int64_t(Sn.first + r) * LR + i] = make_float4(z0.x, z0.y, z1.x, z1.y);
    } else {
      reinterpret_cast<float4*>(u)[(Sn.wbase + up.to[n]) * LR + i] = vsub(up.b2[n], s);
    }
  }
}

// Backward: 32 pivot columns x one chunk of kMultiBwdRows rows per task.  The chunk's panel is copied
// to shared memory by cp.async while the right-hand sides are gathered; lanes are 8 groups of 4
// columns x 4 row pairs, warps S / 4 groups of right-hand sides x row groups.
template <int S>
__global__ void __launch_bounds__(256, 4) k_bwd_multi32(const int4* tasks, const SnDev* sn, const int32_t* rowlist,
                                                        const float2* panels, const float2* zin, float2* x,
                                                        float2* partial, const int4* fins, unsigned int* counters) {
  constexpr int ROWS = kMultiBwdRows, HG = S / 4, KG = 8 / HG, VP = S + kVecPad;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* col = reinterpret_cast<float2*>(smem_raw);                      // 32 x kColPitch; then KG x 32 x S sums
  float2* vec = col + 32 * kColPitch;                                      // ROWS x VP
  __shared__ unsigned int ticket;
  const int4 tk = tasks[blockIdx.x];
  const SnDev Sn = sn[tk.x];
  const int k = Sn.k, m = Sn.m, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int r0 = tk.z * ROWS, r1 = min(m, r0 + ROWS), cnt = r1 - r0, j0 = tk.y * 32;
  for (int e = tid; e < 32 * (ROWS / 2); e += 256) {                       // row pairs (ld % 4 == 0, r0 even)
    const int c = e / (ROWS / 2), r = 2 * (e % (ROWS / 2));
    if (j0 + c < k && r < cnt)
      cp_async16(col + c * kColPitch + r, panels + Sn.paneloff + int64_t(j0 + c) * Sn.ld + r0 + r);
  }
  cp_async_commit();
  const int32_t* rl = rowlist + Sn.rowoff;
  {
    constexpr int LR = S / 2, N = ROWS * LR / 256;
    int32_t at[N];
#pragma unroll
    for (int n = 0; n < N; n++) {
      const int r = r0 + (tid + 256 * n) / LR;
      at[n] = r < r1 && r >= k ? rl[r] : 0;
    }
#pragma unroll
    for (int n = 0; n < N; n++) {
      const int q = (tid + 256 * n) / LR, i = (tid + 256 * n) % LR, r = r0 + q;
      float4 v = vzero<float4>();
      if (r < k) v = r < r1 ? __ldcg(reinterpret_cast<const float4*>(zin) + int64_t(Sn.first + r) * LR + i) : v;
      else if (r < r1) v = vsub(v, __ldcg(reinterpret_cast<const float4*>(x) + int64_t(at[n]) * LR + i));
      *reinterpret_cast<float4*>(vec + q * VP + 2 * i) = v;
    }
  }
  cp_async_wait<0>();
  __syncthreads();
  const int cg = lane >> 2, kl = lane & 3, hg = wid % HG, kg = wid / HG;
  float2 acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) acc[a][b] = make_float2(0.f, 0.f);
  const int jc = j0 + 4 * cg;                                              // this lane's columns jc .. jc + 3
  const float2* pc = col + 4 * cg * kColPitch;
  for (int q = 8 * kg + 2 * kl; q < cnt; q += 8 * KG) {
    const float4* b = reinterpret_cast<const float4*>(vec + q * VP + 4 * hg);
    const float4* b2 = reinterpret_cast<const float4*>(vec + (q + 1) * VP + 4 * hg);
    const int r = r0 + q;
    const bool full = r > jc + 3 && jc + 3 < k;
#pragma unroll
    for (int a = 0; a < 4; a++) {
      float4 p = *reinterpret_cast<const float4*>(pc + a * kColPitch + q);
      if (!full) {                                                         // on or above the diagonal, or beyond the columns
        if (jc + a >= k || r <= jc + a) p.x = p.y = 0.f;
        if (jc + a >= k || r + 1 <= jc + a) p.z = p.w = 0.f;
      }
      if (r + 1 >= r1) p.z = p.w = 0.f;
      mad4(make_float2(p.x, p.y), b, acc[a]);
      mad4(make_float2(p.z, p.w), b2, acc[a]);
    }
  }
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) {
      acc[a][b] = cadd(acc[a][b], shfl_xor(acc[a][b], 1));
      acc[a][b] = cadd(acc[a][b], shfl_xor(acc[a][b], 2));
    }
  __syncthreads();                                                         // the panel is used
  if (kl == 0) {
#pragma unroll
    for (int a = 0; a < 4; a++)
#pragma unroll
      for (int b = 0; b < 4; b++) col[(kg * 32 + 4 * cg + a) * S + 4 * hg + b] = acc[a][b];
  }
  __syncthreads();
  const bool single = m <= ROWS;
  float2* out = partial + int64_t(blockIdx.x) * 32 * S;
  for (int e = tid; e < 32 * S; e += 256) {
    float2 s = col[e];
#pragma unroll
    for (int q = 1; q < KG; q++) s = cadd(s, col[q * 32 * S + e]);
    const int j = j0 + e / S;
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
    const int j = j0 + e / S;
    if (j >= k) continue;
    float2 a = make_float2(0.f, 0.f);
    for (int ch = 0; ch < fin.w; ch++) a = cadd(a, ldv(partial + int64_t(fin.z + ch) * 32 * S + e));
    x[int64_t(Sn.first + j) * S + e % S] = cadd(ldv(zin + int64_t(Sn.first + j) * S + e % S), a);
  }
  if (tid == 0) counters[tk.w] = 0u;
}

template <int S>
static void solve_multi32_t(const FactorDev& F, cudaStream_t st) {
  static const bool attr = [] {
    cudaFuncSetAttribute(k_fwd_multi32<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    cudaFuncSetAttribute(k_bwd_multi32<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    return true;
  }();
  (void)attr;
  constexpr int RT = kFwdRows32<S>, SLOT = kFwdCols32<S> * RT;
  const float2* P = (const float2*)F.panels;
  float2 *t = (float2*)F.mt_loc, *z = (float2*)F.mz_loc, *x = (float2*)F.mx_loc, *u = (float2*)F.mu_ws;
  for (int l = 0; l < F.snlev; l++) {
    const int64_t b = F.h_mfwd_ptr[l], e = F.h_mfwd_ptr[l + 1];
    if (e == b) continue;
    add_launches(1);
    const int kpad = F.h_lev_k[l];
    k_fwd_multi32<S><<<unsigned(e - b), 256, size_t(2 * SLOT + kpad * S) * 8, st>>>(F.mfwd_tasks + b, F.ssn, F.cptr, F.wpos,
                                                                             P, t, z, u, kpad);
  }
  const size_t bsm = size_t(32 * kColPitch + kMultiBwdRows * (S + kVecPad)) * 8;
  for (int l = F.snlev - 1; l >= 0; l--) {
    const int64_t b = F.h_mbwd_ptr[l], e = F.h_mbwd_ptr[l + 1];
    if (e == b) continue;
    add_launches(1);
    k_bwd_multi32<S><<<unsigned(e - b), 256, bsm, st>>>(F.mbwd_tasks + b, F.ssn, F.rowlist, P, z, x,
                                                        (float2*)F.mbwd_partial, F.mbfin_tasks, F.mbwd_counters);
  }
}

void launch_solve_multi32(const FactorDev& F, int S, cudaStream_t st) {
  if (S == 4) solve_multi32_t<4>(F, st);
  else if (S == 8) solve_multi32_t<8>(F, st);
  else solve_multi32_t<16>(F, st);
}

}  // namespace hz
