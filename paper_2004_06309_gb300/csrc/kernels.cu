// CUDA kernels of the hz library (sm_103a).
//
//   * value assembly A(omega) = K - omega^2 M' - i omega B'        (Eq. 2)
//   * batched multifrontal complex-symmetric LDL^T of all A_i and E (the local
//     "direct solver" of the method, factorised once per frequency)
//   * batched supernodal forward / diagonal / backward solves       (Eq. 3-4)
//   * restriction R_i (gather) and PU-weighted prolongation R_i^T D_i
//   * complex CSR SpMV, real-by-complex CSR SpMV (Z, Z^T)
//   * fused CGS2 passes, deterministic reductions, Givens update    (GMRES)
//
// Complex numbers are interleaved (re, im) pairs: double2 (complex128) or
// float2 (complex64).  All reductions are fixed-order (no atomics on values),
// so reruns are bitwise identical.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>

#include "dev.h"
#include "dmath.cuh"

namespace hz {

// Kernel launches issued by this library (for the launch count in hz_stats).
static std::atomic<long long> g_launches{0};
long long launch_count() { return g_launches.load(); }
void add_launches(long long n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
#define HZ_COUNT() add_launches(1)

// widest supernode (pivot columns) any kernel handles
constexpr int kMaxK = 128;

static inline unsigned grid_for(int64_t work, int per_block, int cap = 152 * 16) {
  int64_t g = (work + per_block - 1) / per_block;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return unsigned(g);
}

// ---------------------------------------------------------------------------
// value assembly, Eq. (2): A = K - w^2 M' - i w B'
// ---------------------------------------------------------------------------
__device__ __forceinline__ double2 helmholtz_value(double k, double2 m, double2 b, double w) {
  // K - w^2 (m.x + i m.y) - i w (b.x + i b.y)
  return make_double2(k - w * w * m.x + w * b.y, -w * w * m.y - w * b.x);
}

__global__ void k_fill_values(int64_t nnz, const double* K, const double2* M, const double2* B, double w,
                              double2* out) {
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < nnz; e += int64_t(gridDim.x) * blockDim.x)
    out[e] = helmholtz_value(K[e], M[e], B[e], w);
}

void launch_fill_values(int64_t nnz, const double* K, const double2* M, const double2* B, double w,
                        double2* out, cudaStream_t st) {
  if (nnz == 0) return;
  HZ_COUNT();
  k_fill_values<<<grid_for(nnz, 256), 256, 0, st>>>(nnz, K, M, B, w, out);
}

template <typename V>
__global__ void k_front_fill(int64_t ne, const int64_t* epos, const double* K, const double2* M,
                             const double2* B, double w, V* fronts) {
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < ne; e += int64_t(gridDim.x) * blockDim.x)
    fronts[epos[e]] = from2<V>(helmholtz_value(K[e], M[e], B[e], w));
}

// ---------------------------------------------------------------------------
// complex128: symmetric scaling by powers of two.  The factorisation's products hold their operands as
// digits below the largest entry of a row (digits.cuh), so rows of A of very different size (wave
// speeds spread over 10^12 within a subdomain) would cost the small ones their digits.  With
// S A S, S = 2^-sig, the diagonal is within [1/2, 4), and so the rows of L D^(1/2).  A^{-1} v =
// S (S A S)^{-1} S v: powers of two change no digit of the vectors either.
// ---------------------------------------------------------------------------
constexpr int kMaxSig = 200;
__global__ void k_scaling(int64_t ntot, const int64_t* ediag, const double* K, const double2* M, const double2* B,
                          double w, int16_t* sig) {
  for (int64_t l = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; l < ntot; l += int64_t(gridDim.x) * blockDim.x) {
    const int64_t e = ediag[l];
    int s = 0;
    if (e >= 0) {
      const double2 v = helmholtz_value(K[e], M[e], B[e], w);
      const double a = fmax(fabs(v.x), fabs(v.y));
      if (a > 0.0 && isfinite(a)) s = max(-kMaxSig, min(kMaxSig, ilogb(a) >> 1));
    }
    sig[l] = int16_t(s);
  }
}

void launch_scaling(const FactorDev& F, double w, cudaStream_t st) {
  if (F.ntot == 0) return;
  HZ_COUNT();
  k_scaling<<<grid_for(F.ntot, 256), 256, 0, st>>>(F.ntot, F.ediag, F.ek, F.em, F.eb, w, F.sig);
}

// A's entries of a level's fronts (their pivot columns), after k_front_fill; grid as k_front_zero's
__global__ void __launch_bounds__(256) k_front_scale(const int32_t* lev_sn, const SnDev* sn, const int32_t* rowlist,
                                                     const int16_t* sig, double2* fronts) {
  const SnDev S = sn[lev_sn[blockIdx.x]];
  double2* f = fronts + S.frontoff;
  const int32_t* rl = rowlist + S.rowoff;
  for (int j = blockIdx.y * 8 + (threadIdx.x >> 5); j < S.k; j += 8 * gridDim.y) {
    const int sj = sig[S.first + j];
    for (int r = j + (threadIdx.x & 31); r < S.m; r += 32) {
      const double2 v = f[int64_t(j) * S.m + r];
      if (v.x != 0.0 || v.y != 0.0) {
        const double c = exp2i(-sj - sig[rl[r]]);
        f[int64_t(j) * S.m + r] = make_double2(v.x * c, v.y * c);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// multifrontal factorisation, one assembly-tree level at a time
// ---------------------------------------------------------------------------

// Extend-add: parent front += child's contribution block (lower triangle).
// One warp per contribution column; a launch holds at most one child per parent.  A lane's
// kEaRows entries are loaded together: a column has no row twice, but the compiler cannot know
// and would wait for each entry's store address and load in turn.  349,461 dofs, complex64:
// 7.6 -> 6.7 ms per factorisation.
constexpr int kEaRows = 4;
template <typename V>
__global__ void __launch_bounds__(256) k_extend_add(const int2* tasks, const SnDev* sn, const int32_t* rel,
                                                    const int64_t* reloff, V* fronts) {
  const int2 t = tasks[blockIdx.x];
  const SnDev C = sn[t.x];
  const int r = C.m - C.k;
  const int b = t.y * 8 + (threadIdx.x >> 5);
  if (b >= r) return;
  const SnDev P = sn[C.parent];
  const int32_t* rl = rel + reloff[t.x];
  const V* Fc = fronts + C.frontoff;
  V* Fp = fronts + P.frontoff;
  const int64_t pc = int64_t(rl[b]) * P.m;
  const int64_t cc = int64_t(C.k + b) * C.m + C.k;
  for (int a0 = b + (threadIdx.x & 31); a0 < r; a0 += 32 * kEaRows) {
    int64_t q[kEaRows];
    V p[kEaRows], v[kEaRows];
#pragma unroll
    for (int i = 0; i < kEaRows; i++) q[i] = a0 + 32 * i < r ? pc + rl[a0 + 32 * i] : 0;
#pragma unroll
    for (int i = 0; i < kEaRows; i++)
      if (a0 + 32 * i < r) {
        v[i] = Fc[cc + a0 + 32 * i];
        p[i] = Fp[q[i]];
      }
#pragma unroll
    for (int i = 0; i < kEaRows; i++)
      if (a0 + 32 * i < r) Fp[q[i]] = cadd(p[i], v[i]);
  }
}

// Off-diagonal panel of a complex64 supernode, kWgRows rows per task:
//   W = F21 T^T  (= L21 D), saved to the level scratch for the Schur update,
//   G = W D^{-1} T  (= F21 F11^{-1} = L21 L11^{-1}), written over F21.
// Bound: FP32 arithmetic.  A thread owns 8 rows x 4 columns, its rows in pairs 16 apart: the eight
// lanes that read a column of F21 then take 128 consecutive bytes (with 8 consecutive rows a thread the
// reads conflicted four ways and the load/store unit bounded the kernel).  T is copied 16 columns
// (rows) at a time by cp.async, one stage ahead, and a warp skips the stages that hold only zeros for
// its 16 columns.  349,461 dofs: 15.5 -> 10.9 ms per factorisation (14.7 with the copies alone).
// Every sum keeps the order of the columns.
constexpr int kWgPitch = kWgRows + 2, kWgTPitch = kMaxK + 2;
__global__ void __launch_bounds__(256, 2) k_wg32(const int2* tasks, const SnDev* sn, const int64_t* scr_off,
                                                 float2* fronts, float2* scratch, int kpad) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* Fs = reinterpret_cast<float2*>(smem_raw);          // kpad x kWgPitch: F21, then L21
  float2* Tt = Fs + kpad * kWgPitch;                         // 2 stages of 16 x kWgTPitch
  __shared__ float2 di[kMaxK];
  const int2 t = tasks[blockIdx.x];
  const SnDev S = sn[t.x];
  const int k = S.k, m = S.m, r = m - k, tid = threadIdx.x;
  float2* F = fronts + S.frontoff;
  const int R0 = t.y * kWgRows, nr = min(kWgRows, r - R0);
  float2* F21 = F + k + R0;
  // the warp's 16 columns: warps w and w + 4 share a scheduler, so the second four count down
  // and each scheduler gets the same share of T's triangle
  const int wid = tid >> 5, wj0 = 16 * (wid < 4 ? wid : 11 - wid);
  const int rg = tid & 7, j0 = wj0 + 4 * ((tid >> 3) & 3);   // rows 16 q + 2 rg + 0, 1, columns j0 ..
  auto row_of = [&](int a) { return 16 * (a >> 1) + 2 * rg + (a & 1); };
  const int K16 = (k + 15) / 16 * 16;
  const float2 z = make_float2(0.f, 0.f);
  for (int e = tid; e < K16 * kWgRows; e += 256) {
    const int i = e % kWgRows, j = e / kWgRows;
    Fs[j * kWgPitch + i] = (i < nr && j < k) ? F21[i + int64_t(j) * m] : z;
  }
  for (int j = tid; j < k; j += 256) di[j] = F[j + int64_t(j) * m];
  float2 acc[8][4];
  auto product = [&](const float2* T, int i0) {
#pragma unroll 4
    for (int ii = 0; ii < 16; ii++) {
      const float4* a4 = reinterpret_cast<const float4*>(Fs + (i0 + ii) * kWgPitch + 2 * rg);
      const float4* b4 = reinterpret_cast<const float4*>(T + ii * kWgTPitch + j0);
      const float4 b0 = b4[0], b1 = b4[1];
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const float4 a = a4[8 * q];
        const float2 x = make_float2(a.x, a.y), y = make_float2(a.z, a.w);
        acc[2 * q][0] = cmad(x, make_float2(b0.x, b0.y), acc[2 * q][0]);
        acc[2 * q][1] = cmad(x, make_float2(b0.z, b0.w), acc[2 * q][1]);
        acc[2 * q][2] = cmad(x, make_float2(b1.x, b1.y), acc[2 * q][2]);
        acc[2 * q][3] = cmad(x, make_float2(b1.z, b1.w), acc[2 * q][3]);
        acc[2 * q + 1][0] = cmad(y, make_float2(b0.x, b0.y), acc[2 * q + 1][0]);
        acc[2 * q + 1][1] = cmad(y, make_float2(b0.z, b0.w), acc[2 * q + 1][1]);
        acc[2 * q + 1][2] = cmad(y, make_float2(b1.x, b1.y), acc[2 * q + 1][2]);
        acc[2 * q + 1][3] = cmad(y, make_float2(b1.z, b1.w), acc[2 * q + 1][3]);
      }
    }
  };
  auto start = [&]() {
#pragma unroll
    for (int a = 0; a < 8; a++)
#pragma unroll
      for (int b = 0; b < 4; b++) acc[a][b] = j0 + b < K16 ? Fs[(j0 + b) * kWgPitch + row_of(a)] : z;
  };
  // stage n of W takes T(j, i), i < j, of G T(i, j), i > j: copied while the stage before it is
  // multiplied
  const int ns = (k + 15) / 16;
  auto copy_w = [&](int n) {
    float2* D = Tt + (n & 1) * 16 * kWgTPitch;
    for (int e = tid; e < 16 * K16; e += 256) {
      const int j = e % K16, i = 16 * n + e / K16;
      const bool in = j < k && i < j;
      cp_async8(D + (e / K16) * kWgTPitch + j, in ? F + j + int64_t(i) * m : F, in);
    }
    cp_async_commit();
  };
  auto copy_g = [&](int n) {
    float2* D = Tt + (n & 1) * 16 * kWgTPitch;
    for (int e = tid; e < 16 * K16; e += 256) {
      const int ii = e % 16, i = 16 * n + ii, j = e / 16;
      const bool in = i < k && i > j;
      cp_async8(D + ii * kWgTPitch + j, in ? F + i + int64_t(j) * m : F, in);
    }
    cp_async_commit();
  };
  copy_w(0);
  __syncthreads();
  start();
  for (int n = 0; n < ns; n++) {
    cp_async_wait<0>();
    __syncthreads();                                         // stage n is in, stage n - 1's buffer is free
    if (n + 1 < ns) copy_w(n + 1);
    if (wj0 < K16 && wj0 + 15 > 16 * n) product(Tt + (n & 1) * 16 * kWgTPitch, 16 * n);
  }
  __syncthreads();
  float2* W = scratch + scr_off[t.x];
#pragma unroll
  for (int b = 0; b < 4; b++) {
    const int j = j0 + b;
    if (j >= k) continue;
#pragma unroll
    for (int a = 0; a < 8; a++) {
      const int i = row_of(a);
      if (i < nr) W[(R0 + i) + int64_t(j) * r] = acc[a][b];
      Fs[j * kWgPitch + i] = cmul(acc[a][b], di[j]);         // L21
    }
  }
  copy_g(0);
  __syncthreads();
  start();
  for (int n = 0; n < ns; n++) {
    cp_async_wait<0>();
    __syncthreads();
    if (n + 1 < ns) copy_g(n + 1);
    if (wj0 < K16 && wj0 < 16 * n + 15) product(Tt + (n & 1) * 16 * kWgTPitch, 16 * n);
  }
#pragma unroll
  for (int b = 0; b < 4; b++)
#pragma unroll
    for (int a = 0; a < 8; a++)
      if (j0 + b < k && row_of(a) < nr) F21[row_of(a) + int64_t(j0 + b) * m] = acc[a][b];
}

// ---------------------------------------------------------------------------
// Tensor-core (tcgen05) Schur update of complex64 fronts, one 128 x 128 lower
// tile of the contribution block per CTA (8 warps):
//   F22[a][b] -= sum_i W[a][i] d_i^{-1} W[b][i]      (complex, i < k)
// as two real products over K' = 2k, K' interleaved by complex column (2i: real parts,
// 2i + 1: imaginary parts):
//   Re = A B1^T,  Im = A B2^T,  A = (Wr, Wi),  B1 = (Br, -Bi),  B2 = (Bi, Br),  B = W diag(d^{-1}),
// each in 3xTF32 (hi*hi + hi*lo + lo*hi, hi = TF32 rounding, lo = the remainder),
// accumulated in FP32 in tensor memory (Re: columns 0-127, Im: 128-255).
// Operands are staged K-major in shared memory as 8-row x 16-byte core matrices
// (no swizzle), kTcCols complex columns (2 kTcCols K' values) per stage, in two stages
// (96 KB, two CTAs per SM): while one stage's MMAs run the 256 threads fill the other
// (thread = tile row, half of the stage's columns; every W element is read once per
// tile; a thread's loads of the next stage are issued together, right after the current
// stage's MMAs).  One elected thread issues the MMAs
// and commits each stage to that stage's mbarrier.  Every wait is bounded: a stage
// buffer is refilled only after the commit of the stage that last used it; the polls of
// these waits and of the final one are first_wait.  When one runs out the CTA raises
// status->timeout (bit 0), skips its epilogue and drains the MMAs it issued with a
// second wait of kTcDrainPolls polls on the last commit before it frees its tensor
// memory.  The MMAs read only this CTA's shared memory and write only its tensor
// memory, so they finish in bounded time and the drain ends; should it run out as well
// (a faulty tensor pipe), bit 1 is raised and the memory is still freed, because a CTA
// that exits holding tensor memory would leave later allocations on its SM waiting
// forever.  Either bit makes hz_factor return HZ_ERR_TIMEOUT and leaves the context
// unfactored.
// The epilogue loads 16 front entries of a row together, the first ones before the last wait:
// loaded one by one between the stores, each waited for the memory, 64 times a CTA, and took
// longer than the MMAs.  349,461 dofs: 23.3 -> 12.8 ms per factorisation.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float tf32_rna(float x) {
  uint32_t y;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(y) : "f"(x));
  return __uint_as_float(y);
}
// TF32 high parts and remainders of four values, stored as vectors
__device__ __forceinline__ void tc_split(float4 v, float* hi, float* lo) {
  const float4 h = make_float4(tf32_rna(v.x), tf32_rna(v.y), tf32_rna(v.z), tf32_rna(v.w));
  *reinterpret_cast<float4*>(hi) = h;
  *reinterpret_cast<float4*>(lo) =
      make_float4(tf32_rna(v.x - h.x), tf32_rna(v.y - h.y), tf32_rna(v.z - h.z), tf32_rna(v.w - h.w));
}
// float offset of element (row r, k) in a 128 x 32 K-major tile of core matrices
constexpr int kTcCols = 8;                      // complex columns per stage
constexpr int kTcK = 2 * kTcCols;               // real K' values per stage
constexpr int kTcTile = 128 * kTcK;             // floats of one 128-row operand tile
__device__ __forceinline__ int tc_off(int r, int kk) {
  return ((r >> 3) * (kTcK / 4) + (kk >> 2)) * 32 + (r & 7) * 4 + (kk & 3);
}
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr) {
  // LBO = 128 B (next core matrix along K), SBO = 8 rows x kTcK x 4 B (next 8-row group),
  // version 1, no swizzle
  return uint64_t((saddr >> 4) & 0x3FFF) | (uint64_t(128 >> 4) << 16) | (uint64_t((32 * kTcK) >> 4) << 32) |
         (uint64_t(1) << 46);
}
__device__ __forceinline__ void tc_mma(uint32_t tmem, uint64_t da, uint64_t db, uint32_t acc) {
  // D f32, A/B tf32, both K-major, N = 128, M = 128
  const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
               "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n"
               :: "r"(tmem), "l"(da), "l"(db), "r"(idesc), "r"(acc));
}
constexpr int kTcDrainPolls = 1 << 22;
__device__ __forceinline__ bool tc_wait(uint64_t* mbar, uint32_t phase, int polls) {
  uint32_t done = 0;
  for (int it = 0; it < polls && !done; it++)
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(done) : "r"(smem_addr(mbar)), "r"(phase));
  return done != 0;
}
__device__ __forceinline__ void tc_ld16(uint32_t ta, float* out) {
  uint32_t v[16];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                 "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                 "=r"(v[15])
               : "r"(ta));
  asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
  for (int j = 0; j < 16; j++) out[j] = __uint_as_float(v[j]);
}

// Two stages of kTcCols complex columns: Ah, Al, B1h, B1l, B2h, B2l
// per stage, 96 KB; the MMAs of one stage run while the other is refilled.
constexpr int kTcStage = 6 * kTcTile;
constexpr int kTcSmemFloats = 2 * kTcStage;     // 96 KB: two CTAs per SM
__global__ void __launch_bounds__(256, 2) k_cb_tc(const int4* tasks, const SnDev* sn, const int64_t* scr_off,
                                               float2* fronts, const float2* scratch, DevStatus* status,
                                               int first_wait) {
  extern __shared__ __align__(1024) float tsm[];
  __shared__ float2 dinv[kMaxK];
  __shared__ __align__(8) uint64_t mbar[2];
  __shared__ uint32_t tmem_base;
  const int4 t = tasks[blockIdx.x];
  const SnDev S = sn[t.x];
  const int k = S.k, m = S.m, r = m - k, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row = tid & 127, half = tid >> 7;        // staging: tile row, and which 8 of 16 columns
  const int a0 = t.y * 128, b0 = t.z * 128;
  const float2* W = scratch + scr_off[t.x];          // r x k, column-major (ld r)
  float2* F = fronts + S.frontoff;
  for (int i = tid; i < k; i += blockDim.x) dinv[i] = F[i + int64_t(i) * m];
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 :: "r"(smem_addr(&tmem_base)), "r"(256));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_addr(&mbar[0])), "r"(1));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_addr(&mbar[1])), "r"(1));
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base;
  // K is interleaved by complex column: K' = 2i holds the real parts, 2i + 1 the imaginary
  // ones, so Re = sum A B1^T, Im = sum A B2^T with A = (Wr, Wi), B1 = (Br, -Bi), B2 = (Bi, Br)
  const int nst = (k + kTcCols - 1) / kTcCols;
  constexpr int QH = kTcCols / 2;                   // complex columns per thread per stage
  const int ra = a0 + row, rb = b0 + row;
  // a stage's 16 operand values per thread are loaded into registers in one go, the next
  // stage's right after this stage's MMAs are issued, so the loads overlap the MMAs
  float2 av[QH], bw[QH];
  auto load_stage = [&](int st) {
#pragma unroll
    for (int q = 0; q < QH; q++) {
      const int i = kTcCols * st + QH * half + q;
      av[q] = (i < k && ra < r) ? W[ra + int64_t(i) * r] : make_float2(0.f, 0.f);
      bw[q] = (i < k && rb < r) ? W[rb + int64_t(i) * r] : make_float2(0.f, 0.f);
    }
  };
  load_stage(0);
  bool ok = true;
  int issued = 0;                                    // stages whose MMAs were committed
  for (int st = 0; st < nst; st++) {
    const int b = st & 1;
    if (st >= 2) {                                   // buffer b: stage st - 2's MMAs must be done
      const bool mine = tc_wait(&mbar[b], uint32_t((st - 2) >> 1) & 1u, first_wait);
      ok = __syncthreads_and(mine) != 0;             // block-uniform
      if (!ok) break;
    }
    float* Ah = tsm + b * kTcStage;
    float* Al = Ah + kTcTile;
    float* B1h = Al + kTcTile;
    float* B1l = B1h + kTcTile;
    float* B2h = B1l + kTcTile;
    float* B2l = B2h + kTcTile;
    // two complex columns fill a 16-byte core-matrix row: one conflict-free vector store per operand
#pragma unroll
    for (int q = 0; q < QH; q += 2) {
      const int i = kTcCols * st + QH * half + q;
      const float2 b0 = i < k ? cmul(bw[q], dinv[i]) : make_float2(0.f, 0.f);
      const float2 b1 = i + 1 < k ? cmul(bw[q + 1], dinv[i + 1]) : make_float2(0.f, 0.f);
      const int o = tc_off(row, 2 * (QH * half + q));
      const float4 a = make_float4(av[q].x, av[q].y, av[q + 1].x, av[q + 1].y);
      const float4 c1 = make_float4(b0.x, -b0.y, b1.x, -b1.y), c2 = make_float4(b0.y, b0.x, b1.y, b1.x);
      tc_split(a, Ah + o, Al + o);
      tc_split(c1, B1h + o, B1l + o);
      tc_split(c2, B2h + o, B2l + o);
    }
    asm volatile("fence.proxy.async.shared::cta;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (tid == 0) {
      for (int kk = 0; kk < kTcK / 8; kk++) {
        const uint32_t off = kk * 256;                // two core matrices (8 K values) per MMA
        const uint32_t acc0 = (st > 0 || kk > 0) ? 1u : 0u;
        const uint64_t dah = tc_desc(smem_addr(Ah) + off), dal = tc_desc(smem_addr(Al) + off);
        tc_mma(tmem, dah, tc_desc(smem_addr(B1h) + off), acc0);
        tc_mma(tmem, dah, tc_desc(smem_addr(B1l) + off), 1u);
        tc_mma(tmem, dal, tc_desc(smem_addr(B1h) + off), 1u);
        tc_mma(tmem + 128, dah, tc_desc(smem_addr(B2h) + off), acc0);
        tc_mma(tmem + 128, dah, tc_desc(smem_addr(B2l) + off), 1u);
        tc_mma(tmem + 128, dal, tc_desc(smem_addr(B2h) + off), 1u);
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                   :: "r"(smem_addr(&mbar[b])));
    }
    issued = st + 1;
    if (st + 1 < nst) load_stage(st + 1);
  }
  // the front entries of this thread's row: loaded before their stores, or each would wait for
  // the memory in turn (a >= bb: the lower triangle, and then bb < r too)
  const int q4 = warp & 3, ch = warp >> 2;             // TMEM lanes 32 q4.., columns 64 ch..
  const int a = a0 + q4 * 32 + lane;
  float2* Fa = F + (k + a) + int64_t(k) * m;
  auto load_front = [&](int h, float2* f) {
#pragma unroll
    for (int j = 0; j < 16; j++) {
      const int bb = b0 + ch * 64 + h * 16 + j;
      f[j] = a < r && a >= bb ? Fa[int64_t(bb) * m] : make_float2(0.f, 0.f);
    }
  };
  float2 fv[16];
  load_front(0, fv);
  // the last stage's commit covers every MMA before it (they complete in order)
  const int L = issued - 1;
  uint64_t* lbar = &mbar[L & 1];
  const uint32_t lpar = uint32_t(L >> 1) & 1u;
  if (ok) {
    const bool mine = tc_wait(lbar, lpar, first_wait);
    ok = __syncthreads_and(mine) != 0;
  }
  if (!ok) {
    const bool drained = tc_wait(lbar, lpar, kTcDrainPolls);   // MMAs still in flight
    const bool all = __syncthreads_and(drained) != 0;
    if (tid == 0) atomicOr(&status->timeout, all ? 1u : 3u);
  }
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (ok) {
#pragma unroll 1
    for (int h = 0; h < 4; h++) {
      if (h > 0) load_front(h, fv);
      float re[16], im[16];
      const uint32_t ta = tmem + (uint32_t(q4 * 32) << 16) + ch * 64 + h * 16;
      tc_ld16(ta, re);
      tc_ld16(ta + 128, im);
#pragma unroll
      for (int j = 0; j < 16; j++) {
        const int bb = b0 + ch * 64 + h * 16 + j;
        if (a < r && a >= bb) Fa[int64_t(bb) * m] = make_float2(fv[j].x - re[j], fv[j].y - im[j]);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(256));
}

// Zeroes the lower triangles of a level's fronts (nothing reads above them).  grid.y CTAs
// share a front's columns, one column per warp at a time: bound by writing the fronts, and a
// single CTA per front left the top levels' few tall fronts to a few SMs (28 -> 2 ms per
// factorisation of the 349,461-dof survey model, both precisions' factors).
template <typename V>
__global__ void __launch_bounds__(256) k_front_zero(const int32_t* lev_sn, const SnDev* sn, V* fronts) {
  const SnDev S = sn[lev_sn[blockIdx.x]];
  V* f = fronts + S.frontoff;
  for (int j = blockIdx.y * 8 + (threadIdx.x >> 5); j < S.m; j += 8 * gridDim.y)
    for (int r = j + (threadIdx.x & 31); r < S.m; r += 32) f[int64_t(j) * S.m + r] = czero<V>();
}

// Copies a level's panels from the fronts to the factor store (grid as above); padding rows
// are zero.
template <typename V>
__global__ void __launch_bounds__(256) k_panel_copy(const int32_t* lev_sn, const SnDev* sn, const V* fronts,
                                                    V* panels) {
  const SnDev S = sn[lev_sn[blockIdx.x]];
  const V* src = fronts + S.frontoff;
  V* dst = panels + S.paneloff;
  for (int j = blockIdx.y * 8 + (threadIdx.x >> 5); j < S.k; j += 8 * gridDim.y)
    for (int r = threadIdx.x & 31; r < S.ld; r += 32)
      dst[int64_t(j) * S.ld + r] = (r >= j && r < S.m) ? src[int64_t(j) * S.m + r] : czero<V>();
}

// CTAs per supernode of a level, so that its columns (8 per CTA at a time) and the whole level
// fill the GPU about twice over
static unsigned split_for(int64_t nb, int64_t cols) {
  const int64_t want = std::max<int64_t>(1, 152 * 16 / std::max<int64_t>(nb, 1));
  return unsigned(std::max<int64_t>(1, std::min(want, (cols + 7) / 8)));
}


// One tree level of one factorisation group (whole matrices whose fronts share the
// workspace at once): each task list holds, per level, the groups' tasks in order.
template <typename V>
static void factor_level_t(const FactorDev& F, int lev, int grp, double w, V* fronts, V* scratch,
                           DevStatus* status, double tiny, cudaStream_t st) {
  const int G1 = F.ngrp + 1;
  auto range = [&](const int64_t* gp, int64_t row, int64_t& b, int64_t& e) {
    b = gp[row * G1 + grp];
    e = gp[row * G1 + grp + 1];
  };
  int64_t lb, le;
  range(F.h_lev_g, lev, lb, le);
  const int64_t nb = le - lb;
  const int32_t* lsn = F.lev_sn + lb;
  if (nb > 0) {
    HZ_COUNT();
    k_front_zero<V><<<dim3(unsigned(nb), split_for(nb, F.maxm)), 256, 0, st>>>(lsn, F.sn, fronts);
  }
  int64_t e0, e1;
  range(F.h_ent_g, lev, e0, e1);
  if (e1 > e0) {
    HZ_COUNT();
    k_front_fill<V><<<grid_for(e1 - e0, 256), 256, 0, st>>>(e1 - e0, F.epos + e0, F.ek + e0, F.em + e0, F.eb + e0,
                                                           w, fronts);
  }
  if constexpr (sizeof(V) == 16) {
    if (nb > 0) {
      HZ_COUNT();
      k_front_scale<<<dim3(unsigned(nb), split_for(nb, F.h_flev_k[size_t(lev)])), 256, 0, st>>>(lsn, F.sn, F.rowlist,
                                                                                               F.sig, fronts);
    }
  }
  // extend-add, one child slot per launch so that no parent entry is written twice
  for (int q = 0; q < F.max_slot; q++) {
    int64_t b, e;
    range(F.h_ea_g, int64_t(lev) * F.max_slot + q, b, e);
    if (e > b) {
      HZ_COUNT();
      k_extend_add<V><<<unsigned(e - b), 256, 0, st>>>(F.ea_tasks + b, F.sn, F.rel, F.reloff, fronts);
    }
  }
  if (nb == 0) return;
  const int maxk = F.h_flev_k[size_t(lev)];
  launch_diag(F.precision, nb, maxk, lsn, F.sn, F.sig, fronts, status, tiny, st);
  int64_t wb, we;
  range(F.h_wg_g, lev, wb, we);
  if (we > wb) {
    if constexpr (sizeof(V) == 8) {
      HZ_COUNT();
      const int kpad = (maxk + 15) / 16 * 16;
      k_wg32<<<unsigned(we - wb), 256, size_t(kpad * kWgPitch + 32 * kWgTPitch) * 8, st>>>(F.wg_tasks + wb, F.sn,
                                                                                           F.scr_off, fronts, scratch, kpad);
    } else {
      launch_wg_dig(we - wb, maxk, F.wg_tasks + wb, F, fronts, scratch, status, st);
    }
  }
  if constexpr (sizeof(V) == 8) {
    int64_t tb, te;
    range(F.h_tc_g, lev, tb, te);
    if (te > tb) {
      HZ_COUNT();
      k_cb_tc<<<unsigned(te - tb), 256, kTcSmemFloats * sizeof(float), st>>>(F.tc_tasks + tb, F.sn, F.scr_off,
                                                                            fronts, scratch, status, F.tc_wait);
    }
  } else {
    int64_t cbb, cbe;
    range(F.h_cb_g, lev, cbb, cbe);
    if (cbe > cbb) launch_cb_dig(cbe - cbb, maxk, F.cb_tasks + cbb, F, fronts, scratch, st);
  }
  HZ_COUNT();
  k_panel_copy<V><<<dim3(unsigned(nb), split_for(nb, maxk)), 256, 0, st>>>(lsn, F.sn, fronts, (V*)F.panels);
}

static void set_attrs() {
  static const bool done = [] {
    cudaFuncSetAttribute(k_cb_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmemFloats * int(sizeof(float)));
    cudaFuncSetAttribute(k_wg32, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    return true;
  }();
  (void)done;
}

void launch_factor_level(const FactorDev& F, int lev, int grp, double w, void* fronts, void* scratch,
                         DevStatus* status, double tiny, cudaStream_t st) {
  set_attrs();
  if (F.precision == 0)
    factor_level_t<double2>(F, lev, grp, w, (double2*)fronts, (double2*)scratch, status, tiny, st);
  else
    factor_level_t<float2>(F, lev, grp, w, (float2*)fronts, (float2*)scratch, status, tiny, st);
}

// ---------------------------------------------------------------------------
// batched supernodal solves  (A_i^{-1}: forward with D^{-1}, then backward)
// ---------------------------------------------------------------------------
// a vector entry on its way into the factor's scaling and out of it (complex128 factors)
template <typename V> __device__ __forceinline__ V scaled_in(double2 v, const int16_t* sig, int64_t l) {
  if constexpr (sizeof(V) == 16) {
    const double c = exp2i(-sig[l]);
    return make_double2(v.x * c, v.y * c);
  } else {
    return from2<V>(v);
  }
}
template <typename V> __device__ __forceinline__ double scaled_weight(double pw, const int16_t* sig, int32_t l) {
  if constexpr (sizeof(V) == 16) return pw * exp2i(-sig[l]);
  else return pw;
}
template <typename V>
__global__ void k_gather(int64_t ntot, const int32_t* gidx, const int16_t* sig, const double2* src, V* dst) {
  for (int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; q < ntot; q += int64_t(gridDim.x) * blockDim.x)
    dst[q] = scaled_in<V>(src[gidx[q]], sig, q);
}

// Backward, split over row chunks so that tall supernodes use many CTAs:
//   partial[task][c] = sum over the task's rows r > j of P[r][j] vec[r],
//   vec = (z, -x[ancestor rows]) for 32 pivot columns j of one supernode;
// then x[j] = z[j] + sum of the partials in chunk order (deterministic).
constexpr int kBwdRows = 512;
// complex64 forward, 512 / CG rows of one supernode per task: thread t owns the row
// pair (2p, 2p+1), p = t % (256 / CG), for the pivot columns j = t / (256 / CG) mod CG,
// with 16-byte loads; the right-hand side b1 is gathered once per task.  CG = 2 (256
// rows) where a tree level has many supernodes; CG = 8 (64 rows, each warp one column
// group) on sparse levels, where a task's serial walk over its columns, not bandwidth,
// sets the time.  In both, a thread's first 8 panel values are loaded, and the update
// rows' child contributions b2 gathered, before the barrier that publishes b1, so the
// load chains overlap; with CG = 2 the next kFwdAsync values are also copied into shared
// memory (cp.async) before the gather.  Every sum keeps the order of the column loop
// (even q on one chain, odd q on the other).
constexpr int kFwdAsync = 8, kFwdNarrowAsync = 8;
template <int CG>
__device__ __forceinline__ void fwd_c64_item(const int2 t, const SnDev* sn, const uint32_t* cptr,
                                             const uint32_t* wpos, const float2* panels, const float2* tin,
                                             float2* zout, float2* u) {
  constexpr int NP = 256 / CG;                       // row pairs per task
  constexpr int ROWS = 2 * NP;
  __shared__ float2 b1[kMaxSolveK64];
  __shared__ float2 part[CG][ROWS];
  const SnDev S = sn[t.x];
  const int k = S.k, m = S.m, tid = threadIdx.x;
  const int pr = tid % NP, cg = tid / NP;
  const uint32_t* cp = cptr + S.rowoff + S.id;
  const float2* ub = u + S.ubase;
  const int r = t.y * ROWS + 2 * pr;                 // rows r, r + 1 (r even, ld % 4 == 0)
  const int rr = t.y * ROWS + tid;                   // update row finished by this thread
  // where this thread's child contributions lie and where its update goes: loaded before the
  // wait for the previous level, so that only the contributions themselves come after it
  const bool upd = tid < ROWS && rr >= k && rr < m;
  const uint32_t g0 = tid < k ? cp[tid] : 0u, g1 = tid < k ? cp[tid + 1] : 0u;
  const uint32_t h0 = upd ? cp[rr] : 0u, h1 = upd ? cp[rr + 1] : 0u;
  float2* uw = u + (upd ? S.wbase + wpos[S.rowoff + rr] : 0);
  float2 a0 = make_float2(0.f, 0.f), a1 = a0, c0 = a0, c1 = a0, b2 = a0;
  if constexpr (CG == 8) {
    constexpr int MQ = kMaxK / CG, PF = 8;              // PF of the MQ columns are prefetched,
    constexpr int NA = kFwdNarrowAsync;                 // the next NA copied by cp.async
    __shared__ __align__(16) float4 apf[NA > 0 ? NA * 256 : 1];
    float4 pv[MQ];
    const int j0 = min(r, k), j1 = min(r + 1, k);
    const float4* P4 = reinterpret_cast<const float4*>(panels + S.paneloff + (r < m ? r : 0));
    const int64_t ld4 = S.ld / 2;
#pragma unroll
    for (int q = 0; q < PF; q++) {
      const int j = cg + CG * q;
      pv[q] = (r < m && j < j1) ? P4[int64_t(j) * ld4] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int q = PF; q < PF + NA; q++) {
      const int j = cg + CG * q;
      if (r < m && j < j1) cp_async16(&apf[(q - PF) * 256 + tid], P4 + int64_t(j) * ld4);
    }
    pdl_wait();
    for (int jj = tid; jj < k; jj += 256) {
      const uint32_t c0 = jj == tid ? g0 : cp[jj], c1 = jj == tid ? g1 : cp[jj + 1];
      float2 acc = ldv(tin + S.first + jj);
      for (uint32_t c = c0; c < c1; c++) acc = cadd(acc, ldv(ub + c));
      b1[jj] = acc;
    }
    for (uint32_t c = h0; c < h1; c++) b2 = cadd(b2, ldv(ub + c));
    if constexpr (NA > 0) cp_async_wait_all();        // each thread reads back only its own copies
    __syncthreads();
    if (r < m) {
#pragma unroll
      for (int q = 0; q < MQ; q++) {
        const int j = cg + CG * q;
        if (j < j1) {
          if (q >= PF && q < PF + NA) pv[q] = apf[(q - PF) * 256 + tid];
          else if (q >= PF) pv[q] = P4[int64_t(j) * ld4];
          const float2 bj = b1[j];
          if (q % 2 == 0) {
            a1 = cmad(make_float2(pv[q].z, pv[q].w), bj, a1);
            if (j < j0) a0 = cmad(make_float2(pv[q].x, pv[q].y), bj, a0);
          } else {
            c1 = cmad(make_float2(pv[q].z, pv[q].w), bj, c1);
            if (j < j0) c0 = cmad(make_float2(pv[q].x, pv[q].y), bj, c0);
          }
        }
      }
      // merged solve supernodes wider than kMaxK: the remaining columns, same chains
      int j = cg + CG * MQ;
      for (; j + CG < j1; j += 2 * CG) {
        const float4 p = P4[int64_t(j) * ld4];
        const float4 q = P4[int64_t(j + CG) * ld4];
        const float2 bj = b1[j], bq = b1[j + CG];
        a1 = cmad(make_float2(p.z, p.w), bj, a1);
        c1 = cmad(make_float2(q.z, q.w), bq, c1);
        if (j < j0) a0 = cmad(make_float2(p.x, p.y), bj, a0);
        if (j + CG < j0) c0 = cmad(make_float2(q.x, q.y), bq, c0);
      }
      if (j < j1) {
        const float4 p = P4[int64_t(j) * ld4];
        const float2 bj = b1[j];
        a1 = cmad(make_float2(p.z, p.w), bj, a1);
        if (j < j0) a0 = cmad(make_float2(p.x, p.y), bj, a0);
      }
    }
  } else {
    constexpr int PF = 8;                              // columns q < PF are prefetched
    constexpr int NA = kFwdAsync;                      // columns PF <= q < PF + NA: cp.async
    __shared__ __align__(16) float4 apf[NA > 0 ? NA * 256 : 1];
    float4 pv[PF];
    const int j0 = min(r, k), j1 = min(r + 1, k);
    const float4* P4 = reinterpret_cast<const float4*>(panels + S.paneloff + (r < m ? r : 0));
    const int64_t ld4 = S.ld / 2;
#pragma unroll
    for (int q = 0; q < PF; q++) {
      const int j = cg + CG * q;
      pv[q] = (r < m && j < j1) ? P4[int64_t(j) * ld4] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int q = 0; q < NA; q++) {
      const int j = cg + CG * (PF + q);
      if (r < m && j < j1) cp_async16(&apf[q * 256 + tid], P4 + int64_t(j) * ld4);
    }
    pdl_wait();
    for (int jj = tid; jj < k; jj += 256) {
      const uint32_t c0 = jj == tid ? g0 : cp[jj], c1 = jj == tid ? g1 : cp[jj + 1];
      float2 acc = ldv(tin + S.first + jj);
      for (uint32_t c = c0; c < c1; c++) acc = cadd(acc, ldv(ub + c));
      b1[jj] = acc;
    }
    for (uint32_t c = h0; c < h1; c++) b2 = cadd(b2, ldv(ub + c));
    if constexpr (NA > 0) cp_async_wait_all();        // each thread reads back only its own copies
    __syncthreads();
    if (r < m) {
#pragma unroll
      for (int q = 0; q < PF; q++) {
        const int j = cg + CG * q;
        if (j < j1) {
          const float2 bj = b1[j];
          if (q % 2 == 0) {
            a1 = cmad(make_float2(pv[q].z, pv[q].w), bj, a1);
            if (j < j0) a0 = cmad(make_float2(pv[q].x, pv[q].y), bj, a0);
          } else {
            c1 = cmad(make_float2(pv[q].z, pv[q].w), bj, c1);
            if (j < j0) c0 = cmad(make_float2(pv[q].x, pv[q].y), bj, c0);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < NA; q++) {
        const int j = cg + CG * (PF + q);
        if (j < j1) {
          const float4 p = apf[q * 256 + tid];
          const float2 bj = b1[j];
          if ((PF + q) % 2 == 0) {
            a1 = cmad(make_float2(p.z, p.w), bj, a1);
            if (j < j0) a0 = cmad(make_float2(p.x, p.y), bj, a0);
          } else {
            c1 = cmad(make_float2(p.z, p.w), bj, c1);
            if (j < j0) c0 = cmad(make_float2(p.x, p.y), bj, c0);
          }
        }
      }
      int j = cg + CG * (PF + NA);
      for (; j + CG < j1; j += 2 * CG) {               // two independent chains
        const float4 p = P4[int64_t(j) * ld4];
        const float4 q = P4[int64_t(j + CG) * ld4];
        const float2 bj = b1[j], bq = b1[j + CG];
        a1 = cmad(make_float2(p.z, p.w), bj, a1);
        c1 = cmad(make_float2(q.z, q.w), bq, c1);
        if (j < j0) a0 = cmad(make_float2(p.x, p.y), bj, a0);
        if (j + CG < j0) c0 = cmad(make_float2(q.x, q.y), bq, c0);
      }
      if (j < j1) {
        const float4 p = P4[int64_t(j) * ld4];
        const float2 bj = b1[j];
        a1 = cmad(make_float2(p.z, p.w), bj, a1);
        if (j < j0) a0 = cmad(make_float2(p.x, p.y), bj, a0);
      }
    }
  }
  part[cg][2 * pr] = cadd(a0, c0);
  part[cg][2 * pr + 1] = cadd(a1, c1);
  __syncthreads();
  if (tid < ROWS && rr < m) {
    float2 tot = part[0][tid];
#pragma unroll
    for (int q = 1; q < CG; q++) tot = cadd(tot, part[q][tid]);
    const float2* P = panels + S.paneloff;
    if (rr < k)
      zout[S.first + rr] = cmul(P[rr + int64_t(rr) * S.ld], cadd(b1[rr], tot));
    else
      *uw = csub(b2, tot);
  }
}

template <int CG>
__global__ void __launch_bounds__(256, 4) k_fwd_c64(const int2* tasks, const SnDev* sn, const uint32_t* cptr,
                                                 const uint32_t* wpos, const float2* panels, const float2* tin,
                                                 float2* zout, float2* u) {
  pdl_trigger();
  fwd_c64_item<CG>(tasks[blockIdx.x], sn, cptr, wpos, panels, tin, zout, u);
}

// complex64 backward partial sums with 16-byte loads (two rows per lane), two forms:
//   kBwdAsync  (wide chunks): the first kBwdAsyncIt row pairs per lane and column are copied
//              into shared memory by asynchronous copies (cp.async, no registers held)
//              issued before the gather, so the panel stream starts while the gather's
//              dependent loads are in flight; the rest of each column is loaded in the loop;
//   kBwdPrefetch (narrow chunks of at most 128 rows, sparse levels): each lane's <= 2 row
//              pairs of its 4 columns are loaded into registers before the gather.
// Both keep the column loop's sums in its order.  The panel loads issued before the gather
// do not depend on earlier levels; the kernel waits for the previous level
// (griddepcontrol.wait, a no-op without programmatic dependent launch) only after them,
// before its first read of x.  A supernode that fits in one chunk is finished by
// its own CTA (lane 0 of each column's warp), with the same sums, without the partial-sum
// round trip and ticket of bwd_finish.
enum { kBwdAsync = 1, kBwdPrefetch = 2 };
constexpr int kBwdAsyncIt = 2;
template <int MODE>
__global__ void __launch_bounds__(256, MODE == kBwdPrefetch ? 4 : 6)
    k_bwd_partial_c64(const int4* tasks, const SnDev* sn, const int32_t* rowlist, const float2* panels,
                      const float2* zin, float2* x, float2* partial, int rows, const int4* fins,
                      unsigned int* counters) {
  pdl_trigger();
  __shared__ __align__(16) float2 vec[kBwdRows + 2];
  __shared__ __align__(16) float4 apf[MODE == kBwdAsync ? 4 * kBwdAsyncIt * 256 : 1];
  const int4 t = tasks[blockIdx.x];
  const SnDev S = sn[t.x];
  const int k = S.k, m = S.m, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int r0 = t.z * rows, r1 = min(m, r0 + rows);
  const int32_t* rl = rowlist + S.rowoff;
  float4 pre[4][2];
  if constexpr (MODE == kBwdPrefetch) {
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int j = t.y * 32 + wid + 8 * q;
      const float4* col = reinterpret_cast<const float4*>(panels + S.paneloff + int64_t(j < k ? j : 0) * S.ld);
      const int rs = max(r0, (j + 1) & ~1);
#pragma unroll
      for (int it = 0; it < 2; it++) {
        const int r = rs + 2 * lane + 64 * it;
        pre[q][it] = (j < k && r < r1) ? col[r >> 1] : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  } else if constexpr (MODE == kBwdAsync) {
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int j = t.y * 32 + wid + 8 * q;
      const float4* col = reinterpret_cast<const float4*>(panels + S.paneloff + int64_t(j < k ? j : 0) * S.ld);
      const int rs = max(r0, (j + 1) & ~1);
#pragma unroll
      for (int it = 0; it < kBwdAsyncIt; it++) {
        const int r = rs + 2 * lane + 64 * it;
        if (j < k && r < r1) cp_async16(&apf[(q * kBwdAsyncIt + it) * 256 + tid], col + (r >> 1));
      }
    }
  }
  pdl_wait();
  for (int r = r0 + tid; r < r0 + rows + 2; r += blockDim.x)
    vec[r - r0] = (r < r1) ? ((r < k) ? zin[S.first + r] : cneg(x[rl[r]])) : make_float2(0.f, 0.f);
  if constexpr (MODE == kBwdAsync) cp_async_wait_all();     // each thread reads back only its own copies
  __syncthreads();
  float2* out = partial + int64_t(blockIdx.x) * 32;
  const bool single = m <= rows;                     // the only chunk: finish here, no ticket
  const float4* vec4 = reinterpret_cast<const float4*>(vec);
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const int c = wid + 8 * q;
    const int j = t.y * 32 + c;
    float2 acc = make_float2(0.f, 0.f);
    if (j < k) {
      const int rs = max(r0, (j + 1) & ~1);          // first even row of the pair holding row j + 1
      if constexpr (MODE == kBwdPrefetch) {
#pragma unroll
        for (int it = 0; it < 2; it++) {
          const int r = rs + 2 * lane + 64 * it;
          if (r < r1) {
            const float4 p = pre[q][it];
            const float4 v = vec4[(r - r0) >> 1];
            if (r > j) acc = cmad(make_float2(p.x, p.y), make_float2(v.x, v.y), acc);
            acc = cmad(make_float2(p.z, p.w), make_float2(v.z, v.w), acc);
          }
        }
      } else {
        const float4* col = reinterpret_cast<const float4*>(panels + S.paneloff + int64_t(j) * S.ld);
        int r = rs + 2 * lane;
        if constexpr (MODE == kBwdAsync) {
#pragma unroll
          for (int it = 0; it < kBwdAsyncIt; it++, r += 64) {
            if (r < r1) {
              const float4 p = apf[(q * kBwdAsyncIt + it) * 256 + tid];
              const float4 v = vec4[(r - r0) >> 1];
              if (r > j) acc = cmad(make_float2(p.x, p.y), make_float2(v.x, v.y), acc);
              acc = cmad(make_float2(p.z, p.w), make_float2(v.z, v.w), acc);
            }
          }
        }
#pragma unroll 4
        for (; r < r1; r += 64) {
          const float4 p = col[r >> 1];
          const float4 v = vec4[(r - r0) >> 1];
          if (r > j) acc = cmad(make_float2(p.x, p.y), make_float2(v.x, v.y), acc);
          acc = cmad(make_float2(p.z, p.w), make_float2(v.z, v.w), acc);
        }
      }
    }
    acc = warp_sum(acc);
    if (lane == 0) {
      if (!single)
        out[c] = acc;
      else if (j < k)
        x[S.first + j] = cadd(zin[S.first + j], cadd(make_float2(0.f, 0.f), acc));
    }
  }
  if (!single) bwd_finish<float2>(fins[t.w], S, zin, partial, x, counters + t.w);
}

template <typename V>
__global__ void k_prolong(int64_t n, const int64_t* pptr, const int32_t* pidx, const double* pw, const int16_t* sig,
                          const V* xl, const double2* y, double2* z) {
  for (int64_t g = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; g < n; g += int64_t(gridDim.x) * blockDim.x) {
    double2 acc = y ? y[g] : make_double2(0.0, 0.0);
    for (int64_t q = pptr[g]; q < pptr[g + 1]; q++) {
      const double2 v = to2(xl[pidx[q]]);
      const double c = scaled_weight<V>(pw[q], sig, pidx[q]);
      acc.x = xfma(c, v.x, acc.x);
      acc.y = xfma(c, v.y, acc.y);
    }
    z[g] = acc;
  }
}

static void solve_c64(const FactorDev& F, cudaStream_t st) {
  const float2* P = (const float2*)F.panels;
  float2 *t = (float2*)F.t_loc, *z = (float2*)F.z_loc, *x = (float2*)F.x_loc, *u = (float2*)F.u_ws;
  float2* part = (float2*)F.bwd_partial;
  const bool pdl = pdl_enabled();
  if (F.level_events) cudaEventRecord(F.level_events[0], st);
  for (int l = 0; l < F.snlev; l++) {
    const int64_t b = F.h_fwd_ptr[l], e = F.h_fwd_ptr[l + 1];
    if (e > b) {
      HZ_COUNT();
      const int2* tk = F.fwd_tasks + b;
      if (F.h_fwd_rt[l] == 64)
        launch_level(k_fwd_c64<8>, e - b, 256, 0, st, pdl, tk, F.ssn, F.cptr, F.wpos, P, t, z, u);
      else
        launch_level(k_fwd_c64<2>, e - b, 256, 0, st, pdl, tk, F.ssn, F.cptr, F.wpos, P, t, z, u);
    }
    if (F.level_events) cudaEventRecord(F.level_events[1 + l], st);
  }
  for (int l = F.snlev - 1; l >= 0; l--) {
    const int64_t b = F.h_bwd_ptr[l], e = F.h_bwd_ptr[l + 1];
    if (e > b) {
      HZ_COUNT();
      const int4* tk = F.bwd_tasks + b;
      const int rows = F.h_bwd_rows[l];
      if (rows <= 128)
        launch_level(k_bwd_partial_c64<kBwdPrefetch>, e - b, 256, 0, st, pdl, tk, F.ssn, F.rowlist, P, z, x, part, rows,
                     F.bfin_tasks, F.bwd_counters);
      else
        launch_level(k_bwd_partial_c64<kBwdAsync>, e - b, 256, 0, st, pdl, tk, F.ssn, F.rowlist, P, z, x, part, rows,
                     F.bfin_tasks, F.bwd_counters);
    }
    if (F.level_events) cudaEventRecord(F.level_events[1 + F.snlev + (F.snlev - 1 - l)], st);
  }
}

void launch_gather(const FactorDev& F, const double2* src, cudaStream_t st) {
  if (F.ntot == 0) return;
  if (F.precision == 0) {
    HZ_COUNT();
    k_gather<double2><<<grid_for(F.ntot, 256), 256, 0, st>>>(F.ntot, F.gidx, F.sig, src, (double2*)F.t_loc);
  } else {
    HZ_COUNT();
    k_gather<float2><<<grid_for(F.ntot, 256), 256, 0, st>>>(F.ntot, F.gidx, F.sig, src, (float2*)F.t_loc);
  }
}

void launch_solve(const FactorDev& F, cudaStream_t st) {
  if (F.precision == 0) launch_solve_dig(F, st);
  else solve_c64(F, st);
}

// ---------------------------------------------------------------------------
// merged solve supernodes (complex128 and complex64 factors): a chain s_1 -> s_2 -> ... in which each
// supernode is the only child of the next and its rows below its pivots are exactly the
// next one's rows.  A supernode's panel holds T = L11^{-1} (strict lower part; D^{-1} on the
// diagonal) over G = L21 L11^{-1}.  Appending s (T_s, G_s) to the merged M (T_M, G_M, width
// w, rows P_M, P_s, R_s in that order) gives
//   T' = [[T_M, 0], [-T_s A, T_s]],  G' = [G_M(R_s) - G_s A, G_s],  A = G_M(P_s rows),
// from the block inverse of [[L11^M, 0], [L(P_s, P_M), L11^s]] (T_s taken with a unit
// diagonal in the product).  Same entries, so the sweep reads the same bytes, in fewer
// dependent levels.
// ---------------------------------------------------------------------------
// tmp (ks x w, column-major) = M[w .. w + ks, 0 .. w)
template <typename V>
__global__ void k_merge_save(const V* M, int ldm, int w, int ks, V* tmp) {
  const int64_t n = int64_t(ks) * w;
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < n; e += int64_t(gridDim.x) * blockDim.x) {
    const int q = int(e % ks), c = int(e / ks);
    tmp[e] = M[(w + q) + int64_t(ldm) * c];
  }
}

// M[w + i, c] = (i >= ks ? M[w + i, c] : 0) - sum_q C(i, q) tmp[q, c] for i < ms, c < w, with
// C = [T_s (unit diagonal, upper part 0); G_s] the appended panel.  64 x 32 output tiles,
// 16-deep slices of q staged in shared memory; each thread owns 4 rows x 2 columns.  The
// sums run in the panels' precision (the complex64 factor is itself computed in FP32).
template <typename V>
__global__ void __launch_bounds__(256) k_merge_update(V* M, int ldm, int w, const V* Ps, int lds,
                                                      int ks, int ms, const V* tmp) {
  __shared__ V Cs[16][64];
  __shared__ V As[16][32];
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int i0 = blockIdx.x * 64, c0 = blockIdx.y * 32;
  V acc[4][2];
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 2; b++) acc[a][b] = czero<V>();
  for (int q0 = 0; q0 < ks; q0 += 16) {
#pragma unroll
    for (int t = 0; t < 4; t++) {
      const int e = tid + 256 * t, il = e & 63, ql = e >> 6;
      const int i = i0 + il, q = q0 + ql;
      V v = czero<V>();
      if (i < ms && q < ks) {
        if (i >= ks || i > q) v = Ps[i + int64_t(lds) * q];
        else if (i == q) v = from2<V>(make_double2(1.0, 0.0));
      }
      Cs[ql][il] = v;
    }
#pragma unroll
    for (int t = 0; t < 2; t++) {
      const int e = tid + 256 * t, ql = e & 15, cl = e >> 4;
      const int q = q0 + ql, c = c0 + cl;
      As[ql][cl] = (q < ks && c < w) ? tmp[q + int64_t(ks) * c] : czero<V>();
    }
    __syncthreads();
#pragma unroll
    for (int ql = 0; ql < 16; ql++) {
      const V b0 = As[ql][2 * tx], b1 = As[ql][2 * tx + 1];
#pragma unroll
      for (int a = 0; a < 4; a++) {
        const V cv = Cs[ql][4 * ty + a];
        acc[a][0] = cmad(cv, b0, acc[a][0]);
        acc[a][1] = cmad(cv, b1, acc[a][1]);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < 4; a++) {
    const int i = i0 + 4 * ty + a;
    if (i >= ms) continue;
#pragma unroll
    for (int b = 0; b < 2; b++) {
      const int c = c0 + 2 * tx + b;
      if (c >= w) continue;
      V* o = M + (w + i) + int64_t(ldm) * c;
      *o = csub(i >= ks ? *o : czero<V>(), acc[a][b]);
    }
  }
}

// M[w + i, w + q] = Ps[i, q] for i < ms, q < ks
template <typename V>
__global__ void k_merge_put(V* M, int ldm, int w, const V* Ps, int lds, int ks, int ms) {
  const int64_t n = int64_t(ks) * ms;
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < n; e += int64_t(gridDim.x) * blockDim.x) {
    const int i = int(e % ms), q = int(e / ms);
    M[(w + i) + int64_t(ldm) * (w + q)] = Ps[i + int64_t(lds) * q];
  }
}

template <typename V>
static void merge_panels_t(const FactorDev& F, cudaStream_t st) {
  V* P = (V*)F.panels;
  V* tmp = (V*)F.merge_tmp;
  for (const FactorDev::MergeStep& m : F.merges) {
    V* M = P + m.moff;
    const V* Ps = P + m.soff;
    if (m.w > 0) {
      HZ_COUNT();
      k_merge_save<<<grid_for(int64_t(m.ks) * m.w, 256), 256, 0, st>>>(M, m.ldm, m.w, m.ks, tmp);
      if constexpr (sizeof(V) == 16) {
        launch_merge_dig(M, m.ldm, m.w, Ps, m.lds, m.ks, m.ms, tmp, st);
      } else {
        HZ_COUNT();
        k_merge_update<<<dim3(unsigned((m.ms + 63) / 64), unsigned((m.w + 31) / 32)), 256, 0, st>>>(
            M, m.ldm, m.w, Ps, m.lds, m.ks, m.ms, tmp);
      }
    }
    HZ_COUNT();
    k_merge_put<<<grid_for(int64_t(m.ks) * m.ms, 256), 256, 0, st>>>(M, m.ldm, m.w, Ps, m.lds, m.ks, m.ms);
  }
}

void launch_merge_panels(const FactorDev& F, cudaStream_t st) {
  if (F.merges.empty()) return;
  if (F.precision == 0) merge_panels_t<double2>(F, st);
  else merge_panels_t<float2>(F, st);
}

void launch_prolong(const FactorDev& F, const double2* y, double2* z, cudaStream_t st) {
  if (F.nglob == 0) return;
  if (F.precision == 0) {
    HZ_COUNT();
    k_prolong<double2><<<grid_for(F.nglob, 256), 256, 0, st>>>(F.nglob, F.pptr, F.pidx, F.pw, F.sig,
                                                               (const double2*)F.x_loc, y, z);
  } else {
    HZ_COUNT();
    k_prolong<float2><<<grid_for(F.nglob, 256), 256, 0, st>>>(F.nglob, F.pptr, F.pidx, F.pw, F.sig,
                                                              (const float2*)F.x_loc, y, z);
  }
}

// ---------------------------------------------------------------------------
// batched preconditioner for S right-hand sides (pseudo-block GMRES):
// vectors are interleaved per row, X[r * S + i].  Each factor panel element is
// read once and used for all S right-hand sides.
// ---------------------------------------------------------------------------
template <typename V, int S>
__global__ void k_gather_multi(int64_t ntot, const int32_t* gidx, const int16_t* sig, const double2* src, V* dst) {
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < ntot * S; e += int64_t(gridDim.x) * blockDim.x) {
    const int64_t q = e / S;
    const int i = int(e % S);
    dst[e] = scaled_in<V>(src[int64_t(gidx[q]) * S + i], sig, q);
  }
}

template <typename V, int S>
__global__ void k_prolong_multi(int64_t n, const int64_t* pptr, const int32_t* pidx, const double* pw, const int16_t* sig,
                                const V* xl, const double2* y, double2* z) {
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < n * S; e += int64_t(gridDim.x) * blockDim.x) {
    const int64_t g = e / S;
    const int i = int(e % S);
    double2 acc = y ? y[e] : make_double2(0.0, 0.0);
    for (int64_t q = pptr[g]; q < pptr[g + 1]; q++) {
      const double2 v = to2(xl[int64_t(pidx[q]) * S + i]);
      const double c = scaled_weight<V>(pw[q], sig, pidx[q]);
      acc.x = xfma(c, v.x, acc.x);
      acc.y = xfma(c, v.y, acc.y);
    }
    z[e] = acc;
  }
}

template <typename V, int S>
static void prec_multi_t(const FactorDev& F, const double2* src, const double2* y, double2* dst, cudaStream_t st) {
  V* t = (V*)F.mt_loc;
  HZ_COUNT();
  k_gather_multi<V, S><<<grid_for(F.ntot * S, 256), 256, 0, st>>>(F.ntot, F.gidx, F.sig, src, t);
  if constexpr (sizeof(V) == 8) launch_solve_multi32(F, S, st);
  else launch_solve_dig_multi(F, S, st);
  HZ_COUNT();
  k_prolong_multi<V, S><<<grid_for(F.nglob * S, 256), 256, 0, st>>>(F.nglob, F.pptr, F.pidx, F.pw, F.sig,
                                                                   (const V*)F.mx_loc, y, dst);
}

// dst = y + sum_i R_i^T D_i A_i^{-1} R_i src  (S interleaved right-hand sides)
void launch_local_multi(const FactorDev& F, int S, const double2* src, const double2* y, double2* dst,
                        cudaStream_t st) {
  if (F.precision == 0) {
    if (S == 4) prec_multi_t<double2, 4>(F, src, y, dst, st);
    else if (S == 8) prec_multi_t<double2, 8>(F, src, y, dst, st);
    else prec_multi_t<double2, 16>(F, src, y, dst, st);
  } else {
    if (S == 4) prec_multi_t<float2, 4>(F, src, y, dst, st);
    else if (S == 8) prec_multi_t<float2, 8>(F, src, y, dst, st);
    else prec_multi_t<float2, 16>(F, src, y, dst, st);
  }
}

// interleaved <-> per-right-hand-side column layouts
// Interleaving of per-slot columns: slot i reads (or writes) base + off.o[i] + r; a
// negative offset marks an empty slot, read as zero and never written.
__global__ void k_interleave(int64_t n, int S, SlotCols off, const double2* base, double2* inter) {
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < n * S; e += int64_t(gridDim.x) * blockDim.x) {
    const int64_t r = e / S;
    const int i = int(e % S);
    const int64_t o = off.o[i];
    inter[e] = (o >= 0) ? base[o + r] : make_double2(0.0, 0.0);
  }
}
__global__ void k_deinterleave(int64_t n, int S, SlotCols off, const double2* inter, double2* base) {
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < n * S; e += int64_t(gridDim.x) * blockDim.x) {
    const int64_t r = e / S;
    const int i = int(e % S);
    const int64_t o = off.o[i];
    if (o >= 0) base[o + r] = inter[e];
  }
}
void launch_interleave(int64_t n, int S, const SlotCols& off, const double2* base, double2* inter, cudaStream_t st) {
  HZ_COUNT();
  k_interleave<<<grid_for(n * S, 256), 256, 0, st>>>(n, S, off, base, inter);
}
void launch_deinterleave(int64_t n, int S, const SlotCols& off, const double2* inter, double2* base, cudaStream_t st) {
  HZ_COUNT();
  k_deinterleave<<<grid_for(n * S, 256), 256, 0, st>>>(n, S, off, inter, base);
}

// Column i of S interleaved vectors set from a plain vector (other columns untouched).
__global__ void k_interleave_put(int64_t n, int S, int i, const double2* col, double2* inter) {
  for (int64_t r = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; r < n; r += int64_t(gridDim.x) * blockDim.x)
    inter[r * S + i] = col[r];
}
void launch_interleave_put(int64_t n, int S, int i, const double2* col, double2* inter, cudaStream_t st) {
  HZ_COUNT();
  k_interleave_put<<<grid_for(n, 256), 256, 0, st>>>(n, S, i, col, inter);
}

// Point-source right-hand side written into a zeroed column: out[idx[q]] += val[q].
__global__ void k_point_rhs(PointRhs p, double2* out) {
  if (threadIdx.x == 0)
    for (int q = 0; q < p.cnt; q++) out[p.idx[q]].x += p.val[q];
}
void launch_point_rhs(const PointRhs& p, double2* out, cudaStream_t st) {
  HZ_COUNT();
  k_point_rhs<<<1, 32, 0, st>>>(p, out);
}

// Y = A X (or SUB - A X) for S interleaved vectors; lanes of a warp split the right-hand sides.
template <int S>
__global__ void __launch_bounds__(256) k_spmv_multi(int64_t n, const int64_t* rp, const int32_t* ci,
                                                    const double2* val, const double2* x, const double2* sub,
                                                    double2* y) {
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < n * S; e += int64_t(gridDim.x) * blockDim.x) {
    const int64_t row = e / S;
    const int i = int(e % S);
    double2 a0 = make_double2(0.0, 0.0), a1 = a0;
    const int64_t q1 = rp[row + 1];
    int64_t q = rp[row];
    for (; q + 1 < q1; q += 2) {
      a0 = cmad(val[q], x[int64_t(ci[q]) * S + i], a0);
      a1 = cmad(val[q + 1], x[int64_t(ci[q + 1]) * S + i], a1);
    }
    if (q < q1) a0 = cmad(val[q], x[int64_t(ci[q]) * S + i], a0);
    const double2 acc = cadd(a0, a1);
    y[e] = sub ? csub(sub[e], acc) : acc;
  }
}
template <int S>
__global__ void __launch_bounds__(256) k_spmv_real_multi(int64_t n, const int64_t* rp, const int32_t* ci,
                                                         const double* val, const double2* x, double2* y) {
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < n * S; e += int64_t(gridDim.x) * blockDim.x) {
    const int64_t row = e / S;
    const int i = int(e % S);
    double2 acc = make_double2(0.0, 0.0);
    for (int64_t q = rp[row]; q < rp[row + 1]; q++) {
      const double2 v = x[int64_t(ci[q]) * S + i];
      acc.x = xfma(val[q], v.x, acc.x);
      acc.y = xfma(val[q], v.y, acc.y);
    }
    y[e] = acc;
  }
}
void launch_spmv_multi(int64_t n, int S, const int64_t* rp, const int32_t* ci, const double2* val, const double2* x,
                       const double2* sub, double2* y, cudaStream_t st) {
  HZ_COUNT();
  const unsigned g = grid_for(n * S, 256, 152 * 32);
  if (S == 4) k_spmv_multi<4><<<g, 256, 0, st>>>(n, rp, ci, val, x, sub, y);
  else if (S == 8) k_spmv_multi<8><<<g, 256, 0, st>>>(n, rp, ci, val, x, sub, y);
  else k_spmv_multi<16><<<g, 256, 0, st>>>(n, rp, ci, val, x, sub, y);
}
void launch_spmv_real_multi(int64_t n, int S, const int64_t* rp, const int32_t* ci, const double* val,
                            const double2* x, double2* y, cudaStream_t st) {
  HZ_COUNT();
  const unsigned g = grid_for(n * S, 256, 152 * 32);
  if (S == 4) k_spmv_real_multi<4><<<g, 256, 0, st>>>(n, rp, ci, val, x, y);
  else if (S == 8) k_spmv_real_multi<8><<<g, 256, 0, st>>>(n, rp, ci, val, x, y);
  else k_spmv_real_multi<16><<<g, 256, 0, st>>>(n, rp, ci, val, x, y);
}

// ---------------------------------------------------------------------------
// sparse matrix-vector products
// ---------------------------------------------------------------------------
// Bound by FP64 arithmetic (four FMAs per entry: 66 us for the 9.7M entries of the 349,461-dof
// survey model), a warp taking as long as its longest row: P2 rows hold 10 to 65 entries, and in
// natural order 15 % of the lanes' steps were idle (counted on the 54,925-dof pattern, two lanes per
// row).  SORTED: the rows are walked in an order that sorts them by length within windows of 4,096, which
// keeps the gathers of x local: 3 % idle.  A row's start, length and number lie together in this
// order: the number alone, and then the row's pointers, was one more load in the chain.  Where
// sorting pays: spmv_rows.
template <int TPR, bool SORTED>
__global__ void __launch_bounds__(256) k_spmv(int64_t n, const SpmvRow* rows, const int64_t* rp, const int32_t* ci,
                                              const double2* val, const double2* x, const double2* sub, double2* y) {
  const int lane = threadIdx.x % TPR;
  const int64_t groups = (int64_t(gridDim.x) * blockDim.x) / TPR;
  const int64_t g0 = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) / TPR;
  const int64_t wbase0 = (blockIdx.x * int64_t(blockDim.x) + (threadIdx.x & ~31)) / TPR;
  for (int64_t off = 0; wbase0 + off < n; off += groups) {
    int64_t row = g0 + off;
    const bool in = row < n;
    double2 acc = make_double2(0.0, 0.0);
    if (in) {
      int64_t q, e;
      if constexpr (SORTED) {
        const SpmvRow r = rows[row];
        row = r.row;
        q = r.start;
        e = r.start + r.len;
      } else {
        e = rp[row + 1];
        q = rp[row];
      }
      for (q += lane; q < e; q += TPR) acc = cmad(val[q], x[ci[q]], acc);
    }
    for (int o = TPR / 2; o > 0; o >>= 1) acc = cadd(acc, shfl_xor(acc, o, TPR));
    if (in && lane == 0) y[row] = sub ? csub(sub[row], acc) : acc;
  }
}

__global__ void __launch_bounds__(256) k_spmv_real(int64_t n, const int64_t* rp, const int32_t* ci,
                                                   const double* val, const double2* x, double2* y) {
  constexpr int TPR = 4;
  const int lane = threadIdx.x % TPR;
  const int64_t groups = (int64_t(gridDim.x) * blockDim.x) / TPR;
  const int64_t g0 = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) / TPR;
  const int64_t wbase0 = (blockIdx.x * int64_t(blockDim.x) + (threadIdx.x & ~31)) / TPR;
  for (int64_t off = 0; wbase0 + off < n; off += groups) {
    const int64_t row = g0 + off;
    double2 acc = make_double2(0.0, 0.0);
    if (row < n) {
      const int64_t e = rp[row + 1];
      for (int64_t q = rp[row] + lane; q < e; q += TPR) {
        const double2 v = x[ci[q]];
        acc.x = xfma(val[q], v.x, acc.x);
        acc.y = xfma(val[q], v.y, acc.y);
      }
    }
    for (int o = TPR / 2; o > 0; o >>= 1) acc = cadd(acc, shfl_xor(acc, o, TPR));
    if (row < n && lane == 0) y[row] = acc;
  }
}

// Lanes per row for the complex SpMV (set per context by its autotuner).
static thread_local int g_spmv_tpr = 8;
void set_spmv_lanes(int tpr) { g_spmv_tpr = tpr; }

template <bool SORTED>
static void spmv_lanes(int64_t n, const SpmvRow* rows, const int64_t* rp, const int32_t* ci, const double2* val,
                       const double2* x, const double2* sub, double2* y, cudaStream_t st) {
  const int t = g_spmv_tpr;
  const unsigned g = grid_for(n * t, 256, 152 * 32);
  if (t == 2) k_spmv<2, SORTED><<<g, 256, 0, st>>>(n, rows, rp, ci, val, x, sub, y);
  else if (t == 4) k_spmv<4, SORTED><<<g, 256, 0, st>>>(n, rows, rp, ci, val, x, sub, y);
  else if (t == 16) k_spmv<16, SORTED><<<g, 256, 0, st>>>(n, rows, rp, ci, val, x, sub, y);
  else k_spmv<8, SORTED><<<g, 256, 0, st>>>(n, rows, rp, ci, val, x, sub, y);
}
void launch_spmv(int64_t n, const SpmvRow* rows, const int64_t* rp, const int32_t* ci, const double2* val,
                 const double2* x, const double2* sub, double2* y, cudaStream_t st) {
  if (n == 0) return;
  HZ_COUNT();
  if (rows) spmv_lanes<true>(n, rows, rp, ci, val, x, sub, y, st);
  else spmv_lanes<false>(n, rows, rp, ci, val, x, sub, y, st);
}

void launch_spmv_real(int64_t n, const int64_t* rp, const int32_t* ci, const double* val, const double2* x,
                      double2* y, cudaStream_t st) {
  if (n == 0) return;
  HZ_COUNT();
  k_spmv_real<<<grid_for(n * 4, 256, 152 * 32), 256, 0, st>>>(n, rp, ci, val, x, y);
}

// ---------------------------------------------------------------------------
// GMRES vector updates (the orthogonalisation is in cgs.cu)
// ---------------------------------------------------------------------------
constexpr int kMaxCols = 64;

__global__ void k_scale_slots(int64_t n, SlotScale p) {
  const int i = blockIdx.y;
  if (!p.out[i]) return;
  const double a = *p.s[i];
  for (int64_t r = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; r < n; r += int64_t(gridDim.x) * blockDim.x)
    p.out[i][r] = make_double2(p.w[i][r].x * a, p.w[i][r].y * a);
}
void launch_scale_slots(int64_t n, int S, const SlotScale& p, cudaStream_t st) {
  HZ_COUNT();
  k_scale_slots<<<dim3(std::max(1u, grid_for(n, 256) / unsigned(S)), S), 256, 0, st>>>(n, p);
}

// out[:, q] (+)= sign * (sum_i B1[:, i] coef[i, q] + sum_i B2[:, i] coef[nb1 + i, q]), q < nout:
// linear combinations of two column-major bases (recycled-space updates of GCRO-DR).
// coef is (nb1 + nb2) x nout column-major, staged in shared memory.
constexpr int kComboCols = 80, kComboOut = 16;
__global__ void __launch_bounds__(256) k_combo(int64_t n, int nb1, const double2* B1, int64_t ld1, int nb2,
                                               const double2* B2, int64_t ld2, const double2* coef, int nout,
                                               double2* out, int64_t ldo, double sign, int accumulate) {
  __shared__ double2 cf[kComboCols * kComboOut];
  const int nbt = nb1 + nb2;
  for (int e = threadIdx.x; e < nbt * nout; e += blockDim.x) cf[e] = coef[e];
  __syncthreads();
  for (int64_t r = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; r < n; r += int64_t(gridDim.x) * blockDim.x) {
    double2 acc[kComboOut];
#pragma unroll
    for (int q = 0; q < kComboOut; q++) acc[q] = make_double2(0.0, 0.0);
    for (int i = 0; i < nbt; i++) {
      const double2 v = i < nb1 ? B1[r + int64_t(i) * ld1] : B2[r + int64_t(i - nb1) * ld2];
#pragma unroll
      for (int q = 0; q < kComboOut; q++)
        if (q < nout) acc[q] = cmad(v, cf[q * nbt + i], acc[q]);
    }
    for (int q = 0; q < nout; q++) {
      double2* o = out + r + int64_t(q) * ldo;
      const double2 a = make_double2(sign * acc[q].x, sign * acc[q].y);
      *o = accumulate ? cadd(*o, a) : a;
    }
  }
}
void launch_combo(int64_t n, int nb1, const double2* B1, int64_t ld1, int nb2, const double2* B2, int64_t ld2,
                  const double2* coef, int nout, double2* out, int64_t ldo, double sign, bool accumulate,
                  cudaStream_t st) {
  if (n == 0 || nout == 0) return;
  HZ_COUNT();
  k_combo<<<grid_for(n, 256), 256, 0, st>>>(n, nb1, B1, ld1, nb2, B2, ld2, coef, nout, out, ldo, sign,
                                            accumulate ? 1 : 0);
}

__global__ void k_init_cycle(const double2* nrm2, double2* g, int m, double* invbeta, double* beta) {
  const double b = sqrt(nrm2[kMaxCols].x);
  for (int i = threadIdx.x; i <= m; i += blockDim.x) g[i] = make_double2(i == 0 ? b : 0.0, 0.0);
  if (threadIdx.x == 0) {
    *beta = b;
    *invbeta = 1.0 / b;
  }
}

void launch_init_cycle(const double2* nrm2, double2* g, int m, double* invbeta, double* beta, cudaStream_t st) {
  HZ_COUNT();
  k_init_cycle<<<1, 64, 0, st>>>(nrm2, g, m, invbeta, beta);
}

__global__ void k_scale(int64_t n, const double2* w, const double* s, double2* out) {
  const double a = *s;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    out[i] = make_double2(w[i].x * a, w[i].y * a);
}

void launch_scale(int64_t n, const double2* w, const double* s, double2* out, cudaStream_t st) {
  HZ_COUNT();
  k_scale<<<grid_for(n, 256), 256, 0, st>>>(n, w, s, out);
}

__global__ void k_gemv_add(int64_t n, int k, const double2* y, const double2* Zs, int64_t ldz, double2* x) {
  __shared__ double2 ys[kMaxCols];
  for (int j = threadIdx.x; j < k; j += blockDim.x) ys[j] = y[j];
  __syncthreads();
  for (int64_t r = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; r < n; r += int64_t(gridDim.x) * blockDim.x) {
    double2 acc = x[r];
    for (int j = 0; j < k; j++) acc = cmad(Zs[r + int64_t(j) * ldz], ys[j], acc);
    x[r] = acc;
  }
}

// x += Zs[:, 0:k) y (k <= 64)
void launch_gemv_add(int64_t n, int k, const double2* y, const double2* Zs, int64_t ldz, double2* x, cudaStream_t st) {
  HZ_COUNT();
  k_gemv_add<<<grid_for(n, 256), 256, 0, st>>>(n, k, y, Zs, ldz, x);
}

__global__ void k_add2(int n, const double2* a, const double2* b, double2* out) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) out[i] = cadd(a[i], b[i]);
}

void launch_add2(int n, const double2* a, const double2* b, double2* out, cudaStream_t st) {
  HZ_COUNT();
  k_add2<<<1, 64, 0, st>>>(n, a, b, out);
}

__global__ void k_copy(int64_t n, const double2* a, double2* out) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    out[i] = a[i];
}

void launch_axpby_copy(int64_t n, const double2* a, double2* out, cudaStream_t st) {
  HZ_COUNT();
  k_copy<<<grid_for(n, 256), 256, 0, st>>>(n, a, out);
}

}  // namespace hz
