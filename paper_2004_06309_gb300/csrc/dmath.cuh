// Device helpers shared by the kernel files: complex arithmetic, programmatic dependent
// launch, asynchronous copies, and the last-block finish of the backward sweeps.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdlib>

#include "dev.h"

namespace hz {

// ---------------------------------------------------------------------------
// complex helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ float xfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double xfma(double a, double b, double c) { return __fma_rn(a, b, c); }

template <typename V> struct RealOf;
template <> struct RealOf<float2> { using T = float; };
template <> struct RealOf<double2> { using T = double; };

// 2^e, |e| <= 1000
__device__ __forceinline__ double exp2i(int e) { return __hiloint2double((e + 1023) << 20, 0); }

template <typename V>
__device__ __forceinline__ V mk(typename RealOf<V>::T x, typename RealOf<V>::T y) {
  V v;
  v.x = x;
  v.y = y;
  return v;
}
template <typename V> __device__ __forceinline__ V czero() { return mk<V>(0, 0); }
template <typename V> __device__ __forceinline__ V cadd(V a, V b) { return mk<V>(a.x + b.x, a.y + b.y); }
template <typename V> __device__ __forceinline__ V csub(V a, V b) { return mk<V>(a.x - b.x, a.y - b.y); }
template <typename V> __device__ __forceinline__ V cneg(V a) { return mk<V>(-a.x, -a.y); }
template <typename V> __device__ __forceinline__ V cmul(V a, V b) {
  return mk<V>(xfma(a.x, b.x, -a.y * b.y), xfma(a.x, b.y, a.y * b.x));
}
// c + a b
template <typename V> __device__ __forceinline__ V cmad(V a, V b, V c) {
  c.x = xfma(a.x, b.x, c.x);
  c.x = xfma(-a.y, b.y, c.x);
  c.y = xfma(a.x, b.y, c.y);
  c.y = xfma(a.y, b.x, c.y);
  return c;
}
// c - a b
template <typename V> __device__ __forceinline__ V cmsub(V a, V b, V c) {
  c.x = xfma(-a.x, b.x, c.x);
  c.x = xfma(a.y, b.y, c.x);
  c.y = xfma(-a.x, b.y, c.y);
  c.y = xfma(-a.y, b.x, c.y);
  return c;
}
// c + conj(a) b
template <typename V> __device__ __forceinline__ V cmadc(V a, V b, V c) {
  c.x = xfma(a.x, b.x, c.x);
  c.x = xfma(a.y, b.y, c.x);
  c.y = xfma(a.x, b.y, c.y);
  c.y = xfma(-a.y, b.x, c.y);
  return c;
}
template <typename V> __device__ __forceinline__ V cinv(V a) {
  const typename RealOf<V>::T d = a.x * a.x + a.y * a.y;
  return mk<V>(a.x / d, -a.y / d);
}
template <typename V> __device__ __forceinline__ V from2(double2 a);
template <> __device__ __forceinline__ double2 from2<double2>(double2 a) { return a; }
template <> __device__ __forceinline__ float2 from2<float2>(double2 a) { return make_float2(float(a.x), float(a.y)); }
__device__ __forceinline__ double2 to2(double2 a) { return a; }
__device__ __forceinline__ double2 to2(float2 a) { return make_double2(a.x, a.y); }

template <typename V> __device__ __forceinline__ V shfl_xor(V v, int m, int w = 32) {
  v.x = __shfl_xor_sync(0xffffffffu, v.x, m, w);
  v.y = __shfl_xor_sync(0xffffffffu, v.y, m, w);
  return v;
}
template <typename V> __device__ __forceinline__ V warp_sum(V v) {
  for (int o = 16; o > 0; o >>= 1) v = cadd(v, shfl_xor(v, o));
  return v;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return uint32_t(__cvta_generic_to_shared(p)); }
// Programmatic dependent launch (the triangular sweeps, one launch per tree level): a level's
// kernel lets the next level's grid start as soon as all of its CTAs are running
// (launch_dependents), and the next level reads nothing of the previous levels' results
// before griddepcontrol.wait, which returns once the previous grid has completed and its
// writes are visible.  Loads issued before the wait touch only the factor panels and the
// task descriptors, which no sweep writes.  Without the launch attribute both are no-ops.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
// 16-byte asynchronous copy global -> shared (L2 only), and the wait for all of a thread's copies
__device__ __forceinline__ void cp_async16(void* sdst, const void* gsrc) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(sdst)), "l"(gsrc) : "memory");
}
// 8 bytes, or zeros if !in (gsrc is not read then)
__device__ __forceinline__ void cp_async8(void* sdst, const void* gsrc, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(smem_addr(sdst)), "l"(gsrc), "r"(in ? 8 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// returns when at most N of the thread's committed groups are still in flight
template <int N> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// Loads of solve vectors (t, u, z, x) bypass L1 (ld.global.cg): each value is read
// once per sweep, so caching it in L1 only evicts panel lines.
template <typename V> __device__ __forceinline__ V ldv(const V* p);
template <> __device__ __forceinline__ float2 ldv<float2>(const float2* p) { return __ldcg(p); }
template <> __device__ __forceinline__ double2 ldv<double2>(const double2* p) { return __ldcg(p); }

// ---------------------------------------------------------------------------
// batched sweeps: S right-hand sides per row, moved 16 bytes at a time (one complex128 or two
// complex64 values), 256 threads.  A row's child contributions are adjacent (cptr); the loads of U
// rows, their row pointers, and of each row's first two contributions (a nested-dissection
// supernode has at most two children) are issued together: one after the other, these chains
// held the forward tasks (22 us each at k = 128, S = 16 in complex64, of which 20 were this).
// ---------------------------------------------------------------------------
template <typename V> struct Vec16;
template <> struct Vec16<float2> { using T = float4; };
template <> struct Vec16<double2> { using T = double2; };
__device__ __forceinline__ float4 vadd(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ double2 vadd(double2 a, double2 b) { return cadd(a, b); }
__device__ __forceinline__ float4 vsub(float4 a, float4 b) { return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w); }
__device__ __forceinline__ double2 vsub(double2 a, double2 b) { return csub(a, b); }
template <typename T> __device__ __forceinline__ T vzero();
template <> __device__ __forceinline__ float4 vzero<float4>() { return make_float4(0.f, 0.f, 0.f, 0.f); }
template <> __device__ __forceinline__ double2 vzero<double2>() { return make_double2(0.0, 0.0); }

// a[q] + the contributions c0[q] .. c1[q] - 1 of U rows, lane i of LR per row
template <typename V, int LR, int U, typename T>
__device__ __forceinline__ void add_contributions(T* a, const uint32_t* c0, const uint32_t* c1, const V* u, int i) {
  const T* u16 = reinterpret_cast<const T*>(u) + i;
  T v0[U], v1[U];
#pragma unroll
  for (int q = 0; q < U; q++) {
    v0[q] = c0[q] < c1[q] ? __ldcg(u16 + int64_t(c0[q]) * LR) : vzero<T>();
    v1[q] = c0[q] + 1 < c1[q] ? __ldcg(u16 + int64_t(c0[q] + 1) * LR) : vzero<T>();
  }
#pragma unroll
  for (int q = 0; q < U; q++) {
    a[q] = vadd(vadd(a[q], v0[q]), v1[q]);
    for (uint32_t c = c0[q] + 2; c < c1[q]; c++) a[q] = vadd(a[q], __ldcg(u16 + int64_t(c) * LR));
  }
}

// dst[j] = tin[j] + contributions of row j, j < k
template <typename V, int S>
__device__ __forceinline__ void gather_rows(V* dst, const V* tin, const uint32_t* cp, const V* u, int k) {
  using T = typename Vec16<V>::T;
  constexpr int LR = S * int(sizeof(V)) / 16, RP = 256 / LR, U = 4;
  const int i = threadIdx.x % LR;
  const T* t16 = reinterpret_cast<const T*>(tin) + i;
  for (int j0 = threadIdx.x / LR; j0 < k; j0 += U * RP) {
    uint32_t c0[U], c1[U];
    T a[U];
#pragma unroll
    for (int q = 0; q < U; q++) {
      const int j = j0 + q * RP;
      c0[q] = j < k ? cp[j] : 0u;
      c1[q] = j < k ? cp[j + 1] : 0u;
      a[q] = j < k ? __ldcg(t16 + int64_t(j) * LR) : vzero<T>();
    }
    add_contributions<V, LR, U>(a, c0, c1, u, i);
#pragma unroll
    for (int q = 0; q < U; q++)
      if (j0 + q * RP < k) reinterpret_cast<T*>(dst)[(j0 + q * RP) * LR + i] = a[q];
  }
}

// A forward task's update rows: their contributions and where they go, N 16-byte items per thread
// (rows row0 + item / LR of RT), loaded before the task's products.
template <typename V, int S, int RT> struct UpdateRows {
  using T = typename Vec16<V>::T;
  static constexpr int LR = S * int(sizeof(V)) / 16, N = (RT * LR + 255) / 256;
  T b2[N];
  uint32_t to[N];
  __device__ __forceinline__ void load(const SnDev& Sn, const uint32_t* cp, const uint32_t* wpos, const V* u, int row0) {
    uint32_t c0[N], c1[N];
#pragma unroll
    for (int q = 0; q < N; q++) {
      const int e = threadIdx.x + 256 * q, r = row0 + e / LR;
      const bool ok = e < RT * LR && r >= Sn.k && r < Sn.m;
      c0[q] = ok ? cp[r] : 0u;
      c1[q] = ok ? cp[r + 1] : 0u;
      to[q] = ok ? wpos[Sn.rowoff + r] : 0u;
      b2[q] = vzero<T>();
    }
    add_contributions<V, LR, N>(b2, c0, c1, u + Sn.ubase * S, threadIdx.x % LR);
  }
};

// Fused second stage of the backward sweep ("last block done"), for a (supernode,
// column block) split over several row chunks: every partial-sum CTA of the pair
// publishes its 32 sums, fences, and bumps the pair's counter; the CTA that brings it
// to `chunks` adds the partials in chunk order (deterministic), writes x, and resets
// the counter for the next sweep.  No CTA ever waits on another.  (The single-chunk
// case finishes inside its own CTA and never touches the counter.)
template <typename V>
__device__ __forceinline__ void bwd_finish(const int4 fin, const SnDev& S, const V* zin, const V* partial_level,
                                           V* x, unsigned int* counter) {
  __shared__ unsigned int ticket;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) ticket = atomicAdd(counter, 1u);
  __syncthreads();
  if (ticket != unsigned(fin.w) - 1) return;
  __threadfence();
  const int c = threadIdx.x;
  if (c < 32) {
    const int j = fin.y * 32 + c;
    if (j < S.k) {
      V acc = czero<V>();
      for (int ch = 0; ch < fin.w; ch++) {
        const V* pp = partial_level + int64_t(fin.z + ch) * 32 + c;
        V v;
        if constexpr (sizeof(V) == 8) {
          const float2 t = __ldcg(reinterpret_cast<const float2*>(pp));
          v.x = t.x; v.y = t.y;
        } else {
          const double2 t = __ldcg(reinterpret_cast<const double2*>(pp));
          v.x = t.x; v.y = t.y;
        }
        acc = cadd(acc, v);
      }
      x[S.first + j] = cadd(zin[S.first + j], acc);
    }
    if (c == 0) *counter = 0u;
  }
}

// One tree level of a sweep, launched with programmatic stream serialisation (unless HZ_NO_PDL
// is set), so that a level's CTAs start their panel loads while the previous level's grid
// drains; the kernels wait (pdl_wait) before they read any result of that level.
inline bool pdl_enabled() {
  static const bool on = std::getenv("HZ_NO_PDL") == nullptr;
  return on;
}
template <typename... KArgs, typename... Args>
void launch_level(void (*kern)(KArgs...), int64_t grid, int threads, size_t smem, cudaStream_t st, bool pdl,
                  Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(grid));
  cfg.blockDim = dim3(unsigned(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

}  // namespace hz
