// Device helpers shared by the fused stage kernel (stage.cu) and the adjoint stage kernel
// (adjoint_kernels.cuh).
#pragma once

#include <atomic>

#include "common.cuh"
#include "kernels.hpp"

namespace acm {
namespace {

// Opt `kernel` in to `bytes` of dynamic shared memory (above the default 48 KB) on the current
// device, once per device (the attribute belongs to the device's context).
template <typename K>
void smem_opt_in_stage(K kernel, size_t bytes, std::atomic<unsigned long long>& done) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  const unsigned long long bit = 1ull << dev;
  if (done.load(std::memory_order_relaxed) & bit) return;
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  done.fetch_or(bit);
}

template <typename T>
__device__ __forceinline__ void cp_async_elem(T* dst, const T* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (sizeof(T) == 4) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
  } else {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
  }
}
__device__ __forceinline__ void cp_async_16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
template <typename T>
__device__ __forceinline__ T tmax(T a, T b) { return a > b ? a : b; }

// Pairs of values: FP32 pairs take the packed FP32x2 instructions, FP64 pairs go component by
// component.  Every operation rounds each component once, to nearest.
__host__ __device__ __forceinline__ float2 vset(float v) { return make_float2(v, v); }
__host__ __device__ __forceinline__ double2 vset(double v) { return make_double2(v, v); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) {
  union P { float2 f; unsigned long long u; } x, y, r;
  x.f = a;
  y.f = b;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(x.u), "l"(y.u));
  return r.f;
}
__device__ __forceinline__ double2 vadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 vmul(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ double2 vfma(double2 a, double2 b, double2 c) {
  return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
__device__ __forceinline__ double2 vsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

// h / a_1 times the first difference of a pair from its neighbours at distance 1, 2, 3 (Sec. 2.3).
template <typename K, typename V>
__device__ __forceinline__ V d1_pair(const K& kc, V m1, V p1, V m2, V p2, V m3, V p3) {
  return vfma(kc.r3, vsub(p3, m3), vfma(kc.r2, vsub(p2, m2), vsub(p1, m1)));
}
// -12 h^2 times the second difference (Sec. 2.3): p2 + m2 - 16 (p1 + m1) + 30 c.
template <typename K, typename V>
__device__ __forceinline__ V d2_pair(const K& kc, V c, V m1, V p1, V m2, V p2) {
  return vfma(kc.k30, c, vfma(kc.km16, vadd(p1, m1), vadd(p2, m2)));
}
// The same of a pair's first component.
__device__ __forceinline__ float d2_first(float2 c, float2 m1, float2 p1, float2 m2, float2 p2) {
  return fmaf(30.f, c.x, fmaf(-16.f, p1.x + m1.x, p2.x + m2.x));
}
__device__ __forceinline__ double d2_first(double2 c, double2 m1, double2 p1, double2 m2, double2 p2) {
  return fma(30.0, c.x, fma(-16.0, p1.x + m1.x, p2.x + m2.x));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_inval(unsigned long long* bar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
// orders this thread's earlier shared-memory accesses (and those a barrier published to it) before
// later bulk copies into the same memory
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
// global -> shared bulk copy of `bytes` (both addresses 16-byte aligned, bytes a multiple of 16)
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
               ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
// Waits for the phase of the given parity; after a bounded number of polls (each may suspend the
// thread for a while) it sets *err |= 1 (a bounded wait expired) and goes on.
__device__ __forceinline__ void mbar_wait(unsigned long long* bar, unsigned parity, int* err) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .u32 n;\n mov.u32 n, 0;\n"
      "W%=:\n mbarrier.try_wait.parity.shared::cta.b64 p, [%0], %1;\n @p bra D%=;\n"
      " add.u32 n, n, 1;\n setp.lt.u32 p, n, 4194304;\n @p bra W%=;\n red.global.or.b32 [%2], 1;\n"
      "D%=:\n}\n" ::"r"(smem_u32(bar)), "r"(parity), "l"(err)
      : "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait_group() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Address of one halo value: face F, distance l = 1..3 from the face plane, tangential
// coordinates (t0, t1) = (y, z) for x-faces, (x, z) for y-faces, (x, y) for z-faces.
template <typename T, int BS>
__device__ __forceinline__ const T* halo_ptr(const int (&ftype)[6], const int (&fs)[6][4],
                                             const T* __restrict__ in, const T* __restrict__ slab,
                                             int F, int l, int t0, int t1, int f) {
  using L = Lay<T, BS>;
  constexpr int M = L::M;
  const int ax = F >> 1;
  const bool plus = F & 1;
  const int ty = ftype[F];
  int s, nl, u0 = t0, u1 = t1;
  if (ty == kTypeLeaf) {
    s = fs[F][0];
    nl = plus ? l : M - l;
  } else if (ty == kTypeRefined) {
    const int c0 = t0 > M / 2, c1 = t1 > M / 2;
    s = fs[F][c0 + 2 * c1];
    nl = plus ? 2 * l : M - 2 * l;
    u0 = 2 * t0 - c0 * M;
    u1 = 2 * t1 - c1 * M;
  } else {
    return slab + ((((size_t)fs[F][0] * 4 + f) * 3 + (l - 1)) * BS + t1) * BS + t0;
  }
  int x, y, z;
  if (ax == 0) { x = nl; y = u0; z = u1; }
  else if (ax == 1) { x = u0; y = nl; z = u1; }
  else { x = u0; y = u1; z = nl; }
  return in + (size_t)s * L::BLK + (size_t)f * L::FS + L::idx(x, y, z);
}


// Face table of one block from its face record (TopoK::faces): for each face F the type of the
// neighbour across it and the slots / slab index in fs[F][0..3].  Threads 0..29 fill it; the
// caller synchronises.
__device__ __forceinline__ void stage_faces(int tid, const int32_t* __restrict__ faces, int rank, int (&ftype)[6],
                                            int (&fs)[6][4]) {
  if (tid < 30) {
    const int v = faces[(size_t)rank * kFaceStride + tid];
    if (tid < 6) ftype[tid] = v;
    else (&fs[0][0])[tid - 6] = v;
  }
}

// Global lattice index of a block's point i along axis a; the periodic seam x = L is taken as 0.
__device__ __forceinline__ int lattice_index(const PhysK& ph, int4 bi, int a, int i, int M) {
  const int g = a == 0 ? bi.y : (a == 1 ? bi.z : bi.w);
  const int N = (ph.nroot[a] << bi.x) * M;
  const int gi = g * M + i;                               // in [0, N]
  return gi >= N ? gi - N : gi;
}

// Sponge profile of one block along each axis (Sec. 2.2, sponge terms; the profile's reading is
// the tanh of the distance to the nearest box face minus L_sp), in the field precision: threads
// 0..3 Bs - 1 fill sp[axis][i]; the caller synchronises.
template <typename T, int BS>
__device__ __forceinline__ void stage_sponge(int tid, const PhysK& ph, int4 bi, T (&sp)[3][BS]) {
  constexpr int M = BS - 1;
  if (ph.sponge && tid < 3 * BS) {
    const double h = ph.h[bi.x];
    const int ax = tid / BS, i = tid % BS;
    const int g = ax == 0 ? bi.y : (ax == 1 ? bi.z : bi.w);
    const long long N = ((long long)ph.nroot[ax] << bi.x) * M;
    long long gi = (long long)g * M + i;        // in [0, N]; the seam x = L is taken as 0
    if (gi >= N) gi -= N;
    const double c = (double)gi * h;
    // the profile in the field precision (FP32 fields keep tanh off the FP64 pipe)
    const T dist = T(fmin(c, ph.sp_L[ax] - c));
    sp[ax][i] = T(0.5) * (T(1) - ttanh((dist - T(ph.sp_width)) / T(ph.sp_delta)));
  }
}

}  // namespace
}  // namespace acm
