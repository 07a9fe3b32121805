// Fused right-hand side + RK4 stage kernel of libacm (the hot path).
//
// One CTA updates one block.  Paper, eqs. (u_eqn-1, p_eqn-1):
//   du/dt = -(u.grad)u - grad p + nu lap u - chi/C_eta (u - u_s) - chi_sp/C_sp (u - u_inf)
//   dp/dt = -C_0^2 div u - C_gamma p - chi_sp/C_sp (p - p_inf)
// with the Tam-Webb (or classical) 4th-order first derivative and the classical 4th-order
// second derivative (Sec. 2.3; u_s = 0 unless the body moves), and one stage of classical RK4
// (Sec. 2.3), U = U^n, K_s the right-hand side of stage s:
//   stage 1: Y_2 = U + dt/2 K_1        stage 2: Y_3 = U + dt/2 K_2       stage 3: Y_4 = U + dt K_3
//   stage 4: U^{n+1} = U + [(Y_2 - U) + 2 (Y_3 - U) + (Y_4 - U)] / 3 + dt/6 K_4
//   stage 0 (checks only): out = K
// The last line is U + dt/6 (K_1 + 2 K_2 + 2 K_3 + K_4) with the first three K's taken from the
// stage states, so no accumulator is kept: 13 words per point and component group instead of 16.
// Points that fine wins overwrites in the stage states (on a boundary shared with a finer leaf)
// keep an accumulator, acc = U + dt/6 K_1 + dt/3 K_2 + dt/3 K_3, and take U^{n+1} = acc + dt/6 K_4;
// which points these are depends on the physical point alone, so all copies of a point take the
// same form.
//
// Work layout: a thread owns one (x, y) pencil of the block and marches in z (a block of up to
// 17^3 points is one CTA; a 33^3 block is split by rows over five CTAs, which read the rows
// next to their own from the block like a halo).  The four components of a point travel
// together: the z-stencil (7 points) lives in a register ring of component pairs (u, v), (w, p),
// and the x/y stencils read a shared-memory plane of four-component points with a 3-point halo on
// each side.  A neighbour is then one 16-byte shared load instead of four, and FP32 differences
// run on pairs (add/mul/fma.f32x2).  The ring is indexed by the plane modulo 7 in a loop unrolled
// by 7, so no register moves.  The block's own planes are brought into shared memory by bulk copies
// that one further warp issues, up to three planes ahead, and the x/y halo points by cp.async two
// planes ahead, straight from the neighbour's stored interior (same level: copy; finer: decimation, Sec. 3.1
// restriction) or, across a face to a coarser neighbour, from the halo slab that the coarse-face
// kernel predicted for this stage.  No ghost layer is written to HBM.
//
// What bounds it: the L1 data pipe's wavefronts (68, 55, 55 and 51 % of the cycles in stages 1 to 4 on 4608
// FP32 blocks; 60, 48, 48 and 45 % are shared-memory ones), latency at two CTAs per SM and the prologue of
// a CTA (halo table, first planes), then HBM (1.10 times the algorithmic bytes); FP64: the FP64 pipe.  Measured per launch (mean over the four
// stages), against one point per thread with a point's components apart and the accumulator kept:
// 4608 blocks of 17^3 FP32 0.393 ms (0.434 before); 32768 blocks 2.42 (2.79); 64 blocks 0.0192 (0.0297);
// 33^3 moving plate 1.57 (2.23, its solid-velocity kernel included); FP64 4096 blocks 2.37 (2.63).  Slower
// with the same arithmetic: components apart in the stage states 0.448, 3 CTAs per SM at 64 registers
// (spills) 0.60, two threads per point 0.50, two rows per thread 0.60, all halos by the loading warp 0.44.
#include <algorithm>
#include <type_traits>

#include "stage_common.cuh"
#include "stage_parts.hpp"

namespace acm {

namespace {

template <typename T, int BS>
struct Cfg {
  static constexpr int NS = BS <= 17 ? 1 : 5;      // CTAs per block
  static constexpr int RY = (BS + NS - 1) / NS;    // most rows (y) of a CTA
  // computing threads; one more warp loads.  The 289th pencil of a 17^3 block would take a warp of
  // its own: the loading warp computes it at its end, a lane per plane.
  static constexpr int CORNER = BS == 17 ? 1 : 0;
  static constexpr int NT = ((BS * RY - CORNER + 31) / 32) * 32;
  static constexpr int H = RY + 6;       // plane rows: 3 halo rows each side
  // row stride in points: congruent to BS modulo 8, so that the pencils of a quarter warp that
  // continue on the next row continue on the next 16-byte banks (no bank conflicts)
  static constexpr int W = BS + 8;
  static constexpr int PW = H * W;
  // x/y halo points per plane: x faces 2 x 3 x RY, y faces 2 x 3 x BS
  // (and the corner pencil's point, which no computing thread holds)
  static constexpr int NX = 6 * (RY + BS);
  static constexpr int NH = NX + CORNER;
  static constexpr int HPT = (NH + NT - 1) / NT;
  static constexpr int MINB = sizeof(T) == 4 ? (NT <= 160 ? 4 : 2) : 1;   // CTAs per SM
  static_assert(NS == 1 || sizeof(T) == 4, "row-split blocks are FP32 only");
  static_assert(PW < 0x8000, "plane buffer offsets must fit 15 bits");
  static_assert(parts_are_sound(BS), "the upper halo planes arrive before they are read, for every part");
};

// Shared planes.  FP32: a point's (u, v, w, p) is one float4.  FP64: (u, v) and (w, p) in two
// arrays of double2 (16 bytes per lane either way).
template <typename T, int PW>
struct Plane;
template <int PW>
struct Plane<float, PW> {
  float4 c[PW];
  __device__ __forceinline__ void put(int i, float2 a, float2 b) { c[i] = make_float4(a.x, a.y, b.x, b.y); }
  __device__ __forceinline__ void get(int i, float2& a, float2& b) const {
    const float4 v = c[i];
    a = make_float2(v.x, v.y);
    b = make_float2(v.z, v.w);
  }
  __device__ __forceinline__ float* comp(int i, int f) { return reinterpret_cast<float*>(c + i) + f; }
  __device__ __forceinline__ void copy_point(int i, const float* src) { cp_async_16(c + i, src); }
};
template <int PW>
struct Plane<double, PW> {
  double2 a[PW], b[PW];
  __device__ __forceinline__ void put(int i, double2 va, double2 vb) { a[i] = va; b[i] = vb; }
  __device__ __forceinline__ void get(int i, double2& va, double2& vb) const { va = a[i]; vb = b[i]; }
  __device__ __forceinline__ double* comp(int i, int f) {
    return reinterpret_cast<double*>((f & 2) ? b + i : a + i) + (f & 1);
  }
  __device__ __forceinline__ void copy_point(int i, const double* src) {
    cp_async_16(a + i, src);
    cp_async_16(b + i, src + 2);
  }
};

// Addressing of a register in the component-major layout (the state U) and in the point-major one
// (A: the stage states Y_2 .. Y_4 and the accumulator inside a step): element offset of a point's
// component 0 in its block, strides of components, planes and halo-slab components.  Four components
// side by side make every access of a point one 16-byte instruction and a halo row whole sectors.
template <typename T, int BS, bool A>
struct At {
  using L = Lay<T, BS>;
  static constexpr int CS = A ? 1 : L::FS, PT = A ? 4 : 1, PL = A ? 4 * BS * BS : L::PP;
  static constexpr int SCS = A ? 1 : 3 * BS * BS;           // slab: components
  static constexpr int SLS = BS * BS * PT;                   // slab: layers
  __device__ __forceinline__ static constexpr int idx(int x, int y, int z) { return z * PL + (y * BS + x) * PT; }
  __device__ __forceinline__ static size_t slab(int s, int l, int t0, int t1) {   // layer l = 1..3
    return A ? (((size_t)s * 3 + (l - 1)) * BS * BS + t1 * BS + t0) * 4
             : ((size_t)s * 12 + (l - 1)) * BS * BS + t1 * BS + t0;
  }
  static_assert(4 * BS * BS * BS <= L::BLK, "the point-major form fits the block stride");
};
template <bool A>
__device__ __forceinline__ void load_point(const float* p, int cs, float2& a, float2& b) {
  if (A) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    a = make_float2(v.x, v.y);
    b = make_float2(v.z, v.w);
  } else {
    a = make_float2(p[0], p[cs]);
    b = make_float2(p[2 * cs], p[3 * cs]);
  }
}
template <bool A>
__device__ __forceinline__ void load_point(const double* p, int cs, double2& a, double2& b) {
  if (A) {
    a = reinterpret_cast<const double2*>(p)[0];
    b = reinterpret_cast<const double2*>(p)[1];
  } else {
    a = make_double2(p[0], p[cs]);
    b = make_double2(p[2 * cs], p[3 * cs]);
  }
}
template <bool A>
__device__ __forceinline__ void store_point(float* p, int cs, const float (&v)[4]) {
  if (A) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int f = 0; f < 4; ++f) p[f * cs] = v[f];
  }
}
template <bool A>
__device__ __forceinline__ void store_point(double* p, int cs, const double (&v)[4]) {
  if (A) {
    reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
  } else {
#pragma unroll
    for (int f = 0; f < 4; ++f) p[f * cs] = v[f];
  }
}

// Planes of the block's own points staged in shared memory for an iteration z: the input's plane
// z + 3, and of plane z U (stages 2 to 4), Y_2 and Y_3 (stage 4), and chi.
template <int STAGE>
__host__ __device__ constexpr int staged_arrays(bool mask) {
  return 4 + (STAGE == 2 || STAGE == 3 ? 4 : (STAGE == 4 ? 12 : 0)) + (mask ? 1 : 0);
}
constexpr int kNB = 4;     // plane buffers
constexpr int kND = 3;     // iterations whose data may be in flight
// Elements of one staged plane: a CTA's rows, widened to 16-byte boundaries.
template <typename T, int BS>
__host__ __device__ constexpr int staged_pitch() {
  using L = Lay<T, BS>;
  return Cfg<T, BS>::NS == 1 ? L::PP : ((BS * Cfg<T, BS>::RY + 3 * (L::VEC - 1)) / L::VEC) * L::VEC;
}
template <typename T, int BS, int STAGE>
constexpr size_t stage_smem(bool mask) {
  return kNB * sizeof(Plane<T, Cfg<T, BS>::PW>) +
         (size_t)(kND * staged_arrays<STAGE>(mask) + 12) * staged_pitch<T, BS>() * sizeof(T);
}

// Right-hand side K of one point (components u, v, w, p) whose pair values are ca = (u, v), cb =
// (w, p); get(axis, k, a, b) gives the neighbour's pairs at distance k along the axis (0 x, 1 y,
// 2 z), chi() the mask, solid(us) a moving body's velocity, chi_sp() the sponge profile.  The spacing factors are
// applied once per term (1/h, nu/(12 h^2), C_0^2/h), not to every difference.
template <typename T, typename V, typename G, typename CM, typename US, typename CS>
__device__ __forceinline__ void point_rhs(const StageConst<T>& kc, int mask, int sponge, const T* cst, V ca, V cb,
                                          G&& get, CM&& chi, US&& solid, CS&& chi_sp, T (&K)[4]) {
  const T u = ca.x, v = ca.y, w = cb.x, p = cb.y;
  T K0, K1, K2, div, lapw;
  V lap;
  {
    V m1a, m1b, p1a, p1b, m2a, m2b, p2a, p2b, m3a, m3b, p3a, p3b;
    get(0, -1, m1a, m1b); get(0, 1, p1a, p1b);
    get(0, -2, m2a, m2b); get(0, 2, p2a, p2b);
    get(0, -3, m3a, m3b); get(0, 3, p3a, p3b);
    const V d = d1_pair(kc, m1a, p1a, m2a, p2a, m3a, p3a);
    const V e = d1_pair(kc, m1b, p1b, m2b, p2b, m3b, p3b);
    lap = d2_pair(kc, ca, m1a, p1a, m2a, p2a);
    lapw = d2_first(cb, m1b, p1b, m2b, p2b);
    K0 = fma(u, d.x, e.y);
    K1 = u * d.y;
    K2 = u * e.x;
    div = d.x;
  }
  {
    V m1a, m1b, p1a, p1b, m2a, m2b, p2a, p2b, m3a, m3b, p3a, p3b;
    get(1, -1, m1a, m1b); get(1, 1, p1a, p1b);
    get(1, -2, m2a, m2b); get(1, 2, p2a, p2b);
    get(1, -3, m3a, m3b); get(1, 3, p3a, p3b);
    const V d = d1_pair(kc, m1a, p1a, m2a, p2a, m3a, p3a);
    const V e = d1_pair(kc, m1b, p1b, m2b, p2b, m3b, p3b);
    lap = vadd(lap, d2_pair(kc, ca, m1a, p1a, m2a, p2a));
    lapw += d2_first(cb, m1b, p1b, m2b, p2b);
    K0 = fma(v, d.x, K0);
    K1 = fma(v, d.y, K1) + e.y;
    K2 = fma(v, e.x, K2);
    div += d.y;
  }
  {
    V m1a, m1b, p1a, p1b, m2a, m2b, p2a, p2b, m3a, m3b, p3a, p3b;
    get(2, -1, m1a, m1b); get(2, 1, p1a, p1b);
    get(2, -2, m2a, m2b); get(2, 2, p2a, p2b);
    get(2, -3, m3a, m3b); get(2, 3, p3a, p3b);
    const V d = d1_pair(kc, m1a, p1a, m2a, p2a, m3a, p3a);
    const V e = d1_pair(kc, m1b, p1b, m2b, p2b, m3b, p3b);
    lap = vadd(lap, d2_pair(kc, ca, m1a, p1a, m2a, p2a));
    lapw += d2_first(cb, m1b, p1b, m2b, p2b);
    K0 = fma(w, d.x, K0);
    K1 = fma(w, d.y, K1);
    K2 = fma(w, e.x, K2) + e.y;
    div += e.x;
  }
  const T ih = cst[0], nu_ih2 = cst[1], c0sq_ih = cst[2];
  K[0] = fma(-ih, K0, -nu_ih2 * lap.x);
  K[1] = fma(-ih, K1, -nu_ih2 * lap.y);
  K[2] = fma(-ih, K2, -nu_ih2 * lapw);
  K[3] = fma(-c0sq_ih, div, -kc.cgam * p);
  if (mask) {
    const T cm = chi() * kc.inv_ceta;
    T us[3] = {T(0), T(0), T(0)};
    if (kc.moving) solid(us);
    K[0] = fma(-cm, u - us[0], K[0]);
    K[1] = fma(-cm, v - us[1], K[1]);
    K[2] = fma(-cm, w - us[2], K[2]);
  }
  if (sponge) {
    const T cs = chi_sp() * kc.inv_csp;
    K[0] = fma(-cs, u - kc.uinf[0], K[0]);
    K[1] = fma(-cs, v - kc.uinf[1], K[1]);
    K[2] = fma(-cs, w - kc.uinf[2], K[2]);
    K[3] = fma(-cs, p - kc.pinf, K[3]);
  }
}

// The RK4 combination of a point (see the head of the file): c the stage state's components, U(f),
// y2(f), y3(f) the other values read; at points fine wins overwrites (keep) the accumulator at offset
// oa (component stride cs) is read and written.
template <typename T, bool A, int STAGE, typename FU, typename F2, typename F3>
__device__ __forceinline__ void rk_combine(const StagePtrs<T>& a, size_t oa, int cs, const T (&c)[4], const T (&K)[4],
                                           FU&& U, F2&& y2, F3&& y3, T c_acc, T c_out, bool keep, T (&nv)[4]) {
  using V = typename StageVec<T>::type;
  if (STAGE == 0) {
#pragma unroll
    for (int f = 0; f < 4; ++f) nv[f] = K[f];
  } else if (STAGE == 1) {
#pragma unroll
    for (int f = 0; f < 4; ++f) nv[f] = fma(c_out, K[f], c[f]);
    if (keep) {
      T acc[4];
#pragma unroll
      for (int f = 0; f < 4; ++f) acc[f] = fma(c_acc, K[f], c[f]);
      store_point<A>(a.acc_out + oa, cs, acc);
    }
  } else if (STAGE == 4) {
    if (keep) {
      V aa, ab;
      load_point<A>(a.acc_in + oa, cs, aa, ab);
      nv[0] = fma(c_out, K[0], aa.x);
      nv[1] = fma(c_out, K[1], aa.y);
      nv[2] = fma(c_out, K[2], ab.x);
      nv[3] = fma(c_out, K[3], ab.y);
    } else {
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const T u = U(f);
        const T t = fma(T(2), y3(f) - u, y2(f) - u) + (c[f] - u);
        nv[f] = u + fma(c_out, K[f], t * (T(1) / T(3)));
      }
    }
  } else {
#pragma unroll
    for (int f = 0; f < 4; ++f) nv[f] = fma(c_out, K[f], U(f));
    if (keep) {
      V aa, ab;
      load_point<A>(a.acc_in + oa, cs, aa, ab);
      const T acc[4] = {fma(c_acc, K[0], aa.x), fma(c_acc, K[1], aa.y), fma(c_acc, K[2], ab.x), fma(c_acc, K[3], ab.y)};
      store_point<A>(a.acc_out + oa, cs, acc);
    }
  }
}

// Which planes of pencil (x, y) hold points that fine wins overwrites, from the block's mask of
// refined neighbour boxes: bit 0 all planes, bit 1 plane 0, bit 2 plane M.
template <int M>
__device__ __forceinline__ int fine_win_bits(unsigned m, int x, int y) {
  const int cx = x == 0 ? -1 : (x == M ? 1 : 0), cy = y == 0 ? -1 : (y == M ? 1 : 0);
  const unsigned t = (1u << 4) | (1u << (4 + cx)) | (1u << (4 + 3 * cy)) | (1u << (4 + cx + 3 * cy));
  return (((m >> 9) & t) ? 1 : 0) | ((m & t) ? 2 : 0) | (((m >> 18) & t) ? 4 : 0);
}

// The update of one block (rank `rank` of the topology tp), rows of y part `part` and planes za .. ze - 1
// of it; a: the arrays, kc: the constants.
// MULTI: called again by the same CTA afterwards (the mbarriers are given back at the end).
// PM: the stage states and the accumulator are point-major (see At); U is component-major.
template <typename T, int BS, int STAGE, bool PM, bool MULTI, bool SPLIT>
__device__ __forceinline__ void stage_block(const StagePtrs<T>& a, const StageConst<T>& kc, const TopoK& tp,
                                            const PhysK& ph, int* err, const int rank, const int part,
                                            const int za, const int ze) {
  // (planes 0 .. M, known to the compiler, unless the block is split along z)
  const int z0 = SPLIT ? za : 0, z1 = SPLIT ? ze : BS;
  using L = Lay<T, BS>;
  using C = Cfg<T, BS>;
  using V = typename StageVec<T>::type;
  constexpr int M = L::M, NT = C::NT, RY = C::RY, W = C::W, PW = C::PW, NH = C::NH;
  constexpr bool AI = PM && STAGE >= 2, AO = PM && STAGE >= 1 && STAGE <= 3;   // input, output point-major
  using I = At<T, BS, AI>;
  using O = At<T, BS, AO>;
  using Y = At<T, BS, PM>;               // the accumulator, Y_2 and Y_3

  extern __shared__ __align__(16) unsigned char dsm[];
  Plane<T, PW>* buf = reinterpret_cast<Plane<T, PW>*>(dsm);   // [kNB]
  constexpr int SP = staged_pitch<T, BS>();
  T* zup = reinterpret_cast<T*>(dsm + kNB * sizeof(Plane<T, PW>));   // [3][4][SP]: planes M + 1 .. M + 3
  T* stg = zup + 12 * SP;                                            // [kND][nst][SP]
  __shared__ __align__(8) unsigned long long full[kND];
  __shared__ int ftype[6];
  __shared__ int fs[6][4];
  __shared__ T sp[3][BS];
  // 1/h, nu/(12 h^2), C_0^2/h and the RK coefficients: read where they are used (registers are scarce)
  __shared__ __align__(16) T cst[8];
  // x/y halo points of every plane as affine functions of z (see below)
  __shared__ uint4 htab[NH];

  const int tid = threadIdx.x;
  const int slot = tp.blist[rank];
  const int4 bi = tp.binfo[rank];
  const unsigned fwm = (unsigned)tp.faces[(size_t)rank * kFaceStride + 30];

  if (tid == 0) {
    // iteration z starts when its staged planes have arrived (the announced bytes) and every computing
    // warp has put its part of plane z into its buffer
    for (int k = 0; k < kND; ++k) mbar_init(&full[k], 1 + NT / 32);
    mbar_init_fence();
  }
  stage_faces(tid, tp.faces, rank, ftype, fs);

  const int y0 = part * BS / C::NS, ny = (part + 1) * BS / C::NS - y0;   // this CTA's rows
  const bool act = tid < BS * ny - C::CORNER;
  const int x = act ? tid % BS : 0, y = y0 + (act ? tid / BS : 0);
  const size_t bo = (size_t)slot * L::BLK;
  const T* __restrict__ inb = a.in + bo;
  // register ring: plane zz of the pencil sits in entry (zz - z0 + 3) % 7 (planes z - 3 .. z + 3 of
  // iteration z; plane z + 3 enters at its start); the block's own planes are requested before the
  // first barrier, together with the face record
  V qa[7], qb[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) qa[k] = qb[k] = vset(T(0));
  if (act) {
#pragma unroll
    for (int k = SPLIT ? 0 : 3; k < 6; ++k) {
      const int zz = z0 + k - 3;
      if (!SPLIT || (zz >= 0 && zz <= M)) load_point<AI>(inb + I::idx(x, y, zz), I::CS, qa[k], qb[k]);
    }
  }
  stage_sponge<T, BS>(tid, ph, bi, sp);
  if (tid == NT) {
    cst[0] = kc.ih[bi.x];                  // a_1 / h: the first differences come divided by a_1
    cst[1] = kc.nu * kc.ih2[bi.x];
    cst[2] = kc.c0sq * kc.ih[bi.x];
    // RK coefficients: kernel parameters, or (steps with the time step on the device) the values
    // the time-step kernel left in device memory
    cst[3] = STAGE >= 1 && a.coefp ? T(a.coefp[2 * (STAGE - 1)]) : kc.c_acc;
    cst[4] = STAGE >= 1 && a.coefp ? T(a.coefp[2 * (STAGE - 1) + 1]) : kc.c_out;
  }
  __syncthreads();

  // The values of pencil (px, py) beyond the block's lower (F = 4) or upper (F = 5) z face: the
  // first layer's address, the layers' stride and the components' stride.
  auto z_face = [&](int F, int px, int py, const T*& p, int& ls, int& cs) {
    const int ty = ftype[F];
    const bool plus = F & 1;
    if (ty == kTypeLeaf) {
      p = a.in + (size_t)fs[F][0] * L::BLK + I::idx(px, py, plus ? 1 : M - 1);
      ls = plus ? I::PL : -I::PL;
      cs = I::CS;
    } else if (ty == kTypeRefined) {
      const int cx = px > M / 2, cy = py > M / 2;
      p = a.in + (size_t)fs[F][cx + 2 * cy] * L::BLK + I::idx(2 * px - cx * M, 2 * py - cy * M, plus ? 2 : M - 2);
      ls = plus ? 2 * I::PL : -2 * I::PL;
      cs = I::CS;
    } else {
      p = a.slab + I::slab(fs[F][0], 1, px, py);
      ls = I::SLS;
      cs = I::SCS;
    }
  };
  if (act) {
    if (!SPLIT || z0 < 3) {
      const T* p;
      int ls, cs;
      z_face(4, x, y, p, ls, cs);
#pragma unroll
      for (int k = 0; k < 3; ++k)         // plane z0 + k - 3, if below the block
        if (z0 + k < 3) load_point<AI>(p + (2 - k - z0) * ls, cs, qa[k], qb[k]);
    }
    if (SPLIT && z0 + 2 > M) {
      const T* p;
      int ls, cs;
      z_face(5, x, y, p, ls, cs);
#pragma unroll
      for (int k = 4; k < 6; ++k)         // plane z0 + k - 3, if above it
        if (z0 + k - 3 > M) load_point<AI>(p + (z0 + k - 4 - M) * ls, cs, qa[k], qb[k]);
    }
  }
  // x/y halo points of every plane as affine functions of z: component f of the point of plane z is
  // read at offset (z <= M/2 ? lo : hi) + z * hz + f * cs from the state (or from the slab buffer,
  // flag bit 15) and lands at point dst of the plane buffer: entry = (lo, hi, hz << 16 | slab << 15 |
  // dst, cs).  The offsets are element indices (32-bit: pool and slab sizes are checked at forest
  // creation); hi differs from lo for the upper child of a finer face.  A CTA holding part of the
  // rows reads the rows beyond its own from the block itself, and its x-face entries past its last
  // row are unused (hz = 0).
  for (int i = tid; i < NH; i += NT + 32) {
    int el = i, F, l, t;
    // x-faces take the 3 layers of a row as consecutive elements (one sector), y-faces a row
    if (el >= C::NX) {
      htab[i] = make_uint4((unsigned)(bo + I::idx(M, M, 0)), (unsigned)(bo + I::idx(M, M, 0)),
                           ((unsigned)I::PL << 16) | (unsigned)((M + 3) * W + M + 3), (unsigned)I::CS);
      continue;
    }
    if (el < 6 * RY) {
      F = el / (3 * RY);
      el %= 3 * RY;
      l = el % 3 + 1;
      t = y0 + el / 3;
    } else {
      el -= 6 * RY;
      F = 2 + el / (3 * BS);
      el %= 3 * BS;
      t = el % BS;
      l = el / BS + 1;
    }
    int hx, hy;                                   // plane coordinates, rows from y0
    if (F == 0) { hx = -l; hy = t - y0; }
    else if (F == 1) { hx = M + l; hy = t - y0; }
    else if (F == 2) { hx = t; hy = -l; }
    else { hx = t; hy = ny - 1 + l; }
    const unsigned dst = (unsigned)((hy + 3) * W + hx + 3);
    const int ty = ftype[F];
    const bool plus = F & 1;
    const int ax = F >> 1;
    uint4 e = make_uint4(0u, 0u, 0u, (unsigned)I::CS);
    if (F < 2 && t >= y0 + ny) {
      // past this CTA's rows: unused
    } else if ((F == 2 && y0 > 0) || (F == 3 && y0 + ny - 1 < M)) {
      // a row of this block held by the CTA next to this one
      const int yy = F == 2 ? y0 - l : y0 + ny - 1 + l;
      e.x = e.y = (unsigned)(bo + I::idx(t, yy, 0));
      e.z = ((unsigned)I::PL << 16) | dst;
    } else if (ty == kTypeCoarser) {
      e.x = e.y = (unsigned)I::slab(fs[F][0], l, t, 0);
      e.z = ((unsigned)(BS * I::PT) << 16) | 0x8000u | dst;
      e.w = (unsigned)I::SCS;
    } else if (ty == kTypeLeaf) {
      const int nl = plus ? l : M - l;
      const int xx = ax == 0 ? nl : t, yy = ax == 0 ? t : nl;
      e.x = e.y = (unsigned)((size_t)fs[F][0] * L::BLK + I::idx(xx, yy, 0));
      e.z = ((unsigned)I::PL << 16) | dst;
    } else {
      const int c0 = t > M / 2;
      const int nl = plus ? 2 * l : M - 2 * l;
      const int u0 = 2 * t - c0 * M;
      const int xx = ax == 0 ? nl : u0, yy = ax == 0 ? u0 : nl;
      e.x = (unsigned)((size_t)fs[F][c0] * L::BLK + I::idx(xx, yy, 0));
      // upper child: its plane 2z - M sits at 2z planes - M planes from its base (the sum with z * hz
      // is taken modulo 2^32 and is non-negative)
      e.y = (unsigned)((size_t)fs[F][c0 + 2] * L::BLK + I::idx(xx, yy, 0)) - (unsigned)(M * I::PL);
      e.z = ((unsigned)(2 * I::PL) << 16) | dst;
    }
    htab[i] = e;
  }
  auto halo_src = [&](const uint4& e, int z) -> const T* {
    const unsigned off = (z > M / 2 ? e.y : e.x) + (unsigned)z * (e.z >> 16);
    return ((e.z & 0x8000u) ? a.slab : a.in) + (size_t)off;
  };
  // solid velocity of a moving body at lattice point (i, j, k): omega x (x - x_0)
  auto solid = [&](int i, int j, int k, T (&us)[3]) {
    const T hT = kc.h[bi.x];
    const T rx = T(lattice_index(ph, bi, 0, i, M)) * hT - kc.x0[0];
    const T ry = T(lattice_index(ph, bi, 1, j, M)) * hT - kc.x0[1];
    const T rz = T(lattice_index(ph, bi, 2, k, M)) * hT - kc.x0[2];
    us[0] = kc.om[1] * rz - kc.om[2] * ry;
    us[1] = kc.om[2] * rx - kc.om[0] * rz;
    us[2] = kc.om[0] * ry - kc.om[1] * rx;
  };
  __syncthreads();                        // halo table complete
  auto issue_halos = [&](int z) {
#pragma unroll
    for (int k = 0; k < C::HPT; ++k) {
      const int i = tid + k * NT;
      if (i < NH) {
        const uint4 e = htab[i];
        if (C::NS == 1 || (e.z >> 16) != 0) {
          const unsigned off = (z > M / 2 ? e.y : e.x) + (unsigned)z * (e.z >> 16);
          Plane<T, PW>& B = buf[z & 3];
          const int d = (int)(e.z & 0x7fffu);
          if (AI) {
            B.copy_point(d, ((e.z & 0x8000u) ? a.slab : a.in) + (size_t)off);
          } else if (e.z & 0x8000u) {
            const T* p = a.slab + (size_t)off;
#pragma unroll
            for (int f = 0; f < 4; ++f) cp_async_elem(B.comp(d, f), p + f * I::SCS);
          } else {
            const T* p = a.in + (size_t)off;
#pragma unroll
            for (int f = 0; f < 4; ++f) cp_async_elem(B.comp(d, f), p + f * I::CS);
          }
        }
      }
    }
    cp_async_commit();
  };

  T nm[5] = {T(0), T(0), T(0), T(0), T(0)};   // stage 4: max |u|,|v|,|w|,|p|, |(u,v,w)|^2
  auto norms_of = [&](const T (&nv)[4]) {
#pragma unroll
    for (int f = 0; f < 4; ++f) nm[f] = max_number(nv[f], nm[f]);
    nm[4] = max_number(mag2(nv[0], nv[1], nv[2]), nm[4]);
  };
  const int nst = staged_arrays<STAGE>(ph.mask != 0);
  // this CTA's rows of a plane, widened to 16-byte boundaries inside the padded plane
  const int pf0 = C::NS == 1 ? 0 : ((y0 * BS) & ~(L::VEC - 1));
  const bool work = tid < NT;
  if (!work) {
    // the loading warp: the planes of every iteration by bulk copies, a lane each
    const int lane = tid - NT;
    const int pf1 = C::NS == 1 ? L::PP : (((y0 + ny) * BS + L::VEC - 1) & ~(L::VEC - 1));
    const unsigned bytes = (unsigned)((pf1 - pf0) * sizeof(T)), pbytes = (unsigned)(4 * ny * BS * sizeof(T));
    // lane k brings array k: 0..3 the input, 4..7 U, 8..11 Y_2, 12..15 Y_3 by components (a point-major
    // one whole by its first lane), the last one chi
    const bool is_in = lane < 4, pm = is_in ? AI : PM && STAGE == 4 && lane >= 8 && lane < 16;
    const T* src = nullptr;
    int pl = L::PP;                       // plane stride
    if (lane < nst) {
      const T* r = is_in ? a.in : (STAGE >= 2 && lane < 8 ? a.U : (STAGE == 4 && lane < 12 ? a.y2 : (STAGE == 4 && lane < 16 ? a.y3 : nullptr)));
      if (!r) src = a.chi + (size_t)slot * L::FS + pf0;
      else if (pm) src = (lane & 3) == 0 ? r + bo + 4 * y0 * BS : nullptr;
      else src = r + bo + (size_t)(lane & 3) * L::FS + pf0;
      if (pm) pl = 4 * BS * BS;
      if (is_in && src) src += 3 * pl;
    }
    const unsigned mine = pm ? pbytes : bytes;
    const unsigned in_bytes = AI ? pbytes : 4 * bytes;
    const unsigned other = (STAGE == 2 || STAGE == 3 ? 4 * bytes : (STAGE == 4 ? 4 * bytes + (PM ? 2 * pbytes : 8 * bytes) : 0)) +
                           (ph.mask ? bytes : 0);
    auto fill = [&](int z, int sl) {
      if (lane == 0) {
        fence_async_shared();
        mbar_expect_tx(&full[sl], other + (z + 3 <= M ? in_bytes : 0));
      }
      __syncwarp();
      if (src && (!is_in || z + 3 <= M))
        bulk_g2s(stg + ((size_t)sl * nst + lane) * SP, src + (size_t)z * pl, mine, &full[sl]);
    };
    for (int k = 0; k < kND; ++k)
      if (!SPLIT || z0 + k < z1) fill(z0 + k, k);
    if (C::CORNER && lane >= z0 && lane < z1) {
      // pencil (M, M), plane `lane`
      const int z = lane;
      V ca, cb;
      load_point<AI>(inb + I::idx(M, M, z), I::CS, ca, cb);
      T K[4], nv[4];
      point_rhs(kc, ph.mask, ph.sponge, cst, ca, cb,
                [&](int ax, int k, V& va, V& vb) {
                  if (ax == 2) {
                    if (z + k >= 0 && z + k <= M) {
                      load_point<AI>(inb + I::idx(M, M, z + k), I::CS, va, vb);
                    } else {
                      const T* p;
                      int ls, fcs;
                      z_face(k < 0 ? 4 : 5, M, M, p, ls, fcs);
                      load_point<AI>(p + ((k < 0 ? -(z + k) : z + k - M) - 1) * ls, fcs, va, vb);
                    }
                  } else if (k < 0) {
                    load_point<AI>(inb + (ax == 0 ? I::idx(M + k, M, z) : I::idx(M, M + k, z)), I::CS, va, vb);
                  } else {
                    const uint4 e = htab[ax == 0 ? 3 * RY + 3 * M + k - 1 : 6 * RY + 3 * BS + (k - 1) * BS + M];
                    load_point<AI>(halo_src(e, z), (int)e.w, va, vb);
                  }
                },
                [&]() { return a.chi[(size_t)slot * L::FS + L::idx(M, M, z)]; }, [&](T (&us)[3]) { solid(M, M, z, us); },
                [&]() { return tmax(tmax(sp[0][M], sp[1][M]), sp[2][z]); }, K);
      const int wm = fine_win_bits<M>(fwm, M, M);
      const bool keep = (wm & 1) || (z == 0 && (wm & 2)) || (z == M && (wm & 4));
      const T c[4] = {ca.x, ca.y, cb.x, cb.y};
      const size_t pu = bo + L::idx(M, M, z), py = bo + Y::idx(M, M, z);
      rk_combine<T, PM, STAGE>(a, py, Y::CS, c, K, [&](int f) { return a.U[pu + (size_t)f * L::FS]; },
                               [&](int f) { return a.y2[py + (size_t)f * Y::CS]; },
                               [&](int f) { return a.y3[py + (size_t)f * Y::CS]; }, cst[3], cst[4], keep, nv);
      store_point<AO>(a.out + bo + O::idx(M, M, z), O::CS, nv);
      if (STAGE == 4) norms_of(nv);
    }
    __syncwarp();
    int ds = kND - 1, dp = 0;
    for (int z = z0 + kND; z < z1; ++z) {
      // iteration z - 1 may start: every warp has put plane z - 1, so it has finished iteration z - 3,
      // whose slot is free
      mbar_wait(&full[ds], (unsigned)dp, err);
      ds = ds == kND - 1 ? 0 : ds + 1;
      dp ^= ds == 0;
      fill(z, ds);
    }
  }

  const int ci = (y - y0 + 3) * W + x + 3;
  const int lp = L::idx(x, y, 0) - pf0, lq = 4 * ((y - y0) * BS + x);   // this pencil in a staged plane
  const int wm = fine_win_bits<M>(fwm, x, y);
  // Plane z + 1 goes to shared memory at the start of iteration z (its centre is in the ring), and
  // a warp then tells the others so on an mbarrier: a warp waits for the slowest one only if that
  // is more than an iteration behind, instead of all warps meeting in every plane.  Buffer p & 3:
  // when a warp passes the wait of plane z, every warp has finished iteration z - 2, so the buffers
  // of planes z - 2 and older are free.
  auto publish = [&](int sl) {
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(&full[sl]);
  };
  // The planes beyond the upper z face, needed from iteration M - 2 on (each thread its own pencil's),
  // requested far enough ahead that nobody waits for them; which iteration commits their group is
  // upper_in_prologue / upper_in_loop's rule (stage_parts.hpp).
  auto load_upper = [&]() {
    const T* p;
    int ls, fcs;
    z_face(5, x, y, p, ls, fcs);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (AI) {
#pragma unroll
        for (int q = 0; q < (int)(4 * sizeof(T) / 16); ++q)
          cp_async_16(zup + k * 4 * SP + lq + q * (16 / (int)sizeof(T)), p + k * ls + q * (16 / (int)sizeof(T)));
      } else {
#pragma unroll
        for (int f = 0; f < 4; ++f) cp_async_elem(zup + (k * 4 + f) * SP + lp, p + k * ls + (size_t)f * fcs);
      }
    }
  };
  int ds = 0, dp = 0;                     // slot and phase of the iteration
  if (work) {
    if (SPLIT && act && upper_in_prologue(z0, M)) load_upper();
    issue_halos(z0);
    if (!SPLIT || z0 + 1 < z1) issue_halos(z0 + 1);
    else cp_async_commit();
    if (act) buf[z0 & 3].put(ci, qa[3], qb[3]);
    cp_async_wait_group<1>();
    publish(0);
  }
  Plane<T, PW>* B = buf + (z0 & 3);       // the plane of iteration z
#pragma unroll 1
  for (int zb = z0; zb < z1 && work; zb += 7) {
#pragma unroll
    for (int j = 0; j < 7; ++j) {
      const int z = zb + j;
      if (z >= z1) break;
      // ring entries of planes z - 3 .. z + 3
      auto QA = [&](int k) -> V& { return qa[(j + 3 + k) % 7]; };
      auto QB = [&](int k) -> V& { return qb[(j + 3 + k) % 7]; };
      mbar_wait(&full[ds], (unsigned)dp, err);
      const T* sg = stg + (size_t)ds * nst * SP;
      ds = ds == kND - 1 ? 0 : ds + 1;
      dp ^= ds == 0;
      if (act && upper_in_loop(z, z0, z1, M)) load_upper();
      if (z + 2 < z1) issue_halos(z + 2);
      else cp_async_commit();
      if (z + 1 < z1) {
        if (act) buf[(z + 1) & 3].put(ci, QA(1), QB(1));
        cp_async_wait_group<1>();
        publish(ds);
      }
      if (act) {
        load_point<AI>((z + 3 <= M ? sg : zup + (z + 2 - M) * 4 * SP) + (AI ? lq : lp), SP, QA(3), QB(3));
        T K[4], nv[4];
        const V ca = QA(0), cb = QB(0);
        point_rhs(kc, ph.mask, ph.sponge, cst, ca, cb,
                  [&](int ax, int k, V& va, V& vb) {
                    if (ax == 2) {
                      va = QA(k);
                      vb = QB(k);
                    } else {
                      B->get(ci + (ax == 0 ? k : k * W), va, vb);
                    }
                  },
                  [&]() { return sg[(nst - 1) * SP + lp]; }, [&](T (&us)[3]) { solid(x, y, z, us); },
                  [&]() { return tmax(tmax(sp[0][x], sp[1][y]), sp[2][z]); }, K);
        const bool keep = wm && ((wm & 1) || (z == 0 && (wm & 2)) || (z == M && (wm & 4)));
        const T c[4] = {ca.x, ca.y, cb.x, cb.y};
        T y2[4], y3[4];
        if (STAGE == 4 && PM) {
          V va, vb;
          load_point<PM>(sg + 8 * SP + lq, 1, va, vb);
          y2[0] = va.x; y2[1] = va.y; y2[2] = vb.x; y2[3] = vb.y;
          load_point<PM>(sg + 12 * SP + lq, 1, va, vb);
          y3[0] = va.x; y3[1] = va.y; y3[2] = vb.x; y3[3] = vb.y;
        }
        rk_combine<T, PM, STAGE>(a, bo + Y::idx(x, y, z), Y::CS, c, K, [&](int f) { return sg[(4 + f) * SP + lp]; },
                                 [&](int f) { return PM ? y2[f] : sg[(8 + f) * SP + lp]; },
                                 [&](int f) { return PM ? y3[f] : sg[(12 + f) * SP + lp]; }, cst[3], cst[4], keep, nv);
        store_point<AO>(a.out + bo + O::idx(x, y, z), O::CS, nv);
        if (STAGE == 4) norms_of(nv);
      }
      B = buf + ((z + 1) & 3);
    }
  }
  if (STAGE == 4 && a.norms) {
    // block maxima (the planes are free now), then one atomic maximum per norm and block
    __syncthreads();
    constexpr int NW = NT / 32 + 1;
    T* red = buf[0].comp(0, 0);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      T m = nm[k];
      for (int o = 16; o > 0; o >>= 1) {
        const T t = __shfl_xor_sync(0xffffffffu, m, o);
        m = t > m ? t : m;
      }
      if ((tid & 31) == 0) red[k * NW + (tid >> 5)] = m;
    }
    __syncthreads();
    if (tid < 5) {
      T m = T(0);
      for (int w = 0; w < NW; ++w) m = red[tid * NW + w] > m ? red[tid * NW + w] : m;
      const double d = tid == 4 ? (double)tsqrt(m) : (double)m;
      atomicMax(a.norms + tid, (unsigned long long)__double_as_longlong(d));
    }
  }
  if (MULTI) {
    __syncthreads();
    if (tid == 0) {
      for (int k = 0; k < kND; ++k) mbar_inval(&full[k]);
    }
  }
}

template <typename T, int BS, int STAGE, bool PM, bool SPLIT>
__global__ void __launch_bounds__(Cfg<T, BS>::NT + 32, Cfg<T, BS>::MINB)
k_stage(const StageK<T> a, const TopoK tp, const PhysK ph, int* err, int nz) {
  constexpr int NS = Cfg<T, BS>::NS;
  if (!SPLIT) nz = 1;
  const int rank = blockIdx.x / (NS * nz), q = blockIdx.x % (NS * nz), zp = q / NS;
  stage_block<T, BS, STAGE, PM, false, SPLIT>(a.p, a.kc, tp, ph, err, rank, q % NS, part_begin(zp, nz, BS),
                                              part_begin(zp + 1, nz, BS));
}

// Persistent form over several independent instances: the CTAs walk the work list of
// (instance, rank) pairs, each instance with its own arrays and topology (desc) and the same
// physics and constants; every block gets bitwise the update k_stage gives it.
template <typename T, int BS, int STAGE>
__global__ void __launch_bounds__(Cfg<T, BS>::NT + 32, Cfg<T, BS>::MINB)
k_stage_multi(const StageConst<T> kc, const PhysK ph, const StageInst<T>* desc, const int2* work, int nwork,
              int* err) {
  for (int w = blockIdx.x; w < nwork; w += gridDim.x) {
    const int2 it = work[w];
    const StageInst<T> d = desc[it.x];
    stage_block<T, BS, STAGE, true, true, false>(d.p, kc, d.tp, ph, err, it.y, 0, 0, BS);
    __syncthreads();                   // the next block reuses the shared arrays
  }
}

// Time step of one RK4 step on the device (Sec. 2.3): dt_fixed if > 0, else the CFL rule from the
// velocity max norm of the last reduction (maxbits[4]); writes rk[0] = dt, rk[1] += dt (time)
// and the stage coefficients rk[2..9] = (c_acc, c_out) of stages 1..4, in double, by the same
// expressions as the host path.
__global__ void k_rk_coefs(const unsigned long long* maxbits, RkK p, double* rk) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double dt = p.dt_fixed;
  if (!(dt > 0.0)) {
    const double u = __longlong_as_double((long long)maxbits[4]);
    const double ueig = fabs(u) + sqrt(u * u + p.c0 * p.c0);
    dt = p.cfl * p.h / ueig;
    if (p.mask) dt = fmin(dt, p.cfl_eta * p.C_eta);
    if (p.nu > 0) dt = fmin(dt, p.cfl_nu * p.h * p.h / p.nu);
  }
  rk[0] = dt;
  rk[1] += dt;
  rk[2] = dt / 6.0; rk[3] = dt / 2.0;
  rk[4] = dt / 3.0; rk[5] = dt / 2.0;
  rk[6] = dt / 3.0; rk[7] = dt;
  rk[8] = dt / 3.0; rk[9] = dt / 6.0;
}

// Parts of a block along z, a CTA each.  A CTA costs its start (six extra planes to load and a chain
// of dependent reads, about five planes' time in FP32, one in FP64 where a plane is long) plus its
// planes; the parts are chosen so that the waves of CTAs over the chip cost least: a grid of a few
// dozen blocks would leave most of the SMs idle with one CTA per block.  n: the blocks that run side by
// side (instances of a batch on several streams together fill a chip that one of them would not: with
// each split by its own count a batch of 12 instances took 11.1 ms instead of 9.9).  Measured, us per
// launch with one part and with this rule's: 17^3 FP32 8 blocks 19.0 and 9.4 (six parts), 57 blocks 20.9
// and 13.1 (five), 64 blocks 19.1 and 13.4 (four); FP64 29 blocks 212 and 57 (five), 64 blocks 210 and 114
// (two), 512 blocks 827 and 745 (two); 64 blocks of 33^3 65.0 and 54.8 (three), of 9^3 in FP64 53.3 and 33.0
// (two).  Where it keeps one part, two cost more: 302 blocks of 17^3 FP32 27.8 and 34.2.  A grid that fills
// the chip keeps one part, in a form of the kernel whose plane range the compiler knows (the split form
// spills registers there: 4608 blocks 426 against 393 us, 32768 blocks 2630 against 2420).
template <typename T, int BS>
int z_parts(int64_t n) {
  using C = Cfg<T, BS>;
  return z_parts_rule(n, C::NS, BS, (int64_t)C::MINB * sm_count(), sizeof(T) == 4 ? 5 : 1);
}

template <typename T, int BS, int STAGE, bool PM, bool SPLIT>
void launch_parts(const StageK<T>& s, const TopoK& t, const PhysK& p, int* err, int nz, cudaStream_t st) {
  static std::atomic<unsigned long long> opted{0};
  smem_opt_in_stage(k_stage<T, BS, STAGE, PM, SPLIT>, stage_smem<T, BS, STAGE>(true), opted);
  const size_t dyn = stage_smem<T, BS, STAGE>(p.mask != 0);
  k_stage<T, BS, STAGE, PM, SPLIT>
      <<<(unsigned)(t.n * Cfg<T, BS>::NS * nz), Cfg<T, BS>::NT + 32, dyn, st>>>(s, t, p, err, nz);
}
template <typename T, int BS, int STAGE, bool PM>
void launch_one(const StageK<T>& s, const TopoK& t, const PhysK& p, int* err, cudaStream_t st) {
  const int nz = !PM ? 1 : (s.parts > 0 ? s.parts : z_parts<T, BS>(std::max(t.n, s.side_by_side)));
  if constexpr (PM) {
    if (nz > 1) {
      launch_parts<T, BS, STAGE, PM, true>(s, t, p, err, nz, st);
      return;
    }
  }
  launch_parts<T, BS, STAGE, PM, false>(s, t, p, err, 1, st);
}

template <typename T, int BS>
void launch_stage_bs(int stage, const StageK<T>& s, const TopoK& t, const PhysK& p, int* err, cudaStream_t st) {
  if (t.n <= 0) return;
  switch (stage * 2 + (s.point_major ? 1 : 0)) {
    case 0: case 1: launch_one<T, BS, 0, false>(s, t, p, err, st); break;
    case 2: launch_one<T, BS, 1, false>(s, t, p, err, st); break;
    case 3: launch_one<T, BS, 1, true>(s, t, p, err, st); break;
    case 4: launch_one<T, BS, 2, false>(s, t, p, err, st); break;
    case 5: launch_one<T, BS, 2, true>(s, t, p, err, st); break;
    case 6: launch_one<T, BS, 3, false>(s, t, p, err, st); break;
    case 7: launch_one<T, BS, 3, true>(s, t, p, err, st); break;
    case 8: launch_one<T, BS, 4, false>(s, t, p, err, st); break;
    default: launch_one<T, BS, 4, true>(s, t, p, err, st); break;
  }
}

template <typename T>
StageConst<T> stage_constants(const PhysK& p, double c_acc, double c_out, const MaskK* body = nullptr) {
  StageConst<T> c{};
  c.moving = body != nullptr;
  for (int i = 0; i < 3; ++i) {
    c.om[i] = body ? T(body->p[19 + i]) : T(0);
    c.x0[i] = body ? T(body->p[9 + i]) : T(0);
  }
  c.r2 = vset(T(p.a2 / p.a1)); c.r3 = vset(T(p.a3 / p.a1));
  c.km16 = vset(T(-16)); c.k30 = vset(T(30));
  c.nu = T(p.nu); c.c0sq = T(p.c0sq); c.cgam = T(p.cgamma);
  c.inv_ceta = T(p.inv_ceta); c.inv_csp = T(p.inv_csp);
  for (int i = 0; i < 3; ++i) c.uinf[i] = T(p.uinf[i]);
  c.pinf = T(p.pinf);
  c.c_acc = T(c_acc); c.c_out = T(c_out);
  for (int J = 0; J <= kMaxLevel; ++J) {
    c.ih[J] = T(p.a1 / p.h[J]);
    c.ih2[J] = T(1.0 / (12.0 * p.h[J] * p.h[J]));
    c.h[J] = T(p.h[J]);
  }
  return c;
}

}  // namespace

template <typename T>
void launch_stage_multi(int stage, int Bs, const PhysK& p, const StageInst<T>* desc, const int2* work, int64_t nwork,
                        int* err, cudaStream_t st) {
  if (nwork <= 0 || Bs == 33) return;     // the persistent form takes whole blocks (Bs <= 17)
  const StageConst<T> kc = stage_constants<T>(p, 0.0, 0.0);
  auto go = [&](auto bs, auto sg) {
    constexpr int BS = decltype(bs)::value, SG = decltype(sg)::value;
    const int nb = (int)std::min<int64_t>(nwork, (int64_t)Cfg<T, BS>::MINB * sm_count());
    static std::atomic<unsigned long long> opted{0};
    smem_opt_in_stage(k_stage_multi<T, BS, SG>, stage_smem<T, BS, SG>(true), opted);
    const size_t dyn = stage_smem<T, BS, SG>(p.mask != 0);
    k_stage_multi<T, BS, SG><<<nb, Cfg<T, BS>::NT + 32, dyn, st>>>(kc, p, desc, work, (int)nwork, err);
  };
  auto pick = [&](auto bs) {
    switch (stage) {
      case 1: go(bs, std::integral_constant<int, 1>{}); break;
      case 2: go(bs, std::integral_constant<int, 2>{}); break;
      case 3: go(bs, std::integral_constant<int, 3>{}); break;
      default: go(bs, std::integral_constant<int, 4>{}); break;
    }
  };
  if (Bs == 17) pick(std::integral_constant<int, 17>{});
  else pick(std::integral_constant<int, 9>{});
}

template <typename T>
void launch_stage(int stage, int Bs, const StageK<T>& s, const TopoK& t, const PhysK& p, int* err, cudaStream_t st) {
  StageK<T> a = s;
  a.kc = stage_constants<T>(p, s.c_acc, s.c_out, s.body);
  if (Bs == 33) {
    if constexpr (sizeof(T) == 4) launch_stage_bs<T, 33>(stage, a, t, p, err, st);
  } else if (Bs == 17) {
    launch_stage_bs<T, 17>(stage, a, t, p, err, st);
  } else {
    launch_stage_bs<T, 9>(stage, a, t, p, err, st);
  }
}

void launch_rk_coefs(const unsigned long long* maxbits, const RkK& p, double* rk, cudaStream_t st) {
  k_rk_coefs<<<1, 32, 0, st>>>(maxbits, p, rk);
}

template void launch_stage<float>(int, int, const StageK<float>&, const TopoK&, const PhysK&, int*, cudaStream_t);
template void launch_stage<double>(int, int, const StageK<double>&, const TopoK&, const PhysK&, int*, cudaStream_t);
template void launch_stage_multi<float>(int, int, const PhysK&, const StageInst<float>*, const int2*, int64_t,
                                        int*, cudaStream_t);
template void launch_stage_multi<double>(int, int, const PhysK&, const StageInst<double>*, const int2*, int64_t,
                                         int*, cudaStream_t);

}  // namespace acm
