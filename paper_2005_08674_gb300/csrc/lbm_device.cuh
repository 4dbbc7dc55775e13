// lbm_device.cuh -- device-side building blocks of the D2Q9 + NSBC update
// for sm_103a: storage traits (shifted populations in f64/f32/f16/bf16 with
// 16-byte vector access), the BGK cell update, and the NSBC node update.
//
// Populations are stored as h_i = f_i - w_i (deviation from the rest state),
// so rho = 1 + sum h_i and rho u = sum c_i h_i (sum c_i w_i = 0).  The
// equilibrium in the same shift is
//   h_i^eq = f_i^eq - w_i = w_i (d_rho + rho (3 c_i.u + 4.5 (c_i.u)^2 - 1.5 u.u))
// which is Eq. (feq_1) with cs^2 = 1/3 minus w_i.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>

#include "lbm_check.cuh"

namespace lbmk {

// ---------------------------------------------------------------------------
// Lattice (Fig. 1): c_0=(0,0) c_1=(1,0) c_2=(-1,0) c_3=(0,1) c_4=(0,-1)
// c_5=(1,1) c_6=(-1,-1) c_7=(-1,1) c_8=(1,-1); w = 4/9, 1/9, 1/36.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int cx(int i) {
  return i == 1 || i == 5 || i == 8 ? 1 : (i == 2 || i == 6 || i == 7 ? -1 : 0);
}
__host__ __device__ constexpr int cy(int i) {
  return i == 3 || i == 5 || i == 7 ? 1 : (i == 4 || i == 6 || i == 8 ? -1 : 0);
}
__host__ __device__ constexpr int opp(int i) { return i == 0 ? 0 : (i % 2 == 1 ? i + 1 : i - 1); }
template <typename C>
__host__ __device__ constexpr C wt(int i) {
  return i == 0 ? C(4) / C(9) : (i <= 4 ? C(1) / C(9) : C(1) / C(36));
}

// ---------------------------------------------------------------------------
// Storage traits: compute type C, cells per 16-byte vector V, vector and
// scalar loads (streaming: every population is read once per step) and
// stores.  16-bit types round to nearest even on store.
// ---------------------------------------------------------------------------
template <typename T>
struct Store;

template <>
struct Store<double> {
  using C = double;
  static constexpr int V = 2;
  __device__ static void ld(const double* p, C (&o)[V]) {
    if (!in_bounds(p, 16)) {
      o[0] = o[1] = 0.0;
      return;
    }
    const double2 t = __ldcs(reinterpret_cast<const double2*>(p));
    o[0] = t.x;
    o[1] = t.y;
  }
  __device__ static void st(double* p, const C (&o)[V]) {
    if (!in_bounds(p, 16)) return;
    __stcs(reinterpret_cast<double2*>(p), make_double2(o[0], o[1]));
  }
  static constexpr double kScale = 1.0;
  // shared-memory copies of the stored values (tiles staged by bulk copies)
  __device__ static void lds(const double* p, C (&o)[V]) {
    const double2 t = *reinterpret_cast<const double2*>(p);
    o[0] = t.x;
    o[1] = t.y;
  }
  __device__ static C ld1s(const double* p) { return *p; }
  __device__ static C ld1(const double* p) { return in_bounds(p, 8) ? __ldcs(p) : 0.0; }
  __device__ static C ldg1(const double* p) { return in_bounds(p, 8) ? __ldg(p) : 0.0; }
  __device__ static void st1(double* p, C v) {
    if (in_bounds(p, 8)) *p = v;
  }
  __device__ static void st1r(double* p, C v) {
    if (in_bounds(p, 8)) *p = v;
  }
  __device__ static double cvt(C v) { return v; }
};

template <>
struct Store<float> {
  using C = float;
  static constexpr int V = 4;
  __device__ static void ld(const float* p, C (&o)[V]) {
    if (!in_bounds(p, 16)) {
      o[0] = o[1] = o[2] = o[3] = 0.f;
      return;
    }
    const float4 t = __ldcs(reinterpret_cast<const float4*>(p));
    o[0] = t.x;
    o[1] = t.y;
    o[2] = t.z;
    o[3] = t.w;
  }
  __device__ static void st(float* p, const C (&o)[V]) {
    if (!in_bounds(p, 16)) return;
    __stcs(reinterpret_cast<float4*>(p), make_float4(o[0], o[1], o[2], o[3]));
  }
  static constexpr float kScale = 1.0f;
  __device__ static void lds(const float* p, C (&o)[V]) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    o[0] = t.x;
    o[1] = t.y;
    o[2] = t.z;
    o[3] = t.w;
  }
  __device__ static C ld1s(const float* p) { return *p; }
  __device__ static C ld1(const float* p) { return in_bounds(p, 4) ? __ldcs(p) : 0.f; }
  __device__ static C ldg1(const float* p) { return in_bounds(p, 4) ? __ldg(p) : 0.f; }
  __device__ static void st1(float* p, C v) {
    if (in_bounds(p, 4)) *p = v;
  }
  __device__ static void st1r(float* p, C v) {
    if (in_bounds(p, 4)) *p = v;
  }
  __device__ static float cvt(C v) { return v; }
};

// binary16 holds h_i * 2^12: acoustic deviations of 1e-7..1e-2 would fall
// into binary16's subnormal range (below 6.1e-5), where the absolute spacing
// 6e-8 is a large relative error; scaled by 2^12 they stay normal (down to
// 1.5e-8), and |h| up to 16 still fits.  A power of two scales exactly.
constexpr float kHalfScale = 4096.0f;
constexpr float kHalfUnscale = 1.0f / 4096.0f;

// ld / st / ld1 / st1r move STORED values (s * h, s = kScale) and are used by
// the bulk kernel, whose collision works in stored units; ldg1 / st1 / cvt
// convert to and from h itself for the boundary and the helper kernels.
template <>
struct Store<__half> {
  using C = float;
  static constexpr int V = 8;
  static constexpr float kScale = kHalfScale;
  __device__ static void ld(const __half* p, C (&o)[V]) {
    if (!in_bounds(p, 16)) {
#pragma unroll
      for (int k = 0; k < V; ++k) o[k] = 0.f;
      return;
    }
    const uint4 t = __ldcs(reinterpret_cast<const uint4*>(p));
    const uint32_t w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      __half2 h2;
      memcpy(&h2, &w[k], 4);
      const float2 f = __half22float2(h2);
      o[2 * k] = f.x;
      o[2 * k + 1] = f.y;
    }
  }
  __device__ static void st(__half* p, const C (&o)[V]) {
    if (!in_bounds(p, 16)) return;
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const __half2 h2 = __floats2half2_rn(o[2 * k], o[2 * k + 1]);
      memcpy(&w[k], &h2, 4);
    }
    __stcs(reinterpret_cast<uint4*>(p), make_uint4(w[0], w[1], w[2], w[3]));
  }
  __device__ static void lds(const __half* p, C (&o)[V]) {
    const uint4 t = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      __half2 h2;
      memcpy(&h2, &w[k], 4);
      const float2 f = __half22float2(h2);
      o[2 * k] = f.x;
      o[2 * k + 1] = f.y;
    }
  }
  __device__ static C ld1s(const __half* p) { return __half2float(*p); }
  // half vectors (4 nodes, 8 bytes): shared-memory load and streaming store
  __device__ static void ldsp(const __half* p, C (&o)[4]) {
    const uint2 t = *reinterpret_cast<const uint2*>(p);
    __half2 a, b;
    memcpy(&a, &t.x, 4);
    memcpy(&b, &t.y, 4);
    const float2 fa = __half22float2(a), fb = __half22float2(b);
    o[0] = fa.x;
    o[1] = fa.y;
    o[2] = fb.x;
    o[3] = fb.y;
  }
  __device__ static void stp(__half* p, const C (&o)[4]) {
    if (!in_bounds(p, 8)) return;
    const __half2 a = __floats2half2_rn(o[0], o[1]), b = __floats2half2_rn(o[2], o[3]);
    uint2 t;
    memcpy(&t.x, &a, 4);
    memcpy(&t.y, &b, 4);
    __stcs(reinterpret_cast<uint2*>(p), t);
  }
  __device__ static C ld1(const __half* p) { return in_bounds(p, 2) ? __half2float(*p) : 0.f; }
  __device__ static void st1r(__half* p, C v) {
    if (in_bounds(p, 2)) *p = __float2half_rn(v);
  }
  __device__ static C ldg1(const __half* p) {
    return in_bounds(p, 2) ? __half2float(__ldg(p)) * kHalfUnscale : 0.f;
  }
  __device__ static void st1(__half* p, C v) {
    if (in_bounds(p, 2)) *p = __float2half_rn(v * kHalfScale);
  }
  __device__ static __half cvt(C v) { return __float2half_rn(v * kHalfScale); }
};

template <>
struct Store<__nv_bfloat16> {
  using C = float;
  static constexpr int V = 8;
  __device__ static void ld(const __nv_bfloat16* p, C (&o)[V]) {
    if (!in_bounds(p, 16)) {
#pragma unroll
      for (int k = 0; k < V; ++k) o[k] = 0.f;
      return;
    }
    const uint4 t = __ldcs(reinterpret_cast<const uint4*>(p));
    const uint32_t w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      __nv_bfloat162 b2;
      memcpy(&b2, &w[k], 4);
      const float2 f = __bfloat1622float2(b2);
      o[2 * k] = f.x;
      o[2 * k + 1] = f.y;
    }
  }
  __device__ static void st(__nv_bfloat16* p, const C (&o)[V]) {
    if (!in_bounds(p, 16)) return;
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const __nv_bfloat162 b2 = __floats2bfloat162_rn(o[2 * k], o[2 * k + 1]);
      memcpy(&w[k], &b2, 4);
    }
    __stcs(reinterpret_cast<uint4*>(p), make_uint4(w[0], w[1], w[2], w[3]));
  }
  static constexpr float kScale = 1.0f;
  __device__ static void lds(const __nv_bfloat16* p, C (&o)[V]) {
    const uint4 t = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      __nv_bfloat162 b2;
      memcpy(&b2, &w[k], 4);
      const float2 f = __bfloat1622float2(b2);
      o[2 * k] = f.x;
      o[2 * k + 1] = f.y;
    }
  }
  __device__ static C ld1s(const __nv_bfloat16* p) { return __bfloat162float(*p); }
  __device__ static void ldsp(const __nv_bfloat16* p, C (&o)[4]) {
    const uint2 t = *reinterpret_cast<const uint2*>(p);
    __nv_bfloat162 a, b;
    memcpy(&a, &t.x, 4);
    memcpy(&b, &t.y, 4);
    const float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
    o[0] = fa.x;
    o[1] = fa.y;
    o[2] = fb.x;
    o[3] = fb.y;
  }
  __device__ static void stp(__nv_bfloat16* p, const C (&o)[4]) {
    if (!in_bounds(p, 8)) return;
    const __nv_bfloat162 a = __floats2bfloat162_rn(o[0], o[1]), b = __floats2bfloat162_rn(o[2], o[3]);
    uint2 t;
    memcpy(&t.x, &a, 4);
    memcpy(&t.y, &b, 4);
    __stcs(reinterpret_cast<uint2*>(p), t);
  }
  __device__ static C ld1(const __nv_bfloat16* p) { return in_bounds(p, 2) ? __bfloat162float(*p) : 0.f; }
  __device__ static C ldg1(const __nv_bfloat16* p) { return in_bounds(p, 2) ? __bfloat162float(__ldg(p)) : 0.f; }
  __device__ static void st1(__nv_bfloat16* p, C v) {
    if (in_bounds(p, 2)) *p = __float2bfloat16_rn(v);
  }
  __device__ static void st1r(__nv_bfloat16* p, C v) {
    if (in_bounds(p, 2)) *p = __float2bfloat16_rn(v);
  }
  __device__ static __nv_bfloat16 cvt(C v) { return __float2bfloat16_rn(v); }
};

// Bulk-copy-engine prefetch of [p, p + bytes) into L2 (16-byte aligned,
// bytes a multiple of 16); no registers or shared memory are tied up.
__device__ __forceinline__ void prefetch_l2(const void* p, unsigned bytes) {
  if (!in_bounds(p, bytes)) return;
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// ---------------------------------------------------------------------------
// Moments of shifted populations (Eqs. cf_0, cf_1 as discrete sums).
// ---------------------------------------------------------------------------
template <typename C>
__device__ __forceinline__ void moments(const C (&h)[9], C& drho, C& jx, C& jy) {
  drho = ((h[0] + h[1]) + (h[2] + h[3])) + ((h[4] + h[5]) + (h[6] + h[7])) + h[8];
  jx = (h[1] - h[2]) + (h[5] - h[6]) + (h[8] - h[7]);
  jy = (h[3] - h[4]) + (h[5] - h[6]) + (h[7] - h[8]);
}

// Shifted equilibrium h^eq_i at (d_rho, u), Eq. (feq_1) minus w_i, times the
// storage scale s (1 except for binary16 storage, where it folds into w_i).
template <typename C>
__device__ __forceinline__ void equilibrium(C drho, C ux, C uy, C (&e)[9], C s = C(1)) {
  const C rho = C(1) + drho;
  const C usq = C(1.5) * (ux * ux + uy * uy);
  const C w0 = wt<C>(0) * s, wa = wt<C>(1) * s, wd = wt<C>(5) * s;
  e[0] = w0 * (drho - rho * usq);
  // axis directions: c.u = +-ux, +-uy
  {
    const C a = C(4.5) * ux * ux - usq, b = C(3) * ux;
    e[1] = wa * (drho + rho * (a + b));
    e[2] = wa * (drho + rho * (a - b));
  }
  {
    const C a = C(4.5) * uy * uy - usq, b = C(3) * uy;
    e[3] = wa * (drho + rho * (a + b));
    e[4] = wa * (drho + rho * (a - b));
  }
  {
    const C s = ux + uy;  // c_5 = -c_6 = (1, 1)
    const C a = C(4.5) * s * s - usq, b = C(3) * s;
    e[5] = wd * (drho + rho * (a + b));
    e[6] = wd * (drho + rho * (a - b));
  }
  {
    const C d = uy - ux;  // c_7 = -c_8 = (-1, 1)
    const C a = C(4.5) * d * d - usq, b = C(3) * d;
    e[7] = wd * (drho + rho * (a + b));
    e[8] = wd * (drho + rho * (a - b));
  }
}

// Storage shift.  A stored population is h_i = f_i - f_i^eq(m0) (times the
// storage scale), m0 = (rho0, u0) the far field, so that with a mean flow the
// stored numbers stay as small as the disturbance instead of carrying the
// stream's equilibrium (a 16-bit storage keeps its relative precision for
// what changes); for a far field at rest h_i = f_i - w_i.  The step kernels
// compute in deviations from m0 as well (d = rho - rho0, v = u - u0: cell_sums,
// pair_equilibrium), which needs P_i(u0), u0 and rho0; sh_i = f_i^eq(m0) - w_i
// converts to and from absolute populations outside the step.
template <typename C>
struct Shift {
  C sh[9];        // f_i^eq(m0) - w_i
  C p0[9];        // P_i(u0) = 1 + 3 c_i.u0 + 4.5 (c_i.u0)^2 - 1.5 u0.u0
  C u0[2];        // u0
  C rho0;         // rho0
  double m0[3];   // (rho0, u0x, u0y) in double
  bool on;        // false: far field at rest (rho0 = 1, u0 = 0)
};

// The shift of far field m0 = (rho0, u0x, u0y), formed in double on the host
// (the same expression as equilibrium() below, with rho0 - 1 kept apart).
// Defined once, in lbm_runtime.cu: a host compiler that fuses multiply-adds
// could otherwise round an inline copy differently in each file, and the
// single-domain and batched paths must start from the same bits.
Shift<double> far_field_shift(const double m0[3]);

template <typename C>
__host__ __device__ inline Shift<C> shift_as(const Shift<double>& z) {
  Shift<C> o;
  for (int i = 0; i < 9; ++i) o.sh[i] = C(z.sh[i]);
  for (int i = 0; i < 9; ++i) o.p0[i] = C(z.p0[i]);
  o.u0[0] = C(z.u0[0]);
  o.u0[1] = C(z.u0[1]);
  o.rho0 = C(z.rho0);
  for (int c = 0; c < 3; ++c) o.m0[c] = z.m0[c];
  o.on = z.on;
  return o;
}

// Relaxation rates, and the storage shift the collision needs.
template <typename C>
struct Rates {
  C omega;         // BGK rate 1/tau, also the MRT stress rate omega_nu
  C s_e, s_eps, s_q;
  Shift<C> z;
};

// a * b + c rounded once, in every kernel alike (the shift terms multiply
// loop-invariant values, and a compiler left free to hoist the product in one
// kernel and fuse it in another would round them differently).
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
// a - b rounded on its own (never fused with a product that formed a)
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
// a * b rounded on its own (never fused into a later add)
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// a / rho for the velocity u = (rho u) / rho of the macroscopic fields: in
// float the fast division intrinsic (within 2 ulp for rho in the normal range;
// rho is near 1 here), an IEEE division in double (the parity mode).
__device__ __forceinline__ float div_rho(float a, float rho) { return __fdividef(a, rho); }
__device__ __forceinline__ double div_rho(double a, double rho) { return a / rho; }

// The interior collision's arithmetic, every operation rounded on its own
// (none fused by the compiler), on one node (float, double) or on two nodes
// at once (float2: the paired FP32 instructions of sm_100 and later, whose
// components round exactly as the scalar __fadd_rn / __fmul_rn / __fmaf_rn
// do).  The same sequence of operations therefore gives the same bits for a
// node whether it is collided alone or beside another.
__device__ __forceinline__ float v_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double v_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float2 v_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float v_neg(float a) { return -a; }
__device__ __forceinline__ double v_neg(double a) { return -a; }
__device__ __forceinline__ float2 v_neg(float2 a) { return make_float2(-a.x, -a.y); }
// a - b rounded once (negating a paired operand costs no instruction)
__device__ __forceinline__ float v_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double v_sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float2 v_sub(float2 a, float2 b) { return v_add(a, v_neg(b)); }
__device__ __forceinline__ float v_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double v_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float2 v_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float v_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double v_fma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float2 v_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
template <typename V, typename C>
__device__ __forceinline__ V v_splat(C c) {
  if constexpr (std::is_same<V, float2>::value)
    return make_float2(c, c);
  else
    return V(c);
}
// 1 / a for the velocity u = (rho u) / rho.  float: the hardware's
// approximate reciprocal (0.975 last places measured over [1e-6, 1e6]).
// double: its gross approximation (about 20 bits) and one third-order step of
// Householder's iteration, r (1 + e + e^2) with e = 1 - a r, which leaves an
// error of e^3 (2^-60) before the last rounding (0.508 last places measured,
// and the value of a division in 9,995 cases of 10,000): three FP64
// operations where the IEEE division takes about nine, on a chip whose FP64
// pipe issues one warp instruction in 16 cycles.
__device__ __forceinline__ float v_rcp(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ double v_rcp(double a) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
  const double e = __fma_rn(-a, r, 1.0);
  return __fma_rn(r, __fma_rn(e, e, e), r);
}
// 1 / a as an IEEE division rounds it (one Newton step in float: the same in
// each of four million measured cases; in double the iteration above)
__device__ __forceinline__ float rcp_full(float a) {
  const float r = v_rcp(a);
  return __fmaf_rn(r, __fmaf_rn(-a, r, 1.f), r);
}
__device__ __forceinline__ double rcp_full(double a) { return v_rcp(a); }
__device__ __forceinline__ float2 v_rcp(float2 a) { return make_float2(v_rcp(a.x), v_rcp(a.y)); }

// ---------------------------------------------------------------------------
// The interior collision, from the pairs of opposite populations.
//
// With d = rho - rho0 = sum h, j = sum c h (the momentum's deviation from
// rho0 u0), J = rho (u - u0) = j - d u0, v = u - u0 = J / rho, the deviation
// of the equilibrium (Eq. feq_1) from the far field's is
//   E_i = f_i^eq(rho, u) - f_i^eq(rho0, u0)
//       = w_i [ d + 3 c_i.j + 4.5 c_i c_i : Pi - 1.5 tr Pi ],
//   Pi  = rho u u - rho0 u0 u0 = d u0 u0 + J u0 + u0 J + J v,
// so with a = Pi_xx, b = Pi_yy, c = Pi_xy, q = a + b
//   E_0     = w_0 [ d - 1.5 q ],
//   E_{1,2} = w_1 [ d - 1.5 q + 4.5 a +- 3 j_x ],   E_{3,4} with b, j_y,
//   E_{5,6} = w_5 [ d + 3 q + 9 c +- 3 (j_x + j_y) ],
//   E_{7,8} = w_5 [ d + 3 q - 9 c +- 3 (j_y - j_x) ].
// Every term is of the size of the disturbance, so float rounding is
// relative to it in a mean flow too, and the linear term takes j as summed
// from the populations.  Everything is held in stored units (times the
// storage scale s, a power of two): 1 / (s rho) turns s J into v.
//
// These kernels are bound by instruction issue (f32 and 16 bit) or by the
// FP64 pipe (f64), so the operations are what counts: 55 for BGK and 67 for
// MRT plus the reciprocal.  Forming the nine E_i one by one and relaxing each
// population took 81 and 138 and an IEEE division in f64.  Every operation
// is rounded on its own (v_add / v_mul / v_fma), so the shifted form with a
// zero shift rounds exactly like the plain one, and two nodes at once like
// one at a time.
// ---------------------------------------------------------------------------
template <typename V>
struct CellSums {
  V s1, s3, s5, s7;  // h_i + h_opp(i)
  V t1, t3;          // h_i - h_opp(i)
  V m, p;            // t5 - t7, t5 + t7
  V sa, sd;          // s1 + s3, s5 + s7
  V d, jx, jy;       // moments
  V Jx, Jy, wy;      // J, u_y: Pi_xy = J_x u_y + u0_x (J_y + d u0_y)
  V a, b, q, r;      // Pi_xx, Pi_yy, a + b, a - b
};

template <bool SHIFT, typename V, typename C>
__device__ __forceinline__ void cell_sums(const V (&h)[9], const Shift<C>& z, C s, V vs, CellSums<V>& o) {
  o.s1 = v_add(h[1], h[2]);
  o.t1 = v_sub(h[1], h[2]);
  o.s3 = v_add(h[3], h[4]);
  o.t3 = v_sub(h[3], h[4]);
  o.s5 = v_add(h[5], h[6]);
  o.s7 = v_add(h[7], h[8]);
  const V t5 = v_sub(h[5], h[6]), t7 = v_sub(h[7], h[8]);
  o.m = v_sub(t5, t7);
  o.p = v_add(t5, t7);
  o.sa = v_add(o.s1, o.s3);
  o.sd = v_add(o.s5, o.s7);
  o.d = v_add(v_add(o.sa, o.sd), h[0]);
  o.jx = v_add(o.t1, o.m);
  o.jy = v_add(o.t3, o.p);
  // No sum takes a product here: a paired sum of a paired product may be
  // contracted by the compiler, and would then round differently from the
  // scalar form.
  if constexpr (SHIFT) {
    const C ux = z.u0[0], uy = z.u0[1];
    const V inv = v_rcp(v_add(v_splat<V>(mul_rn(s, z.rho0)), o.d));
    const V u = v_splat<V>(ux), w = v_splat<V>(uy), one = v_splat<V>(C(1)), two = v_splat<V>(C(2));
    const V uyy = v_splat<V>(mul_rn(uy, uy)), uxx = v_splat<V>(mul_rn(ux, ux));
    o.Jx = v_fma(v_neg(u), o.d, o.jx);
    o.Jy = v_fma(v_neg(w), o.d, o.jy);
    const V vx = v_mul(o.Jx, inv), vy = v_mul(o.Jy, inv);
    const V sx = v_fma(two, u, vx), sy = v_fma(two, w, vy);  // s = 2 u0 + v
    o.wy = v_fma(one, w, vy);
    o.a = v_fma(o.d, uxx, v_mul(o.Jx, sx));
    o.b = v_fma(o.d, uyy, v_mul(o.Jy, sy));
    o.q = v_fma(o.Jx, sx, v_fma(o.d, uxx, o.b));
    o.r = v_fma(v_neg(o.Jy), sy, v_fma(v_neg(o.d), uyy, o.a));
  } else {
    const V inv = v_rcp(v_add(vs, o.d));
    const V vx = v_mul(o.jx, inv);
    o.Jx = o.jx;
    o.Jy = o.jy;
    o.wy = v_mul(o.jy, inv);
    o.a = v_mul(o.jx, vx);
    o.b = v_mul(o.jy, o.wy);
    o.q = v_fma(o.jx, vx, o.b);
    o.r = v_fma(v_neg(o.jy), o.wy, o.a);
  }
}

// Pi_xy, and x - Pi_xy
template <bool SHIFT, typename V, typename C>
__device__ __forceinline__ V pi_xy(const CellSums<V>& n, const Shift<C>& z) {
  V c = v_mul(n.Jx, n.wy);
  if constexpr (SHIFT)
    c = v_fma(v_splat<V>(z.u0[0]), n.Jy, v_fma(v_splat<V>(mul_rn(z.u0[0], z.u0[1])), n.d, c));
  return c;
}
template <bool SHIFT, typename V, typename C>
__device__ __forceinline__ V less_pi_xy(const CellSums<V>& n, const Shift<C>& z, V x) {
  if constexpr (SHIFT) {
    x = v_fma(v_splat<V>(-z.u0[0]), n.Jy, x);
    x = v_fma(v_splat<V>(-mul_rn(z.u0[0], z.u0[1])), n.d, x);
  }
  return v_fma(v_neg(n.Jx), n.wy, x);
}

// The constants of the collision of two nodes or one, formed once per kernel.
// PIN (pairs): the compiler would rather rebuild a pair of equal constants
// before each use than keep its two registers; an empty asm it cannot see
// through keeps them.
template <typename V, bool PIN>
__device__ __forceinline__ V v_const(typename std::conditional<std::is_same<V, double>::value, double, float>::type c) {
  V v = v_splat<V>(c);
  if constexpr (PIN && std::is_same<V, float2>::value) {
    unsigned long long u;
    memcpy(&u, &v, 8);
    asm volatile("" : "+l"(u));
    memcpy(&v, &u, 8);
  }
  return v;
}

template <typename V>
struct CellConst {
  V s, two, half;                     // storage scale, 2, 1/2
  V k2, wa, wa15, wa45, wd, wd3, wd6, wd9;  // BGK
  V three, four, ke, kep, kq, kw;     // MRT
};

template <int MODEL, bool PIN, typename V, typename C>
__device__ __forceinline__ CellConst<V> cell_const(const Rates<C>& r, C s) {
  CellConst<V> k;
  k.s = v_const<V, PIN>(s);
  k.two = v_const<V, PIN>(C(2));
  if constexpr (MODEL == 1) {
    k.three = v_const<V, PIN>(C(3));
    k.four = v_const<V, PIN>(C(4));
    k.ke = v_const<V, PIN>(mul_rn(r.s_e, C(1.0 / 36.0)));
    k.kep = v_const<V, PIN>(mul_rn(r.s_eps, C(1.0 / 12.0)));
    k.kq = v_const<V, PIN>(mul_rn(r.s_q, C(1.0 / 12.0)));
    k.kw = v_const<V, PIN>(mul_rn(r.omega, C(0.25)));
  } else {
    const C wa = mul_rn(r.omega, wt<C>(1)), wd = mul_rn(C(0.25), wa);
    k.half = v_const<V, PIN>(C(0.5));
    k.k2 = v_const<V, PIN>(mul_rn(C(0.5), sub_rn(C(1), r.omega)));
    k.wa = v_const<V, PIN>(wa);
    k.wa15 = v_const<V, PIN>(mul_rn(C(1.5), wa));
    k.wa45 = v_const<V, PIN>(mul_rn(C(4.5), wa));
    k.wd = v_const<V, PIN>(wd);
    k.wd3 = v_const<V, PIN>(mul_rn(C(3), wd));
    k.wd6 = v_const<V, PIN>(mul_rn(C(6), wd));
    k.wd9 = v_const<V, PIN>(mul_rn(C(9), wd));
  }
  return k;
}

// BGK collision, Eq. (lbe_1) with dt = 1, on shifted populations held as
// s * h: h* = (1 - omega) h + omega E, by pairs: with S = (h*_i + h*_opp) / 2
// and T = (h*_i - h*_opp) / 2,
//   S_i = keep/2 s_i + omega w_i [ ... ],   X = T_5 - T_7, Y = T_5 + T_7,
// and what the relaxation conserves closes the rest: T_1 = j_x / 2 - X,
// T_3 = j_y / 2 - Y, h*_0 = d - 2 (S_1 + S_3 + S_5 + S_7).  Mass and momentum
// are then kept to the rounding of each sum; relaxing every population with
// its own rounded omega w_i lost up to 1e-7 of the disturbance per step (the
// rounded weights do not add up to omega), which after 100 steps was the
// whole f32 error.
template <bool SHIFT, typename V, typename C>
__device__ __forceinline__ void collide_bgk(V (&h)[9], const Rates<C>& r, C s, const CellConst<V>& k) {
  CellSums<V> n;
  cell_sums<SHIFT>(h, r.z, s, k.s, n);
  const V ba = v_fma(v_neg(k.wa15), n.q, v_mul(k.wa, n.d));
  const V bd = v_fma(k.wd3, n.q, v_mul(k.wd, n.d));
  const V c = pi_xy<SHIFT>(n, r.z);
  const V S1 = v_fma(k.k2, n.s1, v_fma(k.wa45, n.a, ba));
  const V S3 = v_fma(k.k2, n.s3, v_fma(k.wa45, n.b, ba));
  const V S5 = v_fma(k.k2, n.s5, v_fma(k.wd9, c, bd));
  const V S7 = v_fma(k.k2, n.s7, v_fma(v_neg(k.wd9), c, bd));
  const V X = v_fma(k.k2, n.m, v_mul(k.wd6, n.jx)), Y = v_fma(k.k2, n.p, v_mul(k.wd6, n.jy));
  const V T1 = v_fma(k.half, n.jx, v_neg(X)), T3 = v_fma(k.half, n.jy, v_neg(Y));
  const V U5 = v_add(X, Y), U7 = v_sub(Y, X);  // 2 T_5, 2 T_7
  h[0] = v_fma(v_neg(k.two), v_add(v_add(S1, S3), v_add(S5, S7)), n.d);
  h[1] = v_add(S1, T1);
  h[2] = v_sub(S1, T1);
  h[3] = v_add(S3, T3);
  h[4] = v_sub(S3, T3);
  h[5] = v_fma(k.half, U5, S5);
  h[6] = v_fma(v_neg(k.half), U5, S5);
  h[7] = v_fma(k.half, U7, S7);
  h[8] = v_fma(v_neg(k.half), U7, S7);
}

// ---------------------------------------------------------------------------
// MRT collision, Eq. (mrt_lbe): f* = f - M^-1 S (m - m^eq), with the
// Gram-Schmidt moment basis of Sec. 4 in the order of Eq. (mrt_rm):
// (rho, e, eps, jx, qx, jy, qy, pxx, pxy).  Rows scaled to integers:
//   e   = (-4, -1, -1, -1, -1,  2,  2,  2,  2)   |e|^2   = 36
//   eps = ( 4, -2, -2, -2, -2,  1,  1,  1,  1)   |eps|^2 = 36
//   qx  = ( 0, -2,  2,  0,  0,  1, -1, -1,  1)   |qx|^2  = 12
//   qy  = ( 0,  0,  0, -2,  2,  1, -1,  1, -1)   |qy|^2  = 12
//   pxx = ( 0,  1,  1, -1, -1,  0,  0,  0,  0)   |pxx|^2 = 4
//   pxy = ( 0,  0,  0,  0,  0,  1,  1, -1, -1)   |pxy|^2 = 4
// The rows are orthogonal, so M^-1 = M^T diag(1/|row|^2); a row scale does
// not change M^-1 S M.  The conserved moments of f - f^eq vanish, so their
// rates (C_rho, C_jx, C_jy) never enter.  The stress rate is 1/tau.  The
// moments of E (above) are e: -2 d + 3 q, eps: d - 3 q, q: -j, pxx: a - b,
// pxy: c, so the non-equilibrium moments need no equilibrium populations:
//   e   : -2 h0 + sa + 4 sd - 3 q      eps : 3 (h0 - sa + q)
//   qx  : 2 m - t1                     qy  : 2 p - t3
//   pxx : (s1 - s3) - (a - b)          pxy : (s5 - s7) - c
// ---------------------------------------------------------------------------
template <bool SHIFT, typename V, typename C>
__device__ __forceinline__ void collide_mrt(V (&h)[9], const Rates<C>& r, C s, const CellConst<V>& k) {
  CellSums<V> n;
  cell_sums<SHIFT>(h, r.z, s, k.s, n);
  const V two = k.two, mtwo = v_neg(k.two);
  const V me = v_fma(v_neg(k.three), n.q, v_fma(k.four, n.sd, v_fma(mtwo, h[0], n.sa)));
  const V mep = v_add(v_sub(h[0], n.sa), n.q);  // a third of it
  const V mqx = v_fma(two, n.m, v_neg(n.t1)), mqy = v_fma(two, n.p, v_neg(n.t3));
  const V mxx = v_sub(v_sub(n.s1, n.s3), n.r);
  const V mxy = less_pi_xy<SHIFT>(n, r.z, v_sub(n.s5, n.s7));
  const V re = v_mul(k.ke, me), rep = v_mul(k.kep, mep);
  const V rqx = v_mul(k.kq, mqx), rqy = v_mul(k.kq, mqy);
  const V rxx = v_mul(k.kw, mxx), rxy = v_mul(k.kw, mxy);
  const V a0 = v_fma(mtwo, rep, v_neg(re));  // e/eps part of the axis columns
  const V a1 = v_fma(two, re, rep);          // e/eps part of the diagonal columns
  const V ax = v_add(a0, rxx), ay = v_sub(a0, rxx);
  const V d5 = v_add(a1, rxy), d7 = v_sub(a1, rxy);
  const V q5 = v_add(rqx, rqy), q7 = v_sub(rqy, rqx);
  h[0] = v_fma(v_neg(k.four), v_sub(rep, re), h[0]);
  h[1] = v_sub(h[1], v_fma(mtwo, rqx, ax));
  h[2] = v_sub(h[2], v_fma(two, rqx, ax));
  h[3] = v_sub(h[3], v_fma(mtwo, rqy, ay));
  h[4] = v_sub(h[4], v_fma(two, rqy, ay));
  h[5] = v_sub(h[5], v_add(d5, q5));
  h[6] = v_sub(h[6], v_sub(d5, q5));
  h[7] = v_sub(h[7], v_add(d7, q7));
  h[8] = v_sub(h[8], v_sub(d7, q7));
}

// Collision model: 0 = BGK (Eq. lbe_1), 1 = MRT (Eq. mrt_lbe).
template <int MODEL, bool SHIFT, typename V, typename C>
__device__ __forceinline__ void collide(V (&h)[9], const Rates<C>& r, C s, const CellConst<V>& k) {
  if constexpr (MODEL == 1)
    collide_mrt<SHIFT>(h, r, s, k);
  else
    collide_bgk<SHIFT>(h, r, s, k);
}
template <int MODEL, bool SHIFT, typename V, typename C>
__device__ __forceinline__ void collide(V (&h)[9], const Rates<C>& r, C s = C(1)) {
  collide<MODEL, SHIFT>(h, r, s, cell_const<MODEL, false, V>(r, s));
}

// The collision of N nodes held as h[i][k] (population i of node k): with
// PAIRED, in float, two nodes per paired instruction (half the arithmetic
// instructions, at the price of register pairs: worth it where the kernel is
// bound by instruction issue and has registers to spare), otherwise one
// after another; the bits of each node are those of collide() on it alone
// either way.
template <int MODEL, bool SHIFT, bool PAIRED, typename C, int N>
__device__ __forceinline__ void collide_nodes(C (&h)[9][N], const Rates<C>& r, C s = C(1)) {
  if constexpr (PAIRED && std::is_same<C, float>::value && N % 2 == 0) {
#pragma unroll
    for (int k = 0; k < N; k += 2) {
      float2 p[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) p[i] = make_float2(h[i][k], h[i][k + 1]);
      collide<MODEL, SHIFT>(p, r, s);
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        h[i][k] = p[i].x;
        h[i][k + 1] = p[i].y;
      }
    }
  } else {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      C n[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) n[i] = h[i][k];
      collide<MODEL, SHIFT>(n, r, s);
#pragma unroll
      for (int i = 0; i < 9; ++i) h[i][k] = n[i];
    }
  }
}

// ---------------------------------------------------------------------------
// Geometry and NSBC parameters passed by value to the kernels.
// ---------------------------------------------------------------------------
struct Geom {
  int nx, ny, pitch;
  long long plane;  // elements between population planes
};

// A number as the unevaluated sum of two floats (48 bits together).
struct FloatPair {
  float h, l;
};

struct Nsbc {
  double gamma, beta, kappa;
  double m0[3];  // far-field (rho, ux, uy)
  int order;     // 1 or 2
  int corner;    // corner reading: 0 diagonal normal, 1 mean of the two edges' m_c
  int periodic_x, periodic_y;  // axes closed periodically instead of by NSBC edges
  int vel[4];                  // edges (left, right, bottom, top) with a prescribed velocity
  double uw[4][2];             // that velocity
  // the same settings as the float kernels use them (set())
  float kappa_f;
  FloatPair step[2];  // gamma / |n| along an edge's normal and along a corner's diagonal, halved for order 2
  FloatPair keep;     // 1 - beta

  void set(double gamma_, double beta_, double kappa_, int corner_, int order_) {
    gamma = gamma_;
    beta = beta_;
    kappa = kappa_;
    corner = corner_;
    order = order_;
    // (settings past the range of float at its end: an infinity would make 0 of a uniform state a NaN)
    auto pair = [](double v) {
      constexpr double most = 3.4028234663852886e38;
      v = v > most ? most : (v < -most ? -most : v);
      const float h = (float)v;
      return FloatPair{h, (float)(v - (double)h)};
    };
    const double g = order == 2 ? 0.5 * gamma : gamma;
    kappa_f = (float)kappa;
    step[0] = pair(g);
    step[1] = pair(g * 0.70710678118654752);
    keep = pair(1.0 - beta);
  }
};

// Node k of the perimeter (k < 2 nx + 2 (ny - 2)) -> coordinates and outward
// normal.  Order: bottom row, top row, left column, right column (corners
// belong to the rows).
__device__ __forceinline__ void perimeter_node(int k, int nx, int ny, int& x, int& y, int& nxn, int& nyn) {
  if (k < 2 * nx) {
    const bool top = k >= nx;
    x = top ? k - nx : k;
    y = top ? ny - 1 : 0;
    nyn = top ? 1 : -1;
    nxn = x == 0 ? -1 : (x == nx - 1 ? 1 : 0);
  } else {
    k -= 2 * nx;
    const bool right = k >= ny - 2;
    y = 1 + (right ? k - (ny - 2) : k);
    x = right ? nx - 1 : 0;
    nxn = right ? 1 : -1;
    nyn = 0;
  }
}

// Deviations (rho - rho0, u - u0) from the far field at node (x, y) of the
// stored state, in the compute type of the storage: float for f32 / f16 /
// bf16 (the shifted populations keep them free of cancellation, so float
// loses nothing the storage kept), double in the f64 parity mode.
template <typename T>
__device__ __forceinline__ void node_dmoments(const T* __restrict__ A, const Geom& g, int x, int y,
                                              const Shift<typename Store<T>::C>& z, typename Store<T>::C (&m)[3]) {
  using S = Store<T>;
  using C = typename S::C;
  const long long o = (long long)y * g.pitch + x;
  C h[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) h[i] = S::ldg1(A + i * g.plane + o);
  C d, jx, jy;
  moments(h, d, jx, jy);
  const C inv = div_rho(C(1), z.rho0 + d);
  m[0] = d;
  m[1] = fma_rn(-d, z.u0[0], jx) * inv;
  m[2] = fma_rn(-d, z.u0[1], jy) * inv;
}

// Deviations (rho - rho0, u - u0) from the far field of a node's shifted
// populations (physical units) in the compute type of the storage: every
// quantity is of the size of the disturbance, so float is exact to float
// rounding of the perturbation.  For a far field at rest (SHIFT false) they
// are (rho - 1, u).
template <bool SHIFT, typename C>
__device__ __forceinline__ void dmoments_of(const C (&h)[9], C rho0, C u0x, C u0y, C (&m)[3]) {
  C d, jx, jy;
  moments(h, d, jx, jy);
  m[0] = d;
  if constexpr (SHIFT) {
    const C inv = rcp_full(rho0 + d);
    m[1] = mul_rn(fma_rn(-d, u0x, jx), inv);
    m[2] = mul_rn(fma_rn(-d, u0y, jy), inv);
  } else {
    const C inv = rcp_full(C(1) + d);
    m[1] = mul_rn(jx, inv);
    m[2] = mul_rn(jy, inv);
  }
}

}  // namespace lbmk
