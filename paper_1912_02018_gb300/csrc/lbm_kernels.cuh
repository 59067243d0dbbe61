// Kernels of one time step of the CM pseudopotential boiling LBM (arXiv:1912.02018),
// templated on the compute type C (double or float) and population storage type S.
//
// Layout: structure of arrays, every field [ny][pitch] with x fastest; populations are
// 9 such planes, ping-ponged between two buffers.  Here: the building blocks, and the collision of one node per
// lane that the FP64 build, FP16 and FP64 population storage, FP64 psi and single-phase fluids take (the
// energy passes of FP64 and FP16 storage: lbm_energy_f64.cuh, one kernel per Heun stage, and
// lbm_step_f16s.cuh).  The FP32 step: lbm_step_f32.cuh, lbm_flow_f32.cuh (collision with psi in its tiles),
// lbm_collide_f32.cuh (the arithmetic of both collisions), lbm_energy_f32.cuh.
//   k_rho_psi pull f with boundary substitutions, rho, psi(rho, T); writes psi.  Runs only
//             when neither an energy pass made psi nor the collision makes it (first step,
//             after a restore, warm-up).
//   k_collide per 32x8 tile: the pull window of the 9 planes (1-node halo) and the psi tile
//             (2-node halo) staged in shared memory by TMA (edge tiles: plain loads);
//             interaction force, gravity, CM collision; writes f*, rho, u.
//   kb_*      the same passes over the tiles of many domains in one launch per pass.
// The operation order inside each node follows the paper's equations term by term so
// that the FP64 build (compiled without FMA contraction) rounds like a plain reference;
// the FP32 build writes its roundings out (packed FP32x2 stencils, explicit fma) so that
// every kernel that inlines the same code gives the same bits.
#pragma once

#include <cuda_fp16.h>

#include <cstdint>

#include "lbm_internal.h"
#include "lbm_tma.cuh"

namespace lbm {
namespace kern {

// ---------------------------------------------------------------- programmatic dependent launch
// A pass launched with the programmatic-stream-serialization attribute may start while the
// kernel before it in the stream is still running (sm_90+).  wait(): the calling thread blocks
// until that kernel has completed and its writes are visible; trigger(): once every block of
// this pass has called it (or exited), the next such pass may start.  Both are no-ops in a
// pass launched without the attribute.  A pass reads nothing the previous kernel writes, and
// writes nothing at all, before wait().
namespace pdl {
__device__ __forceinline__ void wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
}  // namespace pdl

// ---------------------------------------------------------------- lattice tables
// D2Q9 velocities, Eq. (velVec).
__device__ __forceinline__ constexpr int cxv(int i) {
  return i == 1 || i == 5 || i == 7 ? 1 : (i == 2 || i == 6 || i == 8 ? -1 : 0);
}
__device__ __forceinline__ constexpr int cyv(int i) {
  return i == 3 || i == 5 || i == 8 ? 1 : (i == 4 || i == 6 || i == 7 ? -1 : 0);
}
__device__ __forceinline__ constexpr int oppv(int i) { return i == 0 ? 0 : (i % 2 == 1 ? i + 1 : i - 1); }
// The 24-neighbour stencil of Eq. (interForce) as 12 pairs (e, -e), with w(|e|^2).
__device__ __forceinline__ constexpr int exv(int k) {
  return k == 0 ? 1 : k == 1 ? 2 : k == 2 ? -2 : k == 3 ? -1 : k == 4 ? 0 : k == 5 ? 1 : k == 6 ? 2
       : k == 7 ? -2 : k == 8 ? -1 : k == 9 ? 0 : k == 10 ? 1 : 2;
}
__device__ __forceinline__ constexpr int eyv(int k) { return k < 2 ? 0 : (k < 7 ? 1 : 2); }
__device__ __forceinline__ constexpr double wiso(int k) {
  // |e|^2 = 1: 4/21, 2: 4/45, 4: 1/60, 5: 2/315, 8: 1/5040
  return (exv(k) * exv(k) + eyv(k) * eyv(k)) == 1 ? 4.0 / 21.0
       : (exv(k) * exv(k) + eyv(k) * eyv(k)) == 2 ? 4.0 / 45.0
       : (exv(k) * exv(k) + eyv(k) * eyv(k)) == 4 ? 1.0 / 60.0
       : (exv(k) * exv(k) + eyv(k) * eyv(k)) == 5 ? 2.0 / 315.0
       : 1.0 / 5040.0;
}

// Constants in the compute precision.
template <typename C>
__device__ __forceinline__ const PhysC<C>& pc(const Phys& ph);
template <>
__device__ __forceinline__ const PhysC<double>& pc<double>(const Phys& ph) {
  return ph.d;
}
template <>
__device__ __forceinline__ const PhysC<float>& pc<float>(const Phys& ph) {
  return ph.f;
}

// Division in the compute precision: IEEE in the FP64 build (which must round like the
// reference), the 2-ulp hardware approximation in the FP32 build.
template <typename C>
__device__ __forceinline__ C fdiv(C a, C b) {
  return a / b;
}
template <>
__device__ __forceinline__ float fdiv<float>(float a, float b) {
  return __fdividef(a, b);
}

// a / b with rb = 1 / b rounded to nearest.  FP64: q = a rb corrected by its exact remainder, which is
// the correctly rounded quotient (P. Markstein, IBM J. Res. Dev. 34, 1990; N. Brisebarre, J.-M. Muller,
// S. K. Raina, IEEE Trans. Comput. 53, 2004): 3 operations on the FP64 pipe instead of about 10 where
// the divisor is a constant or used more than once.  FP32: a / b as fdiv.
__device__ __forceinline__ double div_by(double a, double b, double rb) {
  const double q = __dmul_rn(a, rb);
  return __fma_rn(__fma_rn(-q, b, a), rb, q);
}
__device__ __forceinline__ float div_by(float a, float b, float) { return fdiv(a, b); }

// Sums and products whose rounding the source fixes, whatever kernel they are inlined into:
// FP32 fuses a b + c into one fma; FP64 rounds the product and the sum separately, as the
// FP64 build (compiled without contraction) does for every expression.
template <typename C>
__device__ __forceinline__ C mad(C a, C b, C c);
template <>
__device__ __forceinline__ float mad<float>(float a, float b, float c) {
  return __fmaf_rn(a, b, c);
}
template <>
__device__ __forceinline__ double mad<double>(double a, double b, double c) {
  return __dadd_rn(__dmul_rn(a, b), c);
}
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }

// ---------------------------------------------------------------- addressing
// Node coordinate of an arbitrary lattice position for stencil reads: periodic in y; in x
// periodic, or the nearest boundary column (zero-gradient ghost) at the inlet and outlet.
__device__ __forceinline__ int map_y(const Geo& g, int y) {
  if (y >= 0 && y < g.ny) return y;
  if (y < 0 && y + g.ny >= 0) return y + g.ny;
  if (y >= g.ny && y - g.ny < g.ny) return y - g.ny;
  y %= g.ny;  // only for lattices smaller than a tile
  return y < 0 ? y + g.ny : y;
}
__device__ __forceinline__ int map_x(const Geo& g, int x) {
  if (x >= 0 && x < g.nx) return x;
  if (g.periodic_x) {
    if (x < 0 && x + g.nx >= 0) return x + g.nx;
    if (x >= g.nx && x - g.nx < g.nx) return x - g.nx;
    x %= g.nx;
    return x < 0 ? x + g.nx : x;
  }
  return x < 0 ? 0 : g.nx - 1;
}
__device__ __forceinline__ int wrap_y(const Geo& g, int y) {  // offsets |dy| <= 2 < ny
  return y < 0 ? y + g.ny : (y >= g.ny ? y - g.ny : y);
}
// Population storage: FP64 or FP32 values as they are, or shifted FP16 h_i = f_i - w_i rho_l
// (the shift keeps liquid populations near zero, where FP16 is finest).
template <typename C, typename S>
struct PopIO {
  static __device__ __forceinline__ C ld(S v, int, const Phys&) { return static_cast<C>(v); }
  static __device__ __forceinline__ S st(C v, int, const Phys&) { return static_cast<S>(v); }
  static __device__ __forceinline__ double ld_d(S v, int, const Phys&) { return static_cast<double>(v); }
  static __device__ __forceinline__ S st_d(double v, int, const Phys&) { return static_cast<S>(v); }
};
template <typename C>
struct PopIO<C, __half> {
  static __device__ __forceinline__ C ld(__half v, int i, const Phys& ph) {
    return static_cast<C>(__half2float(v) + ph.pop_shift[i]);
  }
  static __device__ __forceinline__ __half st(C v, int i, const Phys& ph) {
    return __float2half_rn(static_cast<float>(v) - ph.pop_shift[i]);
  }
  static __device__ __forceinline__ double ld_d(__half v, int i, const Phys& ph) {
    return static_cast<double>(__half2float(v) + ph.pop_shift[i]);
  }
  static __device__ __forceinline__ __half st_d(double v, int i, const Phys& ph) {
    return __float2half_rn(static_cast<float>(v) - ph.pop_shift[i]);
  }
};
template <typename C, typename S>
__device__ __forceinline__ C ldf(const Geo& g, const Phys& ph, const S* __restrict__ f, int i, int y, int x) {
  return PopIO<C, S>::ld(f[i * g.plane + y * g.pitch + x], i, ph);
}

// ---------------------------------------------------------------- double-float arithmetic
// A double-float value is a pair (hi, lo) of FP32 words standing for the real number hi + lo.
// Building blocks: Knuth's TwoSum and Dekker's FastTwoSum (error-free sums), the FMA-based
// exact product, and products, sums and a quotient of pairs after Joldes, Muller and Popescu,
// "Tight and rigorous error bounds for basic building blocks of double-word arithmetic" (ACM
// TOMS 2017), here in their cheapest forms: results are left unnormalised (|lo| a few ulps of
// hi, never renormalised by a FastTwoSum), the lo * lo term of a product is dropped, and a
// difference uses FastTwoSum of the high words where the order of the operands is known.
// Square roots and the quotient start from the FP32 approximations (rsqrt.approx, rcp.approx)
// and take one correction from an exact residual (Karp and Markstein, "High-precision division
// and square root", ACM TOMS 1997).  Each result carries about 2^-44 relative error.
struct DF {
  float hi, lo;
};
__device__ __forceinline__ DF df_of(F2 v) { return {v.hi, v.lo}; }
__device__ __forceinline__ DF df_neg(DF a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// a * f for an FP32 f
__device__ __forceinline__ DF df_mulf(DF a, float f) {
  const float p = __fmul_rn(a.hi, f);
  return {p, __fmaf_rn(a.lo, f, __fmaf_rn(a.hi, f, -p))};
}
__device__ __forceinline__ DF df_mul(DF a, DF b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  return {p, __fmaf_rn(a.lo, b.hi, e)};
}
__device__ __forceinline__ DF df_sqr(DF a) {
  const float p = __fmul_rn(a.hi, a.hi);
  return {p, __fmaf_rn(__fadd_rn(a.hi, a.hi), a.lo, __fmaf_rn(a.hi, a.hi, -p))};
}
// c - a where |c.hi| >= |a.hi| (FastTwoSum of the high words)
__device__ __forceinline__ DF df_csub(DF c, DF a) {
  const float s = __fsub_rn(c.hi, a.hi);
  const float t = __fsub_rn(__fsub_rn(c.hi, s), a.hi);
  return {s, __fadd_rn(t, __fsub_rn(c.lo, a.lo))};
}
// c - a for an FP32 c with |c| >= |a.hi|
__device__ __forceinline__ DF df_fsub(float c, DF a) {
  const float s = __fsub_rn(c, a.hi);
  const float t = __fsub_rn(__fsub_rn(c, s), a.hi);
  return {s, __fsub_rn(t, a.lo)};
}
// a + b for any magnitudes (TwoSum of the high words)
__device__ __forceinline__ DF df_add(DF a, DF b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float bb = __fsub_rn(s, a.hi);
  const float t = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb));
  return {s, __fadd_rn(t, __fadd_rn(a.lo, b.lo))};
}
// a / b: q1 = a.hi / b.hi from the approximate reciprocal, then the exact remainder
// a - b q1 (a.hi - b.hi q1 is exact by Sterbenz's lemma) divided once more
__device__ __forceinline__ DF df_div(DF a, DF b) {
  const float r = rcp_approx(b.hi);
  const float q1 = __fmul_rn(a.hi, r);
  const float p = __fmul_rn(b.hi, q1);
  const float e = __fmaf_rn(b.lo, q1, __fmaf_rn(b.hi, q1, -p));
  const float d = __fadd_rn(__fsub_rn(a.hi, p), __fsub_rn(a.lo, e));
  return {q1, __fmul_rn(d, r)};
}
// sqrt(a): s = a.hi rsqrt(a.hi), corrected by (a - s^2) / (2 s) with the residual from one fma
__device__ __forceinline__ DF df_sqrt(DF a) {
  const float r = rsqrt_approx(a.hi);
  const float s = __fmul_rn(a.hi, r);
  const float res = __fadd_rn(__fmaf_rn(-s, s, a.hi), a.lo);
  return {s, __fmul_rn(res, __fmul_rn(0.5f, r))};
}

// ---------------------------------------------------------------- thermodynamics
// Peng-Robinson EOS, Eq. (eos), and psi of Eq. (potential) in IEEE FP64.
__device__ __forceinline__ double psi_eos(const Phys& ph, double rho, double T, double& rad) {
  const double cs2 = 1.0 / 3.0;
  const PhysC<double>& k = ph.d;
  double s = 1.0 + k.kappa * (1.0 - sqrt(div_by(T, k.Tc, ph.rTc)));
  double phi = s * s;
  double rep = rho * k.R * T / (1.0 - k.b * rho);
  double att = k.a * phi * rho * rho / (1.0 + 2.0 * k.b * rho - k.b * k.b * rho * rho);
  double p = rep - att;
  rad = div_by(2.0 * (p - rho * cs2), k.G * cs2, ph.rGc);
  return sqrt(rad);
}
// The same in double-float arithmetic (inputs and result FP32), over one denominator: with
// x = b rho and D = 1 + 2x - x^2 = 2 - (1 - x)^2,
//   rad = rho [kR T D - ka phi rho (1 - x) - (k/3)(1 - x) D] / ((1 - x) D),  k = 2/(G cs^2),
//   phi = (K1 - kappa sqrt(T/Tc))^2,  K1 = 1 + kappa
// (kR, ka, k/3, K1 folded on the host).  The numerator has condition number ~2 over the
// liquid-vapour range, so the cheap sums above keep the radicand within ~2^-42 of exact; psi
// is then the correctly rounded FP32 value (checked on 20,000 sampled (rho, T) against a
// 120-bit evaluation in a CPU emulation of these operations).  The FastTwoSum differences need
// kappa sqrt(T/Tc) <= 1 + kappa (T <= 3.5 Tc) and b rho <= 1, which hold wherever Eq. (eos) is
// defined on the lattice.
__device__ __forceinline__ float psi_eos_df(const Phys& ph, float rho, float T, float& rad_hi) {
  const DF sq = df_sqrt(df_mulf(df_of(ph.invTc2), T));
  const DF phi = df_sqr(df_csub(df_of(ph.K12), df_mul(df_of(ph.kappa2), sq)));
  const DF omx = df_fsub(1.0f, df_mulf(df_of(ph.b2), rho));
  const DF D = df_fsub(2.0f, df_sqr(omx));
  const DF den = df_mul(omx, D);
  const DF A = df_mul(df_mulf(df_of(ph.kR2), T), D);
  const DF B = df_mul(df_mulf(df_mul(df_of(ph.ka2), phi), rho), omx);
  const DF num = df_add(df_add(A, df_neg(B)), df_neg(df_mul(df_of(ph.k32), den)));
  const DF rad = df_div(df_mulf(num, rho), den);
  rad_hi = rad.hi;
  const DF r = df_sqrt(rad);
  return __fadd_rn(r.hi, r.lo);
}
// The same in plain FP32 (its FMA contraction is the compiler's; the tests hold its routes to equal bits).
__device__ __forceinline__ float psi_eos_f32(const Phys& ph, float rho, float T, float& rad) {
  float s = 1.0f + ph.kappa2.hi * (1.0f - sqrtf(T * ph.invTc2.hi));
  float phi = s * s;
  float b = ph.b2.hi;
  float rep = rho * ph.R2.hi * T / (1.0f - b * rho);
  float att = ph.a2.hi * phi * rho * rho / (1.0f + 2.0f * b * rho - b * b * rho * rho);
  rad = (rep - att - rho * ph.cs22.hi) * ph.k2.hi;
  return sqrtf(rad);
}
template <typename C, int PSI>
__device__ __forceinline__ C psi_of(const Phys& ph, C rho, C T, int* status) {
  if constexpr (PSI == kPsiDF) {
    float rad;
    float p = psi_eos_df(ph, (float)rho, (float)T, rad);
    if (!(rad > 0.0f)) atomicOr(status, 2);
    return (C)p;
  } else if constexpr (PSI == kPsiF32) {
    float rad;
    float p = psi_eos_f32(ph, (float)rho, (float)T, rad);
    if (!(rad > 0.0f)) atomicOr(status, 2);
    return (C)p;
  } else {
    double rad;
    double p = psi_eos(ph, (double)rho, (double)T, rad);
    if (!(rad > 0.0)) atomicOr(status, 2);
    return (C)p;
  }
}
// Phase fraction for the transport properties, and nu(rho), lambda(rho).
template <typename C>
__device__ __forceinline__ C phase_frac(const Phys& ph, C rho) {
  if (!(pc<C>(ph).rho_l > pc<C>(ph).rho_v)) return C(1);
  C f = div_by(sub(rho, pc<C>(ph).rho_v), sub(pc<C>(ph).rho_l, pc<C>(ph).rho_v), C(ph.rdr));
  f = f < C(0) ? C(0) : f;
  return f > C(1) ? C(1) : f;
}
template <typename C>
__device__ __forceinline__ C nu_of(const Phys& ph, C rho) {
  return mad(phase_frac(ph, rho), sub(pc<C>(ph).nu_l, pc<C>(ph).nu_v), pc<C>(ph).nu_v);
}
template <typename C>
__device__ __forceinline__ C lam_of(const Phys& ph, C rho) {
  C alpha = mad(phase_frac(ph, rho), sub(pc<C>(ph).alpha_l, pc<C>(ph).alpha_v), pc<C>(ph).alpha_v);
  return mul(mul(rho, pc<C>(ph).c_v), alpha);
}

// theta = T - T_sat of a temperature stored in FP32, which the FP32 energy pass and its adjoint work with.  The
// stored T_wall and T_sat stand for their FP64 values: their rounding to FP32 would reach the heat flux as a
// constant error (up to 1e-5 of it at a superheat of 0.01 T_c).  Other wall temperatures, of a profile
// along the wall or of a restored state, keep their rounding.
__device__ __forceinline__ float theta_of(const StepConst& k, float T) {
  if (T == k.T_wall) return k.th_wall;
  const float t = __fsub_rn(T, k.T_sat);
  return t == 0.0f ? 0.0f : __fsub_rn(t, k.dT_sat);
}

// ---------------------------------------------------------------- stencils on tiles (Sec. II.C)
// p points at the stencil centre of a row-major tile with row stride s.
// Isotropic gradient sum_k w_k phi(x+e_k) e_k over +/- pairs.
template <typename C, bool kX = true, bool kY = true>
__device__ __forceinline__ void grad_t(const C* p, int s, C& gx, C& gy) {
  C sx = C(0), sy = C(0);
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const int ex = exv(k), ey = eyv(k);
    if ((kX && ex != 0) || (kY && ey != 0)) {
      // w e is w scaled by a power of two: (w e) d rounds exactly like (w d) e
      C d = sub(p[ey * s + ex], p[-ey * s - ex]);
      if (kX && ex != 0) sx = mad(C(wiso(k) * ex), d, sx);
      if (kY && ey != 0) sy = mad(C(wiso(k) * ey), d, sy);
    }
  }
  gx = sx;
  gy = sy;
}
// ---------------------------------------------------------------- packed FP32 pairs and their stencils
// The FP32 kernels handle two x-adjacent nodes per lane as one packed float2 (sm_100+ FFMA2, FADD2,
// FMUL2: half the instructions, the same lane throughput).  Stencils fold a window row (columns
// -2 .. 3 around the pair) into sums and differences over +/-1 and +/-2 columns, which every stencil
// of the 25-point neighbourhood then takes its share of.
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.0f), a); }
__device__ __forceinline__ float2 nabs2(float2 a) {
  return make_float2(__uint_as_float(__float_as_uint(a.x) | 0x80000000u),
                     __uint_as_float(__float_as_uint(a.y) | 0x80000000u));
}
__device__ __forceinline__ float2 rcp2(float2 a) { return make_float2(rcp_approx(a.x), rcp_approx(a.y)); }

// One window row of a column pair: the pair, and per node the difference and sum of its neighbours
// at +/-1 (X1, S1) and +/-2 (X2, S2) columns.  q: the row's first window element (columns -2, -1).
struct RowSums {
  float2 c, X1, X2, S1, S2;
};
template <bool kX, bool kS>
__device__ __forceinline__ RowSums row_sums(const float2* q) {
  const float2 a = q[0], b = q[1], d = q[2];
  RowSums r;
  r.c = b;
  if (kX) {
    r.X1 = make_float2(__fsub_rn(b.y, a.y), __fsub_rn(d.x, b.x));
    r.X2 = sub2(d, a);
  }
  if (kS) {
    r.S1 = make_float2(__fadd_rn(b.y, a.y), __fadd_rn(d.x, b.x));
    r.S2 = add2(d, a);
  }
  return r;
}
// Stencil weights by row distance k = |d|: of the pair (k, column offset 0, +/-1, +/-2).
__device__ __forceinline__ constexpr float wrow(int k, int c) {
  const int e = k * k + c * c;
  return e == 1 ? float(4.0 / 21.0) : e == 2 ? float(4.0 / 45.0) : e == 4 ? float(1.0 / 60.0)
       : e == 5 ? float(2.0 / 315.0) : e == 8 ? float(1.0 / 5040.0) : 0.0f;
}
// gx += the row's share of sum w e_x phi(x + e), at row distance k
__device__ __forceinline__ void row_gx(const RowSums& r, int k, float2& gx) {
  gx = fma2(f2(wrow(k, 1)), r.X1, fma2(f2(2.0f * wrow(k, 2)), r.X2, gx));
}
// gy += the row's share of sum w e_y phi(x + e), at row offset d != 0
__device__ __forceinline__ void row_gy(const RowSums& r, int d, float2& gy) {
  const int k = d < 0 ? -d : d;
  gy = fma2(f2(d * wrow(k, 0)), r.c, fma2(f2(d * wrow(k, 1)), r.S1, fma2(f2(d * wrow(k, 2)), r.S2, gy)));
}

// The isotropic gradient of a column pair from the window rows -2 .. 2 (q: columns -2, -1 of the
// middle row, row stride ts), and of one node from a 5x5 window (row-major, centre w[12]) with the
// same roundings.  Rows are subtracted before they are weighted: exactly zero on a uniform field.
__device__ __forceinline__ void grad_rows(const float2* q, int ts, float2& gx, float2& gy) {
  gx = gy = f2(0.0f);
  RowSums lo = row_sums<true, true>(q - 2 * ts), hi = row_sums<true, true>(q + 2 * ts);
  row_gx(lo, 2, gx);
  row_gx(hi, 2, gx);
  gy = fma2(f2(2.0f * wrow(2, 0)), sub2(hi.c, lo.c),
            fma2(f2(2.0f * wrow(2, 1)), sub2(hi.S1, lo.S1), fma2(f2(2.0f * wrow(2, 2)), sub2(hi.S2, lo.S2), gy)));
  lo = row_sums<true, true>(q - ts);
  hi = row_sums<true, true>(q + ts);
  row_gx(lo, 1, gx);
  row_gx(hi, 1, gx);
  gy = fma2(f2(wrow(1, 0)), sub2(hi.c, lo.c),
            fma2(f2(wrow(1, 1)), sub2(hi.S1, lo.S1), fma2(f2(wrow(1, 2)), sub2(hi.S2, lo.S2), gy)));
  row_gx(row_sums<true, false>(q), 0, gx);
}
__device__ __forceinline__ void grad_window(const float* w, int s, float& gx, float& gy) {
  gx = gy = 0.0f;
#pragma unroll
  for (int k = 2; k >= 0; --k) {
#pragma unroll
    for (int t = 0; t < (k ? 2 : 1); ++t) {
      const float* q = w + s * (t ? 2 + k : 2 - k);
      gx = __fmaf_rn(wrow(k, 1), __fsub_rn(q[3], q[1]), __fmaf_rn(2.0f * wrow(k, 2), __fsub_rn(q[4], q[0]), gx));
    }
    if (k == 0) continue;
    const float *a = w + s * (2 - k), *b = w + s * (2 + k);
    gy = __fmaf_rn(k * wrow(k, 0), __fsub_rn(b[2], a[2]),
                   __fmaf_rn(k * wrow(k, 1), __fsub_rn(__fadd_rn(b[3], b[1]), __fadd_rn(a[3], a[1])),
                             __fmaf_rn(k * wrow(k, 2), __fsub_rn(__fadd_rn(b[4], b[0]), __fadd_rn(a[4], a[0])), gy)));
  }
}

// ---------------------------------------------------------------- streaming (Sec. IV.A BCs)
// Link fraction q of direction i at a near-wall node: the fraction of the link from the node
// along -c_i that lies in the fluid (smallest root of |d + t c|^2 = r^2, tabulated at creation).
template <typename C>
__device__ __forceinline__ C link_q(const Geo& g, int x, int y, int i) {
  return static_cast<const C*>(g.wall_q)[g.wall_idx[y * g.pitch + x] * 8 + i - 1];
}

// Substitutions of the pull for nodes next to the wall, the inlet or the outlet, on the plainly pulled
// fo: linear interpolated bounce-back on the cylinder, Zou-He inlet, convective outlet.  at(i, dx, dy):
// population i at the node (x + dx, y + dy), |dx|, |dy| <= 1, inside the lattice.  The table of link
// fractions tells which links meet the wall (no node types are read), so the loads of a node wait
// for two others at most.  side_out != nullptr: store the outlet's new streamed values there.
template <typename C, typename At>
__device__ __forceinline__ void pull_special(const Geo& g, const Phys& ph, const C* __restrict__ side_in,
                                             C* __restrict__ side_out, int x, int y, uint8_t m, C fo[9], const At& at) {
  if (m & kNearWall) {
    const C* wq = static_cast<const C*>(g.wall_q) + g.wall_idx[y * g.pitch + x] * 8 - 1;
    C lq[9];
#pragma unroll
    for (int i = 1; i < 9; ++i) lq[i] = wq[i];
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      // the wall lies along c_opp(i); its link fraction is -1 where the pull's source is fluid
      const int io = oppv(i);
      const C q = lq[i];
      if (q >= C(0)) {
        const C a = at(io, 0, 0);
        const C q2 = mul(C(2), q);
        if (q < C(0.5)) {
          const int nxp = x + cxv(i);
          const bool ok = lq[io] < C(0) && (g.periodic_x || (nxp >= 0 && nxp < g.nx));
          fo[i] = ok ? add(mul(q2, a), mul(sub(C(1), q2), at(io, cxv(i), cyv(i)))) : a;
        } else {
          fo[i] = add(fdiv(a, q2), mul(fdiv(sub(q2, C(1)), q2), at(i, 0, 0)));
        }
      }
    }
  }
  if (g.periodic_x) return;
  if (x == 0) {
    // Zou-He velocity inlet, u = (u_in, 0): unknowns f1, f5, f7
    const C u = pc<C>(ph).u_in;
    const C rho = fdiv(add(add(add(fo[0], fo[3]), fo[4]), mul(C(2), add(add(fo[2], fo[6]), fo[8]))), sub(C(1), u));
    fo[1] = add(fo[2], mul(mul(C(2.0 / 3.0), rho), u));
    fo[5] = add(sub(fo[6], mul(C(0.5), sub(fo[3], fo[4]))), fdiv(mul(rho, u), C(6)));
    fo[7] = add(add(fo[8], mul(C(0.5), sub(fo[3], fo[4]))), fdiv(mul(rho, u), C(6)));
  }
  if (x == g.nx - 1) {
    // convective outlet: f(t+1) = (f(t) + U f_{nx-2}(t+1)) / (1 + U) for f2, f6, f8.  FP32 takes
    // the same update as f(t) + k (f_{nx-2}(t+1) - f(t)), k = U / (1 + U) rounded once from FP64:
    // the quotient with 1 + U rounded to FP32 has its fixed point about 1e-6 above the interior
    // value, a steady mass source at the outlet that shifts the open domain's pressure level over
    // long runs (the FP64 build keeps the quotient, term for term as written)
    const C U = pc<C>(ph).U_out;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int i = j == 0 ? 2 : (j == 1 ? 6 : 8);
      const C inner = at(i, 0, -cyv(i));
      const C s0 = side_in[j * g.ny + y];
      C v;
      if constexpr (sizeof(C) == 4) v = mad(pc<C>(ph).U_k, sub(inner, s0), s0);
      else v = fdiv(add(s0, mul(U, inner)), add(C(1), U));
      fo[i] = v;
      if (side_out) side_out[j * g.ny + y] = v;
    }
  }
}

// rho = sum_i f_i of pulled populations: in pairs of opposite directions in FP32 (whose moments use
// the same sums), in the order of the index in FP64, as the reference does, and with FP16 storage.
template <typename C, typename S>
__device__ __forceinline__ C pop_sum(const C f[9]) {
  if constexpr (sizeof(C) == 4 && sizeof(S) != 2) {
    return add(add(f[0], add(add(f[1], f[2]), add(f[3], f[4]))), add(add(f[5], f[6]), add(f[7], f[8])));
  } else {
    C r = f[0];
#pragma unroll
    for (int i = 1; i < 9; ++i) r = r + f[i];
    return r;
  }
}

template <typename C, typename S>
__device__ __forceinline__ void pull_node(const Geo& g, const Phys& ph, const S* __restrict__ f,
                                          const uint8_t* __restrict__ mask, const C* __restrict__ side_in,
                                          C* __restrict__ side_out, int x, int y, uint8_t m, C fo[9]) {
  // the plain pulls are issued before the node type is tested (columns clamped at an open
  // edge), so they overlap the mask read; wall and edge nodes then redo the pull
  const int ym = y == 0 ? g.ny - 1 : y - 1;
  const int yp = y == g.ny - 1 ? 0 : y + 1;
  int xm = x - 1, xp = x + 1;
  if (g.periodic_x) {
    xm = xm < 0 ? g.nx - 1 : xm;
    xp = xp >= g.nx ? 0 : xp;
  } else {
    xm = xm < 0 ? 0 : xm;
    xp = xp >= g.nx ? g.nx - 1 : xp;
  }
  fo[0] = ldf<C>(g, ph, f, 0, y, x);
  fo[1] = ldf<C>(g, ph, f, 1, y, xm);
  fo[2] = ldf<C>(g, ph, f, 2, y, xp);
  fo[3] = ldf<C>(g, ph, f, 3, ym, x);
  fo[4] = ldf<C>(g, ph, f, 4, yp, x);
  fo[5] = ldf<C>(g, ph, f, 5, ym, xm);
  fo[6] = ldf<C>(g, ph, f, 6, yp, xp);
  fo[7] = ldf<C>(g, ph, f, 7, yp, xm);
  fo[8] = ldf<C>(g, ph, f, 8, ym, xp);
  const bool edge = !g.periodic_x && (x == 0 || x == g.nx - 1);
  if ((m & kNearWall) || edge) {
    auto at = [&](int i, int dx, int dy) {
      int sx = x + dx;
      if (g.periodic_x) sx = sx < 0 ? sx + g.nx : (sx >= g.nx ? sx - g.nx : sx);
      return ldf<C>(g, ph, f, i, wrap_y(g, y + dy), sx);
    };
    pull_special<C>(g, ph, side_in, side_out, x, y, m, fo, at);
  }
}

// psi at node (x, y): pull, rho = sum f, Eq. (potential); solid nodes use rho_s.
template <typename C, typename S, int PSI>
__device__ __forceinline__ C psi_node(const Geo& g, const Phys& ph, const S* __restrict__ f,
                                      const C* __restrict__ T, const uint8_t* __restrict__ mask,
                                      const C* __restrict__ side_in, int x, int y, int* status) {
  const int id = y * g.pitch + x;
  const uint8_t m = mask[id];
  const C t = T[id];
  C rho = pc<C>(ph).rho_s;
  if (!(m & kSolid)) {
    C fo[9];
    pull_node<C, S>(g, ph, f, mask, side_in, nullptr, x, y, m, fo);
    rho = pop_sum<C, S>(fo);
  }
  return psi_of<C, PSI>(ph, rho, t, status);
}

}  // namespace kern
}  // namespace lbm
#include "lbm_collide_f32.cuh"
namespace lbm {
namespace kern {

// ---------------------------------------------------------------- CM collision (Sec. II.A-B)
// Raw moments -> central moments k4, k5 (T = N M), post-collision CMs of Eq. (postColl2),
// m* = N(u)^{-1} k* by forward substitution, f* = M^{-1} m*.  Closed form of the 9x9
// algebra, sums in the order of the matrix products.  FP64: products by powers of two are exact, so
// they are moved out of the rounded products or into an FMA with the sum, with the same result.
template <typename C>
__device__ __forceinline__ void collide(const C f[9], C rho, C Fx, C Fy, C Fmx, C Fmy, C psi, C omega, C sigma,
                                        C fs[9], C& ux, C& uy);
template <>
__device__ __forceinline__ void collide<double>(const double f[9], double rho, double Fx, double Fy, double Fmx,
                                                double Fmy, double psi, double omega, double sigma, double fs[9],
                                                double& ux, double& uy) {
  const double m1 = ((((f[1] - f[2]) + f[5]) - f[6]) + f[7]) - f[8];
  const double m2 = ((((f[3] - f[4]) + f[5]) - f[6]) - f[7]) + f[8];
  const double m4 = ((f[1] + f[2]) - f[3]) - f[4];
  const double m5 = ((f[5] + f[6]) - f[7]) - f[8];
  const double ir = 1.0 / rho;
  ux = div_by(__fma_rn(0.5, Fx, m1), rho, ir);
  uy = div_by(__fma_rn(0.5, Fy, m2), rho, ir);
  const double u = ux, v = uy;
  // entries of the shift matrix N(u), App. A, up to sign and powers of two
  const double uu = u * u, vv = v * v, uv = u * v, s2 = uu + vv, d2 = uu - vv, uuv = uu * v, uvv = uv * v;
  const double k4 = __fma_rn(2.0, v * m2, __fma_rn(-2.0, u * m1, d2 * rho)) + m4;
  const double k5 = ((uv * rho - v * m1) - u * m2) + m5;
  // post-collision central moments
  const double alpha = sigma != 0.0 ? sigma / (psi * psi) : 0.0;
  const double Fm2 = Fmx * Fmx + Fmy * Fmy;
  const double ks3 = 2.0 * (div_by(rho, 3.0, 1.0 / 3.0) + alpha * Fm2);
  const double ks4 = (1.0 - omega) * k4;
  const double ks5 = (1.0 - omega) * k5;
  const double fy3 = div_by(Fy, 3.0, 1.0 / 3.0), fx3 = div_by(Fx, 3.0, 1.0 / 3.0);
  const double ks8 = __fma_rn(0.5, (4.0 / 3.0) * alpha * Fm2, div_by(rho, 9.0, 1.0 / 9.0));
  // forward substitution N m* = k*
  const double ms0 = rho;
  const double ms1 = __fma_rn(0.5, Fx, u * ms0);
  const double ms2 = __fma_rn(0.5, Fy, v * ms0);
  const double p1 = u * ms1, p2 = v * ms2;
  const double ms3 = __fma_rn(2.0, p2, __fma_rn(2.0, p1, ks3 - s2 * ms0));
  const double ms4 = __fma_rn(-2.0, p2, __fma_rn(2.0, p1, ks4 - d2 * ms0));
  const double ms5 = ((ks5 - uv * ms0) + v * ms1) + u * ms2;
  double t = __fma_rn(0.5, fy3, uuv * ms0);
  t = __fma_rn(-2.0, uv * ms1, t) - uu * ms2;
  t = __fma_rn(0.5, v * ms4, __fma_rn(0.5, v * ms3, t));
  const double ms6 = __fma_rn(2.0, u * ms5, t);
  t = __fma_rn(0.5, fx3, uvv * ms0);
  t = __fma_rn(-2.0, uv * ms2, t - vv * ms1);
  t = __fma_rn(-0.5, u * ms4, __fma_rn(0.5, u * ms3, t));
  const double ms7 = __fma_rn(2.0, v * ms5, t);
  t = ks8 - uuv * v * ms0;
  t = __fma_rn(2.0, uuv * ms2, __fma_rn(2.0, uvv * ms1, t));
  t = __fma_rn(0.5, d2 * ms4, __fma_rn(-0.5, s2 * ms3, t));
  t = __fma_rn(2.0, v * ms6, __fma_rn(-4.0, uv * ms5, t));
  const double ms8 = __fma_rn(2.0, u * ms7, t);
  // f* = M^{-1} m*
  const double h1 = 0.5 * ms1, h2 = 0.5 * ms2, q5 = 0.25 * ms5;
  auto axis = [&](double a, double s34, double s6) {  // ((a + ms3 / 4) +/- ms4 / 4) +/- ms_6,7 / 2) - ms8 / 2
    return __fma_rn(-0.5, ms8, __fma_rn(0.5, s6, __fma_rn(s34, ms4, __fma_rn(0.25, ms3, a))));
  };
  auto diag = [&](double a, double s6, double s7) {
    return __fma_rn(0.25, ms8, __fma_rn(s7, ms7, __fma_rn(s6, ms6, a)));
  };
  fs[0] = (ms0 - ms3) + ms8;
  fs[1] = axis(h1, 0.25, -ms7);
  fs[2] = axis(-h1, 0.25, ms7);
  fs[3] = axis(h2, -0.25, -ms6);
  fs[4] = axis(-h2, -0.25, ms6);
  fs[5] = diag(q5, 0.25, 0.25);
  fs[6] = diag(q5, -0.25, -0.25);
  fs[7] = diag(-q5, -0.25, 0.25);
  fs[8] = diag(-q5, 0.25, -0.25);
}
// Single-rate BGK on the same equilibrium and forcing, the operator the paper compares the CM
// collision with (Sec. III.B): f* = f + omega (f^eq - f) + (1 - omega/2) F_i, u as above.  T(u) =
// N(u) M is linear and maps f^eq and F_i to k^eq = (rho, 0, 0, 2 rho/3, 0, 0, 0, 0, rho/9) and
// R = (0, F_x, F_y, 0, 0, 0, F_y/3, F_x/3, 0), so f* = (1 - omega) f + M^{-1} N(u)^{-1} k' with
// k' = omega k^eq + (1 - omega/2) R: the forward substitution and reconstruction of the CM
// collision on k'.  No consistency term (it belongs to the CM forcing of Eq. (force2)).
template <typename C>
__device__ __forceinline__ void collide_bgk(const C f[9], C rho, C Fx, C Fy, C omega, C fs[9], C& ux, C& uy) {
  const C m1 = ((((f[1] - f[2]) + f[5]) - f[6]) + f[7]) - f[8];
  const C m2 = ((((f[3] - f[4]) + f[5]) - f[6]) - f[7]) + f[8];
  ux = fdiv(m1 + C(0.5) * Fx, rho);
  uy = fdiv(m2 + C(0.5) * Fy, rho);
  const C u = ux, v = uy;
  // shift matrix N(u), App. A
  const C N10 = -u, N20 = -v;
  const C N30 = u * u + v * v, N31 = C(-2) * u, N32 = C(-2) * v;
  const C N40 = u * u - v * v, N41 = C(-2) * u, N42 = C(2) * v;
  const C N50 = u * v, N51 = -v, N52 = -u;
  const C N60 = -u * u * v, N61 = C(2) * u * v, N62 = u * u, N63 = -v / C(2), N64 = -v / C(2), N65 = C(-2) * u;
  const C N70 = -u * v * v, N71 = v * v, N72 = C(2) * u * v, N73 = -u / C(2), N74 = u / C(2), N75 = C(-2) * v;
  const C N80 = u * u * v * v, N81 = C(-2) * u * v * v, N82 = C(-2) * u * u * v, N83 = (u * u + v * v) / C(2),
          N84 = -(u * u - v * v) / C(2), N85 = C(4) * u * v, N86 = C(-2) * v, N87 = C(-2) * u;
  const C cf = C(1) - C(0.5) * omega;
  const C ks0 = omega * rho;
  const C ks1 = cf * Fx;
  const C ks2 = cf * Fy;
  const C ks3 = omega * div_by(C(2) * rho, C(3), C(1.0 / 3.0));
  const C ks6 = cf * div_by(Fy, C(3), C(1.0 / 3.0));
  const C ks7 = cf * div_by(Fx, C(3), C(1.0 / 3.0));
  const C ks8 = omega * div_by(rho, C(9), C(1.0 / 9.0));
  // forward substitution N m' = k' (k'_4 = k'_5 = 0)
  const C ms0 = ks0;
  const C ms1 = ks1 - N10 * ms0;
  const C ms2 = ks2 - N20 * ms0;
  const C ms3 = ((ks3 - N30 * ms0) - N31 * ms1) - N32 * ms2;
  const C ms4 = ((-N40 * ms0) - N41 * ms1) - N42 * ms2;
  const C ms5 = ((-N50 * ms0) - N51 * ms1) - N52 * ms2;
  const C ms6 = (((((ks6 - N60 * ms0) - N61 * ms1) - N62 * ms2) - N63 * ms3) - N64 * ms4) - N65 * ms5;
  const C ms7 = (((((ks7 - N70 * ms0) - N71 * ms1) - N72 * ms2) - N73 * ms3) - N74 * ms4) - N75 * ms5;
  const C ms8 =
      (((((((ks8 - N80 * ms0) - N81 * ms1) - N82 * ms2) - N83 * ms3) - N84 * ms4) - N85 * ms5) - N86 * ms6) - N87 * ms7;
  // f* = (1 - omega) f + M^{-1} m'
  const C h = C(0.5), q = C(0.25), r = C(1) - omega;
  fs[0] = r * f[0] + ((ms0 - ms3) + ms8);
  fs[1] = r * f[1] + ((((h * ms1 + q * ms3) + q * ms4) - h * ms7) - h * ms8);
  fs[2] = r * f[2] + ((((-h * ms1 + q * ms3) + q * ms4) + h * ms7) - h * ms8);
  fs[3] = r * f[3] + ((((h * ms2 + q * ms3) - q * ms4) - h * ms6) - h * ms8);
  fs[4] = r * f[4] + ((((-h * ms2 + q * ms3) - q * ms4) + h * ms6) - h * ms8);
  fs[5] = r * f[5] + (((q * ms5 + q * ms6) + q * ms7) + q * ms8);
  fs[6] = r * f[6] + (((q * ms5 - q * ms6) - q * ms7) + q * ms8);
  fs[7] = r * f[7] + (((-q * ms5 - q * ms6) + q * ms7) + q * ms8);
  fs[8] = r * f[8] + (((-q * ms5 + q * ms6) - q * ms7) + q * ms8);
}

// ---------------------------------------------------------------- k_rho_psi, k_collide
constexpr int kCollTX = 32, kCollTY = 8;

// psi(rho, T) at every node of tile (bx, by) of 32 x 8 nodes (rho from the pulled
// populations, rho_s in the solid).
template <typename C, typename S, int PSI>
__device__ __forceinline__ void rho_psi_tile(const Geo& g, const Phys& ph, const S* __restrict__ f,
                                             const C* __restrict__ T, const uint8_t* __restrict__ mask,
                                             const C* __restrict__ side_in, C* __restrict__ psi_o, int* status, int bx,
                                             int by) {
  const int x = bx * kCollTX + threadIdx.x, y = by * 8 + threadIdx.y;
  if (x >= g.nx || y >= g.ny) return;
  psi_o[y * g.pitch + x] = psi_node<C, S, PSI>(g, ph, f, T, mask, side_in, x, y, status);
}
// Blocks per SM (FP32 arithmetic): left alone the compiler takes 48 registers with FP16 and 46 with FP64 storage, and
// fewer pulls are in flight: 68 and 99 us at 3000 x 2000 against 58 (7 blocks) and 97 (6).
template <typename C, typename S, int PSI>
__global__ void __launch_bounds__(256, sizeof(C) == 8 ? 1 : sizeof(S) == 2 ? 7 : 6) k_rho_psi(Geo g, Phys ph, const S* __restrict__ f, const C* __restrict__ T,
                                                const uint8_t* __restrict__ mask, const C* __restrict__ side_in,
                                                C* __restrict__ psi_o, int* status) {
  rho_psi_tile<C, S, PSI>(g, ph, f, T, mask, side_in, psi_o, status, blockIdx.x, blockIdx.y);
}

// Shared-memory staging of a collision tile.  Populations: the tile's rows with a 1-row halo,
// columns from x0 - XA (XA elements = 16 bytes, the alignment of a TMA copy's first column);
// psi: a 2-row and PA-column halo.  Tiles whose staged boxes lie inside the lattice (no wrap,
// no open edge) are copied by TMA; the others load psi and pull with plain loads.
template <typename C, typename S, int CTY>
struct CollStage {
  static constexpr int XA = 16 / (int)sizeof(S), FW = kCollTX + 2 * XA, FH = CTY + 2;
  static constexpr int PA = 16 / (int)sizeof(C) < 2 ? 2 : 16 / (int)sizeof(C), PW = kCollTX + 2 * PA, PH = CTY + 4;
  static constexpr int MARGIN = XA > PA ? XA : PA;  // columns a staged tile needs left and right of it
};
template <typename C, typename S, int CTY>
__device__ __forceinline__ bool coll_staged(const Geo& g, int x0, int y0) {
  constexpr int M = CollStage<C, S, CTY>::MARGIN;
  return x0 >= M && x0 + kCollTX + M <= g.nx && y0 >= 2 && y0 + CTY + 2 <= g.ny;
}

// One fluid-or-solid node (x, y) = (x0 + tx, y0 + ty) of a collision tile, mask m: pull (from
// the staged populations s_f of a staged tile, else from global memory with the boundary
// substitutions), interaction force from the psi tile s_psi with its 2-node halo, gravity,
// CM collision (or, with OP = kCollBGK, the BGK comparison operator); writes f* (other
// buffer), rho, u and the outlet's streamed values.
// FP32 arithmetic over FP32 or FP64 populations takes the operations of lbm_collide_f32.cuh, with the bits of the
// column pairs of lbm_flow_f32.cuh.
template <typename C, typename S, int CTY, int OP = kCollCM>
__device__ __forceinline__ void collide_node(const Geo& g, const Phys& ph, const S* __restrict__ f,
                                             S* __restrict__ fn, const C* __restrict__ psi,
                                             const uint8_t* __restrict__ mask, const C* __restrict__ side_in,
                                             C* __restrict__ side_out, C* __restrict__ rho_o, C* __restrict__ ux_o,
                                             C* __restrict__ uy_o, int forcing, int* status, int tx, int ty, int x,
                                             int y, uint8_t m, bool staged, const S* s_f, const C* s_psi,
                                             C* __restrict__ lam_o) {
  using CS = CollStage<C, S, CTY>;
  constexpr int HX = CS::PW;
  const PhysC<C>& k = pc<C>(ph);
  const int id = y * g.pitch + x;
  if (m & kSolid) {
    rho_o[id] = k.rho_s;
    ux_o[id] = C(0);
    uy_o[id] = C(0);
    if (sizeof(C) == 8 && lam_o) lam_o[id] = lam_of(ph, k.rho_s);
    return;
  }
  const bool multiphase = k.G != C(0);
  const bool need_psi = multiphase && forcing;
  C fo[9];
  if (staged) {
#pragma unroll
    for (int i = 0; i < 9; ++i)
      fo[i] = PopIO<C, S>::ld(s_f[(i * CS::FH + ty + 1 - cyv(i)) * CS::FW + tx + CS::XA - cxv(i)], i, ph);
    if (m & kNearWall) {  // a staged tile holds no edge column
      const S* q = s_f + (ty + 1) * CS::FW + tx + CS::XA;
      pull_special<C>(g, ph, side_in, side_out, x, y, m, fo, [&](int i, int dx, int dy) {
        return PopIO<C, S>::ld(q[(i * CS::FH + dy) * CS::FW + dx], i, ph);
      });
    }
  } else {
    pull_node<C, S>(g, ph, f, mask, side_in, side_out, x, y, m, fo);
  }
  const int pc0 = (ty + 2) * HX + tx + CS::PA;  // this node in the psi tile
  if constexpr (sizeof(C) == 4 && sizeof(S) != 2) {
    const Moments<float> M = moments_of(fo);
    float Fx = 0.0f, Fy = 0.0f, aF = 0.0f, ux, uy;
    if (forcing) {
      float gx = 0.0f, gy = 0.0f, psi0 = 0.0f;
      if (multiphase) {
        psi0 = s_psi[pc0];
        grad_window(&s_psi[pc0] - 2 * HX - 2, HX, gx, gy);
        aF = mul2(ph.sc.sg, fma2(gx, gx, mul2(gy, gy)));
      }
      force_of(ph, M.rho, psi0, gx, gy, Fx, Fy);
    }
    auto out = [&](int i, float v) { fn[i * g.plane + id] = PopIO<C, S>::st(v, i, ph); };
    if constexpr (OP == kCollBGK) collide_bgk_of(ph.sc, fo, M, Fx, Fy, ux, uy, out);
    else collide_cm(ph.sc, M, Fx, Fy, aF, ux, uy, out);
    rho_o[id] = M.rho;
    ux_o[id] = ux;
    uy_o[id] = uy;
    if (!(M.rho > 0.0f) || !(ux == ux) || !(uy == uy)) atomicOr(status, 1);
    return;
  }
  C rho = fo[0];
#pragma unroll
  for (int i = 1; i < 9; ++i) rho = rho + fo[i];
  const C cs2 = C(1.0 / 3.0);
  C Fmx = C(0), Fmy = C(0), Fx = C(0), Fy = C(0), psi0 = C(0);
  if (multiphase) psi0 = need_psi ? s_psi[pc0] : psi[id];
  if (need_psi) {
    C sx, sy;
    grad_t(&s_psi[pc0], HX, sx, sy);
    Fmx = -k.G * cs2 * psi0 * sx;
    Fmy = -k.G * cs2 * psi0 * sy;
  }
  if (forcing) {
    Fx = sub(Fmx, mul(sub(rho, k.rho_l), k.g));
    if (k.body_fx != C(0)) Fx = add(Fx, k.body_fx);
    Fy = Fmy;
  }
  const C omega = fdiv(C(1), add(div_by(nu_of(ph, rho), cs2, C(1.0 / (1.0 / 3.0))), C(0.5)));
  const C sig = need_psi ? k.sigma : C(0);
  C fs[9], ux, uy;
  if constexpr (OP == kCollBGK) collide_bgk(fo, rho, Fx, Fy, omega, fs, ux, uy);
  else collide(fo, rho, Fx, Fy, Fmx, Fmy, psi0, omega, sig, fs, ux, uy);
#pragma unroll
  for (int i = 0; i < 9; ++i) fn[i * g.plane + id] = PopIO<C, S>::st(fs[i], i, ph);
  rho_o[id] = rho;
  ux_o[id] = ux;
  uy_o[id] = uy;
  if (sizeof(C) == 8 && lam_o) lam_o[id] = lam_of(ph, rho);
  if (!(rho > C(0)) || !(ux == ux) || !(uy == uy)) atomicOr(status, 1);
}

// The psi tile of tile (x0, y0) with plain loads (periodic in y, clamped or periodic in x).
template <typename C, typename S, int CTY>
__device__ __forceinline__ void psi_tile_plain(const Geo& g, const C* __restrict__ psi, int x0, int y0, C* s_psi) {
  using CS = CollStage<C, S, CTY>;
  for (int p = threadIdx.y * kCollTX + threadIdx.x; p < CS::PW * CS::PH; p += kCollTX * CTY) {
    const int hx = p % CS::PW, hy = p / CS::PW;
    s_psi[p] = psi[map_y(g, y0 + hy - 2) * g.pitch + map_x(g, x0 + hx - CS::PA)];
  }
}

// Collision tile (bx, by) of 32 x CTY nodes.  tm_f, tm_psi: tensor maps of f and psi for TMA
// staging, or null.  FP64 blocks leave the next pass to start when they end: they run for 15 us on the FP64
// pipe, and blocks of the next pass that wait beside them from the start pile up on some SMs (241 x 241,
// single phase: 51 us a step so, 36 us now; 512 x 256: the same).
template <typename C, typename S, int CTY, int OP = kCollCM>
__device__ __forceinline__ void collide_tile(const Geo& g, const Phys& ph, const S* __restrict__ f,
                                             S* __restrict__ fn, const C* __restrict__ psi,
                                             const uint8_t* __restrict__ mask, const C* __restrict__ side_in,
                                             C* __restrict__ side_out, C* __restrict__ rho_o, C* __restrict__ ux_o,
                                             C* __restrict__ uy_o, int forcing, int* status, int bx, int by,
                                             const CUtensorMap* tm_f = nullptr, const CUtensorMap* tm_psi = nullptr,
                                             bool starve = false, bool early_f = false, C* lam_o = nullptr) {
  using CS = CollStage<C, S, CTY>;
  constexpr int HX = CS::PW, HY = CS::PH;
  __shared__ __align__(128) S s_f[9 * CS::FH * CS::FW];
  __shared__ __align__(128) C s_psi[HY * HX];
  __shared__ uint64_t s_bar;
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * kCollTX + tx;
  const int x0 = bx * kCollTX, y0 = by * CTY;
  const int x = x0 + tx, y = y0 + ty;
  const bool need_psi = pc<C>(ph).G != C(0) && forcing;
  const bool staged = tm_f && (!need_psi || tm_psi) && coll_staged<C, S, CTY>(g, x0, y0);
  if (staged) {
    if (tid == 0) tma::bar_init(&s_bar, 1);
    __syncthreads();
    if (tid == 0) {
      const uint32_t bytes = sizeof(S) * 9 * CS::FH * CS::FW + (need_psi ? sizeof(C) * HX * HY : 0);
      tma::bar_expect_tx(&s_bar, bytes);
      // (the test hook leaves the barrier armed with no copy issued)
      if (!starve && early_f) tma::load_3d(s_f, tm_f, &s_bar, x0 - CS::XA, y0 - 1, 0);
    }
    pdl::wait();  // psi is the previous kernel's output
    if (sizeof(C) == 4) pdl::trigger();
    if (tid == 0 && !starve) {
      if (!early_f) tma::load_3d(s_f, tm_f, &s_bar, x0 - CS::XA, y0 - 1, 0);
      if (need_psi) tma::load_2d(s_psi, tm_psi, &s_bar, x0 - CS::PA, y0 - 2);
    }
  } else {
    pdl::wait();
    if (sizeof(C) == 4) pdl::trigger();
    if (need_psi) {
      psi_tile_plain<C, S, CTY>(g, psi, x0, y0, s_psi);
      __syncthreads();
    }
  }
  const bool inside = x < g.nx && y < g.ny;
  const uint8_t m = inside ? mask[y * g.pitch + x] : kSolid;
  const int tries = starve ? tma::kStarveTries : tma::kWaitTries;
  if (staged && !tma::bar_wait(&s_bar, 0, tries)) {
    // the copies did not land in time: report it, give them a second bound to land before the
    // block's shared memory is released, and produce nothing
    if (tid == 0) atomicOr(status, kStatusTimeoutCollide);
    tma::bar_wait(&s_bar, 0, tries);
    return;
  }
  if (!inside) return;
  collide_node<C, S, CTY, OP>(g, ph, f, fn, psi, mask, side_in, side_out, rho_o, ux_o, uy_o, forcing, status, tx, ty,
                              x, y, m, staged, s_f, s_psi, lam_o);
}

template <typename C, typename S, int OP = kCollCM>
// FP32 arithmetic: at most 36 registers, so 7 blocks share an SM and more pulls are in flight (7 blocks
// and a few spilled registers beat 6 without spills: FP16 storage 30.8 vs 32.6 us at 1536 x 768, FP32 30.4 vs
// 32.8 us at 2048 x 1024)
__global__ void __launch_bounds__(kCollTX* kCollTY, sizeof(C) == 4 ? 7 : 1)
    k_collide(Geo g, Phys ph, const S* __restrict__ f, S* __restrict__ fn, const C* __restrict__ psi,
              const uint8_t* __restrict__ mask, const C* __restrict__ side_in, C* __restrict__ side_out,
              C* __restrict__ rho_o, C* __restrict__ ux_o, C* __restrict__ uy_o, int forcing, int* status,
              const __grid_constant__ CUtensorMap tm_f, const __grid_constant__ CUtensorMap tm_psi, int flags,
              C* __restrict__ lam_o) {
  const bool staged = flags & kLaunchStaged;
  collide_tile<C, S, kCollTY, OP>(g, ph, f, fn, psi, mask, side_in, side_out, rho_o, ux_o, uy_o, forcing, status,
                                  blockIdx.x, blockIdx.y, staged ? &tm_f : nullptr, staged ? &tm_psi : nullptr,
                                  (flags & kLaunchStarve) != 0, (flags & kLaunchEarlyF) != 0, lam_o);
}

// ---------------------------------------------------------------- k_energy
// Fixed-shape block sum (warp shuffles, then the first warp over the warp sums).
template <int NT>
__device__ __forceinline__ double block_sum(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  if ((tid & 31) == 0) red[tid >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (tid < 32) {
    s = tid < NT / 32 ? red[tid] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  }
  return s;  // valid in thread 0
}

// Two x-adjacent nodes per thread: a 5x6 window (rows -2..2, columns -2..3 around the
// left node) is read from a shared tile with three aligned 2-vector loads per row; both
// nodes' stencils are then evaluated from registers in the same term order as above.
template <typename C>
struct Vec2;
template <>
struct Vec2<float> {
  using T = float2;
};
template <>
struct Vec2<double> {
  using T = double2;
};
template <typename C>
__device__ __forceinline__ void load_window(const C* p, int s, C w[5][6]) {
  using T2 = typename Vec2<C>::T;
#pragma unroll
  for (int r = 0; r < 5; ++r) {
    const T2* q = reinterpret_cast<const T2*>(p + (r - 2) * s - 2);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const T2 v = q[c];
      w[r][2 * c] = v.x;
      w[r][2 * c + 1] = v.y;
    }
  }
}
template <typename C, bool kX = true, bool kY = true>
__device__ __forceinline__ void grad_w(const C w[5][6], int c0, C& gx, C& gy) {
  C sx = C(0), sy = C(0);
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const int ex = exv(k), ey = eyv(k);
    if ((kX && ex != 0) || (kY && ey != 0)) {
      C d = w[2 + ey][c0 + ex] - w[2 - ey][c0 - ex];
      if (kX && ex != 0) sx = sx + C(wiso(k) * ex) * d;
      if (kY && ey != 0) sy = sy + C(wiso(k) * ey) * d;
    }
  }
  gx = sx;
  gy = sy;
}
template <typename C>
__device__ __forceinline__ C lap_w(const C w[5][6], int c0) {
  const C c = w[2][c0];
  C acc = C(0);
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const int ex = exv(k), ey = eyv(k);
    C d = (w[2 + ey][c0 + ex] + w[2 - ey][c0 - ex]) - C(2) * c;
    acc = acc + C(wiso(k)) * d;
  }
  return C(2) * acc;
}
// Density of the pulled populations, rho = sum_i f*_i(x - c_i), at the nodes (x0, y) and
// (x0 + 1, y), x0 even, for a pair none of whose pulls crosses the lattice edge or meets the
// wall (1 <= x0, x0 + 2 <= nx - 1, 1 <= y <= ny - 2, no near-wall node): the planes with c_x = 0
// are read as aligned vectors, the others as scalars, all from one base address; the sum runs
// in the order i = 0..8, as in the general pull, so both give the same bits.
template <typename S>
struct PairLoad;
template <>
struct PairLoad<float> {
  static __device__ __forceinline__ void ld(const float* q, float& a, float& b) {
    const float2 v = *reinterpret_cast<const float2*>(q);
    a = v.x, b = v.y;
  }
};
template <>
struct PairLoad<double> {
  static __device__ __forceinline__ void ld(const double* q, double& a, double& b) {
    const double2 v = *reinterpret_cast<const double2*>(q);
    a = v.x, b = v.y;
  }
};
template <>
struct PairLoad<__half> {
  static __device__ __forceinline__ void ld(const __half* q, __half& a, __half& b) {
    const __half2 v = *reinterpret_cast<const __half2*>(q);
    a = __low2half(v), b = __high2half(v);
  }
};
template <typename C, typename S>
__device__ __forceinline__ void pair_rho(const Geo& g, const Phys& ph, const S* __restrict__ f, int x0, int y,
                                         C r[2]) {
  const S* p = f + y * g.pitch + x0;
  C v[9][2];
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const S* q = p + i * g.plane - cyv(i) * g.pitch - cxv(i);
    S a, b;
    if (cxv(i) == 0) {
      PairLoad<S>::ld(q, a, b);
    } else {
      a = q[0];
      b = q[1];
    }
    v[i][0] = PopIO<C, S>::ld(a, i, ph);
    v[i][1] = PopIO<C, S>::ld(b, i, ph);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    C t = v[0][k];
#pragma unroll
    for (int i = 1; i < 9; ++i) t = t + v[i][k];
    r[k] = t;
  }
}

// Block-level end of the wall heat flux: FP64 block sums only in the blocks that hold wall
// nodes (the others skip the fence and the counter); the last of those n_wall blocks to
// finish adds all nblocks partials in block order (zero elsewhere), updates the running
// statistics hf and clears the partials for the next launch.  Every thread of the block calls it.
template <int NT>
__device__ __forceinline__ void heat_flux_blocks(double q, int mine, double* partial, unsigned* counter, int n_wall,
                                                 int bid, int nblocks, double* hf, int nb, double* red,
                                                 int* done_last) {
  const int tid = threadIdx.x;
  if (__syncthreads_or(mine)) {
    const double s = block_sum<NT>(q, red);
    if (tid == 0) {
      partial[bid] = s;
      __threadfence();
      *done_last = atomicInc(counter, n_wall - 1) == (unsigned)(n_wall - 1);
    }
    __syncthreads();
    if (*done_last) {
      __threadfence();
      double acc = 0.0;
      for (int i = tid; i < nblocks; i += NT) acc += __ldcg(&partial[i]);
      acc = block_sum<NT>(acc, red);  // its barrier also ends every thread's reads above
      for (int i = tid; i < nblocks; i += NT) partial[i] = 0.0;
      if (tid == 0) {
        const double qv = acc / nb;
        hf[0] = qv;
        hf[1] += qv;
        hf[2] += qv * qv;
        hf[3] += 1.0;
      }
    }
  }
}

}  // namespace kern
}  // namespace lbm
#include "lbm_energy_f64.cuh"
#include "lbm_step_f16s.cuh"
namespace lbm {
namespace kern {

// Planes of the FP64 energy pass in a context's work planes (T1 first).
__device__ __forceinline__ Frozen64 frozen64(double* en64, const Geo& g) {
  const size_t n = g.plane;
  return {en64 + n, en64 + 2 * n, en64 + 3 * n, en64 + 4 * n, en64 + 5 * n, en64 + 6 * n};
}
static __global__ void __launch_bounds__(128)
    k_energy1_f64(Geo g, Phys ph, const double* __restrict__ Tin, double* __restrict__ T1, double* en64,
                  const double* __restrict__ lam, const double* __restrict__ rho, const double* __restrict__ ux,
                  const double* __restrict__ uy, const uint8_t* __restrict__ mask, double* partial, unsigned* counter,
                  double* hf, int nb, int do_hf, int n_wall_tiles, int* status, const __grid_constant__ EnergyMaps maps,
                  int flags) {
  energy1_tile(g, ph, Tin, T1, lam, frozen64(en64, g), rho, ux, uy, mask, partial, counter, hf, nb, do_hf, n_wall_tiles,
               blockIdx.x, blockIdx.y, blockIdx.y * gridDim.x + blockIdx.x, gridDim.x * gridDim.y, status,
               (flags & kLaunchStaged) ? &maps : nullptr, (flags & kLaunchStarve) != 0);
}
static __global__ void __launch_bounds__(128)
    k_energy2_f64(Geo g, Phys ph, const double* __restrict__ Tin, double* __restrict__ Tout,
                  const double* __restrict__ T1, double* en64, const double* __restrict__ lam,
                  const double* __restrict__ rho, const double* __restrict__ ux, const double* __restrict__ uy,
                  const uint8_t* __restrict__ mask, const double* __restrict__ fnew,
                  const double* __restrict__ side_new, double* __restrict__ psi_out, int* status) {
  energy2_tile(g, ph, Tin, Tout, T1, lam, frozen64(en64, g), rho, ux, uy, mask, blockIdx.x, blockIdx.y, fnew, side_new,
               psi_out, status);
}

// ---------------------------------------------------------------- batched passes
// Every block of a batched pass finds its domain through the block -> domain map and its
// tile from its index within that domain; the tile bodies are the single-domain ones.
// psi of the state with population parity p sits in domain buffer p (psi, psi_next): the
// energy pass of a step with parity cur writes psi of the next state into buffer cur ^ 1,
// so the psi pass runs only when the host no longer knows psi (creation, a state change).
template <typename C>
__device__ __forceinline__ C* psi_buf(const BatchDomain& D, int p) {
  return static_cast<C*>(p ? D.d.psi_next : D.d.psi);
}
template <typename C, typename S, int PSI>
__global__ void __launch_bounds__(256) kb_rho_psi(const BatchDomain* __restrict__ doms, const int* __restrict__ map,
                                                 int cur, int tcur) {
  const BatchDomain& D = doms[map[blockIdx.x]];
  if (pc<C>(D.ph).G == C(0)) return;
  const int local = blockIdx.x - D.psi_first;
  rho_psi_tile<C, S, PSI>(D.g, D.ph, static_cast<const S*>(D.d.f[cur]), static_cast<const C*>(D.d.T[tcur]),
                          D.d.mask, static_cast<const C*>(D.d.side[cur]), psi_buf<C>(D, cur), D.d.status,
                          local % D.psi_ntx, local / D.psi_ntx);
}
// A batched launch covers the blocks [block0, block0 + gridDim.x) of a pass, which belong to
// the domains dom0 ..; their tensor maps come as kernel parameters (index k - dom0).
template <typename C, typename S, int CTY>
__global__ void __launch_bounds__(kCollTX* CTY)
    kb_collide(const BatchDomain* __restrict__ doms, const int* __restrict__ map, int cur, long long step,
               int block0, int dom0, const __grid_constant__ CollLaunchMaps maps) {
  const int blk = block0 + blockIdx.x, k = map[blk];
  const BatchDomain& D = doms[k];
  const int local = blk - D.coll_first;
  collide_tile<C, S, CTY>(D.g, D.ph, static_cast<const S*>(D.d.f[cur]), static_cast<S*>(D.d.f[cur ^ 1]),
                          psi_buf<C>(D, cur), D.d.mask, static_cast<const C*>(D.d.side[cur]),
                          static_cast<C*>(D.d.side[cur ^ 1]), static_cast<C*>(D.d.rho), static_cast<C*>(D.d.ux),
                          static_cast<C*>(D.d.uy), step >= D.warmup, D.d.status, local % D.coll_ntx,
                          local / D.coll_ntx, D.tma ? &maps.f[k - dom0] : nullptr,
                          D.tma ? &maps.psi[k - dom0] : nullptr, false, false,
                          sizeof(C) == 8 ? static_cast<C*>(D.d.lam) : nullptr);
}
// FP64 energy pass of a batch: the two stages of the domains that take an energy step; the others
// carry T over in the second.
static __global__ void __launch_bounds__(128)
    kb_energy1_f64(const BatchDomain* __restrict__ doms, const int* __restrict__ map, int tcur, long long step, int block0,
                   int dom0, const __grid_constant__ EnLaunchMaps maps) {
  const int blk = block0 + blockIdx.x, k = map[blk];
  const BatchDomain& D = doms[k];
  const int local = blk - D.en_first;
  if (!D.energy || step < D.warmup) return;
  energy1_tile(D.g, D.ph, static_cast<const double*>(D.d.T[tcur]), static_cast<double*>(D.d.en64),
               static_cast<const double*>(D.d.lam), frozen64(static_cast<double*>(D.d.en64), D.g),
               static_cast<const double*>(D.d.rho), static_cast<const double*>(D.d.ux),
               static_cast<const double*>(D.d.uy), D.d.mask, D.d.partial, D.d.counter, D.d.hf, D.d.nb, D.d.nb > 0,
               D.d.wall_tiles[0], local % D.en_ntx, local / D.en_ntx, local, D.en_nblocks, D.d.status,
               D.tma ? &maps.e[k - dom0] : nullptr, false);
}
static __global__ void __launch_bounds__(128)
    kb_energy2_f64(const BatchDomain* __restrict__ doms, const int* __restrict__ map, int cur, int tcur, long long step) {
  const int k = map[blockIdx.x];
  const BatchDomain& D = doms[k];
  const int local = blockIdx.x - D.en_first, bx = local % D.en_ntx, by = local / D.en_ntx;
  const double* Tin = static_cast<const double*>(D.d.T[tcur]);
  double* Tout = static_cast<double*>(D.d.T[tcur ^ 1]);
  const double* fnew = static_cast<const double*>(D.d.f[cur ^ 1]);
  const double* side_new = static_cast<const double*>(D.d.side[cur ^ 1]);
  double* psi_next = D.ph.d.G != 0.0 ? psi_buf<double>(D, cur ^ 1) : nullptr;
  if (!D.energy || step < D.warmup) {
    // no energy update for this domain this step: carry T over so all domains flip together,
    // and make psi of the next state from the new populations and the unchanged T
    for (int p = threadIdx.x; p < kEnergyTX64 * 8; p += 128) {
      const int x = bx * kEnergyTX64 + p % kEnergyTX64, y = by * 8 + p / kEnergyTX64;
      if (x < D.g.nx && y < D.g.ny) {
        Tout[y * D.g.pitch + x] = Tin[y * D.g.pitch + x];
        if (psi_next)
          psi_next[y * D.g.pitch + x] =
              psi_node<double, double, kPsiF64>(D.g, D.ph, fnew, Tin, D.d.mask, side_new, x, y, D.d.status);
      }
    }
    return;
  }
  energy2_tile(D.g, D.ph, Tin, Tout, static_cast<const double*>(D.d.en64), static_cast<const double*>(D.d.lam),
               frozen64(static_cast<double*>(D.d.en64), D.g), static_cast<const double*>(D.d.rho),
               static_cast<const double*>(D.d.ux), static_cast<const double*>(D.d.uy), D.d.mask, bx, by, fnew, side_new,
               psi_next, D.d.status);
}
template <typename C, typename S, int PSI, int CTY>
int batch_step_impl(const BatchDomain* doms, const int* map_psi, int nb_psi, const int* map_coll, int nb_coll,
                    const int* map_en, int nb_en, int cur, int tcur, long long step, int need_psi,
                    const BatchDomain* hdoms, const DomainMaps* hmaps, int ndom, cudaStream_t s) {
  int n = 0;
  if (need_psi) {
    kb_rho_psi<C, S, PSI><<<nb_psi, dim3(kCollTX, 8), 0, s>>>(doms, map_psi, cur, tcur);
    ++n;
  }
  for (int d0 = 0; d0 < ndom; d0 += kBatchCollDomains) {
    const int d1 = d0 + kBatchCollDomains < ndom ? d0 + kBatchCollDomains : ndom;
    CollLaunchMaps m;
    for (int k = d0; k < d1; ++k) {
      m.f[k - d0] = hmaps[k].f[cur];
      m.psi[k - d0] = hmaps[k].psi[cur];
    }
    const int b0 = hdoms[d0].coll_first, b1 = d1 < ndom ? hdoms[d1].coll_first : nb_coll;
    kb_collide<C, S, CTY><<<b1 - b0, dim3(kCollTX, CTY), 0, s>>>(doms, map_coll, cur, step, b0, d0, m);
    ++n;
  }
  for (int d0 = 0; d0 < ndom; d0 += kBatchEnDomains) {
    const int d1 = d0 + kBatchEnDomains < ndom ? d0 + kBatchEnDomains : ndom;
    EnLaunchMaps m;
    for (int k = d0; k < d1; ++k) m.e[k - d0] = hmaps[k].em[tcur];
    const int b0 = hdoms[d0].en_first, b1 = d1 < ndom ? hdoms[d1].en_first : nb_en;
    kb_energy1_f64<<<b1 - b0, 128, 0, s>>>(doms, map_en, tcur, step, b0, d0, m);
    ++n;
  }
  kb_energy2_f64<<<nb_en, 128, 0, s>>>(doms, map_en, cur, tcur, step);
  ++n;
  return cudaPeekAtLastError() == cudaSuccess ? n : -1;
}

// Tensor maps of one batched domain for tile heights (cty, ety), as the single-domain step
// encodes them per launch (here once per layout: the buffers of a domain do not move).
template <typename C, typename S>
bool batch_maps_impl(BatchDomain& D, DomainMaps& m, int cty, int ety) {
  const Geo& g = D.g;
  const int XA = 16 / (int)sizeof(S), PA = 16 / (int)sizeof(C) < 2 ? 2 : 16 / (int)sizeof(C);
  bool ok = D.d.tma != 0;
  for (int p = 0; p < 2 && ok; ++p) {
    ok = tma::encode<S>(&m.f[p], D.d.f[p], g.nx, g.ny, g.pitch, g.plane, 9, kCollTX + 2 * XA, cty + 2) &&
         tma::encode<C>(&m.psi[p], p ? D.d.psi_next : D.d.psi, g.nx, g.ny, g.pitch, g.plane, 1,
                        kCollTX + 2 * PA, cty + 4) &&
         tma::encode<C>(&m.em[p].T, D.d.T[p], g.nx, g.ny, g.pitch, g.plane, 1, kEnergyTX64 + 4, ety + 4) &&
         static_cast<const C*>(D.d.ux) == static_cast<const C*>(D.d.rho) + g.plane &&
         static_cast<const C*>(D.d.uy) == static_cast<const C*>(D.d.rho) + 2 * (size_t)g.plane &&
         tma::encode<C>(&m.em[p].ruv, D.d.rho, g.nx, g.ny, g.pitch, g.plane, 3, kEnergyTX64 + 4, ety + 4);
  }
  D.tma = ok ? 1 : 0;
  return ok;
}

// ---------------------------------------------------------------- init / export / import
// Fourth-order Hermite equilibrium, Eq. (equi).
__device__ __forceinline__ void feq_hermite(double rho, double ux, double uy, double fe[9]) {
  const double cs2 = 1.0 / 3.0;
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const double w = i == 0 ? 4.0 / 9.0 : (i < 5 ? 1.0 / 9.0 : 1.0 / 36.0);
    const double cx = cxv(i), cy = cyv(i);
    const double Hxx = cx * cx - cs2, Hyy = cy * cy - cs2, Hxy = cx * cy;
    const double Hxxy = cx * cx * cy - cs2 * cy;
    const double Hxyy = cx * cy * cy - cs2 * cx;
    const double Hxxyy = cx * cx * cy * cy - cs2 * (cx * cx + cy * cy) + cs2 * cs2;
    const double t1 = (cx * ux + cy * uy) / cs2;
    const double t2 = (Hxx * ux * ux + 2.0 * Hxy * ux * uy + Hyy * uy * uy) / (2.0 * cs2 * cs2);
    const double t3 = (Hxxy * ux * ux * uy + Hxyy * ux * uy * uy) / (2.0 * cs2 * cs2 * cs2);
    const double t4 = Hxxyy * ux * ux * uy * uy / (4.0 * cs2 * cs2 * cs2 * cs2);
    fe[i] = w * rho * (1.0 + t1 + t2 + t3 + t4);
  }
}

// SplitMix64 (Steele, Lea, Flood 2014): value k of stream `seed`, mapped to [-1, 1).
__device__ __forceinline__ double splitmix_pm1(unsigned long long seed, unsigned long long k) {
  unsigned long long z = seed + (k + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z = z ^ (z >> 31);
  return (double)(z >> 11) * 0x1.0p-53 * 2.0 - 1.0;
}

// in: optional dense [ny][nx] double arrays (rho, drho, ux, uy, T), any NULL.
template <typename C, typename S>
__global__ void __launch_bounds__(256) k_init(Geo g, Phys ph, const double* rho0, const double* drho,
                                             const double* ux0, const double* uy0, const double* T0,
                                             const double* Tw, unsigned long long seed, double noise_amp, S* f,
                                             C* T, C* rho_o,
                                             C* ux_o, C* uy_o, C* side, const uint8_t* __restrict__ mask) {
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = blockIdx.y * 8 + threadIdx.y;
  if (x >= g.nx || y >= g.ny) return;
  const int id = y * g.pitch + x;
  const int k = y * g.nx + x;
  double r = rho0 ? rho0[k] : ph.d.rho_l;
  r = r + (drho ? drho[k] : noise_amp * splitmix_pm1(seed, (unsigned long long)k));
  double u = ux0 ? ux0[k] : ph.d.u_in, v = uy0 ? uy0[k] : 0.0;
  double t = T0 ? T0[k] : ph.d.T_sat;
  if (mask[id] & kSolid) {
    r = ph.d.rho_s;
    u = 0.0;
    v = 0.0;
    t = Tw ? Tw[k] : ph.d.T_wall;
  }
  double fe[9];
  feq_hermite(r, u, v, fe);
#pragma unroll
  for (int i = 0; i < 9; ++i) f[i * g.plane + id] = PopIO<C, S>::st_d(fe[i], i, ph);
  T[id] = (C)t;
  rho_o[id] = (C)r;
  ux_o[id] = (C)u;
  uy_o[id] = (C)v;
  if (!g.periodic_x && x == g.nx - 1) {
    side[0 * g.ny + y] = (C)fe[2];
    side[1 * g.ny + y] = (C)fe[6];
    side[2 * g.ny + y] = (C)fe[8];
  }
}

template <typename E>
__global__ void k_export(Geo g, const E* __restrict__ src, int src_pitch, int rows, double* __restrict__ dst,
                         int ncols) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y;
  if (x >= ncols || y >= rows) return;
  dst[y * ncols + x] = (double)src[y * src_pitch + x];
}

static __global__ void k_export_solid(Geo g, const uint8_t* __restrict__ mask, double* __restrict__ dst) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y;
  if (x >= g.nx || y >= g.ny) return;
  dst[y * g.nx + x] = (mask[y * g.pitch + x] & kSolid) ? 1.0 : 0.0;
}

// Component comp (0: x, 1: y) of the force F = F_m + F_g (+ the body force) that the collision
// applied at every node (Eq. interForce with gravity along -x, Sec. IV.A), recomputed from the
// psi and rho that collision used with the same order of operations and roundings (rows: those of
// force_of and grad_rows, which the FP32 build takes but for FP16 populations; else of collide_node); zero on
// solid nodes and when the step ran without forcing (warm-up).
template <typename C, bool rows>
__global__ void k_export_force(Geo g, Phys ph, const C* __restrict__ psi, const C* __restrict__ rho,
                               const uint8_t* __restrict__ mask, int forcing, int comp, double* __restrict__ dst) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y;
  if (x >= g.nx || y >= g.ny) return;
  const int id = y * g.pitch + x;
  double out = 0.0;
  if (forcing && !(mask[id] & kSolid)) {
    const PhysC<C>& k = pc<C>(ph);
    const C cs2 = C(1.0 / 3.0);
    C Fmx = C(0), Fmy = C(0);
    if (k.G != C(0)) {
      C w[25];
#pragma unroll
      for (int r = 0; r < 5; ++r)
#pragma unroll
        for (int c = 0; c < 5; ++c) w[r * 5 + c] = psi[map_y(g, y + r - 2) * g.pitch + map_x(g, x + c - 2)];
      C sx, sy;
      if constexpr (rows) {
        grad_window(w, 5, sx, sy);
        const C a = mul(ph.sc.gm, w[12]);
        Fmx = mul(a, sx);
        Fmy = mul(a, sy);
      } else {
        grad_t(&w[12], 5, sx, sy);
        Fmx = -k.G * cs2 * w[12] * sx;
        Fmy = -k.G * cs2 * w[12] * sy;
      }
    }
    C Fx;
    if constexpr (rows) Fx = mad(-k.g, sub(rho[id], k.rho_l), Fmx);
    else Fx = sub(Fmx, mul(sub(rho[id], k.rho_l), k.g));
    if (k.body_fx != C(0)) Fx = add(Fx, k.body_fx);
    out = comp == 0 ? (double)Fx : (double)Fmy;
  }
  dst[y * g.nx + x] = out;
}

template <typename C, typename S>
__global__ void k_export_pop(Geo g, Phys ph, const S* __restrict__ src, int i, double* __restrict__ dst) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y;
  if (x >= g.nx || y >= g.ny) return;
  dst[y * g.nx + x] = PopIO<C, S>::ld_d(src[y * g.pitch + x], i, ph);
}
template <typename C, typename S>
__global__ void k_import_pop(Geo g, Phys ph, S* __restrict__ dst, int i, const double* __restrict__ src) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y;
  if (x >= g.nx || y >= g.ny) return;
  dst[y * g.pitch + x] = PopIO<C, S>::st_d(src[y * g.nx + x], i, ph);
}

template <typename E>
__global__ void k_import(Geo g, E* __restrict__ dst, int dst_pitch, int rows, const double* __restrict__ src,
                         int ncols) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y;
  if (x >= ncols || y >= rows) return;
  dst[y * dst_pitch + x] = static_cast<E>(src[y * ncols + x]);
}

}  // namespace kern

// ---------------------------------------------------------------- launchers
// Launch kernel k (smem bytes of dynamic shared memory) on stream s, as a programmatic dependent
// of the kernel before it when pdl is set.
template <typename... KArgs, typename... Args>
cudaError_t launch_dep(bool pdl, dim3 grd, dim3 blk, size_t smem, cudaStream_t s, void (*k)(KArgs...),
                       Args&&... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grd;
  cfg.blockDim = blk;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, static_cast<Args&&>(args)...);
}

// The collision of 32 x 8 tiles, one node per lane, with psi read from memory.
template <typename C, typename S>
void launch_collide(const Geo& g, const Phys& ph, const Dev& d, int cur, int forcing, C* lam, cudaStream_t s) {
  using namespace kern;
  const S* f = static_cast<const S*>(d.f[cur]);
  const C* psi = static_cast<const C*>(d.psi);
  // tensor maps of this step's populations and psi for the TMA-staged tiles (plain loads
  // everywhere when a map cannot be made)
  using CS = CollStage<C, S, kCollTY>;
  CUtensorMap tm_f = {}, tm_psi = {};
  const bool staged = d.tma && tma::encode<S>(&tm_f, f, g.nx, g.ny, g.pitch, g.plane, 9, CS::FW, CS::FH) &&
                      (ph.d.G == 0.0 || tma::encode<C>(&tm_psi, psi, g.nx, g.ny, g.pitch, g.plane, 1, CS::PW, CS::PH));
  const int flags = staged ? (kLaunchStaged | ((d.starve & kStarveCollide) ? kLaunchStarve : 0) |
                              ((d.pdl && d.f_ready) ? kLaunchEarlyF : 0))
                           : 0;
  const dim3 blk(kCollTX, kCollTY), grd((g.nx + kCollTX - 1) / kCollTX, (g.ny + kCollTY - 1) / kCollTY);
  auto go = [&](auto kernel) {
    launch_dep(d.pdl, grd, blk, 0, s, kernel, g, ph, f, static_cast<S*>(d.f[cur ^ 1]), psi, d.mask,
               static_cast<const C*>(d.side[cur]), static_cast<C*>(d.side[cur ^ 1]), static_cast<C*>(d.rho),
               static_cast<C*>(d.ux), static_cast<C*>(d.uy), forcing, d.status, tm_f, tm_psi, flags, lam);
  };
  if (d.collision == kCollBGK) go(k_collide<C, S, kCollBGK>);
  else go(k_collide<C, S, kCollCM>);
}

template <typename C, typename S, int PSI>
int step_impl(const Geo& g, const Phys& ph, const Dev& d, int cur, int tcur, int forcing, int energy, cudaStream_t s,
              const LaunchHook* hook, int* t_flipped, PsiChain* chain) {
  using namespace kern;
  const S* f = static_cast<const S*>(d.f[cur]);
  S* fn = static_cast<S*>(d.f[cur ^ 1]);
  const C* T = static_cast<const C*>(d.T[tcur]);
  C* Tn = static_cast<C*>(d.T[tcur ^ 1]);
  C* rho = static_cast<C*>(d.rho);
  C* ux = static_cast<C*>(d.ux);
  C* uy = static_cast<C*>(d.uy);
  C* psi = static_cast<C*>(d.psi);
  const C* side_in = static_cast<const C*>(d.side[cur]);
  C* side_out = static_cast<C*>(d.side[cur ^ 1]);
  int n = 0;
  auto pre = [&](int k) {
    if (hook) hook->before(hook->self, k);
  };
  auto post = [&](int k) {
    if (hook) hook->after(hook->self, k);
    ++n;
  };
  const dim3 blk(kCollTX, kCollTY), grd((g.nx + kCollTX - 1) / kCollTX, (g.ny + kCollTY - 1) / kCollTY);
  if (ph.d.G != 0.0 && !(chain && chain->have)) {
    pre(kKRhoPsi);
    k_rho_psi<C, S, PSI><<<grd, blk, 0, s>>>(g, ph, f, T, d.mask, side_in, psi, d.status);
    post(kKRhoPsi);
  }
  pre(kKCollide);
  C* const lam = sizeof(C) == 8 && energy && forcing ? static_cast<C*>(d.lam) : nullptr;
  launch_collide<C, S>(g, ph, d, cur, forcing, lam, s);
  post(kKCollide);
  *t_flipped = 0;
  if (energy && forcing) {
    const int do_hf = d.nb > 0;
    const bool fuse = chain && chain->want && ph.d.G != 0.0;
    pre(kKEnergy);
    constexpr bool f64 = sizeof(C) == 8;
    constexpr int TY = f64 ? 8 : EnergyTile16::TY, EH = f64 ? 4 : 8;  // both halos of the tile
    const dim3 blk(kEnergyTX64 * TY / 2), grd((g.nx + kEnergyTX64 - 1) / kEnergyTX64, (g.ny + TY - 1) / TY);
    constexpr int AX = kEnergyTX64 + EH, AY = TY + EH;
    EnergyMaps em;
    const bool ruv = ux == rho + g.plane && uy == rho + 2 * (size_t)g.plane;  // consecutive planes
    const bool e_staged = d.tma && ruv && tma::encode<C>(&em.T, T, g.nx, g.ny, g.pitch, g.plane, 1, AX, AY) &&
                          tma::encode<C>(&em.ruv, rho, g.nx, g.ny, g.pitch, g.plane, 3, AX, AY);
    const int eflags = e_staged ? (kLaunchStaged | ((d.starve & kStarveEnergy) ? kLaunchStarve : 0)) : 0;
    if constexpr (f64) {
      double* en64 = static_cast<double*>(d.en64);
      double* T1 = d.t1_out ? static_cast<double*>(d.t1_out) : en64;
      launch_dep(d.pdl, grd, blk, 0, s, k_energy1_f64, g, ph, T, T1, en64, lam, rho, ux, uy, d.mask, d.partial,
                 d.counter, d.hf, d.nb, do_hf, d.wall_tiles[0], d.status, em, eflags);
      launch_dep(d.pdl, grd, blk, 0, s, k_energy2_f64, g, ph, T, Tn, T1, en64, lam, rho, ux, uy, d.mask,
                 fuse ? static_cast<const double*>(fn) : nullptr, side_out,
                 fuse ? static_cast<double*>(d.psi_next) : nullptr, d.status);
      ++n;
    } else {
      launch_dep(d.pdl, grd, blk, 0, s, k_energy_f16s<PSI>, g, ph, T, Tn, rho, ux, uy, d.mask, d.partial, d.counter,
                 d.hf, d.nb, do_hf, d.wall_tiles[1], fuse ? static_cast<const __half*>(fn) : nullptr,
                 static_cast<const float*>(side_out), fuse ? static_cast<float*>(d.psi_next) : nullptr, d.status, em,
                 eflags);
    }
    post(kKEnergy);
    *t_flipped = 1;
    if (chain) chain->made = fuse ? kPsiFromPlane : kPsiFromPass;
  } else if (chain) {
    chain->made = kPsiFromPass;
  }
  return cudaPeekAtLastError() == cudaSuccess ? n : -1;
}

template <typename C, typename S>
int export_impl(const Geo& g, const Phys& ph, const Dev& d, int cur, int tcur, int which, double* dst, cudaStream_t s) {
  using namespace kern;
  const dim3 blk(256);
  if (which >= 20 && which < 23) {
    const C* src = static_cast<const C*>(d.side[cur]) + (which - 20) * g.ny;
    k_export<C><<<dim3((g.ny + 255) / 256, 1), blk, 0, s>>>(g, src, g.ny, 1, dst, g.ny);
  } else if (which >= 10 && which < 19) {
    const S* src = static_cast<const S*>(d.f[cur]) + (which - 10) * g.plane;
    k_export_pop<C, S><<<dim3((g.nx + 255) / 256, g.ny), blk, 0, s>>>(g, ph, src, which - 10, dst);
  } else if (which == 5) {
    k_export_solid<<<dim3((g.nx + 255) / 256, g.ny), blk, 0, s>>>(g, d.mask, dst);
  } else if (which >= 30 && which < 34) {  // 30 + comp + 2 forcing: the force of the last collision
    k_export_force<C, (sizeof(C) == 4 && sizeof(S) != 2)><<<dim3((g.nx + 255) / 256, g.ny), blk, 0, s>>>(
        g, ph, static_cast<const C*>(d.psi), static_cast<const C*>(d.rho), d.mask, (which - 30) >> 1, (which - 30) & 1,
        dst);
  } else {
    const void* p = which == 0 ? d.rho : which == 1 ? d.ux : which == 2 ? d.uy : which == 3 ? d.T[tcur] : d.psi;
    k_export<C><<<dim3((g.nx + 255) / 256, g.ny), blk, 0, s>>>(g, static_cast<const C*>(p), g.pitch, g.ny, dst, g.nx);
  }
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

template <typename C, typename S>
int import_impl(const Geo& g, const Phys& ph, const Dev& d, int cur, int tcur, int which, const double* src,
                cudaStream_t s) {
  using namespace kern;
  const dim3 blk(256);
  if (which >= 20 && which < 23) {
    C* dst = static_cast<C*>(d.side[cur]) + (which - 20) * g.ny;
    k_import<C><<<dim3((g.ny + 255) / 256, 1), blk, 0, s>>>(g, dst, g.ny, 1, src, g.ny);
  } else if (which >= 10 && which < 19) {
    S* dst = static_cast<S*>(d.f[cur]) + (which - 10) * g.plane;
    k_import_pop<C, S><<<dim3((g.nx + 255) / 256, g.ny), blk, 0, s>>>(g, ph, dst, which - 10, src);
  } else if (which == 3) {
    k_import<C><<<dim3((g.nx + 255) / 256, g.ny), blk, 0, s>>>(g, static_cast<C*>(d.T[tcur]), g.pitch, g.ny, src,
                                                                 g.nx);
  } else {
    return -1;
  }
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

template <typename C, typename S>
int init_impl(const Geo& g, const Phys& ph, const Dev& d, const double* rho0, const double* drho, const double* ux0,
              const double* uy0, const double* T0, const double* Tw, unsigned long long seed, double amp,
              cudaStream_t s) {
  using namespace kern;
  const dim3 blk(32, 8), grd((g.nx + 31) / 32, (g.ny + 7) / 8);
  k_init<C, S><<<grd, blk, 0, s>>>(g, ph, rho0, drho, ux0, uy0, T0, Tw, seed, amp, static_cast<S*>(d.f[0]),
                                   static_cast<C*>(d.T[0]), static_cast<C*>(d.rho), static_cast<C*>(d.ux),
                                   static_cast<C*>(d.uy), static_cast<C*>(d.side[0]), d.mask);
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

}  // namespace lbm
