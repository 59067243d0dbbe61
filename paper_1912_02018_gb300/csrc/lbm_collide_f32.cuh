// FP32 collision of a node (V = float) or of a column pair (V = float2, packed FP32x2 operations, which round
// lane by lane like the scalar ones): moments, force, CM and BGK operators (Sec. II.A-B; included by
// lbm_kernels.cuh).  Every rounding is written out, so that both forms, and every kernel that inlines them, give
// the same bits.  Shifted FP16 populations keep the earlier order of operations (lbm_step_f16s.cuh).
#pragma once

namespace lbm {
namespace kern {

__device__ __forceinline__ float add2(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub2(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul2(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma2(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float rcp2(float a) { return rcp_approx(a); }
// a in every lane
template <typename V>
__device__ __forceinline__ V all(float a);
template <>
__device__ __forceinline__ float all<float>(float a) {
  return a;
}
template <>
__device__ __forceinline__ float2 all<float2>(float a) {
  return f2(a);
}
// a b + c clamped to [0, 1]
__device__ __forceinline__ float satfma(float a, float b, float c) { return __saturatef(__fmaf_rn(a, b, c)); }
__device__ __forceinline__ float2 satfma(float2 a, float b, float c) {
  return make_float2(satfma(a.x, b, c), satfma(a.y, b, c));
}

// Moments of the pulled populations that the collision keeps: rho (in the order of pop_sum), m1, m2, m4, m5
// (App. A), and f_0 and the sum of the other eight.
template <typename V>
struct Moments {
  V rho, m1, m2, m4, m5, f0, sum8;
};
template <typename V>
__device__ __forceinline__ Moments<V> moments_of(const V f[9]) {
  const V s12 = add2(f[1], f[2]), s34 = add2(f[3], f[4]), s56 = add2(f[5], f[6]), s78 = add2(f[7], f[8]);
  const V d56 = sub2(f[5], f[6]), d78 = sub2(f[7], f[8]);
  const V s14 = add2(s12, s34), s58 = add2(s56, s78);
  Moments<V> M;
  M.rho = add2(add2(f[0], s14), s58);
  M.f0 = f[0];
  M.sum8 = add2(s14, s58);
  M.m1 = add2(add2(sub2(f[1], f[2]), d56), d78);
  M.m2 = sub2(add2(sub2(f[3], f[4]), d56), d78);
  M.m4 = sub2(s12, s34);
  M.m5 = sub2(s56, s78);
  return M;
}

// Force F_m = -G cs^2 psi grad psi (Eq. interForce; gx, gy the stencil sums) and F = F_m + gravity (+ the body
// force).
template <typename V>
__device__ __forceinline__ void force_of(const Phys& ph, V rho, V psi, V gx, V gy, V& Fx, V& Fy) {
  const V a = mul2(all<V>(ph.sc.gm), psi);
  Fx = fma2(all<V>(-ph.f.g), sub2(rho, all<V>(ph.f.rho_l)), mul2(a, gx));
  Fy = mul2(a, gy);
  if (ph.f.body_fx != 0.0f) Fx = add2(Fx, all<V>(ph.f.body_fx));
}

// f* = M^{-1} m* from raw moments m20 .. m22 (m10, m01 and the sum rho of all; f0_of(s8): f*_0 from the sum of
// the other eight).  out(i, f*_i): called as each population is ready.
template <typename V, typename F0, typename Out>
__device__ __forceinline__ void populations_of(V m10, V m01, V m20, V m02, V m11, V m21, V m12, V m22, const F0& f0_of,
                                               const Out& out) {
  const V px = sub2(m20, m22), py = sub2(m02, m22);
  out(0, f0_of(add2(m20, py)));
  const V hpx = mul2(all<V>(0.5f), px), qx = sub2(m10, m12);
  out(1, fma2(all<V>(0.5f), qx, hpx));
  out(2, fma2(all<V>(-0.5f), qx, hpx));
  const V hpy = mul2(all<V>(0.5f), py), qy = sub2(m01, m21);
  out(3, fma2(all<V>(0.5f), qy, hpy));
  out(4, fma2(all<V>(-0.5f), qy, hpy));
  const V sp = mul2(all<V>(0.25f), add2(m22, m11)), tp = add2(m21, m12);
  out(5, fma2(all<V>(0.25f), tp, sp));
  out(6, fma2(all<V>(-0.25f), tp, sp));
  const V sm = mul2(all<V>(0.25f), sub2(m22, m11)), tm = sub2(m12, m21);
  out(7, fma2(all<V>(0.25f), tm, sm));
  out(8, fma2(all<V>(-0.25f), tm, sm));
}

// CM collision (Eq. postColl2).  aF = alpha |F_m|^2 with alpha = sigma / psi^2.
// The central moments that relax, with h = F / 2 and u = (m1 + h_x) / rho:
//   k4 = m4 - u (m1 - h_x) + v (m2 - h_y),   k5 = m5 - v m1 + u h_y.
// Raw moments from the post-collision central moments K_ab one axis at a time:
//   M_1b = K_1b + u K_0b,  M_2b = K_2b + u (K_1b + M_1b), then the same with v over b;
// M_10 = m1 + F_x and M_01 = m2 + F_y hold exactly.  f*_0 is f_0 less what the other eight gain
// (their sum after is M_20 + M_02 - M_22): taken from the rounded rho, a quiet liquid's mass drifts by
// up to half of rho's last place a step, the same at every node.
template <typename V, typename Out>
__device__ __forceinline__ void collide_cm(const StepConst& k, const Moments<V>& M, V Fx, V Fy, V aF, V& ux, V& uy,
                                           const Out& out) {
  const V rho = M.rho, m1 = M.m1, m2 = M.m2;
  const V ir = rcp2(rho), hx = mul2(all<V>(0.5f), Fx), hy = mul2(all<V>(0.5f), Fy);
  const V u = mul2(add2(m1, hx), ir), v = mul2(add2(m2, hy), ir);
  const V nu = mul2(all<V>(-1.0f), u), nv = mul2(all<V>(-1.0f), v);
  const V k4 = fma2(nu, sub2(m1, hx), fma2(v, sub2(m2, hy), M.m4));
  const V k5 = fma2(nv, m1, fma2(u, hy, M.m5));
  // 1 - omega = (3 nu - 1/2) / (3 nu + 1/2), nu linear in the phase fraction
  const V n3 = fma2(satfma(rho, k.ph1, k.ph0), all<V>(k.dn3), all<V>(k.nv3));
  const V om = mul2(add2(n3, all<V>(-0.5f)), rcp2(add2(n3, all<V>(0.5f))));
  const V ks4 = mul2(om, k4), K11 = mul2(om, k5);
  const V base = fma2(all<V>(1.0f / 3.0f), rho, aF);
  const V K20 = fma2(all<V>(0.5f), ks4, base), K02 = fma2(all<V>(-0.5f), ks4, base);
  const V K21 = mul2(all<V>(1.0f / 6.0f), Fy), K12 = mul2(all<V>(1.0f / 6.0f), Fx);
  const V K22 = fma2(all<V>(2.0f / 3.0f), aF, mul2(all<V>(1.0f / 9.0f), rho));
  // x axis
  const V m10 = add2(m1, Fx), m01 = add2(m2, Fy);
  const V m20 = fma2(u, add2(hx, m10), K20);
  const V M11 = fma2(u, hy, K11), M21 = fma2(u, add2(K11, M11), K21);
  const V M12 = fma2(u, K02, K12), M22 = fma2(u, add2(K12, M12), K22);
  // y axis
  const V m02 = fma2(v, add2(hy, m01), K02);
  const V m11 = fma2(v, m10, M11), m12 = fma2(v, add2(M11, m11), M12);
  const V m21 = fma2(v, m20, M21), m22 = fma2(v, add2(M21, m21), M22);
  populations_of(m10, m01, m20, m02, m11, m21, m12, m22, [&](V s8) { return add2(M.f0, sub2(M.sum8, s8)); }, out);
  ux = u;
  uy = v;
}

// Single-rate BGK operator on the same equilibrium and forcing (Sec. III.B; collide_bgk of lbm_kernels.cuh has
// the derivation): f* = (1 - omega) f + M^{-1} N(u)^{-1} k' with k' = omega k^eq + (1 - omega / 2) R.
template <typename V, typename Out>
__device__ __forceinline__ void collide_bgk_of(const StepConst& k, const V f[9], const Moments<V>& M, V Fx, V Fy, V& ux,
                                               V& uy, const Out& out) {
  const V ir = rcp2(M.rho);
  const V u = mul2(fma2(all<V>(0.5f), Fx, M.m1), ir), v = mul2(fma2(all<V>(0.5f), Fy, M.m2), ir);
  const V n3 = fma2(satfma(M.rho, k.ph1, k.ph0), all<V>(k.dn3), all<V>(k.nv3));
  const V omega = rcp2(add2(n3, all<V>(0.5f)));
  const V r = sub2(all<V>(1.0f), omega);  // exact: r + omega = 1, or the mass would drift
  const V cf = fma2(all<V>(-0.5f), omega, all<V>(1.0f));
  const V K00 = mul2(omega, M.rho), K10 = mul2(cf, Fx), K01 = mul2(cf, Fy);
  const V K20 = mul2(all<V>(1.0f / 3.0f), K00), K22 = mul2(all<V>(1.0f / 9.0f), K00);  // K02 = K20, K11 = 0
  const V K21 = mul2(all<V>(1.0f / 3.0f), K01), K12 = mul2(all<V>(1.0f / 3.0f), K10);
  // x axis
  const V m10 = fma2(u, K00, K10), m20 = fma2(u, add2(K10, m10), K20);
  const V M11 = mul2(u, K01), M21 = fma2(u, M11, K21);
  const V M12 = fma2(u, K20, K12), M22 = fma2(u, add2(K12, M12), K22);
  // y axis
  const V m01 = fma2(v, K00, K01), m02 = fma2(v, add2(K01, m01), K20);
  const V m11 = fma2(v, m10, M11), m12 = fma2(v, add2(M11, m11), M12);
  const V m21 = fma2(v, m20, M21), m22 = fma2(v, add2(M21, m21), M22);
  populations_of(m10, m01, m20, m02, m11, m21, m12, m22, [&](V s8) { return sub2(K00, s8); },
                 [&](int i, V g) { out(i, fma2(r, f[i], g)); });
  ux = u;
  uy = v;
}

}  // namespace kern
}  // namespace lbm
