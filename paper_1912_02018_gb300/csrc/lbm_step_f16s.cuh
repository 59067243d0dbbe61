// Step kernels of the FP32 arithmetic over shifted FP16 populations (LBM_STORE_F16S; included by
// lbm_kernels.cuh): the collision operator and the energy pass.  A stored population keeps 11 bits,
// so a last-bit difference anywhere in the step flips stored roundings, and a run's velocities then
// differ by 1e-3 within a hundred steps.  These kernels therefore keep one order of operations for good:
// one lane per node in the collision (collide_tile of lbm_kernels.cuh, 32 x 8 tiles), a lane per
// pair in the 32 x 16 energy tiles, whose last part makes psi of the next step.  The reordered
// passes of lbm_flow_f32.cuh, lbm_collide_f32.cuh and lbm_energy_f32.cuh serve FP32 and FP64 populations only.
#pragma once

namespace lbm {
namespace kern {

// The collision of one node with every rounding written out (explicit fma, mul, add), so that the
// result does not depend on which kernel inlines it.  Forward substitution of N(u) m* = k*
// in closed form; m*_1 = k*_1 + u rho = m1 + Fx and m*_2 = m2 + Fy hold exactly since
// u rho = m1 + Fx / 2.
template <>
__device__ __forceinline__ void collide<float>(const float f[9], float rho, float Fx, float Fy, float Fmx, float Fmy,
                                               float psi, float omega, float sigma, float fs[9], float& ux,
                                               float& uy) {
  const float a56 = __fsub_rn(f[5], f[6]), a78 = __fsub_rn(f[7], f[8]);
  const float m1 = __fadd_rn(__fadd_rn(__fsub_rn(f[1], f[2]), a56), a78);
  const float m2 = __fsub_rn(__fadd_rn(__fsub_rn(f[3], f[4]), a56), a78);
  const float m4 = __fsub_rn(__fadd_rn(f[1], f[2]), __fadd_rn(f[3], f[4]));
  const float m5 = __fsub_rn(__fadd_rn(f[5], f[6]), __fadd_rn(f[7], f[8]));
  const float u = __fdividef(__fmaf_rn(0.5f, Fx, m1), rho), v = __fdividef(__fmaf_rn(0.5f, Fy, m2), rho);
  ux = u;
  uy = v;
  const float uu = __fmul_rn(u, u), vv = __fmul_rn(v, v), uv = __fmul_rn(u, v);
  const float s2 = __fadd_rn(uu, vv), d2 = __fsub_rn(uu, vv), u2 = __fmul_rn(2.0f, u), v2 = __fmul_rn(2.0f, v);
  // central moments k4, k5 of the pre-collision populations (Eq. (postColl2) shift)
  const float k4 = __fmaf_rn(d2, rho, __fmaf_rn(v2, m2, __fmaf_rn(-u2, m1, m4)));
  const float k5 = __fmaf_rn(uv, rho, __fmaf_rn(-v, m1, __fmaf_rn(-u, m2, m5)));
  // post-collision central moments with the consistency terms alpha |Fm|^2
  const float alpha = sigma != 0.0f ? __fdividef(sigma, __fmul_rn(psi, psi)) : 0.0f;
  const float aF = __fmul_rn(alpha, __fmaf_rn(Fmx, Fmx, __fmul_rn(Fmy, Fmy)));
  const float om = __fsub_rn(1.0f, omega);
  const float ks3 = __fmaf_rn(2.0f, aF, __fmul_rn(2.0f / 3.0f, rho));
  const float ks4 = __fmul_rn(om, k4), ks5 = __fmul_rn(om, k5);
  const float ks6 = __fmul_rn(1.0f / 6.0f, Fy), ks7 = __fmul_rn(1.0f / 6.0f, Fx);
  const float ks8 = __fmaf_rn(2.0f / 3.0f, aF, __fmul_rn(1.0f / 9.0f, rho));
  // raw moments m* = N(u)^{-1} k*
  const float ms1 = __fadd_rn(m1, Fx), ms2 = __fadd_rn(m2, Fy);
  const float ms3 = __fmaf_rn(u2, ms1, __fmaf_rn(v2, ms2, __fmaf_rn(-s2, rho, ks3)));
  const float ms4 = __fmaf_rn(u2, ms1, __fmaf_rn(-v2, ms2, __fmaf_rn(-d2, rho, ks4)));
  const float ms5 = __fmaf_rn(v, ms1, __fmaf_rn(u, ms2, __fmaf_rn(-uv, rho, ks5)));
  const float uv2 = __fmul_rn(2.0f, uv);
  const float ms6 = __fmaf_rn(u2, ms5, __fmaf_rn(__fmul_rn(0.5f, v), __fadd_rn(ms3, ms4),
                              __fmaf_rn(-uu, ms2, __fmaf_rn(-uv2, ms1, __fmaf_rn(__fmul_rn(uu, v), rho, ks6)))));
  const float ms7 = __fmaf_rn(v2, ms5, __fmaf_rn(__fmul_rn(0.5f, u), __fsub_rn(ms3, ms4),
                              __fmaf_rn(-uv2, ms2, __fmaf_rn(-vv, ms1, __fmaf_rn(__fmul_rn(u, vv), rho, ks7)))));
  const float ms8 = __fmaf_rn(
      u2, ms7,
      __fmaf_rn(v2, ms6,
                __fmaf_rn(__fmul_rn(-2.0f, uv2), ms5,
                          __fmaf_rn(__fmul_rn(0.5f, d2), ms4,
                                    __fmaf_rn(__fmul_rn(-0.5f, s2), ms3,
                                              __fmaf_rn(__fmul_rn(uv2, u), ms2,
                                                        __fmaf_rn(__fmul_rn(uv2, v), ms1,
                                                                  __fmaf_rn(-__fmul_rn(uu, vv), rho, ks8))))))));
  // f* = M^{-1} m*
  const float A = __fmul_rn(0.25f, __fadd_rn(ms3, ms4)), B = __fmul_rn(0.25f, __fsub_rn(ms3, ms4));
  const float c = __fmaf_rn(-0.5f, ms8, A), e = __fmaf_rn(-0.5f, ms8, B);
  const float d = __fmul_rn(0.5f, __fsub_rn(ms1, ms7)), gy = __fmul_rn(0.5f, __fsub_rn(ms2, ms6));
  fs[0] = __fadd_rn(__fsub_rn(rho, ms3), ms8);
  fs[1] = __fadd_rn(c, d);
  fs[2] = __fsub_rn(c, d);
  fs[3] = __fadd_rn(e, gy);
  fs[4] = __fsub_rn(e, gy);
  const float sp = __fadd_rn(ms5, ms8), tp = __fadd_rn(ms6, ms7), wm = __fsub_rn(ms8, ms5), zm = __fsub_rn(ms6, ms7);
  fs[5] = __fmul_rn(0.25f, __fadd_rn(sp, tp));
  fs[6] = __fmul_rn(0.25f, __fsub_rn(sp, tp));
  fs[7] = __fmul_rn(0.25f, __fsub_rn(wm, zm));
  fs[8] = __fmul_rn(0.25f, __fadd_rn(wm, zm));
}

// Eq. (energy) splits into parts that depend on rho and u only, frozen during the step
// (lambda, grad lambda, div u), and parts that depend on the temperature being advanced.
struct FrozenNode {
  float lam0, lx, ly, divu;
};
// FP32: the two nodes of a pair are one packed float2 throughout the stencil sums (sm_100+
// FFMA2/FADD2/FMUL2), halving the FP32 instructions of the energy pass.  The window of a pair
// is kept as aligned column pairs A[r][j] = (c_2j, c_2j+1) and shifted pairs B[r][j] =
// (c_2j+1, c_2j+2); the value pair at offset ex is A[r][1 + ex/2] for even ex, B[r][(1 + ex)/2]
// for odd ex.  Each packed operation rounds like the scalar one it replaces.
struct Win2 {
  float2 A[5][3], B[5][2];
};
__device__ __forceinline__ void load_win2(const float* p, int s, Win2& W) {
#pragma unroll
  for (int r = 0; r < 5; ++r) {
    const float2* q = reinterpret_cast<const float2*>(p + (r - 2) * s - 2);
#pragma unroll
    for (int c = 0; c < 3; ++c) W.A[r][c] = q[c];
    W.B[r][0] = make_float2(W.A[r][0].y, W.A[r][1].x);
    W.B[r][1] = make_float2(W.A[r][1].y, W.A[r][2].x);
  }
}
__device__ __forceinline__ float2 win_at(const Win2& W, int r, int ex) {
  return (ex & 1) ? W.B[r][(1 + ex) / 2] : W.A[r][1 + ex / 2];
}
template <bool kX = true, bool kY = true>
__device__ __forceinline__ void grad_w2(const Win2& W, float2& gx, float2& gy) {
  float2 sx = f2(0.f), sy = f2(0.f);
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const int ex = exv(k), ey = eyv(k);
    if ((kX && ex != 0) || (kY && ey != 0)) {
      const float2 d = sub2(win_at(W, 2 + ey, ex), win_at(W, 2 - ey, -ex));
      if (kX && ex != 0) sx = __ffma2_rn(f2(float(wiso(k) * ex)), d, sx);
      if (kY && ey != 0) sy = __ffma2_rn(f2(float(wiso(k) * ey)), d, sy);
    }
  }
  gx = sx;
  gy = sy;
}
__device__ __forceinline__ float2 lap_w2(const Win2& W) {
  const float2 c = W.A[2][1];
  float2 acc = f2(0.f);
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const int ex = exv(k), ey = eyv(k);
    const float2 d = __ffma2_rn(c, f2(-2.f), __fadd2_rn(win_at(W, 2 + ey, ex), win_at(W, 2 - ey, -ex)));
    acc = __ffma2_rn(f2(float(wiso(k))), d, acc);
  }
  return __fmul2_rn(f2(2.f), acc);
}
// Six times the third-order upwind derivative of the pair along x (row 2) or y (column pair
// 1), each node biased against the sign of its own velocity v.
__device__ __forceinline__ float2 upwind6_w2(const Win2& W, bool along_x, float2 v) {
  float2 q[5];
#pragma unroll
  for (int o = -2; o <= 2; ++o) q[o + 2] = along_x ? win_at(W, 2, o) : W.A[2 + o][1];
  const float2 c = q[2];
  const float2 m2 = sub2(q[0], c), m1 = sub2(q[1], c), p1 = sub2(q[3], c), p2 = sub2(q[4], c);
  const float2 pos = __ffma2_rn(f2(2.f), p1, __ffma2_rn(f2(-6.f), m1, m2));
  const float2 neg = sub2(__ffma2_rn(f2(6.f), p1, __fmul2_rn(f2(-2.f), m1)), p2);
  return make_float2(v.x >= 0.f ? pos.x : neg.x, v.y >= 0.f ? pos.y : neg.y);
}
__device__ __forceinline__ void frozen_pair(const float* lam, const float* u, const float* v, int as,
                                                   FrozenNode fz[2]) {
  Win2 W;
  float2 lx, ly, dxux, dyuy, unused;
  load_win2(lam, as, W);
  fz[0].lam0 = W.A[2][1].x;
  fz[1].lam0 = W.A[2][1].y;
  grad_w2(W, lx, ly);
  load_win2(u, as, W);
  grad_w2<true, false>(W, dxux, unused);
  load_win2(v, as, W);
  grad_w2<false, true>(W, unused, dyuy);
  const float2 dv = __fadd2_rn(dxux, dyuy);
  fz[0].lx = lx.x, fz[0].ly = ly.x, fz[0].divu = dv.x;
  fz[1].lx = lx.y, fz[1].ly = ly.y, fz[1].divu = dv.y;
}
__device__ __forceinline__ float2 pk_div(float2 a, float2 b) {
  return make_float2(__fdividef(a.x, b.x), __fdividef(a.y, b.y));
}
__device__ __forceinline__ void energy_rhs_pair(const Phys& ph, const float* t, int ts, const float* u,
                                                       const float* v, const float* r, const FrozenNode fz[2],
                                                       float L[2]) {
  Win2 W;
  load_win2(t, ts, W);
  const float2 u2 = make_float2(u[0], u[1]), v2 = make_float2(v[0], v[1]);
  const float2 conv6 = __ffma2_rn(u2, upwind6_w2(W, true, u2), __fmul2_rn(v2, upwind6_w2(W, false, v2)));
  float2 gx, gy;
  grad_w2(W, gx, gy);
  const float2 lap = lap_w2(W);
  const float2 diff = __ffma2_rn(make_float2(fz[0].lam0, fz[1].lam0), lap,
                                 __ffma2_rn(make_float2(fz[0].lx, fz[1].lx), gx,
                                            __fmul2_rn(make_float2(fz[0].ly, fz[1].ly), gy)));
  // (dp/dT)_rho of Eq. (eos) with phi = (1 + kappa (1 - sqrt(T/Tc)))^2, dphi/dT = -kappa
  // sqrt(phi) / sqrt(T Tc):  rep + att (kappa (1 + kappa) / sqrt(T Tc) - kappa^2 / Tc), with
  // rep = rho R / (1 - b rho) and att = a rho^2 / (1 + 2 b rho - b^2 rho^2)
  const PhysC<float>& k = ph.f;
  const float2 rho = make_float2(r[0], r[1]), T0 = W.A[2][1];
  const float2 rep = pk_div(__fmul2_rn(f2(k.R), rho), __ffma2_rn(f2(-k.b), rho, f2(1.0f)));
  const float2 att = pk_div(__fmul2_rn(__fmul2_rn(f2(k.a), rho), rho),
                            __ffma2_rn(rho, __ffma2_rn(f2(-k.b * k.b), rho, f2(2.0f * k.b)), f2(1.0f)));
  const float2 rs = make_float2(rsqrtf(T0.x * k.Tc), rsqrtf(T0.y * k.Tc));
  const float2 dpdT = __ffma2_rn(att, __ffma2_rn(f2(ph.dpdT_c1), rs, f2(-ph.dpdT_c2)), rep);
  const float2 work = __fmul2_rn(__fmul2_rn(T0, dpdT), make_float2(fz[0].divu, fz[1].divu));
  const float2 Lp = __ffma2_rn(sub2(diff, work), pk_div(f2(1.0f), __fmul2_rn(f2(k.c_v), rho)),
                               __fmul2_rn(f2(-1.0f / 6.0f), conv6));
  L[0] = Lp.x;
  L[1] = Lp.y;
}

// Heun stage 2 at the pair whose left node is (x, y), T^{n+1} = (T + T1 + L(T1)) / 2, from
// shared tiles: inputs sT, sL, sU, sV, sR, sM (row stride ax, pair at index a) and the stage-1
// temperature sT1 (row stride bx, pair at index b); fz: the pair's frozen parts.  Nodes with
// x >= nx or y >= ylim are skipped.  Writes T^{n+1} and, with psi_out,
// psi of the next step from the pull of the new populations fnew, side_new (Eq. potential);
// adds the pair's wall heat flux -lambda grad T^n . n (Sec. IV.B) to q and sets mine when
// the pair holds a near-wall node.
template <int PSI>
__device__ __forceinline__ void stage2_pair(const Geo& g, const Phys& ph, const float* sT, const float* sL, const float* sU,
                                            const float* sV, const float* sR, const uint8_t* sM, int ax, int a, const float* sT1,
                                            int bx, int b, const FrozenNode* fz_in, int x0, int y, int ylim,
                                            float* __restrict__ Tout, int do_hf,
                                            const __half* __restrict__ fnew, const uint8_t* __restrict__ mask,
                                            const float* __restrict__ side_new, float* __restrict__ psi_out, int* status,
                                            double& q, int& mine) {
  const FrozenNode fz[2] = {fz_in[0], fz_in[1]};
  float L[2];
  energy_rhs_pair(ph, &sT1[b], bx, &sU[a], &sV[a], &sR[a], fz, L);
  float tnew[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int x = x0 + k;
    if (x < g.nx && y < ylim) {
      float out;
      if (sM[a + k] & kSolid) out = sT[a + k];
      else if (!g.periodic_x && x == 0) out = pc<float>(ph).T_sat;
      else out = ((sT[a + k] + sT1[b + k]) + L[k]) * 0.5f;
      Tout[y * g.pitch + x] = out;
      tnew[k] = out;
      if (do_hf && (sM[a + k] & kNearWall)) {
        float gx, gy;
        grad_t(&sT[a + k], ax, gx, gy);
        const double* nv = &g.wall_n[2 * g.wall_idx[y * g.pitch + x]];
        q += -(double)sL[a + k] * ((double)gx * nv[0] + (double)gy * nv[1]);
        mine = 1;
      }
    }
  }
  if (psi_out) {
    const uint8_t m0 = sM[a], m1 = sM[a + 1];
    float r[2];
    // a pair away from the wall, the open edges and the periodic seams pulls from one base
    // address; the others take the general pull with its boundary substitutions
    if (!((m0 | m1) & kNearWall) && y >= 1 && y + 1 < g.ny && x0 >= 1 && x0 + 3 <= g.nx) {
      pair_rho<float, __half>(g, ph, fnew, x0, y, r);
    } else {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        r[k] = 0.0f;
        if (x0 + k < g.nx && y < ylim) {
          float fo[9];
          pull_node<float, __half>(g, ph, fnew, mask, side_new, nullptr, x0 + k, y, k ? m1 : m0, fo);
          float t = fo[0];
#pragma unroll
          for (int i = 1; i < 9; ++i) t = t + fo[i];
          r[k] = t;
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int x = x0 + k;
      if (x < g.nx && y < ylim) {
        const float rho = ((k ? m1 : m0) & kSolid) ? pc<float>(ph).rho_s : r[k];
        psi_out[y * g.pitch + x] = psi_of<float, PSI>(ph, rho, tnew[k], status);
      }
    }
  }
}

// 32 x 16 tiles, a lane per pair
struct EnergyTile16 {
  static constexpr int TX = 32, TY = 16, NT = TX * TY / 2;
};

// Both Heun stages on tile (bx, by); bid, nblocks: this tile's index among the domain's
// nblocks tiles (for the heat-flux partials and the last-block reduction).
// With psi_out set the tile also evaluates psi of the next step at its nodes: the
// pull of the populations this step's collision wrote (fnew, side_new), rho their sum (rho_s
// in the solid), T the new temperature (Eq. potential) -- the next step then needs no psi pass.
// maps: tensor maps of the inputs, with which an interior tile stages them by TMA (else null:
// plain loads).
template <int PSI>
__device__ __forceinline__ void energy_tile16(const Geo& g, const Phys& ph, const float* __restrict__ Tin,
                                            float* __restrict__ Tout, const float* __restrict__ rho, const float* __restrict__ ux,
                                            const float* __restrict__ uy, const uint8_t* __restrict__ mask,
                                            double* partial, unsigned* counter, double* hf, int nb, int do_hf,
                                            int n_wall_tiles, int bx, int by, int bid, int nblocks,
                                            const __half* __restrict__ fnew, const float* __restrict__ side_new,
                                            float* __restrict__ psi_out, int* status, const EnergyMaps* maps, bool starve) {
  constexpr int TX = EnergyTile16::TX, TY = EnergyTile16::TY, NT = EnergyTile16::NT;
  constexpr int H = 4, AX = TX + 2 * H, AY = TY + 2 * H;  // inputs: tile + 4
  constexpr int BX = TX + 4, BY = TY + 4;                 // stage 1: tile + 2
  static_assert(AX * AY * sizeof(float) % 128 == 0 && AX * sizeof(float) % 16 == 0, "TMA boxes of the input tile");
  static_assert(AX % 4 == 0 && (AX * AY) % 4 == 0, "word-wise mask and float4 lambda staging");
  __shared__ __align__(128) float sT[AY * AX];
  __shared__ __align__(128) float sL[AY * AX];
  __shared__ __align__(128) float sRUV[3 * AY * AX];  // rho, u_x, u_y: the planes of one TMA box
  float* const sR = sRUV;
  float* const sU = sRUV + AY * AX;
  float* const sV = sRUV + 2 * AY * AX;
  __shared__ uint64_t s_bar;
  __shared__ __align__(16) float sT1[BY * BX];
  __shared__ FrozenNode sF[TX * TY];
  __shared__ __align__(16) uint8_t sM[AY * AX];
  __shared__ double red[NT / 32];
  __shared__ int done_last;
  const int tid = threadIdx.x;
  const int x0 = bx * TX, y0 = by * TY;
  const bool interior = x0 >= H && y0 >= H && x0 + TX + H <= g.nx && y0 + TY + H <= g.ny;
  if (maps && interior) {
    // the input boxes by TMA (T; rho, u_x, u_y in one 3-plane box; first column x0 - 4:
    // 16-byte aligned); the mask with plain
    // loads while they fly; lambda(rho) once rho has landed
    if (tid == 0) tma::bar_init(&s_bar, 1);
    __syncthreads();
    if (tid == 0) {
      tma::bar_expect_tx(&s_bar, 4 * AX * AY * sizeof(float));
      // T comes from the energy pass before the previous kernel (the collision, which does not
      // write it): its copy starts before that kernel ends; the test hook leaves the barrier
      // armed with no copy issued
      if (!starve) tma::load_2d(sT, &maps->T, &s_bar, x0 - H, y0 - H);
    }
    // the mask as 32-bit words (x0 - 4 and the row pitch are multiples of 4 bytes)
    for (int p = tid; p < (AX / 4) * AY; p += NT) {
      const int r = p / (AX / 4), c = p - r * (AX / 4);
      reinterpret_cast<uint32_t*>(sM)[p] =
          *reinterpret_cast<const uint32_t*>(mask + (y0 + r - H) * g.pitch + x0 - H + 4 * c);
    }
    pdl::wait();  // rho, u and the new populations are the collision's output
    pdl::trigger();
    if (tid == 0 && !starve) tma::load_3d(sRUV, &maps->ruv, &s_bar, x0 - H, y0 - H, 0);
    const int tries = starve ? tma::kStarveTries : tma::kWaitTries;
    const bool landed = tma::bar_wait(&s_bar, 0, tries);
    if (__syncthreads_or(!landed)) {
      // a copy did not land in time: report it, let the copies land (bounded) and stop the tile
      // (a tile that holds wall nodes then misses its heat-flux partial; restoring a state with
      // lbm_set_state resets that bookkeeping)
      if (tid == 0) atomicOr(status, kStatusTimeoutEnergy);
      tma::bar_wait(&s_bar, 0, tries);
      return;
    }
    for (int p = tid; p < AX * AY / 4; p += NT) {  // four nodes per thread
      const float4 r4 = reinterpret_cast<const float4*>(sR)[p];
      reinterpret_cast<float4*>(sL)[p] =
          make_float4(lam_of(ph, r4.x), lam_of(ph, r4.y), lam_of(ph, r4.z), lam_of(ph, r4.w));
    }
  } else {
    pdl::wait();
    pdl::trigger();
    for (int p = tid; p < AX * AY; p += NT) {
      const int gx = x0 + p % AX - H, gy = y0 + p / AX - H;
      const int nid = interior ? gy * g.pitch + gx : map_y(g, gy) * g.pitch + map_x(g, gx);
      const float r = rho[nid];
      sT[p] = Tin[nid];
      sR[p] = r;
      sL[p] = lam_of(ph, r);
      sU[p] = ux[nid];
      sV[p] = uy[nid];
      sM[p] = mask[nid];
    }
  }
  __syncthreads();
  // stage 1: T1 = T + L(T) on the tile and a 2-node halo, two nodes per thread; the frozen
  // parts of the tile's own nodes are kept for stage 2
  for (int p = tid; p < (BX / 2) * BY; p += NT) {
    const int by = p / (BX / 2), bx = (p % (BX / 2)) * 2;
    const int a = (by + 2) * AX + bx + 2;
    FrozenNode fz[2];
    frozen_pair(&sL[a], &sU[a], &sV[a], AX, fz);
    float L[2];
    energy_rhs_pair(ph, &sT[a], AX, &sU[a], &sV[a], &sR[a], fz, L);
    const int tx = bx - 2, ty = by - 2;
    if (tx >= 0 && tx < TX && ty >= 0 && ty < TY) {
      sF[ty * TX + tx] = fz[0];
      sF[ty * TX + tx + 1] = fz[1];
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int gx = x0 + bx + k - 2;
      float t1;
      if (sM[a + k] & kSolid) t1 = sT[a + k];  // solid nodes keep their wall temperature
      else if (!g.periodic_x && gx == 0) t1 = pc<float>(ph).T_sat;
      else t1 = sT[a + k] + L[k];
      sT1[by * BX + bx + k] = t1;  // positions past a non-periodic edge are replaced below
    }
  }
  __syncthreads();
  if (!g.periodic_x && (x0 < 2 || x0 + TX + 2 > g.nx)) {
    for (int p = tid; p < BX * BY; p += NT) {
      const int bx = p % BX, by = p / BX;
      const int gx = x0 + bx - 2;
      if (gx < 0 || gx >= g.nx) sT1[p] = sT1[by * BX + (map_x(g, gx) - x0 + 2)];
    }
    __syncthreads();
  }
  // stage 2 on the tile: T^{n+1} = (T + T1 + L(T1)) / 2
  const int tx = (tid % (TX / 2)) * 2, ty = tid / (TX / 2);
  double q = 0.0;
  int mine = 0;
  stage2_pair<PSI>(g, ph, sT, sL, sU, sV, sR, sM, AX, (ty + H) * AX + tx + H, sT1, BX,
                               (ty + 2) * BX + tx + 2, &sF[ty * TX + tx], x0 + tx, y0 + ty, g.ny, Tout, do_hf,
                               fnew, mask, side_new, psi_out, status, q, mine);
  if (do_hf) heat_flux_blocks<NT>(q, mine, partial, counter, n_wall_tiles, bid, nblocks, hf, nb, red, &done_last);
}
// 64 registers and 4 blocks per SM: the conversions of the psi pull need them (no spills)
template <int PSI>
__global__ void __launch_bounds__(EnergyTile16::NT, 4)
    k_energy_f16s(Geo g, Phys ph, const float* __restrict__ Tin, float* __restrict__ Tout,
                  const float* __restrict__ rho, const float* __restrict__ ux, const float* __restrict__ uy,
                  const uint8_t* __restrict__ mask, double* partial, unsigned* counter, double* hf, int nb, int do_hf,
                  int n_wall_tiles, const __half* __restrict__ fnew, const float* __restrict__ side_new,
                  float* __restrict__ psi_out, int* status, const __grid_constant__ EnergyMaps maps, int flags) {
  energy_tile16<PSI>(g, ph, Tin, Tout, rho, ux, uy, mask, partial, counter, hf, nb, do_hf, n_wall_tiles, blockIdx.x,
                     blockIdx.y, blockIdx.y * gridDim.x + blockIdx.x, gridDim.x * gridDim.y, fnew, side_new, psi_out,
                     status, (flags & kLaunchStaged) ? &maps : nullptr, (flags & kLaunchStarve) != 0);
}

}  // namespace kern
}  // namespace lbm
