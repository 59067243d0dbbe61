// FP32 collision pass of one lattice tile: pull-streaming, rho, psi, interaction force and the CM
// (or BGK) collision (Sec. II.A-B, Sec. IV.A; included by lbm_step_f32.cuh).
//
// Tile: 64 - 2H columns by TY rows with a halo of H = 2 nodes where psi is needed (H = 0 for a
// single-phase fluid).  One warp covers one row of 64 columns, two per lane, so a block is TY + 2H
// warps.  Phase 1: every lane pulls its pair from the populations staged in shared memory (by TMA
// inside the lattice) and evaluates psi of it, the halo rows too, into a shared tile.  Phase 2: the
// warps of the own rows take the force from the psi tile and collide the moments they still hold in
// registers.
//
// Bound by the latency of a block (900 cycles of prologue, 2700 of the copy, 1600 pull, 1400 psi, 1000
// barrier, 1500 collision, 850 stores; two blocks of 16 warps on an SM): 58 us for collision and psi
// at 2048 x 1024, where the one-node-per-lane collision took 38 us and the psi that the energy pass
// made for it 27 us more.  8 to 16 rows, 2 to 4 blocks and a persistent grid that prefetches the
// next tile lie within 5% of it; 64 own columns with a wider halo take 62 us.
//
// psi in the tile (kFlowTile) evaluates psi at 1.42 nodes per node, and reads each population once
// per step (the halo comes from L2).  The other way (kFlowRead) loads psi from global memory, made by the energy pass of the
// step before from a second pull of the populations.
//
// The arithmetic is packed FP32x2 with every rounding written out, so that all variants give the
// same bits.
#pragma once

namespace lbm {
namespace kern {

// Where psi of the collision comes from: nowhere (single phase), global memory, the tile itself.
enum FlowMode { kFlowNone = 0, kFlowRead = 1, kFlowTile = 2 };

__device__ __forceinline__ void pair_set(float2& v, int i, float x) {
  if (i == 0) v.x = x;
  else v.y = x;
}
__device__ __forceinline__ float pair_get(float2 v, int i) { return i == 0 ? v.x : v.y; }

// A pair of populations to storage.
template <typename S>
struct PairStore;
template <>
struct PairStore<float> {
  static __device__ __forceinline__ void st(float* q, float2 v, int, const Phys&) {
    *reinterpret_cast<float2*>(q) = v;
  }
};
template <>
struct PairStore<double> {
  static __device__ __forceinline__ void st(double* q, float2 v, int, const Phys&) {
    *reinterpret_cast<double2*>(q) = make_double2((double)v.x, (double)v.y);
  }
};

// Moments of a pair's pulled populations that the collision keeps: rho (in the order of pop_sum),
// m1, m2, m4, m5 (App. A), and f_0 and the sum of the other eight.
struct PairMoments {
  float2 rho, m1, m2, m4, m5, f0, sum8;
};
__device__ __forceinline__ PairMoments moments_pair(const float2 f[9]) {
  const float2 s12 = add2(f[1], f[2]), s34 = add2(f[3], f[4]), s56 = add2(f[5], f[6]), s78 = add2(f[7], f[8]);
  const float2 d56 = sub2(f[5], f[6]), d78 = sub2(f[7], f[8]);
  PairMoments M;
  const float2 s14 = add2(s12, s34), s58 = add2(s56, s78);
  M.rho = add2(add2(f[0], s14), s58);
  M.f0 = f[0];
  M.sum8 = add2(s14, s58);
  M.m1 = add2(add2(sub2(f[1], f[2]), d56), d78);
  M.m2 = sub2(add2(sub2(f[3], f[4]), d56), d78);
  M.m4 = sub2(s12, s34);
  M.m5 = sub2(s56, s78);
  return M;
}
// rho alone.
__device__ __forceinline__ float2 pop_sum2(const float2 f[9]) {
  return add2(add2(f[0], add2(add2(f[1], f[2]), add2(f[3], f[4]))), add2(add2(f[5], f[6]), add2(f[7], f[8])));
}

// Force of a column pair: F_m = -G cs^2 psi grad psi (Eq. interForce; gx, gy the stencil sums) and
// F = F_m + gravity (+ the body force).
__device__ __forceinline__ void force_pair(const Phys& ph, float2 rho, float2 psi, float2 gx, float2 gy, float2& Fx,
                                           float2& Fy) {
  const StepConst& k = ph.sc;
  const float2 a = mul2(f2(k.gm), psi);
  Fx = fma2(f2(-ph.f.g), sub2(rho, f2(ph.f.rho_l)), mul2(a, gx));
  Fy = mul2(a, gy);
  if (ph.f.body_fx != 0.0f) Fx = add2(Fx, f2(ph.f.body_fx));
}

// CM collision of a column pair (Eq. postColl2).  aF = alpha |F_m|^2 with alpha = sigma / psi^2.
// The central moments that relax, with h = F / 2 and u = (m1 + h_x) / rho:
//   k4 = m4 - u (m1 - h_x) + v (m2 - h_y),   k5 = m5 - v m1 + u h_y.
// Raw moments from the post-collision central moments K_ab one axis at a time:
//   M_1b = K_1b + u K_0b,  M_2b = K_2b + u (K_1b + M_1b), then the same with v over b;
// M_10 = m1 + F_x and M_01 = m2 + F_y hold exactly.  f*_0 is f_0 less what the other eight gain
// (their sum after is M_20 + M_02 - M_22): taken from the rounded rho, a quiet liquid's mass drifts by
// up to half of rho's last place a step, the same at every node.
// out(i, f*_i): called as each population is ready.
template <typename Out>
__device__ __forceinline__ void collide_pair(const StepConst& k, const PairMoments& M, float2 Fx, float2 Fy, float2 aF,
                                             float2& ux, float2& uy, const Out& out) {
  const float2 rho = M.rho, m1 = M.m1, m2 = M.m2, m4 = M.m4, m5 = M.m5;
  const float2 ir = rcp2(rho), hx = mul2(f2(0.5f), Fx), hy = mul2(f2(0.5f), Fy);
  const float2 u = mul2(add2(m1, hx), ir), v = mul2(add2(m2, hy), ir);
  const float2 nu = mul2(f2(-1.0f), u), nv = mul2(f2(-1.0f), v);
  const float2 k4 = fma2(nu, sub2(m1, hx), fma2(v, sub2(m2, hy), m4));
  const float2 k5 = fma2(nv, m1, fma2(u, hy, m5));
  // 1 - omega = (3 nu - 1/2) / (3 nu + 1/2), nu linear in the phase fraction
  const float2 ph = make_float2(__saturatef(__fmaf_rn(rho.x, k.ph1, k.ph0)), __saturatef(__fmaf_rn(rho.y, k.ph1, k.ph0)));
  const float2 n3 = fma2(ph, f2(k.dn3), f2(k.nv3));
  const float2 om = mul2(add2(n3, f2(-0.5f)), rcp2(add2(n3, f2(0.5f))));
  const float2 ks4 = mul2(om, k4), K11 = mul2(om, k5);
  const float2 base = fma2(f2(1.0f / 3.0f), rho, aF);
  const float2 K20 = fma2(f2(0.5f), ks4, base), K02 = fma2(f2(-0.5f), ks4, base);
  const float2 K21 = mul2(f2(1.0f / 6.0f), Fy), K12 = mul2(f2(1.0f / 6.0f), Fx);
  const float2 K22 = fma2(f2(2.0f / 3.0f), aF, mul2(f2(1.0f / 9.0f), rho));
  // x axis
  const float2 m10 = add2(m1, Fx), m01 = add2(m2, Fy);
  const float2 m20 = fma2(u, add2(hx, m10), K20);
  const float2 M11 = fma2(u, hy, K11), M21 = fma2(u, add2(K11, M11), K21);
  const float2 M12 = fma2(u, K02, K12), M22 = fma2(u, add2(K12, M12), K22);
  // y axis
  const float2 m02 = fma2(v, add2(hy, m01), K02);
  const float2 m11 = fma2(v, m10, M11), m12 = fma2(v, add2(M11, m11), M12);
  const float2 m21 = fma2(v, m20, M21), m22 = fma2(v, add2(M21, m21), M22);
  // f* = M^{-1} m*
  const float2 px = sub2(m20, m22), py = sub2(m02, m22);
  out(0, add2(M.f0, sub2(M.sum8, add2(m20, py))));
  const float2 hpx = mul2(f2(0.5f), px), qx = sub2(m10, m12);
  out(1, fma2(f2(0.5f), qx, hpx));
  out(2, fma2(f2(-0.5f), qx, hpx));
  const float2 hpy = mul2(f2(0.5f), py), qy = sub2(m01, m21);
  out(3, fma2(f2(0.5f), qy, hpy));
  out(4, fma2(f2(-0.5f), qy, hpy));
  const float2 sp = mul2(f2(0.25f), add2(m22, m11)), tp = add2(m21, m12);
  out(5, fma2(f2(0.25f), tp, sp));
  out(6, fma2(f2(-0.25f), tp, sp));
  const float2 sm = mul2(f2(0.25f), sub2(m22, m11)), tm = sub2(m12, m21);
  out(7, fma2(f2(0.25f), tm, sm));
  out(8, fma2(f2(-0.25f), tm, sm));
  ux = u;
  uy = v;
}
// BGK operator of a column pair, node by node.
template <typename Out>
__device__ __forceinline__ void collide_bgk_pair(const Phys& ph, const float2 f[9], float2 rho, float2 Fx, float2 Fy,
                                                 float2& ux, float2& uy, const Out& out) {
  float2 fs[9];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    float a[9], b[9], u, v;
#pragma unroll
    for (int q = 0; q < 9; ++q) a[q] = pair_get(f[q], i);
    const float r = pair_get(rho, i);
    const float omega = fdiv(1.0f, add(fdiv(nu_of(ph, r), 1.0f / 3.0f), 0.5f));
    collide_bgk(a, r, pair_get(Fx, i), pair_get(Fy, i), omega, b, u, v);
#pragma unroll
    for (int q = 0; q < 9; ++q) pair_set(fs[q], i, b[q]);
    pair_set(ux, i, u);
    pair_set(uy, i, v);
  }
#pragma unroll
  for (int q = 0; q < 9; ++q) out(q, fs[q]);
}

// Shape of a flow tile: FR rows and FW columns of populations around it, from XL columns left of the
// tile or less (a TMA copy starts on 16 bytes: the column is rounded down).
template <typename S, int MODE, int TY_>
struct FlowTile {
  static constexpr int H = MODE == kFlowNone ? 0 : 2, TX = 64 - 2 * H, TY = TY_, ROWS = TY + 2 * H;
  static constexpr int NT = 32 * ROWS;
  static constexpr int FR = MODE == kFlowTile ? H + 1 : 1, FH = TY + 2 * FR;
  static constexpr int XA = 16 / (int)sizeof(S);
  // columns x0 - H - 1 .. x0 - H + 64 after rounding down (x0 a multiple of 4)
  static constexpr int OFF = sizeof(S) == 4 && !H ? 3 : 1;
  static constexpr int FW = (OFF + 66 + XA - 1) / XA * XA;
  static __host__ __device__ int xbox(int x0) { return (x0 - H - 1) & ~(XA - 1); }
};

// Collision of tile (bx, by).  tm_f: tensor map of the populations for TMA staging, or null.
// psi_g: psi in global memory, read (kFlowRead) or written (kFlowTile).
template <typename S, int PSI, int MODE, int OP, int TY>
__device__ __forceinline__ void flow_tile(const Geo& g, const Phys& ph, const S* __restrict__ f, S* __restrict__ fn,
                                          const float* __restrict__ T, float* psi_g, const uint8_t* __restrict__ mask,
                                          const float* __restrict__ side_in, float* __restrict__ side_out,
                                          float* __restrict__ rho_o, float* __restrict__ ux_o,
                                          float* __restrict__ uy_o, int forcing, int* status, int bx, int by,
                                          const CUtensorMap* tm_f, bool starve, bool early_f) {
  using FT = FlowTile<S, MODE, TY>;
  constexpr int H = FT::H, TX = FT::TX, FH = FT::FH, FW = FT::FW, FR = FT::FR;
  __shared__ __align__(128) S s_f[9 * FH * FW];
  __shared__ __align__(16) float s_psi[H ? FT::ROWS * 64 : 4];
  __shared__ uint64_t s_bar;
  const int tid = threadIdx.x, lane = tid & 31, r = (tid >> 5) - H;  // r: the warp's row in the tile
  const int x0 = bx * TX, y0 = by * TY, xb = FT::xbox(x0);
  const int xl = x0 - H + 2 * lane, y = y0 + r;  // the lane's left node
  const bool own = r >= 0 && r < TY;
  const bool multi = H && ph.f.G != 0.0f;
  constexpr int HR = H > FR ? H : FR;  // rows above and below that the tile reads
  const bool interior = x0 - H >= 1 && x0 - H + 64 < g.nx && y0 >= HR && y0 + TY + HR <= g.ny;
  // TMA also stages the tiles at an inlet or outlet (the columns outside read as zeros).  Tiles whose
  // rows wrap are staged by plain loads of an open lattice, and pull from global memory in a periodic
  // one (shear layer 512 x 512: 4.5 us a step against 6.5 staged; 1536 x 768 open: 4 us the other way)
  const bool staged = tm_f && y0 >= FR && y0 + TY + FR <= g.ny && (interior || !g.periodic_x);
  if (staged && tid == 0) {
    tma::bar_init(&s_bar, 1);
    tma::bar_expect_tx(&s_bar, sizeof(S) * 9 * FH * FW);
    // (the test hook leaves the barrier armed with no copy issued)
    if (!starve && early_f) tma::load_3d(s_f, tm_f, &s_bar, xb, y0 - FR, 0);
  }
  // node types of the pair (bytes 0, 1); positions past an edge stand for the node they repeat
  uint32_t m, ia = y * g.pitch + xl, ib = ia + 1;
  if (interior) {
    m = *reinterpret_cast<const uint16_t*>(mask + ia);
  } else {
    const int row = map_y(g, y) * g.pitch;
    ia = row + map_x(g, xl);
    ib = row + map_x(g, xl + 1);
    m = mask[ia] | (uint32_t)mask[ib] << 8;
  }
  pdl::wait();  // T, and psi where it is read, are the previous kernel's output
  pdl::trigger();
  if (staged && tid == 0 && !starve && !early_f) tma::load_3d(s_f, tm_f, &s_bar, xb, y0 - FR, 0);
  float2 psi = f2(0.0f);  // T of the pair first, where psi is evaluated here
  if (multi) {
    const float* p = MODE == kFlowTile ? T : psi_g;
    psi = interior ? *reinterpret_cast<const float2*>(p + ia) : make_float2(p[ia], p[ib]);
  }
  const bool in_smem = staged || !g.periodic_x;
  if (!staged && in_smem) {
    constexpr int NV = FW / FT::XA;  // 16-byte vectors of a row
#pragma unroll 4
    for (int p = tid; p < 9 * FH * NV; p += FT::NT) {
      const int q = p / NV, c = (p - q * NV) * FT::XA;
      const S* row = f + (q / FH) * g.plane + map_y(g, y0 - FR + q % FH) * g.pitch;
      if (xb + c >= 0 && xb + c < g.pitch)
        *reinterpret_cast<uint4*>(&s_f[q * FW + c]) = *reinterpret_cast<const uint4*>(row + xb + c);
    }
  }
  if (in_smem) __syncthreads();  // the barrier is initialised, or the plain copy complete
  // phase 1: pull, moments, psi
  const int tries = starve ? tma::kStarveTries : tma::kWaitTries;
  bool landed = true;
  if (staged) landed = tma::bar_wait(&s_bar, 0, tries);
  float2 fo[9];
  PairMoments M;
  M.rho = f2(ph.f.rho_s);
  if (own || (MODE == kFlowTile && multi)) {
    if (in_smem) {
      const S* q = s_f + (r + FR) * FW + (x0 - H - xb) + 2 * lane;  // the left node in plane 0
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const S* p = q + (i * FH - cyv(i)) * FW - cxv(i);
        S c, d;
        if (cxv(i) == 0) {
          PairLoad<S>::ld(p, c, d);
        } else {
          c = p[0];
          d = p[1];
        }
        fo[i] = make_float2(PopIO<float, S>::ld(c, i, ph), PopIO<float, S>::ld(d, i, ph));
      }
    } else {
      int row[3], col[4];
#pragma unroll
      for (int k = 0; k < 3; ++k) row[k] = map_y(g, y + k - 1) * g.pitch;
#pragma unroll
      for (int k = 0; k < 4; ++k) col[k] = map_x(g, xl + k - 1);
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const S* p = f + i * g.plane;
        fo[i] = make_float2(PopIO<float, S>::ld(p[(uint32_t)(row[1 - cyv(i)] + col[1 - cxv(i)])], i, ph),
                            PopIO<float, S>::ld(p[(uint32_t)(row[1 - cyv(i)] + col[2 - cxv(i)])], i, ph));
      }
    }
    // nodes next to the wall and in the edge columns of an open lattice take the substitutions (ghost
    // columns repeat the edge column)
    uint32_t slow = ((m & kNearWall) ? 1u : 0u) | ((m & (kNearWall << 8)) ? 2u : 0u), off = 0;
    if (!interior && !g.periodic_x) {
      if (xl <= 0 || xl >= g.nx - 1) slow |= 1u;
      if (xl + 1 <= 0 || xl + 1 >= g.nx - 1) slow |= 2u;
      off = (xl > g.nx + 1 ? 1u : 0u) | (xl + 1 > g.nx + 1 ? 2u : 0u);  // no stencil reads these
      slow &= ~(off | ((m & kSolid) ? 1u : 0u) | ((m & (kSolid << 8)) ? 2u : 0u));
    }
#pragma unroll 1
    for (; slow; slow &= slow - 1) {
      const int i = slow & 1 ? 0 : 1, x = map_x(g, xl + i), yy = map_y(g, y);
      const bool mine = own && lane >= H / 2 && lane < 32 - H / 2 && xl + i < g.nx && y < g.ny;
      const S* n = s_f + (r + FR) * FW + x - xb;  // the node in plane 0 of a staged tile (no column wraps)
      auto at = [&](int i2, int dx, int dy) {
        if (in_smem) return PopIO<float, S>::ld(n[(i2 * FH + dy) * FW + dx], i2, ph);
        return ldf<float>(g, ph, f, i2, wrap_y(g, yy + dy), map_x(g, x + dx));
      };
      float t[9];
#pragma unroll
      for (int q2 = 0; q2 < 9; ++q2) t[q2] = at(q2, -cxv(q2), -cyv(q2));
      // a tile whose copy did not land stores no outlet values
      pull_special<float>(g, ph, side_in, mine && landed ? side_out : nullptr, x, yy, (uint8_t)(m >> (8 * i)), t, at);
#pragma unroll
      for (int q2 = 0; q2 < 9; ++q2) pair_set(fo[q2], i, t[q2]);
    }
    M = moments_pair(fo);
    if (!landed) M.rho = f2(ph.f.rho_s);  // reported below; psi of a density that can be
    if (m & kSolid) M.rho.x = ph.f.rho_s;
    if (m & (kSolid << 8)) M.rho.y = ph.f.rho_s;
    // saturated liquid where no stencil reads: the edge column's T may have no psi at another density
    if (off & 1u) M.rho.x = ph.f.rho_l, psi.x = ph.f.T_sat;
    if (off & 2u) M.rho.y = ph.f.rho_l, psi.y = ph.f.T_sat;
  }
  if (multi) {
    if (MODE == kFlowTile)
      psi = make_float2(psi_of<float, PSI>(ph, M.rho.x, psi.x, status), psi_of<float, PSI>(ph, M.rho.y, psi.y, status));
    reinterpret_cast<float2*>(s_psi)[(r + H) * 32 + lane] = psi;
  }
  if (__syncthreads_or(!landed)) {
    // the copies did not land in time: report it, give them a second bound to land before the
    // block's shared memory is released, and produce nothing
    if (tid == 0) atomicOr(status, kStatusTimeoutCollide);
    tma::bar_wait(&s_bar, 0, tries);
    return;
  }
  // phase 2: force and collision at the own nodes
  if (!own || y >= g.ny || lane < H / 2 || lane >= 32 - H / 2 || xl >= g.nx) return;
  float2 Fx = f2(0.0f), Fy = f2(0.0f), aF = f2(0.0f);
  if (forcing) {
    float2 gx = f2(0.0f), gy = f2(0.0f);
    if (multi) {
      grad_rows(reinterpret_cast<const float2*>(s_psi) + (r + H) * 32 + lane - 1, 32, gx, gy);
      aF = mul2(f2(ph.sc.sg), fma2(gx, gx, mul2(gy, gy)));
    }
    force_pair(ph, M.rho, psi, gx, gy, Fx, Fy);
  }
  const uint32_t id = y * g.pitch + xl;
  float2 ux, uy;
  auto run = [&](auto&& out) {
    if constexpr (OP == kCollBGK) collide_bgk_pair(ph, fo, M.rho, Fx, Fy, ux, uy, out);
    else collide_pair(ph.sc, M, Fx, Fy, aF, ux, uy, out);
  };
  if (!(m & (kSolid * 0x0101u)) && xl + 1 < g.nx) {
    run([&](int i, float2 v) { PairStore<S>::st(fn + i * g.plane + id, v, i, ph); });
    // any NaN, or a density that is not positive
    const float2 w = add2(ux, uy);
    if (!(M.rho.x > 0.0f) || !(M.rho.y > 0.0f) || !(w.x == w.x) || !(w.y == w.y)) atomicOr(status, 1);
  } else {  // solid nodes keep their populations; the right node may lie in the padding of an odd nx
    const bool ox = !(m & kSolid), oy = !(m & (kSolid << 8)) && xl + 1 < g.nx;
    run([&](int i, float2 v) {
      if (ox) fn[i * g.plane + id] = PopIO<float, S>::st(v.x, i, ph);
      if (oy) fn[i * g.plane + id + 1] = PopIO<float, S>::st(v.y, i, ph);
    });
    if (ox && (!(M.rho.x > 0.0f) || !(ux.x == ux.x) || !(uy.x == uy.x))) atomicOr(status, 1);
    if (oy && (!(M.rho.y > 0.0f) || !(ux.y == ux.y) || !(uy.y == uy.y))) atomicOr(status, 1);
    if (!ox) ux.x = uy.x = 0.0f;
    if (!oy) ux.y = uy.y = 0.0f;
  }
  *reinterpret_cast<float2*>(rho_o + id) = M.rho;
  *reinterpret_cast<float2*>(ux_o + id) = ux;
  *reinterpret_cast<float2*>(uy_o + id) = uy;
  if (MODE == kFlowTile && multi) *reinterpret_cast<float2*>(psi_g + id) = psi;
}

}  // namespace kern
}  // namespace lbm
