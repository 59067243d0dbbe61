// FP32 collision pass of one lattice tile with psi evaluated in it: pull-streaming, rho, psi, interaction force
// and the CM (or BGK) collision (Sec. II.A-B, Sec. IV.A; included by lbm_step_f32.cuh).
//
// Tile: 60 columns by TY rows with a halo of H = 2 nodes where psi is needed.  One warp covers one row of
// 64 columns, two per lane, so a block is TY + 4 warps.  Phase 1: every lane pulls its pair from the
// populations staged in shared memory (by TMA inside the lattice) and evaluates psi of it, the halo
// rows too, into a shared tile.  Phase 2: the warps of the own rows take the force from the psi tile and
// collide the moments they still hold in registers.
//
// 56 us for collision and psi at 2048 x 1024, where the one-node-per-lane collision took 38 us and the psi that
// the energy pass made for it 27 us more.  Its 32.0 M warp instructions take 53% of the issue slots, the
// FMA pipe is busy in 37% of the cycles and DRAM in 33%: the two 16-warp blocks of an SM pass copy, pull, psi,
// barrier, collision and stores one after the other, and there are no more warps to fill in.  8 to 16 rows, 2
// to 4 blocks and a persistent grid that prefetches the next tile lie within 5% of it; 64 own columns with
// a wider halo take 62 us.
//
// psi in the tile evaluates psi at 1.42 nodes per node, and reads each population once per step (the halo
// comes from L2).  Collisions that read psi, or need none, run one node per lane (collide_node of
// lbm_kernels.cuh) with the same bits.
#pragma once

namespace lbm {
namespace kern {

__device__ __forceinline__ void pair_set(float2& v, int i, float x) {
  if (i == 0) v.x = x;
  else v.y = x;
}
__device__ __forceinline__ float pair_get(float2 v, int i) { return i == 0 ? v.x : v.y; }

// rho alone.
__device__ __forceinline__ float2 pop_sum2(const float2 f[9]) {
  return add2(add2(f[0], add2(add2(f[1], f[2]), add2(f[3], f[4]))), add2(add2(f[5], f[6]), add2(f[7], f[8])));
}

// Shape of a flow tile: FR rows and FW columns of populations around it, from XL columns left of the
// tile or less (a TMA copy starts on 16 bytes: the column is rounded down).
template <int TY_>
struct FlowTile {
  static constexpr int H = 2, TX = 64 - 2 * H, TY = TY_, ROWS = TY + 2 * H;
  static constexpr int NT = 32 * ROWS;
  static constexpr int FR = H + 1, FH = TY + 2 * FR;
  static constexpr int XA = 4;
  // columns x0 - H - 1 .. x0 - H + 64 after rounding down (x0 a multiple of 4)
  static constexpr int OFF = 1;
  static constexpr int FW = (OFF + 66 + XA - 1) / XA * XA;
  static __host__ __device__ int xbox(int x0) { return (x0 - H - 1) & ~(XA - 1); }
};

// Collision of tile (bx, by).  tm_f: tensor map of the populations for TMA staging, or null.
// psi_o: where psi of the nodes goes.
template <int PSI, int OP, int TY>
__device__ __forceinline__ void flow_tile(const Geo& g, const Phys& ph, const float* __restrict__ f, float* __restrict__ fn,
                                          const float* __restrict__ T, float* __restrict__ psi_o, const uint8_t* __restrict__ mask,
                                          const float* __restrict__ side_in, float* __restrict__ side_out,
                                          float* __restrict__ rho_o, float* __restrict__ ux_o,
                                          float* __restrict__ uy_o, int forcing, int* status, int bx, int by,
                                          const CUtensorMap* tm_f, bool starve, bool early_f) {
  using FT = FlowTile<TY>;
  constexpr int H = FT::H, TX = FT::TX, FH = FT::FH, FW = FT::FW, FR = FT::FR;
  __shared__ __align__(128) float s_f[9 * FH * FW];
  __shared__ __align__(16) float s_psi[FT::ROWS * 64];
  __shared__ uint64_t s_bar;
  const int tid = threadIdx.x, lane = tid & 31, r = (tid >> 5) - H;  // r: the warp's row in the tile
  const int x0 = bx * TX, y0 = by * TY, xb = FT::xbox(x0);
  const int xl = x0 - H + 2 * lane, y = y0 + r;  // the lane's left node
  const bool own = r >= 0 && r < TY;
  const bool multi = ph.f.G != 0.0f;
  const bool interior = x0 - H >= 1 && x0 - H + 64 < g.nx && y0 >= FR && y0 + TY + FR <= g.ny;
  // TMA also stages the tiles at an inlet or outlet (the columns outside read as zeros).  Tiles whose
  // rows wrap are staged by plain loads of an open lattice, and pull from global memory in a periodic
  // one (shear layer 512 x 512: 4.5 us a step against 6.5 staged; 1536 x 768 open: 4 us the other way)
  const bool staged = tm_f && y0 >= FR && y0 + TY + FR <= g.ny && (interior || !g.periodic_x);
  if (staged && tid == 0) {
    tma::bar_init(&s_bar, 1);
    tma::bar_expect_tx(&s_bar, sizeof(float) * 9 * FH * FW);
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
  pdl::wait();  // T is the previous kernel's output
  pdl::trigger();
  if (staged && tid == 0 && !starve && !early_f) tma::load_3d(s_f, tm_f, &s_bar, xb, y0 - FR, 0);
  float2 psi = f2(0.0f);  // T of the pair first
  if (multi) psi = interior ? *reinterpret_cast<const float2*>(T + ia) : make_float2(T[ia], T[ib]);
  const bool in_smem = staged || !g.periodic_x;
  if (!staged && in_smem) {
    constexpr int NV = FW / FT::XA;  // 16-byte vectors of a row
#pragma unroll 4
    for (int p = tid; p < 9 * FH * NV; p += FT::NT) {
      const int q = p / NV, c = (p - q * NV) * FT::XA;
      const float* row = f + (q / FH) * g.plane + map_y(g, y0 - FR + q % FH) * g.pitch;
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
  Moments<float2> M;
  M.rho = f2(ph.f.rho_s);
  if (own || multi) {
    if (in_smem) {
      const float* q = s_f + (r + FR) * FW + (x0 - H - xb) + 2 * lane;  // the left node in plane 0
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const float* p = q + (i * FH - cyv(i)) * FW - cxv(i);
        fo[i] = cxv(i) == 0 ? *reinterpret_cast<const float2*>(p) : make_float2(p[0], p[1]);
      }
    } else {
      int row[3], col[4];
#pragma unroll
      for (int k = 0; k < 3; ++k) row[k] = map_y(g, y + k - 1) * g.pitch;
#pragma unroll
      for (int k = 0; k < 4; ++k) col[k] = map_x(g, xl + k - 1);
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const float* p = f + i * g.plane;
        fo[i] = make_float2(p[(uint32_t)(row[1 - cyv(i)] + col[1 - cxv(i)])],
                            p[(uint32_t)(row[1 - cyv(i)] + col[2 - cxv(i)])]);
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
      const float* n = s_f + (r + FR) * FW + x - xb;  // the node in plane 0 of a staged tile (no column wraps)
      auto at = [&](int i2, int dx, int dy) {
        if (in_smem) return n[(i2 * FH + dy) * FW + dx];
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
    M = moments_of(fo);
    if (!landed) M.rho = f2(ph.f.rho_s);  // reported below; psi of a density that can be
    if (m & kSolid) M.rho.x = ph.f.rho_s;
    if (m & (kSolid << 8)) M.rho.y = ph.f.rho_s;
    // saturated liquid where no stencil reads: the edge column's T may have no psi at another density
    if (off & 1u) M.rho.x = ph.f.rho_l, psi.x = ph.f.T_sat;
    if (off & 2u) M.rho.y = ph.f.rho_l, psi.y = ph.f.T_sat;
  }
  if (multi) {
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
    force_of(ph, M.rho, psi, gx, gy, Fx, Fy);
  }
  const uint32_t id = y * g.pitch + xl;
  float2 ux, uy;
  auto run = [&](auto&& out) {
    if constexpr (OP == kCollBGK) collide_bgk_of(ph.sc, fo, M, Fx, Fy, ux, uy, out);
    else collide_cm(ph.sc, M, Fx, Fy, aF, ux, uy, out);
  };
  if (!(m & (kSolid * 0x0101u)) && xl + 1 < g.nx) {
    run([&](int i, float2 v) { *reinterpret_cast<float2*>(fn + i * g.plane + id) = v; });
    // any NaN, or a density that is not positive
    const float2 w = add2(ux, uy);
    if (!(M.rho.x > 0.0f) || !(M.rho.y > 0.0f) || !(w.x == w.x) || !(w.y == w.y)) atomicOr(status, 1);
  } else {  // solid nodes keep their populations; the right node may lie in the padding of an odd nx
    const bool ox = !(m & kSolid), oy = !(m & (kSolid << 8)) && xl + 1 < g.nx;
    run([&](int i, float2 v) {
      if (ox) fn[i * g.plane + id] = v.x;
      if (oy) fn[i * g.plane + id + 1] = v.y;
    });
    if (ox && (!(M.rho.x > 0.0f) || !(ux.x == ux.x) || !(uy.x == uy.x))) atomicOr(status, 1);
    if (oy && (!(M.rho.y > 0.0f) || !(ux.y == ux.y) || !(uy.y == uy.y))) atomicOr(status, 1);
    if (!ox) ux.x = uy.x = 0.0f;
    if (!oy) ux.y = uy.y = 0.0f;
  }
  *reinterpret_cast<float2*>(rho_o + id) = M.rho;
  *reinterpret_cast<float2*>(ux_o + id) = ux;
  *reinterpret_cast<float2*>(uy_o + id) = uy;
  if (multi) *reinterpret_cast<float2*>(psi_o + id) = psi;
}

}  // namespace kern
}  // namespace lbm
