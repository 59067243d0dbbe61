// FP64 energy pass (Eq. energy; included by lbm_kernels.cuh), bound by the FP64 pipe (2 lanes per SM):
// every operation of a node is worth saving, memory traffic is not.
//
// Two launches, one per Heun stage, so that no node's stage 1 is computed again in a neighbour's
// halo (on 32 x 8 tiles with a 2-node halo that was 1.69 times the work): k_energy1 stores T1 and the
// parts of the right-hand side that are frozen during the step, k_energy2 reads them back.  lambda
// of a node is computed once, by the collision.  Divisors that are used more than once have their
// reciprocals rounded once, and each quotient is then one product and two FMAs (div_by).
// Every result rounds as the plain expressions do (sums in the order of the method's, no contraction).
// 512 x 256 (CUDA events): 312 -> 185 us for the pass and 109 -> 93 us for the collision, 580 and 285
// FP64 instructions per node instead of 978 and 340; the FP64 pipe is 82% busy throughout.
#pragma once

namespace lbm {
namespace kern {

// Planes of the frozen parts, per node: grad lambda, div u; rho R / (1 - b rho); the reciprocals of
// 1 + 2 b rho - b^2 rho^2 and of rho c_v.
struct Frozen64 {
  double *lx, *ly, *divu, *rep, *ratt, *rrc;
};

// The frozen parts at one node, with lambda.
struct NodeFrozen {
  double lam, lx, ly, divu, rep, ratt, rrc;
};
__device__ __forceinline__ double upwind3_f64(const double w[5][6], int c0, bool along_x, double v) {
  const double c = w[2][c0];
  auto at = [&](int o) { return along_x ? w[2][c0 + o] : w[2 + o][c0]; };
  // biased against the sign of v: on the mirrored window, (a2 - 6 a1) + 2 b1 for v >= 0 and
  // (6 a1 - 2 b1) - a2 for v < 0 (products by 2 are exact, so one FMA rounds like product and sum)
  const bool pos = v >= 0.0;
  const double a2 = (pos ? at(-2) : at(2)) - c, a1 = (pos ? at(-1) : at(1)) - c, b1 = (pos ? at(1) : at(-1)) - c;
  const double p6 = 6.0 * a1;
  const double t = __fma_rn(pos ? -1.0 : -2.0, pos ? p6 : b1, pos ? a2 : p6);
  const double s = __fma_rn(pos ? 2.0 : -1.0, pos ? b1 : a2, t);
  return div_by(s, 6.0, 1.0 / 6.0);
}
// Right-hand side of Eq. (energy) at node c0 of a pair whose 5x6 temperature window is w, and the
// temperature gradient there.
__device__ __forceinline__ double energy_rhs_f64(const Phys& ph, const double w[5][6], int c0, double u, double v,
                                                 double rho, const NodeFrozen& z, double& gx, double& gy) {
  const PhysC<double>& k = ph.d;
  const double T = w[2][c0];
  const double conv = u * upwind3_f64(w, c0, true, u) + v * upwind3_f64(w, c0, false, v);
  grad_w(w, c0, gx, gy);
  const double diff = z.lam * lap_w(w, c0) + (z.lx * gx + z.ly * gy);
  const double s = 1.0 + k.kappa * (1.0 - sqrt(div_by(T, k.Tc, ph.rTc)));
  const double dphi = -k.kappa * s / sqrt(T * k.Tc);
  const double D = 1.0 + 2.0 * k.b * rho - k.b * k.b * rho * rho;
  const double dpdT = z.rep - div_by(k.a * dphi * rho * rho, D, z.ratt);
  const double work = T * dpdT * z.divu, rc = rho * k.c_v;
  return -conv + div_by(diff, rc, z.rrc) - div_by(work, rc, z.rrc);
}
// The 5x6 window around the node pair (x, y), (x + 1, y) of a plane, x even: aligned pairs, or node by
// node with the positions past an edge mapped back.
__device__ __forceinline__ void window_global(const Geo& g, const double* __restrict__ p, int x, int y, double w[5][6]) {
  if (x >= 2 && x + 4 <= g.nx && y >= 2 && y + 3 <= g.ny) {
#pragma unroll
    for (int r = 0; r < 5; ++r) {
      const double2* q = reinterpret_cast<const double2*>(p + (y + r - 2) * g.pitch + x - 2);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double2 v = q[c];
        w[r][2 * c] = v.x;
        w[r][2 * c + 1] = v.y;
      }
    }
  } else {
#pragma unroll
    for (int r = 0; r < 5; ++r) {
      const double* q = p + map_y(g, y + r - 2) * g.pitch;
#pragma unroll
      for (int c = 0; c < 6; ++c) w[r][c] = q[map_x(g, x + c - 2)];
    }
  }
}

// Heun stage 1, T1 = T + L(T), at the 32 x 8 nodes of tile (bx, by), two per thread, with the wall heat
// flux of T (Sec. IV.B).  maps: tensor maps of T and of rho, u_x, u_y with the box of the tile and a
// 2-node halo, with which an interior tile stages them by TMA (else null: plain loads).
__device__ __forceinline__ void energy1_tile(const Geo& g, const Phys& ph, const double* __restrict__ Tin,
                                             double* __restrict__ T1, const double* __restrict__ lam,
                                             const Frozen64& fz, const double* __restrict__ rho,
                                             const double* __restrict__ ux, const double* __restrict__ uy,
                                             const uint8_t* __restrict__ mask, double* partial, unsigned* counter,
                                             double* hf, int nb, int do_hf, int n_wall_tiles, int bx, int by, int bid,
                                             int nblocks, int* status, const EnergyMaps* maps, bool starve) {
  constexpr int TX = kEnergyTX64, TY = 8, H = 2, AX = TX + 2 * H, AY = TY + 2 * H, NT = TX * TY / 2;
  __shared__ __align__(128) double sT[AY * AX];
  __shared__ __align__(128) double sRUV[3 * AY * AX];  // rho, u_x, u_y: the planes of one TMA box
  __shared__ __align__(16) double sL[AY * AX];
  __shared__ uint64_t s_bar;
  __shared__ double red[NT / 32];
  __shared__ int done_last;
  double* const sU = sRUV + AY * AX;
  double* const sV = sRUV + 2 * AY * AX;
  const int tid = threadIdx.x;
  const int x0 = bx * TX, y0 = by * TY;
  const bool interior = x0 >= H && y0 >= H && x0 + TX + H <= g.nx && y0 + TY + H <= g.ny;
  const bool staged = maps && interior;
  if (staged) {
    if (tid == 0) tma::bar_init(&s_bar, 1);
    __syncthreads();
    if (tid == 0) {
      tma::bar_expect_tx(&s_bar, 4 * AX * AY * sizeof(double));
      // T comes from the energy pass before the previous kernel (the collision, which does not
      // write it): its copy starts before that kernel ends; the test hook leaves the barrier
      // armed with no copy issued
      if (!starve) tma::load_2d(sT, &maps->T, &s_bar, x0 - H, y0 - H);
    }
  }
  pdl::wait();  // rho, u and lambda are the collision's output
  pdl::trigger();
  if (staged && tid == 0 && !starve) tma::load_3d(sRUV, &maps->ruv, &s_bar, x0 - H, y0 - H, 0);
  for (int p = tid; p < AX * AY; p += NT) {
    const int nid = map_y(g, y0 + p / AX - H) * g.pitch + map_x(g, x0 + p % AX - H);
    sL[p] = lam[nid];
    if (!staged) {
      sT[p] = Tin[nid];
      sRUV[p] = rho[nid];
      sU[p] = ux[nid];
      sV[p] = uy[nid];
    }
  }
  const int tries = starve ? tma::kStarveTries : tma::kWaitTries;
  const bool landed = !staged || tma::bar_wait(&s_bar, 0, tries);
  if (__syncthreads_or(!landed)) {
    // a copy did not land in time: report it, let the copies land (bounded) and stop the tile
    // (a tile that holds wall nodes then misses its heat-flux partial; restoring a state with
    // lbm_set_state resets that bookkeeping)
    if (tid == 0) atomicOr(status, kStatusTimeoutEnergy);
    tma::bar_wait(&s_bar, 0, tries);
    return;
  }
  const int tx = (tid % (TX / 2)) * 2, ty = tid / (TX / 2), a = (ty + H) * AX + tx + H;
  const int y = y0 + ty;
  double q = 0.0;
  int mine = 0;
  if (x0 + tx < g.nx && y < g.ny) {
    const PhysC<double>& k = ph.d;
    const int id = y * g.pitch + x0 + tx;
    NodeFrozen z[2];
    double w[5][6], unused, dxux[2], dyuy;
    load_window(&sL[a], AX, w);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      z[i].lam = w[2][2 + i];
      grad_w(w, 2 + i, z[i].lx, z[i].ly);
    }
    load_window(&sU[a], AX, w);
#pragma unroll
    for (int i = 0; i < 2; ++i) grad_w<double, true, false>(w, 2 + i, dxux[i], unused);
    load_window(&sV[a], AX, w);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      grad_w<double, false, true>(w, 2 + i, unused, dyuy);
      z[i].divu = dxux[i] + dyuy;
    }
    load_window(&sT[a], AX, w);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int x = x0 + tx + i;
      const double r = sRUV[a + i], T = w[2][2 + i];
      z[i].rep = r * k.R / (1.0 - k.b * r);
      z[i].ratt = 1.0 / (1.0 + 2.0 * k.b * r - k.b * k.b * r * r);
      z[i].rrc = 1.0 / (r * k.c_v);
      double gx, gy;
      const double L = energy_rhs_f64(ph, w, 2 + i, sU[a + i], sV[a + i], r, z[i], gx, gy);
      if (x >= g.nx) continue;  // the pair's right node past an odd nx
      const uint8_t m = mask[id + i];
      double t1;
      if (m & kSolid) t1 = T;  // solid nodes keep their wall temperature
      else if (!g.periodic_x && x == 0) t1 = k.T_sat;
      else t1 = T + L;
      T1[id + i] = t1;
      fz.lx[id + i] = z[i].lx;
      fz.ly[id + i] = z[i].ly;
      fz.divu[id + i] = z[i].divu;
      fz.rep[id + i] = z[i].rep;
      fz.ratt[id + i] = z[i].ratt;
      fz.rrc[id + i] = z[i].rrc;
      if (do_hf && (m & kNearWall)) {
        const double* nv = &g.wall_n[2 * g.wall_idx[id + i]];
        q += -z[i].lam * (gx * nv[0] + gy * nv[1]);
        mine = 1;
      }
    }
  }
  if (do_hf) heat_flux_blocks<NT>(q, mine, partial, counter, n_wall_tiles, bid, nblocks, hf, nb, red, &done_last);
}

// Heun stage 2, T^{n+1} = (T + T1 + L(T1)) / 2, at the same nodes; with psi_out set also psi of the next
// step from the pull of the populations this step's collision wrote (fnew, side_new).
__device__ __forceinline__ void energy2_tile(const Geo& g, const Phys& ph, const double* __restrict__ Tin,
                                             double* __restrict__ Tout, const double* __restrict__ T1,
                                             const double* __restrict__ lam, const Frozen64& fz,
                                             const double* __restrict__ rho, const double* __restrict__ ux,
                                             const double* __restrict__ uy, const uint8_t* __restrict__ mask, int bx,
                                             int by, const double* __restrict__ fnew,
                                             const double* __restrict__ side_new, double* __restrict__ psi_out,
                                             int* status) {
  pdl::wait();  // T1 and the frozen parts are the previous kernel's output
  pdl::trigger();
  const int x0 = bx * kEnergyTX64 + (threadIdx.x % (kEnergyTX64 / 2)) * 2, y = by * 8 + threadIdx.x / (kEnergyTX64 / 2);
  if (x0 >= g.nx || y >= g.ny) return;
  const int id = y * g.pitch + x0;
  double w[5][6], tnew[2];
  window_global(g, T1, x0, y, w);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    if (x0 + i >= g.nx) continue;
    const NodeFrozen z = {lam[id + i], fz.lx[id + i], fz.ly[id + i], fz.divu[id + i], fz.rep[id + i], fz.ratt[id + i],
                          fz.rrc[id + i]};
    double gx, gy;
    const double L = energy_rhs_f64(ph, w, 2 + i, ux[id + i], uy[id + i], rho[id + i], z, gx, gy);
    const double T = Tin[id + i];
    double out;
    if (mask[id + i] & kSolid) out = T;
    else if (!g.periodic_x && x0 + i == 0) out = ph.d.T_sat;
    else out = ((T + w[2][2 + i]) + L) * 0.5;
    Tout[id + i] = out;
    tnew[i] = out;
  }
  if (!psi_out) return;
  const uint8_t m0 = mask[id], m1 = mask[id + 1];
  double r[2];
  // a pair away from the wall, the open edges and the periodic seams pulls from one base address;
  // the others take the general pull with its boundary substitutions
  if (!((m0 | m1) & kNearWall) && y >= 1 && y + 1 < g.ny && x0 >= 1 && x0 + 3 <= g.nx) {
    pair_rho<double, double>(g, ph, fnew, x0, y, r);
  } else {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (x0 + i >= g.nx || ((i ? m1 : m0) & kSolid)) continue;
      double fo[9];
      pull_node<double, double>(g, ph, fnew, mask, side_new, nullptr, x0 + i, y, i ? m1 : m0, fo);
      double t = fo[0];
#pragma unroll
      for (int j = 1; j < 9; ++j) t = t + fo[j];
      r[i] = t;
    }
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (x0 + i < g.nx)
      psi_out[id + i] = psi_of<double, kPsiF64>(ph, ((i ? m1 : m0) & kSolid) ? ph.d.rho_s : r[i], tnew[i], status);
}

}  // namespace kern
}  // namespace lbm
