// FP32 energy pass of one lattice tile (Eq. energy; included by lbm_step_f32.cuh).
//
// Tile: 60 x TY nodes.  With the 2-node halo of Heun stage 1 a tile row is 64 columns, two per
// lane: one warp covers it exactly.  Warp w of the TY / 2 first ones owns the tile rows 2w, 2w + 1
// in both stages, so the parts of Eq. (energy) that depend on rho and u only (frozen during the
// step) stay in its registers between the stages; two more warps compute stage 1 on the two halo
// rows below and above the tile.
//
// 40 us at 2048 x 1024 for 23.6 M warp instructions.  No unit is full: 59% of the issue slots, the FMA pipe 53% of
// the cycles (a packed operation holds it for two), DRAM 12%; three 10-warp blocks an SM (64 registers,
// 124 B spilled) wait at the barriers (2.0 cycles an instruction), for the copies (1.8) and for the FMA pipe
// (1.4).  32 x 16 tiles with a lane per pair, separate stencil sums and the psi of the next step took 51.9 M
// and 68 us (30 M and about 27 us of it for that psi).  4-row tiles where 16-row ones would leave SMs idle
// (12.6 us of a 192 x 96 lattice against 18).
//
// Stencils: a lane reads the 6-column window of its column pair row by row (three 8-byte loads)
// and folds each row into sums and differences over +/-1 and +/-2 columns, from which every
// stencil of the row's 25-point neighbourhood takes its share: the gradient, the Laplacian and
// the upwind derivative (written as the centred fourth-order difference plus |u| times a fourth
// difference: no selection by sign) together cost fewer operations than their 12 pairs each, and
// no operand needs a register move.  Two rows per thread share the window rows.
//
// The temperature is staged as theta = T - T_sat: the sums over rows round at the size of the superheat
// instead of T.
//
// Every operation is written out (packed FP32x2 or explicit roundings), so that every kernel that
// inlines the tile gives the same bits.
#pragma once

namespace lbm {
namespace kern {

// The frozen parts of Eq. (energy) of a column pair, divided by rho c_v: twice the diffusivity
// alpha = lambda / (rho c_v), grad lambda / (rho c_v), and the pressure work as T (P + Q / sqrt(T))
// with (dp/dT)_rho = rep + att (kappa (1 + kappa) / sqrt(T Tc) - kappa^2 / Tc), rep = rho R /
// (1 - b rho), att = a rho^2 / (1 + 2 b rho - b^2 rho^2).
struct FrozenPair {
  float2 al2, ax, ay, P, Q;
};
// Frozen parts of two rows of a column pair.  l (lambda / c_v), u, v: window columns -2, -1 of the
// upper row in tiles of row stride ts (pairs); rho: the pair itself.
__device__ __forceinline__ void frozen_rows(const StepConst& k, const float2* l, const float2* u, const float2* v,
                                            const float2* rho, int ts, FrozenPair fz[2]) {
  float2 lx[2] = {f2(0.f), f2(0.f)}, ly[2] = {f2(0.f), f2(0.f)}, dv[2] = {f2(0.f), f2(0.f)}, l0[2];
#pragma unroll
  for (int r = -2; r <= 3; ++r) {
    const RowSums R = row_sums<true, true>(l + r * ts);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int d = r - j;
      if (d < -2 || d > 2) continue;
      row_gx(R, d < 0 ? -d : d, lx[j]);
      if (d != 0) row_gy(R, d, ly[j]);
      else l0[j] = R.c;
    }
  }
#pragma unroll
  for (int r = -2; r <= 3; ++r) {
    const RowSums U = row_sums<true, false>(u + r * ts), V = row_sums<false, true>(v + r * ts);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int d = r - j;
      if (d < -2 || d > 2) continue;
      row_gx(U, d < 0 ? -d : d, dv[j]);
      if (d != 0) row_gy(V, d, dv[j]);
    }
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float2 r = rho[j * ts], ir = rcp2(r);
    fz[j].al2 = mul2(mul2(f2(2.0f), l0[j]), ir);
    fz[j].ax = mul2(lx[j], ir);
    fz[j].ay = mul2(ly[j], ir);
    const float2 rep = mul2(f2(k.rep), rcp2(fma2(f2(-k.b), r, f2(1.0f))));
    const float2 att = mul2(mul2(f2(k.att), r), rcp2(fma2(r, fma2(f2(-k.bb), r, f2(k.b2)), f2(1.0f))));
    fz[j].P = mul2(dv[j], fma2(f2(-k.c2), att, rep));
    fz[j].Q = mul2(mul2(f2(k.c1), att), dv[j]);
  }
}
// Right-hand side of Eq. (energy) at two rows of a column pair for the temperature tile t (theta,
// window columns -2, -1 of the upper row; row stride ts), and the temperature gradient there:
// -u.grad T + alpha lap T + grad lambda.grad T / (rho c_v) - T (P + Q / sqrt(T)), with
// 12 u dT/dx (third-order upwind) = u (8 X1 - X2) + |u| (S2 - 4 S1 + 6 theta).
__device__ __forceinline__ void rhs_rows(const StepConst& k, const float2* t, int ts, const float2 u[2],
                                         const float2 v[2], const FrozenPair fz[2], float2 L[2], float2 gx[2],
                                         float2 gy[2]) {
  // lap holds half the Laplacian; its centre weight is the sum of the 24 others as rounded to FP32
  // (in two parts), so that a uniform theta, however large, contributes nothing
  constexpr double W = 4.0 * wrow(0, 1) + 4.0 * wrow(0, 2) + 4.0 * wrow(1, 1) + 4.0 * wrow(2, 2) + 8.0 * wrow(1, 2);
  constexpr float W0 = float(W), W1 = float(W - double(W0));
  float2 lap[2], c[6], nx[2], mx[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) gx[j] = gy[j] = lap[j] = f2(0.f);
#pragma unroll
  for (int r = -2; r <= 3; ++r) {
    const RowSums R = row_sums<true, true>(t + r * ts);
    c[r + 2] = R.c;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int d = r - j, a = d < 0 ? -d : d;
      if (a > 2) continue;
      row_gx(R, a, gx[j]);
      if (d == 0) {
        lap[j] = fma2(f2(wrow(0, 1)), R.S1, fma2(f2(wrow(0, 2)), R.S2, fma2(f2(-W0), R.c, fma2(f2(-W1), R.c, lap[j]))));
        nx[j] = fma2(f2(-8.0f), R.X1, R.X2);
        mx[j] = fma2(f2(6.0f), R.c, fma2(f2(-4.0f), R.S1, R.S2));
      } else {
        const float2 V = fma2(f2(wrow(a, 0)), R.c, fma2(f2(wrow(a, 1)), R.S1, mul2(f2(wrow(a, 2)), R.S2)));
        gy[j] = fma2(f2(float(d)), V, gy[j]);
        lap[j] = add2(lap[j], V);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float2 c0 = c[j + 2];
    const float2 ny = fma2(f2(-8.0f), sub2(c[j + 3], c[j + 1]), sub2(c[j + 4], c[j]));
    const float2 my = fma2(f2(6.0f), c0, fma2(f2(-4.0f), add2(c[j + 3], c[j + 1]), add2(c[j + 4], c[j])));
    // -12 times the convection
    const float2 cv = fma2(u[j], nx[j], fma2(v[j], ny, fma2(nabs2(u[j]), mx[j], mul2(nabs2(v[j]), my))));
    const float2 T = add2(c0, f2(k.T_sat));
    const float2 rs = make_float2(rsqrt_approx(T.x), rsqrt_approx(T.y));
    const float2 work = mul2(T, fma2(fz[j].Q, rs, fz[j].P));
    const float2 diff = fma2(fz[j].al2, lap[j], fma2(fz[j].ax, gx[j], mul2(fz[j].ay, gy[j])));
    L[j] = fma2(f2(float(1.0 / 12.0)), cv, sub2(diff, work));
  }
}

// Density of the pulled populations at a column pair of row y (neighbour rows ym, yp), from aligned
// pairs: the planes with c_x = +/-1 hand one value to the next or previous lane.  Every lane of the
// warp calls it with consecutive pairs; the first and last lane lack their neighbour.
template <typename S>
__device__ __forceinline__ float2 pull_rho_pair(const Geo& g, const Phys& ph, const S* __restrict__ f, int x, int y,
                                                int ym, int yp) {
  const uint32_t o = y * g.pitch + x, om = ym * g.pitch + x, op = yp * g.pitch + x;
  float2 v[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    S a, b;
    PairLoad<S>::ld(f + i * g.plane + (cyv(i) == 0 ? o : (cyv(i) > 0 ? om : op)), a, b);
    v[i] = make_float2(PopIO<float, S>::ld(a, i, ph), PopIO<float, S>::ld(b, i, ph));
  }
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    if (cxv(i) > 0) v[i] = make_float2(__shfl_up_sync(0xffffffffu, v[i].y, 1), v[i].x);
    if (cxv(i) < 0) v[i] = make_float2(v[i].y, __shfl_down_sync(0xffffffffu, v[i].x, 1));
  }
  return pop_sum2(v);
}

// lambda(rho) / c_v with alpha(rho) linear in the phase fraction, clamped to [0, 1].
__device__ __forceinline__ float lam_cv(const StepConst& k, float rho) {
  return __fmul_rn(rho, __fmaf_rn(__saturatef(__fmaf_rn(rho, k.ph1, k.ph0)), k.da, k.av));
}

// The stored temperature of theta = T - T_sat (theta_of of lbm_kernels.cuh is the way back).
__device__ __forceinline__ float2 T_of(const StepConst& k, float2 theta) {
  // the nearest temperature that can be stored.  The stored T_sat stands for theta = 0 and lies dT_sat off the
  // even spacing, so its two boundaries are dT_sat / 2 off the even ones: rounded evenly there, a bulk that
  // fluctuates about T_sat would drift by a fraction of dT_sat each step
  const float2 d = make_float2(fabsf(theta.x) < k.T_ulp ? k.dT_half : k.dT_sat,
                               fabsf(theta.y) < k.T_ulp ? k.dT_half : k.dT_sat);
  return add2(f2(k.T_sat), add2(theta, d));
}

// Block-level end of the wall heat flux: one FP64 partial per tile column and 4-row group of the
// lattice (two warps), whatever the tile's height, so that tiles of 4, 8 and 16 rows give the same
// bits; only the blocks that hold wall nodes take part.  The last of those n_wall blocks to finish
// adds the partials of the groups that can be nonzero, in the order of 128 threads, updates the
// running statistics hf and clears the partials for the next launch.  Every thread calls it.
template <int TY>
__device__ __forceinline__ void heat_flux_groups(const Geo& g, double q, int mine, double* partial, unsigned* counter,
                                                 int n_wall, int bx, int by, int ntx, double* hf, int nb, double* red,
                                                 int* done_last) {
  const int tid = threadIdx.x;
  if (!__syncthreads_or(mine)) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) q += __shfl_down_sync(0xffffffffu, q, o);
  if ((tid & 31) == 0) red[tid >> 5] = q;
  __syncthreads();
  const int gi = by * (TY / 4) + tid;
  if (tid < TY / 4 && 4 * gi < g.ny) {
    partial[gi * ntx + bx] = red[2 * tid] + red[2 * tid + 1];
    __threadfence();
  }
  __syncthreads();
  if (tid == 0) *done_last = atomicInc(counter, n_wall - 1) == (unsigned)(n_wall - 1);
  __syncthreads();
  if (!*done_last) return;
  __threadfence();
  double acc = 0.0;
  const int first = g.hf_g0 * ntx, last = g.hf_g1 * ntx;
  if (tid < 128)
    for (int i = first + tid; i < last; i += 128) acc += __ldcg(&partial[i]);
  acc = block_sum<128>(acc, red);  // its barrier also ends every thread's reads above
  if (tid < 128)
    for (int i = first + tid; i < last; i += 128) partial[i] = 0.0;
  if (tid == 0) {
    const double qv = acc / nb;
    hf[0] = qv;
    hf[1] += qv;
    hf[2] += qv * qv;
    hf[3] += 1.0;
  }
}

// Both Heun stages on tile (bx, by) of ntx tile columns.  With PULL and psi_out set the
// tile also evaluates psi of the next step at its nodes from the pull of the populations this
// step's collision wrote (fnew, side_new).
// maps: tensor maps of the inputs, with which an interior tile stages them by TMA (else null:
// plain loads); t1_out: where to store theta of stage 1 (the adjoint's recompute).
template <typename S, int PSI, bool PULL, int TY>
__device__ __forceinline__ void energy_strip(const Geo& g, const Phys& ph, const float* __restrict__ Tin,
                                             float* __restrict__ Tout, const float* __restrict__ rho,
                                             const float* __restrict__ ux, const float* __restrict__ uy,
                                             const uint8_t* __restrict__ mask, double* partial, unsigned* counter,
                                             double* hf, int nb, int do_hf, int n_wall_tiles, int bx, int by, int ntx,
                                             const S* __restrict__ fnew, const float* __restrict__ side_new,
                                             float* __restrict__ psi_out, int* status, float* __restrict__ t1_out,
                                             const EnergyMaps* maps, bool starve) {
  using ET = EnergyTile<TY>;
  constexpr int TX = ET::TX, NT = ET::NT, H = 4, AX = TX + 2 * H, AY = TY + 2 * H, BX = TX + 4, BY = TY + 4;
  static_assert(BX == 64 && TY % 2 == 0 && NT == 32 * (TY / 2 + 2), "one warp per two rows of 64 columns");
  static_assert(AX * sizeof(float) % 16 == 0 && AX * AY % 4 == 0, "TMA boxes of the input tile, staged four nodes at a time");
  __shared__ __align__(128) float sT[AY * AX];        // T, then theta
  __shared__ __align__(128) float sRUV[3 * AY * AX];  // rho, u_x, u_y: the planes of one TMA box
  __shared__ __align__(16) float sL[AY * AX];         // lambda / c_v
  __shared__ __align__(16) float sT1[BY * BX];        // theta of stage 1
  __shared__ uint64_t s_bar;
  __shared__ double red[NT / 32];
  __shared__ int done_last;
  const StepConst& k = ph.sc;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int x0 = bx * TX, y0 = by * TY;
  const bool own = warp < TY / 2;
  const int rb = own ? 2 * warp : (warp == TY / 2 ? -2 : TY);  // the warp's upper row in the tile
  const int xl = x0 - 2 + 2 * lane;                             // the lane's left column
  const bool interior = x0 >= H && y0 >= H && x0 + TX + H <= g.nx && y0 + TY + H <= g.ny;
  // TMA also stages the tiles at an inlet or outlet (ghost columns are filled below); tiles whose rows
  // wrap, and the edge columns of a periodic lattice, are copied plainly
  const bool staged = maps && y0 >= H && y0 + TY + H <= g.ny && (interior || !g.periodic_x);
  uint32_t m[2];  // node types of the pair (bytes 0, 1) in the two rows
  if (interior) {
#pragma unroll
    for (int j = 0; j < 2; ++j) m[j] = *reinterpret_cast<const uint16_t*>(mask + (y0 + rb + j) * g.pitch + xl);
  } else {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint8_t* row = mask + map_y(g, y0 + rb + j) * g.pitch;
      m[j] = row[map_x(g, xl)] | (uint32_t)row[map_x(g, xl + 1)] << 8;
    }
  }
  if (staged) {
    // the input boxes by TMA (first column x0 - 4: 16-byte aligned)
    if (tid == 0) {
      tma::bar_init(&s_bar, 1);
      tma::bar_expect_tx(&s_bar, 4 * AX * AY * sizeof(float));
      // T comes from the energy pass before the previous kernel (the collision, which does not
      // write it): its copy starts before that kernel ends; the test hook leaves the barrier
      // armed with no copy issued
      if (!starve) tma::load_2d(sT, &maps->T, &s_bar, x0 - H, y0 - H);
    }
    pdl::wait();  // rho, u and the new populations are the collision's output
    pdl::trigger();
    if (tid == 0 && !starve) tma::load_3d(sRUV, &maps->ruv, &s_bar, x0 - H, y0 - H, 0);
  } else {
    pdl::wait();
    pdl::trigger();
    const float* const src[4] = {Tin, rho, ux, uy};
    if (interior || !g.periodic_x) {
      constexpr int NV = AX / 4;
#pragma unroll
      for (int k4 = 0; k4 < 4; ++k4) {
        float* dst = k4 == 0 ? sT : sRUV + (k4 - 1) * AX * AY;
#pragma unroll 2
        for (int p = tid; p < AY * NV; p += NT) {
          const int r = p / NV, c = (p - r * NV) * 4, gx = x0 - H + c;
          if (gx >= 0 && gx < g.pitch)
            *reinterpret_cast<float4*>(dst + r * AX + c) =
                *reinterpret_cast<const float4*>(src[k4] + map_y(g, y0 + r - H) * g.pitch + gx);
        }
      }
    } else {
#pragma unroll 2
      for (int p = tid; p < AX * AY; p += NT) {
        const int nid = map_y(g, y0 + p / AX - H) * g.pitch + map_x(g, x0 + p % AX - H);
        sT[p] = Tin[nid];
        sRUV[p] = rho[nid];
        sRUV[AX * AY + p] = ux[nid];
        sRUV[2 * AX * AY + p] = uy[nid];
      }
    }
  }
  // density of the next step's pull, while the copies fly
  float2 rn[2];
  if (PULL && psi_out && own) {
    const int xc = xl < 0 ? 0 : (xl > g.pitch - 2 ? g.pitch - 2 : xl);
    uint32_t slow = 0;  // nodes next to the wall or in an edge column: the pull with its substitutions
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int y = y0 + rb + j, yc = y < g.ny ? y : g.ny - 1;
      rn[j] = pull_rho_pair<S>(g, ph, fnew, xc, yc, yc == 0 ? g.ny - 1 : yc - 1, yc == g.ny - 1 ? 0 : yc + 1);
      if (lane >= 1 && lane <= 30 && y < g.ny) {
#pragma unroll
        for (int i = 0; i < 2; ++i)
          if (xl + i < g.nx && !((m[j] >> (8 * i)) & kSolid) &&
              (((m[j] >> (8 * i)) & kNearWall) || xl + i == 0 || xl + i == g.nx - 1))
            slow |= 1u << (2 * j + i);
      }
    }
#pragma unroll 1
    for (; slow; slow &= slow - 1) {
      const int q = __ffs(slow) - 1;
      float fo[9];
      pull_node<float, S>(g, ph, fnew, mask, side_new, nullptr, xl + (q & 1), y0 + rb + (q >> 1),
                          (uint8_t)(m[q >> 1 & 1] >> (8 * (q & 1))), fo);
      const float r = pop_sum<float, S>(fo);
      if (q == 0) rn[0].x = r;
      if (q == 1) rn[0].y = r;
      if (q == 2) rn[1].x = r;
      if (q == 3) rn[1].y = r;
    }
  }
  __syncthreads();  // the barrier is initialised, or the plain loads complete
  const int tries = starve ? tma::kStarveTries : tma::kWaitTries;
  bool landed = true;
  if (staged) landed = tma::bar_wait(&s_bar, 0, tries);
  if (!g.periodic_x && (x0 < H || x0 + TX + H > g.nx)) {
    // ghost columns past an open edge repeat the edge column
    const int cl = H - x0, cr = g.nx - 1 - x0 + H;  // tile columns of x = 0 and x = nx - 1
    __syncthreads();
    for (int p = tid; p < 4 * AY * H; p += NT) {
      const int k4 = p / (AY * H), r = (p / H) % AY, c = p % H;
      float* row = (k4 == 0 ? sT : sRUV + (k4 - 1) * AX * AY) + r * AX;
      if (x0 < H) row[cl - 1 - c] = row[cl];
      if (cr + 1 + c < AX) row[cr + 1 + c] = row[cr];
    }
    __syncthreads();
  }
  for (int p = tid; p < AX * AY / 4; p += NT) {  // lambda and theta, four nodes per thread
    const float4 r = reinterpret_cast<const float4*>(sRUV)[p], t = reinterpret_cast<const float4*>(sT)[p];
    reinterpret_cast<float4*>(sL)[p] = make_float4(lam_cv(k, r.x), lam_cv(k, r.y), lam_cv(k, r.z), lam_cv(k, r.w));
    reinterpret_cast<float4*>(sT)[p] = make_float4(theta_of(k, t.x), theta_of(k, t.y), theta_of(k, t.z), theta_of(k, t.w));
  }
  if (__syncthreads_or(!landed)) {
    // a copy did not land in time: report it, let the copies land (bounded) and stop the tile
    // (a tile that holds wall nodes then misses its heat-flux partial; restoring a state with
    // lbm_set_state resets that bookkeeping)
    if (tid == 0) atomicOr(status, kStatusTimeoutEnergy);
    tma::bar_wait(&s_bar, 0, tries);
    return;
  }
  // stage 1 at the warp's two rows: theta1 = theta + L(theta)
  constexpr int A2 = AX / 2, B2 = BX / 2, AP = AX * AY / 2;
  const float2* const aT = reinterpret_cast<const float2*>(sT) + (rb + H) * A2 + lane;  // window columns -2, -1
  const float2* const aL = reinterpret_cast<const float2*>(sL) + (rb + H) * A2 + lane;
  const float2* const aR = reinterpret_cast<const float2*>(sRUV) + (rb + H) * A2 + lane;
  float2* const bT = reinterpret_cast<float2*>(sT1) + (rb + 2) * B2 + lane;
  FrozenPair fz[2];
  double q = 0.0;
  int mine = 0;
  {
    frozen_rows(k, aL, aR + AP, aR + 2 * AP, aR + 1, A2, fz);
    const float2 u[2] = {aR[AP + 1], aR[AP + A2 + 1]}, v[2] = {aR[2 * AP + 1], aR[2 * AP + A2 + 1]};
    float2 L[2], gx[2], gy[2];
    rhs_rows(k, aT, A2, u, v, fz, L, gx, gy);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float2 t = aT[j * A2 + 1];
      float2 t1 = add2(t, L[j]);
      if (!g.periodic_x && xl == 0) t1.x = 0.0f;  // the inlet column stays at T_sat (xl is even)
      if (m[j] & kSolid) t1.x = t.x;  // solid nodes keep their wall temperature
      if (m[j] & (kSolid << 8)) t1.y = t.y;
      bT[j * B2] = t1;  // positions past a non-periodic edge are replaced below
      if (do_hf && own && (m[j] & (kNearWall * 0x0101u)) && lane >= 1 && lane <= 30 && y0 + rb + j < g.ny) {
        // the wall heat flux -lambda grad T^n . n of the pair's near-wall nodes (Sec. IV.B)
        const float2 l = aL[j * A2 + 1];
#pragma unroll
        for (int i = 0; i < 2; ++i)
          if (((m[j] >> (8 * i)) & kNearWall) && xl + i < g.nx) {
            const double* nv = &g.wall_n[2 * g.wall_idx[(y0 + rb + j) * g.pitch + xl + i]];
            q += -(double)__fmul_rn(ph.f.c_v, i ? l.y : l.x) *
                 ((double)(i ? gx[j].y : gx[j].x) * nv[0] + (double)(i ? gy[j].y : gy[j].x) * nv[1]);
            mine = 1;
          }
      }
    }
  }
  __syncthreads();
  if (!g.periodic_x && (x0 < 2 || x0 + TX + 2 > g.nx)) {
    for (int p = tid; p < BX * BY; p += NT) {
      const int gx = x0 + p % BX - 2;
      if (gx < 0 || gx >= g.nx) sT1[p] = sT1[p - p % BX + (map_x(g, gx) - x0 + 2)];
    }
    __syncthreads();
  }
  // stage 2 at the own rows: T^{n+1} = T_sat + (theta + theta1 + L(theta1)) / 2
  if (own) {
    const int lc = lane < 1 ? 1 : (lane > 30 ? 30 : lane);  // the first and last lane hold halo columns only
    const float2 u[2] = {aR[AP + 1], aR[AP + A2 + 1]}, v[2] = {aR[2 * AP + 1], aR[2 * AP + A2 + 1]};
    float2 L[2], gx[2], gy[2], out[2];
    rhs_rows(k, bT - lane + lc - 1, B2, u, v, fz, L, gx, gy);
    const bool lane_out = lane >= 1 && lane <= 30 && xl < g.nx;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint32_t id = (y0 + rb + j) * g.pitch + xl;
      const float2 t = aT[j * A2 + 1], t1 = bT[j * B2];
      out[j] = T_of(k, mul2(f2(0.5f), add2(add2(t, t1), L[j])));
      if (!lane_out || y0 + rb + j >= g.ny) continue;
      if (!g.periodic_x && xl == 0) out[j].x = k.T_sat;
      if (m[j] & kSolid) out[j].x = Tin[id];
      if ((m[j] & (kSolid << 8)) && xl + 1 < g.nx) out[j].y = Tin[id + 1];
      // the row pitch is even: a pair whose right node lies past an odd nx ends in the padding
      *reinterpret_cast<float2*>(Tout + id) = out[j];
      if (t1_out) *reinterpret_cast<float2*>(t1_out + id) = t1;
    }
    if (PULL && psi_out) {
      if (lane_out) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if (y0 + rb + j >= g.ny) continue;
          const float rs = ph.f.rho_s;
          float2 ps;
          ps.x = psi_of<float, PSI>(ph, (m[j] & kSolid) ? rs : rn[j].x, out[j].x, status);
          ps.y = 0.0f;
          if (xl + 1 < g.nx) ps.y = psi_of<float, PSI>(ph, (m[j] & (kSolid << 8)) ? rs : rn[j].y, out[j].y, status);
          *reinterpret_cast<float2*>(psi_out + (uint32_t)((y0 + rb + j) * g.pitch + xl)) = ps;
        }
      }
    }
  }
  if (do_hf) heat_flux_groups<TY>(g, q, mine, partial, counter, n_wall_tiles, bx, by, ntx, hf, nb, red, &done_last);
}

}  // namespace kern
}  // namespace lbm
