// FP32 step: the kernels of a single domain and of a batch over the tiles of lbm_flow_f32.cuh and
// lbm_energy_f32.cuh, and their launchers.
#pragma once

#include "lbm_kernels.cuh"

namespace lbm {
namespace kern {
// Energy tile of the FP32 build: 60 x TY nodes, a warp per two rows and two for the halo rows.
template <int TY_>
struct EnergyTile {
  static constexpr int TX = kEnergyTX32, TY = TY_;
  static constexpr int NT = 32 * (TY / 2 + 2);
};
}  // namespace kern
}  // namespace lbm

#include "lbm_flow_f32.cuh"
#include "lbm_energy_f32.cuh"

namespace lbm {
namespace kern {

template <int PSI, int OP>
__global__ void __launch_bounds__(FlowTile<kFlowTY>::NT, 2)
    k_collide_f32(Geo g, Phys ph, const float* __restrict__ f, float* __restrict__ fn, const float* __restrict__ T, float* psi,
                  const uint8_t* __restrict__ mask, const float* __restrict__ side_in, float* __restrict__ side_out,
                  float* __restrict__ rho_o, float* __restrict__ ux_o, float* __restrict__ uy_o, int forcing,
                  int* status, const __grid_constant__ CUtensorMap tm_f, int flags) {
  flow_tile<PSI, OP, kFlowTY>(g, ph, f, fn, T, psi, mask, side_in, side_out, rho_o, ux_o, uy_o,
                                                    forcing, status, blockIdx.x, blockIdx.y,
                                                    (flags & kLaunchStaged) ? &tm_f : nullptr,
                                                    (flags & kLaunchStarve) != 0, (flags & kLaunchEarlyF) != 0);
}

template <typename S, int PSI, bool PULL, int TY>
__global__ void __launch_bounds__(EnergyTile<TY>::NT, TY == kEnergyTY ? 3 : 4)
    k_energy_f32(Geo g, Phys ph, const float* __restrict__ Tin, float* __restrict__ Tout, const float* __restrict__ rho,
                 const float* __restrict__ ux, const float* __restrict__ uy, const uint8_t* __restrict__ mask,
                 double* partial, unsigned* counter, double* hf, int nb, int do_hf, int n_wall_tiles,
                 const S* __restrict__ fnew, const float* __restrict__ side_new, float* __restrict__ psi_out,
                 int* status, float* __restrict__ t1_out, const __grid_constant__ EnergyMaps maps, int flags) {
  energy_strip<S, PSI, PULL, TY>(g, ph, Tin, Tout, rho, ux, uy, mask, partial, counter, hf, nb, do_hf, n_wall_tiles,
                                 blockIdx.x, blockIdx.y, gridDim.x, fnew, side_new, psi_out, status, t1_out,
                                 (flags & kLaunchStaged) ? &maps : nullptr, (flags & kLaunchStarve) != 0);
}

// ---------------------------------------------------------------- batched passes
// A batched launch covers the blocks [block0, block0 + gridDim.x) of a pass, which belong to the
// domains dom0 ..; their tensor maps come as kernel parameters (index k - dom0).
template <int CTY>
__global__ void __launch_bounds__(FlowTile<CTY>::NT, CTY == kFlowTY ? 2 : 3)
    kb_collide_f32(const BatchDomain* __restrict__ doms, const int* __restrict__ map, int cur, int tcur, long long step,
                   int block0, int dom0, const __grid_constant__ FlowLaunchMaps maps) {
  const int blk = block0 + blockIdx.x, k = map[blk];
  const BatchDomain& D = doms[k];
  const int local = blk - D.coll_first;
  flow_tile<kPsiDF, kCollCM, CTY>(
      D.g, D.ph, static_cast<const float*>(D.d.f[cur]), static_cast<float*>(D.d.f[cur ^ 1]),
      static_cast<const float*>(D.d.T[tcur]), psi_buf<float>(D, cur), D.d.mask,
      static_cast<const float*>(D.d.side[cur]), static_cast<float*>(D.d.side[cur ^ 1]), static_cast<float*>(D.d.rho),
      static_cast<float*>(D.d.ux), static_cast<float*>(D.d.uy), step >= D.warmup, D.d.status, local % D.coll_ntx,
      local / D.coll_ntx, D.tma ? &maps.f[k - dom0] : nullptr, false, false);
}
template <int ETY>
__global__ void __launch_bounds__(EnergyTile<ETY>::NT, 960 / EnergyTile<ETY>::NT)
    kb_energy_f32(const BatchDomain* __restrict__ doms, const int* __restrict__ map, int cur, int tcur, long long step,
                  int block0, int dom0, const __grid_constant__ EnLaunchMaps maps) {
  const int blk = block0 + blockIdx.x, k = map[blk];
  const BatchDomain& D = doms[k];
  const int local = blk - D.en_first, bx = local % D.en_ntx, by = local / D.en_ntx;
  const float* Tin = static_cast<const float*>(D.d.T[tcur]);
  float* Tout = static_cast<float*>(D.d.T[tcur ^ 1]);
  if (!D.energy || step < D.warmup) {
    // no energy update for this domain this step: carry T over so all domains flip together
    constexpr int TX = EnergyTile<ETY>::TX;
    for (int p = threadIdx.x; p < TX * ETY; p += EnergyTile<ETY>::NT) {
      const int x = bx * TX + p % TX, y = by * ETY + p / TX;
      if (x < D.g.nx && y < D.g.ny) Tout[y * D.g.pitch + x] = Tin[y * D.g.pitch + x];
    }
    return;
  }
  energy_strip<float, kPsiDF, false, ETY>(
      D.g, D.ph, Tin, Tout, static_cast<const float*>(D.d.rho), static_cast<const float*>(D.d.ux),
      static_cast<const float*>(D.d.uy), D.d.mask, D.d.partial, D.d.counter, D.d.hf, D.d.nb, D.d.nb > 0,
      D.d.wall_tiles[ETY == kEnergyTY ? 1 : 0], bx, by, D.en_ntx, nullptr, nullptr, nullptr, D.d.status,
      nullptr, D.tma ? &maps.e[k - dom0] : nullptr, false);
}

// Tensor maps of one batched domain for tile heights (cty, ety).
inline bool batch_maps_impl_f32(BatchDomain& D, DomainMaps& m, int cty, int ety) {
  using FT = FlowTile<8>;
  const Geo& g = D.g;
  bool ok = D.d.tma != 0 && static_cast<const float*>(D.d.ux) == static_cast<const float*>(D.d.rho) + g.plane &&
            static_cast<const float*>(D.d.uy) == static_cast<const float*>(D.d.rho) + 2 * (size_t)g.plane;
  for (int p = 0; p < 2 && ok; ++p)
    ok = tma::encode<float>(&m.f[p], D.d.f[p], g.nx, g.ny, g.pitch, g.plane, 9, FT::FW, cty + 2 * FT::FR) &&
         tma::encode<float>(&m.em[p].T, D.d.T[p], g.nx, g.ny, g.pitch, g.plane, 1, kEnergyTX32 + 8, ety + 8) &&
         tma::encode<float>(&m.em[p].ruv, D.d.rho, g.nx, g.ny, g.pitch, g.plane, 3, kEnergyTX32 + 8, ety + 8);
  D.tma = ok ? 1 : 0;
  return ok;
}

template <int CTY, int ETY>
int batch_step_impl_f32(const BatchDomain* doms, const int* map_coll, int nb_coll, const int* map_en, int nb_en, int cur,
                        int tcur, long long step, const BatchDomain* hdoms, const DomainMaps* hmaps, int ndom,
                        cudaStream_t s) {
  int n = 0;
  for (int d0 = 0; d0 < ndom; d0 += kBatchCollDomains) {
    const int d1 = d0 + kBatchCollDomains < ndom ? d0 + kBatchCollDomains : ndom;
    FlowLaunchMaps m;
    for (int k = d0; k < d1; ++k) m.f[k - d0] = hmaps[k].f[cur];
    const int b0 = hdoms[d0].coll_first, b1 = d1 < ndom ? hdoms[d1].coll_first : nb_coll;
    kb_collide_f32<CTY><<<b1 - b0, FlowTile<CTY>::NT, 0, s>>>(doms, map_coll, cur, tcur, step, b0, d0, m);
    ++n;
  }
  for (int d0 = 0; d0 < ndom; d0 += kBatchEnDomains) {
    const int d1 = d0 + kBatchEnDomains < ndom ? d0 + kBatchEnDomains : ndom;
    EnLaunchMaps m;
    for (int k = d0; k < d1; ++k) m.e[k - d0] = hmaps[k].em[tcur];
    const int b0 = hdoms[d0].en_first, b1 = d1 < ndom ? hdoms[d1].en_first : nb_en;
    kb_energy_f32<ETY><<<b1 - b0, EnergyTile<ETY>::NT, 0, s>>>(doms, map_en, cur, tcur, step, b0, d0, m);
    ++n;
  }
  return cudaPeekAtLastError() == cudaSuccess ? n : -1;
}

}  // namespace kern

// ---------------------------------------------------------------- single-domain step
template <int PSI>
void launch_flow_f32(const Geo& g, const Phys& ph, const Dev& d, int cur, int tcur, int forcing, cudaStream_t s) {
  using namespace kern;
  using FT = FlowTile<kFlowTY>;
  const float* f = static_cast<const float*>(d.f[cur]);
  CUtensorMap tm_f;
  const bool staged = d.tma && tma::encode<float>(&tm_f, f, g.nx, g.ny, g.pitch, g.plane, 9, FT::FW, FT::FH);
  const int flags = staged ? (kLaunchStaged | ((d.starve & kStarveCollide) ? kLaunchStarve : 0) |
                              ((d.pdl && d.f_ready) ? kLaunchEarlyF : 0))
                           : 0;
  const dim3 grd((g.nx + FT::TX - 1) / FT::TX, (g.ny + FT::TY - 1) / FT::TY);
  auto go = [&](auto kernel) {
    launch_dep(d.pdl, grd, dim3(FT::NT), 0, s, kernel, g, ph, f, static_cast<float*>(d.f[cur ^ 1]),
               static_cast<const float*>(d.T[tcur]), static_cast<float*>(d.psi), d.mask,
               static_cast<const float*>(d.side[cur]), static_cast<float*>(d.side[cur ^ 1]), static_cast<float*>(d.rho),
               static_cast<float*>(d.ux), static_cast<float*>(d.uy), forcing, d.status, tm_f, flags);
  };
  if (d.collision == kCollBGK) go(k_collide_f32<PSI, kCollBGK>);
  else go(k_collide_f32<PSI, kCollCM>);
}

template <typename S, int PSI, bool PULL, int TY>
void launch_energy_f32(const Geo& g, const Phys& ph, const Dev& d, int cur, int tcur, bool fuse, cudaStream_t s) {
  using namespace kern;
  using ET = EnergyTile<TY>;
  const float* T = static_cast<const float*>(d.T[tcur]);
  const float* rho = static_cast<const float*>(d.rho);
  const float *ux = static_cast<const float*>(d.ux), *uy = static_cast<const float*>(d.uy);
  const dim3 grd((g.nx + ET::TX - 1) / ET::TX, (g.ny + ET::TY - 1) / ET::TY);
  constexpr int AX = ET::TX + 8, AY = ET::TY + 8;
  EnergyMaps em;
  const bool ruv = ux == rho + g.plane && uy == rho + 2 * (size_t)g.plane;  // consecutive planes
  const bool staged = d.tma && ruv && tma::encode<float>(&em.T, T, g.nx, g.ny, g.pitch, g.plane, 1, AX, AY) &&
                      tma::encode<float>(&em.ruv, rho, g.nx, g.ny, g.pitch, g.plane, 3, AX, AY);
  launch_dep(d.pdl, grd, dim3(ET::NT), 0, s, k_energy_f32<S, PSI, PULL, TY>, g, ph, T,
             static_cast<float*>(d.T[tcur ^ 1]), rho, ux, uy, d.mask, d.partial, d.counter, d.hf, d.nb,
             (int)(d.nb > 0), d.wall_tiles[TY == kEnergyTY ? 1 : 2], fuse ? static_cast<const S*>(d.f[cur ^ 1]) : nullptr,
             static_cast<const float*>(d.side[cur ^ 1]), fuse ? static_cast<float*>(d.psi_next) : nullptr, d.status,
             static_cast<float*>(d.t1_out), em,
             staged ? (kLaunchStaged | ((d.starve & kStarveEnergy) ? kLaunchStarve : 0)) : 0);
}

// The collision of a step: with psi in its tiles (populations stored in FP32, psi in FP32 or double-float), or
// one node per lane (launch_collide) where psi is read, or there is none: FP64 populations and FP64 psi, whose
// tiles would not fit shared memory or cost more than a second pull, and single-phase fluids.  Pairs of columns
// took longer there: FP64 populations 58 us against 49 at 1350 x 600 and 127 against 111 at 2048 x 1024, a single phase
// 6.6 against 3.0 at 241 x 241, 6.3 against 4.5 at 512 x 512 and 36 against 31 at 2048 x 1024 (a step, energy pass off).
// psi that is read comes from the energy pass of the step before or, in a first step, from k_rho_psi.  On
// small lattices (flow_psi_in_tile) a step whose predecessor ran no energy pass (a first step, a warm-up step,
// T fixed) takes psi from k_rho_psi too.
template <typename S, int PSI>
int step_impl_f32(const Geo& g, const Phys& ph, const Dev& d, int cur, int tcur, int forcing, int energy,
                  cudaStream_t s, const LaunchHook* hook, int* t_flipped, PsiChain* chain) {
  using namespace kern;
  constexpr bool can_tile = PSI != kPsiF64 && sizeof(S) != 8;
  const bool multi = ph.d.G != 0.0;
  const bool tile = can_tile && multi && (flow_psi_in_tile(g.nx, g.ny) || (chain && chain->have));
  int n = 0;
  auto pre = [&](int k) {
    if (hook) hook->before(hook->self, k);
  };
  auto post = [&](int k) {
    if (hook) hook->after(hook->self, k);
    ++n;
  };
  if (multi && !tile && !(chain && chain->have)) {
    const dim3 blk(kCollTX, 8), grd((g.nx + kCollTX - 1) / kCollTX, (g.ny + 7) / 8);
    pre(kKRhoPsi);
    k_rho_psi<float, S, PSI><<<grd, blk, 0, s>>>(g, ph, static_cast<const S*>(d.f[cur]),
                                                 static_cast<const float*>(d.T[tcur]), d.mask,
                                                 static_cast<const float*>(d.side[cur]), static_cast<float*>(d.psi),
                                                 d.status);
    post(kKRhoPsi);
  }
  pre(kKCollide);
  if constexpr (!can_tile) {
    launch_collide<float, S>(g, ph, d, cur, forcing, nullptr, s);
  } else {
    if (tile) launch_flow_f32<PSI>(g, ph, d, cur, tcur, forcing, s);
    else launch_collide<float, S>(g, ph, d, cur, forcing, nullptr, s);
  }
  post(kKCollide);
  *t_flipped = 0;
  if (chain) chain->made = kPsiFromPass;
  if (energy && forcing) {
    const bool next = chain && chain->want && multi, small = small_lattice(g.nx, g.ny);
    pre(kKEnergy);
    if (!can_tile && next) {
      if constexpr (!can_tile) {
        if (small) launch_energy_f32<S, PSI, true, kEnergyTYSmall>(g, ph, d, cur, tcur, true, s);
        else launch_energy_f32<S, PSI, true, kEnergyTY>(g, ph, d, cur, tcur, true, s);
      }
    } else {
      if (small) launch_energy_f32<float, kPsiDF, false, kEnergyTYSmall>(g, ph, d, cur, tcur, false, s);
      else launch_energy_f32<float, kPsiDF, false, kEnergyTY>(g, ph, d, cur, tcur, false, s);
    }
    post(kKEnergy);
    *t_flipped = 1;
    if (chain) chain->made = !next ? kPsiFromPass : can_tile ? kPsiFromTile : kPsiFromPlane;
  }
  return cudaPeekAtLastError() == cudaSuccess ? n : -1;
}

}  // namespace lbm
