// FP64 storage (the plain method): fused pull-stream + collide step with all
// arithmetic in FP64, plus the FP64 initialiser, read-out and raw copies.
#include <cuda_runtime.h>

#include "rlbm_kernels.cuh"

namespace rlbm {

// The velocity, gamma and rate the collision uses: constant tau, or the local
// tau = 4 (eta/s) / theta + 0.2546 of Sec. 3.5; a body force shifts the velocity to
// u + a tau (Sec. 3.4). (Branches, uniform per domain: the divisions only run for a
// local tau.)
__device__ __forceinline__ void collision_frame(const DomDev& D, double theta, double& ux, double& uy, double& gam,
                                                double& itau) {
  double tau = D.tau;
  itau = D.inv_tau;
  if (D.eta_s > 0.0) {
    tau = 4.0 * D.eta_s / theta + 0.2546;
    itau = 1.0 / tau;
  }
  if (D.accel_x != 0.0 || D.accel_y != 0.0) {
    ux += D.accel_x * tau;
    uy += D.accel_y * tau;
    gam = 1.0 / sqrt(1.0 - ux * ux - uy * uy);
  }
}

// One fused step for every cell of every tile: pull-stream from fin (its halo
// was filled by the previous step), moments, Landau state, equilibrium,
// relaxation (Eq. 3), store to fout and fill fout's halo.
//
// Bound: the FP64 pipe. One FP64 warp instruction holds its SM sub-partition's unit
// for 64 clocks, whatever its operation and however many lanes are active, so the
// count of FP64 instructions per cell is the time. About 1,000 (MJ): pull 192, moments
// 200, Landau 35 (FP32 start), state and equilibrium moments 65, directional powers
// and rates 45, six shells of 80 (21 projection, 35 synthesis, 24 relaxation). With
// FP64 Newton throughout and harmonic powers applied before the projection it was
// 1,382; conversions (the FP64 unit's too) run on the integer pipe. A 512^2 domain a
// step: MJ 720 -> 513 us, BE 1,000 -> 568 us; the local-tau disc 730 -> 525 us.
// kVw: the launch has velocity walls (StepArgs::halo 3); without them their code and its
// registers are left out (512^2: 569 -> 530 us).
template <int EDF, bool kVw>
__global__ void __launch_bounds__(kThreads, 2) k_step_f64(StepArgs a) {
  extern __shared__ double sm[];
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
    const Tile tl = a.tiles[t];
    const DomDev& D = a.doms[tl.dom];
    int x, y;
    if (!tile_cell(tl, threadIdx.x, threadIdx.y, x, y) || x >= D.nx || y >= D.ny) continue;
    const double* __restrict__ fin = static_cast<const double*>(a.fin) + D.off;
    double* __restrict__ fout = static_cast<double*>(a.fout) + D.off;
    const long long c = cell_rel(D, x, y);
    double N[3], T[6];
    pull_moments64<EDF, StoreF64>(fin, D, x, y, c, sm, tid, N, T);
    CellState S;
    unsigned st = cell_state<EDF, false>(N, T, S);
    const bool ok = !(st & ST_NONPHYSICAL);
    if (ok) {
      double ux = S.ux, uy = S.uy, gam = S.gamma, itau;
      collision_frame(D, S.theta, ux, uy, gam, itau);
      const int oi = D.order - 2;
      const DirPow C = dir_powers(ux, uy);
      // relaxation rates gamma (1 - v_d . u) / tau (Eq. 3): v_d . u = C_1(d), -C_1(d) at d + 6
      const double K = gam * itau;
      double om[12];
#pragma unroll
      for (int d = 0; d < 6; ++d) {
        om[d] = fma(-K, C.c1[d], K);
        om[d + 6] = fma(K, C.c1[d], K);
      }
      double ym[21];
      // a clamped BE state relaxes to its own equilibrium energy 4 pi theta^3 g_3(z_c)
      const double eps_eq = (st & ST_CLAMPED) ? 4.0 * PI * S.theta * S.theta * S.theta * S.g[2] : S.eps;
      eq_moments<EDF>(S.g, S.theta, fma(ux, ux, uy * uy), gam, S.n, eps_eq, ym, oi);
      const bool vw = kVw && touches_vwall(D, x, y), clamped = (st & ST_CLAMPED) != 0;
      VwallGhosts G;
      if (vw) vwall_setup<EDF>(D, x, y, a.images != 0, &G, &st);
#pragma unroll 1
      for (int s = 0; s < 6; ++s) {
        double fe[12];
        feq_shell<EDF>(s, ym, C, fe, oi);
#pragma unroll
        for (int d = 0; d < 12; ++d) {
          const int q = 6 * d + s;
          const double v = sm[q * kThreads + tid];
          const double r = fma(om[d], fe[d] - v, v);
          sm[q * kThreads + tid] = r;
          if (vw) fe[d] = r - fe[d];
        }
        if (vw) {
          const double fw = vwall_shell<EDF>(G, s, oi);
          for (int i = 0; i < G.cnt; ++i) {
#pragma unroll
            for (int d = 0; d < 12; ++d) fout[G.at[i] + plane_off(6 * d + s)] = fw + fe[d];
          }
        }
      }
      if (EDF == EDF_BE && vw && clamped)
        vwall_clamped<true>(D, &G, S.theta, S.n, S.eps, ux, uy, gam, sm + tid, 0xfffu, fout);
    }
    // f* (or the unrelaxed populations of a non-physical cell), a plane pair per store
#pragma unroll 4
    for (int q = 0; q < 72; q += 2)
      *reinterpret_cast<Pair<double>*>(fout + plane_off(q) + c) =
          Pair<double>{sm[q * kThreads + tid], sm[(q + 1) * kThreads + tid]};
    if ((a.images || a.halo) && (x == 0 || x == D.nx - 1 || y == 0 || y == D.ny - 1))
      write_halo64<EDF, StoreF64>(D, x, y, fout, sm, tid, ok, S.n, S.ux, S.uy, S.gamma, st, ok, a.images != 0);
    if (st) atomicOr(a.status, st);
  }
}

// ------------------------------------------------- step of a launch of few warps
// The same update, bit for bit, by three warps per 32 cells (one warp of a tile),
// for launches that leave SM sub-partitions without a warp: there the time is one
// warp's chain of FP64 instructions (64 to 71 clocks each), not their number. Warp W
// pulls, sums, relaxes and stores the directions 2W, 2W + 1 and their opposites; the
// Landau solve runs in one warp (a different one from block to block); then that
// warp forms the equilibrium moments while the next forms the directional powers;
// each warp projects two shells. About 490 instructions in the longest chain instead
// of 1,000. One domain alone, a step: 64^2 44 -> 20.8 us, FD Riemann 2048 x 4 55 -> 35 us,
// 8 x 255 channel 57 -> 37 us.
struct SplitSm {
  double eo[6][4][32];     // e, o of A and B (harmonics_eo) per direction pair
  double cell[6][32];      // u_x, u_y, gamma, n, eps, theta
  double y[21][32];        // equilibrium moments
  double c[20][32];        // DirPow
  double R[6][6][32];      // projection by shell, k
  unsigned st[32], clamped[32];
};
constexpr int kSplitWarps = 3;

// Barrier of the block's three warps, which run code of their own.
__device__ __forceinline__ void split_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(32 * kSplitWarps) : "memory");
}

// Directions 2W + (i & 1) + 6 (i >> 1), i = 0..3, of warp W.
template <int EDF, int W>
__device__ __forceinline__ void split_pull(const double* __restrict__ fin, long long c, const Nbr& nb, double v[4][6],
                                           SplitSm& sm, int lane) {
  double A[4], B[4];
#define RLBM_SPLIT_DIR(i)                                                                        \
  {                                                                                              \
    constexpr int d = 2 * W + ((i) & 1) + 6 * ((i) >> 1);                                        \
    double a_ = 0.0, b_ = 0.0;                                                                   \
    _Pragma("unroll") for (int s = 0; s < 6; s += 2) {                                           \
      const Pair<double> r_ = pull_pair<d, PullF64, StoreF64>(fin + c + plane_off(6 * d + s), nb); \
      v[i][s] = r_.x;                                                                            \
      v[i][s + 1] = r_.y;                                                                        \
      a_ = fma(r_.x, c_p[EDF][s], a_);                                                           \
      b_ = fma(r_.x, c_p2[EDF][s], b_);                                                          \
      a_ = fma(r_.y, c_p[EDF][s + 1], a_);                                                       \
      b_ = fma(r_.y, c_p2[EDF][s + 1], b_);                                                      \
    }                                                                                            \
    A[i] = a_;                                                                                   \
    B[i] = b_;                                                                                   \
  }
  RLBM_SPLIT_DIR(0) RLBM_SPLIT_DIR(1) RLBM_SPLIT_DIR(2) RLBM_SPLIT_DIR(3)
#undef RLBM_SPLIT_DIR
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    sm.eo[2 * W + i][0][lane] = A[i] + A[i + 2];
    sm.eo[2 * W + i][1][lane] = A[i] - A[i + 2];
    sm.eo[2 * W + i][2][lane] = B[i] + B[i + 2];
    sm.eo[2 * W + i][3][lane] = B[i] - B[i + 2];
  }
}

// Relaxation of a warp's directions: v becomes f*; ghost(d, s, f*, f^eq) writes velocity-wall ghosts.
template <int EDF, int W, class Ghost>
__device__ __forceinline__ void split_relax(double K, double v[4][6], const SplitSm& sm, int lane, Ghost ghost) {
  DirPow C;  // the entries of directions 2W, 2W + 1
  constexpr int d0 = 2 * W, d1 = 2 * W + 1;
  C.c1[d0] = sm.c[d0][lane];
  C.c1[d1] = sm.c[d1][lane];
  C.c5[d0] = sm.c[6 + d0][lane];
  C.c5[d1] = sm.c[6 + d1][lane];
  C.c2[d0 % 3] = sm.c[12 + d0 % 3][lane];
  C.c2[d1 % 3] = sm.c[12 + d1 % 3][lane];
  C.c4[d0 % 3] = sm.c[15 + d0 % 3][lane];
  C.c4[d1 % 3] = sm.c[15 + d1 % 3][lane];
  C.w3r = sm.c[18][lane];
  C.w3i = sm.c[19][lane];
  const double om[4] = {fma(-K, C.c1[d0], K), fma(-K, C.c1[d1], K), fma(K, C.c1[d0], K), fma(K, C.c1[d1], K)};
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    double R[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) R[k] = sm.R[s][k][lane];
    const double p3 = R[3] * C.w3r, q3 = R[3] * C.w3i;
    double E[2], O[2];
    synth_dir(d0, R, p3, q3, C, E[0], O[0]);
    synth_dir(d1, R, p3, q3, C, E[1], O[1]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const double fe = i < 2 ? E[i & 1] + O[i & 1] : E[i & 1] - O[i & 1];
      v[i][s] = fma(om[i], fe - v[i][s], v[i][s]);
      ghost(2 * W + (i & 1) + 6 * (i >> 1), s, v[i][s], fe);
    }
  }
}

// Store of a warp's directions at cell offset c.
template <int W>
__device__ __forceinline__ void split_store(double* __restrict__ fout, long long c, const double v[4][6]) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int s = 0; s < 6; s += 2)
      *reinterpret_cast<Pair<double>*>(fout + c + plane_off(6 * (2 * W + (i & 1) + 6 * (i >> 1)) + s)) =
          Pair<double>{v[i][s], v[i][s + 1]};
}

// Equilibrium at (theta, g, u) at a warp's directions, stored at cell offset c.
template <int EDF, int W>
__device__ __noinline__ void split_feq(const DomDev& D, double* __restrict__ fout, long long c, double theta, double n,
                                       double ux, double uy, double gam, unsigned* st) {
  double z, g[6];
  *st |= solve_z_from_n_theta<EDF, false>(n, theta, z, g);
  const double t2 = theta * theta;
  double ym[21], v[4][6];
  eq_moments<EDF>(g, theta, fma(ux, ux, uy * uy), gam, (2.0 * PI) * (t2 * g[1]), (4.0 * PI) * (t2 * theta) * g[2], ym,
                  D.order - 2);
  const DirPow C = dir_powers(ux, uy);
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    double fe[12];
    feq_shell<EDF>(s, ym, C, fe, D.order - 2);
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i][s] = fe[2 * W + (i & 1) + 6 * (i >> 1)];
  }
  split_store<W>(fout, c, v);
}

// Halo cells of a cell, a warp's directions: as write_halo64.
template <int EDF, int W>
__device__ __forceinline__ void split_halo(const DomDev& D, int x, int y, double* __restrict__ fout,
                                           const double v[4][6], bool ok, double n, double ux, double uy, double gam,
                                           bool images, unsigned* st) {
  int hx[8], hy[8], wall[8];
  const int cnt = halo_targets(D, x, y, hx, hy, wall, images);
  for (int i = 0; i < cnt; ++i) {
    const long long h = cell_rel(D, hx[i], hy[i]);
    const int w = wall[i];
    if (w >= 0 && D.bc[w] == BC_VWALL) {
      if (!ok) split_feq<EDF, W>(D, fout, h, D.t_wall[w], D.n_wall, 0.0, 0.0, 1.0, st);
    } else if (w < 0 || !ok) {
      split_store<W>(fout, h, v);
    } else {
      split_feq<EDF, W>(D, fout, h, D.t_wall[w], n, ux, uy, gam, st);
    }
  }
}

template <int EDF, bool kVw, int W>
__device__ __forceinline__ void split_cell(const StepArgs& a, const DomDev& D, int x, int y, bool in, int serial,
                                           SplitSm& sm, int lane) {
  const double* __restrict__ fin = static_cast<const double*>(a.fin) + D.off;
  double* __restrict__ fout = static_cast<double*>(a.fout) + D.off;
  const long long c = cell_rel(D, x, y);
  double v[4][6];
  split_pull<EDF, W>(fin, c, neighbours(D, x, y), v, sm, lane);
  split_sync();
  CellState S;
  unsigned st = 0;
  if (serial == W) {
    double e[6], o[6], N[3], T[6];
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      e[d] = sm.eo[d][0][lane];
      o[d] = sm.eo[d][1][lane];
    }
    const Harm ha = harmonics_eo(e, o, false);
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      e[d] = sm.eo[d][2][lane];
      o[d] = sm.eo[d][3][lane];
    }
    moments_of(ha, harmonics_eo(e, o, true), N, T);
    st = cell_frame(N, T, S);
    sm.st[lane] = st;
    if (!(st & ST_NONPHYSICAL)) {
      sm.cell[0][lane] = S.ux;
      sm.cell[1][lane] = S.uy;
      sm.cell[2][lane] = S.gamma;
      sm.cell[3][lane] = S.n;
      sm.cell[4][lane] = S.eps;
    }
  }
  split_sync();
  const bool ok = !(sm.st[lane] & ST_NONPHYSICAL);
  double K = 0.0, ux = 0.0, uy = 0.0, gam = 1.0;
  if (ok) {
    ux = sm.cell[0][lane];
    uy = sm.cell[1][lane];
    gam = sm.cell[2][lane];
  }
  if (ok && serial == W) {
    st |= cell_theta<EDF, false>(S);
    sm.cell[5][lane] = S.theta;
    sm.clamped[lane] = st & ST_CLAMPED;
  }
  if (D.eta_s > 0.0) split_sync();  // every warp's rate needs theta (uniform per domain)
  if (ok) {
    double itau;
    collision_frame(D, D.eta_s > 0.0 ? sm.cell[5][lane] : 1.0, ux, uy, gam, itau);
    K = gam * itau;
    if (serial == W) {
      const double eps_eq = (st & ST_CLAMPED) ? 4.0 * PI * S.theta * S.theta * S.theta * S.g[2] : S.eps;
      double ym[21];
      eq_moments<EDF>(S.g, S.theta, fma(ux, ux, uy * uy), gam, S.n, eps_eq, ym, D.order - 2);
#pragma unroll
      for (int i = 0; i < 21; ++i) sm.y[i][lane] = ym[i];
    } else if ((serial + 1) % kSplitWarps == W) {
      const DirPow C = dir_powers(ux, uy);
#pragma unroll
      for (int d = 0; d < 6; ++d) {
        sm.c[d][lane] = C.c1[d];
        sm.c[6 + d][lane] = C.c5[d];
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        sm.c[12 + d][lane] = C.c2[d];
        sm.c[15 + d][lane] = C.c4[d];
      }
      sm.c[18][lane] = C.w3r;
      sm.c[19][lane] = C.w3i;
    }
  }
  split_sync();
  if (ok) {
    double ym[21], R[6];
#pragma unroll
    for (int i = 0; i < 21; ++i) ym[i] = sm.y[i][lane];
#pragma unroll
    for (int s = 2 * W; s < 2 * W + 2; ++s) {
      shell_project<EDF>(s, ym, R, D.order - 2);
#pragma unroll
      for (int k = 0; k < 6; ++k) sm.R[s][k][lane] = R[k];
    }
  }
  split_sync();
  const bool vw = kVw && in && ok && touches_vwall(D, x, y);
  VwallGhosts G;
  if (kVw && __any_sync(0xffffffffu, vw)) {
    G.cnt = 0;
    if (vw) vwall_setup<EDF>(D, x, y, a.images != 0, &G, &st);
    if (ok)
      split_relax<EDF, W>(K, v, sm, lane, [&](int d, int s, double r, double fe) {
        if (!vw) return;
        const double g = vwall_shell<EDF>(G, s, D.order - 2) + (r - fe);
        for (int i = 0; i < G.cnt; ++i) fout[G.at[i] + plane_off(6 * d + s)] = g;
      });
  } else if (ok) {
    split_relax<EDF, W>(K, v, sm, lane, [](int, int, double, double) {});
  }
  if (in) {
    split_store<W>(fout, c, v);
    if (EDF == EDF_BE && vw && sm.clamped[lane])
      vwall_clamped<false>(D, &G, sm.cell[5][lane], sm.cell[3][lane], sm.cell[4][lane], ux, uy, gam, fout + c,
                           0xc3u << (2 * W), fout);
    const bool edge = x == 0 || x == D.nx - 1 || y == 0 || y == D.ny - 1;
    if (edge && (a.images || a.halo)) {
      double n = 0.0, hx = 0.0, hy = 0.0, hg = 1.0;
      if (ok) {
        n = sm.cell[3][lane];
        hx = sm.cell[0][lane];
        hy = sm.cell[1][lane];
        hg = sm.cell[2][lane];
      }
      split_halo<EDF, W>(D, x, y, fout, v, ok, n, hx, hy, hg, a.images != 0, &st);
    }
    if (st) atomicOr(a.status, st);
  }
}

template <int EDF, bool kVw>
__global__ void __launch_bounds__(32 * kSplitWarps, 2) k_step_f64_split(StepArgs a) {
  __shared__ SplitSm sm;
  const int lane = threadIdx.x, u = blockIdx.x;
  const Tile tl = a.tiles[u / kTileH];
  const DomDev& D = a.doms[tl.dom];
  int x, y;
  const bool in = tile_cell(tl, lane, u % kTileH, x, y) && x < D.nx && y < D.ny;
  const unsigned some = __ballot_sync(0xffffffffu, in);
  if (!some) return;  // the same in the three warps
  // lanes without a cell follow a lane that has one and store nothing
  const int src = in ? lane : __ffs(some) - 1;
  x = __shfl_sync(0xffffffffu, x, src);
  y = __shfl_sync(0xffffffffu, y, src);
  const int serial = u % kSplitWarps;
  if (threadIdx.y == 0) split_cell<EDF, kVw, 0>(a, D, x, y, in, serial, sm, lane);
  else if (threadIdx.y == 1) split_cell<EDF, kVw, 1>(a, D, x, y, in, serial, sm, lane);
  else split_cell<EDF, kVw, 2>(a, D, x, y, in, serial, sm, lane);
}

template <int EDF>
static cudaError_t prepare_t() {
  cudaError_t e = cudaFuncSetAttribute(k_step_f64<EDF, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem64);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_step_f64<EDF, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem64);
  if (e != cudaSuccess) return e;
  return prepare_common_t<StoreF64, EDF>();
}

// Opt the kernels into 72 KB of dynamic shared memory (once per process).
cudaError_t prepare_f64() {
  cudaError_t e;
  if ((e = prepare_t<EDF_MJ>())) return e;
  if ((e = prepare_t<EDF_FD>())) return e;
  return prepare_t<EDF_BE>();
}

// Most tiles of a launch that takes the split step (unless a grid is asked for): 4 blocks of
// it per tile, two on each of 152 SMs. Measured, plain / split, us a step (MJ): 32^2 47.4 /
// 21.5, 64^2 47.4 / 21.8, 96^2 (72 tiles) 47.4 / 27.5, 112^2 (98) 47.4 / 50.7, 256^2 164 / 171.
constexpr int kSplitTiles = 76;

template <int EDF, bool kVw>
static void launch_step_t(const StepArgs& a, int grid, cudaStream_t s) {
  if (grid == 0 && a.ntiles <= kSplitTiles)
    k_step_f64_split<EDF, kVw><<<a.ntiles * kTileH, dim3(32, kSplitWarps), 0, s>>>(a);
  else
    k_step_f64<EDF, kVw><<<grid > 0 ? grid : a.ntiles, dim3(kTileW, kTileH), kSmem64, s>>>(a);
}

cudaError_t launch_step_f64(int edf, const StepArgs& a, int grid, cudaStream_t s) {
  const bool vw = a.halo >= 3;
  switch (edf) {
    case EDF_MJ: vw ? launch_step_t<EDF_MJ, true>(a, grid, s) : launch_step_t<EDF_MJ, false>(a, grid, s); break;
    case EDF_FD: vw ? launch_step_t<EDF_FD, true>(a, grid, s) : launch_step_t<EDF_FD, false>(a, grid, s); break;
    default: vw ? launch_step_t<EDF_BE, true>(a, grid, s) : launch_step_t<EDF_BE, false>(a, grid, s); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_init_f64(int edf, const InitArgs& a, int nx, int ny, cudaStream_t s) {
  return launch_init_t<StoreF64>(edf, a, nx, ny, s);
}

cudaError_t launch_fields_f64(int edf, const FieldsArgs& a, int nx, int ny, cudaStream_t s) {
  return launch_fields_t<StoreF64>(edf, a, nx, ny, s);
}

cudaError_t launch_copy_f64(const CopyArgs& a, cudaStream_t s) { return launch_copy_t<StoreF64>(a, s); }

}  // namespace rlbm
