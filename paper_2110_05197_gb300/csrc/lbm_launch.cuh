// Launch helper for the fused step kernel (one instantiation per lattice, storage
// precision, model and wall variant).
#pragma once

#include <algorithm>

#include "lbm_internal.cuh"
#include "lbm_step_aa.cuh"
#include "lbm_step_pair.cuh"

namespace lbm {

// rho^N for the repulsion pre-pass, with the step's density bookkeeping; odd: the state
// is in the odd in-place layout
template <class L, class T, class S, class RT>
__global__ void colour_kernel(const S* __restrict__ f, const RT* __restrict__ r, T* __restrict__ colour,
                              RepParams a, int odd, int px, long long ns) {
  for (long long m = blockIdx.x * (long long)blockDim.x + threadIdx.x; m < a.n; m += (long long)gridDim.x * blockDim.x) {
    T rho[2];
    const long long st = stored_index(m, a.nx, px);
    for (int k = 0; k < 2; k++) {
      T g[L::Q];
#pragma unroll
      for (int i = 0; i < L::Q; i++)
        g[i] = ld_s<S, T>(f[odd ? aa_index_n<L>(k, i, m, a.nx, a.ny, a.nz, a.n, odd) : (k * L::Q + i) * ns + st]);
      rho[k] = comp_state<L, T, RT>(g, T(r[k * ns + st])).rho;
    }
    T s0 = rho[0], s1 = rho[1];
    if (a.color_norm) {
      s0 = s0 * T(a.inv_rho_r0);
      s1 = s1 * T(a.inv_rho_b0);
    }
    colour[m] = (s0 - s1) / (s0 + s1);
  }
}

// The same on two nodes a thread (FP32 arithmetic, dense layout of the two-buffer scheme):
// rows of `row` nodes, `pitch` apart, pairs of stored elements aligned.  256^3 FP16: 323 us
// one node at a time, 224 (206 us are its bytes).
template <class L, class S>
__global__ void __launch_bounds__(256) colour2_kernel(const S* __restrict__ f, const float* __restrict__ r,
                                                      float* __restrict__ colour, unsigned row, unsigned pitch,
                                                      unsigned rows, RepParams a, long long ns) {
  using U = typename std::conditional<sizeof(S) == 4, uint2, unsigned>::type;
  const unsigned per = (row + 1) / 2, total = per * rows;
  for (unsigned m = blockIdx.x * blockDim.x + threadIdx.x; m < total; m += gridDim.x * blockDim.x) {
    const unsigned y = m / per, x = 2 * (m - y * per), st = y * pitch + x;
    F2 rho[2];
#pragma unroll
    for (int k = 0; k < 2; k++) {
      F2 g[L::Q];
#pragma unroll
      for (int i = 0; i < L::Q; i++) {
        S e[2];
        *reinterpret_cast<U*>(e) = *reinterpret_cast<const U*>(f + (k * L::Q + i) * ns + st);
        g[i].set(0, ld_s<S, float>(e[0]));
        g[i].set(1, ld_s<S, float>(e[1]));
      }
      rho[k] = comp_state2<L>(g, F2(*reinterpret_cast<const float2*>(r + k * ns + st))).q;
    }
#pragma unroll
    for (int j = 0; j < 2; j++) {
      float s0 = rho[0][j], s1 = rho[1][j];
      if (a.color_norm) {
        s0 = s0 * float(a.inv_rho_r0);
        s1 = s1 * float(a.inv_rho_b0);
      }
      if (x + j < row) colour[y * row + x + j] = (s0 - s1) / (s0 + s1);
    }
  }
}

inline RepParams rep_params(const lbm_ctx* c) {
  RepParams a{};
  a.nx = c->p.nx;
  a.ny = c->p.ny;
  a.nz = c->p.nz;
  a.n = c->N;
  a.color_norm = c->p.color_norm;
  a.psi_kind = c->p.rep_psi_kind;
  a.inv_rho_r0 = 1.0 / c->p.rho_r0;
  a.inv_rho_b0 = 1.0 / c->p.rho_b0;
  a.grad_eps = c->p.grad_eps;
  a.pi = c->p.rep_pi;
  a.chi = c->p.rep_chi;
  return a;
}

// Repulsion force of the current state into c->rep_f.
template <class L, class T, class S, class RT>
cudaError_t launch_rep_prepass_t(lbm_ctx* c, int buf) {
  const RepParams a = rep_params(c);
  const int grid = (int)std::min<long long>((c->N + 255) / 256, 8192);
  const S* f = static_cast<const S*>(c->f[buf]);
  const RT* r = static_cast<const RT*>(c->r[buf]);
  T* colour = static_cast<T*>(c->colour);
  bool two = false;
  if constexpr (sizeof(T) == 4) {
    const bool dense = c->px == c->p.nx;
    const long long row = dense ? c->N : c->p.nx, pitch = dense ? c->N : c->px, rows = c->N / row;
    two = !c->aa && pitch % 2 == 0 && c->NS % 2 == 0 && c->NS < (1LL << 32);
    if (two)
      colour2_kernel<L, S><<<(grid + 1) / 2, 256, 0, c->stream>>>(f, r, colour, (unsigned)row, (unsigned)pitch,
                                                                  (unsigned)rows, a, c->NS);
  }
  if (!two)
    colour_kernel<L, T, S, RT><<<grid, 256, 0, c->stream>>>(f, r, colour, a, c->aa ? (buf & 1) : 0, c->px, c->NS);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // planes per block: long runs share their halo planes, short ones keep the SMs busy
  const long long tiles = (long long)((c->p.nx + kRepTX - 1) / kRepTX) * ((c->p.ny + kRepTY - 1) / kRepTY);
  int chunk = 16;
  while (chunk > 1 && tiles * ((c->p.nz + chunk - 1) / chunk) < 8LL * c->nsm) chunk /= 2;
  const long long blocks = tiles * ((c->p.nz + chunk - 1) / chunk);
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  auto kern = c->has_walls ? rep_force_kernel<L, T, true> : rep_force_kernel<L, T, false>;
  kern<<<(int)blocks, kRepThreads, 0, c->stream>>>(colour, c->solid, static_cast<T*>(c->rep_f), chunk, a);
  c->launches += 2;
  return cudaGetLastError();
}

// Launch of a kernel that begins with await_previous_step().
template <class... P, class... A>
cudaError_t launch_dependent(void (*kern)(P...), int grid, dim3 block, size_t smem, cudaStream_t stream, A... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// Persistent grid: `resident` blocks (or clusters) loop over the units.  The z-chunk count
// trades the halo planes every unit re-reads (2 per unit) against the idle share of the
// last round of units; chunks stay at least 8 planes long.
template <class T>
void persistent_plan(StepParams<T>& sp, int resident) {
  resident = std::max(resident, 1);
  const int max_chunks = std::max(1, sp.nz / 8);
  double best = -1.0;
  int best_n = 1;
  for (int n = 1; n <= max_chunks; n++) {
    const long long units = (long long)sp.ncol * n;
    const long long rounds = (units + resident - 1) / resident;
    const double busy = double(units) / double(rounds * resident);  // share of block-rounds with a unit
    const double planes = double(sp.nz) / n;
    const double score = busy / (1.0 + 1.0 / planes);  // halo planes cost about half a plane each
    if (score > best + 1e-9) {
      best = score;
      best_n = n;
    }
  }
  sp.nchunks = best_n;
  sp.nblk = (int)std::min<long long>((long long)sp.ncol * best_n, resident);
}

template <class L, class T, class S, class RT, int MODEL, bool WALLS>
cudaError_t launch_tma_t(lbm_ctx* c) {
  constexpr int TX = kTmaTX, TY = kTmaTY;
  constexpr size_t smem = tma_smem_bytes<L, T, S, RT, MODEL, WALLS, TX, TY>();
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(step_kernel_tma<L, T, S, RT, MODEL, WALLS, TX, TY>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  dim3 block(kTmaThreads, 1, 1);
  StepParams<T> sp = make_step_params<T>(c);
  if (c->tz == 0) persistent_plan(sp, c->nsm);  // one block per SM (shared memory)
  dim3 grid(sp.nblk, 1, 1);
  const S* fin = static_cast<const S*>(c->f[c->cur]);
  const RT* rin = static_cast<const RT*>(c->r[c->cur]);
  S* fout = static_cast<S*>(c->f[c->cur ^ 1]);
  RT* rout = static_cast<RT*>(c->r[c->cur ^ 1]);
  step_kernel_tma<L, T, S, RT, MODEL, WALLS, TX, TY><<<grid, block, smem, c->stream>>>(
      c->tma[c->cur], fin, rin, fout, rout, c->solid, &c->diag->status, sp);
  return cudaGetLastError();
}

// Pair kernel (lbm_step_pair.cuh): clusters of nx / 32 blocks, each cluster one run of
// (tile row, plane) pairs; TY rows per tile, MB blocks per SM.
template <class L, class T, class S, class RT, int MODEL, int FORM, int TY, int MB, bool REP = false>
cudaError_t launch_pair_tile(lbm_ctx* c) {
  constexpr size_t smem = pair_smem_bytes<L, S, RT, MODEL, TY>(pair_raw<L, S, RT, MODEL, TY, MB>());
  auto kern = step_kernel_pair<L, T, S, RT, MODEL, FORM, TY, MB, REP>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  const int C = (c->p.nx + kPairTX - 1) / kPairTX;
  StepParams<T> sp = make_step_params<T>(c);
  sp.ncx = C;                         // blocks per cluster
  sp.ncol = (c->p.ny + TY - 1) / TY;  // tile rows
  cudaLaunchAttribute attr[2];
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(16 * TY, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = c->stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const void* fn = reinterpret_cast<const void*>(kern);
  if (c->occ_fn != fn || c->occ_tx != -C) {
    int ncl = 0;
    cfg.gridDim = dim3(C, 1, 1);
    // a part of a GPU may hold no cluster of this size (its SMs lie in groups of fewer)
    if (cudaOccupancyMaxActiveClusters(&ncl, kern, &cfg) != cudaSuccess || ncl < 1) {
      cudaGetLastError();
      c->no_clusters = true;
      return cudaErrorNotSupported;
    }
    c->occ_fn = fn;
    c->occ_tx = -C;
    c->occ_ty = 0;
    c->occ_blocks = ncl;
  }
  sp.nblk = (int)std::min<long long>(c->occ_blocks, (long long)sp.ncol * sp.nz);  // clusters
  // a grid of at most one block per SM leaves room for the next step's blocks beside its own: they
  // come before its last collision (32^3 CG FP32 9.3 -> 8.7 us)
  sp.admit_early = sp.nblk * C <= c->nsm;
  cfg.numAttrs = 2;  // the step follows the step before as a programmatic dependent launch
  cfg.gridDim = dim3(sp.nblk * C, 1, 1);
  OutArrays<S, RT, ModelTraits<MODEL>::K * L::Q, ModelTraits<MODEL>::K> out;
  for (int a = 0; a < c->K * c->Q; a++) out.f[a] = static_cast<S*>(c->f[c->cur ^ 1]) + a * c->NS;
  for (int k = 0; k < c->K; k++) out.r[k] = static_cast<RT*>(c->r[c->cur ^ 1]) + k * c->NS;
  return cudaLaunchKernelEx(&cfg, kern, c->tma[c->cur], out, static_cast<const unsigned long long*>(c->walls),
                            static_cast<const uint8_t*>(c->rows_walled), static_cast<const int*>(c->cuts),
                            static_cast<const T*>(c->rep_f), &c->diag->status, sp);
}

// Tile of the pair kernel.  CG keeps a plane's sums in registers (242 of them), two-component
// SC two sets: two blocks of 4 warps per SM.  SC multiphase in FP32 runs 16 warps per SM as
// two blocks of 16 rows, whose halo rows cost 12% of the staging instead of 25% with 8 rows
// (128^3: 68 us against 73), unless 16 rows do not divide ny or there are fewer such tiles
// than blocks to hold them (32^3: 10.4 us against 8.8); in 16-bit storage, whose plane
// buffers are half as large, as four blocks of 8 rows (57.6 against 59.8 us), of which three
// have the registers for walls.
template <class L, class T, class S, class RT, int MODEL, bool WALLS, bool REP>
cudaError_t launch_pair_t(lbm_ctx* c) {
  constexpr int MB = MODEL != kSCMP ? 2 : sizeof(S) == 4 || WALLS ? 3 : 4;
  if constexpr (REP) {
    static_assert(!WALLS, "the repulsion force between walls runs on the generic kernel");
    cudaError_t e = launch_rep_prepass_t<L, T, S, RT>(c, c->cur);
    if (e != cudaSuccess) return e;
    if (c->p.nx % kPairTX != 0 || c->p.ny % 8 != 0) return launch_pair_tile<L, T, S, RT, MODEL, kRagged, 8, MB, true>(c);
    return launch_pair_tile<L, T, S, RT, MODEL, kFull, 8, MB, true>(c);
  } else if constexpr (WALLS) {
    return launch_pair_tile<L, T, S, RT, MODEL, kWalls, 8, MB>(c);
  } else {
    if (c->p.nx % kPairTX != 0 || c->p.ny % 8 != 0) return launch_pair_tile<L, T, S, RT, MODEL, kRagged, 8, MB>(c);
    if constexpr (MODEL == kSCMP && sizeof(S) == 4)
      if (c->p.ny % 16 == 0 && c->N / (32 * 16) >= 2 * c->nsm)
        return launch_pair_tile<L, T, S, RT, MODEL, kFull, 16, 2>(c);
    return launch_pair_tile<L, T, S, RT, MODEL, kFull, 8, MB>(c);
  }
}

// Field-pass step (in-place streaming, or the multirange model): the field pass, then the
// step kernel, both over all nodes.
template <class L, class T, class S, class RT, int MODEL, bool WALLS, bool REP, class I>
cudaError_t launch_fp_i(lbm_ctx* c) {
  if constexpr (REP) {
    cudaError_t e = launch_rep_prepass_t<L, T, S, RT>(c, c->cur);
    if (e != cudaSuccess) return e;
  }
  const StepParams<T> sp = make_step_params<T>(c);
  const int odd = c->aa ? (c->cur & 1) : 0;
  const int mode = c->aa ? 1 + odd : 0;
  const S* fin = static_cast<const S*>(c->f[c->cur]);
  S* fout = static_cast<S*>(c->f[c->cur ^ 1]);  // == fin in place
  const RT* rin = static_cast<const RT*>(c->r[c->cur]);
  RT* rout = static_cast<RT*>(c->r[c->cur ^ 1]);
  T* fld = reinterpret_cast<T*>(c->stage);  // [NF + K][N] of the compute type, fits 6N doubles
  const long long blocks = (c->N + 255) / 256;
  const int grid = (int)std::min<long long>(blocks, (long long)c->nsm * 16);
  fp_fields_kernel<L, T, S, RT, MODEL><<<grid, 256, 0, c->stream>>>(fin, rin, fld, WALLS ? c->solid : nullptr,
                                                                   &c->diag->status, sp, odd);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  c->launches += 1;
  if constexpr (L::D == 3 && MODEL == kSCMR) {
    // belt-2 fields staged in shared memory (halo 2): 2.7x faster than gathering the 92
    // neighbours through L1; for the halo-1 models the L1 gathers measured as fast or
    // faster (in-place SC-MP 128^3: 142 vs 162 us), so they keep fp_step_kernel
    constexpr int H = 2;
    constexpr size_t smem = fpt_smem_bytes<T, MODEL, WALLS, H>();
    auto kern = fpt_step_kernel<L, T, S, RT, MODEL, WALLS, REP, H, I>;
    static int occ = 0;  // resident blocks per SM of this instantiation
    if (occ == 0) {
      if (smem > 48 * 1024) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
      }
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kFpTX * kFpTY, smem);
      if (e != cudaSuccess) return e;
      occ = std::max(occ, 1);
    }
    StepParams<T> tp = sp;
    tp.ncx = (c->p.nx + kFpTX - 1) / kFpTX;
    tp.ncol = tp.ncx * ((c->p.ny + kFpTY - 1) / kFpTY);
    persistent_plan(tp, c->nsm * occ);
    kern<<<tp.nblk, kFpTX * kFpTY, smem, c->stream>>>(fin, fout, rin, rout, fld, c->solid, &c->diag->status, tp,
                                                      static_cast<const T*>(c->rep_f), mode);
  } else {
    fp_step_kernel<L, T, S, RT, MODEL, WALLS, REP, I><<<grid, 256, 0, c->stream>>>(
        fin, fout, rin, rout, fld, c->solid, &c->diag->status, sp, static_cast<const T*>(c->rep_f), mode);
  }
  return cudaGetLastError();
}

// Field-pass step with 32-bit indices where every index fits (FP64 storage: 64-bit).
template <class L, class T, class S, class RT, int MODEL, bool WALLS, bool REP>
cudaError_t launch_fp_t(lbm_ctx* c) {
  if constexpr (sizeof(T) < 8) {
    if ((long long)c->K * c->Q * c->N < (1LL << 31)) return launch_fp_i<L, T, S, RT, MODEL, WALLS, REP, int>(c);
  }
  return launch_fp_i<L, T, S, RT, MODEL, WALLS, REP, long long>(c);
}

// Generic plane-marching step (step_kernel) with index type I.
template <class L, class T, class S, class RT, int MODEL, bool WALLS, bool REP, class I>
cudaError_t launch_generic_t(lbm_ctx* c) {
  const int tx = c->tx;
  int ty = c->ty, tz = c->tz;
  // A lattice with fewer tiles than SMs is cut into smaller ones: the time is that of the
  // fullest SM, whose tiles take a collision per node and a staging (about a quarter of one)
  // per node and halo node.  2D 128^2 CG FP64 (32 x 8 tiles on 64 SMs): 31.8 us, as 32 x 4
  // tiles on 128 19.5.
  const long long tiles_x = (c->p.nx + tx - 1) / tx;
  auto units = [&](int y, int z) {
    return tiles_x * ((c->p.ny + y - 1) / y) * (z > 0 ? (c->p.nz + z - 1) / z : 1);
  };
  if (tz > 0 && units(ty, tz) < c->nsm) {
    auto cost = [&](int y, int z) {
      const long long rounds = (units(y, z) + c->nsm - 1) / c->nsm;
      return double(rounds) * (double(tx) * y * z + 0.25 * (tx + 2) * (y + 2) * (L::D == 3 ? z + 2 : 1));
    };
    double best = cost(ty, tz);
    const int y0 = ty, z0 = tz;
    for (int z = z0; z >= 1; z /= 2)
      for (int y = y0; y >= 1 && tx * y >= 64; y /= 2)
        if (cost(y, z) < best) {
          best = cost(y, z);
          ty = y;
          tz = z;
        }
  }
  const size_t smem = step_smem_bytes<L, T, MODEL, WALLS>(tx, ty);
  static size_t smem_set = 0;  // largest dynamic shared memory opted in so far
  if (smem > 48 * 1024 && smem > smem_set) {
    cudaError_t e = cudaFuncSetAttribute(step_kernel<L, T, S, RT, MODEL, WALLS, REP, I>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    smem_set = smem;
  }
  dim3 block(tx, ty, 1);
  StepParams<T> sp = make_step_params<T>(c);
  sp.ncol = (int)units(ty, 0);
  sp.nchunks = tz > 0 ? (c->p.nz + tz - 1) / tz : 1;
  sp.nblk = sp.ncol * sp.nchunks;
  if (tz == 0) {
    const void* fn = reinterpret_cast<const void*>(step_kernel<L, T, S, RT, MODEL, WALLS, REP, I>);
    if (c->occ_fn != fn || c->occ_tx != tx || c->occ_ty != ty) {
      int nb = 0;
      cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, step_kernel<L, T, S, RT, MODEL, WALLS, REP, I>,
                                                                    tx * ty, smem);
      if (e != cudaSuccess) return e;
      c->occ_fn = fn;
      c->occ_tx = tx;
      c->occ_ty = ty;
      c->occ_blocks = nb > 0 ? nb : 1;
    }
    persistent_plan(sp, c->nsm * c->occ_blocks);
  }
  const S* fin = static_cast<const S*>(c->f[c->cur]);
  S* fout = static_cast<S*>(c->f[c->cur ^ 1]);
  const RT* rin = static_cast<const RT*>(c->r[c->cur]);
  RT* rout = static_cast<RT*>(c->r[c->cur ^ 1]);
  return launch_dependent(step_kernel<L, T, S, RT, MODEL, WALLS, REP, I>, sp.nblk, block, smem, c->stream, fin, fout, rin,
                          rout, c->solid, &c->diag->status, sp, static_cast<const T*>(c->rep_f));
}

template <class L, class T, class S, class RT, int MODEL, bool WALLS, bool REP>
cudaError_t launch_step_t(lbm_ctx* c) {
  if constexpr (MODEL == kSCMR) {
    return launch_fp_t<L, T, S, RT, MODEL, WALLS, REP>(c);
  } else {
  if (c->aa) return launch_fp_t<L, T, S, RT, MODEL, WALLS, REP>(c);
  // the pair kernel, whatever the tiling
  if constexpr (L::D == 3 && sizeof(T) == 4 && !(REP && WALLS))
    if (c->tma_ok && !c->no_clusters && pair_steps(c->p, WALLS)) {
      const cudaError_t e = launch_pair_t<L, T, S, RT, MODEL, WALLS, REP>(c);
      if (!c->no_clusters) return e;  // else, from now on, the kernels below
    }
  if (c->tx * c->ty > 256) {
    // the 512-node tilings run as 32 x 8 persistent tiles
    const int tx = c->tx, ty = c->ty, tz = c->tz;
    c->tx = kTmaTX;
    c->ty = kTmaTY;
    c->tz = 0;
    const cudaError_t e = launch_step_t<L, T, S, RT, MODEL, WALLS, REP>(c);
    c->tx = tx;
    c->ty = ty;
    c->tz = tz;
    return e;
  }
  if constexpr (L::D == 3 && sizeof(T) == 4 && !REP)
    if (c->tma_ok && c->px == c->p.nx && c->p.nx % kTmaTX == 0 && c->p.ny % kTmaTY == 0 && c->tx == kTmaTX &&
        c->ty == kTmaTY)
      return launch_tma_t<L, T, S, RT, MODEL, WALLS>(c);
  if constexpr (REP) {
    cudaError_t e = launch_rep_prepass_t<L, T, S, RT>(c, c->cur);
    if (e != cudaSuccess) return e;
  }
  // 32-bit node and array indices where every index fits (FP64 storage keeps 64-bit ones:
  // its step is bound by the FP64 rate, not by index arithmetic)
  if constexpr (sizeof(T) < 8) {
    if ((long long)c->K * c->Q * c->NS < (1LL << 31)) return launch_generic_t<L, T, S, RT, MODEL, WALLS, REP, int>(c);
  }
  return launch_generic_t<L, T, S, RT, MODEL, WALLS, REP, long long>(c);
  }
}

template <class L, class T, class S, class RT, int MODEL>
cudaError_t dispatch_walls(lbm_ctx* c) {
  const bool w = c->has_walls;
  if constexpr (MODEL == kCG) {
    if (c->rep) return w ? launch_step_t<L, T, S, RT, MODEL, true, true>(c) : launch_step_t<L, T, S, RT, MODEL, false, true>(c);
  }
  return w ? launch_step_t<L, T, S, RT, MODEL, true, false>(c) : launch_step_t<L, T, S, RT, MODEL, false, false>(c);
}

template <class T, class S, class RT, int MODEL>
cudaError_t dispatch_lattice(lbm_ctx* c) {
  if constexpr (MODEL == kSCMR) {
    return dispatch_walls<D3Q19, T, S, RT, MODEL>(c);  // D3Q19 only (lbm_create checks)
  } else {
    if (c->p.lattice == LBM_D3Q19) return dispatch_walls<D3Q19, T, S, RT, MODEL>(c);
    return dispatch_walls<D2Q9, T, S, RT, MODEL>(c);
  }
}

template <class T, class S, class RT>
cudaError_t dispatch_model(lbm_ctx* c) {
  if (c->p.model == LBM_MODEL_CG) return dispatch_lattice<T, S, RT, kCG>(c);
  if (c->p.model == LBM_MODEL_SC_MP) return dispatch_lattice<T, S, RT, kSCMP>(c);
  if (c->p.model == LBM_MODEL_SC_MR) return dispatch_lattice<T, S, RT, kSCMR>(c);
  return dispatch_lattice<T, S, RT, kSC2C>(c);
}


}  // namespace lbm
