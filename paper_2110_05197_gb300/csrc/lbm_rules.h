// Which lattices the pair kernel (lbm_step_pair.cuh) steps: host code without CUDA.
#pragma once

#include "../../include/lbm.h"

namespace lbm {

constexpr int kPairTX = 32;          // columns of a tile
constexpr int kPairMaxCluster = 16;  // tiles of a row, one cluster (the non-portable limit): nx <= 512

// Rows of the pair kernel's lattices: a tensor map needs rows of a multiple of 16 bytes, i.e. 8
// elements of the narrowest storage.
inline int padded_pitch(int nx) { return (nx + 7) / 8 * 8; }

// Whether the pair kernel takes a lattice.  Kind: D3Q19, 32- or 16-bit storage, two buffers, at most
// kPairMaxCluster tiles of 32 columns.  Among those,
// aligned lattices always.  With partial tiles the generic
// kernel's tuned tiles are as fast or faster for narrow lattices (a warp's lanes are columns; us a
// step, generic against pair: CG FP32 9 x 200 x 100 36 : 55, 12 x 100 x 100 30 : 33) and, where a
// plane costs little or storage is 16-bit, for small cross-sections, unless they are long (SC FP32
// 24 x 24 x 24 5.5 : 8.0, x 600 23 : 18; 48 x 48 x 48 11.0 : 12.0, x 150 24 : 18; 75 x 77 x 71 29 :
// 22; CG FP16 40 x 40 x 40 14 : 22, 48 x 48 x 48 16 : 20, x 150 41 : 34); FP32 CG and two-component SC
// without walls gain or are level at every other cross-section.  The rule does not look at nz:
// z-slabs of a lattice (decomp.py) must run the kernel that the whole lattice runs.
// Nor are rows padded where that alone would take the arrays beyond 32-bit indices: the batched
// launch and the generic kernel's 32-bit form take such lattices as long as K Q N < 2^31.
// The pair kernel's own indices reach over one array in 31 bits, and with walls over two.
inline bool pair_takes(const lbm_params& p, bool walls) {
  if (p.lattice != LBM_D3Q19 || p.precision == LBM_FP64 || p.streaming != LBM_STREAM_AB ||
      p.model == LBM_MODEL_SC_MR || p.nx > kPairTX * kPairMaxCluster)
    return false;
  const long long rows = (long long)p.ny * p.nz, all = (p.model == LBM_MODEL_SC_MP ? 19 : 38) * rows, limit = 1LL << 31;
  if (all * p.nx < limit && all * padded_pitch(p.nx) >= limit) return false;
  if (rows * padded_pitch(p.nx) >= (walls ? limit / 2 : limit)) return false;
  if (p.nx % kPairTX == 0 && p.ny % 8 == 0) return true;
  const bool heavy = p.precision == LBM_FP32 && p.model != LBM_MODEL_SC_MP && !walls;
  return p.nx >= 12 && (heavy || (long long)p.nx * p.ny >= (p.precision == LBM_FP32 ? 1500 : 2000));
}

// Whether a lattice is stored for the pair kernel: it takes it with or without walls, which are not
// known when the workspace is laid out.
inline bool pair_lattice(const lbm_params& p) { return pair_takes(p, false) || pair_takes(p, true); }

// Whether the pair kernel steps it.  (The repulsion force between walls runs on the generic kernel.)
inline bool pair_steps(const lbm_params& p, bool walls) {
  return pair_takes(p, walls) && !(walls && p.model == LBM_MODEL_CG && p.rep_pi != 0.0);
}

// Row pitch of the stored arrays; lattices of the other kernels are stored densely.
inline int row_pitch(const lbm_params& p) { return pair_lattice(p) ? padded_pitch(p.nx) : p.nx; }

}  // namespace lbm
