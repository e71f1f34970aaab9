// Colour-gradient repulsion force (Sec. 2.3, Eqs. repForce, potential, normal1, normal2).
//
//   F_rep(x) = Pi psi_rep(rho^N(x)) sum_{i>=1} H(-(n.c_i)(n'_i.c_i)) [(n.c_i) n + (n'_i.c_i) n'_i] / |c_i|
//
// with n the unit colour gradient at x and n'_i the one at x + c_i.  The force needs the
// colour gradient one node away, i.e. rho^N two nodes away, so it is computed before each
// step that has it enabled:
//   colour_kernel   : rho^N(x) from the stored populations (the same density bookkeeping as
//                     the step kernel);
//   rep_force_kernel: n(x) = grad rho^N / |grad rho^N| (zero vector where |grad rho^N| <= eps,
//                     which then contributes nothing), gradient by the isotropic stencil,
//                     and F_rep, of which the step reads its own node's value.
// Readings: psi_rep = (1 - |rho^N|)^chi (or the printed (1 + |rho^N|)^chi), H(0) = 0,
// direction 0 skipped, a wall neighbour contributes nothing.
#pragma once

#include <cstdint>

#include "lbm_lattice.cuh"

namespace lbm {

template <class T>
__device__ __forceinline__ T fpow(T b, T e);
template <>
__device__ __forceinline__ float fpow<float>(float b, float e) { return e == 2.0f ? b * b : powf(b, e); }
template <>
__device__ __forceinline__ double fpow<double>(double b, double e) { return e == 2.0 ? b * b : pow(b, e); }

struct RepParams {
  int nx, ny, nz;
  long long n;
  int color_norm, psi_kind;
  double inv_rho_r0, inv_rho_b0, grad_eps, pi, chi;
};

__device__ __forceinline__ long long wrap_index(int x, int y, int z, int nx, int ny, int nz) {
  x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
  y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
  z = z < 0 ? z + nz : (z >= nz ? z - nz : z);
  return x + (long long)nx * (y + (long long)ny * z);
}

// Tile of rep_force_kernel: 32 x 8 nodes, the planes of normals with one node around it, those
// of rho^N with two.
constexpr int kRepTX = 32, kRepTY = 8, kRepThreads = 128;

// F_rep of every node from rho^N into rep [3][N].  A block marches a tile along z with four
// planes of rho^N and three of normals in shared memory (2D: one plane), so that neither the
// normals nor their 54 gathered neighbours touch global memory.  256^3: normals to global
// memory and gathered by their readers took 188 us and more than 600 of the step's 1560; this
// kernel takes 208.  Instruction issue bounds it; a warp without a normal skips the sum.  chunk: planes per block.
template <class L, class T, bool WALLS>
__global__ void __launch_bounds__(kRepThreads) rep_force_kernel(const T* __restrict__ colour,
                                                                const uint8_t* __restrict__ solid, T* __restrict__ rep,
                                                                int chunk, RepParams a) {
  constexpr int CX = kRepTX + 4, CY = kRepTY + 4, NC = CX * CY;
  constexpr int MX = kRepTX + 2, MY = kRepTY + 2, NM = MX * MY;
  constexpr int H = L::D == 3 ? 1 : 0;  // halo planes of the normals
  __shared__ T col[4][NC];
  __shared__ T nrm[3][3][NM];
  __shared__ uint8_t wall[4][WALLS ? NC : 1];
  const int ncx = (a.nx + kRepTX - 1) / kRepTX, ncy = (a.ny + kRepTY - 1) / kRepTY;
  const int x0 = int(blockIdx.x % ncx) * kRepTX, y0 = int(blockIdx.x / ncx % ncy) * kRepTY;
  const int z0 = int(blockIdx.x / ncx / ncy) * chunk, z1 = min(z0 + chunk, a.nz);
  const int tid = threadIdx.x;
  auto cslot = [](int z) { return (z + 4) & 3; };
  auto mslot = [](int z) { return (z + 3) % 3; };
  // this thread's elements of a staged plane (their place in a plane of the lattice does not
  // change along z)
  constexpr int EL = (NC + kRepThreads - 1) / kRepThreads;
  long long off[EL];
#pragma unroll
  for (int v = 0; v < EL; v++) {
    const int e = tid + v * kRepThreads;
    const int X = (x0 + e % CX - 2 + 2 * a.nx) % a.nx, Y = (y0 + e / CX - 2 + 2 * a.ny) % a.ny;
    off[v] = X + (long long)a.nx * Y;
  }
  auto stage = [&](int z) {  // rho^N of plane z >= -2, of its periodic image outside the lattice
    const int zw = z < 0 || z >= a.nz ? ((z % a.nz) + a.nz) % a.nz : z, s = cslot(z);
    const long long plane = (long long)a.nx * a.ny * zw;
#pragma unroll
    for (int v = 0; v < EL; v++) {
      const int e = tid + v * kRepThreads;
      if (e >= NC) break;
      col[s][e] = colour[plane + off[v]];
      if constexpr (WALLS) wall[s][e] = solid[plane + off[v]];
    }
  };
  auto normals = [&](int z) {
    const int s0 = cslot(z), sp = cslot(z + 1), sm = cslot(z + 3);
#pragma unroll
    for (int v = 0; v < (NM + kRepThreads - 1) / kRepThreads; v++) {
      const int e = tid + v * kRepThreads;
      if (e >= NM) break;
      const int e0 = (e / MX + 1) * CX + e % MX + 1;
      auto at = [&](int dx, int dy, int dz) -> T {
        const int s = dz == 0 ? s0 : dz > 0 ? sp : sm, c = e0 + dy * CX + dx;
        if (WALLS && wall[s][c]) return col[s0][e0];
        return col[s][c];
      };
      T g[3] = {T(0), T(0), T(0)};
#pragma unroll
      for (int q = 0; q < L::NP; q++) {
        const int cx = L::pcx(q), cy = L::pcy(q), cz = L::pcz(q);
        const T v = T(3.0 * L::w(L::pgrp(q))) * (at(cx, cy, cz) - at(-cx, -cy, -cz));
        if (cx) g[0] += T(cx) * v;
        if (cy) g[1] += T(cy) * v;
        if (cz) g[2] += T(cz) * v;
      }
      const T gn = sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
      if (gn > T(a.grad_eps) && !(WALLS && wall[s0][e0])) {
        for (int t = 0; t < 3; t++) g[t] = g[t] / gn;
      } else {
        g[0] = g[1] = g[2] = T(0);
      }
#pragma unroll
      for (int t = 0; t < 3; t++) nrm[mslot(z)][t][e] = g[t];
    }
  };
  if constexpr (H == 1) {
    for (int z = z0 - 2; z <= z0 + 1; z++) stage(z);
    __syncthreads();
    normals(z0 - 1);
    normals(z0);
    __syncthreads();
  }
  for (int z = z0; z < z1; z++) {
    // takes the slot of plane z - 2, which the normals of plane z - 1 read last (two barriers
    // ago; F_rep of plane z - 1 reads the planes z - 1 only)
    stage(z + 2 * H);
    __syncthreads();
    normals(z + H);
    __syncthreads();
    const int ms[3] = {mslot(z + 2), mslot(z), mslot(z + 1)};  // planes z - 1, z, z + 1
#pragma unroll
    for (int e = tid; e < kRepTX * kRepTY; e += kRepThreads) {
      const int x = x0 + e % kRepTX, y = y0 + e / kRepTX;
      if (x >= a.nx || y >= a.ny) continue;
      const int e0 = (e / kRepTX + 1) * MX + e % kRepTX + 1;
      const T n0 = nrm[ms[1]][0][e0], n1 = nrm[ms[1]][1][e0], n2 = nrm[ms[1]][2][e0];
      T F[3] = {T(0), T(0), T(0)};
      if (n0 != T(0) || n1 != T(0) || n2 != T(0)) {  // a normal at x; none on a wall
        T acc[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int i = 1; i < L::Q; i++) {
          const int s = ms[cz<L>(i) + 1], c = e0 + cy<L>(i) * MX + cx<L>(i);
          const T p0 = nrm[s][0][c], p1 = nrm[s][1][c], p2 = nrm[s][2][c];
          const T nc = cx<L>(i) * n0 + cy<L>(i) * n1 + cz<L>(i) * n2;
          const T pc = cx<L>(i) * p0 + cy<L>(i) * p1 + cz<L>(i) * p2;
          if (-(nc * pc) > T(0)) {  // H(0) = 0; an undefined neighbour normal gives pc = 0
            const T il = grp<L>(i) == 1 ? T(1) : T(0.70710678118654752440);
            acc[0] += (nc * n0 + pc * p0) * il;
            acc[1] += (nc * n1 + pc * p1) * il;
            acc[2] += (nc * n2 + pc * p2) * il;
          }
        }
        const T c = col[cslot(z)][(e / kRepTX + 2) * CX + e % kRepTX + 2];
        const T base = a.psi_kind ? T(1) + fabs(c) : T(1) - fabs(c);
        // outward (repulsive, Sec. 2.3): the printed sum points toward the rho^N extremum
        const T s = -T(a.pi) * fpow<T>(base, T(a.chi));
        for (int t = 0; t < 3; t++) F[t] = s * acc[t];
      }
      const long long n = x + (long long)a.nx * (y + (long long)a.ny * z);
      for (int t = 0; t < 3; t++) rep[t * a.n + n] = F[t];
    }
  }
}

}  // namespace lbm
