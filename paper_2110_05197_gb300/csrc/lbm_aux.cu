// Auxiliary kernels: equilibrium initialisation, checkpoint import/export of populations,
// and the FP64 moment / diagnostics reductions (mass, momentum, E_kin, max|u|, blow-up).
//
// Populations are stored as deviations g^k_i = f^k_i - phi^k_i r_k from the rest-state
// equilibrium of a per-node reference density r_k (see lbm_step.cuh); every kernel here
// reconstructs f in FP64 as g + phi r.
#include <cmath>
#include <type_traits>

#include "lbm_launch.cuh"

namespace lbm {

namespace {

__device__ __forceinline__ double to_d(double v) { return v; }
__device__ __forceinline__ double to_d(float v) { return (double)v; }
__device__ __forceinline__ double to_d(__half v) { return (double)__half2float(v); }
__device__ __forceinline__ double to_d(__nv_bfloat16 v) { return (double)__bfloat162float(v); }
template <class S>
__device__ __forceinline__ S from_d(double v);
template <>
__device__ __forceinline__ double from_d<double>(double v) { return v; }
template <>
__device__ __forceinline__ float from_d<float>(double v) { return (float)v; }
template <>
__device__ __forceinline__ __half from_d<__half>(double v) { return __float2half_rn((float)v); }
template <>
__device__ __forceinline__ __nv_bfloat16 from_d<__nv_bfloat16>(double v) { return __float2bfloat16_rn((float)v); }

struct AuxParams {
  int nx, ny, nz;
  long long n;
  int model, enhanced, K;
  double phi[2][3];      // rest-state weights per component and group
  double nu_r, nu_b;
  double G, rho0, irho0; // SC two-component: G = G_eff; irho0 = 1 / rho0
  double body[3];
  int forced;            // there may be a force: body is not 0, or repulsion
  double umax, neg_tol;
  double Ga[2], Gr[2];   // multirange SC self-couplings
  int px;                // row pitch and size of the stored arrays
  long long ns;
  int aa;                // in-place streaming: the state's layout parity is its buffer index
};

AuxParams aux_params(const lbm_ctx* c) {
  const lbm_params& q = c->p;
  AuxParams a{};
  a.nx = q.nx;
  a.ny = q.ny;
  a.nz = q.nz;
  a.n = c->N;
  a.px = c->px;
  a.ns = c->NS;
  a.aa = c->aa;
  a.model = q.model;
  a.enhanced = q.enhanced_eq;
  a.K = c->K;
  rest_weights(q, a.phi);
  a.nu_r = (q.tau_r - 0.5) / 3.0;
  a.nu_b = (q.tau_b - 0.5) / 3.0;
  a.G = (q.model == LBM_MODEL_SC_2C || q.model == LBM_MODEL_SC_MR) ? q.G / (q.rho0_psi * q.rho0_psi) : q.G;
  for (int k = 0; k < 2; k++) {
    a.Ga[k] = q.Ga[k];
    a.Gr[k] = q.Gr[k];
  }
  a.rho0 = q.rho0_psi;
  a.irho0 = 1.0 / q.rho0_psi;
  for (int d = 0; d < 3; d++) a.body[d] = q.body_force[d];
  a.forced = c->rep || a.body[0] != 0 || a.body[1] != 0 || a.body[2] != 0;
  a.umax = q.umax_unstable > 0 ? q.umax_unstable : 0.5;
  double scale = 1.0;
  if (q.model == LBM_MODEL_CG) scale = fmax(scale, fmax(q.rho_r0, q.rho_b0));
  a.neg_tol = kNegDensityTol * scale;
  return a;
}

// The buffer pair holding the current state: the host's index, or the pair frozen by a
// tripped blow-up check (the host cannot know when that happened).
__device__ __forceinline__ int state_index(const lbm_diag* d, int cur) { return d->status ? d->trip_buf : cur; }

// Compute type of the step for a storage type: per-node arithmetic of the auxiliary
// kernels runs in it (FP64 only for FP64 storage); sums over the lattice stay FP64.
template <class S>
using step_t = typename std::conditional<std::is_same<S, double>::value, double, float>::type;

// a value of the compute type in FP64, in integer arithmetic: GB300 runs conversions to FP64
// at its low FP64 rate.  The exponent moves by 1023 - 127 (Inf and NaN: by 2047 - 255); a
// subnormal is scaled to a normal number first.
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v) {
  const bool sub = (__float_as_uint(v) & 0x7f800000u) == 0;
  const unsigned b = __float_as_uint(sub ? v * 0x1p64f : v), m = b & 0x7fffffffu;
  const unsigned up = sub ? 0x34000000u : m >= 0x7f800000u ? 0x70000000u : 0x38000000u;
  return __hiloint2double(int((b & 0x80000000u) | (m == 0 ? 0 : (m >> 3) + up)), int(b << 29));
}

// The nodes a thread of densities_kernel handles at a time: two in FP32, whose packed
// instructions work on both (lbm_vec.cuh), one in FP64.
template <class C>
struct Lanes;
template <>
struct Lanes<float> {
  using V = F2;
  static constexpr int W = 2;
};
template <>
struct Lanes<double> {
  using V = double;
  static constexpr int W = 1;
};
__device__ __forceinline__ double lane(double v, int) { return v; }
__device__ __forceinline__ float lane(const F2& v, int j) { return v[j]; }
__device__ __forceinline__ void set_lane(double& v, int, double x) { v = x; }
__device__ __forceinline__ void set_lane(F2& v, int j, float x) { v.set(j, x); }

// Sum of values of the compute type whose FP64 result is as accurate as FP64 summation.  In
// FP32 the sum is carried as an unevaluated pair s + c and the rounding error of every
// addition is kept exactly (TwoSum), at FP32 cost: GB300's FP64 rate is a small fraction of
// its FP32 rate, and the reductions here would otherwise be FP64 bound.
template <class V>
struct ExactSum;
template <>
struct ExactSum<double> {
  double s;
  __device__ __forceinline__ explicit ExactSum(double v = 0.0) : s(v) {}
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ void sub(double v) { s -= v; }
  __device__ __forceinline__ void add(const ExactSum& o) { s += o.s; }
  __device__ __forceinline__ void sub(const ExactSum& o) { s -= o.s; }
  __device__ __forceinline__ double value(int) const { return s; }
};
template <>
struct ExactSum<F2> {
  F2 s, c;
  __device__ __forceinline__ explicit ExactSum(F2 v = F2(0.f)) : s(v), c(0.f) {}
  __device__ __forceinline__ void add(F2 v) {
    F2 e;
    s = two_sum2(s, v, e);
    c = c + e;
  }
  __device__ __forceinline__ void sub(F2 v) {  // TwoSum of s and -v
    const F2 t = s - v, bb = t - s;
    c = c + ((s - (t - bb)) - (v + bb));
    s = t;
  }
  __device__ __forceinline__ void add(const ExactSum& o) {
    add(o.s);
    c = c + o.c;
  }
  __device__ __forceinline__ void sub(const ExactSum& o) {
    sub(o.s);
    c = c - o.c;
  }
  __device__ __forceinline__ double value(int j) const { return widen(s[j]) + widen(c[j]); }
};

// x, y, z of node n
__device__ __forceinline__ void node_xyz(long long n, const AuxParams& a, int& x, int& y, int& z) {
  node_coords(n, a.nx, a.ny, a.n, x, y, z);
}

// Index of the neighbour of (x, y, z), all steps at most 2 with one periodic wrap.  32-bit: no
// device holds the workspace of 2^32 nodes.
__device__ __forceinline__ unsigned wrapped(int x, int y, int z, const AuxParams& a) {
  x = x < 0 ? x + a.nx : (x >= a.nx ? x - a.nx : x);
  y = y < 0 ? y + a.ny : (y >= a.ny ? y - a.ny : y);
  z = z < 0 ? z + a.nz : (z >= a.nz ? z - a.nz : z);
  return unsigned(x) + unsigned(a.nx) * (unsigned(y) + unsigned(a.ny) * unsigned(z));
}

// 3 sum_i w_i phi_k(x + c_i) c_i of both fields, a wall neighbour replaced by the centre value.
template <class L, class C, class E>
__device__ __forceinline__ void grad_c(const E* phi0, const E* phi1, const uint8_t* solid, unsigned n, int x, int y,
                                       int z, const AuxParams& a, C (&g)[2][3]) {
  const E* const phi[2] = {phi0, phi1};
  C ax[2][3] = {}, dg[2][3] = {};
#pragma unroll
  for (int q = 0; q < L::NP; q++) {
    const int c[3] = {L::pcx(q), L::pcy(q), L::pcz(q)};
    unsigned mp = wrapped(x + c[0], y + c[1], z + c[2], a), mm = wrapped(x - c[0], y - c[1], z - c[2], a);
    if (solid) {
      if (solid[mp]) mp = n;
      if (solid[mm]) mm = n;
    }
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const C d = C(phi[k][mp]) - C(phi[k][mm]);
#pragma unroll
      for (int t = 0; t < 3; t++) {
        if (c[t] == 0) continue;
        if (L::pgrp(q) == 1) ax[k][t] = d;
        else if (c[t] > 0) dg[k][t] += d;
        else dg[k][t] -= d;
      }
    }
  }
  for (int k = 0; k < 2; k++)
    for (int t = 0; t < 3; t++) g[k][t] = C(3.0 * L::w(1)) * ax[k][t] + C(3.0 * L::w(2)) * dg[k][t];
}

// Eq. equiliCG for one colour (phi from Eq. phi, enhanced part optional) or Eq. equiliSC
// (phi = w, no enhanced part), minus phi_i * rref, to emit(i, value); drho = rho_k - rref
// (exact in FP64, then rounded), so every term is a small deviation.  A pair's values are
// even + odd and even - odd in c_i.
template <class L, class C, class EMIT>
__device__ __forceinline__ void feq_dev(C rho_k, const double* phi, C nubar_en, const C u[3], const C g[3], C drho,
                                        const EMIT& emit) {
  const C uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const C ug = u[0] * g[0] + u[1] * g[1] + u[2] * g[2];
  C even[3], quad[3], odd[3], mix[3];
#pragma unroll
  for (int s = 0; s < 3; s++) {
    const C w = C(L::w(s));
    even[s] = nubar_en * (C(L::psi(s)) * ug) + C(phi[s]) * drho - rho_k * w * C(1.5) * uu;
    quad[s] = rho_k * w * C(4.5);
    odd[s] = rho_k * w * C(3);
    mix[s] = nubar_en * C(2.0 * L::xi(s));
  }
  emit(0, even[0]);
#pragma unroll
  for (int q = 0; q < L::NP; q++) {
    const int c[3] = {L::pcx(q), L::pcy(q), L::pcz(q)}, s = L::pgrp(q);
    C cu = C(0), cgr = C(0);
#pragma unroll
    for (int t = 0; t < 3; t++) {
      if (c[t] > 0) { cu += u[t]; cgr += g[t]; }
      if (c[t] < 0) { cu -= u[t]; cgr -= g[t]; }
    }
    const C e = even[s] + cu * (quad[s] * cu + mix[s] * cgr);
    emit(2 * q + 1, e + odd[s] * cu);
    emit(2 * q + 2, e - odd[s] * cu);
  }
}

// Both component densities rounded to the compute type: out[k][n] = C(rho_k[n]).
template <class C>
__global__ void to_compute_kernel(const double* __restrict__ rr, const double* __restrict__ rb, C* __restrict__ out,
                                  long long n) {
  for (long long m = blockIdx.x * (long long)blockDim.x + threadIdx.x; m < n; m += (long long)gridDim.x * blockDim.x) {
    out[m] = C(rr[m]);
    out[n + m] = C(rb[m]);
  }
}

// Both gradients take each neighbour's index once, a pair's two populations share their even
// part, and every population goes out as it is formed (one loop over the directions from
// an array of them: CG 128^3 FP32 150 us, now 90; 470 MB take 69).
template <class L, class S, class RT, int K>
__global__ void __launch_bounds__(256) init_eq_kernel(S* __restrict__ fa, S* __restrict__ fb, RT* __restrict__ ra,
                                                      RT* __restrict__ rb_, const double* __restrict__ rr,
                                                      const double* __restrict__ rb, const double* __restrict__ U,
                                                      const uint8_t* __restrict__ solid,
                                                      const step_t<S>* __restrict__ fc, AuxParams a) {
  using C = step_t<S>;
  const unsigned N = (unsigned)a.n;
  for (unsigned n = blockIdx.x * blockDim.x + threadIdx.x; n < N; n += gridDim.x * blockDim.x) {
    int x, y, z;
    node_xyz(n, a, x, y, z);
    const unsigned st = a.px == a.nx ? n : unsigned(x) + unsigned(a.px) * (unsigned(y) + unsigned(a.ny) * unsigned(z));
    if (solid && solid[n]) {
      for (int k = 0; k < K; k++) {
        ra[k * a.ns + st] = RT(0);
        if (rb_) rb_[k * a.ns + st] = RT(0);
        for (int i = 0; i < L::Q; i++) {
          fa[(k * L::Q + i) * a.ns + st] = from_d<S>(0.0);
          if (fb) fb[(k * L::Q + i) * a.ns + st] = from_d<S>(0.0);
        }
      }
      continue;
    }
    C u[3] = {C(0), C(0), C(0)};
    if (U) {
      u[0] = C(U[n]);
      u[1] = C(U[a.n + n]);
      u[2] = C(U[2 * a.n + n]);
    }
    C en = C(0), g[2][3] = {};
    if (a.model == LBM_MODEL_CG) {
      if (a.enhanced) {
        const C r = fc ? fc[n] : C(rr[n]), b = fc ? fc[a.n + n] : C(rb[n]), rho = r + b;
        en = C(1) / ((r / rho) / C(a.nu_r) + (b / rho) / C(a.nu_b));  // Eq. interpVisc
      }
      if (fc)
        grad_c<L, C>(fc, fc + a.n, solid, n, x, y, z, a, g);
      else
        grad_c<L, C>(rr, rb, solid, n, x, y, z, a, g);
    }
    // Only pair 0 is written for fluid nodes: the first step writes every population and
    // reference density of every fluid node of pair 1.
#pragma unroll
    for (int k = 0; k < K; k++) {
      const double rho = (k == 0 ? rr : rb)[n];
      const RT rref = RT(rho);  // reference density: the initial density, rounded
      ra[k * a.ns + st] = rref;
      feq_dev<L, C>(C(rho), a.phi[k], en, u, g[k], C(rho - (double)rref), [&](int i, C v) {
        fa[(k * L::Q + i) * a.ns + st] = st_s<S, C>(v);
      });
    }
  }
}

__global__ void restore_acc_kernel(const double* __restrict__ plane, double* __restrict__ acc, long long n, bool first) {
  for (long long m = blockIdx.x * (long long)blockDim.x + threadIdx.x; m < n; m += (long long)gridDim.x * blockDim.x)
    acc[m] = first ? plane[m] : acc[m] + plane[m];
}

template <class S, class RT>
__global__ void restore_plane_kernel(S* __restrict__ fa, S* __restrict__ fb, RT* __restrict__ ra,
                                     RT* __restrict__ rb_, const double* __restrict__ plane,
                                     const double* __restrict__ acc, const uint8_t* __restrict__ solid, long long n,
                                     long long off, long long roff, double phi, bool write_ref, int nx, int px) {
  for (long long m = blockIdx.x * (long long)blockDim.x + threadIdx.x; m < n; m += (long long)gridDim.x * blockDim.x) {
    const bool wall = solid && solid[m];
    const RT r = wall ? RT(0) : RT(acc[m]);
    const S v = wall ? from_d<S>(0.0) : from_d<S>(plane[m] - phi * (double)r);
    const long long st = stored_index(m, nx, px);
    fa[off + st] = v;
    if (fb) fb[off + st] = v;
    if (write_ref) {
      ra[roff + st] = r;
      if (rb_) rb_[roff + st] = r;
    }
  }
}

// canonical populations f = g + phi r, FP64; `out` holds planes [first_plane, first_plane+np);
// 0 on wall nodes (whose slots the in-place scheme uses for bounced populations)
template <class L, class S, class RT>
__global__ void export_kernel(const S* __restrict__ f0, const S* __restrict__ f1, const RT* __restrict__ r0,
                              const RT* __restrict__ r1, const lbm_diag* __restrict__ d, int cur, int first_plane,
                              int np, double* __restrict__ out, const uint8_t* __restrict__ solid, AuxParams a) {
  const int b = state_index(d, cur);
  const S* f = b ? f1 : f0;
  const RT* r = b ? r1 : r0;
  const bool odd = a.aa && (b & 1);
  const long long total = (long long)np * a.n;
  for (long long m = blockIdx.x * (long long)blockDim.x + threadIdx.x; m < total; m += (long long)gridDim.x * blockDim.x) {
    const int plane = first_plane + (int)(m / a.n);
    const long long node = m - (long long)(plane - first_plane) * a.n;
    const int k = plane / L::Q, i = plane - k * L::Q;
    const long long st = stored_index(node, a.nx, a.px);
    out[m] = (solid && solid[node])
                 ? 0.0
                 : to_d(f[odd ? aa_index_n<L>(k, i, node, a.nx, a.ny, a.nz, a.n, odd) : (k * L::Q + i) * a.ns + st]) +
                       a.phi[k][grp<L>(i)] * to_d(r[k * a.ns + st]);
  }
}

// stored plane (k, i) of the even layout from the odd in-place layout (0 on wall nodes)
template <class L, class S>
__global__ void aa_gather_kernel(const S* __restrict__ f, S* __restrict__ out, const uint8_t* __restrict__ solid,
                                 int k, int i, AuxParams a) {
  for (long long m = blockIdx.x * (long long)blockDim.x + threadIdx.x; m < a.n; m += (long long)gridDim.x * blockDim.x) {
    out[m] = (solid && solid[m]) ? from_d<S>(0.0) : f[aa_index_n<L>(k, i, m, a.nx, a.ny, a.nz, a.n, true)];
  }
}


// x is finite: its exponent field is not all ones (integer test of the high word; GB300
// runs FP64 compares at its low FP64 rate).
__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// ---- fixed-order block reductions ----
// Ordered 64-bit keys of FP64 values: signed integer comparison orders them (GB300 runs FP64
// compares at its low FP64 rate).
__device__ __forceinline__ long long key_of(double v) {
  const long long b = __double_as_longlong(v);
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double of_key(long long k) {
  return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffLL));
}
constexpr long long kInfKey = 0x7ff0000000000000LL;

// A thread's share of the totals.  SUMS false: only what the blow-up check looks at, for
// callers that do not ask for the totals.
struct Acc {
  double sum[6];             // mass_r, mass_b, momentum, kinetic energy
  long long uu, minr, minb;  // keys of max |u|^2 and of the smallest densities
  int bad;                   // nodes with a value that is not finite
};
__device__ __forceinline__ void acc_init(Acc& a) {
  for (int s = 0; s < 6; s++) a.sum[s] = 0.0;
  a.uu = 0;
  a.minr = a.minb = kInfKey;
  a.bad = 0;
}
template <bool SUMS>
__device__ __forceinline__ void acc_merge(Acc& a, const Acc& b) {
  if constexpr (SUMS)
    for (int s = 0; s < 6; s++) a.sum[s] += b.sum[s];
  a.uu = max(a.uu, b.uu);
  a.minr = min(a.minr, b.minr);
  a.minb = min(a.minb, b.minb);
  a.bad += b.bad;
}
template <bool SUMS>
__device__ void block_reduce(Acc& a) {
  __shared__ Acc sh[kDiagThreads / 32];
  for (int off = 16; off > 0; off >>= 1) {
    Acc o;
    if constexpr (SUMS)
      for (int s = 0; s < 6; s++) o.sum[s] = __shfl_xor_sync(0xffffffffu, a.sum[s], off);
    o.uu = __shfl_xor_sync(0xffffffffu, a.uu, off);
    o.minr = __shfl_xor_sync(0xffffffffu, a.minr, off);
    o.minb = __shfl_xor_sync(0xffffffffu, a.minb, off);
    o.bad = __shfl_xor_sync(0xffffffffu, a.bad, off);
    acc_merge<SUMS>(a, o);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) sh[warp] = a;
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < (int)(blockDim.x >> 5); w++) acc_merge<SUMS>(a, sh[w]);
}

// Fixed-order reduction of the nblk block partials into the totals and the blow-up status
// (all threads of one block take part).
template <bool SUMS>
__device__ void reduce_partials(const double* partials, int nblk, lbm_diag* d, int cur, const AuxParams& a) {
  Acc acc;
  acc_init(acc);
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) {
    const double* p = partials + b * LBM_NTOTALS;
    Acc o;
    if constexpr (SUMS)
      for (int s = 0; s < 6; s++) o.sum[s] = __ldcg(&p[s]);
    o.uu = key_of(__ldcg(&p[6]));
    o.bad = (int)__ldcg(&p[7]);
    o.minr = key_of(__ldcg(&p[8]));
    o.minb = key_of(__ldcg(&p[9]));
    acc_merge<SUMS>(acc, o);
  }
  __syncthreads();  // the block's own reduction is done with the shared array
  block_reduce<SUMS>(acc);
  if (threadIdx.x == 0) {
    // max |u| from max |u|^2 (sqrt is monotonic and correctly rounded)
    const double um = sqrt(of_key(acc.uu)), minr = of_key(acc.minr), minb = of_key(acc.minb);
    int st = 0;
    if (acc.bad > 0) st |= 1;
    if constexpr (SUMS)
      if (!isfinite(acc.sum[0]) || !isfinite(acc.sum[1])) st |= 1;
    if (minr < -a.neg_tol || minb < -a.neg_tol) st |= 2;
    if (!(um <= a.umax)) st |= 4;
    if constexpr (SUMS)
      for (int s = 0; s < 6; s++) d->totals[s] = acc.sum[s];
    d->totals[6] = um;
    d->totals[7] = acc.bad;
    d->totals[8] = minr;
    d->totals[9] = minb;
    if (d->status == 0 && st != 0) d->trip_buf = cur;
    d->status |= st;
  }
}

// Velocity of one node (force-shifted, Eq. guoforce; 0 on walls) and its share of the totals.
template <bool SUMS, bool FORCED = true>
__device__ __forceinline__ void diag_node(bool wall, double r, double b, const double (&j)[3], const double (&F)[3],
                                          double (&u)[3], Acc& acc) {
  u[0] = u[1] = u[2] = 0.0;
  if (wall) return;
  const double rho = r + b;
  const double inv = 1.0 / rho;
  for (int t = 0; t < 3; t++) u[t] = (FORCED ? j[t] + 0.5 * F[t] : j[t]) * inv;
  const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  if constexpr (SUMS) {
    acc.sum[0] += r;
    acc.sum[1] += b;
    acc.sum[2] += j[0];
    acc.sum[3] += j[1];
    acc.sum[4] += j[2];
    acc.sum[5] += 0.5 * rho * uu;
  }
  // fmax / fmin: a NaN does not count (its key is beyond the infinities')
  const long long ku = key_of(uu), kr = key_of(r), kb = key_of(b);
  if (ku <= kInfKey) acc.uu = max(acc.uu, ku);
  if (kr >= ~kInfKey) acc.minr = min(acc.minr, kr);
  if (kb >= ~kInfKey) acc.minb = min(acc.minb, kb);
  acc.bad += !(finite_bits(r) && finite_bits(b) && finite_bits(j[0]) && finite_bits(j[1]) && finite_bits(j[2]));
}

// The block that finishes last reduces every block's partial (in block order, whatever the
// finishing order): partial written, fence, count; the counter goes back to 0.  Slot 6 of
// the partials holds max |u|^2 (its square root is taken in the final pass).
template <bool SUMS>
__device__ __forceinline__ void diag_finish(Acc& acc, double* __restrict__ partials, lbm_diag* __restrict__ d, int cur,
                                            const AuxParams& a) {
  block_reduce<SUMS>(acc);
  __shared__ bool last;
  if (threadIdx.x == 0) {
    double* p = partials + blockIdx.x * LBM_NTOTALS;
    if constexpr (SUMS)
      for (int s = 0; s < 6; s++) p[s] = acc.sum[s];
    p[6] = of_key(acc.uu);
    p[7] = acc.bad;
    p[8] = of_key(acc.minr);
    p[9] = of_key(acc.minb);
    __threadfence();
    last = atomicAdd(&d->done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (last) {
    __threadfence();
    reduce_partials<SUMS>(partials, gridDim.x, d, cur, a);
    if (threadIdx.x == 0) d->done = 0;
  }
}

// One pass over the populations: the component densities rr, rb (FP64, as exact as FP64
// summation), psi of Eq. pseudopotential (SC multiphase, FP64), the momentum
// j = sum_k sum_i c_i f^k_i into jm [3][N] (FP64), and for the multirange model the
// pseudopotentials Psi_s of both species in the step's compute type into mrpsi [2][N].
// FUSED (no stencil: colour gradient; rep, if not null: the repulsion force): the velocity and the totals as well, so that
// neither the densities nor the momentum are read again.
// rb may be null with one component.  `pitch`/`rows`: stored rows of `row` nodes, `pitch`
// apart (one row of N nodes where they are dense); vld: pairs of stored nodes are aligned;
// vst: pairs of FP64 results are.
// Bound by FP32 issue as scalar code: 128^3 CG FP32 107 us, with the reads of diag_kernel
// 274; two nodes a thread and fused 115 us (403 MB: 59 us at the copy rate).
template <class L, class S, class RT, int MODEL, bool FUSED, bool SUMS>
__global__ void __launch_bounds__(kDiagThreads, 2) densities_kernel(
    const S* __restrict__ f0, const S* __restrict__ f1, const RT* __restrict__ r0, const RT* __restrict__ r1,
    lbm_diag* __restrict__ d, int cur, double* __restrict__ rr, double* __restrict__ rb, double* __restrict__ psi,
    double* __restrict__ jm, step_t<S>* __restrict__ mrpsi, const uint8_t* __restrict__ solid,
    double* __restrict__ partials, const step_t<S>* __restrict__ rep, AuxParams a, unsigned row, unsigned pitch, unsigned rows, int vld, int vst) {
  using C = step_t<S>;
  using V = typename Lanes<C>::V;
  constexpr int W = Lanes<C>::W, K = MODEL == LBM_MODEL_SC_MP ? 1 : 2;
  const int b = state_index(d, cur);
  const S* f = b ? f1 : f0;
  const RT* r = b ? r1 : r0;
  const bool odd = a.aa && (b & 1);
  const unsigned per = (row + W - 1) / W, total = per * rows;
  [[maybe_unused]] Acc acc;
  if constexpr (FUSED) acc_init(acc);
  for (unsigned p = blockIdx.x * blockDim.x + threadIdx.x; p < total; p += gridDim.x * blockDim.x) {
    const unsigned y = rows == 1 ? 0 : p / per, x = (p - y * per) * W;
    const unsigned n = y * row + x, st = y * pitch + x;
    const bool two = W == 1 || x + 1 < row;  // else the second node is beyond the row's end
    auto load = [&](auto* arr) -> V {  // of a stored array
      using E = typename std::remove_const<typename std::remove_pointer<decltype(arr)>::type>::type;
      V v;
      if constexpr (W == 1) {
        v = ld_s<E, C>(arr[st]);
      } else {
        E e[2];
        if (vld) {
          using U = typename std::conditional<sizeof(E) == 4, uint2, unsigned>::type;
          *reinterpret_cast<U*>(e) = *reinterpret_cast<const U*>(arr + st);
        } else {
          e[0] = arr[st];
          e[1] = two ? arr[st + 1] : e[0];
        }
        v.set(0, ld_s<E, C>(e[0]));
        v.set(1, ld_s<E, C>(e[1]));
      }
      return v;
    };
    // the shift phi_i r is symmetric in c_i and carries no momentum: opposite pairs of the
    // stored deviations.  The colours' momenta nearly cancel at interfaces, so rounding in
    // the sum would show up in the reported u: exact sums
    ExactSum<V> j[3], s[K];
#pragma unroll
    for (int k = 0; k < K; k++) {
      V g[L::Q];
      if (odd) {
#pragma unroll
        for (int i = 0; i < L::Q; i++)
#pragma unroll
          for (int l = 0; l < W; l++)
            set_lane(g[i], l, ld_s<S, C>(f[aa_index_n<L>(k, i, l && two ? n + l : n, a.nx, a.ny, a.nz, a.n, true)]));
      } else {
#pragma unroll
        for (int i = 0; i < L::Q; i++) g[i] = load(f + (k * L::Q + i) * a.ns);
      }
      s[k] = ExactSum<V>(load(r + k * a.ns));  // sum_i phi_i = 1
#pragma unroll
      for (int i = 0; i < L::Q; i++) s[k].add(g[i]);
#pragma unroll
      for (int q = 0; q < L::NP; q++) {
        ExactSum<V> dq(g[2 * q + 1]);
        dq.sub(g[2 * q + 2]);
        const int c[3] = {L::pcx(q), L::pcy(q), L::pcz(q)};
#pragma unroll
        for (int t = 0; t < 3; t++)
          if (c[t] > 0) j[t].add(dq); else if (c[t] < 0) j[t].sub(dq);
      }
    }
    double out[5][W];  // rr, rb, j or u
#pragma unroll
    for (int l = 0; l < W; l++) {
      out[0][l] = s[0].value(l);
      out[1][l] = K == 2 ? s[K - 1].value(l) : 0.0;
      const double jj[3] = {j[0].value(l), j[1].value(l), j[2].value(l)};
      for (int t = 0; t < 3; t++) out[2 + t][l] = jj[t];
      if (l && !two) break;
      if constexpr (FUSED) {
        double F[3] = {a.body[0], a.body[1], a.body[2]};
        double u[3];
        const bool wall = solid && solid[n + l];
        if (rep)
          for (int t = 0; t < 3; t++) F[t] += widen(rep[t * a.n + n + l]);
        if (a.forced)
          diag_node<SUMS>(wall, out[0][l], out[1][l], jj, F, u, acc);
        else
          diag_node<SUMS, false>(wall, out[0][l], out[1][l], jj, F, u, acc);
        for (int t = 0; t < 3; t++) out[2 + t][l] = u[t];
      }
      // Eq. pseudopotential, once per node (the force stencil reads it 18 times)
      if constexpr (MODEL == LBM_MODEL_SC_MP) psi[n + l] = a.rho0 * (1.0 - exp(-out[0][l] * a.irho0));
      if constexpr (MODEL == LBM_MODEL_SC_MR) {  // Psi_s = rho_0 (1 - exp(-rho_s / rho_0)) in the compute type
        const C c0 = C(a.rho0), ic0 = C(a.irho0);
        for (int k = 0; k < 2; k++) mrpsi[k * a.n + n + l] = c0 * (C(1) - exp(-C(out[k][l]) * ic0));
      }
    }
    double* const dst[5] = {rr, rb, jm, jm + a.n, jm + 2 * a.n};
#pragma unroll
    for (int t = 0; t < 5; t++) {
      if ((t == 1 && K == 1 && !rb) || (FUSED && t >= 2 && !jm)) continue;
      if (W == 2 && vst && two) {
        *reinterpret_cast<double2*>(dst[t] + n) = make_double2(out[t][0], out[t][W - 1]);
      } else {
        dst[t][n] = out[t][0];
        if (W == 2 && two) dst[t][n + 1] = out[t][W - 1];
      }
    }
  }
  if constexpr (FUSED) diag_finish<SUMS>(acc, partials, d, cur, a);
}

// sum_i w_i phi(x + c_i) c_i of one field as opposite-pair differences in FP64 (the force is
// a small difference of O(1) values), in units of the diagonal weight: the axis differences
// weigh w_axis / w_diagonal times as much, so that a component takes one product.
template <class L>
struct Gradient {
  double s[3] = {0.0, 0.0, 0.0};
  double ax[3] = {0.0, 0.0, 0.0};
  __device__ __forceinline__ void add(int q, double dq) {
    const int c[3] = {L::pcx(q), L::pcy(q), L::pcz(q)};
#pragma unroll
    for (int t = 0; t < 3; t++) {
      if (c[t] == 0) continue;
      if (L::pgrp(q) == 1) ax[t] = dq;
      else if (c[t] > 0) s[t] += dq;
      else s[t] -= dq;
    }
  }
  __device__ __forceinline__ double at(int t) const {
    constexpr double ratio = L::D == 3 ? 2.0 : 4.0;  // w(1) / w(2), exact
    return ratio * ax[t] + s[t];
  }
};

// F = body - G (r grad b + b grad r) or body - G psi grad psi, of one node
template <class L, int MODEL, bool WALLS>
__device__ __forceinline__ void sc_force(const double* __restrict__ rr, const double* __restrict__ rb,
                                         const double* __restrict__ psi, const uint8_t* __restrict__ solid, double r,
                                         double b, unsigned n, int x, int y, int z, const AuxParams& a, double (&F)[3]) {
  Gradient<L> g1, g2;
  const double pc = MODEL == LBM_MODEL_SC_MP ? psi[n] : 0.0;
#pragma unroll
  for (int q = 0; q < L::NP; q++) {
    const unsigned mp = wrapped(x + L::pcx(q), y + L::pcy(q), z + L::pcz(q), a);
    const unsigned mm = wrapped(x - L::pcx(q), y - L::pcy(q), z - L::pcz(q), a);
    const bool wp = WALLS && solid[mp], wm = WALLS && solid[mm];
    if constexpr (MODEL == LBM_MODEL_SC_MP) {
      g1.add(q, (wp ? pc : psi[mp]) - (wm ? pc : psi[mm]));
    } else {
      g1.add(q, (wp ? b : rb[mp]) - (wm ? b : rb[mm]));
      g2.add(q, (wp ? r : rr[mp]) - (wm ? r : rr[mm]));
    }
  }
  const double gw = -a.G * L::w(2);
  if constexpr (MODEL == LBM_MODEL_SC_MP) {
    const double gp = gw * pc;
    for (int t = 0; t < 3; t++) F[t] = gp * g1.at(t) + a.body[t];
  } else {
    const double gr = gw * r, gb = gw * b;
    for (int t = 0; t < 3; t++) F[t] = gr * g1.at(t) + (gb * g2.at(t) + a.body[t]);
  }
}

// Per-node velocity and the block partials of the totals, from the staged densities and
// momentum (densities_kernel): no population is read again.  u (force-shifted, Eq.
// guoforce) may be written over jm (uo == jm): each node reads its own momentum first.
// FP64 issue bounds it (2 operations per clock and SM): every factor common to a stencil is
// applied once to its sum.  128^3 SC multiphase 339 -> 183 us, two components 442 ->
// 290 us.
template <class L, int MODEL, bool WALLS, bool SUMS>
__global__ void __launch_bounds__(kDiagThreads) diag_kernel(const double* __restrict__ rr,
                                                            const double* __restrict__ rb,
                                                            const double* __restrict__ psi,
                                                            const double* jm, const uint8_t* __restrict__ solid,
                                                            double* uo, double* __restrict__ partials, AuxParams a,
                                                            lbm_diag* __restrict__ d, int cur) {
  Acc acc;
  acc_init(acc);
  const unsigned N = (unsigned)a.n;
  for (unsigned n = blockIdx.x * blockDim.x + threadIdx.x; n < N; n += gridDim.x * blockDim.x) {
    const bool wall = WALLS && solid[n];
    const double j[3] = {jm[n], jm[a.n + n], jm[2 * a.n + n]};
    const double r = rr[n], b = MODEL == LBM_MODEL_SC_MP ? 0.0 : rb[n];
    double F[3] = {a.body[0], a.body[1], a.body[2]};
    if (!wall) {
      int x, y, z;
      node_xyz(n, a, x, y, z);
      sc_force<L, MODEL, WALLS>(rr, rb, psi, solid, r, b, n, x, y, z, a, F);
    }
    double u[3];
    diag_node<SUMS>(wall, r, b, j, F, u, acc);
    if (uo)
      for (int t = 0; t < 3; t++) uo[t * a.n + n] = u[t];
  }
  diag_finish<SUMS>(acc, partials, d, cur, a);
}

// The same for the multirange model: self forces of Eqs. doublebeltattractiveforce /
// doublebeltrepulsionforce with the staged Psi_s, summed in the step's compute type C as the
// step kernel sums them; a wall neighbour takes the centre value.  Each node reads 92 values
// of either species: a block marches along z over a tile of 32 x 8 nodes with the five
// planes around it in shared memory (two halo nodes).  128x64x64: 674 us with the neighbours
// gathered from global memory, 121 us from the planes (FP64 issue of the
// cross force bounds it).
constexpr int kMrTX = 32, kMrTY = kDiagThreads / kMrTX, kMrEX = kMrTX + 4, kMrEY = kMrTY + 4, kMrZ = 4;
template <class C, bool WALLS, bool SUMS>
__global__ void __launch_bounds__(kDiagThreads) diag_mr_kernel(const double* __restrict__ rr,
                                                               const double* __restrict__ rb,
                                                               const C* __restrict__ mrpsi, const double* jm,
                                                               const uint8_t* __restrict__ solid, double* uo,
                                                               double* __restrict__ partials, AuxParams a,
                                                               lbm_diag* __restrict__ d, int cur) {
  using L = D3Q19;
  constexpr int NE = kMrEX * kMrEY;
  __shared__ C ps[5][2][NE];
  __shared__ uint8_t msk[5][WALLS ? NE : 1];
  Acc acc;
  acc_init(acc);
  const int ncx = (a.nx + kMrTX - 1) / kMrTX, ncy = (a.ny + kMrTY - 1) / kMrTY, ncz = (a.nz + kMrZ - 1) / kMrZ;
  const long long units = (long long)ncx * ncy * ncz;
  const int tx = threadIdx.x % kMrTX, ty = threadIdx.x / kMrTX;
  for (long long w = blockIdx.x; w < units; w += gridDim.x) {
    const int bx = int(w % ncx) * kMrTX, by = int(w / ncx % ncy) * kMrTY, z0 = int(w / ncx / ncy) * kMrZ;
    const int z1 = min(z0 + kMrZ, a.nz);
    auto stage = [&](int z) {  // plane z into slot (z + 5) % 5; beyond the lattice, its periodic image
      const int zw = ((z % a.nz) + a.nz) % a.nz, slot = (z + 5) % 5;
      for (int e = threadIdx.x; e < NE; e += kDiagThreads) {
        const int X = bx + e % kMrEX - 2, Y = by + e / kMrEX - 2;
        const int Xw = (X + 2 * a.nx) % a.nx, Yw = (Y + 2 * a.ny) % a.ny;
        const unsigned m = wrapped(Xw, Yw, zw, a);
        ps[slot][0][e] = mrpsi[m];
        ps[slot][1][e] = mrpsi[a.n + m];
        if constexpr (WALLS) msk[slot][e] = solid[m];
      }
    };
    __syncthreads();  // the last unit's reads are done
    for (int z = z0 - 2; z < z0 + 2; z++) stage(z);
    for (int z = z0; z < z1; z++) {
      stage(z + 2);
      __syncthreads();
      const int x = bx + tx, y = by + ty;
      if (x < a.nx && y < a.ny) {
        const unsigned n = wrapped(x, y, z, a);
        const bool wall = WALLS && solid[n];
        const double j[3] = {jm[n], jm[a.n + n], jm[2 * a.n + n]};
        const double r = rr[n], b = rb[n];
        double F[3] = {a.body[0], a.body[1], a.body[2]};
        if (!wall) {
          sc_force<L, LBM_MODEL_SC_MR, WALLS>(rr, rb, nullptr, solid, r, b, n, x, y, z, a, F);
          int slot[5];
#pragma unroll
          for (int t = 0; t < 5; t++) slot[t] = (z + t + 3) % 5;  // plane z + t - 2
          const int e0 = (ty + 2) * kMrEX + tx + 2;
#pragma unroll
          for (int sp = 0; sp < 2; sp++) {
            const C pc = ps[slot[2]][sp][e0];
            auto psi_at = [&](int dx, int dy, int dz) -> C {
              const int e = e0 + dy * kMrEX + dx, t = slot[dz + 2];
              if (WALLS && msk[t][e]) return pc;
              return ps[t][sp][e];
            };
            C att[3] = {C(0), C(0), C(0)}, rep[3] = {C(0), C(0), C(0)};
#pragma unroll
            for (int dz = 0; dz <= 2; dz++)
#pragma unroll
              for (int dy = -2; dy <= 2; dy++)
#pragma unroll
                for (int dx = -2; dx <= 2; dx++) {
                  const int r2 = dx * dx + dy * dy + dz * dz;
                  if (r2 == 0 || r2 > 8 || mr_weight(r2) == 0.0 || !(dz > 0 || dy > 0 || (dy == 0 && dx > 0))) continue;
                  const C diff = psi_at(dx, dy, dz) - psi_at(-dx, -dy, -dz);
                  const C dr = C(mr_weight(r2)) * diff;
                  if (dx) rep[0] += C(dx) * dr;
                  if (dy) rep[1] += C(dy) * dr;
                  if (dz) rep[2] += C(dz) * dr;
                  if (r2 > 2) continue;
                  const C da = C(L::w(r2)) * diff;
                  if (dx) att[0] += C(dx) * da;
                  if (dy) att[1] += C(dy) * da;
                  if (dz) att[2] += C(dz) * da;
                }
            const double ga = -a.Ga[sp] * widen(pc), gr = -a.Gr[sp] * widen(pc);
            for (int t = 0; t < 3; t++) F[t] += ga * widen(att[t]) + gr * widen(rep[t]);
          }
        }
        double u[3];
        diag_node<SUMS>(wall, r, b, j, F, u, acc);
        if (uo)
          for (int t = 0; t < 3; t++) uo[t * a.n + n] = u[t];
      }
      __syncthreads();
    }
  }
  diag_finish<SUMS>(acc, partials, d, cur, a);
}

// The wall mask as the pair kernel reads it (kWallAny, lbm_step_pair.cuh), one warp per word.
__global__ void wall_words_kernel(const uint8_t* __restrict__ solid, unsigned long long* __restrict__ words, int tiles,
                                  AuxParams a) {
  const int lane = threadIdx.x & 31;
  const unsigned total = unsigned(tiles) * a.ny * a.nz, warps = gridDim.x * (blockDim.x / 32);
  for (unsigned w = (blockIdx.x * blockDim.x + threadIdx.x) / 32; w < total; w += warps) {
    const unsigned row = w / tiles, z = row / a.ny;
    const int y = int(row - z * a.ny), x = int(w - row * tiles) * 32 - 1 + lane;
    unsigned lo = 0, hi = 0, any = 0;
    for (int dz = -1; dz <= 1; dz++)
      for (int dy = -1; dy <= 2; dy++) {
        const unsigned Y = unsigned(y + dy + a.ny) % unsigned(a.ny), Z = unsigned(int(z) + dz + a.nz) % unsigned(a.nz);
        const uint8_t* s = solid + (long long)a.nx * (Y + (long long)a.ny * Z);
        auto wall = [&](int X) { return X <= a.nx && s[X < 0 ? a.nx - 1 : X < a.nx ? X : 0] != 0; };
        const unsigned b = __ballot_sync(0xffffffffu, wall(x));
        const unsigned c = __ballot_sync(0xffffffffu, lane < 2 && wall(x + 32));
        any |= b | c;
        if (dz == 0 && dy == 0) {
          lo = b;
          hi = c;
        }
      }
    if (lane == 0) words[w] = lo | (unsigned long long)hi << 32 | (any ? kWallAny : 0);
  }
}

// The planes of tile rows with walls in sight and the cuts (kWallCost, lbm_step_pair.cuh) of a walled
// lattice, one block: every thread adds up the costs of its share of the positions, and walks them again from the sum of the threads before.
constexpr int kCutThreads = 1024;
__global__ void __launch_bounds__(kCutThreads) wall_cuts_kernel(const unsigned long long* __restrict__ words,
                                                                uint8_t* __restrict__ rows_walled, int* __restrict__ cuts,
                                                                int ncuts, int tiles, AuxParams a) {
  __shared__ long long sums[kCutThreads];
  const long long total = (long long)((a.ny + 7) / 8) * a.nz;
  const long long p0 = total * threadIdx.x / kCutThreads, p1 = total * (threadIdx.x + 1) / kCutThreads;
  auto in_sight = [&](long long pos) {
    const int row = int(pos / a.nz), z = int(pos - (long long)row * a.nz);
    unsigned long long any = 0;
    for (int y = row * 8; y < min(row * 8 + 8, a.ny); y += 2)
      for (int t = 0; t < tiles; t++) any |= words[((long long)z * a.ny + y) * tiles + t];
    return (any & kWallAny) != 0;
  };
  auto cost = [&](long long pos) { return rows_walled[pos] ? kWallCost : kPlainCost; };
  long long own = 0;
  for (long long pos = p0; pos < p1; pos++) {
    rows_walled[pos] = in_sight(pos);
    own += cost(pos);
  }
  sums[threadIdx.x] = own;
  for (int off = 1; off < kCutThreads; off *= 2) {
    __syncthreads();
    const long long before = (int)threadIdx.x >= off ? sums[threadIdx.x - off] : 0;
    __syncthreads();
    sums[threadIdx.x] += before;
  }
  __syncthreads();
  const long long all = sums[kCutThreads - 1];
  long long sum = sums[threadIdx.x] - own;
  if (threadIdx.x == 0) cuts[0] = 0;
  for (long long pos = p0; pos < p1; pos++) {
    const long long first = sum * ncuts / all + 1;
    sum += cost(pos);
    for (long long g = first; g <= sum * ncuts / all; g++) cuts[g] = int(pos + 1);
  }
}

// A warp per row, four 32-bit words of it in flight per lane: the stored rows in whole words (their
// pitch is a multiple of 16 bytes; what lies beyond a row's end is never read), the dense ones in
// units U of their alignment.  w: units of a dense row; pitch, stride: words of a stored row and array.
template <class U>
__global__ void __launch_bounds__(256) pack_rows_kernel(U* __restrict__ dense, unsigned* __restrict__ stored, size_t r0,
                                                        size_t rows, size_t per, unsigned w, unsigned pitch,
                                                        size_t stride, bool to_dense) {
  constexpr unsigned P = 4 / sizeof(U);
  const unsigned lane = threadIdx.x & 31, words = (w + P - 1) / P;
  const size_t warps = (size_t)gridDim.x * (blockDim.x / 32);
  for (size_t r = blockIdx.x * (size_t)(blockDim.x / 32) + threadIdx.x / 32; r < rows; r += warps) {
    const size_t array = (r0 + r) / per;
    unsigned* const s = stored + array * stride + (r0 + r - array * per) * pitch;
    U* const d = dense + r * w;
    for (unsigned x = lane; x < words; x += 128) {
      union {
        unsigned word;
        U unit[P];
      } v[4];
#pragma unroll
      for (unsigned i = 0; i < 4; i++) {
        if (x + 32 * i >= words) continue;
        if (to_dense) v[i].word = s[x + 32 * i];
        else
#pragma unroll
          for (unsigned j = 0; j < P; j++)
            if ((x + 32 * i) * P + j < w) v[i].unit[j] = d[(x + 32 * i) * P + j];
      }
#pragma unroll
      for (unsigned i = 0; i < 4; i++) {
        if (x + 32 * i >= words) continue;
        if (!to_dense) s[x + 32 * i] = v[i].word;
        else
#pragma unroll
          for (unsigned j = 0; j < P; j++)
            if ((x + 32 * i) * P + j < w) d[(x + 32 * i) * P + j] = v[i].unit[j];
      }
    }
  }
}

template <class U>
cudaError_t pack_rows_t(lbm_ctx* c, void* dense, void* stored, size_t r0, size_t rows, size_t per, size_t elt, bool to_dense) {
  const int blocks = (int)std::min<size_t>((rows + 7) / 8, 8 * (size_t)c->nsm);
  c->launches += 1;
  pack_rows_kernel<U><<<blocks, 256, 0, c->stream>>>(static_cast<U*>(dense), static_cast<unsigned*>(stored), r0, rows, per,
                                                     unsigned(c->p.nx * elt / sizeof(U)), unsigned(c->px * elt / 4),
                                                     (size_t)c->NS * elt / 4, to_dense);
  return cudaGetLastError();
}

int grid_for(long long n, int threads, int cap) {
  long long b = (n + threads - 1) / threads;
  if (b > cap) b = cap;
  if (b < 1) b = 1;
  return (int)b;
}

template <class L, class S, class RT>
cudaError_t init_t(lbm_ctx* c, const double* rr, const double* rb, const double* u) {
  using C = step_t<S>;
  const AuxParams a = aux_params(c);
  // CG in a compute type narrower than FP64: the gradient stencil reads each density 19
  // times, so the fields are rounded to the compute type once, into the free tail of the
  // staging buffer ([5N, 6N) doubles hold 2N values of at most 4 bytes); the stencil gives
  // the same values as rounding at every read
  C* fc = nullptr;
  if (sizeof(C) < sizeof(double) && c->p.model == LBM_MODEL_CG) {
    fc = reinterpret_cast<C*>(c->stage + 5 * c->N);
    to_compute_kernel<C><<<grid_for(c->N, 256, 8192), 256, 0, c->stream>>>(rr, rb, fc, c->N);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    c->launches += 1;
  }
  // in-place streaming: one buffer pair (the second pointers alias the first)
  auto kern = c->K == 2 ? init_eq_kernel<L, S, RT, 2> : init_eq_kernel<L, S, RT, 1>;
  kern<<<grid_for(c->N, 256, 8192), 256, 0, c->stream>>>(
      static_cast<S*>(c->f[0]), c->aa ? nullptr : static_cast<S*>(c->f[1]), static_cast<RT*>(c->r[0]),
      c->aa ? nullptr : static_cast<RT*>(c->r[1]), rr, rb, u, c->has_walls ? c->solid : nullptr, fc, a);
  return cudaGetLastError();
}

template <class L, class S, class RT>
cudaError_t restore_t(lbm_ctx* c, const double* plane, int k, int i, const double* acc) {
  double phi[2][3];
  rest_weights(c->p, phi);
  restore_plane_kernel<S, RT><<<grid_for(c->N, 256, 8192), 256, 0, c->stream>>>(
      static_cast<S*>(c->f[0]), c->aa ? nullptr : static_cast<S*>(c->f[1]), static_cast<RT*>(c->r[0]),
      c->aa ? nullptr : static_cast<RT*>(c->r[1]),
      plane, acc + (long long)k * c->N, c->has_walls ? c->solid : nullptr, c->N, (long long)(k * c->Q + i) * c->NS,
      (long long)k * c->NS, phi[k][grp<L>(i)], i == 0, c->p.nx, c->px);
  return cudaGetLastError();
}

template <class L, class S, class RT>
cudaError_t export_t(lbm_ctx* c, double* out, int first_plane, int np) {
  const AuxParams a = aux_params(c);
  export_kernel<L, S, RT><<<grid_for((long long)np * c->N, 256, 16384), 256, 0, c->stream>>>(
      static_cast<const S*>(c->f[0]), static_cast<const S*>(c->f[1]), static_cast<const RT*>(c->r[0]),
      static_cast<const RT*>(c->r[1]), c->diag, c->cur, first_plane, np, out, c->has_walls ? c->solid : nullptr, a);
  return cudaGetLastError();
}

template <class L, class S, class RT>
cudaError_t gather_t(lbm_ctx* c, void* out, int k, int i) {
  const AuxParams a = aux_params(c);
  aa_gather_kernel<L, S><<<grid_for(c->N, 256, 8192), 256, 0, c->stream>>>(
      static_cast<const S*>(c->f[0]), static_cast<S*>(out), c->has_walls ? c->solid : nullptr, k, i, a);
  return cudaGetLastError();
}

// Threads of a block of the moment kernels for `items` of work: fewer on small lattices, whose
// FP64 work then spreads over all SMs (2D 128^2 CG FP64: 20.6 us with 256, 16.0 with this rule;
// the same on lattices that fill the SMs either way).
int diag_threads(const lbm_ctx* c, long long items) {
  int t = kDiagThreads;
  while (t > 64 && items < (long long)t * c->nsm) t /= 2;
  return t;
}

template <class L, class S, class RT, int MODEL, bool FUSED, bool SUMS>
cudaError_t densities_t(lbm_ctx* c, const AuxParams& a, double* rr, double* rb, double* psi, double* jm) {
  using C = step_t<S>;
  constexpr int W = Lanes<C>::W;
  const bool dense = c->px == c->p.nx;
  const long long row = dense ? c->N : c->p.nx, pitch = dense ? c->N : c->px, rows = c->N / row;
  const long long total = (row + W - 1) / W * rows;
  const int threads = diag_threads(c, total);
  const int blocks = (int)std::min<long long>((total + threads - 1) / threads, FUSED ? 2 * c->nsm : c->nblk_diag);
  // pairs are aligned where rows and whole arrays hold an even number of nodes
  const int vld = pitch % 2 == 0 && c->NS % 2 == 0;
  auto at16 = [](const double* p) { return !p || reinterpret_cast<uintptr_t>(p) % 16 == 0; };
  const int vst = row % 2 == 0 && c->N % 2 == 0 && at16(rr) && at16(rb) && at16(jm);
  C* mrpsi = MODEL == LBM_MODEL_SC_MR ? reinterpret_cast<C*>(psi) : nullptr;
  const uint8_t* solid = c->has_walls ? c->solid : nullptr;
  densities_kernel<L, S, RT, MODEL, FUSED, SUMS><<<blocks, threads, 0, c->stream>>>(
      static_cast<const S*>(c->f[0]), static_cast<const S*>(c->f[1]), static_cast<const RT*>(c->r[0]),
      static_cast<const RT*>(c->r[1]), c->diag, c->cur, rr, rb, psi, jm, mrpsi, solid, c->partials,
      c->rep ? static_cast<const C*>(c->rep_f) : nullptr, a, (unsigned)row,
      (unsigned)pitch, (unsigned)rows, vld, vst);
  c->launches += 1;
  return cudaGetLastError();
}

// rr, rb: where the densities go (rb null: a single component's, not asked for); uo: where
// the velocity goes, null if it is not asked for.
template <class L, class S, class RT, int MODEL, bool SUMS>
cudaError_t diag_t(lbm_ctx* c, double* rr, double* rb, double* uo) {
  using C = step_t<S>;
  const AuxParams a = aux_params(c);
  double* jm = c->stage + 2 * c->N;   // momentum, then (if requested here) the velocity
  double* psi = c->stage + 5 * c->N;  // SC multiphase psi (FP64), or the multirange Psi_s
  const uint8_t* solid = c->has_walls ? c->solid : nullptr;
  if constexpr (MODEL == LBM_MODEL_CG) {
    if (c->rep) {
      cudaError_t e = launch_rep_prepass_t<L, C, S, RT>(c, c->cur);
      if (e != cudaSuccess) return e;
    }
    return densities_t<L, S, RT, MODEL, true, SUMS>(c, a, rr, rb, psi, uo);
  } else {
  cudaError_t e = densities_t<L, S, RT, MODEL, false, false>(c, a, rr, rb, psi, jm);
  if (e != cudaSuccess) return e;
  if constexpr (MODEL == LBM_MODEL_SC_MR) {
    auto kern = solid ? diag_mr_kernel<C, true, SUMS> : diag_mr_kernel<C, false, SUMS>;
    const long long units = (long long)((c->p.nx + kMrTX - 1) / kMrTX) * ((c->p.ny + kMrTY - 1) / kMrTY) *
                            ((c->p.nz + kMrZ - 1) / kMrZ);
    kern<<<(int)std::min<long long>(units, c->nblk_diag), kDiagThreads, 0, c->stream>>>(
        rr, rb, reinterpret_cast<const C*>(psi), jm, solid, uo, c->partials, a, c->diag, c->cur);
  } else {
    auto kern = solid ? diag_kernel<L, MODEL, true, SUMS> : diag_kernel<L, MODEL, false, SUMS>;
    const int threads = diag_threads(c, c->N);
    const int blocks = (int)std::min<long long>((c->N + threads - 1) / threads, c->nblk_diag);
    kern<<<blocks, threads, 0, c->stream>>>(rr, rb, psi, jm, solid, uo, c->partials, a, c->diag, c->cur);
  }
  c->launches += 1;
  return cudaGetLastError();
  }
}

// Dispatch on (lattice, storage precision) to an operation templated on <L, S, RT>.
template <template <class, class, class> class F, class... Args>
cudaError_t by_lattice_precision(lbm_ctx* c, Args... args) {
  const bool d3 = c->p.lattice == LBM_D3Q19;
  switch (c->p.precision) {
    case LBM_FP64:
      return d3 ? F<D3Q19, double, double>::run(c, args...) : F<D2Q9, double, double>::run(c, args...);
    case LBM_FP32:
      return d3 ? F<D3Q19, float, float>::run(c, args...) : F<D2Q9, float, float>::run(c, args...);
    case LBM_FP16:
      return d3 ? F<D3Q19, __half, float>::run(c, args...) : F<D2Q9, __half, float>::run(c, args...);
    default:
      return d3 ? F<D3Q19, __nv_bfloat16, float>::run(c, args...) : F<D2Q9, __nv_bfloat16, float>::run(c, args...);
  }
}

template <class L, class S, class RT>
struct InitOp {
  static cudaError_t run(lbm_ctx* c, const double* rr, const double* rb, const double* u) {
    return init_t<L, S, RT>(c, rr, rb, u);
  }
};
template <class L, class S, class RT>
struct RestoreOp {
  static cudaError_t run(lbm_ctx* c, const double* plane, int k, int i, const double* acc) {
    return restore_t<L, S, RT>(c, plane, k, i, acc);
  }
};
template <class L, class S, class RT>
struct ExportOp {
  static cudaError_t run(lbm_ctx* c, double* out, int first, int np) { return export_t<L, S, RT>(c, out, first, np); }
};
template <class L, class S, class RT>
struct GatherOp {
  static cudaError_t run(lbm_ctx* c, void* out, int k, int i) { return gather_t<L, S, RT>(c, out, k, i); }
};
template <class L, class S, class RT>
struct DiagOp {
  static cudaError_t run(lbm_ctx* c, double* rr, double* rb, double* uo, bool totals) {
    // FP64 densities can overflow their sum, which the blow-up check looks at: always summed
    if (totals || std::is_same<S, double>::value) return by_model<true>(c, rr, rb, uo);
    return by_model<false>(c, rr, rb, uo);
  }
  template <bool SUMS>
  static cudaError_t by_model(lbm_ctx* c, double* rr, double* rb, double* uo) {
    switch (c->p.model) {
      case LBM_MODEL_CG:
        return diag_t<L, S, RT, LBM_MODEL_CG, SUMS>(c, rr, rb, uo);
      case LBM_MODEL_SC_MP:
        return diag_t<L, S, RT, LBM_MODEL_SC_MP, SUMS>(c, rr, rb, uo);
      case LBM_MODEL_SC_2C:
        return diag_t<L, S, RT, LBM_MODEL_SC_2C, SUMS>(c, rr, rb, uo);
      default:
        if constexpr (L::D == 3) return diag_t<L, S, RT, LBM_MODEL_SC_MR, SUMS>(c, rr, rb, uo);
        return cudaErrorInvalidValue;
    }
  }
};

}  // namespace

cudaError_t launch_init_eq(lbm_ctx* c, const double* rr, const double* rb, const double* u) {
  c->launches += 1;
  return by_lattice_precision<InitOp>(c, rr, rb, u);
}

cudaError_t launch_wall_words(lbm_ctx* c) {
  const int tiles = (c->p.nx + kPairTX - 1) / kPairTX;
  c->launches += 1;
  wall_words_kernel<<<grid_for((long long)tiles * c->p.ny * c->p.nz, 8, 8192), 256, 0, c->stream>>>(
      c->solid, c->walls, tiles, aux_params(c));
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  c->launches += 1;
  wall_cuts_kernel<<<1, kCutThreads, 0, c->stream>>>(c->walls, c->rows_walled, c->cuts, pair_cuts(c->p), tiles, aux_params(c));
  return cudaGetLastError();
}

// In the largest units that both the elements and the dense buffer's address are multiples of.
cudaError_t launch_pack_rows(lbm_ctx* c, void* dense, void* stored, size_t r0, size_t rows, size_t per, size_t elt,
                             bool to_dense) {
  const size_t units = reinterpret_cast<uintptr_t>(dense) | elt;
  if (units % 4 == 0) return pack_rows_t<unsigned>(c, dense, stored, r0, rows, per, elt, to_dense);
  if (units % 2 == 0) return pack_rows_t<unsigned short>(c, dense, stored, r0, rows, per, elt, to_dense);
  return pack_rows_t<unsigned char>(c, dense, stored, r0, rows, per, elt, to_dense);
}

cudaError_t launch_restore_accumulate(lbm_ctx* c, const double* plane, int k, double* acc, bool first) {
  c->launches += 1;
  restore_acc_kernel<<<grid_for(c->N, 256, 8192), 256, 0, c->stream>>>(plane, acc + (long long)k * c->N, c->N, first);
  return cudaGetLastError();
}

cudaError_t launch_restore_plane(lbm_ctx* c, const double* plane, int k, int i, const double* acc) {
  c->launches += 1;
  return by_lattice_precision<RestoreOp>(c, plane, k, i, acc);
}

cudaError_t launch_export_plane(lbm_ctx* c, double* plane, int k, int i) {
  c->launches += 1;
  return by_lattice_precision<ExportOp>(c, plane, k * c->Q + i, 1);
}

cudaError_t launch_export_all(lbm_ctx* c, double* pops) {
  c->launches += 1;
  return by_lattice_precision<ExportOp>(c, pops, 0, c->K * c->Q);
}

cudaError_t launch_aa_gather_plane(lbm_ctx* c, void* out, int k, int i) {
  c->launches += 1;
  return by_lattice_precision<GatherOp>(c, out, k, i);
}

cudaError_t launch_diagnostics(lbm_ctx* c, double* rho_r, double* rho_b, double* u_out, bool totals) {
  if (!rho_r) rho_r = c->stage;
  if (!rho_b && c->K == 2) rho_b = c->stage + c->N;
  return by_lattice_precision<DiagOp>(c, rho_r, rho_b, u_out, totals);
}

}  // namespace lbm
