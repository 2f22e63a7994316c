// FP64 kernels for the heat-equation model (method of lines, n cells, one control):
//   f_k = (x_{k-1} - 2 x_k + x_{k+1}) / dx^2 - x_k^3,  ghost x_{-1} = u (Dirichlet control),
//   ghost x_n = x_{n-1} (homogeneous Neumann);  0-based cells k = 0..n-1.
// Per-cell derivatives (all other entries are the constant 1/dx^2 of the Laplacian):
//   df_k/dx_k = -2/dx^2 - 3 x_k^2   (k < n-1),   -1/dx^2 - 3 x_k^2   (k = n-1)
//   d2 f_k/dx_k^2 = -6 x_k.
// Row template of component k (the defect of cell k): X cells {k-1, k, k+1} within 0..n-1 on
// each side, plus the control for k = 0, so 6 entries per row except the last cell's 4.
//
// Work decomposition: a CTA covers 32 consecutive nodes (one per lane); in the evaluation and
// H v its one, two, four or eight warps (heat_warps) take the cells in groups of 8, while the
// J + H values, Jv and J^T w run two warps per CTA on units of 16 cells of a tile (at 64 cells four
// times as many CTAs, the same number on every SM).  Row-coupled outputs (defects, Jacobian rows) use tiles that overlap by one node
// (the CTA owns 31 of its 32 nodes); node-local products use disjoint tiles.
// The states of the tile's nodes are staged in shared memory with a padded row (n+1 doubles)
// so that lanes reading different nodes hit different banks; node-major outputs (Hessian
// diagonal, J^T w, H v) are staged the same way and stored with consecutive threads on
// consecutive addresses, except the gradient, stored by each lane for its eight cells.  Component-major outputs (defects, Jacobian rows, Jv)
// are consecutive across lanes and are stored directly or through a per-warp row buffer.
#include <cstring>
#include <type_traits>

#include "follow_on.cuh"
#include "node_kernels.cuh"
#include "ocp_internal.h"

namespace ocpg {

constexpr int HEAT_MAXC = 128;
constexpr int HT_LANES = HEAT_TILE_NODES;
constexpr int HT_WARPS = 8;                          // most warps of a whole-tile CTA
constexpr int HT_THREADS = HT_LANES * HT_WARPS;
// Warps of a whole-tile CTA: one per group of eight cells, 1, 2, 4 or 8, in launches of more than one
// wave of CTAs (with eight for every cell count, seven of eight warps of an 8-cell problem only
// waited: its step at N = 1e5 115 -> 101 us); eight in smaller ones, where all of them stage a tile.
static int heat_warps(int n, int64_t tiles, int num_sms) {
  if (tiles <= (int64_t)5 * num_sms || n > 32) return HT_WARPS;
  return n <= 8 ? 1 : n <= 16 ? 2 : 4;
}

struct HeatArgs {
  const double* __restrict__ x;
  const double* __restrict__ y;
  const double* __restrict__ v;
  const double* __restrict__ v2;  // Jv and J^T w in one launch: the direction of J^T w
  double *f, *c, *g, *jv, *hv, *out;
  double* out2;                   // ... and J^T w
  double* out3;                   // Jv, J^T w and H v in one launch: H v (direction v, multipliers y)
  double* partials;
  unsigned* counter;
  int64_t N, nb, B, E, ntiles, uoff;
  int n, has_final, has_ref, hu;
  double hh, mhh, mhidx2;   // hh, -hh, -hh/dx^2
  double d_in, d_last;      // hh * 2/dx^2, hh * 1/dx^2  (diagonal constant of -hh df_k/dx_k)
  double di_m1, di_p1, dl_m1, dl_p1;  // d_in - 1, d_in + 1, d_last - 1, d_last + 1
  double h3, h6, hidx2;     // 3 hh, 6 hh, hh/dx^2
  double one, mz;           // 1.0 and -0.0 at run time: sums and products are issued as FMAs
  int soft;                 // integer products (soft_mul.cuh): the constants allow them and the launch is large
  double cq_in[HEAT_MAXC + 1], cq_end[HEAT_MAXC + 1];
  double gq_in[HEAT_MAXC + 1], gq_end[HEAT_MAXC + 1];
  double ref[HEAT_MAXC + 1];
  int beside_eval;          // the fused step: the products run beside the evaluation's end
};

// Doubles of the first shared-memory region of k_heat_eval: the staged states (32 rows of n+1),
// and at least the 256 the objective's reductions use when they reuse it.
__host__ __device__ __forceinline__ int heat_xlen(int n) {
  return HT_LANES * (n + 1) > HT_THREADS ? HT_LANES * (n + 1) : HT_THREADS;
}

__device__ __forceinline__ int64_t heat_jbase(const HeatArgs& a, int k) { return a.nb + (int64_t)6 * k * a.N; }

// a + b, a - b, a * b as FMAs against run-time 1 and -0 (same rounding; faster on GB300's FP64 pipe)
__device__ __forceinline__ double hadd(const HeatArgs& a, double u, double v) { return fma(u, a.one, v); }
__device__ __forceinline__ double hsub(const HeatArgs& a, double u, double v) { return fma(-v, a.one, u); }
__device__ __forceinline__ double hmul(const HeatArgs& a, double u, double v) { return fma(u, v, a.mz); }

// The plain products of a cell's work: on the FP64 pipe (ModelConst) or, in large launches, on the
// integer pipes (SoftConst, soft_mul.cuh).  A warp (32 nodes of one cell) decides for each cell,
// from the operands that the cell's inputs give (`ok`); lanes without a node work on ones.  With them
// (64 cells) the step takes 105 us at N = 2e4 and 743 at 2e5 (124 and 914 before), J + H 21.8 (24.8), Jv 23.0
// (27.0), H v 16.9 (19.0), c 25.0 (31.0).
template <bool IP>
__device__ __forceinline__ ModelConst heat_consts(const HeatArgs& a) {
  ModelConst K;
  K.one = a.one; K.mz = a.mz;
  K.soft = IP ? a.soft : 0;
  return K;
}

// Stage the states (and controls) of nodes [r0, r0+nn) into sX[t*(n+1) + k], sX[t*(n+1) + n] = u.
template <int THREADS>
__device__ __forceinline__ void heat_stage(const HeatArgs& a, const double* __restrict__ src, int64_t r0, int nn,
                                           double* sX) {
  const int n = a.n, ld = n + 1;
  const int total = nn * n;
  const double* base = src + (int64_t)n * r0;
  for (int i = threadIdx.x; i < total; i += THREADS) {
    const int t = i / n, k = i - t * n;
    sX[t * ld + k] = __ldg(base + i);
  }
  for (int t = threadIdx.x; t < nn; t += THREADS) sX[t * ld + n] = __ldg(src + a.uoff + r0 + t);
}

// ======================================================================================
// Fused evaluation
// ======================================================================================

// Jacobian rows of cell k for the tile's nodes: the entries on x_k are -1 + dk (left node) and
// +1 + dk (right node), dk = 3 hh x_k^2 + d (d = hh 2/dx^2, or hh/dx^2 at the Neumann end),
// written fma(3 hh, x_k^2, d -+ 1); every other entry is the constant c = -hh/dx^2.  Lane t
// writes the whole row (k, r0 + t): its own left entry, the right entry of lane t+1 (shuffle),
// the constants; entries by position (left X cells, right X cells, then the control's left
// and right entries for k = 0):
//   k = 0:        [jl, c, jr', c, c, c]        interior:  [c, jl, c, c, jr', c]
//   k = n-1:      [c, jl, c, jr']
// A row is 48 (or 32) bytes: three (two) 16-byte stores when the component's rows start on a
// 16-byte boundary, scalar stores otherwise; consecutive lanes write consecutive rows.
__device__ __forceinline__ void heat_jrows(const HeatArgs& a, int k, bool LAST, int t, bool act, int nrows,
                                           int64_t r0, double x2) {
  const double jl = fma(a.h3, x2, LAST ? a.dl_m1 : a.di_m1);
  const double jr = fma(a.h3, x2, LAST ? a.dl_p1 : a.di_p1);
  const double jrn = __shfl_down_sync(0xffffffffu, jr, 1);   // the right node's entry on x_k
  if (!(act && t < nrows)) return;
  const double c = a.mhidx2;
  const int cnt = LAST ? 4 : 6;
  double* rp = a.jv + heat_jbase(a, k) + (r0 + t) * cnt;
  double v[6];
  if (k == 0) { v[0] = jl; v[1] = c; v[2] = jrn; v[3] = c; v[4] = c; v[5] = c; }
  else if (LAST) { v[0] = c; v[1] = jl; v[2] = c; v[3] = jrn; v[4] = c; v[5] = c; }
  else { v[0] = c; v[1] = jl; v[2] = c; v[3] = c; v[4] = jrn; v[5] = c; }
  if ((reinterpret_cast<uintptr_t>(rp) & 15u) == 0) {
    double2* r2 = reinterpret_cast<double2*>(rp);
    r2[0] = make_double2(v[0], v[1]);
    r2[1] = make_double2(v[2], v[3]);
    if (!LAST) r2[2] = make_double2(v[4], v[5]);
  } else {
#pragma unroll
    for (int e = 0; e < 6; ++e)
      if (e < cnt) rp[e] = v[e];
  }
}

// boundary rows X_{0,k} (and X_{N,k}): one constant entry each
__device__ __forceinline__ void heat_jbound(const HeatArgs& a, int k, int64_t j) {
  if (j == 0) a.jv[k] = 1.0;
  if (a.has_final && j == a.N) a.jv[a.n + k] = 1.0;
}

// Hessian diagonal of cell k at node j: 6 hh ybar_k x_k + the objective's sigma w q_k (ybar_k =
// y_{k,j-1} + y_{k,j}, zero beyond the first and last rows)
template <class KC>
__device__ __forceinline__ double heat_hdiag(const HeatArgs& a, const KC& K, int k, bool endp, double xk, double yb) {
  const double ty = fmul(K, a.h6, yb);
  return fma(ty, xk, endp ? a.cq_end[k] : a.cq_in[k]);
}
// y_{k,j-1} + y_{k,j}
__device__ __forceinline__ double heat_ybar(const HeatArgs& a, int k, int64_t j) {
  const double yl = (j >= 1) ? __ldg(a.y + a.nb + (int64_t)k * a.N + j - 1) : 0.0;
  const double yr = (j < a.N) ? __ldg(a.y + a.nb + (int64_t)k * a.N + j) : 0.0;
  return hadd(a, yl, yr);
}

// gradient entry of cell k at node j and its objective term (d = x_k - ref_k)
template <class KC>
__device__ __forceinline__ void heat_grad(const HeatArgs& a, const KC& K, int k, int64_t j, bool endp, double d, bool WG,
                                          bool WF, double obj0, double& objacc) {
  const double gk = fmul_w<MUL_G>(K, endp ? a.gq_end[k] : a.gq_in[k], d);
  if (WF) objacc = fma(gk, d, obj0);
  if (WG) a.g[(int64_t)a.n * j + k] = gk;
}

// tile_sum and finish_tiles for a CTA of W warps, in the order that HT_WARPS warps give (the
// missing ones add nothing to a tile; the tiles' sums go to HT_THREADS places whatever the CTA).
template <int W>
__device__ __forceinline__ double heat_tile_sum(double v, double* red, double one) {
  red[threadIdx.x] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 32) {
    s = red[threadIdx.x];
    #pragma unroll
    for (int i = 1; i < W; ++i) s = fma(red[threadIdx.x + 32 * i], one, s);
    s = warp_sum(s, one);
  }
  return s;
}
template <int W>
__device__ __forceinline__ void heat_finish(const HeatArgs& a, double* red) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = (atomicAdd(a.counter, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // a warp takes the places of HT_WARPS / W warps at once, eight or sixteen loads before the first sum (a lone warp that
  // took them in turn, a load at a time, was the longest part of eval_obj: 5 cells, N = 1e5, 25.0 us so, 16.8 now)
  // (eight warps, also those of launches with few tiles, take one load at a time: each further sum of zeros costs them
  // 64 cycles)
  constexpr int PER = HT_WARPS / W, DEPTH = PER == 1 ? 1 : PER > 4 ? 16 / PER : 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double s[PER] = {};
  for (int64_t i0 = 32 * warp + lane; i0 < a.ntiles; i0 += DEPTH * HT_THREADS) {
    double v[DEPTH][PER];
#pragma unroll
    for (int d = 0; d < DEPTH; ++d)
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        const int64_t i = i0 + HT_THREADS * d + 32 * W * q;
        v[d][q] = i < a.ntiles ? __ldcg(a.partials + i) : 0.0;   // (a sum that starts at +0 is the same with +0 added)
      }
#pragma unroll
    for (int d = 0; d < DEPTH; ++d)
#pragma unroll
      for (int q = 0; q < PER; ++q) s[q] = s[q] + v[d][q];
  }
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const double sum = warp_sum(s[q], 1.0);
    if (lane == 0) red[warp + W * q] = sum;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < HT_WARPS; ++w) s = fma(red[w], 1.0, s);
    *a.f = 0.5 * s;
    *a.counter = 0u;
  }
}

template <unsigned OUT, bool IP, int W>
__global__ void __launch_bounds__(32 * W, (OUT & O_C) ? (W > 1 ? 40 / W : 32) : (W > 1 ? 64 / W : 32)) k_heat_eval(const __grid_constant__ HeatArgs a) {
  constexpr bool CF = OUT & O_F, CC = OUT & O_C, CG = OUT & O_G, CJ = OUT & O_J, CH = OUT & O_H;
  // the full kernel also serves output subsets: NULL outputs are skipped
  const bool WF = CF && a.f, WC = CC && a.c, WG = CG && a.g, WJ = CJ && a.jv, WH = CH && a.hv;
  constexpr int THREADS = 32 * W;
  extern __shared__ __align__(16) double sm[];
  start_follow_on();
  if (OUT == O_ALL && a.beside_eval) let_next_start();   // (the fused step's products: heat_step_overlaps)
  const int n = a.n, ld = n + 1;
  // shared memory: states, then only the staging buffers this variant needs.  The gradient
  // is stored straight from the cell loop (a lane's eight cells of a group fill whole 32-byte
  // sectors) and the objective's reduction reuses the states' buffer once the tile's stores
  // are done: the full evaluation fits five CTAs per SM (one wave of 646 tiles at N = 2e4).
  double* sX = sm;                                             // 32 * ld
  double* sN = sX + heat_xlen(n);                              // Hessian diagonal, 31 * ld
  double* red = sX;                                            // reduction, 256 (after the stores)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double objacc = 0.0;
  const ModelConst K0 = heat_consts<IP>(a);
  constexpr unsigned SOFT = IP ? MUL_ALL : 0u;

  for (int64_t tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
    const int64_t r0 = a.B + tile * (HT_LANES - 1);
    const int64_t own_end = min(r0 + HT_LANES - 1, a.E);
    const int64_t row_end = min(own_end, a.N);
    const int64_t eval_end = row_end + 1;
    const int nn = (int)(eval_end - r0);
    const int nown = (int)(own_end - r0);
    const int nrows = (int)max(row_end - r0, (int64_t)0);
    const int t = lane;
    const int64_t j = r0 + t;
    const bool act = t < nn;
    const bool own = t < nown;
    const bool endp = (j == 0) || (j == a.N);
    heat_stage<THREADS>(a, a.x, r0, nn, sX);
    __syncthreads();
    // ---- Hessian diagonal of every owned (node, cell), elementwise: warps take whole cells
    // (lanes = nodes, the multipliers' rows coalesced), so no load waits inside the cell loop
    // (measured: the separate pass speeds up the full evaluation; J + H alone is faster with
    // the diagonal computed in its cell loop)
    if (CC && WH) {
#pragma unroll 2
      for (int k = warp; k < n; k += W) {
        const double yb = own ? heat_ybar(a, k, j) : 1.0, xk = own ? sX[t * ld + k] : 1.0;
        with_products<SOFT>(K0, true, soft_value(yb), [&](const auto& K) __attribute__((always_inline)) {
          const double h = heat_hdiag(a, K, k, endp, xk, yb);
          if (own) sN[t * ld + k] = h;
        });
      }
    }

    // ---- control entries (warp 0): gradient, objective, Hessian (u,u)
    if (warp == 0 && own) {
      const double u = sX[t * ld + n];
      if (WG || WF) {
        const double d = a.has_ref ? hsub(a, u, a.ref[n]) : u;
        const double gu = hmul(a, endp ? a.gq_end[n] : a.gq_in[n], d);
        if (WG) a.g[a.uoff + j] = gu;
        if (WF) objacc = fma(gu, d, objacc);
      }
      if (WH && a.hu) a.hv[(int64_t)n * (a.N + 1) + j] = endp ? a.cq_end[n] : a.cq_in[n];
    }

    const int ngroups = (n + 7) / 8;
    if constexpr (CC) {
      // One cell k of the tile's nodes; LAST: k is the Neumann end n-1.  The end cell is
      // peeled out of the loop so that its Laplacian and diagonal constant are compile-time
      // choices: a run-time select between two FP64 results issues both on every cell.
      // (xl, xk, xr: the left neighbour (the control for k = 0), the cell, its right neighbour)
      auto cell = [&](const int k, auto last_tag, const double xl, const double xk, const double xr) {
        constexpr bool LAST = decltype(last_tag)::value;
        const double d = ((WG || WF) && a.has_ref) ? hsub(a, xk, a.ref[k]) : xk;
        const double obj0 = objacc;
        const bool ok = !act || (soft_value(xk) & soft_value(d));
        with_products<SOFT>(K0, true, ok, [&](const auto& K) __attribute__((always_inline)) {
          const double x2 = fmul(K, xk, xk);
          if (WJ) heat_jrows(a, k, LAST, t, act, nrows, r0, x2);
          if (WC) {
            // hh f_k = hh (lap / dx^2 - x^3)
            // pa = x + hh f, pb = x - hh f, with hh f = hh/dx^2 lap - hh x^3
            const double lap = LAST ? hsub(a, xl, xk) : fma(-2.0, xk, hadd(a, xl, xr));
            const double x3 = fmul(K, x2, xk);
            const double pa = fma(a.hidx2, lap, fma(a.mhh, x3, xk));
            const double pb = fma(-a.hidx2, lap, fma(a.hh, x3, xk));
            const double nb = __shfl_down_sync(0xffffffffu, pb, 1);
            if (t < nrows) a.c[a.nb + (int64_t)k * a.N + j] = hsub(a, nb, pa);
          }
          if (own && (WG || WF)) heat_grad(a, K, k, j, endp, d, WG, WF, obj0, objacc);
        });
        if (WJ && own) heat_jbound(a, k, j);
        if (WC) {
          if (own && j == 0) a.c[k] = xk;
          if (own && a.has_final && j == a.N) a.c[n + k] = xk;
        }
      };
      auto state = [&](int k) { return act ? sX[t * ld + k] : 1.0; };
      for (int gi = warp; gi < ngroups; gi += W) {
        const int k0 = gi * 8, k1 = min(k0 + 8, n);
        const int kin = min(k1, n - 1);  // interior cells of the group: k0 .. kin-1
        double xl = state(k0 == 0 ? n : k0 - 1), xk = state(k0);
#pragma unroll 1
        for (int k = k0; k < kin; ++k) {
          const double xr = state(k + 1);
          cell(k, std::false_type{}, xl, xk, xr);
          xl = xk;
          xk = xr;
        }
        if (k1 == n) cell(n - 1, std::true_type{}, xl, xk, xk);
      }
    } else {
      // without the constraints one loop body for every cell (smaller and measured faster)
      for (int gi = warp; gi < ngroups; gi += W) {
        const int k0 = gi * 8, k1 = min(k0 + 8, n);
        for (int k = k0; k < k1; ++k) {
          const bool last = (k == n - 1);
          const double xk = act ? sX[t * ld + k] : 1.0;
          if (WJ) heat_jrows(a, k, last, t, act, nrows, r0, hmul(a, xk, xk));
          if (WJ && own) heat_jbound(a, k, j);
          if (own && WH) sN[t * ld + k] = heat_hdiag(a, K0, k, endp, xk, heat_ybar(a, k, j));
          if (own && (WG || WF)) heat_grad(a, K0, k, j, endp, a.has_ref ? hsub(a, xk, a.ref[k]) : xk, WG, WF, objacc, objacc);
        }
      }
    }
    __syncthreads();
    if (WH) {
      const int total = nown * n;
      double* dst = a.hv + (int64_t)n * r0;
      for (int i = threadIdx.x; i < total; i += THREADS) {
        const int tt = i / n, k = i - tt * n;
        dst[i] = sN[tt * ld + k];
      }
    }
    if (WF) {
      __syncthreads();  // red is the states' buffer, read by the loop above
      const double ts = heat_tile_sum<W>(objacc, red, a.one);
      if (threadIdx.x == 0) a.partials[tile] = ts;
      objacc = 0.0;
    }
    __syncthreads();
  }
  if (WF) heat_finish<W>(a, red);
}

// ======================================================================================
// Jacobian and Hessian values alone (no objective, defects or gradient).  Each entry depends on
// its own cell only, so a CTA of two warps takes one tile's 32 nodes (31 owned) and 16 of its
// cells, eight per warp: a problem splits into ceil(n/16) times as many CTAs as tiles, spread
// evenly over the SMs (at N = 2e4 and 64 cells: 2584 CTAs, 17 per SM in one wave, where the
// 646 CTAs of whole tiles put 4 on some SMs and 5 on others).  Every entry is computed by the
// same expressions as in k_heat_eval, so the values are bit-identical.
// ======================================================================================
constexpr int HJ_CELLS = 16, HJ_WARPS = 2, HJ_THREADS = 32 * HJ_WARPS, HJ_LD = HJ_CELLS + 1;

template <unsigned OUT, bool IP>
__global__ void __launch_bounds__(HJ_THREADS, 18) k_heat_jh(const __grid_constant__ HeatArgs a, int cgroups) {
  constexpr bool CJ = OUT & O_J, CH = OUT & O_H;
  const bool WJ = CJ && a.jv, WH = CH && a.hv;
  // the states of the unit's cells, node-major in padded rows, overwritten in place by the
  // Hessian diagonal; the multipliers y_{k, r0-1 .. r0+30} of its cells, cell-major
  __shared__ double sX[HT_LANES * HJ_LD];
  __shared__ double sY[HJ_CELLS * HT_LANES];
  const int n = a.n;
  const int t = threadIdx.x & 31, warp = threadIdx.x >> 5;
  start_follow_on();
  const ModelConst K0 = heat_consts<IP>(a);
  constexpr unsigned SOFT = IP ? MUL_ALL : 0u;
  const int64_t units = a.ntiles * cgroups;
  for (int64_t unit = blockIdx.x; unit < units; unit += gridDim.x) {
    const int64_t tile = unit / cgroups;
    const int c0 = (int)(unit - tile * cgroups) * HJ_CELLS;
    const int nc = min(HJ_CELLS, n - c0);
    const int64_t r0 = a.B + tile * (HT_LANES - 1);
    const int64_t own_end = min(r0 + HT_LANES - 1, a.E);
    const int64_t row_end = min(own_end, a.N);
    const int nn = (int)(row_end + 1 - r0);
    const int nown = (int)(own_end - r0);
    const int nrows = (int)max(row_end - r0, (int64_t)0);
    const int64_t j = r0 + t;
    const bool act = t < nn;
    const bool own = t < nown;
    const bool endp = (j == 0) || (j == a.N);
    for (int i = threadIdx.x; i < nn * nc; i += HJ_THREADS) {
      const int tt = i / nc, kk = i - tt * nc;
      sX[tt * HJ_LD + kk] = __ldg(a.x + (int64_t)n * (r0 + tt) + c0 + kk);
    }
    if (WH) {
      // rows outside [0, N) stage as zero: y_{k,j-1} for j = 0 and y_{k,j} for j = N
      for (int i = threadIdx.x; i < nc * HT_LANES; i += HJ_THREADS) {
        const int kk = i / HT_LANES;
        const int64_t jj = r0 - 1 + (i - kk * HT_LANES);
        sY[i] = (jj >= 0 && jj < a.N) ? __ldg(a.y + a.nb + (int64_t)(c0 + kk) * a.N + jj) : 0.0;
      }
    }
    __syncthreads();
    // the control's Hessian entry (u, u), by the unit of the first cells
    if (c0 == 0 && warp == 0 && own && WH && a.hu) a.hv[(int64_t)n * (a.N + 1) + j] = endp ? a.cq_end[n] : a.cq_in[n];
    const int k1 = min(8 * warp + 8, nc);
    for (int kk = 8 * warp; kk < k1; ++kk) {
      const int k = c0 + kk;
      const double xk = act ? sX[t * HJ_LD + kk] : 1.0;
      // an owned lane t <= 30 reads the multipliers of rows j-1 and j at positions t and t+1
      const double yb = (own && WH) ? hadd(a, sY[kk * HT_LANES + t], sY[kk * HT_LANES + t + 1]) : 1.0;
      with_products<SOFT>(K0, true, (!WJ || soft_value(xk)) & soft_value(yb), [&](const auto& K) __attribute__((always_inline)) {
        if (WJ) heat_jrows(a, k, k == n - 1, t, act, nrows, r0, fmul(K, xk, xk));
        if (WH) {
          const double h = heat_hdiag(a, K, k, endp, xk, yb);
          if (own) sX[t * HJ_LD + kk] = h;
        }
      });
      if (WJ && own) heat_jbound(a, k, j);
    }
    __syncthreads();
    if (WH) {
      double* dst = a.hv + (int64_t)n * r0 + c0;
      for (int i = threadIdx.x; i < nown * nc; i += HJ_THREADS) {
        const int tt = i / nc, kk = i - tt * nc;
        dst[(int64_t)n * tt + kk] = sX[tt * HJ_LD + kk];
      }
    }
    __syncthreads();
  }
}

// ======================================================================================
// H v (node-local):    out_a = (2 sigma w q_a + 6 hh ybar_a x_a) v_a,  out_u = 2 sigma w r v_u
// (whole tiles of 32 nodes and their 64 cells: measured faster than the 16-cell units of the
// other products, 23.3 against 24.3 us at N = 2e4, 39.4 against 41.1 at N = 5e4); at most 51
// registers: five CTAs per SM, one wave of 626 tiles at N = 2e4 (measured faster)
// ======================================================================================
template <bool IP, int W>
__global__ void __launch_bounds__(32 * W, W > 1 ? 40 / W : 32) k_heat_hprod(const __grid_constant__ HeatArgs a) {
  constexpr int THREADS = 32 * W;
  extern __shared__ __align__(16) double sm[];
  const int n = a.n, ld = n + 1;
  double* sX = sm;
  double* sV = sX + HT_LANES * ld;  // the direction
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  start_follow_on();
  const ModelConst K0 = heat_consts<IP>(a);
  constexpr unsigned SOFT = IP ? MUL_ALL : 0u;
  for (int64_t tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
    const int64_t r0 = tile * HT_LANES;
    const int nn = (int)min((int64_t)HT_LANES, a.N + 1 - r0);
    const int t = lane;
    const int64_t j = r0 + t;
    const bool act = t < nn;
    const bool endp = (j == 0) || (j == a.N);
    heat_stage<THREADS>(a, a.x, r0, nn, sX);
    heat_stage<THREADS>(a, a.v, r0, nn, sV);
    __syncthreads();
    const int ngroups = (n + 7) / 8;
    for (int gi = warp; gi < ngroups; gi += W) {
      const int k0 = gi * 8, k1 = min(k0 + 8, n);
      // elementwise: the group's multiplier rows are loaded before any arithmetic needs them
      double yl[8], yr[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int k = k0 + q;
        yl[q] = (act && k < k1 && j >= 1) ? __ldg(a.y + a.nb + (int64_t)k * a.N + j - 1) : 0.0;
        yr[q] = (act && k < k1 && j < a.N) ? __ldg(a.y + a.nb + (int64_t)k * a.N + j) : 0.0;
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int k = k0 + q;
        if (k >= k1) continue;   // (warp-uniform)
        const double xk = act ? sX[t * ld + k] : 1.0, vk = act ? sV[t * ld + k] : 1.0;
        const double yb = act ? hadd(a, yl[q], yr[q]) : 1.0;
        with_products<SOFT>(K0, true, soft_value(vk) & soft_value(yb), [&](const auto& K) __attribute__((always_inline)) {
          const double h = fmul(K, heat_hdiag(a, K, k, endp, xk, yb), vk);
          if (act) sX[t * ld + k] = h;   // in place: x no longer needed for cell k
        });
      }
    }
    if (warp == 0 && act) {
      const double cu = a.hu ? (endp ? a.cq_end[n] : a.cq_in[n]) : 0.0;
      sX[t * ld + n] = hmul(a, cu, sV[t * ld + n]);
    }
    __syncthreads();
    {
      const int total = nn * n;
      double* dst = a.out + (int64_t)n * r0;
      for (int i = threadIdx.x; i < total; i += THREADS) {
        const int tt = i / n, k = i - tt * n;
        dst[i] = sX[tt * ld + k];
      }
      for (int tt = threadIdx.x; tt < nn; tt += THREADS) a.out[a.uoff + r0 + tt] = sX[tt * ld + n];
    }
    __syncthreads();
  }
}

// ======================================================================================
// Jv and J^T w on units of one tile and 16 cells (two warps of 8 cells each, as in k_heat_jh),
// so that the work spreads evenly over the SMs (at N = 2e4: Jv 35.0 -> 31.4 us, J^T w 31.8 ->
// 28.9 us, against whole tiles of 32 nodes and 64 cells).
//   Jv:     p_k(j) = -hh grad f_k(z_j) . v_{z_j};
//           row (k,j) = (p_k(j) - v_{X_j,k}) + (p_k(j+1) + v_{X_{j+1},k})
//           on tiles overlapping by one node (its rows couple nodes j and j+1); the direction of
//           cells c0-1 .. c0+16 is staged, the control's in place of cell -1.
//   J^T w:  out_a = (w_{a,j-1} - w_{a,j}) + wbar_a dd_a - hh/dx^2 (wbar_{a-1} + wbar_{a+1}),
//           out_u = -hh/dx^2 wbar_0  (dd_a = -hh df_a/dx_a), node-local on disjoint tiles; the
//           result is staged and stored node by node in runs of the unit's cells.
//   All three (the heat model's fused step): the products of the same unit in one launch, on the
//           tiles of Jv; J^T w for the owned nodes, its result written over the staged states
//           (where Jv leaves -hh df_a/dx_a, which J^T w needs of them); H v of the owned nodes, each
//           entry formed in Jv's cell loop from the same state and direction values and stored by
//           its lane.  Each entry by the same expressions as the separate launches.
// ======================================================================================
enum : int { HP_JPROD = 0, HP_JTPROD = 1, HP_ALL3 = 3 };
constexpr int HP_LDV = HJ_CELLS + 3;  // padded row of the staged direction (or J^T w result)

template <int KIND, bool IP>
__global__ void __launch_bounds__(HJ_THREADS, 18) k_heat_prod_unit(const __grid_constant__ HeatArgs a, int cgroups) {
  constexpr bool ALL3 = KIND == HP_ALL3, JP = KIND == HP_JPROD || ALL3, JT = KIND == HP_JTPROD || ALL3;
  constexpr int LDV = JP ? HP_LDV : HJ_LD;
  __shared__ double sX[HT_LANES * HJ_LD];  // states of the unit's cells (both: then the J^T w result)
  __shared__ double sV[HT_LANES * LDV];    // Jv: the direction; J^T w alone: the result
  double* const sO = ALL3 ? sX : sV;       // the J^T w result (row length HJ_LD either way)
  const double* const wv = ALL3 ? a.v2 : a.v;
  double* const wout = ALL3 ? a.out2 : a.out;
  const int n = a.n;
  const int t = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (!ALL3 || !a.beside_eval) start_follow_on();
  const ModelConst K0 = heat_consts<IP>(a);
  constexpr unsigned SOFT = IP ? MUL_ALL : 0u;
  const int64_t units = a.ntiles * cgroups;
  for (int64_t unit = blockIdx.x; unit < units; unit += gridDim.x) {
    const int64_t tile = unit / cgroups;
    const int c0 = (int)(unit - tile * cgroups) * HJ_CELLS;
    const int nc = min(HJ_CELLS, n - c0);
    const int kb = 8 * warp, ke = min(8 * warp + 8, nc);  // this warp's cells c0 + [kb, ke)
    int64_t r0;
    int nn, nrows = 0, nown = 0;
    bool bnd = false;
    if (JP) {
      r0 = tile * (HT_LANES - 1);
      const int64_t own_end = min(r0 + HT_LANES - 1, a.N + 1);
      const int64_t row_end = min(own_end, a.N);
      nn = (int)(row_end + 1 - r0);
      nrows = (int)max(row_end - r0, (int64_t)0);
      nown = (int)(own_end - r0);
    } else {
      r0 = tile * HT_LANES;
      nn = (int)min((int64_t)HT_LANES, a.N + 1 - r0);
      bnd = (tile == 0) || (r0 + HT_LANES > a.N);
    }
    if (ALL3) bnd = (r0 == 0) || (r0 + nown == a.N + 1);  // the tile holds node 0 or node N
    const int64_t j = r0 + t;
    const bool act = t < nn;
    const bool jown = ALL3 ? (t < nown) : act;  // J^T w: the owned nodes
    for (int i = threadIdx.x; i < nn * nc; i += HJ_THREADS) {
      const int tt = i / nc, kk = i - tt * nc;
      sX[tt * HJ_LD + kk] = __ldg(a.x + (int64_t)n * (r0 + tt) + c0 + kk);
    }
    if (JP) {
      const int w = nc + 2;  // cells c0-1 .. c0+nc at positions 0 .. nc+1
      for (int i = threadIdx.x; i < nn * w; i += HJ_THREADS) {
        const int tt = i / w, e = i - tt * w, k = c0 - 1 + e;
        double val = 0.0;
        if (k < 0) val = __ldg(a.v + a.uoff + r0 + tt);
        else if (k < n) val = __ldg(a.v + (int64_t)n * (r0 + tt) + k);
        sV[tt * HP_LDV + e] = val;
      }
    }
    __syncthreads();
    if (JP) {
      const bool endp = (j == 0) || (j == a.N);
      if (ALL3 && c0 == 0 && warp == 0 && jown) {  // H v, the control: 2 sigma w r v_u
        const double cu = a.hu ? (endp ? a.cq_end[n] : a.cq_in[n]) : 0.0;
        a.out3[a.uoff + j] = hmul(a, cu, sV[t * HP_LDV]);
      }
      for (int kk = kb; kk < ke; ++kk) {
        const int k = c0 + kk;
        const bool last = (k == n - 1);
        const double xk = act ? sX[t * HJ_LD + kk] : 1.0, vk = act ? sV[t * HP_LDV + kk + 1] : 1.0;
        const double yb = (ALL3 && jown) ? heat_ybar(a, k, j) : 1.0;
        // the left neighbour's entry (the control's for k = 0), plus the right one's
        const double vl = sV[t * HP_LDV + kk];
        const double nsum = last ? vl : hadd(a, vl, sV[t * HP_LDV + kk + 2]);
        with_products<SOFT>(K0, true, soft_value(xk) & soft_value(vk) & soft_value(yb), [&](const auto& K) __attribute__((always_inline)) {
          if (ALL3) {  // H v: (2 sigma w q_k + 6 hh ybar_k x_k) v_k
            const double h = fmul(K, heat_hdiag(a, K, k, endp, xk, yb), vk);
            if (jown) a.out3[(int64_t)n * j + k] = h;
          }
          const double dk = fma(a.h3, fmul(K, xk, xk), last ? a.d_last : a.d_in);
          if (JT) sX[t * HJ_LD + kk] = dk;   // J^T w needs of the state only this, in this thread
          const double p = fma(a.mhidx2, nsum, fmul(K, dk, vk));
          const double right = __shfl_down_sync(0xffffffffu, hadd(a, p, vk), 1);
          if (t < nrows) a.out[a.nb + (int64_t)k * a.N + j] = hadd(a, hsub(a, p, vk), right);
        });
        if (act && j == 0) a.out[k] = vk;
        if (act && a.has_final && j == a.N && t < nown) a.out[n + k] = vk;
      }
    }
    if (JT && kb < ke) {
      // wbar of cells k0-1 .. k1 (clamped), rolling window
      auto wbar = [&](int k, double& wl, double& wr) {
        const double* row = wv + a.nb + (int64_t)k * a.N;
        wl = (j >= 1) ? __ldg(row + j - 1) : 0.0;
        wr = (j < a.N) ? __ldg(row + j) : 0.0;
      };
      const int k0 = c0 + kb, k1 = c0 + ke;
      double wbm = 0.0, wbc = 0.0, wbp = 0.0, wlc = 0.0, wrc = 0.0;
      if (jown) {
        if (k0 > 0) { double l2, r2; wbar(k0 - 1, l2, r2); wbm = hadd(a, l2, r2); }
        wbar(k0, wlc, wrc);
        wbc = hadd(a, wlc, wrc);
        if (k0 == 0) wout[a.uoff + j] = hmul(a, a.mhidx2, wbc);  // control column: -hh/dx^2 wbar_0
      }
      for (int k = k0; k < k1; ++k) {
        if (jown) {
          double wlp = 0.0, wrp = 0.0;
          if (k + 1 < n) { wbar(k + 1, wlp, wrp); wbp = hadd(a, wlp, wrp); } else wbp = 0.0;
          double dk = sX[t * HJ_LD + (k - c0)];
          if (!JP) dk = fma(a.h3, hmul(a, dk, dk), k == n - 1 ? a.d_last : a.d_in);   // (the state until here)
          double s = fma(wbc, dk, hsub(a, wlc, wrc));
          s = fma(a.mhidx2, hadd(a, wbm, wbp), s);
          if (bnd) {  // only the CTAs holding node 0 or node N (uniform branch)
            if (j == 0) s = hadd(a, s, __ldg(wv + k));
            if (a.has_final && j == a.N) s = hadd(a, s, __ldg(wv + n + k));
          }
          sO[t * HJ_LD + (k - c0)] = s;
          wbm = wbc; wbc = wbp; wlc = wlp; wrc = wrp;
        }
      }
    }
    __syncthreads();
    if (JT) {
      // node-major results of the unit's cells, in runs of nc per node
      double* dst = wout + (int64_t)n * r0 + c0;
      const int nst = ALL3 ? nown : nn;
      for (int i = threadIdx.x; i < nst * nc; i += HJ_THREADS) {
        const int tt = i / nc, kk = i - tt * nc;
        dst[(int64_t)n * tt + kk] = sO[tt * HJ_LD + kk];
      }
    }
    __syncthreads();
  }
  if (ALL3 && a.beside_eval) wait_for_previous();   // (they read nothing that the evaluation writes: heat_step_overlaps)
}

// ======================================================================================
// Host side
// ======================================================================================
static void heat_fill(const ocp* h, double sigma, HeatArgs& a) {
  memset(&a, 0, sizeof(a));
  const int n = h->nx;
  const double idx2 = (double)n * (double)n;  // 1/dx^2 with dx = 1/n
  a.N = h->N;
  a.nb = h->pat.nb;
  a.uoff = (int64_t)n * (h->N + 1);
  a.n = n;
  a.has_final = h->has_final;
  a.has_ref = h->has_ref;
  a.hu = h->pat.hu;
  a.hh = h->hh;
  a.mhh = -h->hh;
  a.mhidx2 = -h->hh * idx2;
  a.hidx2 = h->hh * idx2;
  a.d_in = h->hh * (2.0 * idx2);
  a.d_last = h->hh * idx2;
  a.di_m1 = a.d_in - 1.0;
  a.di_p1 = a.d_in + 1.0;
  a.dl_m1 = a.d_last - 1.0;
  a.dl_p1 = a.d_last + 1.0;
  a.h3 = 3.0 * h->hh;
  a.h6 = 6.0 * h->hh;
  a.one = 1.0;
  a.mz = -0.0;
  for (int v = 0; v <= n; ++v) {
    const double w = v < n ? h->q[v] : h->r[0];
    a.gq_in[v] = 2.0 * h->h * w;
    a.gq_end[v] = h->h * w;
    a.cq_in[v] = sigma * (2.0 * h->h * w);
    a.cq_end[v] = sigma * (h->h * w);
    a.ref[v] = v < n ? h->xref[v] : h->uref[0];
  }
  a.partials = h->d_partials;
  a.counter = h->d_counter;
  // (a thread takes eight cells of a node, so a node counts n / 8 times)
  auto fits = [](double v) { return v >= 0x1p-64 && v < 0x1p64; };
  a.soft = large_launch((h->N + 1) * (int64_t)n / 8, h->num_sms) && fits(a.h6) && finite_cost(h);
}

// Calls fn with the number of warps as a compile-time constant.
template <class Fn>
static cudaError_t with_warps(int w, Fn&& fn) {
  switch (w) {
    case 1: return fn(std::integral_constant<int, 1>{});
    case 2: return fn(std::integral_constant<int, 2>{});
    case 4: return fn(std::integral_constant<int, 4>{});
    default: return fn(std::integral_constant<int, HT_WARPS>{});
  }
}

constexpr int HEAT_STEP_CARVEOUT = 81;   // percent of 228 KB: 18 CTAs of the products, 9 KB and 1 KB of the system's each

template <unsigned OUT>
static ocp_status heat_eval_t(ocp* h, const EvalCall& c, cudaStream_t s) {
  HeatArgs a;
  heat_fill(h, c.sigma, a);
  a.x = c.x; a.y = c.y; a.f = c.f; a.c = c.c; a.g = c.g; a.jv = c.jv; a.hv = c.hv;
  a.beside_eval = c.products_beside;
  a.B = c.B; a.E = c.E;
  const int64_t nodes = c.E - c.B;
  a.ntiles = (nodes + (HT_LANES - 2)) / (HT_LANES - 1);
  if (a.ntiles < 1) a.ntiles = 1;
  if (a.ntiles > h->max_partials) return set_err(h, OCP_EDIM, "too many tiles for the reduction scratch");
  const int ld = h->nx + 1;
  const size_t smem = sizeof(double) * ((size_t)heat_xlen(h->nx) + ((OUT & O_H) ? (HT_LANES - 1) * ld : 0));
  constexpr bool MUL = (OUT & O_C) != 0;   // integer products (the other instances are bound by other things)
  auto go = [&](auto w) -> cudaError_t {
    constexpr int W = decltype(w)::value;
    auto kern = (MUL && a.soft) ? k_heat_eval<OUT, MUL, W> : k_heat_eval<OUT, false, W>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if constexpr (OUT == O_ALL) {
      // An SM splits its memory between L1 and shared memory for the kernel that it runs, and takes CTAs that
      // need another split only when it is empty.  The products' CTAs ask for 18 x 10 KB, and beside an
      // evaluation of fewer than 64 cells, whose five CTAs fit in a split of 164 KB, they all went to the SMs
      // without one (16 cells, N = 4300: 36.9 us, 27.8 in order, 20.5 with their split).
      const bool ask = c.products_beside && a.ntiles <= h->num_sms && 5 * (smem + 1024) <= 164 * 1024;
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 ask ? HEAT_STEP_CARVEOUT : cudaSharedmemCarveoutDefault);
    }
    if (e != cudaSuccess) return e;
    return launch(!c.products_beside, kern, occupancy_grid(h, (const void*)kern, 32 * W, smem, a.ntiles), 32 * W, smem, s, a);
  };
  return cuda_err(h, with_warps(heat_warps(h->nx, a.ntiles, h->num_sms), go), "k_heat_eval launch");
}

// Jacobian and / or Hessian values alone: units of one tile and 16 cells (k_heat_jh)
template <unsigned OUT>
static ocp_status heat_jh_t(ocp* h, const EvalCall& c, cudaStream_t s) {
  HeatArgs a;
  heat_fill(h, c.sigma, a);
  a.x = c.x; a.y = c.y; a.jv = c.jv; a.hv = c.hv;
  a.B = c.B; a.E = c.E;
  const int64_t nodes = c.E - c.B;
  a.ntiles = (nodes + (HT_LANES - 2)) / (HT_LANES - 1);
  if (a.ntiles < 1) a.ntiles = 1;
  const int cgroups = (h->nx + HJ_CELLS - 1) / HJ_CELLS;
  auto kern = a.soft ? k_heat_jh<OUT, true> : k_heat_jh<OUT, false>;
  const int grid = occupancy_grid(h, (const void*)kern, HJ_THREADS, 0, a.ntiles * cgroups);
  if (grid <= 0) return set_err(h, OCP_ECUDA, "occupancy query failed");
  return cuda_err(h, launch(true, kern, grid, HJ_THREADS, 0, s, a, cgroups), "k_heat_jh launch");
}

ocp_status heat_eval(ocp* h, unsigned out, const EvalCall& c, cudaStream_t s) {
  switch (out) {
    case O_F: return heat_eval_t<O_F>(h, c, s);
    case O_C: return heat_eval_t<O_C>(h, c, s);
    case O_G: return heat_eval_t<O_G>(h, c, s);
    case O_J: return heat_jh_t<O_J>(h, c, s);
    case O_H: return heat_jh_t<O_H>(h, c, s);
    case O_J | O_H: return heat_jh_t<O_J | O_H>(h, c, s);
    default: return heat_eval_t<O_ALL>(h, c, s);
  }
}

// Whether the fused step's products may run beside the evaluation's last CTAs.  They read nothing
// that the evaluation writes and write nothing that it touches, unless the caller's arrays share
// memory; then (and with path or boundary terms, whose launch comes between) they come after it.
// With at most one evaluation CTA per SM they always do: heat_eval_t has those SMs' memory split so that the
// products' CTAs find room on all of them (2 to 128 cells, N = 60 to 4650, 119 sizes: 0.48 to 0.89 of
// the time in order; 64 cells, N = 3000: 33.6 and 22.7 us).  With more, FP64 work is bound by the fullest
// SM, and the products' CTAs crowd some of them (14 cells, N = 9041: 28.6 us in order, 59.6 beside each other; 37
// cells, N = 20000: 63.0 and 69.8; but 64 cells, N = 1e4: 57.2 and 46.8), unless they fill the chip in any
// case, HJ_CTAS on every SM or nearly so: at 16 to 24 per SM 0.76 to 1.05 of the time in order (64 cells,
// N = 2e4, 17 per SM: 92.9 us in order, 79.3 so; 128 cells, N = 1e4: 103.4 and 93.6; 33 cells, N = 28000: 83.0 and
// 86.1), at 14 and 15 0.88 to 1.07 (50 cells, N = 16500).
constexpr int HJ_CTAS = 18;   // (the register cap of k_heat_prod_unit)
bool heat_step_overlaps(const ocp* h, const EvalCall& e, const double* vn, const double* vm, const double* Jv,
                        const double* Jtv, const double* Hv) {
  const Pattern& P = h->pat;
  if (P.npath > 0 || P.nbin > 0 || h->has_bol) return false;
  const int64_t tiles = (h->N + 1 + (HT_LANES - 2)) / (HT_LANES - 1), ctas = tiles * ((h->nx + HJ_CELLS - 1) / HJ_CELLS);
  if (tiles > h->num_sms && ctas < (int64_t)(HJ_CTAS - 2) * h->num_sms) return false;
  struct Range { const double* p; int64_t n; };
  const Range eval_in[] = {{e.x, P.n}, {e.y, P.m}};
  const Range eval_out[] = {{e.f, 1}, {e.c, P.m}, {e.g, P.n}, {e.jv, P.nnzj}, {e.hv, P.nnzh}};
  const Range prod_in[] = {{e.x, P.n}, {e.y, P.m}, {vn, P.n}, {vm, P.m}};
  const Range prod_out[] = {{Jv, P.m}, {Jtv, P.n}, {Hv, P.n}};
  auto apart = [](const Range& a, const Range& b) { return a.p + a.n <= b.p || b.p + b.n <= a.p; };
  bool ok = true;
  for (const Range& o : eval_out) {
    for (const Range& r : prod_in) ok &= apart(o, r);
    for (const Range& w : prod_out) ok &= apart(o, w);
  }
  for (const Range& w : prod_out)
    for (const Range& r : eval_in) ok &= apart(w, r);
  return ok;
}

// Jv (jp.v -> jp.out), J^T w (jt.v -> jt.out) and H v (hp.y, hp.sigma, the direction jp.v ->
// hp.out) of the heat model in one launch (the fused step); after_eval: the launch before it on the
// stream is the evaluation's kernel, and the two may overlap
ocp_status heat_prod3(ocp* h, const ProdCall& jp, const ProdCall& jt, const ProdCall& hp, bool after_eval, cudaStream_t s) {
  HeatArgs a;
  heat_fill(h, hp.sigma, a);
  a.x = jp.x; a.v = jp.v; a.out = jp.out; a.v2 = jt.v; a.out2 = jt.out;
  a.y = hp.y; a.out3 = hp.out;
  const int cgroups = (h->nx + HJ_CELLS - 1) / HJ_CELLS;
  a.ntiles = (h->N + 1 + (HT_LANES - 2)) / (HT_LANES - 1);
  auto k = a.soft ? k_heat_prod_unit<HP_ALL3, true> : k_heat_prod_unit<HP_ALL3, false>;
  const int grid = occupancy_grid(h, (const void*)k, HJ_THREADS, 0, a.ntiles * cgroups);
  if (grid <= 0) return set_err(h, OCP_ECUDA, "occupancy query failed");
  a.beside_eval = after_eval;
  return cuda_err(h, launch(true, k, grid, HJ_THREADS, 0, s, a, cgroups), "heat product launch");
}

ocp_status heat_prod(ocp* h, const ProdCall& c, cudaStream_t s) {
  HeatArgs a;
  heat_fill(h, c.sigma, a);
  a.x = c.x; a.y = c.y; a.v = c.v; a.out = c.out;
  if (c.kind == P_HPROD) {
    a.ntiles = (h->N + 1 + HT_LANES - 1) / HT_LANES;
    const size_t smem = sizeof(double) * (size_t)HT_LANES * (h->nx + 1) * 2;  // states and direction
    auto go = [&](auto w) -> cudaError_t {
      constexpr int W = decltype(w)::value;
      auto k = a.soft ? k_heat_hprod<true, W> : k_heat_hprod<false, W>;
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      return launch(true, k, occupancy_grid(h, (const void*)k, 32 * W, smem, a.ntiles), 32 * W, smem, s, a);
    };
    return cuda_err(h, with_warps(heat_warps(h->nx, a.ntiles, h->num_sms), go), "heat product launch");
  }
  const int cgroups = (h->nx + HJ_CELLS - 1) / HJ_CELLS;
  if (c.kind == P_JPROD) a.ntiles = (h->N + 1 + (HT_LANES - 2)) / (HT_LANES - 1);
  else a.ntiles = (h->N + 1 + HT_LANES - 1) / HT_LANES;
  // (J^T w has one plain product per cell, left to the FP64 pipe)
  auto k = c.kind == P_JTPROD ? k_heat_prod_unit<HP_JTPROD, false>
                              : a.soft ? k_heat_prod_unit<HP_JPROD, true> : k_heat_prod_unit<HP_JPROD, false>;
  const int grid = occupancy_grid(h, (const void*)k, HJ_THREADS, 0, a.ntiles * cgroups);
  if (grid <= 0) return set_err(h, OCP_ECUDA, "occupancy query failed");
  return cuda_err(h, launch(true, k, grid, HJ_THREADS, 0, s, a, cgroups), "heat product launch");
}

}  // namespace ocpg
