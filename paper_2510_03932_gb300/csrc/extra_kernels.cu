// The terms beside the transcription proper, all in the quadratic-plus-linear family
//     sum_v [ a_v (z_v - b_v)^2 + l_v z_v ]      (derivatives 2 a_v (z_v - b_v) + l_v and 2 a_v):
//   path inequalities (paper Sec. 3: c(X_i, U_i) <= 0 at every node with a control)
//       c_p(z) = sum_v [...] - r_p,  rows nb + nx N + p nun + i after the defect rows;
//   boundary inequalities (paper Sec. 3: b(X_0, X_N) <= 0)
//       b_q(z) = sum_v [...] - r_q,  z = (X_0, X_N),  rows nb + nx N + npath nun + q;
//   boundary cost (paper Sec. 3, the Bolza term)  g(X_0, X_N) = sum_v [...], added to F.
//
// One launch after the model's kernel of the same call on the same stream writes the rows of c, J
// and J v and adds the terms to f, the gradient, the Hessian diagonals, J^T w and H v.  Each entry's
// additions keep one order: the path rows in order, the boundary rows in order, the boundary cost.
//   Path rows: one thread per node (a node's entries belong to it alone).
//   Boundary terms: block 0, when there are any.  They couple only the nodes 0 and N, so this
//   block also does those two nodes' path rows first; then its threads take a term each (the
//   rows' sums run in term order over terms staged in shared memory) and a variable each (its
//   additions run over the rows in order, then the boundary cost).
// (A kernel per kind and output, the boundary ones on a single thread, took six launches of 4 to
// 5.5 us each for the boundary terms of an evaluation: the quadrotor's at N = 33333, with
// path rows, 40 of its 68 us.)
//
// What bounds the path rows is the FP64 pipe: a plain term costs six FP64 instructions for c alone.  Most
// terms are squared only or linear only, the same at every node, so each kind skips what its
// zero coefficient would multiply; a warp with a value that is infinite, NaN or beyond 2^900 (0
// times what it gives is NaN) evaluates the full form.
#include <algorithm>
#include <cstring>

#include "follow_on.cuh"
#include "ocp_internal.h"

namespace ocpg {

constexpr int EX_THREADS = 256;
constexpr int EX_CHUNK = 512;   // boundary terms staged at once

struct ExtraArgs {
  const double* __restrict__ x;
  const double* __restrict__ y;
  const double* __restrict__ vn;
  const double* __restrict__ vm;
  double *f, *g, *c, *jv, *hv, *ojv, *ojtv, *ohv;
  // path rows: terms poff[p] .. poff[p+1]-1 of row p with variable pv and a, b, l, 2a (4 per
  // term), then r (npath); first J slot of each row block
  const int32_t* poff;
  const int32_t* pv;
  const double* pcoef;
  const int64_t* jpbase;
  // boundary rows, the same (variables of z = (X_0, X_N)); by variable: the terms voff[v] ..
  // voff[v+1]-1 in row order, each a (row, term) pair; the boundary cost's a, b, l, 2 nx each
  const int32_t* boff;
  const int32_t* bv;
  const double* bcoef;
  const int64_t* jbbase;
  const int32_t* voff;
  const int32_t* vterm;
  const double* bol;
  double sigma;
  int64_t N, nun, B, E, uoff, prow0, brow0, hbase_u, xN;
  int nx, nu, npath, npterms, nbin, nbterms, hx, hu, has_bol, ends;
  int16_t hdiag[256];    // position of (v, v) in the node's X or U block (-1: none)
};

__device__ __forceinline__ int64_t path_col(const ExtraArgs& a, int64_t i, int v) {
  return v < a.nx ? (int64_t)a.nx * i + v : a.uoff + (int64_t)a.nu * i + (v - a.nx);
}

// -0 -> +0 (what adding it to +0 gives)
__device__ __forceinline__ double pos_zero(double v) { return __double_as_longlong(v) == (long long)0x8000000000000000ull ? 0.0 : v; }
// |v| < 2^900 (v - b is then finite for every finite b) in the whole warp
__device__ __forceinline__ bool all_moderate(double v) {
  return __all_sync(__activemask(), (__double2hiint(v) & 0x7ff00000) < 0x78300000);
}

// value (a d^2 + l z, d = z - b) and derivative (2 a d + l) of one term; a2 = 2 a
template <bool VAL, bool DER>
__device__ __forceinline__ void ex_term(double z, double av, double bv, double lv, double a2, double& val, double& der) {
  if (av == 0.0 && all_moderate(z)) {          // linear (the coefficients are the launch's: a uniform branch)
    if (VAL) val = pos_zero(lv * z);
    if (DER) der = lv;
    return;
  }
  const double d = z - bv;
  if (lv == 0.0 && all_moderate(z)) {          // squared
    if (VAL) val = pos_zero(av * d * d);
    if (DER) der = pos_zero(a2 * d);
    return;
  }
  if (VAL) val = av * d * d + lv * z;
  if (DER) der = a2 * d + lv;
}

// The path rows of node i.
template <bool WC, bool WJ, bool WH, bool WJV, bool WJTV, bool WHV>
__device__ __forceinline__ void path_node(const ExtraArgs& a, int64_t i) {
  const double* pr = a.pcoef + 4 * (int64_t)a.npterms;
  for (int p = 0; p < a.npath; ++p) {
    const int64_t row = a.prow0 + (int64_t)p * a.nun + i;
    const int t0 = __ldg(a.poff + p), t1 = __ldg(a.poff + p + 1);
    const double yp = (WH || WHV) ? __ldg(a.y + row) : 0.0;
    const double wp = WJTV ? __ldg(a.vm + row) : 0.0;
    double cv = 0.0, jvv = 0.0;
    for (int t = t0; t < t1; ++t) {
      const int v = __ldg(a.pv + t);
      const double av = __ldg(a.pcoef + 4 * t), a2 = __ldg(a.pcoef + 4 * t + 3);
      const int64_t col = path_col(a, i, v);
      if (WC || WJ || WJV || WJTV) {
        double val = 0.0, dv = 0.0;
        ex_term<WC, WJ || WJV || WJTV>(__ldg(a.x + col), av, __ldg(a.pcoef + 4 * t + 1), __ldg(a.pcoef + 4 * t + 2), a2, val, dv);
        if (WC) cv = (t == t0) ? pos_zero(val) : cv + val;
        if (WJ) a.jv[__ldg(a.jpbase + p) + i * (t1 - t0) + (t - t0)] = dv;
        if (WJV) {
          const double w = dv * __ldg(a.vn + col);
          jvv = (t == t0) ? pos_zero(w) : jvv + w;
        }
        if (WJTV) a.ojtv[col] = a.ojtv[col] + wp * dv;
      }
      if ((WH || WHV) && av != 0.0) {  // the squared term's diagonal
        const double h2 = a2 * yp;
        if (WH) {
          const int e = a.hdiag[v];
          const int64_t slot = v < a.nx ? (int64_t)a.hx * i + e : a.hbase_u + (int64_t)a.hu * i + e;
          a.hv[slot] = a.hv[slot] + h2;
        }
        if (WHV) a.ohv[col] = a.ohv[col] + h2 * __ldg(a.vn + col);
      }
    }
    if (WC) a.c[row] = cv - __ldg(pr + p);
    if (WJV) a.ojv[row] = jvv;
  }
}

// The boundary inequalities and the boundary cost (one block).
template <bool WC, bool WJ, bool WH, bool WJV, bool WJTV, bool WHV>
__device__ __forceinline__ void end_block(const ExtraArgs& a) {
  __shared__ double s_c[EX_CHUNK], s_j[EX_CHUNK];
  const int t = threadIdx.x;
  if (a.npath > 0) {   // the path rows of nodes 0 and N come first
    if (t == 0 && a.B == 0 && a.E > 0) path_node<WC, WJ, WH, WJV, WJTV, WHV>(a, 0);
    if (t == 32 && a.N < a.E && a.N > 0) path_node<WC, WJ, WH, WJV, WJTV, WHV>(a, a.N);
  }
  __syncthreads();
  auto column = [&](int v) { return v >= a.nx ? a.xN + (v - a.nx) : (int64_t)v; };
  // ---- by variable: the additions to J^T w, H and H v, then the boundary cost's
  for (int v = t; v < 2 * a.nx; v += EX_THREADS) {
    const bool fin = v >= a.nx;
    const int k = fin ? v - a.nx : v;
    const int64_t col = column(v);
    const int64_t slot = (fin ? a.N * a.hx : 0) + a.hdiag[k];
    const double z = a.x[col];
    const double vv = WHV ? a.vn[col] : 0.0;
    double jt = 0.0, hd = 0.0, ho = 0.0;
    bool tj = false, th = false;   // entries loaded
    const int e0 = a.nbin ? a.voff[v] : 0, e1 = a.nbin ? a.voff[v + 1] : 0;
    for (int e = e0; e < e1; ++e) {
      const int q = a.vterm[2 * e], b = a.vterm[2 * e + 1];
      const double av = a.bcoef[4 * b], a2 = a.bcoef[4 * b + 3];
      if (WJTV) {
        double val, dv;
        ex_term<false, true>(z, av, a.bcoef[4 * b + 1], a.bcoef[4 * b + 2], a2, val, dv);
        if (!tj) jt = a.ojtv[col];
        tj = true;
        jt = jt + a.vm[a.brow0 + q] * dv;
      }
      if ((WH || WHV) && av != 0.0) {
        const double h2 = a2 * a.y[a.brow0 + q];
        if (!th) { if (WH) hd = a.hv[slot]; if (WHV) ho = a.ohv[col]; }
        th = true;
        if (WH) hd = hd + h2;
        if (WHV) ho = ho + h2 * vv;
      }
    }
    if (a.has_bol) {
      const double av = a.bol[v], bv = a.bol[2 * a.nx + v], lv = a.bol[4 * a.nx + v];
      if (a.g && (av != 0.0 || lv != 0.0)) a.g[col] = a.g[col] + (2.0 * av * (z - bv) + lv);
      if ((WH || WHV) && av != 0.0) {
        const double h2 = a.sigma * (2.0 * av);
        if (!th) { if (WH) hd = a.hv[slot]; if (WHV) ho = a.ohv[col]; }
        th = true;
        if (WH) hd = hd + h2;
        if (WHV) ho = ho + h2 * vv;
      }
    }
    if (WJTV && tj) a.ojtv[col] = jt;
    if (WH && th) a.hv[slot] = hd;
    if (WHV && th) a.ohv[col] = ho;
  }
  // ---- by term: the rows of c, J and J v (their sums in term order, thread q for row q)
  if (a.nbin > 0 && (WC || WJ || WJV)) {
    double cv = 0.0, jvv = 0.0;
    for (int b0 = 0; b0 < a.nbterms; b0 += EX_CHUNK) {
      const int n = min(EX_CHUNK, a.nbterms - b0);
      for (int i = t; i < n; i += EX_THREADS) {
        const int b = b0 + i;
        const int64_t col = column(a.bv[b]);
        double val = 0.0, dv = 0.0;
        ex_term<WC, WJ || WJV>(a.x[col], a.bcoef[4 * b], a.bcoef[4 * b + 1], a.bcoef[4 * b + 2], a.bcoef[4 * b + 3], val, dv);
        if (WC) s_c[i] = val;
        if (WJ) a.jv[a.jbbase[0] + b] = dv;
        if (WJV) s_j[i] = dv * a.vn[col];
      }
      __syncthreads();
      if (t < a.nbin && (WC || WJV)) {
        const int lo = max(a.boff[t], b0), hi = min(a.boff[t + 1], b0 + n);
        for (int b = lo; b < hi; ++b) {
          if (WC) cv = cv + s_c[b - b0];
          if (WJV) jvv = jvv + s_j[b - b0];
        }
      }
      __syncthreads();
    }
    if (t < a.nbin) {
      if (WC) a.c[a.brow0 + t] = cv - a.bcoef[4 * (int64_t)a.nbterms + t];
      if (WJV) a.ojv[a.brow0 + t] = jvv;
    }
  }
  // ---- the boundary cost's value, in variable order (2 nx <= EX_CHUNK)
  if (a.has_bol && a.f) {
    for (int v = t; v < 2 * a.nx; v += EX_THREADS) {
      const double av = a.bol[v], lv = a.bol[4 * a.nx + v], z = a.x[column(v)], d = z - a.bol[2 * a.nx + v];
      s_c[v] = av * d * d + lv * z;
      s_j[v] = (av != 0.0 || lv != 0.0) ? 1.0 : 0.0;
    }
    __syncthreads();
    if (t == 0) {
      double gs = 0.0;
      for (int v = 0; v < 2 * a.nx; ++v)
        if (s_j[v] != 0.0) gs = gs + s_c[v];
      a.f[0] = a.f[0] + gs;
    }
  }
}

template <bool WC, bool WJ, bool WH, bool WJV, bool WJTV, bool WHV>
__global__ void __launch_bounds__(EX_THREADS) k_extra(const __grid_constant__ ExtraArgs a) {
  start_follow_on();
  if (a.ends && blockIdx.x == 0) {
    end_block<WC, WJ, WH, WJV, WJTV, WHV>(a);
    return;
  }
  const int nblk = gridDim.x - a.ends, blk = blockIdx.x - a.ends;
  const int64_t stride = (int64_t)nblk * EX_THREADS;
  for (int64_t i = a.B + (int64_t)blk * EX_THREADS + threadIdx.x; i < a.E; i += stride) {
    if (a.ends && (i == 0 || i == a.N)) continue;   // by the boundary terms' block
    path_node<WC, WJ, WH, WJV, WJTV, WHV>(a, i);
  }
}

// The launch for the outputs `m` (O_C, O_J, O_H, O_JV, O_JTV, O_HV of the rows; f and g of the
// boundary cost by their pointers in `a`) on the nodes [B, E).
static ocp_status extra_launch(ocp* h, ExtraArgs& a, unsigned m, int64_t B, int64_t E, cudaStream_t s) {
  const Pattern& P = h->pat;
  if (P.nz > 256 || 2 * P.nx > EX_CHUNK) return set_err(h, OCP_EDIM, "too many variables per node for path or boundary terms");
  const bool rows = m != 0;
  a.npath = rows ? P.npath : 0;
  a.nbin = rows ? P.nbin : 0;
  a.has_bol = h->has_bol && (a.f || a.g || (m & (O_H | O_HV)));
  a.ends = (a.nbin > 0 || a.has_bol) ? 1 : 0;
  if (!a.npath && !a.ends) return OCP_OK;
  a.poff = h->d_poff; a.pv = h->d_pv; a.pcoef = h->d_pcoef; a.jpbase = h->d_pbase;
  a.boff = h->d_boff; a.bv = h->d_bv; a.bcoef = h->d_bcoef; a.jbbase = h->d_bbase;
  a.voff = h->d_boff + P.nbin + 1; a.vterm = a.voff + 2 * P.nx + 1;
  a.N = h->N; a.nun = P.nun;
  a.B = B; a.E = std::min(E, P.nun);
  a.uoff = (int64_t)h->nx * (h->N + 1);
  a.prow0 = P.nb + (int64_t)h->nx * h->N;
  a.brow0 = a.prow0 + (int64_t)P.npath * P.nun;
  a.hbase_u = P.hbase_u;
  a.xN = (int64_t)h->nx * h->N;
  a.nx = h->nx; a.nu = h->nu; a.hx = P.hx; a.hu = P.hu;
  for (int p = 0; p < P.npath; ++p) a.npterms += (int)P.psupp[p].size();
  for (int q = 0; q < P.nbin; ++q) a.nbterms += (int)P.bsupp[q].size();
  a.bol = h->d_bcoef + 4 * (int64_t)a.nbterms + P.nbin;
  for (int v = 0; v < P.nz; ++v) a.hdiag[v] = (int16_t)P.hdiag[v];
  const int64_t n = a.npath ? a.E - a.B : 0;
  int64_t blocks = n > 0 ? std::min<int64_t>((n + EX_THREADS - 1) / EX_THREADS, (int64_t)h->num_sms * 8) : 0;
  blocks += a.ends;
  if (blocks < 1) return OCP_OK;
  cudaError_t e = cudaSuccess;
  auto go = [&](auto kern) { e = launch(true, kern, blocks, EX_THREADS, 0, s, a); };
  switch (m) {
    case 0:          // f and g alone
    case O_C: go(k_extra<true, false, false, false, false, false>); break;
    case O_J: go(k_extra<false, true, false, false, false, false>); break;
    case O_H: go(k_extra<false, false, true, false, false, false>); break;
    case O_C | O_J: go(k_extra<true, true, false, false, false, false>); break;
    case O_C | O_H: go(k_extra<true, false, true, false, false, false>); break;
    case O_J | O_H: go(k_extra<false, true, true, false, false, false>); break;
    case O_C | O_J | O_H: go(k_extra<true, true, true, false, false, false>); break;
    case O_JV: go(k_extra<false, false, false, true, false, false>); break;
    case O_JTV: go(k_extra<false, false, false, false, true, false>); break;
    case O_HV: go(k_extra<false, false, false, false, false, true>); break;
    case O_JV | O_JTV | O_HV: go(k_extra<false, false, false, true, true, true>); break;
    default: go(k_extra<true, true, true, true, true, true>); break;   // the fused step: every output
  }
  return cuda_err(h, e, "path and boundary terms launch");
}

static bool any_extra(const ocp* h) { return h->pat.npath > 0 || h->pat.nbin > 0 || h->has_bol; }

ocp_status extra_eval(ocp* h, const EvalCall& c, cudaStream_t s) {
  if (!any_extra(h)) return OCP_OK;
  if (c.range && h->pat.nbin > 0) return set_err(h, OCP_EMODEL, "node ranges are not provided with boundary inequalities");
  if (c.range && h->has_bol) return set_err(h, OCP_EMODEL, "node ranges are not provided with a boundary cost");
  ExtraArgs a;
  memset(&a, 0, sizeof(a));
  a.x = c.x; a.y = c.y; a.vn = c.vn; a.vm = c.vm; a.sigma = c.sigma;
  a.f = c.f; a.g = c.g; a.c = c.c; a.jv = c.jv; a.hv = c.hv; a.ojv = c.ojv; a.ojtv = c.ojtv; a.ohv = c.ohv;
  unsigned m = (c.c ? O_C : 0u) | (c.jv ? O_J : 0u) | (c.hv ? O_H : 0u);
  if (c.ojv || c.ojtv || c.ohv) m = O_STEP;
  return extra_launch(h, a, m, c.B, c.E, s);
}

ocp_status extra_prod(ocp* h, const ProdCall& c, cudaStream_t s) {
  if (!any_extra(h)) return OCP_OK;
  ExtraArgs a;
  memset(&a, 0, sizeof(a));
  a.x = c.x; a.y = c.y; a.sigma = c.sigma;
  const int64_t B = (c.kind == P_JTPROD) ? c.B : 0, E = (c.kind == P_JTPROD && c.E >= 0) ? c.E : h->N + 1;
  if (c.kind == P_JPROD) { a.vn = c.v; a.ojv = c.out; return extra_launch(h, a, O_JV, B, E, s); }
  if (c.kind == P_JTPROD) { a.vm = c.v; a.ojtv = c.out; return extra_launch(h, a, O_JTV, B, E, s); }
  a.vn = c.v; a.ohv = c.out;
  return extra_launch(h, a, O_HV, B, E, s);
}

// The three products of one fused step in one launch (jp and hp share their direction).
ocp_status extra_prod3(ocp* h, const ProdCall& jp, const ProdCall& jt, const ProdCall& hp, cudaStream_t s) {
  if (!any_extra(h)) return OCP_OK;
  ExtraArgs a;
  memset(&a, 0, sizeof(a));
  a.x = hp.x; a.y = hp.y; a.sigma = hp.sigma; a.vn = jp.v; a.vm = jt.v;
  a.ojv = jp.out; a.ojtv = jt.out; a.ohv = hp.out;
  return extra_launch(h, a, O_JV | O_JTV | O_HV, 0, h->N + 1, s);
}

// a, b, l and 2a of a term
static void push_term(std::vector<double>& coef, double a, double b, double l) {
  coef.push_back(a);
  coef.push_back(b);
  coef.push_back(l);
  coef.push_back(2.0 * a);
}

// Device tables of the path rows (terms, coefficients, slot bases); called after every
// pattern rebuild.
ocp_status path_upload(ocp* h) {
  cudaFree(h->d_poff); cudaFree(h->d_pv); cudaFree(h->d_pcoef); cudaFree(h->d_pbase);
  h->d_poff = nullptr; h->d_pv = nullptr; h->d_pcoef = nullptr; h->d_pbase = nullptr;
  const Pattern& P = h->pat;
  std::vector<int32_t> poff(1, 0), pv;
  std::vector<double> coef;
  for (int p = 0; p < P.npath; ++p) {
    for (int v : P.psupp[p]) {
      pv.push_back(v);
      push_term(coef, h->path_a[p * P.nz + v], h->path_b[p * P.nz + v], h->path_l[p * P.nz + v]);
    }
    poff.push_back((int32_t)pv.size());
  }
  for (int p = 0; p < P.npath; ++p) coef.push_back(h->path_r[p]);
  std::vector<int64_t> base(P.jpbase);
  base.insert(base.end(), P.kpbase.begin(), P.kpbase.end());
  if (pv.empty()) pv.push_back(0);
  if (coef.empty()) coef.push_back(0.0);
  cudaError_t e;
  if ((e = ocpg::dev_malloc(&h->d_poff, poff.size() * 4)) != cudaSuccess ||
      (e = ocpg::dev_malloc(&h->d_pv, pv.size() * 4)) != cudaSuccess ||
      (e = ocpg::dev_malloc(&h->d_pcoef, coef.size() * 8)) != cudaSuccess ||
      (e = ocpg::dev_malloc(&h->d_pbase, base.size() * 8)) != cudaSuccess)
    return cuda_err(h, e, "cudaMalloc(path tables)");
  if ((e = ocpg::dev_upload(h->d_poff, poff.data(), poff.size() * 4)) != cudaSuccess ||
      (e = ocpg::dev_upload(h->d_pv, pv.data(), pv.size() * 4)) != cudaSuccess ||
      (e = ocpg::dev_upload(h->d_pcoef, coef.data(), coef.size() * 8)) != cudaSuccess ||
      (e = ocpg::dev_upload(h->d_pbase, base.data(), base.size() * 8)) != cudaSuccess)
    return cuda_err(h, e, "cudaMemcpy(path tables)");
  return OCP_OK;
}

// Device tables of the boundary inequalities (terms by row and by variable, coefficients, slot
// bases) and of the boundary cost; called after every pattern rebuild.
ocp_status bin_upload(ocp* h) {
  cudaFree(h->d_boff); cudaFree(h->d_bv); cudaFree(h->d_bcoef); cudaFree(h->d_bbase);
  h->d_boff = nullptr; h->d_bv = nullptr; h->d_bcoef = nullptr; h->d_bbase = nullptr;
  const Pattern& P = h->pat;
  const int bz = 2 * P.nx;
  std::vector<int32_t> boff(1, 0), bv, var(1, 0), vterm;
  std::vector<double> coef;
  for (int q = 0; q < P.nbin; ++q) {
    for (int v : P.bsupp[q]) {
      bv.push_back(v);
      push_term(coef, h->bin_a[q * bz + v], h->bin_b[q * bz + v], h->bin_l[q * bz + v]);
    }
    boff.push_back((int32_t)bv.size());
  }
  if (P.nbin > 0) {
    for (int v = 0; v < bz; ++v) {
      for (int q = 0; q < P.nbin; ++q)
        for (int t = boff[q]; t < boff[q + 1]; ++t)
          if (bv[t] == v) { vterm.push_back(q); vterm.push_back(t); }
      var.push_back((int32_t)(vterm.size() / 2));
    }
    boff.insert(boff.end(), var.begin(), var.end());
    boff.insert(boff.end(), vterm.begin(), vterm.end());
  }
  for (int q = 0; q < P.nbin; ++q) coef.push_back(h->bin_r[q]);
  if (h->has_bol)
    for (const auto* t : {&h->bol_a, &h->bol_b, &h->bol_l}) coef.insert(coef.end(), t->begin(), t->end());
  std::vector<int64_t> base(P.jbbase);
  base.insert(base.end(), P.kbbase.begin(), P.kbbase.end());
  if (bv.empty()) bv.push_back(0);
  if (coef.empty()) coef.push_back(0.0);
  cudaError_t e;
  if ((e = ocpg::dev_malloc(&h->d_boff, boff.size() * 4)) != cudaSuccess ||
      (e = ocpg::dev_malloc(&h->d_bv, bv.size() * 4)) != cudaSuccess ||
      (e = ocpg::dev_malloc(&h->d_bcoef, coef.size() * 8)) != cudaSuccess ||
      (e = ocpg::dev_malloc(&h->d_bbase, base.size() * 8)) != cudaSuccess)
    return cuda_err(h, e, "cudaMalloc(boundary tables)");
  if ((e = ocpg::dev_upload(h->d_boff, boff.data(), boff.size() * 4)) != cudaSuccess ||
      (e = ocpg::dev_upload(h->d_bv, bv.data(), bv.size() * 4)) != cudaSuccess ||
      (e = ocpg::dev_upload(h->d_bcoef, coef.data(), coef.size() * 8)) != cudaSuccess ||
      (e = ocpg::dev_upload(h->d_bbase, base.data(), base.size() * 8)) != cudaSuccess)
    return cuda_err(h, e, "cudaMemcpy(boundary tables)");
  return OCP_OK;
}

}  // namespace ocpg
