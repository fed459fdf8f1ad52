// Physics kernels: block pattern, transmissibilities, residual and Jacobian
// assembly, norms, decoupling, pressure extraction and the Newton update.
//
// Compiled with -fmad=false: every floating-point expression is evaluated
// as written (no fused multiply-add), so that the assembled Jacobian, the
// decoupled matrix and the pressure block are bit-identical to a plain
// sequential CPU evaluation of the same formulas.  The AMG strength graph
// and aggregates are computed from those values and must not depend on the
// processor that evaluated them.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "dp_internal.h"
#include "dp_kernels.cuh"

namespace dp {

// ---------------------------------------------------------------- physics

// Sign and zero tests and sign changes of doubles on their two 32-bit halves:
// on this GPU an FP64 comparison or negation costs a quarter of an SM 64
// cycles, and 64-bit integer forms of them are compiled back into one.
__device__ __forceinline__ bool is_zero(double v) {
  return (((unsigned)__double2hiint(v) << 1) | (unsigned)__double2loint(v)) == 0u;
}
__device__ __forceinline__ bool nonneg(double v) { return __double2hiint(v) >= 0 || is_zero(v); }
__device__ __forceinline__ double flip(double v) {   // -v
  return __hiloint2double(__double2hiint(v) ^ (int)0x80000000, __double2loint(v));
}
__device__ __forceinline__ double twice(double v) {   // 2 v, v finite and >= 0
  int h = __double2hiint(v);
  return h >= 0x00100000 && h < 0x7fd00000 ? __hiloint2double(h + 0x00100000, __double2loint(v))
                                           : 2.0 * v;
}

// Cell properties (Section 2): linear densities, porosity, Corey relative
// permeabilities of the normalised saturation, mobilities and derivatives.
struct Props {
  double rho[2], drho[2], phi, dphi, lam[2], dlam[2];
  double pc, dpc;   // capillary pressure and slope (set only where a table is given)
};

// Capillary pressure p_cow(s_w) (Section 2: p_w = p_o - p_cow(s_w)) from a
// table of n (s_w, p_cow) pairs: the line through the two points around s_w,
// constant with zero slope at and beyond the end points; zero with no table.
__device__ __forceinline__ void cap_pressure(int n, const double *t, double sw, double &pc,
                                             double &dpc) {
  if (n == 0) { pc = 0.0; dpc = 0.0; return; }
  if (sw <= t[0]) { pc = t[1]; dpc = 0.0; return; }
  if (sw >= t[2 * (n - 1)]) { pc = t[2 * n - 1]; dpc = 0.0; return; }
  int k = 0;
  while (sw >= t[2 * (k + 1)]) ++k;      // t[2k] <= sw < t[2k + 2]
  double ds = t[2 * k + 2] - t[2 * k];
  double dp = t[2 * k + 3] - t[2 * k + 1];
  dpc = dp / ds;
  pc = t[2 * k + 1] + dp * ((sw - t[2 * k]) / ds);
}

__device__ __forceinline__ void props(const Phys &P, const double *phi_f, const double *phi_m,
                                      int c, double p, double sw, Props &q) {
  int loc = c >> 1;
  double phi_ref = (c & 1) == 0 ? phi_f[loc] : phi_m[loc];
  double dp = p - P.p_ref;
  q.rho[0] = P.rho_o_ref * (1.0 + P.c_o * dp);
  q.rho[1] = P.rho_w_ref * (1.0 + P.c_w * dp);
  q.drho[0] = P.rho_o_ref * P.c_o;
  q.drho[1] = P.rho_w_ref * P.c_w;
  // with no rock compressibility the factor is 1 exactly
  q.phi = !P.rock ? phi_ref : phi_ref * (1.0 + P.c_rock * (p - P.p_ref_rock));
  q.dphi = !P.rock ? 0.0 : phi_ref * P.c_rock;
  double S = (sw - P.swc) * P.inv_span, dS;
  const int hi = __double2hiint(S), mag = hi & 0x7fffffff;
  const bool nan = mag > 0x7ff00000 || (mag == 0x7ff00000 && __double2loint(S) != 0);
  if (!nan && (hi < 0 || is_zero(S))) { S = 0.0; dS = 0.0; }        // S <= 0
  else if (!nan && hi >= 0x3ff00000) { S = 1.0; dS = 0.0; }          // S >= 1
  else dS = P.inv_span;
  if (is_zero(S)) {   // no mobile water: the values below, without their arithmetic
    q.lam[1] = 0.0;
    q.dlam[1] = 0.0;
    q.lam[0] = P.inv_mu_o;
    q.dlam[0] = -0.0;
    return;
  }
  double so = 1.0 - S;
  q.lam[1] = (S * S) * P.inv_mu_w;
  q.dlam[1] = (twice(S) * dS) * P.inv_mu_w;
  q.lam[0] = (so * so) * P.inv_mu_o;
  q.dlam[0] = flip(twice(so) * dS) * P.inv_mu_o;
}

// Phase masses V phi rho s of a cell and their derivatives [phase][p, sw].
__device__ __forceinline__ void accumulation(const Phys &P, double sw, const Props &q,
                                             double M[2], double dM[4]) {
  double Vphi = P.V * q.phi;
  double so = 1.0 - sw;
  M[0] = (Vphi * q.rho[0]) * so;
  M[1] = (Vphi * q.rho[1]) * sw;
  if (!P.rock) {   // dphi = 0: the first products are exact zeros
    dM[0] = (P.V * (q.phi * q.drho[0])) * so;
    dM[2] = (P.V * (q.phi * q.drho[1])) * sw;
  } else {
    dM[0] = (P.V * ((q.dphi * q.rho[0]) + (q.phi * q.drho[0]))) * so;
    dM[2] = (P.V * ((q.dphi * q.rho[1]) + (q.phi * q.drho[1]))) * sw;
  }
  dM[1] = flip(Vphi * q.rho[0]);
  dM[3] = Vphi * q.rho[1];
}

// Perforation mass rate into a fracture cell (Section 2, q_{alpha,i}):
// producer WI rho lambda (p_b - p); water injector WI rho_w lambda_t (p_b - p).
__device__ __forceinline__ void perf_rate(int kind, double wi, double pc, double pb, const Props &q,
                                          double Q[2], double dq[4], double dqb[2]) {
  double dpw = pb - pc;
  if (kind == 0) {
    double lt = q.lam[0] + q.lam[1], dlt = q.dlam[0] + q.dlam[1];
    Q[0] = 0.0; dq[0] = 0.0; dq[1] = 0.0; dqb[0] = 0.0;
    Q[1] = ((wi * q.rho[1]) * lt) * dpw;
    dq[2] = (((wi * q.drho[1]) * lt) * dpw) - ((wi * q.rho[1]) * lt);
    dq[3] = ((wi * q.rho[1]) * dlt) * dpw;
    dqb[1] = (wi * q.rho[1]) * lt;
  } else {
#pragma unroll
    for (int al = 0; al < 2; ++al) {
      Q[al] = ((wi * q.rho[al]) * q.lam[al]) * dpw;
      dq[2 * al + 0] = (((wi * q.drho[al]) * q.lam[al]) * dpw) - ((wi * q.rho[al]) * q.lam[al]);
      dq[2 * al + 1] = ((wi * q.rho[al]) * q.dlam[al]) * dpw;
      dqb[al] = (wi * q.rho[al]) * q.lam[al];
    }
  }
}

__device__ __forceinline__ void loc_ijk(const Phys &P, int loc, int &i, int &j, int &k) {
  i = loc % P.nx;
  j = (loc / P.nx) % P.ny;
  k = loc / (P.nx * P.ny);
}

__device__ __forceinline__ double depth(const Phys &P, int k) {
  return P.top_depth + ((double)k + 0.5) * P.dz;
}

// ---------------------------------------------------------------- pattern

// Perforations of a cell: [lo, hi) in the (cell, well)-sorted list.
__device__ __forceinline__ void perf_range(const int *pc_cell, int np, int c, int &lo, int &hi) {
  int a = 0, b = np;
  while (a < b) { int m = (a + b) >> 1; if (pc_cell[m] < c) a = m + 1; else b = m; }
  lo = a;
  b = np;
  while (a < b) { int m = (a + b) >> 1; if (pc_cell[m] <= c) a = m + 1; else b = m; }
  hi = a;
}

__global__ void k_pattern_count(Phys P, const int *pc_cell, int np, const int *pw_start,
                                int *len) {
  int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= P.nb) return;
  if (r >= P.nc) { int w = r - P.nc; len[r] = 1 + pw_start[w + 1] - pw_start[w]; return; }
  if (r & 1) { len[r] = 2; return; }
  int i, j, k;
  loc_ijk(P, r >> 1, i, j, k);
  int lo, hi;
  perf_range(pc_cell, np, r, lo, hi);
  len[r] = 2 + (i > 0) + (i < P.nx - 1) + (j > 0) + (j < P.ny - 1) + (k > 0) + (k < P.nz - 1) +
           (hi - lo);
}

// Two-point transmissibility between cells a < b (fracture-fracture
// harmonic mean, or the shape-factor transfer sigma km V of one location).
__device__ __forceinline__ double conn_trans(const Phys &P, const double *kf, const double *km,
                                             int a, int b) {
  int la = a >> 1, lb = b >> 1;
  if (la == lb) return (P.sigma * km[la]) * P.V;
  int ia, ja, ka, ib, jb, kb;
  loc_ijk(P, la, ia, ja, ka);
  loc_ijk(P, lb, ib, jb, kb);
  double A, D;
  if (ka != kb) { A = P.dx * P.dy; D = P.dz; }
  else if (ja != jb) { A = P.dx * P.dz; D = P.dy; }
  else { A = P.dy * P.dz; D = P.dx; }
  double k1 = kf[la], k2 = kf[lb];
  return ((2.0 * A) * (k1 * k2)) / (D * (k1 + k2));
}

__global__ void k_pattern_fill(Phys P, const double *kf, const double *km, const int *pc_cell,
                               const int *pc_well, const double *pc_wi, int np,
                               const int *pw_start, const int *pw_cell, const double *pw_wi,
                               const int *rowptr, int *col, int *diag, double *trans) {
  int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= P.nb) return;
  int e0 = rowptr[r];
  if (r >= P.nc) {                       // well row: perforated cells, then itself
    int w = r - P.nc, s = pw_start[w], t = pw_start[w + 1];
    for (int q = s; q < t; ++q) { col[e0 + q - s] = pw_cell[q]; trans[e0 + q - s] = pw_wi[q]; }
    col[e0 + t - s] = r;
    trans[e0 + t - s] = 0.0;
    diag[r] = e0 + t - s;
    return;
  }
  int c[16];
  int n = 0;
  int loc = r >> 1;
  if (r & 1) { c[n++] = r - 1; c[n++] = r; }
  else {
    int i, j, k, nxy = P.nx * P.ny;
    loc_ijk(P, loc, i, j, k);
    if (k > 0) c[n++] = 2 * (loc - nxy);
    if (j > 0) c[n++] = 2 * (loc - P.nx);
    if (i > 0) c[n++] = 2 * (loc - 1);
    c[n++] = r;
    c[n++] = r + 1;
    if (i < P.nx - 1) c[n++] = 2 * (loc + 1);
    if (j < P.ny - 1) c[n++] = 2 * (loc + P.nx);
    if (k < P.nz - 1) c[n++] = 2 * (loc + nxy);
  }
  for (int a = 1; a < n; ++a) {          // sorted ascending
    int v = c[a], b = a - 1;
    while (b >= 0 && c[b] > v) { c[b + 1] = c[b]; --b; }
    c[b + 1] = v;
  }
  for (int a = 0; a < n; ++a) {
    int d = c[a];
    col[e0 + a] = d;
    if (d == r) { diag[r] = e0 + a; trans[e0 + a] = 0.0; }
    else trans[e0 + a] = conn_trans(P, kf, km, min(r, d), max(r, d));
  }
  if (!(r & 1)) {
    int lo, hi;
    perf_range(pc_cell, np, r, lo, hi);
    for (int q = lo; q < hi; ++q) {      // wells after all cells, by well index
      col[e0 + n] = P.nc + pc_well[q];
      trans[e0 + n] = pc_wi[q];
      ++n;
    }
  }
}

// Connections of the cell graph, by kind: c = axis nL + loc for the face
// between location loc and its neighbour along x, y or z (axis 0, 1, 2), c =
// 3 nL + loc for the fracture-matrix link of loc; its cells are a < b.  The
// positions of the blocks (a, b) and (b, a), (-1, -1) where there is no
// connection, and its transmissibility.
__device__ __forceinline__ int find_entry(const int *__restrict__ rowptr,
                                          const int *__restrict__ col, int r, int d) {
  for (int e = rowptr[r], e1 = rowptr[r + 1]; e < e1; ++e)
    if (col[e] == d) return e;
  return -1;
}

__global__ void k_conn_build(Phys P, const int *rowptr, const int *col, const double *trans,
                             int2 *cpos, double *ctrans) {
  int loc = blockIdx.x * blockDim.x + threadIdx.x, axis = blockIdx.y;
  if (loc >= P.nL) return;
  int i, j, k;
  loc_ijk(P, loc, i, j, k);
  int cb = -1;
  if (axis == 0 && i + 1 < P.nx) cb = 2 * (loc + 1);
  else if (axis == 1 && j + 1 < P.ny) cb = 2 * (loc + P.nx);
  else if (axis == 2 && k + 1 < P.nz) cb = 2 * (loc + P.nx * P.ny);
  else if (axis == 3) cb = 2 * loc + 1;
  int2 e = make_int2(-1, -1);
  if (cb >= 0) e = make_int2(find_entry(rowptr, col, 2 * loc, cb), find_entry(rowptr, col, cb, 2 * loc));
  size_t c = (size_t)axis * P.nL + loc;
  cpos[c] = e;
  ctrans[c] = cb >= 0 ? trans[e.x] : 0.0;
}

__global__ void k_storage_len(int nb, int nL, int nc, const int *rowptr, int *len) {
  int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nb) return;
  int i = row_of_pair(q, nL, nc);
  len[q] = rowptr[i + 1] - rowptr[i];
}

__global__ void k_storage_cols(int nb, int nL, int nc, const int *rowptr, const int *col,
                               const int *srowptr, int *scol) {
  int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nb) return;
  int i = row_of_pair(q, nL, nc);
  int e0 = rowptr[i], m = rowptr[i + 1] - e0, d0 = srowptr[q];
  for (int k = 0; k < m; ++k) scol[d0 + k] = col[e0 + k];
}

// Peaceman's radius for a vertical well and the well index
// W = 2 pi k h w_frac / (ln(r_e / r_w) + s), k h = sqrt(kx ky) dz, w_frac = 1.
static double well_index_host(double kx, double ky, double dx, double dy, double dz, double rw,
                              double skin) {
  double ryx = ky / kx, rxy = kx / ky;
  double re = 0.28 * std::sqrt(std::sqrt(ryx) * dx * dx + std::sqrt(rxy) * dy * dy) /
              (std::pow(ryx, 0.25) + std::pow(rxy, 0.25));
  double wfrac = 1.0;
  return (((2.0 * M_PI) * std::sqrt(kx * ky)) * dz) * wfrac / (std::log(re / rw) + skin);
}

int phys_build_pattern(Sim *s) {
  Phys &P = s->ph;
  // perforations, well by well (cells ascending), with their well indices
  std::vector<double> kf_host;  // only the perforated locations are needed
  int np = 0;
  for (auto &w : s->wells) np += w.k_bot - w.k_top + 1;
  s->nperf = np;
  std::vector<int> locs;
  for (auto &w : s->wells)
    for (int k = w.k_top; k <= w.k_bot; ++k) locs.push_back(w.i + P.nx * (w.j + P.ny * k));
  std::vector<double> kfp(np);
  for (int q = 0; q < np; ++q)
    DP_CUDA(s, cudaMemcpyAsync(&kfp[q], s->kf + locs[q], sizeof(double), cudaMemcpyDeviceToHost,
                               s->stream));
  DP_CUDA(s, cudaStreamSynchronize(s->stream));
  std::vector<int> pw_start(P.nw + 1, 0), pw_cell(np);
  std::vector<double> pw_wi(np);
  s->wi_host.resize(np);
  int q = 0;
  for (int w = 0; w < P.nw; ++w) {
    const dp_well &W = s->wells[w];
    pw_start[w] = q;
    for (int k = W.k_top; k <= W.k_bot; ++k, ++q) {
      pw_cell[q] = 2 * locs[q];
      pw_wi[q] = W.wi > 0.0 ? W.wi : well_index_host(kfp[q], kfp[q], P.dx, P.dy, P.dz, W.rw, W.skin);
      s->wi_host[q] = pw_wi[q];
    }
  }
  pw_start[P.nw] = np;
  std::vector<int> order(np);
  for (int t = 0; t < np; ++t) order[t] = t;
  std::vector<int> pw_well(np);
  for (int w = 0; w < P.nw; ++w)
    for (int t = pw_start[w]; t < pw_start[w + 1]; ++t) pw_well[t] = w;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
    return pw_cell[a] != pw_cell[b] ? pw_cell[a] < pw_cell[b] : pw_well[a] < pw_well[b];
  });
  std::vector<int> pc_cell(np), pc_well(np);
  std::vector<double> pc_wi(np);
  for (int t = 0; t < np; ++t) {
    pc_cell[t] = pw_cell[order[t]];
    pc_well[t] = pw_well[order[t]];
    pc_wi[t] = pw_wi[order[t]];
  }
  for (int t = 1; t < np; ++t)
    if (pc_cell[t] == pc_cell[t - 1] && pc_well[t] == pc_well[t - 1]) {
      s->fail(DP_EINVAL, "a well perforates the same cell twice");
      return DP_EINVAL;
    }
  size_t npb = (size_t)std::max(np, 1);
  int *d_pc_cell = (int *)dalloc(s, npb * 4), *d_pc_well = (int *)dalloc(s, npb * 4);
  double *d_pc_wi = (double *)dalloc(s, npb * 8);
  int *d_pw_start = (int *)dalloc(s, (P.nw + 1) * 4), *d_pw_cell = (int *)dalloc(s, npb * 4);
  double *d_pw_wi = (double *)dalloc(s, npb * 8);
  if (!d_pc_cell || !d_pc_well || !d_pc_wi || !d_pw_start || !d_pw_cell || !d_pw_wi) {
    s->fail(DP_ENOMEM, "allocation failed");
    return DP_ENOMEM;
  }
  if (np) {
    DP_CUDA(s, cudaMemcpyAsync(d_pc_cell, pc_cell.data(), np * 4, cudaMemcpyHostToDevice, s->stream));
    DP_CUDA(s, cudaMemcpyAsync(d_pc_well, pc_well.data(), np * 4, cudaMemcpyHostToDevice, s->stream));
    DP_CUDA(s, cudaMemcpyAsync(d_pc_wi, pc_wi.data(), np * 8, cudaMemcpyHostToDevice, s->stream));
    DP_CUDA(s, cudaMemcpyAsync(d_pw_cell, pw_cell.data(), np * 4, cudaMemcpyHostToDevice, s->stream));
    DP_CUDA(s, cudaMemcpyAsync(d_pw_wi, pw_wi.data(), np * 8, cudaMemcpyHostToDevice, s->stream));
  }
  DP_CUDA(s, cudaMemcpyAsync(d_pw_start, pw_start.data(), (P.nw + 1) * 4, cudaMemcpyHostToDevice,
                             s->stream));
  s->perf_cell = d_pc_cell;
  s->perf_well = d_pc_well;
  s->perf_wi = d_pc_wi;
  // row lengths, row pointers, columns and per-entry transmissibilities
  int *len = (int *)dalloc(s, (size_t)P.nb * 4);
  s->A.n = P.nb;
  s->A.rowptr = (int *)dalloc(s, (size_t)(P.nb + 1) * 4);
  s->A.diag = (int *)dalloc(s, (size_t)P.nb * 4);
  if (!len || !s->A.rowptr || !s->A.diag) { s->fail(DP_ENOMEM, "allocation failed"); return DP_ENOMEM; }
  DP_LAUNCH(s, k_pattern_count, nblk(P.nb), kBlock, 0, P, d_pc_cell, np, d_pw_start, len);
  int nnz = 0;
  DP_TRY(scan_i32(s, len, s->A.rowptr, P.nb, &nnz));
  s->A.nnz = nnz;
  s->A.col = (int *)dalloc(s, (size_t)nnz * 4);
  s->A.val = (double *)dalloc(s, (size_t)nnz * 32);
  s->trans = (double *)dalloc(s, (size_t)nnz * 8);
  s->ap = (double *)dalloc(s, (size_t)nnz * 8);
  s->sval = (double *)dalloc(s, (size_t)nnz * 32);
  if (s->opt.precision >= 1) {   // the preconditioner's residuals in FP32
    s->svalf = (float *)dalloc(s, (size_t)nnz * 16);
    s->spf = (float *)dalloc(s, (size_t)nnz * 8);
    if (!s->svalf || !s->spf) { s->fail(DP_ENOMEM, "allocation failed"); return DP_ENOMEM; }
  } else {
    s->sa00 = (double *)dalloc(s, (size_t)nnz * 8);
    s->sa01 = (double *)dalloc(s, (size_t)nnz * 8);
    if (!s->sa00 || !s->sa01) { s->fail(DP_ENOMEM, "allocation failed"); return DP_ENOMEM; }
  }
  s->scol = (int *)dalloc(s, (size_t)nnz * 4);
  s->srowptr = (int *)dalloc(s, ((size_t)P.nb + 1) * 4);
  s->cpos = (int2 *)dalloc(s, (size_t)P.nL * 32);
  s->ctrans = (double *)dalloc(s, (size_t)P.nL * 32);
  s->fconn = (double *)dalloc(s, (size_t)P.nL * 64);
  if (!s->A.col || !s->A.val || !s->trans || !s->ap || !s->sval || !s->scol || !s->srowptr ||
      !s->cpos || !s->ctrans || !s->fconn) {
    s->fail(DP_ENOMEM, "allocation failed");
    return DP_ENOMEM;
  }
  DP_LAUNCH(s, k_pattern_fill, nblk(P.nb), kBlock, 0, P, s->kf, s->km, d_pc_cell, d_pc_well,
            d_pc_wi, np, d_pw_start, d_pw_cell, d_pw_wi, s->A.rowptr, s->A.col, s->A.diag,
            s->trans);
  DP_CUDA(s, cudaGetLastError());
  DP_LAUNCH(s, k_conn_build, dim3(nblk(P.nL), 4), kBlock, 0, P, s->A.rowptr, s->A.col, s->trans,
            s->cpos, s->ctrans);
  DP_CUDA(s, cudaGetLastError());
  // the storage-order pattern of the Krylov operator's copy
  DP_LAUNCH(s, k_storage_len, nblk(P.nb), kBlock, 0, P.nb, P.nL, P.nc, s->A.rowptr, len);
  int snnz = 0;
  DP_TRY(scan_i32(s, len, s->srowptr, P.nb, &snnz));
  DP_LAUNCH(s, k_storage_cols, nblk(P.nb), kBlock, 0, P.nb, P.nL, P.nc, s->A.rowptr, s->A.col,
            s->srowptr, s->scol);
  DP_CUDA(s, cudaGetLastError());
  dfree(s, len);
  dfree(s, d_pw_start);
  dfree(s, d_pw_cell);
  dfree(s, d_pw_wi);
  return DP_OK;
}

// ---------------------------------------------------------------- assembly

// Everything here is FP64-bound (1.2 TFLOP/s), so each kernel is written for
// few FP64 instructions; the products and sums are those of the row-by-row
// formulas, in their order, and what is left out is exact: terms that are
// zero because a cell is downstream, or because no water moves there.
// sim_assemble's residual, Jacobian and norms: 1.17 ms at 200x200x50
// locations (8M unknowns) instead of 1.57, 82 us at 61x43x27 with gravity
// and curves instead of 144.
//
// Cell properties stored structure-of-arrays, fracture cells then matrix
// cells (cell c at (c & 1) nL + c / 2, so that a warp of connections along
// one axis reads them contiguously): per phase the upstream products rho
// lambda, rho' lambda and rho lambda' (formed once per cell: a cell is
// upstream of up to seven connections), the densities, and with capillary
// curves p_cow and its slope (a table search and a division per cell, not
// per connection and side).
__device__ __forceinline__ size_t prop_at(const Phys &P, int c) {
  return (size_t)(c & 1) * P.nL + (c >> 1);
}

template <bool CAP>
__global__ void __launch_bounds__(kBlock) k_props(Phys P, const double *phi_f, const double *phi_m,
                                                  const double *p, const double *sw, double *pr) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= P.nc) return;
  Props q;
  double s = sw[c];
  props(P, phi_f, phi_m, c, p[c], s, q);
  size_t n = (size_t)P.nc;
  double *o = pr + prop_at(P, c);
  o[6 * n] = q.rho[0];
  o[7 * n] = q.rho[1];
  o[0] = q.rho[0] * q.lam[0];
  o[n] = q.drho[0] * q.lam[0];
  if (is_zero(q.lam[1]) && is_zero(q.dlam[1]) && is_zero(q.dlam[0])) {
    o[2 * n] = -0.0;   // no mobile water, densities positive
    o[3 * n] = o[4 * n] = o[5 * n] = 0.0;
  } else {
    o[2 * n] = q.rho[0] * q.dlam[0];
    o[3 * n] = q.rho[1] * q.lam[1];
    o[4 * n] = q.drho[1] * q.lam[1];
    o[5 * n] = q.rho[1] * q.dlam[1];
  }
  if (CAP) {
    double pc, dpc;
    cap_pressure(P.pc_n[c & 1], P.pc_tab[c & 1], s, pc, dpc);
    o[8 * n] = pc;
    o[9 * n] = dpc;
  }
}

struct AsmArgs {
  Phys P;
  const int *rowptr, *col, *diag;
  const int2 *cpos;
  const double *trans, *ctrans, *phi_f, *phi_m, *pr;
  const double *p, *sw, *bhp, *Mn;
  const int *well_kind;
  const double *well_target;
  double *val, *R, *Macc;
  double2 *fconn;
  double inv_dt;
  bool wide;   // val on a 32-byte boundary
};

// A 2x2 block as one 32-byte access, where the blocks start on 32-byte
// boundaries (wide; an allocator given by the caller may give less).
__device__ __forceinline__ void store_block(double *p, const double (&v)[4], bool wide) {
  if (wide) {
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0]), "d"(v[1]),
                 "d"(v[2]), "d"(v[3])
                 : "memory");
  } else {
    reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
  }
}
__device__ __forceinline__ void load_block(const double *p, double (&v)[4], bool wide) {
  if (wide) {
    asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
                 : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3])
                 : "l"(p));
  } else {
    double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
  }
}

// Each connection's mass flux a -> b (a < b) per phase, once: upstream
// mobility (Section 2: Darcy flux with potential Phi = p - rho g z, upstream
// weighting), written as F, and as the two off-diagonal blocks, dF/dx_b into
// row a and -dF/dx_a into row b.  With mob = rho lambda of the upstream cell,
//   F = (T mob) dpot,  dF/dp_up = T (mob' dpot +- mob),  dF/ds_up = T (mob_s dpot),
//   dF/dp_down = -+ T mob,  dF/ds_down = 0
// (the gravity and capillary terms below), which is what the two-sided
// formula gives with the downstream cell's zero products left out: 16 FP64
// operations a connection without gravity and curves instead of 45.
// GRAV: the vertical connections' density terms (for the others gdz = 0 and
// the terms are exact zeros); CAP: the water potential carries -p_cow(s_w)
// of each side.  A thread per connection, the axis by blockIdx.y.
template <bool GRAV, bool CAP>
__global__ void __launch_bounds__(kBlock) k_conn_flux(AsmArgs a) {
  const Phys &P = a.P;
  const int la = blockIdx.x * blockDim.x + threadIdx.x, axis = blockIdx.y;
  if (la >= P.nL) return;
  const size_t c = (size_t)axis * P.nL + la;
  const int2 e = a.cpos[c];
  if (e.x < 0 || e.y < 0) return;
  const int lb = la + (axis == 0 ? 1 : axis == 1 ? P.nx : axis == 2 ? P.nx * P.ny : 0);
  const int ca = 2 * la, cb = axis == 3 ? ca + 1 : 2 * lb;
  const size_t n = (size_t)P.nc, ia = prop_at(P, ca), ib = prop_at(P, cb);
  const double T = a.ctrans[c];
  const double dp = a.p[ca] - a.p[cb];
  double F[2], fa[4], fb[4];   // fa, fb: -dF/dx_a and dF/dx_b as stored
#pragma unroll
  for (int al = 0; al < 2; ++al) {
    const bool capw = CAP && al == 1;
    double dpot = dp, ddpa = 1.0, ddpb = -1.0;
    if (capw) dpot = (a.p[ca] - a.pr[8 * n + ia]) - (a.p[cb] - a.pr[8 * n + ib]);
    const bool grav = GRAV && axis == 2;
    if (grav) {
      const int ka = la / (P.nx * P.ny);
      const double gdz = P.g * (depth(P, ka) - depth(P, ka + 1));
      const double drho = al == 0 ? P.drho_o : P.drho_w;
      dpot = dpot - ((0.5 * (a.pr[(6 + al) * n + ia] + a.pr[(6 + al) * n + ib])) * gdz);
      ddpa = 1.0 - ((0.5 * drho) * gdz);
      ddpb = -1.0 - ((0.5 * drho) * gdz);
    }
    const bool up_a = nonneg(dpot);
    const size_t iu = up_a ? ia : ib;
    const double mob = a.pr[(3 * al) * n + iu], mp = a.pr[(3 * al + 1) * n + iu],
                 ms = a.pr[(3 * al + 2) * n + iu];
    // up- and downstream derivatives; zeros keep the two-sided formula's signs
    // (0 dpot is -0 for dpot < 0)
    double fl = 0.0, pu = up_a ? 0.0 : -0.0, su = up_a ? ms : flip(ms), pd = 0.0;
    double sd = pu;
    // a phase that does not move (residual saturation upstream): all zeros
    if (capw || !(is_zero(mob) && is_zero(mp) && is_zero(ms))) {
      const double tm = T * mob;
      fl = tm * dpot;
      if (grav) {
        pu = T * ((mp * dpot) + (mob * (up_a ? ddpa : ddpb)));
        pd = T * (mob * (up_a ? ddpb : ddpa));
      } else {
        pu = T * ((mp * dpot) + (up_a ? mob : flip(mob)));
        pd = up_a ? flip(tm) : tm;
      }
      if (is_zero(mob)) pd = 0.0;
      su = ms * dpot;
      if (capw) {   // - mob p_cow'(a) on a's side, + mob p_cow'(b) on b's
        const double ga = mob * a.pr[9 * n + ia], gb = mob * a.pr[9 * n + ib];
        su = up_a ? su - ga : su + gb;
        sd = T * (up_a ? (is_zero(gb) ? 0.0 : gb) : flip(ga));
      }
      su = T * su;
    }
    F[al] = fl;
    const double pa = up_a ? pu : pd, sa = up_a ? su : sd;
    fa[2 * al] = flip(pa);
    fa[2 * al + 1] = flip(sa);
    fb[2 * al] = up_a ? pd : pu;
    fb[2 * al + 1] = up_a ? sd : su;
  }
  store_block(a.val + 4 * (size_t)e.x, fb, a.wide);
  store_block(a.val + 4 * (size_t)e.y, fa, a.wide);
  a.fconn[c] = make_double2(F[0], F[1]);
}

// A perforated cell's properties, as the cell's own row evaluates them.
__device__ __forceinline__ void cell_props(const AsmArgs &a, int c, Props &q) {
  props(a.P, a.phi_f, a.phi_m, c, a.p[c], a.sw[c], q);
}

// The well rows, a warp per row: the lanes evaluate 32 perforations at once
// (a serial loop over them was the longest chain of the launch: 55 us at
// twenty perforations), then their terms are added one by one in the row's
// order, so that the sums are the serial ones.
__device__ __forceinline__ void well_row(const AsmArgs &a, int w, int lane) {
  const Phys &P = a.P;
  const int r = P.nc + w, e0 = a.rowptr[r], e1 = a.rowptr[r + 1], kind = a.well_kind[w];
  const double pb = a.bhp[w];
  double acc = 0.0, accd = 0.0;
  for (int base = e0; base < e1; base += 32) {
    const int e = base + lane;
    const bool in = e < e1 && a.col[e] != r;
    double q = 0.0, dqb0 = 0.0;
    if (in) {
      const int c = a.col[e];
      double2 o = make_double2(0.0, 0.0);
      if (kind == 0 || kind == 2) {
        Props qc;
        cell_props(a, c, qc);
        const double wi = a.trans[e];
        if (kind == 0) {
          double lt = qc.lam[0] + qc.lam[1], dlt = qc.dlam[0] + qc.dlam[1];
          double wl = wi * lt;
          q = wl * (pb - a.p[c]);
          dqb0 = wl;
          o = make_double2(-wl, (wi * dlt) * (pb - a.p[c]));
        } else {
          // oil-rate producer: the perforation oil rates into the cells sum to
          // minus the target (the oil leaving the reservoir equals the target)
          double Q[2], dq[4], dqb[2];
          perf_rate(2, wi, a.p[c], pb, qc, Q, dq, dqb);
          q = Q[0];
          dqb0 = dqb[0];
          o = make_double2(dq[0], dq[1]);
        }
      }
      double2 *off = reinterpret_cast<double2 *>(a.val + 4 * (size_t)e);
      off[0] = o;
      off[1] = make_double2(0.0, 0.0);
    }
    const unsigned m = __ballot_sync(0xffffffffu, in);
    if (kind != 0 && kind != 2) continue;
    for (int k = 0; k < 32; ++k) {
      double qk = __shfl_sync(0xffffffffu, q, k), dk = __shfl_sync(0xffffffffu, dqb0, k);
      if ((m >> k) & 1u) {
        acc = acc + qk;
        accd = accd + dk;
      }
    }
  }
  if (lane != 0) return;
  double d = 1.0, res;
  if (kind == 0) { res = acc - a.well_target[w]; d = accd; }
  else if (kind == 2) { res = acc + a.well_target[w]; d = accd; }
  else res = pb - a.well_target[w];
  double *dg = a.val + 4 * (size_t)a.diag[r];
  dg[0] = d; dg[1] = 0.0; dg[2] = 0.0; dg[3] = 1.0;
  a.R[2 * r] = res;
  a.R[2 * r + 1] = 0.0;
}

// One thread per cell row, after k_conn_flux; threads [0, nL) take the
// fracture rows, [nL, nc) the matrix rows, and the blocks from cell_blocks on
// the well rows.  Cell rows: accumulation, then the connections in increasing
// column order (the neighbours below along z, y, x, the matrix cell, the
// neighbours above along x, y, z): a neighbour d adds +F (d > r) or -F (d <
// r) of their connection to the residual and minus the transposed block (d,
// r) to the diagonal block (that block is -dF/dx_r written by k_conn_flux,
// so this adds exactly the dF/dx_r of the row-wise evaluation); then the
// perforations.  Zero terms are not added (the sum is the same).
__global__ void __launch_bounds__(kBlock) k_assemble(AsmArgs a, int cell_blocks) {
  const Phys &P = a.P;
  if ((int)blockIdx.x >= cell_blocks) {
    int w = ((blockIdx.x - cell_blocks) * blockDim.x + threadIdx.x) >> 5;
    if (w < P.nw) well_row(a, w, threadIdx.x & 31);   // whole warps
    return;
  }
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= P.nc) return;
  const bool mat = t >= P.nL;
  const int loc = mat ? t - P.nL : t, r = 2 * loc + (mat ? 1 : 0);
  const double sw = a.sw[r];
  Props qc;
  const size_t n = (size_t)P.nc, at = prop_at(P, r);
  qc.rho[0] = a.pr[6 * n + at];
  qc.rho[1] = a.pr[7 * n + at];
  qc.drho[0] = P.drho_o;
  qc.drho[1] = P.drho_w;
  const double phi_ref = mat ? a.phi_m[loc] : a.phi_f[loc];
  qc.phi = !P.rock ? phi_ref : phi_ref * (1.0 + P.c_rock * (a.p[r] - P.p_ref_rock));
  qc.dphi = !P.rock ? 0.0 : phi_ref * P.c_rock;
  double M[2], dM[4];
  accumulation(P, sw, qc, M, dM);
  reinterpret_cast<double2 *>(a.Macc)[r] = make_double2(M[0], M[1]);
  const double2 mn = reinterpret_cast<const double2 *>(a.Mn)[r];
  double r0 = (M[0] - mn.x) * a.inv_dt, r1 = (M[1] - mn.y) * a.inv_dt;
  double d0 = dM[0] * a.inv_dt, d1 = dM[1] * a.inv_dt;
  double d2 = dM[2] * a.inv_dt, d3 = dM[3] * a.inv_dt;
  // connection c[q] (none: not there) of which this row is cell a (low) or
  // cell b: the positions and fluxes of all N first, then their blocks, then
  // the sums
  auto conns = [&](auto &c, const auto &there, auto low) {
    constexpr int N = sizeof(c) / sizeof(c[0]);
    int te[N];
    double2 F[N];
    double tb[N][4];
#pragma unroll
    for (int q = 0; q < N; ++q) {
      te[q] = -1;
      if (there[q]) {
        const int2 e = a.cpos[c[q]];
        te[q] = low.value ? e.y : e.x;
        F[q] = a.fconn[c[q]];
      }
    }
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (te[q] >= 0) load_block(a.val + 4 * (size_t)te[q], tb[q], a.wide);
#pragma unroll
    for (int q = 0; q < N; ++q) {
      if (te[q] < 0) continue;
      r0 = low.value ? r0 + F[q].x : r0 - F[q].x;
      d0 = d0 - tb[q][0];
      if (!is_zero(tb[q][1])) d1 = d1 - tb[q][1];
      if (!(is_zero(F[q].y) && is_zero(tb[q][2]))) {
        r1 = low.value ? r1 + F[q].y : r1 - F[q].y;
        d2 = d2 - tb[q][2];
      }
      if (!is_zero(tb[q][3])) d3 = d3 - tb[q][3];
    }
  };
  const size_t nL = (size_t)P.nL;
  if (mat) {
    const size_t c[1] = {3 * nL + loc};
    const bool there[1] = {true};
    conns(c, there, std::false_type{});
  } else {
    int i, j, k;
    loc_ijk(P, loc, i, j, k);
    {
      const size_t c[3] = {2 * nL + loc - (size_t)P.nx * P.ny, nL + loc - P.nx, (size_t)loc - 1};
      const bool there[3] = {k > 0, j > 0, i > 0};
      conns(c, there, std::false_type{});
    }
    {
      const size_t c[4] = {3 * nL + loc, (size_t)loc, nL + loc, 2 * nL + loc};
      const bool there[4] = {true, i < P.nx - 1, j < P.ny - 1, k < P.nz - 1};
      conns(c, there, std::true_type{});
    }
    // the perforations come after all cells
    const int cells = 2 + (i > 0) + (j > 0) + (k > 0) + (i < P.nx - 1) + (j < P.ny - 1) +
                      (k < P.nz - 1);
    for (int e = a.rowptr[r] + cells, e1 = a.rowptr[r + 1]; e < e1; ++e) {
      const int w = a.col[e] - P.nc;
      Props q;
      cell_props(a, r, q);
      double Q[2], dq[4], dqb[2];
      perf_rate(a.well_kind[w], a.trans[e], a.p[r], a.bhp[w], q, Q, dq, dqb);
      r0 = r0 - Q[0]; r1 = r1 - Q[1];
      d0 = d0 - dq[0]; d1 = d1 - dq[1]; d2 = d2 - dq[2]; d3 = d3 - dq[3];
      double *off = a.val + 4 * (size_t)e;
      off[0] = -dqb[0]; off[1] = 0.0; off[2] = -dqb[1]; off[3] = 0.0;
    }
  }
  const double dg[4] = {d0, d1, d2, d3};
  store_block(a.val + 4 * (size_t)a.diag[r], dg, a.wide);
  reinterpret_cast<double2 *>(a.R)[r] = make_double2(r0, r1);
}

__global__ void k_save_old(Phys P, const double *phi_f, const double *phi_m, const double *p,
                           const double *sw, const double *bhp, double *pn, double *swn,
                           double *bhpn, double *Mn) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < P.nw) bhpn[c] = bhp[c];
  if (c >= P.nc) return;
  Props q;
  props(P, phi_f, phi_m, c, p[c], sw[c], q);
  double M[2], dM[4];
  accumulation(P, sw[c], q, M, dM);
  pn[c] = p[c];
  swn[c] = sw[c];
  Mn[2 * c] = M[0];
  Mn[2 * c + 1] = M[1];
}

int phys_save_old(Sim *s) {
  Phys &P = s->ph;
  int n = std::max(P.nc, P.nw);
  DP_LAUNCH(s, k_save_old, nblk(n), kBlock, 0, P, s->phi_f, s->phi_m, s->p, s->sw, s->bhp, s->pn,
            s->swn, s->bhpn, s->Mn);
  DP_CUDA(s, cudaGetLastError());
  return DP_OK;
}

// Per well, the oil and water mass rates into the reservoir summed over its
// perforations (Section 2's perforation rates).  One thread per well; the
// perforations are sorted by (cell, well), so a well's own perforations come
// in increasing cell order, from the top layer down.
__global__ void k_well_rates(Phys P, const double *phi_f, const double *phi_m, const double *p,
                             const double *sw, const double *bhp, const int *perf_cell,
                             const int *perf_well, const double *perf_wi, int np,
                             const int *well_kind, double *q_oil, double *q_water) {
  int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= P.nw) return;
  double qo = 0.0, qw = 0.0;
  for (int t = 0; t < np; ++t) {
    if (perf_well[t] != w) continue;
    int c = perf_cell[t];
    Props q;
    props(P, phi_f, phi_m, c, p[c], sw[c], q);
    double Q[2], dq[4], dqb[2];
    perf_rate(well_kind[w], perf_wi[t], p[c], bhp[w], q, Q, dq, dqb);
    qo = qo + Q[0];
    qw = qw + Q[1];
  }
  q_oil[w] = qo;
  q_water[w] = qw;
}

int phys_well_rates(Sim *s, double *q) {
  if (s->ph.nw == 0) return DP_OK;
  DP_LAUNCH(s, k_well_rates, nblk(s->ph.nw), kBlock, 0, s->ph, s->phi_f, s->phi_m, s->p, s->sw,
            s->bhp, s->perf_cell, s->perf_well, s->perf_wi, s->nperf, s->well_kind, q,
            q + s->ph.nw);
  DP_CUDA(s, cudaGetLastError());
  return DP_OK;
}

// Well controls.  restore: every well back on its own control (start of a
// timestep).  Otherwise, after a Newton update: an injector above its BHP
// limit, or an oil-rate producer below it, goes on BHP control at the limit.
__global__ void k_well_controls(int nw, int restore, const int *ctl_kind, const double *ctl_target,
                                const double *limit, const double *bhp, int *kind, double *target) {
  int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= nw) return;
  if (restore) {
    kind[w] = ctl_kind[w];
    target[w] = ctl_target[w];
    return;
  }
  double lim = limit[w];
  if (lim <= 0.0) return;
  int k = kind[w];
  if ((k == 0 && bhp[w] > lim) || (k == 2 && bhp[w] < lim)) {
    kind[w] = 1;
    target[w] = lim;
  }
}

int phys_well_controls(Sim *s, bool restore) {
  if (s->ph.nw == 0) return DP_OK;
  DP_LAUNCH(s, k_well_controls, nblk(s->ph.nw), kBlock, 0, s->ph.nw, restore ? 1 : 0,
            s->well_ctl_kind, s->well_ctl_target, s->well_limit, s->bhp, s->well_kind,
            s->well_target);
  DP_CUDA(s, cudaGetLastError());
  return DP_OK;
}

int phys_assemble(Sim *s) {
  const Phys &P = s->ph;
  bool grav = P.g != 0.0, cap = P.pc_n[0] > 0 || P.pc_n[1] > 0;
  if (cap)
    DP_LAUNCH(s, k_props<true>, nblk(P.nc), kBlock, 0, P, s->phi_f, s->phi_m, s->p, s->sw, s->pr);
  else
    DP_LAUNCH(s, k_props<false>, nblk(P.nc), kBlock, 0, P, s->phi_f, s->phi_m, s->p, s->sw, s->pr);
  AsmArgs a;
  a.P = P;
  a.rowptr = s->A.rowptr; a.col = s->A.col; a.diag = s->A.diag; a.cpos = s->cpos;
  a.trans = s->trans; a.ctrans = s->ctrans;
  a.phi_f = s->phi_f; a.phi_m = s->phi_m; a.pr = s->pr; a.Macc = s->Macc;
  a.p = s->p; a.sw = s->sw; a.bhp = s->bhp; a.Mn = s->Mn;
  a.well_kind = s->well_kind; a.well_target = s->well_target;
  a.val = s->A.val; a.R = s->R;
  a.fconn = reinterpret_cast<double2 *>(s->fconn);
  a.inv_dt = s->inv_dt;
  a.wide = ((uintptr_t)s->A.val & 31) == 0;
  void (*k_conn_flux_sel)(AsmArgs) =
      cap ? (grav ? k_conn_flux<true, true> : k_conn_flux<false, true>)
          : (grav ? k_conn_flux<true, false> : k_conn_flux<false, false>);
  DP_LAUNCH(s, k_conn_flux_sel, dim3(nblk(P.nL), 4), kBlock, 0, a);
  int cells = nblk(P.nc), wells = P.nw ? nblk(32LL * P.nw) : 0;
  DP_LAUNCH(s, k_assemble, cells + wells, kBlock, 0, a, cells);
  DP_CUDA(s, cudaGetLastError());
  return DP_OK;
}

// ---------------------------------------------------------------- norms
// Scaled residual (cell rows by dt / (rho_ref phi_ref V), well rows by
// their target), phase residual sums, mass change and well inflow.  Two
// passes with a fixed reduction order (deterministic for a given size).

// max of non-negative doubles as integers (a NaN counts as 0, as fmax drops it)
__device__ __forceinline__ long long max_bits(double v) {
  long long b = __double_as_longlong(v) & 0x7fffffffffffffffll;
  return b > 0x7ff0000000000000ll ? 0 : b;
}
__device__ __forceinline__ double warp_max_bits(long long b) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    long long t = __shfl_xor_sync(0xffffffffu, b, o);
    if (t > b) b = t;
  }
  return __longlong_as_double(b);
}
// Eight sums over a warp in nine FP64 additions a lane instead of forty: the
// lanes halve the values between them while they exchange.  Lane 4 k returns
// the sum of v[k] (all lanes of that group of four).
__device__ __forceinline__ double warp_sum8(const double (&v)[8], int lane) {
  double a[4], b[2], c;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    double keep = lane & 16 ? v[k + 4] : v[k], send = lane & 16 ? v[k] : v[k + 4];
    a[k] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    double keep = lane & 8 ? a[k + 2] : a[k], send = lane & 8 ? a[k] : a[k + 2];
    b[k] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
  {
    double keep = lane & 4 ? b[1] : b[0], send = lane & 4 ? b[0] : b[1];
    c = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  }
  c += __shfl_xor_sync(0xffffffffu, c, 2);
  c += __shfl_xor_sync(0xffffffffu, c, 1);
  return c;
}

// The cell rows' weights of the scaled residual, 1 / (rho_ref phi_ref V) per
// cell and phase, formed once (an FP64 division per entry is a long
// instruction sequence on this GPU; the norms then multiply).
__global__ void k_norm_weights(Phys P, const double *phi_f, const double *phi_m, double *w) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= P.nc) return;
  int loc = c >> 1;
  double phi_ref = (c & 1) == 0 ? phi_f[loc] : phi_m[loc];
  w[2 * c] = 1.0 / ((P.rho_o_ref * phi_ref) * P.V);
  w[2 * c + 1] = 1.0 / ((P.rho_w_ref * phi_ref) * P.V);
}

int phys_norm_weights(Sim *s) {
  DP_LAUNCH(s, k_norm_weights, nblk(s->ph.nc), kBlock, 0, s->ph, s->phi_f, s->phi_m, s->norm_w);
  DP_CUDA(s, cudaGetLastError());
  return DP_OK;
}

// With lq (the linear residual of the last solve; null when the forcing term
// does not use it) also the squared scaled norm of lq, in the scaling of the
// residual norm, and with diff (forcing term 1) that of R - lq.
__global__ void __launch_bounds__(kBlock) k_norms_part(Phys P, const double *__restrict__ w,
                                                       const double *R,
                                                       const double *Macc, const double *Mn,
                                                       const int *well_kind,
                                                       const double *well_target, double dt,
                                                       const double *__restrict__ lq, int diff,
                                                       double *part) {
  // s2, (the max, apart), sro, srw, dmo, dmw, |lq|^2, |R-lq|^2
  double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  long long mx = 0;
  const double2 *R2 = reinterpret_cast<const double2 *>(R);
  const double2 *M2 = reinterpret_cast<const double2 *>(Macc);
  const double2 *O2 = reinterpret_cast<const double2 *>(Mn);
  const double2 *W2 = reinterpret_cast<const double2 *>(w);
  const double2 *L2 = reinterpret_cast<const double2 *>(lq);
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < P.nb; r += gridDim.x * blockDim.x) {
    if (r < P.nc) {   // explicit FMAs: this kernel is FP64-bound
      double2 Rr = R2[r], M = M2[r], O = O2[r], W = W2[r];
      const double w0 = W.x * dt, w1 = W.y * dt;
      double x0 = Rr.x * w0, x1 = Rr.y * w1;
      v[0] = fma(x0, x0, v[0]);
      v[0] = fma(x1, x1, v[0]);
      mx = max(mx, max(max_bits(x0), max_bits(x1)));
      if (lq) {
        double2 l = L2[r];
        double a0 = l.x * w0, a1 = l.y * w1;
        v[6] = fma(a0, a0, v[6]);
        v[6] = fma(a1, a1, v[6]);
        if (diff) {
          double e0 = x0 - a0, e1 = x1 - a1;   // R~(R - lq), scaled as R and lq are
          v[7] = fma(e0, e0, v[7]);
          v[7] = fma(e1, e1, v[7]);
        }
      }
      v[2] += Rr.x;
      v[3] += Rr.y;
      v[4] += M.x - O.x;
      v[5] += M.y - O.y;
    } else {
      int wl = r - P.nc;
      double sc = well_kind[wl] == 0 ? fmax(well_target[wl], 1e-12) : well_target[wl];
      double x = R[2 * r] / sc;
      v[0] = fma(x, x, v[0]);
      mx = max(mx, max_bits(x));
      if (lq) {
        double a = lq[2 * r] / sc, d = (R[2 * r] - lq[2 * r]) / sc;
        v[6] = fma(a, a, v[6]);
        v[7] = fma(d, d, v[7]);
      }
    }
  }
  __shared__ double sh[kBlock / 32][8];
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double t = warp_sum8(v, lane), m = warp_max_bits(mx);
  if ((lane & 3) == 0) sh[wid][lane >> 2] = lane == 4 ? m : t;
  __syncthreads();
  if (threadIdx.x < 8) {
    int k = threadIdx.x;
    double t = 0.0;
    for (int q = 0; q < kBlock / 32; ++q) t = k == 1 ? fmax(t, sh[q][k]) : t + sh[q][k];
    part[blockIdx.x * 8 + k] = t;
  }
}

// One block: partials and perforation rates summed in a fixed order.
__global__ void __launch_bounds__(kBlock) k_norms_final(Phys P, const double *phi_f,
                                                        const double *phi_m, const double *p,
                                                        const double *sw, const double *bhp,
                                                        const int *perf_cell, const int *perf_well,
                                                        const double *perf_wi, int np,
                                                        const int *well_kind, const double *part,
                                                        int nparts, double *out) {
  // v: s2, |R-lq|^2, sro, srw, dmo, dmw, the wells' oil and water; apart: max, |lq|^2
  double v[8] = {0, 0, 0, 0, 0, 0, 0, 0}, l2 = 0.0;
  long long mx = 0;
  for (int b = threadIdx.x; b < nparts; b += blockDim.x) {
    const double *q = part + b * 8;
    v[0] += q[0];
    mx = max(mx, max_bits(q[1]));
    for (int k = 2; k < 6; ++k) v[k] += q[k];
    l2 += q[6];
    v[1] += q[7];
  }
  for (int t = threadIdx.x; t < np; t += blockDim.x) {
    int c = perf_cell[t], w = perf_well[t];
    Props q;
    props(P, phi_f, phi_m, c, p[c], sw[c], q);
    double Q[2], dq[4], dqb[2];
    perf_rate(well_kind[w], perf_wi[t], p[c], bhp[w], q, Q, dq, dqb);
    v[6] += Q[0];
    v[7] += Q[1];
  }
  __shared__ double sh[kBlock / 32][10];
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double t = warp_sum8(v, lane), m = warp_max_bits(mx);
  l2 = warp_sum(l2);
  // out's order: 1 the max, 8 |lq|^2, 9 |R-lq|^2
  if ((lane & 3) == 0) sh[wid][lane == 4 ? 9 : lane >> 2] = t;
  if (lane == 0) {
    sh[wid][1] = m;
    sh[wid][8] = l2;
  }
  __syncthreads();
  int k = threadIdx.x;
  if (k >= 10) return;
  double o = 0.0;
  for (int q = 0; q < kBlock / 32; ++q) o = k == 1 ? fmax(o, sh[q][k]) : o + sh[q][k];
  out[k] = k == 0 || k >= 8 ? sqrt(o) : o;   // 8: ||R~(lq)||_2, 9: ||R~(R - lq)||_2
}

int phys_norms(Sim *s) {
  Phys &P = s->ph;
  bool lin = s->have_lq && (s->opt.eta_mode == 1 || s->opt.eta_mode == 2);
  DP_LAUNCH(s, k_norms_part, s->norm_blocks, kBlock, 0, P, s->norm_w, s->R, s->Macc,
            s->Mn, s->well_kind, s->well_target, s->dt, lin ? s->lq : nullptr,
            s->opt.eta_mode == 1 ? 1 : 0, s->norm_part);
  DP_LAUNCH(s, k_norms_final, 1, kBlock, 0, P, s->phi_f, s->phi_m, s->p, s->sw, s->bhp, s->perf_cell,
            s->perf_well, s->perf_wi, s->nperf, s->well_kind, s->norm_part, s->norm_blocks,
            s->norm_out);
  DP_CUDA(s, cudaGetLastError());
  return DP_OK;
}

// ---------------------------------------------------------------- decoupling
// Per cell block row (Eq. "decoupled-eq"), well rows unchanged; the pressure
// block takes entry (0,0) of every decoupled block.  Mode 0: the paper's
// modified Gauss-Jordan step, read as the elimination of the pressure row's
// saturation coefficient by the water row of the diagonal block, D_i^-1 =
// [[1, -a01/a11], [0, 1]] (the per-cell Quasi-IMPES form); mode 1: ABF,
// D_i^-1 = the inverse of the diagonal block; mode 2: True-IMPES, the weight
// c01/c11 from the sums of block column i over all rows, in increasing row
// order (read through the transpose positions of row i's entries).
//
// Two passes: one thread per row takes the row's weight or inverse (the
// divisions once per row) and the right-hand side; then one thread per
// entry, in natural order (coalesced reads of the Jacobian), writes the
// decoupled block wherever it is consumed: the pressure block ap (natural
// order), the storage-order copy of the Krylov operator (sval, and
// sa00/sa01 for the pressure residual), the ILU(0) factor's starting values
// in its split layout and precision, and the colour-ordered level-0 copy of
// the Gauss-Seidel sweeps.  The Jacobian itself is left as assembled.
__global__ void __launch_bounds__(kBlock) k_decouple_rows(int nb, int nc, int mode,
                                                          const int *rowptr, const int *diag,
                                                          const int *tpos, const double *val,
                                                          const double *R, double *fct,
                                                          double *bh) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nb) return;
  double b0 = -R[2 * i], b1 = -R[2 * i + 1];
  if (i >= nc) {
    bh[2 * i] = b0;
    bh[2 * i + 1] = b1;
    return;
  }
  const double *dg = val + 4 * (size_t)diag[i];
  if (mode == 1) {
    double d00 = dg[0], d01 = dg[1], d10 = dg[2], d11 = dg[3];
    double det = (d00 * d11) - (d01 * d10);
    double *f = fct + 4 * (size_t)i;
    if (fabs(det) < 1e-300) {
      f[0] = 1.0; f[1] = 0.0; f[2] = 0.0; f[3] = 1.0;   // row left as it is
      bh[2 * i] = b0;
      bh[2 * i + 1] = b1;
      return;
    }
    double i00 = d11 / det, i01 = (-d01) / det, i10 = (-d10) / det, i11 = d00 / det;
    f[0] = i00; f[1] = i01; f[2] = i10; f[3] = i11;
    bh[2 * i] = (i00 * b0) + (i01 * b1);
    bh[2 * i + 1] = (i10 * b0) + (i11 * b1);
    return;
  }
  double w;
  if (mode == 2) {
    double c01 = 0.0, c11 = 0.0;
    for (int e = rowptr[i]; e < rowptr[i + 1]; ++e) {
      const double *a = val + 4 * (size_t)tpos[e];
      c01 = c01 + a[1];
      c11 = c11 + a[3];
    }
    w = fabs(c11) < 1e-300 ? 0.0 : c01 / c11;
  } else {
    double a01 = dg[1], a11 = dg[3];
    w = fabs(a11) < 1e-300 ? 0.0 : a01 / a11;
  }
  fct[i] = w;
  bh[2 * i] = b0 - (w * b1);
  bh[2 * i + 1] = b1;
}

struct DecArgs {
  long long nnz;
  int nc, sL, sc, mode;   // rows below nc are cell rows; storage mapping (sL, sc)
  const int *erow, *rowptr, *srowptr, *ilupos, *l0pos;
  const double *val, *fct;
  double *ap, *sval, *sa00, *sa01;
  float *svalf, *spf;   // FP32 copies for the preconditioner's residuals, or null
  void *lu;         // split-layout factor values (float or double), or null
  void *l0;         // colour-ordered level-0 pressure values, or null
};

template <typename T>
__global__ void __launch_bounds__(kBlock) k_decouple(DecArgs a) {
  long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= a.nnz) return;
  int i = __ldg(a.erow + e);
  const double2 *v2 = reinterpret_cast<const double2 *>(a.val) + 2 * e;
  double2 u = v2[0], w = v2[1];
  double n0 = u.x, n1 = u.y, n2 = w.x, n3 = w.y;
  if (i < a.nc) {
    if (a.mode == 1) {
      const double *f = a.fct + 4 * (size_t)i;
      double i00 = f[0], i01 = f[1], i10 = f[2], i11 = f[3];
      bool keep = i00 == 1.0 && i01 == 0.0 && i10 == 0.0 && i11 == 1.0;   // singular pivot
      double v0 = n0, v1 = n1, v2 = n2, v3 = n3;
      if (!keep) {
        n0 = (i00 * v0) + (i01 * v2);
        n1 = (i00 * v1) + (i01 * v3);
        n2 = (i10 * v0) + (i11 * v2);
        n3 = (i10 * v1) + (i11 * v3);
      }
    } else {
      double f = a.fct[i];
      n0 = n0 - (f * n2);
      n1 = n1 - (f * n3);
    }
  }
  a.ap[e] = n0;
  int si = storage_row(i, a.sL, a.sc);
  size_t q = (size_t)(__ldg(a.srowptr + si) + (int)(e - __ldg(a.rowptr + i)));
  double2 *sv = reinterpret_cast<double2 *>(a.sval) + 2 * q;
  sv[0] = make_double2(n0, n1);
  sv[1] = make_double2(n2, n3);
  if (a.sa00) {
    a.sa00[q] = n0;
    a.sa01[q] = n1;
  }
  // converted once, stored as blocks: 200 x 200 x 50 cells, 457 -> 424 us
  const T t[4] = {narrow_to<T>(n0), narrow_to<T>(n1), narrow_to<T>(n2), narrow_to<T>(n3)};
  if constexpr (sizeof(T) == 4)
    if (a.svalf) {
      Blk<float>::store(a.svalf + 4 * q, t);
      reinterpret_cast<float2 *>(a.spf)[q] = make_float2(t[0], t[1]);
    }
  if (a.lu) Blk<T>::store(reinterpret_cast<T *>(a.lu) + 4 * (size_t)__ldg(a.ilupos + e), t);
  if (a.l0) reinterpret_cast<T *>(a.l0)[__ldg(a.l0pos + e)] = t[0];
}

int phys_decouple_extract(Sim *s) {
  int mode = s->opt.decouple;
  const Bsr &K = s->K;
  DP_LAUNCH(s, k_decouple_rows, nblk(K.n), kBlock, 0, K.n, s->sv_cells, mode, K.rowptr, K.diag,
            s->btpos, K.val, s->Rk, s->fct, s->bh);
  DecArgs a;
  a.nnz = K.nnz; a.nc = s->sv_cells; a.sL = s->sv_sL; a.sc = s->sv_sc; a.mode = mode;
  a.erow = s->erow; a.rowptr = K.rowptr; a.srowptr = s->srowptr;
  a.ilupos = s->ilupos; a.l0pos = s->l0pos;
  a.val = K.val; a.fct = s->fct;
  a.ap = s->ap; a.sval = s->sval; a.sa00 = s->sa00; a.sa01 = s->sa01;
  a.svalf = s->svalf; a.spf = s->spf;
  bool f32 = s->opt.precision >= 1;
  a.lu = s->opt.precond >= 1 ? (f32 ? (void *)s->lu_valf : (void *)s->lu_val) : nullptr;
  a.l0 = s->l0_lu ? (f32 ? (void *)s->l0_pvf : (void *)s->l0_pv) : nullptr;
  if (f32) DP_LAUNCH(s, k_decouple<float>, nblk(K.nnz), kBlock, 0, a);
  else DP_LAUNCH(s, k_decouple<double>, nblk(K.nnz), kBlock, 0, a);
  DP_CUDA(s, cudaGetLastError());
  return DP_OK;
}

// The decoupled matrix in natural order, from its storage-order copy (test
// access: the Jacobian itself stays as assembled).
__global__ void k_natural_from_storage(long long nnz, int nc, int nL, const int *erow,
                                       const int *rowptr, const int *srowptr, const double *sval,
                                       double *out) {
  long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nnz) return;
  int i = erow[e];
  size_t q = (size_t)(srowptr[storage_row(i, nL, nc)] + (int)(e - rowptr[i]));
  for (int k = 0; k < 4; ++k) out[4 * e + k] = sval[4 * q + k];
}

int phys_decoupled_natural(Sim *s, double *out) {
  DP_LAUNCH(s, k_natural_from_storage, nblk(s->K.nnz), kBlock, 0, (long long)s->K.nnz, s->sv_sc,
            s->sv_sL, s->erow, s->K.rowptr, s->srowptr, s->sval, out);
  DP_CUDA(s, cudaGetLastError());
  return DP_OK;
}

// ---------------------------------------------------------------- Schur option
// Exact elimination of the matrix continuum: a matrix cell m of location loc
// couples only to itself and to its fracture cell f, so y_m = A_mm^-1 (-R_m
// - A_mf y_f), and the fracture row takes S_ff = A_ff - A_fm A_mm^-1 A_mf and
// the residual R_f - A_fm A_mm^-1 R_m.  K keeps the fracture rows (row loc)
// and the well rows (row nL + w); its other blocks are copies of A's.  The
// formulas are evaluated as written, in the order the oracle uses.

__device__ __forceinline__ int kcol(int c, int nL, int nc) {   // -1: a matrix column, dropped
  return c >= nc ? nL + (c - nc) : ((c & 1) ? -1 : c >> 1);
}

__global__ void k_schur_len(int nk, int nL, int nc, const int *rowptr, const int *col, int *len) {
  int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= nk) return;
  int jr = r < nL ? 2 * r : nc + (r - nL), c = 0;
  for (int e = rowptr[jr]; e < rowptr[jr + 1]; ++e) c += kcol(col[e], nL, nc) >= 0;
  len[r] = c;
}

__global__ void k_schur_fill(int nk, int nL, int nc, const int *rowptr, const int *col,
                             const int *krowptr, int *kcolv, int *kdiag, int *kmap) {
  int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= nk) return;
  int jr = r < nL ? 2 * r : nc + (r - nL), k = krowptr[r];
  for (int e = rowptr[jr]; e < rowptr[jr + 1]; ++e) {
    int c = kcol(col[e], nL, nc);
    if (c < 0) continue;
    kcolv[k] = c;
    kmap[k] = (r < nL && c == r) ? -1 : e;
    if (c == r) kdiag[r] = k;
    ++k;
  }
}

__device__ __forceinline__ int find_col_in(const int *col, int lo, int hi, int c) {
  while (lo < hi) {
    int m = (lo + hi) >> 1;
    if (col[m] == c) return m;
    if (col[m] < c) lo = m + 1; else hi = m;
  }
  return -1;
}

__global__ void k_schur_pos(int nL, const int *rowptr, const int *col, int *pos_fm, int *pos_mf) {
  int loc = blockIdx.x * blockDim.x + threadIdx.x;
  if (loc >= nL) return;
  int f = 2 * loc, m = f + 1;
  pos_fm[loc] = find_col_in(col, rowptr[f], rowptr[f + 1], m);
  pos_mf[loc] = find_col_in(col, rowptr[m], rowptr[m + 1], f);
}

__global__ void k_schur_copy(long long nnzk, const int *kmap, const double *val, double *kval) {
  long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nnzk) return;
  int e = kmap[k];
  if (e < 0) return;
  const double2 *src = reinterpret_cast<const double2 *>(val) + 2 * (size_t)e;
  double2 *dst = reinterpret_cast<double2 *>(kval) + 2 * k;
  dst[0] = src[0];
  dst[1] = src[1];
}

__global__ void k_schur_loc(int nL, int nc, int nw, const int *diag, const int *pos_fm,
                            const int *pos_mf, const int *kdiag, const double *val,
                            const double *R, double *kval, double *RK, double *Minv) {
  int loc = blockIdx.x * blockDim.x + threadIdx.x;
  if (loc < nw) {
    RK[2 * (nL + loc)] = R[2 * (nc + loc)];
    RK[2 * (nL + loc) + 1] = R[2 * (nc + loc) + 1];
  }
  if (loc >= nL) return;
  int f = 2 * loc, m = f + 1;
  const double *amm = val + 4 * (size_t)diag[m];
  const double *amf = val + 4 * (size_t)pos_mf[loc];
  const double *afm = val + 4 * (size_t)pos_fm[loc];
  const double *aff = val + 4 * (size_t)diag[f];
  double det = (amm[0] * amm[3]) - (amm[1] * amm[2]);
  double m0, m1, m2, m3;
  if (fabs(det) < 1e-300) { m0 = 0.0; m1 = 0.0; m2 = 0.0; m3 = 0.0; }
  else { m0 = amm[3] / det; m1 = (-amm[1]) / det; m2 = (-amm[2]) / det; m3 = amm[0] / det; }
  double *mi = Minv + 4 * (size_t)loc;
  mi[0] = m0; mi[1] = m1; mi[2] = m2; mi[3] = m3;
  double x00 = (afm[0] * m0) + (afm[1] * m2);
  double x01 = (afm[0] * m1) + (afm[1] * m3);
  double x10 = (afm[2] * m0) + (afm[3] * m2);
  double x11 = (afm[2] * m1) + (afm[3] * m3);
  double *sk = kval + 4 * (size_t)kdiag[loc];
  sk[0] = aff[0] - ((x00 * amf[0]) + (x01 * amf[2]));
  sk[1] = aff[1] - ((x00 * amf[1]) + (x01 * amf[3]));
  sk[2] = aff[2] - ((x10 * amf[0]) + (x11 * amf[2]));
  sk[3] = aff[3] - ((x10 * amf[1]) + (x11 * amf[3]));
  double rm0 = R[2 * m], rm1 = R[2 * m + 1];
  RK[2 * loc] = R[2 * f] - ((x00 * rm0) + (x01 * rm1));
  RK[2 * loc + 1] = R[2 * f + 1] - ((x10 * rm0) + (x11 * rm1));
}

__global__ void k_schur_back(int nL, int nc, int nw, const int *pos_mf, const double *val,
                             const double *Minv, const double *R, const double *yk, double *y) {
  int loc = blockIdx.x * blockDim.x + threadIdx.x;
  if (loc < nw) {
    y[2 * (nc + loc)] = yk[2 * (nL + loc)];
    y[2 * (nc + loc) + 1] = yk[2 * (nL + loc) + 1];
  }
  if (loc >= nL) return;
  int f = 2 * loc, m = f + 1;
  double yf0 = yk[2 * loc], yf1 = yk[2 * loc + 1];
  const double *amf = val + 4 * (size_t)pos_mf[loc];
  const double *mi = Minv + 4 * (size_t)loc;
  double t0 = (-R[2 * m]) - ((amf[0] * yf0) + (amf[1] * yf1));
  double t1 = (-R[2 * m + 1]) - ((amf[2] * yf0) + (amf[3] * yf1));
  y[2 * f] = yf0;
  y[2 * f + 1] = yf1;
  y[2 * m] = (mi[0] * t0) + (mi[1] * t1);
  y[2 * m + 1] = (mi[2] * t0) + (mi[3] * t1);
}

int phys_solver_view(Sim *s) {
  Phys &P = s->ph;
  if (!s->opt.schur) {
    s->K = s->A;
    s->sv_sL = P.nL; s->sv_sc = P.nc; s->sv_cells = P.nc; s->sv_long0 = P.nc;
    s->Rk = s->R;
    s->yk = s->y;
    return DP_OK;
  }
  Bsr &K = s->K;
  int nk = P.nL + P.nw;
  K.n = nk;
  K.rowptr = (int *)dalloc(s, ((size_t)nk + 1) * 4);
  K.diag = (int *)dalloc(s, (size_t)nk * 4);
  int *len = (int *)dalloc(s, (size_t)nk * 4);
  if (!K.rowptr || !K.diag || !len) { s->fail(DP_ENOMEM, "allocation failed"); return DP_ENOMEM; }
  DP_LAUNCH(s, k_schur_len, nblk(nk), kBlock, 0, nk, P.nL, P.nc, s->A.rowptr, s->A.col, len);
  int nnz = 0;
  DP_TRY(scan_i32(s, len, K.rowptr, nk, &nnz));
  K.nnz = nnz;
  K.col = (int *)dalloc(s, (size_t)nnz * 4);
  K.val = (double *)dalloc(s, (size_t)nnz * 32);
  s->kmap = (int *)dalloc(s, (size_t)nnz * 4);
  s->pos_fm = (int *)dalloc(s, (size_t)P.nL * 4);
  s->pos_mf = (int *)dalloc(s, (size_t)P.nL * 4);
  s->Minv = (double *)dalloc(s, (size_t)P.nL * 32);
  s->Rk = (double *)dalloc(s, (size_t)nk * 16);
  s->yk = (double *)dalloc(s, (size_t)nk * 16);
  if (!K.col || !K.val || !s->kmap || !s->pos_fm || !s->pos_mf || !s->Minv || !s->Rk || !s->yk) {
    s->fail(DP_ENOMEM, "allocation failed");
    return DP_ENOMEM;
  }
  DP_LAUNCH(s, k_schur_fill, nblk(nk), kBlock, 0, nk, P.nL, P.nc, s->A.rowptr, s->A.col, K.rowptr,
            K.col, K.diag, s->kmap);
  DP_LAUNCH(s, k_schur_pos, nblk(P.nL), kBlock, 0, P.nL, s->A.rowptr, s->A.col, s->pos_fm,
            s->pos_mf);
  dfree(s, len);
  // K's rows are already grouped (fracture rows, then wells): its storage
  // order is its natural order
  dfree(s, s->srowptr);
  dfree(s, s->scol);
  s->srowptr = K.rowptr;
  s->scol = K.col;
  s->sv_sL = 0; s->sv_sc = 0; s->sv_cells = P.nL; s->sv_long0 = P.nL;
  DP_CUDA(s, cudaGetLastError());
  return DP_OK;
}

int phys_schur_reduce(Sim *s) {
  Phys &P = s->ph;
  DP_LAUNCH(s, k_schur_copy, nblk(s->K.nnz), kBlock, 0, (long long)s->K.nnz, s->kmap, s->A.val,
            s->K.val);
  DP_LAUNCH(s, k_schur_loc, nblk(std::max(P.nL, P.nw)), kBlock, 0, P.nL, P.nc, P.nw, s->A.diag,
            s->pos_fm, s->pos_mf, s->K.diag, s->A.val, s->R, s->K.val, s->Rk, s->Minv);
  DP_CUDA(s, cudaGetLastError());
  return DP_OK;
}

int phys_schur_back(Sim *s) {
  Phys &P = s->ph;
  DP_LAUNCH(s, k_schur_back, nblk(std::max(P.nL, P.nw)), kBlock, 0, P.nL, P.nc, P.nw, s->pos_mf,
            s->A.val, s->Minv, s->R, s->yk, s->y);
  DP_CUDA(s, cudaGetLastError());
  return DP_OK;
}

// ---------------------------------------------------------------- update
__global__ void k_update(int nc, int nw, double ds_max, const double *y, double *p, double *sw,
                         double *bhp) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < nw) bhp[c] += y[2 * (nc + c)];
  if (c >= nc) return;
  p[c] += y[2 * c];
  double ds = y[2 * c + 1];
  if (ds > ds_max) ds = ds_max;
  if (ds < -ds_max) ds = -ds_max;
  double v = sw[c] + ds;
  if (v < 0.0) v = 0.0;
  if (v > 1.0) v = 1.0;
  sw[c] = v;
}

int phys_update(Sim *s) {
  int n = std::max(s->ph.nc, s->ph.nw);
  DP_LAUNCH(s, k_update, nblk(n), kBlock, 0, s->ph.nc, s->ph.nw, s->opt.ds_max, s->y, s->p, s->sw,
            s->bhp);
  DP_CUDA(s, cudaGetLastError());
  return DP_OK;
}

}  // namespace dp
