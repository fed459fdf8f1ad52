// The coarse part of the AMG V-cycle in one launch of one thread-block
// cluster.
//
// Below a size threshold every level of the hierarchy is small, but its
// multicolour Gauss-Seidel still needs one ordered phase per colour (17-46
// colours per level on the 8M-unknown problem), and even l1-Jacobi needs a
// few phases per level.  Launching a kernel per phase costs more than the
// phase's work.  Here one cluster of CTAs (up to
// 16 CTAs of 512 threads, one per SM of a GPC) runs all phases of levels l0..L-1: the colour
// sweeps, residuals, restrictions, the dense coarsest solve and the
// prolongations, separated by hardware cluster barriers (barrier.cluster
// with release/acquire semantics).
//
// What bounds it is latency: a phase has a few hundred rows, and its chain
// of dependent steps (colour bounds, entries, gathers, sum, store, barrier)
// was five L2 round trips, 2.2-5.1 us a phase.  So every CTA keeps a replica
// of the levels' vectors in its own shared memory: a row's result goes to
// all replicas at once (a row's lanes split the CTAs between them, stores
// through distributed shared memory), the gathers read the CTA's own copy,
// and between its arrival at a barrier and its wait a thread loads what the
// next phase needs that no phase writes (its rows' columns, values, 1/a_ii).
// What is left of a phase is the barrier, a warp's own instructions (an FP64
// one holds its quarter of the SM for 64 cycles), local gathers and the
// stores, 1.2 us in FP32 and 1.9 us in FP64: a cycle over 1205, 186 and 26
// rows in FP64 60 us instead of 87, over 3285, 458 and 58 rows 155 instead
// of 306, over 15308 rows down 250 instead of 405 (FP32, Gauss-Seidel on the
// finest only, 1205 rows down: 25 instead of 40).  The right-hand sides and
// residuals are replicated too when everything fits (kCycleSmem), else they
// stay in global memory, written and read through L2 (st/ld.global.cg) so
// that no stale L1 line is used after a barrier; a level whose x does not
// fit is not taken.  A CTA running small levels by itself, with CTA barriers
// and no exchange, was no faster (60 against 62 us; 166 against 136 us from
// 810 rows): the loads of a phase's entries then have no barrier to hide
// behind.  256 threads a CTA, or 8 CTAs: 5-15% slower on the larger levels.
#include <cooperative_groups.h>

#include <algorithm>

#include "dp_internal.h"

namespace cg = cooperative_groups;

namespace dp {

template <typename T>
struct LevelDev {
  int n, ncolour, lanes;
  int l1;                         // l1-Jacobi smoothing; dinv = 1 / sum_j |a_ij|
  const int *rowptr, *col, *clist;
  const T *val, *dinv;
  const int *r_rowptr, *r_col;   // restriction to the next level
  const T *r_val;
  int nn;                         // rows of the next level
  int r_lanes, p_lanes;
  const int *p_rowptr, *p_col;   // prolongation from the next level
  const T *p_val;
  T *x, *b, *r;
  int xo, bo, ro;                 // their replicas' places in shared memory (elements)
  // padded copy of the rows of each colour, G lanes a row and U (even)
  // entries a lane: lane g of the t-th row of colour c holds its entries
  // g, g + G, ... at off + (t G + g) U; ell_desc[c] = (first row slot,
  // rows, off, U 32 + log2 G), ell_dinv[slot] = 1/a_ii
  const int *ell_col;
  const int *ell_desc;
  const T *ell_val, *ell_dinv;
};

constexpr int kClusterThreads = 512;

// The two halves of the cluster barrier (release at the arrival, acquire at
// the wait), by whole warps: the barrier counts warps, so a warp's lanes meet
// first.
__device__ __forceinline__ void cl_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cl_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// A vector replicated in the shared memory of every CTA of the cluster, at
// the same place in each: s is the CTA's own copy.
__device__ __forceinline__ void st_cluster(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
template <typename T>
struct Rep {
  T *s;
  __device__ __forceinline__ T get(int i) const { return s[i]; }
  // by all G lanes of a row's group, which hold the same v: lane gl stores to
  // CTAs gl, gl + G, ...
  __device__ __forceinline__ void put(int i, T v, int gl, int G, int C) const {
    uint32_t a = (uint32_t)__cvta_generic_to_shared(s + i);
    for (int c = gl; c < C; c += G) {
      uint32_t ra;
      asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(c));
      st_cluster(ra, v);
    }
  }
};
// A vector in global memory, through L2.
template <typename T>
struct Glob {
  T *g;
  __device__ __forceinline__ T get(int i) const { return __ldcg(g + i); }
  __device__ __forceinline__ void put(int i, T v, int gl, int, int) const {
    if (gl == 0) __stcg(g + i, v);
  }
};
// the right-hand sides and residuals: replicated (REP) or global
template <typename T, bool REP> struct Side { using t = Rep<T>; };
template <typename T> struct Side<T, false> { using t = Glob<T>; };

template <typename T>
__device__ __forceinline__ T group_reduce(T v, int G) {
  for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, G);
  return v;
}

// The rows of a phase in groups of G lanes (a power of two).  The warps of
// the cluster are numbered across the CTAs (warp w of CTA r is w C + r), so
// that a short phase uses every SM (FP64 adds are scarce on each), and a
// warp's rows are consecutive.
struct RowMap {
  int gl, q, step;    // lane in the group, first row, rows per trip
  int sub;            // the row's place in the warp
  bool any;           // the warp has a row in this trip (uniform)
  __device__ __forceinline__ RowMap() {}
  __device__ __forceinline__ RowMap(int G, int count, int rank, int C) {
    const int lane = threadIdx.x & 31, lg = 31 - __clz(G), lr = 5 - lg;
    const int first = ((threadIdx.x >> 5) * C + rank) << lr;
    gl = lane & (G - 1);
    sub = lane >> lg;
    q = first + sub;
    step = ((kClusterThreads / 32) * C) << lr;
    any = first < count;
  }
  __device__ __forceinline__ bool next(int count) {
    q += step;
    any = q - sub < count;
    return any;
  }
};

// The first kHead entries a lane of a row's group has in a CSR row, loaded
// while the barrier before is still pending.
constexpr int kHead = 4;
template <typename T>
struct CsrHead {
  int e, e1, c[kHead];
  T v[kHead];
  __device__ __forceinline__ void load(bool valid, int i, int gl, int G,
                                       const int *__restrict__ rowptr,
                                       const int *__restrict__ col, const T *__restrict__ val) {
    e = valid ? __ldg(rowptr + i) + gl : 0;
    e1 = valid ? __ldg(rowptr + i + 1) : 0;
#pragma unroll
    for (int u = 0; u < kHead; ++u) {
      bool h = e + u * G < e1;
      c[u] = h ? __ldg(col + e + u * G) : -1;
      v[u] = h ? __ldg(val + e + u * G) : T(0);
    }
  }
  template <typename F>
  __device__ __forceinline__ T dot(int G, const int *__restrict__ col, const T *__restrict__ val,
                                   F X) const {
    T s0 = T(0), s1 = T(0);
#pragma unroll
    for (int u = 0; u < kHead; u += 2) {
      if (c[u] >= 0) s0 = fma(v[u], X(c[u]), s0);
      if (c[u + 1] >= 0) s1 = fma(v[u + 1], X(c[u + 1]), s1);
    }
    for (int k = e + kHead * G; k < e1; k += 2 * G) {
      int c0 = __ldg(col + k), c1 = k + G < e1 ? __ldg(col + k + G) : -1;
      T v0 = __ldg(val + k), v1 = c1 >= 0 ? __ldg(val + k + G) : T(0);
      s0 = fma(v0, X(c0), s0);
      if (c1 >= 0) s1 = fma(v1, X(c1), s1);
    }
    return s0 + s1;
  }
};

// One phase over the rows of a CSR operator: s_i = sum_j a_ij X(j), then
// done(i, s_i, o_i, lane of the group) on every lane of the row's group.
// o_i = own(i) is what the row reads of its own entry: every lane has read it
// before any lane stores, as a put writes this CTA's copy too.
template <typename T, typename F, typename O, typename D>
__device__ __forceinline__ void csr_phase(int count, int G, int rank, int C,
                                          const int *__restrict__ rowptr,
                                          const int *__restrict__ col, const T *__restrict__ val,
                                          F X, O own, D done) {
  RowMap m(G, count, rank, C);
  CsrHead<T> h;
  if (m.any) h.load(m.q < count, m.q, m.gl, G, rowptr, col, val);
  cl_wait();
  while (m.any) {
    const T o = m.q < count ? own(m.q) : T(0);
    T s = group_reduce<T>(h.dot(G, col, val, X), G);
    __syncwarp();
    if (m.q < count) done(m.q, s, o, m.gl);
    if (m.next(count)) h.load(m.q < count, m.q, m.gl, G, rowptr, col, val);
  }
  cl_arrive();
}

// Two neighbouring values as one load.
__device__ __forceinline__ double2 ld2(const double *p) {
  return __ldg(reinterpret_cast<const double2 *>(p));
}
__device__ __forceinline__ float2 ld2(const float *p) {
  return __ldg(reinterpret_cast<const float2 *>(p));
}
// v == 0 without the FP64 pipe's comparison
__device__ __forceinline__ bool is_zero(double v) {
  return (((unsigned)__double2hiint(v) << 1) | (unsigned)__double2loint(v)) == 0u;
}
__device__ __forceinline__ bool is_zero(float v) { return v == 0.f; }

// One Gauss-Seidel sweep over the colours of a level from its padded copy: a
// phase per colour, the next colour's bounds loaded a phase ahead, a row's
// columns, values and 1/a_ii before the wait.  A warp's own instructions are
// what a phase costs besides the barrier (an FP64 one holds its quarter of
// the SM for 64 cycles), so a lane's entries come in pairs by vector loads,
// padding (the row itself times 0) takes no predicates, and the sum starts
// from -b_i: x_i - (sum_j a_ij x_j - b_i) / a_ii in one chain.
constexpr int kEll = 8;   // entries a lane held in registers
template <typename T, typename VB>
__device__ void gs_sweep_cl(const LevelDev<T> &Ld, const VB b, const Rep<T> x, bool forward,
                            int rank, int C) {
  const int ncolour = Ld.ncolour;
  if (ncolour <= 0) return;
  const int *__restrict__ clist = Ld.clist;
  const int *__restrict__ desc = Ld.ell_desc;
  const int *__restrict__ ecol = Ld.ell_col;
  const T *__restrict__ eval = Ld.ell_val;
  const T *__restrict__ edinv = Ld.ell_dinv;
  int4 d;
  auto bounds = [&](int c) {
    d = make_int4(__ldg(desc + 4 * c), __ldg(desc + 4 * c + 1), __ldg(desc + 4 * c + 2),
                  __ldg(desc + 4 * c + 3));
  };
  bounds(forward ? 0 : ncolour - 1);
  for (int t = 0; t < ncolour; ++t) {
    const int r0 = d.x, ncr = d.y, off = d.z, U = d.w >> 5, G = 1 << (d.w & 31);
    if (t + 1 < ncolour) bounds(forward ? t + 1 : ncolour - 2 - t);
    RowMap m(G, ncr, rank, C);
    int i = 0;
    int2 c[kEll / 2];
    T di = T(0);
    decltype(ld2(eval)) v[kEll / 2];
    const int *cp = ecol;
    const T *vp = eval;
    auto load = [&]() {   // a row past the end: the last one's, never stored
      int q = min(m.q, ncr - 1);
      size_t at = (size_t)off + (size_t)(q * G + m.gl) * U;
      cp = ecol + at;
      vp = eval + at;
      i = __ldg(clist + r0 + q);
      di = __ldg(edinv + r0 + q);
#pragma unroll
      for (int u = 0; u < kEll / 2; ++u) {
        if (2 * u >= U) break;
        c[u] = __ldg(reinterpret_cast<const int2 *>(cp) + u);
        v[u] = ld2(vp + 2 * u);
      }
    };
    if (m.any) load();
    cl_wait();
    while (m.any) {
      T s = m.gl == 0 ? -b.get(i) : T(0), xi = x.get(i);
#pragma unroll
      for (int u = 0; u < kEll / 2; ++u) {
        if (2 * u >= U) break;
        s = fma(v[u].x, x.get(c[u].x), s);
        s = fma(v[u].y, x.get(c[u].y), s);
      }
      for (int u = kEll; u < U; u += 2) {   // rows of more than 32 kEll entries
        int2 ce = __ldg(reinterpret_cast<const int2 *>(cp + u));
        auto ve = ld2(vp + u);
        s = fma(ve.x, x.get(ce.x), s);
        s = fma(ve.y, x.get(ce.y), s);
      }
      s = group_reduce<T>(s, G);
      __syncwarp();   // xi is read on every lane before a put writes this CTA's copy
      if (m.q < ncr && !is_zero(di)) x.put(i, fma(-s, di, xi), m.gl, G, C);
      if (m.next(ncr)) load();
    }
    cl_arrive();
  }
}

// Dense solve with the FP64 LU factors and row pivots of the coarsest level,
// by the first CTA of the cluster only; xs: n doubles of shared memory.
template <typename T, typename VB>
__device__ void dense_solve_cta(int n, const double *a, const int *piv, const VB b,
                                const Rep<T> x, double *xs, int C) {
  int t = threadIdx.x, nt = blockDim.x;
  for (int i = t; i < n; i += nt) xs[i] = double(b.get(i));
  __syncthreads();
  if (t == 0)   // every row exchange first (see k_dense_solve)
    for (int k = 0; k < n; ++k) {
      int p = piv[k];
      if (p != k && p >= 0 && p < n) { double tmp = xs[k]; xs[k] = xs[p]; xs[p] = tmp; }
    }
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    double xk = xs[k];
    for (int i = k + 1 + t; i < n; i += nt) xs[i] -= a[(size_t)i * n + k] * xk;
    __syncthreads();
  }
  for (int i = n - 1; i >= 0; --i) {
    if (t == 0) { double d = a[(size_t)i * n + i]; xs[i] = d != 0.0 ? xs[i] / d : 0.0; }
    __syncthreads();
    double xi = xs[i];
    for (int r = t; r < i; r += nt) xs[r] -= a[(size_t)r * n + i] * xi;
    __syncthreads();
  }
  for (int i = t; i < n; i += nt) x.put(i, T(xs[i]), 0, 1, C);
}

// l1-Jacobi pre-smoothing from zero and the residual in one phase:
// x_i = b_i d_i, r_i = b_i - sum_j a_ij b_j d_j (d constant, loaded with the
// row's head before the wait).
template <typename T, typename VB>
__device__ void jacobi_pre_cl(const LevelDev<T> &L, const VB b, const Rep<T> x, const VB r,
                              int rank, int C) {
  const int G = L.lanes, n = L.n;
  const int *__restrict__ rowptr = L.rowptr;
  const int *__restrict__ col = L.col;
  const T *__restrict__ val = L.val;
  const T *__restrict__ d = L.dinv;
  RowMap m(G, n, rank, C);
  CsrHead<T> h;
  T dh[kHead], di = T(0);
  auto load = [&]() {
    bool valid = m.q < n;
    h.load(valid, m.q, m.gl, G, rowptr, col, val);
    di = valid ? __ldg(d + m.q) : T(0);
#pragma unroll
    for (int u = 0; u < kHead; ++u) dh[u] = h.c[u] >= 0 ? __ldg(d + h.c[u]) : T(0);
  };
  if (m.any) load();
  cl_wait();
  while (m.any) {
    T s0 = T(0), s1 = T(0);
#pragma unroll
    for (int u = 0; u < kHead; u += 2) {
      if (h.c[u] >= 0) s0 = fma(h.v[u], b.get(h.c[u]) * dh[u], s0);
      if (h.c[u + 1] >= 0) s1 = fma(h.v[u + 1], b.get(h.c[u + 1]) * dh[u + 1], s1);
    }
    for (int k = h.e + kHead * G; k < h.e1; k += G) {
      int c = __ldg(col + k);
      s0 = fma(__ldg(val + k), b.get(c) * __ldg(d + c), s0);
    }
    T s = group_reduce<T>(s0 + s1, G);
    if (m.q < n) {
      T bi = b.get(m.q);
      x.put(m.q, bi * di, m.gl, G, C);
      r.put(m.q, bi - s, m.gl, G, C);
    }
    if (m.next(n)) load();
  }
  cl_arrive();
}

// One l1-Jacobi sweep from x into t: t_i = x_i + (b_i - (A x)_i) d_i.
template <typename T, typename VB>
__device__ void jacobi_post_cl(const LevelDev<T> &L, const VB b, const Rep<T> x, const VB t,
                               int rank, int C) {
  const int G = L.lanes;
  const T *__restrict__ d = L.dinv;
  csr_phase<T>(
      L.n, G, rank, C, L.rowptr, L.col, L.val, [&](int c) { return x.get(c); },
      [&](int i) { return x.get(i); },
      [&](int i, T s, T o, int gl) { t.put(i, fma(b.get(i) - s, __ldg(d + i), o), gl, G, C); });
}

// x = inv b for the coarsest level from its explicit FP64 inverse: one phase
template <typename T, typename VB>
__device__ void dense_mv_cl(int n, const double *__restrict__ inv, const VB b, const Rep<T> x,
                            int rank, int C) {
  int G = 1;
  while (G < 32 && 4 * G < n) G <<= 1;
  RowMap m(G, n, rank, C);
  double a[kHead];
  auto load = [&]() {
#pragma unroll
    for (int u = 0; u < kHead; ++u)
      a[u] = m.q < n && m.gl + u * G < n ? __ldg(inv + (size_t)m.q * n + m.gl + u * G) : 0.0;
  };
  if (m.any) load();
  cl_wait();
  while (m.any) {
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int u = 0; u < kHead; u += 2) {
      if (m.gl + u * G < n) s0 = fma(a[u], double(b.get(m.gl + u * G)), s0);
      if (m.gl + (u + 1) * G < n) s1 = fma(a[u + 1], double(b.get(m.gl + (u + 1) * G)), s1);
    }
    if (m.q < n)
      for (int j = m.gl + kHead * G; j < n; j += G)
        s0 = fma(__ldg(inv + (size_t)m.q * n + j), double(b.get(j)), s0);
    double s = group_reduce<double>(s0 + s1, G);
    if (m.q < n) x.put(m.q, T(s), m.gl, G, C);
    if (m.next(n)) load();
  }
  cl_arrive();
}

// Every phase loads its constants, waits for the phase before, works and
// arrives; the launch starts with the replicas' initial values (x = 0, the
// right-hand side of level l0) and an arrival, and ends with a wait, after
// which no CTA writes to another's shared memory any more.  REP: b and r
// are replicated too.
template <typename T, bool REP>
__global__ void __launch_bounds__(kClusterThreads, 1)
    k_coarse_cycle(const LevelDev<T> *__restrict__ lv, int l0, int nl, const T *b0, T *x0,
                   const double *lu, const int *piv, const double *inv, int dense_n,
                   int dense_smem, int trig) {
  extern __shared__ __align__(16) unsigned char cyc_smem[];
  T *sm = reinterpret_cast<T *>(cyc_smem);
  using VB = typename Side<T, REP>::t;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), C = (int)cl.num_blocks();
  const int gt = rank * blockDim.x + threadIdx.x, nt = C * blockDim.x;
  auto xv = [&](int l) { return Rep<T>{sm + lv[l].xo}; };
  auto bv = [&](int l) -> VB {
    if constexpr (REP) return VB{sm + lv[l].bo};
    else return VB{l == l0 ? const_cast<T *>(b0) : lv[l].b};   // b0 is only read
  };
  auto rv = [&](int l) -> VB {
    if constexpr (REP) return VB{sm + lv[l].ro};
    else return VB{lv[l].r};
  };
  griddep_wait();
  if (trig) griddep_launch_dependents();
  for (int l = l0; l < nl; ++l) {
    if (lv[l].l1) continue;   // an l1-Jacobi level writes its x whole
    T *x = sm + lv[l].xo;
    for (int i = threadIdx.x; i < lv[l].n; i += blockDim.x) x[i] = T(0);
  }
  if (REP)
    for (int i = threadIdx.x; i < lv[l0].n; i += blockDim.x) sm[lv[l0].bo + i] = __ldcg(b0 + i);
  __syncthreads();
  cl_arrive();
  // descending half: pre-smoothing, residual, restriction
  for (int l = l0; l < nl - 1; ++l) {
    const LevelDev<T> &L = lv[l];
    const Rep<T> x = xv(l);
    const VB b = bv(l), r = rv(l), nb = bv(l + 1);
    if (L.l1) {
      jacobi_pre_cl<T>(L, b, x, r, rank, C);
    } else {
      gs_sweep_cl<T>(L, b, x, true, rank, C);
      const int G = L.lanes;
      csr_phase<T>(
          L.n, G, rank, C, L.rowptr, L.col, L.val, [&](int c) { return x.get(c); },
          [&](int i) { return b.get(i); },
          [&](int i, T s, T o, int gl) { r.put(i, o - s, gl, G, C); });
    }
    const int rG = L.r_lanes;
    csr_phase<T>(
        L.nn, rG, rank, C, L.r_rowptr, L.r_col, L.r_val, [&](int c) { return r.get(c); },
        [](int) { return T(0); }, [&](int I, T s, T, int gl) { nb.put(I, s, gl, rG, C); });
  }
  // coarsest level; in_r: a level's result is in its r (after an l1-Jacobi
  // post-smoothing), else in its x
  bool in_r = false;
  {
    const LevelDev<T> &L = lv[nl - 1];
    const Rep<T> x = xv(nl - 1);
    const VB b = bv(nl - 1), r = rv(nl - 1);
    if (dense_n == L.n && L.n > 0 && inv) {
      dense_mv_cl<T>(L.n, inv, b, x, rank, C);
    } else if (dense_n == L.n && L.n > 0) {
      cl_wait();
      if (rank == 0)
        dense_solve_cta<T>(L.n, lu, piv, b, x,
                           reinterpret_cast<double *>(cyc_smem + dense_smem), C);
      cl_arrive();
    } else if (L.l1) {
      jacobi_pre_cl<T>(L, b, x, r, rank, C);
      jacobi_post_cl<T>(L, b, x, r, rank, C);
      in_r = true;
    } else {
      gs_sweep_cl<T>(L, b, x, true, rank, C);
      gs_sweep_cl<T>(L, b, x, false, rank, C);
    }
  }
  // ascending half: prolongation, post-smoothing
  for (int l = nl - 2; l >= l0; --l) {
    const LevelDev<T> &L = lv[l];
    const Rep<T> x = xv(l), nx = xv(l + 1);
    const VB b = bv(l), r = rv(l), nr = rv(l + 1);
    const int pG = L.p_lanes;
    auto own = [&](int i) { return x.get(i); };
    auto add = [&](int i, T s, T o, int gl) { x.put(i, o + s, gl, pG, C); };
    if (in_r)
      csr_phase<T>(
          L.n, pG, rank, C, L.p_rowptr, L.p_col, L.p_val, [&](int c) { return nr.get(c); },
          own, add);
    else
      csr_phase<T>(
          L.n, pG, rank, C, L.p_rowptr, L.p_col, L.p_val, [&](int c) { return nx.get(c); },
          own, add);
    in_r = L.l1;
    if (L.l1) jacobi_post_cl<T>(L, b, x, r, rank, C);
    else gs_sweep_cl<T>(L, b, x, false, rank, C);
  }
  cl_wait();
  const Rep<T> x = xv(l0);
  const VB r = rv(l0);
  for (int i = gt; i < lv[l0].n; i += nt) x0[i] = in_r ? r.get(i) : x.get(i);
}

// lanes per row inside the cluster: rows are few, so shorten the chains, in
// FP64 less so (the reduction's adds take the SM's FP64 issue)
template <typename T>
static int cluster_lanes(double mean_len) {
  int g = 1;
  while (g < 32 && (sizeof(T) == 8 ? 8.0 : 4.0) * g < mean_len) g *= 2;
  return g;
}

template <typename T>
static const T *pick(const double *d, const float *f) {
  if constexpr (sizeof(T) == 8) return (const T *)d; else return (const T *)f;
}
template <typename T>
static T *pickw(double *d, float *f) {
  if constexpr (sizeof(T) == 8) return (T *)d; else return (T *)f;
}

// Places of the replicas in the shared memory of a CTA: x of every level
// from `first` down, and the right-hand sides and residuals when all of it
// fits (rep).  Returns the bytes used, 0 when not even x fits.  At 16 CTAs
// the whole budget of an SM may be used: the cluster takes its SMs alone.
constexpr size_t kCycleSmem = 224 * 1024;
template <typename T>
static size_t rep_plan(const Sim *s, int first, std::vector<LevelDev<T>> &h, bool *rep,
                       size_t *dense_smem) {
  int nl = (int)s->lev.size();
  h.resize(nl);
  bool lu = s->coarse_n == s->lev[nl - 1].n && s->coarse_n > 0 && !s->coarse_inv;
  size_t room = kCycleSmem - (lu ? (size_t)s->coarse_n * 8 : 0), one = 0, used = 0;
  auto bytes = [&](int l) { return ((size_t)s->lev[l].n * sizeof(T) + 15) & ~(size_t)15; };
  for (int l = first; l < nl; ++l) one += bytes(l);
  if (one > room) return 0;
  *rep = 3 * one <= room;
  for (int v = 0; v < 3; ++v)
    for (int l = 0; l < nl; ++l) {
      bool put = l >= first && (v == 0 || *rep);
      (v == 0 ? h[l].xo : v == 1 ? h[l].bo : h[l].ro) = put ? (int)(used / sizeof(T)) : 0;
      if (put) used += bytes(l);
    }
  *dense_smem = used;
  return used + (lu ? (size_t)s->coarse_n * 8 : 0);
}

template <typename T>
static int upload_levels(Sim *s, void **dst, int first, int *smem, int *dense_smem, bool *rep) {
  int nl = (int)s->lev.size();
  std::vector<LevelDev<T>> h;
  size_t ds = 0;
  *smem = (int)rep_plan<T>(s, first, h, rep, &ds);
  *dense_smem = (int)ds;
  for (int l = 0; l < nl; ++l) {
    Level &L = s->lev[l];
    LevelDev<T> &d = h[l];
    d.n = L.n;
    d.l1 = L.l1 ? 1 : 0;
    d.ncolour = L.ncolour;
    d.lanes = cluster_lanes<T>(L.n ? (double)L.nnz / L.n : 0.0);
    d.rowptr = L.rowptr; d.col = L.col; d.clist = L.clist;
    d.val = pick<T>(L.val, L.valf);
    d.dinv = pick<T>(L.dinv, L.dinvf);
    d.x = pickw<T>(L.x, L.xf); d.b = pickw<T>(L.b, L.bf); d.r = pickw<T>(L.r, L.rf);
    d.ell_col = L.ell_col;
    d.ell_desc = L.ell_desc;
    d.ell_val = pick<T>(L.ell_val, L.ell_valf);
    d.ell_dinv = pick<T>(L.ell_dinv, L.ell_dinvf);
    if (l + 1 < nl) {
      d.nn = s->lev[l + 1].n;
      d.r_rowptr = L.r_rowptr; d.r_col = L.r_col; d.r_val = pick<T>(L.r_val, L.r_valf);
      d.p_rowptr = L.p_rowptr; d.p_col = L.p_col; d.p_val = pick<T>(L.p_val, L.p_valf);
      d.r_lanes = cluster_lanes<T>(d.nn ? (double)L.r_nnz / d.nn : 0.0);
      d.p_lanes = cluster_lanes<T>(L.n ? (double)L.p_nnz / L.n : 0.0);
    } else {
      d.nn = 0; d.r_rowptr = d.r_col = d.p_rowptr = d.p_col = nullptr;
      d.r_val = d.p_val = nullptr; d.r_lanes = d.p_lanes = 1;
    }
  }
  if (!*dst) {
    *dst = dalloc(s, sizeof(LevelDev<T>) * std::max(nl, 1));
    if (!*dst) { s->fail(DP_ENOMEM, "allocation failed"); return DP_ENOMEM; }
  }
  DP_CUDA(s, cudaMemcpyAsync(*dst, h.data(), sizeof(LevelDev<T>) * nl, cudaMemcpyHostToDevice,
                             s->stream));
  DP_CUDA(s, cudaStreamSynchronize(s->stream));
  return DP_OK;
}

__global__ void k_ell_maxlen(int n, const int *rowptr, const int *colour, int *K) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) atomicMax(&K[colour[i]], rowptr[i + 1] - rowptr[i]);
}

// Fill the padded copy (LevelDev): padding entries point at the row itself
// with source -1 (value 0).
__global__ void k_ell_fill(int n, const int *clist, const int *colour, const int *desc,
                           const int *rowptr, const int *col, int *ecol, int *esrc) {
  int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  int i = clist[q];
  const int *d = desc + 4 * colour[i];
  int t = q - d[0], U = d[3] >> 5, G = 1 << (d[3] & 31);
  int e0 = rowptr[i], len = rowptr[i + 1] - e0;
  for (int g = 0; g < G; ++g)
    for (int u = 0; u < U; ++u) {
      size_t p = (size_t)d[2] + ((size_t)t * G + g) * U + u;
      int k = g + u * G;
      ecol[p] = k < len ? col[e0 + k] : i;
      esrc[p] = k < len ? e0 + k : -1;
    }
}

// the padded values, then 1/a_ii by row slot
template <typename T>
__global__ void k_ell_values(long long total, const int *esrc, const T *val, T *eval, int n,
                             const int *clist, const T *dinv, T *edinv) {
  long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p < total) { int q = esrc[p]; eval[p] = q >= 0 ? val[q] : T(0); }
  else if (p < total + n) edinv[p - total] = dinv[clist[p - total]];
}

static int ell_build(Sim *s, Level &L) {
  int nc = L.ncolour, m4 = std::max(nc, 1);
  L.ell_desc = (int *)dalloc(s, (size_t)m4 * 16);
  int *K_dev = (int *)dalloc(s, (size_t)m4 * 4);
  if (!L.ell_desc || !K_dev) { s->fail(DP_ENOMEM, "allocation failed"); return DP_ENOMEM; }
  DP_CUDA(s, cudaMemsetAsync(K_dev, 0, (size_t)m4 * 4, s->stream));
  DP_LAUNCH(s, k_ell_maxlen, nblk(L.n), kBlock, 0, L.n, L.rowptr, L.colour, K_dev);
  std::vector<int> K(m4), desc((size_t)m4 * 4, 0);
  DP_CUDA(s, cudaMemcpyAsync(K.data(), K_dev, (size_t)m4 * 4, cudaMemcpyDeviceToHost, s->stream));
  DP_CUDA(s, cudaStreamSynchronize(s->stream));
  dfree(s, K_dev);
  long long total = 0;
  for (int c = 0; c < nc; ++c) {
    int lg = 0;
    while (lg < 5 && (kEll << lg) < K[c]) ++lg;
    int U = (K[c] + (1 << lg) - 1) >> lg;
    U = std::max(2, (U + 1) & ~1);
    desc[4 * c] = L.cstart[c];
    desc[4 * c + 1] = L.cstart[c + 1] - L.cstart[c];
    desc[4 * c + 2] = (int)total;
    desc[4 * c + 3] = U * 32 + lg;
    total += (long long)desc[4 * c + 1] * U << lg;
    if (total >= (1LL << 31)) { s->fail(DP_EINVAL, "coarse level too large for its padded copy"); return DP_EINVAL; }
  }
  L.ell_total = total;
  size_t m = (size_t)std::max(total, 1LL), n = (size_t)std::max(L.n, 1);
  L.ell_col = (int *)dalloc(s, m * 4);
  L.ell_src = (int *)dalloc(s, m * 4);
  // in the precision of the V-cycle
  if (s->opt.precision >= 1) {
    L.ell_valf = (float *)dalloc(s, m * 4);
    L.ell_dinvf = (float *)dalloc(s, n * 4);
  } else {
    L.ell_val = (double *)dalloc(s, m * 8);
    L.ell_dinv = (double *)dalloc(s, n * 8);
  }
  if (!L.ell_col || !L.ell_src || !(L.ell_val || L.ell_valf) || !(L.ell_dinv || L.ell_dinvf)) {
    s->fail(DP_ENOMEM, "allocation failed");
    return DP_ENOMEM;
  }
  DP_CUDA(s, cudaMemcpyAsync(L.ell_desc, desc.data(), desc.size() * 4, cudaMemcpyHostToDevice,
                             s->stream));
  DP_CUDA(s, cudaStreamSynchronize(s->stream));
  DP_LAUNCH(s, k_ell_fill, nblk(L.n), kBlock, 0, L.n, L.clist, L.colour, L.ell_desc, L.rowptr,
            L.col, L.ell_col, L.ell_src);
  DP_CUDA(s, cudaGetLastError());
  return DP_OK;
}

// Copy the current level values into the padded copies when the hierarchy's
// values have been refreshed (with their FP32 copies); otherwise (coarse =
// false) only level 0's 1/a_ii, in FP64: its sweeps keep the entries of the
// last refresh, and in FP32 all of level 0 is of that refresh (mixed_refresh).
// With the current entries a timestep took as many iterations (0.7% fewer over
// 400 timesteps of 11k and 16k rows) and one in sixteen ended more than the
// Newton tolerance away from the state it ends in so.
int cluster_refresh(Sim *s, bool coarse) {
  if (s->cl_level < 0) return DP_OK;
  bool f32 = s->opt.precision >= 1;
  for (int l = s->cl_level; l < (int)s->lev.size() && (coarse || l == 0); ++l) {
    Level &L = s->lev[l];
    if (!L.ell_src) continue;
    long long total = coarse ? L.ell_total : 0;
    if (f32)
      DP_LAUNCH(s, k_ell_values<float>, nblk(total + L.n), kBlock, 0, total, L.ell_src, L.valf,
                L.ell_valf, L.n, L.clist, L.dinvf, L.ell_dinvf);
    else
      DP_LAUNCH(s, k_ell_values<double>, nblk(total + L.n), kBlock, 0, total, L.ell_src, L.val,
                L.ell_val, L.n, L.clist, L.dinv, L.ell_dinv);
  }
  DP_CUDA(s, cudaGetLastError());
  return DP_OK;
}

// Cluster size: 16 CTAs if the GPU can place them, else 8, else 0.  Asked
// once on each device: the occupancy queries cost more than the rest of
// cluster_setup, and they serialise the set-ups of several host threads.
static int cluster_ctas() {
  static PerDevice per;
  return per([] {
    using Cycle64 = void (*)(const LevelDev<double> *, int, int, const double *, double *,
                             const double *, const int *, const double *, int, int, int);
    using Cycle32 = void (*)(const LevelDev<float> *, int, int, const float *, float *,
                             const double *, const int *, const double *, int, int, int);
    const Cycle64 k64[2] = {k_coarse_cycle<double, false>, k_coarse_cycle<double, true>};
    const Cycle32 k32[2] = {k_coarse_cycle<float, false>, k_coarse_cycle<float, true>};
    for (int k = 0; k < 2; ++k) {
      cudaFuncSetAttribute(k64[k], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCycleSmem);
      cudaFuncSetAttribute(k32[k], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCycleSmem);
    }
    int csize = 0;
    for (int c : {16, 8}) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(c);
      cfg.blockDim = dim3(kClusterThreads);
      cfg.dynamicSmemBytes = kCycleSmem;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = c; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      bool fits = true;
      for (int k = 0; k < 2; ++k) {
        if (c > 8) {
          cudaFuncSetAttribute(k64[k], cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
          cudaFuncSetAttribute(k32[k], cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        }
        int nc1 = 0, nc2 = 0;
        fits = fits && cudaOccupancyMaxActiveClusters(&nc1, k64[k], &cfg) == cudaSuccess &&
               cudaOccupancyMaxActiveClusters(&nc2, k32[k], &cfg) == cudaSuccess && nc1 > 0 &&
               nc2 > 0;
      }
      if (fits) {
        csize = c;
        break;
      }
      cudaGetLastError();
    }
    return csize;
  });
}

// Decide the first level run by the cluster kernel and the cluster size; copy
// the level descriptors and colour starts to the device.  Called after the
// hierarchy is built.
int cluster_setup(Sim *s) {
  s->cl_level = -1;
  if (s->lev.empty()) return DP_OK;
  const int csize = cluster_ctas();
  s->cl_size = csize;
  if (csize == 0 || !s->opt.use_graphs) return DP_OK;  // the per-launch cycle stays in use
  int rows = s->opt.cluster_rows == 0 ? kClusterMaxRows : s->opt.cluster_rows;
  int first = -1;
  bool f32 = s->opt.precision >= 1;
  for (int l = 0; l < (int)s->lev.size() && rows > 0; ++l) {
    if (s->lev[l].n > rows) continue;
    std::vector<LevelDev<double>> h64;
    std::vector<LevelDev<float>> h32;
    bool rep;
    size_t ds;
    if (f32 ? !rep_plan<float>(s, l, h32, &rep, &ds) : !rep_plan<double>(s, l, h64, &rep, &ds))
      continue;   // its vectors do not fit
    first = l;
    break;
  }
  if (first < 0) return DP_OK;
  // By default the cluster runs only where it saves launches: a level with
  // multicolour Gauss-Seidel has one phase per colour, an l1-Jacobi level
  // five, and on GB300 five full-GPU launches of a small level (graph
  // launched) cost less than the same phases on the cluster's 16 SMs.
  bool gs = false;
  for (int l = first; l < (int)s->lev.size(); ++l) gs |= !s->lev[l].l1;
  if (s->opt.cluster_rows == 0 && !gs) return DP_OK;
  for (int l = first; l < (int)s->lev.size(); ++l)
    if (!s->lev[l].l1) DP_TRY(ell_build(s, s->lev[l]));   // Gauss-Seidel levels only
  // the levels in the precision of the V-cycle
  if (f32)
    DP_TRY(upload_levels<float>(s, &s->cl_lev, first, &s->cl_smem, &s->cl_dense, &s->cl_rep));
  else
    DP_TRY(upload_levels<double>(s, &s->cl_lev, first, &s->cl_smem, &s->cl_dense, &s->cl_rep));
  s->cl_level = first;
  return DP_OK;
}

template <typename T>
int coarse_cycle(Sim *s, int l0, const T *b, T *x) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(s->cl_size);
  cfg.blockDim = dim3(kClusterThreads);
  cfg.dynamicSmemBytes = s->cl_smem;
  cfg.stream = s->stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = s->cl_size; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  const bool pdl = s->pdl_small && (pdl_mode() & kPdlSmall);
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 2 : 1;
  const LevelDev<T> *lv = (const LevelDev<T> *)s->cl_lev;
  int nl = (int)s->lev.size();
  {
    LaunchScope ls(s, "k_coarse_cycle");
    DP_CUDA(s, cudaLaunchKernelEx(&cfg, s->cl_rep ? k_coarse_cycle<T, true> : k_coarse_cycle<T, false>,
                                  lv, l0, nl, b, x, (const double *)s->coarse_lu,
                                  (const int *)s->coarse_piv, (const double *)s->coarse_inv,
                                  s->coarse_n, s->cl_dense, pdl && pdl_trigger() ? 1 : 0));
  }
  return DP_OK;
}

template int coarse_cycle<double>(Sim *, int, const double *, double *);
template int coarse_cycle<float>(Sim *, int, const float *, float *);

}  // namespace dp
