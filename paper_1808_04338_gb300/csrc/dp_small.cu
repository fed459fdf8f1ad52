// The CPR-FPF preconditioner of a small realisation in two cluster launches
// around the V-cycle.
//
// Below some ten thousand block rows every kernel of an application (two
// ILU(0) solves of two sweeps over the colours, the two stage residuals, the
// injection, the gathers) has less work than a launch costs: 17 launches of
// 3 to 5 us each.  Here one thread-block cluster runs the phases before the
// V-cycle (part 0: z1 = F r and the pressure residual) in one launch and
// those after it (part 1: z2 = z1 + P e, r - A z2, z = z2 + F (r - A z2)) in
// another, with a hardware cluster barrier between phases instead of a
// launch.  A phase loads what no phase writes (its rows' pointers, first
// blocks and columns) between its arrival at the barrier before and its wait;
// vectors that another CTA has written are read through L2 (ld.global.cg).
// The row formulas and the order of their sums are those of the kernels of
// one launch each.  Timestep of 602 rows with these and k_orth_small 8.4 ms
// -> 7.0, of 5765 rows in FP64 43.3 -> 36.6, with the FP32 preconditioner 6.5
// -> 5.8 (k_orth_small is a bit more than half of that).
#include <cooperative_groups.h>

#include <algorithm>

#include "dp_internal.h"
#include "dp_kernels.cuh"

namespace cg = cooperative_groups;

namespace dp {

constexpr int kSmallThreads = 512, kSmallColours = 8;

template <typename T>
struct SmallArgs {
  int n, nL, ncol, last;                 // factor: rows, L blocks, colours, last non-empty colour
  int cstart[kSmallColours + 1];
  int lng;                               // bit c: colour c has long rows (a warp each)
  const int *perm, *iperm, *Lptr, *Uptr, *colp;
  const T *lu;
  T *zp, *zp2;                           // results of the first and second ILU(0) solve
  // the operator's storage-order copy
  int sL, sc, long0;
  const int *srowptr, *scol;             // scol: columns as positions in x of the stage residuals
  const double *sval, *a00, *a01;        // FP64
  const float *svalf;                    // FP32
  const float2 *spf;
  const double *r;                       // v_j
  double *z1, *r1, *rp, *xp;             // FP64 stage vectors
  float *z1f, *r1f, *z2c, *bf, *xf;      // FP32 stage vectors, level 0's b and x
  const int *omap;                       // level 0 in colour order: its position of each row
  X0Init xi;
  double *z;                             // the result
};

__device__ __forceinline__ void small_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void small_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The cluster's threads, its warps numbered across the CTAs.
struct Lanes {
  int t, nt;     // thread, threads
  __device__ __forceinline__ int warp() const { return t >> 5; }
  __device__ __forceinline__ int nwarp() const { return nt >> 5; }
};

template <typename T> __device__ __forceinline__ typename V2<T>::t ld2cg(const T *p, size_t k) {
  return __ldcg(reinterpret_cast<const typename V2<T>::t *>(p) + k);
}

// Rows [r0, r1) of one sweep, two lanes a row (one output component each):
// the first kPre blocks' row of that component and columns are loaded before
// the wait.  done(row, comp, s) on both lanes (the trip count is uniform in a
// warp, so the lanes may exchange).
constexpr int kPre = 4;
template <typename T, typename D>
__device__ __forceinline__ void sweep_rows(const Lanes &L, int r0, int r1,
                                           const int *__restrict__ ptr, size_t base,
                                           const int *__restrict__ colp, const T *__restrict__ lu,
                                           const T *x, D done) {
  using T2 = typename V2<T>::t;
  const int comp = L.t & 1;
  int q = r0 + (L.t >> 1), e = 0, e1 = 0, c[kPre];
  T2 a[kPre];
  const T2 *v2 = reinterpret_cast<const T2 *>(lu) + comp;
  auto load = [&]() {
    const bool in = q < r1;
    e = in ? __ldg(ptr + q) : 0;
    e1 = in ? __ldg(ptr + q + 1) : 0;
#pragma unroll
    for (int k = 0; k < kPre; ++k)
      if (e + k < e1) {
        a[k] = __ldg(v2 + 2 * (base + e + k));
        c[k] = __ldg(colp + base + e + k);
      }
  };
  const int first = r0 + ((L.t & ~31) >> 1);   // the warp's first row (uniform)
  int w = first;
  if (w < r1) load();
  small_wait();
  while (w < r1) {
    T s = T(0);
#pragma unroll
    for (int k = 0; k < kPre; ++k)
      if (e + k < e1) {
        T2 xk = ld2cg<T>(x, c[k]);
        s = fma(a[k].x, xk.x, s);
        s = fma(a[k].y, xk.y, s);
      }
    for (int k = e + kPre; k < e1; ++k) {
      T2 ak = __ldg(v2 + 2 * (base + k));
      T2 xk = ld2cg<T>(x, __ldg(colp + base + k));
      s = fma(ak.x, xk.x, s);
      s = fma(ak.y, xk.y, s);
    }
    done(q, comp, s, q < r1);
    q += L.nt >> 1;
    w += L.nt >> 1;
    if (w < r1) load();
  }
}

// Long rows (the wells), a warp per row: s0, s1 on every lane.
template <typename T, typename D>
__device__ __forceinline__ void sweep_long(const Lanes &L, int r0, int r1,
                                           const int *__restrict__ ptr, size_t base,
                                           const int *__restrict__ colp, const T *__restrict__ lu,
                                           const T *x, D done) {
  using T2 = typename V2<T>::t;
  const int lane = L.t & 31;
  small_wait();
  for (int r = r0 + L.warp(); r < r1; r += L.nwarp()) {
    T s0 = T(0), s1 = T(0);
    for (int e = __ldg(ptr + r) + lane, eb = __ldg(ptr + r + 1); e < eb; e += 32) {
      T a[4];
      V4<T>::load(lu + 4 * (base + e), a);
      T2 xk = ld2cg<T>(x, __ldg(colp + base + e));
      s0 = fma(a[0], xk.x, fma(a[1], xk.y, s0));
      s1 = fma(a[2], xk.x, fma(a[3], xk.y, s1));
    }
    done(r, lane, warp_sum(s0), warp_sum(s1));
  }
}

// (LU)^-1 rhs into zp (colour order): the forward sweep over the colours (the
// first a copy; a last colour of long rows with its pivots applied), then the
// backward sweep.  Every phase waits for the one before and arrives.
template <typename T, typename TR>
__device__ __forceinline__ void small_ilu(const Lanes &L, const SmallArgs<T> &A, const TR *rhs,
                                          T *zp) {
  using T2 = typename V2<T>::t;
  using R2 = typename V2<TR>::t;
  const size_t ub = (size_t)A.nL + A.n;
  bool first = true;
  for (int c = 0; c < A.ncol; ++c) {
    const int r0 = A.cstart[c], r1 = A.cstart[c + 1];
    if (r1 <= r0) continue;
    const bool lng = (A.lng >> c) & 1;
    if (first && !lng) {
      int q = r0 + L.t, p = q < r1 ? __ldg(A.perm + q) : 0;
      small_wait();
      for (; q < r1; q += L.nt, p = q < r1 ? __ldg(A.perm + q) : 0) {
        R2 v = __ldcg(reinterpret_cast<const R2 *>(rhs) + p);
        T2 o;
        o.x = T(v.x);
        o.y = T(v.y);
        __stcg(reinterpret_cast<T2 *>(zp) + q, o);
      }
    } else if (lng) {
      sweep_long<T>(L, r0, r1, A.Lptr, 0, A.colp, A.lu, zp, [&](int r, int lane, T s0, T s1) {
        if (lane != 0) return;
        const int i = __ldg(A.perm + r);
        T y0 = T(__ldcg(rhs + 2 * (size_t)i)) - s0, y1 = T(__ldcg(rhs + 2 * (size_t)i + 1)) - s1;
        T2 o;
        o.x = y0;
        o.y = y1;
        if (c == A.last) {
          T d[4];
          V4<T>::load(A.lu + 4 * ((size_t)A.nL + r), d);
          o.x = fma(d[0], y0, d[1] * y1);
          o.y = fma(d[2], y0, d[3] * y1);
        }
        __stcg(reinterpret_cast<T2 *>(zp) + r, o);
      });
    } else {
      sweep_rows<T>(L, r0, r1, A.Lptr, 0, A.colp, A.lu, zp, [&](int q, int comp, T s, bool in) {
        if (!in) return;
        const int i = __ldg(A.perm + q);
        __stcg(zp + 2 * (size_t)q + comp, T(__ldcg(rhs + 2 * (size_t)i + comp)) - s);
      });
    }
    first = false;
    small_arrive();
  }
  for (int c = A.ncol - 1; c >= 0; --c) {
    const int r0 = A.cstart[c], r1 = A.cstart[c + 1];
    if (r1 <= r0) continue;
    const bool lng = (A.lng >> c) & 1;
    if (lng && c == A.last) continue;   // done with the forward sweep
    if (lng) {
      sweep_long<T>(L, r0, r1, A.Uptr, ub, A.colp, A.lu, zp, [&](int r, int lane, T s0, T s1) {
        if (lane != 0) return;
        T2 y = ld2cg<T>(zp, r), o;
        T y0 = y.x - s0, y1 = y.y - s1, d[4];
        V4<T>::load(A.lu + 4 * ((size_t)A.nL + r), d);
        o.x = fma(d[0], y0, d[1] * y1);
        o.y = fma(d[2], y0, d[3] * y1);
        __stcg(reinterpret_cast<T2 *>(zp) + r, o);
      });
    } else {
      sweep_rows<T>(L, r0, r1, A.Uptr, ub, A.colp, A.lu, zp, [&](int q, int comp, T s, bool in) {
        T y = (in ? __ldcg(zp + 2 * (size_t)q + comp) : T(0)) - s;
        T o = __shfl_xor_sync(0xffffffffu, y, 1);
        if (!in) return;
        T2 d = __ldg(reinterpret_cast<const T2 *>(A.lu + 4 * ((size_t)A.nL + q)) + comp);
        T y0 = comp ? o : y, y1 = comp ? y : o;
        __stcg(zp + 2 * (size_t)q + comp, fma(d.x, y0, d.y * y1));
      });
    }
    small_arrive();
  }
}

// Pressure rows of r - A x into rp (FP64) or, with the pre-smoothing's start,
// into level 0's right-hand side (FP32), as k_bsr_presid and
// k_bsr_presid_f32_b.
template <typename T>
__device__ __forceinline__ void small_presid(const Lanes &L, const SmallArgs<T> &A, const T *x) {
  using T2 = typename V2<T>::t;
  auto pair = [&](int e) {
    if constexpr (sizeof(T) == 8) return make_double2(__ldg(A.a00 + e), __ldg(A.a01 + e));
    else return __ldg(A.spf + e);
  };
  auto put = [&](int row, T v) {
    const int pos = A.omap ? __ldg(A.omap + row) : row;
    if constexpr (sizeof(T) == 8) A.rp[pos] = v;
    else put_b0(A.bf, pos, v, A.xi);
  };
  int q = L.t, e = 0, e1 = 0;
  if (q < A.long0) { e = __ldg(A.srowptr + q); e1 = __ldg(A.srowptr + q + 1); }
  small_wait();
  while (q < A.long0) {
    T s = T(0);
    for (; e < e1; ++e) {
      T2 a = pair(e), xj = ld2cg<T>(x, __ldg(A.scol + e));
      s = fma(a.x, xj.x, s);
      s = fma(a.y, xj.y, s);
    }
    const int row = row_of_pair(q, A.sL, A.sc);
    put(row, T(A.r[2 * (size_t)row]) - s);
    q += L.nt;
    if (q < A.long0) { e = __ldg(A.srowptr + q); e1 = __ldg(A.srowptr + q + 1); }
  }
  const int lane = L.t & 31;
  for (int row = A.long0 + L.warp(); row < A.n; row += L.nwarp()) {
    T s = T(0);
    for (int k = __ldg(A.srowptr + row) + lane, k1 = __ldg(A.srowptr + row + 1); k < k1; k += 32) {
      T2 a = pair(k), xj = ld2cg<T>(x, __ldg(A.scol + k));
      s = fma(a.x, xj.x, fma(a.y, xj.y, s));
    }
    s = warp_sum(s);
    if (lane == 0) put(row, T(A.r[2 * (size_t)row]) - s);
  }
  small_arrive();
}

// y = r - A x, two lanes a row, as k_bsr_spmv_b<1> and k_bsr_resid_f32_b.
template <typename T>
__device__ __forceinline__ void small_resid(const Lanes &L, const SmallArgs<T> &A, const T *x,
                                            T *y) {
  using T2 = typename V2<T>::t;
  const T *val;
  if constexpr (sizeof(T) == 8) val = A.sval; else val = A.svalf;
  const int comp = L.t & 1;
  const T2 *v2 = reinterpret_cast<const T2 *>(val);
  int q = L.t >> 1, e = 0, e1 = 0;
  if (q < A.long0) { e = __ldg(A.srowptr + q); e1 = __ldg(A.srowptr + q + 1); }
  small_wait();
  while (q < A.long0) {
    T s = T(0);
#pragma unroll 4
    for (int k = e; k < e1; ++k) {
      T2 a = __ldg(v2 + 2 * (size_t)k + comp), xj = ld2cg<T>(x, __ldg(A.scol + k));
      s = fma(a.x, xj.x, s);
      s = fma(a.y, xj.y, s);
    }
    const size_t k = 2 * (size_t)row_of_pair(q, A.sL, A.sc) + comp;
    __stcg(y + k, T(A.r[k]) - s);
    q += L.nt >> 1;
    if (q < A.long0) { e = __ldg(A.srowptr + q); e1 = __ldg(A.srowptr + q + 1); }
  }
  const int lane = L.t & 31;
  for (int row = A.long0 + L.warp(); row < A.n; row += L.nwarp()) {
    T s0 = T(0), s1 = T(0);
    for (int k = __ldg(A.srowptr + row) + lane, k1 = __ldg(A.srowptr + row + 1); k < k1; k += 32) {
      T2 a = __ldg(v2 + 2 * (size_t)k), c = __ldg(v2 + 2 * (size_t)k + 1);
      T2 xj = ld2cg<T>(x, __ldg(A.scol + k));
      s0 = fma(a.x, xj.x, fma(a.y, xj.y, s0));
      s1 = fma(c.x, xj.x, fma(c.y, xj.y, s1));
    }
    s0 = warp_sum(s0);
    s1 = warp_sum(s1);
    if (lane == 0) {
      __stcg(y + 2 * (size_t)row, T(A.r[2 * (size_t)row]) - s0);
      __stcg(y + 2 * (size_t)row + 1, T(A.r[2 * (size_t)row + 1]) - s1);
    }
  }
  small_arrive();
}

template <typename T, int PART>
__global__ void __launch_bounds__(kSmallThreads, 1) k_cpr_small(const SmallArgs<T> A, int trig) {
  using T2 = typename V2<T>::t;
  constexpr bool kF32 = sizeof(T) == 4;
  cg::cluster_group cl = cg::this_cluster();
  Lanes L;
  L.t = ((int)(threadIdx.x >> 5) * (int)cl.num_blocks() + (int)cl.block_rank()) * 32 +
        (int)(threadIdx.x & 31);
  L.nt = (int)cl.num_blocks() * kSmallThreads;
  griddep_wait();
  if (trig) griddep_launch_dependents();
  small_arrive();
  if (PART == 0) {
    small_ilu<T, double>(L, A, A.r, A.zp);
    // z1: in the colour order (FP32, level 0 in that order), else gathered
    if (!kF32 || !A.z2c) {
      small_wait();
      T *out;
      if constexpr (kF32) out = A.z1f; else out = A.z1;
      for (int i = L.t; i < A.n; i += L.nt)
        __stcg(reinterpret_cast<T2 *>(out) + i, ld2cg<T>(A.zp, __ldg(A.iperm + i)));
      small_arrive();
      small_presid<T>(L, A, out);
    } else {
      small_presid<T>(L, A, A.zp);
    }
  } else {
    // z2 = z1 + P e
    small_wait();
    if constexpr (!kF32) {
      for (int i = L.t; i < A.n; i += L.nt) {
        const double e = A.xp[A.omap ? __ldg(A.omap + i) : i];
        __stcg(A.z1 + 2 * (size_t)i, A.z1[2 * (size_t)i] + e);
      }
    } else if (A.z2c) {
      for (int q = L.t; q < A.n; q += L.nt) {
        float2 v = reinterpret_cast<const float2 *>(A.zp)[q];
        v.x += A.xf[q];
        __stcg(reinterpret_cast<float2 *>(A.z2c) + q, v);
      }
    } else {
      for (int i = L.t; i < A.n; i += L.nt)
        __stcg(A.z1f + 2 * (size_t)i,
               A.z1f[2 * (size_t)i] + A.xf[A.omap ? __ldg(A.omap + i) : i]);
    }
    small_arrive();
    if constexpr (kF32) small_resid<float>(L, A, A.z2c ? A.z2c : A.z1f, A.r1f);
    else small_resid<double>(L, A, A.z1, A.r1);
    if constexpr (kF32) small_ilu<float, float>(L, A, A.r1f, A.zp2);
    else small_ilu<double, double>(L, A, A.r1, A.zp2);
    // z = z2 + F (r - A z2)
    small_wait();
    for (int i = L.t; i < A.n; i += L.nt) {
      const int p = __ldg(A.iperm + i);
      T2 v = ld2cg<T>(A.zp2, p);
      double2 b;
      if constexpr (kF32) {   // z2 from the first result and the correction, in FP64
        float2 u = reinterpret_cast<const float2 *>(A.zp)[p];
        b = make_double2(double(u.x), double(u.y));
        b.x = b.x + double(A.xf[A.omap ? p : i]);
      } else {
        b = __ldcg(reinterpret_cast<const double2 *>(A.z1) + i);
      }
      reinterpret_cast<double2 *>(A.z)[i] = make_double2(b.x + double(v.x), b.y + double(v.y));
    }
    small_arrive();
  }
  small_wait();
}

// One cluster of s->cl_size CTAs, as a programmatic dependent (kPdlSmall).
template <typename K, typename Args>
static int launch_cluster(Sim *s, const char *name, K kern, const Args &A) {
  if (s->alloc_failed) return DP_ENOMEM;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(s->cl_size);
  cfg.blockDim = dim3(kSmallThreads);
  cfg.stream = s->stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = s->cl_size; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  const bool pdl = s->pdl_small && (pdl_mode() & kPdlSmall);
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 2 : 1;
  LaunchScope ls(s, name);
  DP_CUDA(s, cudaLaunchKernelEx(&cfg, kern, A, pdl && pdl_trigger() ? 1 : 0));
  return DP_OK;
}

template <typename T, int PART>
static int launch_small(Sim *s, const SmallArgs<T> &A) {
  // clusters of 16 CTAs
  DP_CUDA(s, (kernel_attribute<k_cpr_small<T, PART>,
                               cudaFuncAttributeNonPortableClusterSizeAllowed>(1)));
  return launch_cluster(s, "k_cpr_small", k_cpr_small<T, PART>, A);
}

// The sizes where the cluster launches beat the launches of a phase each:
// its 16 SMs are 10-20% faster over a timestep up to 7845 rows, equal from
// 11565 (FP32 7.8 and 7.8 ms, FP64 65.4 and 66.9) and slower at 33125 (FP32
// 8.4 against 6.8 ms).  With other streams on the GPU too: 1, 4, 8 and 16
// realisations, a thread and a stream each, cluster launches and a launch a
// phase (ms a timestep): 602 rows FP64 18.0 and 20.7, 4.99 and 5.99, 3.15 and
// 3.59, 2.14 and 2.24, FP32 3.73 and 4.00, 1.27 and 1.30, 1.07 and 1.05, 1.07
// and 1.04; 8002 rows FP64 47.2 and 48.4, 12.3 and 13.7, 8.51 and 9.95, 7.11
// and 7.92, FP32 4.59 and 4.64, 1.56 and 1.63, 1.07 and 1.12, 0.92 and 0.94.
// cluster_rows < 0 asks for no cluster launch.
constexpr int kSmallRows = 8192;

bool cpr_small(const Sim *s) {
  return s->opt.precond == 2 && s->opt.use_graphs && s->opt.cluster_rows >= 0 && s->cl_size > 0 &&
         s->ncolour <= kSmallColours &&
         s->K.n <= kSmallRows;
}

template <typename T>
int cpr_small_part(Sim *s, int part, const double *r, double *z, const int *omap,
                   const X0Init &xi, bool colour_z) {
  SmallArgs<T> A{};
  A.n = s->K.n;
  A.nL = s->lu_nL;
  A.ncol = s->ncolour;
  A.last = s->ncolour - 1;
  while (A.last >= 0 && s->lu_cstart[A.last + 1] <= s->lu_cstart[A.last]) --A.last;
  for (int c = 0; c <= s->ncolour; ++c) A.cstart[c] = s->lu_cstart[c];
  for (int c = 0; c < s->ncolour; ++c)
    if (s->lu_cmaxlen[c] > kLongRow) A.lng |= 1 << c;
  A.perm = s->perm; A.iperm = s->iperm; A.Lptr = s->lu_Lptr; A.Uptr = s->lu_Uptr;
  A.colp = s->lu_colp;
  A.sL = s->sv_sL; A.sc = s->sv_sc; A.long0 = s->sv_long0;
  A.srowptr = s->srowptr;
  A.scol = s->scol;
  A.r = r; A.z = z; A.omap = omap;
  if constexpr (sizeof(T) == 8) {
    A.lu = s->lu_val;
    A.zp = A.zp2 = s->ilu_zp;
    A.sval = s->sval; A.a00 = s->sa00; A.a01 = s->sa01;
    A.z1 = s->z1; A.r1 = s->r1; A.rp = s->rp; A.xp = s->xp;
  } else {
    A.lu = s->lu_valf;
    A.zp = reinterpret_cast<float *>(s->ilu_zp);
    A.zp2 = reinterpret_cast<float *>(s->ilu_zp2);
    A.svalf = s->svalf;
    A.spf = reinterpret_cast<const float2 *>(s->spf);
    A.z1f = s->z1f; A.r1f = s->r1f; A.bf = s->lev[0].bf; A.xf = s->lev[0].xf;
    if (colour_z) {
      A.z2c = s->z2c;
      A.scol = s->scolc;
    }
    A.xi = xi;
  }
  return part == 0 ? launch_small<T, 0>(s, A) : launch_small<T, 1>(s, A);
}

template int cpr_small_part<double>(Sim *, int, const double *, double *, const int *,
                                    const X0Init &, bool);
template int cpr_small_part<float>(Sim *, int, const double *, double *, const int *,
                                   const X0Init &, bool);

// ---------------------------------------------------------------- Arnoldi step
// The rest of a small realisation's Arnoldi step in one cluster launch: w = A
// z_j, classical Gram-Schmidt against v_0..v_j with the DGKS test (the second
// pass only when it asks for one), v_{j+1}, and the Givens rotations of the
// new column, where one launch each takes 9 to 15, most of them shorter than
// a launch.  Every CTA keeps its slice of w in shared memory; the partial
// projections go to all CTAs through distributed shared memory, so each sums
// them in the same order to the same bits and takes the same branch.
constexpr int kOrthSlice = 2048;   // doubles of w a CTA

struct OrthArgs {
  int n, sL, sc, long0, j, m;
  const int *rowptr, *col;
  const double *val, *z, *V;
  double *vnext, *H, *cs, *sn, *g, *scal;
  double reorth;
};

__global__ void __launch_bounds__(kSmallThreads, 1) k_orth_small(const OrthArgs A, int trig) {
  __shared__ double ws[kOrthSlice];
  __shared__ double part[2][16][32];   // by pass, CTA and vector (31: w . w)
  __shared__ double h[32], hc[32], dec[3];   // projections, their sum, (again, beta, 1 / beta)
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), C = (int)cl.num_blocks();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = kSmallThreads / 32;
  const long long N = 2LL * A.n;
  const int chunk = (int)((N + 2 * C - 1) / (2 * C)) * 2;
  const int lo = min(rank * chunk, (int)N), len = min(chunk, (int)N - lo), nv = A.j + 1;
  small_arrive();   // waited for before the first store to another CTA's shared memory
  griddep_wait();
  if (trig) griddep_launch_dependents();
  {   // w = A z over the slice's rows, as k_bsr_spmv_b<0>
    const double2 *x2 = reinterpret_cast<const double2 *>(A.z);
    for (int t = threadIdx.x; t < len; t += kSmallThreads) {
      const int i = (lo + t) >> 1, comp = t & 1;   // lo is even
      if (i >= A.long0) continue;
      const int q = storage_row(i, A.sL, A.sc);
      const double2 *v2 = reinterpret_cast<const double2 *>(A.val) + comp;
      double s = 0.0;
#pragma unroll 4
      for (int e = __ldg(A.rowptr + q), e1 = __ldg(A.rowptr + q + 1); e < e1; ++e) {
        double2 a = __ldg(v2 + 2 * (size_t)e), xj = x2[__ldg(A.col + e)];
        s = fma(a.x, xj.x, s);
        s = fma(a.y, xj.y, s);
      }
      ws[t] = s;
    }
    const double2 *v2 = reinterpret_cast<const double2 *>(A.val);
    for (int i = max(A.long0, lo >> 1) + warp; 2 * i < lo + len; i += nw) {
      double s0 = 0.0, s1 = 0.0;
      for (int e = __ldg(A.rowptr + i) + lane, e1 = __ldg(A.rowptr + i + 1); e < e1; e += 32) {
        double2 a = __ldg(v2 + 2 * (size_t)e), c = __ldg(v2 + 2 * (size_t)e + 1);
        double2 xj = x2[__ldg(A.col + e)];
        s0 = fma(a.x, xj.x, fma(a.y, xj.y, s0));
        s1 = fma(c.x, xj.x, fma(c.y, xj.y, s1));
      }
      s0 = warp_sum(s0);
      s1 = warp_sum(s1);
      if (lane == 0) {
        ws[2 * i - lo] = s0;
        ws[2 * i + 1 - lo] = s1;
      }
    }
  }
  __syncthreads();
  small_wait();   // every CTA of the cluster has started: its shared memory may be written
  for (int pass = 0; pass < 2; ++pass) {
    for (int k = warp; k <= nv; k += nw) {   // a warp per vector (nv: w itself)
      const double *v = A.V + (k < nv ? k : 0) * N + lo;
      double s0 = 0.0, s1 = 0.0;
      int t = lane;
      for (; t + 32 < len; t += 64) {
        double a = k < nv ? v[t] : ws[t], b = k < nv ? v[t + 32] : ws[t + 32];
        s0 = fma(a, ws[t], s0);
        s1 = fma(b, ws[t + 32], s1);
      }
      if (t < len) s0 = fma(k < nv ? v[t] : ws[t], ws[t], s0);
      s0 = warp_sum(s0 + s1);
      if (lane < C) *cl.map_shared_rank(&part[pass][rank][k < nv ? k : 31], lane) = s0;
    }
    cl.sync();
    {   // vector 2 warp + (lane / 16): its C partials
      const int k = 2 * warp + (lane >> 4), r = lane & 15;
      double v = r < C && (k < nv || k == 31) ? part[pass][r][k] : 0.0;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, 16);
      if (r == 0) h[k] = v;
    }
    __syncthreads();
    if (warp == 0) {
      const double v = lane < nv ? h[lane] : 0.0;
      const double hh = warp_sum(v * v), ww = h[31], b2 = ww - hh;
      hc[lane] = pass == 0 ? v : hc[lane] + v;
      if (lane == 0) {
        const bool again = pass == 0 && (A.reorth >= 1.0 || b2 < A.reorth * ww);
        const double beta = sqrt(b2 > 0.0 ? b2 : 0.0);
        dec[0] = again ? 1.0 : 0.0;
        dec[1] = beta;
        dec[2] = beta != 0.0 ? 1.0 / beta : 0.0;
      }
    }
    __syncthreads();
    const bool again = dec[0] != 0.0;
    const double rb = dec[2];
    for (int t = threadIdx.x; t < len; t += kSmallThreads) {
      double acc = ws[t];
      const double *v = A.V + lo + t;
#pragma unroll 4
      for (int k = 0; k < nv; ++k) acc = fma(-h[k], v[k * N], acc);
      if (again) ws[t] = acc;
      else A.vnext[lo + t] = acc * rb;
    }
    if (!again) break;   // the same in every CTA
    __syncthreads();
  }
  if (rank != 0 || warp != 0) return;
  // the Givens rotations of column j (k_givens_b): lane 0 forms the rotated
  // entry, lane 1 the one carried on
  const int j = A.j, m = A.m;
  const double beta = dec[1];
  const double c0 = lane < j ? A.cs[lane] : 0.0, s0 = lane < j ? A.sn[lane] : 0.0;
  double a = hc[0], out = 0.0;
  for (int i = 0; i < j; ++i) {
    const double ci = __shfl_sync(0xffffffffu, c0, i), si = __shfl_sync(0xffffffffu, s0, i);
    const double c = hc[i + 1];
    const double r = fma(lane == 0 ? si : ci, c, (lane == 0 ? ci : -si) * a);
    const double top = __shfl_sync(0xffffffffu, r, 0);
    if (lane == i) out = top;
    a = __shfl_sync(0xffffffffu, r, 1);
  }
  const double rr = sqrt(a * a + beta * beta);
  const double cj = rr == 0.0 ? 1.0 : a / rr, sj = rr == 0.0 ? 0.0 : beta / rr;
  if (lane < j) A.H[(size_t)lane * m + j] = out;
  if (lane == 0) {
    A.cs[j] = cj;
    A.sn[j] = sj;
    A.H[(size_t)j * m + j] = rr;
    A.H[(size_t)(j + 1) * m + j] = 0.0;
    const double gj = A.g[j], gn = -sj * gj;
    A.g[j + 1] = gn;
    A.g[j] = cj * gj;
    A.scal[2] = beta;
    A.scal[3] = fabs(gn);
    A.scal[4] = 0.0;
  }
}

bool orth_small(const Sim *s) {
  return s->opt.precond == 2 && s->opt.use_graphs && s->opt.cluster_rows >= 0 && s->cl_size > 0 &&
         s->K.n <= kSmallRows && 2LL * s->K.n <= (long long)s->cl_size * (kOrthSlice - 2);
}

int orth_small_step(Sim *s, int j, const double *z, double *vnext) {
  OrthArgs A;
  A.n = s->K.n; A.sL = s->sv_sL; A.sc = s->sv_sc; A.long0 = s->sv_long0;
  A.j = j; A.m = s->m;
  A.rowptr = s->srowptr; A.col = s->scol; A.val = s->sval;
  A.z = z; A.V = s->V; A.vnext = vnext;
  A.H = s->H; A.cs = s->cs; A.sn = s->sn; A.g = s->g; A.scal = s->scal;
  A.reorth = s->opt.reorth;
  DP_CUDA(s, (kernel_attribute<k_orth_small, cudaFuncAttributeNonPortableClusterSizeAllowed>(1)));
  return launch_cluster(s, "k_orth_small", k_orth_small, A);
}

}  // namespace dp
