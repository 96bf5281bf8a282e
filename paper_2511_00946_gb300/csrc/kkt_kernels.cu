// Kernels of the partitioned block Cholesky factorization and solve of an SPD
// block-tridiagonal-arrow KKT matrix (arXiv 2511.00946, Algorithms 1-3), and
// of the FP64 residual used by mixed-precision iterative refinement.
//
// One CTA per segment task. Per stage the CTA keeps the pivot block, the
// stacked panel Z = [E; G; W] and the Schur accumulator T in shared memory
// (row-major, odd leading dimensions: row- and column-wise accesses are free
// of bank conflicts) and runs
//   D-hat = chol(D)  ->  Z <- Z D-hat^{-T}  ->  T -= Z Z^T (lower triangle)
// FP64 is the scarce resource on this part: one FP64 warp-instruction occupies
// a sub-partition's FP64 pipe for about 64-76 cycles whether 1 or 32 lanes are
// active, and FP32 runs about 70x faster. So the loops issue FP64 instructions
// from full warps only (lower triangles are enumerated linearly instead of
// masked squares). FP64 tasks (k_factor_fp64, k_factor_clus) eliminate the pivot
// block without square roots in blocks of eight columns, the panel solve beside
// it (ldl_sweep), and take the Schur products of blocks n >= kDigMin from the
// tensor cores by exact digit splitting (kkt_oz.cuh). Mixed tasks (k_factor) keep
// the pivot Cholesky and the Schur accumulator in FP64: the panel solve and the
// dot products run in FP32 and each dot product is subtracted from the FP64
// accumulator once. Blocks n <= kWarpMaxN run one warp per task (k_factor_w).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <unordered_map>

#include "kkt_internal.h"
#include "kkt_bulk.cuh"
#include "kkt_numerics.cuh"
#include "kkt_oz.cuh"
#include "kkt_tc.cuh"

namespace kkt {
namespace {

constexpr int kMaxDevices = 64;  // devices whose kernel attributes are recorded

__device__ __forceinline__ int odd(int c) { return c | 1; }

// e / d for 0 <= e < 2^20 / d (every block: at most 112 x 48 elements, d <= 113)
// by a multiplication: an integer division costs about 20 instructions, and
// the block loops below run one per element.
struct Div {
  unsigned inv;
  __device__ __forceinline__ explicit Div(int d) : inv((1u << 20) / (unsigned)d + 1u) {}
  __device__ __forceinline__ int operator()(int e) const { return (int)((unsigned)e * inv >> 20); }
};

// Row-by-row enumeration of a lower triangle (diagonal included):
// e -> (a, b) with 0 <= b <= a, e = a(a+1)/2 + b.
__device__ __forceinline__ void tri_rc(int e, int& a, int& b) {
  int r = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
  while (r * (r + 1) / 2 > e) --r;
  while ((r + 1) * (r + 2) / 2 <= e) ++r;
  a = r;
  b = e - r * (r + 1) / 2;
}

__device__ void record_status(Info* info, int status, int sys, int stage, int level) {
  if (atomicCAS(&info->status, 0, -1) == 0) {
    info->system = sys;
    info->stage = stage;
    info->level = level;
    __threadfence();
    atomicExch(&info->status, status);
  }
}
__device__ void record_breakdown(Info* info, int sys, int stage, int level) {
  record_status(info, 3 /* KKT_ERR_NOT_SPD */, sys, stage, level);
}
// a bounded device wait ran out (the kernel carries on; its results are invalid)
__device__ void record_timeout(Info* info, int sys, int stage, int level) {
  record_status(info, 5 /* KKT_ERR_TIMEOUT */, sys, stage, level);
}

// Debug build (compiled with -DKKT_DEBUG): index checks on entry to every
// segment task and residual task. A task whose geometry does not fit its
// system (segment index, stage range, separator, block sizes) or whose
// shared-memory layout does not fit the launch's dynamic shared memory is
// skipped, and the first such failure is recorded (status 8,
// KKT_ERR_BOUNDS) in a device record that kkt_get_info reports. Nothing
// traps. In the normal build the checks compile to nothing.
#ifdef KKT_DEBUG
__device__ Info g_debug_info;
#endif
extern __shared__ __align__(16) unsigned char kkt_dyn_smem[];
__device__ __forceinline__ bool dbg_ok(bool cond, const LevelDesc& d) {
#ifdef KKT_DEBUG
  if (!cond) record_status(&g_debug_info, 8, d.sys, -1, d.level);
  return cond;
#else
  (void)d;
  return cond || true;
#endif
}
__device__ __forceinline__ bool task_geometry_ok(const LevelDesc& d, int seg, const void* sm, int bytes) {
#ifdef KKT_DEBUG
  unsigned dyn;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
  const long long off = (long long)__cvta_generic_to_shared(sm) - (long long)__cvta_generic_to_shared(kkt_dyn_smem);
  bool ok = d.n >= 1 && d.n <= kMaxN && d.m >= 0 && d.m <= kMaxM && d.N >= 1 && d.P >= 1 && seg >= 0 &&
            seg < d.P && d.mr >= 0 && d.mr <= d.m;
  if (ok) {
    const int f = d.seg[seg], e = d.seg[seg + 1] - 2;  // first and last stage of the segment
    ok = f >= (seg ? 1 : 0) && e >= f && e < d.N && d.seg[d.P] == d.N + 1;
    if (ok) ok = d.nat[f] >= 0 && d.nat[e] < d.Nnat && (seg == 0 || d.nat[f - 1] >= 0);
  }
  ok = ok && off >= 0 && off + bytes <= (long long)dyn;
  return dbg_ok(ok, d);
#else
  (void)d; (void)seg; (void)sm; (void)bytes;
  return true;
#endif
}

// A group of threads working on one role of a CTA: thread index within the
// group, group size and the named barrier that synchronizes it (0 = the whole
// CTA, __syncthreads; -1 = a single warp, __syncwarp).
struct Grp {
  int tid, nt, bar;
};
__device__ __forceinline__ Grp cta_grp() { return Grp{(int)threadIdx.x, (int)blockDim.x, 0}; }

__device__ __forceinline__ void group_bar(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
__device__ __forceinline__ void gsync(const Grp& g) {
  if (g.bar == 0) __syncthreads();
  else if (g.bar < 0) __syncwarp();
  else group_bar(g.bar, g.nt);
}

// dst (rows x cols, smem, ld) <- A (+ B) from global row-major [rows][cols],
// or the transpose of A (+ B) given as [cols][rows] when `trans`. A null A
// loads zeros. Coalesced over the global array.
// The three source cases are separate loops: a predicated-off FP64 add still
// holds the FP64 pipe on this part.
// U > 1: every thread issues U loads before their stores. The stores go to
// shared memory, which the compiler cannot prove disjoint from A and B, so
// with U = 1 each load's latency is waited out in turn (U = 1 keeps the
// register footprint of the warp kernels).
template <int U = 1, typename T>
__device__ void load_blk(T* dst, int ld, const double* A, const double* B, int rows, int cols,
                         bool trans, Grp g = cta_grp()) {
  const int tot = rows * cols;
  const Div by(trans ? rows : cols);
  auto at = [&](int e) {
    int r, c;
    if (trans) { c = by(e); r = e - c * rows; }
    else { r = by(e); c = e - r * cols; }
    return r * ld + c;
  };
  auto batched = [&](auto get) {
    for (int e0 = g.tid; e0 < tot; e0 += U * g.nt) {
      double v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = e0 + u * g.nt;
        v[u] = e < tot ? get(e) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = e0 + u * g.nt;
        if (e < tot) dst[at(e)] = (T)v[u];
      }
    }
  };
  if (A && B) {
    if constexpr (U > 1) batched([&](int e) { return A[e] + B[e]; });
    else for (int e = g.tid; e < tot; e += g.nt) dst[at(e)] = (T)(A[e] + B[e]);
  } else if (A) {
    if constexpr (U > 1) batched([&](int e) { return A[e]; });
    else for (int e = g.tid; e < tot; e += g.nt) dst[at(e)] = (T)A[e];
  } else {
    for (int e = g.tid; e < tot; e += g.nt) dst[at(e)] = T(0);
  }
}

// global row-major [rows][cols] <- src (smem), or the transpose when `trans`
// (dst is then [cols][rows]). `lower` writes zeros above the diagonal.
template <typename TD, typename TS>
__device__ void store_blk(TD* dst, const TS* src, int ld, int rows, int cols, bool trans,
                          bool lower, Grp g = cta_grp()) {
  const int tot = rows * cols;
  const Div by(trans ? rows : cols);
  for (int e = g.tid; e < tot; e += g.nt) {
    int r, c;
    if (trans) { c = by(e); r = e - c * rows; }
    else { r = by(e); c = e - r * cols; }
    TS v = src[r * ld + c];
    if (lower && c > r) v = TS(0);
    dst[e] = (TD)v;
  }
}

// smem -> smem copy of a rows x cols block (with conversion)
template <typename TD, typename TS>
__device__ void copy_blk(TD* dst, int ldd, const TS* src, int lds, int rows, int cols,
                         Grp g = cta_grp()) {
  const Div by(cols);
  for (int e = g.tid; e < rows * cols; e += g.nt) {
    const int r = by(e), c = e - r * cols;
    dst[r * ldd + c] = (TD)src[r * lds + c];
  }
}

// Element table of the trailing updates of an n x n Cholesky: the pairs
// (i, k) with 2 <= k <= i < n ordered by k descending (packed i << 16 | k),
// so that the updates applied by column j form the prefix of length
// (n-2-j)(n-1-j)/2. Built once per CTA (it depends on n only).
__device__ void potrf_table(int* tab, int n) {
  const int np = (n - 2) * (n - 1) / 2;
  for (int e = threadIdx.x; e < np; e += blockDim.x) {
    int a, b;
    tri_rc(e, a, b);
    const int k = n - 1 - a;
    tab[e] = (k + b) << 16 | k;
  }
}

// Column steps of the in-place lower Cholesky of A (n x n, FP64, n <= 64),
// right-looking with a one-column look-ahead: in the phase of column j
// (final and scaled), warp 0 alone updates column j+1, computes its pivot
// from the register holding the diagonal and scales it, so the serial pivot
// chain runs on a sub-pipe of its own, while warps 1-3 walk the prefix of the
// element table `tab` for the trailing columns. Every loop has a runtime trip
// count: on this part a predicated-off FP64 instruction still holds the FP64
// pipe, so no FP64 work is issued for inactive elements. On a pivot that is
// not positive *bad is set (first column + 1) and the factorization carries
// on (NaNs propagate; no trap). rinv[j] = 1 / L_jj.
__device__ __forceinline__ void potrf_col0(double* A, int ld, int n, double* rinv, int* bad, int lane) {
  const double d = A[0];
  const double r = pivot_rsqrt(d);
  if (lane == 0) {
    if (not_positive(d) && *bad == 0) *bad = 1;
    rinv[0] = r;
  }
  // (lane 0 scales the diagonal: L_00 = d r)
  for (int i = lane; i < n; i += 32) A[i * ld] *= r;
}

// warp 0 in the phase of column j: column j+1 updated, pivoted and scaled
__device__ __forceinline__ void potrf_lookahead(double* A, int ld, int n, double* rinv, int* bad, int j,
                                                int lane) {
  const double lj = A[(j + 1) * ld + j];
  const int i0 = j + 1 + lane, i1 = i0 + 32;
  const bool two = j + 33 < n;  // warp-uniform: a second row per lane
  double v0 = 0.0, v1 = 0.0;
  if (i0 < n) v0 = fma(-A[i0 * ld + j], lj, A[i0 * ld + j + 1]);
  if (two) {
    if (i1 < n) v1 = fma(-A[i1 * ld + j], lj, A[i1 * ld + j + 1]);
  }
  double r = 0.0;
  if (lane == 0) {  // v0 is the diagonal element (j+1, j+1)
    if (not_positive(v0) && *bad == 0) *bad = j + 2;
    r = pivot_rsqrt(v0);
    rinv[j + 1] = r;
  }
  r = __shfl_sync(0xffffffffu, r, 0);
  // one FP64 multiply for the whole column, the diagonal L_{j+1,j+1} = v0 r on lane 0
  if (i0 < n) A[i0 * ld + j + 1] = v0 * r;
  if (two) {
    if (i1 < n) A[i1 * ld + j + 1] = v1 * r;
  }
}

// warps 1-3 in the phase of column j: the updates of columns j+2.. by column j
__device__ __forceinline__ void potrf_trailing(double* A, int ld, int n, const int* tab, int j, int t,
                                               int nt) {
  const int cnt = (n - 2 - j) * (n - 1 - j) / 2;
  for (int e = t; e < cnt; e += nt) {
    const int p = tab[e], i = p >> 16, k = p & 0xffff;
    A[i * ld + k] = fma(-A[i * ld + j], A[k * ld + j], A[i * ld + k]);
  }
}

// Fused pivot factorization (FP64) and panel solve (in the panel type TZ: FP32
// in the mixed variant) by the whole CTA: the Cholesky above and Z[r0, r1) <-
// Z[r0, r1) L^{-T} in the division-free form of trsm_panel (the same operations
// in the same order). Warp 0 runs the pivot chain; in the phase of column j the
// other warps run, each as a tight strided loop,
//   - the trailing updates of columns j+2.. by column j,
//   - the panel operand column M[c][j] = L[c][j] / L[j][j] (c > j),
//   - the panel updates z_c -= z_{j-1} M[c][j-1] (c >= j) of every row,
// so the panel lags the factorization by two columns and runs beside the
// pivot chain instead of after it. x_c = z_c / L_cc closes the sweep. One
// barrier per phase; the caller synchronizes the CTA before the results are read.
template <typename TZ>
__device__ void potrf_trsm_sm(double* A, int ld, int n, double* rinv, TZ* M, const int* tab, int* bad,
                              TZ* Z, int ldz, int r0, int r1) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int w = tid - 32;  // worker index
  const int nwk = kFactorThreads - 32;
  const int rows = r1 - r0;
  // panel mapping: `per` workers on a row, each on every per-th column
  const int per = rows > 0 ? max(1, nwk / rows) : 0;
  const bool pact = tid >= 32 && w < rows * per;
  const int pr = pact ? w % rows : 0, pc = pact ? w / rows : 0;
  TZ* zr = Z + (r0 + pr) * ldz;
  if (tid < 32) potrf_col0(A, ld, n, rinv, bad, lane);
  group_bar(1, kFactorThreads);
  for (int j = 0; j < n; ++j) {
    if (tid < 32) {
      if (j + 1 < n) potrf_lookahead(A, ld, n, rinv, bad, j, lane);
    } else {
      potrf_trailing(A, ld, n, tab, j, w, nwk);
      for (int c = j + 1 + w; c < n; c += nwk) M[c * ld + j] = (TZ)(A[c * ld + j] * rinv[j]);
      if (pact && j >= 1) {
        const TZ zj = zr[j - 1];
        for (int c = j + pc; c < n; c += per) zr[c] = fma(-zj, M[c * ld + j - 1], zr[c]);
      }
    }
    group_bar(1, kFactorThreads);
  }
  if (tid >= 32)
    for (int e = w; e < rows * n; e += nwk) {
      const int r = e / n, c = e - r * n;
      Z[(r0 + r) * ldz + c] *= (TZ)rinv[c];
    }
}

// Z[r0:r1) <- Z[r0:r1) L^{-T} with the pre-scaled columns M (M_cj = L_cj /
// L_jj), in the panel type TZ: for each row, u_c = z_c - sum_{k<c} u_k M_ck
// (in k order) and x_c = u_c / L_cc (times rinv). Column sweep: every thread
// works on every column (FP64 from full warps), thread t owning row
// r0 + t % rows and every (nt/rows)-th column. The group needs at least as
// many threads as rows (true for every panel: at most 2 kMaxN + kMaxM rows).
template <typename TZ>
__device__ void trsm_panel(TZ* Z, int ldz, int r0, int r1, const TZ* M, int ldm, int n, const TZ* rinv,
                           Grp g) {
  const int rows = r1 - r0;
  if (rows <= 0) return;
  const int per = g.nt / rows;  // threads per row (>= 1)
  const int rr = g.tid % rows, cc = g.tid / rows;
  const bool act = cc < per;
  TZ* zr = Z + (r0 + rr) * ldz;
  for (int j = 0; j < n - 1; ++j) {
    if (act) {
      const TZ zj = zr[j];
      for (int c = j + 1 + cc; c < n; c += per) zr[c] = fma(-zj, M[c * ldm + j], zr[c]);
    }
    gsync(g);
  }
  if (act)
    for (int c = cc; c < n; c += per) zr[c] *= rinv[c];
  gsync(g);
}

// T[a][b] -= sum_t Z[a][t] Z[b][t] for ra0 <= a < ra1, cb0 <= b <= a (cb0 <=
// ra0: a rectangle of full rows beside a lower triangle; ra0 = cb0 is a plain
// lower triangle). Panel rows below `zsplit` are read from Zlo, the others
// from Z (same leading dimension and row numbering). FP64 panels: T_ab takes
// the rank-1 updates of the columns t = 0, 1, .. in turn, each one fma. FP32
// panels (mixed variant): the dot product is formed in FP32 and subtracted
// from the FP64 accumulator once.
template <typename TZ>
__device__ void syrk_trap(double* T, int ldt, const TZ* Zlo, const TZ* Z, int zsplit, int ldz, int ra0,
                          int ra1, int cb0, int n, Grp g) {
  const int w0 = ra0 - cb0, h = ra1 - ra0;
  const int tot = h * w0 + h * (h + 1) / 2;  // row a holds a - cb0 + 1 elements
  // (a, b) of element g.tid, then advanced by g.nt along the rows
  int a = ra0, b = cb0 + g.tid;
  while (a < ra1 && b > a) { b -= a - cb0 + 1; ++a; }
  for (int e = g.tid; e < tot; e += g.nt) {
    if (e != g.tid) {
      b += g.nt;
      while (b > a) { b -= a - cb0 + 1; ++a; }
    }
    const TZ* zi = (a < zsplit ? Zlo : Z) + a * ldz;
    const TZ* zj = (b < zsplit ? Zlo : Z) + b * ldz;
    if (sizeof(TZ) == 8) {
      // FP64: rank-1 updates in column order, T_ab = fma(-z_at, z_bt, T_ab): no
      // partial sums to combine, and one dependent chain per element already
      // keeps an FP64 pipe busy on this part
      double acc = T[a * ldt + b];
      for (int t = 0; t < n; ++t) acc = fma(-(double)zi[t], (double)zj[t], acc);
      T[a * ldt + b] = acc;
    } else {
      TZ s0 = 0, s1 = 0, s2 = 0, s3 = 0;
      int t = 0;
      for (; t + 3 < n; t += 4) {
        s0 = fma(zi[t], zj[t], s0);
        s1 = fma(zi[t + 1], zj[t + 1], s1);
        s2 = fma(zi[t + 2], zj[t + 2], s2);
        s3 = fma(zi[t + 3], zj[t + 3], s3);
      }
      for (; t < n; ++t) s0 = fma(zi[t], zj[t], s0);
      T[a * ldt + b] -= (double)((s0 + s1) + (s2 + s3));
    }
  }
  gsync(g);
}

// ---------------------------------------------------------------------------
// FP64 Schur products on the tensor cores (kkt_oz.cuh).
// ---------------------------------------------------------------------------

// Smallest block whose Schur products take digits; smaller ones take FP64 FMAs
// (syrk_trap) and keep their doubles. A tile costs the same 28 products per 16
// columns however few rows and columns are left, so small panels are faster in
// FMAs, most of all where a task has its SM to itself. Digits against FMAs, us:
// one system of N = 300, m = 4 in one pass, n = 17 309, 289, n = 19 321, 314, n = 20
// 328, 323, n = 22 344, 338; 160 systems of four segments, N = 40, n = 17 542, 586,
// n = 19 577, 705, n = 20 600, 745. One line for every layout, whose results agree
// bit for bit.
constexpr int kDigMin = 20;

// T[a][b] -= sum_t Z[a][t] Z[b][t] for ra0 <= a < ra1, cb0 <= b <= a (cb0 <=
// ra0), rows in digits (panel_out; n < kDigMin: doubles). Panel rows below `zsplit` are read from
// (Zlo, flo), the others from (Z, fz). One 16 x 8 tile per warp at a time.
// Every element is one sum rounded once, so the result does not depend on the
// tiling.
// BORDER: row ry is a bordered right-hand side. Its entries have no common
// scale (a right-hand side may hold numbers 10^12 apart that nothing couples),
// so it keeps its doubles and its products are FP64 FMAs against the solved
// rows in device memory, Pd (row-major, n columns; complete): two lanes a row,
// jobs of sixteen rows ahead of the tiles in the warps' list, where the FP64 pipe
// is idle beside the other warps' tiles (1172 us for N = 777, n = 45; behind the
// tiles 1175, four lanes a row 1177 and 1190).
// Ends with the group's barrier.
template <bool BORDER>
__device__ void oz_syrk(double* T, int ldt, const double* Zlo, const int* flo, const double* Z, const int* fz,
                        int zsplit, int ldz, int ra0, int ra1, int cb0, int n, int ry, const double* Pd, Grp G) {
  if (n < kDigMin) {
    syrk_trap(T, ldt, Zlo, Z, zsplit, ldz, ra0, ra1, cb0, n, G);
    return;
  }
  const int lane = G.tid & 31, nw = G.nt >> 5, w0 = ra0 - cb0;
  int i = 0, j = G.tid >> 5;
  if constexpr (BORDER) {
    // (ry, b) for cb0 <= b < ry, then (a, ry) for the rows a behind ry
    const int left = ry >= ra0 && ry < ra1 ? ry - cb0 : 0, a0 = max(ra0, ry + 1), tot = left + max(0, ra1 - a0);
    const double* const y = (ry < zsplit ? Zlo : Z) + ry * ldz;
    for (; 16 * j < tot; j += nw) {
      const int e = 16 * j + (lane >> 1), ee = min(e, tot - 1), o = ee < left ? cb0 + ee : a0 + ee - left;
      const double* const p = Pd + (size_t)o * n;
      double acc = 0.0;
#pragma unroll 1
      for (int k0 = 0; k0 < n; k0 += 16) {
        double v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int k = k0 + 2 * q + (lane & 1);
          v[q] = k < n ? p[k] : 0.0;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int k = k0 + 2 * q;
          if (k < n) acc = fma(v[q], k + (lane & 1) < n ? y[k + (lane & 1)] : 0.0, acc);  // (warp-uniform)
        }
      }
      acc += __shfl_xor_sync(0xffffffffu, acc, 1);
      if (e < tot && (lane & 1) == 0) T[max(o, ry) * ldt + min(o, ry)] -= acc;
    }
    j -= (tot + 15) >> 4;
  }
  // row tile i has cols(i) column tiles; this warp takes every nw-th tile
  for (;;) {
    for (; ra0 + 16 * i < ra1; ++i) {
      const int cols = (w0 + min(16 * i + 16, ra1 - ra0) + 7) >> 3;
      if (j < cols) break;
      j -= cols;
    }
    if (ra0 + 16 * i >= ra1) break;
    oz::tile<BORDER>(T, ldt, Zlo, flo, Z, fz, zsplit, ldz, ra0 + 16 * i, ra1, cb0 + 8 * j, ra1, n, lane, ry);
    j += nw;
  }
  gsync(G);
}

// ---------------------------------------------------------------------------
// Pivot factorization and panel solve of one FP64 stage, in blocks of eight
// columns. Within a block the columns are eliminated in the square-root-free
// form: with v_c the column after the earlier updates and d_c = v_cc, m_c =
// v_c / d_c (the panel operand L_rc / L_cc) and v_i -= v_c m_ic. So the chain
// from one pivot to the next is a shuffle, a reciprocal in integer arithmetic
// (pivot_rcp), one multiply and one FMA (the lanes keep their own diagonal
// elements up to date), against six dependent FP64 instructions and a block
// barrier per column before (1080-1250 cycles a column); 1 / L_cc =
// 1 / sqrt(d_c) is formed off the chain. The panel behind a block (u m^T, u the
// unscaled solution) is updated by FP64 FMAs, one element per lane. (Digit
// products of eight columns took the FMAs off the FP64 pipe but stood longer in
// the sweep: encoding, a barrier and a tile of 28 products for eight columns.
// Digits against FMAs, us: one system of N = 300, m = 4, n = 26 438, 396, n = 32
// 485, 453, n = 48 853, 818; 1200 systems of N = 40, n = 26 3396, 2898, n = 32
// 4274, 4132, n = 48 10703, 10946.)
// Schedule: warp 0 eliminates block J. Meanwhile the other warps finish block
// J - 1: the pivot block's columns beyond block J, the panel's block J - 1
// (one row per thread, or eight lanes per row where the rows are few) and the
// panel behind it. Then all warps update the pivot block's next eight columns.
// ---------------------------------------------------------------------------
constexpr int kLB = 8;         // columns per block
constexpr int kBarSweep = 2;   // barrier of warps 1 and up

// Warp 0: columns [c0, c0 + cn) of the pivot block A (row-major FP64, updated
// by the blocks before), rows c0 + lane + 32 q: v and d into A, m into M (same
// ld). Every lane keeps its own row's diagonal element up to date, d_r -=
// v_rc^2 / d_c with the square formed beforehand, so the chain from pivot to
// pivot is one shuffle, one reciprocal and one FMA. FULL: cn = kLB. Without SAFE
// the code has no branch inside (the updates fill the reciprocal's latency:
// 4.3k cycles a block against 5.5k) and returns false, with nothing written to A,
// where a pivot fails pivot_rcp_ok; SAFE forms no square, divides by the pivots
// that fail it and takes any, *bad is then the first column + 1 that is not
// positive. Blocks that a handle runs one warp per task (potrf_w) take SAFE at
// once: its operations are potrf_w's, and kkt_solve_noalloc then agrees with a
// handle on systems so ill-conditioned that no other rounding would.
template <int SL, bool FULL, bool SAFE>
__device__ __forceinline__ bool ldl_block_t(double* A, double* M, int ld, int n, int c0, int cn, int* bad, int lane) {
  double v[SL][kLB];
#pragma unroll
  for (int q = 0; q < SL; ++q) {
    const int r = c0 + lane + 32 * q;
#pragma unroll
    for (int c = 0; c < kLB; ++c) v[q][c] = r < n && (FULL || c < cn) && c0 + c < r ? A[r * ld + c0 + c] : 0.0;
  }
  double dg = lane < cn ? A[(c0 + lane) * ld + c0 + lane] : 1.0;  // this lane's diagonal element
  double vv = v[0][0] * v[0][0];
  int first = 0;
  bool ok = true;
#pragma unroll
  for (int c = 0; c < kLB; ++c) {
    if (FULL || c < cn) {  // warp-uniform
      const double d = __shfl_sync(0xffffffffu, dg, c);
      double m[SL], dn;
      if (SAFE) {
        if (not_positive(d) && first == 0) first = c0 + c + 1;
#pragma unroll
        for (int q = 0; q < SL; ++q)
          m[q] = pivot_rcp_ok(d)   ? v[q][c] * pivot_rcp(d)
                 : not_positive(d) ? __longlong_as_double(0x7ff8000000000000LL)
                                   : v[q][c] / d;
        dn = fma(-v[0][c], m[0], dg);
      } else {
        ok = ok && pivot_rcp_ok(d);
        const double ri = pivot_rcp(d);
        dn = fma(-vv, ri, dg);
#pragma unroll
        for (int q = 0; q < SL; ++q) m[q] = v[q][c] * ri;
      }
      dg = lane > c ? dn : dg;  // (lane c keeps d)
#pragma unroll
      for (int q = 0; q < SL; ++q) {
        const int r = c0 + lane + 32 * q;
        if (r < n && r > c0 + c) M[r * ld + c0 + c] = m[q];
      }
      __syncwarp();
#pragma unroll
      for (int i = c + 1; i < kLB; ++i) {
        if (FULL || i < cn) {
          const double mi = M[(c0 + i) * ld + c0 + c];
#pragma unroll
          for (int q = 0; q < SL; ++q) v[q][i] = fma(-v[q][c], mi, v[q][i]);
        }
        if (!SAFE && i == c + 1) vv = v[0][i] * v[0][i];
      }
    }
  }
  if (!SAFE && !ok) return false;
#pragma unroll
  for (int q = 0; q < SL; ++q) {
    const int r = c0 + lane + 32 * q;
#pragma unroll
    for (int c = 1; c < kLB; ++c)
      if (r < n && (FULL || c < cn) && c0 + c < r) A[r * ld + c0 + c] = v[q][c];
  }
  if (lane < cn) A[(c0 + lane) * ld + c0 + lane] = dg;
  if (SAFE && lane == 0 && first && *bad == 0) *bad = first;
  return true;
}
template <int SL>
__device__ __noinline__ void ldl_block_safe(double* A, double* M, int ld, int n, int c0, int cn, int* bad, int lane) {
  ldl_block_t<SL, false, true>(A, M, ld, n, c0, cn, bad, lane);
}
__device__ __forceinline__ void ldl_block(double* A, double* M, int ld, int n, int c0, int cn, int* bad, int lane) {
  if (n <= kWarpMaxN) {
    ldl_block_safe<1>(A, M, ld, n, c0, cn, bad, lane);
    return;
  }
  const bool done = cn < kLB      ? ldl_block_t<1, false, false>(A, M, ld, n, c0, cn, bad, lane)
                    : n - c0 > 32 ? ldl_block_t<2, true, false>(A, M, ld, n, c0, cn, bad, lane)
                                  : ldl_block_t<1, true, false>(A, M, ld, n, c0, cn, bad, lane);
  if (!done) ldl_block_safe<2>(A, M, ld, n, c0, cn, bad, lane);
}

// Columns [c0, c0 + cn) of the panel rows [r0, r1): u_i = z_i - sum_{c < i} u_c
// m_ic, c in order: one row per thread, or eight lanes per row (a lane per
// column: 7 shuffle and FMA steps instead of 28 FMAs) where that fits the
// group at once. The same operations per element.
__device__ __forceinline__ void ldl_rows(double* Z, int ldz, int r0, int r1, const double* M, int ld, int c0, int cn,
                                         Grp G) {
  if (8 * (r1 - r0) <= G.nt) {
    if ((G.tid & ~31) < 8 * (r1 - r0)) {  // whole warps
      const int sub = G.tid & 7, r = min(r0 + (G.tid >> 3), r1 - 1);
      const bool on = sub < cn && r0 + (G.tid >> 3) < r1;
      double u = on ? Z[r * ldz + c0 + sub] : 0.0;
      for (int c = 0; c + 1 < cn; ++c) {
        const double uc = __shfl_sync(0xffffffffu, u, c, 8);
        const double mi = on && sub > c ? M[(c0 + sub) * ld + c0 + c] : 0.0;
        const double w = fma(-uc, mi, u);
        if (sub > c) u = w;
      }
      if (on) Z[r * ldz + c0 + sub] = u;
    }
    return;
  }
  for (int r = r0 + G.tid; r < r1; r += G.nt) {
    double* z = Z + r * ldz + c0;
    double u[kLB];
#pragma unroll
    for (int c = 0; c < kLB; ++c) u[c] = c < cn ? z[c] : 0.0;
#pragma unroll
    for (int c = 0; c < kLB - 1; ++c) {
      if (c + 1 < cn) {
#pragma unroll
        for (int i = c + 1; i < kLB; ++i)
          if (i < cn) u[i] = fma(-u[c], M[(c0 + i) * ld + c0 + c], u[i]);
      }
    }
#pragma unroll
    for (int c = 1; c < kLB; ++c)
      if (c < cn) z[c] = u[c];
  }
}

// Panel rows [r0, r1) behind the solved block [c0, c0 + kLB): Z[r][c] -= u_r
// m_c^T for c >= c0 + kLB, in column order; by group G, which synchronizes before
// (u) and after.
__device__ __forceinline__ void ldl_panel_update(double* Z, int ldz, int n, int r0, int r1, const double* M, int ld,
                                                 int c0, Grp G) {
  const int cb = c0 + kLB, w = n - cb;
  const Div by(w);
  for (int e = G.tid; e < (r1 - r0) * w; e += G.nt) {
    const int q = by(e), c = cb + e - q * w;
    double* const z = Z + (r0 + q) * ldz;
    const double* const mc = M + c * ld + c0;
    double x = z[c];
#pragma unroll
    for (int k = 0; k < kLB; ++k) x = fma(-z[c0 + k], mc[k], x);
    z[c] = x;
  }
}

// element (a, b) of the pivot block behind block [c0, c0 + kLB)
__device__ __forceinline__ void ldl_trail(double* A, const double* M, int ld, int c0, int a, int b) {
  const double *va = A + a * ld + c0, *mb = M + b * ld + c0;
  double x = A[a * ld + b];
#pragma unroll
  for (int k = 0; k < kLB; ++k) x = fma(-va[k], mb[k], x);
  A[a * ld + b] = x;
}

// Pivot factorization of A and panel solve Z[r0, r1) <- Z L^{-T} diag(L) by the
// whole CTA (at least two warps). On return A holds v (strict lower part, L_rc
// = v_rc / L_cc) and d on its diagonal, M the panel operand L_rc / L_cc, rinv
// 1 / L_cc and Z the unscaled solution u (x_c = u_c rinv_c). The inputs are
// complete on entry; ends with a block barrier.
__device__ void ldl_sweep(double* A, int ld, int n, double* M, double* rinv, int* bad, double* Z, int ldz, int r0,
                          int r1) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  const Grp W{tid - 32, nt - 32, kBarSweep};
  for (int c0 = 0; c0 < n + kLB; c0 += kLB) {
    const int cn = min(kLB, n - c0), cb = c0 + kLB;
    if (tid < 32) {
      if (cn > 0) ldl_block(A, M, ld, n, c0, cn, bad, lane);
    } else if (c0 > 0) {
      const int p0 = c0 - kLB, pn = min(kLB, n - p0);
      if (W.tid >= W.nt - kLB && p0 + W.tid - (W.nt - kLB) < n) {
        const int c = p0 + W.tid - (W.nt - kLB);
        rinv[c] = pivot_rsqrt(A[c * ld + c]);
      }
      // the pivot block behind block J - 1 from column cb on
      const int h = max(n - cb, 0);
      for (int e = W.tid; e < h * (h + 1) / 2; e += W.nt) {
        int a, b;
        tri_rc(e, a, b);
        ldl_trail(A, M, ld, p0, cb + a, cb + b);
      }
      ldl_rows(Z, ldz, r0, r1, M, ld, p0, pn, W);
      if (cn > 0) {
        gsync(W);
        ldl_panel_update(Z, ldz, n, r0, r1, M, ld, p0, W);
      }
    }
    __syncthreads();
    if (cb < n) {  // the pivot block's next columns
      const int w = min(kLB, n - cb);
      for (int e = tid; e < (n - cb) * kLB; e += nt) {
        const int a = cb + (e >> 3), b = cb + (e & 7);
        if ((e & 7) < w && b <= a) ldl_trail(A, M, ld, c0, a, b);
      }
      __syncthreads();
    }
  }
}

// Panel rows [r0, r1) against a pivot block received as M: the operations of
// ldl_sweep (u, unscaled). By the whole CTA; ends with a block barrier.
__device__ void ldl_panel(double* Z, int ldz, int r0, int r1, const double* M, int ld, int n) {
  const Grp C = cta_grp();
  for (int c0 = 0; c0 < n; c0 += kLB) {
    ldl_rows(Z, ldz, r0, r1, M, ld, c0, min(kLB, n - c0), C);
    __syncthreads();
    if (c0 + kLB < n) {
      ldl_panel_update(Z, ldz, n, r0, r1, M, ld, c0, C);
      __syncthreads();
    }
  }
}

// The solved panel rows [r0, r1): x = u rinv to Pd (row-major, n columns), and in
// digits (n >= kDigMin) into Z with the exponents in rowf; BORDER: the bordered row ry as doubles
// into Z, and to ydst with stride yld. Rows [z0, r0) and [r1, z1) of Pd
// are zeroed. Eight lanes a row; by the whole group, which synchronizes
// before and after.
template <bool BORDER>
__device__ void panel_out(double* Z, int ldz, int r0, int r1, int n, const double* rinv, int* rowf, double* Pd, int z0,
                          int z1, int ry, double* ydst, long long yld, Grp G) {
  const int sub = G.tid & 7, span = r0 + ((r1 - r0 + 3) & ~3);  // (whole warps: four rows each)
  for (int r = r0 + (G.tid >> 3); r < span; r += G.nt >> 3) {
    double* z = Z + min(r, r1 - 1) * ldz;
    double x[kMaxN / 8];
    int em = 0;
#pragma unroll
    for (int q = 0; q < kMaxN / 8; ++q) {
      const int k = sub + 8 * q;
      if (8 * q < n) {  // warp-uniform
        x[q] = k < n ? z[k] * rinv[k] : 0.0;
        em = max(em, oz::mag(oz::dbits(x[q])));
      }
    }
    for (int o = 4; o > 0; o >>= 1) em = max(em, __shfl_xor_sync(0xffffffffu, em, o));
    const int f = n < kDigMin ? oz::kFp64Row : BORDER && r == ry ? 0 : oz::row_exp(em);
    if (r < r1) {
      if (sub == 0) rowf[r] = f;
#pragma unroll
      for (int q = 0; q < kMaxN / 8; ++q) {
        const int k = sub + 8 * q;
        if (k < n) {
          Pd[(size_t)r * n + k] = x[q];
          if (BORDER && r == ry) ydst[(size_t)k * yld] = x[q];
          if (f == oz::kFp64Row || (BORDER && r == ry)) z[k] = x[q];
          else ((oz::u64*)z)[k] = oz::encode(oz::dbits(x[q]), f);
        }
      }
    }
  }
  for (int e = G.tid + z0 * n; e < r0 * n; e += G.nt) Pd[e] = 0.0;
  for (int e = G.tid + r1 * n; e < z1 * n; e += G.nt) Pd[e] = 0.0;
}

// Tensor-core form of the mixed Schur update (whole-CTA layout, eight warps):
// T[a][b] -= (Z Z^T)[a][b] for r0 <= b <= a < pr1, with Z (FP32, ld ldz)
// rounded to TF32 or BF16 and the products accumulated in FP32 by tcgen05
// MMAs (M = 128 rows, N = pr1 rounded up to 16, K = n padded to the
// instruction's 8 or 16), then subtracted from the FP64 accumulator once per
// element, in the element order of syrk_trap. `buf` (shared memory, 16-byte
// aligned) holds the operand, pr1 rows of K, and afterwards the FP32
// products as a packed lower triangle; the tensor core reads 128 rows of
// operand address range from it (rows from pr1 on are arbitrary data inside
// the CTA's shared memory and feed only accumulator rows that are never
// read). `tmem`: the accumulator's tensor-memory address; `bar`: the
// completion mbarrier, waited on with `parity` (its completions so far, mod
// 2); mode 1 = TF32, 2 = BF16. Returns false when the MMAs did not complete
// within the bounded wait (T is then left without the update).
// (out of line: inlined into the stage loop it enlarges the loop's code past
// what the instruction cache holds, and every mixed launch slowed down)
__device__ __noinline__ bool syrk_tc(double* T, int ldt, const float* Z, int ldz, int r0, int pr1, int n,
                                     unsigned char* buf, uint32_t tmem, uint64_t* bar, uint32_t parity, int mode) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const bool bf = mode == 2;
  const int kin = bf ? 16 : 8, epc = bf ? 8 : 4, eb = bf ? 2 : 4;
  const int Kp = (n + kin - 1) / kin * kin;
  const uint32_t LBO = 128, SBO = (uint32_t)(Kp / epc) * 128;
  __syncthreads();  // earlier readers of the buffer (the pivot blocks) are done
  for (int e = tid; e < pr1 * Kp; e += nt) {
    const int r = e / Kp, k = e - r * Kp;
    const float v = k < n ? Z[r * ldz + k] : 0.0f;
    const uint32_t off = (uint32_t)(r >> 3) * SBO + (uint32_t)(k / epc) * LBO + (uint32_t)(r & 7) * 16 +
                         (uint32_t)(k % epc) * eb;
    if (bf) *(__nv_bfloat16*)(buf + off) = __float2bfloat16_rn(v);
    else *(uint32_t*)(buf + off) = tc::to_tf32(v);
  }
  tc::fence_async_smem();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (tid == 0) {
    const int N = (pr1 + 15) & ~15;
    const uint32_t idesc = tc::instr_desc(bf ? 1u : 2u, 128, N);
    const uint32_t a0 = tc::smem_u32(buf);
    for (int ks = 0; ks < Kp / kin; ++ks) {
      const uint64_t d = tc::smem_desc(a0 + (uint32_t)ks * 2 * LBO, LBO, SBO);
      tc::mma(bf, tmem, d, d, idesc, ks > 0);
    }
    tc::commit(bar);
  }
  const bool ok = tc::wait(bar, parity);
  tc::fence_after();
  // products -> packed lower triangle S[a (a + 1) / 2 + b]: warp w reads the
  // TMEM lanes (rows) 32 (w % 4) .. + 31, warps w and w + 4 take alternate
  // 8-column chunks
  float* S = (float*)buf;
  const int warp = tid >> 5, lane = tid & 31, row0 = 32 * (warp & 3);
  if (ok && row0 < pr1 && row0 + 31 >= r0) {
    const int a = row0 + lane;
    for (int c0 = 8 * (warp >> 2); c0 < pr1 && c0 <= row0 + 31; c0 += 16) {
      float v[8];
      tc::ld8(tmem + ((uint32_t)row0 << 16) + (uint32_t)c0, v);
      if (a < pr1 && a >= r0) {
        float* Sa = S + a * (a + 1) / 2;
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (c0 + i >= r0 && c0 + i <= a) Sa[c0 + i] = v[i];
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  if (ok) {
    // the subtraction, enumerated like syrk_trap (a rectangle of width 0
    // beside the triangle of rows and columns [r0, pr1))
    const int h = pr1 - r0, tot = h * (h + 1) / 2;
    int a = r0, b = r0 + tid;
    while (a < pr1 && b > a) { b -= a - r0 + 1; ++a; }
    for (int e = tid; e < tot; e += nt) {
      if (e != tid) {
        b += nt;
        while (b > a) { b -= a - r0 + 1; ++a; }
      }
      T[a * ldt + b] -= (double)S[a * (a + 1) / 2 + b];
    }
  }
  __syncthreads();
  return ok;
}

// Thread-block-cluster primitives (a factor task may run as a pair of CTAs).
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// split-phase hardware barrier over every thread of the cluster; arrive
// releases this thread's earlier writes (local and remote shared memory),
// wait acquires the other CTAs'
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// shared::cluster address of this CTA's shared-memory location p in CTA `rank`
__device__ __forceinline__ unsigned cluster_addr(const void* p, unsigned rank) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(unsigned addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(unsigned addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}

// sum_{p < np} part(p, o) for every output o < nout, by the whole CTA, in a
// fixed order that depends only on (nout, np, group size): `sp` adjacent lanes
// (a power of two, at most 32) per output each add every sp-th partial into
// two accumulators, then a shuffle tree combines the lanes; out(o, sum) is
// called once per output. Many partials (one per segment of every lower
// level) are summed with all FP64 sub-pipes instead of one dependent chain
// per output.
// The partials live in L2 (written by earlier launches); the loads of four
// steps are issued before their adds, which keep the order above, so a lane
// waits for one L2 round trip per four steps instead of one per step.
template <typename Fpart, typename Fout>
__device__ void sum_partials(Grp G, int nout, int np, Fpart part, Fout out) {
  // (the split, and with it the order of the sum, of a whole CTA is that of
  // kFactorThreads threads also where it runs with half of them)
  const int nt = G.nt == kFactorThreads / 2 ? kFactorThreads : G.nt;
  int sp = 1;
  while (sp < 32 && sp * 2 * nout <= nt) sp *= 2;
  const int groups = G.nt / sp, sub = G.tid & (sp - 1);
  for (int o0 = 0; o0 < nout; o0 += groups) {
    const int o = o0 + G.tid / sp;
    double a0 = 0.0, a1 = 0.0;
    if (o < nout) {
      int p = sub;
      for (; p + 7 * sp < np; p += 8 * sp) {
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = part(p + u * sp, o);
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
          a0 += v[u];
          a1 += v[u + 1];
        }
      }
      for (; p + sp < np; p += 2 * sp) {
        a0 += part(p, o);
        a1 += part(p + sp, o);
      }
      if (p < np) a0 += part(p, o);
    }
    double a = a0 + a1;
    for (int s = sp >> 1; s > 0; s >>= 1) a += __shfl_xor_sync(0xffffffffu, a, s);
    if (o < nout && sub == 0) out(o, a);
  }
}

struct SegGeom {
  int f, len, hasW, hasF;
};

__device__ __forceinline__ SegGeom seg_geom(const LevelDesc& d, int k) {
  SegGeom g;
  g.f = d.seg[k];
  g.len = d.seg[k + 1] - d.seg[k] - 1;
  g.hasW = (k >= 1);
  g.hasF = (k < d.P - 1);
  return g;
}

// ---------------------------------------------------------------------------
// Factorization: Algorithm 1 for one segment (parallel phase); the top level
// (P = 1) is the sequential phase on the reduced system and also factors the
// corner R-hat = chol(R + sum of every R~_k partial).
// FP64 tasks: factor_task_fp64. Mixed tasks (FP64 pivots and Schur accumulator,
// FP32 panel, FP32 factor copy written for the correction solves): factor_task.
//
// Roles. The panel rows of a segment with fill-in (k >= 1) fall into two
// groups. The producer runs the chain of Algorithm 1 proper: potrf(D_i), the
// E- and G-rows, and their Schur updates D_{i+1}, G_{i+1}, R~_k. The consumer
// runs the fill-in rows: W_i D-hat_i^{-T} and the updates A~_k, Q~_k^T and
// W_{i+1}, which read the producer's D-hat_i, E-hat_i and G-hat_i but feed
// nothing back into the chain, so the consumer may lag a stage behind. Two
// layouts (`mode`):
//   kWhole  one CTA runs both;
//   kPair   a cluster of two CTAs (levels with few segments): CTA 0 is the
//           producer, CTA 1 the consumer, each on an SM of its own. After its
//           panel solve of stage i the producer stores the pivot factor and
//           the E- and G-rows into buffer i % 2 of the consumer's shared
//           memory and arrives at cluster barrier phase i; the consumer
//           arrives at phase i when it is done with stage i-1 and waits for
//           it before stage i; the producer waits for phase i-1 before it
//           overwrites buffer i % 2 (double buffering). A last phase, after
//           every remote store, ends the task.
// ---------------------------------------------------------------------------
static_assert(kFactorThreads == 256, "the factor roles assume 8 warps per CTA");
constexpr int kWhole = 0, kPair = 2;

// Pairs (i, k) with 1 <= k <= i < n ordered by k descending (packed
// i << 16 | k): the updates by column j are the prefix of length
// (n-1-j)(n-j)/2.
__device__ void pair_table_w(int* tab, int n, int lane) {
  const int np = (n - 1) * n / 2;
  for (int e = lane; e < np; e += 32) {
    int a, b;
    tri_rc(e, a, b);
    const int k = n - 1 - a;
    tab[e] = (k + b) << 16 | k;
  }
  __syncwarp();
}

// In-place lower Cholesky of A (n x n, FP64, n <= kWarpMaxN) by one warp,
// right-looking and square-root-free: column j is m = v / d (kept in row j of the
// upper triangle) and the trailing update v_i m_k over the pair table, with 1/d
// in integer arithmetic (pivot_rcp). The reciprocal roots of all pivots are then
// taken at once, L_ij = v_ij rinv_j, and the panel operand M (null: not
// wanted) is m. Two FP64 instructions per column where a root per column took
// seven: the tasks of small blocks are bound by the FP64 pipe (64 cycles an
// instruction whatever its lanes): 2.98 -> 2.31 ms for the first level of 64
// systems of 8192 stages, n = 6, m = 2. Returns the first bad
// column + 1 (0 if every pivot was positive).
template <typename TZ>
__device__ int potrf_w(double* A, int ld, int n, double* rinv, TZ* M, const int* tab, int lane) {
  int bad = 0;
  for (int j = 0; j < n; ++j) {
    const double d = A[j * ld + j];  // (warp-uniform)
    if (not_positive(d) && bad == 0) bad = j + 1;
    const int i = j + 1 + lane;
    if (pivot_rcp_ok(d)) {
      const double r = pivot_rcp(d);
      if (i < n) A[j * ld + i] = A[i * ld + j] * r;
    } else if (i < n) {
      A[j * ld + i] = not_positive(d) ? __longlong_as_double(0x7ff8000000000000LL) : A[i * ld + j] / d;
    }
    __syncwarp();
    const int cnt = (n - 1 - j) * (n - j) / 2;
    for (int e = lane; e < cnt; e += 32) {
      const int p = tab[e], r = p >> 16, k = p & 0xffff;
      A[r * ld + k] = fma(-A[r * ld + j], A[j * ld + k], A[r * ld + k]);
    }
    __syncwarp();
  }
  if (lane < n) {
    const double d = A[lane * ld + lane], r = pivot_rsqrt(d);
    rinv[lane] = r;
    A[lane * ld + lane] = d * r;
  }
  __syncwarp();
  for (int e = lane; e < (n - 1) * n / 2; e += 32) {
    const int p = tab[e], r = p >> 16, c = (p & 0xffff) - 1;  // (i, k): element (i, k - 1) of the strict lower triangle
    A[r * ld + c] *= rinv[c];
    if (M) M[r * ld + c] = (TZ)A[c * ld + r];
  }
  __syncwarp();
  return bad;
}

// Corner of the top level: R-hat = chol(Rs) on the leading m - mr rows (Rs, ld
// ldR, m x m, in shared memory, already summed); the last mr rows hold
// bordered right-hand sides, which are solved against it instead of pivoted
// (their diagonal is never formed): row r gets (Rs[r][k] - sum_{t<k}
// Rs[r][t] R-hat[k][t]) / R-hat[k][k], the forward solution y_g of the
// corner. Writes R-hat (m x m, upper part zero) and 1/diag. By one warp, G.
__device__ void corner_factor(double* Rs, int ldR, int m, int mr, double* rinv, int* tab, const LevelDesc& d,
                              Info* info, Grp G) {
  const int mk = m - mr;
  pair_table_w(tab, mk, G.tid);
  const int bd = potrf_w<double>(Rs, ldR, mk, rinv, nullptr, tab, G.tid);
  if (G.tid == 0 && bd) record_breakdown(info, d.sys, d.Nnat, d.level);
  // bordered rows: a forward substitution with the corner factor, one row per thread
  for (int r = mk + G.tid; r < m; r += G.nt) {
    double* z = Rs + r * ldR;
    for (int k = 0; k < mk; ++k) {
      double a = z[k];
      for (int t = 0; t < k; ++t) a = fma(-z[t], Rs[k * ldR + t], a);
      z[k] = a * rinv[k];
    }
    for (int k = mk; k < m; ++k) z[k] = 0.0;
  }
  gsync(G);
  store_blk(d.Rhat, Rs, ldR, m, m, false, true, G);
  for (int e = G.tid; e < m; e += G.nt) d.Rri[e] = e < mk ? rinv[e] : 0.0;
}

// Shared-memory view and per-stage bookkeeping of one segment task of
// Algorithm 1: where the stage's blocks live, the loads of its inputs (the
// caller's arrays at level 1, the slots of the level below otherwise), the
// stores of its factor blocks and the next level's slots. Used by the CTA
// kernel (k_factor) and the warp kernel (k_factor_w) alike.
template <typename TZ, int LU>
struct FacCtx {
  static constexpr bool mixed = sizeof(TZ) == 4;
  const LevelDesc* d;
  int n, m, R, ldD, ldZ, ldT, oG, oW, s;
  int ry;  // panel row of a bordered right-hand side (the last arrow row), -1 without one
  size_t nn, mn;
  SegGeom g;
  double *Dfac, *rinv, *T;
  TZ *M, *rinvZ, *Z;
  int* tab;
  const double *Din, *D2, *Ein, *Gin, *G2;

  __device__ FacCtx(const LevelDesc& dd, int seg, unsigned char* sm, const FacLayout& lay, const double* uD,
                    const double* uE, const double* uG) {
    d = &dd;
    n = dd.n; m = dd.m; R = 2 * n + m;
    ldD = odd(n); ldZ = lay.ldZ; ldT = lay.ldT;
    oG = n; oW = n + m;  // panel row offsets
    ry = dd.mr ? oW - 1 : -1;
    g = seg_geom(dd, seg);
    s = g.f - 1;         // separator of this segment (k >= 1)
    nn = (size_t)n * n; mn = (size_t)m * n;
    Dfac = (double*)(sm + lay.oDfac);
    M = (TZ*)(sm + lay.oM);
    rinv = (double*)(sm + lay.oRinv);
    rinvZ = (TZ*)(sm + lay.oRinvZ);
    Z = (TZ*)(sm + lay.oZ);
    T = (double*)(sm + lay.oT);
    tab = (int*)(sm + lay.oTab);
    Din = dd.level == 1 ? uD + dd.offD : dd.Dw;
    D2 = dd.level == 1 ? nullptr : dd.D2w;
    Ein = dd.level == 1 ? uE + dd.offE : dd.Ew;
    Gin = dd.level == 1 ? (m ? uG + dd.offG : nullptr) : dd.Gw;
    G2 = dd.level == 1 ? nullptr : dd.G2w;
  }
  __device__ const double* Dp(const double* b, int j) const { return b ? b + (size_t)j * nn : nullptr; }
  __device__ const double* Gp(const double* b, int j) const { return b ? b + (size_t)j * mn : nullptr; }

  // the pivot block D_j (on levels >= 2 the sum of its two slots) into dst (ld ldD)
  __device__ void load_D(double* dst, int j, Grp G) const {
    load_blk<LU>(dst, ldD, Dp(Din, j), Dp(D2, j), n, n, false, G);
  }

  // the first stage's inputs: pivot block, E- and G-rows and the next D, G
  // (eg); the fill-in rows W_1 = E[s]^T, A_k and Q_k^T (wr)
  __device__ void load_first(bool eg, bool wr, Grp G) const {
    const double* none = nullptr;
    if (eg) {
      load_blk<LU>(Dfac, ldD, Dp(Din, g.f), Dp(D2, g.f), n, n, false, G);
      if (g.len > 1 || g.hasF) load_blk<LU>(Z, ldZ, Dp(Ein, g.f), none, n, n, false, G);
      if (m) load_blk<LU>(Z + oG * ldZ, ldZ, Gp(Gin, g.f), Gp(G2, g.f), m, n, false, G);
      if (g.len > 1) {
        load_blk<LU>(T, ldT, Dp(Din, g.f + 1), Dp(D2, g.f + 1), n, n, false, G);          // D_{2}
        if (m) load_blk<LU>(T + oG * ldT, ldT, Gp(Gin, g.f + 1), Gp(G2, g.f + 1), m, n, false, G);
      }
    }
    if (wr) {
      load_blk<LU>(Z + oW * ldZ, ldZ, Dp(Ein, s), none, n, n, true, G);                 // W_1 = B_k = E[s]^T
      load_blk<LU>(T + oW * ldT + oW, ldT, Dp(Din, s), Dp(D2, s), n, n, false, G);       // A_k
      if (m) load_blk<LU>(T + oW * ldT + oG, ldT, Gp(Gin, s), Gp(G2, s), n, m, true, G);  // Q_k^T
    }
  }

  // factor blocks of stage j from the pivot factor L (Dp_, ld ldD) and
  // rv = 1/diag: Ld = L, LdR = L with its rows divided by their diagonal
  // (backward substitution, row-major), LdM = L with its columns divided by
  // their diagonal (forward substitution: the panel operand Ms when given,
  // else formed here with the same rounding), stored transposed so that
  // column c of L is the contiguous row c of LdM, Lri = rv. Strict lower
  // triangles are computed (no FP64 multiply for an upper half), the
  // diagonals of LdR and LdM hold rv (a substitution reads the reciprocal
  // from the block it streams in) and the rest is zero.
  __device__ void store_pivot(int j, const double* Dp_, const double* rv, const TZ* Ms, Grp G) const {
    store_blk(d->Ld + (size_t)j * nn, Dp_, ldD, n, n, false, true, G);
    TZ* LdRj = mixed ? (TZ*)(d->LdRf + (size_t)j * nn) : (TZ*)(d->LdR + (size_t)j * nn);
    TZ* LdMj = mixed ? (TZ*)(d->LdMf + (size_t)j * nn) : (TZ*)(d->LdM + (size_t)j * nn);
    for (int e = G.tid; e < n * n; e += G.nt) LdRj[e] = TZ(0);
    if (Ms) store_blk(LdMj, Ms, ldD, n, n, true, true, G);
    else
      for (int e = G.tid; e < n * n; e += G.nt) LdMj[e] = TZ(0);
    gsync(G);
    for (int e = G.tid; e < (n - 1) * n / 2; e += G.nt) {
      int a, b;
      tri_rc(e, a, b);
      const int r = a + 1, c = b;
      LdRj[r * n + c] = (TZ)(Dp_[r * ldD + c] * rv[r]);
      if (!Ms) LdMj[c * n + r] = (TZ)(Dp_[r * ldD + c] * rv[c]);
    }
    for (int e = G.tid; e < n; e += G.nt) {
      LdRj[e * n + e] = (TZ)rv[e];
      LdMj[e * n + e] = (TZ)rv[e];
    }
    if (mixed)
      for (int e = G.tid; e < n; e += G.nt) d->Lrif[(size_t)j * n + e] = (float)rv[e];
    for (int e = G.tid; e < n; e += G.nt) d->Lri[(size_t)j * n + e] = rv[e];
  }

  // bordered pass: the last arrow row of the solved panel is y_j^T (the
  // forward substitution of stage j), written where the solve keeps it
  // (the caller's b at level 1, this level's X otherwise)
  __device__ void store_y(int j, double* b, int ldb, Grp G) const {
    const TZ* yr = Z + (oG + m - d->mr) * ldZ;
    double* dst;
    long long ld;
    if (d->level == 1) { dst = b + (size_t)(d->offB + (long long)j * n) * ldb; ld = ldb; }
    else { dst = d->X + (size_t)j * n * kRhsChunk; ld = kRhsChunk; }
    for (int e = G.tid; e < n; e += G.nt) dst[(size_t)e * ld] = (double)yr[e];
  }

  // where y_j of a bordered pass goes (stride ld; null without one), as store_y
  __device__ double* y_dst(int j, double* b, int ldb, long long& ld) const {
    if (!d->mr) return nullptr;
    if (d->level == 1) { ld = ldb; return b + (size_t)(d->offB + (long long)j * n) * ldb; }
    ld = kRhsChunk;
    return d->X + (size_t)j * n * kRhsChunk;
  }

  // store_pivot from the square-root-free form: A holds v (L_rc = v_rc rv_c) and
  // d on its diagonal, Mp the panel operand L_rc / L_cc
  __device__ void store_pivot_ldl(int j, const double* A, const double* Mp, const double* rv, Grp G) const {
    double *Ldj = d->Ld + (size_t)j * nn, *LdRj = d->LdR + (size_t)j * nn, *LdMj = d->LdM + (size_t)j * nn;
    const Div by(n);
    for (int e = G.tid; e < n * n; e += G.nt) {
      const int r = by(e), c = e - r * n;
      if (c > r) {
        Ldj[e] = 0.0;
        LdRj[e] = 0.0;
      }
      // (LdM is stored transposed: element e is (c, r))
      LdMj[e] = c > r ? Mp[c * ldD + r] : c == r ? rv[r] : 0.0;
    }
    for (int e = G.tid; e < n * (n + 1) / 2; e += G.nt) {
      int r, c;
      tri_rc(e, r, c);
      const double l = A[r * ldD + c] * rv[c], lr = l * rv[r];
      Ldj[r * n + c] = l;
      LdRj[r * n + c] = r == c ? rv[r] : lr;
    }
    for (int e = G.tid; e < n; e += G.nt) d->Lri[(size_t)j * n + e] = rv[e];
  }

  // panel rows [0, rows) of Lp for stage j: rows outside [r0, r1) are zero
  // (a consumer writes the W-rows of a split or paired segment)
  __device__ void store_panel(int j, int r0, int r1, int rows, Grp G) const {
    double* Pd = d->Lp + (size_t)j * R * n;
    float* Pf = mixed ? d->Lpf + (size_t)j * R * n : nullptr;
    const Div by(n);
    for (int e = G.tid; e < rows * n; e += G.nt) {
      const int r = by(e), c = e - r * n;
      const TZ v = (r >= r0 && r < r1) ? Z[r * ldZ + c] : TZ(0);
      Pd[e] = (double)v;
      if (mixed) Pf[e] = (float)v;
    }
  }

  // rotate the panel after the Schur update of stage i: the updated blocks
  // become stage i+1's inputs, the next ones are loaded
  __device__ void rotate(int i, int j, bool withW, Grp G) const {
    const double* none = nullptr;
    if (m) copy_blk(Z + oG * ldZ, ldZ, T + oG * ldT, ldT, m, n, G);          // G_{i+1}
    if (withW) copy_blk(Z + oW * ldZ, ldZ, T + oW * ldT, ldT, n, n, G);      // W_{i+1}
    if ((i + 1 < g.len - 1) || g.hasF) load_blk<LU>(Z, ldZ, Dp(Ein, j + 1), none, n, n, false, G);
    gsync(G);
    if (withW) load_blk<LU>(T + oW * ldT, ldT, none, none, n, n, false, G);     // W_{i+2} <- 0
    if (i + 2 < g.len) {
      load_blk<LU>(T, ldT, Dp(Din, j + 2), Dp(D2, j + 2), n, n, false, G);
      if (m) load_blk<LU>(T + oG * ldT, ldT, Gp(Gin, j + 2), Gp(G2, j + 2), m, n, false, G);
    } else {
      load_blk<LU>(T, ldT, none, none, n, n, false, G);
      if (m) load_blk<LU>(T + oG * ldT, ldT, none, none, m, n, false, G);
    }
    gsync(G);
  }

  // rotate for the FP64 CTA tasks, with D_{i+1} to Dfac: the loads of stage i+1's
  // E and of D and G of stage i+2 go out first, up to ten per thread, and their
  // latency passes during the copies within shared memory
  __device__ void rotate_cta(int i, int j, bool withW, Grp G) const {
    const bool e1 = (i + 1 < g.len - 1) || g.hasF, d2 = i + 2 < g.len;
    const double *pE = e1 ? Dp(Ein, j + 1) : nullptr, *pD = d2 ? Dp(Din, j + 2) : nullptr,
                 *qD = d2 ? Dp(D2, j + 2) : nullptr, *pG = d2 && m ? Gp(Gin, j + 2) : nullptr,
                 *qG = d2 && m ? Gp(G2, j + 2) : nullptr;
    constexpr int U = 4;
    double ve[U], vd[U], vg;
    auto at = [&](const double* p, const double* q, int e, int tot) {
      return p && e < tot ? (q ? p[e] + q[e] : p[e]) : 0.0;
    };
#pragma unroll
    for (int u = 0; u < U; ++u) {
      ve[u] = at(pE, nullptr, G.tid + u * G.nt, n * n);
      vd[u] = at(pD, qD, G.tid + u * G.nt, n * n);
    }
    vg = at(pG, qG, G.tid, m * n);
    copy_blk(Dfac, ldD, T, ldT, n, n, G);                                 // D_{i+1}
    if (m) copy_blk(Z + oG * ldZ, ldZ, T + oG * ldT, ldT, m, n, G);      // G_{i+1}
    if (withW) copy_blk(Z + oW * ldZ, ldZ, T + oW * ldT, ldT, n, n, G);  // W_{i+1}
    const Div by(n);
    if (e1) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = G.tid + u * G.nt, r = by(e);
        if (e < n * n) Z[r * ldZ + e - r * n] = (TZ)ve[u];
      }
      for (int e = G.tid + U * G.nt; e < n * n; e += G.nt) Z[by(e) * ldZ + e - by(e) * n] = (TZ)pE[e];
    }
    gsync(G);
    if (withW) load_blk<1>(T + oW * ldT, ldT, (const double*)nullptr, (const double*)nullptr, n, n, false, G);  // W_{i+2} <- 0
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = G.tid + u * G.nt, r = by(e);
      if (e < n * n) T[r * ldT + e - r * n] = vd[u];
    }
    for (int e = G.tid + U * G.nt; e < n * n; e += G.nt) T[by(e) * ldT + e - by(e) * n] = at(pD, qD, e, n * n);
    for (int e = G.tid; e < m * n; e += G.nt) {
      const int r = by(e);
      T[(oG + r) * ldT + e - r * n] = e < G.nt ? vg : at(pG, qG, e, m * n);
    }
    gsync(G);
  }

  // stages j+1's E and j+2's D and G towards L2 (rotate_cta reads them at the end
  // of the current stage)
  __device__ void prefetch_next(int i, int j, Grp G) const {
    auto pull = [&](const double* p, int cnt) {
      if (p)
        for (int e = 16 * G.tid; e < cnt; e += 16 * G.nt) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + e));
    };
    if (i + 1 >= g.len) return;
    if ((i + 1 < g.len - 1) || g.hasF) pull(Dp(Ein, j + 1), n * n);
    if (i + 2 < g.len) {
      pull(Dp(Din, j + 2), n * n);
      if (m) pull(Gp(Gin, j + 2), m * n);
    }
  }

  // the next level's slots of segment k (not on the top level)
  __device__ void store_slots(int k, bool eg, bool wr, Grp G) const {
    if (eg && g.hasF) {
      store_blk(d->DB + (size_t)k * nn, T, ldT, n, n, false, true, G);             // -F^ F^T
      if (m) store_blk(d->GB + (size_t)k * mn, T + oG * ldT, ldT, m, n, false, false, G);  // -G^ F^T
    }
    if (wr) {
      store_blk(d->DA + (size_t)(k - 1) * nn, T + oW * ldT + oW, ldT, n, n, false, true, G);  // A~_k
      if (m) store_blk(d->GA + (size_t)(k - 1) * mn, T + oW * ldT + oG, ldT, n, m, true, false, G);  // Q~_k
      if (g.hasF) store_blk(d->EN + (size_t)(k - 1) * nn, T + oW * ldT, ldT, n, n, true, false, G);  // H~_k
    }
    if (eg && m) store_blk(d->Rpart + (size_t)k * m * m, T + oG * ldT + oG, ldT, m, m, false, true, G);
  }
};

// Forward substitution task of the solve kernels (defined below); the factor
// kernel of a bordered pass runs it for the top level (corner solve and the
// backward sweep of the top level) right after the corner.
// KIND: how the tasks share the chip.
constexpr int kAlone = 0;  // a CTA each, at most two on an SM: registers for the loads ahead
constexpr int kWarp = 1;   // a warp each (small blocks)
constexpr int kDense = 2;  // a CTA each, several on an SM hide the latency for one another
template <typename TS, int KIND = kAlone>
__device__ void forward_task(const Task tk, const LevelDesc* __restrict__ descs, double* b, int ldb, int nr,
                             const int* skip, unsigned char* smraw, Grp G, int fwd_done, int c0 = 0);

// One FP64 segment task by the whole CTA or, with `pair`, by this CTA's half
// of a two-CTA cluster: the body of k_factor_fp64, also run task after task by
// the persistent kernel. In a pair CTA 0 runs the chain (pivot, E- and
// G-rows), CTA 1 the fill-in rows one stage behind with the panel operand and
// the E- and G-rows received through distributed shared memory (buffer i % 2);
// see the roles above. Every element is computed by the same operations
// whatever the layout.
template <bool BORDER>
__device__ __forceinline__ void factor_task_fp64(const Task tk, const LevelDesc* __restrict__ descs,
                                               const double* __restrict__ uD, const double* __restrict__ uE,
                                               const double* __restrict__ uG, const double* __restrict__ uR,
                                               Info* info, int pair, double* yb, int ldyb, int top_solve,
                                               unsigned char* smraw, int& bad) {
  const unsigned rank = pair ? cluster_rank() : 0u;
  const LevelDesc& d = descs[tk.desc];
  const FacLayout lay = cta_layout(d.n, d.m, d.P > 1);
  if (!task_geometry_ok(d, tk.seg, smraw, lay.total)) return;  // debug build only (both CTAs of a pair alike)
  const FacCtx<double, 4> cx(d, tk.seg, smraw, lay, uD, uE, uG);
  const int n = cx.n, m = cx.m, R = cx.R, ldD = cx.ldD, ldZ = cx.ldZ, ldT = cx.ldT, oG = cx.oG, oW = cx.oW;
  double* const Dfac = cx.Dfac;
  double* const rinv = cx.rinv;
  double* const T = cx.T;
  double* const Z = cx.Z;
  double* const M = cx.M;
  const SegGeom g = cx.g;
  // the consumer's buffer 1 reuses the pivot block, rinv and the first rows of
  // T, which a consumer CTA has no other use for
  auto Mbuf = [&](int b) { return b ? Dfac : M; };
  auto rinvbuf = [&](int b) { return b ? rinv : cx.rinvZ; };
  auto Zbuf = [&](int b) { return b ? T : Z; };
  auto fbuf = [&](int b) { return (int*)(smraw + lay.oF[b]); };  // exponents of the solved rows
  int* const rowf = fbuf(0);
  const bool eg = !pair || rank == 0;             // this CTA holds the E/G rows
  const bool wr = g.hasW && (!pair || rank == 1);  // this CTA holds the W rows
  const Grp C = cta_grp();
  if (threadIdx.x == 0) bad = 0;
  for (int e = threadIdx.x; e < lay.Rs * ldT; e += blockDim.x) T[e] = 0.0;
  __syncthreads();
  cx.load_first(eg, wr, C);
  __syncthreads();
  if (pair) {
    // both CTAs have started before any remote store
    cluster_arrive();
    cluster_wait();
  }
  if (eg) {
    const int pr1 = n + m + (wr ? n : 0);  // end of the CTA's panel rows
    const bool push = pair && g.hasW;
    for (int i = 0; i < g.len; ++i) {
      const int j = g.f + i;
      const bool eRows = (i < g.len - 1) || g.hasF;
      const int r0 = eRows ? 0 : n;
      if (d.level == 1) cx.prefetch_next(i, j, C);
      ldl_sweep(Dfac, ldD, n, M, rinv, &bad, Z, ldZ, r0, pr1);
      if (threadIdx.x == 0 && bad) { record_breakdown(info, d.sys, d.nat[j], d.level); bad = 0; }
      long long yld = 1;
      double* const yd = cx.y_dst(j, yb, ldyb, yld);
      double* const Pd = d.Lp + (size_t)j * R * n;
      panel_out<BORDER>(Z, ldZ, r0, pr1, n, rinv, rowf, Pd, 0, pair ? n + m : R, cx.ry, yd, yld, C);
      __syncthreads();
      if (push) {
        if (i > 0) cluster_wait();  // the consumer is done with stage i-2 (buffer i % 2)
        const int b = i & 1;
        const unsigned aM = cluster_addr(Mbuf(b), 1), aR = cluster_addr(rinvbuf(b), 1), aF = cluster_addr(fbuf(b), 1),
                       aZ = cluster_addr(Zbuf(b), 1);
        for (int e = C.tid; e < (n - 1) * n / 2; e += C.nt) {
          int a, c;
          tri_rc(e, a, c);
          const int off = (a + 1) * ldD + c;
          st_cluster(aM + off * 8u, M[off]);
        }
        for (int e = C.tid; e < n; e += C.nt) st_cluster(aR + e * 8u, rinv[e]);
        for (int e = r0 + C.tid; e < n + m; e += C.nt) st_cluster(aF + e * 4u, __int_as_float(rowf[e]));
        for (int e = C.tid; e < (n + m - r0) * n; e += C.nt) {
          const int r = r0 + e / n, c = e - (r - r0) * n;
          st_cluster(aZ + (r * ldZ + c) * 8u, Z[r * ldZ + c]);
        }
        cluster_arrive();
      }
      cx.store_pivot_ldl(j, Dfac, M, rinv, C);
      oz_syrk<BORDER>(T, ldT, Z, rowf, Z, rowf, 0, ldZ, r0, pr1, r0, n, cx.ry, Pd, C);
      if (i + 1 < g.len) cx.rotate_cta(i, j, wr, C);
    }
    if (push) cluster_wait();  // phase of the last stage
  } else if (wr) {
    // fill-in rows W of a pair
    for (int i = 0; i < g.len; ++i) {
      const int j = g.f + i;
      const bool eRows = (i < g.len - 1) || g.hasF;
      const int r0 = eRows ? 0 : n, b = i & 1;
      cluster_arrive();  // done with stage i-1
      cluster_wait();    // stage i's blocks are in buffer b
      ldl_panel(Z, ldZ, oW, R, Mbuf(b), ldD, n);
      // (the W-rows' exponents live in buffer 0's array, of which the producer
      // writes the rows below oW only)
      double* const Pd = d.Lp + (size_t)j * R * n;
      panel_out<false>(Z, ldZ, oW, R, n, rinvbuf(b), rowf, Pd, oW, R, -1, nullptr, 1, C);
      __syncthreads();
      oz_syrk<BORDER>(T, ldT, Zbuf(b), fbuf(b), Z, rowf, oW, ldZ, oW, R, r0, n, cx.ry, Pd, C);
      if (i + 1 < g.len) {
        copy_blk(Z + oW * ldZ, ldZ, T + oW * ldT, ldT, n, n, C);  // W_{i+1}
        gsync(C);
        load_blk(T + oW * ldT, ldT, (const double*)nullptr, (const double*)nullptr, n, n, false, C);  // W_{i+2} <- 0
        gsync(C);
      }
    }
  }
  __syncthreads();

  if (!d.is_top) {
    cx.store_slots(tk.seg, eg, wr, C);
  } else if (m) {
    // corner: R-hat = chol(R + sum_k R~_k over every level), in a fixed order:
    // the lower levels' partials are summed by the pair's idle CTA while this
    // one runs the stages (or here, without a pair), then R and this level's
    // own partial are added
    double* Psum = (double*)(smraw + lay.oCorner);
    auto part = [&](int p, int o) { return d.Rpart_all[(size_t)p * m * m + o]; };
    if (pair && rank == 1) {
      const unsigned aP = cluster_addr(Psum, 0);
      sum_partials(C, m * m, d.nRpart_all, part,
                   [&](int o, double v) { st_cluster(aP + o * (unsigned)sizeof(double), v); });
    } else if (!pair) {
      sum_partials(C, m * m, d.nRpart_all, part, [&](int o, double v) { Psum[o] = v; });
    }
    if (pair) {
      cluster_arrive();
      cluster_wait();
    } else {
      __syncthreads();
    }
  }
  if (d.is_top && eg && m) {
    double* Psum = (double*)(smraw + lay.oCorner);
    double* Rs = Dfac;  // reuse
    const int ldR = odd(m);
    const double* Ru = uR + d.offR;
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
      const int r = e / m, c = e - r * m;
      Rs[r * ldR + c] = (Ru[e] + Psum[e]) + T[(oG + r) * ldT + oG + c];
    }
    __syncthreads();
    // by one warp: at m <= 16 a per-column block barrier costs more than the
    // column's work
    if (threadIdx.x < 32)
      corner_factor(Rs, ldR, m, d.mr, rinv, cx.tab, d, info, Grp{(int)threadIdx.x, 32, -1});
    __syncthreads();
  }
  // bordered pass, top level: the corner solve x_g = R-hat^{-T} y_g and the
  // backward sweep of the top level's stages (Algorithm 3, sequential phase)
  // here instead of in a launch of their own; the blocks it reads were
  // written by this CTA, and the shared memory is free by now
  if constexpr (BORDER) {
    if (top_solve && d.is_top && d.mr && yb && eg) {
      __syncthreads();
      forward_task<double>(tk, descs, yb, ldyb, 1, nullptr, smraw, C, 1);
    }
  }
  if (pair) {
    // a segment without fill-in leaves its consumer idle; every CTA of the
    // pair then meets once more, after which no remote store is in flight
    cluster_arrive();
    cluster_wait();
  }
}

// Two CTAs of 256 threads per SM: up to 128 registers (the products' fragments).
// BORDER: bordered descriptors (kkt_factor_solve); the others carry none of that code.
template <bool BORDER>
__global__ void __launch_bounds__(kFactorThreads, 2) k_factor_fp64(const LevelDesc* __restrict__ descs,
                                                                 const Task* __restrict__ tasks,
                                                                 const double* __restrict__ uD,
                                                                 const double* __restrict__ uE,
                                                                 const double* __restrict__ uG,
                                                                 const double* __restrict__ uR, Info* info, int pair,
                                                                 double* yb, int ldyb, int top_solve) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int bad;
  factor_task_fp64<BORDER>(tasks[pair ? blockIdx.x >> 1 : blockIdx.x], descs, uD, uE, uG, uR, info, pair, yb, ldyb, top_solve,
                   smraw, bad);
}

// One segment task of the mixed factorization by the whole CTA (or, with `pair`,
// by this CTA's half of a two-CTA cluster): the body of k_factor, also run
// task after task by the persistent kernel. `bad`, `tslot`, `tbar`: shared
// variables of the caller (breakdown flag, TMEM address slot, mbarrier).
template <bool TC>
__device__ __forceinline__ void factor_task(const Task tk, const LevelDesc* __restrict__ descs,
                                            const double* __restrict__ uD, const double* __restrict__ uE,
                                            const double* __restrict__ uG, const double* __restrict__ uR,
                                            Info* info, int pair,
                                            int tcm, unsigned char* smraw, int& bad, uint32_t& tslot,
                                            uint64_t& tbar) {
  const unsigned rank = pair ? cluster_rank() : 0u;
  const LevelDesc& d = descs[tk.desc];
  const FacLayout lay = fac_layout(d.n, d.m, (int)sizeof(float), d.P > 1);
  if (!task_geometry_ok(d, tk.seg, smraw, lay.total)) return;  // debug build only (both CTAs of a pair alike)
  const FacCtx<float, 4> cx(d, tk.seg, smraw, lay, uD, uE, uG);
  const int n = cx.n, m = cx.m, R = cx.R, ldD = cx.ldD, ldZ = cx.ldZ, ldT = cx.ldT, oG = cx.oG, oW = cx.oW;
  double* const Dfac = cx.Dfac;
  double* const rinv = cx.rinv;
  double* const T = cx.T;
  float* const M = cx.M;
  float* const rinvZ = cx.rinvZ;
  float* const Z = cx.Z;
  int* const tab = cx.tab;
  const SegGeom g = cx.g;
  const int mode = pair ? kPair : kWhole;
  // consumer buffers of the pair layout: buffer 0 is (M, rinvZ, Z rows [0, n+m)),
  // buffer 1 reuses the pivot block, rinv and the first rows of T, which a
  // consumer CTA has no other use for
  auto Mbuf = [&](int b) { return b ? (float*)Dfac : M; };
  auto rinvbuf = [&](int b) { return b ? (float*)rinv : rinvZ; };
  auto Zbuf = [&](int b) { return b ? (float*)T : Z; };
  const bool eg = mode != kPair || rank == 0;       // this CTA holds the E/G rows
  const bool wr = g.hasW && (mode != kPair || rank == 1);  // this CTA holds the W rows

  // tensor-core Schur products (mixed whole-CTA layout; the pivot buffers'
  // region stages the operands)
  const bool use_tc = TC && tcm && mode == kWhole;
  const uint32_t tc_cols = ((lay.Rs + 15) & ~15) <= 64 ? 64u : 128u;
  uint32_t tmem = 0u, tphase = 0u;
  if constexpr (TC) {
    if (use_tc) {
      if (threadIdx.x < 32) tc::alloc(&tslot, tc_cols);
      if (threadIdx.x == 0) tc::mbar_init(&tbar);
      tc::fence_before();
    }
  }
  if (threadIdx.x == 0) bad = 0;
  for (int e = threadIdx.x; e < lay.Rs * ldT; e += blockDim.x) T[e] = 0.0;
  if (eg) potrf_table(tab, n);
  __syncthreads();
  if constexpr (TC) {
    if (use_tc) {
      tc::fence_after();
      tmem = tslot;
    }
  }
  cx.load_first(eg, wr, cta_grp());
  __syncthreads();
  if (mode == kPair) {
    // both CTAs have started before any remote store
    cluster_arrive();
    cluster_wait();
  }

  const bool producer = mode == kWhole || rank == 0;
  auto store_pivot = [&](int j, const double* Dp_, const double* rv, const float* Ms, Grp G) {
    cx.store_pivot(j, Dp_, rv, Ms, G);
  };
  auto store_panel = [&](int j, int r0, int r1, int rows, Grp G) { cx.store_panel(j, r0, r1, rows, G); };
  // hand the trsm operand (strict lower triangle of Msrc, ld ldD), its
  // 1/diag and panel rows [r0, r1) of stage i to the consumer CTA of a pair
  auto push_stage = [&](int i, const float* Msrc, const float* rsrc, int r0, int r1, Grp G) {
    const int b = i & 1;
    const unsigned aM = cluster_addr(Mbuf(b), 1), aR = cluster_addr(rinvbuf(b), 1),
                   aZ = cluster_addr(Zbuf(b), 1);
    const int ntri = (n - 1) * n / 2;
    for (int e = G.tid; e < ntri; e += G.nt) {
      int a, c;
      tri_rc(e, a, c);
      const int off = (a + 1) * ldD + c;
      st_cluster(aM + off * (unsigned)sizeof(float), Msrc[off]);
    }
    for (int e = G.tid; e < n; e += G.nt) st_cluster(aR + e * (unsigned)sizeof(float), rsrc[e]);
    for (int e = G.tid; e < (r1 - r0) * n; e += G.nt) {
      const int r = r0 + e / n, c = e - (r - r0) * n;
      const int off = r * ldZ + c;
      st_cluster(aZ + off * (unsigned)sizeof(float), Z[off]);
    }
  };
  auto rotate = [&](int i, int j, bool withW, Grp G) { cx.rotate(i, j, withW, G); };

  if (producer) {
    // Whole CTA on the E- and G-rows (and the W-rows in the whole layout). Per
    // stage: the fused pivot factorization and panel solve, the pivot blocks'
    // store, then the hand-off to the consumer, the Schur update and the rotation.
    const Grp P = cta_grp();
    const int pr1 = n + m + (mode == kWhole && g.hasW ? n : 0);  // end of the CTA's panel rows
    const bool push = mode == kPair && g.hasW;
    for (int i = 0; i < g.len; ++i) {
      const int j = g.f + i;
      const bool eRows = (i < g.len - 1) || g.hasF;
      const int r0 = eRows ? 0 : n;
      potrf_trsm_sm(Dfac, ldD, n, rinv, M, tab, &bad, Z, ldZ, r0, pr1);
      __syncthreads();
      if (threadIdx.x == 0 && bad) { record_breakdown(info, d.sys, d.nat[j], d.level); bad = 0; }
      store_pivot(j, Dfac, rinv, nullptr, P);  // read before the copy of D_{i+1} below
      if (push) {
        for (int e = P.tid; e < n; e += P.nt) rinvZ[e] = (float)rinv[e];
        __syncthreads();
        if (i > 0) cluster_wait();  // the consumer is done with stage i-2 (buffer i % 2)
        push_stage(i, M, rinvZ, r0, n + m, P);
        cluster_arrive();
      }
      store_panel(j, r0, pr1, mode == kWhole ? R : n + m, P);
      bool tc_done = false;
      if constexpr (TC) {
        if (use_tc) {
          if (!syrk_tc(T, ldT, (const float*)Z, ldZ, r0, pr1, n, smraw + lay.oDfac, tmem, &tbar, tphase & 1, tcm) &&
              threadIdx.x == 0)
            record_timeout(info, d.sys, d.nat[j], d.level);
          ++tphase;
          tc_done = true;
        }
      }
      if (!tc_done) syrk_trap(T, ldT, Z, Z, 0, ldZ, r0, pr1, r0, n, P);
      if (i + 1 < g.len) {
        copy_blk(Dfac, ldD, T, ldT, n, n, P);  // D_{i+1}
        rotate(i, j, mode == kWhole && g.hasW, P);
      }
    }
    if (push) cluster_wait();  // phase of the last stage
  } else if (wr) {
    // fill-in rows W
    const Grp C = cta_grp();
    for (int i = 0; i < g.len; ++i) {
      const int j = g.f + i;
      const bool eRows = (i < g.len - 1) || g.hasF;
      const int r0 = eRows ? 0 : n;
      const int b = i & 1;
      cluster_arrive();  // done with stage i-1
      cluster_wait();    // stage i's blocks are in buffer b
      trsm_panel(Z, ldZ, oW, R, Mbuf(b), ldD, n, rinvbuf(b), C);
      {
        double* Pd = d.Lp + (size_t)j * R * n + (size_t)oW * n;
        float* Pf = d.Lpf + (size_t)j * R * n + (size_t)oW * n;
        for (int e = C.tid; e < n * n; e += C.nt) {
          const int r = e / n, c = e - r * n;
          const float v = Z[(oW + r) * ldZ + c];
          Pd[e] = (double)v;
          Pf[e] = v;
        }
      }
      syrk_trap(T, ldT, Zbuf(b), Z, oW, ldZ, oW, R, r0, n, C);
      if (i + 1 < g.len) {
        copy_blk(Z + oW * ldZ, ldZ, T + oW * ldT, ldT, n, n, C);               // W_{i+1}
        gsync(C);
        load_blk(T + oW * ldT, ldT, (const double*)nullptr, (const double*)nullptr, n, n, false, C);  // W_{i+2} <- 0
        gsync(C);
      }
    }
  }
  __syncthreads();

  if (!d.is_top) {
    cx.store_slots(tk.seg, eg, wr, cta_grp());
  } else if (m) {
    // corner: R-hat = chol(R + sum_k R~_k over every level), in a fixed order:
    // the lower levels' partials are summed by the pair's idle CTA while this
    // one runs the stages (or here, without a pair), then R and this level's
    // own partial are added
    double* Psum = (double*)(smraw + lay.oCorner);
    auto part = [&](int p, int o) { return d.Rpart_all[(size_t)p * m * m + o]; };
    if (mode == kPair && rank == 1) {
      const unsigned aP = cluster_addr(Psum, 0);
      sum_partials(cta_grp(), m * m, d.nRpart_all, part,
                   [&](int o, double v) { st_cluster(aP + o * (unsigned)sizeof(double), v); });
    } else if (mode != kPair) {
      sum_partials(cta_grp(), m * m, d.nRpart_all, part, [&](int o, double v) { Psum[o] = v; });
    }
    if (mode == kPair) {
      cluster_arrive();
      cluster_wait();
    } else {
      __syncthreads();
    }
  }
  if (d.is_top && eg && m) {
    double* Psum = (double*)(smraw + lay.oCorner);
    double* Rs = Dfac;  // reuse
    const int ldR = odd(m);
    const double* Ru = uR + d.offR;
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
      const int r = e / m, c = e - r * m;
      Rs[r * ldR + c] = (Ru[e] + Psum[e]) + T[(oG + r) * ldT + oG + c];
    }
    __syncthreads();
    // by one warp: at m <= 16 a per-column block barrier costs more than the
    // column's work
    if (threadIdx.x < 32)
      corner_factor(Rs, ldR, m, d.mr, rinv, tab, d, info, Grp{(int)threadIdx.x, 32, -1});
    __syncthreads();
  }
  if (mode == kPair) {
    // a segment without fill-in leaves its consumer idle; every CTA of the
    // pair then meets once more, after which no remote store is in flight
    cluster_arrive();
    cluster_wait();
  }
  if constexpr (TC) {
    if (use_tc) {
      tc::fence_before();
      __syncthreads();
      if (threadIdx.x < 32) tc::dealloc(tmem, tc_cols);
    }
  }
}

// MINB: CTAs per SM the register allocation must allow. Launches of CTA pairs
// (one CTA per SM, latency-bound) take the unconstrained allocation (1);
// the others four (at most 64 registers), so that several segment CTAs share
// an SM when shared memory allows it.
// TC: the instantiation with the tensor-core Schur products (mixed launches
// that use them); the others carry none of that code.
template <int MINB, bool TC = false>
__global__ void __launch_bounds__(kFactorThreads, MINB) k_factor(const LevelDesc* __restrict__ descs,
                                                           const Task* __restrict__ tasks,
                                                           const double* __restrict__ uD,
                                                           const double* __restrict__ uE,
                                                           const double* __restrict__ uG,
                                                           const double* __restrict__ uR,
                                                           Info* info, int pair,
                                                           int tcm) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int bad;
  __shared__ uint32_t tslot;               // TMEM address of the tensor-core accumulator
  __shared__ __align__(8) uint64_t tbar;   // its completion mbarrier
  factor_task<TC>(tasks[pair ? blockIdx.x >> 1 : blockIdx.x], descs, uD, uE, uG, uR, info, pair,
                      tcm, smraw, bad, tslot, tbar);
}

// ---------------------------------------------------------------------------
// One-stage segments on a cluster of C CTAs (2 <= C <= 8), FP64. On the deep
// levels of a recursive plan every segment is a single stage (its pivot
// block with the E-, G- and W-rows of its panel), and the levels have few
// tasks: one or two CTAs per task leave most SMs idle while the stage's
// panel solve and Schur update (Alg. 1) run at two FP64 FMAs per clock per
// SM. Here the stage is spread over the cluster:
//   - every CTA factors the pivot block itself and solves a contiguous band
//     of about 1/C of the panel rows (ldl_sweep),
//     then stores its solved rows into every other CTA's shared memory;
//   - every CTA applies the Schur update to a band of trapezoid rows holding
//     about 1/C of the elements and stores the results into the shared
//     memory of the CTA that writes that block's slots for the next level
//     (rank 0: E- and G-rows, rank 1: W-rows);
//   - the last rank writes the pivot blocks, each CTA its panel rows.
// Three split-phase cluster barriers order the exchanges. Every element is
// computed by the same operations in the same order as in the one- and
// two-CTA layouts, so the results are bitwise theirs.
// ---------------------------------------------------------------------------
template <bool BORDER>
__device__ __forceinline__ void clus_task(const Task tk, const LevelDesc* __restrict__ descs,
                                          const double* __restrict__ uD, const double* __restrict__ uE,
                                          const double* __restrict__ uG, Info* info, double* yb, int ldyb, int C,
                                          unsigned char* smraw, int& bad) {
  const int rank = (int)cluster_rank();
  const LevelDesc& d = descs[tk.desc];
  const FacLayout lay = cta_layout(d.n, d.m);
  if (!task_geometry_ok(d, tk.seg, smraw, lay.total)) return;  // debug build only (every CTA alike)
  const FacCtx<double, 4> cx(d, tk.seg, smraw, lay, uD, uE, uG);
  const int n = cx.n, m = cx.m, ldD = cx.ldD, ldZ = cx.ldZ, ldT = cx.ldT, oG = cx.oG, oW = cx.oW;
  const SegGeom g = cx.g;
  const int j = g.f, s = cx.s, tid = threadIdx.x, nt = blockDim.x;
  double* const Dfac = cx.Dfac;
  double* const rinv = cx.rinv;
  double* const T = cx.T;
  double* const M = cx.M;
  double* const Z = cx.Z;
  int* const rowf = (int*)(smraw + lay.oF[0]);
  // panel rows [r0, r1): the E-rows when a next separator exists, the G-rows,
  // the W-rows when a previous one does
  const int r0 = g.hasF ? 0 : n, r1 = g.hasW ? cx.R : n + m, h = r1 - r0;
  // this CTA's band of the panel solve: equal row counts
  const int t0 = r0 + h * rank / C, t1 = r0 + h * (rank + 1) / C;
  // its band of the Schur update: row r0 + a holds a + 1 elements; band q
  // starts at the first row whose preceding rows hold >= q/C of the total
  const int tot = h * (h + 1) / 2;
  auto band0 = [&](int q) {
    const int want = (tot * q + C - 1) / C;
    int a = 0;
    while (a < h && a * (a + 1) / 2 < want) ++a;
    return r0 + a;
  };
  const int s0 = band0(rank), s1 = band0(rank + 1);
  cluster_arrive();  // this CTA runs: the others may store into its shared memory after their wait
  if (tid == 0) bad = 0;
  // inputs: the pivot block D_j, the panel rows of the solve band, and the
  // initial values of the Schur band (A_k and Q_k^T in its W-rows, zero
  // elsewhere). Every load is an L2 round trip, so the three sets form one
  // list whose loads go out eight per thread before any store: element e
  // of the list is D_j's (e < nD), then the band's panel rows (< nD + nZ),
  // then the W-row part [oG, R) of the Schur band's rows (the rest of those
  // rows is zeroed separately). Sums of two slots add in the order of
  // load_blk, so the values are those of the other layouts.
  {
    const int nD = n * n, nZ = (t1 - t0) * n;
    const int wa0 = max(s0, oW), nTr = max(0, s1 - wa0), nTc = m + n;
    const int nIn = nD + nZ + nTr * nTc;
    const double* const D1 = cx.Din + (size_t)j * cx.nn;
    const double* const D2 = cx.D2 ? cx.D2 + (size_t)j * cx.nn : nullptr;
    constexpr int U = 8;
    for (int e0 = tid; e0 < nIn; e0 += U * nt) {
      double v[U];
      int dst[U];  // offset in doubles from smraw's Dfac (Dfac, Z and T are one allocation)
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = e0 + u * nt;
        dst[u] = -1;
        v[u] = 0.0;
        if (e < nD) {
          const int r = e / n, c = e - r * n;
          v[u] = D2 ? D1[e] + D2[e] : D1[e];
          dst[u] = (int)(&Dfac[r * ldD + c] - Dfac);
        } else if (e < nD + nZ) {
          const int f = e - nD, r = t0 + f / n, c = f - (r - t0) * n;
          if (r < n) v[u] = cx.Ein[(size_t)j * cx.nn + r * n + c];  // E_j
          else if (r < oW) {                                         // G_j (+ its second slot)
            const size_t o = (size_t)j * cx.mn + (r - oG) * n + c;
            v[u] = cx.G2 ? cx.Gin[o] + cx.G2[o] : cx.Gin[o];
          } else v[u] = cx.Ein[(size_t)s * cx.nn + c * n + (r - oW)];  // W_1 = E[s]^T
          dst[u] = (int)(&Z[r * ldZ + c] - Dfac);
        } else if (e < nIn) {
          const int f = e - nD - nZ, a = wa0 + f / nTc, b = oG + (f - (a - wa0) * nTc);
          if (b >= oW) {  // A_k = D_s (+ its second slot)
            const size_t o = (size_t)s * cx.nn + (a - oW) * n + (b - oW);
            v[u] = cx.D2 ? cx.Din[o] + cx.D2[o] : cx.Din[o];
          } else {        // Q_k^T = G_s^T
            const size_t o = (size_t)s * cx.mn + (b - oG) * n + (a - oW);
            v[u] = cx.G2 ? cx.Gin[o] + cx.G2[o] : cx.Gin[o];
          }
          dst[u] = (int)(&T[a * ldT + b] - Dfac);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (dst[u] >= 0) Dfac[dst[u]] = v[u];
    }
    // the rest of the Schur band's rows: zero
    for (int e = tid; e < (s1 - s0) * ldT; e += nt) {
      const int a = s0 + e / ldT, b = e - (a - s0) * ldT;
      if (!(a >= oW && b >= oG && b < cx.R)) T[a * ldT + b] = 0.0;
    }
  }
  __syncthreads();
  ldl_sweep(Dfac, ldD, n, M, rinv, &bad, Z, ldZ, t0, t1);
  // its panel rows to device memory (rank 0 also writes the zero rows [0, r0);
  // the bordered row is y_j of the forward substitution), then in digits to the
  // other CTAs
  double* const Pd = d.Lp + (size_t)j * cx.R * n;
  {
    long long yld = 1;
    double* const yd = cx.y_dst(j, yb, ldyb, yld);
    panel_out<BORDER>(Z, ldZ, t0, t1, n, rinv, rowf, Pd, rank == 0 ? 0 : t0, t1, cx.ry, yd, yld, cta_grp());
  }
  __syncthreads();
  cluster_wait();  // every CTA of the cluster runs
  {
    for (int q = 1; q < C; ++q) {
      const unsigned af = cluster_addr(rowf, (unsigned)((rank + q) % C));
      for (int r = t0 + tid; r < t1; r += nt) st_cluster(af + r * 4u, __int_as_float(rowf[r]));
      const unsigned az = cluster_addr(Z, (unsigned)((rank + q) % C));
      for (int e = tid; e < (t1 - t0) * n; e += nt) {
        const int r = t0 + e / n, c = e - (r - t0) * n;
        const unsigned off = (unsigned)(r * ldZ + c) * 8u;
        st_cluster(az + off, Z[r * ldZ + c]);
      }
    }
  }
  cluster_arrive();
  // the pivot blocks: by the last rank, which stores no slots when C > 2
  if (rank == C - 1) {
    if (tid == 0 && bad) record_breakdown(info, d.sys, d.nat[j], d.level);
    cx.store_pivot_ldl(j, Dfac, M, rinv, cta_grp());
  }
  cluster_wait();  // every solved panel row is here (and in device memory)
  oz_syrk<BORDER>(T, ldT, Z, rowf, Z, rowf, 0, ldZ, s0, s1, r0, n, cx.ry, Pd, cta_grp());
  {
    const unsigned a0 = cluster_addr(T, 0u), a1 = cluster_addr(T, 1u);
    const int w0 = s0 - r0;  // row s0 + i holds w0 + i + 1 elements
    const int cnt = (s1 - s0) * w0 + (s1 - s0) * (s1 - s0 + 1) / 2;
    // (a, b) of element tid of the band, then advanced by nt along the rows
    int a = s0, b = r0 + tid;
    while (a < s1 && b > a) { b -= a - r0 + 1; ++a; }
    for (int e = tid; e < cnt; e += nt) {
      if (e != tid) {
        b += nt;
        while (b > a) { b -= a - r0 + 1; ++a; }
      }
      const int owner = a < oW ? 0 : 1;
      if (owner != rank)
        st_cluster((owner ? a1 : a0) + (unsigned)(a * ldT + b) * 8u, T[a * ldT + b]);
    }
  }
  cluster_arrive();
  cluster_wait();  // the slot owners hold their rows of the update
  if (rank == 0) cx.store_slots(tk.seg, true, false, cta_grp());
  else if (rank == 1) cx.store_slots(tk.seg, false, g.hasW, cta_grp());
}

template <bool BORDER>
__global__ void __launch_bounds__(kFactorThreads, 2) k_factor_clus(const LevelDesc* __restrict__ descs,
                                                                   const Task* __restrict__ tasks,
                                                                   const double* __restrict__ uD,
                                                                   const double* __restrict__ uE,
                                                                   const double* __restrict__ uG, Info* info,
                                                                   double* yb, int ldyb, int C) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int bad;
  clus_task<BORDER>(tasks[blockIdx.x / C], descs, uD, uE, uG, info, yb, ldyb, C, smraw, bad);
}


// ---------------------------------------------------------------------------
// Small blocks (n <= kWarpMaxN): one warp per segment task, every step of a
// stage warp-synchronous, several tasks per CTA with a shared-memory slice
// each. The CTA kernel's role split needs blocks large enough to keep eight
// warps busy; at n = 6 a stage is a few hundred FMAs, and what counts is how
// many independent stage chains an SM interleaves.
// ---------------------------------------------------------------------------

// Z[r0:r1) <- Z[r0:r1) L^{-T} by one warp, one panel row per lane: the
// division-free substitution of trsm_panel, in the same order per element.
template <typename TZ>
__device__ void trsm_w(TZ* Z, int ldz, int r0, int r1, const TZ* M, int ldm, int n, const TZ* rinv, int lane) {
  for (int r = r0 + lane; r < r1; r += 32) {
    TZ* z = Z + r * ldz;
    for (int j = 0; j < n - 1; ++j) {
      const TZ zj = z[j];
      for (int c = j + 1; c < n; ++c) z[c] = fma(-zj, M[c * ldm + j], z[c]);
    }
    for (int c = 0; c < n; ++c) z[c] *= rinv[c];
  }
  __syncwarp();
}

// One small-block segment task by one warp in its shared-memory slice `sm`:
// the body of k_factor_w, also run by the persistent kernel.
template <typename TZ>
__device__ __forceinline__ void factor_task_w(const Task tk, const LevelDesc* __restrict__ descs,
                                              const double* __restrict__ uD, const double* __restrict__ uE,
                                              const double* __restrict__ uG, const double* __restrict__ uR,
                                              Info* info, unsigned char* sm, int lane, double* yb, int ldyb) {
  const LevelDesc& d = descs[tk.desc];
  const FacLayout lay = fac_layout_w(d.n, d.m, (int)sizeof(TZ), d.P > 1);
  if (!task_geometry_ok(d, tk.seg, sm, lay.total)) return;  // debug build only
  const FacCtx<TZ, 1> cx(d, tk.seg, sm, lay, uD, uE, uG);
  const int n = cx.n, m = cx.m, R = cx.R, ldD = cx.ldD, ldZ = cx.ldZ, ldT = cx.ldT, oG = cx.oG;
  const SegGeom g = cx.g;
  const Grp W{lane, 32, -1};
  for (int e = lane; e < lay.Rs * ldT; e += 32) cx.T[e] = 0.0;
  pair_table_w(cx.tab, n, lane);
  cx.load_first(true, g.hasW, W);
  __syncwarp();
  const int pr1 = n + m + (g.hasW ? n : 0);
  for (int i = 0; i < g.len; ++i) {
    const int j = g.f + i;
    const bool eRows = (i < g.len - 1) || g.hasF;
    const int r0 = eRows ? 0 : n;
    const int bad = potrf_w<TZ>(cx.Dfac, ldD, n, cx.rinv, cx.M, cx.tab, lane);
    if (lane == 0 && bad) record_breakdown(info, d.sys, d.nat[j], d.level);
    for (int e = lane; e < n; e += 32) cx.rinvZ[e] = (TZ)cx.rinv[e];
    __syncwarp();
    trsm_w(cx.Z, ldZ, r0, pr1, cx.M, ldD, n, cx.rinvZ, lane);
    if (d.mr) cx.store_y(j, yb, ldyb, W);
    cx.store_pivot(j, cx.Dfac, cx.rinv, cx.M, W);
    cx.store_panel(j, r0, pr1, R, W);
    syrk_trap(cx.T, ldT, cx.Z, cx.Z, 0, ldZ, r0, pr1, r0, n, W);
    if (i + 1 < g.len) {
      copy_blk(cx.Dfac, ldD, cx.T, ldT, n, n, W);                                  // D_{i+1}
      __syncwarp();
      cx.rotate(i, j, g.hasW, W);
    }
  }
  __syncwarp();
  if (!d.is_top) {
    cx.store_slots(tk.seg, true, g.hasW, W);
  } else if (m) {
    // corner: R-hat = chol((R + sum of the lower levels' partials) + this level's)
    double* Rs = cx.Dfac;  // reuse (n >= m is not needed: the slice has room for q x q)
    double* Psum = (double*)(sm + lay.oCorner);
    const int ldR = odd(m);
    for (int o = lane; o < m * m; o += 32) {
      double a0 = 0.0, a1 = 0.0;
      int p = 0;
      for (; p + 1 < d.nRpart_all; p += 2) {
        a0 += d.Rpart_all[(size_t)p * m * m + o];
        a1 += d.Rpart_all[(size_t)(p + 1) * m * m + o];
      }
      if (p < d.nRpart_all) a0 += d.Rpart_all[(size_t)p * m * m + o];
      Psum[o] = a0 + a1;
    }
    __syncwarp();
    const double* Ru = uR + d.offR;
    for (int e = lane; e < m * m; e += 32) {
      const int r = e / m, c = e - r * m;
      Rs[r * ldR + c] = (Ru[e] + Psum[e]) + cx.T[(oG + r) * ldT + oG + c];
    }
    __syncwarp();
    corner_factor(Rs, ldR, m, d.mr, cx.rinv, cx.tab, d, info, W);
  }
}

template <typename TZ>
__global__ void __launch_bounds__(256, 4) k_factor_w(const LevelDesc* __restrict__ descs,
                                                  const Task* __restrict__ tasks, int ntasks,
                                                  const double* __restrict__ uD, const double* __restrict__ uE,
                                                  const double* __restrict__ uG, const double* __restrict__ uR,
                                                  Info* info, int slice, double* yb, int ldyb) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int t = blockIdx.x * (blockDim.x >> 5) + wid;
  if (t >= ntasks) return;  // whole warp
  factor_task_w<TZ>(tasks[t], descs, uD, uE, uG, uR, info, smraw + (size_t)wid * slice, lane, yb, ldyb);
}

// ---------------------------------------------------------------------------
// Persistent factorization: one launch runs every segment task of every level
// (Algorithm 1's parallel phase and, level by level, the reduced systems of
// Eq. (7)). CTAs take work items by ticket (atomicAdd) from a list in
// topological order: level by level, and within a level the most expensive
// first (longest-processing-time order), so long systems start first and the
// short ones fill the tail. An item of level >= 2 reads slots written by its
// feeder tasks one level down; its CTA waits (thread 0, acquire loads with a
// growing sleep, bounded by wait_cycles) until the feeders' release
// increments reach `need`. A CTA only ever waits on items with smaller
// tickets, which CTAs already running hold, so every wait has a producer in
// progress. A wait that runs out records KKT_ERR_TIMEOUT (with the waiting
// task's system, natural stage and level), skips its task and still releases
// its consumers, so nothing waits forever.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void red_release_gpu(int* p) {
  asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p) : "memory");
}
__device__ __forceinline__ int ld_acquire_gpu(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

template <typename TZ>
__global__ void __launch_bounds__(kFactorThreads, sizeof(TZ) == 8 ? 2 : 3)
    k_factor_persist(const LevelDesc* __restrict__ descs, const Task* __restrict__ tasks,
                     const PItem* __restrict__ items, int nitems, const PCons* __restrict__ cons, int* ready,
                     const double* __restrict__ uD, const double* __restrict__ uE, const double* __restrict__ uG,
                     const double* __restrict__ uR, Info* info, int slice, long long wait_cycles) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int bad;
  __shared__ uint32_t tslot;
  __shared__ __align__(8) uint64_t tbar;
  __shared__ int cur, ok;
  int* const ticket = ready + nitems;
  for (;;) {
    if (threadIdx.x == 0) cur = atomicAdd(ticket, 1);
    __syncthreads();
    const int it = cur;
    if (it >= nitems) break;
    const PItem w = items[it];
    if (threadIdx.x == 0) {
      int good = 1;
      if (w.need > 0) {
        const long long t0 = clock64();
        unsigned ns = 64;
        while (ld_acquire_gpu(ready + it) < w.need) {
          if (clock64() - t0 > wait_cycles) {
            good = 0;
            break;
          }
          __nanosleep(ns);
          if (ns < 2048) ns *= 2;
        }
        __threadfence();
      }
      ok = good;
      if (!good) {
        const Task tk = tasks[w.first];
        const LevelDesc& d = descs[tk.desc];
        record_timeout(info, d.sys, d.nat[d.seg[tk.seg]], d.level);
      }
    }
    __syncthreads();
    if (ok) {
      if (!w.warp) {
        if constexpr (sizeof(TZ) == 8)
          factor_task_fp64<false>(tasks[w.first], descs, uD, uE, uG, uR, info, 0, nullptr, 1, 0, smraw, bad);
        else
          factor_task<false>(tasks[w.first], descs, uD, uE, uG, uR, info, 0, 0, smraw, bad, tslot, tbar);
      } else {
        const int wid = threadIdx.x >> 5;
        if (wid < w.cnt)
          factor_task_w<TZ>(tasks[w.first + wid], descs, uD, uE, uG, uR, info, smraw + (size_t)wid * slice,
                            threadIdx.x & 31, nullptr, 1);
      }
    }
    __syncthreads();
    // release: every thread's writes of this item precede the barrier; the
    // fence makes them visible device-wide before the counters move
    if (threadIdx.x == 0) {
      __threadfence();
      for (int c = 0; c < w.ncons; ++c) atomicAdd(ready + cons[w.cons0 + c].item, cons[w.cons0 + c].weight);
    }
  }
}

// ---------------------------------------------------------------------------
// Solve. TS = double: FP64 factor and vectors. TS = float: the FP32 factor
// copy of a mixed level and FP32 vectors (the correction solves of iterative
// refinement). Global vectors are FP64 in both cases.
// ---------------------------------------------------------------------------

// rhs / solution rows of stage j at this level: the caller's b at level 1
// (rows offB + j n, stride ldb), this level's X array otherwise.
struct VecView {
  double* p;
  int ld;
};

__device__ __forceinline__ VecView level_vec(const LevelDesc& d, double* b, int ldb, int j, int c0) {
  VecView v;
  if (d.level == 1) { v.p = b + (size_t)(d.offB + (long long)j * d.n) * ldb; v.ld = ldb; }
  else { v.p = d.X + (size_t)j * d.n * kRhsChunk + c0; v.ld = kRhsChunk; }
  return v;
}

// level_vec of every stage (the descriptor is read once: a level's fields would
// be loaded again behind every store)
struct VecViews {
  double* p;
  size_t step;
  int ld;
  __device__ VecViews(const LevelDesc& d, double* b, int ldb, int c0) {
    const VecView v = level_vec(d, b, ldb, 0, c0);
    p = v.p;
    ld = v.ld;
    step = (size_t)d.n * ld;
  }
  __device__ double* at(int j) const { return p + j * step; }
};

// dst (rows x nr, smem ld) <- src rows (global, stride lds) (+ src2, stride kRhsChunk)
template <typename TS>
__device__ void load_vec(TS* dst, int ldd, const double* src, int lds, const double* src2, int rows,
                         int nr, Grp G) {
  if (src2) {
#pragma unroll 2
    for (int e = G.tid; e < rows * nr; e += G.nt) {
      const int r = e / nr, c = e - r * nr;
      dst[r * ldd + c] = (TS)(src[(size_t)r * lds + c] + src2[(size_t)r * kRhsChunk + c]);
    }
  } else {
#pragma unroll 2
    for (int e = G.tid; e < rows * nr; e += G.nt) {
      const int r = e / nr, c = e - r * nr;
      dst[r * ldd + c] = (TS)src[(size_t)r * lds + c];
    }
  }
}

template <typename TS>
__device__ void store_vec(double* dst, int ldd, const TS* src, int lds, int rows, int nr, Grp G) {
#pragma unroll 2
  for (int e = G.tid; e < rows * nr; e += G.nt) {
    const int r = e / nr, c = e - r * nr;
    dst[(size_t)r * ldd + c] = (double)src[r * lds + c];
  }
}

// load_vec in two parts: the loads into registers, and the stores some work
// later (up to U elements per thread; further ones are loaded late). U = 3:
// kMaxN x kRhsChunk elements by 256 threads.
template <int U>
struct VecPrefetch {
  double v[U + 1], w[U + 1];
  const double *src, *src2;
  int lds;
  __device__ __forceinline__ void load(const double* s, int ld, const double* s2, int rows, int nr, const Div& by,
                                       Grp G) {
    src = s;
    src2 = s2;
    lds = ld;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = G.tid + u * G.nt, r = by(e), c = e - r * nr;
      w[u] = 0.0;
      if (G.tid >= 0 && e < rows * nr) {
        v[u] = s[(size_t)r * ld + c];
        if (s2) w[u] = s2[(size_t)r * kRhsChunk + c];
      }
    }
  }
  template <typename TS>
  __device__ __forceinline__ void store(TS* dst, int ldd, int rows, int nr, const Div& by, Grp G) const {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = G.tid + u * G.nt, r = by(e);
      if (G.tid >= 0 && e < rows * nr) dst[r * ldd + e - r * nr] = (TS)(src2 ? v[u] + w[u] : v[u]);
    }
    if (G.tid < 0) return;
#pragma unroll 1
    for (int e = G.tid + U * G.nt; e < rows * nr; e += G.nt) {
      const int r = by(e), c = e - r * nr;
      const double x = src[(size_t)r * lds + c];
      dst[r * ldd + c] = (TS)(src2 ? x + src2[(size_t)r * kRhsChunk + c] : x);
    }
  }
};

__device__ __forceinline__ double shfl_idx(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ float shfl_idx(float v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// Asynchronous global -> shared copy of one 4- or 8-byte element (no
// register staging; completes at cp_async_wait).
template <typename T>
__device__ __forceinline__ void cp_async_elem(T* dst, const T* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if (sizeof(T) == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// every group but the two most recent ones complete
__device__ __forceinline__ void cp_async_wait_2() { asm volatile("cp.async.wait_group 2;" ::: "memory"); }

// cp.async of `cnt` contiguous elements by the group: 16 bytes at a time where both ends are aligned
template <typename T>
__device__ __forceinline__ void cp_async_flat(T* dst, const T* src, int cnt, Grp G) {
  constexpr int V = 16 / (int)sizeof(T);
  if ((((size_t)dst | (size_t)src) & 15) == 0 && cnt % V == 0) {
#pragma unroll 2
    for (int e = V * G.tid; e < cnt; e += V * G.nt)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst + e)),
                   "l"(src + e)
                   : "memory");
  } else {
#pragma unroll 2
    for (int e = G.tid; e < cnt; e += G.nt) cp_async_elem(dst + e, src + e);
  }
}

// t <- L^{-1} t (forward) or t <- L^{-T} t (backward) for nr columns, warp-
// synchronous, without the group's barrier. Rows i and i + 32 of a column live
// in lane i. M holds the multipliers of step j as its row j (forward: columns
// of L divided by their diagonal, backward: rows of L): u_i -= M_ji u_j for the
// rows i behind j, x = u * rinv.
// A step is the broadcast of u_j and one FP64 FMA: 115 cycles in a row (a
// device probe), 83 per column where a warp takes two (NC = 2), against 163
// with a branch per step and its multipliers' latency: they are read four steps
// ahead. (A broadcast through shared memory takes 119; one broadcast for two steps and
// another FMA in its place, 133.)
// LEAN, for tasks that share an SM by the dozen: their number hides the latency,
// the FP64 pipe and the registers are the limit, so no step too many and four
// multipliers at a time (eight in flight cost registers: 8 systems of 2000 stages, n = 12
// in 300 segments solved in 3847 us against 3367; of 4000 stages, n = 8, 64 systems 1388
// against 1317).
template <typename TS, int NC, bool TWO, bool BW, bool LEAN = false>
__device__ __forceinline__ void trsv_cols(TS* t, int ldt, const TS* M, int ldl, const TS* rinv, int n, int c, int dc,
                                          int lane) {
  const int i0 = lane, i1 = lane + 32, r0 = min(i0, n - 1), r1 = min(i1, n - 1);  // (r: rows for addresses)
  TS u0[NC], u1[NC], ma0[4], ma1[4], mb0[4], mb1[4];
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    u0[q] = i0 < n ? t[i0 * ldt + c + q * dc] : TS(0);
    u1[q] = TWO && i1 < n ? t[i1 * ldt + c + q * dc] : TS(0);
  }
  const int steps = n - 1;
  auto load = [&](int s0, TS* m0, TS* m1) {
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const int k = min(s0 + s, steps), j = BW ? n - 1 - k : k;
      m0[s] = M[j * ldl + r0];
      m1[s] = TWO ? M[j * ldl + r1] : TS(0);
    }
  };
  // four steps (those past the last one change dead rows only; LEAN leaves them
  // out); no branch a lane could take alone
  auto run = [&](int s0, const TS* m0, const TS* m1) {
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      if (LEAN && s0 + s >= steps) break;
      const int j = BW ? n - 1 - s0 - s : s0 + s;
      TS x[NC];
#pragma unroll
      for (int q = 0; q < NC; ++q) x[q] = shfl_idx(TWO && j >= 32 ? u1[q] : u0[q], j & 31);
      if (!TWO || BW || j < 31) {
#pragma unroll
        for (int q = 0; q < NC; ++q) {
          const TS v = fma(-m0[s], x[q], u0[q]);
          u0[q] = (BW ? i0 < j : i0 > j) ? v : u0[q];
        }
      }
      if (TWO && (!BW || j > 32)) {
#pragma unroll
        for (int q = 0; q < NC; ++q) {
          const TS v = fma(-m1[s], x[q], u1[q]);
          u1[q] = (BW ? i1 < j : i1 > j) ? v : u1[q];
        }
      }
    }
  };
  load(0, ma0, ma1);
#pragma unroll 1
  for (int s0 = 0; s0 < steps; s0 += 4) {
    if (LEAN) {
      run(s0, ma0, ma1);
      if (s0 + 4 < steps) load(s0 + 4, ma0, ma1);
      continue;
    }
    load(s0 + 4, mb0, mb1);
    run(s0, ma0, ma1);
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      ma0[s] = mb0[s];
      ma1[s] = mb1[s];
    }
  }
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    if (i0 < n) t[i0 * ldt + c + q * dc] = u0[q] * rinv[i0];
    if (TWO && i1 < n) t[i1 * ldt + c + q * dc] = u1[q] * rinv[i1];
  }
}
template <typename TS, bool BW>
__device__ __noinline__ void trsv_warp(TS* t, int ldt, const TS* M, int ldl, const TS* rinv, int n, int nr, Grp G) {
  const int lane = G.tid & 31, nw = G.nt >> 5;
  for (int c = G.tid >> 5; c < nr; c += 2 * nw) {
    const bool two = c + nw < nr;
    if (n <= 32) {
      if (two) trsv_cols<TS, 2, false, BW>(t, ldt, M, ldl, rinv, n, c, nw, lane);
      else trsv_cols<TS, 1, false, BW>(t, ldt, M, ldl, rinv, n, c, nw, lane);
    } else {
      if (two) trsv_cols<TS, 2, true, BW>(t, ldt, M, ldl, rinv, n, c, nw, lane);
      else trsv_cols<TS, 1, true, BW>(t, ldt, M, ldl, rinv, n, c, nw, lane);
    }
  }
}
// (kWarp, kDense: a column at a time; one-warp tasks have n <= 32)
template <typename TS, int KIND, bool BW>
__device__ __forceinline__ void trsv_group(TS* t, int ldt, const TS* M, int ldl, const TS* rinv, int n, int nr,
                                           Grp G) {
  if (KIND == kAlone) {
    trsv_warp<TS, BW>(t, ldt, M, ldl, rinv, n, nr, G);
    return;
  }
  const int lane = G.tid & 31;
  for (int c = KIND == kWarp ? 0 : G.tid >> 5; c < nr; c += KIND == kWarp ? 1 : G.nt >> 5) {
    if (KIND == kWarp || n <= 32) trsv_cols<TS, 1, false, BW, true>(t, ldt, M, ldl, rinv, n, c, 0, lane);
    else trsv_cols<TS, 1, true, BW, true>(t, ldt, M, ldl, rinv, n, c, 0, lane);
  }
}

// Shared-memory view of a substitution task: double-buffered factor blocks
// (selected by value, not by a run-time array index, which would put the
// pointers in local memory), the panel vector V and the stage vector t.
template <typename TS>
struct SolveSmem {
  TS *L0, *L1, *ri0, *ri1, *Z0, *Z1, *V, *t;
  int ldL, ldZ, ldV, Rs;  // Rs: panel rows held (2n + m, or n + m on a level with P = 1)
  __device__ TS* L(int q) const { return q ? L1 : L0; }
  __device__ TS* rinv(int q) const { return q ? ri1 : ri0; }
  __device__ TS* Z(int q) const { return q ? Z1 : Z0; }
};

template <typename TS>
__device__ __forceinline__ SolveSmem<TS> solve_smem(unsigned char* sm, int n, int m, bool fill) {
  SolveSmem<TS> S;
  const SolLayout L = sol_layout(n, m, (int)sizeof(TS), fill);
  S.Rs = L.R;
  S.ldL = n;
  S.ldZ = L.ldZ;
  S.ldV = L.ldV;
  S.L0 = (TS*)(sm + L.oL[0]);
  S.L1 = (TS*)(sm + L.oL[1]);
  S.ri0 = (TS*)(sm + L.oRinv[0]);
  S.ri1 = (TS*)(sm + L.oRinv[1]);
  S.Z0 = (TS*)(sm + L.oZ[0]);
  S.Z1 = (TS*)(sm + L.oZ[1]);
  S.V = (TS*)(sm + L.oV);
  S.t = (TS*)(sm + L.oT);
  return S;
}

template <typename TS>
struct FactorView {
  const TS *M, *MR, *ri, *P;
};
__device__ __forceinline__ FactorView<double> factor_view(const LevelDesc& d, double) {
  return FactorView<double>{d.LdM, d.LdR, d.Lri, d.Lp};
}
__device__ __forceinline__ FactorView<float> factor_view(const LevelDesc& d, float) {
  return FactorView<float>{d.LdMf, d.LdRf, d.Lrif, d.Lpf};
}

// Start the asynchronous load of the factor blocks of stage j into buffer q
// (the multipliers of trsv_warp, both stored as its rows, 1/diag, panel rows
// [r0, r1)).
template <typename TS>
__device__ void prefetch_stage_factor(const SolveSmem<TS>& S, int q, const FactorView<TS>& F, int n, int m, int j,
                                      int r0, int r1, bool backward, Grp G) {
  if (G.tid < 0) return;
  const int R = 2 * n + m;
  cp_async_flat(S.L(q), (backward ? F.MR : F.M) + (size_t)j * n * n, n * n, G);
  for (int e = G.tid; e < n; e += G.nt) cp_async_elem(S.rinv(q) + e, F.ri + (size_t)j * n + e);
  const TS* P = F.P + (size_t)j * R * n;
  const Div by(n);
#pragma unroll 2
  for (int e = G.tid + r0 * n; e < r1 * n; e += G.nt) {
    const int r = by(e), c = e - r * n;
    cp_async_elem(S.Z(q) + r * S.ldZ + c, P + e);
  }
  cp_async_commit();
}

// the warps without a column of trsv_warp, for the copies beside it; all of them
// where every warp has one
__device__ __forceinline__ Grp beside(Grp G, int nr) {
  const int used = 32 * nr < G.nt ? 32 * nr : 0;
  return Grp{G.tid - used, G.nt - used, G.bar};
}

__device__ __forceinline__ void stage_rows(const SegGeom& g, int i, int n, int m, int& r0, int& r1) {
  const bool eRows = (i < g.len - 1) || g.hasF;
  r0 = eRows ? 0 : n;
  r1 = n + m + (g.hasW ? n : 0);
}

// Backward substitution over the stages of one segment (Algorithm 3,
// parallel phase; for the top level the whole sequential sweep). On entry
// S.V holds [x_next (E rows); x_g (G rows); x_sep (W rows)]. The factor
// blocks of the next stage stream in while the current one is solved.
// (prefetched: the last stage's factor blocks were already requested into
// buffer 0, see backward_prefetch)
template <typename TS, int KIND>
__device__ void backward_segment(const SolveSmem<TS>& S, const LevelDesc& d, const SegGeom& g,
                                 double* b, int ldb, int nr, int c0, Grp G, bool prefetched = false) {
  const int n = d.n, m = d.m;
  int r0, r1;
  stage_rows(g, g.len - 1, n, m, r0, r1);
  const FactorView<TS> F = factor_view(d, TS(0));
  const VecViews X(d, b, ldb, c0);
  const Grp B = beside(G, nr);
  if (!prefetched) prefetch_stage_factor(S, 0, F, n, m, g.f + g.len - 1, r0, r1, true, G);
  const Div by(nr);
  TS *t = S.t, *xe = S.V;  // y_j, then x_j; the E-rows of v: x_{j+1}
  load_vec(t, S.ldV, (const double*)X.at(g.f + g.len - 1), X.ld, (const double*)nullptr, n, nr, G);
  for (int i = g.len - 1; i >= 0; --i) {
    const int j = g.f + i, q = (g.len - 1 - i) & 1;
    stage_rows(g, i, n, m, r0, r1);
    VecPrefetch<KIND == kAlone ? 3 : 0> yp;  // y_{j-1}: its loads pass during this stage
    cp_async_wait_all();
    gsync(G);
    if (i > 0) {
      yp.load(X.at(j - 1), X.ld, nullptr, n, nr, by, B);
    }
    const TS* Z = S.Z(q);
    // t = y_j - Z^T v over the active panel rows: four lanes per output (each
    // a quarter of the rows, two partial sums), shuffle-reduced
    {
      const int outs = n * nr, span = (outs * 4 + 31) & ~31, rows = r1 - r0;
      auto v = [&](int r, int c) { return (r < n ? xe : S.V)[r * S.ldV + c]; };
#pragma unroll 1
      for (int e = G.tid; e < span; e += G.nt) {
        const int o = e >> 2, qq = e & 3;
        const bool act = o < outs;
        const int oo = act ? o : 0;
        const int c2 = by(oo), c = oo - c2 * nr;
        const int ra = r0 + ((qq * rows) >> 2), rb = r0 + (((qq + 1) * rows) >> 2);
        TS a0 = 0, a1 = 0;
        int r = ra;
        if (act) {
#pragma unroll(KIND == kAlone ? 4 : 1)
          for (; r + 1 < rb; r += 2) {
            a0 = fma(Z[r * S.ldZ + c2], v(r, c), a0);
            a1 = fma(Z[(r + 1) * S.ldZ + c2], v(r + 1, c), a1);
          }
          if (r < rb) a0 = fma(Z[r * S.ldZ + c2], v(r, c), a0);
        }
        TS a = a0 + a1;
        a += __shfl_xor_sync(0xffffffffu, a, 1);
        a += __shfl_xor_sync(0xffffffffu, a, 2);
        if (act && qq == 0) t[c2 * S.ldV + c] -= a;
      }
    }
    gsync(G);
    if (i > 0) {
      int p0, p1;
      stage_rows(g, i - 1, n, m, p0, p1);
      prefetch_stage_factor(S, q ^ 1, F, n, m, j - 1, p0, p1, true, B);
    }
    trsv_group<TS, KIND, true>(t, S.ldV, S.L(q), S.ldL, S.rinv(q), n, nr, G);
    if (i > 0) yp.store(xe, S.ldV, n, nr, by, B);
    gsync(G);
    store_vec(X.at(j), X.ld, t, S.ldV, n, nr, G);
    TS* const sw = t;
    t = xe;
    xe = sw;
  }
  gsync(G);
}

// Forward substitution (Algorithm 2) for one segment; the top level (P = 1)
// also solves the corner and runs its own backward sweep (Algorithm 3,
// sequential phase). `skip`: per-system flags; a set flag returns at once.
template <typename TS, int KIND>
__device__ void forward_task(const Task tk, const LevelDesc* __restrict__ descs, double* b, int ldb, int nr,
                             const int* skip, unsigned char* smraw, Grp G, int fwd_done, int c0) {
  const LevelDesc& d = descs[tk.desc];
  if (skip && skip[d.sys]) return;
  if (fwd_done && !d.is_top) return;  // the factorization carried this forward sweep
  if (!task_geometry_ok(d, tk.seg, smraw, sol_layout(d.n, d.m, (int)sizeof(TS), d.P > 1).total)) return;
  const int n = d.n, m = d.m, mg = d.m - d.mr;  // mg: rows of the real arrow
  const SolveSmem<TS> S = solve_smem<TS>(smraw, n, m, d.P > 1);
  const int oG = n, oW = n + m;
  const SegGeom g = seg_geom(d, tk.seg);
  const int k = tk.seg;
  int r0, r1;
  stage_rows(g, 0, n, m, r0, r1);
  const FactorView<TS> F = factor_view(d, TS(0));
  const VecViews X(d, b, ldb, c0);
  // right-hand side of stage j of this level: the caller's, or RA + RB
  const double* const ra = d.level == 1 ? X.p : d.RA + c0;
  const double* const rb = d.level == 1 ? nullptr : d.RB + c0;
  const int ldr = d.level == 1 ? X.ld : kRhsChunk;
  const Grp B = beside(G, nr);
  if (!fwd_done) prefetch_stage_factor(S, 0, F, n, m, g.f, r0, r1, false, G);
  // V_G <- 0, V_W <- rhs of the separator, t <- rhs of the first stage
  for (int e = G.tid; e < S.Rs * S.ldV; e += G.nt) S.V[e] = TS(0);
  gsync(G);
  auto rhs = [&](int j, TS* dst) {
    const size_t o = (size_t)j * n * ldr;
    load_vec(dst, S.ldV, ra + o, ldr, rb ? rb + o : nullptr, n, nr, G);
  };
  if (g.hasW) rhs(g.f - 1, S.V + oW * S.ldV);
  rhs(g.f, S.t);
  const Div by(nr);
  // this stage's vector, and the E-rows of the panel product: the next stage's
  TS *t = S.t, *tn = S.V;
  // a bordered factorization already carried this forward sweep (fwd_done)
  for (int i = 0; i < (fwd_done ? 0 : g.len); ++i) {
    const int j = g.f + i, q = i & 1;
    const bool more = i + 1 < g.len;
    stage_rows(g, i, n, m, r0, r1);
    VecPrefetch<KIND == kAlone ? 3 : 0> bp;  // the next stage's rhs: its loads pass during the solve
    if (more) {
      const size_t o = (size_t)(j + 1) * n * ldr;
      bp.load(ra + o, ldr, rb ? rb + o : nullptr, n, nr, by, B);
    }
    cp_async_wait_all();
    gsync(G);
    if (more) {
      int p0, p1;
      stage_rows(g, i + 1, n, m, p0, p1);
      prefetch_stage_factor(S, q ^ 1, F, n, m, j + 1, p0, p1, false, B);
    }
    trsv_group<TS, KIND, false>(t, S.ldV, S.L(q), S.ldL, S.rinv(q), n, nr, G);
    if (more) bp.store(tn, S.ldV, n, nr, by, B);
    else
      for (int e = G.tid; e < n * S.ldV; e += G.nt) tn[e] = TS(0);  // the F-hat term
    gsync(G);
    store_vec(X.at(j), X.ld, t, S.ldV, n, nr, G);
    // [V_E; V_G; V_W] -= Z y over the active panel rows: four lanes per output
    // (each a quarter of the dot product, two partial sums), shuffle-reduced
    const TS* Z = S.Z(q);
    {
      const int outs = (r1 - r0) * nr, span = (outs * 4 + 31) & ~31;
#pragma unroll 1
      for (int e = G.tid; e < span; e += G.nt) {
        const int o = e >> 2, qq = e & 3;
        const bool act = o < outs;
        const int oo = act ? o : 0;
        const int r = r0 + by(oo), c = oo - (r - r0) * nr;
        const int k0 = (qq * n) >> 2, k1 = ((qq + 1) * n) >> 2;
        TS a0 = 0, a1 = 0;
        int t2 = k0;
        if (act) {
#pragma unroll(KIND == kAlone ? 4 : 1)
          for (; t2 + 1 < k1; t2 += 2) {
            a0 = fma(Z[r * S.ldZ + t2], t[t2 * S.ldV + c], a0);
            a1 = fma(Z[r * S.ldZ + t2 + 1], t[(t2 + 1) * S.ldV + c], a1);
          }
          if (t2 < k1) a0 = fma(Z[r * S.ldZ + t2], t[t2 * S.ldV + c], a0);
        }
        TS a = a0 + a1;
        a += __shfl_xor_sync(0xffffffffu, a, 1);
        a += __shfl_xor_sync(0xffffffffu, a, 2);
        if (act && qq == 0) (r < n ? tn : S.V)[r * S.ldV + c] -= a;
      }
    }
    TS* const sw = t;
    t = tn;
    tn = sw;
  }
  gsync(G);
  if (!d.is_top) {
    if (g.hasF) store_vec(d.YB + (size_t)k * n * kRhsChunk + c0, kRhsChunk, t, S.ldV, n, nr, G);
    if (g.hasW)
      store_vec(d.YA + (size_t)(k - 1) * n * kRhsChunk + c0, kRhsChunk, S.V + oW * S.ldV, S.ldV, n, nr, G);
    if (m) store_vec(d.ygpart + (size_t)k * m * kRhsChunk + c0, kRhsChunk, S.V + oG * S.ldV, S.ldV, m, nr, G);
    return;
  }
  // top level: corner y_g = R-hat^{-1} (r_g + sum of every yg partial + own),
  // x_g = R-hat^{-T} y_g, written to the caller's b; then the backward sweep.
  // After a bordered factorization y_g is the bordered row of R-hat itself.
  if (mg) {
    double* bg = b + (size_t)d.rowG * ldb;
    TS* gv = S.t;
    const int ldR = odd(mg);
    if (fwd_done) {
      for (int e = G.tid; e < mg * nr; e += G.nt) {
        const int r = e / nr, c = e - r * nr;
        gv[r * S.ldV + c] = (TS)d.Rhat[(size_t)(mg + c) * m + r];
      }
    } else {
      sum_partials(
          G, mg * nr, d.nyg_all,
          [&](int p, int o) { return d.yg_all[((size_t)p * m + o / nr) * kRhsChunk + c0 + o % nr]; },
          [&](int o, double v) {
            const int r = o / nr, c = o - r * nr;
            gv[r * S.ldV + c] = (TS)((bg[(size_t)r * ldb + c] + v) + (double)S.V[(oG + r) * S.ldV + c]);
          });
    }
    for (int e = G.tid; e < mg * mg; e += G.nt) {  // R-hat: columns scaled (transposed), rows scaled
      const int r = e / mg, c = e - r * mg;
      S.L(0)[c * ldR + r] = (TS)(d.Rhat[r * m + c] * d.Rri[c]);
      S.L(1)[r * ldR + c] = (TS)(d.Rhat[r * m + c] * d.Rri[r]);
    }
    for (int e = G.tid; e < mg; e += G.nt) S.rinv(0)[e] = (TS)d.Rri[e];
    gsync(G);
    if (!fwd_done) {
      trsv_group<TS, KIND, false>(gv, S.ldV, S.L(0), ldR, S.rinv(0), mg, nr, G);
      gsync(G);
    }
    trsv_group<TS, KIND, true>(gv, S.ldV, S.L(1), ldR, S.rinv(0), mg, nr, G);
    gsync(G);
    store_vec(bg, ldb, gv, S.ldV, mg, nr, G);
  }
  // V <- [0; x_g; 0; -] for the backward sweep of the top level (bordered rows 0)
  for (int e = G.tid; e < S.Rs * S.ldV; e += G.nt) {
    const int r = e / S.ldV;
    if (r < oG || r >= oG + mg) S.V[e] = TS(0);
    else S.V[e] = S.t[(r - oG) * S.ldV + (e - r * S.ldV)];
  }
  gsync(G);
  backward_segment<TS, KIND>(S, d, g, b, ldb, nr, c0, G);
}

// Backward substitution (Algorithm 3, parallel phase) for one segment below
// the top level: needs x_g (already in b), the separator solutions of the
// next level (x at s_k and s_{k+1}), and this level's y.
template <typename TS, int KIND = kAlone>
__device__ void backward_task(const Task tk, const LevelDesc* __restrict__ descs, double* b, int ldb, int nr,
                              const int* skip, unsigned char* smraw, Grp G, int c0 = 0, bool prefetched = false) {
  const LevelDesc& d = descs[tk.desc];
  if (skip && skip[d.sys]) return;
  if (!task_geometry_ok(d, tk.seg, smraw, sol_layout(d.n, d.m, (int)sizeof(TS), d.P > 1).total)) return;
  const int n = d.n, m = d.m;
  const SolveSmem<TS> S = solve_smem<TS>(smraw, n, m, d.P > 1);
  const int oG = n, oW = n + m;
  const SegGeom g = seg_geom(d, tk.seg);
  const int k = tk.seg;
  const double* none = nullptr;
  for (int e = G.tid; e < S.Rs * S.ldV; e += G.nt) S.V[e] = TS(0);
  gsync(G);
  if (g.hasF) load_vec(S.V, S.ldV, d.Xnext + (size_t)k * n * kRhsChunk + c0, kRhsChunk, none, n, nr, G);
  if (d.m - d.mr) load_vec(S.V + oG * S.ldV, S.ldV, b + (size_t)d.rowG * ldb, ldb, none, d.m - d.mr, nr, G);
  if (g.hasW) {
    load_vec(S.V + oW * S.ldV, S.ldV, d.Xnext + (size_t)(k - 1) * n * kRhsChunk + c0, kRhsChunk, none, n,
             nr, G);
    gsync(G);
    const VecView xs = level_vec(d, b, ldb, g.f - 1, c0);  // this level's copy of x at s_k
    store_vec(xs.p, xs.ld, S.V + oW * S.ldV, S.ldV, n, nr, G);
  }
  gsync(G);
  backward_segment<TS, KIND>(S, d, g, b, ldb, nr, c0, G, prefetched);
}

// The factor blocks of the backward sweep's first stage (the segment's last)
// into buffer 0: they do not depend on x, so a task can request them before
// the solutions it needs exist.
template <typename TS>
__device__ void backward_prefetch(const Task tk, const LevelDesc& d, unsigned char* smraw, Grp G) {
  const SolveSmem<TS> S = solve_smem<TS>(smraw, d.n, d.m, d.P > 1);
  const SegGeom g = seg_geom(d, tk.seg);
  int r0, r1;
  stage_rows(g, g.len - 1, d.n, d.m, r0, r1);
  prefetch_stage_factor(S, 0, factor_view(d, TS(0)), d.n, d.m, g.f + g.len - 1, r0, r1, true, G);
}


// One CTA per task (blocks above kWarpMaxN), or one warp per task with a
// shared-memory slice each (small blocks; `slice` bytes per warp).
template <typename TS, int KIND>
__global__ void __launch_bounds__(kSolveThreads, KIND == kDense ? 4 : 2) k_forward(const LevelDesc* __restrict__ descs,
                                                           const Task* __restrict__ tasks, double* b,
                                                           int ldb, int nr, const int* skip, int fwd_done,
                                                           int split) {
  extern __shared__ __align__(16) unsigned char smraw[];
  // `split` CTAs per task, each on its own group of right-hand-side columns
  const int cg = blockIdx.x % split, nc = (nr + split - 1) / split, c0 = cg * nc, cn = min(nc, nr - c0);
  if (cn <= 0) return;
  forward_task<TS, KIND>(tasks[blockIdx.x / split], descs, b + c0, ldb, cn, skip, smraw, cta_grp(), fwd_done, c0);
}
template <typename TS, int KIND>
__global__ void __launch_bounds__(kSolveThreads, KIND == kDense ? 4 : 2) k_backward(const LevelDesc* __restrict__ descs,
                                                            const Task* __restrict__ tasks, double* b,
                                                            int ldb, int nr, const int* skip, int split) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int cg = blockIdx.x % split, nc = (nr + split - 1) / split, c0 = cg * nc, cn = min(nc, nr - c0);
  if (cn <= 0) return;
  backward_task<TS, KIND>(tasks[blockIdx.x / split], descs, b + c0, ldb, cn, skip, smraw, cta_grp(), c0);
}
template <typename TS>
__global__ void __launch_bounds__(256, 3) k_forward_w(const LevelDesc* __restrict__ descs,
                                                   const Task* __restrict__ tasks, int ntasks, double* b,
                                                   int ldb, int nr, const int* skip, int slice, int fwd_done) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int wid = threadIdx.x >> 5, t = blockIdx.x * (blockDim.x >> 5) + wid;
  if (t >= ntasks) return;  // whole warp
  forward_task<TS, kWarp>(tasks[t], descs, b, ldb, nr, skip, smraw + (size_t)wid * slice,
                   Grp{(int)(threadIdx.x & 31), 32, -1}, fwd_done);
}
template <typename TS>
__global__ void __launch_bounds__(256, 3) k_backward_w(const LevelDesc* __restrict__ descs,
                                                    const Task* __restrict__ tasks, int ntasks, double* b,
                                                    int ldb, int nr, const int* skip, int slice) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int wid = threadIdx.x >> 5, t = blockIdx.x * (blockDim.x >> 5) + wid;
  if (t >= ntasks) return;  // whole warp
  backward_task<TS, kWarp>(tasks[t], descs, b, ldb, nr, skip, smraw + (size_t)wid * slice,
                    Grp{(int)(threadIdx.x & 31), 32, -1});
}

// Every backward level below the top (Algorithm 3, parallel phase of each
// level, top down) in one launch. Items are (segment task, column group)
// pairs in chain order: the levels from the one below the top down to level
// 1, each level's items together. CTAs take items by ticket, so a CTA only
// ever waits for items taken before its own, which running CTAs hold. An
// item first requests its stage's factor blocks (they do not depend on x),
// then waits until every item of the level above has released its counter
// (thread 0 polls with ld.acquire.gpu, bounded by `wait` clock cycles; a
// wait that runs out records KKT_ERR_TIMEOUT and skips the item), solves,
// and releases its own level's counter. ctr[0] is the ticket, ctr[1 + li]
// the finished items of chain level li; the host zeroes them before the
// launch. unmet: every wait expects one item more than its level has (a
// test of the timeout path).
template <typename TS>
__global__ void __launch_bounds__(kSolveThreads, 2) k_backward_chain(const LevelDesc* __restrict__ descs,
                                                                  const Task* __restrict__ tasks, ChainPlan cp,
                                                                  int* ctr, double* b, int ldb, int nr,
                                                                  const int* skip, Info* info,
                                                                  long long wait_cycles, int unmet) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int cur, ok;
  const int total = cp.nlev > 0 ? cp.end[cp.nlev - 1] : 0;
  for (;;) {
    if (threadIdx.x == 0) cur = atomicAdd(ctr, 1);
    __syncthreads();
    const int t = cur;
    if (t >= total) break;
    int li = 0;
    while (t >= cp.end[li]) ++li;
    const int u = t - (li ? cp.end[li - 1] : 0), sp = cp.split[li];
    const Task tk = tasks[cp.off[li] + u / sp];
    const LevelDesc& d = descs[tk.desc];
    const int nc = (nr + sp - 1) / sp, c0 = (u % sp) * nc, cn = min(nc, nr - c0);
    bool work = cn > 0 && !(skip && skip[d.sys]) &&
                task_geometry_ok(d, tk.seg, smraw, sol_layout(d.n, d.m, (int)sizeof(TS), d.P > 1).total);
    if (work) backward_prefetch<TS>(tk, d, smraw, cta_grp());
    if (threadIdx.x == 0) {
      int good = 1;
      if (li > 0) {
        const int need = cp.end[li - 1] - (li >= 2 ? cp.end[li - 2] : 0) + unmet;
        const long long t0 = clock64();
        while (ld_acquire_gpu(ctr + li) < need) {
          if (clock64() - t0 > wait_cycles) {
            good = 0;
            break;
          }
        }
      }
      ok = good;
      if (!good) record_timeout(info, d.sys, d.nat[d.seg[tk.seg]], d.level);
    }
    __syncthreads();
    work = work && ok;
    if (work) backward_task<TS>(tk, descs, b + c0, ldb, cn, nullptr, smraw, cta_grp(), c0, true);
    cp_async_wait_all();  // (a skipped item's requested blocks)
    __syncthreads();
    // release: the item's writes precede the barrier, and the release
    // reduction orders them (cumulatively) before the counter's increment
    if (threadIdx.x == 0) red_release_gpu(ctr + 1 + li);
  }
}

// ---------------------------------------------------------------------------
// Whole substitution of a system whose level plan is one level with P = 1
// (the sequential method), one right-hand side, one warp per system:
// Algorithm 2 over the N stages, the corner of Eq. (7), Algorithm 3 back.
// Stage j's n x n multipliers and its panel rows (the E-hat rows when a next
// stage exists, then the arrow rows) arrive by two bulk copies into one of
// `nbuf` (2 to 4) shared-memory buffers; the 2N stage visits (forward, then
// backward) form one sequence whose next nbuf - 1 visits are in flight while
// one is solved (the backward sweep's first stages arrive during the last
// forward stages and the corner). A
// lane owns rows `lane` (and `lane + 32` when RPL = 2) of a stage, so the
// warp needs no block barrier. Every shared-memory read is free of bank
// conflicts on the unpadded blocks: the forward multipliers are stored
// transposed (column c of L contiguous), the backward ones row-major, the
// backward panel product reads columns and the forward one walks a skewed
// diagonal (lane r reads column (r + kk) mod n of row r at step kk). The
// arrow rows' sums sum_j G-hat_j y_j stay in registers over the forward
// sweep (per lane, over its own rows) and are reduced across the warp once,
// before the corner. The right-hand side (forward) and y (backward) rows of
// the stages three ahead stream into a ring of shared-memory slots by
// cp.async, so no register waits on a load in flight.
// ---------------------------------------------------------------------------

// forward chain u_r -= (L_rc / L_cc) u_c for c < r; MT holds column c of L
// (divided by its diagonal) as row c
template <typename TS, int RPL>
__device__ __forceinline__ void seq_fwd_chain(TS& u0, TS& u1, const TS* MT, int n, int lane) {
  if (RPL == 1) {
    const int r0 = lane < n ? lane : n - 1;
    int c = 0;
#pragma unroll
    for (; c + 4 < n; c += 4) {  // multipliers of four steps loaded ahead
      const TS m0 = MT[c * n + r0], m1 = MT[(c + 1) * n + r0], m2 = MT[(c + 2) * n + r0],
               m3 = MT[(c + 3) * n + r0];
      TS uc = shfl_idx(u0, c);
      if (lane > c) u0 = fma(-m0, uc, u0);
      uc = shfl_idx(u0, c + 1);
      if (lane > c + 1) u0 = fma(-m1, uc, u0);
      uc = shfl_idx(u0, c + 2);
      if (lane > c + 2) u0 = fma(-m2, uc, u0);
      uc = shfl_idx(u0, c + 3);
      if (lane > c + 3) u0 = fma(-m3, uc, u0);
    }
#pragma unroll
    for (; c < n - 1; ++c) {
      const TS uc = shfl_idx(u0, c);
      if (lane > c) u0 = fma(-MT[c * n + r0], uc, u0);
    }
  } else {
    const int r1 = lane + 32 < n ? lane + 32 : n - 1;
#pragma unroll
    for (int c = 0; c < n - 1; ++c) {
      const TS m0 = MT[c * n + lane], m1 = MT[c * n + r1];
      const TS uc = shfl_idx(c < 32 ? u0 : u1, c & 31);
      if (lane > c) u0 = fma(-m0, uc, u0);
      if (lane + 32 > c && lane + 32 < n) u1 = fma(-m1, uc, u1);
    }
  }
}

// backward chain u_r -= (L_cr / L_cc) u_c for c > r; MR holds row c of L
// (divided by its diagonal)
template <typename TS, int RPL>
__device__ __forceinline__ void seq_bwd_chain(TS& u0, TS& u1, const TS* MR, int n, int lane) {
  if (RPL == 1) {
    const int r0 = lane < n ? lane : n - 1;
    int c = n - 1;
#pragma unroll
    for (; c - 3 > 0; c -= 4) {
      const TS m0 = MR[c * n + r0], m1 = MR[(c - 1) * n + r0], m2 = MR[(c - 2) * n + r0],
               m3 = MR[(c - 3) * n + r0];
      TS uc = shfl_idx(u0, c);
      if (lane < c) u0 = fma(-m0, uc, u0);
      uc = shfl_idx(u0, c - 1);
      if (lane < c - 1) u0 = fma(-m1, uc, u0);
      uc = shfl_idx(u0, c - 2);
      if (lane < c - 2) u0 = fma(-m2, uc, u0);
      uc = shfl_idx(u0, c - 3);
      if (lane < c - 3) u0 = fma(-m3, uc, u0);
    }
#pragma unroll
    for (; c > 0; --c) {
      const TS uc = shfl_idx(u0, c);
      if (lane < c) u0 = fma(-MR[c * n + r0], uc, u0);
    }
  } else {
    const int r1 = lane + 32 < n ? lane + 32 : n - 1;
#pragma unroll
    for (int c = n - 1; c > 0; --c) {
      const TS m0 = MR[c * n + lane], m1 = MR[c * n + r1];
      const TS uc = shfl_idx(c < 32 ? u0 : u1, c & 31);
      if (lane < c) u0 = fma(-m0, uc, u0);
      if (lane + 32 < c) u1 = fma(-m1, uc, u1);
    }
  }
}

// a_r = sum_k Z[r][k] y_k for the rows r = lane (a0) and lane + 32 (a1) of
// an n x n block, y_k held by lane k (k < 32, y0) or lane k - 32 (y1);
// lane r starts its walk over k at column r, so that the warp's reads of
// one step fall in distinct banks
template <typename TS, int RPL>
__device__ __forceinline__ void seq_fwd_panel(TS& a0, TS& a1, const TS* Z, TS y0, TS y1, int n, int lane) {
  if (RPL == 1) {
    const int r0 = lane < n ? lane : n - 1;
    const TS* zr = Z + r0 * n;
    int k = r0;
    TS s0 = TS(0), s1 = TS(0);
    int kk = 0;
#pragma unroll
    for (; kk + 1 < n; kk += 2) {
      const TS ya = shfl_idx(y0, k);
      const TS za = zr[k];
      k = k + 1 == n ? 0 : k + 1;
      const TS yb = shfl_idx(y0, k);
      const TS zb = zr[k];
      k = k + 1 == n ? 0 : k + 1;
      s0 = fma(za, ya, s0);
      s1 = fma(zb, yb, s1);
    }
    if (kk < n) s0 = fma(zr[k], shfl_idx(y0, k), s0);
    a0 = s0 + s1;
    a1 = TS(0);
  } else {
    const int r1 = lane + 32 < n ? lane + 32 : n - 1, h = n - 32;
    const TS *z0 = Z + lane * n, *z1 = Z + r1 * n;
    TS s0 = TS(0), s1 = TS(0);
#pragma unroll
    for (int kk = 0; kk < 32; ++kk) {  // columns 0..31: y from y0
      const int k = (lane + kk) & 31;
      const TS yk = shfl_idx(y0, k);
      s0 = fma(z0[k], yk, s0);
      s1 = fma(z1[k], yk, s1);
    }
    int k = lane % h;
#pragma unroll
    for (int kk = 0; kk < h; ++kk) {  // columns 32..n-1: y from y1
      const TS yk = shfl_idx(y1, k);
      s0 = fma(z0[32 + k], yk, s0);
      s1 = fma(z1[32 + k], yk, s1);
      k = k + 1 == h ? 0 : k + 1;
    }
    a0 = s0;
    a1 = s1;
  }
}

// NT > 0: every system of the launch has n = NT (the loops unroll with
// constant offsets); NT = 0: n from the descriptor, RPL rows per lane
template <typename TS, int RPL, int NT>
__global__ void __launch_bounds__(32) k_seq_solve(const LevelDesc* __restrict__ descs,
                                                  const Task* __restrict__ tasks, double* b, int ldb,
                                                  const int* skip, Info* info, long long wait_cycles,
                                                  int unmet, int nbuf) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int sb = (int)sizeof(TS);
  const int lane = threadIdx.x;
  const Task tk = tasks[blockIdx.x];
  const LevelDesc& d = descs[tk.desc];
  if (skip && skip[d.sys]) return;
  const int n = NT > 0 ? NT : d.n, m = d.m, N = d.N, R = 2 * n + m, mg = m - d.mr;
#ifdef KKT_DEBUG
  {
    unsigned dyn;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
    if (!dbg_ok(d.n == n && d.is_top && d.P == 1 && d.level == 1 && tk.seg == 0 && N >= 1 && seq_shape_ok(n, m, sb) &&
                    n <= 32 * RPL && mg >= 0 && d.nyg_all >= 0 && nbuf >= 2 && nbuf <= kSeqMaxBuf &&
                    seq_slice_bytes(n, m, sb, nbuf) <= (int)dyn,
                d))
      return;
  }
#endif
  uint64_t* bar = reinterpret_cast<uint64_t*>(smraw);  // one mbarrier per buffer
  const int bufB = seq_buf_bytes(n, m, sb);
  auto bufp = [&](int q) { return reinterpret_cast<TS*>(smraw + kSeqHeader + q * bufB); };
  const int zo = seq_zoff_bytes(n, sb) / sb;  // panel rows follow the multipliers
  const size_t nn = (size_t)n * n;
  const FactorView<TS> F = factor_view(d, TS(0));
  double* const bs = b + (size_t)d.offB * ldb;  // the system's stage rows
  const bool own0 = lane < n, own1 = RPL == 2 && lane + 32 < n;
  const int c0 = own0 ? lane : n - 1, c1 = own1 ? lane + 32 : n - 1;  // rows for addresses
  if (lane == 0) {
    for (int q = 0; q < nbuf; ++q) bulk::init(bar + q);
    bulk::fence_async();
  }
  __syncwarp();
  uint32_t phase = 0, pend = 0;  // bit q: parity of buffer q's next phase; buffer q's copies in flight
  // visit t of the sequence (t < N: forward stage t; else backward stage
  // 2N - 1 - t) into buffer t % nbuf: lane 0 copies the stage's multipliers
  // and panel rows; every lane notes the copies in flight
  auto issue = [&](int t) {
    const bool backward = t >= N;
    const int j = backward ? 2 * N - 1 - t : t, q = t & (nbuf - 1);
    if (lane == 0) {
      const int e0 = j < N - 1 ? 0 : n;  // E-hat rows exist above the last stage only
      const uint32_t bM = (uint32_t)(nn * sb), bZ = (uint32_t)((n + m - e0) * n * sb);
      TS* B = bufp(q);
      bulk::fence_async();
      bulk::expect_tx(bar + q, bM + bZ + (unmet ? 16u : 0u));  // unmet: a phase that never completes
      bulk::g2s(B, (backward ? F.MR : F.M) + (size_t)j * nn, bM, bar + q);
      if (bZ) bulk::g2s(B + zo, F.P + ((size_t)j * R + e0) * n, bZ, bar + q);
    }
    pend |= 1u << q;
  };
  auto wait_buf = [&](int q) -> bool {
    const bool got = __all_sync(0xffffffffu, bulk::wait(bar + q, (phase >> q) & 1u, wait_cycles));
    if (got) {
      phase ^= 1u << q;
      pend &= ~(1u << q);
    }
    return got;
  };
  // a copy that did not arrive: record it; the copies still in flight land
  // in this warp's buffers, so wait for them (bounded) before returning
  auto fail = [&](int stage) {
    if (lane == 0) record_timeout(info, d.sys, stage, 1);
    for (int q = 0; q < nbuf; ++q)
      if ((pend >> q) & 1u) (void)bulk::wait(bar + q, (phase >> q) & 1u, wait_cycles);
    cp_async_wait_all();  // the ring's copies too
  };
  // ring of kSeqRing slots (rows lane and lane + 32 of one stage each);
  // stage j's rows of bs go to slot j % kSeqRing, one commit group per stage
  double* const ring = reinterpret_cast<double*>(smraw + kSeqHeader + nbuf * bufB);
  auto ring_load = [&](int j) {
    if (j >= 0 && j < N) {
      double* sl = ring + (j & (kSeqRing - 1)) * 64;
      if (own0) cp_async_elem(sl + lane, bs + ((size_t)j * n + lane) * ldb);
      if (own1) cp_async_elem(sl + 32 + lane, bs + ((size_t)j * n + lane + 32) * ldb);
    }
    cp_async_commit();
  };
  auto ring_get = [&](int j, TS& v0, TS& v1) {  // after the wait for stage j's group
    const double* sl = ring + (j & (kSeqRing - 1)) * 64;
    v0 = own0 ? (TS)sl[lane] : TS(0);
    v1 = own1 ? (TS)sl[32 + lane] : TS(0);
  };
  constexpr int kAhead = kSeqRing - 1;  // stages in flight besides the one read

  // ---- forward sweep (Algorithm 2): L y = b
  for (int jj = 0; jj < kAhead; ++jj) ring_load(jj);
  cp_async_wait_2();
  TS t0, t1;
  ring_get(0, t0, t1);
  TS pg[kMaxM];  // this lane's terms of sum_j G-hat_j y_j, per arrow row
#pragma unroll
  for (int g = 0; g < kMaxM; ++g) pg[g] = TS(0);
  for (int t = 0; t < nbuf - 1 && t < 2 * N; ++t) issue(t);
  for (int j = 0; j < N; ++j) {
    const int q = j & (nbuf - 1);
    if (!wait_buf(q)) {
      fail(j);
      return;
    }
    __syncwarp();  // every lane is done with the buffer of the previous visit
    if (j + nbuf - 1 < 2 * N) issue(j + nbuf - 1);
    ring_load(j + kAhead);
    const TS* MT = bufp(q);
    const TS* Z = MT + zo;
    TS u0 = t0, u1 = t1;
    seq_fwd_chain<TS, RPL>(u0, u1, MT, n, lane);
    const TS y0 = own0 ? u0 * MT[c0 * n + c0] : TS(0);
    const TS y1 = own1 ? u1 * MT[c1 * n + c1] : TS(0);
    if (own0) bs[((size_t)j * n + lane) * ldb] = (double)y0;
    if (own1) bs[((size_t)j * n + lane + 32) * ldb] = (double)y1;
    const int e0 = j < N - 1 ? 0 : n;
    const TS* ZG = Z + (size_t)(n - e0) * n;  // arrow rows
#pragma unroll
    for (int g = 0; g < kMaxM; ++g) {
      if (g >= m) break;  // warp-uniform; full unrolling keeps pg in registers
      pg[g] = fma(ZG[g * n + c0], y0, pg[g]);
      if (RPL == 2) pg[g] = fma(ZG[g * n + c1], y1, pg[g]);
    }
    if (j + 1 < N) {  // t_{j+1} = b_{j+1} - E-hat_j y_j
      TS a0, a1;
      seq_fwd_panel<TS, RPL>(a0, a1, Z, y0, y1, n, lane);
      cp_async_wait_2();  // stage j + 1's group (two newer ones may be in flight)
      TS bn0, bn1;
      ring_get(j + 1, bn0, bn1);
      t0 = bn0 - a0;
      t1 = bn1 - a1;
    }
  }

  // ---- corner (Eq. (7)): R-hat R-hat^T x_g = b_g - sum_j G-hat_j y_j
  TS vg = TS(0);  // lane g: sum_j G-hat_j y_j of arrow row g
#pragma unroll
  for (int g = 0; g < kMaxM; ++g) {
    if (g >= m) break;
    TS v = pg[g];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == g) vg = v;
  }
  TS xgl = TS(0);  // lane g: x_g of arrow row g (0 for a bordered row)
  if (mg > 0) {
    const int gl = lane < mg ? lane : 0;
    double bsum = 0.0;
    if (lane < mg) {
      double v = 0.0;
      for (int p = 0; p < d.nyg_all; ++p) v += d.yg_all[((size_t)p * m + lane) * kRhsChunk];
      bsum = b[(size_t)(d.rowG + lane) * ldb] + v;
    }
    TS u = lane < mg ? (TS)(bsum + (double)(-vg)) : TS(0);
    double rrow[kMaxM], rcol[kMaxM];  // row and column gl of R-hat
#pragma unroll
    for (int p = 0; p < kMaxM; ++p) {
      rrow[p] = p < mg ? d.Rhat[gl * m + p] : 0.0;
      rcol[p] = p < mg ? d.Rhat[p * m + gl] : 0.0;
    }
    // R-hat y = u: u_g -= (R_gp / R_pp) u_p for p < g, y_g = u_g / R_gg
#pragma unroll
    for (int p = 0; p < kMaxM - 1; ++p) {
      if (p >= mg - 1) break;
      const TS up = shfl_idx(u, p);
      if (lane > p && lane < mg) u = fma(-(TS)(rrow[p] * d.Rri[p]), up, u);
    }
    u = u * (TS)d.Rri[gl];
    // R-hat^T x = y: u_g -= (R_pg / R_pp) u_p for p > g, x_g = u_g / R_gg
#pragma unroll
    for (int p = kMaxM - 1; p >= 1; --p) {
      if (p >= mg) continue;
      const TS up = shfl_idx(u, p);
      if (lane < p) u = fma(-(TS)(rcol[p] * d.Rri[p]), up, u);
    }
    const TS x = u * (TS)d.Rri[gl];
    if (lane < mg) b[(size_t)(d.rowG + lane) * ldb] = (double)x;
    xgl = lane < mg ? x : TS(0);
  }
  TS xg[kMaxM];  // x_g, every lane
#pragma unroll
  for (int g = 0; g < kMaxM; ++g) xg[g] = g < m ? shfl_idx(xgl, g) : TS(0);

  // ---- backward sweep (Algorithm 3): L^T x = y
  TS xn0 = TS(0), xn1 = TS(0);  // x of stage j + 1
  __threadfence_block();  // this lane's y stores before its asynchronous reads of them
  for (int jj = 0; jj < kAhead; ++jj) ring_load(N - 1 - jj);
  cp_async_wait_2();
  TS yc0, yc1;
  ring_get(N - 1, yc0, yc1);
  for (int s = 0; s < N; ++s) {
    const int j = N - 1 - s, t = N + s, q = t & (nbuf - 1);
    if (!wait_buf(q)) {
      fail(j);
      return;
    }
    __syncwarp();
    if (t + nbuf - 1 < 2 * N) issue(t + nbuf - 1);
    ring_load(j - kAhead);
    const TS* MR = bufp(q);
    const TS* Z = MR + zo;
    const int e0 = j < N - 1 ? 0 : n;
    const TS* ZG = Z + (size_t)(n - e0) * n;
    // t_c = y_c - sum_g G-hat_j[g][c] x_g - sum_r E-hat_j[r][c] x_{j+1, r}
    TS s0 = TS(0), s1 = TS(0), s0b = TS(0), s1b = TS(0);
#pragma unroll
    for (int g = 0; g < kMaxM; ++g) {
      if (g >= m) break;
      s0 = fma(ZG[g * n + c0], xg[g], s0);
      if (RPL == 2) s1 = fma(ZG[g * n + c1], xg[g], s1);
    }
    if (e0 == 0) {
#pragma unroll
      for (int r = 0; r < n; ++r) {
        const TS xr = shfl_idx(RPL == 2 && r >= 32 ? xn1 : xn0, r & 31);
        s0b = fma(Z[r * n + c0], xr, s0b);
        if (RPL == 2) s1b = fma(Z[r * n + c1], xr, s1b);
      }
    }
    TS u0 = yc0 - (s0 + s0b), u1 = yc1 - (s1 + s1b);
    seq_bwd_chain<TS, RPL>(u0, u1, MR, n, lane);
    xn0 = u0 * MR[c0 * n + c0];
    xn1 = u1 * MR[c1 * n + c1];
    if (own0) bs[((size_t)j * n + lane) * ldb] = (double)xn0;
    if (own1) bs[((size_t)j * n + lane + 32) * ldb] = (double)xn1;
    if (j > 0) {
      cp_async_wait_2();  // stage j - 1's group
      ring_get(j - 1, yc0, yc1);
    }
  }
  cp_async_wait_all();  // (only empty groups remain)
}

// ---------------------------------------------------------------------------
// Iterative refinement support (FP64): x += c; c = b - Psi x with the blocks
// of Eq. (3) (lower triangles of D and R read); eta = ||c||_inf /
// (||Psi||_inf ||x||_inf + ||b||_inf), maxima taken over all right-hand
// sides of the system together.
// ---------------------------------------------------------------------------

// x += c over the stage rows of one chunk; each system's first chunk also
// does the g rows. c has leading dimension kRhsChunk.
__global__ void k_axpy(const LevelDesc* __restrict__ descs, const ResTask* __restrict__ tasks,
                       double* x, int ldx, const double* c, int nr, const int* skip) {
  const ResTask tk = tasks[blockIdx.x];
  const LevelDesc& d = descs[tk.desc];
  if (skip && skip[d.sys]) return;
  const int j1 = min(tk.j0 + kResChunk, d.N);
  const long long row0 = d.offB + (long long)tk.j0 * d.n;
  const int rows = (j1 - tk.j0) * d.n;
  for (int e = threadIdx.x; e < rows * nr; e += blockDim.x) {
    const int r = e / nr, col = e - r * nr;
    x[(size_t)(row0 + r) * ldx + col] += c[(size_t)(row0 + r) * kRhsChunk + col];
  }
  if (tk.part == 0)
    for (int e = threadIdx.x; e < d.m * nr; e += blockDim.x) {
      const int r = e / nr, col = e - r * nr;
      x[(size_t)(d.rowG + r) * ldx + col] += c[(size_t)(d.rowG + r) * kRhsChunk + col];
    }
}

// |v| as an integer of the same order, 0 for NaN (which fmax passes over): the
// largest of a task without an FP64 instruction
__device__ __forceinline__ long long abs_order(double v) {
  const long long a = __double_as_longlong(v) & 0x7fffffffffffffffLL;
  return a > 0x7ff0000000000000LL ? 0 : a;
}

// FP64 residual c = b - Psi x (blocks of Eq. (3)) over the stage rows of one
// residual task (kResChunk consecutive stages of one system) per CTA. The task's
// rows, all stages in one list, go to the warps in groups of 32, one row per
// lane, since an FP64 instruction costs its issue slot whether a lane has a row
// or not. Each lane forms, for its row i of stage j,
//   (E_{j-1} x_{j-1} + D_j x_j + E_j^T x_{j+1} + G_j^T x_g)_i
// from the blocks in global memory (lower triangle of D_j by symmetry) as
// three independent FMA chains, with the x rows of the task (and its neighbour
// stages') staged in shared memory, so Psi is read once. A matrix-vector
// product does 2 flop per 8-byte element, more than the FP64 units sustain
// at full HBM bandwidth on this part, so the kernel keeps FP64 work to the
// products themselves: the row sums of |Psi| (for eta) are only formed when
// `norms` is set (the first sweep of a refinement; they depend on the matrix
// alone). Per task it writes the g-row partials sum_j G_j x_j (m x nr),
// max|c|, max|x|, max|b| and, with `norms`, the largest stage-row sum of
// |Psi| and the |G| sums of the g rows, each the warps' partials in warp order;
// k_residual_final combines them per system. MB: registers for up to MB arrow rows.
//
// Bound by the FP64 pipe (75 % busy; 1824 tasks of mixed sizes). With one warp
// per task, three rows per lane, it was bound by the latency of its loads: 150
// -> 27 us a sweep for one system of N = 256, n = 32, m = 8 (32 warps on the
// whole chip), 2.7 -> 1.9 ms for 2048 uneven systems.
template <int MB>
__global__ void __launch_bounds__(256, MB <= 8 ? 3 : 2) k_residual(const LevelDesc* __restrict__ descs,
                                                  const ResTask* __restrict__ tasks,
                                                  const double* __restrict__ uD, const double* __restrict__ uE,
                                                  const double* __restrict__ uG, const double* __restrict__ b,
                                                  int ldb, const double* __restrict__ x, int ldx, double* c,
                                                  int nr, double* parts, const int* skip, int norms,
                                                  int xs_doubles) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  const int t = blockIdx.x;
  const ResTask tk = tasks[t];
  const LevelDesc& d = descs[tk.desc];
  if (skip && skip[d.sys]) return;
  const int n = d.n, m = d.m, N = d.N;
  if (!dbg_ok(tk.j0 >= 0 && tk.j0 < d.N && d.n <= kMaxN && d.m <= MB && tk.part < tk.nparts &&
                  (kResChunk + 2) * n <= xs_doubles,
              d))
    return;
  const int j0 = tk.j0, cnt = min(kResChunk, N - j0), rows = cnt * n;
  const size_t nn = (size_t)n * n, mn = (size_t)m * n;
  const double* D = uD + d.offD;
  const double* E = uE ? uE + d.offE : nullptr;
  const double* G = m ? uG + d.offG : nullptr;
  const Div by(n);
  // x rows of stages j0 - 1 .. j0 + cnt: xs[(s + 1) n + k] is row k of stage j0 + s
  // (zero outside 0..N-1)
  double* const xs = reinterpret_cast<double*>(smraw);
  // the warps' partials: kMaxM x kRhsChunk g rows, maxima and sums
  double* const wpart = xs + xs_doubles;
  double* const part = wpart + wid * kResWarpDoubles;
  long long mr = 0, mx = 0, mb = 0;
  float mrow = 0.0f;
  for (int col = 0; col < nr; ++col) {
    const double xg_l = lane < m ? x[(size_t)(d.rowG + lane) * ldx + col] : 0.0;  // x_g, lane q holds row q
    double gacc[MB];  // this lane's terms of sum_j G_j x_j per g row
#pragma unroll
    for (int q = 0; q < MB; ++q) gacc[q] = 0.0;
    if (col) __syncthreads();  // the previous column is done with xs
    {
      const long long r0 = (long long)(j0 - 1) * n;  // first row, below 0 at the system's start
      for (int e = tid; e < (cnt + 2) * n; e += nt) {
        const long long r = r0 + e;
        xs[e] = r >= 0 && r < (long long)N * n ? x[(size_t)(d.offB + r) * ldx + col] : 0.0;
      }
    }
    __syncthreads();
    for (int g0 = wid * 32; g0 < rows; g0 += nw * 32) {
      const bool ok = g0 + lane < rows;
      const int r = ok ? g0 + lane : 0, s = by(r), i = r - s * n, j = j0 + s;
      const double* Dj = D + (size_t)j * nn;
      const bool hp = E && j > 0, hn = E && j < N - 1;
      const double* Ep = hp ? E + (size_t)(j - 1) * nn : D;
      const double* En = hn ? E + (size_t)j * nn : D;
      const double* xp = xs + (size_t)s * n;  // x_{j-1}, x_j, x_{j+1} follow at n apart
      // E_{j-1} x_{j-1}, D_j x_j (lower triangle by symmetry) and E_j^T
      // x_{j+1} as three independent chains over k, then summed
      double aP = 0.0, aD = 0.0, aN = 0.0;
      float rs = 0.0f;
#pragma unroll 4
      for (int k = 0; k < n; ++k) {
        const double dv = k <= i ? Dj[i * n + k] : Dj[k * n + i];
        const double pv = hp ? Ep[i * n + k] : 0.0, qv = hn ? En[k * n + i] : 0.0;
        aP = fma(pv, xp[k], aP);
        aD = fma(dv, xp[n + k], aD);
        aN = fma(qv, xp[2 * n + k], aN);
        if (norms) rs += (abs_lo(dv) + abs_lo(pv)) + abs_lo(qv);
      }
      double acc = (aP + aD) + aN;
      const double xo = ok ? xp[n + i] : 0.0;  // this row's x
      if (m) {
        const double* Gj = G + (size_t)j * mn;
#pragma unroll
        for (int g = 0; g < MB; ++g) {
          if (g >= m) break;  // warp-uniform; full unrolling keeps gacc in registers
          const double xq = __shfl_sync(0xffffffffu, xg_l, g);
          const double gv = Gj[g * n + i];
          acc = fma(gv, xq, acc);
          gacc[g] = fma(gv, xo, gacc[g]);  // xo = 0 on lanes without a row
          if (norms) rs += abs_lo(gv);
        }
      }
      if (ok) {
        const size_t row = (size_t)(d.offB + (long long)j * n + i);
        const double bv = b ? b[row * ldb + col] : 0.0, res = bv - acc;
        c[row * kRhsChunk + col] = res;
        mr = max(mr, abs_order(res)); mb = max(mb, abs_order(bv)); mx = max(mx, abs_order(xo));
        if (norms) mrow = fmaxf(mrow, rs);
      }
    }
    // g-row partials of this column: the lanes halve the rows between them at each
    // step of the tree while there are rows to halve, MB + log2(32 / MB) - 1 FP64
    // additions a warp instead of five a row (with eight warps to a task those
    // were a quarter of its FP64 instructions: a sweep of 512 systems of N = 256,
    // n = 32, m = 8 took 2255 us, 1875 with this and the maxima in integers)
    if (m) {
      int q = 0;  // the row this lane ends with
#pragma unroll
      for (int o = 16, left = MB; o > 0; o >>= 1) {
        const bool up = lane & o;
        if (left > 1) {
          left >>= 1;
          q = 2 * q + (up ? 1 : 0);
#pragma unroll
          for (int i = 0; i < MB / 2; ++i) {
            if (i >= left) break;
            const double send = up ? gacc[i] : gacc[i + left], keep = up ? gacc[i + left] : gacc[i];
            gacc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
          }
        } else {
          gacc[0] += __shfl_xor_sync(0xffffffffu, gacc[0], o);
        }
      }
      if (lane % (32 / MB) == 0 && q < m) part[q * kRhsChunk + col] = gacc[0];
    }
  }
  float gab = 0.0f;  // |G| sum of g row `lane` (lane < m) over the warp's stages
  if (norms && m && lane < m)
    for (int j = j0 + wid; j < j0 + cnt; j += nw) {
      const double* Gj = G + (size_t)j * mn;
      for (int i = 0; i < n; ++i) gab += abs_lo(Gj[lane * n + i]);
    }
  for (int o = 16; o > 0; o >>= 1) {
    mr = max(mr, __shfl_xor_sync(0xffffffffu, mr, o));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
    if (norms) mrow = fmaxf(mrow, __shfl_xor_sync(0xffffffffu, mrow, o));
  }
  double* const pm = part + kMaxM * kRhsChunk;
  if (lane == 0) {
    pm[0] = __longlong_as_double(mr); pm[1] = __longlong_as_double(mx); pm[2] = __longlong_as_double(mb);
    if (norms) pm[3] = (double)mrow;
  }
  if (norms && lane < m) pm[4 + lane] = (double)gab;
  __syncthreads();
  double* const slot = parts + (size_t)t * kResPartDoubles;
  for (int e = tid; e < m * nr; e += nt) {
    const int q = e / nr, o = q * kRhsChunk + (e - q * nr);
    double v = wpart[o];
    for (int w = 1; w < nw; ++w) v += wpart[w * kResWarpDoubles + o];
    slot[o] = v;
  }
  if (tid < (norms ? 4 + m : 3)) {
    const double* const wm = wpart + kMaxM * kRhsChunk + tid;
    double v = wm[0];
    for (int w = 1; w < nw; ++w) {
      const double u = wm[w * kResWarpDoubles];
      v = tid < 4 ? fmax(v, u) : v + u;
    }
    slot[kMaxM * kRhsChunk + tid] = v;
  }
}

// Finish the g rows of one system from the chunk partials, then eta and the
// stop flag (`stall`: the fallback is enabled, flag 3 below): 1 when eta <= tol, 2 when eta is at the rounding level of the
// FP64 residual (kEtaFloor) and the sweep cut the previous sweep's eta by
// less than 10 % (refinement has reached its floor; above that level a slow
// sweep is not taken as the end, since the normwise eta of an
// ill-conditioned system need not fall monotonically); 3 (only with `stall`)
// when eta is above that level and the sweep did not halve it (refinement
// stalls: the system is handed to the preconditioned conjugate-gradient
// fallback); a stopped system skips the remaining sweeps.
constexpr double kEtaFloor = 4.0 * 1.1102230246251565e-16;  // 4 u
__global__ void k_residual_final(const LevelDesc* __restrict__ descs, const int* __restrict__ sys_desc,
                                 const int* __restrict__ part0, const double* __restrict__ uG,
                                 const double* __restrict__ uR, const double* __restrict__ b, int ldb,
                                 const double* __restrict__ x, int ldx, double* c, int nr,
                                 const double* __restrict__ parts, double tol, double* eta_out,
                                 const double* __restrict__ eta_prev, int* converged, int stall) {
  __shared__ double red[4][256];
  __shared__ double gsum[kMaxM];
  const int s = blockIdx.x;
  const LevelDesc& d = descs[sys_desc[s]];
  if (converged && converged[s]) {  // keeps the eta of its converging sweep
    if (threadIdx.x == 0 && eta_prev) eta_out[s] = eta_prev[s];
    return;
  }
  const int m = d.m;
  const int p0 = part0[s], np = (d.N + kResChunk - 1) / kResChunk;
  const double* R = m ? uR + d.offR : nullptr;
  double mr = 0.0, mx = 0.0, mb = 0.0, mrow = 0.0;
  for (int p = threadIdx.x; p < np; p += blockDim.x) {
    const double* pm = parts + (size_t)(p0 + p) * kResPartDoubles + kMaxM * kRhsChunk;
    mr = fmax(mr, pm[0]); mx = fmax(mx, pm[1]); mb = fmax(mb, pm[2]); mrow = fmax(mrow, pm[3]);
  }
  // a warp per g row, its lanes over the chunks
  const int lane = threadIdx.x & 31;
  auto warp_sum = [](double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  for (int q = threadIdx.x >> 5; q < m; q += blockDim.x >> 5) {
    double ga = 0.0;
    for (int p = lane; p < np; p += 32) ga += parts[(size_t)(p0 + p) * kResPartDoubles + kMaxM * kRhsChunk + 4 + q];
    if (lane < m) ga += fabs(lane <= q ? R[q * m + lane] : R[lane * m + q]);
    ga = warp_sum(ga);
    if (lane == 0) gsum[q] = ga;
  }
  __syncthreads();
  for (int e = threadIdx.x >> 5; e < m * nr; e += blockDim.x >> 5) {
    const int q = e / nr, col = e - q * nr;
    const size_t row = (size_t)(d.rowG + q);
    const double bv = b ? b[row * ldb + col] : 0.0, xv = x[row * ldx + col];
    double acc = 0.0;
    for (int p = lane; p < np; p += 32) acc += parts[(size_t)(p0 + p) * kResPartDoubles + q * kRhsChunk + col];
    if (lane < m) acc = fma(lane <= q ? R[q * m + lane] : R[lane * m + q], x[(size_t)(d.rowG + lane) * ldx + col], acc);
    const double r = bv - warp_sum(acc);
    if (lane == 0) c[row * kRhsChunk + col] = r;
    mr = fmax(mr, fabs(r));
    mb = fmax(mb, fabs(bv));
    mx = fmax(mx, fabs(xv));
  }
  for (int q = threadIdx.x; q < m; q += blockDim.x) mrow = fmax(mrow, gsum[q]);
  red[0][threadIdx.x] = mr; red[1][threadIdx.x] = mx; red[2][threadIdx.x] = mb; red[3][threadIdx.x] = mrow;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w)
      for (int q = 0; q < 4; ++q) red[q][threadIdx.x] = fmax(red[q][threadIdx.x], red[q][threadIdx.x + w]);
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double eta = red[0][0] / (red[3][0] * red[1][0] + red[2][0]);
    eta_out[s] = eta;
    // stop: 1 = eta <= tol; 2 = eta is at the rounding level of the FP64
    // residual (<= 4 u) and this sweep cut it by less than 10 %
    if (converged) {
      if (eta <= tol) converged[s] = 1;
      else if (tol >= 0.0 && eta_prev && eta <= kEtaFloor && eta > 0.9 * eta_prev[s]) converged[s] = 2;
      else if (stall && eta_prev && eta > kEtaFloor && eta > 0.5 * eta_prev[s]) converged[s] = 3;
    }
  }
}

// Gradients of a loss L(x), x = Psi^{-1} b, with respect to the stored
// blocks, given x and bbar = Psi^{-1} xbar (xbar = dL/dx): dPsi = -bbar x^T
// restricted to the blocks, each symmetric pair of entries perturbed
// together, summed over the right-hand sides:
//   dD_j[r][c] = -(bbar_r x_c + bbar_c x_r) (r > c), -bbar_r x_r (r = c), 0 above
//   dE_j       = -(bbar_{j+1} x_j^T + x_{j+1} bbar_j^T)
//   dG_j       = -(bbar_g x_j^T + x_g bbar_j^T),   dR like dD on the g rows.
__global__ void k_adjoint_grad(const LevelDesc* __restrict__ descs, const ResTask* __restrict__ tasks,
                               const double* __restrict__ x, int ldx, const double* __restrict__ xb,
                               int ldxb, int nr, double* dD, double* dE, double* dG, double* dR) {
  const ResTask tk = tasks[blockIdx.x];
  const LevelDesc& d = descs[tk.desc];
  const int n = d.n, m = d.m, N = d.N;
  const int j1 = min(tk.j0 + kResChunk, N);
  const size_t nn = (size_t)n * n, mn = (size_t)m * n;
  auto xr = [&](long long row, int c) { return x[(size_t)row * ldx + c]; };
  auto br = [&](long long row, int c) { return xb[(size_t)row * ldxb + c]; };
  // Every element costs two FP64 fmas per right-hand side, issued by every
  // lane alike (a predicated-off FP64 instruction still takes its issue
  // slot): v = fma(-a_r, b_c, fma(-a'_c, b'_r, v)). On a symmetric block's
  // diagonal the second term's factor is zeroed by an integer select (the
  // entry is one parameter: -bbar_r x_r); above it the stored value is 0.
  auto sym = [&](long long r0, long long c0, int r, int c) {  // dD / dR entry (r, c)
    double v = 0.0;
    for (int q = 0; q < nr; ++q) {
      const double bc = __longlong_as_double(c == r ? 0LL : __double_as_longlong(br(c0 + c, q)));
      v = fma(-br(r0 + r, q), xr(c0 + c, q), fma(-bc, xr(r0 + r, q), v));
    }
    return c > r ? 0.0 : v;
  };
  for (int j = tk.j0; j < j1; ++j) {
    const long long rj = d.offB + (long long)j * n;
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
      const int r = e / n, c = e - r * n;
      dD[d.offD + (size_t)j * nn + e] = sym(rj, rj, r, c);
    }
    if (j < N - 1)
      for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
        const int r = e / n, c = e - r * n;
        double v = 0.0;
        for (int q = 0; q < nr; ++q) v = fma(-br(rj + n + r, q), xr(rj + c, q), fma(-xr(rj + n + r, q), br(rj + c, q), v));
        dE[d.offE + (size_t)j * nn + e] = v;
      }
    for (int e = threadIdx.x; e < m * n; e += blockDim.x) {
      const int r = e / n, c = e - r * n;
      double v = 0.0;
      for (int q = 0; q < nr; ++q) v = fma(-br(d.rowG + r, q), xr(rj + c, q), fma(-xr(d.rowG + r, q), br(rj + c, q), v));
      dG[d.offG + (size_t)j * mn + e] = v;
    }
  }
  if (tk.part == 0)
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
      const int r = e / m, c = e - r * m;
      dR[d.offR + e] = sym(d.rowG, d.rowG, r, c);
    }
}

// ---------------------------------------------------------------------------
// Fallback of iterative refinement: preconditioned conjugate gradients on
// Psi x = b (Psi is SPD), preconditioned by the mixed factor, for the systems
// whose refinement stalled (flag 3) or ran out of sweeps (flag 0), as
// proposed for GMRES/CG-based refinement with a low-precision factor
// (Carson and Higham, SIAM J. Sci. Comput. 40, 2018). Vectors are FP64 with
// leading dimension kRhsChunk; per system and right-hand side the scalars rho
// and p^T q live in small device arrays, so the iteration needs no host
// synchronization.
// ---------------------------------------------------------------------------

// out[s][q] = sum over the system's rows of u[row][q] v[row][q] (rows offB ..
// offB + N n + m, contiguous), for the systems whose mask entry is set; a
// fixed-order tree over the CTA
__global__ void k_sys_dot(const LevelDesc* __restrict__ descs, const int* __restrict__ sys_desc,
                          const int* __restrict__ conv, const double* __restrict__ u, const double* __restrict__ v,
                          int nr, double* out) {
  __shared__ double red[256];
  const int s = blockIdx.x;
  if (conv[s] == 1 || conv[s] == 2) return;  // converged: not in the fallback
  const LevelDesc& d = descs[sys_desc[s]];
  const long long r0 = d.offB, rows = (long long)d.N * d.n + d.m;
  for (int q = 0; q < nr; ++q) {
    double a = 0.0;
    for (long long r = threadIdx.x; r < rows; r += blockDim.x)
      a = fma(u[(size_t)(r0 + r) * kRhsChunk + q], v[(size_t)(r0 + r) * kRhsChunk + q], a);
    red[threadIdx.x] = a;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
      if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
      __syncthreads();
    }
    if (threadIdx.x == 0) out[(size_t)s * kRhsChunk + q] = red[0];
    __syncthreads();
  }
}

// mode 0: alpha = rho / (p^T Psi p) with Qn = -Psi p and pq = p^T Qn:
//         x += alpha p, r += alpha Qn (i.e. r -= alpha Psi p)
// mode 1: beta = rho_new / rho_old: p = z + beta p
// over the stage rows of each residual task (the g rows with the system's
// first task); systems outside the fallback are skipped
__global__ void k_pcg_update(const LevelDesc* __restrict__ descs, const ResTask* __restrict__ tasks,
                             const int* __restrict__ conv, int mode, int nr, double* x, int ldx, double* rr,
                             const double* __restrict__ qn, double* p, const double* __restrict__ z,
                             const double* __restrict__ num, const double* __restrict__ den) {
  const ResTask tk = tasks[blockIdx.x];
  const LevelDesc& d = descs[tk.desc];
  const int cs = conv[d.sys];
  if (cs == 1 || cs == 2) return;
  const int j1 = min(tk.j0 + kResChunk, d.N);
  const long long row0 = d.offB + (long long)tk.j0 * d.n;
  const int rows = (j1 - tk.j0) * d.n + (tk.part == 0 ? 0 : 0);
  auto one = [&](long long row, int col) {
    const size_t sc = (size_t)d.sys * kRhsChunk + col, i = (size_t)row * kRhsChunk + col;
    const double dn = den[sc];
    if (mode == 0) {
      const double alpha = dn != 0.0 ? -num[sc] / dn : 0.0;
      x[(size_t)row * ldx + col] = fma(alpha, p[i], x[(size_t)row * ldx + col]);
      rr[i] = fma(alpha, qn[i], rr[i]);
    } else {
      const double beta = dn != 0.0 ? num[sc] / dn : 0.0;
      p[i] = fma(beta, p[i], z[i]);
    }
  };
  for (int e = threadIdx.x; e < rows * nr; e += blockDim.x) one(row0 + e / nr, e % nr);
  if (tk.part == 0)
    for (int e = threadIdx.x; e < d.m * nr; e += blockDim.x) one(d.rowG + e / nr, e % nr);
}

// fallback mask for the solves and the matrix products: skip[s] = 1 unless
// the system's refinement stalled or did not converge
__global__ void k_pcg_mask(const int* __restrict__ conv, int* skip, int count) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < count) skip[s] = (conv[s] == 1 || conv[s] == 2) ? 1 : 0;
}

// Identity pivot blocks and corner for every system of a batch (synthetic
// inputs of the autotuner: the kernels' run time does not depend on values).
__global__ void k_fill_identity(const LevelDesc* __restrict__ descs, const int* __restrict__ sys_desc,
                                double* D, double* R) {
  const LevelDesc& d = descs[sys_desc[blockIdx.x]];
  const long long nn = (long long)d.n * d.n, tot = (long long)d.N * nn;
  for (long long e = threadIdx.x; e < tot; e += blockDim.x) {
    const long long r = e % nn;
    D[d.offD + e] = (r % (d.n + 1) == 0) ? 1.0 : 0.0;
  }
  for (int e = threadIdx.x; e < d.m * d.m; e += blockDim.x) R[d.offR + e] = (e % (d.m + 1) == 0) ? 1.0 : 0.0;
}

// Bordered inputs for a fused factor-and-solve pass: Gb_j = [G_j; b_j^T],
// Rb = [[R, b_g], [b_g^T, 0]]; db holds the bordered level-1 descriptors (m + 1
// arrow rows, offG and offR into Gb and Rb). Grid: x strides over a system's
// elements (one stage's row per 32-lane chunk), y = system.
__global__ void k_border(const LevelDesc* __restrict__ descs, const int* __restrict__ sys_desc,
                         const double* __restrict__ G, const double* __restrict__ R, const double* __restrict__ b,
                         int ldb, double* Gb, double* Rb, int j0, int j1, int corner) {
  const LevelDesc& d = descs[sys_desc[blockIdx.y]];
  const int n = d.n, mb = d.m, m = mb - 1, N = d.N;
  const long long offG = d.offGu, offR = d.offRu;  // the caller's arrays
  const int je = min(j1, N);
  const long long rows = je > j0 ? (long long)(je - j0) * mb : 0;  // rows of Gb of stages [j0, je)
  const long long base = (long long)j0 * mb * n;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < rows * n;
       e += (long long)gridDim.x * blockDim.x) {
    const long long row = e / n, j = j0 + row / mb;
    const int r = (int)(row - (j - j0) * mb), c = (int)(e - row * n);
    Gb[d.offG + base + e] = r < m ? G[offG + (j * m + r) * n + c] : b[(size_t)(d.offB + j * n + c) * ldb];
  }
  if (corner && blockIdx.x == 0)
    for (int e = threadIdx.x; e < mb * mb; e += blockDim.x) {
      const int r = e / mb, c = e - r * mb;
      double v = 0.0;
      if (r < m && c < m) v = R[offR + r * m + c];
      else if (r == m && c < m) v = b[(size_t)(d.rowG + c) * ldb];
      else if (c == m && r < m) v = b[(size_t)(d.rowG + r) * ldb];
      Rb[d.offR + e] = v;
    }
}

// Raises a kernel's dynamic shared memory limit to `bytes` on the current
// device (never lowers it: a captured graph replays earlier launches of the
// same kernel, which may need more than the latest one). The attribute is
// per device, so the record of what was granted is keyed by (device, kernel).
int set_smem(const void* fn, size_t bytes) {
  static std::mutex mu;
  static std::unordered_map<const void*, size_t> granted[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return (int)cudaErrorInvalidDevice;
  if (dev < 0 || dev >= kMaxDevices)  // not recorded: set every time
    return (int)cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  std::lock_guard<std::mutex> lock(mu);
  size_t& g = granted[dev][fn];
  if (bytes <= g) return 0;
  const int e = (int)cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (!e) g = bytes;
  return e;
}

}  // namespace

size_t factor_smem_bytes(int n, int m, int mixed, int fill) {
  return (size_t)(mixed ? fac_layout(n, m, 4, fill != 0).total : cta_layout(n, m, fill != 0).total);
}

int debug_info(Info* out, int clear) {
#ifdef KKT_DEBUG
  if (cudaMemcpyFromSymbol(out, g_debug_info, sizeof(Info)) != cudaSuccess) return 1;
  if (clear) {
    const Info zero{};
    if (cudaMemcpyToSymbol(g_debug_info, &zero, sizeof(Info)) != cudaSuccess) return 1;
  }
#else
  *out = Info{};
  (void)clear;
#endif
  return 0;
}

size_t factor_w_slice_bytes(int n, int m, int mixed, int fill) {
  return (size_t)fac_layout_w(n, m, mixed ? 4 : 8, fill != 0).total;
}

int persist_occupancy(int mixed, size_t smem, int threads) {
  const void* fn = mixed ? (const void*)k_factor_persist<float> : (const void*)k_factor_persist<double>;
  if (set_smem(fn, smem)) return 0;
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, smem) != cudaSuccess) return 0;
  return occ;
}

int launch_factor_persist(const LevelDesc* d, const Task* t, const PItem* items, int nitems, const PCons* cons,
                          int* ready, int mixed, const double* D, const double* E, const double* G,
                          const double* R, Info* info, int grid, int threads, size_t smem, int slice,
                          long long wait_cycles, void* stream) {
  if (nitems <= 0) return 0;
  const void* fn = mixed ? (const void*)k_factor_persist<float> : (const void*)k_factor_persist<double>;
  int e = set_smem(fn, smem);
  if (e) return e;
  cudaStream_t st = (cudaStream_t)stream;
  if (mixed)
    k_factor_persist<float><<<grid, threads, smem, st>>>(d, t, items, nitems, cons, ready, D, E, G, R, info, slice,
                                                         wait_cycles);
  else
    k_factor_persist<double><<<grid, threads, smem, st>>>(d, t, items, nitems, cons, ready, D, E, G, R, info, slice,
                                                          wait_cycles);
  return (int)cudaGetLastError();
}

size_t solve_smem_bytes(int n, int m, int single, int fill) {
  return (size_t)sol_layout(n, m, single ? 4 : 8, fill != 0).total;
}

int launch_factor_w(const LevelDesc* d, const Task* t, int ntasks, int maxn, int maxm, int mixed,
                    const double* D, const double* E, const double* G, const double* R, Info* info,
                    void* stream, double* b, int ldb, int fill) {
  if (ntasks <= 0) return 0;
  const int slice = fac_layout_w(maxn, maxm, mixed ? 4 : 8, fill != 0).total;
  const int wpc = std::max(1, std::min(8, (200 * 1024) / slice));  // tasks (warps) per CTA
  const size_t sm = (size_t)wpc * slice;
  const void* fn = mixed ? (const void*)k_factor_w<float> : (const void*)k_factor_w<double>;
  int e = set_smem(fn, sm);
  if (e) return e;
  const int grid = (ntasks + wpc - 1) / wpc;
  if (mixed)
    k_factor_w<float><<<grid, 32 * wpc, sm, (cudaStream_t)stream>>>(d, t, ntasks, D, E, G, R, info, slice, b, ldb);
  else
    k_factor_w<double><<<grid, 32 * wpc, sm, (cudaStream_t)stream>>>(d, t, ntasks, D, E, G, R, info, slice, b, ldb);
  return (int)cudaGetLastError();
}

// Tensor-core Schur products for a mixed launch of blocks n >= 32 when the
// pivot-buffer region can stage the operand (Rs rows of K) and the packed
// product triangle, and the layout spans the 128 operand rows the MMA
// addresses; 0 otherwise.
int tc_mode_for(int tc, int mixed, int pair, int maxn, int maxm, int fill) {
  if (!tc || !mixed || pair || maxn < 32) return 0;
  const FacLayout L = fac_layout(maxn, maxm, 4, fill != 0);
  const int kin = tc == 2 ? 16 : 8, eb = tc == 2 ? 2 : 4;
  const long Kp = (maxn + kin - 1) / kin * kin;
  const long cap = L.oZ - L.oDfac;
  const bool fits = L.Rs <= 128 && (long)L.Rs * Kp * eb <= cap && (long)L.Rs * (L.Rs + 1) / 2 * 4 <= cap &&
                    128 * Kp * eb <= L.total;
  return fits ? tc : 0;
}

int launch_factor(const LevelDesc* d, const Task* t, int ntasks, int maxn, int maxm, int mixed, int pair,
                  const double* D, const double* E, const double* G, const double* R, Info* info,
                  void* stream, double* b, int ldb, int fill, int top_solve, int tc) {
  if (ntasks <= 0) return 0;
  top_solve = top_solve && b && !mixed;
  const int tcm = tc_mode_for(tc, mixed, pair, maxn, maxm, fill);
  size_t sm = factor_smem_bytes(maxn, maxm, mixed, fill);
  if (top_solve) sm = std::max(sm, solve_smem_bytes(maxn, maxm, 0, fill));
  const void* fn = !mixed ? (b ? (const void*)k_factor_fp64<true> : (const void*)k_factor_fp64<false>)
                   : pair ? (const void*)k_factor<1>
                   : tcm  ? (const void*)k_factor<4, true>
                          : (const void*)k_factor<4>;
  const int e = set_smem(fn, sm);
  if (e) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3((unsigned)(pair ? 2 * ntasks : ntasks));
  cfg.blockDim = dim3(kFactorThreads);
  if (!mixed && !pair) {
    // more tasks than CTAs of 256 threads fit at once, and half as many threads
    // let twice as many tasks share the SMs: their pivot chains then overlap
    // (512 systems of n = 32: 19.1 against 21.9 ms; where shared memory allows two
    // CTAs in either case, n = 48, the larger CTA is faster: 57.6 against 64.9 ms
    // on 4096 uneven systems)
    int dev = 0, sms = 0, o1 = 0, o2 = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o1, fn, kFactorThreads, sm) == cudaSuccess &&
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o2, fn, kFactorThreads / 2, sm) == cudaSuccess &&
        ntasks > o1 * sms && o2 >= 2 * o1)
      cfg.blockDim = dim3(kFactorThreads / 2);
  }
  cfg.dynamicSmemBytes = sm;
  cfg.stream = (cudaStream_t)stream;
  if (pair) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  }
  const int p = pair ? 1 : 0;
  if (!mixed)
    return b ? (int)cudaLaunchKernelEx(&cfg, k_factor_fp64<true>, d, t, D, E, G, R, info, p, b, ldb, top_solve)
             : (int)cudaLaunchKernelEx(&cfg, k_factor_fp64<false>, d, t, D, E, G, R, info, p, b, ldb, top_solve);
  return pair ? (int)cudaLaunchKernelEx(&cfg, k_factor<1>, d, t, D, E, G, R, info, p, 0)
         : tcm ? (int)cudaLaunchKernelEx(&cfg, k_factor<4, true>, d, t, D, E, G, R, info, p, tcm)
               : (int)cudaLaunchKernelEx(&cfg, k_factor<4>, d, t, D, E, G, R, info, p, 0);
}

int factor_clus_size(int ntasks, int maxn, int maxm, int sms) {
  if (ntasks <= 0) return 0;
  const size_t sm = factor_smem_bytes(maxn, maxm, 0, 1);
  if (set_smem((const void*)k_factor_clus<false>, sm)) return 0;
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_factor_clus<false>, kFactorThreads, sm) != cudaSuccess ||
      occ < 1)
    return 0;
  occ = std::min(occ, 2);
  for (int C = 8; C >= 2; C /= 2) {
    if ((long long)C * ntasks > (long long)occ * sms) continue;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(C * ntasks));
    cfg.blockDim = dim3(kFactorThreads);
    cfg.dynamicSmemBytes = sm;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int ncl = 0;
    if (cudaOccupancyMaxActiveClusters(&ncl, k_factor_clus<false>, &cfg) == cudaSuccess && ncl >= ntasks) return C;
  }
  return 0;
}

int launch_factor_clus(const LevelDesc* d, const Task* t, int ntasks, int maxn, int maxm, int C, const double* D,
                       const double* E, const double* G, Info* info, void* stream, double* b, int ldb) {
  if (ntasks <= 0) return 0;
  if (C < 2 || C > 8) return (int)cudaErrorInvalidValue;
  const size_t sm = factor_smem_bytes(maxn, maxm, 0, 1);
  const int e = set_smem(b ? (const void*)k_factor_clus<true> : (const void*)k_factor_clus<false>, sm);
  if (e) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(C * ntasks));
  cfg.blockDim = dim3(kFactorThreads);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = (cudaStream_t)stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return b ? (int)cudaLaunchKernelEx(&cfg, k_factor_clus<true>, d, t, D, E, G, info, b, ldb, C)
           : (int)cudaLaunchKernelEx(&cfg, k_factor_clus<false>, d, t, D, E, G, info, b, ldb, C);
}

// The substitution kernel of a launch of `grid` CTAs: the dense one (64 registers,
// four CTAs per SM where shared memory allows) if the launch has more CTAs than the
// other one (128 registers, loads a stage ahead, two columns a warp) holds at once.
// Alone against dense, us: 1000 systems of N = 40, m = 4, n = 17 796, 472 (one
// column) and 2289, 1686 (eight), n = 33 1885, 1168, n = 41, sixteen 12793, 12942;
// 400 systems, m = 0, n = 33 929, 549.
template <typename F>
static F pick_solve(F alone, F dense, unsigned grid, size_t sm, int* err) {
  int dev = 0, sms = 0, o1 = 0, o2 = 0;
  *err = set_smem((const void*)alone, sm);
  if (*err) return alone;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || grid <= (unsigned)sms)
    return alone;
  if (set_smem((const void*)dense, sm) == 0 &&
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o1, alone, kSolveThreads, sm) == cudaSuccess &&
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o2, dense, kSolveThreads, sm) == cudaSuccess && o2 > o1 &&
      grid > (unsigned)(o1 * sms))
    return dense;
  return alone;
}

int launch_forward(const LevelDesc* d, const Task* t, int ntasks, int maxn, int maxm, int single,
                   double* b, int ldb, int nrhs, const int* skip, void* stream, int fwd_done, int split, int fill) {
  if (ntasks <= 0) return 0;
  const size_t sm = solve_smem_bytes(maxn, maxm, single, fill);
  split = std::max(1, std::min(split, nrhs));
  const unsigned grid = (unsigned)(ntasks * split);
  int e = 0;
  auto* const fn = single ? pick_solve(k_forward<float, kAlone>, k_forward<float, kDense>, grid, sm, &e)
                          : pick_solve(k_forward<double, kAlone>, k_forward<double, kDense>, grid, sm, &e);
  if (e) return e;
  fn<<<grid, kSolveThreads, sm, (cudaStream_t)stream>>>(d, t, b, ldb, nrhs, skip, fwd_done, split);
  return (int)cudaGetLastError();
}

int launch_backward(const LevelDesc* d, const Task* t, int ntasks, int maxn, int maxm, int single,
                    double* b, int ldb, int nrhs, const int* skip, void* stream, int split, int fill) {
  if (ntasks <= 0) return 0;
  const size_t sm = solve_smem_bytes(maxn, maxm, single, fill);
  split = std::max(1, std::min(split, nrhs));
  const unsigned grid = (unsigned)(ntasks * split);
  int e = 0;
  auto* const fn = single ? pick_solve(k_backward<float, kAlone>, k_backward<float, kDense>, grid, sm, &e)
                          : pick_solve(k_backward<double, kAlone>, k_backward<double, kDense>, grid, sm, &e);
  if (e) return e;
  fn<<<grid, kSolveThreads, sm, (cudaStream_t)stream>>>(d, t, b, ldb, nrhs, skip, split);
  return (int)cudaGetLastError();
}

int launch_backward_chain(const LevelDesc* d, const Task* t, const ChainPlan& cp, int* ctr, int maxn, int maxm,
                          int single, double* b, int ldb, int nrhs, const int* skip, Info* info, long long wait,
                          int unmet, int sms, void* stream) {
  if (cp.nlev <= 0) return 0;
  if (cp.nlev > kChainMax) return (int)cudaErrorInvalidValue;
  const size_t sm = solve_smem_bytes(maxn, maxm, single, 1);
  const void* fn = single ? (const void*)k_backward_chain<float> : (const void*)k_backward_chain<double>;
  int e = set_smem(fn, sm);
  if (e) return e;
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, kSolveThreads, sm) != cudaSuccess || occ < 1)
    return (int)cudaErrorInvalidConfiguration;
  const int total = cp.end[cp.nlev - 1];
  const unsigned grid = (unsigned)std::max(1, std::min(total, occ * std::max(sms, 1)));
  const cudaError_t me = cudaMemsetAsync(ctr, 0, sizeof(int) * (cp.nlev + 1), (cudaStream_t)stream);
  if (me != cudaSuccess) return (int)me;
  if (single)
    k_backward_chain<float><<<grid, kSolveThreads, sm, (cudaStream_t)stream>>>(d, t, cp, ctr, b, ldb, nrhs, skip,
                                                                               info, wait, unmet ? 1 : 0);
  else
    k_backward_chain<double><<<grid, kSolveThreads, sm, (cudaStream_t)stream>>>(d, t, cp, ctr, b, ldb, nrhs, skip,
                                                                                info, wait, unmet ? 1 : 0);
  return (int)cudaGetLastError();
}

// warp-per-task substitutions (blocks n <= kWarpMaxN)
int launch_solve_w(bool backward, const LevelDesc* d, const Task* t, int ntasks, int maxn, int maxm, int single,
                   double* b, int ldb, int nrhs, const int* skip, void* stream, int fwd_done, int fill) {
  if (ntasks <= 0) return 0;
  const int slice = (int)solve_smem_bytes(maxn, maxm, single, fill);
  const int wpc = std::max(1, std::min(8, (200 * 1024) / slice));
  const size_t sm = (size_t)wpc * slice;
  const void* fn = backward ? (single ? (const void*)k_backward_w<float> : (const void*)k_backward_w<double>)
                            : (single ? (const void*)k_forward_w<float> : (const void*)k_forward_w<double>);
  int e = set_smem(fn, sm);
  if (e) return e;
  const int grid = (ntasks + wpc - 1) / wpc;
  cudaStream_t st = (cudaStream_t)stream;
  if (backward) {
    if (single) k_backward_w<float><<<grid, 32 * wpc, sm, st>>>(d, t, ntasks, b, ldb, nrhs, skip, slice);
    else k_backward_w<double><<<grid, 32 * wpc, sm, st>>>(d, t, ntasks, b, ldb, nrhs, skip, slice);
  } else {
    if (single) k_forward_w<float><<<grid, 32 * wpc, sm, st>>>(d, t, ntasks, b, ldb, nrhs, skip, slice, fwd_done);
    else k_forward_w<double><<<grid, 32 * wpc, sm, st>>>(d, t, ntasks, b, ldb, nrhs, skip, slice, fwd_done);
  }
  return (int)cudaGetLastError();
}

int launch_seq_solve(const LevelDesc* d, const Task* t, int ntasks, int maxn, int maxm, int single, double* b,
                     int ldb, const int* skip, Info* info, long long wait, int unmet, int sms, int uniform,
                     void* stream) {
  if (ntasks <= 0) return 0;
  const int sb = single ? 4 : 8;
  if (maxn < 2 || maxn % 2 || maxn > kMaxN || maxm < 0 || maxm > kMaxM) return (int)cudaErrorInvalidValue;
  const int nbuf = seq_nbuf(maxn, maxm, sb, ntasks, sms);
  const size_t sm = (size_t)seq_slice_bytes(maxn, maxm, sb, nbuf);
  // block sizes with their own unrolled kernel (every system of the launch the same n)
  const int nt = uniform && (maxn == 12 || maxn == 24 || maxn == 32 || maxn == 48) ? maxn : 0;
  const bool two = maxn > 32;
  cudaStream_t st = (cudaStream_t)stream;
  auto go = [&](auto kern) -> int {
    const int e = set_smem((const void*)kern, sm);
    if (e) return e;
    kern<<<ntasks, 32, sm, st>>>(d, t, b, ldb, skip, info, wait, unmet, nbuf);
    return (int)cudaGetLastError();
  };
  if (single) {
    switch (nt) {
      case 12: return go(k_seq_solve<float, 1, 12>);
      case 24: return go(k_seq_solve<float, 1, 24>);
      case 32: return go(k_seq_solve<float, 1, 32>);
      case 48: return go(k_seq_solve<float, 2, 48>);
      default: return two ? go(k_seq_solve<float, 2, 0>) : go(k_seq_solve<float, 1, 0>);
    }
  }
  switch (nt) {
    case 12: return go(k_seq_solve<double, 1, 12>);
    case 24: return go(k_seq_solve<double, 1, 24>);
    case 32: return go(k_seq_solve<double, 1, 32>);
    case 48: return go(k_seq_solve<double, 2, 48>);
    default: return two ? go(k_seq_solve<double, 2, 0>) : go(k_seq_solve<double, 1, 0>);
  }
}

int launch_axpy(const LevelDesc* d, const ResTask* t, int ntasks, double* x, int ldx, const double* c,
                int nr, const int* skip, void* stream) {
  if (ntasks <= 0) return 0;
  k_axpy<<<ntasks, 256, 0, (cudaStream_t)stream>>>(d, t, x, ldx, c, nr, skip);
  return (int)cudaGetLastError();
}

int launch_fill_identity(const LevelDesc* d, const int* sys_desc, int count, double* D, double* R,
                         void* stream) {
  if (count <= 0) return 0;
  k_fill_identity<<<count, 256, 0, (cudaStream_t)stream>>>(d, sys_desc, D, R);
  return (int)cudaGetLastError();
}

int launch_border(const LevelDesc* db, const int* sys_desc, int count, long long max_elems, const double* G,
                  const double* R, const double* b, int ldb, double* Gb, double* Rb, void* stream, int j0, int j1,
                  int corner) {
  if (count <= 0) return 0;
  const long long bx = std::min<long long>(std::max<long long>((max_elems + 255) / 256, 1), 2048);
  k_border<<<dim3((unsigned)bx, (unsigned)count), 256, 0, (cudaStream_t)stream>>>(db, sys_desc, G, R, b, ldb, Gb,
                                                                                  Rb, j0, j1, corner);
  return (int)cudaGetLastError();
}

int launch_sys_dot(const LevelDesc* d, const int* sys_desc, const int* conv, int count, const double* u,
                   const double* v, int nr, double* out, void* stream) {
  if (count <= 0) return 0;
  k_sys_dot<<<count, 256, 0, (cudaStream_t)stream>>>(d, sys_desc, conv, u, v, nr, out);
  return (int)cudaGetLastError();
}

int launch_pcg_update(const LevelDesc* d, const ResTask* t, int ntasks, const int* conv, int mode, int nr,
                      double* x, int ldx, double* r, const double* qn, double* p, const double* z,
                      const double* num, const double* den, void* stream) {
  if (ntasks <= 0) return 0;
  k_pcg_update<<<ntasks, 256, 0, (cudaStream_t)stream>>>(d, t, conv, mode, nr, x, ldx, r, qn, p, z, num, den);
  return (int)cudaGetLastError();
}

int launch_pcg_mask(const int* conv, int* skip, int count, void* stream) {
  if (count <= 0) return 0;
  k_pcg_mask<<<(count + 255) / 256, 256, 0, (cudaStream_t)stream>>>(conv, skip, count);
  return (int)cudaGetLastError();
}

int launch_adjoint_grad(const LevelDesc* d, const ResTask* t, int ntasks, const double* x, int ldx,
                        const double* xb, int ldxb, int nr, double* dD, double* dE, double* dG,
                        double* dR, void* stream) {
  if (ntasks <= 0) return 0;
  k_adjoint_grad<<<ntasks, 256, 0, (cudaStream_t)stream>>>(d, t, x, ldx, xb, ldxb, nr, dD, dE, dG, dR);
  return (int)cudaGetLastError();
}

int launch_residual(const LevelDesc* d, const ResTask* t, int ntasks, const double* D, const double* E,
                    const double* G, const double* b, int ldb, const double* x, int ldx, double* c, int nr,
                    double* parts, const int* skip, int norms, void* stream, int maxn, int maxm) {
  if (ntasks <= 0) return 0;
  const int xs_doubles = (kResChunk + 2) * maxn;
  cudaStream_t st = (cudaStream_t)stream;
  const int nw = std::min(8, (kResChunk * maxn + 31) / 32);  // a warp per 32 rows of a task
  const size_t sm = ((size_t)xs_doubles + nw * kResWarpDoubles) * sizeof(double);
  auto go = [&](auto kern) -> int {
    const int e = set_smem((const void*)kern, sm);
    if (e) return e;
    kern<<<ntasks, 32 * nw, sm, st>>>(d, t, D, E, G, b, ldb, x, ldx, c, nr, parts, skip, norms, xs_doubles);
    return (int)cudaGetLastError();
  };
  if (maxm <= 4) return go(k_residual<4>);
  if (maxm <= 8) return go(k_residual<8>);
  return go(k_residual<kMaxM>);
}

int launch_residual_final(const LevelDesc* d, const int* sys_desc, const int* part0, int count,
                          const double* G, const double* R, const double* b, int ldb, const double* x,
                          int ldx, double* c, int nr, const double* parts, double tol, double* eta_out,
                          const double* eta_prev, int* converged, void* stream, int stall) {
  if (count <= 0) return 0;
  k_residual_final<<<count, 256, 0, (cudaStream_t)stream>>>(d, sys_desc, part0, G, R, b, ldb, x, ldx, c,
                                                            nr, parts, tol, eta_out, eta_prev, converged, stall);
  return (int)cudaGetLastError();
}

}  // namespace kkt
