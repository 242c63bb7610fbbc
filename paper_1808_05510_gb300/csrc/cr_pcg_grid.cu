// Grid-wide Jacobi PCG for the ALS sub-systems (Eq. ALS_linsys, u side;
// Eq. ALS_linsys_v, v side) on voxel grids too large for one thread-block
// cluster's shared memory.  Vectors stream from HBM; every SM takes part.
//
// One persistent cooperative launch runs the whole solve.  Block b owns the
// contiguous rows [b*chunk, (b+1)*chunk).  Each PCG iteration is three
// sweeps separated by a bounded grid barrier (the v side adds one short
// sweep: block a adds column a of the per-block partial X^T p, so that every
// block then reads y = s o X^T p for its data term X diag(s) X^T p):
//   A2a  p = z + beta p_old (z = D^-1 r) and t = (L + cI) p.  Row i needs p on
//        its one-hop neighbourhood, recomputed from z and p_old (p is double
//        buffered), so no barrier separates the p update from the stencil;
//   A2b  q = lam ((L + cI) t + e p) + data(p), and the block's partial <p, q>;
//   B    alpha = rho / <p, q>, x += alpha p, r -= alpha q, z = D^-1 r, and the
//        partials of rho' = <r, z> and |r|^2; four rows per thread and load.
// The operator holds (L + cI)^2; splitting it through t keeps every row's
// loads one hop deep, with the neighbour indices fetched before the values.
// Reads of data that other blocks wrote before the last grid barrier are
// ordinary (L1-cached) loads: the barrier's acquire at GPU scope, taken before
// the block passes its CTA barrier, makes those writes visible, and adjacent
// rows share most of their neighbourhoods in L1.
// Every block adds the per-block partial sums itself, in one fixed order, so
// all blocks hold bit-identical scalars and take identical decisions.
// T = float: float32 vectors and arithmetic with double-float (two-float)
// accumulation of the inner products per thread, float64 between threads;
// T = double: float64 throughout (on GB300 the float64 form is bound by float64
// arithmetic, not by HBM).
// Neighbour tables: a unit-weight graph Laplacian with at most six neighbours
// per row, none further than 32,767 rows away, stores the six distances as
// 16-bit integers (12 B per row instead of 24 B, and L_ii is their count);
// every other matrix keeps 32-bit indices, weights and L_ii.
// Bytes per row and iteration in float32 with the 16-bit table: A2a reads z,
// p_old, the table and writes p, t (28 B); A2b reads t, p, omega, the table and
// writes q (28 B); B reads x, p, r, q, D^-1 and writes x, r, z (32 B): 88 B
// (120 B with 32-bit indices, L_ii, and z formed from r and D^-1 at every
// neighbour, which also took seven gathers more).
// Measured with it against that form (us per iteration, ellipsoidal shells):
// float32 200,160 voxels 38 -> 18, 1.0M 61 -> 26, 3.0M 158 -> 69 (3.8 TB/s of the
// 88 B); float64 1.0M 102 -> 75, 3.0M 267 -> 201.
#include <algorithm>

#include "cr_common.cuh"
#include "cr_df.cuh"
#include "cr_grid_bar.cuh"

namespace cr {

namespace {

// One CTA of 1,024 threads per SM with the 16-bit table; with the general one CTAs of 512, one per SM
// or, from kGTwoRows rows on, two (up to six neighbours; more take 128 registers a thread).  A second
// CTA lengthens the barriers and the sums behind them, and keeps twice the loads in flight: weighted
// grids, us per iteration in float64 with one and with two, 60,000 rows 22 and 27, 500,000 60 and 59,
// 3.0M 466 and 300.
constexpr int kGThreads16 = 1024, kGThreads = 512;
constexpr int kGTwoRows = 500000;
constexpr int kMaxInj = 4096;  // injections of a problem

struct GridPcg {
  DevLap L;
  double lam;
  const double* coef;  // device [2]: c, d of the shifted operator
  int side;            // 0: u side (omega data term), 1: v side (X diag(s) X^T)
  int m;
  const double* s;     // v side [m]
  const int* xr_ptr;   // v side: X by rows (CSR)
  const int* xr_col;
  const double* xr_val;
  const int* xc_ptr;   // v side: X by columns (CSC, rows ascending)
  const int* xc_row;
  const double* xc_val;
  const double* b;     // [n] right side (float64)
  double* x;           // [n] in: x0, out: solution (float64)
  const double* dinv64;  // [n] Jacobi inverse diagonal (float64)
  const double* omt64;   // [n] u side omega (float64)
  void* xs;            // [n] T work: x
  void* rs;            // [n] T: r
  void* p0;            // [n] T: p, two buffers (old / new)
  void* p1;
  void* qs;            // [n] T: q = A_hat p
  void* ts;            // [n] T: t = (L + cI) p
  void* ds;            // [n] T: D^-1
  void* os;            // [n] T: omega (u side)
  void* gs;            // [n] T: L_ii (32-bit table)
  void* zs;            // [n] T: z = D^-1 r
  const uint32_t* idx; // [3 * n] six 16-bit neighbour distances per row (0: none), or null
  double* part;        // [nb * kParts] per-block partial sums
  double* ypart;       // v side [nb * m] per-block partial X^T p
  double* yglob;       // v side [m] y = s o X^T p
  unsigned* bar;       // barrier counter
  int* err;            // barrier timeout flag
  int nb, chunk;
  double tol;
  int maxit;
  PcgStat* stat;
};

constexpr int kParts = 4;  // (p,q), rho, |r|^2, |b|^2

// Accumulator of an inner product: double-float for float32 vectors, double otherwise.
template <class T>
struct Acc;
template <>
struct Acc<float> {
  DF v{0.f, 0.f};
  __device__ void add(float a, float b) { v = df_add(v, df_prod(a, b)); }
  __device__ double get() const { return (double)v.hi + (double)v.lo; }
};
template <>
struct Acc<double> {
  double v = 0.0;
  __device__ void add(double a, double b) { v = fma(a, b, v); }
  __device__ double get() const { return v; }
};

// four consecutive rows of a vector
__device__ __forceinline__ void ld4(float (&v)[4], const float* p) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x;
  v[1] = q.y;
  v[2] = q.z;
  v[3] = q.w;
}
__device__ __forceinline__ void ld4(double (&v)[4], const double* p) {
  const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
  v[0] = a.x;
  v[1] = a.y;
  v[2] = b.x;
  v[3] = b.y;
}
__device__ __forceinline__ void st4(float* p, const float (&v)[4]) {
  *reinterpret_cast<float4*>(p) = float4{v[0], v[1], v[2], v[3]};
}
__device__ __forceinline__ void st4(double* p, const double (&v)[4]) {
  *reinterpret_cast<double2*>(p) = double2{v[0], v[1]};
  *reinterpret_cast<double2*>(p + 2) = double2{v[2], v[3]};
}

// Block sums of NV accumulators in float64 and a fixed tree order; results in out[] of thread 0.
// Float64 adds take 16 issue cycles a warp, so a shuffle tree over every warp costs 2,560 of them per
// value at 1,024 threads: instead 128 threads add eight values each from shared memory.  sh: NV
// blockDim doubles of the kernel's one buffer (a static array in each instantiation came to 49,696 B).
template <class T, int NV>
__device__ __forceinline__ void block_reduce(Acc<T> (&v)[NV], double* sh, double* out) {
  __shared__ double sw[4][NV];
  const int nt = blockDim.x;  // 512 or 1,024
#pragma unroll
  for (int k = 0; k < NV; ++k) sh[k * nt + threadIdx.x] = v[k].get();
  __syncthreads();
  if (threadIdx.x < 128) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double q[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) q[u] = threadIdx.x + 128 * u < nt ? sh[k * nt + threadIdx.x + 128 * u] : 0.0;
      double t = ((q[0] + q[1]) + (q[2] + q[3])) + ((q[4] + q[5]) + (q[6] + q[7]));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
      if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5][k] = t;
    }
  }
  __syncthreads();
  if (threadIdx.x < NV) out[threadIdx.x] = ((sw[0][threadIdx.x] + sw[1][threadIdx.x]) + sw[2][threadIdx.x]) + sw[3][threadIdx.x];
  __syncthreads();
}

// Sums of part[b * kParts + k] over all blocks b, k < NV, in the same order in every block.
template <int NV>
__device__ __forceinline__ void sum_parts(const double* part, int nb, int first, double (&out)[NV]) {
  __shared__ double res[NV];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (w < NV) {
    double t = 0.0;
    for (int b = lane; b < nb; b += 8 * 32) {
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = b + 32 * u < nb ? __ldcg(part + (size_t)(b + 32 * u) * kParts + first + w) : 0.0;
      t += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) res[w] = t;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) out[k] = res[k];
  __syncthreads();
}

// Neighbours of row i (KM slots; -1 = none).  The table is never written during
// the solve: read-only path.  Returns L_ii where the table holds 16-bit distances.
template <bool F16, int KM>
__device__ __forceinline__ int load_nbrs(const GridPcg& a, int i, int (&q)[KM]) {
  if constexpr (F16) {
    const int n = a.L.n;
    int deg = 0;
    uint32_t w[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) w[k] = __ldg(a.idx + (size_t)k * n + i);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const int d = (int)(int16_t)(k & 1 ? w[k >> 1] >> 16 : w[k >> 1] & 0xFFFFu);
      q[k] = d ? i + d : -1;
      deg += d ? 1 : 0;
    }
    return deg;
  } else {
#pragma unroll
    for (int sl = 0; sl < KM; ++sl) q[sl] = sl < a.L.K ? __ldg(a.L.nbr + (size_t)sl * a.L.n + i) : -1;
    return 0;
  }
}

// Row i of (L + cI) v with the neighbours already loaded; vi = v(i), v(l) from the functor.
template <class T, bool F16, int KM, class VF>
__device__ __forceinline__ T shifted_row(const GridPcg& a, const T* gs, int i, const int (&q)[KM], int deg, T c, T vi,
                                         const VF& v) {
  if constexpr (F16) {
    T w[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) w[k] = q[k] >= 0 ? v(q[k]) : (T)0;
    return ((T)deg + c) * vi - (((w[0] + w[1]) + (w[2] + w[3])) + (w[4] + w[5]));
  } else {
    T acc = (gs[i] + c) * vi;
#pragma unroll
    for (int sl = 0; sl < KM; ++sl) {
      if (q[sl] >= 0) {
        const T w = a.L.offw ? (T)__ldg(a.L.offw + (size_t)sl * a.L.n + i) : (T)-1;
        acc = fma(w, v(q[sl]), acc);
      }
    }
    return acc;
  }
}

// f(i, q, deg) over the block's rows.  With the general table two rows per thread
// and step, both rows' neighbours loaded before either row's values, so that each
// thread keeps two rows' loads in flight (the sweeps are bound by memory latency);
// with the 16-bit table one row, which leaves registers for twice the threads.
template <bool F16, int KM, class F>
__device__ __forceinline__ void for_rows(const GridPcg& a, int lo, int hi, const F& f) {
  const int bd = blockDim.x;
  if constexpr (F16) {
    for (int i = lo + threadIdx.x; i < hi; i += bd) {
      int q[KM];
      const int deg = load_nbrs<F16, KM>(a, i, q);
      f(i, q, deg);
    }
  } else {
    for (int i0 = lo + threadIdx.x; i0 < hi; i0 += 2 * bd) {
      const int i1 = i0 + bd;
      int q0[KM], q1[KM];
      load_nbrs<F16, KM>(a, i0, q0);
      if (i1 < hi) load_nbrs<F16, KM>(a, i1, q1);
      f(i0, q0, 0);
      if (i1 < hi) f(i1, q1, 0);
    }
  }
}

// Column sums of X restricted to rows [lo, hi): out[a] = sum_i X_ia v_i, one
// warp per column, the column's row range found by binary search (rows of a
// CSC column ascend), lanes summed in a fixed order.
template <class T>
__device__ __forceinline__ void xt_partial(const GridPcg& a, int lo, int hi, const T* v, double* out) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int col = w; col < a.m; col += nw) {
    int b0 = a.xc_ptr[col], b1 = a.xc_ptr[col + 1];
    // first entry with row >= lo
    int l = b0, h = b1;
    while (l < h) {
      const int mid = (l + h) >> 1;
      if (a.xc_row[mid] < lo) l = mid + 1; else h = mid;
    }
    const int s0 = l;
    h = b1;
    while (l < h) {
      const int mid = (l + h) >> 1;
      if (a.xc_row[mid] < hi) l = mid + 1; else h = mid;
    }
    const int s1 = l;
    double t = 0.0;
    for (int q = s0 + lane; q < s1; q += 32) t = fma(a.xc_val[q], (double)v[a.xc_row[q]], t);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) out[col] = t;
  }
}

// Second stage of the v side's X^T v: block a adds column a of the per-block
// partials (fixed order) and stores y_a = s_a (X^T v)_a.
__device__ __forceinline__ void reduce_y_global(const GridPcg& a) {
  __shared__ double sh[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int col = blockIdx.x; col < a.m; col += a.nb) {
    double t = 0.0;
    for (int b = threadIdx.x; b < a.nb; b += blockDim.x) t += __ldcg(a.ypart + (size_t)b * a.m + col);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) sh[w] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
      double u = 0.0;
      for (int q = 0; q < (int)(blockDim.x >> 5); ++q) u += sh[q];
      a.yglob[col] = a.s[col] * u;
    }
    __syncthreads();
  }
}

// y into shared memory for the block's data-term rows
__device__ __forceinline__ void load_y(const GridPcg& a, double* ys) {
  for (int col = threadIdx.x; col < a.m; col += blockDim.x) ys[col] = __ldcg(a.yglob + col);
  __syncthreads();
}

// Data term of row i: omega_i v_i (u side) or sum_a X_ia y_a (v side, y in shared memory).
template <class T>
__device__ __forceinline__ T data_row(const GridPcg& a, const T* om, const double* ys, int i, T vi) {
  if (a.side == 0) return om[i] * vi;
  T acc = (T)0;
  for (int q = a.xr_ptr[i]; q < a.xr_ptr[i + 1]; ++q) acc = fma((T)a.xr_val[q], (T)ys[a.xr_col[q]], acc);
  return acc;
}

template <class T, int KM, bool F16>
__global__ void __launch_bounds__(F16 ? kGThreads16 : kGThreads, !F16 && KM == 6 ? 2 : 1) pcg_grid_kernel(const GridPcg a) {
  extern __shared__ double ys[];  // v side: y = s o (X^T v), m entries
  __shared__ double red[kParts], sums[3 * (F16 ? kGThreads16 : kGThreads)];
  T* xs = (T*)a.xs;
  T* rs = (T*)a.rs;
  T* qs = (T*)a.qs;
  T* ts = (T*)a.ts;
  T* dv = (T*)a.ds;
  T* om = (T*)a.os;
  T* gs = (T*)a.gs;
  T* zs = (T*)a.zs;
  GridBar bar = grid_bar(a.bar, a.err);
  const int n = a.L.n;
  const int lo = min(n, blockIdx.x * a.chunk), hi = min(n, lo + a.chunk);
  const double cd = a.coef[0], dd = a.coef[1];
  const T c = (T)cd, e = (T)(dd - cd * cd), lam = (T)a.lam;
  int it = 0, status = 0;
  double rho = 0.0, rr = 0.0, bb = 0.0;

  // ---- set-up: T copies of x0, D^-1, omega, L_ii
  for (int i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    xs[i] = (T)a.x[i];
    dv[i] = (T)a.dinv64[i];
    if (!F16) gs[i] = (T)a.L.diag[i];
    if (a.side == 0) om[i] = (T)a.omt64[i];
  }
  if (!grid_bar_sync(bar)) goto done;
  // ---- t = (L + cI) x0; v side partial X^T x0
  {
    auto xv = [&](int l) { return xs[l]; };
    for_rows<F16, KM>(a, lo, hi, [&](int i, const int (&q)[KM], int deg) {
      ts[i] = shifted_row<T, F16, KM>(a, gs, i, q, deg, c, xs[i], xv);
    });
  }
  if (a.side == 1) xt_partial<T>(a, lo, hi, xs, a.ypart + (size_t)blockIdx.x * a.m);
  if (!grid_bar_sync(bar)) goto done;
  if (a.side == 1) {
    reduce_y_global(a);
    if (!grid_bar_sync(bar)) goto done;
    load_y(a, ys);
  }
  // ---- r0 = b - A_hat x0; partial rho, |r|^2, |b|^2
  {
    auto tv = [&](int l) { return ts[l]; };
    Acc<T> acc[3];
    for_rows<F16, KM>(a, lo, hi, [&](int i, const int (&q)[KM], int deg) {
      const T xi = xs[i];
      const T bi = (T)a.b[i];
      const T ri = bi - (lam * (shifted_row<T, F16, KM>(a, gs, i, q, deg, c, ts[i], tv) + e * xi) + data_row<T>(a, om, ys, i, xi));
      const T zi = dv[i] * ri;
      rs[i] = ri;
      zs[i] = zi;
      acc[0].add(ri, zi);
      acc[1].add(ri, ri);
      acc[2].add(bi, bi);
    });
    block_reduce(acc, sums, red);
    if (threadIdx.x == 0) {
      double* pb = a.part + (size_t)blockIdx.x * kParts;
      pb[1] = red[0];
      pb[2] = red[1];
      pb[3] = red[2];
    }
  }
  if (!grid_bar_sync(bar)) goto done;
  {
    double v[3];
    sum_parts<3>(a.part, a.nb, 1, v);
    rho = v[0];
    rr = v[1];
    bb = v[2];
  }
  if (bb > 0.0) {
    const double tol2 = a.tol * a.tol * bb;
    double rho_prev = 1.0;
    for (;;) {
      if (rr <= tol2) break;
      if (it >= a.maxit) {
        status = 1;
        break;
      }
      T* pold = (T*)((it & 1) ? a.p1 : a.p0);
      T* pnew = (T*)((it & 1) ? a.p0 : a.p1);
      // ---- sweep A2a: p = D^-1 r + beta p_old (recomputed on the one-hop
      //      neighbourhood), t = (L + cI) p; v side partial X^T p
      {
        const bool first = it == 0;
        const T beta = (T)(first ? 0.0 : rho / rho_prev);
        auto pn = [&](int l) -> T { return first ? zs[l] : fma(beta, pold[l], zs[l]); };
        for_rows<F16, KM>(a, lo, hi, [&](int i, const int (&q)[KM], int deg) {
          const T pi = pn(i);
          pnew[i] = pi;
          ts[i] = shifted_row<T, F16, KM>(a, gs, i, q, deg, c, pi, pn);
        });
      }
      if (a.side == 1) {
        __syncthreads();
        xt_partial<T>(a, lo, hi, pnew, a.ypart + (size_t)blockIdx.x * a.m);
      }
      if (!grid_bar_sync(bar)) goto done;
      if (a.side == 1) {
        reduce_y_global(a);
        if (!grid_bar_sync(bar)) goto done;
        load_y(a, ys);
      }
      // ---- sweep A2b: q = lam ((L + cI) t + e p) + data(p); partial <p, q>
      {
        auto tv = [&](int l) { return ts[l]; };
        Acc<T> acc[1];
        for_rows<F16, KM>(a, lo, hi, [&](int i, const int (&q)[KM], int deg) {
          const T pi = pnew[i];
          const T qi = lam * (shifted_row<T, F16, KM>(a, gs, i, q, deg, c, ts[i], tv) + e * pi) + data_row<T>(a, om, ys, i, pi);
          qs[i] = qi;
          acc[0].add(pi, qi);
        });
        block_reduce(acc, sums, red);
        if (threadIdx.x == 0) a.part[(size_t)blockIdx.x * kParts + 0] = red[0];
      }
      if (!grid_bar_sync(bar)) goto done;
      double pqv[1];
      sum_parts<1>(a.part, a.nb, 0, pqv);
      const double pq = pqv[0];
      if (!(pq > 0.0)) {
        status = 2;
        break;
      }
      // ---- sweep B: x += alpha p, r -= alpha q; partial rho, |r|^2
      {
        const T alpha = (T)(rho / pq);
        Acc<T> acc[2];
        // chunk and vector starts are multiples of four rows
        for (int i = lo + 4 * threadIdx.x; i < hi; i += 4 * blockDim.x) {
          T xv[4], pv[4], rv[4], qv[4], dd4[4], zv[4];
          ld4(xv, xs + i);
          ld4(pv, pnew + i);
          ld4(rv, rs + i);
          ld4(qv, qs + i);
          ld4(dd4, dv + i);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            xv[u] = fma(alpha, pv[u], xv[u]);
            rv[u] = fma(-alpha, qv[u], rv[u]);
            zv[u] = dd4[u] * rv[u];
            if (i + u < hi) {
              acc[0].add(rv[u], zv[u]);
              acc[1].add(rv[u], rv[u]);
            }
          }
          st4(xs + i, xv);
          st4(rs + i, rv);
          st4(zs + i, zv);
        }
        block_reduce(acc, sums, red);
        if (threadIdx.x == 0) {
          double* pb = a.part + (size_t)blockIdx.x * kParts;
          pb[1] = red[0];
          pb[2] = red[1];
        }
      }
      ++it;
      if (!grid_bar_sync(bar)) goto done;
      double v2[2];
      sum_parts<2>(a.part, a.nb, 1, v2);
      rho_prev = rho;
      rho = v2[0];
      rr = v2[1];
    }
  }
  for (int i = lo + threadIdx.x; i < hi; i += blockDim.x) a.x[i] = (double)xs[i];
done:
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    PcgStat st;
    st.iters = it;
    st.status = *(volatile int*)a.err ? 3 : status;
    st.relres = bb > 0.0 ? sqrt(fmax(rr, 0.0) / bb) : 0.0;
    st.bnorm = sqrt(bb);
    *a.stat = st;
  }
}

}  // namespace
}  // namespace cr

namespace cr {

// Threads per block and largest block count that is co-resident for the kernel
// variant (float32 or float64; neighbour table), at most one block of 1,024 or one
// or two of 512 threads per SM (cooperative launch); 0 if it cannot run.
static int grid_threads(const DevLap& L) { return L.nbr16 ? kGThreads16 : kGThreads; }
const void* grid_kernel_fn(bool fp32, const DevLap& L) {
  if (L.nbr16) return fp32 ? (const void*)pcg_grid_kernel<float, 6, true> : (const void*)pcg_grid_kernel<double, 6, true>;
  const bool k6 = L.K <= 6;
  return fp32 ? (k6 ? (const void*)pcg_grid_kernel<float, 6, false> : (const void*)pcg_grid_kernel<float, kMaxSlots, false>)
              : (k6 ? (const void*)pcg_grid_kernel<double, 6, false>
                    : (const void*)pcg_grid_kernel<double, kMaxSlots, false>);
}

int pcg_grid_blocks(bool fp32, int m, const DevLap& L) {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const size_t smem = sizeof(double) * (size_t)std::max(m, 1);
  const void* fn = grid_kernel_fn(fp32, L);
  // y and the sums together may exceed the 48 KB that need no opt-in (m up to 4,096: 32 KB + 25 KB)
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(double) * kMaxInj) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, grid_threads(L), smem) != cudaSuccess || per < 1) {
    cudaGetLastError();
    return 0;
  }
  return sms * std::min(per, L.nbr16 || L.n < kGTwoRows ? 1 : 2);
}

// vectors start at multiples of 16 rows, so that four rows load at once
static size_t grid_stride(int n) { return ((size_t)n + 15) / 16 * 16; }
size_t pcg_grid_work_elems(int n) { return 10 * grid_stride(n); }

cudaError_t pcg_grid_launch(const PcgArgs& a, int side, const int* xc_ptr, const int* xc_row, const double* xc_val,
                            double* work, double* part, double* ypart, double* yglob, unsigned* bar, int* err,
                            int nb, cudaStream_t st) {
  const int n = a.L.n;
  if (nb < 1 || n < 1) return cudaErrorInvalidValue;
  GridPcg g{};
  g.L = a.L;
  g.lam = a.lam;
  g.coef = a.coef;
  g.side = side;
  g.m = a.m;
  g.s = a.s;
  g.xr_ptr = a.X.xr_ptr;
  g.xr_col = a.X.xr_col;
  g.xr_val = a.X.xr_val;
  g.xc_ptr = xc_ptr;
  g.xc_row = xc_row;
  g.xc_val = xc_val;
  g.b = a.b;
  g.x = a.x;
  g.dinv64 = a.dinv;
  g.omt64 = a.omt;
  const size_t word = a.fp32 ? sizeof(float) : sizeof(double);
  char* w = reinterpret_cast<char*>(work);
  void** slots[10] = {&g.xs, &g.rs, &g.p0, &g.p1, &g.qs, &g.ts, &g.ds, &g.os, &g.gs, &g.zs};
  for (int k = 0; k < 10; ++k) *slots[k] = w + (size_t)k * grid_stride(n) * word;
  g.idx = a.L.nbr16;
  g.part = part;
  g.ypart = ypart;
  g.yglob = yglob;
  g.bar = bar;
  g.err = err;
  g.nb = nb;
  g.chunk = ((n + nb - 1) / nb + 3) / 4 * 4;
  g.tol = a.tol;
  g.maxit = a.maxit;
  g.stat = a.stat;
  cudaError_t e = cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(err, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  void* args[] = {&g};
  const size_t smem = sizeof(double) * (size_t)std::max(a.m, 1);
  count_launch();
  return cudaLaunchCooperativeKernel(grid_kernel_fn(a.fp32 != 0, a.L), dim3(nb), dim3(grid_threads(a.L)), args, smem, st);
}

}  // namespace cr
