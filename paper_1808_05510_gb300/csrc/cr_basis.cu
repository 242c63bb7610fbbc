// Growth of the residual-norm bases and of the Galerkin eigenbases by one greedy
// step (see cr_api.cu), both grids in every launch.
//
// A step appends the three columns [u, L u, L^2 u] to the orthonormal basis of
// each grid.  Taken one column at a time that was 27 launches and three host round
// trips per grid, and every column re-read the basis four times.  Here the three
// are projected together against the basis, twice (block classical Gram-Schmidt
// with reorthogonalisation), each projection followed by their own
// orthonormalisation in one cluster: eight launches for both grids and one read-back
// (how many columns were accepted).  The float64 rate bounds the projections
// (GB300: two FMAs per SM and clock): 12 n k FMAs per grid and step for a basis of
// k columns, and 3 n k for the coefficients behind them, whatever the blocking; the
// blocking saves launches, round trips and memory passes.  Factors of rank 240 on grids of 7,500 voxels, 28 injections, set and
// projected: 302 ms a pass, 100 of them in these products, before, and 177 ms after.
#include <cooperative_groups.h>

#include <algorithm>

#include "cr_common.cuh"

namespace cg = cooperative_groups;

namespace cr {

namespace {

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// out[p + s * ldo] = A(:, p)^T w_s, s < 3 (column s at at[s] if given, and mirrored into a row with
// stride ldrow if given); one CTA per column p and grid, fixed-order sums.
// MAG: grid 0 also gives mag[p] = sum_i |A(i, p)| |w_0(i)|
template <bool MAG>
__global__ void __launch_bounds__(256) panel_t_kernel(const PanelArgs a) {
  const int g = blockIdx.y, p = blockIdx.x, n = a.n[g];
  if (p >= a.k[g]) return;
  const double* A = a.A[g] + (int64_t)p * a.lda[g];
  const double* w = a.w[g];
  const int64_t ldw = a.ldw[g];
  constexpr int NV = 3, NS = MAG ? NV + 1 : NV;
  double acc[NS][2];
#pragma unroll
  for (int s = 0; s < NS; ++s) acc[s][0] = acc[s][1] = 0.0;
  int i = threadIdx.x;
  for (; i + 256 < n; i += 512) {
    const double x0 = A[i], x1 = A[i + 256];
#pragma unroll
    for (int s = 0; s < NV; ++s) {
      acc[s][0] = fma(x0, w[i + s * ldw], acc[s][0]);
      acc[s][1] = fma(x1, w[i + 256 + s * ldw], acc[s][1]);
    }
    if (MAG && g == 0) {
      acc[NS - 1][0] = fma(fabs(x0), fabs(w[i]), acc[NS - 1][0]);
      acc[NS - 1][1] = fma(fabs(x1), fabs(w[i + 256]), acc[NS - 1][1]);
    }
  }
  if (i < n) {
    const double x0 = A[i];
#pragma unroll
    for (int s = 0; s < NV; ++s) acc[s][0] = fma(x0, w[i + s * ldw], acc[s][0]);
    if (MAG && g == 0) acc[NS - 1][0] = fma(fabs(x0), fabs(w[i]), acc[NS - 1][0]);
  }
  // one warp per value adds the 256 partial sums (a shuffle tree in every warp costs three times
  // the float64 issue slots)
  __shared__ double sh[NS][256];
#pragma unroll
  for (int s = 0; s < NS; ++s) sh[s][threadIdx.x] = acc[s][0] + acc[s][1];
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (wid < NS) {
    double q[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) q[u] = sh[wid][lane + 32 * u];
    const double t = wsum(((q[0] + q[1]) + (q[2] + q[3])) + ((q[4] + q[5]) + (q[6] + q[7])));
    if (MAG && wid == NV) {
      if (lane == 0 && g == 0) a.mag[p] = t;
    } else if (lane == 0) {
      (a.at[g][wid] ? a.at[g][wid] : a.out[g] + wid * a.ldo[g])[p] = t;
      if (a.row[g][wid]) a.row[g][wid][(int64_t)p * a.ldrow] = t;
    }
  }
}

// w_s(i) -= sum_p A(i, p) c[p + s * ldc], s < 3: 32 rows per CTA, the columns split between its
// eight warps in eight fixed ranges whose sums are added in order
__global__ void __launch_bounds__(256) panel_n_kernel(const PanelArgs a) {
  const int g = blockIdx.y, n = a.n[g], k = a.k[g];
  if (blockIdx.x * 32 >= n) return;
  extern __shared__ double cs[];  // [3][k]
  for (int t = threadIdx.x; t < 3 * k; t += 256) cs[t] = a.out[g][t % k + (t / k) * a.ldo[g]];
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  const int kc = (k + 7) / 8, p0 = min(k, wid * kc), p1 = min(k, p0 + kc);
  double acc[3] = {0.0, 0.0, 0.0};
  if (i < n) {
    const double* A = a.A[g] + i;
    const int64_t lda = a.lda[g];
    int p = p0;
    for (; p + 3 < p1; p += 4) {
      double x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = A[(int64_t)(p + u) * lda];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int s = 0; s < 3; ++s) acc[s] = fma(x[u], cs[p + u + s * k], acc[s]);
    }
    for (; p < p1; ++p) {
      const double x = A[(int64_t)p * lda];
#pragma unroll
      for (int s = 0; s < 3; ++s) acc[s] = fma(x, cs[p + s * k], acc[s]);
    }
  }
  __shared__ double part[3][8][33];
#pragma unroll
  for (int s = 0; s < 3; ++s) part[s][wid][lane] = acc[s];
  __syncthreads();
  if (wid < 3 && i < n) {
    double t = 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q) t += part[wid][q][lane];
    double* w = const_cast<double*>(a.w[g]) + i + wid * a.ldw[g];
    *w -= t;
  }
}

// w_s = src_s, s < 3
__global__ void __launch_bounds__(256) panel_copy_kernel(const PanelArgs a) {
  const int g = blockIdx.y, i = blockIdx.x * 256 + threadIdx.x;
  if (i >= a.n[g]) return;
#pragma unroll
  for (int s = 0; s < 3; ++s)
    const_cast<double*>(a.w[g])[i + s * a.ldw[g]] = a.src[g][i + s * a.lds[g]];
}

constexpr int kOrthCtas = 8;

// Orthonormalises the three columns w_s (one cluster per grid).  first: a column whose norm has
// fallen to 1e-12 of its source column's, or to zero, is dropped; the accepted ones move to the
// front, the rest is zeroed, and their number goes to a.count.
__global__ void __cluster_dims__(kOrthCtas, 1, 1) __launch_bounds__(256) panel_orth_kernel(const PanelArgs a, int first) {
  cg::cluster_group cl = cg::this_cluster();
  const int g = blockIdx.y, n = a.n[g], rank = (int)cl.block_rank();
  double* w = const_cast<double*>(a.w[g]);
  const int64_t ldw = a.ldw[g];
  const int step = kOrthCtas * 256, i0 = rank * 256 + threadIdx.x;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __shared__ double sh[8][6], red[2][6], tot[6];
  int parity = 0;
  // sums of v[] over the cluster, in a fixed order, the same in every CTA
  auto total = [&](double (&v)[6], int cnt) {
    for (int q = 0; q < cnt; ++q) v[q] = wsum(v[q]);
    if (lane == 0)
      for (int q = 0; q < cnt; ++q) sh[wid][q] = v[q];
    __syncthreads();
    if (threadIdx.x < cnt) {
      double t = 0.0;
      for (int q = 0; q < 8; ++q) t += sh[q][threadIdx.x];
      red[parity][threadIdx.x] = t;
    }
    cl.sync();
    if (threadIdx.x < cnt) {
      double t = 0.0;
      for (int r = 0; r < kOrthCtas; ++r) t += cl.map_shared_rank(&red[parity][0], r)[threadIdx.x];
      tot[threadIdx.x] = t;
    }
    __syncthreads();
    for (int q = 0; q < cnt; ++q) v[q] = tot[q];
    parity ^= 1;
  };
  double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
  for (int i = i0; i < n; i += step) {
    const double x = w[i], y = w[i + ldw], z = w[i + 2 * ldw];
    v[0] = fma(x, x, v[0]);
    v[1] = fma(x, y, v[1]);
    v[2] = fma(x, z, v[2]);
    if (first)
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        const double b = a.src[g][i + s * a.lds[g]];
        v[3 + s] = fma(b, b, v[3 + s]);
      }
  }
  total(v, first ? 6 : 3);
  const double nb0 = v[3], nb1 = v[4], nb2 = v[5];
  auto accepted = [&](double na, double nb) { return first ? nb > 0.0 && sqrt(na / nb) > 1e-12 : na > 0.0; };
  const bool ok0 = accepted(v[0], nb0);
  const double inv0 = ok0 ? 1.0 / sqrt(v[0]) : 0.0, r01 = v[1] * inv0, r02 = v[2] * inv0;
  double u[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
  for (int i = i0; i < n; i += step) {
    const double x = w[i] * inv0;
    const double y = fma(-r01, x, w[i + ldw]), z = fma(-r02, x, w[i + 2 * ldw]);
    w[i] = x;
    w[i + ldw] = y;
    w[i + 2 * ldw] = z;
    u[0] = fma(y, y, u[0]);
    u[1] = fma(y, z, u[1]);
  }
  total(u, 2);
  const bool ok1 = accepted(u[0], nb1);
  const double inv1 = ok1 ? 1.0 / sqrt(u[0]) : 0.0, r12 = u[1] * inv1;
  double t[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
  for (int i = i0; i < n; i += step) {
    const double y = w[i + ldw] * inv1, z = fma(-r12, y, w[i + 2 * ldw]);
    w[i + ldw] = y;
    w[i + 2 * ldw] = z;
    t[0] = fma(z, z, t[0]);
  }
  total(t, 1);
  const bool ok2 = accepted(t[0], nb2);
  const double inv2 = ok2 ? 1.0 / sqrt(t[0]) : 0.0;
  // accepted columns first, in order; zeros behind them
  const int at1 = ok0 ? 1 : 0, at2 = at1 + (ok1 ? 1 : 0), cnt = at2 + (ok2 ? 1 : 0);
#pragma unroll 4
  for (int i = i0; i < n; i += step) {
    const double x = w[i], y = w[i + ldw], z = w[i + 2 * ldw] * inv2;
    double o[3] = {0.0, 0.0, 0.0};
    if (ok0) o[0] = x;
    if (ok1) o[at1] = y;
    if (ok2) o[at2] = z;
#pragma unroll
    for (int s = 0; s < 3; ++s) w[i + s * ldw] = o[s];
  }
  if (first && rank == 0 && threadIdx.x == 0) *a.count[g] = (double)cnt;
  cl.sync();  // no CTA leaves while another can still read its shared memory
}

// Next border of both eigenbases: z_p = Q(:, p)^T A(:, q) for p < q, z_q = A(q, q), Q(q, q) = 1
__global__ void __launch_bounds__(128) basis_border_kernel(int q, int64_t ld, double* Qa, double* Qb, const double* A1,
                                                           const double* B1, double* za, double* zb) {
  const int p = blockIdx.x;
  double* Q = blockIdx.y == 0 ? Qa : Qb;
  const double* A = (blockIdx.y == 0 ? A1 : B1) + (int64_t)q * ld;
  double* z = blockIdx.y == 0 ? za : zb;
  if (p == q) {
    if (threadIdx.x == 0) {
      Q[q + (int64_t)q * ld] = 1.0;
      z[q] = A[q];
    }
    return;
  }
  const double* c = Q + (int64_t)p * ld;
  double acc = 0.0;
  for (int i = threadIdx.x; i < q; i += 128) acc = fma(c[i], A[i], acc);
  acc = wsum(acc);
  __shared__ double sh[4];
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) z[p] = ((sh[0] + sh[1]) + sh[2]) + sh[3];
}

// O_g = Q_g W_g, g = 0, 1 (n1 x n1; Q, O with leading dimension ld, W with n1): 16 x 16 tiles, the
// next 16 columns' operands loaded while the current ones are multiplied
__global__ void __launch_bounds__(256) basis_product_kernel(int n1, int64_t ld, const double* Qa, const double* Qb,
                                                            const double* Wa, const double* Wb, double* Oa, double* Ob) {
  __shared__ double As[2][16][17], Bs[2][16][17];
  const double* Q = blockIdx.z == 0 ? Qa : Qb;
  const double* W = blockIdx.z == 0 ? Wa : Wb;
  double* O = blockIdx.z == 0 ? Oa : Ob;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int i0 = blockIdx.x * 16, l0 = blockIdx.y * 16;
  auto la = [&](int k0) { return i0 + tx < n1 && k0 + ty < n1 ? Q[i0 + tx + (int64_t)(k0 + ty) * ld] : 0.0; };
  auto lb = [&](int k0) { return k0 + tx < n1 && l0 + ty < n1 ? W[k0 + tx + (int64_t)(l0 + ty) * n1] : 0.0; };
  double ra = la(0), rb = lb(0), acc = 0.0;
  int cur = 0;
  for (int k0 = 0; k0 < n1; k0 += 16) {
    As[cur][ty][tx] = ra;  // [k][i]
    Bs[cur][ty][tx] = rb;  // [l][k]
    __syncthreads();
    ra = la(k0 + 16);
    rb = lb(k0 + 16);
#pragma unroll
    for (int k = 0; k < 16; ++k) acc = fma(As[cur][k][tx], Bs[cur][ty][k], acc);
    cur ^= 1;
  }
  if (i0 + tx < n1 && l0 + ty < n1) O[i0 + tx + (int64_t)(l0 + ty) * ld] = acc;
}

// G_a(p, q) = sum_i Omega_ia u_p(i) u_q(i) for p <= q, from D(p) = u_p^T u_q and the shorter of each
// injection's row lists: the unobserved rows (full[a] = 1: D minus their products) or the observed
// ones; one warp per (p, a), both triangles written.  The shorter list needs at most half of the
// products of a masked copy of u_q times U (gemm: 20.7 of 141 ms at rank 240, 28 injections), and
// bounds the launch by its gathers from L2.  The difference carries the rounding of all rows'
// products: it is taken where the unobserved rows hold at most half of T(p) = sum_i |u_p(i)| |u_q(i)|,
// which keeps its error within three times the observed rows' own; elsewhere the sum runs over the
// observed rows themselves.
__global__ void __launch_bounds__(256) omega_border_kernel(int q, int m, const double* __restrict__ UU, int64_t ldu,
                                                           const double* __restrict__ D, const double* __restrict__ T,
                                                           const int* __restrict__ zp, const int* __restrict__ zrow,
                                                           const uint8_t* __restrict__ full, const uint8_t* __restrict__ Om,
                                                           int n, double* __restrict__ G, int64_t ld) {
  const int lane = threadIdx.x & 31;
  const int64_t t = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (t >= (int64_t)m * (q + 1)) return;
  const int p = (int)(t % (q + 1)), a = (int)(t / (q + 1));
  const double *up = UU + p * ldu, *uq = UU + q * ldu;
  double acc = 0.0, mag = 0.0;
#pragma unroll 4
  for (int k = zp[a] + lane; k < zp[a + 1]; k += 32) {
    const int i = zrow[k];
    acc = fma(up[i], uq[i], acc);
    mag = fma(fabs(up[i]), fabs(uq[i]), mag);
  }
  acc = wsum(acc);
  double g = acc;
  if (full[a]) {
    g = D[p] - acc;
    if (!(2.0 * wsum(mag) <= T[p])) {
      acc = 0.0;
      for (int i = lane; i < n; i += 32)
        if (Om[i + (int64_t)a * n]) acc = fma(up[i], uq[i], acc);
      g = wsum(acc);
    }
  }
  if (lane == 0) {
    double* Ga = G + (int64_t)a * ld * ld;
    Ga[p + (int64_t)q * ld] = g;
    Ga[q + (int64_t)p * ld] = g;
  }
}

}  // namespace

void omega_border(int q, int m, const double* UU, int64_t ldu, const double* D, const double* T, const int* zp,
                  const int* zrow, const uint8_t* full, const uint8_t* Om, int n, double* G, int64_t ld, cudaStream_t st) {
  const int64_t t = (int64_t)m * (q + 1);
  if (t <= 0) return;
  count_launch();
  omega_border_kernel<<<(unsigned)((t + 7) / 8), 256, 0, st>>>(q, m, UU, ldu, D, T, zp, zrow, full, Om, n, G, ld);
}

void panel_t(const PanelArgs& a, cudaStream_t st) {
  const int k = std::max(a.k[0], a.k[1]);
  if (k <= 0) return;
  count_launch();
  if (a.mag)
    panel_t_kernel<true><<<dim3(k, 2), 256, 0, st>>>(a);
  else
    panel_t_kernel<false><<<dim3(k, 2), 256, 0, st>>>(a);
}

void panel_n(const PanelArgs& a, cudaStream_t st) {
  constexpr int kChunk = 1536;  // columns whose coefficients fit a CTA's static share of shared memory
  const int k = std::max(a.k[0], a.k[1]);
  for (int p0 = 0; p0 < k; p0 += kChunk) {
    PanelArgs b = a;
    for (int g = 0; g < 2; ++g) {
      b.k[g] = std::max(0, std::min(kChunk, a.k[g] - p0));
      b.A[g] = a.A[g] + (int64_t)p0 * a.lda[g];
      b.out[g] = a.out[g] + p0;
    }
    count_launch();
    panel_n_kernel<<<dim3((std::max(a.n[0], a.n[1]) + 31) / 32, 2), 256,
                     sizeof(double) * 3 * std::max(b.k[0], b.k[1]), st>>>(b);
  }
}

void panel_copy(const PanelArgs& a, cudaStream_t st) {
  count_launch();
  panel_copy_kernel<<<dim3((std::max(a.n[0], a.n[1]) + 255) / 256, 2), 256, 0, st>>>(a);
}

void panel_orth(const PanelArgs& a, bool first, cudaStream_t st) {
  count_launch();
  panel_orth_kernel<<<dim3(kOrthCtas, 2), 256, 0, st>>>(a, first ? 1 : 0);
}

void basis_border(int q, int64_t ld, double* Qa, double* Qb, const double* A1, const double* B1, double* za, double* zb,
                  cudaStream_t st) {
  count_launch();
  basis_border_kernel<<<dim3(q + 1, 2), 128, 0, st>>>(q, ld, Qa, Qb, A1, B1, za, zb);
}

void basis_product(int n1, int64_t ld, const double* Qa, const double* Qb, const double* Wa, const double* Wb, double* Oa,
                   double* Ob, cudaStream_t st) {
  count_launch();
  basis_product_kernel<<<dim3((n1 + 15) / 16, (n1 + 15) / 16, 2), 256, 0, st>>>(n1, ld, Qa, Qb, Wa, Wb, Oa, Ob);
}

}  // namespace cr
