// Cluster-resident float32 Jacobi PCG for the inner solves of the mixed form's
// ALS sub-problems (Sec. 2.3, Eqs. ALS_linsys and ALS_linsys_v) on unit-weight
// Laplacians with at most six neighbours per row (the operator, the split and
// the Chronopoulos-Gear recurrence of cr_pcg.cu, from a zero initial guess).
//
// What bounds it.  One cluster holds a whole solve on chip, so an iteration is
// a chain of latencies: cluster barriers, reads of other CTAs' shared memory
// (a round trip each), and sums.  Here values are pushed instead of fetched:
//  - u = D^-1 r goes by st.shared::cluster into the shared memory of every CTA
//    that needs it, before the barrier that publishes it, so that every later
//    read is local.  Each CTA receives the rows within two hops of its own and
//    forms t = (L + cI) u on its own rows and their neighbours, which saves the
//    barrier between the two stencils: two cluster barriers per iteration
//    instead of three.
//  - v side: the CTA's part of X^T u is pushed to all CTAs before the same
//    barrier, one warp per receiving CTA so that the stores of a warp share
//    packets (scattered, one lane per CTA, they cost more than they saved); the
//    CTA's rows of X lie in shared memory by rows (four entries a
//    load) and by columns (eight lanes a column), instead of dependent global
//    loads.
//  - inner products: each CTA's three sums are pushed to all CTAs, and one warp
//    adds them from its own shared memory after the barrier.
// Sums are double-float (cr_df.cuh) in a fixed order, so every CTA forms the
// same scalars and results repeat bit for bit.
// Measured (16 CTAs, us per iteration, launches included) against the kernel that
// fetched neighbours through distributed shared memory: 7,526 voxels u side
// 3.70 -> 2.65, v side with 28 injections 5.83 -> 3.26; 15,000 voxels, v side
// with 100 injections 10.07 -> 5.42.  What is left of the 2.65: two barriers
// 0.8, the sums 1.0, push and stencils 0.6; the v side adds 0.8 for X^T u.
#include <cooperative_groups.h>

#include "cr_common.cuh"
#include "cr_df.cuh"

namespace cg = cooperative_groups;

namespace cr {

namespace {

constexpr int kPushWarps = kPcgThreads / 32;

__device__ __forceinline__ uint32_t push_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t push_mapa(uint32_t a, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}

__device__ __forceinline__ void st_remote(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t a, DF v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.hi), "f"(v.lo) : "memory");
}

__device__ __forceinline__ DF df_pick(bool b, DF x, DF y) { return DF{b ? x.hi : y.hi, b ? x.lo : y.lo}; }
__device__ __forceinline__ DF df_xor(DF v, int o) {
  return DF{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}

// Sums of three values over the warp: every lane of lanes 0-7 gets a's, 8-15 b's, 16-23 c's.  The
// first two steps also split the values between the lanes, so that six double-float additions are
// issued instead of fifteen (four warps share a scheduler: the tree is bound by issue).
__device__ __forceinline__ DF warp_sum3(DF a, DF b, DF c) {
  const int lane = threadIdx.x & 31;
  const bool h = lane & 16, q = lane & 8;
  const DF z{0.f, 0.f};
  const DF x = df_add(df_pick(h, c, a), df_xor(df_pick(h, a, c), 16));
  const DF y = df_add(df_pick(h, z, b), df_xor(df_pick(h, b, z), 16));
  DF v = df_add(df_pick(q, y, x), df_xor(df_pick(q, x, y), 8));
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v = df_add(v, df_xor(v, o));
  return v;
}

// byte offsets of the shared-memory sections
struct PushLayout {
  int xv, xc, slots, wsum, ub, tb, ys, yl, sy, ss, push, hn, hd, ac, ab, cv, cr, scal, bytes;
};

__host__ __device__ inline PushLayout push_layout(const DevPush& D, int m) {
  PushLayout l{};
  int at = 0;
  auto sect = [&](int bytes) {
    const int a = at;
    at += (bytes + 15) / 16 * 16;
    return a;
  };
  const bool v = D.xq_max >= 0, xs = v && D.x_smem;
  l.xv = sect(xs ? 16 * D.xq_max : 0);
  l.xc = sect(xs ? 8 * D.xq_max : 0);
  l.slots = sect(8 * 3 * D.csize);
  l.wsum = sect(8 * 3 * kPushWarps);
  l.ub = sect(4 * D.ext);
  l.tb = sect(4 * D.ext);
  l.ys = sect(v ? 4 * D.csize * m : 0);
  l.yl = sect(v ? 4 * m : 0);
  l.sy = sect(v ? 4 * m : 0);
  l.ss = sect(v ? 4 * m : 0);
  l.push = sect(4 * D.P * D.chunk);
  l.hn = sect(16 * D.hmax);
  l.hd = sect(4 * D.hmax);
  l.ac = sect(xs ? 4 * D.xa_max : 0);
  l.ab = sect(xs ? 4 * (D.xa_max + 1) : 0);
  l.cv = sect(xs ? 4 * D.xc_max : 0);
  l.cr = sect(xs ? 2 * D.xc_max : 0);
  l.scal = sect(32);
  l.bytes = at;
  return l;
}

// XS: the CTA's part of X lies in shared memory (else, where it does not fit, in global memory)
template <int KIND, int VPT, bool XS>
__global__ void __launch_bounds__(kPcgThreads, 1) pcg_push_kernel(const PcgArgs A, const DevPush D) {
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks();
  const int rank = (int)cl.block_rank();
  const DevLap& L = A.L;
  const int chunk = D.chunk, beg = rank * chunk;
  const int nloc = max(0, min(L.n - beg, chunk));
  const int m = A.m;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  extern __shared__ __align__(16) char sm[];
  const PushLayout lay = push_layout(D, m);
  float* ub = reinterpret_cast<float*>(sm + lay.ub);
  float* tb = reinterpret_cast<float*>(sm + lay.tb);
  DF* slots = reinterpret_cast<DF*>(sm + lay.slots);
  DF* wsum = reinterpret_cast<DF*>(sm + lay.wsum);
  uint32_t* ptab = reinterpret_cast<uint32_t*>(sm + lay.push);
  uint4* hn = reinterpret_cast<uint4*>(sm + lay.hn);
  float* hd = reinterpret_cast<float*>(sm + lay.hd);
  float* ys = reinterpret_cast<float*>(sm + lay.ys);
  float* yl = reinterpret_cast<float*>(sm + lay.yl);
  float* sY = reinterpret_cast<float*>(sm + lay.sy);
  float* sS = reinterpret_cast<float*>(sm + lay.ss);
  const float4* xv = reinterpret_cast<float4*>(sm + lay.xv);
  const ushort4* xc = reinterpret_cast<ushort4*>(sm + lay.xc);
  const int* ac = reinterpret_cast<int*>(sm + lay.ac);
  const int* ab = reinterpret_cast<int*>(sm + lay.ab);
  const float* cv = reinterpret_cast<float*>(sm + lay.cv);
  const uint16_t* crow = reinterpret_cast<uint16_t*>(sm + lay.cr);
  float* scal = reinterpret_cast<float*>(sm + lay.scal);

  const float lam = (float)A.lam;
  const double cd = A.coef[0];
  const float e = (float)(A.coef[1] - cd * cd);
  const int nh = D.hcnt[rank];
  for (int k = tid; k < D.ext; k += kPcgThreads) ub[k] = tb[k] = 0.f;
  for (int k = tid; k < D.P * chunk; k += kPcgThreads) {
    const uint32_t q = D.push[(size_t)rank * D.P * chunk + k];
    ptab[k] = q == 0xFFFFFFFFu ? 0u : push_mapa(push_smem(ub + (q & 0xFFFFu)), q >> 16);
  }
  for (int h = tid; h < nh; h += kPcgThreads) {
    hn[h] = D.hn[(size_t)rank * D.hmax + h];
    hd[h] = (float)(D.hdiag[(size_t)rank * D.hmax + h] + cd);
  }
  int na = 0, nent = 0;  // v side: columns with an entry in this CTA, entries
  if (KIND == 1) {
    const int q0 = D.xq_off[rank], nq = D.xq_off[rank + 1] - q0;
    const int a0 = D.xa_off[rank], e0 = D.xc_off[rank], ne = D.xc_off[rank + 1] - e0;
    na = D.xa_off[rank + 1] - a0;
    nent = ne;
    if (XS) {
      float4* xv_s = reinterpret_cast<float4*>(sm + lay.xv);
      ushort4* xc_s = reinterpret_cast<ushort4*>(sm + lay.xc);
      int *ac_s = reinterpret_cast<int*>(sm + lay.ac), *ab_s = reinterpret_cast<int*>(sm + lay.ab);
      float* cv_s = reinterpret_cast<float*>(sm + lay.cv);
      uint16_t* cr_s = reinterpret_cast<uint16_t*>(sm + lay.cr);
      for (int k = tid; k < nq; k += kPcgThreads) {
        xv_s[k] = D.xr_v[q0 + k];
        xc_s[k] = D.xr_c[q0 + k];
      }
      for (int k = tid; k <= na; k += kPcgThreads) {
        if (k < na) ac_s[k] = D.xa_col[a0 + k];
        ab_s[k] = k < na ? D.xa_beg[a0 + k] : ne;
      }
      for (int k = tid; k < ne; k += kPcgThreads) {
        cv_s[k] = D.xc_v[e0 + k];
        cr_s[k] = D.xc_r[e0 + k];
      }
    } else {
      xv = D.xr_v + q0;
      xc = D.xr_c + q0;
      ac = D.xa_col + a0;
      ab = D.xa_beg + a0;
      cv = D.xc_v + e0;
      crow = D.xc_r + e0;
    }
    for (int k = tid; k < C * m; k += kPcgThreads) ys[k] = 0.f;
    for (int k = tid; k < m; k += kPcgThreads) {
      sS[k] = (float)A.s[k];
      yl[k] = 0.f;
    }
  }

  float x[VPT], r[VPT], p[VPT], sv[VPT], dpc[VPT], dinv[VPT], omt[VPT];
  uint32_t na3[VPT][3];  // neighbours as pairs of 16-bit indices
  // v side: the row's quads of X, the first kQ of them in registers
  constexpr int kQ = KIND == 1 && VPT == 1 ? 1 : 0;
  float4 qv[VPT][kQ > 0 ? kQ : 1];
  ushort4 qc[VPT][kQ > 0 ? kQ : 1];
  int q0r[VPT], q1r[VPT];
  bool own[VPT];
#pragma unroll
  for (int k = 0; k < VPT; ++k) {
    const int li = tid + k * kPcgThreads;
    own[k] = li < nloc;
    x[k] = r[k] = p[k] = sv[k] = 0.f;
    dpc[k] = dinv[k] = omt[k] = 0.f;
    q0r[k] = q1r[k] = 0;
    const uint32_t zz = (uint32_t)(D.ext - 1) * 0x10001u;
    na3[k][0] = na3[k][1] = na3[k][2] = zz;
    if (own[k]) {
      const int i = beg + li;
      const uint4 q = D.own[i];
      na3[k][0] = q.x;
      na3[k][1] = q.y;
      na3[k][2] = q.z;
      dpc[k] = (float)(L.diag[i] + cd);
      dinv[k] = (float)A.dinv[i];
      if (KIND == 0) omt[k] = (float)A.omt[i];
      if (KIND == 1) {
        q0r[k] = D.xr_q[(size_t)rank * (chunk + 1) + li];
        q1r[k] = D.xr_q[(size_t)rank * (chunk + 1) + li + 1];
      }
      r[k] = (float)A.b[i];
    }
  }
#pragma unroll
  for (int k = 0; k < VPT; ++k)
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
      const bool in = q0r[k] + q < q1r[k];
      const int at = D.xq_off[rank] + q0r[k] + q;
      qv[k][q] = in ? D.xr_v[at] : float4{0.f, 0.f, 0.f, 0.f};
      qc[k][q] = in ? D.xr_c[at] : ushort4{0, 0, 0, 0};
    }
  // (L + cI) v minus its diagonal part: the six neighbours from shared memory, fixed order
  auto nsum = [&](const float* v, uint32_t a, uint32_t b, uint32_t d) -> float {
    const float v0 = v[a & 0xFFFFu], v1 = v[a >> 16], v2 = v[b & 0xFFFFu], v3 = v[b >> 16], v4 = v[d & 0xFFFFu],
                v5 = v[d >> 16];
    return ((v0 + v1) + (v2 + v3)) + (v4 + v5);
  };
  cl.sync();  // every CTA's shared memory is initialised before anyone pushes into it

  // lanes per column of X: the CTA's columns fill its warps
  const int cgl = na <= kPushWarps ? 32 : na <= 2 * kPushWarps ? 16 : 8;
  int it = 0, status = 0;
  DF rho{0.f, 0.f}, bb{0.f, 0.f};
  // thread 0: 1 / gamma and 1 / alpha of the step before, gamma and alpha's denominator of this one
  DF gam_prev{1.f, 0.f}, alpha_prev{1.f, 0.f}, gcur{1.f, 0.f}, dcur{1.f, 0.f};
  float tol2 = 0.f;
  const float tt2 = (float)(A.tol * A.tol);
  for (;;) {
    float u[VPT], t[VPT], w[VPT];
#pragma unroll
    for (int k = 0; k < VPT; ++k) {
      const int li = tid + k * kPcgThreads;
      u[k] = r[k] * dinv[k];
      if (own[k]) {
        ub[li] = u[k];
        for (int q = 0; q < D.P; ++q) {
          const uint32_t a = ptab[q * chunk + li];
          if (a) st_remote(a, u[k]);
        }
      }
    }
    if (KIND == 1) {
      __syncthreads();
      // columns of X with rows in this CTA, cgl lanes each
      const int grp = tid / cgl, ln = tid % cgl;
      for (int a0 = 0; a0 < na; a0 += kPcgThreads / cgl) {
        const int a = a0 + grp;
        float acc = 0.f;
        if (a < na) {
          const int q1 = XS || a + 1 < na ? ab[a + 1] : nent;
          for (int q = ab[a] + ln; q < q1; q += 8 * cgl) {
            float v8[8];
#pragma unroll
            for (int s = 0; s < 8; ++s) v8[s] = q + cgl * s < q1 ? cv[q + cgl * s] * ub[crow[q + cgl * s]] : 0.f;
            acc += ((v8[0] + v8[1]) + (v8[2] + v8[3])) + ((v8[4] + v8[5]) + (v8[6] + v8[7]));
          }
        }
        for (int o = cgl >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (a < na && ln == 0) yl[ac[a]] = acc;
      }
      __syncthreads();
      for (int q = wid; q < C; q += kPushWarps) {
        const uint32_t to = push_mapa(push_smem(ys + rank * m), q);
        for (int a = lane; a < m; a += 32) st_remote(to + 4u * a, yl[a]);
      }
    }
    cl.barrier_arrive();
    if (tid == 0 && it > 0) {
      gam_prev = df_div(DF{1.f, 0.f}, gcur);
      alpha_prev = df_mul(dcur, gam_prev);
    }
    cl.barrier_wait();
#pragma unroll
    for (int k = 0; k < VPT; ++k) {
      t[k] = own[k] ? dpc[k] * u[k] - nsum(ub, na3[k][0], na3[k][1], na3[k][2]) : 0.f;
      if (own[k]) tb[tid + k * kPcgThreads] = t[k];
    }
    for (int h = tid; h < nh; h += kPcgThreads) {
      const uint4 q = hn[h];
      tb[q.w] = hd[h] * ub[q.w] - nsum(ub, q.x, q.y, q.z);
    }
    if (KIND == 1) {
      // (from the last thread down: the first ones have a neighbour row besides their own)
      for (int a = kPcgThreads - 1 - tid; a < m; a += kPcgThreads) {
        float v[kMaxCluster];
#pragma unroll
        for (int q = 0; q < kMaxCluster; ++q) v[q] = q < C ? ys[q * m + a] : 0.f;
#pragma unroll
        for (int o = kMaxCluster / 2; o > 0; o >>= 1)
#pragma unroll
          for (int q = 0; q < o; ++q) v[q] += v[q + o];
        sY[a] = sS[a] * v[0];
      }
    }
    __syncthreads();
    DF v0{0.f, 0.f}, v1{0.f, 0.f}, v2{0.f, 0.f};
#pragma unroll
    for (int k = 0; k < VPT; ++k) {
      w[k] = 0.f;
      if (own[k]) {
        float dt = 0.f;
        if (KIND == 0) {
          dt = omt[k] * u[k];
        } else {
#pragma unroll
          for (int q = 0; q < kQ; ++q)
            dt += (qv[k][q].x * sY[qc[k][q].x] + qv[k][q].y * sY[qc[k][q].y]) +
                  (qv[k][q].z * sY[qc[k][q].z] + qv[k][q].w * sY[qc[k][q].w]);
          for (int q = q0r[k] + kQ; q < q1r[k]; ++q) {
            const float4 xa = xv[q];
            const ushort4 ca = xc[q];
            dt += (xa.x * sY[ca.x] + xa.y * sY[ca.y]) + (xa.z * sY[ca.z] + xa.w * sY[ca.w]);
          }
        }
        w[k] = lam * (dpc[k] * t[k] - nsum(tb, na3[k][0], na3[k][1], na3[k][2]) + e * u[k]) + dt;
      }
      // inner products from exact float products, summed in double-float
      v0 = df_add(v0, df_prod(r[k], u[k]));
      v1 = df_add(v1, df_prod(u[k], w[k]));
      v2 = df_add(v2, df_prod(r[k], r[k]));
    }
    {
      const DF v = warp_sum3(v0, v1, v2);
      if ((lane & 7) == 0 && lane < 24) wsum[(lane >> 3) * kPushWarps + wid] = v;
    }
    __syncthreads();
    if (wid == 0) {
      const DF z{0.f, 0.f};
      const bool in = lane < kPushWarps;
      const DF v = warp_sum3(in ? wsum[lane] : z, in ? wsum[kPushWarps + lane] : z, in ? wsum[2 * kPushWarps + lane] : z);
      // eight lanes hold each sum: they push it to two CTAs each
      if (lane < 24)
        for (int q = lane & 7; q < C; q += 8) st_remote(push_mapa(push_smem(slots + 3 * rank + (lane >> 3)), q), v);
    }
    cl.sync();
    if (wid == 0) {
      const DF z{0.f, 0.f};
      const bool in = lane < C;
      const DF v = warp_sum3(in ? slots[3 * lane] : z, in ? slots[3 * lane + 1] : z, in ? slots[3 * lane + 2] : z);
      const DF g = v;  // lane 0
      const DF dl{__shfl_sync(0xffffffffu, v.hi, 8), __shfl_sync(0xffffffffu, v.lo, 8)};
      const DF rh{__shfl_sync(0xffffffffu, v.hi, 16), __shfl_sync(0xffffffffu, v.lo, 16)};
      if (lane == 0) {
        if (it == 0) {
          bb = rh;
          tol2 = tt2 * rh.hi;
        }
        float flag = 0.f;
        DF alpha{0.f, 0.f}, beta{0.f, 0.f};
        if (rh.hi <= tol2) {
          flag = 1.f;
        } else if (it >= A.maxit) {
          flag = 2.f;
        } else {
          // gam_prev and alpha_prev hold the reciprocals of the step before, formed while the
          // first barrier completes: one division stays on the chain
          DF den = dl;
          if (it > 0) {
            beta = df_mul(g, gam_prev);
            den = df_sub(dl, df_mul(df_mul(beta, g), alpha_prev));
          }
          if (!(den.hi > 0.f) || !isfinite(den.hi)) {
            flag = 3.f;
          } else {
            alpha = df_div(g, den);
          }
          gcur = g;
          dcur = den;
        }
        rho = rh;
        scal[0] = flag;
        scal[1] = alpha.hi;
        scal[2] = beta.hi;
      }
    }
    __syncthreads();
    const float flag = scal[0], alpha = scal[1], beta = scal[2];
    if (flag != 0.f) {
      status = flag == 2.f ? 1 : flag == 3.f ? 2 : 0;
      break;
    }
#pragma unroll
    for (int k = 0; k < VPT; ++k) {
      p[k] = it == 0 ? u[k] : u[k] + beta * p[k];
      sv[k] = it == 0 ? w[k] : w[k] + beta * sv[k];
      x[k] += alpha * p[k];
      r[k] -= alpha * sv[k];
    }
    ++it;
  }
#pragma unroll
  for (int k = 0; k < VPT; ++k)
    if (own[k]) A.x[beg + tid + k * kPcgThreads] = (double)x[k];
  if (rank == 0 && tid == 0) {
    const double b2 = (double)bb.hi + (double)bb.lo, rr = (double)rho.hi + (double)rho.lo;
    A.stat->iters = it;
    A.stat->status = status;
    A.stat->relres = b2 > 0.0 ? sqrt(fmax(rr, 0.0) / b2) : 0.0;
    A.stat->bnorm = sqrt(fmax(b2, 0.0));
  }
}

const void* push_fn(int side, const DevPush& d) {
  const int vpt = d.chunk <= kPcgThreads ? 1 : d.chunk <= 2 * kPcgThreads ? 2 : 4;
  if (side == 0)
    return vpt == 1 ? (const void*)pcg_push_kernel<0, 1, false>
                    : vpt == 2 ? (const void*)pcg_push_kernel<0, 2, false> : (const void*)pcg_push_kernel<0, 4, false>;
  if (d.x_smem)
    return vpt == 1 ? (const void*)pcg_push_kernel<1, 1, true>
                    : vpt == 2 ? (const void*)pcg_push_kernel<1, 2, true> : (const void*)pcg_push_kernel<1, 4, true>;
  return vpt == 1 ? (const void*)pcg_push_kernel<1, 1, false>
                  : vpt == 2 ? (const void*)pcg_push_kernel<1, 2, false> : (const void*)pcg_push_kernel<1, 4, false>;
}

cudaLaunchConfig_t push_config(const DevPush& d, int m, cudaStream_t st, cudaLaunchAttribute* at) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(d.csize);
  cfg.blockDim = dim3(kPcgThreads);
  cfg.dynamicSmemBytes = (size_t)push_layout(d, m).bytes;
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = d.csize;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

}  // namespace

bool pcg_push_prepare(DevPush& d, int m, int side) {
  for (d.x_smem = side; d.x_smem >= 0; --d.x_smem) {
    const void* fn = push_fn(side, d);
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = push_config(d, m, nullptr, at);
    int ncl = 0;
    if (push_layout(d, m).bytes <= 227 * 1024 &&
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) == cudaSuccess &&
        cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&ncl, fn, &cfg) == cudaSuccess && ncl > 0)
      return true;
    cudaGetLastError();
  }
  return false;
}

cudaError_t pcg_push_launch(const PcgArgs& a, const DevPush& d, int side, cudaStream_t st) {
  cudaLaunchAttribute at[1];
  const cudaLaunchConfig_t cfg = push_config(d, a.m, st, at);
  PcgArgs a2 = a;
  DevPush d2 = d;
  void* args[] = {&a2, &d2};
  count_launch();
  return cudaLaunchKernelExC(&cfg, push_fn(side, d), args);
}

}  // namespace cr
