// Grid-wide multigrid-preconditioned CG for the ALS sub-problems (Sec. 2.3,
// Eqs. ALS_linsys and ALS_linsys_v): the preconditioner of cr_mg.cu
// (M^-1 = (1 / lam) V(V(.)), V one V-cycle of L + sigma I with two damped-Jacobi
// sweeps before and after the coarse correction), spread over many SMs in one
// cooperative launch.
//
// What bounds it.  A V-cycle is a chain of short dependent sweeps, so the time
// is (number of phases) x (barrier + one gather).  Two things shorten it:
//  - Fewer phases.  With x1 = w D^-1 R, t1 = R - A x1, s1 = w D^-1 t1 the
//    pre-smoothed iterate is x1 + s1 and its residual tt = t1 - A s1, so
//      restriction      P^T tt = S^T t1,            S = P - w D^-1 A P
//      correction + first post-sweep:  y1 = z + S xc,  z = x1 + s1 + w D^-1 tt
//      second post-sweep:              y2 = y1 + w D^-1 (R - A y1):
//    two phases down and two up per level instead of three and three.  On the
//    level above the coarsest, S times the coarsest inverse is formed once per
//    launch (own rows x nc, dense), which leaves no coarse-solve phase.  A
//    three-level PCG iteration takes 19 barriers (the cluster kernel: 28), two more
//    with the v side's Woodbury step.
//  - Many SMs.  The float64 pipe of GB300 issues one warp operation per 16 cycles,
//    so a level-0 sweep over 470 rows per CTA (16-CTA cluster, 7,530 voxels) is
//    1.2 us of float64 arithmetic alone; 76 CTAs hold 99 rows each, and every
//    table of the solve fits shared memory up to about 30,000 rows.  The chain
//    leaves an SM idle most of the time, so its registers and shared memory are
//    kept to a half or a third of it, and CTAs of other handles' solves run beside
//    it (the split and its figures: build_mg_grid in cr_api.cu).
// Vectors that other CTAs gather live in global memory (L2) and are read with
// ld.global.cg after a barrier; everything a row needs for itself stays in the
// CTA's shared memory.  Barriers are those of cr_grid_bar.cuh (bounded).  Sums run
// in a fixed order and every CTA forms the same scalars, so results repeat bit for
// bit and all CTAs take the same branches.
// Measured against the cluster kernel (ms per solve): 7,500 voxels, float64, v side
// with 28 injections 3.00 -> 2.08; 45,000 voxels, float32, u side 6.41 -> 2.62.  An
// iteration of that v side is 102 -> 55 us: 21 barriers and the gathers between them.
// With all 152 SMs for one solve these were 1.91 and 2.27 ms, and eight handles on
// eight threads took turns: 1.22 ms a u-side solve of 7,500 voxels against 0.32 in
// clusters, 0.33 now.
#include <algorithm>

#include "cr_common.cuh"
#include "cr_grid_bar.cuh"

namespace cr {

namespace {

constexpr double kOm = 2.0 / 3.0;

__device__ __forceinline__ double warp_sum_all(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <class T>
__device__ __forceinline__ T lanes_sum(T v, int G) {
  for (int o = G >> 1; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o, G);
  return v;
}

template <int N>
struct Int {
  static constexpr int value = N;
};

template <int KIND, class T, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == kMgGridFew ? kMgGridFewCtas : 2) pcg_mg_grid_kernel(const PcgArgs A, const DevMg G, const DevMgGrid D) {
  const int b = blockIdx.x, nb = D.nb;
  const int tid = threadIdx.x, nth = blockDim.x;
  const int lane = tid & 31, wid = tid >> 5, nw = nth >> 5;
  const DevLap& L = A.L;
  const int m = A.m, nc = G.nc, nlev = G.nlev;
  const int K = L.K;
  const bool smw = KIND == 1 && G.smw;
  extern __shared__ __align__(16) char smraw[];
  __shared__ double scal[16];
  __shared__ double scr[3 * 32];
  double* sS = reinterpret_cast<double*>(smraw + D.o_m);  // [m] xi^2 or s
  double* sY = sS + m;                                    // [m]
  double* smw_ci = sY + m;                                // [m * m] (smw)
  double* smw_g = smw_ci + (smw ? m * m : 0);             // [m]
  char* tab = D.tab_smem ? smraw + D.o_tab : D.tab_glob + (size_t)b * D.tab_bytes;

  const double lam = A.lam, c = A.coef[0], d = A.coef[1], e = d - c * c;
  const T om = (T)kOm;

  GridBar bar = grid_bar(D.bar, D.err);
  auto gsync = [&]() { grid_bar_sync(bar); };

  auto nown = [&](int l) -> int { return max(0, min(G.lev[l].n - b * D.lev[l].chunk, D.lev[l].chunk)); };
  auto gbeg = [&](int l) -> int { return b * D.lev[l].chunk; };
  // own vector k of level l in shared memory
  auto own = [&](int l, int k) -> T* {
    return reinterpret_cast<T*>(smraw + D.lev[l].o_own) + (size_t)k * D.lev[l].chunk;
  };
  // global vector k of level l: 0 x1, 1 t1, 2 s1, 3 y1, 4 xc (level 0: u), 5 (level 0: t)
  auto gv = [&](int l, int k) -> T* { return reinterpret_cast<T*>(D.lev[l].g) + (size_t)k * G.lev[l].n; };
  // lanes per row for `rows` rows of this CTA
  auto gsize = [&](int rows) -> int {
    int g = 1;
    while (g < 32 && 2 * g * rows <= nth) g *= 2;
    return g;
  };
  const int beg0 = gbeg(0), n0 = nown(0);
  enum { O_R, O_X1, O_S1, O_Z, O_Y1, O_DI, O_T1, O_U, O_P, O_SV, O_X, O_OM, O_W, O_TT, O_RR, O_DG };  // level 0
  // levels >= 1 use O_R .. O_T1

  // ---- set-up: data weights, shift ----------------------------------------------------
  for (int a = tid; a < m; a += nth) sS[a] = KIND == 0 ? A.xi[a] * A.xi[a] : A.s[a];
  __syncthreads();
  if (wid == 0) {
    double wb = 0.0;
    for (int a = lane; a < m; a += 32) wb += KIND == 0 ? sS[a] : sS[a] * G.xn2[a];
    wb = warp_sum_all(wb);
    if (lane == 0) {
      // (float64 divisions and roots cost hundreds of cycles and share one pipe: one thread forms them)
      if (KIND == 1) wb /= (double)L.n;
      const double sig_now = sqrt(fmax(d + wb / lam, 1e-12));
      // the v side's correction keeps the shift its cache was formed with while the new one
      // stays within 25 % of it (same inputs in every CTA: same decision)
      double sg = sig_now, build = 0.0;
      if (smw) {
        const double sref = G.smw_sig[0];
        build = G.smw_sig[1] == (double)sizeof(T) && sref > 0.0 && fabs(sig_now / sref - 1.0) <= 0.25 ? 0.0 : 1.0;
        if (build == 0.0) sg = sref;
      }
      scal[0] = sg;
      scal[1] = build;
      scal[3] = 1.0 / lam;
    }
  }
  __syncthreads();
  const double sigd = scal[0];
  const bool smw_build = smw && scal[1] != 0.0;
  const T sig = (T)sigd;
  // inverse diagonals of every level (global: the coefficients of S^T need the owners' values)
  for (int l = 0; l < nlev - 1; ++l) {
    T* di = own(l, O_DI);
    for (int li = tid; li < nown(l); li += nth) {
      const int i = gbeg(l) + li;
      const double dd = l == 0 ? L.diag[i] + sigd : G.lev[l].dl[i] + sigd * G.lev[l].dm[i];
      const double inv = dd > 0.0 ? 1.0 / dd : 0.0;
      D.lev[l].dinv[i] = inv;
      di[li] = om * (T)inv;
      if (l == 0) own(0, O_DG)[li] = (T)L.diag[i];
    }
  }
  for (int li = tid; li < n0; li += nth) {
    const double x0 = A.x[beg0 + li];
    own(0, O_X)[li] = (T)x0;
    gv(0, 4)[beg0 + li] = (T)x0;
  }
  if (KIND == 0) {
    // omega_tilde of the own rows, a lane group per row
    const int g = gsize(D.lev[0].chunk), rpp = nth / g, ln = tid % g;
    for (int base = 0; base < n0; base += rpp) {
      const int li = base + tid / g;
      double o = 0.0;
      if (li < n0) {
        const uint8_t* om8 = A.Om + beg0 + li;
#pragma unroll 4
        for (int a = ln; a < m; a += g) o += (double)om8[(int64_t)a * A.ldo] * sS[a];
      }
      o = lanes_sum(o, g);
      if (li < n0 && ln == 0) own(0, O_OM)[li] = (T)o;
    }
  }
  // level 0 neighbour table
  int* nbt = reinterpret_cast<int*>(tab + D.o_nb);
  T* nbw = D.o_nbw >= 0 ? reinterpret_cast<T*>(tab + D.o_nbw) : nullptr;
  const int ch0 = D.lev[0].chunk;
  for (int t = tid; t < K * n0; t += nth) {
    const int k = t / n0, li = t % n0;
    const int q = L.nbr[(size_t)k * L.n + beg0 + li];
    nbt[k * ch0 + li] = q;
    if (nbw) nbw[k * ch0 + li] = q >= 0 ? (T)L.offw[(size_t)k * L.n + beg0 + li] : (T)0;
  }
  gsync();
  // tables: operator rows (levels >= 1), S rows (all but the last fine level), S^T rows
  for (int l = 0; l < nlev - 1; ++l) {
    const DevMgLevel& V = G.lev[l];
    const DevMgGridLevel& W = D.lev[l];
    const int no = nown(l), gb = gbeg(l);
    if (l >= 1 && no > 0) {
      int* rp = reinterpret_cast<int*>(tab + W.o_rp);
      int* ci = reinterpret_cast<int*>(tab + W.o_ci);
      T* cv = reinterpret_cast<T*>(tab + W.o_cv);
      const int q0 = V.rp[gb], q1 = V.rp[gb + no];
      for (int li = tid; li <= no; li += nth) rp[li] = V.rp[gb + li] - q0;
      for (int q = q0 + tid; q < q1; q += nth) {
        const int pk = V.cp[q];
        ci[q - q0] = V.dist ? (pk >> 24) * V.chunk + (pk & 0xFFFFFF) : pk;
        cv[q - q0] = (T)(V.lv[q] + sigd * V.mv[q]);
      }
    }
    if (l < nlev - 2 && no > 0) {
      int* rp = reinterpret_cast<int*>(tab + W.o_srp);
      int* ci = reinterpret_cast<int*>(tab + W.o_sci);
      T* cv = reinterpret_cast<T*>(tab + W.o_scv);
      const int q0 = W.srp[gb];
      for (int li = tid; li <= no; li += nth) rp[li] = W.srp[gb + li] - q0;
      const int g = gsize(W.chunk), rpp = nth / g, ln = tid % g;
      for (int li = tid / g; li < no; li += rpp) {
        const double wd = kOm * __ldcg(W.dinv + gb + li);
        for (int q = W.srp[gb + li] + ln; q < W.srp[gb + li + 1]; q += g) {
          ci[q - q0] = W.sci[q];
          cv[q - q0] = (T)(W.sp[q] - wd * (W.sl[q] + sigd * W.sm[q]));
        }
      }
    }
    const int n1 = nown(l + 1), g1 = gbeg(l + 1);
    if (n1 > 0) {
      int* rp = reinterpret_cast<int*>(tab + W.o_trp);
      int* ci = reinterpret_cast<int*>(tab + W.o_tci);
      T* cv = reinterpret_cast<T*>(tab + W.o_tcv);
      const int q0 = W.trp[g1], q1 = W.trp[g1 + n1];
      for (int li = tid; li <= n1; li += nth) rp[li] = W.trp[g1 + li] - q0;
      for (int q = q0 + tid; q < q1; q += nth) {
        const int i = W.tci[q];
        ci[q - q0] = i;
        cv[q - q0] = (T)(W.tp[q] - kOm * __ldcg(W.dinv + i) * (W.tl[q] + sigd * W.tm[q]));
      }
    }
  }
  {
    // level above the coarsest: rows of S (L_c + sigma M_c)^-1 = S Q diag(1 / (mu + sigma)) Q^T
    const int l = nlev - 2, no = nown(l), gb = gbeg(l);
    const DevMgGridLevel& W = D.lev[l];
    T* Tm = reinterpret_cast<T*>(tab + W.o_scv);  // own rows x nc
    double* sq = reinterpret_cast<double*>(tab + W.o_sq);  // own rows x nc
    for (int t = tid; t < no * nc; t += nth) {
      const int li = t / nc, q = t % nc;
      double acc = 0.0;
      for (int s = W.srp[gb + li]; s < W.srp[gb + li + 1]; ++s) {
        const double sv = W.sp[s] - kOm * __ldcg(W.dinv + gb + li) * (W.sl[s] + sigd * W.sm[s]);
        acc += sv * G.cQ[W.sci[s] + (size_t)q * nc];
      }
      sq[t] = acc / (fmax(G.cmu[q], 0.0) + sigd);
    }
    __syncthreads();
    for (int t = tid; t < no * nc; t += nth) {
      const int li = t / nc, k = t % nc;
      double acc = 0.0;
      for (int q = 0; q < nc; ++q) acc += sq[li * nc + q] * G.cQ[k + (size_t)q * nc];
      Tm[t] = (T)acc;
    }
  }
  __syncthreads();

  T* const DG = own(0, O_DG);
  // ---- row helpers ----------------------------------------------------------------------
  // (L + shift I) x on level 0, own row li; x the published vector, xo its own value
  auto lap0 = [&](int li, const T* x, T xo, T shift) -> T {
    T acc = (DG[li] + shift) * xo;
    if (K <= 6) {
      T nv[6];
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const int q = k < K ? nbt[k * ch0 + li] : -1;
        nv[k] = q >= 0 ? __ldcg(x + q) : (T)0;
      }
      if (nbw) {
#pragma unroll
        for (int k = 0; k < 6; ++k)
          if (k < K) acc += nbw[k * ch0 + li] * nv[k];
      } else {
        acc -= ((nv[0] + nv[1]) + (nv[2] + nv[3])) + (nv[4] + nv[5]);
      }
      return acc;
    }
    for (int k = 0; k < K; ++k) {
      const int q = nbt[k * ch0 + li];
      if (q >= 0) acc += (nbw ? nbw[k * ch0 + li] : (T)-1) * __ldcg(x + q);
    }
    return acc;
  };
  // this lane's share of table row li against the published vector x
  auto trow = [&](int64_t o_rp, int64_t o_ci, int64_t o_cv, int li, int ln, int g, const T* x) -> T {
    const int* rp = reinterpret_cast<const int*>(tab + o_rp);
    const int* ci = reinterpret_cast<const int*>(tab + o_ci);
    const T* cv = reinterpret_cast<const T*>(tab + o_cv);
    T acc = (T)0;
    const int q1 = rp[li + 1];
    for (int q = rp[li] + ln; q < q1; q += 8 * g) {  // eight entries in flight per lane
      T v[8], w[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int qq = q + u * g;
        w[u] = qq < q1 ? cv[qq] : (T)0;
        v[u] = qq < q1 ? __ldcg(x + ci[qq]) : (T)0;
      }
      acc += ((w[0] * v[0] + w[1] * v[1]) + (w[2] * v[2] + w[3] * v[3])) +
             ((w[4] * v[4] + w[5] * v[5]) + (w[6] * v[6] + w[7] * v[7]));
    }
    return acc;
  };
  // f(li, sum) for every own row of level l: sum = part(li, lane, g) added over the row's group of
  // g lanes; threads [t0, t0 + nt) take part (whole warps)
  auto grows = [&](int l, int g, int t0, int nt, auto&& part, auto&& fin) {
    const int tt = tid - t0;
    if (tt < 0 || tt >= nt) return;
    const int no = nown(l);
    const int rpp = nt / g, ln = tt % g;
    for (int base = 0; base < no; base += rpp) {
      const int li = base + tt / g;
      T s = li < no ? part(li, ln, g) : (T)0;
      s = lanes_sum(s, g);
      if (li < no && ln == 0) fin(li, s);
    }
  };
  // A_l x for own rows: fin(li, (A x)_li); xk = own copy of x (level 0)
  auto arows = [&](int l, int t0, int nt, const T* x, const T* xo, auto&& fin) {
    if (l == 0) {
      if (tid >= t0)
        for (int li = tid - t0; li < n0; li += nt) fin(li, lap0(li, x, xo[li], sig));
    } else {
      const DevMgGridLevel& W = D.lev[l];
      grows(l, W.g_op, t0, nt, [&](int li, int ln, int g) { return trow(W.o_rp, W.o_ci, W.o_cv, li, ln, g, x); }, fin);
    }
  };
  // partial q added over the CTAs, in every lane of the calling warp
  auto part_total = [&](int q) -> double {
    double t = 0.0;
    for (int k = lane; k < nb; k += 8 * 32) {
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = k + 32 * u < nb ? __ldcg(D.part + 4 * (k + 32 * u) + q) : 0.0;
      t += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
    return warp_sum_all(t);
  };
  // |r|^2 <= tol^2 |b|^2 decided inside the first V-cycle of an iteration: the last warp adds
  // the partials while the others work on the first sweep
  double tol2 = 0.0;
  // V-cycle of the right side in own(0, O_R), x1 published; result through fin(li, y2).
  // check: stop (return false) when the residual norm published with x1 meets the target.
  auto vcycle = [&](bool check, auto&& fin) -> bool {
    if (check && wid == nw - 1) {
      const double t = part_total(3);
      if (lane == 0) scal[8] = t;
    }
    for (int l = 0; l < nlev - 1; ++l) {
      T* R = own(l, O_R);
      T* X1 = own(l, O_X1);
      T* S1 = own(l, O_S1);
      T* T1 = own(l, O_T1);
      T* Z = own(l, O_Z);
      T* DI = own(l, O_DI);
      const int gb = gbeg(l);
      T *gt = gv(l, 1) + gb, *gs = gv(l, 2) + gb;
      arows(l, 0, nth, gv(l, 0), X1, [&](int li, T ax) {
        const T t1 = R[li] - ax, s1 = DI[li] * t1;
        T1[li] = t1;
        S1[li] = s1;
        gt[li] = t1;
        gs[li] = s1;
      });
      gsync();
      if (check && l == 0 && (scal[8] <= tol2 || bar.dead)) return false;
      {
        const DevMgGridLevel& W = D.lev[l];
        const T* x = gv(l, 1);
        const int g1 = gbeg(l + 1);
        auto part = [&](int li, int ln, int g) { return trow(W.o_trp, W.o_tci, W.o_tcv, li, ln, g, x); };
        if (l + 1 == nlev - 1) {
          T* rc = reinterpret_cast<T*>(D.rc);
          grows(l + 1, W.g_t, 0, nth / 2, part, [&](int li, T v) { rc[g1 + li] = v; });
        } else {
          T *R1 = own(l + 1, O_R), *X11 = own(l + 1, O_X1), *DI1 = own(l + 1, O_DI), *gx = gv(l + 1, 0) + g1;
          grows(l + 1, W.g_t, 0, nth / 2, part, [&](int li, T v) {
            const T x1 = DI1[li] * v;
            R1[li] = v;
            X11[li] = x1;
            gx[li] = x1;
          });
        }
      }
      // the other half of the warps: nothing reads z before the way up
      arows(l, nth / 2, nth / 2, gv(l, 2), S1, [&](int li, T as) { Z[li] = X1[li] + S1[li] + DI[li] * (T1[li] - as); });
      gsync();
    }
    for (int l = nlev - 2; l >= 0; --l) {
      T* R = own(l, O_R);
      T* Y1 = own(l, O_Y1);
      T* Z = own(l, O_Z);
      T* DI = own(l, O_DI);
      const DevMgGridLevel& W = D.lev[l];
      const int gb = gbeg(l);
      T* gy = gv(l, 3) + gb;
      auto put = [&](int li, T v) {
        const T y = Z[li] + v;
        Y1[li] = y;
        gy[li] = y;
      };
      if (l == nlev - 2) {
        const T* rc = reinterpret_cast<const T*>(D.rc);
        const T* Tm = reinterpret_cast<const T*>(tab + W.o_scv);
        grows(l, W.g_s, 0, nth,
              [&](int li, int ln, int g) {
                T acc = (T)0;
                for (int k = ln; k < nc; k += 8 * g) {
                  T v[8];
#pragma unroll
                  for (int u = 0; u < 8; ++u) v[u] = k + u * g < nc ? __ldcg(rc + k + u * g) : (T)0;
#pragma unroll
                  for (int u = 0; u < 8; ++u) v[u] *= k + u * g < nc ? Tm[li * nc + k + u * g] : (T)0;
                  acc += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
                }
                return acc;
              },
              put);
      } else {
        const T* x = gv(l + 1, 4);
        grows(l, W.g_s, 0, nth, [&](int li, int ln, int g) { return trow(W.o_srp, W.o_sci, W.o_scv, li, ln, g, x); }, put);
      }
      gsync();
      if (l > 0) {
        T* gx = gv(l, 4) + gb;
        arows(l, 0, nth, gv(l, 3), Y1, [&](int li, T ay) { gx[li] = Y1[li] + DI[li] * (R[li] - ay); });
        gsync();
      } else {
        arows(0, 0, nth, gv(0, 3), Y1, [&](int li, T ay) { fin(li, Y1[li] + DI[li] * (R[li] - ay)); });
      }
    }
    return true;
  };
  T* const R0 = own(0, O_R);
  T* const X10 = own(0, O_X1);
  T* const DI0 = own(0, O_DI);
  T* const U0 = own(0, O_U);
  // publish x1 = w D^-1 R for the V-cycle of R
  auto start = [&](int li, T r) {
    const T x1 = DI0[li] * r;
    R0[li] = r;
    X10[li] = x1;
    gv(0, 0)[beg0 + li] = x1;
  };
  // y_a = X_a^T x of the published vector x, one CTA per column, into D.ytot (half the warps: the
  // sum over a CTA costs float64 issue slots per warp)
  auto xt_cols = [&](const T* x) {
    const int nt = nth / 2, w0 = nw / 2;  // the upper warps: the lower ones work on t
    for (int a = b; a < m; a += nb) {
      const int p0 = D.xc_ptr[a], p1 = D.xc_ptr[a + 1];
      if (wid >= w0) {
        double acc = 0.0;
        for (int q = p0 + tid - nt; q < p1; q += 4 * nt) {
          double v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int qq = q + u * nt;
            v[u] = qq < p1 ? D.xc_val[qq] * (double)__ldcg(x + D.xc_row[qq]) : 0.0;
          }
          acc += (v[0] + v[1]) + (v[2] + v[3]);
        }
        acc = warp_sum_all(acc);
        if (lane == 0) scr[wid - w0] = acc;
      }
      __syncthreads();
      if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < w0; ++w) t += scr[w];
        D.ytot[a] = t;
      }
      if (a + nb < m) __syncthreads();
    }
  };
  auto data = [&](int li, T xo) -> T {
    if (KIND == 0) return own(0, O_OM)[li] * xo;
    const int i = beg0 + li;
    double acc = 0.0;
    const int q1 = A.X.xr_ptr[i + 1];
    for (int q = A.X.xr_ptr[i]; q < q1; ++q) acc += A.X.xr_val[q] * sY[A.X.xr_col[q]];
    return (T)acc;
  };
  // sums of v[0..CNT) over the CTA (rows sit in the first `aw` warps), partials to D.part
  const int aw = min(nw, (ch0 + 31) / 32);
  auto partials = [&](auto& v, auto cnt, int first) {
    constexpr int CNT = decltype(cnt)::value;
    if (wid < aw) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < CNT; ++q) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
      if (lane == 0)
#pragma unroll
        for (int q = 0; q < CNT; ++q) scr[q * 32 + wid] = v[q];
    }
    __syncthreads();
    if (tid < CNT) {
      double t = 0.0;
      for (int w = 0; w < aw; ++w) t += scr[tid * 32 + w];
      D.part[4 * b + first + tid] = t;
    }
  };
  const T cT = (T)c, lamT = (T)lam, eT = (T)e, ilam = (T)scal[3];
  T* const TT = own(0, O_TT);
  T* const W0 = own(0, O_W);
  T* const Xs = own(0, O_X);
  T* const gu = gv(0, 4);
  T* const gt0 = gv(0, 5);

  // ---- v side: Sherman-Morrison-Woodbury correction (see cr_mg.cu) ----------------------
  T* const mx = reinterpret_cast<T*>(G.smw_mx);
  if (smw) {
    if (smw_build) {
      for (int a = 0; a < m; ++a) {
        for (int li = tid; li < n0; li += nth) {
          const int i = beg0 + li;
          double xa = 0.0;
          for (int q = A.X.xr_ptr[i]; q < A.X.xr_ptr[i + 1]; ++q)
            if (A.X.xr_col[q] == a) xa += A.X.xr_val[q];
          start(li, (T)xa);
        }
        gsync();
        vcycle(false, [&](int li, T y) { start(li, y); });
        gsync();
        vcycle(false, [&](int li, T y) { mx[(size_t)(beg0 + li) * m + a] = ilam * y; });
      }
      gsync();
      // X^T MX: column a of X against every column of MX
      for (int a = b; a < m; a += nb) {
        const int p0 = D.xc_ptr[a], p1 = D.xc_ptr[a + 1];
        for (int w2 = wid; w2 < m; w2 += nw) {
          double acc = 0.0;
          for (int q = p0 + lane; q < p1; q += 32)
            acc += D.xc_val[q] * (double)__ldcg(mx + (size_t)D.xc_row[q] * m + w2);
          acc = warp_sum_all(acc);
          if (lane == 0) G.smw_xx[a * m + w2] = acc;
        }
      }
      if (b == 0 && tid == 0 && !bar.dead) {
        G.smw_sig[0] = sigd;
        G.smw_sig[1] = (double)sizeof(T);
      }
      gsync();
    }
    // (I + D X^T MX D)^-1 by Gauss-Jordan (symmetric positive definite: no pivoting), in every CTA
    for (int idx = tid; idx < m * m; idx += nth) {
      const int a = idx / m, q = idx % m;
      smw_ci[idx] = (a == q ? 1.0 : 0.0) + sqrt(fmax(sS[a], 0.0)) * __ldcg(G.smw_xx + idx) * sqrt(fmax(sS[q], 0.0));
    }
    __syncthreads();
    for (int k = 0; k < m; ++k) {
      if (tid < 32) {  // row and column k before the step, the row scaled (m <= 32)
        const double piv = smw_ci[k * m + k];
        const double cc = tid < m ? smw_ci[tid * m + k] : 0.0, rr = tid < m ? smw_ci[k * m + tid] : 0.0;
        const double pinv = 1.0 / piv;
        __syncwarp();
        if (tid < m) {
          smw_g[tid] = cc;
          smw_ci[k * m + tid] = (tid == k ? 1.0 : rr) * pinv;
        }
      }
      __syncthreads();
      for (int idx = tid; idx < m * m; idx += nth) {
        const int a = idx / m, q = idx % m;
        if (a != k) smw_ci[idx] = (q == k ? 0.0 : smw_ci[idx]) - smw_g[a] * smw_ci[k * m + q];
      }
      __syncthreads();
    }
    for (int idx = tid; idx < m * m; idx += nth)
      smw_ci[idx] *= sqrt(fmax(sS[idx / m], 0.0)) * sqrt(fmax(sS[idx % m], 0.0));  // Q = D C^-1 D
    __syncthreads();
    // With y = X^T u0 (u0 = M0^-1 r) the correction is u = u0 - MX Q y: the rows of MX Q are formed
    // here for the own rows (MX of the own rows was written by this CTA, so ordinary loads see it).
    // The operator is then applied to the u that enters x.  Its data term also follows from y
    // (S X^T u = Q y), and t from stored rows of (L + cI) MX Q, which would save a phase, but in the
    // span of X u0 is much larger than u, and A u then differs from that of the rounded u by u0's
    // rounding: float64 solves for 1e-13 (3,000 rows, 5 to 32 injections, lambda 1 to 300) left
    // 1.4e-13 to 4.7e-12 of the right side, against 5e-14 to 1.2e-13.
    for (int idx = tid; idx < n0 * m; idx += nth) {
      const int li = idx / m, q = idx % m, i = beg0 + li;
      const T* row = mx + (size_t)i * m;
      double acc = 0.0;
#pragma unroll 4
      for (int a = 0; a < m; ++a) acc += (double)row[a] * smw_ci[a * m + q];
      reinterpret_cast<T*>(D.smw_rows)[(size_t)i * m + q] = (T)acc;
    }
    __syncthreads();
  }
  // after the barrier behind u0 (published): the corrected u of the own rows, published
  auto smw_correct = [&]() {
    xt_cols(gu);
    gsync();
    for (int a = tid; a < m; a += nth) sY[a] = __ldcg(D.ytot + a);
    __syncthreads();
    // two lanes per row: sums over more lanes would add to the float64 pipe's work
    const int ln = tid % 2, rpp = nth / 2;
    for (int base = 0; base < n0; base += rpp) {
      const int li = base + tid / 2;
      T acc = (T)0;
      if (li < n0) {
        const T* row = reinterpret_cast<const T*>(D.smw_rows) + (size_t)(beg0 + li) * m;
#pragma unroll 4
        for (int q = ln; q < m; q += 2) acc += row[q] * (T)sY[q];
      }
      acc += __shfl_xor_sync(0xffffffffu, acc, 1);
      if (li < n0 && ln == 0) {
        const T u = U0[li] - acc;
        U0[li] = u;
        gu[beg0 + li] = u;
      }
    }
    gsync();
  };

  // ---- r0 = b - A x0 --------------------------------------------------------------------
  auto op_t = [&](const T* uo) {  // t = (L + cI) u published; v side: X^T u
    for (int li = tid; li < n0; li += nth) {
      const T t = lap0(li, gu, uo[li], cT);
      TT[li] = t;
      gt0[beg0 + li] = t;
    }
    if (KIND == 1) xt_cols(gu);
  };
  auto load_y = [&]() {
    if (KIND == 1) {
      for (int a = tid; a < m; a += nth) sY[a] = sS[a] * __ldcg(D.ytot + a);
      __syncthreads();
    }
  };
  gsync();
  op_t(Xs);
  gsync();
  load_y();
  {
    double v[2] = {0.0, 0.0};
    for (int li = tid; li < n0; li += nth) {
      const T xi = Xs[li];
      const T wi = lamT * (lap0(li, gt0, TT[li], cT) + eT * xi) + data(li, xi);
      const double bi = A.b[beg0 + li];
      const T r = (T)(bi - (double)wi);
      start(li, r);
      v[0] += bi * bi;
      v[1] += (double)r * (double)r;
    }
    partials(v, Int<2>{}, 2);  // |b|^2 and |r|^2
  }
  gsync();
  if (wid == 0) {
    const double t = part_total(2);
    if (lane == 0) scal[2] = t;
  }
  __syncthreads();
  const double bb = scal[2];
  tol2 = A.tol * A.tol * bb;
  int it = 0, status = 0;
  double igam_prev = 1.0, ialpha_prev = 1.0;  // 1 / gamma and 1 / alpha of the step before (thread 0)
  // own copy of r: the V-cycles overwrite O_R
  T* const Pv = own(0, O_P);
  T* const Sv = own(0, O_SV);
  T* const Rr = own(0, O_RR);
  for (int li = tid; li < n0; li += nth) Rr[li] = R0[li];
  while (bb > 0.0 && !bar.dead) {
    // u = M^-1 r = (1 / lam) V(V(r))
    if (!vcycle(true, [&](int li, T y) { start(li, y); })) break;
    if (it >= A.maxit) {
      status = 1;
      break;
    }
    gsync();
    vcycle(false, [&](int li, T y) {
      const T u = ilam * y;
      U0[li] = u;
      gu[beg0 + li] = u;
    });
    gsync();
    if (smw) smw_correct();
    op_t(U0);
    gsync();
    load_y();
    double v[2] = {0.0, 0.0};
    for (int li = tid; li < n0; li += nth) {
      const T ui = U0[li];
      const T wi = lamT * (lap0(li, gt0, TT[li], cT) + eT * ui) + data(li, ui);
      W0[li] = wi;
      v[0] += (double)Rr[li] * (double)ui;
      v[1] += (double)ui * (double)wi;
    }
    partials(v, Int<2>{}, 0);
    gsync();
    // the recurrence's scalars, formed once per CTA: one division on the dependent chain
    if (wid < 2) {
      const double t = part_total(wid);
      if (lane == 0) scal[wid] = t;
    }
    __syncthreads();
    if (tid == 0) {
      const double gam = scal[0], del = scal[1];
      double beta = 0.0, den = del;
      if (it > 0) {
        beta = gam * igam_prev;
        den = del - beta * gam * ialpha_prev;
      }
      const bool bad = !(den > 0.0) || !isfinite(den);
      scal[4] = bad ? 0.0 : gam / den;
      scal[5] = beta;
      scal[6] = bad ? 1.0 : 0.0;
      igam_prev = 1.0 / gam;
      ialpha_prev = den * igam_prev;
    }
    __syncthreads();
    if (scal[6] != 0.0) {
      status = 2;
      break;
    }
    const T aT = (T)scal[4], bT = (T)scal[5];
    double rr[1] = {0.0};
    for (int li = tid; li < n0; li += nth) {
      const T pi = it == 0 ? U0[li] : U0[li] + bT * Pv[li];
      const T si = it == 0 ? W0[li] : W0[li] + bT * Sv[li];
      Pv[li] = pi;
      Sv[li] = si;
      Xs[li] += aT * pi;
      const T r = Rr[li] - aT * si;
      Rr[li] = r;
      start(li, r);
      rr[0] += (double)r * (double)r;
    }
    partials(rr, Int<1>{}, 3);
    ++it;
    gsync();
  }
  __syncthreads();
  for (int li = tid; li < n0; li += nth) A.x[beg0 + li] = bb > 0.0 ? (double)Xs[li] : 0.0;
  if (b == 0 && tid == 0) {
    const double rho = scal[8];
    A.stat->iters = it;
    A.stat->status = bar.dead ? 3 : status;
    A.stat->relres = bb > 0.0 ? sqrt(rho / bb) : 0.0;
    A.stat->bnorm = sqrt(bb);
  }
}

template <int THREADS>
const void* mg_grid_fn_t(int side, bool f32) {
  if (f32)
    return side == 0 ? (const void*)pcg_mg_grid_kernel<0, float, THREADS> : (const void*)pcg_mg_grid_kernel<1, float, THREADS>;
  return side == 0 ? (const void*)pcg_mg_grid_kernel<0, double, THREADS> : (const void*)pcg_mg_grid_kernel<1, double, THREADS>;
}

const void* mg_grid_fn(int side, bool f32, int threads) {
  return threads == kMgGridFew ? mg_grid_fn_t<kMgGridFew>(side, f32) : mg_grid_fn_t<kMgGridMany>(side, f32);
}

}  // namespace

bool mg_grid_prepare(const DevMgGrid& D) {
  for (int side = 0; side < 2; ++side)
    for (int f = 0; f < 2; ++f) {
      int per = 0;
      if (cudaFuncSetAttribute(mg_grid_fn(side, f == 0, D.threads), cudaFuncAttributeMaxDynamicSharedMemorySize,
                               kMgGridSmemMax) != cudaSuccess ||
          cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, mg_grid_fn(side, f == 0, D.threads), D.threads, D.smem) !=
              cudaSuccess ||
          per < 1) {
        cudaGetLastError();
        return false;
      }
    }
  return true;
}

cudaError_t mg_grid_launch(const PcgArgs& a, const DevMg& g, const DevMgGrid& d, int side, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(d.bar, 0, 2 * sizeof(unsigned), st);  // the barrier's counter and error word
  if (e != cudaSuccess) return e;
  PcgArgs a2 = a;
  DevMg g2 = g;
  DevMgGrid d2 = d;
  void* args[] = {&a2, &g2, &d2};
  count_launch();
  return cudaLaunchCooperativeKernel(mg_grid_fn(side, a.fp32 != 0, d.threads), dim3(d.nb), dim3(d.threads), args, d.smem, st);
}

}  // namespace cr
