// The solution pass over W = P V^T (P = U Z) on the tensor cores, exact to the
// last step (Secs. 3 and 4; the float64 form is in cr_post.cu).
//
// The pass is 2 (j + j*) flops per entry of W, and GB300's float64 rate (1.26
// TFLOP/s) bounds it: 24.5 ms at 7,530^2 with ranks 100 and 140.  Here each row of
// P and of V is scaled by a power of two and written as eight signed 8-bit digits
// (integers in [-128, 128], exact in bfloat16), the scheme of Ozaki, Ogita, Oishi
// and Rump for error-free products:
//   P(i, k) = 2^(eP_i - 7) sum_s p_s(i, k) 2^(-8 s),   V(c, k) likewise,
//   W(i, c) = 2^(eP_i + eV_c - 14) sum_l 2^(-8 l) L_l,  L_l = sum_{s + t = l} sum_k p_s v_t.
// Every product is an integer of at most 2^14 and every partial sum of a level over
// at most 112 columns stays below 2^24, so bfloat16 matrix instructions with float32
// accumulation form L_0 .. L_7 without a rounding error.  Two 48-bit integers hold
// the eight levels; one float64 FMA and one scaled addition per 112 columns turn them
// into W.
// What is left out, levels 8 and up (seven products of at most 2^14 2^-64 a column and
// less behind them) and the factors' digits 9 and up, is below E = 9.1 K 2^-50 in units
// of 2^(eP_i + eV_c - 14).  A float64 sum rounds by K 2^-53 S, S = sum_k |P(i, k)| |V(c, k)|
// in the same units, however much smaller than the rows' largest entries S is.  So
// post_check_kernel first forms T = sum_k |p_0| |v_0|, one matrix product of the 36: a
// digit that is not zero is at most twice its entry, hence S >= T / 4, and T >= 512
// makes E at most 0.57 of the float64 sum's bound.  Tiles of 64 x 64 entries in which
// some T is smaller (rows whose large entries do not meet, and the sign and size of W
// there) go to the float64 pass, the others come from the digits.
// Measured (7,530^2 entries, ms per report): rank 100 against rank 140 25.2 -> 5.8 (0.4
// of them the check), rank 100 alone 11.8 -> 2.5, rank 1 2.6 -> 1.6 (what the
// statistics' float64 operations take); W's error against extended precision
// 6.6e-16 -> 3.9e-16 at rank 140.  A warp holds 16 x 16 entries (eight levels: 64 accumulators), eight warps a
// CTA and two CTAs an SM; W and the statistics wait in shared memory meanwhile (kept
// in registers they spilled: 5.8 ms; one CTA of 64 x 64 entries: 6.7 ms).  At rank 100
// alone the float64 pipe is 63 % busy (level sums, statistics) and the tensor pipe 41 %,
// in turns: the two CTAs of an SM overlap the phases only in part.  The check's 0.21 ms
// are latency of its operand loads.
#include <cuda_bf16.h>

#include <algorithm>

#include "cr_common.cuh"
#include "cr_post_stats.cuh"

namespace cr {

namespace {

constexpr int kS = 8;               // digits
constexpr int kTm = 64, kTn = 32;   // tile of W
constexpr int kKs = 16;             // columns staged at once: one matrix step
constexpr int kStageP = kS * kTm * kKs * 2, kStageV = kS * kTn * kKs * 2;  // bytes
constexpr int kNt = 2;              // 8-column matrix tiles per warp (4 x 2 warps of 16 x 16)
// two stages, the tiles of W and of the reference, and the threads' statistics: 97 KB, two CTAs per SM
constexpr int kSmem = 2 * (kStageP + kStageV) + (2 * 4 * kNt + PS_N) * 8 * 256;
constexpr int kChunk = 112;         // columns whose level sums stay below 2^24
constexpr int kPcThreads = 256;

// exponent e with |x| < 2^e for every |x| <= m
__device__ __forceinline__ int pow2_above(double m) {
  int e = 0;
  frexp(m, &e);
  return e;
}

// Digits of the rows of A (n x K, A(r, k) at A[r + k lda]): plane s of row r at
// out + (s * n + r) * Kp (k contiguous, zero-padded to Kp), scale[r] = 2^(e_r - 35) (0: a row of zeros).
// One thread per row and group of eight columns.  *odd is set where a row holds a
// value that is not finite or is too large or small to scale (the caller's float64
// pass then runs instead).
__global__ void __launch_bounds__(256) post_digits_kernel(int n, int K, int Kp, const double* __restrict__ A, int64_t lda,
                                                          __nv_bfloat16* __restrict__ out, double* __restrict__ scale,
                                                          int* __restrict__ odd) {
  __shared__ double red[8][32];
  const int r = blockIdx.x * 32 + (threadIdx.x & 31), w = threadIdx.x >> 5;
  double m = 0.0;
  bool fin = true;
  if (r < n)
    for (int k = w; k < K; k += 8) {
      const double x = A[r + (int64_t)k * lda];
      fin = fin && isfinite(x);
      m = fmax(m, fabs(x));
    }
  red[w][threadIdx.x & 31] = fin ? m : INFINITY;
  __syncthreads();
  m = 0.0;
#pragma unroll
  for (int q = 0; q < 8; ++q) m = fmax(m, red[q][threadIdx.x & 31]);
  const bool bad = !(m < 1e140) || (m > 0.0 && m < 1e-140);
  const int e = m > 0.0 && !bad ? pow2_above(m) : 0;
  if (r >= n) return;
  if (w == 0) {
    scale[r] = m > 0.0 ? ldexp(1.0, e - 35) : 0.0;
    if (bad) *odd = 1;
  }
  const double up = ldexp(1.0, 7 - e);
  for (int k0 = 8 * w; k0 < Kp; k0 += 64) {
    double y[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) y[u] = !bad && k0 + u < K ? A[r + (int64_t)(k0 + u) * lda] * up : 0.0;
#pragma unroll
    for (int s = 0; s < kS; ++s) {
      __align__(16) __nv_bfloat16 d[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const double q = rint(y[u]);
        d[u] = __float2bfloat16_rn((float)q);
        y[u] = (y[u] - q) * 256.0;
      }
      *reinterpret_cast<uint4*>(out + ((int64_t)s * n + r) * Kp + k0) = *reinterpret_cast<const uint4*>(d);
    }
  }
}

__device__ __forceinline__ uint32_t pc_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void ldsm4(uint32_t a, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, "
      "%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

struct DigitMat {
  const __nv_bfloat16* d;  // planes
  const double* scale;
  int n, Kp;
};

// Whether T = sum_k |p_0| |v_0| reaches 512 in the thread's entries of the 64 x 64 tile at (i0, c0),
// rows past the matrix and rows of zeros aside: eight warps of 16 x 32 entries, the operands
// read from global memory as the matrix instruction's fragments hold them.
__device__ __forceinline__ bool tile_covered(const DigitMat& P, const DigitMat& V, int K, int i0, int c0, int ny, int cend) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, g = lane >> 2, q = lane & 3;
  const int i = i0 + (wid & 3) * 16 + g, c = c0 + (wid >> 2) * 32;
  auto word = [&](const DigitMat& M, int row, int end, int k) -> uint32_t {  // two digits' sizes
    return row < end ? __ldg(reinterpret_cast<const uint32_t*>(M.d + (int64_t)row * M.Kp + k)) & 0x7FFF7FFFu : 0u;
  };
  float acc[4][4];
#pragma unroll
  for (int t = 0; t < 4; ++t)
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[t][u] = 0.f;
  __syncwarp();
  for (int k = 0; k < K; k += 16) {
    const uint32_t a[4] = {word(P, i, ny, k + 2 * q), word(P, i + 8, ny, k + 2 * q), word(P, i, ny, k + 2 * q + 8),
                           word(P, i + 8, ny, k + 2 * q + 8)};
#pragma unroll
    for (int t = 0; t < 4; ++t)
      mma16816(acc[t], a, word(V, c + 8 * t + g, cend, k + 2 * q), word(V, c + 8 * t + g, cend, k + 2 * q + 8));
  }
  bool ok = true;
#pragma unroll
  for (int t = 0; t < 4; ++t)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int ii = i + 8 * (u >> 1), cc = c + 8 * t + 2 * q + (u & 1);
      if (ii < ny && cc < cend && acc[t][u] < 512.f) ok = ok && (P.scale[ii] == 0.0 || V.scale[cc] == 0.0);
    }
  return ok;
}

// wide[t] = 1 for the 64 x 64 tiles t (row tile fastest) that the float64 pass has to take
__global__ void __launch_bounds__(kPcThreads) post_check_kernel(const int* __restrict__ odd, int ny, int j, DigitMat P,
                                                                DigitMat V, int jr, DigitMat Pr, DigitMat Vr, int col0,
                                                                int ncols, uint8_t* __restrict__ wide) {
  const int rt = (ny + 63) / 64, cend = col0 + ncols;
  const int64_t ntiles = (int64_t)rt * ((ncols + 63) / 64);
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int i0 = (int)(tile % rt) * 64, c0 = col0 + (int)(tile / rt) * 64;
    bool ok = !*odd;  // the same in all threads, as is jr: the matrix instructions take whole warps
    if (ok) {
      ok = tile_covered(P, V, j, i0, c0, ny, cend);
      const bool ref = jr == 0 || tile_covered(Pr, Vr, jr, i0, c0, ny, cend);
      ok = ok && ref;
    }
    const int bad = __syncthreads_or(!ok);
    if (threadIdx.x == 0) wide[tile] = bad ? 1 : 0;
  }
}

// byte offset of 16-byte piece q of a staged row: the pieces of every second group of four rows are
// swapped, which puts those of eight consecutive rows in distinct banks
__device__ __forceinline__ uint32_t piece(int row, int q) { return (uint32_t)(row * (kKs * 2) + 16 * (q ^ ((row >> 2) & 1))); }

// Stage columns [k0, k0 + 16) of all digits of R rows from r0 on (rows past n: zeros).
template <int R>
__device__ __forceinline__ void stage(char* dst, const DigitMat& M, int r0, int k0) {
#pragma unroll
  for (int t = threadIdx.x; t < kS * R * 2; t += kPcThreads) {
    const int q = t & 1, r = (t >> 1) & (R - 1), s = t / (2 * R);
    const bool in = r0 + r < M.n;
    const __nv_bfloat16* src = in ? M.d + ((int64_t)s * M.n + r0 + r) * M.Kp + k0 + 8 * q : M.d;
    const uint32_t to = pc_smem(dst) + piece(s * R + r, q);
    const int bytes = in ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(src), "r"(bytes) : "memory");
  }
}

// The thread's eight entries of the warp's 16 x 16 part of the tile, rows i0 + .., columns c0 + ..
// of P V^T, into w[(4 nt + q) * kPcThreads] (shared memory: the level sums take the registers)
__device__ __forceinline__ void tile_product(char* buf, const DigitMat& P, const DigitMat& V, int K, int i0, int c0,
                                             double* w) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, wr = wid & 3, wc = wid >> 2;
  const int steps = (K + 15) / 16;
#pragma unroll
  for (int k = 0; k < 4 * kNt; ++k) w[k * kPcThreads] = 0.0;
  float acc[kS][kNt][4];
#pragma unroll
  for (int l = 0; l < kS; ++l)
#pragma unroll
    for (int t = 0; t < kNt; ++t)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[l][t][q] = 0.f;
  __syncthreads();  // the buffers' last readers are done
  stage<kTm>(buf, P, i0, 0);
  stage<kTn>(buf + kStageP, V, c0, 0);
  asm volatile("cp.async.commit_group;" ::: "memory");
  // this lane's row and 16-byte piece of a 16 x 16 block of P (x4: rows 0-7, 8-15, then the upper
  // columns) and of V (two matrix tiles: columns 0-7, 8-15 of each)
  const uint32_t offa = piece(wr * 16 + (lane & 15), lane >> 4);
  const uint32_t offb = piece(wc * 16 + (lane & 7) + ((lane >> 4) << 3), (lane >> 3) & 1);
  int in_chunk = 0;
  for (int st = 0; st < steps; ++st) {
    char* cur = buf + (st & 1) * (kStageP + kStageV);
    if (st + 1 < steps) {
      char* nxt = buf + ((st + 1) & 1) * (kStageP + kStageV);
      stage<kTm>(nxt, P, i0, (st + 1) * kKs);
      stage<kTn>(nxt + kStageP, V, c0, (st + 1) * kKs);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const uint32_t sa = pc_smem(cur) + offa, sb = pc_smem(cur + kStageP) + offb;
    uint32_t a[kS][4];
#pragma unroll
    for (int s = 0; s < kS; ++s) ldsm4(sa + (uint32_t)(s * kTm * kKs * 2), a[s]);
#pragma unroll
    for (int t = 0; t < kS; ++t) {
      uint32_t b[4];
      ldsm4(sb + (uint32_t)(t * kTn * kKs * 2), b);
#pragma unroll
      for (int s = 0; s < kS - t; ++s) {
        mma16816(acc[s + t][0], a[s], b[0], b[1]);
        mma16816(acc[s + t][1], a[s], b[2], b[3]);
      }
    }
    in_chunk += 16;
    if (in_chunk == kChunk || st == steps - 1) {
      // the level sums are integers below 2^24: two 48-bit integers, then float64
      in_chunk = 0;
#pragma unroll
      for (int t = 0; t < kNt; ++t)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          long long hi = 0, lo = 0;
#pragma unroll
          for (int l = 0; l < 4; ++l) {
            hi = hi * 256 + (long long)__float2int_rn(acc[l][t][q]);
            lo = lo * 256 + (long long)__float2int_rn(acc[4 + l][t][q]);
            acc[l][t][q] = 0.f;
            acc[4 + l][t][q] = 0.f;
          }
          w[(4 * t + q) * kPcThreads] += fma((double)hi, 4294967296.0, (double)lo);
        }
    }
    __syncthreads();
  }
  // value = 2^(eP + eV - 14 - 56) (hi 2^32 + lo); the rows' scales are 2^(e - 35)
  const int g = lane >> 2, c = 2 * (lane & 3);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = i0 + wr * 16 + g + 8 * (q >> 1);
    const double sp = i < P.n ? P.scale[i] : 0.0;
#pragma unroll
    for (int t = 0; t < kNt; ++t) {
      const int cc = c0 + wc * 16 + 8 * t + c + (q & 1);
      w[(4 * t + q) * kPcThreads] *= sp * (cc < V.n ? V.scale[cc] : 0.0);
    }
  }
}

// Statistics of a finite w, as stat_add but with the comparisons and the count on the integer
// units: a double's order is that of its bits (negative ones reversed).
struct TcStats {
  long long nneg = 0, mn = 0x7FF0000000000000ll, mx = ~0x7FF0000000000000ll;
  unsigned long long ma = 0;
  double w2 = 0.0, neg2 = 0.0, ref2 = 0.0, diff2 = 0.0;
  __device__ static long long key(double w) {
    const long long b = __double_as_longlong(w);
    return b ^ (long long)((unsigned long long)(b >> 63) >> 1);
  }
  __device__ static double val(long long k) {
    return __longlong_as_double(k ^ (long long)((unsigned long long)(k >> 63) >> 1));
  }
  __device__ void save(double* s) const {
    const long long b[4] = {nneg, mn, mx, (long long)ma};
    const double d[4] = {w2, neg2, ref2, diff2};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      s[k * kPcThreads] = __longlong_as_double(b[k]);
      s[(4 + k) * kPcThreads] = d[k];
    }
  }
  __device__ void load(const double* s) {
    nneg = __double_as_longlong(s[0]);
    mn = __double_as_longlong(s[kPcThreads]);
    mx = __double_as_longlong(s[2 * kPcThreads]);
    ma = (unsigned long long)__double_as_longlong(s[3 * kPcThreads]);
    w2 = s[4 * kPcThreads];
    neg2 = s[5 * kPcThreads];
    ref2 = s[6 * kPcThreads];
    diff2 = s[7 * kPcThreads];
  }
  __device__ double add(double w, double wr, int nonneg) {
    const long long b = __double_as_longlong(w), k = key(w);
    const bool neg = b < 0 && (b << 1) != 0;
    mn = k < mn ? k : mn;
    mx = k > mx ? k : mx;
    w2 = fma(w, w, w2);
    if (neg) {
      ++nneg;
      neg2 = fma(w, w, neg2);
    }
    const double pw = nonneg && neg ? 0.0 : w;
    const double d = pw - wr;
    ref2 = fma(wr, wr, ref2);
    diff2 = fma(d, d, diff2);
    const unsigned long long da = (unsigned long long)__double_as_longlong(d) & 0x7FFFFFFFFFFFFFFFull;
    ma = da > ma ? da : ma;
    return pw;
  }
};

// As post_tile_kernel (cr_post.cu), on the digit planes of P, V and the reference's
// factors; passes the tiles by that post_check_kernel marked.
__global__ void __launch_bounds__(kPcThreads, 2) post_tc_kernel(const uint8_t* __restrict__ wide, int ny, int j, DigitMat P,
                                                           DigitMat V, int jr, DigitMat Pr, DigitMat Vr, int nonneg, int col0,
                                                           int ncols, double* __restrict__ out, int64_t ldo,
                                                           double* __restrict__ part) {
  extern __shared__ __align__(16) char buf[];  // see kSmem
  double* wt = reinterpret_cast<double*>(buf + 2 * (kStageP + kStageV)) + threadIdx.x;
  double* rt_ = wt + 4 * kNt * kPcThreads;
  double* st = rt_ + 4 * kNt * kPcThreads;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, wr = wid & 3, wc = wid >> 2;
  const int g = lane >> 2, cb = 2 * (lane & 3);
  const int rt = (ny + kTm - 1) / kTm, ct = (ncols + kTn - 1) / kTn;
  const int64_t ntiles = (int64_t)rt * ct;
  const int cend = col0 + ncols;
  TcStats ts;
  ts.save(st);
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int i0 = (int)(tile % rt) * kTm, c0 = col0 + (int)(tile / rt) * kTn;
    if (wide[tile % rt + tile / rt / 2 * rt]) continue;  // its half of a 64 x 64 tile
    if (jr > 0) tile_product(buf, Pr, Vr, jr, i0, c0, rt_);
    tile_product(buf, P, V, j, i0, c0, wt);
    ts.load(st);
#pragma unroll
    for (int t = 0; t < kNt; ++t)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = i0 + wr * 16 + g + 8 * (q >> 1), c = c0 + wc * 16 + 8 * t + cb + (q & 1);
        if (i >= ny || c >= cend) continue;
        const int k = (4 * t + q) * kPcThreads;
        const double pw = ts.add(wt[k], jr > 0 ? rt_[k] : 0.0, nonneg);
        if (out) out[(int64_t)i + (int64_t)(c - col0) * ldo] = pw;
      }
    ts.save(st);
  }
  ts.load(st);
  double s[PS_N];
  s[PS_NNEG] = (double)ts.nneg;
  s[PS_MIN] = TcStats::val(ts.mn);
  s[PS_MAX] = TcStats::val(ts.mx);
  s[PS_W2] = ts.w2;
  s[PS_NEG2] = ts.neg2;
  s[PS_REF2] = ts.ref2;
  s[PS_DIFF2] = ts.diff2;
  s[PS_MAXABS] = __longlong_as_double((long long)ts.ma);
  block_stats<kPcThreads>(s, part + (int64_t)blockIdx.x * PS_N);
}

int padded(int K) { return (K + 15) / 16 * 16; }

}  // namespace

int post_tc_blocks() {
  static const int nb = [] {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaFuncSetAttribute(post_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, post_tc_kernel, kPcThreads, kSmem) != cudaSuccess || per < 1) {
      cudaGetLastError();
      return 0;
    }
    return sms * per;
  }();
  return nb;
}

int post_tc_parts(int ny, int ncols) {
  const int64_t ntiles = (int64_t)((ny + kTm - 1) / kTm) * ((ncols + kTn - 1) / kTn);
  return (int)std::min<int64_t>(post_tc_blocks(), std::max<int64_t>(ntiles, 1));
}

size_t post_tc_digit_elems(int n, int K) { return (size_t)kS * n * padded(K); }

void post_tc_digits(int n, int K, const double* A, int64_t lda, void* digits, double* scale, int* odd, cudaStream_t st) {
  if (K <= 0) return;
  count_launch();
  post_digits_kernel<<<(n + 31) / 32, 256, 0, st>>>(n, K, padded(K), A, lda, (__nv_bfloat16*)digits, scale, odd);
}

size_t post_wide_tiles(int ny, int ncols) { return (size_t)((ny + 63) / 64) * ((ncols + 63) / 64); }

void post_tc_tiles(const int* odd, uint8_t* wide, int ny, int nx, int j, const void* P, const double* sP, const void* V,
                   const double* sV, int jr, const void* Pr, const double* sPr, const void* Vr, const double* sVr,
                   int nonneg, int col0, int ncols, double* out, int64_t ldo, double* part, cudaStream_t st) {
  auto mat = [&](const void* d, const double* s, int n, int K) {
    return DigitMat{(const __nv_bfloat16*)d, s, n, padded(K)};
  };
  const DigitMat mP = mat(P, sP, ny, j), mV = mat(V, sV, nx, j), mPr = mat(Pr, sPr, ny, jr), mVr = mat(Vr, sVr, nx, jr);
  count_launch();
  post_check_kernel<<<(unsigned)std::min<size_t>(post_wide_tiles(ny, ncols), 1 << 16), kPcThreads, 0, st>>>(
      odd, ny, j, mP, mV, jr, mPr, mVr, col0, ncols, wide);
  count_launch();
  post_tc_kernel<<<post_tc_parts(ny, ncols), kPcThreads, kSmem, st>>>(wide, ny, j, mP, mV, jr, mPr, mVr, nonneg, col0,
                                                                      ncols, out, ldo, part);
}

}  // namespace cr
