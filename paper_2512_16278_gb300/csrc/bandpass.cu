// bandpass.cu - Section 3.1 bandpass normalisation with ArPLS, and the CCM
// under the bandpass-centred reading of Eq. 1.
//
// For a fit interval of F sub-integrations the bandpass of beam a is its
// time-aggregated spectrum y_a(j), the mean of channel j over the
// interval's samples; here it comes exactly from the Gram sums already
// formed (sum of S_a over the interval's cells over the sum of their n).
// Its baseline z_a(j) is fitted over channels with ArPLS (asymmetrically
// reweighted penalized least squares; Baek, Park, Ahn and Ahn 2015, the
// method Section 3.1 names, with the lam / ratio / itermax parameters of
// Section 4.5): weights w start at 1; each step solves
// (W + lam D^T D) z = W y (D: second differences), takes the mean m and
// population deviation s of the negative residuals d = y - z, and moves to
// w_i = 1 / (1 + exp(2 (d_i - (2 s - m)) / s)) until the weights change by
// less than `ratio` (relative Euclidean norm) or itermax solves.
//
// The CCM of a cell about the bandpass is
//   C_ab = (1/n) sum_t (x_a - z_a)(x_b - z_b) = cov_ab / n^2 + d_a d_b,
// cov_ab = n S_ab - S_a S_b the exact int64 covariance numerator and
// d_a = S_a / n - z_a the cell mean's offset from the bandpass: no
// cancellation between large terms, so FP32 suffices for C.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "internal.h"

namespace cg = cooperative_groups;

namespace mraid {
namespace {

constexpr int kArThreads = 512;
constexpr int kArWarps = kArThreads / 32;
constexpr int kCrArrays = 13;  // per block row: A (3), C (4), saved left coupling (4), F (2)

// Sums of two values over the block in a fixed order; every thread gets the
// totals. One warp adds the warps' sums: FP64 issue is scarce (two lanes per
// cycle and SM on GB300), and every warp adding all 16 cost 2 us a sum.
__device__ void block_sum2(double& a, double& b, double (*red)[2]) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  __syncthreads();
  if (lane == 0) {
    red[warp][0] = a;
    red[warp][1] = b;
  }
  __syncthreads();
  if (warp == 0) {
    a = lane < kArWarps ? red[lane][0] : 0.0;
    b = lane < kArWarps ? red[lane][1] : 0.0;
#pragma unroll
    for (int o = kArWarps / 2; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if (lane == 0) {
      red[kArWarps][0] = a;
      red[kArWarps][1] = b;
    }
  }
  __syncthreads();
  a = red[kArWarps][0];
  b = red[kArWarps][1];
}

// Entries of D^T D for D the (n-2) x n second-difference matrix (rows
// 1, -2, 1): the contributions of the rows k that touch i.
__device__ __forceinline__ double dtd0(int i, int n) {  // (i, i)
  return (i >= 2 ? 1.0 : 0.0) + (i >= 1 && i - 1 <= n - 3 ? 4.0 : 0.0) + (i <= n - 3 ? 1.0 : 0.0);
}
__device__ __forceinline__ double dtd1(int i, int n) {  // (i, i + 1)
  return (i >= 1 && i - 1 <= n - 3 ? -2.0 : 0.0) + (i <= n - 3 ? -2.0 : 0.0);
}

struct M2 {  // [[a, b], [c, d]]
  double a, b, c, d;
};
__device__ __forceinline__ M2 mm(const M2& x, const M2& y) {
  return {fma(x.a, y.a, x.b * y.c), fma(x.a, y.b, x.b * y.d), fma(x.c, y.a, x.d * y.c),
          fma(x.c, y.b, x.d * y.d)};
}
__device__ __forceinline__ M2 tr(const M2& x) { return {x.a, x.c, x.b, x.d}; }

struct CrArrays {  // m block rows each
  double *aa, *ab, *ad;            // A_i = [[aa, ab], [ab, ad]]; the inverse once eliminated
  double *c00, *c01, *c10, *c11;   // C_i: coupling of row i to the next active row
  double *l00, *l01, *l10, *l11;   // left coupling of a row, saved when it is eliminated
  double *f0, *f1;                 // right side, then the solution
  __device__ CrArrays(double* p, int m)
      : aa(p), ab(p + m), ad(p + 2 * m), c00(p + 3 * m), c01(p + 4 * m), c10(p + 5 * m),
        c11(p + 6 * m), l00(p + 7 * m), l01(p + 8 * m), l10(p + 9 * m), l11(p + 10 * m),
        f0(p + 11 * m), f1(p + 12 * m) {}
  __device__ M2 C(int i) const { return {c00[i], c01[i], c10[i], c11[i]}; }
  __device__ M2 A(int i) const { return {aa[i], ab[i], ab[i], ad[i]}; }
};

// (W + lam D^T D) z = W y by block cyclic reduction. Unknowns in pairs
// X_i = (z_2i, z_2i+1) make the pentadiagonal matrix block tridiagonal with
// 2 x 2 blocks (row i: C_{i-1}^T X_{i-1} + A_i X_i + C_i X_{i+1}); m block
// rows, a power of two (rows past n are identity rows with no coupling).
// Each level eliminates the odd rows of the active set (stride s) into the
// even ones; then the single remaining row is solved and the eliminated
// rows are recovered level by level. It is Gaussian elimination of the
// symmetric positive definite matrix in an odd-even order, so it needs no
// pivoting, and every level is parallel over its rows.
//
// A cluster of K CTAs shares one spectrum: CTA r holds block rows [r mk,
// (r + 1) mk), mk = m / K. A level reads one row of the CTA before (the last
// leaving one); when one row per CTA is left, CTA 0 solves those K rows.

// Row j leaves: its A becomes the inverse, its left coupling is kept.
__device__ __forceinline__ void cr_leave(const CrArrays& r, int j, const M2& Cprev) {
  const double a = r.aa[j], b = r.ab[j], d = r.ad[j];
  const double inv = 1.0 / fma(a, d, -b * b);
  r.aa[j] = d * inv;
  r.ab[j] = -b * inv;
  r.ad[j] = a * inv;
  const M2 L = tr(Cprev);
  r.l00[j] = L.a;
  r.l01[j] = L.b;
  r.l10[j] = L.c;
  r.l11[j] = L.d;
}

// Row i takes in the row before it (rp, jp; jp < 0: none) and the row jn after it
// (jn < 0: none).
__device__ __forceinline__ void cr_stay(const CrArrays& r, int i, const CrArrays& rp, int jp,
                                        int jn) {
  M2 Ai = r.A(i);
  double g0 = r.f0[i], g1 = r.f1[i];
  if (jp >= 0) {
    const M2 Cj = rp.C(jp);
    M2 al = mm(tr(Cj), rp.A(jp));
    al = {-al.a, -al.b, -al.c, -al.d};
    const M2 t = mm(al, Cj);
    Ai = {Ai.a + t.a, Ai.b + t.b, Ai.c + t.c, Ai.d + t.d};
    g0 = fma(al.a, rp.f0[jp], fma(al.b, rp.f1[jp], g0));
    g1 = fma(al.c, rp.f0[jp], fma(al.d, rp.f1[jp], g1));
  }
  M2 Cn = {0.0, 0.0, 0.0, 0.0};
  if (jn >= 0) {
    const M2 Ci = r.C(i);
    M2 ga = mm(Ci, r.A(jn));
    ga = {-ga.a, -ga.b, -ga.c, -ga.d};
    const M2 t = mm(ga, tr(Ci));
    Ai = {Ai.a + t.a, Ai.b + t.b, Ai.c + t.c, Ai.d + t.d};
    g0 = fma(ga.a, r.f0[jn], fma(ga.b, r.f1[jn], g0));
    g1 = fma(ga.c, r.f0[jn], fma(ga.d, r.f1[jn], g1));
    Cn = mm(ga, r.C(jn));
  }
  r.aa[i] = Ai.a;
  r.ab[i] = 0.5 * (Ai.b + Ai.c);
  r.ad[i] = Ai.d;
  r.c00[i] = Cn.a;
  r.c01[i] = Cn.b;
  r.c10[i] = Cn.c;
  r.c11[i] = Cn.d;
  r.f0[i] = g0;
  r.f1[i] = g1;
}

// The eliminated row j from the solutions before it (row j - s) and after
// it: row j + s, or (y0, y1) of the next CTA's first row.
__device__ __forceinline__ void cr_back(const CrArrays& r, int j, int s, int m, double y0, double y1) {
  const double x0 = r.f0[j - s], x1 = r.f1[j - s];
  double g0 = r.f0[j] - fma(r.l00[j], x0, r.l01[j] * x1);
  double g1 = r.f1[j] - fma(r.l10[j], x0, r.l11[j] * x1);
  if (j + s < m) {
    y0 = r.f0[j + s];
    y1 = r.f1[j + s];
  }
  g0 -= fma(r.c00[j], y0, r.c01[j] * y1);
  g1 -= fma(r.c10[j], y0, r.c11[j] * y1);
  r.f0[j] = fma(r.aa[j], g0, r.ab[j] * g1);
  r.f1[j] = fma(r.ab[j], g0, r.ad[j] * g1);
}

__device__ __forceinline__ void cr_last(const CrArrays& r) {  // the one row left
  const double a = r.aa[0], b = r.ab[0], d = r.ad[0];
  const double inv = 1.0 / fma(a, d, -b * b);
  const double g0 = r.f0[0], g1 = r.f1[0];
  r.f0[0] = (d * g0 - b * g1) * inv;
  r.f1[0] = (a * g1 - b * g0) * inv;
}

constexpr int kArMaxCtas = 8;
constexpr size_t kArSmem = 214 * 1024;  // for the arrays of one CTA

// K = cluster.num_blocks() CTAs; base: the store of each CTA's CrArrays;
// top: kCrArrays x kArMaxCtas doubles (CTA 0's are used); next_x: the next
// CTA's first solution.
__device__ void cr_solve(const cg::cluster_group& cl, double* base, double* top, double* next_x,
                         int mk, const double* w, const double* y, int n, double lam) {
  const int K = (int)cl.num_blocks(), rank = (int)cl.block_rank(), row0 = rank * mk;
  const CrArrays r(base, mk);
  for (int l = threadIdx.x; l < mk; l += blockDim.x) {
    const int r0 = 2 * (row0 + l), r1 = r0 + 1;
    const bool v0 = r0 < n, v1 = r1 < n;
    r.aa[l] = v0 ? w[r0] + lam * dtd0(r0, n) : 1.0;
    r.ab[l] = v1 ? lam * dtd1(r0, n) : 0.0;
    r.ad[l] = v1 ? w[r1] + lam * dtd0(r1, n) : 1.0;
    r.c00[l] = r0 + 2 < n ? lam : 0.0;                 // (r0, r0 + 2)
    r.c01[l] = 0.0;                                     // (r0, r0 + 3)
    r.c10[l] = r1 + 1 < n ? lam * dtd1(r1, n) : 0.0;    // (r1, r1 + 1)
    r.c11[l] = r1 + 2 < n ? lam : 0.0;                  // (r1, r1 + 2)
    r.f0[l] = v0 ? w[r0] * y[r0] : 0.0;
    r.f1[l] = v1 ? w[r1] * y[r1] : 0.0;
  }
  __syncthreads();
  // the CTA before: its rows are read while they are the leaving ones, which
  // nothing changes until the solution comes back
  const CrArrays rp(K > 1 && rank > 0 ? cl.map_shared_rank(base, rank - 1) : base, mk);
  auto sync = [&]() {
    if (K > 1) cl.sync();
    else __syncthreads();
  };
  for (int s = 1; s < mk; s *= 2) {
    for (int j = s + 2 * s * threadIdx.x; j < mk; j += 2 * s * blockDim.x) cr_leave(r, j, r.C(j - s));
    sync();
    for (int i = 2 * s * threadIdx.x; i < mk; i += 2 * s * blockDim.x) {
      if (i > 0) cr_stay(r, i, r, i - s, i + s);
      else cr_stay(r, i, rp, rank > 0 ? mk - s : -1, i + s);
    }
    __syncthreads();
  }
  if (K == 1) {
    if (threadIdx.x == 0) cr_last(r);
    __syncthreads();
  } else {
    // CTA 0 gathers the K rows left, reduces and solves them
    cl.sync();
    if (rank == 0) {
      const CrArrays t(top, kArMaxCtas);
      if (threadIdx.x < (unsigned)K) {
        const CrArrays q(cl.map_shared_rank(base, threadIdx.x), mk);
        const int l = threadIdx.x;
        t.aa[l] = q.aa[0];
        t.ab[l] = q.ab[0];
        t.ad[l] = q.ad[0];
        t.c00[l] = q.c00[0];
        t.c01[l] = q.c01[0];
        t.c10[l] = q.c10[0];
        t.c11[l] = q.c11[0];
        t.f0[l] = q.f0[0];
        t.f1[l] = q.f1[0];
      }
      __syncthreads();
      for (int s = 1; s < K; s *= 2) {
        const int j = s + 2 * s * threadIdx.x, i = 2 * s * threadIdx.x;
        if (j < K) cr_leave(t, j, t.C(j - s));
        __syncthreads();
        if (i < K) cr_stay(t, i, t, i - s, i + s < K ? i + s : -1);
        __syncthreads();
      }
      if (threadIdx.x == 0) cr_last(t);
      __syncthreads();
      for (int s = K / 2; s >= 1; s /= 2) {
        const int j = s + 2 * s * threadIdx.x;
        if (j < K) cr_back(t, j, s, K, 0.0, 0.0);
        __syncthreads();
      }
    }
    cl.sync();
    if (threadIdx.x < 2) {  // this CTA's first solution and the next one's
      const CrArrays t(cl.map_shared_rank(top, 0), kArMaxCtas);
      const double* f = threadIdx.x == 0 ? t.f0 : t.f1;
      (threadIdx.x == 0 ? r.f0 : r.f1)[0] = f[rank];
      next_x[threadIdx.x] = rank + 1 < K ? f[rank + 1] : 0.0;
    }
    __syncthreads();
  }
  const double y0 = K > 1 ? next_x[0] : 0.0, y1 = K > 1 ? next_x[1] : 0.0;
  for (int s = mk / 2; s >= 1; s /= 2) {
    for (int j = s + 2 * s * threadIdx.x; j < mk; j += 2 * s * blockDim.x)
      cr_back(r, j, s, mk, y0, y1);
    __syncthreads();
  }
}

__host__ __device__ constexpr int cr_rows(int n) {  // block rows: a power of two >= n / 2
  int m = 1;
  while (2 * m < n) m *= 2;
  return m;
}

struct ArplsArgs {
  const double* y;   // [sys][n]
  double* z;         // [sys][n]
  float* zf;         // [sys][n] float copy, or null
  int32_t* iters;    // [sys], or null
  double* work;      // [sys][2][n] weights and new weights, then [sys][13 m] when the
                     // reduction arrays are not in shared memory
  int n, n_sys, itermax, in_smem;
  double lam, ratio;
};

// One cluster of K CTAs per spectrum (K = 1: one CTA): the weighted solves by
// block cyclic reduction, the residual statistics and the reweighting, all
// parallel over the cluster. FP64 issue bounds it (two lanes per cycle and
// SM on GB300; a solve and reweighting of 4096 channels is about 4e5
// operations) and the levels' latency.
__global__ void __launch_bounds__(kArThreads, 1) arpls_kernel(ArplsArgs g) {
  extern __shared__ double ar_sm[];
  __shared__ double red[kArWarps + 1][2];
  __shared__ double top[kCrArrays * kArMaxCtas];
  __shared__ double next_x[2];
  __shared__ double parts[2][kArMaxCtas][2];
  const cg::cluster_group cl = cg::this_cluster();
  const int K = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int sys = blockIdx.x / K, n = g.n, mk = cr_rows(n) / K;
  double* w = g.work + (size_t)sys * 2 * n;
  double* wt = w + n;
  double* base = g.in_smem ? ar_sm
                           : g.work + (size_t)g.n_sys * 2 * n + (size_t)sys * kCrArrays * mk;
  const CrArrays r(base, mk);
  const double* y = g.y + (size_t)sys * n;
  // this CTA's channels
  const int i0 = 2 * rank * mk, i1 = min(n, i0 + 2 * mk);
  auto z = [&](int i) { return (i & 1) ? r.f1[(i - i0) >> 1] : r.f0[(i - i0) >> 1]; };
  // sums of two values over the cluster, in a fixed order
  int buf = 0;
  auto sum2 = [&](double& a, double& b) {
    block_sum2(a, b, red);
    if (K == 1) return;
    if (threadIdx.x < (unsigned)K) {
      double* dst = cl.map_shared_rank(&parts[buf][rank][0], threadIdx.x);
      dst[0] = a;
      dst[1] = b;
    }
    cl.sync();
    if (threadIdx.x < 2) {  // two threads: FP64 issue is scarce
      double t = 0.0;
      for (int c = 0; c < K; ++c) t += parts[buf][c][threadIdx.x];
      red[kArWarps][threadIdx.x] = t;
    }
    __syncthreads();
    a = red[kArWarps][0];
    b = red[kArWarps][1];
    buf ^= 1;  // the other buffer's readers passed this barrier
  };
  for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) w[i] = 1.0;
  __syncthreads();
  int solves = 0;
  double w2 = (double)n;  // sum of the squared weights
  while (solves < g.itermax) {
    cr_solve(cl, base, top, next_x, mk, w, y, n, g.lam);
    ++solves;
    double sn = 0.0, cn = 0.0;
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
      const double d = y[i] - z(i);
      if (d < 0.0) {
        sn += d;
        cn += 1.0;
      }
    }
    sum2(sn, cn);
    if (cn == 0.0) break;
    const double mneg = sn / cn;
    double s2 = 0.0, unused = 0.0;
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
      const double d = y[i] - z(i);
      if (d < 0.0) s2 += (d - mneg) * (d - mneg);
    }
    sum2(s2, unused);
    const double sd = sqrt(s2 / cn);
    if (!(sd > 0.0)) break;
    const double thr = 2.0 * sd - mneg, scale = 2.0 / sd;
    double dw2 = 0.0, wn2 = 0.0;
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
      const double d = y[i] - z(i);
      const double wn = 1.0 / (1.0 + exp((d - thr) * scale));
      dw2 += (w[i] - wn) * (w[i] - wn);
      wn2 += wn * wn;
      wt[i] = wn;
    }
    sum2(dw2, wn2);
    if (sqrt(dw2) / sqrt(w2) < g.ratio) break;
    w2 = wn2;
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) w[i] = wt[i];
    __syncthreads();
  }
  __syncthreads();
  for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    const double zi = z(i);
    g.z[(size_t)sys * n + i] = zi;
    if (g.zf) g.zf[(size_t)sys * n + i] = (float)zi;
  }
  if (rank == 0 && threadIdx.x == 0 && g.iters) g.iters[sys] = solves;
  if (K > 1) cl.sync();  // no CTA leaves while another may read its rows
}

// y[(I * N + a) * n_chan + j]: mean of beam a, channel j over interval I,
// from the Gram sums [cell][P].
__global__ void bandpass_input_kernel(const int64_t* __restrict__ sums, int n_beam, int n_chan,
                                      int n_sub, int n_samp_sub, int interval, int psum,
                                      double* __restrict__ y, int64_t total) {
  const int N1 = n_beam + 1;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(idx % n_chan);
    const int64_t ia = idx / n_chan;
    const int a = (int)(ia % n_beam);
    const int I = (int)(ia / n_beam);
    const int e_sa = a * N1 - a * (a - 1) / 2 + (n_beam - a);  // S_a
    const int k0 = I * interval;
    const int k1 = k0 + interval < n_sub ? k0 + interval : n_sub;
    int64_t s = 0;
    for (int k = k0; k < k1; ++k) s += sums[((int64_t)k * n_chan + j) * psum + e_sa];
    y[idx] = (double)s / (double)((int64_t)(k1 - k0) * n_samp_sub);
  }
}

// One warp per cell: C_ab = cov_ab / n^2 + d_a d_b, packed upper triangle.
__global__ void ccm_bandpass_kernel(const int64_t* __restrict__ sums, int64_t n_cells, int n_beam, int n_chan, int interval,
                                    int psum, int np, const double* __restrict__ z,
                                    float* __restrict__ ccm) {
  extern __shared__ unsigned char bp_raw[];
  const int warps = blockDim.x / 32;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  int64_t* S = reinterpret_cast<int64_t*>(bp_raw) + (size_t)warp * psum;
  float* dv = reinterpret_cast<float*>(reinterpret_cast<int64_t*>(bp_raw) + (size_t)warps * psum) +
              (size_t)warp * kMaxBeam;
  const int64_t cell = (int64_t)blockIdx.x * warps + warp;
  if (cell >= n_cells) return;
  const int N1 = n_beam + 1;
  const int64_t* src = sums + cell * psum;
  for (int e = lane; e < psum; e += 32) S[e] = src[e];
  __syncwarp();
  const int64_t n = S[psum - 1];
  const int k = (int)(cell / n_chan), j = (int)(cell % n_chan);
  const int I = k / interval;
  // FP32 throughout (this GPU's FP64 rate is low): S_a < 2^24 is exact
  // in float, and the offsets d_a are O(1), so rounding the mean and the
  // baseline to float costs ~1e-5 absolute in d_a, ~1e-7 of C
  const float inv_n = 1.f / (float)n;
  for (int a = lane; a < n_beam; a += 32) {
    const int64_t sa = S[a * N1 - a * (a - 1) / 2 + (n_beam - a)];
    dv[a] = fmaf((float)sa, inv_n, -(float)z[((int64_t)I * n_beam + a) * n_chan + j]);
  }
  __syncwarp();
  const float inv_n2 = inv_n * inv_n;
  float* dst = ccm + cell * np;
  int a = 0, rowlen = n_beam, row_start = 0;
  for (int e = lane; e < np; e += 32) {
    while (e >= row_start + rowlen) {
      row_start += rowlen;
      --rowlen;
      ++a;
    }
    const int b = a + (e - row_start);
    const int64_t sa = S[a * N1 - a * (a - 1) / 2 + (n_beam - a)];
    const int64_t sb = S[b * N1 - b * (b - 1) / 2 + (n_beam - b)];
    const int64_t cov = n * S[a * N1 - a * (a - 1) / 2 + (b - a)] - sa * sb;
    dst[e] = fmaf(dv[a], dv[b], (float)cov * inv_n2);
  }
}

}  // namespace

// Shared memory of one of k CTAs; 0: the arrays do not fit
size_t arpls_smem_bytes(int n, int k) {
  const size_t b = (size_t)kCrArrays * (cr_rows(n) / k) * sizeof(double);
  return b <= kArSmem ? b : 0;
}

// CTAs per spectrum with the arrays in shared memory: two for long spectra
// that leave SMs idle, and as many as it takes for the arrays to fit; 0 where
// eight do not. Measured on GB300, us a call of 5 to 6 solves with 1 / 2 / 4 /
// 8 CTAs: 38 spectra of 4096 channels 904 / 696 / 994 / 1290, 190 spectra 1650
// / 1845 / 2793 / 5303, 38 spectra of 1000 channels 420 / 431 / 649 / 1093 (the
// cluster's barriers and the serial top outweigh the share of the FP64 work).
int arpls_ctas(int n, int n_sys, int sm_count) {
  const int m = cr_rows(n);
  int k = m >= 1024 && (int64_t)n_sys * 2 <= sm_count ? 2 : 1;
  while (k < kArMaxCtas && !arpls_smem_bytes(n, k)) k *= 2;
  return arpls_smem_bytes(n, k) ? k : 0;
}

// True where one CTA per spectrum on global memory is the faster way: many
// spectra that need a cluster for their arrays. A cluster of 2 / 4 / 8 is 1.67 /
// 3.05 / 5.4 times as fast as such a CTA, but 152 SMs hold 76 / 34 / 15 of them
// at a time (not every SM has neighbours left for a cluster). Measured, clusters
// against global memory: 760 spectra of 8192 channels 8.70 ms against 6.84, 190
// 2.51 against 2.79; 760 of 16 384 18.7 against 13.0, 38 1.71 against 2.52; 400
// of 32 768 23.5 against 16.0, 38 2.62 against 4.76.
bool arpls_on_global(const mraid_plan_s* pl, int n, int n_sys) {
  const int sm_count = pl->sm_count, k = arpls_ctas(n, n_sys, sm_count);
  if (k == 0) return true;
  if (arpls_smem_bytes(n, 1) || pl->ar_work_short) return false;
  const double gain = k == 2 ? 1.67 : (k == 4 ? 3.05 : 5.4);
  const int held = k == 2 ? sm_count / 2 : (k == 4 ? sm_count * 9 / 40 : sm_count / 10);
  const int64_t rounds = ((int64_t)n_sys + held - 1) / held;
  return (double)(((int64_t)n_sys + sm_count - 1) / sm_count) * gain < (double)rounds;
}

// the weights always; the reduction arrays when they are not in shared memory
size_t arpls_work_doubles(int n, int n_sys, bool on_global) {
  return (size_t)2 * n * n_sys + (on_global ? (size_t)kCrArrays * cr_rows(n) * n_sys : 0);
}

cudaError_t launch_arpls(const mraid_plan_s* pl, const double* d_y, int n_sys, int n, double lam,
                         double ratio, int itermax, double* d_z, float* d_zf, int32_t* d_iters,
                         double* d_work) {
  if (n_sys <= 0) return cudaSuccess;
  if (!d_work) return cudaErrorInvalidValue;
  ArplsArgs g;
  g.y = d_y;
  g.z = d_z;
  g.zf = d_zf;
  g.iters = d_iters;
  g.work = d_work;
  g.n = n;
  g.n_sys = n_sys;
  g.itermax = itermax;
  g.lam = lam;
  g.ratio = ratio;
  const bool on_global = arpls_on_global(pl, n, n_sys);
  const int k = on_global ? 1 : arpls_ctas(n, n_sys, pl->sm_count);
  const size_t smem = on_global ? 0 : arpls_smem_bytes(n, k);
  g.in_smem = on_global ? 0 : 1;
  cudaError_t e = cudaFuncSetAttribute(arpls_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)n_sys * k);
  cfg.blockDim = dim3(kArThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = pl->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim = {(unsigned)k, 1, 1};
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, arpls_kernel, g);
}

cudaError_t launch_bandpass_input(const mraid_plan_s* pl, const int64_t* d_sums, int interval, double* d_y) {
  const int n_int = (pl->p.n_sub + interval - 1) / interval;
  const int64_t total = (int64_t)n_int * pl->p.n_beam * pl->p.n_chan;
  int64_t blocks = (total + 255) / 256;
  if (blocks > (int64_t)pl->sm_count * 16) blocks = (int64_t)pl->sm_count * 16;
  if (blocks < 1) return cudaSuccess;
  bandpass_input_kernel<<<(unsigned)blocks, 256, 0, pl->stream>>>(
      d_sums, pl->p.n_beam, pl->p.n_chan, pl->p.n_sub, pl->p.n_samp_sub, interval, pl->psum,
      d_y, total);
  return cudaGetLastError();
}

cudaError_t launch_ccm_bandpass(const mraid_plan_s* pl, const int64_t* d_sums, int interval, const double* d_z, float* d_ccm) {
  const int psum = pl->psum;
  int warps = (int)(40960 / ((size_t)psum * 8 + kMaxBeam * 4));
  warps = warps < 1 ? 1 : (warps > 8 ? 8 : warps);
  const size_t smem = (size_t)warps * ((size_t)psum * 8 + kMaxBeam * 4);
  cudaError_t e = cudaFuncSetAttribute(ccm_bandpass_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t blocks = (pl->n_cells + warps - 1) / warps;
  if (blocks > 0)
    ccm_bandpass_kernel<<<(unsigned)blocks, warps * 32, smem, pl->stream>>>(
        d_sums, pl->n_cells, pl->p.n_beam, pl->p.n_chan, interval, psum,
        pl->np, d_z, d_ccm);
  return cudaGetLastError();
}

}  // namespace mraid

namespace mraid {
namespace {
mraid_status check_bandpass_params(const mraid_bandpass_params* bp) {
  if (!bp || !(bp->lam > 0.0) || !(bp->lam < 1e300) || !(bp->ratio > 0.0) || bp->itermax < 1 ||
      bp->itermax > 1000 || bp->interval < 1) {
    set_error("bandpass parameters: lam > 0, ratio > 0, itermax in 1..1000, interval >= 1");
    return MRAID_ERR_INVALID_ARG;
  }
  return MRAID_OK;
}

// ArPLS weights, and the arrays of spectra that are solved on global memory; if
// these do not fit it and clusters can do without, the weights alone, and the
// plan stays on clusters
mraid_status ensure_arpls_work(mraid_plan_s* pl, int n, int n_sys) {
  size_t need = arpls_work_doubles(n, n_sys, arpls_on_global(pl, n, n_sys));
  if (need <= pl->ar_work_elems) return MRAID_OK;
  cudaFree(pl->ar_work);
  pl->ar_work = nullptr;
  pl->ar_work_elems = 0;
  cudaError_t e = cudaMalloc(&pl->ar_work, need * sizeof(double));
  if (e != cudaSuccess && arpls_ctas(n, n_sys, pl->sm_count) > 0) {
    cudaGetLastError();
    pl->ar_work_short = true;
    need = arpls_work_doubles(n, n_sys, false);
    e = cudaMalloc(&pl->ar_work, need * sizeof(double));
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return cuda_fail(e, "arpls work allocation");
  }
  pl->ar_work_elems = need;
  return MRAID_OK;
}
}  // namespace
}  // namespace mraid

// ---------------------------------------------------------------------------
// Entry points (include/mraid.h)

using namespace mraid;

void mraid_default_bandpass_params(mraid_bandpass_params* bp) {
  if (!bp) return;
  bp->lam = 1e5;
  bp->ratio = 1e-3;
  bp->itermax = 50;
  bp->interval = 20;
}

mraid_status mraid_arpls(mraid_plan_t pl, const double* d_y, int32_t n_sys, int32_t n,
                         const mraid_bandpass_params* bp, double* d_z, int32_t* d_iters) {
  mraid_status st = check_plan(pl);
  if (st != MRAID_OK) return st;
  st = check_bandpass_params(bp);
  if (st != MRAID_OK) return st;
  if (!d_y || !d_z || n < 3 || n > (1 << 20) || n_sys < 0) {
    set_error("mraid_arpls: d_y and d_z are required, 3 <= n <= 2^20, n_sys >= 0");
    return MRAID_ERR_INVALID_ARG;
  }
  st = ensure_arpls_work(pl, n, n_sys);
  if (st != MRAID_OK) return st;
  cudaError_t e = MRAID_PROF(pl, K_ARPLS,
                             launch_arpls(pl, d_y, n_sys, n, bp->lam, bp->ratio, bp->itermax, d_z,
                                          nullptr, d_iters, pl->ar_work));
  return e == cudaSuccess ? MRAID_OK : cuda_fail(e, "arpls launch");
}

mraid_status mraid_run_bandpass(mraid_plan_t pl, const void* d_data,
                                const mraid_bandpass_params* bp, float* d_bandpass,
                                float* d_evals, float* d_q1, float* d_stat, uint8_t* d_flags,
                                mraid_flag_info* info) {
  mraid_status st = check_plan(pl);
  if (st != MRAID_OK) return st;
  st = check_bandpass_params(bp);
  if (st != MRAID_OK) return st;
  if (!d_data || !d_stat || !d_flags) {
    set_error("mraid_run_bandpass: d_data, d_stat and d_flags are required");
    return MRAID_ERR_INVALID_ARG;
  }
  if (pl->p.bit_depth != 8 || pl->p.n_chan < 3 || pl->p.n_chan > (1 << 20)) {
    set_error("mraid_run_bandpass: 8-bit samples and 3 to 2^20 channels");
    return MRAID_ERR_UNSUPPORTED;
  }
  // an interval at least as long as the block is one interval of the
  // block: the same partition, and no int arithmetic on a huge interval
  const int interval = bp->interval < pl->p.n_sub ? bp->interval : pl->p.n_sub;
  const int n_int = (int)(((int64_t)pl->p.n_sub + interval - 1) / interval);
  if ((int64_t)n_int * pl->p.n_beam > INT32_MAX) {
    set_error("mraid_run_bandpass: %d intervals x %d beams exceed 2^31 - 1 spectra", n_int,
              pl->p.n_beam);
    return MRAID_ERR_UNSUPPORTED;
  }
  const int n_sys = n_int * pl->p.n_beam;
  const size_t elems = (size_t)n_sys * pl->p.n_chan;
  st = ensure_workspace(pl, (size_t)pl->n_cells);
  if (st != MRAID_OK) return st;
  cudaError_t e = cudaSuccess;
  if (elems > pl->bp_elems || (size_t)n_sys > pl->bp_sys) {
    cudaFree(pl->bp_y);
    cudaFree(pl->bp_z);
    cudaFree(pl->bp_iters);
    pl->bp_y = pl->bp_z = nullptr;
    pl->bp_iters = nullptr;
    pl->bp_elems = pl->bp_sys = 0;
    e = cudaMalloc(&pl->bp_y, elems * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&pl->bp_z, elems * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&pl->bp_iters, (size_t)n_sys * sizeof(int32_t));
    if (e != cudaSuccess) {
      cudaGetLastError();
      return cuda_fail(e, "bandpass workspace allocation");
    }
    pl->bp_elems = elems;
    pl->bp_sys = (size_t)n_sys;
  }
  st = ensure_arpls_work(pl, pl->p.n_chan, n_sys);
  if (st != MRAID_OK) return st;
  if (d_q1) {
    st = evals_for_q1(pl, (size_t)pl->n_cells, &d_evals);
    if (st != MRAID_OK) return st;
  }
  e = cudaMemsetAsync(pl->d_sweeps, 0, 3 * sizeof(unsigned long long), pl->stream);
  if (e != cudaSuccess) return cuda_fail(e, "memset");
  st = ccm_range(pl, d_data, 0, pl->p.n_sub, pl->ws.sums, nullptr);
  if (st != MRAID_OK) return st;
  // the sums pass may count zero-variance beams; nothing is normalised here
  e = cudaMemsetAsync(pl->d_degenerate, 0, sizeof(unsigned long long), pl->stream);
  if (e == cudaSuccess)
    e = MRAID_PROF(pl, K_BP_INPUT,
                   launch_bandpass_input(pl, pl->ws.sums, interval, pl->bp_y));
  if (e == cudaSuccess)
    e = MRAID_PROF(pl, K_ARPLS,
                   launch_arpls(pl, pl->bp_y, n_sys, pl->p.n_chan, bp->lam, bp->ratio,
                                bp->itermax, pl->bp_z, d_bandpass, pl->bp_iters, pl->ar_work));
  if (e == cudaSuccess)
    e = MRAID_PROF(pl, K_CCM_BP,
                   launch_ccm_bandpass(pl, pl->ws.sums, interval, pl->bp_z, pl->ws.corr));
  if (e != cudaSuccess) return cuda_fail(e, "bandpass kernels");
  e = MRAID_PROF(pl, K_EIG, launch_eig(pl, pl->ws.corr, pl->n_cells, d_evals, d_q1, d_stat));
  if (e != cudaSuccess) return cuda_fail(e, "eig launch");
  e = MRAID_PROF(pl, K_FLAG, launch_flag(pl, d_stat, d_flags));
  if (e != cudaSuccess) return cuda_fail(e, "flag launch");
  e = cudaMemcpyAsync(&pl->d_info->n_degenerate, pl->d_degenerate, sizeof(int64_t),
                      cudaMemcpyDeviceToDevice, pl->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(&pl->d_info->jacobi_sweeps, pl->d_sweeps, 2 * sizeof(int64_t),
                        cudaMemcpyDeviceToDevice, pl->stream);
  if (e == cudaSuccess)  // the FP64 q1 count (low half of the counter)
    e = cudaMemcpyAsync(&pl->d_info->q1_refined, pl->d_sweeps + 2, sizeof(int32_t),
                        cudaMemcpyDeviceToDevice, pl->stream);
  if (e != cudaSuccess) return cuda_fail(e, "counter copy");
  return enqueue_info_copy(pl, info);
}
