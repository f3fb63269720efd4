// flag.cu - iterative Gaussian-fit masking of the normalised dominant
// eigenvalue (Section 3.3 masking paragraph; threshold multiple k from
// Section 4.5; preserved channels from Section 4.3).
//
// Up to kClCells cells per CTA of one cluster (16 CTAs: 860 000 cells; the
// 10 s FAST block has 819 200), flag_cluster_kernel: the statistic is read
// once into the cluster's shared memory and every pass runs from there, with
// a cluster barrier per pass. Larger blocks take flag_kernel.
//
// flag_kernel: one cooperative launch runs the whole iteration: every pass
// masks the cells above the previous threshold, reduces (count, sum s,
// sum s^2) over the cells still unmasked and unpreserved (per thread in
// FP32 over its ~10 cells, then in FP64; the per-cell tests are FP32 and
// decide exactly as FP64 would), and
// derives mu, sigma (population) and mu + k sigma. The fit stops when a
// pass masks nothing new (the unmasked count is unchanged) or after
// max_clip_iter fits. Block partial sums are combined in a fixed order by
// every block, so the result is deterministic.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "internal.h"

namespace cg = cooperative_groups;

namespace mraid {
namespace {

constexpr int kFlagThreads = 512;

struct FlagArgs {
  const float* stat;
  int64_t n_cells;
  int n_chan;
  const uint8_t* keep;  // device [n_chan] or nullptr
  double k_sigma;
  int max_iter;
  uint8_t* flags;
  double* partials;     // [2][gridDim.x][3]
  mraid_flag_info* info;
};

// Block totals of (a, b, c): a fixed shuffle tree per warp, then the warps'
// totals in a fixed order. Only thread 0 receives the block totals (it alone
// publishes them); the other threads skip that FP64 loop, which GB300 would
// otherwise issue once per warp at a small fraction of the FP32 rate.
__device__ __forceinline__ void block_sum3(double& a, double& b, double& c, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
    c += __shfl_xor_sync(0xffffffffu, c, o);
  }
  const int w = threadIdx.x / 32, nw = blockDim.x / 32;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) {
    red[3 * w] = a;
    red[3 * w + 1] = b;
    red[3 * w + 2] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a = b = c = 0.0;
    for (int i = 0; i < nw; ++i) {  // fixed order
      a += red[3 * i];
      b += red[3 * i + 1];
      c += red[3 * i + 2];
    }
  }
}

// Sum of the per-block partials [nb][3] in a fixed order: lane l takes
// blocks l, l+32, ... sequentially, then a fixed shuffle tree; every block
// computes the same bits. Result broadcast through shared memory.
__device__ __forceinline__ void grid_total3(const double* part, int nb, double* bcast, double& a,
                                            double& b, double& c) {
  if (threadIdx.x < 32) {
    double x = 0.0, y = 0.0, z = 0.0;
    for (int i = threadIdx.x; i < nb; i += 32) {
      x += part[3 * i];
      y += part[3 * i + 1];
      z += part[3 * i + 2];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      x += __shfl_xor_sync(0xffffffffu, x, o);
      y += __shfl_xor_sync(0xffffffffu, y, o);
      z += __shfl_xor_sync(0xffffffffu, z, o);
    }
    if (threadIdx.x == 0) {
      bcast[0] = x;
      bcast[1] = y;
      bcast[2] = z;
    }
  }
  __syncthreads();
  a = bcast[0];
  b = bcast[1];
  c = bcast[2];
  __syncthreads();
}

// Unroll of the per-cell loop: a thread issues the loads of kFlagUnroll
// cells before it uses them (and before any store), in its usual cell order.
constexpr int kFlagUnroll = 4;

__global__ void __launch_bounds__(kFlagThreads) flag_kernel(FlagArgs f) {
  cg::grid_group grid = cg::this_grid();
  __shared__ double red[3 * (kFlagThreads / 32)];
  __shared__ double bcast[3];
  // the fit's state, kept by thread 0: mu, sigma, cells used, previous count
  __shared__ double fit_state[4];
  __shared__ double fit_thresh;
  __shared__ int fit_stop;
  const float* __restrict__ stat = f.stat;
  uint8_t* __restrict__ flags = f.flags;
  const uint8_t* __restrict__ keep = f.keep;
  const int64_t n = f.n_cells;
  const uint32_t n_chan = (uint32_t)f.n_chan;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nthr = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = tid; i < n; i += nthr) flags[i] = 0;

  double thresh = INFINITY;
  int fits = 0, converged = 0;
  if (threadIdx.x == 0) {
    fit_state[0] = 0.0;   // mu
    fit_state[1] = 0.0;   // sigma
    fit_state[2] = 0.0;   // cells in the last fit
    fit_state[3] = -1.0;  // unmasked count of the last fit
  }
  for (int pass = 0;; ++pass) {
    // The mask test v > thresh for a float v equals v > tf with tf the
    // largest float <= thresh: no float lies in (tf, thresh]. So the cells
    // need no FP64 (GB300 runs it at a small fraction of the FP32 rate).
    const float tf = __double2float_rd(thresh);
    // a thread's few cells sum in FP32 in a fixed order; blocks and the
    // grid combine in FP64, fixed order
    int cnt_t = 0;
    float s1_t = 0.f, s2_t = 0.f;
    for (int64_t i0 = tid; i0 < n; i0 += kFlagUnroll * nthr) {
      float v[kFlagUnroll];
      uint8_t m[kFlagUnroll];
#pragma unroll
      for (int u = 0; u < kFlagUnroll; ++u) {
        const int64_t i = i0 + u * nthr;
        const bool mine = i < n && !(keep && keep[(uint32_t)i % n_chan]);
        v[u] = mine ? stat[i] : 0.f;
        m[u] = mine ? flags[i] : (uint8_t)2;  // 2: past the end or preserved
      }
#pragma unroll
      for (int u = 0; u < kFlagUnroll; ++u) {
        if (m[u] == 0 && v[u] > tf) {
          m[u] = 1;
          flags[i0 + u * nthr] = 1;
        }
        if (m[u] == 0) {
          ++cnt_t;
          s1_t += v[u];
          s2_t = fmaf(v[u], v[u], s2_t);
        }
      }
    }
    double cnt = (double)cnt_t, s1 = (double)s1_t, s2 = (double)s2_t;
    block_sum3(cnt, s1, s2, red);
    double* part = f.partials + (size_t)(pass & 1) * gridDim.x * 3;
    if (threadIdx.x == 0) {
      part[3 * blockIdx.x] = cnt;
      part[3 * blockIdx.x + 1] = s1;
      part[3 * blockIdx.x + 2] = s2;
    }
    grid.sync();
    grid_total3(part, gridDim.x, bcast, cnt, s1, s2);
    // Thread 0 of every block makes the same decision and fit from the same
    // totals; its block takes the threshold and the decision from it. The
    // fit's state (fit_state, fits, converged) is thread 0's, and block 0's
    // thread 0 writes the report.
    if (threadIdx.x == 0) {
      int stop = 0;
      if (pass >= 1 && cnt == fit_state[3]) {  // the last threshold masked nothing
        converged = 1;
        stop = 1;
      } else if (fits == f.max_iter) {  // mask already holds max_iter markings
        stop = 1;
      } else if (cnt == 0.0) {  // nothing left to fit
        fit_state[0] = fit_state[1] = 0.0;
        thresh = INFINITY;
        fit_state[2] = 0.0;
        ++fits;
        converged = 1;
        stop = 1;
      } else {
        const double mu = s1 / cnt;
        const double sigma = sqrt(fmax(s2 / cnt - mu * mu, 0.0));
        thresh = mu + f.k_sigma * sigma;
        fit_state[0] = mu;
        fit_state[1] = sigma;
        fit_state[2] = cnt;
        fit_state[3] = cnt;
        ++fits;
      }
      fit_thresh = thresh;
      fit_stop = stop;
    }
    // the next pass writes these only after its own block barriers
    __syncthreads();
    thresh = fit_thresh;
    if (fit_stop) break;
  }
  // totals for the report. "Near" is |s - thresh| <= 2e-4 s, evaluated in
  // FP32 and redone in FP64 only within 1 % of the boundary: tfin is within
  // one float ulp (1.2e-7 relative) of thresh and the FP32 difference
  // carries a rounding error of the same order, far inside the 1 % band,
  // so every decision outside the band is the FP64 one.
  const float tfin = __double2float_rd(thresh);
  int nflag_t = 0, nnear_t = 0;
  for (int64_t i = tid; i < n; i += nthr) {
    nflag_t += flags[i];
    if (keep && keep[(uint32_t)i % n_chan]) continue;
    const float v = stat[i];
    const float a = fabsf(v - tfin), b = 2e-4f * v;
    bool near;
    if (!(b > 1e-30f) || fabsf(a - b) <= 1e-2f * b)
      near = fabs((double)v - thresh) <= 2e-4 * (double)v;
    else
      near = a < b;
    nnear_t += near;
  }
  double nflag = (double)nflag_t, nnear = (double)nnear_t, dummy = 0.0;
  block_sum3(nflag, nnear, dummy, red);
  grid.sync();  // everyone has read this pass's partials before they are reused
  double* part = f.partials;
  if (threadIdx.x == 0) {
    part[3 * blockIdx.x] = nflag;
    part[3 * blockIdx.x + 1] = nnear;
    part[3 * blockIdx.x + 2] = 0.0;
  }
  grid.sync();
  if (blockIdx.x == 0) {
    double tf = 0.0, tn = 0.0, unused = 0.0;
    grid_total3(part, gridDim.x, bcast, tf, tn, unused);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const double tf = bcast[0], tn = bcast[1];
    mraid_flag_info* o = f.info;
    o->mu = fit_state[0];
    o->sigma = fit_state[1];
    o->thresh = thresh;
    o->iterations = fits;
    o->converged = converged;
    o->n_flagged = (int64_t)tf;
    o->n_used = (int64_t)fit_state[2];
    o->n_near = (int64_t)tn;
  }
}

// ---------------------------------------------------------------------------
// The same iteration on one cluster. What bounds it is latency: a pass costs
// its cells' issue (about 8 instructions a cell) plus one cluster barrier,
// where the cooperative kernel pays a grid barrier and a trip of the partial
// sums through L2. Measured on GB300 (call to call, 4 to 9 fits; cooperative
// kernel, this one): 1 024 cells 62 and 24 us, 16 384 77 and 38, 77 824 78-88
// and 38-40, 409 600 107-114 and 63-66, 819 200 112-124 and 87; past 868 352
// cells (16 CTAs) the cooperative kernel, 113.
//
// Sums are taken about a pivot (the last fit's mean; for the first fit the
// mean of the block's first cells): four cells in FP32, then two floats per
// moment (value and rounding error) through a fixed tree over lanes, warps and
// CTAs, the same bits in every CTA. FP64 sums would cost more than the rest of
// a pass; the fit itself is FP64. The cells' own roundings leave the variance
// s2 / n - m^2 (m the mean's distance from the pivot) an error of 4e-7 s2 / n at
// most, so it is only used where it is at least a tenth of s2 / n. Where it is
// less (the last threshold took out cells that had moved the mean by more than
// three deviations, or the first cells were unlike the rest) the sums are taken
// again about the new mean, at the same threshold.
// Against one FP32 sum for s2 the second float and its tree cost 10 us of 75 at
// 819 200 cells and nothing at 1 024 (two-sums of eight cells instead of four
// gained 1 us).
//
// A cell out of the fit is marked in the shared copy by a NaN of its own
// (kMasked, kOutside); NaNs of the caller's are made the canonical one.
constexpr int kClThreads = 1024;
constexpr int kClCells = 53 * 1024;  // per CTA: 212 KB of shared memory
constexpr int kClMaxCtas = 16;
constexpr int kMasked = 0x7ffffffe, kOutside = 0x7fffffff;  // as int bits: above every other cell

constexpr int kClMoves = 8;  // pivots per fit: each lies 1e7 times closer to the mean

struct alignas(16) ClPart {
  float n, s1, s2, e1, e2;  // n < 2^24: exact; the moments are s1 + e1 and s2 + e2
};

__device__ __forceinline__ void cl_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cl_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// A pivot near c: sixteen significant bits, so that v - pivot is exact for v
// from pivot / 2 to 256 pivot (to 2 pivot by Sterbenz's lemma, beyond as a
// multiple of v's last bit) and, for smaller v, rounds by v's low bits alone:
// it does not lean one way over cells of like values. No shift for
// infinities and NaN.
__device__ __forceinline__ float pivot_near(float c) {
  return fabsf(c) < 1e30f ? __uint_as_float(__float_as_uint(c) & 0xffffff00u) : 0.f;
}
// s + e = a + b exactly (Knuth's two-sum)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float t = s - a;
  e = (a - (s - t)) + (b - t);
}
// one level of a butterfly over the lanes
__device__ __forceinline__ void add_lanes(ClPart& p, int o) {
  const float n = __shfl_xor_sync(0xffffffffu, p.n, o);
  const float s1 = __shfl_xor_sync(0xffffffffu, p.s1, o), e1 = __shfl_xor_sync(0xffffffffu, p.e1, o);
  const float s2 = __shfl_xor_sync(0xffffffffu, p.s2, o), e2 = __shfl_xor_sync(0xffffffffu, p.e2, o);
  float t1, r1, t2, r2;
  two_sum(p.s1, s1, t1, r1);
  two_sum(p.s2, s2, t2, r2);
  p = ClPart{p.n + n, t1, t2, r1 + (p.e1 + e1), r2 + (p.e2 + e2)};
}
// s + e (no error term beside an infinity or NaN)
__device__ __forceinline__ double moment(float s, float e) {
  return (double)s + (isfinite(s) ? (double)e : 0.0);
}
// part (in this CTA's shared memory) of CTA `rank`
__device__ __forceinline__ void cl_store(ClPart* part, int rank, const ClPart& p) {
  uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(part)), r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(r), "f"(p.n), "f"(p.s1),
               "f"(p.s2), "f"(p.e1)
               : "memory");
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(r + 16), "f"(p.e2) : "memory");
}

__global__ void __launch_bounds__(kClThreads, 1) flag_cluster_kernel(FlagArgs f, int per, int vec) {
  extern __shared__ __align__(16) int4 quads[];  // four cells each, as bits
  __shared__ ClPart red[kClThreads / 32];
  __shared__ ClPart part[2][kClMaxCtas];
  __shared__ double fit_thresh;
  __shared__ float fit_pivot;
  __shared__ int fit_stop;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x, rank = blockIdx.x;
  // a CTA's shared memory may be written only once it has started: every CTA
  // arrives here and waits before its first store to the others
  if (G > 1) cl_arrive();
  const int64_t base = (int64_t)rank * per;
  const int mine = (int)max((int64_t)0, min((int64_t)per, f.n_cells - base));
  const int nq = (mine + 3) / 4;
  auto load = [&](int i) -> int {  // cell i of this CTA
    if (i >= mine) return kOutside;
    if (f.keep && f.keep[(uint32_t)(base + i) % (uint32_t)f.n_chan]) return kOutside;
    const float v = f.stat[base + i];
    return v != v ? 0x7fc00000 : __float_as_int(v);
  };
  if (vec && !f.keep) {
    const float4* src = reinterpret_cast<const float4*>(f.stat + base);
#pragma unroll 8
    for (int q = tid; q < mine / 4; q += kClThreads) {
      const float4 v = src[q];
      quads[q] = make_int4(v.x != v.x ? 0x7fc00000 : __float_as_int(v.x),
                           v.y != v.y ? 0x7fc00000 : __float_as_int(v.y),
                           v.z != v.z ? 0x7fc00000 : __float_as_int(v.z),
                           v.w != v.w ? 0x7fc00000 : __float_as_int(v.w));
    }
    if (tid == 0 && mine % 4)
      quads[nq - 1] = make_int4(load(4 * nq - 4), load(4 * nq - 3), load(4 * nq - 2), load(4 * nq - 1));
  } else {
    for (int q = tid; q < nq; q += kClThreads)
      quads[q] = make_int4(load(4 * q), load(4 * q + 1), load(4 * q + 2), load(4 * q + 3));
  }

  // block totals of per-thread parts in every lane of warp 0
  auto block3 = [&](ClPart p) -> ClPart {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) add_lanes(p, o);
    if (lane == 0) red[warp] = p;
    __syncthreads();
    if (warp == 0) {
      p = red[lane];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) add_lanes(p, o);
    }
    return p;
  };
  // the CTAs' totals of buffer `buf` summed, in every lane of warp 0 (the
  // other warps only take part in the barrier)
  auto cluster3 = [&](int buf, ClPart p) -> ClPart {
    if (G == 1) return p;
    if (warp == 0 && lane < G) cl_store(&part[buf][rank], lane, p);
    cl_arrive();
    cl_wait();
    if (warp == 0) {
      p = lane < G ? part[buf][lane] : ClPart{};
#pragma unroll
      for (int o = kClMaxCtas / 2; o > 0; o >>= 1) add_lanes(p, o);
    }
    return p;
  };

  // first pivot: the mean of the block's first cells (the same in every CTA)
  {
    const bool use = tid < f.n_cells && !(f.keep && f.keep[tid % f.n_chan]);
    const float v = use ? f.stat[tid] : 0.f;
    const ClPart p = block3(ClPart{use ? 1.f : 0.f, v});
    if (tid == 0) {
      const float c = p.s1 / fmaxf(p.n, 1.f);
      fit_pivot = pivot_near(c);
    }
    __syncthreads();
  }
  float pivot = fit_pivot;
  double mu = 0.0, sigma = 0.0, thresh = INFINITY;  // thread 0's
  float used = 0.f, prev = -1.f;
  int fits = 0, converged = 0, pass = 0, moves = 0;
  if (G > 1) cl_wait();
  for (;; ++pass) {
    // v > thresh for a float v equals v > tf, tf the largest float <= thresh
    const float tf = __double2float_rd(thresh);
    int cnt = 0;
    float s1 = 0.f, s2 = 0.f, e1 = 0.f, e2 = 0.f;
#pragma unroll 4
    for (int q = tid; q < nq; q += kClThreads) {
      int4 w = quads[q];
      bool changed = false;
      float quad = 0.f, quad2 = 0.f;
      auto cell = [&](int& x) {
        const float v = __int_as_float(x);
        if (v > tf) {  // false for the marks
          x = kMasked;
          changed = true;
        } else if (x < kMasked) {
          const float d = v - pivot;
          ++cnt;
          quad += d;
          quad2 = fmaf(d, d, quad2);
        }
      };
      cell(w.x);
      cell(w.y);
      cell(w.z);
      cell(w.w);
      if (changed) quads[q] = w;
      float e;
      two_sum(s1, quad, s1, e);
      e1 += e;
      two_sum(s2, quad2, s2, e);
      e2 += e;
    }
    const ClPart p = cluster3(pass & 1, block3(ClPart{(float)cnt, s1, s2, e1, e2}));
    if (tid == 0) {
      int stop = 0;
      bool again = false;
      if (pass >= 1 && p.n == prev) {  // the last threshold masked nothing
        converged = 1;
        stop = 1;
      } else if (fits == f.max_iter) {  // mask already holds max_iter markings
        stop = 1;
      } else if (p.n == 0.f) {  // nothing left to fit
        mu = sigma = 0.0;
        used = 0.f;
        thresh = INFINITY;
        ++fits;
        converged = 1;
        stop = 1;
      } else {
        const double inv = 1.0 / (double)p.n;
        const double m = moment(p.s1, p.e1) * inv, q = moment(p.s2, p.e2) * inv;
        mu = (double)pivot + m;
        fit_pivot = pivot_near((float)mu);
        if (m * m > 0.9 * q && moves < kClMoves) {
          // too far: the same cells about the new mean, by all its bits where
          // the coarse pivot is the one that was too far
          if (moves > 0 || fit_pivot == pivot) fit_pivot = (float)mu;
          again = fit_pivot != pivot;
        }
        if (again) {
          ++moves;
        } else {
          sigma = sqrt(fmax(q - m * m, 0.0));
          thresh = mu + f.k_sigma * sigma;
          used = prev = p.n;
          moves = 0;
          fit_pivot = pivot_near((float)mu);
          ++fits;
        }
      }
      fit_thresh = thresh;
      fit_stop = stop;
    }
    __syncthreads();
    thresh = fit_thresh;
    pivot = fit_pivot;
    if (fit_stop) break;
  }
  // the flags and the report ("near": |s - thresh| <= 2e-4 s, in FP64 only
  // within 1 % of that boundary)
  const float tfin = __double2float_rd(thresh);
  int near = 0, hits = 0;
  for (int q = tid; q < nq; q += kClThreads) {
    const int4 w = quads[q];
    const int x[4] = {w.x, w.y, w.z, w.w};
    uint32_t bytes = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float v = __int_as_float(x[i]);
      if (x[i] == kMasked) {
        bytes |= 1u << (8 * i);
        ++hits;
        v = f.stat[base + 4 * q + i];
      }
      const float a = fabsf(v - tfin), b = 2e-4f * v;
      bool is = a < b;
      if (!(b > 1e-30f) || fabsf(a - b) <= 1e-2f * b)
        is = fabs((double)v - thresh) <= 2e-4 * (double)v;
      near += x[i] != kOutside && is;
    }
    uint8_t* dst = f.flags + base + 4 * q;
    if (vec && 4 * q + 4 <= mine) {
      *reinterpret_cast<uint32_t*>(dst) = bytes;
    } else {
      for (int i = 0; i < 4 && 4 * q + i < mine; ++i) dst[i] = (uint8_t)(bytes >> (8 * i));
    }
  }
  // the buffer of the pass before: a CTA may still read the last pass's
  const ClPart p = cluster3((pass + 1) & 1, block3(ClPart{(float)hits, (float)near}));
  if (rank == 0 && tid == 0) {
    mraid_flag_info* o = f.info;
    o->mu = mu;
    o->sigma = sigma;
    o->thresh = thresh;
    o->iterations = fits;
    o->converged = converged;
    o->n_flagged = (int64_t)p.n;
    o->n_used = (int64_t)used;
    o->n_near = (int64_t)p.s1;
  }
}

}  // namespace

int flag_cluster_ctas(int device) {
  static const int sizes[] = {16, 8};
  (void)device;
  for (int g : sizes) {
    if (cudaFuncSetAttribute(flag_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed,
                             1) != cudaSuccess ||
        cudaFuncSetAttribute(flag_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kClCells * (int)sizeof(float)) != cudaSuccess)
      break;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(g);
    cfg.blockDim = dim3(kClThreads);
    cfg.dynamicSmemBytes = kClCells * sizeof(float);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim = {(unsigned)g, 1, 1};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, flag_cluster_kernel, &cfg) == cudaSuccess &&
        clusters >= 1)
      return g;
  }
  cudaGetLastError();
  return 0;
}

int flag_grid_blocks(int device, int sm_count) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, flag_kernel, kFlagThreads, 0) !=
          cudaSuccess ||
      per_sm < 1)
    return 0;
  (void)device;
  return sm_count;  // one block per SM: fewer partials to combine
}

cudaError_t launch_flag(mraid_plan_s* pl, const float* d_stat, uint8_t* d_flags, int64_t n_cells,
                        mraid_flag_info* d_info) {
  FlagArgs f;
  f.stat = d_stat;
  f.n_cells = n_cells >= 0 ? n_cells : pl->n_cells;
  f.n_chan = pl->p.n_chan;
  f.keep = pl->d_keep;
  f.k_sigma = pl->p.eig_k;
  f.max_iter = pl->p.max_clip_iter;
  f.flags = d_flags;
  f.partials = pl->d_partials;
  f.info = d_info ? d_info : pl->d_info;
  if (f.n_cells <= (int64_t)pl->flag_ctas * kClCells) {
    // CTAs of up to 16 K cells: there a pass's cells (16 a thread, ~0.6 us)
    // cost what a cluster barrier does, so a narrower cluster would not gain
    int g = 1;
    while (g < pl->flag_ctas && f.n_cells > (int64_t)g * 16384) g *= 2;
    const int64_t per = ((f.n_cells + g - 1) / g + 3) / 4 * 4;
    const int vec = ((reinterpret_cast<uintptr_t>(d_stat) & 15) |
                     (reinterpret_cast<uintptr_t>(d_flags) & 3)) == 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(g);
    cfg.blockDim = dim3(kClThreads);
    cfg.dynamicSmemBytes = (size_t)per * sizeof(float);
    cfg.stream = pl->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim = {(unsigned)g, 1, 1};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, flag_cluster_kernel, f, (int)per, vec);
  }
  // cooperative launch (all blocks co-resident for the grid barrier), in the
  // form that stream capture accepts
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(pl->flag_blocks);
  cfg.blockDim = dim3(kFlagThreads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = pl->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, flag_kernel, f);
}

}  // namespace mraid
