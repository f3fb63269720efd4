// gram_mma.cu - exact augmented Gram sums of 8-bit multi-beam data for 2..39
// beams, fused with the correlation.
//
// Section 3.2, Eq. 1. For a cell (channel j, sub-integration k) with samples
// x_b(t), the kernel forms G = Y Y^T with Y = [x - 128; 1]. The centred
// values are exact in f16, products are integers of magnitude <= 2^14 and
// sums over <= 1024 samples are integers of magnitude <= 2^24, so FP32
// accumulation is exact; longer sub-integrations are added up every 1024
// samples, as int32 in shared memory for up to 127 such pieces and as int64
// in the sums beyond that. cov_ab = n G_ab - G_a G_b is exact in int64 and
// r_ab = cov_ab / sqrt(var_a var_b) is rounded to float once. The raw sums
// are S_ab = G_ab + 128 (G_a + G_b) + 128^2 n and S_a = G_a + 128 n.
//
// Why register fragments (mma.sync) and not tcgen05: a cell's Gram is 40 x 40
// at most, and the samples lie channel by channel in memory. A 128-row
// tcgen05 tile of 16 beams x 8 channels keeps 1/8 of its products, and its
// operands cross shared memory 5 times as f16; that kernel was bound by
// shared memory at 3.4 TB/s of samples. Here a warp owns 8 channels (4 from 24 beams on) and every
// product is of one channel: a lane reads the warp's channels of one beam
// and one sample, a pair of samples becomes an f16x2 register by byte
// permutes (x in the low mantissa bits of 1024, minus 1152), and that
// register is at once an A and a B fragment of its channel's Gram, because
// the order of the samples within K is free. Products per channel and 16
// samples: each pair of 8-beam block rows x the block columns from its first
// on, and the last block of an odd count by itself.
//
// Layout: a work item is one sub-integration x 32, 64, 96 or 128 channels
// (4, 8, 12 or 16 warps, as many as the accumulators leave registers for; 32
// channels and 8 warps from 24 beams on; 16 channels and 2 warps for narrow
// blocks; items of 4 warps and fewer share an SM);
// stages of 16 samples x all beams come by TMA with a swizzle under which a
// warp's 8-byte loads meet two-way conflicts at most, into a ring as deep as
// shared memory allows; the warps take turns to issue the copies. Wide rows
// on their own multiples matter: 16- and 32-byte rows stream
// at 4.7-4.8 TB/s on GB300, 64-byte ones at 6.3-6.7, 128-byte ones at 7.1.
// Layouts that no tensor map takes (odd channel counts, misaligned buffers)
// fill the same ring by cp.async, or at odd addresses from pairs of aligned
// words (36 beams x 1001 channels x 1000 samples x 20 1.15 ms, on dp4a 5.7; x
// 1000 channels, in 8-byte copies, 0.64).
//
// Measured on GB300 (50 sub-integrations x 4096 channels x 1024 samples):
// 19 beams 0.89 ms (4.5 TB/s of samples; the tcgen05 kernel 1.20 ms), 13
// beams 0.54 ms (0.91), 7 beams 0.35 ms (0.84); with 128 samples per
// sub-integration, where the epilogue weighs most, 1.70, 0.98 and 0.63 ms
// (6.27, 4.64 and 4.21). 1000 channels x 1000 samples x 40 (no tensor map)
// 0.38 ms, on dp4a 0.62 ms. With more than 1024 samples and from 24 beams on,
// correlation included: 36 beams x 2048 channels x 2048 samples x 38 1.58 ms
// (tcgen05 with two channels per 128-row tile 3.52 + 0.17), 24 beams x 4096 x
// 1024 x 20 0.66 ms (1.27 + 0.09), 39 beams x 2048 x 1024 x 38 0.87 ms (1.82
// + 0.22); at 40 beams the accumulators of four channels would no longer fit
// a warp's registers. Without its copies the 19-beam kernel takes 0.75
// ms, without its products 0.8: bound by both, the permutes' and MMAs' issue
// at 3 warps per scheduler and the copies that pause in the epilogue.
//
// Every wait is bounded by the plan's limit; on expiry the kernel records an
// error word, waits (again bounded) for its copies in flight and returns.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

#include "internal.h"
#include "tc_ptx.h"

namespace mraid {
namespace {

constexpr int kMmLag = 1;  // stages between a slot's last read and its refill
constexpr int kMmT = 16;                     // samples per stage: one K step
constexpr int kMmMaxD = 12;                  // ring depth bound
constexpr int kMmPiece = 1024;               // samples accumulated before a flush
constexpr int kMmLongMax = kMmPieceMax;      // samples whose int32 sums cannot overflow (127 pieces)
constexpr size_t kMmSmem = 226 * 1024;
constexpr int kMmEpi = 2;                    // channels staged at a time by the epilogue

// NB 8-beam blocks; kHalf: the last one holds at most four slots, and its
// fragment carries them for two channels (lanes of rows 0..3 the even one,
// 4..7 the odd one); A_, B_: channels of a stage's two boxes (B_ 0: one box).
// kLong_: sub-integrations of several pieces, added as int32 in shared memory.
template <int NB_, bool kHalf_, int A_, int B_, int CW_ = 8, bool kLong_ = false>
struct MmCfg {
  static constexpr bool kLong = kLong_;
  static constexpr int kCW = CW_;  // channels per warp
  static constexpr int NB = NB_, kChA = A_, kChB = B_, kCh = A_ + B_;
  static constexpr bool kHalf = kHalf_;
  static constexpr int kWarps = kCh / kCW, kThreads = 32 * kWarps;
  // CTAs per SM where there are more items than SMs: four warps leave an SM
  // idle between the steps of their chain (with one CTA, 19 beams x 16 channels
  // x 1024 samples x 250 took 81 us, so 55; 7 beams x 24 channels x 166 95 and
  // 54)
  static constexpr int kCtas = (kWarps > 4 ? 1 : (NB_ == 1 ? 3 : 2)) * (kWarps == 2 ? 2 : 1);
  static constexpr int kTile = kMmT * kCh;  // bytes of one beam in a stage
  // One channel's products in the epilogue, in floats: per block row pair
  // (2p, 2p + 1) the 8 x 8 of the diagonal block 2p, then 16 x 8 for every
  // later block column; the last block of an odd count by itself.
  __host__ __device__ static constexpr int pair_at(int p) {
    int at = 0;
    for (int q = 0; q < p; ++q) at += 64 + 128 * (NB - 1 - 2 * q);
    return at;
  }
  static constexpr int kG = kHalf ? 272 : pair_at(NB / 2) + (NB & 1 ? 64 : 0);
  using Sum = typename std::conditional<kLong, int32_t, float>::type;
  struct Shared {
    uint64_t full[kMmMaxD], empty[kMmMaxD];
    uint32_t lut[(8 * NB) * (8 * NB + 1) / 2];  // G offset | a << 16 | b << 24
    // a group of channels' products; of several pieces, every channel's sums
    alignas(16) Sum g[kWarps][kLong ? kCW : kMmEpi][kG];
    int2 row[kWarps][kMmEpi][8 * NB];  // per beam: sum of the centred samples, 1/sqrt(var)
  };
  // Where the pair (a, b), a <= b, lies in a channel's products.
  __host__ __device__ static constexpr int off(int a, int b) {
    const int ba = a >> 3, bb = b >> 3, e = (a & 7) * 8 + (b & 7);
    if (kHalf && bb == 2)
      return ba < 2 ? 192 + a * 4 + (b & 7) : 256 + (a & 7) * 4 + (b & 7);
    int at = 0;
    for (int q = 0; q < ba / 2; ++q) at += 64 + 128 * (NB - 1 - 2 * q);
    if (bb == (ba & ~1)) return at + e;
    return at + 64 + (bb - (ba & ~1) - 1) * 128 + (ba & 1) * 64 + e;
  }
  static constexpr size_t kFixed = 1024 + sizeof(Shared);
  static constexpr int stage_bytes(int n_beam) { return (n_beam + 2) * kTile; }
  static constexpr int depth(int n_beam, int ctas) {
    const size_t room = ctas > 1 ? kMmSmem / ctas - 1024 : kMmSmem;
    const int d = (int)((room - kFixed) / (size_t)stage_bytes(n_beam));
    return d < kMmMaxD ? d : kMmMaxD;
  }
};

struct MmArgs {
  const uint8_t* data;  // plain copies: the samples, beams beam_stride apart
  int64_t beam_stride;
  const uint8_t* data_end;  // one past the last sample
  int vec;  // plain copies: bytes per copy (8 or 4: cp.async; 1: any address)
  int n_beam, n_chan, n_samp_sub, sub0, n_sub;
  int depth;  // ring stages
  int64_t* sums;
  float* corr;
  unsigned long long* degenerate;
  unsigned* error;
  unsigned long long wait_ns;
  long long withhold;
};

__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9},"
      " {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// (float)x for |x| < 2^44, rounded once: both parts are exact in float
// (taken as mantissa bits: the integer conversions run at a quarter of the
// add rate).
__device__ __forceinline__ float i64_to_float(int64_t x) {
  const int hi = (int)(x >> 23);
  const uint32_t lo = (uint32_t)x & 0x7fffffu;
  return fmaf(__int_as_float(0x4b400000 + hi) - 12582912.f, 8388608.f,
              __uint_as_float(0x4b000000u | lo) - 8388608.f);
}

template <bool kLong>
__device__ __forceinline__ float cov_to_float(int64_t x) {
  if constexpr (kLong) return (float)x;  // beyond the two mantissas
  else return i64_to_float(x);
}

__device__ __forceinline__ uint32_t f16_sub(uint32_t x, uint32_t y) {
  uint32_t r;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(y));
  return r;
}

template <int kImm>
__device__ __forceinline__ void lds_word(uint32_t addr, uint2& v) {
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2+%3];" : "=r"(v.x), "=r"(v.y) : "r"(addr), "n"(kImm));
}
template <int kImm>
__device__ __forceinline__ void lds_word(uint32_t addr, uint1& v) {
  asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v.x) : "r"(addr), "n"(kImm));
}
__device__ __forceinline__ uint32_t word(const uint2& v, int q) { return q ? v.y : v.x; }
__device__ __forceinline__ uint32_t word(const uint1& v, int) { return v.x; }
template <class F, int... I>
__device__ __forceinline__ void static_loop_(F&& f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}
template <int K, class F>
__device__ __forceinline__ void static_loop(F&& f) {  // f(constant 0 .. K - 1)
  static_loop_(f, std::make_integer_sequence<int, K>{});
}
// A lane constant that the compiler keeps instead of computing it again.
__device__ __forceinline__ void pin(uint32_t& x) { asm volatile("" : "+r"(x)); }

// The XOR that a tensor map's swizzle of `pitch` bytes applies to the 16-byte
// column of row r (rows `pitch` bytes apart).
__device__ __forceinline__ int swizzle(int pitch, int r) {
  return pitch == 128 ? r & 7 : (pitch == 64 ? (r >> 1) & 3 : (pitch == 32 ? (r >> 2) & 1 : 0));
}

// One cp.async of kBytes; the barrier's phase completes when every thread's
// copies have landed.
template <int kBytes>
__device__ __forceinline__ void copy_async(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(kBytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive_copies(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

template <class C, bool kTma>
__global__ void __launch_bounds__(C::kThreads, C::kCtas)
gram_mma_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                const MmArgs g) {
  constexpr int NB = C::NB;
  constexpr bool kHalf = C::kHalf;
  using Shared = typename C::Shared;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* ring = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int N = g.n_beam, D = g.depth;
  const int stage_bytes = (N + 2) * C::kTile, box_a = (N + 2) * kMmT * C::kChA;
  Shared* s = reinterpret_cast<Shared*>(ring + (size_t)D * stage_bytes);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int chunks = (g.n_chan + C::kCh - 1) / C::kCh;
  const int items = g.n_sub * chunks;
  const int stages = (g.n_samp_sub + kMmT - 1) / kMmT;
  const int my_items =
      ((int)blockIdx.x < items) ? (items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  const int total = my_items * stages;  // a CTA's share of device memory: far below 2^31

  if (threadIdx.x == 0) {
    for (int i = 0; i < D; ++i) {
      mbar_init(&s->full[i], kTma ? 1 : C::kThreads);
      mbar_init(&s->empty[i], C::kWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the constant beams of every stage: x - 128 = 1 in beam N, 0 in beam N + 1
  for (int i = threadIdx.x; i < D * 2 * C::kTile / 4; i += C::kThreads) {
    const int st = i / (2 * C::kTile / 4), j = 4 * (i % (2 * C::kTile / 4));
    constexpr int kA2 = 2 * kMmT * C::kChA;
    const bool one = j < kA2 ? j < kA2 / 2 : j - kA2 < kMmT * C::kChB;
    const int at = j < kA2 ? N * kMmT * C::kChA + j : box_a + N * kMmT * C::kChB + (j - kA2);
    *reinterpret_cast<uint32_t*>(ring + (size_t)st * stage_bytes + at) = one ? 0x81818181u : 0x80808080u;
  }
  const int N1 = N + 1, P = N1 * (N1 + 1) / 2;
  for (int e = threadIdx.x; e < P; e += C::kThreads) {
    int a = 0, r = e;
    while (r >= N1 - a) {
      r -= N1 - a;
      ++a;
    }
    s->lut[e] = (uint32_t)C::off(a, a + r) | ((uint32_t)a << 16) | ((uint32_t)(a + r) << 24);
  }
  __syncthreads();

  // stage r of this CTA into its ring slot by bulk tensor copies (one lane)
  auto issue = [&](int r) {
    const int it = blockIdx.x + r / stages * gridDim.x, st = r % stages, slot = r % D;
    const int k = it / chunks, ch0 = it % chunks * C::kCh;
    const int t0 = (g.sub0 + k) * g.n_samp_sub + st * kMmT;
    if (blockIdx.x == 0 && r == g.withhold) return;  // injected fault: the wait for it expires
    unsigned char* dst = ring + (size_t)slot * stage_bytes;
    mbar_expect_tx(&s->full[slot], (uint32_t)(N * C::kTile));
    tma_load_3d(dst, &map_a, ch0, t0, 0, &s->full[slot]);
    if constexpr (C::kChB > 0)
      tma_load_3d(dst + box_a, &map_b, ch0 + C::kChA, t0, 0, &s->full[slot]);
  };
  // the same by every thread's own copies, for layouts that no tensor map
  // takes; a stage has kPlaces8 or kPlaces4 places of 8 or 4 bytes a beam, and
  // the kGroups8 or kGroups4 groups of that many threads share the beams. A
  // thread's place is worked out anew each time: kept in registers it made few
  // beams 15 % faster but 19 beams x 1000 x 1000 x 40 0.52 ms instead of 0.38
  // (spills)
  constexpr int kPlaces8 = C::kCh / 8 * kMmT, kPlaces4 = C::kCh / 4 * kMmT;
  constexpr int kGroups8 = C::kThreads / kPlaces8, kGroups4 = C::kThreads / kPlaces4;
  static_assert(kGroups8 * kPlaces8 == C::kThreads && kGroups4 * kPlaces4 == C::kThreads,
                "every thread has a place, and no two the same");
  const int group4 = kGroups4 > 1 ? threadIdx.x / kPlaces4 : 0;
  int f_it = blockIdx.x, f_st = 0, f_slot = 0;  // next stage to fill
  auto fill = [&](int r) {
    const int v = g.vec, words = v == 8 ? C::kCh / 8 : C::kCh / 4;
    const int col = threadIdx.x % words, row = threadIdx.x / words % kMmT;
    const int k = f_it / chunks, cc = col * (C::kCh / words), ch = f_it % chunks * C::kCh + cc;
    const int nv = g.n_samp_sub - f_st * kMmT;
    const uint8_t* src = g.data + ((int64_t)(g.sub0 + k) * g.n_samp_sub + f_st * kMmT + row) * g.n_chan + ch;
    const bool b_box = cc >= C::kChA;
    const int pitch = b_box ? C::kChB : C::kChA, c16 = (b_box ? cc - C::kChA : cc) >> 4;
    uint32_t dst = smem_u32(ring) + (uint32_t)(f_slot * stage_bytes) + (b_box ? box_a : 0) +
                   row * pitch + ((c16 ^ swizzle(pitch, row)) << 4) + (cc & 15);
    const bool mine = row < nv && ch < g.n_chan && !(blockIdx.x == 0 && r == g.withhold);
    if (v == 8) {
      for (int b = threadIdx.x / kPlaces8; b < N; b += kGroups8)
        if (mine) copy_async<8>(dst + b * kMmT * pitch, src + b * g.beam_stride);
    } else if (v == 4) {
      for (int b = group4; b < N; b += kGroups4)
        if (mine) copy_async<4>(dst + b * kMmT * pitch, src + b * g.beam_stride);
    } else if (mine) {
      const int nc = g.n_chan - ch;
      // four bytes at any address: of the two aligned words about them, where
      // the first and the last beam's lie within the samples (one branch for
      // all beams, so that eight beams' loads are in flight)
      auto word = [](const uint8_t* p) { return p - (reinterpret_cast<uintptr_t>(p) & 3); };
      if (nc >= 4 && word(src) >= g.data &&
          word(src + (N - 1) * g.beam_stride) + 8 <= g.data_end) {
        for (int b0 = 8 * group4; b0 < N; b0 += 8 * kGroups4) {
          uint32_t lo[8], hi[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint8_t* p = src + min(b0 + j, N - 1) * g.beam_stride;
            const uint32_t* w = reinterpret_cast<const uint32_t*>(word(p));
            lo[j] = __ldg(w);
            hi[j] = __ldg(w + 1);
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int b = min(b0 + j, N - 1);
            const uint32_t at = (uint32_t)reinterpret_cast<uintptr_t>(src + b * g.beam_stride) & 3;
            const uint32_t x = __funnelshift_r(lo[j], hi[j], at * 8);
            asm volatile("st.shared.u32 [%0], %1;" ::"r"(dst + b * kMmT * pitch), "r"(x) : "memory");
          }
        }
      } else {
#pragma unroll 4
        for (int b = group4; b < N; b += kGroups4) {
          const uint8_t* p = src + b * g.beam_stride;
          uint32_t x = p[0];
          if (nc > 1) x |= (uint32_t)p[1] << 8;
          if (nc > 2) x |= (uint32_t)p[2] << 16;
          if (nc > 3) x |= (uint32_t)p[3] << 24;
          asm volatile("st.shared.u32 [%0], %1;" ::"r"(dst + b * kMmT * pitch), "r"(x) : "memory");
        }
      }
    }
    if (!(blockIdx.x == 0 && r == g.withhold)) {
      if (v == 1) mbar_arrive(&s->full[f_slot]);
      else mbar_arrive_copies(&s->full[f_slot]);
    }
    if (++f_slot == D) f_slot = 0;
    if (++f_st == stages) {
      f_st = 0;
      f_it += gridDim.x;
    }
  };
  int last_issued = -1;
  if constexpr (kTma) {
    if (threadIdx.x == 0) {
      for (int i = 0; i < D && i < total; ++i) issue(i);
      last_issued = min(D, total) - 1;
    }
  } else {
    for (int i = 0; i < D && i < total; ++i) fill(i);
  }

  // ---- this lane's places: beam row g8 of each 8-beam block, times t of
  // every 4; odd beams read the two halves of an 8-sample group in the
  // opposite order (their pairs are put back by the permute selectors)
  const int g8 = lane >> 2, t = lane & 3, odd = g8 & 1;
  const bool in_a = warp < C::kChA / C::kCW;
  const int pitch = in_a ? C::kChA : C::kChB;                       // bytes per row
  const int wc = in_a ? warp >> 1 : (warp - C::kChA / C::kCW) >> 1;   // 16-byte column
  const int cb = C::kCW * warp - (in_a ? 0 : C::kChA);
  auto place = [&](int r) {  // this warp's bytes of row r, swizzled
    if constexpr (C::kCW == 8) return r * pitch + ((wc ^ swizzle(pitch, r)) << 4) + ((warp & 1) << 3);
    return r * pitch + (((cb >> 4) ^ swizzle(pitch, r)) << 4) + (cb & 15);
  };
  const int q0 = place(t + (odd ? 4 : 0)), q1 = place(t + (odd ? 0 : 4));
  uint32_t sel_lo = odd ? 0x1504u : 0x5140u;
  uint32_t sel_half = g8 < 4 ? (odd ? 0x2604u : 0x6240u) : (odd ? 0x3715u : 0x7351u);
  uint32_t mask_even = g8 < 4 ? ~0u : 0u;
  const uint32_t magic = 0x64646464u, bias = 0x64806480u;  // 1024 + x, minus 1152
  const int last_slot = 8 * (NB - 1) + (kHalf ? g8 & 3 : g8);
  const int tile0 = in_a ? 0 : box_a;  // this warp's box within a stage
  // shared addresses of this lane's rows in ring slot 0 (slots past N: zeros)
  const uint32_t ring32 = smem_u32(ring) + tile0;
  uint32_t A0 = ring32 + g8 * kMmT * pitch + q0, A1 = ring32 + g8 * kMmT * pitch + q1;
  uint32_t L0 = ring32 + min(last_slot, N + 1) * kMmT * pitch + q0, L1 = L0 - q0 + q1;
  pin(sel_lo);
  if (kHalf) pin(sel_half);
  if (kHalf) pin(mask_even);
  pin(A0);
  pin(A1);
  pin(L0);
  pin(L1);

  // accumulator tiles per channel
  constexpr int kAcc = kHalf ? 2 : (NB / 2) * ((NB + 1) / 2 + 1) + (NB & 1);
  constexpr int kFull = kHalf ? NB - 1 : NB;

  int slot = 0;
  uint32_t ph = 0;
  int cnt = 0;
  uint32_t fill_ph = 0;  // parity of the slot's read that a plain refill waits for
  int duty = warp;       // this warp's next stage to issue: d % C::kWarps == warp, d >= D
  while (duty < D) duty += C::kWarps;
  bool ok = true;
  for (int it = blockIdx.x; it < items && ok; it += gridDim.x) {
    const int k = it / chunks, ch0 = it % chunks * C::kCh + C::kCW * warp;
    for (int piece0 = 0; piece0 < stages && ok; piece0 += kMmPiece / kMmT) {
      const int piece1 = min(stages, piece0 + kMmPiece / kMmT);
      float acc[C::kCW][kAcc][4];
      float acc2[kHalf ? C::kCW / 2 : 1][2][4];  // of two channels: blocks (0, 1) x last, last x last
#pragma unroll
      for (int c = 0; c < C::kCW; ++c)
#pragma unroll
        for (int m = 0; m < kAcc; ++m)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[c][m][i] = 0.f;
#pragma unroll
      for (int c = 0; c < (kHalf ? C::kCW / 2 : 1); ++c)
#pragma unroll
        for (int i = 0; i < 8; ++i) acc2[c][i / 4][i % 4] = 0.f;
      auto run = [&](auto pitch_c) {
        constexpr int kPitch = decltype(pitch_c)::value;
        using Word = typename std::conditional<C::kCW == 8, uint2, uint1>::type;
        for (int st = piece0; st < piece1; ++st) {
          ok = mbar_wait(&s->full[slot], ph, g.error, g.wait_ns);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          unsigned char* stage = ring + slot * stage_bytes;
          const int nv = g.n_samp_sub - st * kMmT;
          if (nv < kMmT) {  // samples of the next sub-integration: the centre value
            for (int i = lane; i < (kMmT - nv) * N; i += 32) {
              const int r = nv + i / N, b = i % N;
              Word* at = reinterpret_cast<Word*>(stage + tile0 + b * kMmT * kPitch + place(r));
              if constexpr (C::kCW == 8) *at = make_uint2(0x80808080u, 0x80808080u);
              else *at = make_uint1(0x80808080u);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
          }
          Word w[NB][2][2];
          {
            const uint32_t so = (uint32_t)(slot * stage_bytes);
            static_loop<NB>([&](auto bb) {
              constexpr int b = decltype(bb)::value;
              const uint32_t p0 = b == NB - 1 ? L0 + so : A0 + so;
              const uint32_t p1 = b == NB - 1 ? L1 + so : A1 + so;
              constexpr int o = b == NB - 1 ? 0 : b * 8 * kMmT * kPitch;
              lds_word<o>(p0, w[b][0][0]);
              lds_word<o>(p1, w[b][0][1]);
              lds_word<o + 8 * kPitch>(p0, w[b][1][0]);
              lds_word<o + 8 * kPitch>(p1, w[b][1][1]);
            });
          }
          // the stage is in registers: release it before the products
          __syncwarp();
          if (lane == 0) mbar_arrive(&s->empty[slot]);
          if (++slot == D) {
            slot = 0;
            ph ^= 1;
          }
          if constexpr (kTma) {
            // the warps take turns to refill the slot used kMmLag stages ago
            if (cnt + D - kMmLag == duty) {
              if (lane == 0 && duty < total &&
                  mbar_wait(&s->empty[duty % D], (uint32_t)((duty / D - 1) & 1), g.error, g.wait_ns)) {
                issue(duty);
                last_issued = duty;
              }
              __syncwarp();
              duty += C::kWarps;
            }
          } else {
            const int r = cnt + D - kMmLag;
            if (cnt >= kMmLag && r < total) {
              ok = mbar_wait(&s->empty[f_slot], fill_ph, g.error, g.wait_ns);
              ok = __all_sync(0xffffffffu, ok);
              if (!ok) break;
              fill(r);
              if (f_slot == 0) fill_ph ^= 1;
            }
          }
#pragma unroll
          for (int q = 0; q < C::kCW / 4; ++q) {
            // f: blocks 0.., f2: the half block, of two channels
            uint32_t f[4][kFull][2], f2[2][2];
#pragma unroll
            for (int b = 0; b < NB; ++b)
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const uint32_t x = word(w[b][h][0], q), y = word(w[b][h][1], q);
                if (b < kFull) {
                  const uint32_t lo = __byte_perm(x, y, sel_lo), hi = __byte_perm(x, y, sel_lo + 0x2222u);
#pragma unroll
                  for (int c = 0; c < 4; ++c) {
                    const uint32_t u = __byte_perm(c < 2 ? lo : hi, magic, c & 1 ? 0x4342 : 0x4140);
                    f[c][b][h] = f16_sub(u, bias);
                  }
                } else {
                  const uint32_t v = __byte_perm(x, y, sel_half);
#pragma unroll
                  for (int c = 0; c < 2; ++c) {
                    const uint32_t u = __byte_perm(v, magic, c ? 0x4342 : 0x4140);
                    f2[c][h] = f16_sub(u, bias);
                  }
                }
              }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              float(&d)[kAcc][4] = acc[4 * q + c];
              if constexpr (NB == 2 || NB == 3) {
#pragma unroll
                for (int z = 0; z < kFull; ++z)
                  mma16816(d[z], f[c][0][0], f[c][1][0], f[c][0][1], f[c][1][1], f[c][z][0],
                           f[c][z][1]);
              } else {
                int m = 0;
#pragma unroll
                for (int p = 0; p < NB / 2; ++p)
#pragma unroll
                  for (int z = 2 * p; z < kFull; ++z, ++m)
                    mma16816(d[m], f[c][2 * p][0], f[c][2 * p + 1][0], f[c][2 * p][1],
                             f[c][2 * p + 1][1], f[c][z][0], f[c][z][1]);
              }
              if constexpr (kHalf) {
                // the other channel's columns are zero here, so both add into one tile
                const uint32_t mk = c & 1 ? ~mask_even : mask_even;
                mma16816(acc2[2 * q + c / 2][0], f[c][0][0], f[c][1][0], f[c][0][1],
                         f[c][1][1], f2[c / 2][0] & mk, f2[c / 2][1] & mk);
              } else if constexpr (NB & 1) {
                constexpr int L = NB - 1;
                const int p = c & ~1;
                mma16816(d[kAcc - 1], f[p][L][0], f[p + 1][L][0], f[p][L][1], f[p + 1][L][1],
                         f[c][L][0], f[c][L][1]);
              }
            }
            if constexpr (kHalf) {
#pragma unroll
              for (int p = 0; p < 2; ++p)
                mma16816(acc2[2 * q + p][1], f2[0][0], f2[1][0], f2[0][1], f2[1][1], f2[p][0],
                         f2[p][1]);
            }
          }
          ++cnt;
        }
      };
      if (C::kChB == 0 || in_a) run(std::integral_constant<int, C::kChA>{});
      else run(std::integral_constant<int, C::kChB>{});
      if (!ok) break;
      if (ch0 >= g.n_chan) continue;
      // ---- epilogue: a few channels at a time through the warp's staging area
      const int n = C::kLong ? g.n_samp_sub : min(g.n_samp_sub - piece0 * kMmT, kMmPiece);
      // channel c's accumulators into sg, or (several pieces) added to it
      auto stage_out = [&](auto cc, typename C::Sum* sg) {
        constexpr int c = decltype(cc)::value;
        auto put = [&](int at, const float* d) {
          if constexpr (C::kLong) {
            int2* p = reinterpret_cast<int2*>(sg + at);
            int2 v = make_int2(__float2int_rn(d[0]), __float2int_rn(d[1]));
            if (piece0 > 0) {
              v.x += p->x;
              v.y += p->y;
            }
            *p = v;
          } else {
            *reinterpret_cast<float2*>(sg + at) = make_float2(d[0], d[1]);
          }
        };
        const int e = g8 * 8 + 2 * t;
        int m = 0;
#pragma unroll
        for (int p = 0; p < NB / 2; ++p) {
          const int at = C::pair_at(p) + e;
#pragma unroll
          for (int z = 2 * p; z < kFull; ++z, ++m) {
            if (z == 2 * p) {
              put(at, acc[c][m]);  // the other half is block (2p, 2p + 1) again
            } else {
              put(at + 64 + 128 * (z - 2 * p - 1), acc[c][m]);
              put(at + 128 + 128 * (z - 2 * p - 1), acc[c][m] + 2);
            }
          }
        }
        if constexpr (!kHalf && (NB & 1)) put(C::kG - 64 + e, acc[c][kAcc - 1] + 2 * (c & 1));
        if constexpr (kHalf) {
          if ((t >> 1) == (c & 1)) {  // this channel's four of the eight columns
            const int e4 = g8 * 4 + 2 * (t & 1);
            put(192 + e4, acc2[c / 2][0]);
            put(224 + e4, acc2[c / 2][0] + 2);
            if ((g8 >> 2) == (c & 1))
              put(256 + (g8 & 3) * 4 + 2 * (t & 1), acc2[c / 2][1] + ((c / 2) & 1 ? 2 : 0));
          }
        }
      };
      if constexpr (C::kLong) {
        static_loop<C::kCW>([&](auto c) {
          constexpr int e = decltype(c)::value;
          stage_out(c, s->g[warp][e]);
        });
        if (piece1 < stages) continue;  // more pieces of this sub-integration
      }
      const int off_s = lane < N ? C::off(lane, N) : 0, off_d = lane < N ? C::off(lane, lane) : 0;
      constexpr int kE = ((8 * NB) * (8 * NB + 1) / 2 + 31) / 32;  // entries per lane
#pragma unroll 1
      for (int c0 = 0; c0 < C::kCW; c0 += kMmEpi) {
        const int nu = min(kMmEpi, g.n_chan - (ch0 + c0));  // channels of the group that exist
        if (nu <= 0) break;
        __syncwarp();
        if constexpr (!C::kLong && NB <= 3) {
          // the same as stage_out for these blocks, written out: with stage_out here
          // too the kernels of up to 23 beams were 4 to 5 % slower
#pragma unroll
          for (int gr = 0; gr < C::kCW / kMmEpi; ++gr) {
            if (gr * kMmEpi != c0) continue;
#pragma unroll
            for (int u = 0; u < kMmEpi; ++u) {
              const int c = gr * kMmEpi + u;
              float* sg = reinterpret_cast<float*>(s->g[warp][u]);
              auto put = [&](int at, const float* d) {
                *reinterpret_cast<float2*>(sg + at) = make_float2(d[0], d[1]);
              };
              const int e = g8 * 8 + 2 * t;
              if constexpr (NB == 1) {
                put(e, acc[c][0] + 2 * (c & 1));
              } else {
                put(e, acc[c][0]);            // block 0 x 0
                put(64 + e, acc[c][1]);       // 0 x 1
                put(128 + e, acc[c][1] + 2);  // 1 x 1
                if constexpr (NB == 3 && !kHalf) {
                  put(192 + e, acc[c][2]);
                  put(256 + e, acc[c][2] + 2);
                  put(320 + e, acc[c][3] + 2 * (c & 1));
                }
                if constexpr (kHalf) {
                  if ((t >> 1) == (c & 1)) {  // this channel's four of the eight columns
                    const int e4 = g8 * 4 + 2 * (t & 1);
                    put(192 + e4, acc2[c / 2][0]);
                    put(224 + e4, acc2[c / 2][0] + 2);
                    if ((g8 >> 2) == (c & 1))
                      put(256 + (g8 & 3) * 4 + 2 * (t & 1), acc2[c / 2][1] + ((c / 2) & 1 ? 2 : 0));
                  }
                }
              }
            }
          }
        } else if constexpr (!C::kLong) {
          // registers cannot be indexed: the staging of each group is its own code
          static_loop<C::kCW / kMmEpi>([&](auto gr) {
            constexpr int e = decltype(gr)::value * kMmEpi;
            if (e == c0)
              static_loop<kMmEpi>([&](auto u) {
                constexpr int k = decltype(u)::value;
                stage_out(std::integral_constant<int, e + k>{}, s->g[warp][k]);
              });
          });
        }
        typename C::Sum(*sg)[C::kG] = s->g[warp] + (C::kLong ? c0 : 0);
        __syncwarp();
        auto beam = [&](int a, int off_s, int off_d) {
#pragma unroll
          for (int u = 0; u < kMmEpi; ++u) {
            const int32_t sa = (int)sg[u][off_s];
            const int64_t var = (int64_t)n * (int)sg[u][off_d] - (int64_t)sa * sa;
            float inv = 0.f;
            if (var > 0) {
              const float vf = cov_to_float<C::kLong>(var);
              inv = rsqrtf(vf);
              inv = inv * (1.5f - 0.5f * vf * inv * inv);
            } else if (g.corr && u < nu) {
              atomicAdd(g.degenerate, 1ull);
            }
            s->row[warp][u][a] = make_int2(sa, __float_as_int(inv));
          }
        };
        if constexpr (NB <= 3) {
          if (lane < N) beam(lane, off_s, off_d);
        } else {
          for (int a = lane; a < N; a += 32) beam(a, C::off(a, N), C::off(a, a));
        }
        __syncwarp();
        const int64_t cell = (int64_t)k * g.n_chan + ch0 + c0;
        if (g.corr) {
          const int np = N * (N + 1) / 2;
          float* dc = g.corr + cell * (int64_t)np + lane;
#pragma unroll(NB <= 3 ? kE : 2)
          for (int i = 0; i < kE; ++i) {
            if (32 * i >= P) break;
            if (lane + 32 * i < P) {
              const uint32_t l = s->lut[lane + 32 * i];
              const int a = (l >> 16) & 255, b = l >> 24;
              if (b < N) {
#pragma unroll
                for (int u = 0; u < kMmEpi; ++u) {
                  const int2 ra = s->row[warp][u][a], rb = s->row[warp][u][b];
                  const int64_t cov =
                      (int64_t)n * (int)sg[u][l & 0xffff] - (int64_t)ra.x * rb.x;
                  const float r = cov_to_float<C::kLong>(cov) * __int_as_float(ra.y) * __int_as_float(rb.y);
                  if (u < nu) dc[u * np + 32 * i - a] = a == b ? 1.f : r;
                }
              }
            }
          }
        }
        if (g.sums) {
          int64_t* ds = g.sums + cell * P + lane;
#pragma unroll 1
          for (int i = 0; lane + 32 * i < P; ++i) {
            const uint32_t l = s->lut[lane + 32 * i];
            const int a = (l >> 16) & 255, b = l >> 24;
#pragma unroll
            for (int u = 0; u < kMmEpi; ++u) {
              int64_t v = n;
              if (a < N) {
                v = (int64_t)(int)sg[u][l & 0xffff] +
                    128 * (int64_t)(b == N ? n : s->row[warp][u][a].x + s->row[warp][u][b].x);
                if (b < N) v += 16384 * n;
              }
              int64_t* o = ds + u * P + 32 * i;
              if (u < nu) *o = !C::kLong && piece0 > 0 ? *o + v : v;
            }
          }
        }
      }
    }
  }
  // After an expired wait the copies in flight land before the CTA exits:
  // each issuing lane waits for those of its stages it has not waited for.
  if constexpr (kTma) {
    if (!ok && lane == 0)
      for (int d = cnt; d <= last_issued; ++d)
        if ((d < D ? warp == 0 : d % C::kWarps == warp) && !(blockIdx.x == 0 && d == g.withhold))
          mbar_drain(&s->full[d % D], (uint32_t)((d / D) & 1), g.error, g.wait_ns);
  } else {
    asm volatile("cp.async.wait_all;" ::: "memory");
  }
}

template <class C>
cudaError_t launch_cfg(const mraid_plan_s* pl, MmArgs& a, bool tma) {
  CUtensorMap ma = {}, mb = {};
  const mraid_params& p = pl->p;
  if (tma) {
    cuuint64_t dims[3] = {(cuuint64_t)p.n_chan, (cuuint64_t)(a.sub0 + a.n_sub) * p.n_samp_sub,
                          (cuuint64_t)p.n_beam};
    cuuint64_t strides[2] = {(cuuint64_t)p.n_chan, (cuuint64_t)pl->beam_stride};
    cuuint32_t estr[3] = {1, 1, 1};
    auto encode = [&](CUtensorMap* m, int ch, CUtensorMapSwizzle swz) {
      cuuint32_t box[3] = {(cuuint32_t)ch, (cuuint32_t)kMmT, (cuuint32_t)p.n_beam};
      return encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint8_t*>(a.data), dims,
                         strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                         CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    };
    if (encode(&ma, C::kChA, C::kChA == 128  ? CU_TENSOR_MAP_SWIZZLE_128B
                           : C::kChA == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                           : C::kChA == 32 ? CU_TENSOR_MAP_SWIZZLE_32B
                                           : CU_TENSOR_MAP_SWIZZLE_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
    mb = ma;
    if (C::kChB > 0 && encode(&mb, C::kChB, CU_TENSOR_MAP_SWIZZLE_32B) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  const int64_t items = (int64_t)a.n_sub * ((p.n_chan + C::kCh - 1) / C::kCh);
  if (items < 1) return cudaSuccess;
  const int ctas = items > pl->sm_count ? C::kCtas : 1;
  const int64_t slots = (int64_t)pl->sm_count * ctas;
  const int grid = (int)(items < slots ? items : slots);
  a.depth = C::depth(a.n_beam, ctas);
  const size_t smem = C::kFixed + (size_t)a.depth * C::stage_bytes(a.n_beam);
  auto kern = tma ? gram_mma_kernel<C, true> : gram_mma_kernel<C, false>;
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<grid, C::kThreads, smem, pl->stream>>>(ma, mb, a);
  return cudaGetLastError();
}

// Bytes of a plain copy: 8 or 4 where every row of every beam allows it.
int copy_bytes(const mraid_plan_s* pl, const void* d_data) {
  const uint64_t align =
      (uint64_t)pl->p.n_chan | (uint64_t)pl->beam_stride | (uint64_t)(uintptr_t)d_data;
  return align % 8 == 0 ? 8 : (align % 4 == 0 ? 4 : 1);
}

// Time of a launch with work items of `width` channels, in arbitrary units:
// rounds of items over the SMs, each as long as its width over the rate of
// that width (percent of the 64-channel one).
int64_t item_cost(int n_sub, int n_chan, int sm_count, int width, int rate) {
  const int64_t items = (int64_t)n_sub * ((n_chan + width - 1) / width);
  return (items + sm_count - 1) / sm_count * width * 1000 / rate;
}

// Channels of a work item: the wider ones run more warps per SM (measured
// per sample, 64 channels = 100: 128 channels 137 for up to 15 beams, 96
// channels 113 for 16 to 19; 32 channels, half the warps, 55), the narrower
// ones leave less of the last round over the SMs empty. Sub-integrations of
// several pieces keep int32 sums of every channel in shared memory:
// 64-channel items for 16 beams and more, whose sums leave the ring of wider
// ones too shallow. From 24 beams on 32. Blocks of up to 16 channels and more
// sub-integrations than SMs take 16 (19 beams x 16 channels x 512 samples x 500
// 39 us, in 32-channel items 61).
int item_width(const mraid_plan_s* pl, int n_sub) {
  const mraid_params& p = pl->p;
  const bool lng = p.n_samp_sub > kMmPiece && p.n_samp_sub <= kMmLongMax;
  if (p.n_beam > 23) return 32;
  if (p.n_chan <= 16 && n_sub > pl->sm_count && !lng) return 16;
  auto cost = [&](int width, int rate) {
    return item_cost(n_sub, p.n_chan, pl->sm_count, width, rate);
  };
  const int64_t c32 = cost(32, 55), c64 = cost(64, 100);
  if (lng && p.n_beam <= 15) return c32 < cost(128, 137) ? 32 : 128;
  if (lng || p.n_beam > 19) return c32 < c64 ? 32 : 64;
  const int wide = p.n_beam <= 15 ? 128 : 96;
  const int64_t cw = p.n_beam <= 15 ? cost(128, 137) : cost(96, 113);
  return c32 < c64 && c32 < cw ? 32 : (cw <= c64 ? wide : 64);
}

// Microseconds of a call here and on dp4a, from 2 066 timed pairs (2 to 39
// beams, 1 to 4 096 channels, 8 to 65 536 samples, 1 to 20 000
// sub-integrations, copies of every kind; within 15 % for most). A stage of 16
// samples takes an item its time whatever its channels, so a block of few
// channels pays for 32; dp4a's small blocks share an SM and take the channels
// there are. At a few blocks per SM it is bound by a chunk's latency. (Its
// correlation is a second launch, 3 us.) By these figures the slower route is
// taken in 21 of the pairs by more than 20 %, at the worst by 42 %.
double mma_us(const mraid_plan_s* pl, const void* d_data) {
  const mraid_params& p = pl->p;
  const int N = p.n_beam, width = item_width(pl, p.n_sub);
  const int64_t items = (int64_t)p.n_sub * ((p.n_chan + width - 1) / width);
  const int ctas = width > 32 || N > 23 || items <= pl->sm_count ? 1
                   : (N <= 7 ? 3 : 2) * (width == 16 ? 2 : 1);
  const int64_t slots = (int64_t)pl->sm_count * ctas;
  const int kind = copy_bytes(pl, d_data);
  double stage = N <= 7 ? 0.31 : N <= 15 ? 0.40 : N <= 31 ? 0.51 : 0.69;
  const bool tail = kind == 1 && p.n_chan % 4 != 0 && p.n_chan <= 32;  // single bytes in every row
  if (tail) stage = N <= 23 ? 1.1 + 0.13 * N : 1.0 + 0.11 * N;
  else if (kind == 1) stage = (0.7 + 0.05 * N) * (width == 64 || width == 96 ? 1.4 : 1.0);
  else if (!gram_mma_bulk(pl, d_data)) stage += 0.33 + (kind == 8 ? 0.007 : 0.012) * N;
  stage *= width == 32 ? (ctas > 1 ? 1.17 : 1.0) : (width == 64 ? 1.15 : 1.4);
  const double epilogue = (N <= 7 ? 1.0 : N <= 15 ? 2.3 : N <= 23 ? 3.5 : N <= 31 ? 5.0 : 9.0) *
                          width / 32 * (width > 32 ? 0.75 : 1.0);
  const int stages = (p.n_samp_sub + kMmT - 1) / kMmT;
  return 6.0 + (double)((items + slots - 1) / slots) * (stage * stages + epilogue * ctas);
}
double dp4a_us(const mraid_plan_s* pl, const void* d_data) {
  const mraid_params& p = pl->p;
  int cpb, tiles;
  gram_u8_shape(p.n_beam, p.n_chan, &cpb, &tiles);
  const int tasks = cpb * tiles;
  const double bytes = cpb % 4 == 0 && copy_bytes(pl, d_data) >= 4 ? 0.0 : p.n_beam * cpb;  // loaded singly
  const double per_sm = (double)p.n_sub * ((p.n_chan + cpb - 1) / cpb) / pl->sm_count;
  const double latency = 0.8 + 0.0045 * tasks + 0.025 * bytes;
  const double issue = per_sm * (0.2 + (p.n_beam < 32 ? 0.006 : 0.0045) * tasks + 0.016 * bytes);
  const double chunks = (p.n_samp_sub + 31) / 32 * (bytes > 0 && p.n_samp_sub > 2048 ? 1.3 : 1.0);
  return 9.0 + chunks * (latency > issue ? latency : issue) + per_sm * (0.2 + cpb * (0.03 + 0.0008 * pl->psum));
}

}  // namespace

// Bulk tensor copies take rows of whole 16-byte channel groups; other
// layouts go by plain copies.
bool gram_mma_bulk(const mraid_plan_s* pl, const void* d_data) {
  const mraid_params& p = pl->p;
  return p.n_chan % 16 == 0 && pl->beam_stride % 16 == 0 &&
         (reinterpret_cast<uintptr_t>(d_data) & 15) == 0 &&
         (int64_t)p.n_sub * p.n_samp_sub <= 2147483647ll /* TMA time coordinate */ &&
         encode_fn() != nullptr;
}

// Narrow blocks, and few beams by plain copies, are faster on dp4a where there
// are enough of them (measured, dp4a against here): 19 beams x 1 channel x
// 1024 samples x 2 000 193 us against 505, 7 x 4 x 1024 x 1 000 65 against 127,
// 13 x 8 x 1024 x 38 40 against 58, 7 beams x 40 channels x 512 x 200 42
// against 58; but 19 x 16 x 1024 x 250 92 against 50, 19 x 17 x 1024 x 250 454
// against 237, and from 32 channels on, by bulk copies, never. By the plan's
// shape, so that ranges of one plan take one route.
bool gram_mma_takes(const mraid_plan_s* pl, const void* d_data) {
  if (!gram_mma_supported(pl)) return false;
  if (pl->p.n_chan > 16 && gram_mma_bulk(pl, d_data)) return true;
  return mma_us(pl, d_data) <= dp4a_us(pl, d_data);
}

bool gram_mma_has_forms(const mraid_plan_s* pl) {
  const mraid_params& p = pl->p;
  return p.n_beam <= 23 && (p.n_samp_sub <= kMmPiece || p.n_samp_sub > kMmLongMax) &&
         item_width(pl, p.n_sub) != 64;
}

bool gram_mma_supported(const mraid_plan_s* pl) {
  return pl->p.bit_depth == 8 && pl->p.n_beam >= 2 && pl->p.n_beam <= 39;
}

cudaError_t launch_gram_mma(const mraid_plan_s* pl, const uint8_t* d_data, int sub0, int n_sub,
                            int64_t* d_sums, float* d_corr) {
  const mraid_params& p = pl->p;
  if (!gram_mma_supported(pl) || (d_corr && p.n_samp_sub > kMmLongMax)) return cudaErrorNotSupported;
  MmArgs a;
  a.data = d_data;
  a.beam_stride = pl->beam_stride;
  a.vec = copy_bytes(pl, d_data);
  a.data_end = d_data + (int64_t)(p.n_beam - 1) * pl->beam_stride +
               (int64_t)(sub0 + n_sub) * p.n_samp_sub * p.n_chan;
  a.n_beam = p.n_beam;
  a.n_chan = p.n_chan;
  a.n_samp_sub = p.n_samp_sub;
  a.sub0 = sub0;
  a.n_sub = n_sub;
  a.sums = d_sums;
  a.corr = d_corr;
  a.degenerate = pl->d_degenerate;
  a.error = pl->d_error;
  a.wait_ns = pl->wait_ns;
  a.withhold = pl->inject_withhold;
  const bool tma = gram_mma_bulk(pl, d_data);
  const bool lng = p.n_samp_sub > kMmPiece && p.n_samp_sub <= kMmLongMax;
  const int pick = pl->tc_variant == 1 && !lng ? 64 : item_width(pl, n_sub);
  if (lng) {
    if (p.n_beam <= 7)
      return pick == 32 ? launch_cfg<MmCfg<1, false, 32, 0, 8, true>>(pl, a, tma)
                        : launch_cfg<MmCfg<1, false, 128, 0, 8, true>>(pl, a, tma);
    if (p.n_beam <= 15)
      return pick == 32 ? launch_cfg<MmCfg<2, false, 32, 0, 8, true>>(pl, a, tma)
                        : launch_cfg<MmCfg<2, false, 128, 0, 8, true>>(pl, a, tma);
    if (p.n_beam <= 19)
      return pick == 32 ? launch_cfg<MmCfg<3, true, 32, 0, 8, true>>(pl, a, tma)
                        : launch_cfg<MmCfg<3, true, 64, 0, 8, true>>(pl, a, tma);
    if (p.n_beam <= 23)
      return pick == 32 ? launch_cfg<MmCfg<3, false, 32, 0, 8, true>>(pl, a, tma)
                        : launch_cfg<MmCfg<3, false, 64, 0, 8, true>>(pl, a, tma);
    if (p.n_beam <= 31) return launch_cfg<MmCfg<4, false, 32, 0, 4, true>>(pl, a, tma);
    return launch_cfg<MmCfg<5, false, 32, 0, 4, true>>(pl, a, tma);
  }
  if (p.n_beam > 31) return launch_cfg<MmCfg<5, false, 32, 0, 4>>(pl, a, tma);
  if (p.n_beam > 23) return launch_cfg<MmCfg<4, false, 32, 0, 4>>(pl, a, tma);
  if (p.n_beam <= 7)
    return pick == 16   ? launch_cfg<MmCfg<1, false, 16, 0>>(pl, a, tma)
           : pick == 32 ? launch_cfg<MmCfg<1, false, 32, 0>>(pl, a, tma)
           : pick == 64 ? launch_cfg<MmCfg<1, false, 64, 0>>(pl, a, tma)
                        : launch_cfg<MmCfg<1, false, 128, 0>>(pl, a, tma);
  if (p.n_beam <= 15)
    return pick == 16   ? launch_cfg<MmCfg<2, false, 16, 0>>(pl, a, tma)
           : pick == 32 ? launch_cfg<MmCfg<2, false, 32, 0>>(pl, a, tma)
           : pick == 64 ? launch_cfg<MmCfg<2, false, 64, 0>>(pl, a, tma)
                        : launch_cfg<MmCfg<2, false, 128, 0>>(pl, a, tma);
  if (p.n_beam <= 19)
    return pick == 16   ? launch_cfg<MmCfg<3, true, 16, 0>>(pl, a, tma)
           : pick == 32 ? launch_cfg<MmCfg<3, true, 32, 0>>(pl, a, tma)
           : pick == 64 ? launch_cfg<MmCfg<3, true, 64, 0>>(pl, a, tma)
                        : launch_cfg<MmCfg<3, true, 64, 32>>(pl, a, tma);
  return pick == 16   ? launch_cfg<MmCfg<3, false, 16, 0>>(pl, a, tma)
         : pick == 32 ? launch_cfg<MmCfg<3, false, 32, 0>>(pl, a, tma)
                      : launch_cfg<MmCfg<3, false, 64, 0>>(pl, a, tma);
}

}  // namespace mraid
