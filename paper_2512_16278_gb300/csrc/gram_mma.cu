// gram_mma.cu - exact augmented Gram sums of 8-bit multi-beam data for 2..23
// beams, fused with the correlation.
//
// Section 3.2, Eq. 1. For a cell (channel j, sub-integration k) with samples
// x_b(t), the kernel forms G = Y Y^T with Y = [x - 128; 1]. The centred
// values are exact in f16, products are integers of magnitude <= 2^14 and
// sums over <= 1024 samples are integers of magnitude <= 2^24, so FP32
// accumulation is exact; longer sub-integrations are flushed as int64 every
// 1024 samples. cov_ab = n G_ab - G_a G_b is exact in int64 and
// r_ab = cov_ab / sqrt(var_a var_b) is rounded to float once. The raw sums
// are S_ab = G_ab + 128 (G_a + G_b) + 128^2 n and S_a = G_a + 128 n.
//
// Why register fragments (mma.sync) and not tcgen05: a cell's Gram is 24 x 24
// at most, and the samples lie channel by channel in memory. A 128-row
// tcgen05 tile of 16 beams x 8 channels keeps 1/8 of its products, and its
// operands cross shared memory 5 times as f16; that kernel was bound by
// shared memory at 3.4 TB/s of samples. Here a warp owns 8 channels and every
// product is of one channel: a lane reads 8 bytes (8 channels) of one beam
// and one sample, a pair of samples becomes an f16x2 register by byte
// permutes (x in the low mantissa bits of 1024, minus 1152), and that
// register is at once an A and a B fragment of its channel's Gram, because
// the order of the samples within K is free. Products per channel and 16
// samples: block rows (0, 1) x every block column, and the last block of an
// odd count by itself.
//
// Layout: a work item is one sub-integration x 32, 64, 96 or 128 channels
// (4, 8, 12 or 16 warps, as many as the accumulators leave registers for);
// stages of 16 samples x all beams come by TMA with a swizzle under which a
// warp's 8-byte loads meet two-way conflicts at most, into a ring as deep as
// shared memory allows; the warps take turns to issue the copies. Rows of 64
// bytes and more on their own multiples matter: 16- and 32-byte rows stream
// at 4.7-4.8 TB/s on GB300, 64-byte ones at 6.3-6.7, 128-byte ones at 7.1.
// Layouts that no tensor map takes (odd channel counts, misaligned buffers)
// fill the same ring by cp.async or byte loads.
//
// Measured on GB300 (50 sub-integrations x 4096 channels x 1024 samples):
// 19 beams 0.89 ms (4.5 TB/s of samples; the tcgen05 kernel 1.20 ms), 13
// beams 0.54 ms (0.91), 7 beams 0.35 ms (0.84); with 128 samples per
// sub-integration, where the epilogue weighs most, 1.70, 0.98 and 0.63 ms
// (6.27, 4.64 and 4.21). 1000 channels x 1000 samples x 40 (no tensor map)
// 0.38 ms, on dp4a 0.62 ms. Without its copies the 19-beam kernel takes 0.75
// ms, without its products 0.8: bound by both, the permutes' and MMAs' issue
// at 3 warps per scheduler and the copies that pause in the epilogue.
//
// Every wait is bounded by the plan's limit; on expiry the kernel records an
// error word, waits (again bounded) for its copies in flight and returns.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "internal.h"
#include "tc_ptx.h"

namespace mraid {
namespace {

constexpr int kCW = 8;                       // channels per warp
constexpr int kMmLag = 1;  // stages between a slot's last read and its refill
constexpr int kMmT = 16;                     // samples per stage: one K step
constexpr int kMmMaxD = 12;                  // ring depth bound
constexpr int kMmPiece = 1024;               // samples accumulated before a flush
constexpr size_t kMmSmem = 226 * 1024;
constexpr int kMmEpi = 2;                    // channels staged at a time by the epilogue

// NB 8-beam blocks; kHalf: the last one holds at most four slots, and its
// fragment carries them for two channels (lanes of rows 0..3 the even one,
// 4..7 the odd one); A_, B_: channels of a stage's two boxes (B_ 0: one box).
template <int NB_, bool kHalf_, int A_, int B_>
struct MmCfg {
  static constexpr int NB = NB_, kChA = A_, kChB = B_, kCh = A_ + B_;
  static constexpr bool kHalf = kHalf_;
  static constexpr int kWarps = kCh / kCW, kThreads = 32 * kWarps;
  static constexpr int kTile = kMmT * kCh;  // bytes of one beam in a stage
  // floats of one channel's products in the epilogue
  static constexpr int kG = NB == 1 ? 64 : (NB == 2 ? 192 : (kHalf ? 272 : 384));
  struct Shared {
    uint64_t full[kMmMaxD], empty[kMmMaxD];
    uint32_t lut[(8 * NB) * (8 * NB + 1) / 2];  // G offset | a << 16 | b << 24
    alignas(16) float g[kWarps][kMmEpi][kG];
    int2 row[kWarps][kMmEpi][8 * NB];  // per beam: sum of the centred samples, 1/sqrt(var)
  };
  // Where the pair (a, b), a <= b, lies in a channel's products.
  __host__ __device__ static constexpr int off(int a, int b) {
    const int ba = a >> 3, bb = b >> 3, e = (a & 7) * 8 + (b & 7);
    if (bb == 0) return e;
    if (bb == 1) return 64 + a * 8 + (b & 7);
    if (kHalf) return ba < 2 ? 192 + a * 4 + (b & 7) : 256 + (a & 7) * 4 + (b & 7);
    return ba < 2 ? 192 + a * 8 + (b & 7) : 320 + e;
  }
  static constexpr size_t kFixed = 1024 + sizeof(Shared);
  static constexpr int stage_bytes(int n_beam) { return (n_beam + 2) * kTile; }
  static constexpr int depth(int n_beam) {
    const int d = (int)((kMmSmem - kFixed) / (size_t)stage_bytes(n_beam));
    return d < kMmMaxD ? d : kMmMaxD;
  }
};

struct MmArgs {
  const uint8_t* data;  // plain copies: the samples, beams beam_stride apart
  int64_t beam_stride;
  int vec;  // plain copies: bytes per copy (8 or 4: cp.async; 1: byte loads)
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

__device__ __forceinline__ uint32_t f16_sub(uint32_t x, uint32_t y) {
  uint32_t r;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(y));
  return r;
}

template <int kImm>
__device__ __forceinline__ uint2 lds64(uint32_t addr) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2+%3];" : "=r"(v.x), "=r"(v.y) : "r"(addr), "n"(kImm));
  return v;
}
// A lane constant that the compiler keeps instead of computing it again.
__device__ __forceinline__ void pin(uint32_t& x) { asm volatile("" : "+r"(x)); }

// The XOR that a tensor map's swizzle of `pitch` bytes applies to the 16-byte
// column of row r (rows `pitch` bytes apart).
__device__ __forceinline__ int swizzle(int pitch, int r) {
  return pitch == 128 ? r & 7 : (pitch == 64 ? (r >> 1) & 3 : (r >> 2) & 1);
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
__global__ void __launch_bounds__(C::kThreads, 1)
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
  // takes; a thread fills one place of every beam (or of every other one)
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
      for (int b = threadIdx.x / (words * kMmT); b < N; b += 2)
        if (mine) copy_async<8>(dst + b * kMmT * pitch, src + b * g.beam_stride);
    } else if (v == 4) {
      for (int b = 0; b < N; ++b)
        if (mine) copy_async<4>(dst + b * kMmT * pitch, src + b * g.beam_stride);
    } else if (mine) {
      const int nc = min(4, g.n_chan - ch);
#pragma unroll 4
      for (int b = 0; b < N; ++b) {
        const uint8_t* p = src + b * g.beam_stride;
        uint32_t x = p[0];
        if (nc > 1) x |= (uint32_t)p[1] << 8;
        if (nc > 2) x |= (uint32_t)p[2] << 16;
        if (nc > 3) x |= (uint32_t)p[3] << 24;
        asm volatile("st.shared.u32 [%0], %1;" ::"r"(dst + b * kMmT * pitch), "r"(x) : "memory");
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
      last_issued = D - 1;
    }
  } else {
    for (int i = 0; i < D && i < total; ++i) fill(i);
  }

  // ---- this lane's places: beam row g8 of each 8-beam block, times t of
  // every 4; odd beams read the two halves of an 8-sample group in the
  // opposite order (their pairs are put back by the permute selectors)
  const int g8 = lane >> 2, t = lane & 3, odd = g8 & 1;
  const bool in_a = warp < C::kChA / kCW;
  const int pitch = in_a ? C::kChA : C::kChB;                       // bytes per row
  const int wc = in_a ? warp >> 1 : (warp - C::kChA / kCW) >> 1;   // 16-byte column
  auto place = [&](int r) {  // this warp's 8 bytes of row r, swizzled
    return r * pitch + ((wc ^ swizzle(pitch, r)) << 4) + ((warp & 1) << 3);
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

  constexpr int kAcc = kHalf || NB == 2 ? 2 : (NB == 1 ? 1 : 4);  // per channel
  constexpr int kFull = kHalf ? NB - 1 : NB;

  int slot = 0;
  uint32_t ph = 0;
  int cnt = 0;
  uint32_t fill_ph = 0;  // parity of the slot's read that a plain refill waits for
  int duty = warp;       // this warp's next stage to issue: d % C::kWarps == warp, d >= D
  while (duty < D) duty += C::kWarps;
  bool ok = true;
  for (int it = blockIdx.x; it < items && ok; it += gridDim.x) {
    const int k = it / chunks, ch0 = it % chunks * C::kCh + kCW * warp;
    for (int piece0 = 0; piece0 < stages && ok; piece0 += kMmPiece / kMmT) {
      const int piece1 = min(stages, piece0 + kMmPiece / kMmT);
      float acc[kCW][kAcc][4];
      float acc2[kHalf ? kCW / 2 : 1][2][4];  // of two channels: blocks (0, 1) x last, last x last
#pragma unroll
      for (int c = 0; c < kCW; ++c)
#pragma unroll
        for (int m = 0; m < kAcc; ++m)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[c][m][i] = 0.f;
#pragma unroll
      for (int c = 0; c < (kHalf ? kCW / 2 : 1); ++c)
#pragma unroll
        for (int i = 0; i < 8; ++i) acc2[c][i / 4][i % 4] = 0.f;
      auto run = [&](auto pitch_c) {
        constexpr int kPitch = decltype(pitch_c)::value;
        for (int st = piece0; st < piece1; ++st) {
          ok = mbar_wait(&s->full[slot], ph, g.error, g.wait_ns);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          unsigned char* stage = ring + slot * stage_bytes;
          const int nv = g.n_samp_sub - st * kMmT;
          if (nv < kMmT) {  // samples of the next sub-integration: the centre value
            for (int i = lane; i < (kMmT - nv) * N; i += 32) {
              const int r = nv + i / N, b = i % N;
              *reinterpret_cast<uint2*>(stage + tile0 + b * kMmT * kPitch + place(r)) =
                  make_uint2(0x80808080u, 0x80808080u);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
          }
          uint2 w[NB][2][2];
          {
            const uint32_t so = (uint32_t)(slot * stage_bytes);
#pragma unroll
            for (int b = 0; b < NB; ++b) {
              const uint32_t p0 = b == NB - 1 ? L0 + so : A0 + so;
              const uint32_t p1 = b == NB - 1 ? L1 + so : A1 + so;
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                constexpr int kBlk = 8 * kMmT * kPitch;
                if (b == 0 || b == NB - 1) {
                  w[b][h][0] = h ? lds64<8 * kPitch>(p0) : lds64<0>(p0);
                  w[b][h][1] = h ? lds64<8 * kPitch>(p1) : lds64<0>(p1);
                } else {
                  w[b][h][0] = h ? lds64<kBlk + 8 * kPitch>(p0) : lds64<kBlk>(p0);
                  w[b][h][1] = h ? lds64<kBlk + 8 * kPitch>(p1) : lds64<kBlk>(p1);
                }
              }
            }
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
          for (int q = 0; q < kCW / 4; ++q) {
            // f: blocks 0.., f2: the half block, of two channels
            uint32_t f[4][kFull][2], f2[2][2];
#pragma unroll
            for (int b = 0; b < NB; ++b)
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const uint32_t x = q ? w[b][h][0].y : w[b][h][0].x;
                const uint32_t y = q ? w[b][h][1].y : w[b][h][1].x;
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
              if constexpr (NB >= 2) {
#pragma unroll
                for (int z = 0; z < kFull; ++z)
                  mma16816(d[z], f[c][0][0], f[c][1][0], f[c][0][1], f[c][1][1], f[c][z][0],
                           f[c][z][1]);
              }
              if constexpr (kHalf) {
                // the other channel's columns are zero here, so both add into one tile
                const uint32_t mk = c & 1 ? ~mask_even : mask_even;
                mma16816(acc2[2 * q + c / 2][0], f[c][0][0], f[c][1][0], f[c][0][1],
                         f[c][1][1], f2[c / 2][0] & mk, f2[c / 2][1] & mk);
              } else if constexpr (NB != 2) {
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
      const int n = min(g.n_samp_sub - piece0 * kMmT, kMmPiece);
      constexpr int kE = ((8 * NB) * (8 * NB + 1) / 2 + 31) / 32;  // entries per lane
      const int off_s = lane < N ? C::off(lane, N) : 0;
      const int off_d = lane < N ? C::off(lane, lane) : 0;
#pragma unroll 1
      for (int c0 = 0; c0 < kCW; c0 += kMmEpi) {
        const int nu = min(kMmEpi, g.n_chan - (ch0 + c0));  // channels of the group that exist
        if (nu <= 0) break;
        __syncwarp();
        // registers cannot be indexed: the staging of each group is its own code
#pragma unroll
        for (int gr = 0; gr < kCW / kMmEpi; ++gr) {
          if (gr * kMmEpi != c0) continue;
#pragma unroll
          for (int u = 0; u < kMmEpi; ++u) {
            const int c = gr * kMmEpi + u;
            float* sg = s->g[warp][u];
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
        __syncwarp();
        if (lane < N) {
#pragma unroll
          for (int u = 0; u < kMmEpi; ++u) {
            const int32_t sa = (int)s->g[warp][u][off_s];
            const int64_t var = (int64_t)n * (int)s->g[warp][u][off_d] - (int64_t)sa * sa;
            float inv = 0.f;
            if (var > 0) {
              const float vf = i64_to_float(var);
              inv = rsqrtf(vf);
              inv = inv * (1.5f - 0.5f * vf * inv * inv);
            } else if (g.corr && u < nu) {
              atomicAdd(g.degenerate, 1ull);
            }
            s->row[warp][u][lane] = make_int2(sa, __float_as_int(inv));
          }
        }
        __syncwarp();
        const int64_t cell = (int64_t)k * g.n_chan + ch0 + c0;
        if (g.corr) {
          const int np = N * (N + 1) / 2;
          float* dc = g.corr + cell * (int64_t)np + lane;
#pragma unroll
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
                      (int64_t)n * (int)s->g[warp][u][l & 0xffff] - (int64_t)ra.x * rb.x;
                  const float r = i64_to_float(cov) * __int_as_float(ra.y) * __int_as_float(rb.y);
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
                v = (int64_t)(int)s->g[warp][u][l & 0xffff] +
                    128 * (int64_t)(b == N ? n : s->row[warp][u][a].x + s->row[warp][u][b].x);
                if (b < N) v += 16384 * n;
              }
              int64_t* o = ds + u * P + 32 * i;
              if (u < nu) *o = piece0 > 0 ? *o + v : v;
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
                                           : CU_TENSOR_MAP_SWIZZLE_32B) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
    mb = ma;
    if (C::kChB > 0 && encode(&mb, C::kChB, CU_TENSOR_MAP_SWIZZLE_32B) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  const int64_t items = (int64_t)a.n_sub * ((p.n_chan + C::kCh - 1) / C::kCh);
  if (items < 1) return cudaSuccess;
  const int grid = (int)(items < pl->sm_count ? items : pl->sm_count);
  a.depth = C::depth(a.n_beam);
  const size_t smem = C::kFixed + (size_t)a.depth * C::stage_bytes(a.n_beam);
  auto kern = tma ? gram_mma_kernel<C, true> : gram_mma_kernel<C, false>;
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<grid, C::kThreads, smem, pl->stream>>>(ma, mb, a);
  return cudaGetLastError();
}

// Time of a launch with work items of `width` channels, in arbitrary units:
// rounds of items over the SMs, each as long as its width over the rate of
// that width (percent of the 64-channel one).
int64_t item_cost(const MmArgs& a, int sm_count, int width, int rate) {
  const int64_t items = (int64_t)a.n_sub * ((a.n_chan + width - 1) / width);
  return (items + sm_count - 1) / sm_count * width * 1000 / rate;
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

bool gram_mma_supported(const mraid_plan_s* pl) {
  return pl->p.bit_depth == 8 && pl->p.n_beam >= 2 && pl->p.n_beam <= 23;
}

cudaError_t launch_gram_mma(const mraid_plan_s* pl, const uint8_t* d_data, int sub0, int n_sub,
                            int64_t* d_sums, float* d_corr) {
  const mraid_params& p = pl->p;
  if (!gram_mma_supported(pl) || (d_corr && p.n_samp_sub > kMmPiece)) return cudaErrorNotSupported;
  MmArgs a;
  a.data = d_data;
  a.beam_stride = pl->beam_stride;
  const uint64_t align = (uint64_t)p.n_chan | (uint64_t)pl->beam_stride | (uint64_t)(uintptr_t)d_data;
  a.vec = align % 8 == 0 ? 8 : (align % 4 == 0 ? 4 : 1);
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
  // The width of a work item: the wider ones run more warps per SM (measured
  // per sample, 64 channels = 100: 128 channels 137 for up to 15 beams, 96
  // channels 113 for 16 to 19; 32 channels, half the warps, 55), the
  // narrower ones leave less of the last round over the SMs empty.
  const bool narrow = pl->tc_variant & 1;
  const int64_t c64 = item_cost(a, pl->sm_count, 64, 100);
  const int64_t c32 = item_cost(a, pl->sm_count, 32, 55);
  const int64_t cw = p.n_beam <= 15   ? item_cost(a, pl->sm_count, 128, 137)
                     : p.n_beam <= 19 ? item_cost(a, pl->sm_count, 96, 113)
                                      : INT64_MAX;
  const int pick = narrow ? 64 : (c32 < c64 && c32 < cw ? 32 : (cw <= c64 ? 128 : 64));
  if (p.n_beam <= 7)
    return pick == 32   ? launch_cfg<MmCfg<1, false, 32, 0>>(pl, a, tma)
           : pick == 64 ? launch_cfg<MmCfg<1, false, 64, 0>>(pl, a, tma)
                        : launch_cfg<MmCfg<1, false, 128, 0>>(pl, a, tma);
  if (p.n_beam <= 15)
    return pick == 32   ? launch_cfg<MmCfg<2, false, 32, 0>>(pl, a, tma)
           : pick == 64 ? launch_cfg<MmCfg<2, false, 64, 0>>(pl, a, tma)
                        : launch_cfg<MmCfg<2, false, 128, 0>>(pl, a, tma);
  if (p.n_beam <= 19)
    return pick == 32   ? launch_cfg<MmCfg<3, true, 32, 0>>(pl, a, tma)
           : pick == 64 ? launch_cfg<MmCfg<3, true, 64, 0>>(pl, a, tma)
                        : launch_cfg<MmCfg<3, true, 64, 32>>(pl, a, tma);
  return pick == 32 ? launch_cfg<MmCfg<3, false, 32, 0>>(pl, a, tma)
                    : launch_cfg<MmCfg<3, false, 64, 0>>(pl, a, tma);
}

}  // namespace mraid
