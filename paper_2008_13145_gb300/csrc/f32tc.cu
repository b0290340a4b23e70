// FP32 GEMM on the fifth-generation tensor cores, at FP32 accuracy.
//
// Every FP32 operand element is split on its way into shared memory into three
// BF16 parts that add up to it exactly (x = p0 + p1 + p2: 24 significand bits
// in three roundings to 8), and the six products of parts whose indexes sum to
// at most 2 are accumulated; the three left out add up to at most 2^-23 |xy|.  The
// tensor core truncates each addition into its accumulator, so a K chunk of 32
// is all that one accumulator sums: the small products first, then the two
// steps of p0 q0.  The chunk sums are then added in FP32, rounded to nearest,
// in registers.  Relative error against 64 bits at 4096 x 4096 x 4096, uniform
// [-1, 1): 2.1e-7 (a chain of FP32 FMAs over K: 1.15e-6); f32tc_plan uses the
// kernel only where it is the more exact of the two on dense operands.  Where a
// row has fewer than about 24 non-zero terms an FMA chain, which rounds once a
// term, is the more exact: a diagonal times a matrix has 0.77 2^-24 of rms error a
// result (at most 2.6) against 0.42 (1.0), 8 terms 0.55 against 0.42, 32 terms 0.39
// against 0.41.  Products by 0, by powers of two and of integers are exact.
//
// Bound: six 16-bit products, 315 TFLOP/s of the measured BF16 rate; the FP32
// pipe's peak is 80.  4096 x 4096 x 4096: 572 us, 240 TFLOP/s (A B^T 547; up to 10 %
// more once the clocks fall under the power cap; the last of four rounds of 256 x
// 256 tiles is a third full: 4864 x 4096 x 4096 takes as long, 285 TFLOP/s) against
// 2,525 us for the SIMT kernel.  What holds it is the converting
// warps' chain of latencies (load, split, store, fence per chunk), then
// shared-memory bandwidth: the MMAs of 128-wide tiles alone read 128 bytes a clock.
//
// A split that is not exact (infinities, NaN, magnitudes whose low bits fall
// below BF16's range, values that round past the largest BF16) is seen while
// converting -- the third remainder then has bits below BF16's 16 -- and an
// accumulator that overflowed is seen when it is read.  A reading warp leaves
// its part of such a tile unwritten and marks it; when all of the CTA's chunks
// are summed, so that no role waits, the reading warps compute the marked parts
// by plain FP32 FMAs over K (redo), so such inputs give what the FP32 SIMT family
// gives.  One NaN takes 2048 x 2048 x 2048 from 83 to 564 us (SIMT kernel: 365, on
// any values), an infinity in every row of 4096 x 4096 x 4096 from 578 to 4,400
// (SIMT: 2,525): the parts of a tile stay with its SM.  (Computed where they were
// met, by lanes with a row each: 11,640 and 101,000 us.)
//
// One persistent CTA per SM, five warpgroups.
//   8..15  : two groups that convert alternate chunks.  A thread loads its part
//            of the next chunk of its group (any alignment, either storage order)
//            as soon as it has stored the part before, so its loads have two
//            chunks' time to arrive.  They take the registers that 16..19 give up;
//   0..7   : read each chunk's accumulator from TMEM (two take turns), add it to
//            their part of the tile and write C;
//   16     : issues the MMAs.  It does nothing else: the tensor core accepts few
//            of them ahead, so the issuing thread waits for most of their time.
// Converting inside the kernel rather than in a pre-pass reads each operand
// slice from L2 once as 4-byte elements (a pre-pass writes 6 bytes an element
// to memory and every tile reads those back).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace ks {
namespace f32tc {

using namespace tc;

constexpr int kReaders = 8;     // accumulator-reading warps
constexpr int kGroups = 2;      // converting groups of four warps
constexpr int kIssuer = kReaders + 4 * kGroups;  // the MMA-issuing warp
constexpr int kThreads = 32 * (kIssuer + 4);
// Registers a thread as launched; the warpgroups then share out their sum, 640 x 96.
constexpr int kRegsLaunch = 96, kRegsIssue = 32;
constexpr int kBM = 128;
constexpr int kBK = 32;                       // K elements per chunk: one 64-byte BF16 row per part
constexpr int kParts = 3;
constexpr int kStoreBytes = 2048;             // staging of a reading warp's stores
constexpr int kMarks = 16;                    // more than the chunks under way at once
constexpr int kMaxItems = 1024;               // items of one CTA or pair: a byte each of `lost`

// Stages: what fits in 164 KB, so that 92 KB are left as L1, where the FP32
// loads under way land (with 28 KB left, the 256 x 256 tiles of 4096 x 4096 x
// 4096 took 27 % longer).
template <int BN>
struct Cfg {
  static constexpr int A_PART = kBM * 64;  // bytes of one part of a slice
  static constexpr int B_PART = BN * 64;
  static constexpr int STAGE = kParts * (A_PART + B_PART);
  static constexpr int STAGES = BN == 128 ? 3 : 4;
  static constexpr int SMEM = STAGES * STAGE + kReaders * kStoreBytes + 1024;
  static constexpr int TMEM = 2 * BN;  // two accumulators
  static constexpr int G = BN / 8;     // accumulator columns per reading warp and quarter
  // 128 x 32 + 256 x (112 + 112) or 256 x (128 + 96): at BN 128 a reading thread
  // holds 64 accumulators (with 96 registers it spills: a third slower at 4096 x
  // 4096 x 4096, A B^T), at BN 64 the converting ones gain more.
  static constexpr int REGS_CONVERT = BN == 128 ? 112 : 128, REGS_READ = BN == 128 ? 112 : 96;
};

struct Args {
  GemmArgs g;
  int tiles_m, tiles_n, tiles;  // tiles: all batch entries
  int splits, kchunk, items;    // items = tiles * splits
  int group_m;
  int vec8;  // C takes 32-byte stores
  int* status;
  // 3 x 3 convolution (kConv): A is the NHWC image; bias and ReLU go with the stores.
  int H, W, Ch;
  const float* bias;  // N values or null
  int relu;
};

// How A reaches the kernel: stored with K contiguous, with M contiguous, or as
// the image that its rows are the 3 x 3 neighbourhoods of.
enum : int { kRows = 0, kCols = 1, kConv = 2 };

// Tile row (or column) r of an R-wide operand slice sits in shared-memory row
// (r % 4) * (R / 4) + r / 4.  A thread that loads four consecutive elements
// along M or N (operands stored MN-contiguous) then stores to rows a quarter
// apart while its neighbours store to neighbouring rows, free of bank
// conflicts; and the accumulator columns q, q + BN/4, q + BN/2, q + 3BN/4 are
// four consecutive columns of C in one thread.

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}

// Both elements' three parts; the third remainder's bits are collected in
// `rem`: its low 16 bits are zero exactly when the split is exact.
__device__ __forceinline__ void split2(float a, float b, uint32_t (&p)[kParts], uint32_t& rem) {
  const float2 minus = make_float2(-1.f, -1.f);
  p[0] = pack_bf16(a, b);
  float2 r = __ffma2_rn(make_float2(__uint_as_float(p[0] << 16), __uint_as_float(p[0] & 0xffff0000u)), minus,
                        make_float2(a, b));
  p[1] = pack_bf16(r.x, r.y);
  r = __ffma2_rn(make_float2(__uint_as_float(p[1] << 16), __uint_as_float(p[1] & 0xffff0000u)), minus, r);
  p[2] = __byte_perm(__float_as_uint(r.x), __float_as_uint(r.y), 0x7632);
  rem |= __float_as_uint(r.x) | __float_as_uint(r.y);
}

__device__ __forceinline__ uint32_t swz64(int row, int byte) {  // 64-byte rows, 64-byte swizzle
  return (uint32_t)(row * 64 + (byte ^ (((row >> 1) & 3) << 4)));
}

__device__ __forceinline__ void sts64(uint32_t addr, uint32_t x, uint32_t y) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(x), "r"(y) : "memory");
}
// Elements of operand `op` (0 = A, 1 = B); zero where the debug build finds them out of bounds.
__device__ __forceinline__ float load1(const GemmArgs& g, int op, const float* p) {
  return ks_in_bounds(g, op, p, 4) ? __ldg(p) : 0.f;
}
__device__ __forceinline__ float4 load4(const GemmArgs& g, int op, const float* p) {
  return ks_in_bounds(g, op, p, 16) ? __ldg(reinterpret_cast<const float4*>(p)) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// One operand's slice of R rows (M of A, N of B) x 32 K as this thread loads and
// stores it.
template <int R, int KIND>
struct Slice;

// The slice is stored and the next one loaded part by part (`parts` of them),
// each part's registers being reloaded as soon as they are stored.

// K contiguous: a warp instruction covers 4 rows x 128 bytes of K; part t is 4
// consecutive K of one row.  Warp w of the group has rows w, w + 4, ...
template <int R>
struct Slice<R, kRows> {
  static constexpr int PARTS = R / 16, N = 4;
  const float* ptr;  // (row of part 0, K) of the chunk to load
  int64_t step;      // 16 rows on
  int row, lim, kq, sm;
  __device__ __forceinline__ void place(int warp, int lane) {
    row = 4 * (lane >> 3) + warp;
    sm = warp * (R / 4) + (lane >> 3);
    kq = lane & 7;
  }
  __device__ __forceinline__ void start(const Args&, const float* base, int64_t ld, int r0, int rows, int k0) {
    lim = rows - r0 - row;  // part t's row exists when 16 t < lim
    ptr = base + (int64_t)(r0 + row) * ld + k0 + 4 * kq;
    step = 16 * ld;
  }
  __device__ __forceinline__ void advance() { ptr += kBK; }
  __device__ __forceinline__ void load(const GemmArgs& g, int op, int t, float (&v)[N], bool fast, bool vec,
                                       int kleft) const {
    const float* p = ptr + t * step;
    const int left = fast ? kBK : kleft - 4 * kq;
    const bool in = fast || 16 * t < lim;
    if (fast || (in && vec && left >= 4)) {
      const float4 x = load4(g, op, p);
      v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = (in && e < left) ? load1(g, op, p + e) : 0.f;
    }
  }
  __device__ __forceinline__ void store(int t, const float (&v)[N], uint32_t base, uint32_t& rem) const {
    uint32_t x[kParts], y[kParts];
    split2(v[0], v[1], x, rem);
    split2(v[2], v[3], y, rem);
    const uint32_t at = base + swz64(sm + 4 * t, 8 * kq);
#pragma unroll
    for (int s = 0; s < kParts; ++s) sts64(at + s * (R * 64), x[s], y[s]);
  }
};

// R contiguous: part t is 4 consecutive rows x 4 consecutive K; a warp's part
// covers 32 rows x 16 K, each of its loads 4 K rows x 128 bytes.
template <int R>
struct Slice<R, kCols> {
  static constexpr int PARTS = R / 64, N = 16;
  const float* ptr;
  int64_t ld;
  int row, lim, k, sm;
  __device__ __forceinline__ void place(int warp, int lane) {
    constexpr int MB = R / 32;  // blocks of 32 rows: 4 (a warp has both K halves) or 2
    sm = (warp % MB) * 8 + ((lane >> 1) & 7);  // 8-byte stores: 16 lanes = 8 rows x one 16-byte piece
    row = 4 * sm;
    k = 16 * (warp / MB) + 4 * ((lane & 1) | ((lane >> 3) & 2));
  }
  __device__ __forceinline__ void start(const Args&, const float* base, int64_t ld_, int r0, int rows, int k0) {
    ld = ld_;
    lim = rows - r0 - row;  // rows that exist of this thread's 4
    ptr = base + (int64_t)(k0 + k) * ld + r0 + row;
  }
  __device__ __forceinline__ void advance() { ptr += kBK * ld; }
  __device__ __forceinline__ void load(const GemmArgs& g, int op, int t, float (&v)[N], bool fast, bool vec,
                                       int kleft) const {
    const float* p = ptr + 16 * t * ld;
#pragma unroll
    for (int e = 0; e < 4; ++e, p += ld) {
      const bool in = fast || k + 16 * t + e < kleft;
      if (fast || (in && vec && lim >= 4)) {
        const float4 x = load4(g, op, p);
        v[4 * e] = x.x; v[4 * e + 1] = x.y; v[4 * e + 2] = x.z; v[4 * e + 3] = x.w;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) v[4 * e + j] = (in && j < lim) ? load1(g, op, p + j) : 0.f;
      }
    }
  }
  __device__ __forceinline__ void store(int t, const float (&v)[N], uint32_t base, uint32_t& rem) const {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint32_t x[kParts], y[kParts];
      split2(v[j], v[4 + j], x, rem);
      split2(v[8 + j], v[12 + j], y, rem);
      const uint32_t at = base + swz64(sm + j * (R / 4), 2 * k + 32 * t);
#pragma unroll
      for (int s = 0; s < kParts; ++s) sts64(at + s * (R * 64), x[s], y[s]);
    }
  }
};

// Neighbourhoods of an NHWC image with a multiple of 32 channels: column
// (kh * 3 + kw) * Ch + c of row (n, h, w) is x[n, h + kh - 1, w + kw - 1, c], zero
// outside.  A chunk then lies in one tap, and moving a tap on moves every row's
// address by the same distance, so this is the K-contiguous slice with rows of
// Ch, plus one bit per row and tap that says whether the tap is inside.  (Written
// out by a separate pass, the neighbourhoods are nine times the image: VGG16 on
// 16 images took 5.06 ms with that pass, and one for bias and ReLU, against 3.62.)
template <int R>
struct Slice<R, kConv> : Slice<R, kRows> {
  using Base = Slice<R, kRows>;
  using Base::N;
  using Base::PARTS;
  uint32_t inside[(PARTS + 2) / 3];  // nine bits a part, three parts a word
  int c, tap;
  int64_t down;  // from the end of a tap's channels to the next row of taps
  int channels;
  __device__ __forceinline__ void start(const Args& p, const float* x, int64_t, int r0, int rows, int k0) {
    channels = p.Ch;
    tap = k0 / p.Ch;
    c = k0 - tap * p.Ch;
    down = (int64_t)(p.W - 3) * p.Ch;
    this->step = 16 * (int64_t)p.Ch;
    this->ptr = x + ((int64_t)(r0 + this->row) + (tap / 3 - 1) * p.W + (tap % 3 - 1)) * p.Ch + c + 4 * this->kq;
#pragma unroll
    for (int i = 0; i < (PARTS + 2) / 3; ++i) inside[i] = 0;
#pragma unroll
    for (int t = 0; t < PARTS; ++t) {
      const int m = r0 + this->row + 16 * t, hw = m % (p.H * p.W), h = hw / p.W, w = hw - h * p.W;
      uint32_t in = 0;
      if (m < rows) {
        const uint32_t cols = (w > 0 ? 1u : 0u) | 2u | (w + 1 < p.W ? 4u : 0u);
        in = (h > 0 ? cols : 0u) | cols << 3 | (h + 1 < p.H ? cols << 6 : 0u);
      }
      inside[t / 3] |= in << (9 * (t % 3));
    }
  }
  __device__ __forceinline__ void advance() {
    this->ptr += kBK;
    c += kBK;
    if (c == channels) {
      c = 0;
      if (++tap % 3 == 0) this->ptr += down;
    }
  }
  __device__ __forceinline__ void load(const GemmArgs& g, int op, int t, float (&v)[N], bool, bool, int) const {
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if ((inside[t / 3] >> (9 * (t % 3) + tap)) & 1)
      x = load4(g, op, this->ptr + t * this->step);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
  }
};

// G consecutive accumulator columns of this thread's TMEM lane.
template <int G>
__device__ __forceinline__ void tmem_ld(uint32_t a, uint32_t (&r)[G]) {
  if constexpr (G == 16) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(a));
  } else {
    static_assert(G == 8, "column groups of 8 or 16");
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(a));
  }
}

// Shared-memory descriptor of a K-major tile of 64-byte rows, 64-byte swizzle
// (mode 4): groups of 8 rows 512 bytes apart.
__device__ __forceinline__ uint64_t desc64(uint32_t addr) { return smem_desc_sw128(addr, 16, 512, 4); }

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// A whole warp's bounded wait: its lanes go on, or give up, together.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, int* status, int code) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, status, code));
}

// The last chunks' slots are freed by commits that nobody else waits for; their
// arrivals have to come (bounded) before the CTA that holds the barriers may exit.
// The issuing thread waits for its own (in the converting warps the wait cost
// registers that spill: 323 x 312 x 3945 x 8 A^T B 89 us instead of 83), the pair's
// converting warps for the first CTA's.
template <int STAGES>
__device__ __forceinline__ void wait_freed(uint64_t* empty, int total, int* status) {
  for (int i = max(0, total - STAGES); i < total; ++i)
    if (!mbar_wait(&empty[i % STAGES], (i / STAGES) & 1, status, kStatusTimeoutEmpty)) break;
}

struct Item {
  int b, m0, n0, kbeg, kend;
  int64_t slab;  // batch entry, or (batch entry, split) of the workspace
};

template <int BN, int BM = kBM>
__device__ __forceinline__ Item item_of(const Args& p, int item) {
  const int s = item % p.splits, tile = item / p.splits;
  const int per = p.tiles_m * p.tiles_n;
  Item it;
  it.b = tile / per;
  const int t = tile - it.b * per;
  const int per_group = p.group_m * p.tiles_n, g = t / per_group, first = g * p.group_m;
  const int rows = min(p.group_m, p.tiles_m - first), r = t - g * per_group;
  it.m0 = (first + r % rows) * BM;
  it.n0 = (r / rows) * BN;
  it.kbeg = s * p.kchunk;
  it.kend = min(p.g.K, it.kbeg + p.kchunk);
  it.slab = (int64_t)it.b * p.splits + s;
  return it;
}

__device__ __forceinline__ int chunks(const Item& it) { return (it.kend - it.kbeg + kBK - 1) / kBK; }

// The 12 MMAs of one chunk (small products first) and the commits that free its
// slot and announce its accumulator; one thread.
template <int BN>
__device__ __forceinline__ void issue_mmas(uint32_t a0, uint32_t d, uint64_t* slot_free, uint64_t* acc_full) {
  using C = Cfg<BN>;
  constexpr uint32_t idesc = instr_desc<false>(kBM, BN, false, false);
  constexpr int pa[6] = {1, 0, 2, 0, 1, 0}, pb[6] = {1, 2, 0, 1, 0, 0};
  tc_fence_after();
  const uint64_t da = desc64(a0), db = desc64(a0 + kParts * C::A_PART);
#pragma unroll
  for (int g = 0; g < 6; ++g)
#pragma unroll
    for (int k = 0; k < kBK / 16; ++k)  // the address field counts 16-byte units
      mma<false>(d, da + (pa[g] * C::A_PART + k * 32) / 16, db + (pb[g] * C::B_PART + k * 32) / 16, idesc,
                 (g | k) != 0 ? 1u : 0u);
  mma_commit(slot_free);
  mma_commit(acc_full);
}

// Bias and ReLU of column n, where the launch has them.
template <bool ACT>
__device__ __forceinline__ float act(const Args& p, int n, float v) {
  if constexpr (ACT) {
    if (p.bias) v += __ldg(p.bias + n);
    if (p.relu) v = fmaxf(v, 0.f);
  }
  return v;
}

// Up to four (`left`) consecutive columns of one row of C, from column n on.
template <bool ACT>
__device__ __forceinline__ void store4(const Args& p, float* dst, int n, int left, const float (&v)[4]) {
  const GemmArgs& g = p.g;
  float o[4] = {g.alpha * v[0], g.alpha * v[1], g.alpha * v[2], g.alpha * v[3]};
  if (!ks_in_bounds(g, 2, dst, 4 * min(left, 4))) return;
  if (g.vecC && left >= 4) {
    if (g.beta != 0.f) {
      const float4 c = *reinterpret_cast<const float4*>(dst);
      o[0] = fmaf(g.beta, c.x, o[0]); o[1] = fmaf(g.beta, c.y, o[1]);
      o[2] = fmaf(g.beta, c.z, o[2]); o[3] = fmaf(g.beta, c.w, o[3]);
    }
    *reinterpret_cast<float4*>(dst) =
        make_float4(act<ACT>(p, n, o[0]), act<ACT>(p, n + 1, o[1]), act<ACT>(p, n + 2, o[2]), act<ACT>(p, n + 3, o[3]));
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (e < left) dst[e] = act<ACT>(p, n + e, g.beta != 0.f ? fmaf(g.beta, dst[e], o[e]) : o[e]);
  }
}

// The warp's rows of a tile: lane l has row row0 + 4 l, acc[j][q] its column
// col + 4 q + j.  With 32-byte-aligned rows every lane writes whole 32-byte
// sectors of its own row.  Otherwise 16 columns at a time go through the
// warp's 2 KB of shared memory (16-byte piece x of row l at x ^ (l / 2 % 4), free
// of bank conflicts both ways) and leave as 64-byte runs of a row: lanes
// writing 4 bytes of 32 different rows took 109 us against 34 (SIMT kernel) at
// 1433 x 2406 x 18 x 16 with odd rows.
template <int G, bool ACT>
__device__ __forceinline__ void store_rows(const Args& p, const Item& it, int row0, int col, const float (&acc)[4][G],
                                           uint32_t stage, int lane) {
  const float alpha = p.g.alpha, beta = p.g.beta;
  float* base = p.g.C + it.slab * p.g.strideC + col;
  if (p.vec8 && col + 4 * G <= p.g.N) {
    if (row0 + 4 * lane >= p.g.M) return;
    float* crow = base + (int64_t)(row0 + 4 * lane) * p.g.ldc;
#pragma unroll
    for (int q = 0; q < G; q += 2) {
      float o[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) o[e] = alpha * acc[e & 3][q + (e >> 2)];
      float* dst = crow + 4 * q;
      if (!ks_in_bounds(p.g, 2, dst, 32)) continue;
      if (beta != 0.f) {
        const float4 c0 = *reinterpret_cast<const float4*>(dst), c1 = *reinterpret_cast<const float4*>(dst + 4);
        o[0] = fmaf(beta, c0.x, o[0]); o[1] = fmaf(beta, c0.y, o[1]);
        o[2] = fmaf(beta, c0.z, o[2]); o[3] = fmaf(beta, c0.w, o[3]);
        o[4] = fmaf(beta, c1.x, o[4]); o[5] = fmaf(beta, c1.y, o[5]);
        o[6] = fmaf(beta, c1.z, o[6]); o[7] = fmaf(beta, c1.w, o[7]);
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) o[e] = act<ACT>(p, col + 4 * q + e, o[e]);
      asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "f"(o[0]), "f"(o[1]),
                   "f"(o[2]), "f"(o[3]), "f"(o[4]), "f"(o[5]), "f"(o[6]), "f"(o[7])
                   : "memory");
    }
    return;
  }
#pragma unroll
  for (int blk = 0; blk < G / 4; ++blk) {
    const int left = p.g.N - col - 16 * blk;  // columns of the block that exist
    if (left <= 0) return;
    __syncwarp();
#pragma unroll
    for (int x = 0; x < 4; ++x)
      asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(stage + lane * 64 + ((x ^ ((lane >> 1) & 3)) << 4)),
                   "f"(acc[0][4 * blk + x]), "f"(acc[1][4 * blk + x]), "f"(acc[2][4 * blk + x]),
                   "f"(acc[3][4 * blk + x])
                   : "memory");
    __syncwarp();
    if (p.g.vecC) {
#pragma unroll 2
      for (int i = 0; i < 4; ++i) {
        const int r = 8 * i + (lane >> 2), c = 4 * (lane & 3), row = row0 + 4 * r;
        float o[4];
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(o[0]), "=f"(o[1]), "=f"(o[2]), "=f"(o[3])
                     : "r"(stage + r * 64 + (((lane & 3) ^ ((r >> 1) & 3)) << 4))
                     : "memory");
        if (row < p.g.M && c < left)
          store4<ACT>(p, base + (int64_t)row * p.g.ldc + 16 * blk + c, col + 16 * blk + c, left - c, o);
      }
    } else {
#pragma unroll 4
      for (int i = 0; i < 16; ++i) {
        const int r = 2 * i + (lane >> 4), c = lane & 15, row = row0 + 4 * r;
        float o;
        asm volatile("ld.shared.f32 %0, [%1];"
                     : "=f"(o)
                     : "r"(stage + r * 64 + (((c >> 2) ^ ((r >> 1) & 3)) << 4) + 4 * (c & 3))
                     : "memory");
        if (row < p.g.M && c < left) {
          float* dst = base + (int64_t)row * p.g.ldc + 16 * blk + c;
          if (!ks_in_bounds(p.g, 2, dst, 4)) continue;
          o *= alpha;
          *dst = act<ACT>(p, col + 16 * blk + c, beta != 0.f ? fmaf(beta, *dst, o) : o);
        }
      }
    }
  }
}

// A block of an item, 32 rows row0 + 4 i by CW columns from col on, by plain FP32
// FMAs over its K range, in K order; one warp, in its part of the emptied ring.  A
// lane has 8 rows x 4 (CW 32) or 8 columns.  Eight K at a time go K-major into
// shared memory by asynchronous copies of an element (any alignment, either
// storage order; K-contiguous operands four rows of 32 bytes an instruction),
// several steps ahead: what bounds a warp is their latency.  Pitches of 4 modulo 32
// words keep the copies and the reads free of bank conflicts.
template <int CW>
struct Redo {
  static constexpr int K = 8, APITCH = 36, BPITCH = CW + 4;
  static constexpr int STEP = K * (APITCH + BPITCH);  // floats of one step
  static constexpr int STEPS = CW == 32 ? 7 : 5;
  static constexpr int FLOATS = STEPS * STEP;  // of one warp
};

// One element of operand `op`, or zero (its base `any` is then the address given).
__device__ __forceinline__ void copy_async(const GemmArgs& g, int op, uint32_t dst, const float* src,
                                           const float* any, bool in) {
  in = in && ks_in_bounds(g, op, src, 4);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(in ? src : any), "r"(in ? 4 : 0)
               : "memory");
}

template <int CW, int AK, bool B_MN>
__device__ __forceinline__ void redo_block(const Args& p, const Item& it, int row0, int col, const float* buf,
                                           int lane) {
  using R = Redo<CW>;
  const GemmArgs& g = p.g;
  const float* A = static_cast<const float*>(g.A) + (int64_t)it.b * g.strideA;
  const float* B = static_cast<const float*>(g.B) + (int64_t)it.b * g.strideB;
  const int four = lane >> 3, kk = lane & 7;  // K-contiguous: rows (columns) 4 e + four, K kk
  uint32_t inside[AK == kConv ? 3 : 1];       // nine bits a row, three rows a word
  if constexpr (AK == kConv) {
#pragma unroll
    for (int i = 0; i < 3; ++i) inside[i] = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int m = row0 + 4 * (4 * e + four), hw = m % (p.H * p.W), h = hw / p.W, w = hw - h * p.W;
      uint32_t in = 0;
      if (m < g.M) {
        const uint32_t cols = (w > 0 ? 1u : 0u) | 2u | (w + 1 < p.W ? 4u : 0u);
        in = (h > 0 ? cols : 0u) | cols << 3 | (h + 1 < p.H ? cols << 6 : 0u);
      }
      inside[e / 3] |= in << (9 * (e % 3));
    }
  }
  const uint32_t sbuf = smem_u32(buf);
  // INNER: every element of the step exists, which spares the copies their tests.
  auto copies = [&](int k0, uint32_t sa, uint32_t sb, auto inner) {
    constexpr bool INNER = decltype(inner)::value;
    const int left = it.kend - k0;
    if constexpr (AK == kCols) {
      const float* a = A + k0 * g.lda + row0 + 4 * lane;
      const bool row = row0 + 4 * lane < g.M;
#pragma unroll
      for (int e = 0; e < R::K; ++e, a += g.lda)
        copy_async(g, 0, sa + 4 * (e * R::APITCH + lane), a, A, INNER || (row && e < left));
    } else if constexpr (AK == kConv) {
      const int tap = k0 / p.Ch;  // a step is in one tap
      const float* a =
          A + ((int64_t)row0 + 4 * four + (tap / 3 - 1) * p.W + (tap % 3 - 1)) * p.Ch + (k0 - tap * p.Ch) + kk;
#pragma unroll
      for (int e = 0; e < 8; ++e, a += 16 * p.Ch)
        copy_async(g, 0, sa + 4 * (kk * R::APITCH + 4 * e + four), a, A, (inside[e / 3] >> (9 * (e % 3) + tap)) & 1);
    } else {
      const float* a = A + (int64_t)(row0 + 4 * four) * g.lda + k0 + kk;
#pragma unroll
      for (int e = 0; e < 8; ++e, a += 16 * g.lda)
        copy_async(g, 0, sa + 4 * (kk * R::APITCH + 4 * e + four), a, A,
                   INNER || (row0 + 4 * (4 * e + four) < g.M && kk < left));
    }
    if constexpr (B_MN) {
      const float* b = B + k0 * g.ldb + col + lane;
#pragma unroll
      for (int e = 0; e < R::K; ++e, b += g.ldb)
#pragma unroll
        for (int c = 0; c < CW; c += 32)
          copy_async(g, 1, sb + 4 * (e * R::BPITCH + c + lane), b + c, B, INNER || (col + c + lane < g.N && e < left));
    } else {
      const float* b = B + (int64_t)(col + four) * g.ldb + k0 + kk;
#pragma unroll
      for (int e = 0; e < CW / 4; ++e, b += 4 * g.ldb)
        copy_async(g, 1, sb + 4 * (kk * R::BPITCH + 4 * e + four), b, B,
                   INNER || (col + 4 * e + four < g.N && kk < left));
    }
  };
  // (Not with A^T: the pair kernel of A^T B then takes 24 % longer at 4096 x 4096 x
  // 4096 on values that all split.)
  const bool whole = AK != kCols && row0 + 4 * 31 < g.M && col + CW <= g.N;
  auto load = [&](int step) {
    const int k0 = it.kbeg + step * R::K;
    const uint32_t sa = sbuf + 4 * (step % R::STEPS * R::STEP), sb = sa + 4 * R::K * R::APITCH;
    if (whole && k0 + R::K <= it.kend) copies(k0, sa, sb, std::true_type());
    else if (k0 < it.kend) copies(k0, sa, sb, std::false_type());
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int r0 = 8 * (lane >> 3), c0 = 4 * (lane & 7), steps = (it.kend - it.kbeg + R::K - 1) / R::K;
  float v[8][CW / 8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < CW / 8; ++j) v[i][j] = 0.f;
  __syncwarp();  // the block before is summed
#pragma unroll 1
  for (int s = 0; s < R::STEPS - 1; ++s) load(s);
#pragma unroll 1
  for (int s = 0; s < steps; ++s) {
    asm volatile("cp.async.wait_group %0;" ::"n"(R::STEPS - 2) : "memory");
    __syncwarp();
    load(s + R::STEPS - 1);
    const float* sa = buf + s % R::STEPS * R::STEP;
    const float* sb = sa + R::K * R::APITCH;
#pragma unroll
    for (int k = 0; k < R::K; ++k) {  // past the range both operands are zero
      float a[8], b[CW / 8];
#pragma unroll
      for (int i = 0; i < 8; i += 4) {
        const float4 t = *reinterpret_cast<const float4*>(sa + k * R::APITCH + r0 + i);
        a[i] = t.x; a[i + 1] = t.y; a[i + 2] = t.z; a[i + 3] = t.w;
      }
#pragma unroll
      for (int j = 0; j < CW / 8; j += 4) {
        const float4 t = *reinterpret_cast<const float4*>(sb + k * R::BPITCH + 8 * j + c0);
        b[j] = t.x; b[j + 1] = t.y; b[j + 2] = t.z; b[j + 3] = t.w;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < CW / 8; ++j) v[i][j] = fmaf(a[i], b[j], v[i][j]);
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int row = row0 + 4 * (r0 + i);
    float* crow = g.C + it.slab * g.strideC + (int64_t)row * g.ldc;
#pragma unroll
    for (int j = 0; j < CW / 8; j += 4) {
      const int n = col + 8 * j + c0;
      const float o[4] = {v[i][j], v[i][j + 1], v[i][j + 2], v[i][j + 3]};
      if (row < g.M && n < g.N) store4<AK == kConv>(p, crow + n, n, g.N - n, o);
    }
  }
}

// What the reading warps left unwritten: byte o of `lost` has a bit for each
// warp's part of the CTA's item first + o * step.  The parts, or halves of a pair's,
// go round the reading warps.
template <int BN, int BM, int G, int AK, bool B_MN>
__device__ __forceinline__ void redo(const Args& p, const uint32_t* lost, int first, int step, int m_off,
                                     const float* ring, int warp, int lane) {
  constexpr int CW = G == 8 ? 32 : 64;
  int turn = 0;
#pragma unroll 1
  for (int o = 0; first + (int64_t)o * step < p.items; ++o) {
    uint32_t bits = (lost[o >> 2] >> (8 * (o & 3))) & 255u;
    if (!bits) continue;
    const Item it = item_of<BN, BM>(p, first + o * step);
#pragma unroll 1
    for (; bits; bits &= bits - 1) {
      const int w = __ffs(bits) - 1, row0 = it.m0 + m_off + (w & 3), col = it.n0 + 4 * G * (w >> 2);
#pragma unroll 1
      for (int c = col; c < min(col + 4 * G, p.g.N); c += CW)
        if (turn++ % kReaders == warp)
          redo_block<CW, AK, B_MN>(p, it, row0, c, ring + warp * Redo<CW>::FLOATS, lane);
    }
  }
}

// The reading warps have all left their loops.
__device__ __forceinline__ void readers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(32 * kReaders) : "memory"); }

template <int BN, int AK, bool B_MN>
__global__ void __launch_bounds__(kThreads, 1) f32tc_kernel(const __grid_constant__ Args p) {
  using C = Cfg<BN>;
  constexpr int G = C::G;
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full[C::STAGES], empty[C::STAGES], accf[2], acce[2];
  __shared__ int inexact[kMarks];  // chunk i left its mark i + 1 in slot i % kMarks when a split lost bits
  __shared__ uint32_t lost_sh[kMaxItems / 4];  // see redo
  __shared__ int any_lost;
  __shared__ uint32_t tmem_sh;
  const uint32_t smem = (smem_u32(smem_raw) + 1023) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(&full[s], 4);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&accf[a], 1);
      mbar_init(&acce[a], kReaders);
    }
    fence_barrier_init();
  }
  if (threadIdx.x < kMarks) inexact[threadIdx.x] = 0;
  if (threadIdx.x < kMaxItems / 4) lost_sh[threadIdx.x] = 0;
  if (threadIdx.x == 0) any_lost = 0;
  if (warp == kIssuer) tmem_alloc<C::TMEM>(&tmem_sh);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_sh;
  int total = 0;  // chunks of all of this CTA's items
  for (int i = blockIdx.x; i < p.items; i += gridDim.x) total += chunks(item_of<BN>(p, i));
  pdl_wait();
  pdl_launch_dependents();

  if (warp >= kIssuer) {
    // ---------------------------------------------------------------- MMAs
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsIssue));
    if (warp == kIssuer && elect_one()) {
      for (int i = 0; i < total; ++i) {
        const int stage = i % C::STAGES;
        if (!mbar_wait(&acce[i & 1], ((i >> 1) & 1) ^ 1, p.status, kStatusTimeoutAccEmpty)) break;
        if (!mbar_wait(&full[stage], (i / C::STAGES) & 1, p.status, kStatusTimeoutFull)) break;
        issue_mmas<BN>(smem + stage * C::STAGE, tmem + (uint32_t)((i & 1) * BN), &empty[stage], &accf[i & 1]);
      }
      wait_freed<C::STAGES>(empty, total, p.status);
    }
  } else if (warp >= kReaders) {
    // ---------------------------------------------------------------- load and convert
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(C::REGS_CONVERT));
    const int group = (warp - kReaders) >> 2;
    using SA = Slice<kBM, AK>;
    using SB = Slice<BN, B_MN ? kCols : kRows>;
    SA sa;
    SB sb;
    sa.place(warp & 3, lane);
    sb.place(warp & 3, lane);
    float va[SA::PARTS][SA::N], vb[SB::PARTS][SB::N];
    int item = (int)blockIdx.x - (int)gridDim.x, left = 0;  // K elements from the chunk at the pointers to the item's end
    bool fa = false, fb = false;                             // the item's tile is interior and 16-byte loads are legal
    auto next_item = [&]() {
      item += gridDim.x;
      const Item it = item_of<BN>(p, item);
      sa.start(p, static_cast<const float*>(p.g.A) + (int64_t)it.b * p.g.strideA, p.g.lda, it.m0, p.g.M, it.kbeg);
      sb.start(p, static_cast<const float*>(p.g.B) + (int64_t)it.b * p.g.strideB, p.g.ldb, it.n0, p.g.N, it.kbeg);
      left = it.kend - it.kbeg;
      fa = p.g.vecA && it.m0 + kBM <= p.g.M;
      fb = p.g.vecB && it.n0 + BN <= p.g.N;
    };
    auto skip = [&]() {  // one chunk on, into the next item if need be
      left -= kBK;
      if (left <= 0) {
        next_item();
      } else {
        sa.advance();
        sb.advance();
      }
    };
    if (group < total) {
      next_item();
      for (int s = 0; s < group; ++s) skip();
      const bool wa = fa && left >= kBK, wb = fb && left >= kBK;
#pragma unroll
      for (int t = 0; t < SA::PARTS; ++t) sa.load(p.g, 0, t, va[t], wa, p.g.vecA, left);
#pragma unroll
      for (int t = 0; t < SB::PARTS; ++t) sb.load(p.g, 1, t, vb[t], wb, p.g.vecB, left);
    }
    for (int i = group; i < total; i += kGroups) {
      const int stage = i % C::STAGES;
      const bool more = i + kGroups < total;
      if (more)
        for (int s = 0; s < kGroups; ++s) skip();
      if (!warp_wait(&empty[stage], ((i / C::STAGES) & 1) ^ 1, p.status, kStatusTimeoutEmpty)) break;
      uint32_t rem = 0;
      const uint32_t a0 = smem + stage * C::STAGE, b0 = a0 + kParts * C::A_PART;
      if (more && fa && fb && left >= kBK) {
#pragma unroll
        for (int t = 0; t < SA::PARTS; ++t) sa.store(t, va[t], a0, rem);
#pragma unroll
        for (int t = 0; t < SA::PARTS; ++t) sa.load(p.g, 0, t, va[t], true, true, left);
#pragma unroll
        for (int t = 0; t < SB::PARTS; ++t) sb.store(t, vb[t], b0, rem);
#pragma unroll
        for (int t = 0; t < SB::PARTS; ++t) sb.load(p.g, 1, t, vb[t], true, true, left);
      } else {
#pragma unroll
        for (int t = 0; t < SA::PARTS; ++t) sa.store(t, va[t], a0, rem);
#pragma unroll
        for (int t = 0; t < SB::PARTS; ++t) sb.store(t, vb[t], b0, rem);
        if (more) {
#pragma unroll
          for (int t = 0; t < SA::PARTS; ++t) sa.load(p.g, 0, t, va[t], false, p.g.vecA, left);
#pragma unroll
          for (int t = 0; t < SB::PARTS; ++t) sb.load(p.g, 1, t, vb[t], false, p.g.vecB, left);
        }
      }
      if (rem & 0xffffu) inexact[i % kMarks] = i + 1;
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[stage]);
    }
  } else {
    // ---------------------------------------------------------------- accumulators, C
    if constexpr (C::REGS_READ > kRegsLaunch) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(C::REGS_READ));
    float acc[4][G];
    int item = blockIdx.x, at = 0, n = 0;  // the item being summed, chunks of it added, its chunks
    bool lost = false, whole = true;
    const uint32_t t_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * G);
    const uint32_t stage = smem + C::STAGES * C::STAGE + warp * kStoreBytes;
    for (int c = 0; c < total; ++c) {
      if (at == 0) {
        n = chunks(item_of<BN>(p, item));
        lost = false;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int q = 0; q < G; ++q) acc[j][q] = 0.f;
      }
      if (!(whole = warp_wait(&accf[c & 1], (c >> 1) & 1, p.status, kStatusTimeoutAcc))) break;
      __syncwarp();  // lanes without a row of C may have been elsewhere
      tc_fence_after();
      lost |= *(volatile int*)&inexact[c % kMarks] == c + 1;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint32_t r[G];
        tmem_ld<G>(t_lane + (uint32_t)((c & 1) * BN + j * (BN / 4)), r);
        tmem_ld_wait();
        if (j == 3) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acce[c & 1]);
        }
#pragma unroll
        for (int q = 0; q < G; ++q) acc[j][q] += __uint_as_float(r[q]);
      }
      if (++at < n) continue;
      at = 0;
      const Item it = item_of<BN>(p, item);
      item += gridDim.x;
      const int row0 = it.m0 + (warp & 3), col = it.n0 + 4 * G * (warp >> 2);
      if (row0 >= p.g.M || col >= p.g.N) continue;
      // A split that lost bits or an accumulator that overflowed: left to redo().
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < G; ++q) lost |= !(fabsf(acc[j][q]) <= 3.402823466e38f);
      if (!__any_sync(0xffffffffu, lost)) {
        store_rows<G, AK == kConv>(p, it, row0, col, acc, stage, lane);
      } else if (lane == 0) {
        const int o = (item - (int)blockIdx.x) / (int)gridDim.x - 1;
        atomicOr(&lost_sh[o >> 2], 1u << (8 * (o & 3) + warp));
        any_lost = 1;
      }
    }
    readers_sync();
    if (whole && *(volatile int*)&any_lost)
      redo<BN, kBM, G, AK, B_MN>(p, lost_sh, blockIdx.x, gridDim.x, 0,
                                 reinterpret_cast<float*>(smem_raw + (smem - smem_u32(smem_raw))), warp, lane);
  }
  __syncthreads();
  if (warp == kIssuer) {
    tc_fence_after();
    tmem_dealloc<C::TMEM>(tmem);
  }
}

// CTAs or pairs of a launch: as many as are resident at once, and whole multiples
// of that where each would have more items than it can mark.
int units_for(int items, int resident) {
  const int64_t most = (int64_t)resident * kMaxItems;
  return (int)std::min<int64_t>(items, resident * ((items + most - 1) / most));
}

template <int BN, int AK, bool B_MN>
cudaError_t launch(const Args& a, int sms, cudaStream_t s) {
  auto kern = f32tc_kernel<BN, AK, B_MN>;
  static unsigned long long done_mask = 0;  // devices whose attribute is set
  int dev = 0;
  cudaGetDevice(&dev);
  const unsigned long long bit = 1ull << (dev & 63);
  if (!(__atomic_load_n(&done_mask, __ATOMIC_ACQUIRE) & bit)) {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, kern);
    if (e != cudaSuccess) return e;
    if (fa.numRegs != kRegsLaunch) return cudaErrorInvalidConfiguration;  // setmaxnreg counts on it
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<BN>::SMEM);
    if (e != cudaSuccess) return e;
    __atomic_fetch_or(&done_mask, bit, __ATOMIC_ACQ_REL);
  }
  return launch_pdl(kern, dim3((unsigned)units_for(a.items, sms)), dim3(kThreads), Cfg<BN>::SMEM, s, nullptr, 0, a);
}

template <int BN>
cudaError_t launch_bn(const Args& a, int sms, cudaStream_t s) {
  const bool bm = a.g.transB == 0;
  if (a.Ch > 0) return launch<BN, kConv, false>(a, sms, s);
  if (a.g.transA) return bm ? launch<BN, kCols, true>(a, sms, s) : launch<BN, kCols, false>(a, sms, s);
  return bm ? launch<BN, kRows, true>(a, sms, s) : launch<BN, kRows, false>(a, sms, s);
}

// ---------------------------------------------------------------- two CTAs on one 256 x 256 tile
// The same with tcgen05's cta_group::2: each CTA of the pair converts its 128
// rows of A and its 128 columns of B and holds its 128 rows' accumulators; the
// first CTA issues MMAs that read both CTAs' shared memory.  Against 128 x 128
// tiles this halves what is read from L2 per product and takes the operand
// reads of the MMAs from 128 to 64 bytes a clock and SM.  One converting group
// has A, the other B, and each of the eight reading warps 128 accumulators.
constexpr int kPairRegsConvert = 64, kPairRegsIssue = 24, kPairRegsRead = 160;  // 256 x 64 + 128 x 24 + 256 x 160 <= 640 x 96

struct Pair {
  static constexpr int BM = 256, BN = 256, G = 32;
  static constexpr int PART = 128 * 64;
  static constexpr int STAGE = 2 * kParts * PART;
  static constexpr int STAGES = 3;
  static constexpr int SMEM = STAGES * STAGE + kReaders * kStoreBytes + 1024;
  static constexpr int TMEM = 512;
};

// A converting group of the pair kernel: its operand's 128 rows of every chunk.
template <class S>
__device__ __forceinline__ void convert_pair(const Args& p, int total, bool is_a, uint32_t rank, uint32_t smem,
                                             uint64_t* full, uint64_t* empty, int* inexact, int warp, int lane) {
  S sl;
  sl.place(warp & 3, lane);
  float v[S::PARTS][S::N];
  const bool vec = is_a ? p.g.vecA : p.g.vecB;
  int item = ((int)blockIdx.x >> 1) - ((int)gridDim.x >> 1), left = 0;
  bool inner = false;
  auto skip = [&]() {
    left -= kBK;
    if (left > 0) {
      sl.advance();
      return;
    }
    item += (int)gridDim.x >> 1;
    const Item it = item_of<Pair::BN, Pair::BM>(p, item);
    const int r0 = (is_a ? it.m0 : it.n0) + 128 * (int)rank, rows = is_a ? p.g.M : p.g.N;
    const float* base = static_cast<const float*>(is_a ? p.g.A : p.g.B) +
                        (int64_t)it.b * (is_a ? p.g.strideA : p.g.strideB);
    sl.start(p, base, is_a ? p.g.lda : p.g.ldb, r0, rows, it.kbeg);
    left = it.kend - it.kbeg;
    inner = vec && r0 + 128 <= rows;
  };
  if (total > 0) {
    skip();
    const bool whole = inner && left >= kBK;
#pragma unroll
    for (int t = 0; t < S::PARTS; ++t) sl.load(p.g, is_a ? 0 : 1, t, v[t], whole, vec, left);
  }
  for (int i = 0; i < total; ++i) {
    const int stage = i % Pair::STAGES;
    const bool more = i + 1 < total;
    if (more) skip();
    if (!warp_wait(&empty[stage], ((i / Pair::STAGES) & 1) ^ 1, p.status, kStatusTimeoutEmpty)) break;
    uint32_t rem = 0;
    const uint32_t at = smem + stage * Pair::STAGE + (is_a ? 0 : kParts * Pair::PART);
    // Registers are reloaded as soon as they are stored: after each half of the
    // eight K-contiguous parts (4096 x 4096 x 4096, A B^T: 10 % slower with the
    // loads after all parts, 26 % after each), after both MN-contiguous ones
    // (A B: 9 % slower after each).
    constexpr int H = S::PARTS == 8 ? 4 : S::PARTS;
    if (more && inner && left >= kBK) {
#pragma unroll
      for (int h = 0; h < S::PARTS; h += H) {
#pragma unroll
        for (int t = h; t < h + H; ++t) sl.store(t, v[t], at, rem);
#pragma unroll
        for (int t = h; t < h + H; ++t) sl.load(p.g, is_a ? 0 : 1, t, v[t], true, true, left);
      }
    } else {
#pragma unroll
      for (int t = 0; t < S::PARTS; ++t) sl.store(t, v[t], at, rem);
      if (more) {
#pragma unroll
        for (int t = 0; t < S::PARTS; ++t) sl.load(p.g, is_a ? 0 : 1, t, v[t], false, vec, left);
      }
    }
    if (rem & 0xffffu) {  // B's columns are in both CTAs' rows of C
      const uint32_t mark = smem_u32(&inexact[i % kMarks]);
      asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(in_cta(mark, rank)), "r"(i + 1) : "memory");
      if (!is_a) asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(in_cta(mark, rank ^ 1)), "r"(i + 1) : "memory");
      asm volatile("fence.acq_rel.cluster;" ::: "memory");
    }
    fence_async_smem();
    __syncwarp();
    if (lane == 0) arrive_cluster(in_cta(smem_u32(&full[stage]), 0));
  }
  wait_freed<Pair::STAGES>(empty, total, p.status);
}

template <int AK, bool B_MN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    f32tc_pair_kernel(const __grid_constant__ Args p) {
  constexpr int G = Pair::G;
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full[Pair::STAGES], empty[Pair::STAGES], accf[2], acce[2];
  __shared__ int inexact[kMarks];
  __shared__ uint32_t lost_sh[kMaxItems / 4];
  __shared__ int any_lost;
  __shared__ uint32_t tmem_sh;
  const uint32_t smem = (smem_u32(smem_raw) + 1023) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int unit = (int)blockIdx.x >> 1, units = (int)gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < Pair::STAGES; ++s) {
      mbar_init(&full[s], 2 * 4 * kGroups);  // used in the first CTA: both CTAs' converting warps
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&accf[a], 1);
      mbar_init(&acce[a], 2 * kReaders);  // used in the first CTA
    }
    fence_barrier_init();
  }
  if (threadIdx.x < kMarks) inexact[threadIdx.x] = 0;
  if (threadIdx.x < kMaxItems / 4) lost_sh[threadIdx.x] = 0;
  if (threadIdx.x == 0) any_lost = 0;
  if (warp == kIssuer) tmem_alloc_pair<Pair::TMEM>(&tmem_sh);
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem = tmem_sh;
  int total = 0;
  for (int i = unit; i < p.items; i += units) total += chunks(item_of<Pair::BN, Pair::BM>(p, i));
  pdl_wait();
  pdl_launch_dependents();

  if (warp >= kIssuer) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPairRegsIssue));
    if (rank == 0 && warp == kIssuer && elect_one()) {
      constexpr uint32_t idesc = instr_desc<false>(Pair::BM, Pair::BN, false, false);
      constexpr int pa[6] = {1, 0, 2, 0, 1, 0}, pb[6] = {1, 2, 0, 1, 0, 0};
      for (int i = 0; i < total; ++i) {
        const int stage = i % Pair::STAGES;
        if (!mbar_wait(&acce[i & 1], ((i >> 1) & 1) ^ 1, p.status, kStatusTimeoutAccEmpty)) break;
        if (!mbar_wait(&full[stage], (i / Pair::STAGES) & 1, p.status, kStatusTimeoutFull)) break;
        tc_fence_after();
        const uint32_t a0 = smem + stage * Pair::STAGE, d = tmem + (uint32_t)((i & 1) * Pair::BN);
        const uint64_t da = desc64(a0), db = desc64(a0 + kParts * Pair::PART);
#pragma unroll
        for (int g = 0; g < 6; ++g)
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k)
            mma_pair<false>(d, da + (pa[g] * Pair::PART + k * 32) / 16, db + (pb[g] * Pair::PART + k * 32) / 16, idesc,
                     (g | k) != 0 ? 1u : 0u);
        commit_pair(&empty[stage]);
        commit_pair(&accf[i & 1]);
      }
    }
  } else if (warp >= kReaders) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPairRegsConvert));
    if (warp < kReaders + 4) convert_pair<Slice<128, AK>>(p, total, true, rank, smem, full, empty, inexact, warp, lane);
    else convert_pair<Slice<128, B_MN ? kCols : kRows>>(p, total, false, rank, smem, full, empty, inexact, warp, lane);
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kPairRegsRead));
    float acc[4][G];
    int item = unit, at = 0, n = 0;
    bool lost = false, whole = true;
    const uint32_t t_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * 128);
    const uint32_t stage = smem + Pair::STAGES * Pair::STAGE + warp * kStoreBytes;
    for (int c = 0; c < total; ++c) {
      if (at == 0) {
        n = chunks(item_of<Pair::BN, Pair::BM>(p, item));
        lost = false;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int q = 0; q < G; ++q) acc[j][q] = 0.f;
      }
      if (!(whole = warp_wait(&accf[c & 1], (c >> 1) & 1, p.status, kStatusTimeoutAcc))) break;
      __syncwarp();
      tc_fence_after();
      lost |= *(volatile int*)&inexact[c % kMarks] == c + 1;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        uint32_t r[16];
        tmem_ld<16>(t_lane + (uint32_t)((c & 1) * Pair::BN + u * 16), r);
        tmem_ld_wait();
        if (u == 7) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) arrive_cluster(in_cta(smem_u32(&acce[c & 1]), 0));
        }
#pragma unroll
        for (int q = 0; q < 16; ++q) acc[u >> 1][(u & 1) * 16 + q] += __uint_as_float(r[q]);
      }
      if (++at < n) continue;
      at = 0;
      const Item it = item_of<Pair::BN, Pair::BM>(p, item);
      item += units;
      const int row0 = it.m0 + 128 * (int)rank + (warp & 3), col = it.n0 + 128 * (warp >> 2);
      if (row0 >= p.g.M || col >= p.g.N) continue;
      // A split that lost bits or an accumulator that overflowed: left to redo().
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < G; ++q) lost |= !(fabsf(acc[j][q]) <= 3.402823466e38f);
      if (!__any_sync(0xffffffffu, lost)) {
        store_rows<G, AK == kConv>(p, it, row0, col, acc, stage, lane);
      } else if (lane == 0) {
        const int o = (item - unit) / units - 1;
        atomicOr(&lost_sh[o >> 2], 1u << (8 * (o & 3) + warp));
        any_lost = 1;
      }
    }
    readers_sync();
    if (whole && *(volatile int*)&any_lost)
      redo<Pair::BN, Pair::BM, G, AK, B_MN>(p, lost_sh, unit, units, 128 * (int)rank,
                                            reinterpret_cast<float*>(smem_raw + (smem - smem_u32(smem_raw))), warp,
                                            lane);
  }
  __syncthreads();
  cluster_sync();  // neither CTA leaves while the other's MMAs or arrivals may reach it
  if (warp == kIssuer) {
    tc_fence_after();
    tmem_dealloc_pair<Pair::TMEM>(tmem);
  }
}

template <int AK, bool B_MN>
cudaError_t launch_pair(const Args& a, int sms, cudaStream_t s) {
  auto kern = f32tc_pair_kernel<AK, B_MN>;
  static unsigned long long done_mask = 0;
  int dev = 0;
  cudaGetDevice(&dev);
  const unsigned long long bit = 1ull << (dev & 63);
  if (!(__atomic_load_n(&done_mask, __ATOMIC_ACQUIRE) & bit)) {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, kern);
    if (e != cudaSuccess) return e;
    if (fa.numRegs != kRegsLaunch) return cudaErrorInvalidConfiguration;  // setmaxnreg counts on it
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Pair::SMEM);
    if (e != cudaSuccess) return e;
    __atomic_fetch_or(&done_mask, bit, __ATOMIC_ACQ_REL);
  }
  const int pairs = units_for(a.items, sms / 2);
  return launch_pdl(kern, dim3((unsigned)(2 * pairs)), dim3(kThreads), Pair::SMEM, s, nullptr, 0, a);
}

}  // namespace f32tc

// Runs the kernel with BN-wide tiles.  With splits > 1, `g` describes the
// workspace of partial products (alpha 1, beta 0, one M x ldc slab per batch
// entry and split, strideC apart), split s covering K [s * kchunk, (s + 1) * kchunk).
// `conv`: A is an NHWC image and M = its positions, K = 9 x its channels (see Conv3x3).
cudaError_t f32tc_launch(int bn, const GemmArgs& g, int splits, int kchunk, int sms, int* status, cudaStream_t s,
                         const Conv3x3* conv) {
  f32tc::Args a;
  a.H = a.W = a.Ch = a.relu = 0;
  a.bias = nullptr;
  if (conv) {
    a.H = conv->H;
    a.W = conv->W;
    a.Ch = conv->C;
    a.bias = conv->bias;
    a.relu = conv->relu;
  }
  a.g = g;
  const int bm = bn == 256 ? 256 : f32tc::kBM;
  a.tiles_m = (g.M + bm - 1) / bm;
  a.tiles_n = (g.N + bn - 1) / bn;
  a.tiles = a.tiles_m * a.tiles_n * g.batch;
  a.splits = splits;
  a.kchunk = kchunk;
  a.items = a.tiles * splits;
  a.group_m = std::max(1, std::min(a.tiles_m, bm == 256 ? 4 : 8));
  a.vec8 = ((uintptr_t)g.C % 32 == 0) && g.ldc % 8 == 0 && (g.batch * splits == 1 || g.strideC % 8 == 0);
  a.status = status;
  if (bn == 64) return f32tc::launch_bn<64>(a, sms, s);
  if (bn == 128) return f32tc::launch_bn<128>(a, sms, s);
  if (bn == 256) {
    using namespace f32tc;
    const bool bmn = g.transB == 0;
    if (a.Ch > 0) return launch_pair<kConv, false>(a, sms, s);
    if (g.transA) return bmn ? launch_pair<kCols, true>(a, sms, s) : launch_pair<kCols, false>(a, sms, s);
    return bmn ? launch_pair<kRows, true>(a, sms, s) : launch_pair<kRows, false>(a, sms, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ks
