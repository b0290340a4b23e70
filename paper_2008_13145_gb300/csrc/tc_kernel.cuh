// Persistent warp-specialised tcgen05 GEMM for sm_103a.
//
// C[b] = alpha * A[b] * B[b]^T + beta * C[b] with A (M x K) and B (N x K)
// K-contiguous in global memory (BF16, or FP32 read as TF32); an operand may
// instead be MN-contiguous (A stored K x M, B stored K x N), in which case it
// is staged as MN-major tiles and the MMA reads it transposed.  Tiles of
// 128 x BN outputs are distributed over persistent CTAs; each CTA runs
//   warps 0..3  : epilogue, tcgen05.ld of their 32-lane quadrant, alpha/beta,
//                 vector stores of C (BN 256: warps 0..7, two per quadrant);
//   next warp   : TMA producer (one elected lane) filling a STAGES-deep ring
//                 of 128-byte-swizzled A/B slices, 128 bytes of K per slice;
//   last warp   : TMEM allocator and MMA issuer (one elected lane), 4
//                 tcgen05.mma per slice into an FP32 accumulator in TMEM.
// Two TMEM accumulators (2 x BN columns) let the epilogue of tile i overlap
// the MMAs of tile i+1.  With GROUPED, the launch covers an uneven group of
// problems: the global tile index is mapped to (problem, tile) by binary
// search over the problems' first-tile offsets, and each problem brings its
// own tensor maps, C and K.
#pragma once
#include "common.cuh"
#include "tc_ptx.cuh"

namespace ks {
namespace tc {

struct TcArgs {
  int M, N, K, batch;
  int tiles_m, tiles_n, num_tiles, k_blocks;
  int raster;   // 0: consecutive tiles walk M (reuse the B slice), 1: walk N,
                // 2: groups of group_m tile rows, each walked along N (L2 locality)
  int group_m;  // raster 2: tile rows (units) per group, >= 1
  float alpha, beta;
  float* C;
  int64_t ldc, strideC;
  int vecC;  // C takes 16-byte accesses (1) or 32-byte ones (2)
  int a_mn, b_mn;  // operand staged MN-major
  // Split-BF16 products: each operand holds nseg segments of seg_blocks
  // K-slices (its BF16 split parts, largest first) and segment g of the K'
  // loop multiplies A's part seg_map bits [2g, 2g + 2) by B's part seg_map bits
  // [16 + 2g, 16 + 2g + 2); seg_blocks is 0 for the other families.
  int seg_blocks, seg_map;
  int* status;
};

// One problem of a grouped launch, in device memory: its two tensor maps
// (128-byte aligned by their type, beyond the 64 bytes TMA requires), its C,
// and its first global tile index.
struct alignas(128) GroupDesc {
  CUtensorMap tmA;
  CUtensorMap tmB;
  float* C;
  int64_t ldc;
  int M, N, k_blocks, tiles_m, tiles_n, tile_start, vecC;
  int a_mn, b_mn, seg_blocks, seg_map;
  float alpha, beta;
};

struct GroupArgs {
  const GroupDesc* descs;
  int count;  // problems; descs[i].tile_start is ascending
};

constexpr int kBM = 128;

template <int BN, int STAGES, bool TF32>
struct TcCfg {
  static constexpr int ELEM = TF32 ? 4 : 2;
  static constexpr int BK = 128 / ELEM;        // K elements per slice (one 128-byte row)
  static constexpr int KMMA = TF32 ? 8 : 16;   // K per tcgen05.mma
  static constexpr int A_BYTES = kBM * 128;
  static constexpr int B_BYTES = BN * 128;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int TMEM_COLS = 2 * BN;     // 128, 256 or 512: power of two >= 32
  // Epilogue warps: two per TMEM lane quadrant, each with half of the columns,
  // where one CTA has the SM to itself; one where two or three share it.
  static constexpr int EPI_WARPS = BN == 256 ? 8 : 4;
  static constexpr int THREADS = 32 * (EPI_WARPS + 2);
  // Epilogue staging: 32 rows x STORE_COLS FP32 columns per epilogue warp.
  static constexpr int STORE_COLS = BN == 256 ? 32 : 16;
  static constexpr int EPI_BYTES = EPI_WARPS * 32 * STORE_COLS * 4;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + EPI_BYTES + 1024;
  // MN-major staging: one TMA box is MN_BOX MN elements (a 128-byte row) by
  // BK K rows; the boxes of a slice lie MN-block after MN-block.  The swizzle
  // atom is 8 K rows of one box for BF16 (128-byte swizzle, SBO 1 KB) and 4 K
  // rows for TF32 (128-byte swizzle of 32-byte pieces, SBO 512 bytes); the
  // descriptor steps one MN block by MN_BOX_BYTES (LBO), and each MMA's K range
  // starts KMMA rows (KMMA x 128 bytes) further on.
  static constexpr int MN_BOX = 128 / ELEM;
  static constexpr int MN_BOX_BYTES = BK * 128;
  static constexpr uint32_t MN_SBO = TF32 ? 512 : 1024;
  static constexpr uint32_t MN_MODE = TF32 ? kSw128Atom32 : kSw128;
};

__device__ __forceinline__ void tile_coords(const TcArgs& p, int tile, int& b, int& tm, int& tn) {
  const int per = p.tiles_m * p.tiles_n;
  b = tile / per;
  const int t = tile - b * per;
  if (p.raster == 2) {
    // Tile rows in groups of group_m (the last group may be shorter); inside a
    // group the index runs down the group's rows first, then along N, so the
    // tiles in flight at once share a few A and B slices that stay in L2.
    const int per_group = p.group_m * p.tiles_n;
    const int g = t / per_group;
    const int first = g * p.group_m;
    const int rows = min(p.group_m, p.tiles_m - first);
    const int r = t - g * per_group;
    tm = first + r % rows;
    tn = r / rows;
  } else if (p.raster == 0) {
    tm = t % p.tiles_m;
    tn = t / p.tiles_m;
  } else {
    tn = t % p.tiles_n;
    tm = t / p.tiles_n;
  }
}

// Where tile `tile` of the launch lives: operand maps, C and its geometry.
struct TileLoc {
  const CUtensorMap* ma;
  const CUtensorMap* mb;
  float* C;
  int64_t ldc, strideC;
  int M, N, k_blocks, b, tm, tn, vecC, a_mn, b_mn, seg_blocks, seg_map;
  float alpha, beta;
};

// First tiles of a group's problems, kept in shared memory: all of them for up
// to kStarts problems, else every `step`-th.  Each role looks up each of its tiles;
// eight dependent reads of descriptors in L2 (256 problems) held the loads back: the
// grouped call of the 256-problem group took 421 us against 386 so.
constexpr int kStarts = 448;
struct GroupIndex {
  const int* starts;
  int n, step;
};

template <bool GROUPED>
__device__ __forceinline__ TileLoc locate(const TcArgs& p, const GroupArgs& g, const GroupIndex& x,
                                          const CUtensorMap* ma, const CUtensorMap* mb, int tile) {
  TileLoc L;
  if constexpr (GROUPED) {
    int lo = 0, hi = x.n - 1;  // last problem whose tile_start <= tile
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (x.starts[mid] <= tile) lo = mid; else hi = mid - 1;
    }
    if (x.step > 1) {
      lo *= x.step;
      hi = min(lo + x.step, g.count) - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (g.descs[mid].tile_start <= tile) lo = mid; else hi = mid - 1;
      }
    }
    const GroupDesc& d = g.descs[lo];
    const int t = tile - d.tile_start;
    L.ma = &d.tmA; L.mb = &d.tmB; L.C = d.C; L.ldc = d.ldc; L.strideC = 0;
    L.M = d.M; L.N = d.N; L.k_blocks = d.k_blocks; L.b = 0; L.vecC = d.vecC; L.a_mn = d.a_mn; L.b_mn = d.b_mn;
    L.seg_blocks = d.seg_blocks; L.seg_map = d.seg_map;
    L.alpha = d.alpha; L.beta = d.beta;
    if (p.raster == 0) { L.tm = t % d.tiles_m; L.tn = t / d.tiles_m; } else { L.tn = t % d.tiles_n; L.tm = t / d.tiles_n; }
  } else {
    L.ma = ma; L.mb = mb; L.C = p.C; L.ldc = p.ldc; L.strideC = p.strideC;
    L.M = p.M; L.N = p.N; L.k_blocks = p.k_blocks; L.vecC = p.vecC; L.alpha = p.alpha; L.beta = p.beta;
    L.a_mn = p.a_mn; L.b_mn = p.b_mn; L.seg_blocks = p.seg_blocks; L.seg_map = p.seg_map;
    tile_coords(p, tile, L.b, L.tm, L.tn);
  }
  return L;
}

// Stores one 32 x 32 chunk of C (rows row0 + lane of this warp's 32-row
// quadrant, columns n0 .. n0 + 31) from the registers of tcgen05.ld, where
// lane t holds row t.  When every row of C starts on 32 bytes, each lane writes
// whole 32-byte sectors of its own row.  Otherwise SC (16 or 32) columns at a
// time go through this warp's staging buffer (the 16-byte piece q of row t sits
// at q ^ t, or q ^ (t / 2) within 64-byte rows, so both passes are free of bank
// conflicts) and leave as contiguous runs of a row: 16 bytes a lane where C
// allows it, else 4.  beta != 0 reads C the same way.  Together with the second
// epilogue warp per quadrant this took f32mix 1733 x 912 x 1408 x 2 from 77 to 48
// us, an uneven BF16 group of 256 from 509 to 443 and, with rows of 637 floats,
// BF16 2185 x 637 x 95 x 16 from 87 to 63 (its lanes wrote 4 bytes every 16).
// RUNS: rows on 32 bytes go through the staging buffer too unless C is read
// (the CTA-pair tiles: 128-byte runs took BF16 3634 x 1712 x 408 x 8 from 68 to 58
// us; with beta != 0, f32mix 1733 x 912 x 1408 x 2, they took 54 us against 45, and
// an uneven group of 128-row tiles 446 against 428).
template <int SC, bool RUNS = false>
__device__ __forceinline__ void store_chunk32(const TileLoc& p, float* cbase, int row0, int n0, float* stage,
                                              const uint32_t (&r)[32], int lane) {
  if (p.vecC == 2 && n0 + 32 <= p.N && !(RUNS && p.beta == 0.f)) {
    if (row0 + lane >= p.M) return;
    float* dst = cbase + (int64_t)(row0 + lane) * p.ldc + n0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float o[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) o[e] = p.alpha * __uint_as_float(r[8 * q + e]);
      if (p.beta != 0.f) {
        const float4 c0 = *reinterpret_cast<const float4*>(dst + 8 * q);
        const float4 c1 = *reinterpret_cast<const float4*>(dst + 8 * q + 4);
        o[0] = fmaf(p.beta, c0.x, o[0]); o[1] = fmaf(p.beta, c0.y, o[1]);
        o[2] = fmaf(p.beta, c0.z, o[2]); o[3] = fmaf(p.beta, c0.w, o[3]);
        o[4] = fmaf(p.beta, c1.x, o[4]); o[5] = fmaf(p.beta, c1.y, o[5]);
        o[6] = fmaf(p.beta, c1.z, o[6]); o[7] = fmaf(p.beta, c1.w, o[7]);
      }
      asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + 8 * q), "f"(o[0]),
                   "f"(o[1]), "f"(o[2]), "f"(o[3]), "f"(o[4]), "f"(o[5]), "f"(o[6]), "f"(o[7])
                   : "memory");
    }
    return;
  }
  constexpr int P = SC / 4;              // 16-byte pieces of a staged row
  constexpr int SH = SC == 16 ? 1 : 0;   // rows that share a 128-byte line, as a shift
#pragma unroll
  for (int h = 0; h < 32 / SC; ++h) {
#pragma unroll
    for (int q = 0; q < P; ++q) {
      const int c = SC * h + 4 * q;
      const float4 v = make_float4(__uint_as_float(r[c]), __uint_as_float(r[c + 1]), __uint_as_float(r[c + 2]),
                                   __uint_as_float(r[c + 3]));
      *reinterpret_cast<float4*>(stage + lane * SC + ((q ^ ((lane >> SH) & (P - 1))) << 2)) = v;
    }
    __syncwarp();
    if (p.vecC) {
      const int q = lane & (P - 1), n = n0 + SC * h + 4 * q;
#pragma unroll 2
      for (int i = 0; i < P; ++i) {
        const int rr = (32 / P) * i + lane / P, row = row0 + rr;
        const float4 v = *reinterpret_cast<const float4*>(stage + rr * SC + ((q ^ ((rr >> SH) & (P - 1))) << 2));
        if (row >= p.M || n >= p.N) continue;
        float* crow = cbase + (int64_t)row * p.ldc;
        if (n + 3 < p.N) {
          float4 o = make_float4(p.alpha * v.x, p.alpha * v.y, p.alpha * v.z, p.alpha * v.w);
          if (p.beta != 0.f) {
            const float4 c = *reinterpret_cast<const float4*>(crow + n);
            o.x = fmaf(p.beta, c.x, o.x); o.y = fmaf(p.beta, c.y, o.y);
            o.z = fmaf(p.beta, c.z, o.z); o.w = fmaf(p.beta, c.w, o.w);
          }
          *reinterpret_cast<float4*>(crow + n) = o;
        } else {
          const float e4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (n + e < p.N) {
              float o = p.alpha * e4[e];
              if (p.beta != 0.f) o = fmaf(p.beta, crow[n + e], o);
              crow[n + e] = o;
            }
          }
        }
      }
    } else {
      const int c = lane & (SC - 1), n = n0 + SC * h + c;
#pragma unroll 4
      for (int i = 0; i < SC; ++i) {
        const int rr = (32 / SC) * i + lane / SC, row = row0 + rr;
        const float v = stage[rr * SC + (((c >> 2) ^ ((rr >> SH) & (P - 1))) << 2) + (c & 3)];
        if (row < p.M && n < p.N) {
          float* dst = cbase + (int64_t)row * p.ldc + n;
          float o = p.alpha * v;
          if (p.beta != 0.f) o = fmaf(p.beta, *dst, o);
          *dst = o;
        }
      }
    }
    __syncwarp();  // the staging buffer is refilled by the next part
  }
}

template <int BN, int STAGES, bool TF32, bool GROUPED>
__global__ void __launch_bounds__(TcCfg<BN, STAGES, TF32>::THREADS, 1)
    tc_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const TcArgs p,
                   const GroupArgs g) {
  using Cfg = TcCfg<BN, STAGES, TF32>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full_bar[STAGES], empty_bar[STAGES], accf_bar[2], acce_bar[2];
  __shared__ uint32_t tmem_base_sh;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int unit0 = (int)blockIdx.x;
  const int units = (int)gridDim.x;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&accf_bar[a], 1);
      mbar_init(&acce_bar[a], 32 * Cfg::EPI_WARPS);
    }
    fence_barrier_init();
  }
  if (!GROUPED && warp == Cfg::EPI_WARPS && lane == 0) {
    tma_prefetch(&tmA);
    tma_prefetch(&tmB);
  }
  if (warp == Cfg::EPI_WARPS + 1) tmem_alloc<Cfg::TMEM_COLS>(&tmem_base_sh);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_sh;
  // The prologue above (barriers, TMEM, tensor-map prefetch) touches no global
  // memory, so it may overlap the previous kernel's tail.
  pdl_wait();
  pdl_launch_dependents();
  __shared__ int starts_sh[GROUPED ? kStarts : 1];
  GroupIndex index{starts_sh, 0, 1};
  if constexpr (GROUPED) {
    index.step = (g.count + kStarts - 1) / kStarts;
    index.n = (g.count + index.step - 1) / index.step;
    for (int i = threadIdx.x; i < index.n; i += Cfg::THREADS) starts_sh[i] = g.descs[i * index.step].tile_start;
    __syncthreads();
  }

  if (warp == Cfg::EPI_WARPS) {
    // ---------------------------------------------------------------- TMA producer
    if (elect_one()) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int tile = unit0; tile < p.num_tiles && ok; tile += units) {
        const TileLoc L = locate<GROUPED>(p, g, index, &tmA, &tmB, tile);
        for (int kb = 0; kb < L.k_blocks; ++kb) {
          if (!(ok = mbar_wait(&empty_bar[stage], phase ^ 1, p.status, kStatusTimeoutEmpty))) break;
          uint8_t* sa = smem + stage * Cfg::STAGE_BYTES;
          // K coordinates of this slice in A and B (split products: segment g
          // of the K' loop reads the parts of A and B that seg_map names).
          int xa = kb * Cfg::BK, xb = kb * Cfg::BK;
          if (!TF32 && L.seg_blocks > 0) {
            const int g = kb / L.seg_blocks, kk = kb - g * L.seg_blocks;
            xa = (((L.seg_map >> (2 * g)) & 3) * L.seg_blocks + kk) * Cfg::BK;
            xb = (((L.seg_map >> (16 + 2 * g)) & 3) * L.seg_blocks + kk) * Cfg::BK;
          }
          mbar_arrive_expect_tx(&full_bar[stage], Cfg::STAGE_BYTES);
          if (L.a_mn) {
#pragma unroll
            for (int j = 0; j < kBM / Cfg::MN_BOX; ++j)
              tma_load_3d(sa + j * Cfg::MN_BOX_BYTES, L.ma, &full_bar[stage], L.tm * kBM + j * Cfg::MN_BOX, xa,
                          L.b);
          } else {
            tma_load_3d(sa, L.ma, &full_bar[stage], xa, L.tm * kBM, L.b);
          }
          if (L.b_mn) {
#pragma unroll
            for (int j = 0; j < BN / Cfg::MN_BOX; ++j)
              tma_load_3d(sa + Cfg::A_BYTES + j * Cfg::MN_BOX_BYTES, L.mb, &full_bar[stage],
                          L.tn * BN + j * Cfg::MN_BOX, xb, L.b);
          } else {
            tma_load_3d(sa + Cfg::A_BYTES, L.mb, &full_bar[stage], xb, L.tn * BN, L.b);
          }
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1;
          }
        }
      }
      // Wait (bounded) until every issued slice has landed before the CTA can exit.
      if (ok) {
        for (int s = 0; s < STAGES; ++s) {
          if (!mbar_wait(&empty_bar[stage], phase ^ 1, p.status, kStatusTimeoutEmpty)) break;
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1;
          }
        }
      }
    }
  } else if (warp == Cfg::EPI_WARPS + 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (elect_one()) {
      int stage = 0;
      uint32_t phase = 0;
      int acc = 0;
      uint32_t acc_phase = 0;
      bool ok = true;
      for (int tile = unit0; tile < p.num_tiles && ok; tile += units) {
        int k_blocks = p.k_blocks, a_mn = p.a_mn, b_mn = p.b_mn;
        if constexpr (GROUPED) {
          const TileLoc L = locate<true>(p, g, index, &tmA, &tmB, tile);
          k_blocks = L.k_blocks;
          a_mn = L.a_mn;
          b_mn = L.b_mn;
        }
        const uint32_t idesc = instr_desc<TF32>(kBM, BN, a_mn != 0, b_mn != 0);
        // K-major: the next MMA's K range starts KMMA elements along the swizzled
        // 128-byte row; MN-major: KMMA K rows further on, MN blocks MN_BOX_BYTES apart.
        const uint32_t a_step = a_mn ? Cfg::KMMA * 128 : Cfg::KMMA * Cfg::ELEM;
        const uint32_t b_step = b_mn ? Cfg::KMMA * 128 : Cfg::KMMA * Cfg::ELEM;
        const uint32_t a_lbo = a_mn ? Cfg::MN_BOX_BYTES : 16;
        const uint32_t b_lbo = b_mn ? Cfg::MN_BOX_BYTES : 16;
        if (!(ok = mbar_wait(&acce_bar[acc], acc_phase ^ 1, p.status, kStatusTimeoutAccEmpty))) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
        for (int kb = 0; kb < k_blocks; ++kb) {
          if (!(ok = mbar_wait(&full_bar[stage], phase, p.status, kStatusTimeoutFull))) break;
          tc_fence_after();
          const uint32_t a_addr = smem_u32(smem + stage * Cfg::STAGE_BYTES);
          const uint32_t b_addr = a_addr + Cfg::A_BYTES;
#pragma unroll
          for (int k = 0; k < Cfg::BK / Cfg::KMMA; ++k) {
            const uint64_t ad = a_mn ? smem_desc_sw128(a_addr + (uint32_t)k * a_step, a_lbo, Cfg::MN_SBO, Cfg::MN_MODE)
                                     : smem_desc_sw128(a_addr + (uint32_t)k * a_step, a_lbo, 1024);
            const uint64_t bd = b_mn ? smem_desc_sw128(b_addr + (uint32_t)k * b_step, b_lbo, Cfg::MN_SBO, Cfg::MN_MODE)
                                     : smem_desc_sw128(b_addr + (uint32_t)k * b_step, b_lbo, 1024);
            mma<TF32>(d_tmem, ad, bd, idesc, (kb | k) != 0 ? 1u : 0u);
          }
          mma_commit(&empty_bar[stage]);  // frees the slot once these MMAs have read it
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1;
          }
        }
        if (!ok) break;
        mma_commit(&accf_bar[acc]);  // accumulator complete
        if (++acc == 2) {
          acc = 0;
          acc_phase ^= 1;
        }
      }
    }
  } else {
    // ---------------------------------------------------------------- epilogue (warps 0..EPI_WARPS - 1)
    int acc = 0;
    uint32_t acc_phase = 0;
    for (int tile = unit0; tile < p.num_tiles; tile += units) {
      const bool ok = mbar_wait(&accf_bar[acc], acc_phase, p.status, kStatusTimeoutAcc);
      if (!__all_sync(0xffffffffu, ok)) break;  // a warp's lanes go on, or give up, together
      tc_fence_after();
      const TileLoc L = locate<GROUPED>(p, g, index, &tmA, &tmB, tile);
      const int quad = warp & 3, row0 = L.tm * kBM + quad * 32;
      constexpr int COLS = BN / (Cfg::EPI_WARPS / 4);  // columns of this warp
      const int col0 = (warp >> 2) * COLS;
      float* cbase = L.C + (int64_t)L.b * L.strideC;
      float* stage = reinterpret_cast<float*>(smem + STAGES * Cfg::STAGE_BYTES) + warp * 32 * Cfg::STORE_COLS;
      const uint32_t tbase = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * BN);
#pragma unroll 1
      for (int c0 = col0; c0 < col0 + COLS; c0 += 32) {
        uint32_t r[32];
        tmem_ld_32x32b_x32(tbase + (uint32_t)c0, r);
        tmem_ld_wait();
        if (row0 < L.M && L.tn * BN + c0 < L.N)
          store_chunk32<Cfg::STORE_COLS>(L, cbase, row0, L.tn * BN + c0, stage, r, lane);
        __syncwarp();  // lanes past M return early; the next load and the fence want the whole warp
      }
      tc_fence_before();
      mbar_arrive(&acce_bar[acc]);
      if (++acc == 2) {
        acc = 0;
        acc_phase ^= 1;
      }
    }
  }

  __syncthreads();
  if (warp == Cfg::EPI_WARPS + 1) {
    tc_fence_after();
    tmem_dealloc<Cfg::TMEM_COLS>(tmem_base);
  }
}

// ---------------------------------------------------------------- two CTAs on one 256 x 256 tile
// The same with tcgen05's cta_group::2: each CTA of the pair loads its 128 rows
// of A and its 128 of B and holds its 128 rows' accumulators; the first CTA
// issues MMAs that read both CTAs' shared memory.  A slice of K then costs an SM
// 32 KB of loads and shared memory instead of 48 for the same products, which
// leaves room for six stages.  What bounds the 128 x 256 tiles is feeding the
// MMAs (36 % tensor-pipe time at 3634 x 1714 x 406 x 8 TF32).  BF16 8192 cubed A B^T
// 685 -> 575 us (1,910 TFLOP/s), A B 672 -> 535; 4096 cubed 100 -> 80; TF32 8192
// cubed 1360 -> 1060; TF32 3634 x 1714 x 406 x 8 102 -> 86.  Same bits.
template <bool TF32>
struct PairCfg {
  static constexpr int ELEM = TF32 ? 4 : 2;
  static constexpr int BM = 256, BN = 256, HALF = 128;
  static constexpr int BK = 128 / ELEM, KMMA = TF32 ? 8 : 16;
  static constexpr int PART = HALF * 128;  // bytes of one operand's half slice
  static constexpr int STAGE_BYTES = 2 * PART, STAGES = 6;
  static constexpr int EPI_WARPS = 8, THREADS = 32 * (EPI_WARPS + 2);
  static constexpr int STORE_COLS = 32, EPI_BYTES = EPI_WARPS * 32 * STORE_COLS * 4;
  static constexpr int TMEM_COLS = 2 * BN;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + EPI_BYTES + 1024;
  static constexpr int MN_BOX = 128 / ELEM, MN_BOX_BYTES = BK * 128;
  static constexpr uint32_t MN_SBO = TF32 ? 512 : 1024;
  static constexpr uint32_t MN_MODE = TF32 ? kSw128Atom32 : kSw128;
};

template <bool TF32>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PairCfg<TF32>::THREADS, 1)
    tc_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const TcArgs p) {
  using Cfg = PairCfg<TF32>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full_bar[Cfg::STAGES], empty_bar[Cfg::STAGES], accf_bar[2], acce_bar[2];
  __shared__ uint32_t tmem_base_sh;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank();
  const int unit0 = (int)blockIdx.x >> 1, units = (int)gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < Cfg::STAGES; ++s) {
      mbar_init(&full_bar[s], 1);  // used in the first CTA, for both CTAs' loads
      mbar_init(&empty_bar[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&accf_bar[a], 1);
      mbar_init(&acce_bar[a], 2 * Cfg::EPI_WARPS);  // used in the first CTA
    }
    fence_barrier_init();
  }
  if (warp == Cfg::EPI_WARPS && lane == 0) {
    tma_prefetch(&tmA);
    tma_prefetch(&tmB);
  }
  if (warp == Cfg::EPI_WARPS + 1) tmem_alloc_pair<Cfg::TMEM_COLS>(&tmem_base_sh);
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_sh;
  pdl_wait();
  pdl_launch_dependents();

  if (warp == Cfg::EPI_WARPS) {
    if (elect_one()) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int tile = unit0; tile < p.num_tiles && ok; tile += units) {
        int b, tm, tn;
        tile_coords(p, tile, b, tm, tn);
        const int row = tm * Cfg::BM + rank * Cfg::HALF, col = tn * Cfg::BN + rank * Cfg::HALF;
        for (int kb = 0; kb < p.k_blocks; ++kb) {
          // Freed in both CTAs at once; the first CTA's full barrier is then in this
          // slice's phase, so the other's bytes may be counted before they are expected.
          if (!(ok = mbar_wait(&empty_bar[stage], phase ^ 1, p.status, kStatusTimeoutEmpty))) break;
          uint8_t* sa = smem + stage * Cfg::STAGE_BYTES;
          uint8_t* sb = sa + Cfg::PART;
          int xa = kb * Cfg::BK, xb = kb * Cfg::BK;
          if (!TF32 && p.seg_blocks > 0) {
            const int g = kb / p.seg_blocks, kk = kb - g * p.seg_blocks;
            xa = (((p.seg_map >> (2 * g)) & 3) * p.seg_blocks + kk) * Cfg::BK;
            xb = (((p.seg_map >> (16 + 2 * g)) & 3) * p.seg_blocks + kk) * Cfg::BK;
          }
          const uint32_t bar = in_cta(smem_u32(&full_bar[stage]), 0);
          if (rank == 0) mbar_arrive_expect_tx(&full_bar[stage], 2 * Cfg::STAGE_BYTES);
          if (p.a_mn) {
#pragma unroll
            for (int j = 0; j < Cfg::HALF / Cfg::MN_BOX; ++j)
              tma_load_3d_pair(sa + j * Cfg::MN_BOX_BYTES, &tmA, bar, row + j * Cfg::MN_BOX, xa, b);
          } else {
            tma_load_3d_pair(sa, &tmA, bar, xa, row, b);
          }
          if (p.b_mn) {
#pragma unroll
            for (int j = 0; j < Cfg::HALF / Cfg::MN_BOX; ++j)
              tma_load_3d_pair(sb + j * Cfg::MN_BOX_BYTES, &tmB, bar, col + j * Cfg::MN_BOX, xb, b);
          } else {
            tma_load_3d_pair(sb, &tmB, bar, xb, col, b);
          }
          if (++stage == Cfg::STAGES) {
            stage = 0;
            phase ^= 1;
          }
        }
      }
      // Wait (bounded) until every issued slice has been read before the CTA can exit.
      if (ok) {
        for (int s = 0; s < Cfg::STAGES; ++s) {
          if (!mbar_wait(&empty_bar[stage], phase ^ 1, p.status, kStatusTimeoutEmpty)) break;
          if (++stage == Cfg::STAGES) {
            stage = 0;
            phase ^= 1;
          }
        }
      }
    }
  } else if (warp == Cfg::EPI_WARPS + 1) {
    if (rank == 0 && elect_one()) {
      const uint32_t idesc = instr_desc<TF32>(Cfg::BM, Cfg::BN, p.a_mn != 0, p.b_mn != 0);
      const uint32_t a_step = p.a_mn ? Cfg::KMMA * 128 : Cfg::KMMA * Cfg::ELEM;
      const uint32_t b_step = p.b_mn ? Cfg::KMMA * 128 : Cfg::KMMA * Cfg::ELEM;
      const uint32_t a_lbo = p.a_mn ? Cfg::MN_BOX_BYTES : 16, b_lbo = p.b_mn ? Cfg::MN_BOX_BYTES : 16;
      const uint32_t a_sbo = p.a_mn ? Cfg::MN_SBO : 1024, b_sbo = p.b_mn ? Cfg::MN_SBO : 1024;
      const uint32_t a_mode = p.a_mn ? Cfg::MN_MODE : kSw128, b_mode = p.b_mn ? Cfg::MN_MODE : kSw128;
      int stage = 0, acc = 0;
      uint32_t phase = 0, acc_phase = 0;
      bool ok = true;
      for (int tile = unit0; tile < p.num_tiles && ok; tile += units) {
        if (!(ok = mbar_wait(&acce_bar[acc], acc_phase ^ 1, p.status, kStatusTimeoutAccEmpty))) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * Cfg::BN);
        for (int kb = 0; kb < p.k_blocks; ++kb) {
          if (!(ok = mbar_wait(&full_bar[stage], phase, p.status, kStatusTimeoutFull))) break;
          tc_fence_after();
          const uint32_t a_addr = smem_u32(smem + stage * Cfg::STAGE_BYTES), b_addr = a_addr + Cfg::PART;
#pragma unroll
          for (int k = 0; k < Cfg::BK / Cfg::KMMA; ++k)
            mma_pair<TF32>(d_tmem, smem_desc_sw128(a_addr + (uint32_t)k * a_step, a_lbo, a_sbo, a_mode),
                           smem_desc_sw128(b_addr + (uint32_t)k * b_step, b_lbo, b_sbo, b_mode), idesc,
                           (kb | k) != 0 ? 1u : 0u);
          commit_pair(&empty_bar[stage]);
          if (++stage == Cfg::STAGES) {
            stage = 0;
            phase ^= 1;
          }
        }
        if (!ok) break;
        commit_pair(&accf_bar[acc]);
        if (++acc == 2) {
          acc = 0;
          acc_phase ^= 1;
        }
      }
    }
  } else {
    const int quad = warp & 3, half = warp >> 2;
    float* stage = reinterpret_cast<float*>(smem + Cfg::STAGES * Cfg::STAGE_BYTES) + warp * 32 * Cfg::STORE_COLS;
    TileLoc L;
    L.ldc = p.ldc; L.M = p.M; L.N = p.N; L.vecC = p.vecC; L.alpha = p.alpha; L.beta = p.beta;
    int acc = 0;
    uint32_t acc_phase = 0;
    for (int tile = unit0; tile < p.num_tiles; tile += units) {
      const bool ok = mbar_wait(&accf_bar[acc], acc_phase, p.status, kStatusTimeoutAcc);
      if (!__all_sync(0xffffffffu, ok)) break;  // a warp's lanes go on, or give up, together
      tc_fence_after();
      int b, tm, tn;
      tile_coords(p, tile, b, tm, tn);
      const int row0 = tm * Cfg::BM + rank * Cfg::HALF + quad * 32;
      float* cbase = p.C + (int64_t)b * p.strideC;
      const uint32_t tbase = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * Cfg::BN);
#pragma unroll 1
      for (int c0 = half * Cfg::HALF; c0 < (half + 1) * Cfg::HALF; c0 += 32) {
        uint32_t r[32];
        tmem_ld_32x32b_x32(tbase + (uint32_t)c0, r);
        tmem_ld_wait();
        if (row0 < p.M && tn * Cfg::BN + c0 < p.N)
          store_chunk32<Cfg::STORE_COLS, true>(L, cbase, row0, tn * Cfg::BN + c0, stage, r, lane);
        __syncwarp();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) arrive_cluster(in_cta(smem_u32(&acce_bar[acc]), 0));
      if (++acc == 2) {
        acc = 0;
        acc_phase ^= 1;
      }
    }
  }

  __syncthreads();
  cluster_sync();  // neither CTA leaves while the other's loads, MMAs or arrivals may reach it
  if (warp == Cfg::EPI_WARPS + 1) {
    tc_fence_after();
    tmem_dealloc_pair<Cfg::TMEM_COLS>(tmem_base);
  }
}

}  // namespace tc
}  // namespace ks
