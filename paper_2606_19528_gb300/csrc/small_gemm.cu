// Fused LoRA contraction for few tokens (at most 128 rows), tcgen05, sm_103a:
// the products of fused_gemm.cu,
//     y[T, N]  = [x | su] . [W | B]^T      and      dx[T, K] = [dy | sv] . [W ; A],
// with W in bf16 or as 4-bit codes dequantized on the fly.
//
// With so few rows the weight stream bounds the contraction: bytes from HBM
// with bf16 weights, and with 4-bit weights the MMAs' issue and the
// dequantization.  The CTA pairs of fused_gemm.cu give every 256-row MMA at
// least 128 empty rows, so half their tensor time is spent on padding, and their
// 256 x 512 tiles leave 76 workers with unequal shares.  Here every CTA works by
// itself: a 128 x 256 tile, one M = 128, N = 256, K = 16 MMA per 16-deep step
// (512 tensor cycles per 64-deep block of 256 weight columns, where a pair's
// CTA takes 1024), only the rows that exist loaded, 152 workers, and two TMEM
// accumulators so that a tile's epilogue runs under the next tile's MMAs.
// Against the pairs, in the same calls: Llama-shaped layer forward at T = 32
// (201 MB of bf16 weights) 48.6 -> 43.2 us, forward and backward at T = 64 with
// 4-bit weights 124 -> 91 us, Qwen-shaped layer forward and backward at T = 32,
// r = 4 117 -> 95 us; with what came after (contractions that start beside the
// rank-r products, clusters, su^T and B^T made earlier) 41.7, 82 and 86 us.  From 129
// rows on, a pair's MMAs are as full as a CTA's.
//   warp 0      tile scheduler and TMA producer: 4 stages of [activation 16 KB |
//               weight 32 KB] (4-bit: 3 stages; the weight part is dequantized)
//   warp 1      TMEM allocation; tcgen05.mma issuer (one elected lane)
//   warps 2..9  epilogue: TMEM -> registers -> bf16 (or the fp32 partial of a
//               split) -> swizzled shared-memory block -> TMA store
//               (warps 2..5 with 4-bit weights)
//   4-bit:      warps 6..13 dequantize, two groups of four taking alternate
//               blocks; warp 14 streams codes and (s, b) pairs by TMA
// Every wait is bounded.
//
// Cluster form (kCl), for launches whose tiles leave most CTAs idle (one
// projection): a cluster of S = 2, 4 or 8 CTAs shares a tile, CTA j contracting
// the j-th part of its blocks.  Then every CTA's ring is idle and the parts are
// summed through distributed shared memory: CTA j owns 256 / S of the tile's
// columns, gets the other CTAs' fp32 values for them by bulk copies, adds them
// in CTA order, rounds once and stores.  No partials in memory, no reduce
// launch, and a forward without a workspace gives the same bits.
#include "common.cuh"
#include "kernels.h"

namespace lora {

namespace {

constexpr int kM = 128;                      // tile rows: TMEM lanes
constexpr int kN = 256;                      // tile columns
constexpr int kBK = 64;
constexpr uint32_t kABytes = kM * kBK * 2;   // 16 KB
constexpr uint32_t kWBytes = kN * kBK * 2;   // 32 KB
constexpr uint32_t kBox = 64 * kBK * 2;      // one 64-column box of an MN-major weight tile, 8 KB
constexpr uint32_t kStage = kABytes + kWBytes;
constexpr uint32_t kEpiStage = 32 * 128;     // per-warp output block, 4 KB
constexpr uint32_t kTmemCols = 512;
constexpr int kConvWarps = 8, kConvGroups = 2, kGroupWarps = kConvWarps / kConvGroups;
constexpr int kTileRing = 4;
constexpr int kMaxStages = 4;
constexpr int kQMaxStages = 6;
constexpr long long kDrainNs = 1000000000ll;
constexpr long long kAbortDrainNs = 10000000ll;  // 10 ms per armed stage on the abort path

// 4-bit code slots.  Forward: 2 contraction blocks of 256 weight rows (64
// code bytes a row, 64-byte swizzle) and the rows' 4 (s, b) groups around them.
// Backward: one block, 64 contraction rows of 256 columns (128 bytes a row,
// 128-byte swizzle) and their 4 groups.
template <bool kBMn>
struct QSlot {
  static constexpr int kBlocks = kBMn ? 1 : 2;
  static constexpr uint32_t kCodes = kBMn ? 8192 : 16384;
  static constexpr uint32_t kParams = kBMn ? 1024 : 4096;
  static constexpr uint32_t kBytes = kCodes + kParams;
  static constexpr int kStages = kBMn ? 6 : 3;
  static_assert(kStages <= kQMaxStages && kBytes % 1024 == 0, "code slots");
};
constexpr uint32_t kQRing = 61440;

template <bool kQ>
struct Cfg {
  static constexpr int kStages = kQ ? 3 : 4;
  static constexpr int kEpi = kQ ? 4 : 8;
  static constexpr int kPartCols = kN / (kEpi / 4);  // columns of a tile per epilogue warp
  static constexpr uint32_t kRing = kStages * kStage + (kQ ? kQRing : 0);
  static constexpr int kThreads = (2 + kEpi + (kQ ? kConvWarps + 1 : 0)) * 32;
};
static_assert(QSlot<false>::kStages * QSlot<false>::kBytes <= kQRing, "forward code slots");
static_assert(QSlot<true>::kStages * QSlot<true>::kBytes <= kQRing, "backward code slots");

struct __align__(8) Ctl {
  uint64_t full[kMaxStages];       // a stage's TMA boxes landed
  uint64_t wfull[kMaxStages];      // 4-bit: a stage's weight tile dequantized (adapter block: landed)
  uint64_t empty[kMaxStages];      // the MMAs finished reading a stage
  uint64_t qfull[kQMaxStages];     // 4-bit: codes and (s, b) of a slot landed
  uint64_t qempty[kQMaxStages];    // 4-bit: every dequantizing warp is past a slot
  uint64_t tfull[2], tempty[2];    // accumulator complete / drained
  uint64_t tile_full[kTileRing], tile_empty[kTileRing];
  uint64_t drain;
  uint64_t xchg;                   // kCl: the other CTAs' values of this CTA's columns arrived
  int tile_id[kTileRing];
  uint32_t tmem_base;
  int abort;
  int fills, qfills;
};

template <bool kQ>
constexpr size_t smem_bytes() {
  return 1024 + (size_t)Cfg<kQ>::kRing + (size_t)Cfg<kQ>::kEpi * kEpiStage + sizeof(Ctl);
}
static_assert(smem_bytes<true>() <= 232448 && smem_bytes<false>() <= 232448, "shared memory of a CTA");

// Problem p, first column n0 of tile t, its split ks and blocks [kb0, kb1) (one row tile per problem).
struct Tile {
  int p, n0, ks, kb0, kb1;
};
__device__ __forceinline__ Tile decode(const GemmBatch& b, int t) {
  Tile w;
  w.p = 0;
  while (w.p + 1 < b.num_problems && t >= b.prob[w.p + 1].tile_begin) ++w.p;
  const GemmProblem& Q = b.prob[w.p];
  const int local = t - Q.tile_begin;
  w.ks = local / Q.num_n_tiles;
  w.n0 = (local - w.ks * Q.num_n_tiles) * kN;
  w.kb0 = w.ks * Q.kb_split;
  w.kb1 = min(Q.kb_total, w.kb0 + Q.kb_split);
  return w;
}

// Dequantizes one contraction block of the tile's 256 weight columns from a
// code slot into the 128-byte-swizzled operand layout.  Forward: row r (0..255)
// is W row n0 + r, its codes 32 bytes of the slot's 64-byte row (16-byte chunk u
// at u ^ (r / 2 mod 4)).  Backward: row r (0..63) is W row 64 kb + r, its codes
// 128 bytes (chunk u at u ^ (r mod 8)), two chunks per 64-column box.  A thread
// takes 16-byte chunks (32 codes); lanes are ordered so that a quarter warp's
// loads and stores each fall on the eight bank groups once.
template <bool kBMn>
__device__ __forceinline__ void dequant_block(uint32_t slot, uint32_t wdst, int ct, int n0, int kb, int ncols) {
  constexpr int kThr = kGroupWarps * 32;
  const uint32_t params = slot + QSlot<kBMn>::kCodes;
#pragma unroll
  for (int rep = 0; rep < 512 / kThr; ++rep) {
    const int hu = ct + rep * kThr;
    uint32_t csrc, psrc, dst_row;
    int half, sw;
    if (kBMn) {
      const int r = (hu >> 6) * 8 + (hu & 7), u = (hu >> 3) & 7, j = u >> 1;
      if (n0 + j * 64 >= ncols) continue;  // never stored
      half = u & 1;
      sw = r & 7;
      csrc = slot + (uint32_t)(r * 128 + ((u ^ sw) << 4));
      psrc = params + (uint32_t)(r * 16 + j * 4);
      dst_row = wdst + (uint32_t)(j * kBox + r * 128);
    } else {
      const int r = (hu >> 4) * 8 + (hu & 7);
      if (n0 + r >= ncols) continue;
      half = (hu >> 3) & 1;
      sw = r & 7;
      const int u = (kb & 1) * 2 + half;
      csrc = slot + (uint32_t)(r * 64 + ((u ^ ((r >> 1) & 3)) << 4));
      psrc = params + (uint32_t)(r * 16 + (kb & 3) * 4);
      dst_row = wdst + (uint32_t)(r * 128);
    }
    uint32_t w[4], sb;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(csrc) : "memory");
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(sb) : "r"(psrc) : "memory");
    const uint32_t s2 = (sb & 0xFFFFu) * 0x10001u, b2 = (sb >> 16) * 0x10001u;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const uint32_t o0 = dq_pair(w[m], s2, b2), o1 = dq_pair(w[m] >> 4, s2, b2);
      const uint32_t o2 = dq_pair(w[m] >> 8, s2, b2), o3 = dq_pair(w[m] >> 12, s2, b2);
      const uint32_t dst = dst_row + (uint32_t)((((half * 4 + m) ^ sw) & 7) << 4);
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(o0), "r"(o1), "r"(o2), "r"(o3)
                   : "memory");
    }
  }
}

template <bool kBMn, bool kQ, bool kCl>
__global__ void __launch_bounds__(Cfg<kQ>::kThreads, 1) small_lora_gemm(const __grid_constant__ GemmBatch b) {
  using C = Cfg<kQ>;
  using QS = QSlot<kBMn>;
  constexpr int kStages = C::kStages, kEpi = C::kEpi;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  const uint32_t epi_base = base + C::kRing;
  Ctl* ctl = reinterpret_cast<Ctl*>(smem_raw + (base - raw) + (size_t)C::kRing + (size_t)kEpi * kEpiStage);
  volatile int* abort_flag = &ctl->abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const WaitCtl wc{b.status, b.limit_ns};
  auto a_tile = [&](int s) { return base + (uint32_t)s * kStage; };
  auto w_tile = [&](int s) { return base + (uint32_t)s * kStage + kABytes; };
  auto q_slot = [&](int s) { return base + kStages * kStage + (uint32_t)s * QS::kBytes; };

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&ctl->full[s]), 1);
      mbar_init(smem_u32(&ctl->wfull[s]), kGroupWarps);
      mbar_init(smem_u32(&ctl->empty[s]), 1);
    }
    for (int q = 0; q < QS::kStages; ++q) {
      mbar_init(smem_u32(&ctl->qfull[q]), 1);
      mbar_init(smem_u32(&ctl->qempty[q]), kConvWarps);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(smem_u32(&ctl->tfull[h]), 1);
      mbar_init(smem_u32(&ctl->tempty[h]), kEpi);
    }
    for (int k = 0; k < kTileRing; ++k) {
      mbar_init(smem_u32(&ctl->tile_full[k]), 1);
      mbar_init(smem_u32(&ctl->tile_empty[k]), 1 + kEpi + (kQ ? kConvWarps + 1 : 0));
    }
    mbar_init(smem_u32(&ctl->drain), 1);
    mbar_init(smem_u32(&ctl->xchg), 1);
    ctl->abort = 0;
    ctl->fills = 0;
    ctl->qfills = 0;
    fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    for (int q = 0; q < b.num_problems; ++q) {
      tma_prefetch_desc(&b.tmA[q]);
      tma_prefetch_desc(kQ ? &b.tmQ[q] : &b.tmB[q]);
    }
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&ctl->tmem_base), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // with early inputs only the producers of the adapter slab wait for the previous grid, and every CTA before it ends
  if (!b.early_inputs) griddep_wait();
  const uint32_t tmem_base = ctl->tmem_base;
  // kCl: cluster size, this CTA's part of the tile's blocks
  const int S = kCl ? b.cluster : 1;
  const int crank = kCl ? (int)cluster_ctarank() : 0;
  auto tile_of = [&](int t) {
    Tile w = decode(b, t);
    if (kCl) {
      const int kt = b.prob[w.p].kb_total, L = (kt + S - 1) / S;
      w.kb0 = crank * L;
      w.kb1 = min(kt, w.kb0 + L);
    }
    return w;
  };

  // tile of the consumers' iteration `it`, or -1 (all tiles done, or a wait gave up); whole warps call it
  auto next_tile = [&](int it) {
    const int slot = it % kTileRing;
    bool got = mbar_wait(smem_u32(&ctl->tile_full[slot]), (uint32_t)((it / kTileRing) & 1), wc, abort_flag);
    got = __all_sync(0xffffffffu, got);
    if (!got) return -1;
    int t = *reinterpret_cast<volatile int*>(&ctl->tile_id[slot]);
    t = __shfl_sync(0xffffffffu, t, 0);
    if (lane == 0) mbar_arrive(smem_u32(&ctl->tile_empty[slot]));
    return t;
  };
  // loads the weight-side boxes of an adapter block (or of a bf16 block) into the tile at dst
  auto load_w = [&](uint32_t dst, const CUtensorMap* m, uint32_t bar, int n0, int N, int kc) {
    if (kBMn) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (n0 + j * 64 < N) tma_load_2d(dst + (uint32_t)j * kBox, m, bar, n0 + j * 64, kc);
    } else {
      tma_load_2d(dst, m, bar, kc, n0);  // 256 rows, zeros past N
    }
  };
  auto w_bytes = [&](int n0, int N) { return kBMn ? (uint32_t)min(4, (N - n0 + 63) / 64) * kBox : kWBytes; };

  if (warp == 0) {
    // ------------------------------------------------------------ scheduler + producer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      int fills = 0;
      bool waited = !b.early_inputs;
      for (int it = 0;; ++it) {
        const int slot = it % kTileRing;
        if (!mbar_wait(smem_u32(&ctl->tile_empty[slot]), (uint32_t)(((it / kTileRing) & 1) ^ 1), wc, abort_flag)) break;
        int t;
        if (kCl)
          t = it == 0 ? (int)blockIdx.x / S : b.total_tiles;
        else if (b.total_tiles <= (int)gridDim.x)  // at most one tile per CTA: no counter
          t = it == 0 ? (int)blockIdx.x : b.total_tiles;
        else
          t = atomicAdd(b.tile_counter, 1);
        if (t >= b.total_tiles) t = -1;
        ctl->tile_id[slot] = t;
        mbar_arrive(smem_u32(&ctl->tile_full[slot]));
        if (t < 0) {
          griddep_launch_dependents();
          break;
        }
        const Tile w = tile_of(t);
        const GemmProblem& Q = b.prob[w.p];
        const uint32_t a_bytes = (uint32_t)((Q.M + 7) & ~7) * 128u;  // the map's box rows
        const uint32_t tx = a_bytes + (kQ ? 0u : w_bytes(w.n0, Q.N));
        bool ok = true;
        for (int kb = w.kb0; kb < w.kb1; ++kb) {
          if (!mbar_wait(smem_u32(&ctl->empty[stage]), phase ^ 1u, wc, abort_flag)) {
            ok = false;
            break;
          }
          const bool main = kb < Q.kb_main;
          if (!main && !waited) {
            griddep_wait();  // su or sv comes from the previous grid
            waited = true;
          }
          const uint32_t bar = smem_u32(&ctl->full[stage]);
          const int kc = main ? kb * kBK : (kb - Q.kb_main) * kBK;
          mbar_arrive_expect_tx(bar, tx);
          ++fills;
          if (!kQ) load_w(w_tile(stage), main ? &b.tmB[w.p] : &b.tmB2[w.p], bar, w.n0, Q.N, kc);
          tma_load_2d(a_tile(stage), main ? &b.tmA[w.p] : &b.tmA2[w.p], bar, kc, 0);
          if (++stage == kStages) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (!ok) break;
      }
      ctl->fills = fills;
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (converged warp, one elected lane)
    constexpr uint32_t idesc = idesc_bf16_f32(kM, kN, 0, kBMn ? 1 : 0);
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int it = 0; ok; ++it) {
      const int t = next_tile(it);
      if (t < 0) break;
      const Tile w = tile_of(t);
      const GemmProblem& Q = b.prob[w.p];
      const int buf = it & 1;
      ok = mbar_wait(smem_u32(&ctl->tempty[buf]), (uint32_t)(((it >> 1) & 1) ^ 1), wc, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const uint32_t d = tmem_base + (uint32_t)(buf * kN);
      for (int kb = w.kb0; kb < w.kb1; ++kb) {
        bool got = mbar_wait(smem_u32(&ctl->full[stage]), phase, wc, abort_flag);
        if (kQ && got) got = mbar_wait(smem_u32(&ctl->wfull[stage]), phase, wc, abort_flag);
        ok = __all_sync(0xffffffffu, got);
        if (!ok) break;
        tc_fence_after();
        const uint64_t ad = sw128_desc(a_tile(stage), 16, 1024);
        const uint64_t bd = kBMn ? sw128_desc(w_tile(stage), kBox, 1024) : sw128_desc(w_tile(stage), 16, 1024);
        const int nk = kb < Q.kb_main ? kBK / 16 : min(kBK / 16, (Q.r - (kb - Q.kb_main) * kBK + 15) / 16);
        if (elect_one()) {
          if (kb != w.kb0 && nk == kBK / 16) {
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k)
              umma_bf16(d, ad + (uint64_t)(2 * k), bd + (uint64_t)((kBMn ? 128 : 2) * k), idesc, 1u);
          } else {
            for (int k = 0; k < nk; ++k)
              umma_bf16(d, ad + (uint64_t)(2 * k), bd + (uint64_t)((kBMn ? 128 : 2) * k), idesc,
                        (kb != w.kb0 || k != 0) ? 1u : 0u);
          }
          umma_commit(smem_u32(&ctl->empty[stage]));
        }
        __syncwarp();
        if (++stage == kStages) {
          stage = 0;
          phase ^= 1u;
        }
      }
      if (!ok) break;
      if (elect_one()) umma_commit(smem_u32(&ctl->tfull[buf]));
      __syncwarp();
    }
    // completes once every MMA issued above has finished
    __syncwarp();
    if (elect_one()) umma_commit(smem_u32(&ctl->drain));
  } else if (warp < 2 + kEpi) {
    // ------------------------------------------------------------ epilogue
    const int q = warp & 3;            // TMEM lane quadrant this warp may access
    const int part = (warp - 2) >> 2;  // which kPartCols columns of the tile
    const uint32_t stg = epi_base + (uint32_t)(warp - 2) * kEpiStage;
    const int row0 = q * 32;
    for (int it = 0;; ++it) {
      const int t = next_tile(it);
      if (t < 0) break;
      const Tile w = tile_of(t);
      const GemmProblem& Q = b.prob[w.p];
      const int buf = it & 1;
      bool ok = mbar_wait(smem_u32(&ctl->tfull[buf]), (uint32_t)((it >> 1) & 1), wc, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      if (kCl) continue;                 // the exchange follows below, after every role
      const bool f32 = Q.splits > 1;  // the fp32 partial of one split: 32-column blocks
      const int block_cols = f32 ? 32 : 64;
      const int row_st = (f32 ? w.ks * Q.m_pad : 0) + row0;
      for (int cc = 0; cc < C::kPartCols; cc += block_cols) {
        const int col = part * C::kPartCols + cc;
        if (w.n0 + col >= Q.N || row0 >= Q.M) break;  // uniform across the warp
        const uint32_t ta = tmem_base + ((uint32_t)row0 << 16) + (uint32_t)(buf * kN + col);
        uint32_t v[32], u[32];
        tmem_ld_32x32b_x32(ta, v);
        if (!f32) tmem_ld_32x32b_x32(ta + 32u, u);
        tmem_ld_wait();
        if (lane == 0) bulk_wait_read0();  // the previous block's store has read the staging block
        __syncwarp();
        const uint32_t rbase = stg + (uint32_t)lane * 128u;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          uint32_t o[4];
          if (f32) {
#pragma unroll
            for (int e = 0; e < 4; ++e) o[e] = v[4 * k + e];
          } else {
            const uint32_t* src = k < 4 ? &v[k * 8] : &u[(k - 4) * 8];
#pragma unroll
            for (int e = 0; e < 4; ++e)
              o[e] = pack_bf16x2(__uint_as_float(src[2 * e]), __uint_as_float(src[2 * e + 1]));
          }
          const uint32_t dst = rbase + (uint32_t)(((k ^ (lane & 7)) & 7) << 4);
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3])
                       : "memory");
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          tma_store_2d(&b.tmOut[w.p], stg, w.n0 + col, row_st);
          bulk_commit();
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctl->tempty[buf]));
    }
    if (lane == 0) bulk_wait0();  // the output must be written before the CTA exits
  } else if (kQ && warp < 2 + kEpi + kConvWarps) {
    // ------------------------------------------------------------ weight dequantizers
    const int cw = (warp - 2 - kEpi) % kGroupWarps, grp = (warp - 2 - kEpi) / kGroupWarps;
    const int ct = cw * 32 + lane;
    int stage = 0, qs = 0;
    uint32_t phase = 0, qpar = 0;
    uint32_t wseq = 0;  // contraction blocks so far
    bool ok = true;
    for (int it = 0; ok; ++it) {
      const int t = next_tile(it);
      if (t < 0) break;
      const Tile w = tile_of(t);
      const GemmProblem& Q = b.prob[w.p];
      const int kq1 = min(w.kb1, Q.kb_main);  // end of the blocks taken from codes
      for (int kb = w.kb0; kb < w.kb1; ++kb, ++wseq) {
        const bool main = kb < Q.kb_main;
        const bool mine = (int)(wseq % kConvGroups) == grp;
        const uint32_t wfull = smem_u32(&ctl->wfull[stage]);
        if (mine) {
          // the stage's previous contents are consumed by the MMAs
          ok = mbar_wait(smem_u32(&ctl->empty[stage]), phase ^ 1u, wc, abort_flag);
          if (ok && main) ok = mbar_wait(smem_u32(&ctl->qfull[qs]), qpar, wc, abort_flag);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
        }
        if (main) {
          if (mine) {
            dequant_block<kBMn>(q_slot(qs), w_tile(stage), ct, w.n0, kb, Q.N);
            fence_proxy_async_smem();  // the tensor core reads what these threads wrote
            __syncwarp();
          }
          // Past the slot's last block of this tile.  A warp's arrival must count for this fill of the slot and no
          // earlier one.  Forward: a warp arrives once the fill has landed, which the fill before it had to be
          // released for; a slot of one block (a split's range that starts or ends inside a slot) is waited for
          // by the group that owns none of it as well.  Backward: when a warp passes block i, block i - 4 is
          // consumed, so every warp is past block i - 6, the slot's last (waiting there too took the 4-bit
          // Llama-shaped layer at T = 64 from 81.7 to 87.0 us).
          if ((kb + 1) % QS::kBlocks == 0 || kb + 1 == kq1) {
            if (!mine && !kBMn && kb == max(w.kb0, kb / QS::kBlocks * QS::kBlocks)) {
              ok = mbar_wait(smem_u32(&ctl->qfull[qs]), qpar, wc, abort_flag);
              ok = __all_sync(0xffffffffu, ok);
              if (!ok) break;
            }
            if (lane == 0) mbar_arrive(smem_u32(&ctl->qempty[qs]));
            if (++qs == QS::kStages) {
              qs = 0;
              qpar ^= 1u;
            }
          }
        } else if (mine) {
          // adapter block: the bf16 rank side goes straight into the weight tile by TMA (an input, or padded
          // before the row products, which had waited for that when this grid started)
          if (cw == 0 && lane == 0) {
            mbar_expect_tx(wfull, w_bytes(w.n0, Q.N));
            load_w(w_tile(stage), &b.tmB2[w.p], wfull, w.n0, Q.N, (kb - Q.kb_main) * kBK);
          }
          __syncwarp();
        }
        if (mine && lane == 0) mbar_arrive(wfull);
        if (++stage == kStages) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
  } else if (kQ) {
    // ------------------------------------------------------------ code producer
    int qs = 0;
    uint32_t qpar = 0;
    int qfills = 0;
    bool ok = true;
    for (int it = 0; ok; ++it) {
      const int t = next_tile(it);
      if (t < 0) break;
      const Tile w = tile_of(t);
      const GemmProblem& Q = b.prob[w.p];
      for (int kb = w.kb0; kb < min(w.kb1, Q.kb_main); kb = (kb / QS::kBlocks + 1) * QS::kBlocks) {
        ok = mbar_wait(smem_u32(&ctl->qempty[qs]), qpar ^ 1u, wc, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        if (lane == 0) {
          const uint32_t qbar = smem_u32(&ctl->qfull[qs]);
          const uint32_t codes = q_slot(qs), params = codes + QS::kCodes;
          mbar_arrive_expect_tx(qbar, QS::kBytes);
          if (kBMn) {
            tma_load_2d(codes, &b.tmQ[w.p], qbar, w.n0 / 2, kb * kBK);
            tma_load_2d(params, &b.tmP[w.p], qbar, (w.n0 >> 6) * 2, kb * kBK);
          } else {
            tma_load_2d(codes, &b.tmQ[w.p], qbar, (kb & ~1) * 32, w.n0);
            tma_load_2d(params, &b.tmP[w.p], qbar, (kb & ~3) * 2, w.n0);
          }
        }
        ++qfills;
        if (++qs == QS::kStages) {
          qs = 0;
          qpar ^= 1u;
        }
      }
    }
    if (lane == 0) ctl->qfills = qfills;
  }

  if constexpr (kCl) {
    // ------------------------------------------------------------ sum of the parts
    // Send and receive areas lie in the idle ring, each (S - 1) / S of rows x 1 KB (the host keeps both
    // within it): one region per peer of `rows` rows x 1024 / S bytes, 16-byte chunk u of row r at
    // u ^ (r mod 8).
    tc_fence_before();
    cluster_sync_all();
    tc_fence_after();
    if (warp >= 2 && warp < 2 + kEpi && !*abort_flag) {
      const Tile w = tile_of((int)blockIdx.x / S);
      const GemmProblem& Q = b.prob[w.p];
      const int q = warp & 3, part = (warp - 2) >> 2;
      const int row0 = q * 32, row = row0 + lane;
      const int groups = (Q.M + 31) / 32;                // 32-row groups holding rows
      const uint32_t cols = (uint32_t)(kN / S), row_b = cols * 4u, region = (uint32_t)groups * 32u * row_b;
      const uint32_t recv = base, send = base + (uint32_t)(S - 1) * region;
      auto slot = [&](int owner, int from) { return (uint32_t)(from < owner ? from : from - 1) * region; };
      auto chunk = [&](uint32_t u) { return (uint32_t)row * row_b + (((u ^ (uint32_t)row) & 7u) | (u & ~7u)) * 16u; };
      const uint32_t tl = tmem_base + ((uint32_t)row0 << 16);
      if (row0 < Q.M) {  // uniform across the warp
        // the slices of this warp's columns that other CTAs own
        for (int k = 0; k < S; ++k) {
          const int c0 = k * (int)cols;
          if (k == crank || c0 >= (part + 1) * C::kPartCols || c0 + (int)cols <= part * C::kPartCols) continue;
          const uint32_t dst = send + slot(crank, k);
          for (uint32_t cc = 0; cc < cols; cc += 32) {
            uint32_t v[32];
            tmem_ld_32x32b_x32(tl + (uint32_t)c0 + cc, v);
            tmem_ld_wait();
#pragma unroll
            for (int u = 0; u < 8; ++u)
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + chunk(cc / 4 + (uint32_t)u)),
                           "r"(v[4 * u]), "r"(v[4 * u + 1]), "r"(v[4 * u + 2]), "r"(v[4 * u + 3])
                           : "memory");
          }
          fence_proxy_async_smem();  // the bulk copy reads what these threads wrote
          __syncwarp();
          if (lane == 0) {
            const uint32_t off = (uint32_t)row0 * row_b;
            bulk_copy_to_peer(mapa_shared(recv + slot(k, crank) + off, (uint32_t)k), dst + off, 32u * row_b,
                              mapa_shared(smem_u32(&ctl->xchg), (uint32_t)k));
          }
        }
        // this CTA's own columns
        const int c0 = crank * (int)cols;
        if (c0 < (part + 1) * C::kPartCols && c0 + (int)cols > part * C::kPartCols) {
          if (q == 0 && lane == 0) mbar_arrive_expect_tx(smem_u32(&ctl->xchg), (uint32_t)(S - 1) * region);
          bool got = mbar_wait(smem_u32(&ctl->xchg), 0u, wc, abort_flag);
          got = __all_sync(0xffffffffu, got);
          __nv_bfloat16* out = static_cast<__nv_bfloat16*>(Q.out) + (size_t)row * Q.ldo + w.n0 + c0;
          for (uint32_t cc = 0; got && cc < cols; cc += 32) {
            uint32_t v[32];
            tmem_ld_32x32b_x32(tl + (uint32_t)c0 + cc, v);
            tmem_ld_wait();
            float a[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) a[e] = 0.f;
            for (int s = 0; s < S; ++s) {  // in CTA order
              if (s == crank) {
#pragma unroll
                for (int e = 0; e < 32; ++e) a[e] += __uint_as_float(v[e]);
              } else {
                const uint32_t src = recv + slot(crank, s);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                  float o[4];
                  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                               : "=f"(o[0]), "=f"(o[1]), "=f"(o[2]), "=f"(o[3])
                               : "r"(src + chunk(cc / 4 + (uint32_t)u))
                               : "memory");
#pragma unroll
                  for (int e = 0; e < 4; ++e) a[4 * u + e] += o[e];
                }
              }
            }
            if (row < Q.M) {
#pragma unroll
              for (int u = 0; u < 4; ++u)  // N is a multiple of 8: whole 16-byte pieces
                if (w.n0 + c0 + (int)cc + 8 * u < Q.N)
                  *reinterpret_cast<uint4*>(out + cc + 8 * u) =
                      make_uint4(pack_bf16x2(a[8 * u], a[8 * u + 1]), pack_bf16x2(a[8 * u + 2], a[8 * u + 3]),
                                 pack_bf16x2(a[8 * u + 4], a[8 * u + 5]), pack_bf16x2(a[8 * u + 6], a[8 * u + 7]));
            }
          }
        }
      }
    }
  }

  // ------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) {
    // every MMA has finished before tensor memory is released
    if (!mbar_wait_drain(smem_u32(&ctl->drain), 0, b.limit_ns > kDrainNs ? b.limit_ns : kDrainNs))
      atomicCAS(b.status, 0, kStatusTimeout);
    if (*abort_flag) {
      // a wait gave up: let the copies still in flight land before the shared memory is released (bounded);
      // an adapter block's boxes, tracked by wfull only, get a fixed margin
      const int nf = ctl->fills, nq = ctl->qfills;
      for (int i = nf - 1; i >= 0 && i >= nf - kStages; --i)
        if (!mbar_wait_drain(smem_u32(&ctl->full[i % kStages]), (uint32_t)((i / kStages) & 1), kAbortDrainNs))
          atomicCAS(b.status, 0, kStatusTimeout);
      if (kQ)
        for (int i = nq - 1; i >= 0 && i >= nq - QS::kStages; --i)
          if (!mbar_wait_drain(smem_u32(&ctl->qfull[i % QS::kStages]), (uint32_t)((i / QS::kStages) & 1), kAbortDrainNs))
            atomicCAS(b.status, 0, kStatusTimeout);
      const uint64_t t0 = global_timer_ns();
      while (global_timer_ns() - t0 < 50000ull) {
      }
    }
    // this grid's completion implies the previous grid's (the next grid waits for this one only)
    if (b.early_inputs) griddep_wait();
  }
  __syncthreads();
  if (kCl) cluster_sync_all();  // no copy into or out of a peer is pending
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

template <bool kBMn, bool kQ>
cudaError_t launch_variant(const GemmBatch& batch, int ctas, cudaStream_t stream) {
  constexpr size_t smem = smem_bytes<kQ>();
  if (batch.cluster > 1) {
    static std::atomic<unsigned long long> cl_done{0};
    const cudaError_t e = set_smem_once(small_lora_gemm<kBMn, kQ, true>, (int)smem, cl_done);
    if (e != cudaSuccess) return e;
    return launch_kernel(small_lora_gemm<kBMn, kQ, true>, dim3((unsigned)(batch.total_tiles * batch.cluster)),
                         dim3(Cfg<kQ>::kThreads), smem, stream, batch.cluster, batch);
  }
  static std::atomic<unsigned long long> attr_done{0};
  const cudaError_t e = set_smem_once(small_lora_gemm<kBMn, kQ, false>, (int)smem, attr_done);
  if (e != cudaSuccess) return e;
  return launch_kernel(small_lora_gemm<kBMn, kQ, false>, dim3((unsigned)ctas), dim3(Cfg<kQ>::kThreads), smem, stream, 1,
                       batch);
}

template <bool kBMn, bool kQ>
int query_clusters(int size) {
  constexpr size_t smem = smem_bytes<kQ>();
  static std::atomic<unsigned long long> attr_done{0};
  if (set_smem_once(small_lora_gemm<kBMn, kQ, true>, (int)smem, attr_done) != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(size * 128));
  cfg.blockDim = dim3(Cfg<kQ>::kThreads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)size;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int k = 0;
  if (cudaOccupancyMaxActiveClusters(&k, small_lora_gemm<kBMn, kQ, true>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return k;
}

}  // namespace

int gemm_small_max_clusters(bool b_mn_major, bool q4, int size) {
  // per device, form and cluster size 2, 4, 8; 0: not asked yet, -1: none
  static std::atomic<int> cache[64][4][3];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  std::atomic<int>& c = cache[dev][(b_mn_major ? 2 : 0) + (q4 ? 1 : 0)][size == 8 ? 2 : size == 4 ? 1 : 0];
  int v = c.load(std::memory_order_acquire);
  if (v == 0) {
    v = b_mn_major ? (q4 ? query_clusters<true, true>(size) : query_clusters<true, false>(size))
                   : (q4 ? query_clusters<false, true>(size) : query_clusters<false, false>(size));
    if (v <= 0) v = -1;
    c.store(v, std::memory_order_release);
  }
  return v > 0 ? v : 0;
}

// Rows whose send and receive areas, (size - 1) / size of 2 KB each, fit the ring.
int gemm_small_cluster_rows(int size) {
  const int rows = (int)(Cfg<false>::kRing / (2u * 1024u * (unsigned)(size - 1) / (unsigned)size));
  return rows / 32 * 32 < kM ? rows / 32 * 32 : kM;
}

cudaError_t launch_small_gemm(const GemmBatch& batch, bool b_mn_major, bool q4, int num_sms, cudaStream_t stream) {
  if (batch.total_tiles <= 0) return cudaSuccess;
  const int ctas = batch.total_tiles < num_sms ? batch.total_tiles : num_sms;
  if (q4)
    return b_mn_major ? launch_variant<true, true>(batch, ctas, stream) : launch_variant<false, true>(batch, ctas, stream);
  return b_mn_major ? launch_variant<true, false>(batch, ctas, stream) : launch_variant<false, false>(batch, ctas, stream);
}

int gemm_small_rows() { return kM; }
int gemm_tile_n_small() { return kN; }

}  // namespace lora
