// Top-k similarity table of a frozen embedding (Section "Softmax
// Approximation", "Choosing the Reduced Vocabulary Set"): token vectors are
// normalised, C = E~ E~^T holds the cosine similarities, and row i of the
// table lists the k most similar tokens in descending order (lower index
// first on ties).  The V x V matrix is never formed.
//   row_norms           ||E_i||, the sum of squares accumulated in fp32 in index
//                       order (squares of bf16 are exact), correctly rounded sqrt
//   scale_rows          E~_i = bf16(E_i / ||E_i||), the division correctly rounded
// Rows shorter than 32768 tokens (the host runs chunks of rows):
//   topk_short          (up to 8192 tokens) per row of a chunk's fp32 similarities
//                       (tcgen05 contraction in fused_gemm.cu): the values from
//                       the k-th largest one's histogram bin up, sorted as the
//                       long rows' candidates are
//   topk_select         (over 8192 tokens, and any row whose list came out short
//                       or long) over 8192 tokens the values above a threshold
//                       from a sample of the row, sorted on (similarity
//                       descending, index ascending); otherwise, and where those
//                       are too few or too many, radix select on an
//                       order-preserving uint32 image (11-bit histograms,
//                       then 11, then 10 bits) until the candidates at or
//                       above the chosen prefix fit in shared memory, then the
//                       sort
// Rows of at least 32768 tokens:
//   topk_gather_sample  up to 8192 evenly spread tokens
//   topk_tau            each row's threshold from its similarities to them
//   (fused_gemm.cu)     the upper triangle of C, each value appended to the
//                       candidate lists of both its rows when it reaches
//                       their thresholds
//   topk_sort_warp,     each row's candidates sorted: a warp per list of up
//   topk_sort           to 1024 in registers, a block for longer lists
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace lora {

namespace {

constexpr int kSelThreads = 1024;
constexpr int kCap = 4096;  // candidates held in shared memory

// Row norms, one warp per 32 rows.  The sum of squares is a chain in index
// order, so a row belongs to one lane; the warp stages 64 columns of its 32 rows
// at a time through shared memory with coalesced 16-byte copies (cp.async,
// kNormStages chunks in flight) and each lane adds its own row's.  Then one
// element-wise pass divides (scale_rows).  HBM-bound: E twice in, E~ once out (735
// MB at V = 40000, d = 3072).  Measured there: one thread per row, reading its row
// straight from memory and dividing it, 355 us; these two 46 + 99 us.

// bf16(x / n) with the division correctly rounded to fp32 first, as
// __float2bfloat16_rn(__fdiv_rn(x, n)).  x * (1 / n), both rounded, is within 2
// units in the last place of x / n and the rounded quotient within half of
// one, so both round to the same bf16 unless the product's low 16 bits are within
// 3 of the midpoint 0x8000: those elements (1 in 9000) are divided.  `fast` is false
// for a divisor whose reciprocal or quotients could leave the normal range;
// quotients below 2^-100 are divided as well.
__device__ __forceinline__ float divide_bf16(float x, float n, float rn, bool fast) {
  const float q = x * rn;
  const uint32_t u = __float_as_uint(q), lo = (u & 0xFFFFu) - (0x8000u - 4u);
  if (fast && lo > 8u && (fabsf(q) >= 0x1p-100f || x == 0.f)) return q;
  return __fdiv_rn(x, n);
}

constexpr int kNormWarps = 2, kNormStages = 4;
constexpr int kNormPitch = 144;  // bytes of a staged row: 128 + 16, so that lanes reading 16 bytes of 32 rows spread

__global__ void __launch_bounds__(kNormWarps * 32) row_norms_kernel(const __nv_bfloat16* __restrict__ E, int V, int d,
                                                                   float* __restrict__ norm) {
  griddep_wait();
  griddep_launch_dependents();
  __shared__ __align__(16) uint8_t stage[kNormWarps][kNormStages][32 * kNormPitch];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i0 = (blockIdx.x * kNormWarps + warp) * 32;
  if (i0 >= V) return;  // whole warps
  const int rows = min(32, V - i0);
  const int nv = d / 8, chunks = (nv + 7) / 8;  // 16-byte vectors of a row, 8 per chunk
  const uint4* src = reinterpret_cast<const uint4*>(E) + (long long)i0 * nv;
  const int cr = lane >> 3, cv = lane & 7;  // this lane's row (of four) and vector in a copy step
  auto fetch = [&](int c) {
    if (c < chunks && c * 8 + cv < nv) {
      const uint32_t dst = smem_u32(stage[warp][c % kNormStages]) + (uint32_t)cv * 16u;
#pragma unroll
      for (int r = 0; r < 32; r += 4)
        if (r + cr < rows)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + (uint32_t)((r + cr) * kNormPitch)),
                       "l"(src + (long long)(r + cr) * nv + c * 8 + cv)
                       : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int c = 0; c < kNormStages - 1; ++c) fetch(c);
  float s = 0.f;
  for (int c = 0; c < chunks; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kNormStages - 2) : "memory");
    __syncwarp();  // every lane's copies of chunk c have landed, and chunk c - 1 is read
    fetch(c + kNormStages - 1);
    const uint4* row = reinterpret_cast<const uint4*>(stage[warp][c % kNormStages] + lane * kNormPitch);
    const int n = min(8, nv - c * 8);
    if (lane < rows)
      for (int v = 0; v < n; ++v) {
        const uint4 q = row[v];
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float lo = __uint_as_float(w[e] << 16), hi = __uint_as_float(w[e] & 0xFFFF0000u);
          s = __fadd_rn(s, __fmul_rn(lo, lo));  // each square is exact; index order
          s = __fadd_rn(s, __fmul_rn(hi, hi));
        }
      }
  }
  if (lane < rows) norm[i0 + lane] = __fsqrt_rn(s);
}

// En[i] = bf16(E[i] / norm[i]) (zero rows stay zero): eight 16-byte vectors per thread, all loads first.
__global__ void __launch_bounds__(256) scale_rows_kernel(const __nv_bfloat16* __restrict__ E, int V, int d,
                                                         const float* __restrict__ norm,
                                                         __nv_bfloat16* __restrict__ En) {
  griddep_wait();
  griddep_launch_dependents();
  constexpr int kU = 8;
  const int nv = d / 8;
  const long long total = (long long)V * nv, e0 = (long long)blockIdx.x * (256 * kU) + threadIdx.x;
  const uint4* src = reinterpret_cast<const uint4*>(E);
  uint4* dst = reinterpret_cast<uint4*>(En);
  uint4 q[kU];
  float nr[kU];
#pragma unroll
  for (int u = 0; u < kU; ++u) {
    const long long e = e0 + 256 * u;
    q[u] = e < total ? __ldg(src + e) : make_uint4(0u, 0u, 0u, 0u);
    nr[u] = e < total ? __ldg(norm + e / nv) : 1.f;
  }
#pragma unroll
  for (int u = 0; u < kU; ++u) {
    const long long e = e0 + 256 * u;
    const float n = nr[u];
    const bool fast = n > 0x1p-60f && n < 0x1p60f;
    const float rn = __frcp_rn(n);
    const uint32_t w[4] = {q[u].x, q[u].y, q[u].z, q[u].w};
    uint32_t o[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const float lo = __uint_as_float(w[h] << 16), hi = __uint_as_float(w[h] & 0xFFFF0000u);
      const float x = n > 0.f ? divide_bf16(lo, n, rn, fast) : 0.f, y = n > 0.f ? divide_bf16(hi, n, rn, fast) : 0.f;
      o[h] = pack_bf16x2(x, y);
    }
    if (e < total) dst[e] = make_uint4(o[0], o[1], o[2], o[3]);
  }
}

// Exclusive scan of one value per thread over the block; returns the total.
__device__ __forceinline__ int scan_block(int v, int* excl, int* warp_tot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int w = warp_tot[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    warp_tot[lane] = w;
  }
  __syncthreads();
  *excl = (warp > 0 ? warp_tot[warp - 1] : 0) + x - v;
  const int total = warp_tot[31];
  __syncthreads();
  return total;
}

struct SelShared {
  int hist[2048];
  uint32_t ckey[kCap];
  int cidx[kCap];
  int warp_tot[32];
  int bin, above, ncand;
  uint32_t smin, smax;
};

// Bin (of nbins, by descending bin index) where the k_rem-th largest falls,
// and the count in higher bins.
__device__ void find_bin(SelShared& sh, int nbins, int k_rem) {
  const int per = nbins / kSelThreads;  // 1 or 2
  const int t = threadIdx.x;
  int b0 = nbins - 1 - t * per;
  int local = 0;
  for (int q = 0; q < per; ++q) local += sh.hist[b0 - q];
  int excl;
  scan_block(local, &excl, sh.warp_tot);
  if (excl < k_rem && k_rem <= excl + local) {
    int acc = excl;
    for (int q = 0; q < per; ++q) {
      const int h = sh.hist[b0 - q];
      if (k_rem <= acc + h) {
        sh.bin = b0 - q;
        sh.above = acc;
        break;
      }
      acc += h;
    }
  }
  __syncthreads();
}

// A candidate as one 64-bit value, larger first: the order key above, the
// complement of the index below (equal keys: the lower index first).
__device__ __forceinline__ uint64_t pack_cand(uint32_t key, int idx) {
  return ((uint64_t)key << 32) | (uint32_t)(0xffffffffu - (uint32_t)idx);
}
__device__ __forceinline__ int cand_index(uint64_t v) { return (int)(0xffffffffu - (uint32_t)v); }

// Bitonic sort, descending, of p2 = kT * E packed candidates held in
// registers: slot e of thread t is position t + e * kT.  Strides below 32 are
// exchanged by warp shuffles, 32 .. kT / 2 through the shared buffer x (p2
// entries; 2 p2 with kTwo, whose halves alternate so that a stage needs one barrier
// instead of two), kT and up within the thread (fully unrolled, so the slots stay in
// registers).  Only the first n positions hold candidates (the rest zeros, below
// them all): the sort ends with the first runs of at least n.  Every thread of the
// block takes part.  Bound by the barriers' latency: whole tables of V = 12000, d =
// 2048, k = 64 with all sizes and two barriers a stage 1099 us, so 951; of V = 29747,
// d = 1120, k = 150: 4414 / 4231; of V = 24000, d = 512, k = 800: 2976 / 2943.
template <int kT, int E, bool kTwo>
__device__ void bitonic_sort(uint64_t (&v)[E], uint64_t* x, int n) {
  constexpr int p2 = kT * E;
  const int tid = (int)threadIdx.x;
  int half = 0;
  // fully unrolled: every stage's exchange form and masks are compile-time constants
#pragma unroll
  for (int size = 2; size <= p2; size <<= 1) {
    if (size >= 2 * n) break;
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      if (stride >= kT) {
#pragma unroll
        for (int lg = 0; (1 << lg) < E; ++lg) {
          if (stride == (kT << lg)) {
#pragma unroll
            for (int e = 0; e < E; ++e) {
              const int f = e | (1 << lg);
              if ((e & (1 << lg)) == 0 && f < E) {
                const bool up = ((tid + e * kT) & size) == 0;
                if ((v[f] > v[e]) == up) {
                  const uint64_t t = v[e];
                  v[e] = v[f];
                  v[f] = t;
                }
              }
            }
          }
        }
      } else {
        const bool via_smem = stride >= 32;
        if (via_smem) {
#pragma unroll
          for (int e = 0; e < E; ++e) x[half + tid + e * kT] = v[e];
          __syncthreads();
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int p = tid + e * kT;
          const uint64_t q = via_smem ? x[half + (p ^ stride)] : __shfl_xor_sync(0xffffffffu, v[e], stride);
          const bool up = (p & size) == 0, lo = (p & stride) == 0;
          const bool q_first = q > v[e];
          // an ascending run keeps the first of the pair at the lower position
          if (lo ? q_first == up : q_first != up) v[e] = q;
        }
        if (via_smem && !kTwo) __syncthreads();
        if (via_smem && kTwo) half ^= p2;
      }
    }
  }
}

// One warp sorts 32 * E packed candidates, descending: slot e of lane l is
// position l * E + e, so every exchange at a stride below E stays within a lane
// and only the log2(32) + ... + 1 = 15 steps at strides E .. 16 E are warp
// shuffles (with position e * 32 + l, 40 of the 55 steps of 1024 candidates
// shuffled two words of every slot, and the shuffle unit set the pace: 1092 us
// for 40000 rows of about 800 candidates).
template <int E>
__device__ __forceinline__ void warp_sort(uint64_t (&v)[E]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int size = 2; size <= 32 * E; size <<= 1) {
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      if (stride >= E) {
        const bool up = size > 16 * E || (lane & (size / E)) == 0, lo = (lane & (stride / E)) == 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const uint64_t q = __shfl_xor_sync(0xffffffffu, v[e], stride / E);
          // the lower position of the pair keeps the larger in a descending run
          if ((q > v[e]) == (lo == up)) v[e] = q;
        }
      } else {
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int f = e | stride;
          if ((e & stride) == 0 && f < E) {
            const bool up = size < E ? (e & size) == 0 : size > 16 * E || (lane & (size / E)) == 0;
            if ((v[f] > v[e]) == up) {
              const uint64_t t = v[e];
              v[e] = v[f];
              v[f] = t;
            }
          }
        }
      }
    }
  }
}

// A warp loads n <= 32 * E candidates, sorts them and writes the first k
// indices to out through its 32 * E words of shared memory (whole lines).
template <int E>
__device__ void warp_sort_write(const uint2* __restrict__ c, int n, int k, int32_t* __restrict__ buf,
                                int32_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  uint64_t v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {  // any order will do: the loads coalesce
    const int p = lane + e * 32;
    v[e] = 0ull;
    if (p < n) {
      const uint2 q = c[p];
      v[e] = pack_cand(q.x, (int)q.y);
    }
  }
  warp_sort<E>(v);
  // position l * E + e at word (l * E + e) ^ l: lanes write to different banks
#pragma unroll
  for (int e = 0; e < E; ++e) buf[(lane * E + e) ^ lane] = cand_index(v[e]);
  __syncwarp();
  for (int p = lane; p < k; p += 32) out[p] = buf[p ^ (p / E)];
  __syncwarp();
}

// Loads n <= kT * E candidates (get(p) -> (key, index)), sorts them and writes
// the first k indices to out; padding sorts below every real candidate.
template <int kT, int E, bool kTwo = false, typename Get>
__device__ void sort_write_e(Get get, int n, int k, uint64_t* x, int32_t* __restrict__ out) {
  const int tid = (int)threadIdx.x;
  uint64_t v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int p = tid + e * kT;
    if (p < n) {
      const uint2 c = get(p);
      v[e] = pack_cand(c.x, (int)c.y);
    } else {
      v[e] = 0ull;
    }
  }
  __syncthreads();  // the candidates may live in the exchange buffer
  bitonic_sort<kT, E, kTwo>(v, x, n);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int p = tid + e * kT;
    if (p < k) out[p] = cand_index(v[e]);
  }
}

// Sorts the n candidates in shared memory (n <= kCap; the selection kernel's
// 1024 threads) and writes the first k indices to out.
__device__ void sort_and_write(SelShared& sh, int n, int k, int32_t* __restrict__ out) {
  auto get = [&](int p) { return make_uint2(sh.ckey[p], (uint32_t)sh.cidx[p]); };
  uint64_t* x = reinterpret_cast<uint64_t*>(sh.ckey);  // ckey and cidx together: 4096 x 8 bytes
  if (n <= kSelThreads)
    sort_write_e<kSelThreads, 1, true>(get, n, k, x, out);
  else if (n <= 2 * kSelThreads)
    sort_write_e<kSelThreads, 2, true>(get, n, k, x, out);
  else
    sort_write_e<kSelThreads, 4>(get, n, k, x, out);
}

constexpr int kSample = 8 * kSelThreads;
constexpr int kSampleMinV = 4 * kSample;
constexpr float kOver = 1.6f;

// Rank of the sample value that sets the threshold: about kOver * k of a
// row's V values are expected at or above the rs-th largest of ns sampled ones.
__device__ __forceinline__ int sample_rank(int V, int k, int ns) {
  return min(ns, max(1, (int)ceilf(kOver * (float)k * (float)ns / (float)V)));
}

// Sampled threshold for rows of more than kRowSampleMinV values: a linear
// histogram of kRowSample evenly spread values over their [min, max] gives the
// lower edge of the bin of their rs-th largest, rs four standard deviations
// above the k * kRowSample / V of them expected among the row's top k (a row falls
// short about once in 30000); then one streaming pass appends every value at or
// above that edge, one ballot per 16-byte load and, for a warp with hits, one
// shared-memory atomic.  A value left out is strictly below every candidate,
// so when the candidates number between k and kCap they contain the exact
// top k.  Returns false (and the caller falls back to the full radix select)
// otherwise and for a row with a NaN, which the radix select orders by its key.
// Bound by the row's reads from L2 (one and an eighth to one and a half times, the
// radix select three times) and the block sort.  Whole tables, radix select before /
// this: V = 29747, d = 1120, k = 150: 5570 / 4986 us; V = 12000, d = 2048, k = 64: 1269
// / 1200 (with the sort's ten sizes); with more than 1024 candidates only once they are narrowed: V = 17003, d =
// 512, k = 1000: 2939 / 2811 without, about 2410 with.
constexpr int kRowSample = 4 * kSelThreads;
constexpr int kRowSampleMinV = 2 * kRowSample;

// The smallest and largest of the block's keys, each thread's own in kmin and
// kmax, into sh.smin and sh.smax (read after the barrier it ends with).
__device__ __forceinline__ void block_key_range(SelShared& sh, uint32_t kmin, uint32_t kmax) {
  if (threadIdx.x == 0) {
    sh.smin = 0xffffffffu;
    sh.smax = 0u;
  }
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&sh.smin, kmin);
    atomicMax(&sh.smax, kmax);
  }
  __syncthreads();
}

// Of the n candidates (k <= n <= kCap, all written before the caller's last
// barrier) keeps those from the bin of the k-th largest up, in 2048 bins linear in
// the keys; returns their number.  A sort of 2048 costs more than twice one of 1024.
__device__ int narrow_candidates(SelShared& sh, int n, int k) {
  const int t = threadIdx.x, lane = t & 31;
  uint32_t key[4];
  int idx[4];
  uint32_t kmin = 0xffffffffu, kmax = 0u;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int p = t + e * kSelThreads;
    key[e] = p < n ? sh.ckey[p] : 0u;
    idx[e] = p < n ? sh.cidx[p] : 0;
    if (p < n) {
      kmin = min(kmin, key[e]);
      kmax = max(kmax, key[e]);
    }
  }
  sh.hist[t] = 0;
  sh.hist[t + kSelThreads] = 0;
  block_key_range(sh, kmin, kmax);
  kmin = sh.smin;
  const int shift = max(0, 21 - __clz((int)(sh.smax - kmin)));  // 11 bits of the range
#pragma unroll
  for (int e = 0; e < 4; ++e)
    if (t + e * kSelThreads < n) atomicAdd(&sh.hist[(key[e] - kmin) >> shift], 1);
  if (t == 0) sh.ncand = 0;
  __syncthreads();
  find_bin(sh, 2048, k);
  const uint32_t bin = (uint32_t)sh.bin;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const bool keep = t + e * kSelThreads < n && ((key[e] - kmin) >> shift) >= bin;
    const uint32_t m = __ballot_sync(0xffffffffu, keep);
    int base = 0;
    if (lane == 0 && m) base = atomicAdd(&sh.ncand, __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0) + __popc(m & ((1u << lane) - 1u));
    if (keep) {
      sh.ckey[base] = key[e];
      sh.cidx[base] = idx[e];
    }
  }
  __syncthreads();
  return sh.ncand;
}

// f: this thread's 4 sample values.
__device__ float sample_threshold(SelShared& sh, const float (&f)[4], int rs) {
  const int t = threadIdx.x;
  sh.hist[t] = 0;
  sh.hist[t + kSelThreads] = 0;
  uint32_t kmin = 0xffffffffu, kmax = 0u;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    kmin = min(kmin, ord_key(f[e]));
    kmax = max(kmax, ord_key(f[e]));
  }
  block_key_range(sh, kmin, kmax);
  auto value = [](uint32_t key) { return __uint_as_float((key & 0x80000000u) ? (key & 0x7fffffffu) : ~key); };
  const float lo = value(sh.smin), hi = value(sh.smax);
  const float scale = hi > lo ? 2048.f / (hi - lo) : 0.f;
#pragma unroll
  for (int e = 0; e < 4; ++e) atomicAdd(&sh.hist[min(2047, max(0, (int)((f[e] - lo) * scale)))], 1);
  __syncthreads();
  find_bin(sh, 2048, rs);
  return lo + (float)sh.bin * ((hi - lo) / 2048.f);
}

__device__ bool sampled_select(SelShared& sh, const float* __restrict__ s, int V, int k, int32_t* __restrict__ out) {
  const float4* s4 = reinterpret_cast<const float4*>(s);
  const int n4 = V / 4;
  const int lane = threadIdx.x & 31;
  const float4 q0 = __ldg(s4 + (int)(((long long)threadIdx.x * n4) / kSelThreads));  // evenly spread over the row
  const float sample[4] = {q0.x, q0.y, q0.z, q0.w};
  const float rk = (float)k * (float)kRowSample / (float)V;
  const float tf = sample_threshold(sh, sample, min(kRowSample, (int)ceilf(rk + 4.f * sqrtf(rk)) + 2));
  bool nan = false;
  if (threadIdx.x == 0) sh.ncand = 0;
  __syncthreads();
  // appends this lane's hits among its first nv values of q (positions j0 + e); whole warps call it
  auto append4 = [&](const float4 q, int nv, int j0) {
    const float f[4] = {q.x, q.y, q.z, q.w};
    nan = nan || !(q.x == q.x && q.y == q.y && q.z == q.z && q.w == q.w);
    const int c = (nv > 0 && f[0] >= tf) + (nv > 1 && f[1] >= tf) + (nv > 2 && f[2] >= tf) + (nv > 3 && f[3] >= tf);
    if (__ballot_sync(0xffffffffu, c > 0) == 0u) return;
    int x = c;  // inclusive scan of the hit counts over the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    int base = 0;
    if (lane == 31) base = atomicAdd(&sh.ncand, x);
    int slot = __shfl_sync(0xffffffffu, base, 31) + x - c;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (e < nv && f[e] >= tf) {
        if (slot < kCap) {
          sh.ckey[slot] = ord_key(f[e]);
          sh.cidx[slot] = j0 + e;
        }
        ++slot;
      }
    }
  };
  // every thread runs the same iterations, so the ballots see whole warps
  for (int base4 = 0; base4 < n4; base4 += 4 * kSelThreads) {
    float4 q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j4 = base4 + u * kSelThreads + (int)threadIdx.x;
      q[u] = j4 < n4 ? __ldcs(s4 + j4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j4 = base4 + u * kSelThreads + (int)threadIdx.x;
      append4(q[u], j4 < n4 ? 4 : 0, 4 * j4);
    }
  }
  if (threadIdx.x < 32) {  // the last V mod 4 values, one warp
    const int j = 4 * n4 + lane;
    append4(make_float4(j < V ? s[j] : 0.f, 0.f, 0.f, 0.f), j < V ? 1 : 0, j);
  }
  const bool any_nan = __syncthreads_or(nan);
  int n = sh.ncand;
  if (any_nan || n < k || n > kCap) return false;  // uniform: read after the barrier
  if (n > kSelThreads) n = narrow_candidates(sh, n, k);
  sort_and_write(sh, n, k, out);
  return true;
}

// Similarity row s to table row trow.
__device__ __forceinline__ void select_row(SelShared& sh, const float* __restrict__ s, int V, int k, long long trow,
                           int32_t* __restrict__ table, int* __restrict__ status) {
  if (V > kRowSampleMinV) {
    if (sampled_select(sh, s, V, k, table + trow * k)) return;
    __syncthreads();  // the fallback reuses the shared buffers
  }
  // levels: (shift of the level's digit, digit bits); the prefix so far selects candidates
  const int shifts[3] = {21, 10, 0}, bits[3] = {11, 11, 10};
  uint32_t prefix = 0;  // chosen digits so far, as key >> shift of the current level
  int k_rem = k, above_total = 0, lvl_found = -1;
  for (int lvl = 0; lvl < 3; ++lvl) {
    const int nb = 1 << bits[lvl], sh_ = shifts[lvl];
    for (int b = threadIdx.x; b < nb; b += kSelThreads) sh.hist[b] = 0;
    __syncthreads();
    const int hi_shift = sh_ + bits[lvl];  // bits above this level's digit
    auto count = [&](float f) {
      const uint32_t key = ord_key(f);
      if (lvl == 0 || (key >> hi_shift) == prefix) atomicAdd(&sh.hist[(key >> sh_) & (nb - 1)], 1);
    };
    const float4* s4 = reinterpret_cast<const float4*>(s);
    const int n4 = V / 4;
    int j4 = threadIdx.x;
    for (; j4 + 3 * kSelThreads < n4; j4 += 4 * kSelThreads) {  // four loads in flight per thread
      float4 q[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) q[u] = __ldg(s4 + j4 + u * kSelThreads);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        count(q[u].x);
        count(q[u].y);
        count(q[u].z);
        count(q[u].w);
      }
    }
    for (; j4 < n4; j4 += kSelThreads) {
      const float4 q = __ldg(s4 + j4);
      count(q.x);
      count(q.y);
      count(q.z);
      count(q.w);
    }
    for (int j = (V & ~3) + (int)threadIdx.x; j < V; j += kSelThreads) count(s[j]);
    __syncthreads();
    find_bin(sh, nb, k_rem);
    prefix = (lvl == 0 ? 0u : prefix << bits[lvl]) | (uint32_t)sh.bin;
    above_total += sh.above;
    k_rem -= sh.above;
    const int ncand = above_total + sh.hist[sh.bin];
    if (ncand <= kCap) {
      lvl_found = lvl;
      break;
    }
    __syncthreads();
  }
  if (lvl_found < 0) {
    if (threadIdx.x == 0) atomicCAS(status, 0, kStatusTopkTies);  // more ties at the k-th value than fit
    return;
  }
  // collect every key whose prefix at the chosen level is >= the chosen prefix
  const int sh_ = shifts[lvl_found];
  if (threadIdx.x == 0) sh.ncand = 0;
  __syncthreads();
  auto take = [&](float f, int j) {
    const uint32_t key = ord_key(f);
    if ((key >> sh_) >= prefix) {
      const int slot = atomicAdd(&sh.ncand, 1);
      sh.ckey[slot] = key;
      sh.cidx[slot] = j;
    }
  };
  {
    const float4* s4 = reinterpret_cast<const float4*>(s);
    const int n4 = V / 4;
    int j4 = threadIdx.x;
    for (; j4 + 3 * kSelThreads < n4; j4 += 4 * kSelThreads) {
      float4 q[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) q[u] = __ldcs(s4 + j4 + u * kSelThreads);  // last read of the row
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j = 4 * (j4 + u * kSelThreads);
        take(q[u].x, j);
        take(q[u].y, j + 1);
        take(q[u].z, j + 2);
        take(q[u].w, j + 3);
      }
    }
    for (; j4 < n4; j4 += kSelThreads) {
      const float4 q = __ldcs(s4 + j4);
      take(q.x, 4 * j4);
      take(q.y, 4 * j4 + 1);
      take(q.z, 4 * j4 + 2);
      take(q.w, 4 * j4 + 3);
    }
  }
  for (int j = (V & ~3) + (int)threadIdx.x; j < V; j += kSelThreads) take(s[j], j);
  __syncthreads();
  sort_and_write(sh, sh.ncand, k, table + trow * k);
}

// One block per row r of S [.., lds], for table row rows[r] (row0 + r without
// rows); kList: the first *n_list entries of rows are table rows whose similarities
// are S's rows rows[i] - row0 (a short launch that usually finds none).
template <bool kList>
__global__ void __launch_bounds__(kSelThreads, 2) topk_select_kernel(const float* __restrict__ S, long long lds, int V,
                                                                  int k, int row0, const int32_t* __restrict__ rows,
                                                                  const int* __restrict__ n_list,
                                                                  int32_t* __restrict__ table,
                                                                  int* __restrict__ status) {
  griddep_wait();
  griddep_launch_dependents();
  extern __shared__ uint8_t smem_raw[];
  SelShared& sh = *reinterpret_cast<SelShared*>(smem_raw);
  // lds is a multiple of 4: 16-byte aligned rows
  if constexpr (!kList) {
    select_row(sh, S + (long long)blockIdx.x * lds, V, k,
               rows ? rows[blockIdx.x] : row0 + (int)blockIdx.x, table, status);
  } else {
    const int n = *n_list;
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
      select_row(sh, S + (long long)(rows[i] - row0) * lds, V, k, rows[i], table, status);
      __syncthreads();  // the shared buffers are free for the next row
    }
  }
}

// Candidates of rows of at most kShortMaxV values: one block per row of S, the row
// in registers.  A linear histogram of 2048 bins over the row's [min, max] gives
// the bin of its k-th largest value; every value from that bin up goes to the
// row's list (a value left out is in a lower bin, so below every candidate: with
// k to cap of them they hold the exact top k, and the warp sort finishes; any
// other row, for instance thousands of ties, goes to the radix select).  The radix
// select alone, a 1024-thread block with a three-level histogram and a block sort
// per row, took 118 us for 2048 rows of 8000 (k = 200); this 39 us, the sort 8 us.
// For longer rows (512 rows of 24000, k = 800) this form on 1024 threads (47 us) and a
// sort of few rows (31 us) took longer than one block per row (topk_select).
constexpr int kShortThreads = 256;
constexpr int kShortRegs = 8;  // float4 per thread
constexpr int kShortMaxV = 4 * kShortRegs * kShortThreads;

__global__ void __launch_bounds__(kShortThreads, 4) topk_short_kernel(const float* __restrict__ S, long long lds, int V,
                                                                     int k, uint2* __restrict__ cand, int cap,
                                                                     int* __restrict__ cnt) {
  griddep_wait();
  griddep_launch_dependents();
  __shared__ int hist[2048];
  __shared__ float red[2][kShortThreads / 32];
  __shared__ int wsum[kShortThreads / 32];
  __shared__ int s_bin, s_n;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float* s = S + (long long)blockIdx.x * lds;
  const float4* s4 = reinterpret_cast<const float4*>(s);
  const int n4 = (V + 3) / 4;  // lds is a multiple of 4: the last group is readable, its tail not counted
  float4 v[kShortRegs];
#pragma unroll
  for (int u = 0; u < kShortRegs; ++u) {
    const int j4 = tid + u * kShortThreads;
    v[u] = j4 < n4 ? __ldg(s4 + j4) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // f(value, index) over this thread's values
  auto each = [&](auto f) {
#pragma unroll
    for (int u = 0; u < kShortRegs; ++u) {
      const float x[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
      const int j = 4 * (tid + u * kShortThreads);
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (j + e < V) f(x[e], j + e);
    }
  };
  float lo = INFINITY, hi = -INFINITY;
  bool nan = false;
  each([&](float x, int) {
    lo = fminf(lo, x);
    hi = fmaxf(hi, x);
    nan = nan || x != x;
  });
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (__syncthreads_or(nan)) {  // the radix select orders NaNs by their keys
    if (tid == 0) cnt[blockIdx.x] = cap + 1;
    return;
  }
  for (int b = tid; b < 2048; b += kShortThreads) hist[b] = 0;
  if (lane == 0) {
    red[0][warp] = lo;
    red[1][warp] = hi;
  }
  if (tid == 0) {
    s_bin = 0;
    s_n = 0;
  }
  __syncthreads();
  lo = red[0][0];
  hi = red[1][0];
#pragma unroll
  for (int w = 1; w < kShortThreads / 32; ++w) {
    lo = fminf(lo, red[0][w]);
    hi = fmaxf(hi, red[1][w]);
  }
  const float scale = hi > lo ? 2048.f / (hi - lo) : 0.f;
  auto bin_of = [&](float x) { return min(2047, max(0, (int)((x - lo) * scale))); };
  each([&](float x, int) { atomicAdd(&hist[bin_of(x)], 1); });
  __syncthreads();
  // bins by descending index: thread t holds bins 2047 - 8t .. 2040 - 8t
  int local = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) local += hist[2047 - 8 * tid - q];
  int x = local;  // inclusive scan over the block
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  int excl = x - local;
  for (int w = 0; w < warp; ++w) excl += wsum[w];
  if (excl < k && k <= excl + local) {
    int acc = excl;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int h = hist[2047 - 8 * tid - q];
      if (k <= acc + h) {
        s_bin = 2047 - 8 * tid - q;
        break;
      }
      acc += h;
    }
  }
  __syncthreads();
  const int bstar = s_bin;
  uint2* dst = cand + (long long)blockIdx.x * cap;
  each([&](float f, int j) {
    if (bin_of(f) >= bstar) {
      const int slot = atomicAdd(&s_n, 1);
      if (slot < cap) dst[slot] = make_uint2(ord_key(f), (uint32_t)j);
    }
  });
  __syncthreads();
  if (tid == 0) cnt[blockIdx.x] = s_n;
}

// Sample tokens of the rows' thresholds (topk_sample_for): about kSampleRank of
// them lie at or above the threshold, so the candidates above it number kOver k
// give or take 1 / sqrt(kSampleRank) (13 %): one row in 700 falls short of k and
// is redone on the fallback path, about a batch of rows for tables of 30000 to
// 130000 tokens, a few tens of microseconds there.  At V = 40000, k = 500 that
// is 3072 tokens: against 8192 (a fifth of V) the sample contractions take 512 us
// instead of 1253 and the thresholds 245 us instead of 368; 3 rows fell short and
// took 85 us.
constexpr int kSampleRank = 56;

// Rows of the sample similarities Z [rows, ns]: each row's threshold,
// the smallest sample value in the bin of a 2048-bin linear histogram over
// [min, max] of the row's sample that holds its rs-th largest value, so that
// between rs and rs + (that bin's count) sample values are at or above it.
// 256 threads, up to 32 values each (ns a multiple of 512).
constexpr int kTauThreads = 256;

template <int kTauPer>  // values per thread: ns <= kTauPer * kTauThreads
__global__ void __launch_bounds__(kTauThreads, kTauPer > 16 ? 4 : 6) topk_tau_kernel(const float* __restrict__ Z, int V, int k, int ns,
                                                                float* __restrict__ tau) {
  griddep_wait();
  griddep_launch_dependents();
  __shared__ int hist[2048];
  __shared__ float red[2][kTauThreads / 32];
  __shared__ int s_bin;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float4* z4 = reinterpret_cast<const float4*>(Z + (long long)blockIdx.x * ns);
  // values u of this thread beyond the sample repeat its first one, and are not counted (mine: how many count)
  const int mine = tid * 4 < ns ? ((ns / 4 - tid + kTauThreads - 1) / kTauThreads) * 4 : 0;
  float v[kTauPer];
#pragma unroll
  for (int u = 0; u < kTauPer / 4; ++u) {
    const float4 q = __ldcs(z4 + (u * 4 < mine ? tid + u * kTauThreads : tid * 4 < ns ? tid : 0));
    v[4 * u] = q.x;
    v[4 * u + 1] = q.y;
    v[4 * u + 2] = q.z;
    v[4 * u + 3] = q.w;
  }
  float lo = v[0], hi = v[0];
#pragma unroll
  for (int e = 1; e < kTauPer; ++e) {
    lo = fminf(lo, v[e]);
    hi = fmaxf(hi, v[e]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  for (int b = tid; b < 2048; b += kTauThreads) hist[b] = 0;
  if (lane == 0) {
    red[0][warp] = lo;
    red[1][warp] = hi;
  }
  __syncthreads();
  lo = red[0][0];
  hi = red[1][0];
#pragma unroll
  for (int w = 1; w < kTauThreads / 32; ++w) {
    lo = fminf(lo, red[0][w]);
    hi = fmaxf(hi, red[1][w]);
  }
  const float scale = hi > lo ? 2048.f / (hi - lo) : 0.f;
  auto bin_of = [&](float x) { return min(2047, max(0, (int)((x - lo) * scale))); };
#pragma unroll
  for (int e = 0; e < kTauPer; ++e)
    if (e < mine) atomicAdd(&hist[bin_of(v[e])], 1);
  __syncthreads();
  // bins by descending index: thread t holds bins 2047 - 8t .. 2040 - 8t
  const int rs = sample_rank(V, k, ns);
  int local = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) local += hist[2047 - 8 * tid - q];
  int x = local;  // inclusive scan over the block
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  __shared__ int wsum[kTauThreads / 32];
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  int excl = x - local;
  for (int w = 0; w < warp; ++w) excl += wsum[w];
  if (excl < rs && rs <= excl + local) {
    int acc = excl;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int h = hist[2047 - 8 * tid - q];
      if (rs <= acc + h) {
        s_bin = 2047 - 8 * tid - q;
        break;
      }
      acc += h;
    }
  }
  __syncthreads();
  // the smallest sample value in the chosen bin
  const int bstar = s_bin;
  float m = INFINITY;
#pragma unroll
  for (int e = 0; e < kTauPer; ++e)
    if (bin_of(v[e]) == bstar) m = fminf(m, v[e]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
  __syncthreads();
  if (lane == 0) red[0][warp] = m;
  __syncthreads();
  if (tid == 0) {
    float t = red[0][0];
    for (int w = 1; w < kTauThreads / 32; ++w) t = fminf(t, red[0][w]);
    tau[blockIdx.x] = t;
  }
}

// Each row's cnt[r] candidates (order key, token) appended by the similarity
// contraction; with k <= n <= cap they hold the exact top k.  One warp per row
// sorts lists of up to 1024 in registers (32 lanes x up to 32 slots); longer lists go to a
// list for the block sort below; rows outside [k, cap] join the fallback list.
constexpr int kWarpSortMax = 1024;
constexpr int kSortThreads = 256;

__global__ void __launch_bounds__(kSortThreads, 2) topk_sort_warp_kernel(
    const uint2* __restrict__ cand, const int* __restrict__ cnt, int cap, int k, int row0, int nrows,
    int32_t* __restrict__ table, int32_t* __restrict__ big_rows, int* __restrict__ big_count,
    int32_t* __restrict__ fail_rows, int* __restrict__ fail_count) {
  griddep_wait();
  griddep_launch_dependents();
  __shared__ int32_t buf[kSortThreads / 32][kWarpSortMax];
  const int r = blockIdx.x * (kSortThreads / 32) + (int)(threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= nrows) return;  // whole warps
  const int n = cnt[r];
  if (n < k || n > cap || n > kCap) {
    if (lane == 0) fail_rows[atomicAdd(fail_count, 1)] = row0 + r;
    return;
  }
  if (n > kWarpSortMax) {
    if (lane == 0) big_rows[atomicAdd(big_count, 1)] = r;
    return;
  }
  const uint2* c = cand + (long long)r * cap;
  int32_t* out = table + (long long)(row0 + r) * k;
  int32_t* x = buf[threadIdx.x >> 5];
  if (n <= 128)
    warp_sort_write<4>(c, n, k, x, out);
  else if (n <= 256)
    warp_sort_write<8>(c, n, k, x, out);
  else if (n <= 512)
    warp_sort_write<16>(c, n, k, x, out);
  else
    warp_sort_write<32>(c, n, k, x, out);
}

// The rows the warp sort listed (more than 1024 candidates): one block of 256
// threads per row (up to 16 register slots each), rows taken from the list.
__global__ void __launch_bounds__(kSortThreads, 4) topk_sort_kernel(const uint2* __restrict__ cand,
                                                                   const int* __restrict__ cnt, int cap, int k,
                                                                   int row0, const int32_t* __restrict__ big_rows,
                                                                   const int* __restrict__ big_count,
                                                                   int32_t* __restrict__ table) {
  griddep_wait();
  griddep_launch_dependents();
  __shared__ uint64_t xs[kCap];
  const int nbig = *big_count;
  for (int i = blockIdx.x; i < nbig; i += gridDim.x) {
    const int r = big_rows[i];
    const int n = cnt[r];  // kWarpSortMax < n <= kCap
    const uint2* c = cand + (long long)r * cap;
    auto get = [&](int p) { return c[p]; };
    int32_t* out = table + (long long)(row0 + r) * k;
    if (n <= 8 * kSortThreads)
      sort_write_e<kSortThreads, 8>(get, n, k, xs, out);
    else
      sort_write_e<kSortThreads, 16>(get, n, k, xs, out);
    __syncthreads();  // the exchange buffer is free for the next row
  }
}

// Es[i, :] = En[floor(i * V / ns), :] for i < ns: the sample tokens, evenly spread.
__global__ void topk_gather_sample_kernel(const __nv_bfloat16* __restrict__ En, int V, int d, int ns,
                                          __nv_bfloat16* __restrict__ Es) {
  griddep_wait();
  griddep_launch_dependents();
  const int vpr = d / 8;
  const long long total = (long long)ns * vpr;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(e / vpr), v = (int)(e % vpr);
    const long long src = (long long)i * V / ns;
    reinterpret_cast<uint4*>(Es + (long long)i * d)[v] = reinterpret_cast<const uint4*>(En + src * d)[v];
  }
}

}  // namespace

cudaError_t launch_normalize_rows(const __nv_bfloat16* E, int V, int d, float* norm, __nv_bfloat16* En,
                                  cudaStream_t st) {
  const int per = 32 * kNormWarps;
  const cudaError_t e = launch_kernel(row_norms_kernel, dim3((V + per - 1) / per), dim3(kNormWarps * 32), 0, st, 1, E, V, d,
                                      norm);
  if (e != cudaSuccess) return e;
  const long long blocks = ((long long)V * (d / 8) + 256 * 8 - 1) / (256 * 8);
  return launch_kernel(scale_rows_kernel, dim3((unsigned)blocks), dim3(256), 0, st, 1, E, V, d, (const float*)norm, En);
}

// Sets the dynamic shared-memory size of the selection kernel (once per device).
template <bool kList>
cudaError_t sel_attrs() {
  static std::atomic<unsigned long long> attr_done{0};
  return set_smem_once(topk_select_kernel<kList>, (int)sizeof(SelShared), attr_done);
}

cudaError_t launch_topk_select(const float* S, long long lds, int V, int k, int row0, const int32_t* rows, int nrows,
                               const int* n_list, int32_t* table, int* status, cudaStream_t st) {
  const cudaError_t e = n_list ? sel_attrs<true>() : sel_attrs<false>();
  if (e != cudaSuccess) return e;
  return launch_kernel(n_list ? topk_select_kernel<true> : topk_select_kernel<false>, dim3(nrows), dim3(kSelThreads), (int)sizeof(SelShared), st, 1, S, lds, V,
                       k, row0, rows, n_list, table, status);
}

cudaError_t launch_topk_short(const float* S, long long lds, int V, int k, int nrows, uint2* cand, int cap, int* cnt,
                              cudaStream_t st) {
  return launch_kernel(topk_short_kernel, dim3(nrows), dim3(kShortThreads), 0, st, 1, S, lds, V, k, cand, cap, cnt);
}

cudaError_t launch_topk_tau(const float* Z, int V, int k, int ns, int nrows, float* tau, cudaStream_t st) {
  auto kernel = ns <= 16 * kTauThreads ? topk_tau_kernel<16> : topk_tau_kernel<kSample / kTauThreads>;
  return launch_kernel(kernel, dim3(nrows), dim3(kTauThreads), 0, st, 1, Z, V, k, ns, tau);
}

cudaError_t launch_topk_sort(const uint2* cand, int* cnt, int cap, int k, int row0, int nrows, int32_t* table,
                             int32_t* big_rows, int* big_count, int32_t* fail_rows, int* fail_count, int num_sms,
                             cudaStream_t st) {
  const int per = kSortThreads / 32;
  cudaError_t e = launch_kernel(topk_sort_warp_kernel, dim3((nrows + per - 1) / per), dim3(kSortThreads), 0, st, 1,
                                cand, (const int*)cnt, cap, k, row0, nrows, table, big_rows, big_count, fail_rows,
                                fail_count);
  if (e != cudaSuccess) return e;
  return launch_kernel(topk_sort_kernel, dim3(std::min(nrows, 4 * num_sms)), dim3(kSortThreads), 0, st, 1, cand,
                       (const int*)cnt, cap, k, row0, (const int32_t*)big_rows, (const int*)big_count, table);
}

cudaError_t launch_topk_gather_sample(const __nv_bfloat16* En, int V, int d, int ns, __nv_bfloat16* Es, int num_sms,
                                      cudaStream_t st) {
  return launch_kernel(topk_gather_sample_kernel, dim3(num_sms * 4), dim3(256), 0, st, 1, En, V, d, ns, Es);
}

int topk_sample() { return kSample; }
int topk_sample_for(int V, int k) {
  const long long n = (long long)((double)kSampleRank * V / (kOver * (double)k)) + 1;
  return (int)std::min<long long>(kSample, std::max<long long>(1024, (n + 511) / 512 * 512));
}
int topk_sample_min_v() { return kSampleMinV; }
int topk_cap() { return kCap; }
int topk_short_cap() { return kCap / 2; }
int topk_short_max_v() { return kShortMaxV; }

int topk_max_k() { return kSelThreads; }

}  // namespace lora
