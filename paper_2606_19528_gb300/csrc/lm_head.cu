// Reduced-vocabulary LM-head cross entropy with logits masking (Sections
// "Softmax Approximation" and "Logits Masking"): the index and element-wise
// passes around the two tensor-core contractions (fused_gemm.cu), which
// compute the logits of the trainable positions over the reduced vocabulary
// J and the hidden-state gradient.
//   vocab_mark      J = union of the trainable targets' first k top-k entries
//   compact         J and the trainable positions as ascending lists and the
//                   latter's inverse map: 128 blocks take a vocabulary segment
//                   each, counting the flags before it themselves (tables past
//                   2^20 tokens: vocab_count first), one block the positions,
//                   with the check of their targets
//   prepare_rows    rows of h (trainable positions) and of E (J) made dense, each
//                   trainable target's column in J, zeros in the other rows of dh
//                   and the other positions' losses;
//                   it reads the counts on the device, so it runs while the host
//                   waits for them
//   ce_rows         per trainable position: log-sum-exp over J merged from the
//                   logits contraction's per-group partials, its loss, and G =
//                   softmax_J - onehot(target) in bf16 for the dh contraction in
//                   one streaming pass over the logits; the last block writes the
//                   losses' sum in a fixed order
//   scatter_rows    dh rows of trainable positions
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace lora {

namespace {

constexpr int kScanThreads = 1024;

// One block of 128 threads per position t: if t is trainable, flags[v] = 1
// for the k entries v of its target's table row (per 1024 entries, all loads
// of a thread issued before its stores).
constexpr int kMarkThreads = 128;

__global__ void __launch_bounds__(kMarkThreads) vocab_mark_kernel(const int32_t* __restrict__ targets,
                                                                  const uint8_t* __restrict__ mask, int T,
                                                                  const int32_t* __restrict__ topk, long long ld,
                                                                  int k, int V, uint8_t* __restrict__ flags,
                                                                  int32_t* __restrict__ counts) {
  griddep_wait();
  griddep_launch_dependents();
  for (int t = blockIdx.x; t < T; t += gridDim.x) {
    if (mask && !mask[t]) continue;
    const int y = targets[t];
    if (y < 0 || y >= V) {
      if (threadIdx.x == 0) counts[2] = 1;  // invalid target
      continue;
    }
    const int32_t* row = topk + (long long)y * ld;
    for (int j0 = 0; j0 < k; j0 += 8 * kMarkThreads) {
      int v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int j = j0 + threadIdx.x + q * kMarkThreads;
        v[q] = j < k ? row[j] : 0;
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (j0 + threadIdx.x + q * kMarkThreads < k) {
          if (v[q] < 0 || v[q] >= V)
            counts[2] = 1;  // invalid table entry
          else
            flags[v[q]] = 1;
        }
      }
    }
  }
}

// Exclusive scan of one value per thread over the block; returns the total.
__device__ __forceinline__ int block_scan(int v, int* excl) {
  __shared__ int warp_tot[kScanThreads / 32];
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
    int w = lane < kScanThreads / 32 ? warp_tot[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < kScanThreads / 32) warp_tot[lane] = w;  // inclusive
  }
  __syncthreads();
  const int before = (warp > 0 ? warp_tot[warp - 1] : 0) + x - v;
  const int total = warp_tot[kScanThreads / 32 - 1];
  __syncthreads();
  *excl = before;
  return total;
}

// Ascending compaction of the set entries of [0, n) (flag(i) != 0): list[k] =
// first + the k-th set i, and inv[i] = its position or -1.  One block.
template <typename Flag>
__device__ int compact(int n, Flag flag, int first, int32_t* list, int32_t* inv) {
  const int per = (n + kScanThreads - 1) / kScanThreads;
  const int b0 = min(n, (int)threadIdx.x * per), b1 = min(n, b0 + per);
  int cnt = 0;
  for (int i = b0; i < b1; ++i) cnt += flag(i) ? 1 : 0;
  int off;
  const int total = block_scan(cnt, &off);
  for (int i = b0; i < b1; ++i) {
    if (flag(i)) {
      list[off] = first + i;
      if (inv) inv[i] = off;
      ++off;
    } else if (inv) {
      inv[i] = -1;
    }
  }
  return total;
}

constexpr int kSegs = 128;  // vocabulary segments of the multi-block compaction

// Set flags per vocabulary segment (every token in full-vocabulary mode).
__global__ void __launch_bounds__(256) vocab_count_kernel(const uint8_t* __restrict__ flags, int V, int full,
                                                          int32_t* __restrict__ seg_counts) {
  griddep_wait();
  griddep_launch_dependents();
  const int seg = (V + kSegs - 1) / kSegs;
  const int b0 = min(V, (int)blockIdx.x * seg), b1 = min(V, b0 + seg);
  int c = 0;
  for (int i = b0 + threadIdx.x; i < b1; i += blockDim.x) c += (full || flags[i]) ? 1 : 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  __shared__ int wsum[8];
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < 8; ++w) t += wsum[w];
    seg_counts[blockIdx.x] = t;
  }
}

// Set flags (bytes 0 or 1) in [0, n), by the whole block; every thread gets the sum.
__device__ int count_flags(const uint8_t* __restrict__ flags, int n) {
  const int n16 = n / 16;
  const uint4* f4 = reinterpret_cast<const uint4*>(flags);
  int c = 0;
  for (int i = threadIdx.x; i < n16; i += kScanThreads) {
    const uint4 q = f4[i];
    c += __popc(q.x) + __popc(q.y) + __popc(q.z) + __popc(q.w);
  }
  const int t = 16 * n16 + (int)threadIdx.x;
  if (threadIdx.x < 16 && t < n) c += flags[t];
  int excl;
  return block_scan(c, &excl);
}

// Blocks 0 .. kSegs - 1: their segment of J (ascending); block kSegs: the
// trainable positions, their inverse map, the counts, and the check that every
// trainable target lies in J.  seg_counts null: each block counts the flags
// before its segment (at most 2^20 bytes, from L2) instead of a launch of its own
// counting the segments first.
__global__ void __launch_bounds__(kScanThreads) compact_kernel(const uint8_t* __restrict__ flags, int V, int full,
                                                               const int32_t* __restrict__ seg_counts,
                                                               const uint8_t* __restrict__ mask, int T,
                                                               const int32_t* __restrict__ targets, int32_t* J,
                                                               int32_t* tl, int32_t* tpos, int32_t* counts) {
  griddep_wait();
  griddep_launch_dependents();
  if (blockIdx.x < kSegs) {
    const int seg = (V + kSegs - 1) / kSegs;
    const int b0 = min(V, (int)blockIdx.x * seg), b1 = min(V, b0 + seg);
    int base = b0;
    if (!full) {
      base = 0;
      if (seg_counts)
        for (int b = 0; b < (int)blockIdx.x; ++b) base += seg_counts[b];
      else
        base = count_flags(flags, b0);
    }
    const int n = compact(b1 - b0, [&](int i) { return full || flags[b0 + i] != 0; }, b0, J + base, nullptr);
    if (blockIdx.x == kSegs - 1 && threadIdx.x == 0) counts[1] = base + n;
    return;
  }
  auto trainable = [&](int t) { return !mask || mask[t] != 0; };
  const int nT = compact(T, trainable, 0, tl, tpos);
  for (int t = threadIdx.x; t < T; t += kScanThreads) {
    if (!trainable(t)) continue;
    const int y = targets[t];
    if (y < 0 || y >= V || (!full && flags[y] == 0)) counts[2] = 1;  // out of range or outside J
  }
  if (threadIdx.x == 0) counts[0] = nT;
}

__global__ void gather_rows_kernel(const __nv_bfloat16* __restrict__ src, long long ld,
                                   const int32_t* __restrict__ idx, int n, int d, __nv_bfloat16* __restrict__ dst) {
  griddep_wait();
  griddep_launch_dependents();
  const int vpr = d / 8;  // 16-byte vectors per row
  const long long total = (long long)n * vpr;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(e / vpr), v = (int)(e % vpr);
    const uint4* s = reinterpret_cast<const uint4*>(src + (long long)idx[i] * ld) + v;
    reinterpret_cast<uint4*>(dst + (long long)i * d)[v] = __ldg(s);
  }
}

// One warp per row, four 16-byte loads in flight per lane: the trainable rows of
// h (and their targets' columns in the ascending J, by a 32-way search), the rows
// of E in J (not when J is the whole vocabulary: E is read in place), and zeros in
// the rows of dh and the losses outside the trainable set (not after a failed check: the call's
// outputs stay untouched).
__global__ void __launch_bounds__(256) prepare_rows_kernel(const __nv_bfloat16* __restrict__ h,
                                                           const __nv_bfloat16* __restrict__ E, int d, int T, int V,
                                                           const int32_t* __restrict__ tl,
                                                           const int32_t* __restrict__ tpos,
                                                           const int32_t* __restrict__ J,
                                                           const int32_t* __restrict__ targets,
                                                           const int32_t* __restrict__ counts,
                                                           __nv_bfloat16* __restrict__ ht, __nv_bfloat16* __restrict__ ej,
                                                           int32_t* __restrict__ ycol, __nv_bfloat16* __restrict__ dh,
                                                           float* __restrict__ token_loss) {
  griddep_wait();
  griddep_launch_dependents();
  const int nT = counts[0], nJ = counts[1];
  if (counts[2] != 0) return;
  const int nE = nJ < V ? nJ : 0;
  const int vpr = d / 8, lane = threadIdx.x & 31;
  const long long warps = (long long)gridDim.x * 8, total = (long long)nT + nE + (dh || token_loss ? T : 0);
  for (long long w = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); w < total; w += warps) {
    if (w >= (long long)nT + nE) {
      const int t = (int)(w - nT - nE);
      if (tpos[t] < 0) {
        if (dh)
          for (int v = lane; v < vpr; v += 32)
            reinterpret_cast<uint4*>(dh + (long long)t * d)[v] = make_uint4(0u, 0u, 0u, 0u);
        if (token_loss && lane == 0) token_loss[t] = 0.f;
      }
      continue;
    }
    const bool isT = w < nT;
    const int i = (int)(isT ? w : w - nT);
    const int src = isT ? tl[i] : J[i];
    const uint4* s = reinterpret_cast<const uint4*>((isT ? h : E) + (long long)src * d);
    uint4* o = reinterpret_cast<uint4*>((isT ? ht : ej) + (long long)i * d);
    for (int v0 = lane; v0 < vpr; v0 += 4 * 32) {
      uint4 q[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (v0 + u * 32 < vpr) q[u] = __ldg(s + v0 + u * 32);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (v0 + u * 32 < vpr) o[v0 + u * 32] = q[u];
    }
    if (isT) {
      // J[lo] <= y < J[hi] (J[nJ] beyond every token); y is in J
      const int y = targets[src];
      int lo = 0, hi = nJ;
      while (hi - lo > 1) {  // uniform across the warp
        const int step = (hi - lo + 31) / 32, p = lo + lane * step;
        const unsigned le = __ballot_sync(0xffffffffu, p < hi && J[min(p, nJ - 1)] <= y);
        const int k = 31 - __clz((int)le);  // lane 0's probe, J[lo], always counts
        const int l2 = lo + k * step;
        hi = min(hi, l2 + step);
        lo = l2;
      }
      if (lane == 0) ycol[i] = lo;
    }
  }
}

// Combine two (max, sum of exp(x - max)) pairs.
__device__ __forceinline__ void lse_merge(float& m, float& s, float m2, float s2) {
  if (m2 > m) {
    s = s * expf(m - m2) + s2;
    m = m2;
  } else if (m2 > -INFINITY) {
    s += s2 * expf(m2 - m);
  }
}

// The losses' sum in a fixed order (fp64), by one block of 256 threads.
__device__ void finish_body(const float* rowloss, int nT, float* loss) {
  __shared__ double part[256];
  double acc = 0.0;
  for (int i = threadIdx.x; i < nT; i += blockDim.x) acc += (double)rowloss[i];
  part[threadIdx.x] = acc;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *loss = (float)part[0];
}

// One block per (trainable position i, chunk of its logits).  It merges the
// row's log-sum-exp from the logits contraction's per-group (max, sum of exp)
// partials (every block of a row the same way, so the same bits; its first logits
// are on their way meanwhile) and writes G[i, :] = bf16(exp(z - lse_i) - [j ==
// ycol_i]) of its chunk, zeros in [nJ, ldg): one read of the fp32 logits, 16-byte
// loads and 8-byte stores.  The block of a row's first chunk also writes its loss
// lse - z[i, ycol[i]]; the last of those to finish sums them.  Rows are cut so that
// about eight blocks per SM run, in multiples of kGradStep columns: more blocks
// would repeat the merge.  (As two launches, one for the rows and one for G: 12.2
// + 9.8 us for 614 positions and 8648 tokens; this 17.5 us.)
constexpr int kGradStep = 4096;  // four 16-byte loads per thread

__global__ void __launch_bounds__(256) ce_rows_kernel(const float2* __restrict__ part, int ld_part, int ngroups,
                                                      const float* __restrict__ Z, int ldz, int nJ,
                                                      const int32_t* __restrict__ ycol, int nT, int chunk,
                                                      __nv_bfloat16* __restrict__ G, int ldg, float* rowloss,
                                                      const int32_t* __restrict__ tl, float* __restrict__ token_loss,
                                                      float* __restrict__ loss, int* __restrict__ done) {
  griddep_wait();
  griddep_launch_dependents();
  __shared__ float sm[8], ss[8];
  __shared__ int s_last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunks = (ldg + chunk - 1) / chunk;
  const int i = (int)blockIdx.x / chunks, c = (int)blockIdx.x % chunks;
  const float* z = Z + (long long)i * ldz;
  __nv_bfloat16* g = G + (long long)i * ldg;
  const int j_end = min(ldg, (c + 1) * chunk);
  float4 q[4];
  auto fetch = [&](int j0) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = j0 + 1024 * u;
      // ldz >= j + 4: inside the row
      q[u] = j < nJ && j < j_end ? __ldcs(reinterpret_cast<const float4*>(z + j)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  int j0 = c * chunk + 4 * (int)threadIdx.x;
  fetch(j0);
  const float2* pr = part + (long long)i * ld_part;
  float m = -INFINITY, s = 0.f;
  for (int p = threadIdx.x; p < ngroups; p += blockDim.x) {
    const float2 w = pr[p];
    lse_merge(m, s, w.x, w.y);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, m, o), s2 = __shfl_xor_sync(0xffffffffu, s, o);
    lse_merge(m, s, m2, s2);
  }
  if (lane == 0) {
    sm[warp] = m;
    ss[warp] = s;
  }
  const int yc = ycol[i];
  __syncthreads();
  float M = sm[0], Sm = ss[0];
#pragma unroll
  for (int w = 1; w < 8; ++w) lse_merge(M, Sm, sm[w], ss[w]);
  const float lse = M + logf(Sm);
  for (; j0 < j_end; j0 += kGradStep) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = j0 + 1024 * u;
      if (j < j_end) {
        const float zv[4] = {q[u].x, q[u].y, q[u].z, q[u].w};
        float o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) o[e] = j + e < nJ ? expf(zv[e] - lse) - (j + e == yc ? 1.f : 0.f) : 0.f;
        *reinterpret_cast<uint2*>(g + j) = make_uint2(pack_bf16x2(o[0], o[1]), pack_bf16x2(o[2], o[3]));
      }
    }
    if (j0 + kGradStep < j_end) fetch(j0 + kGradStep);
  }
  if (c != 0) return;  // uniform across the block
  if (threadIdx.x == 0) {
    const float l = lse - z[yc];
    rowloss[i] = l;
    if (token_loss) token_loss[tl[i]] = l;
    __threadfence();
    s_last = atomicAdd(done, 1) == nT - 1;
  }
  __syncthreads();
  if (s_last) {  // every rowloss is written and visible
    __threadfence();
    finish_body(rowloss, nT, loss);
  }
}

// dst[idx[i], :] = src[i, :] for i < n.
__global__ void scatter_rows_kernel(const __nv_bfloat16* __restrict__ src, const int32_t* __restrict__ idx, int n, int d,
                                    __nv_bfloat16* __restrict__ dst) {
  griddep_wait();
  griddep_launch_dependents();
  const int vpr = d / 8;
  const long long total = (long long)n * vpr;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(e / vpr), v = (int)(e % vpr);
    reinterpret_cast<uint4*>(dst + (long long)idx[i] * d)[v] = reinterpret_cast<const uint4*>(src + (long long)i * d)[v];
  }
}

int grid_for(long long n, int threads, int cap) {
  long long b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > cap) b = cap;
  return (int)b;
}

}  // namespace

cudaError_t launch_ce_index(const CeIndex& a, cudaStream_t st) {
  cudaError_t e;
  if (a.topk) {
    e = launch_kernel(vocab_mark_kernel, dim3(std::min(a.T, 65535)), dim3(kMarkThreads), 0, st, 1, a.targets,
                      a.mask, a.T, a.topk, a.ld_topk, a.k, a.V, a.flags, a.counts);
    if (e != cudaSuccess) return e;
  }
  const int full = a.topk ? 0 : 1;
  const bool counted = !full && a.V > (1 << 20);
  if (counted) {
    e = launch_kernel(vocab_count_kernel, dim3(kSegs), dim3(256), 0, st, 1, (const uint8_t*)a.flags, a.V, full,
                      a.seg_counts);
    if (e != cudaSuccess) return e;
  }
  return launch_kernel(compact_kernel, dim3(kSegs + 1), dim3(kScanThreads), 0, st, 1, (const uint8_t*)a.flags, a.V,
                       full, (const int32_t*)(counted ? a.seg_counts : nullptr), a.mask, a.T, a.targets, a.J, a.tl,
                       a.tpos, a.counts);
}

cudaError_t launch_ce_prepare(const CeIndex& a, const __nv_bfloat16* h, const __nv_bfloat16* E, int d,
                              __nv_bfloat16* ht, __nv_bfloat16* ej, __nv_bfloat16* dh, float* token_loss, int num_sms,
                              cudaStream_t st) {
  return launch_kernel(prepare_rows_kernel, dim3(num_sms * 8), dim3(256), 0, st, 1, h, E, d, a.T, a.V,
                       (const int32_t*)a.tl, (const int32_t*)a.tpos, (const int32_t*)a.J, a.targets,
                       (const int32_t*)a.counts, ht, ej, a.ycol, dh, token_loss);
}

cudaError_t launch_gather_rows(const __nv_bfloat16* src, long long ld, const int32_t* idx, int n, int d,
                               __nv_bfloat16* dst, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  return launch_kernel(gather_rows_kernel, dim3(grid_for((long long)n * (d / 8), 256, 8192)), dim3(256), 0, st, 1,
                       src, ld, idx, n, d, dst);
}

cudaError_t launch_ce_rows(const float2* lse_part, int ld_part, const float* Z, int ldz, int nJ, const int32_t* ycol,
                           int nT, float* rowloss, const int32_t* tl, float* token_loss, float* loss, int* done,
                           __nv_bfloat16* G, int ldg, int num_sms, cudaStream_t st) {
  if (nT <= 0) return cudaSuccess;
  const int ngroups = (nJ + gemm_lse_group() - 1) / gemm_lse_group();
  // columns per block: rows cut into as many parts as give eight blocks per SM
  const int steps = (ldg + kGradStep - 1) / kGradStep, parts = std::min(steps, std::max(1, (8 * num_sms + nT - 1) / nT));
  const int chunk = (steps + parts - 1) / parts * kGradStep;
  const long long blocks = (long long)nT * ((ldg + chunk - 1) / chunk);
  return launch_kernel(ce_rows_kernel, dim3((unsigned)blocks), dim3(256), 0, st, 1, lse_part, ld_part, ngroups, Z, ldz,
                       nJ, ycol, nT, chunk, G, ldg, rowloss, tl, token_loss, loss, done);
}

cudaError_t launch_scatter_rows(const __nv_bfloat16* src, const int32_t* idx, int n, int d, __nv_bfloat16* dst,
                                cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  return launch_kernel(scatter_rows_kernel, dim3(grid_for((long long)n * (d / 8), 256, 8192)), dim3(256), 0, st, 1,
                       src, idx, n, d, dst);
}

}  // namespace lora
