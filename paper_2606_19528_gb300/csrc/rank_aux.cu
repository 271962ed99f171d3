// Small passes around the rank-r products (those run on the tensor cores,
// rank_tc.cu): the in-order sum of a split tile's fp32 partials, batched
// transposes with zero padding (rank sides as K-major operands), and
// zero-padded copies of rank-r matrices whose rank is not a multiple of 8.
#include <algorithm>

#include "rank_store.cuh"

namespace lora {

namespace {

// Second pass: out = sum of a tile's unit partials, in unit order.  One thread
// per 8 consecutive rank columns (a sector of each partial) of one row of
// [tile][tile_rows][rpad]; the loads of all units are independent and issued
// together.  2 or 4 lanes lie along the columns (64 bytes, or a whole line of
// a partial), the others along the rows, so that the transposed outputs (su^T, sv^T
// and dA) are stored in pieces of 16 to 64 bytes.  Launched early, this kernel shares
// its SMs with the product kernel, whose shared memory leaves little L1 to hold
// loads in flight: with all lanes along the rows a load touched a line per lane,
// and su at T = 2048, r = 64 (Qwen-shaped layer) took 43 us with its products where
// it now takes 32, the forward of a 11008 x 64 projection at T = 8192, r = 64 93 us
// where it now takes 77.
template <typename Batch, bool kRow>
__global__ void __launch_bounds__(256) reduce_partials_kernel(const __grid_constant__ Batch b, int total8) {
  if (b.early_next) griddep_launch_dependents();
  griddep_wait();
  if (!b.early_next) griddep_launch_dependents();
  const int i8 = blockIdx.x * blockDim.x + threadIdx.x;
  if (i8 >= total8) return;
  int pi = 0;
  while (pi + 1 < b.n && i8 >= (int)b.p[pi + 1].red_begin / 8) ++pi;
  const auto& P = b.p[pi];
  const int e = i8 - P.red_begin / 8;
  const int rpad = P.rpad, upt = P.upt, tr = b.tile_rows;
  const int per = tr * (rpad / 8);  // threads of a tile
  const int tile = e / per, k = e % per;
  const int g = (rpad & 31) == 0 ? 4 : 2;  // lanes along the columns
  const int j = (k / (tr * g) * g + k % g) * 8, lr = k / g % tr;
  const size_t blk = (size_t)tr * rpad;
  const float* src = b.partials + P.part_off + (size_t)tile * upt * blk + (size_t)lr * rpad + j;
  float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
  for (int u = 0; u < upt; ++u) {
    const float4 lo = __ldcg(reinterpret_cast<const float4*>(src + (size_t)u * blk));
    const float4 hi = __ldcg(reinterpret_cast<const float4*>(src + (size_t)u * blk) + 1);
    v[0] += lo.x, v[1] += lo.y, v[2] += lo.z, v[3] += lo.w;
    v[4] += hi.x, v[5] += hi.y, v[6] += hi.z, v[7] += hi.w;
  }
  uint32_t w[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) w[q] = __float_as_uint(v[q]);
  const int row = tile * tr + lr;
  if constexpr (kRow) {
    if (row < P.T) row_store8(P, row, j, w);
  } else {
    if (row < P.C) col_store8(P, row, j, w);
  }
}

// Batched transposes with zero padding (the rank sides as K-major operands of
// the tensor cores): job blockIdx.y, 64 source rows per block, through shared
// memory, 16 bytes per load (ranks that are multiples of 8) and per store.  Beside
// a contraction these blocks get few warps, so what each one waits for counts:
// element by element, 32 source rows per warp load, the transposes of a
// Qwen-shaped layer (T = 4096, r = 64) took 26 us alone and 129 us there, on the side
// stream's critical path; this takes 45 us there, the fork from the forward's
// stream included.
constexpr int kTrRows = 64, kTrMaxR = 128;

__global__ void __launch_bounds__(256) transposes_kernel(const __grid_constant__ TransposeJobs jobs) {
  griddep_wait();
  griddep_launch_dependents();
  __shared__ __align__(16) __nv_bfloat16 tile[kTrRows * (kTrMaxR + 8)];
  const int k = blockIdx.y;
  const int n = jobs.n[k], r = jobs.r[k], r8 = jobs.r8[k], ld = jobs.ld[k];
  const int c0 = blockIdx.x * kTrRows;
  if (c0 >= n) return;  // the whole block
  const int rows = min(kTrRows, n - c0), pitch = r8 + 8;
  const __nv_bfloat16* src = jobs.src[k] + (size_t)c0 * ld;
  if (r == r8 && (ld & 7) == 0) {  // 16-byte rows (every source is 16-byte aligned)
    const int vpr = r8 / 8;
    for (int e = threadIdx.x; e < rows * vpr; e += 256) {
      const int c = e / vpr, v = e % vpr;
      *reinterpret_cast<uint4*>(tile + c * pitch + v * 8) = __ldg(reinterpret_cast<const uint4*>(src + (size_t)c * ld) + v);
    }
  } else {
    for (int e = threadIdx.x; e < rows * r8; e += 256) {
      const int c = e / r8, j = e % r8;
      tile[c * pitch + j] = j < r ? src[(size_t)c * ld + j] : __float2bfloat16_rn(0.f);
    }
  }
  __syncthreads();
  const int groups = rows / 8;  // n is a multiple of 8
  for (int e = threadIdx.x; e < r8 * groups; e += 256) {
    const int j = e / groups, g = e % groups;
    __align__(16) __nv_bfloat16 o[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) o[i] = tile[(g * 8 + i) * pitch + j];
    *reinterpret_cast<uint4*>(jobs.dst[k] + (size_t)j * n + c0 + g * 8) = *reinterpret_cast<const uint4*>(o);
  }
}

__global__ void pad_cols_kernel(const __nv_bfloat16* __restrict__ src, int rows, int r,
                                __nv_bfloat16* __restrict__ dst, int ld_dst) {
  griddep_wait();
  griddep_launch_dependents();
  const size_t n = (size_t)rows * ld_dst;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const size_t row = i / ld_dst;
    const int j = (int)(i % ld_dst);
    dst[i] = j < r ? src[row * r + j] : __float2bfloat16_rn(0.f);
  }
}

// Failure-detection self-check: one thread waits, with the library's bounded
// wait, on a barrier that nothing arrives on; the wait gives up after
// limit_ns, records the timeout in the status word and the kernel returns.
__global__ void wait_probe_kernel(int* status, long long limit_ns) {
  griddep_wait();
  griddep_launch_dependents();
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    abort_flag = 0;
    fence_mbar_init();
    const WaitCtl wc{status, limit_ns};
    mbar_wait(smem_u32(&bar), 0, wc, &abort_flag);
  }
}

int grid_for(size_t n, int threads) {
  size_t b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > 65535) b = 65535;
  return (int)b;
}

}  // namespace

cudaError_t launch_transposes(const TransposeJobs& jobs, cudaStream_t st) {
  if (jobs.count <= 0 || jobs.max_n <= 0) return cudaSuccess;
  return launch_kernel(transposes_kernel, dim3((jobs.max_n + kTrRows - 1) / kTrRows, jobs.count), dim3(256), 0, st, 1,
                       jobs);
}

cudaError_t launch_reduce_rows(const RowBatch& b, cudaStream_t st) {
  if (b.red_total <= 0) return cudaSuccess;
  const int total8 = b.red_total / 8;
  return launch_kernel(reduce_partials_kernel<RowBatch, true>, dim3((total8 + 255) / 256), dim3(256), 0, st, 1, b,
                       total8);
}

cudaError_t launch_wait_probe(int* status, long long limit_ns, cudaStream_t st) {
  return launch_kernel(wait_probe_kernel, dim3(1), dim3(32), 0, st, 1, status, limit_ns);
}

cudaError_t launch_reduce_cols(const ColBatch& b, cudaStream_t st) {
  if (b.red_total <= 0) return cudaSuccess;
  const int total8 = b.red_total / 8;
  return launch_kernel(reduce_partials_kernel<ColBatch, false>, dim3((total8 + 255) / 256), dim3(256), 0, st, 1, b,
                       total8);
}

cudaError_t launch_pad_cols(const __nv_bfloat16* src, int rows, int r, __nv_bfloat16* dst, int ld_dst,
                            cudaStream_t st) {
  const size_t n = (size_t)rows * ld_dst;
  return launch_kernel(pad_cols_kernel, dim3(grid_for(n, 256)), dim3(256), 0, st, 1, src, rows, r, dst, ld_dst);
}

}  // namespace lora
