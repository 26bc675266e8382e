// Chain state between the device layout (variable-major, n x Bp) and the
// ABI's (chain-major, B x n), and the best assignment over the chains.
//   k_state_out / k_state_in  transposes through a shared-memory tile, so that
//                both sides are read and written in runs of 32 elements and the
//                host copies one contiguous block.
//   k_best_chain one block per formula: its lowest best cost, ties to the
//                lowest chain.
//   k_best_copy  that chain's best assignment as consecutive bytes.
#include <algorithm>
#include <cstdint>

#include "internal.h"

namespace rbmsat {

namespace {

template <typename V>
__global__ void k_state_out(const V* __restrict__ src, int Bp, int n, int b_begin, int b_count,
                            V* __restrict__ dst) {
  __shared__ V tile[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int i0 = (int)blockIdx.y * 32; i0 < n; i0 += (int)gridDim.y * 32) {
    const int b = (int)blockIdx.x * 32 + tx;
    for (int r = ty; r < 32; r += 8)
      if (i0 + r < n && b < b_count) tile[r][tx] = src[(size_t)(i0 + r) * Bp + b_begin + b];
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {
      const int bo = (int)blockIdx.x * 32 + r;
      if (bo < b_count && i0 + tx < n) dst[(size_t)bo * n + i0 + tx] = tile[tx][r];
    }
    __syncthreads();
  }
}

__device__ __forceinline__ uint8_t as_state(uint8_t v) { return v != 0; }
__device__ __forceinline__ float as_state(float v) { return v; }

template <typename V>
__global__ void k_state_in(const V* __restrict__ src, int Bp, int n, int b_begin, int b_count,
                           V* __restrict__ dst) {
  __shared__ V tile[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int i0 = (int)blockIdx.y * 32; i0 < n; i0 += (int)gridDim.y * 32) {
    for (int r = ty; r < 32; r += 8) {
      const int bo = (int)blockIdx.x * 32 + r;
      if (bo < b_count && i0 + tx < n) tile[r][tx] = as_state(src[(size_t)bo * n + i0 + tx]);
    }
    __syncthreads();
    const int b = (int)blockIdx.x * 32 + tx;
    for (int r = ty; r < 32; r += 8)
      if (i0 + r < n && b < b_count) dst[(size_t)(i0 + r) * Bp + b_begin + b] = tile[tx][r];
    __syncthreads();
  }
}

__global__ void __launch_bounds__(256) k_best_chain(const int64_t* __restrict__ best, int Bp, int B,
                                                    int64_t* __restrict__ cost,
                                                    int32_t* __restrict__ chain) {
  __shared__ int64_t s_c[256];
  __shared__ int32_t s_b[256];
  const int64_t* row = best + (size_t)blockIdx.x * Bp;
  int64_t c = INT64_MAX;
  int32_t at = INT32_MAX;
  for (int b = threadIdx.x; b < B; b += 256) {
    const int64_t v = row[b];
    if (v < c || (v == c && b < at)) {
      c = v;
      at = b;
    }
  }
  s_c[threadIdx.x] = c;
  s_b[threadIdx.x] = at;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) {
      const int64_t v = s_c[threadIdx.x + h];
      const int32_t o = s_b[threadIdx.x + h];
      if (v < s_c[threadIdx.x] || (v == s_c[threadIdx.x] && o < s_b[threadIdx.x])) {
        s_c[threadIdx.x] = v;
        s_b[threadIdx.x] = o;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    cost[blockIdx.x] = s_c[0];
    chain[blockIdx.x] = s_b[0];
  }
}

__global__ void __launch_bounds__(256) k_best_copy(const uint8_t* __restrict__ best_xt, int Bp,
                                                   int n, const int2* __restrict__ var_inst,
                                                   const int32_t* __restrict__ chain,
                                                   uint8_t* __restrict__ out) {
  const int i = (int)blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  const int k = var_inst ? __ldg(var_inst + i).x : 0;
  out[i] = best_xt[(size_t)i * Bp + __ldg(chain + k)];
}

dim3 tile_grid(int b_count, int n) {
  return dim3((unsigned)((b_count + 31) / 32), (unsigned)std::min((n + 31) / 32, 65535));
}

}  // namespace

cudaError_t launch_state_out(const uint8_t* src, int Bp, int n, int b_begin, int b_count,
                             uint8_t* dst, cudaStream_t st) {
  k_state_out<uint8_t><<<tile_grid(b_count, n), 256, 0, st>>>(src, Bp, n, b_begin, b_count, dst);
  return cudaGetLastError();
}
cudaError_t launch_state_out(const float* src, int Bp, int n, int b_begin, int b_count, float* dst,
                             cudaStream_t st) {
  k_state_out<float><<<tile_grid(b_count, n), 256, 0, st>>>(src, Bp, n, b_begin, b_count, dst);
  return cudaGetLastError();
}
cudaError_t launch_state_in(const uint8_t* src, int Bp, int n, int b_begin, int b_count,
                            uint8_t* dst, cudaStream_t st) {
  k_state_in<uint8_t><<<tile_grid(b_count, n), 256, 0, st>>>(src, Bp, n, b_begin, b_count, dst);
  return cudaGetLastError();
}
cudaError_t launch_state_in(const float* src, int Bp, int n, int b_begin, int b_count, float* dst,
                            cudaStream_t st) {
  k_state_in<float><<<tile_grid(b_count, n), 256, 0, st>>>(src, Bp, n, b_begin, b_count, dst);
  return cudaGetLastError();
}

cudaError_t launch_best(const DevFormula& F, const DevChains& C, int64_t* cost, int32_t* chain,
                        uint8_t* assign, cudaStream_t st) {
  k_best_chain<<<F.n_inst, 256, 0, st>>>(C.best, C.Bp, C.B, cost, chain);
  if (assign)
    k_best_copy<<<(F.n + 255) / 256, 256, 0, st>>>(C.best_xt, C.Bp, F.n, F.var_inst, chain, assign);
  return cudaGetLastError();
}

}  // namespace rbmsat
