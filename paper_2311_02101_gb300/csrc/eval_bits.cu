// Exact cost evaluation on assignments packed to one bit per variable.
//
// The weighted unsatisfied cost (Sec. 1) needs, for every clause and
// assignment, one bit: whether no literal is true. Packed 32 assignments to a
// word, a clause of K literals is K word loads and ORs for 32 assignments,
// where the byte gather (k_gather<kEval>) takes K 8-byte loads for 8 of them
// and the FP8 product a column of a 128 x 256 tile. What is left to do is the
// weighted sum, and reading the assignments once (B n bytes).
//   k_pack_bits  assignments (B x n bytes) -> X[word][variable], 32
//                assignments per word; zeroes the costs. One warp = 32
//                assignments x 128 variables: rows read 128 bytes at a time,
//                8 rows folded into the bytes of one register by shifts, a
//                4 x 4 byte transpose, one 16-byte store per lane.
//   k_pack_rows  the same from variable-major bytes (n x Bp, 0 / 1; columns past
//                the last assignment may hold anything).
//   k_bits_cost  one block = one word of assignments x a run of clauses. The
//                word's row of X (4 bytes per variable) is staged in shared
//                memory; a warp takes 32 consecutive clauses, one per lane, so
//                each lane ends with its clause's unsatisfied bits of 32
//                assignments. A 32 x 32 bit transpose gives each lane one
//                assignment's 32 clause bits, and eight look-ups of subset
//                sums of four weights (built by the warp for these 32
//                clauses) add their weights. Integers throughout: exact in
//                any order.
//   k_bits_slabs, once per formula: its clauses in order of length, 32 to a
//                slab, literal j of the 32 side by side. (A warp walks as many
//                literals as its longest clause has, and reads a literal of 32
//                clauses as one line: at lengths 2-12, n = 20000, m = 100000,
//                1000 assignments an evaluation on the lists as they came took
//                64 us, on lists in order of length 58, on slabs 25.)
// Bound by shared-memory look-ups (a literal's 32 random words over 32 banks
// take about 3.5 passes) and the transpose's shuffles.
#include <algorithm>
#include <cstdint>

#include "internal.h"
#include "dense_common.cuh"
#include "pdl.cuh"

namespace rbmsat {

namespace {

// 4 bytes from p, any alignment; [lo, hi) is the readable range
__device__ __forceinline__ uint32_t load4(const uint8_t* p, const uint8_t* lo, const uint8_t* hi) {
  const uint8_t* a = reinterpret_cast<const uint8_t*>(reinterpret_cast<uintptr_t>(p) & ~(uintptr_t)3);
  if (a >= lo && a + 8 <= hi) {
    const uint32_t w0 = reinterpret_cast<const uint32_t*>(a)[0];
    const uint32_t w1 = reinterpret_cast<const uint32_t*>(a)[1];
    return __funnelshift_r(w0, w1, 8u * (uint32_t)(p - a));
  }
  uint32_t v = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (p + k < hi) v |= (uint32_t)p[k] << (8 * k);
  return v;
}

// Variables i .. i + 3 of `rows` (at most 32) assignments of n bytes from row:
// word k has bit r set when byte i + k of assignment r is nonzero. A: the base
// and n are multiples of 4 (every row segment is an aligned word).
template <bool A>
__device__ __forceinline__ uint4 pack4(const uint8_t* row, int rows, int i, int n,
                                       const uint8_t* lo, const uint8_t* hi) {
  uint32_t a[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    uint32_t v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      v[r] = 0u;
      if (i < n && g * 8 + r < rows) {
        const uint8_t* q = row + i + (size_t)(g * 8 + r) * n;
        v[r] = A ? *reinterpret_cast<const uint32_t*>(q) : load4(q, lo, hi);
      }
    }
    // bit r of byte k: row r's byte k is nonzero
    uint32_t acc = 0u;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const uint32_t nz = ((v[r] & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | v[r];
      acc = ((acc >> 1) & 0x7F7F7F7Fu) | (nz & 0x80808080u);
    }
    a[g] = acc;
  }
  // byte k of a[0..3] -> the word of variable i + k
  const uint32_t t0 = __byte_perm(a[0], a[1], 0x5140u), t1 = __byte_perm(a[2], a[3], 0x5140u);
  const uint32_t t2 = __byte_perm(a[0], a[1], 0x7362u), t3 = __byte_perm(a[2], a[3], 0x7362u);
  return make_uint4(__byte_perm(t0, t1, 0x5410u), __byte_perm(t0, t1, 0x7632u),
                    __byte_perm(t2, t3, 0x5410u), __byte_perm(t2, t3, 0x7632u));
}

template <bool A>
__global__ void __launch_bounds__(256) k_pack_bits(const uint8_t* assign, int B, int n, int W,
                                                   int nstride, uint32_t* X, int64_t* cost,
                                                   size_t n_cost) {
  pdl_release();
  // X and the costs may still be read or added into by the launch before
  pdl_wait();
  const size_t threads = (size_t)gridDim.x * blockDim.x;
  const size_t self = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (size_t k = self; k < n_cost; k += threads) cost[k] = 0;
  const int lane = threadIdx.x & 31;
  const int groups = (n + 127) / 128;  // of 128 variables
  const size_t tasks = (size_t)groups * W, warps = threads / 32;
  const uint8_t* end = assign + (size_t)B * n;
  for (size_t task = self / 32; task < tasks; task += warps) {
    const int w = (int)(task / groups), i = (int)(task % groups) * 128 + lane * 4;
    const uint4 words =
        pack4<A>(assign + (size_t)w * 32 * n, min(32, B - w * 32), i, n, assign, end);
    if (i < nstride)  // variables n .. nstride - 1 are padding, never read
      *reinterpret_cast<uint4*>(X + (size_t)w * nstride + i) = words;
  }
}

// the low bits of the four bytes of v as 4 bits (byte k -> bit k). The mask keeps
// the other bits of bytes that nobody wrote (columns past the last assignment)
// out of the products of their neighbours.
__device__ __forceinline__ uint32_t bytes_to_bits(uint32_t v) {
  return ((v & 0x01010101u) * 0x10204080u) >> 28;
}

__global__ void __launch_bounds__(256) k_pack_rows(const uint8_t* __restrict__ xt, int Bp, int n,
                                                   int W, int nstride, uint32_t* __restrict__ X) {
  const int lane = threadIdx.x & 31;
  const int i = (int)blockIdx.x * 32 + lane;
  for (int w = (int)(blockIdx.y * 8 + (threadIdx.x >> 5)); w < W; w += (int)gridDim.y * 8) {
    if (i >= n) continue;
    const uint4* q = reinterpret_cast<const uint4*>(xt + (size_t)i * Bp + (size_t)w * 32);
    const uint4 a = __ldg(q), b = __ldg(q + 1);
    X[(size_t)w * nstride + i] =
        bytes_to_bits(a.x) | bytes_to_bits(a.y) << 4 | bytes_to_bits(a.z) << 8 |
        bytes_to_bits(a.w) << 12 | bytes_to_bits(b.x) << 16 | bytes_to_bits(b.y) << 20 |
        bytes_to_bits(b.z) << 24 | bytes_to_bits(b.w) << 28;
  }
}

// Subset sums of the warp's 32 weights (w: this lane's) in groups of four:
// lut[16 g + s] = sum of weights 4 g + k over the bits k of s.
template <typename V>
__device__ __forceinline__ void build_subset_sums(V* lut, V w, int lane) {
  const int g = lane >> 2;
  const V w0 = __shfl_sync(0xFFFFFFFFu, w, 4 * g), w1 = __shfl_sync(0xFFFFFFFFu, w, 4 * g + 1);
  const V w2 = __shfl_sync(0xFFFFFFFFu, w, 4 * g + 2), w3 = __shfl_sync(0xFFFFFFFFu, w, 4 * g + 3);
  const V hi = ((lane & 1) ? w2 : V(0)) + ((lane & 2) ? w3 : V(0));
  V* o = lut + 4 * lane;  // entries 16 g + 4 (lane % 4) + 0 .. 3
  o[0] = hi;
  o[1] = hi + w0;
  o[2] = hi + w1;
  o[3] = hi + w0 + w1;
}

// sum of the weights of the 32 clauses whose bit is set
template <typename V>
__device__ __forceinline__ V weigh(const V* lut, uint32_t bits) {
  V s = 0;
#pragma unroll
  for (int g = 0; g < 8; ++g) s += lut[16 * g + ((bits >> (4 * g)) & 15u)];
  return s;
}

// One thread per position of the slabs: copies its clause's literals and
// weight. A literal is its variable within the formula, bit 31 set when
// negated; positions past a clause's end name a word that is always zero.
__global__ void __launch_bounds__(256) k_bits_slabs(BitsFormula F, int n_pos) {
  const int pos = (int)(blockIdx.x * 256 + threadIdx.x);
  if (pos >= n_pos) return;
  const int lane = pos & 31;
  const int4 sl = F.slabs[pos >> 5];
  const int rows = F.slabs[(pos >> 5) + 1].x - sl.x;
  const int c = lane >= sl.w ? -1 : F.perm ? F.perm[pos] : sl.z + lane;
  const int2 vs = F.inst_vars[sl.y];
  int32_t* out = F.slab_lits + (size_t)sl.x * 32 + lane;
  int o = 0, len = 0;
  if (c >= 0) {
    o = F.off[c];
    len = F.off[c + 1] - o;
  }
  F.slab_w[pos] = c >= 0 ? F.w[c] : 0;
  for (int j = 0; j < rows; ++j) out[32 * j] = j < len ? F.lits[o + j] - vs.x : (vs.y + 3) / 4 * 4;
}

// V: int32_t when every 32 clauses of a slab weigh less than 2^31, else
// int64_t. RAW: a caller's DIMACS arrays, not checked before.
// PACK (one formula, one block per word): the block packs its 32 assignments
// itself and writes their costs; assign stands for X.
template <typename V, bool RAW, int WARPS, bool PACK>
__global__ void __launch_bounds__(32 * WARPS) k_bits_cost(BitsFormula F, RawFormula R,
                                                          const uint32_t* X,
                                                          const uint8_t* assign, int nstride,
                                                          int B, unsigned long long* out) {
  extern __shared__ __align__(16) uint32_t s_row[];
  __shared__ V s_lut[WARPS][128];
  __shared__ long long s_sum[WARPS][32];
  pdl_release();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int word = (int)blockIdx.x;
  // this block's clauses (RAW) or slabs begin .. end - 1, and its formula's
  // variables
  int begin, end, inst = 0, v0 = 0, nv;
  if (RAW || !F.items) {
    const int runs = RAW ? (R.m + 31) / 32 : F.n_slabs;
    begin = (int)((long long)runs * blockIdx.y / gridDim.y);
    end = (int)((long long)runs * (blockIdx.y + 1) / gridDim.y);
    nv = RAW ? R.n : F.n;
  } else {
    const int4 it = __ldg(F.items + blockIdx.y);
    begin = it.x;
    end = it.y;
    inst = it.z;
    const int2 vs = __ldg(F.inst_vars + inst);
    v0 = vs.x;
    nv = vs.y;
  }
  pdl_wait();
  const uint32_t* row = X + (size_t)word * nstride + v0;
  if constexpr (PACK) {
    const uint8_t *rows = assign + (size_t)word * 32 * nv, *end = assign + (size_t)B * nv;
    const bool aligned = ((reinterpret_cast<uintptr_t>(assign) | (uintptr_t)nv) & 3u) == 0;
    for (int k = threadIdx.x * 4; k < nv; k += 128 * WARPS)
      *reinterpret_cast<uint4*>(s_row + k) =
          aligned ? pack4<true>(rows, min(32, B - word * 32), k, nv, assign, end)
                  : pack4<false>(rows, min(32, B - word * 32), k, nv, assign, end);
  } else if ((v0 & 3) == 0) {
#pragma unroll 8
    for (int k = threadIdx.x * 4; k < nv; k += 128 * WARPS)
      *reinterpret_cast<uint4*>(s_row + k) = *reinterpret_cast<const uint4*>(row + k);
  } else {
    for (int k = threadIdx.x; k < nv; k += 32 * WARPS) s_row[k] = row[k];
  }
  if (threadIdx.x == 0) s_row[(nv + 3) / 4 * 4] = 0u;
  __syncthreads();
  V* lut = s_lut[warp];
  long long sum = 0;
  for (int k = begin + warp; k < end; k += WARPS) {
    uint32_t sat = 0;
    V w = 0;
    if constexpr (RAW) {
      const int c = 32 * k + lane;
      if (c < R.m) {
        w = R.w ? (V)R.w[c] : V(1);
        const int64_t o0 = min(max(R.off[c], (int64_t)0), R.n_lits);
        const int64_t o1 = min(max(R.off[c + 1], o0), R.n_lits);
        for (int64_t j = o0; j < o1; j += 4) {
          int32_t l[4];  // four literals in flight
#pragma unroll
          for (int u = 0; u < 4; ++u) l[u] = j + u < o1 ? R.lits[j + u] : 0;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            // |INT32_MIN| does not fit an int: such a literal is out of range
            const int64_t v = (l[u] > 0 ? (int64_t)l[u] : -(int64_t)l[u]) - 1;
            if (l[u] != 0 && v < nv) sat |= s_row[v] ^ (uint32_t)(l[u] >> 31);
          }
        }
      }
    } else {
      w = (V)__ldg(F.slab_w + 32 * k + lane);
      const int r0 = __ldg(&F.slabs[k].x), r1 = __ldg(&F.slabs[k + 1].x);
      const int32_t* q = F.slab_lits + (size_t)r0 * 32 + lane;
      int r = r0;
      for (; r + 4 <= r1; r += 4, q += 128) {
        int32_t l[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) l[u] = __ldg(q + 32 * u);
#pragma unroll
        for (int u = 0; u < 4; ++u) sat |= s_row[l[u] & 0x7FFFFFFF] ^ (uint32_t)(l[u] >> 31);
      }
      int32_t l[3];
#pragma unroll
      for (int u = 0; u < 3; ++u) l[u] = r + u < r1 ? __ldg(q + 32 * u) : (nv + 3) / 4 * 4;
#pragma unroll
      for (int u = 0; u < 3; ++u) sat |= s_row[l[u] & 0x7FFFFFFF] ^ (uint32_t)(l[u] >> 31);
    }
    __syncwarp();  // the previous 32 clauses' sums are read
    build_subset_sums<V>(lut, w, lane);
    const uint32_t bits = tc::transpose32(~sat, lane);  // lane = assignment
    __syncwarp();
    sum += (long long)weigh<V>(lut, bits);
  }
  s_sum[warp][lane] = sum;
  __syncthreads();
  if (warp == 0) {
    long long c = 0;
#pragma unroll
    for (int k = 0; k < WARPS; ++k) c += s_sum[k][lane];
    const int b = word * 32 + lane;
    if (PACK) {
      if (b < B) out[b] = (unsigned long long)c;
    } else if (b < B && c != 0) {
      atomicAdd(out + (size_t)inst * B + b, (unsigned long long)c);
    }
  }
}

int sms() {
  static int count = 0;
  if (!count) {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1)
      v = 1;
    count = v;
  }
  return count;
}

int row_bytes(int nv) { return 4 * ((nv + 3) / 4 * 4) + 16; }  // with the zero word

// Formulas scored by one launch: a block packs its own 32 assignments (32 n
// bytes) and its 8 warps take all runs of 32 clauses, at most 4 each. Back to
// back, one / two launches: m = 420, 16 assignments 3.2 / 5.0 us; m = 1280, 16 to
// 2048 assignments 4.8-5.1 / 4.9-5.8, 4096 7.6 / 7.4; m = 2048, 16 to 8192
// assignments 6.4-12.3 / 5.0-11.3. The start of a launch bounds both.
constexpr int kOneLaunchVars = 1024, kOneLaunchClauses = 1024;

// blocks of 8 warps that share an SM: room for the staged rows
int cost_blocks_per_sm(int nv) { return 226 * 1024 / (row_bytes(nv) + 11 * 1024); }

// blocks per word: about three on every SM, but no more than fit at once; each
// warp with at least two runs of 32 clauses
int cost_chunks(int W, int runs, int nv) {
  const int want = (3 * sms() + W - 1) / W;
  const int fit = std::max(1, std::min(6, cost_blocks_per_sm(nv)) * sms() / W);
  return std::max(1, std::min(std::min(want, fit), (runs + 15) / 16));
}

template <typename V, bool RAW, int WARPS, bool PACK>
cudaError_t cost_variant(const BitsFormula& F, const RawFormula& R, const uint32_t* X,
                         const uint8_t* assign, int nstride, int B, int nv, int chunks,
                         int64_t* cost, cudaStream_t st) {
  auto kern = k_bits_cost<V, RAW, WARPS, PACK>;
  const int smem = row_bytes(nv), fixed = WARPS * (128 * (int)sizeof(V) + 256);
  if (smem + fixed > 48 * 1024) {
    const cudaError_t e = allow_dynamic_smem(kern, smem);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(kern, dim3((unsigned)((B + 31) / 32), (unsigned)chunks), 32 * WARPS, smem, st,
                    F, R, X, assign, nstride, B, reinterpret_cast<unsigned long long*>(cost));
}

// rows so long that at most two blocks share an SM get blocks of 16 warps
template <typename V, bool RAW>
cudaError_t cost_launch(const BitsFormula& F, const RawFormula& R, const uint32_t* X, int nstride,
                        int B, int nv, int chunks, int64_t* cost, cudaStream_t st) {
  return cost_blocks_per_sm(nv) <= 2
             ? cost_variant<V, RAW, 16, false>(F, R, X, nullptr, nstride, B, nv, chunks, cost, st)
             : cost_variant<V, RAW, 8, false>(F, R, X, nullptr, nstride, B, nv, chunks, cost, st);
}

}  // namespace

cudaError_t launch_pack_bits(const uint8_t* assign, int B, int n, int nstride, uint32_t* X,
                             int64_t* cost, size_t n_cost, cudaStream_t st) {
  const int W = (B + 31) / 32;
  const size_t tasks = (size_t)((n + 127) / 128) * W;
  const unsigned grid = (unsigned)std::min<size_t>((tasks + 7) / 8, (size_t)8 * sms());
  const bool aligned = ((reinterpret_cast<uintptr_t>(assign) | (uintptr_t)n) & 3u) == 0;
  return launch_pdl(aligned ? k_pack_bits<true> : k_pack_bits<false>, dim3(grid), 256, 0, st, assign,
                      B, n, W, nstride, X, cost, n_cost);
}

cudaError_t launch_pack_rows(const uint8_t* xt, int Bp, int B, int n, int nstride, uint32_t* X,
                             cudaStream_t st) {
  const int W = (B + 31) / 32;
  const dim3 grid((unsigned)((n + 31) / 32), (unsigned)std::min((W + 7) / 8, 65535));
  k_pack_rows<<<grid, 256, 0, st>>>(xt, Bp, n, W, nstride, X);
  return cudaGetLastError();
}

cudaError_t launch_bits_slabs(const BitsFormula& F, cudaStream_t st) {
  if (F.n_slabs == 0) return cudaSuccess;
  k_bits_slabs<<<(unsigned)((F.n_slabs + 7) / 8), 256, 0, st>>>(F, 32 * F.n_slabs);
  return cudaGetLastError();
}

cudaError_t launch_bits_cost(const BitsFormula& F, const uint32_t* X, int nstride, int B,
                             int64_t* cost, cudaStream_t st) {
  if (F.m == 0) return cudaSuccess;
  const int chunks = F.items ? F.n_items : cost_chunks((B + 31) / 32, F.n_slabs, F.n);
  return F.wide ? cost_launch<int64_t, false>(F, RawFormula{}, X, nstride, B, F.n, chunks, cost, st)
                : cost_launch<int32_t, false>(F, RawFormula{}, X, nstride, B, F.n, chunks, cost, st);
}

bool bits_one_launch(int n, int64_t m) { return n <= kOneLaunchVars && m <= kOneLaunchClauses; }

cudaError_t launch_bits_eval(const BitsFormula& F, const uint8_t* assign, int B, int64_t* cost,
                             cudaStream_t st) {
  return F.wide ? cost_variant<int64_t, false, 8, true>(F, RawFormula{}, nullptr, assign, 0, B, F.n,
                                                        1, cost, st)
                : cost_variant<int32_t, false, 8, true>(F, RawFormula{}, nullptr, assign, 0, B, F.n,
                                                        1, cost, st);
}

cudaError_t launch_bits_eval_raw(const RawFormula& R, const uint8_t* assign, int B, int64_t* cost,
                                 cudaStream_t st) {
  return cost_variant<int64_t, true, 8, true>(BitsFormula{}, R, nullptr, assign, 0, B, R.n, 1, cost,
                                              st);
}

cudaError_t launch_bits_cost_raw(const RawFormula& R, const uint32_t* X, int nstride, int B,
                                 int64_t* cost, cudaStream_t st) {
  if (R.m == 0) return cudaSuccess;
  return cost_launch<int64_t, true>(BitsFormula{}, R, X, nstride, B, R.n,
                                    cost_chunks((B + 31) / 32, (R.m + 31) / 32, R.n), cost, st);
}

}  // namespace rbmsat
