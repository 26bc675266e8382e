// Learned proposal: a message-passing network over the variable-clause
// incidence of a formula, trained on the solver's own best assignments, that
// supplies the chains' initial assignments (the paper names learned initial
// assignments as complementary to RbmSAT, Sec. 2).
//
//   f_v = [pos_v / deg_v - 1/2, log(1 + deg_v) / 4, 1],  g_c = [log(w_c) / 8, len_c / 4, 1]
//   h_v^0 = relu(Wf f_v),  h_c^0 = relu(Wg g_c)                      (H = 64)
//   layer l: m_c = mean_{(v,s) in c} s h_v^{l-1}
//            h_c^l = relu(Wc_l [m_c ; h_c^{l-1}] + bc_l)
//            a_v = mean_{(c,s) : v in c} s h_c^l
//            h_v^l = relu(Wv_l [a_v ; h_v^{l-1}] + bv_l)
//   z_v = wo . h_v^L + bo,  p_v = sigmoid(z_v),  loss = mean_v softplus(z_v) - y_v z_v
//
// Weight matrices are used in BF16 (rounded from FP32 master weights after
// every Adam step); activations, biases and all sums are FP32. Every kernel is
// hand-written. A step of the network is one launch per layer and side:
//   k_mp_embed   input features and both projections (h_v^0, h_c^0)
//   k_mp_fwd     64 rows at a time: the signed means of the other side's rows
//                (gathered along the clause or variable incidence lists the
//                Gibbs round walks), then relu(W [mean ; own] + b) on the
//                tensor cores
//   k_mp_out     read-out, loss, and its gradient
//   k_mp_bwd     64 rows at a time: the rows' gradient (gathered signed sums of
//                the other side's gradient plus the gradient of their own row),
//                masked by relu, stays on the chip and feeds both the input
//                gradient and the weight gradient
//   k_mp_embed_bwd, k_mp_sum  the projections' gradients; all partial sums
// What bounds a step is moving the rows (64 floats, 256 bytes) through HBM:
// the means, the layers' inputs and the masked gradients are formed in shared
// memory as the tensor cores' operands instead of passing through memory as
// FP32 arrays between launches. Weight gradients are summed in a fixed order
// (per block in registers over its rows, then over blocks); no atomics.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>
#include <vector>

#include "internal.h"
#include "pdl.cuh"
#include "philox.cuh"

namespace rbmsat {

namespace {

constexpr int kH = 64;
__device__ __forceinline__ float relu(float x) { return x > 0.f ? x : 0.f; }

constexpr int kTile = 64;      // rows per tile of the layer kernels
constexpr int kLdD = kH + 8;   // BF16 elements per row of a 64-column operand tile
constexpr int kLdX = 2 * kH + 8;  // and of a 128-column one (both: 16-byte rows, ldmatrix
                                  // without bank conflicts)
constexpr int kWCount = kH * 2 * kH;   // weights of a layer
constexpr int kPart = kWCount + kH;    // a block's weight and bias gradient

// ------------------------------------------------------- features, projections
// relu(W x) of three inputs for output columns 2 lane, 2 lane + 1
struct Proj3 {
  float w[6];
  __device__ __forceinline__ void load(const __nv_bfloat16* W, int lane) {
#pragma unroll
    for (int k = 0; k < 6; ++k) w[k] = __bfloat162float(W[6 * lane + k]);
  }
  __device__ __forceinline__ float2 apply(float x0, float x1, float x2) const {
    float a = w[0] * x0, b = w[3] * x0;
    a = fmaf(w[1], x1, a);
    b = fmaf(w[4], x1, b);
    a = fmaf(w[2], x2, a);
    b = fmaf(w[5], x2, b);
    return make_float2(relu(a), relu(b));
  }
};

// One warp = 32 rows: each lane computes one row's features, then the warp
// writes the 32 rows' projections one after another (256 bytes each). Blocks
// below nbv take variables, the others clauses.
__global__ void __launch_bounds__(256) k_mp_embed(DevFormula F, const __nv_bfloat16* Wf,
                                                  const __nv_bfloat16* Wg, int nbv, float* f,
                                                  float* g, float* inv_len, float* inv_deg,
                                                  float* hv, float* hc) {
  pdl_wait();
  pdl_release();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool var = (int)blockIdx.x < nbv;
  const int rows = var ? F.n : F.m;
  const int r0 = (((int)blockIdx.x - (var ? 0 : nbv)) * 8 + warp) * 32;
  if (r0 >= rows) return;
  Proj3 P;
  P.load(var ? Wf : Wg, lane);
  const int r = r0 + lane;
  float x0 = 0.f, x1 = 0.f;
  if (r < rows) {
    if (var) {
      const int j0 = F.var_off[r], j1 = F.var_off[r + 1];
      int pos = 0;
      for (int j = j0; j < j1; ++j) pos += F.var_inc[j].y >= 0 ? 1 : 0;
      const int deg = j1 - j0;
      x0 = deg > 0 ? (float)pos / (float)deg - 0.5f : 0.f;
      x1 = log1pf((float)deg) * 0.25f;
      inv_deg[r] = deg > 0 ? 1.f / (float)deg : 0.f;
    } else {
      const int len = F.cl_off[r + 1] - F.cl_off[r];
      x0 = logf((float)F.cl_w[r]) * 0.125f;
      x1 = (float)len * 0.25f;
      inv_len[r] = len > 0 ? 1.f / (float)len : 0.f;
    }
    float* o = (var ? f : g) + 3 * (size_t)r;
    o[0] = x0;
    o[1] = x1;
    o[2] = 1.f;
  }
  float* out = var ? hv : hc;
  const int cnt = min(32, rows - r0);
  for (int k = 0; k < cnt; ++k) {
    const float a = __shfl_sync(0xFFFFFFFFu, x0, k), b = __shfl_sync(0xFFFFFFFFu, x1, k);
    reinterpret_cast<float2*>(out + (size_t)(r0 + k) * kH)[lane] = P.apply(a, b, 1.f);
  }
}

// ------------------------------------------------------------ dense layers
// The three 64 x 128 contractions of a layer (forward, input gradient, weight
// gradient) run on the tensor cores: mma.sync m16n8k16 with BF16 operands and
// FP32 accumulation. The weights are BF16 already; an FP32 activation or
// gradient v enters as three BF16 terms hi + mid + lo (hi = bf16(v), mid =
// bf16(v - hi), lo = bf16(v - hi - mid)), so that products with BF16 weights
// sum to FP32 accuracy; the weight gradient, a product of two FP32 operands,
// keeps the three leading cross terms (hi x hi, hi x mid, mid x hi). The terms
// are written to shared memory once per value and read as fragments by
// ldmatrix.

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, "
      "{%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <bool TRANS>
__device__ __forceinline__ void ldm4(uint32_t (&r)[4], const __nv_bfloat16* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  if constexpr (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);  // .x (low half) = lo
  return *reinterpret_cast<const uint32_t*>(&v);
}

// the leading BF16 term of a pair; the pair becomes its remainder (exact)
__device__ __forceinline__ uint32_t take_term(float& x0, float& x1) {
  const uint32_t t = pack_bf16(x0, x1);
  x0 -= __uint_as_float(t << 16);
  x1 -= __uint_as_float(t & 0xFFFF0000u);
  return t;
}

// the first TERMS BF16 terms of four values into tiles `tile` elements apart
template <int TERMS>
__device__ __forceinline__ void store_terms(__nv_bfloat16* dst, int tile, float4 v) {
#pragma unroll
  for (int k = 0; k < TERMS; ++k) {
    uint2 w;
    w.x = take_term(v.x, v.y);
    w.y = take_term(v.z, v.w);
    *reinterpret_cast<uint2*>(dst + (size_t)k * tile) = w;
  }
}

// A row's list: its clause's literals (CL) or its variable's occurrences. The 16
// lanes that share the row hold its first 16 entries, one each: the other side's
// index, bit 31 when negated.
struct RowList {
  int j0, cnt;
  int32_t entry;
};

template <bool CL>
__device__ __forceinline__ int32_t list_entry(const DevFormula& F, int j) {
  if constexpr (CL) {
    return __ldg(F.lit_var + j);
  } else {
    const int2 inc = __ldg(reinterpret_cast<const int2*>(F.var_inc + j));
    return inc.x | (inc.y & (int32_t)0x80000000);
  }
}

// where the lists of the thread's four rows (16 apart from r0) begin and end
struct RowRanges {
  int j0[4], j1[4];
};

template <bool CL>
__device__ __forceinline__ RowRanges row_ranges(const DevFormula& F, int r0, int rows) {
  RowRanges R;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int r = r0 + 16 * k;
    const bool in = r < rows;
    R.j0[k] = in ? __ldg((CL ? F.cl_off : F.var_off) + r) : 0;
    R.j1[k] = in ? __ldg((CL ? F.cl_off : F.var_off) + r + 1) : 0;
  }
  return R;
}

template <bool CL>
__device__ __forceinline__ void row_lists(const DevFormula& F, const RowRanges& R, int c,
                                          RowList (&L)[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    L[k].j0 = R.j0[k];
    L[k].cnt = R.j1[k] - R.j0[k];
    L[k].entry = c < L[k].cnt ? list_entry<CL>(F, R.j0[k] + c) : 0;
  }
}

// The signed sums of two rows (16 lanes each, columns 4 c .. 4 c + 3): sum s *
// scale[other] * src[other] in list order (scale NULL = 1). Four entries of both
// rows are loaded together.
template <bool CL>
__device__ __forceinline__ void gather_pair(const DevFormula& F, const float* src,
                                            const float* scale, const RowList& L0,
                                            const RowList& L1, int c, float4 (&acc)[2]) {
  const unsigned mask = 0xFFFFu << (threadIdx.x & 16);
  acc[0] = acc[1] = make_float4(0.f, 0.f, 0.f, 0.f);
  const int most = max(L0.cnt, L1.cnt);
  int32_t e0 = L0.entry, e1 = L1.entry;
  for (int base = 0; base < most; base += 16) {
    if (base > 0) {
      e0 = base + c < L0.cnt ? list_entry<CL>(F, L0.j0 + base + c) : 0;
      e1 = base + c < L1.cnt ? list_entry<CL>(F, L1.j0 + base + c) : 0;
    }
    const int lim = min(16, most - base);
    for (int u = 0; u < lim; u += 4) {
      float s[2][4];
      float4 x[2][4];
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const int32_t e = __shfl_sync(mask, q ? e1 : e0, u + v, 16);
          s[q][v] = 0.f;
          x[q][v] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (base + u + v < (q ? L1.cnt : L0.cnt)) {
            const int o = e & 0x7FFFFFFF;
            s[q][v] = e < 0 ? -1.f : 1.f;
            if (scale) s[q][v] *= scale[o];
            x[q][v] = *(reinterpret_cast<const float4*>(src + (size_t)o * kH) + c);
          }
        }
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          acc[q].x = fmaf(s[q][v], x[q][v].x, acc[q].x);
          acc[q].y = fmaf(s[q][v], x[q][v].y, acc[q].y);
          acc[q].z = fmaf(s[q][v], x[q][v].z, acc[q].z);
          acc[q].w = fmaf(s[q][v], x[q][v].w, acc[q].w);
        }
    }
  }
}

__device__ __forceinline__ float4 row4(const float* p, int r, bool in, int c) {
  return in ? *(reinterpret_cast<const float4*>(p + (size_t)r * kH) + c)
            : make_float4(0.f, 0.f, 0.f, 0.f);
}

// the layer's BF16 weights (64 x 128) as rows of kLdX
__device__ __forceinline__ void stage_weights(__nv_bfloat16* Ws, const __nv_bfloat16* W) {
  // W is 4-byte aligned only (parameter offsets)
  const uint32_t* src = reinterpret_cast<const uint32_t*>(W);
  for (int e = threadIdx.x; e < kH * kH; e += 256)
    *reinterpret_cast<uint32_t*>(Ws + (e >> 6) * kLdX + 2 * (e & 63)) = src[e];
}

// The layer kernels walk tiles of 64 rows with resident blocks of 8 warps. A
// tile's rows hang on a chain of three loads (where the lists begin, their
// entries, the rows those name): the first two are made one and two tiles ahead,
// in registers, so that only the rows themselves are waited for. At 318000
// clauses and 53000 variables a clause layer takes 105 us forward and 174
// backward (290 with the chain in turn), a variable layer 68 and 75, with events
// around each launch. (The rows are read by plain loads, as a launch in flight may
// still write them; by read-only loads the backward layers took 194 and 93: the
// compiler then keeps fewer values in flight, 24 bytes of spills against 72. 16 warps
// of which half fetched and half multiplied were slower, 131 and 262 us; rows of
// the whole next tile in registers no faster, 115 us forward.) A launch stages
// its weights and first lists while its predecessor ends: eight launches of a
// prediction at n = 2000, m = 12000 take 31.9 us, 40.6 one after another.
// Tiles whose weight gradient one accumulator sums before it is added to the
// block's sums in shared memory: the tensor cores' accumulation rounds less
// exactly than an addition, and with one accumulator for all of a block's rows
// (1045 at 318000 clauses) a step's error against 64 bits was a fifth larger
// than with sums of 256 rows (2.7e-6 against 2.3e-6; now equal, at the same time).
constexpr int kSumTiles = 4;
constexpr int kFwdSmem = (3 * kTile + kH) * kLdX * 2;

// out[r] = relu(W [agg ; self[r]] + b), agg = out_scale[r] * signed sum of src;
// agg also goes to agg_out when given (the backward pass reads it). The three
// BF16 terms of [agg ; self] are the A operand; a warp multiplies 16 rows x 32
// outputs.
template <bool CL>
__global__ void __launch_bounds__(256, 3) k_mp_fwd(DevFormula F, const float* src,
                                                   const float* out_scale, const float* self,
                                                   int rows, const __nv_bfloat16* W,
                                                   const float* b, float* agg_out, float* out) {
  extern __shared__ __align__(16) __nv_bfloat16 sm[];
  __nv_bfloat16* xs = sm;                     // [3][kTile][kLdX]
  __nv_bfloat16* Ws = sm + 3 * kTile * kLdX;  // [kH][kLdX]
  stage_weights(Ws, W);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int hr = tid >> 4, c = tid & 15;  // 16 lanes per row, 16 rows at a time
  const int tiles = (rows + kTile - 1) / kTile, step = (int)gridDim.x;
  RowList lists[4];
  row_lists<CL>(F, row_ranges<CL>(F, (int)blockIdx.x * kTile + hr, rows), c, lists);
  RowRanges next = row_ranges<CL>(F, ((int)blockIdx.x + step) * kTile + hr, rows);
  pdl_wait();
  pdl_release();
  for (int tile = blockIdx.x; tile < tiles; tile += step) {
    __syncthreads();  // weights staged; the previous tile's fragments are read
#pragma unroll
    for (int k = 0; k < 4; k += 2) {
      float4 own[2], v[2];
      float sc[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int r = tile * kTile + hr + 16 * (k + q);
        own[q] = row4(self, r, r < rows, c);
        sc[q] = r < rows ? out_scale[r] : 0.f;
      }
      gather_pair<CL>(F, src, nullptr, lists[k], lists[k + 1], c, v);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int lr = hr + 16 * (k + q), r = tile * kTile + lr;
        __nv_bfloat16* row = xs + lr * kLdX + 4 * c;
        v[q] = make_float4(sc[q] * v[q].x, sc[q] * v[q].y, sc[q] * v[q].z, sc[q] * v[q].w);
        if (agg_out && r < rows) *(reinterpret_cast<float4*>(agg_out + (size_t)r * kH) + c) = v[q];
        store_terms<3>(row, kTile * kLdX, v[q]);
        store_terms<3>(row + kH, kTile * kLdX, own[q]);
      }
    }
    row_lists<CL>(F, next, c, lists);
    next = row_ranges<CL>(F, (tile + 2 * step) * kTile + hr, rows);
    __syncthreads();
    {
      const int rt = (warp & 3) * 16, ch = (warp >> 2) * 32, g = lane >> 2, t = lane & 3;
      float acc[4][4];
#pragma unroll
      for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[nt][q] = 0.f;
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) {
        uint32_t bw[2][4];
#pragma unroll
        for (int p = 0; p < 2; ++p)
          ldm4<false>(bw[p], Ws + (ch + p * 16 + (lane & 7) + ((lane >> 4) << 3)) * kLdX + ks * 16 +
                                 ((lane >> 3) & 1) * 8);
#pragma unroll
        for (int term = 0; term < 3; ++term) {
          uint32_t a[4];
          ldm4<false>(a, xs + (term * kTile + rt + (lane & 15)) * kLdX + ks * 16 + (lane >> 4) * 8);
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            mma_bf16(acc[2 * p], a, bw[p][0], bw[p][1]);
            mma_bf16(acc[2 * p + 1], a, bw[p][2], bw[p][3]);
          }
        }
      }
#pragma unroll
      for (int nt = 0; nt < 4; ++nt) {
        const int j = ch + nt * 8 + 2 * t, ra = tile * kTile + rt + g, rb = ra + 8;
        const float b0 = __ldg(b + j), b1 = __ldg(b + j + 1);
        if (ra < rows)
          *reinterpret_cast<float2*>(out + (size_t)ra * kH + j) =
              make_float2(relu(acc[nt][0] + b0), relu(acc[nt][1] + b1));
        if (rb < rows)
          *reinterpret_cast<float2*>(out + (size_t)rb * kH + j) =
              make_float2(relu(acc[nt][2] + b0), relu(acc[nt][3] + b1));
      }
    }
  }
}

constexpr int kBwdSmem = (3 * kTile * kLdD + (2 * kTile + kH) * kLdX) * 2 + 32 * 256 * 4;

// Gradient of a layer for tiles of 64 rows. The gradient of row r of the
// layer's output is carry[r] + sum s * in_scale[other] * src[other] (carry may
// be absent), or dz[r] wo at the top; delta is that where out > 0. Then dA / dB
// = the two halves of delta W, and part[block] = this block's sums of delta^T
// [agg ; self] (64 x 128) and delta (64). carry and dB may be the same array (a
// tile's rows are read before they are written, and only by their block).
template <bool CL>
__global__ void __launch_bounds__(256, 2)
    k_mp_bwd(DevFormula F, const float* src, const float* in_scale, const float* carry,
             const float* dz, const float* wo, const float* out, const float* agg,
             const float* self, int rows, const __nv_bfloat16* W, float* dA, float* dB,
             float* part) {
  extern __shared__ __align__(16) __nv_bfloat16 sm[];
  __nv_bfloat16* ds = sm;                     // [3][kTile][kLdD]
  __nv_bfloat16* xs = ds + 3 * kTile * kLdD;  // [2][kTile][kLdX]
  __nv_bfloat16* Ws = xs + 2 * kTile * kLdX;  // [kH][kLdX]
  stage_weights(Ws, W);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int q4 = warp & 3, half = warp >> 2;
  const int hr = tid >> 4, c = tid & 15;
  const int tiles = (rows + kTile - 1) / kTile, step = (int)gridDim.x;
  float wacc[8][4];
#pragma unroll
  for (int nt = 0; nt < 8; ++nt)
#pragma unroll
    for (int q = 0; q < 4; ++q) wacc[nt][q] = 0.f;
  float4 bacc = make_float4(0.f, 0.f, 0.f, 0.f);
  RowList lists[4];
  RowRanges next{};
  if (!dz) {
    row_lists<CL>(F, row_ranges<CL>(F, (int)blockIdx.x * kTile + hr, rows), c, lists);
    next = row_ranges<CL>(F, ((int)blockIdx.x + step) * kTile + hr, rows);
  }
  pdl_wait();
  pdl_release();
  float* sums = reinterpret_cast<float*>(Ws + kH * kLdX) + tid;  // [32][256], this thread's own
  auto move_sums = [&](bool first) {
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float& s = sums[(nt * 4 + q) * 256];
        s = first ? wacc[nt][q] : s + wacc[nt][q];
        wacc[nt][q] = 0.f;
      }
  };
  int summed = 0;
  for (int tile = blockIdx.x; tile < tiles; tile += step, ++summed) {
    if (summed > 0 && summed % kSumTiles == 0) move_sums(summed == kSumTiles);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; k += 2) {
      float4 e[2], d[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int r = tile * kTile + hr + 16 * (k + q);
        e[q] = row4(carry, r, r < rows && carry != nullptr && dz == nullptr, c);
      }
      if (dz) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int r = tile * kTile + hr + 16 * (k + q);
          const float z = r < rows ? dz[r] : 0.f;
          d[q] = make_float4(z * __ldg(wo + 4 * c), z * __ldg(wo + 4 * c + 1),
                             z * __ldg(wo + 4 * c + 2), z * __ldg(wo + 4 * c + 3));
        }
      } else {
        gather_pair<CL>(F, src, in_scale, lists[k], lists[k + 1], c, d);
#pragma unroll
        for (int q = 0; q < 2; ++q)
          d[q] = make_float4(d[q].x + e[q].x, d[q].y + e[q].y, d[q].z + e[q].z, d[q].w + e[q].w);
      }
      float4 xa[2], xb[2], o[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int r = tile * kTile + hr + 16 * (k + q);
        xa[q] = row4(agg, r, r < rows, c);
        xb[q] = row4(self, r, r < rows, c);
        o[q] = row4(out, r, r < rows, c);
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int lr = hr + 16 * (k + q);
        d[q] = make_float4(o[q].x > 0.f ? d[q].x : 0.f, o[q].y > 0.f ? d[q].y : 0.f,
                           o[q].z > 0.f ? d[q].z : 0.f, o[q].w > 0.f ? d[q].w : 0.f);
        bacc = make_float4(bacc.x + d[q].x, bacc.y + d[q].y, bacc.z + d[q].z, bacc.w + d[q].w);
        store_terms<3>(ds + lr * kLdD + 4 * c, kTile * kLdD, d[q]);
        store_terms<2>(xs + lr * kLdX + 4 * c, kTile * kLdX, xa[q]);
        store_terms<2>(xs + lr * kLdX + kH + 4 * c, kTile * kLdX, xb[q]);
      }
    }
    if (!dz) {
      row_lists<CL>(F, next, c, lists);
      next = row_ranges<CL>(F, (tile + 2 * step) * kTile + hr, rows);
    }
    __syncthreads();
    {
      {  // input gradient: 16 rows x the 64 columns of one half
        float acc[8][4];
#pragma unroll
        for (int nt = 0; nt < 8; ++nt)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[nt][q] = 0.f;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          uint32_t a[3][4];
#pragma unroll
          for (int term = 0; term < 3; ++term)
            ldm4<false>(a[term], ds + (term * kTile + q4 * 16 + (lane & 15)) * kLdD + ks * 16 +
                                     (lane >> 4) * 8);
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            uint32_t bw[4];
            ldm4<true>(bw,
                       Ws + (ks * 16 + (lane & 15)) * kLdX + half * kH + p * 16 + (lane >> 4) * 8);
#pragma unroll
            for (int term = 0; term < 3; ++term) {
              mma_bf16(acc[2 * p], a[term], bw[0], bw[1]);
              mma_bf16(acc[2 * p + 1], a[term], bw[2], bw[3]);
            }
          }
        }
        float* dst = half ? dB : dA;
        const int ra = tile * kTile + q4 * 16 + g, rb = ra + 8;
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
          const int k = nt * 8 + 2 * t;
          if (ra < rows)
            *reinterpret_cast<float2*>(dst + (size_t)ra * kH + k) =
                make_float2(acc[nt][0], acc[nt][1]);
          if (rb < rows)
            *reinterpret_cast<float2*>(dst + (size_t)rb * kH + k) =
                make_float2(acc[nt][2], acc[nt][3]);
        }
      }
      // weight gradient: outputs 16 q4 .. + 15, inputs of one half, over the rows
#pragma unroll
      for (int ks = 0; ks < kTile / 16; ++ks) {
        uint32_t ah[4], am[4];
        const __nv_bfloat16* ap = ds + (ks * 16 + (lane & 7) + ((lane >> 4) << 3)) * kLdD + q4 * 16 +
                                  ((lane >> 3) & 1) * 8;
        ldm4<true>(ah, ap);
        ldm4<true>(am, ap + kTile * kLdD);
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          uint32_t bh[4], bm[4];
          const __nv_bfloat16* bp =
              xs + (ks * 16 + (lane & 15)) * kLdX + half * kH + p * 16 + (lane >> 4) * 8;
          ldm4<true>(bh, bp);
          ldm4<true>(bm, bp + kTile * kLdX);
          mma_bf16(wacc[2 * p], ah, bh[0], bh[1]);
          mma_bf16(wacc[2 * p], ah, bm[0], bm[1]);
          mma_bf16(wacc[2 * p], am, bh[0], bh[1]);
          mma_bf16(wacc[2 * p + 1], ah, bh[2], bh[3]);
          mma_bf16(wacc[2 * p + 1], ah, bm[2], bm[3]);
          mma_bf16(wacc[2 * p + 1], am, bh[2], bh[3]);
        }
      }
    }
  }
  float* pt = part + (size_t)blockIdx.x * kPart;
  if (summed > kSumTiles) {
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
#pragma unroll
      for (int q = 0; q < 4; ++q) wacc[nt][q] += sums[(nt * 4 + q) * 256];
  }
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    const int j = q4 * 16 + g, k = half * kH + nt * 8 + 2 * t;
    *reinterpret_cast<float2*>(pt + j * 2 * kH + k) = make_float2(wacc[nt][0], wacc[nt][1]);
    *reinterpret_cast<float2*>(pt + (j + 8) * 2 * kH + k) = make_float2(wacc[nt][2], wacc[nt][3]);
  }
  // bias: the 16 row slots' sums, in order
  __syncthreads();
  float* sb = reinterpret_cast<float*>(sm);  // [16][kH]
  *reinterpret_cast<float4*>(sb + hr * kH + 4 * c) = bacc;
  __syncthreads();
  if (tid < kH) {
    float v = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) v += sb[k * kH + tid];
    pt[kWCount + tid] = v;
  }
}

// ------------------------------------------------- gradient of the projections
// Per block: sum_r delta[r][j] x[r][k] (64 x 3), delta = (carry[r] + signed sum
// of src) where h0 > 0. Blocks below nbv take variables (with the sum), the
// others clauses (carry only). A warp takes rows strided over its side's warps.
__global__ void __launch_bounds__(256) k_mp_embed_bwd(DevFormula F, int nbv, const float* src,
                                                      const float* in_scale, const float* carry_v,
                                                      const float* hv, const float* f,
                                                      const float* carry_c, const float* hc,
                                                      const float* g, float* part) {
  __shared__ float s[8][3 * kH];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool var = (int)blockIdx.x < nbv;
  const int rows = var ? F.n : F.m;
  const int blocks = var ? nbv : (int)gridDim.x - nbv;
  const int first = ((int)blockIdx.x - (var ? 0 : nbv)) * 8 + warp, step = blocks * 8;
  float acc[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  pdl_wait();
  pdl_release();
  auto add = [&](float2 d, float2 h, const float* x) {
    const float d0 = h.x > 0.f ? d.x : 0.f, d1 = h.y > 0.f ? d.y : 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float xk = x[k];
      acc[k] = fmaf(d0, xk, acc[k]);
      acc[3 + k] = fmaf(d1, xk, acc[3 + k]);
    }
  };
  if (var) {
    for (int r = first; r < rows; r += step) {
      float2 a = make_float2(0.f, 0.f);
      const int j0 = __ldg(F.var_off + r), j1 = __ldg(F.var_off + r + 1);
#pragma unroll 4
      for (int j = j0; j < j1; ++j) {
        const int2 inc = __ldg(reinterpret_cast<const int2*>(F.var_inc + j));
        const float sc = (inc.y < 0 ? -1.f : 1.f) * in_scale[inc.x];
        const float2 x = reinterpret_cast<const float2*>(src + (size_t)inc.x * kH)[lane];
        a.x = fmaf(sc, x.x, a.x);
        a.y = fmaf(sc, x.y, a.y);
      }
      const float2 e = reinterpret_cast<const float2*>(carry_v + (size_t)r * kH)[lane];
      add(make_float2(a.x + e.x, a.y + e.y), reinterpret_cast<const float2*>(hv + (size_t)r * kH)[lane],
          f + 3 * (size_t)r);
    }
  } else {
    for (int r = first; r < rows; r += 4 * step) {
      float2 d[4], h[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (r + u * step < rows) {
          d[u] = reinterpret_cast<const float2*>(carry_c + (size_t)(r + u * step) * kH)[lane];
          h[u] = reinterpret_cast<const float2*>(hc + (size_t)(r + u * step) * kH)[lane];
        }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (r + u * step < rows) add(d[u], h[u], g + 3 * (size_t)(r + u * step));
    }
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) s[warp][6 * lane + k] = acc[k];
  __syncthreads();
  if (threadIdx.x < 3 * kH) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) v += s[w][threadIdx.x];
    part[(size_t)blockIdx.x * 3 * kH + threadIdx.x] = v;
  }
}

// dst[e] = sum over blocks b of part[b stride + e], e < count, for every set
// (blockIdx.y). A block takes 32 entries: warp w sums blocks w, w + 8, ... in
// order (32 consecutive entries per load), then the eight sums in order.
__global__ void __launch_bounds__(256) k_mp_sum(MpSums S) {
  __shared__ float s[8][32];
  pdl_wait();
  pdl_release();
  const MpSums::Set set = S.set[blockIdx.y];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int e = (int)blockIdx.x * 32 + lane;
  if ((int)blockIdx.x * 32 >= set.count) return;
  float v = 0.f;
  if (e < set.count) {
#pragma unroll 8
    for (int b = warp; b < set.blocks; b += 8) v += set.part[(size_t)b * set.stride + e];
  }
  s[warp][lane] = v;
  __syncthreads();
  if (warp == 0 && e < set.count) {
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += s[w][lane];
    set.dst[e] = t;
  }
}

// ---------------------------------------------------------------- read-out
// z = wo . h + bo, p = sigmoid(z); with labels: dz = (p - y) / n, per block the
// loss terms softplus(z) - y z and the sums of dz h (64) and dz. One warp = one
// row, two columns per lane.
__global__ void __launch_bounds__(256) k_mp_out(const float* h, int n, const float* wo,
                                                const float* bo, const uint8_t* y, float* prob,
                                                float* dz, double* loss_part, float* part) {
  __shared__ double lp[8];
  __shared__ float sg[8][kH + 1];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float2 o = make_float2(__ldg(wo + 2 * lane), __ldg(wo + 2 * lane + 1));
  const float b = __ldg(bo);
  pdl_wait();
  pdl_release();
  double term = 0.0;
  float2 gw = make_float2(0.f, 0.f);
  float gb = 0.f;
  for (int r = (int)blockIdx.x * 8 + w; r < n; r += (int)gridDim.x * 8) {
    const float2 x = reinterpret_cast<const float2*>(h + (size_t)r * kH)[lane];
    float acc = fmaf(x.x, o.x, x.y * o.y);
    for (int s = 16; s > 0; s >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, s);
    const float z = acc + b;
    const float p = 1.f / (1.f + expf(-z));
    if (prob && lane == 0) prob[r] = p;
    if (y) {
      const float yy = y[r] ? 1.f : 0.f;
      const float d = (p - yy) / (float)n;
      gw.x = fmaf(d, x.x, gw.x);
      gw.y = fmaf(d, x.y, gw.y);
      gb += d;
      if (lane == 0) {
        dz[r] = d;
        term += (double)(z > 0.f ? z + log1pf(expf(-z)) : log1pf(expf(z))) - (double)(yy * z);
      }
    }
  }
  if (!y) return;
  if (lane == 0) {
    lp[w] = term;
    sg[w][kH] = gb;
  }
  sg[w][2 * lane] = gw.x;
  sg[w][2 * lane + 1] = gw.y;
  __syncthreads();
  if (threadIdx.x <= kH) {
    float v = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) v += sg[k][threadIdx.x];
    part[(size_t)blockIdx.x * (kH + 1) + threadIdx.x] = v;
  }
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int k = 0; k < 8; ++k) v += lp[k];
    loss_part[blockIdx.x] = v;
  }
}

// --------------------------------------------------------------- optimiser
__global__ void k_mp_adam(float* P, const float* G, float* M, float* V, int count, float lr,
                          float b1, float b2, float eps, float c1, float c2) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= count) return;
  const float g = G[e];
  const float m = b1 * M[e] + (1.f - b1) * g;
  const float v = b2 * V[e] + (1.f - b2) * g * g;
  M[e] = m;
  V[e] = v;
  P[e] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
}

__global__ void k_mp_to_bf16(const float* P, __nv_bfloat16* Pb, int count) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < count) Pb[e] = __float2bfloat16_rn(P[e]);
}

// ------------------------------------------------ biased initial states
// x = [u < P_v] with the initial-draw Philox counter (variable, chain octet,
// 0, init phase | instance << 8): P_v = 32768 everywhere gives exactly the
// states of maxsat_reset. Sparse layout (variable-major) and dense layout.
__global__ void k_init_probs_sparse(DevFormula F, DevChains C, const uint32_t* P, int vg0) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g8 = blockIdx.x * 32 + lane, b0 = g8 * 8;
  const int i = (vg0 + blockIdx.y) * 8 + warp;
  if (i >= F.n) return;
  const int2 vi = F.var_inst ? F.var_inst[i] : make_int2(0, i);
  const uint4 r = philox4x32_10(make_uint4((uint32_t)vi.y, (uint32_t)(g8 + C.g8_off), 0u,
                                           kPhaseInit | ((uint32_t)vi.x << 8)),
                                C.keys);
  const uint32_t Pi = P[i];
  uint64_t x = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) x |= (uint64_t)(lane16(r, q) < Pi) << (8 * q);
  const size_t o = (size_t)i * C.Bp + b0;
  *reinterpret_cast<uint64_t*>(C.xt + o) = x;
  *reinterpret_cast<uint64_t*>(C.best_xt + o) = x;
}

__global__ void k_init_probs_dense(int n, int n_pad, DevChains C, const uint32_t* P, uint8_t* X,
                                   uint8_t* best_x, uint8_t one, uint8_t minus_one, int vg0) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g8 = blockIdx.x * 32 + lane, b0 = g8 * 8;
  const int i = (vg0 + blockIdx.y) * 8 + warp;
  if (i >= n) return;
  const uint4 r = philox4x32_10(make_uint4((uint32_t)i, (uint32_t)(g8 + C.g8_off), 0u, kPhaseInit),
                                C.keys);
  const uint32_t Pi = P[i];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const bool bit = lane16(r, q) < Pi;
    const size_t o = (size_t)(b0 + q) * n_pad + i;
    X[o] = bit ? one : minus_one;
    best_x[o] = bit ? 1 : 0;
  }
}

}  // namespace

// ====================================================================== host
int mp_layout(int L, MpLayout* out) {
  if (L < 1 || L > kMpMaxLayers) return -1;
  int o = 0;
  out->L = L;
  out->Wf = o, o += kH * 3;
  out->Wg = o, o += kH * 3;
  for (int l = 0; l < L; ++l) {
    out->Wc[l] = o, o += kH * 2 * kH;
    out->bc[l] = o, o += kH;
    out->Wv[l] = o, o += kH * 2 * kH;
    out->bv[l] = o, o += kH;
  }
  out->wo = o, o += kH;
  out->bo = o, o += 1;
  out->total = o;
  return 0;
}

namespace {
inline int blocks(long long count, int per) { return (int)((count + per - 1) / per); }

int mp_sms() {
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
}  // namespace

int mp_bwd_blocks(int rows) { return std::max(1, std::min(blocks(rows, kTile), 2 * mp_sms())); }
int mp_out_blocks(int n) { return std::max(1, std::min(blocks(n, 16), 8 * mp_sms())); }
// about five variables a warp: each waits on its list, then on its rows
int mp_embed_bwd_var_blocks(int n) { return std::max(1, std::min(blocks(n, 16), 8 * mp_sms())); }
int mp_embed_bwd_clause_blocks(int m) { return std::max(1, std::min(blocks(m, 64), 3 * mp_sms())); }
int mp_part_floats() { return kPart; }

cudaError_t mp_launch_embed(const DevFormula& F, const __nv_bfloat16* Wf, const __nv_bfloat16* Wg,
                            float* f, float* g, float* inv_len, float* inv_deg, float* hv,
                            float* hc, cudaStream_t st) {
  const int nbv = blocks(F.n, 256), nbc = blocks(F.m, 256);
  return launch_pdl(k_mp_embed, nbv + nbc, 256, 0, st, F, Wf, Wg, nbv, f, g, inv_len, inv_deg, hv,
                    hc);
}

cudaError_t mp_launch_fwd(const DevFormula& F, bool clauses, const float* src,
                          const float* out_scale, const float* self, const __nv_bfloat16* W,
                          const float* b, float* agg_out, float* out, cudaStream_t st) {
  const int rows = clauses ? F.m : F.n;
  if (rows <= 0) return cudaSuccess;
  auto kern = clauses ? k_mp_fwd<true> : k_mp_fwd<false>;
  const cudaError_t e = allow_dynamic_smem(kern, kFwdSmem);
  if (e != cudaSuccess) return e;
  const int grid = std::min(blocks(rows, kTile), 3 * mp_sms());
  return launch_pdl(kern, grid, 256, kFwdSmem, st, F, src, out_scale, self, rows, W, b, agg_out,
                    out);
}

cudaError_t mp_launch_bwd(const DevFormula& F, bool clauses, const float* src,
                          const float* in_scale, const float* carry, const float* dz,
                          const float* wo, const float* out, const float* agg, const float* self,
                          const __nv_bfloat16* W, float* dA, float* dB, float* part,
                          cudaStream_t st) {
  const int rows = clauses ? F.m : F.n;
  auto kern = clauses ? k_mp_bwd<true> : k_mp_bwd<false>;
  const cudaError_t e = allow_dynamic_smem(kern, kBwdSmem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, mp_bwd_blocks(rows), 256, kBwdSmem, st, F, src, in_scale, carry, dz, wo,
                    out, agg, self, rows, W, dA, dB, part);
}

cudaError_t mp_launch_embed_bwd(const DevFormula& F, const float* src, const float* in_scale,
                                const float* carry_v, const float* hv, const float* f,
                                const float* carry_c, const float* hc, const float* g, float* part,
                                cudaStream_t st) {
  const int nbv = mp_embed_bwd_var_blocks(F.n), nbc = mp_embed_bwd_clause_blocks(F.m);
  return launch_pdl(k_mp_embed_bwd, nbv + nbc, 256, 0, st, F, nbv, src, in_scale, carry_v, hv, f,
                    carry_c, hc, g, part);
}

cudaError_t mp_launch_sums(const MpSums& S, cudaStream_t st) {
  int most = 0;
  for (int k = 0; k < S.sets; ++k) most = std::max(most, S.set[k].count);
  return launch_pdl(k_mp_sum, dim3(blocks(most, 32), S.sets), 256, 0, st, S);
}

cudaError_t mp_launch_out(const float* h, int n, const float* wo, const float* bo,
                          const uint8_t* y, float* prob, float* dz, double* loss_part, float* part,
                          cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  return launch_pdl(k_mp_out, mp_out_blocks(n), 256, 0, st, h, n, wo, bo, y, prob, dz, loss_part,
                    part);
}

cudaError_t mp_launch_adam(float* P, const float* G, float* M, float* V, int count, float lr,
                           float b1, float b2, float eps, int step, __nv_bfloat16* Pb,
                           cudaStream_t st) {
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  k_mp_adam<<<blocks(count, 256), 256, 0, st>>>(P, G, M, V, count, lr, b1, b2, eps, c1, c2);
  k_mp_to_bf16<<<blocks(count, 256), 256, 0, st>>>(P, Pb, count);
  return cudaGetLastError();
}

cudaError_t mp_launch_to_bf16(const float* P, __nv_bfloat16* Pb, int count, cudaStream_t st) {
  k_mp_to_bf16<<<blocks(count, 256), 256, 0, st>>>(P, Pb, count);
  return cudaGetLastError();
}

cudaError_t launch_init_probs_sparse(const DevFormula& F, const DevChains& C, const uint32_t* P,
                                     cudaStream_t st) {
  const int groups = (F.n + 7) / 8;
  for (int vg0 = 0; vg0 < groups; vg0 += 65535) {
    dim3 grid(C.Bp / kChainTile, std::min(65535, groups - vg0));
    k_init_probs_sparse<<<grid, 256, 0, st>>>(F, C, P, vg0);
  }
  return cudaGetLastError();
}

cudaError_t launch_init_probs_dense(int n, int n_pad, const DevChains& C, const uint32_t* P,
                                    uint8_t* X, uint8_t* best_x, uint8_t one, uint8_t minus_one,
                                    cudaStream_t st) {
  const int groups = (n + 7) / 8;
  for (int vg0 = 0; vg0 < groups; vg0 += 65535) {
    dim3 grid(C.Bp / kChainTile, std::min(65535, groups - vg0));
    k_init_probs_dense<<<grid, 256, 0, st>>>(n, n_pad, C, P, X, best_x, one, minus_one, vg0);
  }
  return cudaGetLastError();
}

}  // namespace rbmsat
