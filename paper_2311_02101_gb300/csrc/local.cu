// Local rounds: all Gibbs rounds of eight chains inside one block.
//
// A small formula of clauses of at most 3 literals fits an SM: its clause and
// incidence lists, and for one octet of chains (the eight chains that share a
// Philox block) the states, the hidden patterns and nu. Chains never meet, so
// one block then runs any number of rounds of its octet from shared memory with
// two block barriers a round, while the resident rounds (k_rounds) of such a
// formula wait on L2 latencies and on barriers between blocks: 256 chains of n =
// 50, m = 215 take 6.6 us a round there, almost all of it waiting (14 blocks,
// 3000 cycles of gathering, 9700 of barriers).
//
// Here a thread takes a clause (its eight chains' draws from three Philox
// blocks, as gather3_clauses) and TPV neighbouring threads take a variable: each
// sums every TPV-th incidence by byte permutes (as k_visible_nib), a
// reduce-scatter leaves each with 8 / TPV chains, whose draws, nu and states it
// updates. Costs are summed over the block (integers); the free energy is
// accumulated every round and reduced in a fixed order in the last round of a
// launch. Results are those of the two-launch round (free energy: another
// summation order).
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "internal.h"
#include "round_ops.cuh"

namespace rbmsat {

namespace {

struct LocalLayout {  // byte offsets into dynamic shared memory
  int rec, ptab, pva, cl, w, inc, off, x, best, nu, h, fe, total;
};

__host__ __device__ inline int up16(int v) { return (v + 15) & ~15; }

__host__ __device__ inline LocalLayout local_layout(int n, int m, int nnz, int groups,
                                                    int ptab_stride, int pv_len, int threads) {
  LocalLayout L;
  int at = 0;
  L.rec = at, at += groups * 256;               // the octet's temperature (and the next one's)
  L.ptab = at, at += 2 * ptab_stride;           // contributions at both
  L.pva = at, at += up16(pv_len * 8);
  L.cl = at, at += up16(m * 8);
  L.w = at, at += up16(m * 4);
  L.inc = at, at += up16(nnz * 4);
  L.off = at, at += up16((n + 1) * 4);
  L.x = at, at += up16(n * 8);
  L.best = at, at += up16(n * 8);
  L.nu = at, at += n * 32;
  L.h = at, at += up16(m * 4);
  L.fe = at, at += (threads / 32) * 8 * 4;
  L.total = at + 256;  // the record blocks start at a 256-byte boundary
  return L;
}

template <int TPV, int T, bool PLAIN3>
__global__ void __launch_bounds__(T) k_rounds_local(DevFormula F, DevTables Tb, DevChains C,
                                                    LocalFormula P, uint32_t t0, int rounds,
                                                    float keep) {
  constexpr int CPL = 8 / TPV;  // chains per thread of a variable
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(16) int32_t s_cost[2][8];
  const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(smem_raw);
  const uint32_t sb = (s0 + 255u) & ~255u;
  unsigned char* sm = smem_raw + (sb - s0);
  const int n = F.n, m = F.m, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const LocalLayout L =
      local_layout(n, m, F.nnz, Tb.n_groups, Tb.ptab_stride, Tb.pv_len, T);
  const int g8 = blockIdx.x, b0 = g8 * 8;
  const int E = Tb.n_temps, gb0 = C.g8_off * 8 + b0;
  const int e0 = temp_of(gb0, E, C.B_total, C.inv_B_total);
  // first chain of the octet at the next temperature (8: none)
  const int split = e0 == temp_of(gb0 + 7, E, C.B_total, C.inv_B_total)
                        ? 8
                        : (int)(((long long)(e0 + 1) * C.B_total + E - 1) / E) - gb0;
  const int e1 = split < 8 ? e0 + 1 : e0;
  // ---- the formula's lists and tables, the octet's state
  auto copy16 = [&](int at, const void* src, int bytes) {
    const int4* s = reinterpret_cast<const int4*>(src);
    int4* d = reinterpret_cast<int4*>(sm + at);
    for (int k = tid; k < bytes / 16; k += T) d[k] = __ldg(s + k);
  };
  for (int k = tid; k < Tb.n_groups * 16; k += T)
    reinterpret_cast<int4*>(sm + L.rec)[k] = __ldg(
        reinterpret_cast<const int4*>(Tb.rec3) + (size_t)((k >> 4) * E + e0) * 16 + (k & 15));
  copy16(L.ptab, reinterpret_cast<const char*>(Tb.ptab) + (size_t)e0 * Tb.ptab_stride,
         Tb.ptab_stride);
  copy16(L.ptab + Tb.ptab_stride,
         reinterpret_cast<const char*>(Tb.ptab) + (size_t)e1 * Tb.ptab_stride, Tb.ptab_stride);
  copy16(L.pva, Tb.pva, up16(Tb.pv_len * 8));
  copy16(L.cl, P.cl, up16(m * 8));
  copy16(L.inc, P.inc, up16(F.nnz * 4));
  int32_t* s_w = reinterpret_cast<int32_t*>(sm + L.w);
  for (int k = tid; k < m; k += T) s_w[k] = (int32_t)__ldg(F.cl_w + k);
  int32_t* s_off = reinterpret_cast<int32_t*>(sm + L.off);
  for (int k = tid; k <= n; k += T) s_off[k] = __ldg(F.var_off + k);
  uint64_t* s_x = reinterpret_cast<uint64_t*>(sm + L.x);
  uint64_t* s_best = reinterpret_cast<uint64_t*>(sm + L.best);
  float* s_nu = reinterpret_cast<float*>(sm + L.nu);
  for (int k = tid; k < n; k += T) {
    const size_t o = (size_t)k * C.Bp + b0;
    s_x[k] = *reinterpret_cast<const uint64_t*>(C.xt + o);
    s_best[k] = *reinterpret_cast<const uint64_t*>(C.best_xt + o);
    reinterpret_cast<float4*>(s_nu)[2 * k] = reinterpret_cast<const float4*>(C.nu + o)[0];
    reinterpret_cast<float4*>(s_nu)[2 * k + 1] = reinterpret_cast<const float4*>(C.nu + o)[1];
  }
  uint32_t* s_h = reinterpret_cast<uint32_t*>(sm + L.h);
  const uint2* pva = reinterpret_cast<const uint2*>(sm + L.pva);
  const uint2* s_cl = reinterpret_cast<const uint2*>(sm + L.cl);
  const uint32_t* s_inc = reinterpret_cast<const uint32_t*>(sm + L.inc);
  const uint32_t rec_tab = sb + (uint32_t)L.rec;
  const uint32_t tab = sb + (uint32_t)L.ptab, tab1 = tab + (uint32_t)Tb.ptab_stride;
  // every thread keeps the octet's best costs (the host runs this kernel only
  // when all weights together stay below 2^31 - 1)
  int32_t best[8];
  uint32_t kept = 0;  // bit q: chain q improved in this launch
#pragma unroll
  for (int q = 0; q < 8; ++q)
    best[q] = (int32_t)max(min(C.best[b0 + q], (int64_t)INT32_MAX), (int64_t)-1);
  if (tid < 16) s_cost[tid >> 3][tid & 7] = 0;
  const uint64_t up = split < 8 ? 0x8080808080808080ull << (8 * split) : 0ull;
  const uint32_t up_lo = (uint32_t)up, up_hi = (uint32_t)(up >> 32);
  uint32_t mk[4];
  nib_masks(split, mk);
  const RoundKeys& K = C.keys;
  const uint32_t octet = (uint32_t)(g8 + C.g8_off);
  __syncthreads();

  for (int r = 0; r < rounds; ++r) {
    const uint32_t t = t0 + (uint32_t)r;
    const bool last = r + 1 == rounds;
    // ---- gather
    const HiddenThread Q = hidden_thread(octet, t, K);
    int32_t cost[8];
    float fe[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      cost[q] = 0;
      fe[q] = 0.f;
    }
    for (int c = tid; c < m; c += T) {
      const uint2 cl = s_cl[c];
      const uint32_t info = cl.y >> 16;  // group << 6 | saturated << 5 | negated << 2 | length
      const int len = PLAIN3 ? 3 : (int)(info & 3u);
      const uint64_t xa = s_x[cl.x & 0xFFFFu], xb = s_x[cl.x >> 16], xc = s_x[cl.y & 0xFFFFu];
      const uint64_t flip = ((info >> 2) & 7u) * 0x0101010101010101ull;
      uint64_t pat = xa + 2 * xb + 4 * xc;  // absent literals point at a variable and are masked
      if (!PLAIN3) pat &= ((1u << len) - 1u) * 0x0101010101010101ull;
      pat ^= flip;
      const uint32_t lo = (uint32_t)pat, hi = (uint32_t)(pat >> 32);
      const int32_t w = s_w[c];
      const uint32_t u_lo = (~(lo + 0x7F7F7F7Fu) & 0x80808080u) >> 7;
      const uint32_t u_hi = (~(hi + 0x7F7F7F7Fu) & 0x80808080u) >> 7;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        cost[q] += (int32_t)__byte_perm(u_lo, 0u, 0x4440u | q) * w;
        cost[q + 4] += (int32_t)__byte_perm(u_hi, 0u, 0x4440u | q) * w;
      }
      if (!PLAIN3 && len == 0) continue;
      uint4 R[3];
      hidden_blocks3(Q, (uint32_t)c, kPhaseHidden, K, R);
      const uint32_t rb = rec_tab + (info >> 6) * 256u;
      uint32_t h = 0, unused = 0;
      if (PLAIN3 || !((info >> 5) & 1u))
        octet_draws<false, true>((lo << 4) | up_lo, (hi << 4) | up_hi, rb, R, fe, h, unused);
      else
        octet_draws<true, true>((lo << 4) | up_lo, (hi << 4) | up_hi, rb, R, fe, h, unused);
      s_h[c] = h;
    }
    int32_t mine = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int32_t v = __reduce_add_sync(0xFFFFFFFFu, cost[q]);
      if (lane == q) mine = v;
    }
    if (lane < 8 && mine != 0) atomicAdd(&s_cost[r & 1][lane], mine);
    if (last) {  // the free energy of the last state, summed in a fixed order
      float* s_fe = reinterpret_cast<float*>(sm + L.fe);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        float v = fe[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
        if (lane == 0) s_fe[warp * 8 + q] = v;
      }
    }
    __syncthreads();
    // ---- best-keep
    uint32_t imp = 0;  // bit q: chain q improved
    const int4 ca = *reinterpret_cast<const int4*>(&s_cost[r & 1][0]);
    const int4 cb = *reinterpret_cast<const int4*>(&s_cost[r & 1][4]);
    const int32_t cs[8] = {ca.x, ca.y, ca.z, ca.w, cb.x, cb.y, cb.z, cb.w};
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (cs[q] < best[q]) {
        best[q] = cs[q];
        imp |= 1u << q;
      }
    kept |= imp;
    if (tid < 8) {
      s_cost[(r & 1) ^ 1][tid] = 0;  // the next round's sums (last read a round ago)
      if (last) {
        const float* s_fe = reinterpret_cast<const float*>(sm + L.fe);
        float f = 0.f;
        for (int w = 0; w < T / 32; ++w) f += s_fe[w * 8 + tid];
        C.cost[b0 + tid] = s_cost[r & 1][tid];
        C.fe[b0 + tid] = f;
        C.improved[b0 + tid] = (imp >> tid) & 1u;
      }
    }
    // ---- visible update: TPV threads per variable (whole warps take part in
    // the shuffles; a variable past the end has no incidence)
    const int sub = tid & (TPV - 1);
    for (int v0 = 0; v0 < n; v0 += T / TPV) {
      const int v = v0 + tid / TPV;
      const int j0 = v < n ? s_off[v] : 0, j1 = v < n ? s_off[v + 1] : 0;
      int z[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) z[q] = 0;
      for (int j = j0 + sub; j < j1; j += 32 * TPV) {
        uint32_t acc[4] = {0u, 0u, 0u, 0u};
        int cnt = 0;
        for (int k = j; k < j1 && cnt < 32; k += TPV, ++cnt) {
          const uint32_t inc = s_inc[k];  // clause | contribution row << 16
          const uint32_t h = s_h[inc & 0xFFFFu], row = (inc >> 16) * 16u;
          if (split == 8)
            nib_add(lds128(tab + row), h, acc);
          else
            nib_add2(lds128(tab + row), lds128(tab1 + row), h, mk, acc);
        }
        nib_flush(acc, cnt * Tb.ptab_bias, z);
      }
      // reduce-scatter over the TPV threads: thread `sub` ends with chains
      // CPL sub .. CPL sub + CPL - 1
#pragma unroll
      for (int half = 4; half >= CPL; half >>= 1) {
        const int step = half / CPL;  // lane distance
        const bool upper = (sub & step) != 0;
#pragma unroll
        for (int k = 0; k < half; ++k) {
          const int send = upper ? z[k] : z[k + half];
          const int keepv = upper ? z[k + half] : z[k];
          z[k] = keepv + __shfl_xor_sync(0xFFFFFFFFu, send, step);
        }
      }
      if (v < n) {
        const uint4 rn = philox4x32_10(make_uint4((uint32_t)v, octet, t, kPhaseVisible), K);
        uint8_t* xb = reinterpret_cast<uint8_t*>(s_x + v) + sub * CPL;
        uint8_t* bb = reinterpret_cast<uint8_t*>(s_best + v) + sub * CPL;
        float* nu = s_nu + v * 8 + sub * CPL;
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
          const int q = sub * CPL + k;
          const uint2 pv = pva[__viaddmin_s32_relu(z[k], Tb.qmax, 2 * Tb.qmax)];
          if ((imp >> q) & 1u) bb[k] = xb[k];
          nu[k] = __fmaf_rn(keep, nu[k], __uint_as_float(pv.y));
          const uint32_t word = q < 2 ? rn.x : q < 4 ? rn.y : q < 6 ? rn.z : rn.w;
          const uint32_t u = (q & 1) ? word >> 16 : word & 0xFFFFu;
          xb[k] = u < pv.x ? 1 : 0;
        }
      }
    }
    __syncthreads();
  }
  // ---- the octet's state back to the chains
  for (int k = tid; k < n; k += T) {
    const size_t o = (size_t)k * C.Bp + b0;
    *reinterpret_cast<uint64_t*>(C.xt + o) = s_x[k];
    *reinterpret_cast<uint64_t*>(C.best_xt + o) = s_best[k];
    reinterpret_cast<float4*>(C.nu + o)[0] = reinterpret_cast<const float4*>(s_nu)[2 * k];
    reinterpret_cast<float4*>(C.nu + o)[1] = reinterpret_cast<const float4*>(s_nu)[2 * k + 1];
  }
  if (tid < 8) {
    int32_t b = best[0];
#pragma unroll
    for (int q = 1; q < 8; ++q)
      if (tid == q) b = best[q];
    if ((kept >> tid) & 1u) C.best[b0 + tid] = b;
  }
}

using LocalFn = void (*)(DevFormula, DevTables, DevChains, LocalFormula, uint32_t, int, float);

template <int TPV>
LocalFn local_fn(int threads, bool plain3) {
  if (threads == 128) return plain3 ? k_rounds_local<TPV, 128, true> : k_rounds_local<TPV, 128, false>;
  if (threads == 256) return plain3 ? k_rounds_local<TPV, 256, true> : k_rounds_local<TPV, 256, false>;
  return plain3 ? k_rounds_local<TPV, 512, true> : k_rounds_local<TPV, 512, false>;
}

LocalFn local_kernel(const LocalPlan& P, bool plain3) {
  switch (P.tpv) {
    case 8: return local_fn<8>(P.threads, plain3);
    case 4: return local_fn<4>(P.threads, plain3);
    case 2: return local_fn<2>(P.threads, plain3);
    default: return local_fn<1>(P.threads, plain3);
  }
}

}  // namespace

// Shape of the local rounds, threads = 0 when the tables they read are not
// built, the formula does not fit or the resident rounds would be faster.
LocalPlan local_plan(const DevFormula& F, const DevTables& T, int Bp) {
  LocalPlan P;
  if (!T.rec3 || !T.ptab || !T.pva) return P;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    return P;
  // a thread per clause up to 512 (one block per SM at its registers), 256 when
  // there are octets for more than one block per SM; as many threads per
  // variable as keep all of them busy
  const double octets = Bp / 8;
  const int threads = F.m <= 192 ? 128 : F.m <= 768 || octets > sms ? 256 : 512;
  int tpv = 8;
  while (tpv > 1 && F.n * tpv > 2 * threads) tpv /= 2;
  P.tpv = tpv;
  P.threads = threads;
  const int smem = local_layout(F.n, F.m, F.nnz, T.n_groups, T.ptab_stride, T.pv_len, threads).total;
  auto kern = local_kernel(P, T.plain3 != 0);
  int per_sm = 0;
  if (smem > 220 * 1024 || allow_dynamic_smem(kern, smem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    P.threads = 0;
    return P;
  }
  // Cycles of a round, fitted to both forms over n = 50 .. 900, m = 215 .. 4000,
  // 64 .. 4096 chains (local / resident us a round: n = 50, m = 215: 1.9 / 6.9 at
  // 256 chains, 5.0 / 8.3 at 4096; n = 317, m = 1571: 6.0 / 7.7, 24 / 21; n = 600,
  // m = 3600: 12.7 / 10.5, 50 / 36): warp instructions at 2.2 a cycle and SM;
  // the local form runs its blocks in waves, the resident form waits on its
  // barriers and on L2 latencies whatever the work.
  const double instr = (F.m * 300.0 + F.nnz * 20.0 + F.n * 200.0) / 32.0;
  const double waves = std::ceil(octets / ((double)per_sm * sms));
  const double per_wave = std::min((double)per_sm, std::ceil(octets / sms));
  const double local = 1.2 * waves * (1500.0 + per_wave * instr / 2.2);
  const double resident =
      14000.0 + 7000.0 * std::min(1.0, F.m / 3000.0) + octets * instr / 2.2 / sms;
  if (local > resident) P.threads = 0;
  return P;
}

cudaError_t launch_rounds_local(const DevFormula& F, const DevTables& T, const DevChains& C,
                                const LocalFormula& L, const LocalPlan& P, uint32_t t0, int rounds,
                                float alpha, cudaStream_t st) {
  auto kern = local_kernel(P, T.plain3 != 0);
  const int smem = local_layout(F.n, F.m, F.nnz, T.n_groups, T.ptab_stride, T.pv_len, P.threads).total;
  const cudaError_t e = allow_dynamic_smem(kern, smem);
  if (e != cudaSuccess) return e;
  volatile float one = 1.0f;
  const float keep = one - alpha;
  kern<<<C.Bp / 8, P.threads, smem, st>>>(F, T, C, L, t0, rounds, keep);
  return cudaGetLastError();
}

}  // namespace rbmsat
