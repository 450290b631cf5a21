// KVQuant-style b-bit KV cache (Section 2.1, KVQuant paragraph): calibration,
// quantization (prefill bulk and per-step append) and the table preparation
// used by the fused-dequant decode kernel (decode_kvq.cu).
//
// Codes are decided with correctly rounded fp32 operations (__fsub_rn,
// __fdiv_rn, __fmul_rn, rintf) so that they are defined bit for bit:
//   uniform: code = clamp(rint((x - lo) / scale), 0, 2^b - 1)
//   NUQ:     code = #{j : x > mu_j},  mu_j = (c_j + c_{j+1}) * 0.5 in fp32
// Key outliers: x < t_lo or x > t_hi (per channel); value outliers: the n_v
// entries of largest |x| per token (ties: lower channel).  Outliers keep the
// code of their clamped value and are stored exactly in fp16 on the side.
#include <math.h>

#include <algorithm>

#include "mkv_common.cuh"
#include "mkv_internal.h"
#include "mkv_quant_token.cuh"

namespace mkv {

namespace {

__device__ uint32_t g_status_kvquant;

// ----------------------------------------------------------------- prepare

// k_dq[h][c][j] = k_lo + j * k_scale (uniform) or the fp16 centroid (NUQ);
// v_tbl[h][c][j] = j (uniform) or the fp16 value centroid (NUQ).
__global__ void prepare_kernel(int n, int K, int nuq, const float* k_lo, const float* k_scale,
                               const uint16_t* k_cb, const uint16_t* v_cb, float* k_dq, uint16_t* v_tbl) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * K; e += gridDim.x * blockDim.x) {
    const int hc = e / K, j = e % K;
    if (nuq) {
      k_dq[e] = h2f(k_cb[e]);
      v_tbl[e] = v_cb[e];
    } else {
      k_dq[e] = __fadd_rn(k_lo[hc], __fmul_rn((float)j, k_scale[hc]));
      v_tbl[e] = __half_as_ushort(__float2half_rn((float)j));
    }
  }
}

// ----------------------------------------------------------------- quantize

struct QuantArgs {
  const __half* k_pre;   // [B][Hkv][n][D]
  const __half* v;
  int64_t n_tokens;
  int Hkv, D, bits, nuq, n_v;
  const float* t_lo;     // [Hkv][D]
  const float* t_hi;
  const float* k_lo;
  const float* k_scale;
  const uint16_t* k_cb;  // [Hkv][D][K]
  const uint16_t* v_cb;
  int32_t* T_len;
  uint8_t* k_codes;      // [B][Hkv][T_cap][row]
  uint8_t* v_codes;
  float2* v_params;      // [B][Hkv][T_cap]
  uint32_t* v_out;       // [B][Hkv][T_cap][n_v]
  int32_t* k_out_off;    // [B][Hkv][T_cap+1]
  uint32_t* k_out;       // [B][Hkv][k_out_cap]
  int64_t k_out_cap;
  int64_t T_cap;
  int trigger;           // let the decode of the same step start (mkv_kvquant_step)
  int tickets;           // 0: more kv-heads than the tickets in T_len's top 8 bits count; advance_kernel follows
};

// One CTA per (batch, kv-head), one thread per channel; tokens in order so the
// key-outlier CSR is appended sequentially.  Every CTA reads T_len[b] once; the
// last CTA of batch entry b to finish stores the new length: during the launch
// the top 8 bits of T_len[b] count the finished CTAs (readers mask them off).
__global__ void quantize_kernel(const QuantArgs a) {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");   // (no-op in a plain launch)
  if (a.trigger) asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  extern __shared__ uint8_t sm[];
  const int D = a.D, K = 1 << a.bits, L = K - 1;
  const int bh = blockIdx.x;
  const int b = bh / a.Hkv, h = bh % a.Hkv;
  const int c = threadIdx.x;   // channel
  uint8_t* kcode = sm;                       // [D]
  uint8_t* vcode = kcode + D;                // [D]
  float* absx = reinterpret_cast<float*>(vcode + D);   // [D] value magnitudes
  uint32_t* words = reinterpret_cast<uint32_t*>(absx + D);   // [2][D*bits/32] packed rows
  __shared__ int s_cnt[32];
  __shared__ float s_lo[32], s_hi[32];
  __shared__ uint32_t s_max[2][32];

  // Every load that does not depend on the length is issued before it: the channel's parameters and
  // codebooks, and the first token's key and value; then the length and the CSR offset it selects.
  const float tlo = a.t_lo[h * D + c], thi = a.t_hi[h * D + c];
  const float klo = a.k_lo ? a.k_lo[h * D + c] : 0.f, ksc = a.k_scale ? a.k_scale[h * D + c] : 0.f;
  uint16_t kr[16], vr[16];                   // all codebook loads in flight at once (K <= 16)
  if (a.nuq) {
    const uint16_t* kc = a.k_cb + ((int64_t)h * D + c) * K;
    const uint16_t* vc = a.v_cb + ((int64_t)h * D + c) * K;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      if (j < K) {
        kr[j] = __ldg(kc + j);
        vr[j] = __ldg(vc + j);
      }
    }
  }
  const int64_t src0 = (int64_t)bh * a.n_tokens * D + c;
  __half xk_next = a.n_tokens > 0 ? a.k_pre[src0] : __ushort_as_half(0);
  __half xv_next = a.n_tokens > 0 ? a.v[src0] : __ushort_as_half(0);
  const int64_t t_base = a.T_len[b] & 0xffffff;
  int32_t* off_row = a.k_out_off + (int64_t)bh * (a.T_cap + 1);
  const bool room = t_base + a.n_tokens <= a.T_cap;
  int32_t off = (t_base == 0 || !room) ? 0 : off_row[t_base];
  // the last CTA of batch entry b stores its new length (after every thread of this CTA read it)
  auto finish = [&](int64_t len) {
    __syncthreads();
    if (c == 0 && a.tickets) {
      const unsigned old = atomicAdd(reinterpret_cast<unsigned*>(a.T_len) + b, 1u << 24);
      if ((int)(old >> 24) == a.Hkv - 1) a.T_len[b] = (int32_t)len;
    }
  };
  if (!room) {                            // no room: drop, flag, keep T_len
    if (c == 0 && h == 0) atomicOr(&g_status_kvquant, MKV_FLAG_CACHE_FULL);
    finish(t_base);
    return;
  }
  float kmu[15], vmu[15];
  if (a.nuq) {
#pragma unroll
    for (int j = 0; j < 15; ++j) {
      if (j < L) {
        kmu[j] = fl32_mid(h2f(kr[j]), h2f(kr[j + 1]));
        vmu[j] = fl32_mid(h2f(vr[j]), h2f(vr[j + 1]));
      }
    }
  }
  if (t_base == 0 && c == 0) off_row[0] = 0;
  const QTokDst dst{a.k_out + (int64_t)bh * a.k_out_cap, a.k_out_cap, a.v_out + (int64_t)bh * a.T_cap * a.n_v,
                    a.v_params + (int64_t)bh * a.T_cap, a.k_codes + (int64_t)bh * a.T_cap * (D * a.bits / 8),
                    a.v_codes + (int64_t)bh * a.T_cap * (D * a.bits / 8), off_row};
  const QTokSmem scr{kcode, vcode, absx, words, s_cnt, s_lo, s_hi, &s_max[0][0]};
  for (int64_t i = 0; i < a.n_tokens; ++i) {
    const __half xk = xk_next, xv = xv_next;     // this token's key and value; the next one's in flight
    if (i + 1 < a.n_tokens) {
      xk_next = a.k_pre[src0 + (i + 1) * D];
      xv_next = a.v[src0 + (i + 1) * D];
    }
    off = quantize_token(c, D, a.bits, a.nuq != 0, a.n_v, kmu, vmu, tlo, thi, klo, ksc, xk, xv, t_base + i, off, dst,
                         scr, &g_status_kvquant, [] { __syncthreads(); });
  }
  finish(t_base + a.n_tokens);
}

// The new lengths where quantize_kernel did not store them.
__global__ void advance_kernel(int32_t* T_len, int B, int32_t n, int64_t T_cap) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < B && (int64_t)T_len[b] + n <= T_cap) T_len[b] += n;
}

// ----------------------------------------------------------------- bulk quantize (a prompt)
//
// Many tokens at once: the prompt of every (batch, kv-head) is cut into P * kBulkWarps runs of
// tokens, one warp each, and a warp quantizes its tokens by itself, without barriers.
// The CSR of the key outliers needs each run's first entry: quantize_count_kernel counts the runs'
// outliers (one more pass over the keys), the last CTA of a batch entry turns the counts into entry
// offsets, and both pass through the CSR slot of the run's first token, which the run overwrites.
//
// B = 8, 8 kv-heads, T = 8192, D = 128, 4 bits: 0.32 ms (count 33 us, quantize 287 us), where one CTA
// per unit with its tokens in order took 13.4 ms (64 CTAs, a barrier chain of ~1.6 us a token).  Bound
// by instruction issue (about 400 warp instructions a token, IPC 2.5) rather than by its 349 MB, so:
//  * key codes and outliers are decided on fp16 pairs: for fp16 x, x > mu is x > (mu rounded down),
//    x < t is x < (t rounded up);
//  * codebook searches descend a tree of thresholds (ascending midpoints; a codebook out of order is
//    counted linearly, as quantize_token does): the keys' in registers, the values' upper levels in
//    registers and their last two in one 16-byte shared-memory read, which keeps 16 warps per SM;
//  * the n_v largest |x| and the value range of a token are warp reductions (redux.sync) over
//    order-preserving integer keys;
//  * a warp takes two tokens at a time, so that their dependent chains overlap (one at a time: 0.50 ms).

constexpr int kBulkWarps = 8;
constexpr int64_t kBulkMinTokens = 6;

// Token run of warp w of a unit: [w * per_w, (w + 1) * per_w) of the call's n tokens.
struct BulkSplit {
  int P;          // CTAs per (batch, kv-head); P * Hkv <= 256 (the tickets in T_len's top 8 bits)
  int64_t per_w;
};

// Streaming read of two or four fp16 (volatile: issued where written, so that several are in flight)
__device__ __forceinline__ uint32_t ld_stream4(const void* p) {
  uint32_t x;
  asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];\n" : "=r"(x) : "l"(p));
  return x;
}
__device__ __forceinline__ uint2 ld_stream8(const void* p) {
  uint2 x;
  asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];\n" : "=r"(x.x), "=r"(x.y) : "l"(p));
  return x;
}

template <int D>
__global__ void __launch_bounds__(kBulkWarps * 32) quantize_count_kernel(const QuantArgs a, const BulkSplit sp) {
  constexpr int NH = D / 64;               // fp16 pairs per lane
  const int64_t bh = blockIdx.y;
  const int b = (int)(bh / a.Hkv), h = (int)(bh % a.Hkv);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ int s_last;
  const int64_t t_base = a.T_len[b] & 0xffffff, n = a.n_tokens;
  if (t_base + n > a.T_cap) return;        // no room: quantize_bulk_kernel raises the flag
  __half2 lo[NH], hi[NH];                  // channels NH * 2 * lane ..
#pragma unroll
  for (int i = 0; i < NH; ++i) {
    const int64_t c = (int64_t)h * D + (lane * NH + i) * 2;
    lo[i] = __halves2half2(__float2half_ru(a.t_lo[c]), __float2half_ru(a.t_lo[c + 1]));
    hi[i] = __halves2half2(__float2half_rd(a.t_hi[c]), __float2half_rd(a.t_hi[c + 1]));
  }
  int32_t* off_row = a.k_out_off + bh * (a.T_cap + 1);
  const int64_t w0 = ((int64_t)blockIdx.x * kBulkWarps + warp) * sp.per_w, w1 = min(n, w0 + sp.per_w);
  const int m = (int)max((int64_t)0, w1 - w0);
  const __half* src = a.k_pre + (bh * n + w0) * D + lane * NH * 2;
  int cnt = 0;
  constexpr int U = 8;                     // rows in flight
  for (int t = 0; t < m; t += U) {
    uint32_t x[U][NH];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const __half* p = src + (int64_t)min(t + u, m - 1) * D;
      if constexpr (NH == 2) {
        const uint2 y = ld_stream8(p);
        x[u][0] = y.x;
        x[u][1] = y.y;
      } else {
        x[u][0] = ld_stream4(p);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t live = t + u < m ? 0x00010001u : 0u;
#pragma unroll
      for (int i = 0; i < NH; ++i) {
        const __half2 v = *reinterpret_cast<const __half2*>(&x[u][i]);
        cnt += __popc((__hlt2_mask(v, lo[i]) | __hgt2_mask(v, hi[i])) & live);
      }
    }
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if (lane == 0 && w0 < w1) off_row[t_base + w0 + 1] = cnt;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned old = atomicAdd(reinterpret_cast<unsigned*>(a.T_len) + b, 1u << 24);
    s_last = (int)(old >> 24) == (int)gridDim.x * a.Hkv - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int hh = warp; hh < a.Hkv; hh += kBulkWarps) {   // counts -> first entries, one warp per kv-head
    int32_t* row = a.k_out_off + ((int64_t)b * a.Hkv + hh) * (a.T_cap + 1) + t_base;
    int32_t run = t_base == 0 ? 0 : __ldcg(row);
    for (int i0 = 0; i0 < sp.P * kBulkWarps; i0 += 32) {
      const int64_t t = (int64_t)(i0 + lane) * sp.per_w;
      const bool in = i0 + lane < sp.P * kBulkWarps && t < n;
      const int32_t c = in ? __ldcg(row + t + 1) : 0;
      int32_t incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (in) row[t + 1] = run + incl - c;
      run += __shfl_sync(0xffffffffu, incl, 31);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) a.T_len[b] = (int32_t)t_base;   // the tickets cleared
}

// #{j : x > m_j} of the 2^BITS - 1 ascending thresholds of a channel: the upper BITS - 2 levels of
// the search tree in registers (top), then one 16-byte shared-memory read of the three thresholds
// left, as (middle, lower, upper).  `leaf` is the thread's entry of quadrant 0, STRIDE apart.
template <int BITS, int STRIDE>
__device__ __forceinline__ int tree_code(float x, const float (&top)[BITS == 4 ? 3 : 1], const float4* leaf) {
  int q = 0;
  if constexpr (BITS == 4) {               // top = m_7, m_3, m_11
    const bool up = x > top[0];
    q = (up ? 2 : 0) + (x > (up ? top[2] : top[1]) ? 1 : 0);
  } else if constexpr (BITS == 3) {        // top = m_3
    q = x > top[0] ? 1 : 0;
  }
  const float4 m = leaf[q * STRIDE];
  const bool up = x > m.x;
  return 4 * q + (up ? 2 : 0) + (x > (up ? m.z : m.y) ? 1 : 0);
}
// the linear count (any order of the thresholds)
template <int BITS, int STRIDE>
__device__ __forceinline__ int count_code(float x, const float (&top)[BITS == 4 ? 3 : 1], const float4* leaf) {
  int code = 0;
#pragma unroll
  for (int q = 0; q < (1 << (BITS - 2)); ++q) {
    const float4 m = leaf[q * STRIDE];
    code += (x > m.x) + (x > m.y) + (x > m.z);
    if (q + 1 < (1 << (BITS - 2))) code += x > top[q];
  }
  return code;
}
// the same for two fp16 values at once; codes in the two halves
template <int BITS>
__device__ __forceinline__ uint32_t tree_code2(__half2 x, const uint32_t (&m)[(1 << BITS) - 1]) {
  uint32_t cur[(1 << BITS) - 1];
#pragma unroll
  for (int i = 0; i < (1 << BITS) - 1; ++i) cur[i] = m[i];
  uint32_t code = 0;
#pragma unroll
  for (int l = BITS - 1; l >= 0; --l) {
    const int half = (1 << l) - 1;
    const uint32_t up = __hgt2_mask(x, *reinterpret_cast<const __half2*>(&cur[half]));
    code |= up & (0x00010001u << l);
#pragma unroll
    for (int i = 0; i < half; ++i) cur[i] = (up & cur[half + 1 + i]) | (~up & cur[i]);
  }
  return code;
}

// RN(d / s) for r = RN(1 / s): Markstein's correction (IBM J. Res. Dev. 34, 1990) applied twice, so
// that the second starts from a faithful quotient.  s is a difference of two fp16 values (or 1/3,
// 1/7, 1/15 of one) and d one of an fp16 value and such, so no remainder underflows; a quotient
// beyond 2^30 (d infinite, or far outside the range) is past every code's limit as it is.
__device__ __forceinline__ float div_rn(float d, float s, float r) {
  const float q0 = __fmul_rn(d, r);
  const float q1 = __fmaf_rn(__fmaf_rn(-q0, s, d), r, q0);
  const float q2 = __fmaf_rn(__fmaf_rn(-q1, s, d), r, q1);
  return fabsf(q0) < 1073741824.f ? q2 : q0;
}

__device__ __forceinline__ float f32_from_key(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? k & 0x7fffffffu : ~k);
}

// A token's code row from the 2 * BITS * (D / 64) bits of each lane's pairs, in lane order.
template <int D, int BITS>
__device__ __forceinline__ void store_codes(uint8_t* row, uint32_t x, int lane, bool live) {
  constexpr int LB = 2 * BITS * (D / 64);
  if constexpr (LB == 16) {
    if (live) reinterpret_cast<uint16_t*>(row)[lane] = (uint16_t)x;
  } else if constexpr (LB == 8) {
    if (live) row[lane] = (uint8_t)x;
  } else if constexpr (LB == 4) {
    const uint32_t y = __shfl_down_sync(0xffffffffu, x, 1);
    if (live && (lane & 1) == 0) row[lane >> 1] = (uint8_t)(x | (y << 4));
  } else {                                 // 12 or 6 bits: four lanes fill three 16- or 8-bit units
    constexpr int S = LB / 3;
    const uint32_t y = __shfl_down_sync(0xffffffffu, x, 1);
    const int j = lane & 3, at = (lane >> 2) * 3 + j;
    const uint32_t w = (x >> (S * j)) | (y << (LB - S * j));
    if (live && j < 3) {
      if constexpr (LB == 12)
        reinterpret_cast<uint16_t*>(row)[at] = (uint16_t)w;
      else
        row[at] = (uint8_t)w;
    }
  }
}

template <int D, int BITS, bool NUQ>
__global__ void __launch_bounds__(kBulkWarps * 32, 2) quantize_bulk_kernel(const QuantArgs a, const BulkSplit sp) {
  constexpr int NH = D / 64, NC = 2 * NH;  // fp16 pairs and channels per lane
  constexpr int K = 1 << BITS, L = K - 1, NQ = K / 4, ROW = D * BITS / 8;
  __shared__ uint32_t s_kmu[NUQ ? NH * L * 32 : 1];   // [pair][threshold][lane] key midpoints rounded down
  __shared__ float4 s_leaf[NUQ ? NQ * NC * 32 : 1];   // [quadrant][channel][lane] value midpoints
  const int64_t bh = blockIdx.y;
  const int b = (int)(bh / a.Hkv), h = (int)(bh % a.Hkv);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t_base = a.T_len[b] & 0xffffff, n = a.n_tokens;
  if (t_base + n > a.T_cap) {              // no room: drop, flag, keep T_len
    if (blockIdx.x == 0 && h == 0 && threadIdx.x == 0) atomicOr(&g_status_kvquant, MKV_FLAG_CACHE_FULL);
    return;
  }
  // channel j of lane l: D = 128: 2 l, 2 l + 1, 64 + 2 l, 65 + 2 l; D = 64: l, 32 + l
  auto chan_of = [](int j, int l) { return NH == 2 ? 2 * l + (j & 1) + (j >> 1) * 64 : l + j * 32; };
  auto chan = [&](int j) { return chan_of(j, lane); };
  bool sorted = true;
  if constexpr (NUQ) {
    for (int e = threadIdx.x; e < NC * 32 * L; e += kBulkWarps * 32) {
      const int j = e / (32 * L), l = e / L % 32, m = e % L;
      const int64_t hc = ((int64_t)h * D + chan_of(j, l)) * K + m;
      const float c0 = h2f(a.k_cb[hc]), c1 = h2f(a.k_cb[hc + 1]), v0 = h2f(a.v_cb[hc]), v1 = h2f(a.v_cb[hc + 1]);
      const float km = fl32_mid(c0, c1), vm = fl32_mid(v0, v1);
      sorted = sorted && c0 <= c1 && v0 <= v1 && km == km && vm == vm;   // then the midpoints ascend too
      reinterpret_cast<__half*>(s_kmu)[(((j >> 1) * L + m) * 32 + l) * 2 + (j & 1)] =
          __float2half_rd(km);
      // quadrant m / 4 holds m_4q .. m_4q+2 as (middle, lower, upper, the threshold after it)
      constexpr int at[4] = {1, 0, 2, 3};
      reinterpret_cast<float*>(s_leaf)[(((m >> 2) * NC + j) * 32 + l) * 4 + at[m & 3]] = vm;
    }
  }
  sorted = __syncthreads_and(sorted);
  uint32_t lo2[NH], hi2[NH];               // outlier thresholds as fp16 pairs
  uint32_t kmu[NH][L];
  float top[NC][BITS == 4 ? 3 : 1];        // the value search's upper levels
  float klo[NC], ksc[NC];                  // uniform: key grid
#pragma unroll
  for (int i = 0; i < NH; ++i) {
    uint16_t lo[2], hi[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int j = 2 * i + e;
      const int64_t hc = (int64_t)h * D + chan(j);
      lo[e] = __half_as_ushort(__float2half_ru(a.t_lo[hc]));
      hi[e] = __half_as_ushort(__float2half_rd(a.t_hi[hc]));
      if constexpr (NUQ) {
        if constexpr (BITS == 4) {
          top[j][0] = s_leaf[(1 * NC + j) * 32 + lane].w;
          top[j][1] = s_leaf[(0 * NC + j) * 32 + lane].w;
          top[j][2] = s_leaf[(2 * NC + j) * 32 + lane].w;
        } else {
          top[j][0] = BITS == 3 ? s_leaf[j * 32 + lane].w : 0.f;
        }
      } else {
        klo[j] = a.k_lo[hc];
        ksc[j] = a.k_scale[hc];
      }
    }
    lo2[i] = (uint32_t)lo[0] | ((uint32_t)lo[1] << 16);
    hi2[i] = (uint32_t)hi[0] | ((uint32_t)hi[1] << 16);
    if constexpr (NUQ) {
#pragma unroll
      for (int m = 0; m < L; ++m) kmu[i][m] = s_kmu[(i * L + m) * 32 + lane];
    }
  }

  const int64_t w0 = ((int64_t)blockIdx.x * kBulkWarps + warp) * sp.per_w, w1 = min(n, w0 + sp.per_w);
  int32_t* off_row = a.k_out_off + bh * (a.T_cap + 1) + t_base;
  if (w0 < w1) {
    const int m = (int)(w1 - w0);          // this warp's tokens
    uint32_t* k_out = a.k_out + bh * a.k_out_cap;
    const int32_t cap = (int32_t)min(a.k_out_cap, (int64_t)INT32_MAX);
    const int64_t d0 = bh * a.T_cap + t_base + w0;
    uint32_t* v_out = a.v_out + d0 * a.n_v;
    float2* v_par = a.v_params + d0;
    uint8_t* kc = a.k_codes + d0 * ROW;
    uint8_t* vc = a.v_codes + d0 * ROW;
    const uint8_t* ks = reinterpret_cast<const uint8_t*>(a.k_pre + (bh * n + w0) * D) + lane * (NH == 2 ? 4 : 2);
    const uint8_t* vs = reinterpret_cast<const uint8_t*>(a.v + (bh * n + w0) * D) + lane * (NH == 2 ? 4 : 2);
    const int t0 = (int)((t_base + w0) & 63);
    off_row += w0 + 1;
    int32_t off = off_row[0];              // the run's first entry (from quantize_count_kernel)
    __syncwarp();
    const unsigned lt = (1u << lane) - 1u;
    auto load = [&](const uint8_t* base, int t, uint32_t (&x)[NH]) {
      const uint8_t* p = base + (int64_t)min(t, m - 1) * (D * 2);
      if constexpr (NH == 2) {
        x[0] = ld_stream4(p);
        x[1] = ld_stream4(p + 128);
      } else {
        x[0] = (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(p)) |
               ((uint32_t)__ldg(reinterpret_cast<const uint16_t*>(p + 64)) << 16);
      }
    };
    uint32_t kn[2][NH], vn[2][NH];         // the next two tokens' rows, in flight
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      load(ks, e, kn[e]);
      load(vs, e, vn[e]);
    }
    int32_t my_off = 0;                    // of token 32 * i + lane of the run: end of its entries,
    float2 my_par = make_float2(0.f, 0.f); // value range
    // two tokens at a time: their dependent chains (searches, warp reductions, divisions) overlap
    for (int t = 0; t < m; t += 2) {
      uint32_t kx[2][NH], vx[2][NH];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
#pragma unroll
        for (int i = 0; i < NH; ++i) {
          kx[e][i] = kn[e][i];
          vx[e][i] = vn[e][i];
        }
        load(ks, t + 2 + e, kn[e]);
        load(vs, t + 2 + e, vn[e]);
      }
      const bool two = t + 1 < m;
      // a lane's pairs in order: D = 128: (2 lane, 64 + 2 lane), (2 lane + 1, ..); D = 64: (lane, 32 + lane)
      auto pack = [&](const uint32_t (&c)[NH]) -> uint32_t {
        if constexpr (NH == 2) {
          const uint32_t w = c[0] | (c[1] << BITS);
          return (w & 0xffffu) | ((w >> 16) << (2 * BITS));
        } else {
          return (c[0] & 0xffffu) | ((c[0] >> 16) << BITS);
        }
      };
      // ---- values: the n_v largest |x| (ties: lower channel), each found by a warp maximum over
      // unique keys (|x| as fp16 bits, 255 - channel, sign)
      uint32_t key[2][NC];
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int j = 0; j < NC; ++j) {
          const uint32_t x = (vx[e][j >> 1] >> (16 * (j & 1))) & 0xffffu;
          key[e][j] = ((x & 0x7fffu) << 9) | (x >> 15) | (uint32_t)((255 - chan(j)) << 1);
        }
#pragma unroll 1
      for (int r = 0; r < a.n_v; ++r) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          uint32_t mx = key[e][0];
#pragma unroll
          for (int j = 1; j < NC; ++j) mx = max(mx, key[e][j]);
          const uint32_t w = __reduce_max_sync(0xffffffffu, mx);
#pragma unroll
          for (int j = 0; j < NC; ++j) key[e][j] = key[e][j] == w ? 0u : key[e][j];   // live keys are nonzero
          if (lane == 0 && (e == 0 || two))
            v_out[e * a.n_v + r] = ((255u - ((w >> 1) & 255u)) << 16) | (w >> 9) | ((w & 1u) << 15);
        }
      }
      v_out += 2 * a.n_v;
      // ---- keys: codes (packed by pairs of channels) and outliers
      uint32_t code[2][NH], om[2][NH];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
#pragma unroll
        for (int i = 0; i < NH; ++i) {
          const __half2 x = *reinterpret_cast<const __half2*>(&kx[e][i]);
          om[e][i] = __hlt2_mask(x, *reinterpret_cast<const __half2*>(&lo2[i])) |
                     __hgt2_mask(x, *reinterpret_cast<const __half2*>(&hi2[i]));
          if constexpr (NUQ) {
            code[e][i] = tree_code2<BITS>(x, kmu[i]);
          } else {
            const float2 f = __half22float2(x);
            code[e][i] = (uint32_t)uniform_code(f.x, klo[2 * i], ksc[2 * i], L) |
                         ((uint32_t)uniform_code(f.y, klo[2 * i + 1], ksc[2 * i + 1], L) << 16);
          }
        }
      }
      if (NUQ && !sorted) {
#pragma unroll 1
        for (int e = 0; e < 2; ++e) {
#pragma unroll
          for (int i = 0; i < NH; ++i) {
            uint32_t c = 0;
#pragma unroll
            for (int q = 0; q < L; ++q) {
              const uint32_t x = e ? kx[1][i] : kx[0][i];
              c += __hgt2_mask(*reinterpret_cast<const __half2*>(&x), *reinterpret_cast<const __half2*>(&kmu[i][q])) &
                   0x00010001u;
            }
            (e ? code[1][i] : code[0][i]) = c;
          }
        }
      }
      store_codes<D, BITS>(kc, pack(code[0]), lane, true);
      store_codes<D, BITS>(kc + ROW, pack(code[1]), lane, two);
      kc += 2 * ROW;
      // ---- value ranges
      float x[2][NC], lo[2], hi[2], scale[2], u[2][NC];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        lo[e] = INFINITY;
        hi[e] = -INFINITY;
#pragma unroll
        for (int j = 0; j < NC; ++j) {
          x[e][j] = h2f((uint16_t)(vx[e][j >> 1] >> (16 * (j & 1))));
          lo[e] = fminf(lo[e], key[e][j] == 0u ? INFINITY : x[e][j]);
          hi[e] = fmaxf(hi[e], key[e][j] == 0u ? -INFINITY : x[e][j]);
        }
        lo[e] = f32_from_key(__reduce_min_sync(0xffffffffu, f32_key(lo[e])));
        hi[e] = f32_from_key(__reduce_max_sync(0xffffffffu, f32_key(hi[e])));
        if (lo[e] > hi[e]) lo[e] = hi[e] = 0.f;   // no inlier
        const float width = __fsub_rn(hi[e], lo[e]);
        scale[e] = NUQ ? width : __fdiv_rn(width, (float)L);
        const float rcp = __frcp_rn(scale[e]);
#pragma unroll
        for (int j = 0; j < NC; ++j) {
          x[e][j] = __fsub_rn(x[e][j], lo[e]);
          u[e][j] = div_rn(x[e][j], scale[e], rcp);
        }
      }
      if (!(scale[0] > 0.f && scale[0] < INFINITY && scale[1] > 0.f && scale[1] < INFINITY)) {
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
          for (int j = 0; j < NC; ++j) u[e][j] = scale[e] == 0.f ? 0.f : __fdiv_rn(x[e][j], scale[e]);
      }
      // ---- value codes
#pragma unroll
      for (int e = 0; e < 2; ++e) {
#pragma unroll
        for (int i = 0; i < NH; ++i) code[e][i] = 0;
#pragma unroll
        for (int j = 0; j < NC; ++j) {
          int cj;
          if constexpr (NUQ)
            cj = sorted ? tree_code<BITS, NC * 32>(u[e][j], top[j], s_leaf + j * 32 + lane)
                        : count_code<BITS, NC * 32>(u[e][j], top[j], s_leaf + j * 32 + lane);
          else
            cj = (int)fminf(fmaxf(rintf(u[e][j]), 0.f), (float)L);
          code[e][j >> 1] |= (uint32_t)cj << (16 * (j & 1));
        }
      }
      store_codes<D, BITS>(vc, pack(code[0]), lane, true);
      store_codes<D, BITS>(vc + ROW, pack(code[1]), lane, two);
      vc += 2 * ROW;

      // ---- key-outlier entries in channel order: (D = 128) the lanes' first pairs of channels, then
      // their second; then the token's range and end of entries, kept by one lane and stored 32 tokens
      // at a time
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        if (e == 1 && !two) break;
        if (__any_sync(0xffffffffu, (om[e][0] | om[e][NH - 1]) != 0u)) {
          const uint32_t tag = (uint32_t)((t0 + t + e) & 63) << 24;
          auto put = [&](int32_t at, int j, uint32_t bits) {
            if (at < cap)
              k_out[at] = tag | ((uint32_t)chan(j) << 16) | bits;
            else
              atomicOr(&g_status_kvquant, MKV_FLAG_K_OUTLIER_OVERFLOW);
          };
#pragma unroll
          for (int i = 0; i < NH; ++i) {
            const bool o0 = om[e][i] & 0xffffu, o1 = om[e][i] >> 16;
            const unsigned b0 = __ballot_sync(0xffffffffu, o0), b1 = __ballot_sync(0xffffffffu, o1);
            if constexpr (NH == 2) {
              const int32_t at = off + __popc(b0 & lt) + __popc(b1 & lt);
              if (o0) put(at, 2 * i, kx[e][i] & 0xffffu);
              if (o1) put(at + (o0 ? 1 : 0), 2 * i + 1, kx[e][i] >> 16);
            } else {
              if (o0) put(off + __popc(b0 & lt), 0, kx[e][i] & 0xffffu);
              if (o1) put(off + __popc(b0) + __popc(b1 & lt), 1, kx[e][i] >> 16);
            }
            off += __popc(b0) + __popc(b1);
          }
        }
        const int at = (t + e) & 31;
        if (lane == at) {
          my_off = off;
          my_par = make_float2(lo[e], scale[e]);
        }
        if (at == 31 || t + e + 1 == m) {
          if (lane <= at) {
            off_row[t + e - at + lane] = my_off;
            v_par[t + e - at + lane] = my_par;
          }
        }
      }
    }
  }
  if (t_base == 0 && blockIdx.x == 0 && threadIdx.x == 0) a.k_out_off[bh * (a.T_cap + 1)] = 0;
  __syncthreads();                         // every thread of this CTA has read T_len
  if (threadIdx.x == 0) {
    const unsigned old = atomicAdd(reinterpret_cast<unsigned*>(a.T_len) + b, 1u << 24);
    if ((int)(old >> 24) == (int)gridDim.x * a.Hkv - 1) a.T_len[b] = (int32_t)(t_base + n);
  }
}

template <int D, int BITS>
cudaError_t launch_bulk_t(const QuantArgs& a, int B, cudaStream_t st) {
  // CTAs per unit: fewest (waves of two CTAs per SM) x (tokens per warp + a run's fixed cost, about
  // eight tokens)
  BulkSplit sp{};
  int64_t best = INT64_MAX;
  for (int64_t p = 1; p <= std::min<int64_t>(256 / a.Hkv, ceil_div(a.n_tokens, kBulkWarps)); ++p) {
    const int64_t per = ceil_div(a.n_tokens, p * kBulkWarps);
    const int64_t cost = ceil_div(p * B * a.Hkv, 2 * kNumSMs) * (per + 8);
    if (cost < best) {
      best = cost;
      sp.per_w = per;
    }
  }
  sp.P = (int)ceil_div(a.n_tokens, sp.per_w * kBulkWarps);
  const dim3 grid(sp.P, B * a.Hkv);
  quantize_count_kernel<D><<<grid, kBulkWarps * 32, 0, st>>>(a, sp);
  const cudaError_t e = cudaPeekAtLastError();
  if (e != cudaSuccess) return e;
  if (a.nuq)
    quantize_bulk_kernel<D, BITS, true><<<grid, kBulkWarps * 32, 0, st>>>(a, sp);
  else
    quantize_bulk_kernel<D, BITS, false><<<grid, kBulkWarps * 32, 0, st>>>(a, sp);
  return cudaPeekAtLastError();
}

template <int D>
cudaError_t launch_bulk_d(const QuantArgs& a, int B, cudaStream_t st) {
  if (a.bits == 4) return launch_bulk_t<D, 4>(a, B, st);
  if (a.bits == 3) return launch_bulk_t<D, 3>(a, B, st);
  return launch_bulk_t<D, 2>(a, B, st);
}

// ----------------------------------------------------------------- calibrate

// Per (kv-head, calibration token): u = fl32((x - lo) / s) of the token's inlier values, kMasked for
// its outliers.  One warp per token (the warp reductions of quantize_bulk_kernel).
constexpr uint32_t kMasked = 0xffffffffu;   // no result of fp32 arithmetic has these bits
template <int D>
__global__ void __launch_bounds__(256) calib_values_kernel(const __half* v_cal, int64_t N, int64_t row_stride,
                                                           int64_t n_rows, int n_v, float* u_out) {
  constexpr int NC = D / 32;               // channels 2 NC' lane ..: pairs (2 lane, 2 lane + 1), + 64
  const int lane = threadIdx.x & 31;
  const int64_t ht = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (ht >= n_rows) return;
  const __half* row = v_cal + (ht / N * row_stride + ht % N) * D;
  uint32_t key[NC];
  float x[NC];
  auto chan = [&](int j) { return 2 * lane + (j & 1) + (j >> 1) * 64; };
#pragma unroll
  for (int j = 0; j < NC; ++j) {
    const uint32_t b = __half_as_ushort(row[chan(j)]);
    x[j] = h2f((uint16_t)b);
    key[j] = ((b & 0x7fffu) << 8) | (uint32_t)(255 - chan(j));
  }
  for (int r = 0; r < n_v; ++r) {          // the n_v largest |x| (ties: lower channel)
    uint32_t m = key[0];
#pragma unroll
    for (int j = 1; j < NC; ++j) m = max(m, key[j]);
    m = __reduce_max_sync(0xffffffffu, m);
#pragma unroll
    for (int j = 0; j < NC; ++j) key[j] = key[j] == m ? 0u : key[j];
  }
  float lo = INFINITY, hi = -INFINITY;
#pragma unroll
  for (int j = 0; j < NC; ++j) {
    lo = fminf(lo, key[j] == 0u ? INFINITY : x[j]);
    hi = fmaxf(hi, key[j] == 0u ? -INFINITY : x[j]);
  }
  lo = f32_from_key(__reduce_min_sync(0xffffffffu, f32_key(lo)));
  hi = f32_from_key(__reduce_max_sync(0xffffffffu, f32_key(hi)));
  if (lo > hi) lo = hi = 0.f;
  const float s = __fsub_rn(hi, lo);
#pragma unroll
  for (int j = 0; j < NC; ++j) {
    const float u = s == 0.f ? 0.f : __fdiv_rn(__fsub_rn(x[j], lo), s);
    u_out[ht * D + chan(j)] = key[j] == 0u ? __uint_as_float(kMasked) : u;
  }
}

// Ascending sort of the CTA's kCalThr * E values, value i = thread * E + e (blocked): a bitonic network
// whose merges begin with the mirrored comparison (i against i ^ (k - 1)), so every comparison puts the
// smaller value at the lower index.  Partners in the same thread meet in registers, in the same warp
// through shuffles, else through shared memory (sx, kCalThr * E floats).
constexpr int kCalThr = 512;
template <int E>
__device__ __forceinline__ void calib_sort(float (&v)[E], float* sx) {
  const int t = threadIdx.x;
  // the values of thread t ^ tm, element e from e (or mirrored): the smaller or the larger one stays
  auto exchange = [&](int tm, bool mirror, bool lower) {
    float o[E];
    if (tm < 32) {
#pragma unroll
      for (int e = 0; e < E; ++e) o[e] = __shfl_xor_sync(0xffffffffu, mirror ? v[E - 1 - e] : v[e], tm);
    } else {
      __syncthreads();
#pragma unroll
      for (int e = 0; e < E; ++e) sx[e * kCalThr + t] = v[e];
      __syncthreads();
#pragma unroll
      for (int e = 0; e < E; ++e) o[e] = sx[(mirror ? E - 1 - e : e) * kCalThr + (t ^ tm)];
    }
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = (v[e] < o[e]) == lower ? v[e] : o[e];
  };
  auto in_thread = [&](int m) {            // compare e with e ^ m
#pragma unroll
    for (int e = 0; e < E; ++e) {
      if ((e ^ m) > e) {
        const float x = v[e], y = v[e ^ m];
        v[e] = fminf(x, y);
        v[e ^ m] = fmaxf(x, y);
      }
    }
  };
#pragma unroll
  for (int k = 2; k <= E; k <<= 1) {
    in_thread(k - 1);
#pragma unroll
    for (int j = k / 4; j > 0; j >>= 1) in_thread(j);
  }
#pragma unroll 1
  for (int kt = 2; kt <= kCalThr; kt <<= 1) {   // merges of runs of kt threads' values
    exchange(kt - 1, true, (t & (kt / 2)) == 0);
#pragma unroll 1
    for (int j = kt / 4; j > 0; j >>= 1) exchange(j, false, (t & j) == 0);
#pragma unroll
    for (int j = E / 2; j > 0; j >>= 1) in_thread(j);
  }
}

__device__ uint16_t fp16_next_up(uint16_t bits) {
  if (bits == 0x8000u || bits == 0u) return 0x0001u;
  return (bits & 0x8000u) ? (uint16_t)(bits - 1u) : (uint16_t)(bits + 1u);
}

// Centroids rounded to fp16: sorted by value, then made strictly increasing.
__device__ void finish_codebook(int K, uint16_t* cb) {
  for (int j = 1; j < K; ++j) {
    const uint16_t v = cb[j];
    int m = j - 1;
    while (m >= 0 && __hgt(__ushort_as_half(cb[m]), __ushort_as_half(v))) {
      cb[m + 1] = cb[m];
      --m;
    }
    cb[m + 1] = v;
  }
  for (int j = 1; j < K; ++j) {
    if (__hle(__ushort_as_half(cb[j]), __ushort_as_half(cb[j - 1]))) cb[j] = fp16_next_up(cb[j - 1]);
  }
}

// 1-D Lloyd k-means on sorted data x[0..n): quantile start, 25 iterations,
// nearest centroid (ties: lower index), means summed in ascending order in fp64,
// empty clusters keep their centroid; then fp16, sorted, made strictly increasing.
__device__ void lloyd_codebook(const float* x, int n, int K, uint16_t* out, double* cent, uint8_t* asg) {
  const int tid = threadIdx.x;
  if (tid < K) {
    int idx = (int)floor((tid + 0.5) * (double)n / K);
    cent[tid] = n > 0 ? (double)x[min(n - 1, idx)] : 0.0;
  }
  __syncthreads();
  for (int it = 0; it < 25 && n > 0; ++it) {
    for (int i = tid; i < n; i += blockDim.x) {
      const double xv = (double)x[i];
      int best = 0;
      double bd = fabs(xv - cent[0]);
      for (int j = 1; j < K; ++j) {
        const double d = fabs(xv - cent[j]);
        if (d < bd) {
          bd = d;
          best = j;
        }
      }
      asg[i] = (uint8_t)best;
    }
    __syncthreads();
    if (tid < K) {
      double sum = 0.0;
      int cnt = 0;
      for (int i = 0; i < n; ++i) {
        if (asg[i] == tid) {
          sum += (double)x[i];
          ++cnt;
        }
      }
      if (cnt > 0) cent[tid] = sum / (double)cnt;
    }
    __syncthreads();
  }
  if (tid == 0) {
    for (int j = 0; j < K; ++j) out[j] = __half_as_ushort(__double2half(cent[j]));
    finish_codebook(K, out);
  }
  __syncthreads();
}

// The same codebook by one warp from the sorted data and its exact integer prefix sums
// P[i] = sum_{e < i} x[e] * scale (mod 2^64, scale a power of two): a cluster is a run of the sorted data,
// found by a binary search and summed by one subtraction.  Where every partial sum of lloyd_codebook is
// exact (the caller checks), sums and therefore centroids are the same bits; they are kept in units of
// 1 / scale.  The nearest centroid by fp64 distances is kept exactly: between centroids a < b, "b is
// nearer" changes once along the data, and it is evaluated in fp64 on the two values around the
// boundary found unless they are clear of the midpoint by 2^-20 of the data's magnitude; centroids
// closer together than that, or out of order, could tie by rounding elsewhere.  In either case the warp
// gives up (false) and the caller takes lloyd_codebook.  (fp64 runs at two lanes a clock on this chip:
// one division and three conversions per iteration are left of it.)
__device__ __forceinline__ bool lloyd_sorted(const float* x, const unsigned long long* P, int n, int K, float scale,
                                             uint16_t* out) {
  const int lane = threadIdx.x;            // centroid
  const bool act = lane < K;
  const float inv = 1.f / scale;
  const float tol = fmaxf(fabsf(x[0]), fabsf(x[n - 1])) * 0x1p-20f;
  const double tol_s = (double)tol * scale;
  double c = 0.0;
  float cf = 0.f;                          // the centroid itself, to fp32
  if (act) {
    cf = x[min(n - 1, (int)floor((lane + 0.5) * (double)n / K))];
    c = (double)cf * scale;
  }
  int bnd = lane == 0 ? 0 : n;             // first value of the lane's cluster
  for (int it = 0; it < 25; ++it) {
    const double cp = __shfl_up_sync(0xffffffffu, c, 1);
    const float cpf = __shfl_up_sync(0xffffffffu, cf, 1);
    bool ok = true;
    if (act && lane > 0) {
      const float m = 0.5f * (cpf + cf);
      auto search = [&](float t) {         // first i with x[i] >= t, near the last boundary if it is there
        int lo = max(0, bnd - 32), hi = min(n, bnd + 32);
        if (!((lo == 0 || x[lo - 1] < t) && (hi == n || x[hi] >= t))) {
          lo = 0;
          hi = n;
        }
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (x[mid] >= t)
            hi = mid;
          else
            lo = mid + 1;
        }
        return lo;
      };
      auto nearer = [&](int i) {           // (tie: the lower centroid)
        const double xv = (double)x[i] * scale;
        return fabs(xv - c) < fabs(xv - cp);
      };
      bnd = search(m);
      const bool below = bnd == 0 || x[bnd - 1] < m - tol, above = bnd == n || x[bnd] > m + tol;
      ok = cf - cpf > 4.f * tol;
      if (!(below && above)) {
        ok = ok && c - cp > 2.0 * tol_s;
        // the midpoint to fp32 may fall on the wrong side of a value (and of its duplicates)
        if (bnd > 0 && nearer(bnd - 1))
          bnd = search(x[bnd - 1]);
        else if (bnd < n && !nearer(bnd))
          bnd = search(nextafterf(x[bnd], INFINITY));
        ok = ok && (bnd == 0 || !nearer(bnd - 1)) && (bnd == n || nearer(bnd));
      }
    }
    if (!__all_sync(0xffffffffu, ok)) return false;
    int end = __shfl_down_sync(0xffffffffu, bnd, 1);
    if (lane == K - 1) end = n;
    bool same = true;
    if (act && end > bnd) {
      const double cn = (double)(long long)(P[end] - P[bnd]) / (double)(end - bnd);
      same = __double_as_longlong(cn) == __double_as_longlong(c);
      c = cn;
      cf = (float)cn * inv;
    }
    if (__all_sync(0xffffffffu, same)) break;   // a fixed point: the iterations left change nothing
  }
  const __half h = __double2half(c * (double)inv);
  const __half hp = __ushort_as_half((unsigned short)__shfl_up_sync(0xffffffffu, (unsigned)__half_as_ushort(h), 1));
  if (!__all_sync(0xffffffffu, !act || lane == 0 || __hlt(hp, h))) {   // sort and nudge: one thread
    for (int j = 0; j < K; ++j) {
      const unsigned hj = __shfl_sync(0xffffffffu, (unsigned)__half_as_ushort(h), j);
      if (lane == 0) out[j] = (uint16_t)hj;
    }
    if (lane == 0) finish_codebook(K, out);
  } else if (act) {
    out[lane] = __half_as_ushort(h);
  }
  return true;
}

struct CalibArgs {
  const __half* k_cal;   // [Hkv][row_stride][D]
  const float* u;        // [Hkv][N][D], kMasked for outliers
  int64_t N, row_stride;
  int D, bits, nuq, nt, all_out;
  float* t_lo;
  float* t_hi;
  float* k_lo;
  float* k_scale;
  uint16_t* k_cb;
  uint16_t* v_cb;
};

// First index of s[0..n) (ascending) whose value is >= t (or > t).
__device__ __forceinline__ int first_at(const float* s, int n, float t, bool above) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (above ? s[mid] > t : s[mid] >= t)
      hi = mid;
    else
      lo = mid + 1;
  }
  return lo;
}

// grid (Hkv*D, 2): y = 0 keys, y = 1 values (NUQ only).  One channel per CTA: its N values sorted
// (E per thread), prefix sums, then one warp runs Lloyd's iterations.  4 bits, N = 4096, 8 x 128
// channels: the values' kernel 13 us, this one 240 us, the whole call 0.26 ms (55 ms with a brute-force
// fp64 search and sequential sums on every iteration); bound by the sort's instructions (45 thousand per
// channel) and the latency of the one warp that iterates.
template <int E>
__global__ void __launch_bounds__(kCalThr) calib_channel_kernel(const CalibArgs a) {
  constexpr int NP2 = kCalThr * E;
  extern __shared__ __align__(16) uint8_t smem[];
  unsigned long long* P = reinterpret_cast<unsigned long long*>(smem);   // [NP2 + 2] prefix sums
  float* s = reinterpret_cast<float*>(P + NP2 + 2);                      // [NP2]
  __shared__ unsigned long long s_warp[kCalThr / 32];
  __shared__ int s_cnt, s_fast, s_a, s_b;
  __shared__ double cent[16];
  const int hc = blockIdx.x;
  const int h = hc / a.D, c = hc % a.D;
  const bool values = blockIdx.y == 1;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int N = (int)a.N, K = 1 << a.bits, L = K - 1;
  if (t == 0) s_cnt = 0;
  float v[E];
  int cnt = 0;
#pragma unroll
  for (int e = 0; e < E; ++e) {            // any order: the values are sorted next
    const int i = e * kCalThr + t;
    v[e] = INFINITY;
    if (i < N) {
      if (!values) {
        v[e] = __half2float(a.k_cal[((int64_t)h * a.row_stride + i) * a.D + c]);
      } else {
        const float u = a.u[((int64_t)h * N + i) * a.D + c];
        if (__float_as_uint(u) != kMasked) {
          v[e] = u;
          ++cnt;
        }
      }
    }
  }
  calib_sort<E>(v, s);
  __syncthreads();
#pragma unroll
  for (int e = 0; e < E; ++e) s[t * E + e] = v[e];
  if (values) {
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) atomicAdd(&s_cnt, cnt);
  }
  // exact prefix sums: keys are multiples of 2^-24; normalized values of at least 2^-18 (checked
  // below) multiples of 2^-41
  const float scale = values ? 0x1p41f : 0x1p24f;
  unsigned long long q[E], run = 0;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    q[e] = run;
    run += (unsigned long long)__float2ll_rn(v[e] * scale);
  }
  unsigned long long incl = run;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  unsigned long long base = incl - run;
  for (int w = 0; w < warp; ++w) base += s_warp[w];
#pragma unroll
  for (int e = 0; e < E; ++e) P[t * E + e] = base + q[e];
  if (t == kCalThr - 1) P[NP2] = base + run;
  __syncthreads();
  if (warp == 0) {
    int ia = 0, ib = s_cnt;
    if (!values) {
      float tl = INFINITY, th = -INFINITY;
      ib = 0;
      if (!a.all_out) {                    // inliers: the sorted range with tl <= x <= th
        tl = s[a.nt];
        th = s[N - 1 - a.nt];
        ia = first_at(s, N, tl, false);
        ib = first_at(s, N, th, true);
      }
      if (lane == 0) {
        a.t_lo[hc] = tl;
        a.t_hi[hc] = th;
        const float lo = a.all_out ? 0.f : tl, hi = a.all_out ? 0.f : th;
        if (a.k_lo) a.k_lo[hc] = lo;
        if (a.k_scale) a.k_scale[hc] = __fdiv_rn(__fsub_rn(hi, lo), (float)L);
      }
    }
    bool fast = a.nuq && ib > ia;
    if (fast) {                            // finite; keys: |sums| < 2^28; values: in [0, 1], none in (0, 2^-18)
      fast = s[ia] > -INFINITY && s[ib - 1] < INFINITY;
      if (values) {
        const int z = first_at(s, ib, 0.f, true);
        fast = fast && s[ia] >= 0.f && s[ib - 1] <= 1.f && (z == ib || s[z] >= 0x1p-18f);
      }
    }
    if (fast)
      fast = lloyd_sorted(s + ia, P + ia, ib - ia, K, scale,
                          (values ? a.v_cb : a.k_cb) + (int64_t)hc * K);
    if (lane == 0) {
      s_fast = fast;
      s_a = ia;
      s_b = ib;
    }
  }
  __syncthreads();
  if (a.nuq && !s_fast)                    // the prefix sums' room takes the assignments
    lloyd_codebook(s + s_a, s_b - s_a, K, (values ? a.v_cb : a.k_cb) + (int64_t)hc * K, cent,
                   reinterpret_cast<uint8_t*>(P));
}

template <int E>
cudaError_t launch_calib_t(const CalibArgs& a, int channels, cudaStream_t st) {
  constexpr int smem = (kCalThr * E + 2) * 8 + kCalThr * E * 4;
  const cudaError_t e = cudaFuncSetAttribute(calib_channel_kernel<E>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  calib_channel_kernel<E><<<dim3(channels, a.nuq ? 2 : 1), kCalThr, smem, st>>>(a);
  return cudaPeekAtLastError();
}

}  // namespace

cudaError_t launch_quant_prepare(const mkv_config& c, const mkv_quant_params& qp, cudaStream_t st) {
  const int n = c.Hkv * c.D, K = 1 << c.bits;
  prepare_kernel<<<(int)ceil_div((int64_t)n * K, 256), 256, 0, st>>>(
      n, K, c.quant_mode == MKV_QUANT_NUQ, qp.k_lo, qp.k_scale, qp.k_cb, qp.v_cb, qp.k_dq, qp.v_tbl);
  return cudaPeekAtLastError();
}

cudaError_t launch_quantize(const mkv_config& c, const mkv_quant_params& qp, const void* k_pre, const void* v,
                            int64_t n_tokens, const mkv_cache& cache, cudaStream_t st, bool step) {
  QuantArgs a{};
  a.trigger = step;
  a.tickets = c.Hkv <= 256;
  a.k_pre = static_cast<const __half*>(k_pre);
  a.v = static_cast<const __half*>(v);
  a.n_tokens = n_tokens;
  a.Hkv = c.Hkv;
  a.D = c.D;
  a.bits = c.bits;
  a.nuq = c.quant_mode == MKV_QUANT_NUQ;
  a.n_v = std::min(c.D, (int)ceil((double)c.outlier_frac * c.D));
  a.t_lo = qp.t_lo;
  a.t_hi = qp.t_hi;
  a.k_lo = qp.k_lo;
  a.k_scale = qp.k_scale;
  a.k_cb = qp.k_cb;
  a.v_cb = qp.v_cb;
  a.T_len = cache.T_len;
  a.k_codes = cache.k_codes;
  a.v_codes = cache.v_codes;
  a.v_params = reinterpret_cast<float2*>(cache.v_params);
  a.v_out = cache.v_out;
  a.k_out_off = cache.k_out_off;
  a.k_out = cache.k_out;
  a.k_out_cap = cache.k_out_cap;
  a.T_cap = cache.T_cap;
  // Runs of tokens on many warps from kBulkMinTokens tokens on (two launches: 11 us at 64 units, 8 us at
  // 2 units for 8 tokens); fewer (the decode step's one) take one CTA per unit, token after token (one
  // launch: 5.0 us for one token, 10.0 / 8.5 us for 4, 13.5 / 12.0 us for 6).  The runs read fp16 rows in up to 8-byte pieces and store
  // codes in 2-byte ones.
  if (n_tokens >= kBulkMinTokens && ((uintptr_t)k_pre | (uintptr_t)v) % 8 == 0 &&
      ((uintptr_t)a.k_codes | (uintptr_t)a.v_codes) % 2 == 0)
    return c.D == 128 ? launch_bulk_d<128>(a, c.B, st) : launch_bulk_d<64>(a, c.B, st);
  const int nwords = (c.D * c.bits / 8 + 3) / 4;
  const size_t smem = 2 * c.D + 4 * c.D + 2 * nwords * 4 + 16;
  if (!a.tickets) {
    a.trigger = 0;
    quantize_kernel<<<c.B * c.Hkv, c.D, smem, st>>>(a);
    const cudaError_t e = cudaPeekAtLastError();
    if (e != cudaSuccess) return e;
    advance_kernel<<<(unsigned)ceil_div(c.B, 256), 256, 0, st>>>(cache.T_len, c.B, (int32_t)n_tokens, cache.T_cap);
    return cudaPeekAtLastError();
  }
  // in a step, beside the previous layer's draining decode; two plain launches in a graph measured 1.5 %
  // faster than with the attribute on one of them only
  if (step) return launch_pdl(quantize_kernel, dim3(c.B * c.Hkv), dim3(c.D), smem, st, a);
  quantize_kernel<<<c.B * c.Hkv, c.D, smem, st>>>(a);
  return cudaPeekAtLastError();
}

cudaError_t launch_calibrate(const mkv_config& c, const void* k_cal, const void* v_cal, int64_t N,
                             int64_t row_stride, const mkv_quant_params& qp, const CalibWs& ws, cudaStream_t st) {
  const bool nuq = c.quant_mode == MKV_QUANT_NUQ;
  const int n_v = std::min(c.D, (int)ceil((double)c.outlier_frac * c.D));
  if (nuq) {
    const int64_t rows = (int64_t)c.Hkv * N;
    auto values = c.D == 128 ? calib_values_kernel<128> : calib_values_kernel<64>;
    values<<<(unsigned)ceil_div(rows, 8), 256, 0, st>>>(static_cast<const __half*>(v_cal), N, row_stride, rows, n_v,
                                                        ws.u);
    cudaError_t e = cudaPeekAtLastError();
    if (e != cudaSuccess) return e;
  }
  CalibArgs a{};
  a.k_cal = static_cast<const __half*>(k_cal);
  a.u = ws.u;
  a.N = N;
  a.row_stride = row_stride;
  a.D = c.D;
  a.bits = c.bits;
  a.nuq = nuq;
  a.nt = (int)ceil((double)c.outlier_frac / 2.0 * (double)N);
  a.all_out = 2 * a.nt >= N;
  a.t_lo = qp.t_lo;
  a.t_hi = qp.t_hi;
  a.k_lo = qp.k_lo;
  a.k_scale = qp.k_scale;
  a.k_cb = qp.k_cb;
  a.v_cb = qp.v_cb;
  // values per thread: the smallest power of two that holds N
  const int channels = c.Hkv * c.D;
  if (N <= kCalThr) return launch_calib_t<1>(a, channels, st);
  if (N <= 2 * kCalThr) return launch_calib_t<2>(a, channels, st);
  if (N <= 4 * kCalThr) return launch_calib_t<4>(a, channels, st);
  return launch_calib_t<8>(a, channels, st);
}

cudaError_t take_status_kvquant(uint32_t* flags, cudaStream_t st) {
  uint32_t zero = 0, v = 0;
  cudaError_t e = cudaMemcpyFromSymbolAsync(&v, g_status_kvquant, sizeof(v), 0, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(g_status_kvquant, &zero, sizeof(zero), 0, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  *flags |= v;
  return e;
}

}  // namespace mkv
