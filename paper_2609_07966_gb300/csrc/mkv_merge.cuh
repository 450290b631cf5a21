// Split-KV merge done by the last CTA of each (batch, kv-head) inside the decode
// kernels: every CTA writes its partial (m, l, o) and takes a ticket; the CTA
// that takes the last ticket merges all splits of the group's query heads,
//   out_h = sum_s 2^(m_s - M) o_s / sum_s 2^(m_s - M) l_s,  M = max_s m_s,
// writes the output, and resets the ticket counter to zero for the next call.
#pragma once

#include "mkv_common.cuh"

namespace mkv {

struct MergeArgs {
  const float* part_m;   // [B][Hq][n_split]
  const float* part_l;
  const float* part_o;   // [B][Hq][n_split][D]
  int* counters;         // [B][Hkv], zero between calls
  __half* out;           // [B][Hq][D]
  float* m_tot;          // H2O: [B][Hq] (or null)
  float* l_tot;
  int Hq, G, n_split;
};

// `scratch`: 16-byte aligned shared memory the caller no longer needs, `cap` floats of it.  `n_parts`:
// the partials of this group (slots 0 .. n_parts-1 of a.n_split; default all).
//
// Bound by the latency of two dependent reads of L2 (the partials' m and l, then o), so each is one round
// of independent loads: a thread takes four dims of a head and every SL-th split, with the o partials of
// its first splits requested before the weights are known.  FP16 step, batch 1, 32/8 heads, T = 4096 (33
// splits): 13.5 us a step, 17.7 with one thread per head summing l and four o loads in flight; H2O, batch 16,
// 3,277 slots: 48.7 and 49.9.
template <int D, int NT>
__device__ __forceinline__ void merge_if_last(const MergeArgs& a, int64_t bh, int b, int kvh, float* scratch,
                                              int cap, int n_parts = -1) {
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const int t = atomicAdd(&a.counters[bh], 1);
    s_last = (t == (n_parts > 0 ? n_parts : a.n_split) - 1);
    if (s_last) a.counters[bh] = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int ns = n_parts > 0 ? n_parts : a.n_split, stride = a.n_split, G = a.G;
  const int64_t hq0 = (int64_t)b * a.Hq + (int64_t)kvh * G;
  // (a workspace that is not 16-byte aligned takes the direct loop below)
  if (2 * G * ns + 2 * G + 4 * NT + 4 <= cap && (reinterpret_cast<uintptr_t>(a.part_o) & 15) == 0) {
    const int quads = G * (D / 4);               // (head, four dims)
    const int SL = quads < NT ? NT / quads : 1;  // slices of the splits per quad
    float* f = scratch;                          // [G][ns] m, then the weights 2^(m_s - M)
    float* fl = f + G * ns;                      // [G][ns] l
    float* tot = fl + G * ns;                    // [G] M, [G] L
    float4* part = reinterpret_cast<float4*>(scratch + ((2 * G * ns + 2 * G + 3) & ~3));   // [SL][quads]
    constexpr int U = 8;                         // o partials in flight per thread
    const int sl = threadIdx.x / quads, q0 = threadIdx.x - sl * quads;
    auto o_of = [&](int quad, int s) {
      const int row = quad / (D / 4), d = quad % (D / 4) * 4;
      return __ldcg(reinterpret_cast<const float4*>(a.part_o + ((hq0 + row) * stride + s) * D + d));
    };
    float4 x[U];
    if (sl < SL) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (sl + u * SL < ns) x[u] = o_of(q0, sl + u * SL);
    }
    for (int e = threadIdx.x; e < G * ns; e += NT) {
      f[e] = __ldcg(a.part_m + (hq0 + e / ns) * stride + e % ns);
      fl[e] = __ldcg(a.part_l + (hq0 + e / ns) * stride + e % ns);
    }
    __syncthreads();
    for (int row = threadIdx.x / 32; row < G; row += NT / 32) {   // a warp per head
      const int lane = threadIdx.x % 32;
      float M = -INFINITY;
      for (int s = lane; s < ns; s += 32) M = fmaxf(M, f[row * ns + s]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
      float L = 0.f;
      for (int s = lane; s < ns; s += 32) {
        const float ms = f[row * ns + s];
        const float w = (M == -INFINITY || ms == -INFINITY) ? 0.f : exp2f(ms - M);
        f[row * ns + s] = w;
        L += fl[row * ns + s] * w;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
      if (lane == 0) {
        tot[row] = M;
        tot[G + row] = L;
      }
    }
    __syncthreads();
    for (int quad = q0; quad < quads; quad += NT) {   // (SL > 1: one pass)
      const float* fw = f + quad / (D / 4) * ns;
      float4 O = make_float4(0.f, 0.f, 0.f, 0.f);
      if (sl < SL) {
        for (int s0 = sl; s0 < ns; s0 += U * SL) {
          if (s0 != sl || quad != q0) {
#pragma unroll
            for (int u = 0; u < U; ++u)
              if (s0 + u * SL < ns) x[u] = o_of(quad, s0 + u * SL);
          }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            if (s0 + u * SL < ns) {
              const float w = fw[s0 + u * SL];
              O.x += x[u].x * w;
              O.y += x[u].y * w;
              O.z += x[u].z * w;
              O.w += x[u].w * w;
            }
          }
        }
      }
      if (SL > 1) {
        if (sl < SL) part[sl * quads + quad] = O;
        __syncthreads();
        if (sl == 0) {
          for (int k = 1; k < SL; ++k) {
            const float4 y = part[k * quads + quad];
            O.x += y.x;
            O.y += y.y;
            O.z += y.z;
            O.w += y.w;
          }
        }
      }
      if (sl == 0) {
        const int row = quad / (D / 4), d = quad % (D / 4) * 4;
        const float L = tot[G + row];
        store_out4(a.out + (hq0 + row) * D + d, L > 0.f ? O.x / L : 0.f, L > 0.f ? O.y / L : 0.f,
                   L > 0.f ? O.z / L : 0.f, L > 0.f ? O.w / L : 0.f);
        if (a.m_tot != nullptr && d == 0) {
          a.m_tot[hq0 + row] = tot[row];
          a.l_tot[hq0 + row] = L;
        }
      }
    }
    return;
  }
  for (int e = threadIdx.x; e < G * D; e += NT) {      // many splits: direct loop
    const int row = e / D, d = e % D;
    const int64_t hq = hq0 + row;
    const float* pm = a.part_m + hq * stride;
    const float* pl = a.part_l + hq * stride;
    float M = -INFINITY;
    for (int s = 0; s < ns; ++s) M = fmaxf(M, __ldcg(pm + s));
    float L = 0.f, O = 0.f;
    if (M != -INFINITY) {
      for (int s = 0; s < ns; ++s) {
        const float ms = __ldcg(pm + s);
        if (ms == -INFINITY) continue;
        const float w = exp2f(ms - M);
        L += __ldcg(pl + s) * w;
        O += __ldcg(a.part_o + (hq * stride + s) * D + d) * w;
      }
    }
    a.out[hq * D + d] = __float2half_rn(L > 0.f ? O / L : 0.f);
    if (a.m_tot != nullptr && d == 0) {
      a.m_tot[hq] = M;
      a.l_tot[hq] = L;
    }
  }
}

// The same with one thread per head for the weights and one dim of a head per thread: fewer registers
// and less code, for the KVQuant kernel, whose loops ptxas schedules 3 to 10 % slower beside the other
// (8 x 8K, 4 bits, quantize + decode: 101.4 us with this one, 102.7 to 112 with 2 to 8 o partials in
// flight per thread); its merges are of at most 20 parts over 640 threads.
template <int D, int NT>
__device__ __forceinline__ void merge_if_last_lean(const MergeArgs& a, int64_t bh, int b, int kvh, float* scratch,
                                              int cap, int n_parts = -1) {
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const int t = atomicAdd(&a.counters[bh], 1);
    s_last = (t == (n_parts > 0 ? n_parts : a.n_split) - 1);
    if (s_last) a.counters[bh] = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int ns = n_parts > 0 ? n_parts : a.n_split, stride = a.n_split, G = a.G;
  const int64_t hq0 = (int64_t)b * a.Hq + (int64_t)kvh * G;
  if (2 * G * ns + 2 * G <= cap) {
    // weights f[row][s] = 2^(m_s - M) and totals, then independent loads of the o partials
    float* f = scratch;                 // [G][ns]
    float* tot = scratch + G * ns;      // [G] M, [G] L
    for (int e = threadIdx.x; e < G * ns; e += NT) f[e] = __ldcg(a.part_m + (hq0 + e / ns) * stride + e % ns);
    __syncthreads();
    if (threadIdx.x < G) {
      const int row = threadIdx.x;
      float M = -INFINITY;
      for (int s = 0; s < ns; ++s) M = fmaxf(M, f[row * ns + s]);
      float L = 0.f;
      for (int s = 0; s < ns; ++s) {
        const float ms = f[row * ns + s];
        const float w = (M == -INFINITY || ms == -INFINITY) ? 0.f : exp2f(ms - M);
        f[row * ns + s] = w;
        L += __ldcg(a.part_l + (hq0 + row) * stride + s) * w;
      }
      tot[row] = M;
      tot[G + row] = L;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < G * D; e += NT) {
      const int row = e / D, d = e % D;
      const float* po = a.part_o + ((hq0 + row) * stride) * D + d;
      const float* fw = f + row * ns;
      float O0 = 0.f, O1 = 0.f, O2 = 0.f, O3 = 0.f;
      int s = 0;
      for (; s + 4 <= ns; s += 4) {
        O0 += __ldcg(po + (int64_t)(s + 0) * D) * fw[s + 0];
        O1 += __ldcg(po + (int64_t)(s + 1) * D) * fw[s + 1];
        O2 += __ldcg(po + (int64_t)(s + 2) * D) * fw[s + 2];
        O3 += __ldcg(po + (int64_t)(s + 3) * D) * fw[s + 3];
      }
      for (; s < ns; ++s) O0 += __ldcg(po + (int64_t)s * D) * fw[s];
      const float O = (O0 + O1) + (O2 + O3);
      const float L = tot[G + row];
      a.out[(hq0 + row) * D + d] = __float2half_rn(L > 0.f ? O / L : 0.f);
      if (a.m_tot != nullptr && d == 0) {
        a.m_tot[hq0 + row] = tot[row];
        a.l_tot[hq0 + row] = L;
      }
    }
    return;
  }
  for (int e = threadIdx.x; e < G * D; e += NT) {      // many splits: direct loop
    const int row = e / D, d = e % D;
    const int64_t hq = hq0 + row;
    const float* pm = a.part_m + hq * stride;
    const float* pl = a.part_l + hq * stride;
    float M = -INFINITY;
    for (int s = 0; s < ns; ++s) M = fmaxf(M, __ldcg(pm + s));
    float L = 0.f, O = 0.f;
    if (M != -INFINITY) {
      for (int s = 0; s < ns; ++s) {
        const float ms = __ldcg(pm + s);
        if (ms == -INFINITY) continue;
        const float w = exp2f(ms - M);
        L += __ldcg(pl + s) * w;
        O += __ldcg(a.part_o + (hq * stride + s) * D + d) * w;
      }
    }
    a.out[hq * D + d] = __float2half_rn(L > 0.f ? O / L : 0.f);
    if (a.m_tot != nullptr && d == 0) {
      a.m_tot[hq] = M;
      a.l_tot[hq] = L;
    }
  }
}

}  // namespace mkv
