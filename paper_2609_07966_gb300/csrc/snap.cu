// RocketKV (Section 2.1, RocketKV paragraph).
// Stage 1, SnapKV prefill compression: the observation window's aggregated
// scores of the prefix (prefill.cu), max-pooled over |j' - j| <= pool/2,
// the keep - W best prefix positions under (pooled desc, position asc) plus
// the window, gathered in ascending position; per-page key min/max of the
// compact cache.
// Stage 2, page choice at decode: dims = the topq_dims largest sum_h |q_h,i|
// (dim asc on ties), page score = sum_h sum_{i in dims}
// max(q_h,i kmin_i, q_h,i kmax_i) over full pages before the newest token's,
// best topk_pages under (score desc, page asc), listed ascending.
#include <math.h>

#include "mkv_common.cuh"
#include "mkv_internal.h"
#include "mkv_select.cuh"

namespace mkv {

namespace {

constexpr int kSelThreads = 1024;
constexpr int kSelPages = 256;          // page selection: pages whose bounds are prefetched for every dim
constexpr int kSelRow = kSelPages + 8;  // halves per prefetched row (room for the 16-byte alignment offset)
constexpr int kSelChunks = kSelRow / 8; // 16-byte copies per prefetched row

// ---------------------------------------------------------------- keep list
// One cluster of kKeepCl CTAs per (batch, kv-head), each over an equal run of the prefix positions: its
// pooled scores stay in shared memory (in the workspace when they do not fit), and the k-th largest
// score key is found by histograms of 256 bins that every CTA sends to all CTAs (distributed shared
// memory).  The first histogram spans exactly the keys' range, so its bins are spread; later ones divide
// the bin that holds the k-th key, until that bin is kept whole or holds one key (exact ties: the lower
// positions).  Then each CTA lists its kept positions after those of the CTAs before it.
// 32736 positions, 32 units: one 1024-thread CTA per unit left 120 SMs idle and took 100 us of a call of
// 255 us; this one takes 23 us (latency: eight cluster barriers, and the shared-memory additions of the
// first histogram: one per run of equal neighbours, 30 us with one per position).
constexpr int kKeepCl = 8;
constexpr int kKeepThreads = 512;
constexpr int kKeepWords = 128;         // positions / 32 listed at a time (counts fit in 16 bits)
constexpr int kKeepSmem = 160 * 1024;   // bytes a CTA's scores and pooled scores may take in shared memory

struct KeepArgs {
  const float* score;    // [units][T]
  const float* score2;   // [units][T] second part of the sums, or null
  float* pooled_ws;      // [units][T] pooled scores that do not fit in shared memory
  int32_t* keep;         // [units][T]
  int64_t T;
  int W, pool, keep_n, in_smem;
};

__device__ __forceinline__ uint32_t keep_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
  return r;
}
__device__ __forceinline__ void keep_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void keep_send(uint32_t* p, uint32_t rank, uint32_t v) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
  asm volatile("st.shared::cluster.u32 [%0], %1;\n" ::"r"(a), "r"(v) : "memory");
}

__global__ void __cluster_dims__(kKeepCl, 1, 1) __launch_bounds__(kKeepThreads) snap_keep_kernel(const KeepArgs a) {
  extern __shared__ float pooled_sm[];
  __shared__ uint32_t hist[256];
  __shared__ uint32_t all[2][kKeepCl][256];   // the CTAs' histograms (two rounds: one is read, one arrives)
  __shared__ uint32_t edge[kKeepCl][2];       // the CTAs' smallest and largest key, later kept counts
  __shared__ uint32_t sum[256], s_bin, s_left, s_cnt;
  __shared__ uint2 word[kKeepWords];          // flags of 32 positions: kept for sure, equal to the threshold
  __shared__ uint32_t word_before[kKeepWords + 1];
  const int rank = (int)keep_rank();
  const int64_t bh = blockIdx.y;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t n = a.T - a.W;                // prefix positions compete
  const int64_t per = ceil_div_dev(n, kKeepCl), j0 = min(n, rank * per), m64 = min(n, j0 + per) - j0;
  const int m = (int)m64;                     // this CTA's positions j0 ..
  const float* s = a.score + bh * a.T;
  const float* s2 = a.score2 ? a.score2 + bh * a.T : nullptr;
  const bool in_smem = a.in_smem != 0;
  const int r = a.pool / 2;
  float* pooled = in_smem ? pooled_sm : a.pooled_ws + bh * a.T + j0;
  // max over |j' - j| <= r within the prefix, from the run's scores and r more on either side
  uint32_t mn = 0xffffffffu, mx = 0u;
  if (in_smem && m > 0) {
    float* raw = pooled_sm + per;
    const int64_t e0 = max((int64_t)0, j0 - r), e1 = min(n, j0 + m + r);
    const int cnt = (int)(e1 - e0);
    constexpr int U = 4;                      // loads in flight
    for (int i0 = tid; i0 < cnt; i0 += U * kKeepThreads) {
      float x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = min(i0 + u * kKeepThreads, cnt - 1);
        x[u] = s[e0 + i] + (s2 ? s2[e0 + i] : 0.f);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (i0 + u * kKeepThreads < cnt) raw[i0 + u * kKeepThreads] = x[u];
    }
    __syncthreads();
    const int d = (int)(j0 - e0);             // position j0 in raw
    for (int i = tid; i < m; i += kKeepThreads) {
      const int lo = max(0, d + i - r), hi = min(cnt - 1, d + i + r);
      float v = -INFINITY;
      for (int x = lo; x <= hi; ++x) v = fmaxf(v, raw[x]);
      pooled[i] = v;
      const uint32_t key = f32_key(v);
      mn = min(mn, key);
      mx = max(mx, key);
    }
  } else {
    for (int i = tid; i < m; i += kKeepThreads) {
      const int64_t j = j0 + i, lo = max((int64_t)0, j - r), hi = min(n - 1, j + r);
      float v = -INFINITY;
      for (int64_t x = lo; x <= hi; ++x) v = fmaxf(v, s[x] + (s2 ? s2[x] : 0.f));
      pooled[i] = v;
      const uint32_t key = f32_key(v);
      mn = min(mn, key);
      mx = max(mx, key);
    }
  }
  mn = __reduce_min_sync(0xffffffffu, mn);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (tid == 0) {
    s_bin = 0xffffffffu;
    s_left = 0u;
  }
  __syncthreads();
  if (lane == 0) {
    atomicMin(&s_bin, mn);
    atomicMax(&s_left, mx);
  }
  __syncthreads();
  keep_sync();                                // every CTA runs (and has read its scores: keep shares score2's room)
  if (tid < kKeepCl) {
    keep_send(&edge[rank][0], tid, s_bin);
    keep_send(&edge[rank][1], tid, s_left);
  }
  keep_sync();
  for (int c = 0; c < kKeepCl; ++c) {
    mn = min(mn, edge[c][0]);
    mx = max(mx, edge[c][1]);
  }
  const int k = a.keep_n - a.W;               // of the prefix; k < n
  uint32_t lo = mn, span = mx - mn;           // the k-th largest key lies in [lo, lo + span]
  uint32_t left = (uint32_t)k;                // its rank among the keys there
  bool ge = false;                            // keys >= lo are kept (else > lo, and the first `left` equal ones)
  if (k > 0) {
    int sh = max(0, 32 - __clz((int)(mx - mn)) - 8);
    for (int round = 0;; ++round) {
      __syncthreads();
      if (tid < 256) hist[tid] = 0u;
      __syncthreads();
      // neighbours share pooled scores: one addition per run of lanes with the same bin
      for (int i0 = warp * 32; i0 < m; i0 += kKeepThreads) {
        const int i = i0 + lane;
        const uint32_t key = i < m ? f32_key(pooled[i]) : 0u;
        const bool in = i < m && key >= lo && key - lo <= span;
        const uint32_t d = in ? (key - lo) >> sh : 0xffffffffu;    // span >> sh <= 255
        const uint32_t prev = __shfl_up_sync(0xffffffffu, d, 1);
        const bool head = lane == 0 || d != prev;
        const uint32_t after = __ballot_sync(0xffffffffu, head) & (0xfffffffeu << lane);   // heads past this lane
        if (head && in) atomicAdd(&hist[d], (uint32_t)((after ? __ffs((int)after) - 1 : 32) - lane));
      }
      __syncthreads();
      for (int e = tid; e < 256 * kKeepCl; e += kKeepThreads)
        keep_send(&all[round & 1][rank][e & 255], e >> 8, hist[e & 255]);
      keep_sync();
      if (tid < 256) {
        uint32_t c = 0;
#pragma unroll
        for (int x = 0; x < kKeepCl; ++x) c += all[round & 1][x][tid];
        sum[tid] = c;
      }
      __syncthreads();
      if (warp == 0) {                        // lane l owns bins 255 - 8 l .. 248 - 8 l (descending)
        uint32_t cnt = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) cnt += sum[255 - 8 * lane - j];
        uint32_t incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += y;
        }
        const uint32_t excl = incl - cnt;
        if (excl < left && incl >= left) {    // exactly one lane
          uint32_t rem = left - excl;
          int bin = 255 - 8 * lane;
          for (int j = 0; j < 7 && sum[bin] < rem; ++j, --bin) rem -= sum[bin];
          s_bin = (uint32_t)bin;
          s_left = rem;
          s_cnt = sum[bin];
        }
      }
      __syncthreads();
      lo += s_bin << sh;
      left = s_left;
      if (s_cnt == left) {                    // the whole bin is kept
        ge = true;
        left = 0;
        break;
      }
      if (sh == 0) break;
      span = (1u << sh) - 1u;
      sh = max(0, sh - 8);
    }
  }
  // kept positions of this CTA: above (or at) the threshold for sure, and the equal ones
  auto flags = [&](int i, bool& above, bool& tie) {
    const uint32_t key = i < m ? f32_key(pooled[i]) : 0u;
    above = i < m && k > 0 && (ge ? key >= lo : key > lo);
    tie = i < m && k > 0 && !ge && key == lo;
  };
  uint32_t gt = 0, eq = 0;
  for (int i = tid; i < m; i += kKeepThreads) {
    bool above, tie;
    flags(i, above, tie);
    gt += above ? 1u : 0u;
    eq += tie ? 1u : 0u;
  }
  gt = __reduce_add_sync(0xffffffffu, gt);
  eq = __reduce_add_sync(0xffffffffu, eq);
  __syncthreads();                            // every thread has read the last round's words
  if (tid == 0) s_left = s_cnt = 0u;
  __syncthreads();
  if (lane == 0) {
    atomicAdd(&s_left, gt);
    atomicAdd(&s_cnt, eq);
  }
  __syncthreads();
  if (tid < kKeepCl) {
    keep_send(&edge[rank][0], tid, s_left);
    keep_send(&edge[rank][1], tid, s_cnt);
  }
  keep_sync();
  uint32_t base_g = 0, base_e = 0;
  for (int c = 0; c < rank; ++c) {
    base_g += edge[c][0];
    base_e += edge[c][1];
  }
  int32_t* out = a.keep + bh * a.T;
  for (int c0 = 0; c0 < m; c0 += 32 * kKeepWords) {   // kKeepWords words of 32 positions at a time
    for (int w = warp; w < kKeepWords; w += kKeepThreads / 32) {
      bool above, tie;
      flags(c0 + 32 * w + lane, above, tie);
      const uint32_t bg = __ballot_sync(0xffffffffu, above), be = __ballot_sync(0xffffffffu, tie);
      if (lane == 0) word[w] = make_uint2(bg, be);
    }
    __syncthreads();
    if (warp == 0) {                          // kept and equal counts before each word
      uint32_t run = 0;
#pragma unroll
      for (int w0 = 0; w0 < kKeepWords; w0 += 32) {
        const uint2 f = word[w0 + lane];
        const uint32_t mine = __popc(f.x) | (__popc(f.y) << 16);
        uint32_t incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += y;
        }
        word_before[w0 + lane] = run + incl - mine;
        run += __shfl_sync(0xffffffffu, incl, 31);
      }
      if (lane == 0) word_before[kKeepWords] = run;
    }
    __syncthreads();
    for (int w = warp; w < kKeepWords; w += kKeepThreads / 32) {
      const uint2 f = word[w];
      const uint32_t before = word_before[w], lt = (1u << lane) - 1u;
      const uint32_t g = base_g + (before & 0xffffu) + __popc(f.x & lt), q = base_e + (before >> 16) + __popc(f.y & lt);
      if (((f.x >> lane) & 1u) || (((f.y >> lane) & 1u) && q < left))
        out[g + min(q, left)] = (int32_t)(j0 + c0 + 32 * w + lane);
    }
    const uint32_t x = word_before[kKeepWords];
    base_g += x & 0xffffu;
    base_e += x >> 16;
    __syncthreads();
  }
  // the window, kept whole
  if (rank == kKeepCl - 1)
    for (int i = tid; i < a.W; i += kKeepThreads) out[k + i] = (int32_t)(n + i);
}

// Gather kept rows (keep list, or the identity when keep >= T) into slots 0..n-1, eight pages of 16 slots
// per CTA, and the per-dim key min / max of its full pages.  Thread (row, column): 16 bytes of a row,
// four pages in flight.  4096 of 32768 rows, 32 units: 134 MB in 22 us (6.1 TB/s); a copy and a separate
// pass over the copied keys took about 48 us.
constexpr int kGatherPages = 8;
template <int D>
__global__ void __launch_bounds__(kPage * D / 8) snap_gather_kernel(
    const __half* __restrict__ full_k, const __half* __restrict__ full_v, const int32_t* __restrict__ keep,
    int identity, int64_t T, int64_t n, int Hkv, int64_t T_cap, __half* k, __half* v, int32_t* kept_pos,
    int32_t* T_len, __half* kmin, __half* kmax) {
  constexpr int NC = D / 8, NT = kPage * NC;
  __shared__ uint4 rows[4][kPage][NC + 1];    // four pages' keys
  __shared__ __half mm[2][D][kGatherPages];
  const int64_t bh = blockIdx.y;
  const int col = threadIdx.x % NC, row = threadIdx.x / NC;
  const int64_t p0 = (int64_t)blockIdx.x * kGatherPages, np = n / kPage, npc = T_cap / kPage;
  constexpr int U = 4;                        // pages in flight
#pragma unroll 1
  for (int u0 = 0; u0 < kGatherPages; u0 += U) {
    int64_t p[U];
    uint4 x[U], y[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t sl = (p0 + u0 + u) * kPage + row;
      p[u] = sl >= n ? -1 : identity ? sl : keep[bh * T + sl];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      x[u] = y[u] = make_uint4(0u, 0u, 0u, 0u);
      if (p[u] >= 0) {
        x[u] = __ldcs(reinterpret_cast<const uint4*>(full_k + (bh * T + p[u]) * D) + col);
        y[u] = __ldcs(reinterpret_cast<const uint4*>(full_v + (bh * T + p[u]) * D) + col);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t sl = (p0 + u0 + u) * kPage + row;
      if (p[u] >= 0) {
        reinterpret_cast<uint4*>(k + (bh * T_cap + sl) * D)[col] = x[u];
        reinterpret_cast<uint4*>(v + (bh * T_cap + sl) * D)[col] = y[u];
        if (col == 0 && kept_pos) kept_pos[bh * n + sl] = (int32_t)p[u];
      }
      rows[u][row][col] = x[u];
    }
    __syncthreads();
    // thread (dim, page) takes the page's 16 values of its dim in row order
    for (int e = threadIdx.x; e < U * D; e += NT) {
      const int u = e / D, dim = e % D;
      const __half* c = reinterpret_cast<const __half*>(&rows[u][0][0]) + dim;
      __half lo = c[0], hi = c[0];
#pragma unroll
      for (int j = 1; j < kPage; ++j) {
        const __half z = c[j * (NC + 1) * 8];
        lo = __hlt(z, lo) ? z : lo;
        hi = __hgt(z, hi) ? z : hi;
      }
      mm[0][dim][u0 + u] = lo;
      mm[1][dim][u0 + u] = hi;
    }
    __syncthreads();
  }
  const int have = (int)max((int64_t)0, min((int64_t)kGatherPages, np - p0));
  for (int e = threadIdx.x; e < 2 * D * kGatherPages; e += NT) {
    const int u = e % kGatherPages, d = e / kGatherPages % D, w = e / (kGatherPages * D);
    if (u < have) (w ? kmax : kmin)[(bh * D + d) * npc + p0 + u] = mm[w][d][u];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0 && bh % Hkv == 0) T_len[bh / Hkv] = (int32_t)n;
}

// One CTA per (batch, kv-head): dims, page scores, top-k pages.
// Page selection (RocketKV stage 2).  With max(q kmin, q kmax) = q kmax for q >= 0 and q kmin
// otherwise (kmin <= kmax), a page's score over the selected dims t is
//   sum_t (kmax_t P_t + kmin_t N_t),  P_t = sum_h max(q_h,t, 0),  N_t = sum_h min(q_h,t, 0).
// Up to kSelPages candidate pages (the common case) the bounds of every dim are prefetched into
// shared memory while the dims are being chosen; larger caches stage the chosen dims' bounds
// 256 pages at a time.
__global__ void __launch_bounds__(kSelThreads) rocket_select_kernel(const __half* __restrict__ q, const __half* __restrict__ kmin,
                                                                    const __half* __restrict__ kmax,
                                                                    const int32_t* __restrict__ T_len, int Hkv, int G, int D,
                                                                    int64_t T_cap, int kp, int rd, int32_t* __restrict__ out) {
  extern __shared__ __align__(16) float sm[];
  const int64_t npc = T_cap / kPage;
  float* qs = sm;                       // [G][D]
  float* ssc = qs + G * D;              // [npc] page scores
  float* part = ssc + ((npc + 3) & ~3ll);                     // [4][kSelPages] partial scores
  __half* bmn = reinterpret_cast<__half*>(part + 4 * kSelPages);   // fast path: [D][kSelRow]
  __half* bmx = bmn + D * kSelRow;
  __shared__ int hist[256];
  __shared__ int warp_sums[32];
  __shared__ int dims[128];
  __shared__ __align__(16) float a_dim[128];
  __shared__ float pn[2][128];          // P_t, N_t of the selected dims
  const int64_t bh = blockIdx.x;
  const int b = (int)(bh / Hkv), kvh = (int)(bh % Hkv);
  const int n = (int)min((int64_t)T_len[b], T_cap);
  const int ns = n > 0 ? (n - 1) / kPage : 0;
  const bool fast = ns <= kSelPages;
  if (fast && ns > 0) {
    // every dim's bounds of pages [0, ns): 16-byte copies from the row start rounded down to
    // 16 bytes (the first copy may begin in the previous row), the last one cut at the row end
    for (int e = threadIdx.x; e < 2 * D * kSelChunks; e += blockDim.x) {
      const int which = e / (D * kSelChunks), rem = e % (D * kSelChunks);
      const int dim = rem / kSelChunks, ch = rem % kSelChunks;
      const int64_t start = (bh * D + dim) * npc;           // first half of the row
      const int64_t h0 = (start & ~7ll) + ch * 8;
      const int64_t end = start + ns;
      if (h0 < end) {
        const int bytes = (int)min((int64_t)16, (end - h0) * 2);
        cp_async16((which ? bmx : bmn) + dim * kSelRow + ch * 8, (which ? kmax : kmin) + h0, bytes);
      }
    }
    cp_async_commit();
  }
  for (int e = threadIdx.x; e < G * D; e += blockDim.x) qs[e] = __half2float(q[((int64_t)b * Hkv * G + (int64_t)kvh * G) * D + e]);
  __syncthreads();
  if (threadIdx.x < D) {
    float a = 0.f;
    for (int h = 0; h < G; ++h) a += fabsf(qs[h * D + threadIdx.x]);
    a_dim[threadIdx.x] = a;
  }
  __syncthreads();
  if (threadIdx.x < D) {
    // rank under (sum |q| desc, dim asc): four dims per shared-memory read, unrolled so the
    // reads overlap; the sums' bits, as in rocket_fused_kernel: every rank is taken once, with NaNs too
    const int i = threadIdx.x;
    const int ai = __float_as_int(a_dim[i]);
    int rank = 0;
#pragma unroll 4
    for (int j = 0; j < D; j += 4) {
      const int4 v = *reinterpret_cast<const int4*>(a_dim + j);
      rank += (v.x > ai || (v.x == ai && j < i)) + (v.y > ai || (v.y == ai && j + 1 < i)) +
              (v.z > ai || (v.z == ai && j + 2 < i)) + (v.w > ai || (v.w == ai && j + 3 < i));
    }
    if (rank < rd) dims[rank] = i;
  }
  __syncthreads();
  if (threadIdx.x < rd) {
    const int d = dims[threadIdx.x];
    float P = 0.f, N = 0.f;
    for (int h = 0; h < G; ++h) {
      const float v = qs[h * D + d];
      P += fmaxf(v, 0.f);
      N += fminf(v, 0.f);
    }
    pn[0][threadIdx.x] = P;
    pn[1][threadIdx.x] = N;
  }
  if (fast) {
    cp_async_wait<0>();
    __syncthreads();
    // thread (page p, slice sl) sums the dims t = sl, sl + 4, ...; the four slices are added after
    const int p = threadIdx.x % kSelPages, sl = threadIdx.x / kSelPages;
    if (sl < 4) {
      float acc = 0.f;
      if (p < ns) {
        for (int t = sl; t < rd; t += 4) {
          const int d = dims[t];
          const int off = (int)(((bh * D + d) * npc) & 7);
          const int i = d * kSelRow + off + p;
          acc += __half2float(bmx[i]) * pn[0][t] + __half2float(bmn[i]) * pn[1][t];
        }
      }
      part[sl * kSelPages + p] = acc;
    }
    __syncthreads();
    if (threadIdx.x < ns)
      ssc[threadIdx.x] = (part[threadIdx.x] + part[kSelPages + threadIdx.x]) +
                         (part[2 * kSelPages + threadIdx.x] + part[3 * kSelPages + threadIdx.x]);
    __syncthreads();
  } else {
    __syncthreads();
    // the selected dims' min/max rows staged 256 pages at a time with coalesced loads (dim-major
    // layout), then each thread scores one page from shared memory
    __half* smn = bmn;                                          // [rd][256]
    __half* smx = smn + rd * 256;
    for (int p0 = 0; p0 < ns; p0 += 256) {
      const int np = min(256, ns - p0);
      for (int e = threadIdx.x; e < rd * 256; e += blockDim.x) {
        const int t = e / 256, pp = e % 256;
        if (pp < np) {
          const int64_t src = (bh * D + dims[t]) * npc + p0 + pp;
          smn[e] = kmin[src];
          smx[e] = kmax[src];
        }
      }
      __syncthreads();
      if (threadIdx.x < np) {
        float sc = 0.f;
        for (int t = 0; t < rd; ++t)
          sc += __half2float(smx[t * 256 + threadIdx.x]) * pn[0][t] + __half2float(smn[t * 256 + threadIdx.x]) * pn[1][t];
        ssc[p0 + threadIdx.x] = sc;
      }
      __syncthreads();
    }
  }
  const int k = min(kp, ns);
  int base = 0;
  if (ns <= (int)blockDim.x) {
    // few pages: each thread ranks its page by counting the pages ahead of it under
    // (score desc, page asc).  The scores' order-preserving keys are counted: with a NaN among the scores (infinite
    // keys) a comparison of values would give several pages one rank and list more than k.
    const int i = threadIdx.x;
    int flag = 0;
    uint32_t* keys = reinterpret_cast<uint32_t*>(ssc);
    if (i < ((ns + 3) & ~3)) keys[i] = i < ns ? f32_key(ssc[i]) : 0u;   // (its own score; pads never rank ahead)
    __syncthreads();
    if (i < ns && k > 0) {
      const uint32_t own = keys[i];
      int rank = 0;
#pragma unroll 4
      for (int j = 0; j < ns; j += 4) {
        const uint4 v = *reinterpret_cast<const uint4*>(keys + j);
        rank += (v.x > own || (v.x == own && j < i)) + (v.y > own || (v.y == own && j + 1 < i)) +
                (v.z > own || (v.z == own && j + 2 < i)) + (v.w > own || (v.w == own && j + 3 < i));
      }
      flag = rank < k;
    }
    int total;
    const int before = block_exclusive_scan(flag, warp_sums, &total);
    if (flag) out[bh * kp + before] = i;
    base = total;
  } else {
    uint64_t thr = ~0ull;
    if (k > 0) thr = block_kth_largest_score(ns, k, [&](int i) { return ssc[i]; }, hist);
    for (int i0 = 0; i0 < ns; i0 += blockDim.x) {
      const int i = i0 + threadIdx.x;
      const int flag = (i < ns && k > 0 && rank_key(ssc[i], (uint32_t)i) >= thr) ? 1 : 0;
      int total;
      const int before = block_exclusive_scan(flag, warp_sums, &total);
      if (flag) out[bh * kp + base + before] = i;
      base += total;
    }
  }
  for (int i = base + threadIdx.x; i < kp; i += blockDim.x) out[bh * kp + i] = -1;
}

}  // namespace

cudaError_t launch_snap_keep(const mkv_config& c, const void* full_k, const void* full_v, int64_t T,
                             const mkv_cache& cache, int32_t* kept_pos, const PrefillWs& ws, cudaStream_t st) {
  const int units = c.B * c.Hkv;
  const bool identity = T <= c.snap_keep;
  const int64_t n = identity ? T : c.snap_keep;
  if (!identity) {
    KeepArgs a{};
    a.score = ws.score;
    a.score2 = prefill_second_sums(c, c.snap_window, ws);
    a.pooled_ws = reinterpret_cast<float*>(ws.row_st);
    a.keep = ws.keep;
    a.T = T;
    a.W = c.snap_window;
    a.pool = c.snap_pool;
    a.keep_n = c.snap_keep;
    const int64_t per = ceil_div(T - c.snap_window, kKeepCl);
    const int64_t bytes = (2 * per + 2 * (c.snap_pool / 2)) * (int64_t)sizeof(float);
    a.in_smem = bytes <= kKeepSmem;
    const int smem = a.in_smem ? (int)bytes : 0;
    cudaError_t ea = allow_all_smem<snap_keep_kernel>();
    if (ea != cudaSuccess) return ea;
    snap_keep_kernel<<<dim3(kKeepCl, units), kKeepThreads, smem, st>>>(a);
    cudaError_t e = cudaPeekAtLastError();
    if (e != cudaSuccess) return e;
  }
  const dim3 grid((unsigned)ceil_div(n, kPage * kGatherPages), units);
  auto gather = c.D == 128 ? snap_gather_kernel<128> : snap_gather_kernel<64>;
  gather<<<grid, kPage * c.D / 8, 0, st>>>(
      static_cast<const __half*>(full_k), static_cast<const __half*>(full_v), ws.keep, identity ? 1 : 0, T, n, c.Hkv,
      cache.T_cap, static_cast<__half*>(cache.k), static_cast<__half*>(cache.v), kept_pos, cache.T_len,
      static_cast<__half*>(cache.kmin), static_cast<__half*>(cache.kmax));
  return cudaPeekAtLastError();
}

cudaError_t launch_rocket_select(const mkv_config& c, const void* q, const mkv_cache& cache, int32_t* page_idx,
                                 cudaStream_t st) {
  const int G = c.Hq / c.Hkv;
  const int64_t npc = cache.T_cap / kPage;
  const size_t smem = ((size_t)G * c.D + ((npc + 3) & ~3ll) + 4 * kSelPages) * sizeof(float) +
                      std::max<size_t>(2 * (size_t)c.D * kSelRow * 2, 2 * (size_t)c.topq_dims * 256 * 2);
  cudaError_t e = allow_all_smem<rocket_select_kernel>();
  if (e != cudaSuccess) return e;
  rocket_select_kernel<<<c.B * c.Hkv, kSelThreads, smem, st>>>(
      static_cast<const __half*>(q), static_cast<const __half*>(cache.kmin), static_cast<const __half*>(cache.kmax),
      cache.T_len, c.Hkv, G, c.D, cache.T_cap, c.topk_pages, c.topq_dims, page_idx);
  return cudaPeekAtLastError();
}

}  // namespace mkv
