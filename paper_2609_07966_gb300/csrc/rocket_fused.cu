// Fused RocketKV decode (Section 2.1, RocketKV paragraph, stage 2): the page choice and the
// sparse exact attention of one decode step in a single launch.
//
// One thread-block cluster of CL = 8, 4, 2 or 1 CTAs per (batch, kv-head):
//  1. each CTA chooses the top-r_d dims of sum_h |q_h,i| (redundantly, it is 128 keys) and
//     scores its 1/CL share of the candidate pages (the full pages before the newest token's
//     page): score_p = sum_t (kmax_t,p P_t + kmin_t,p N_t) over the chosen dims t, where
//     P_t / N_t are the group's positive / negative query parts (max(q kmin, q kmax) is q kmax
//     for q >= 0, q kmin otherwise, since kmin <= kmax).  Only the chosen dims' bounds are
//     read, by cp.async once the dims are known; meanwhile one warp attends to the newest page;
//  2. every score is stored into every CTA of the cluster (st.async to distributed shared memory,
//     counted by the receiver's mbarrier: a CTA waits for the scores only, not for the cluster);
//  3. every CTA finds the k-th best score for itself and lists the kept pages in ascending order;
//     the newest token's partial page is always attended;
//  4. the attended pages are dealt round-robin over the cluster's 8 CL warps; a warp loads its page's
//     16 K and V rows straight into tensor-core operands (16 tokens = one mma slab) and has the next
//     two pages brought into L2 while it works on this one;
//  5. the CTA merges its warps' partials (m, l, o), sends its partial to CTA 0 (st.async), which
//     merges the CL partials and writes the output.
// No workspace, no global round trip of scores, page ids or partials.
//
// Bound by the latency of the chain (launch, dims, bounds, scores, choice: about 8 us at one page) and,
// with many units and pages, by HBM.  32/8 heads, D = 128: 64 of 256 pages, batch 4: 13.5 us (16.9 with
// the pages' rows staged through shared memory and three cluster barriers); 256 of 1021 pages, batch 16:
// 60 us, 4.5 TB/s (308 us).  Requesting the next K rows before the PV product instead (more registers
// than there are) took 65 us.
//
// With k_new / v_new (mkv_rocket_step) the launch also appends the step's token first, as
// mkv_append_kv does: every CTA takes the length as T_len + 1, the warp that stages the newest
// page takes the new row from the input and writes it into the cache, completes the page's
// per-dim min/max when the row fills it, and the last CTA of the batch entry to finish stores
// the new length.  During the launch the top 8 bits of T_len[b] count the finished CTAs of
// batch entry b (every reader masks them off); the last one writes the clean length.
#include <math.h>

#include <algorithm>

#include "mkv_common.cuh"
#include "mkv_internal.h"
#include "mkv_tc.cuh"

namespace mkv {

__device__ uint32_t g_status_rocket;   // MKV_FLAG_* bits raised by this unit

namespace {

constexpr int kRfWarps = 8;
constexpr int kRfThreads = kRfWarps * 32;
// Up to this many candidate pages are ranked by counting the pages ahead of each (one pass over them), more by
// bits of the k-th key, a barrier a bit or, beyond 256 pages, two.  Counting against bits: 8/2 heads, D = 64,
// batch 1, us a launch: 18 pages 8.0 -> 7.1, 62 pages 8.7 -> 7.5, 124 pages 9.4 -> 8.5, 156
// pages 9.3 both, 256 pages (64 kept) 9.2 -> 10.1.  Two bits against one:
// 361 pages 12.0 -> 10.7, 999 pages (256 kept) 13.5 -> 12.1; up to 256 pages, where the barrier itself counts
// a bit, two took 0.1 to 0.4 us longer.
constexpr int kRankPages = 128;

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
  return r;
}
// the address of a shared variable of this CTA in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_addr(const void* p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
  return r;
}
// Stores into a CTA of the cluster that count as received bytes of that CTA's mbarrier
__device__ __forceinline__ void st_async(uint32_t dst, float v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];\n" ::"r"(dst),
               "r"(__float_as_uint(v)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void st_async4(uint32_t dst, float4 v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];\n" ::"r"(
                   dst),
               "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)),
               "r"(__float_as_uint(v.w)), "r"(bar)
               : "memory");
}
// Wait for the bytes of phase 0, at most a second: then MKV_FLAG_WAIT_TIMEOUT, and the CTA goes on with
// what it has (page indexes stay in range whatever the scores are)
__device__ __forceinline__ void wait_received(uint64_t* bar) {
  uint64_t t0 = 0;
  for (int spin = 0;; ++spin) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(smem_addr(bar))
        : "memory");
    if (ok) return;
    if (spin == 0) t0 = globaltimer_ns();
    else if (globaltimer_ns() - t0 > 1000000000ull) break;
  }
  atomicOr(&g_status_rocket, MKV_FLAG_WAIT_TIMEOUT);
}

// an 8x8 b16 matrix held as rows becomes the column-major operand of the next product
__device__ __forceinline__ uint32_t movm_trans(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(y) : "r"(x));
  return y;
}

// 16 bytes of a cache row, or zeros; volatile: issued where written, so that a page's rows are in flight
// together
__device__ __forceinline__ uint4 ld_row16(const __half* p, bool ok) {
  uint4 x;
  asm volatile(
      "{ .reg .pred p;\n setp.ne.b32 p, %5, 0;\n mov.b32 %0, 0;\n mov.b32 %1, 0;\n mov.b32 %2, 0;\n mov.b32 %3, 0;\n"
      " @p ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];\n}"
      : "=&r"(x.x), "=&r"(x.y), "=&r"(x.z), "=&r"(x.w)
      : "l"(p), "r"((int)ok));
  return x;
}

__host__ __device__ constexpr int a16(int x) { return (x + 15) & ~15; }

// Shared-memory layout (bytes); every region 16-byte aligned.  `rs` = halves per bounds row.
struct RfLayout {
  int qs, sc, part, flags, sel, bounds, cpart, wpart, bytes;
  __host__ __device__ RfLayout(int D, int G, int64_t npc, int kp, int rd, int rs, int cl) {
    qs = 0;                                              // float [G][D]
    sc = a16(qs + G * D * 4);                            // float [npc] page scores
    part = a16(sc + (int)npc * 4);                       // float [warps][sp] partial scores
    flags = a16(part + kRfWarps * (int)((npc + cl - 1) / cl) * 4);   // u32 [pages / 32][2] kept, equal to the k-th
    sel = a16(flags + (int)((npc + 31) / 32) * 8);       // int [min(kp, npc)] chosen pages
    bounds = a16(sel + (int)(kp < npc ? kp : npc) * 4);  // half [2][rd][rs]; later CTA 0's
    cpart = bounds;                                      // float [cl][G][D + 2] partials of the cluster
    const int bb = 2 * rd * rs * 2, cb = cl * G * (D + 2) * 4;
    wpart = a16(bounds + (bb > cb ? bb : cb));           // float [warps][G][D + 2]
    bytes = wpart + kRfWarps * G * (D + 2) * 4;
  }
};

struct RfArgs {
  const __half* q;          // [B][Hq][D]
  __half* k;                // [B][Hkv][T_cap][D]
  __half* v;
  __half* kmin;             // [B][Hkv][D][npc]
  __half* kmax;
  int32_t* T_len;           // low 24 bits: length; top 8: finished CTAs during an appending launch
  const __half* k_new;      // [B][Hkv][D], or null: no append
  const __half* v_new;
  int64_t T_cap, npc;
  int Hq, Hkv, G, kp, rd, rs;
  float scale_log2;
  int32_t* page_idx;        // optional [B][Hkv][kp]
  __half* out;              // [B][Hq][D]
};

// CL: CTAs of a (batch, kv-head)'s cluster
template <int D, int CL>
__global__ void __launch_bounds__(kRfThreads, 2) rocket_fused_kernel(const RfArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int G = a.G;
  const RfLayout L(D, G, a.npc, a.kp, a.rd, a.rs, CL);
  float* qs = reinterpret_cast<float*>(smem + L.qs);
  float* sc = reinterpret_cast<float*>(smem + L.sc);
  float* part = reinterpret_cast<float*>(smem + L.part);
  uint32_t* flags = reinterpret_cast<uint32_t*>(smem + L.flags);
  int* sel = reinterpret_cast<int*>(smem + L.sel);
  __half* bmn = reinterpret_cast<__half*>(smem + L.bounds);
  __half* bmx = bmn + a.rd * a.rs;
  __shared__ int dims[128];
  __shared__ __align__(16) float a_dim[128];
  __shared__ float pn[2][128];
  __shared__ int boff[128];             // first page of a chosen dim's staged row
  __shared__ uint32_t red[kRfWarps * 2];
  __shared__ uint64_t bar[2];
  __shared__ __align__(16) int cnt[2][kRfWarps];
  static_assert(kRfWarps == 8, "two 16-byte reads of the warps' counts");
  __shared__ __align__(16) uint32_t qh2[8][64 + 4];   // query as fp16 pairs, rows padded

  const int rank = CL > 1 ? (int)cluster_rank() : 0;
  if constexpr (CL > 1) {
    // no CTA writes into another before that one runs and has its mbarriers: bar[0] for the pages'
    // scores, bar[1] (CTA 0) for the partials
    if (threadIdx.x == 0) {
      tc_mbar_init(&bar[0], 1);
      tc_mbar_init(&bar[1], 1);
      tc_fence_mbar_init();
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
  }
  const int64_t bh = blockIdx.y;
  const int b = (int)(bh / a.Hkv), kvh = (int)(bh % a.Hkv);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, r = lane & 3;
  // this CTA's share of the pages, by the capacity
  const int sp = (int)((a.npc + CL - 1) / CL);          // pages per CTA
  const int p0 = min((int)a.npc, rank * sp);

  // the group's query (fp16) and the cache length
  constexpr int kQW = (8 * D / 2 + kRfThreads - 1) / kRfThreads;   // query words per thread (G <= 8)
  const uint32_t* qg = reinterpret_cast<const uint32_t*>(a.q + ((int64_t)b * a.Hq + (int64_t)kvh * G) * D);
  uint32_t qw[kQW];
#pragma unroll
  for (int k = 0; k < kQW; ++k) {
    const int e = tid + k * kRfThreads;
    qw[k] = e < G * (D / 2) ? __ldg(qg + e) : 0u;
  }
  const bool append = a.k_new != nullptr;
  const int n_old = (int)min((int64_t)(a.T_len[b] & 0xffffff), a.T_cap);
  const bool room = append && (int64_t)n_old + 1 <= a.T_cap;
  const int n = room ? n_old + 1 : n_old;              // the step's token included
  // the newest token's page, always attended, goes to one warp, which attends to it before the choice
  const int ns = n > 0 ? (n - 1) / kPage : 0;          // candidate (full) pages; page ns is the newest
  const bool tail_warp = rank == CL - 1 && warp == kRfWarps - 1 && n > 0;
  const int tail_valid = n - ns * kPage;               // 1 .. 16 rows
  if (tail_warp && room) {                             // the new row into the cache
    for (int e = lane; e < 2 * (D / 8); e += 32) {
      const int kv = e / (D / 8), ch = e % (D / 8);
      const uint4 x = __ldg(reinterpret_cast<const uint4*>((kv ? a.v_new : a.k_new) + bh * D) + ch);
      reinterpret_cast<uint4*>((kv ? a.v : a.k) + (bh * a.T_cap + (int64_t)n_old) * D)[ch] = x;
    }
  }
  const int np = max(0, min(ns, p0 + sp) - p0);        // of the candidate pages, this CTA's
#pragma unroll
  for (int k = 0; k < kQW; ++k) {
    const int e = tid + k * kRfThreads;
    if (e < G * (D / 2)) {
      const int row = e / (D / 2), w = e % (D / 2);
      qh2[row][w] = qw[k];
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&qw[k]));
      qs[row * D + 2 * w] = f.x;
      qs[row * D + 2 * w + 1] = f.y;
    }
  }
  __syncthreads();
  if (tid < D) {
    float s = 0.f;
    for (int h = 0; h < G; ++h) s += fabsf(qs[h * D + tid]);
    a_dim[tid] = s;
  }
  __syncthreads();
  {
    // rank under (sum |q| desc, dim asc): two threads per dim, half the dims each, four at a time; dims
    // before i count when >= a_i, that is > a_i - 1, dims after it when > a_i.  The sums' bits are ranked (in the order
    // of the values, since none is negative; a NaN comes first): every rank is taken once whatever the query holds.
    const int i = tid >> 1, half = tid & 1;
    int rk = 0;
    if (i < D) {
      const int ai = __float_as_int(a_dim[i]), below = ai - 1;
#pragma unroll 8
      for (int j = half * (D / 2); j < (half + 1) * (D / 2); j += 4) {
        const int4 v = *reinterpret_cast<const int4*>(a_dim + j);
        rk += (v.x > (j < i ? below : ai)) + (v.y > (j + 1 < i ? below : ai)) + (v.z > (j + 2 < i ? below : ai)) +
              (v.w > (j + 3 < i ? below : ai));
      }
    }
    rk += __shfl_xor_sync(0xffffffffu, rk, 1);
    if (i < D && half == 0 && rk < a.rd) dims[rk] = i;
  }
  __syncthreads();
  // ---- 1. the chosen dims' bounds of this CTA's candidate pages, row t for the t-th dim (16-byte copies
  // from the row start rounded down to 16 bytes, the last one cut at the end of the pages).  With no candidate
  // page nothing is copied: CTA 0's bounds are also where it receives the cluster's partials, and only its
  // scores tell the other CTAs that its copies have landed.
  for (int row = tid >> 3; row < 2 * a.rd; row += kRfThreads / 8) {   // eight threads per row
    const int which = row >= a.rd ? 1 : 0, t = which ? row - a.rd : row;
    const int64_t start = (bh * D + dims[t]) * a.npc + p0;
    const __half* src = (which ? a.kmax : a.kmin) + (start & ~7ll);
    __half* dst = (which ? bmx : bmn) + t * a.rs;
    const int off = (int)(start & 7), left = np > 0 ? off + np : 0;   // halves from the first copy's start
    if (which == 0 && (tid & 7) == 0) boff[t] = t * a.rs + off;
    for (int h = (tid & 7) * 8; h < left; h += 64) cp_async16(dst + h, src + h, min(16, (left - h) * 2));
  }
  cp_async_commit();
  if (tid < a.rd) {
    const int d = dims[tid];
    float P = 0.f, N = 0.f;
    for (int h = 0; h < G; ++h) {
      const float v = qs[h * D + d];
      P += fmaxf(v, 0.f);
      N += fminf(v, 0.f);
    }
    pn[0][tid] = P;
    pn[1][tid] = N;
  }

  // Attention state.  S^T (tokens x heads) = K q^T and O^T (dims x heads) = V^T P^T, so K and V fill the
  // 16 rows of the tensor-core product and the heads its 8 columns.  A page's 16 K and V rows go from
  // global memory straight into the operands of the lanes that use them, in 16-byte pieces: the dims of
  // a K row are taken in the order that gives lane r whole pieces (the query's fragments follow the same
  // order), those of a V row in the order that gives lane g whole pieces (undone when the output is
  // written).
  constexpr int KJ = D / 32;                           // 16-byte pieces of a K row per lane
  constexpr int VH = D / 64;                           // 16-byte pieces of a V row per lane
  const bool real = g < G;
  const uint4* qrow = reinterpret_cast<const uint4*>(qh2[real ? g : 0]) + r;
  float o[D / 16][4];                                  // rows: dims, columns: heads 2r, 2r + 1
#pragma unroll
  for (int i = 0; i < D / 16; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
  float m_run[2] = {-INFINITY, -INFINITY}, l_part[2] = {0.f, 0.f};   // heads 2r, 2r + 1
  const __half* klane = a.k + bh * a.T_cap * D + g * D + r * 8;   // this lane's pieces of page 0
  const __half* vlane = a.v + bh * a.T_cap * D + 2 * r * D + g * 8;
  int n_att = 0;                                       // chosen pages
  uint4 kx[2][KJ], vx[4][VH];                          // K rows g, g + 8; V rows 2r, 2r + 1, 2r + 8, 2r + 9
  auto load_k = [&](int page, bool ok) {
    const __half* src = klane + (int64_t)page * (kPage * D);
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int j = 0; j < KJ; ++j) kx[t][j] = ld_row16(src + t * 8 * D + j * 32, ok);
  };
  auto load_v = [&](int page, bool ok) {
    const __half* src = vlane + (int64_t)page * (kPage * D);
#pragma unroll
    for (int t = 0; t < 4; ++t)
#pragma unroll
      for (int h = 0; h < VH; ++h) vx[t][h] = ld_row16(src + ((t & 1) + (t >> 1) * 8) * D + h * 64, ok);
  };
  // the pages after the next one on their way into L2 (a page's K and V rows: 16 D halves each)
  auto prefetch = [&](int at) {
    if (lane < 2 && at < n_att) {
      const __half* src = (lane ? vlane - 2 * D : klane) + (int64_t)sel[at] * (kPage * D);
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(src), "r"(kPage * D * 2) : "memory");
    }
  };
  // the newest page: rows past its length zero, the step's token from the input
  auto load_tail = [&]() {
    const int fresh = room ? tail_valid - 1 : kPage;
    const __half* kbase = a.k + (bh * a.T_cap + (int64_t)ns * kPage) * D;
    const __half* vbase = a.v + (bh * a.T_cap + (int64_t)ns * kPage) * D;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int row = g + 8 * t;
      const __half* src = row == fresh ? a.k_new + bh * D : kbase + row * D;
#pragma unroll
      for (int j = 0; j < KJ; ++j) kx[t][j] = ld_row16(src + (4 * j + r) * 8, row < tail_valid);
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int row = 2 * r + (t & 1) + (t >> 1) * 8;
      const __half* src = row == fresh ? a.v_new + bh * D : vbase + row * D;
#pragma unroll
      for (int h = 0; h < VH; ++h) vx[t][h] = ld_row16(src + h * 64 + g * 8, row < tail_valid);
    }
  };

  // Pass 0: the warp of the newest page attends to it while the bounds are in flight.  Pass 1: the page
  // choice, then every warp's chosen pages.
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    int i = tail_warp ? 0 : 1, step = 1, end = 1;
    if (pass == 1) {
      cp_async_wait<0>();
      __syncthreads();
      // ---- scores of this CTA's pages: lane = page, warp w sums the dims t = w (mod kRfWarps), four at
      // a time
      for (int t0 = warp; t0 < a.rd; t0 += 4 * kRfWarps) {
        int at[4];
        float P[4], N[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int t = t0 + u * kRfWarps, tc = t < a.rd ? t : t0;
          at[u] = boff[tc];
          P[u] = t < a.rd ? pn[0][tc] : 0.f;
          N[u] = t < a.rd ? pn[1][tc] : 0.f;
        }
        for (int pl = lane; pl < np; pl += 32) {
          float acc = t0 == warp ? 0.f : part[warp * sp + pl];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float hi = __half2float(bmx[at[u] + pl]) * P[u] + __half2float(bmn[at[u] + pl]) * N[u];
            if (t0 + u * kRfWarps < a.rd) acc += hi;
          }
          part[warp * sp + pl] = acc;
        }
      }
      __syncthreads();
      // ---- 2. every score into every CTA of the cluster
      if constexpr (CL > 1) {
        if (tid == 0) {
          tc_mbar_expect_tx(&bar[0], (uint32_t)ns * 4u);
          if (rank == 0) tc_mbar_expect_tx(&bar[1], (uint32_t)(CL * G * (D + 2)) * 4u);
        }
        asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
      }
      const int nw = min(kRfWarps, a.rd);              // warps that had dims
      for (int pl = tid; pl < np; pl += kRfThreads) {
        float s = 0.f;
        for (int w = 0; w < nw; ++w) s += part[w * sp + pl];
        if constexpr (CL > 1) {
#pragma unroll
          for (int dst = 0; dst < CL; ++dst)
            st_async(cluster_addr(sc + p0 + pl, dst), s, cluster_addr(&bar[0], dst));
        } else {
          sc[p0 + pl] = s;
        }
      }
      if constexpr (CL > 1) {
        // (waited for before the end: a CTA that does not wait for scores, since it found no candidate page or its
        // bounded wait ran out, stays until the others have sent theirs)
        asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::: "memory");
        if (ns > 0) wait_received(&bar[0]);
      } else {
        __syncthreads();
      }

      // ---- 3. the k best pages under (score desc, page asc), by every CTA for itself.  Few pages are ranked
      // by counting; of more, the k-th largest score key is found bit by bit, from the highest bit in which the
      // keys differ, the keys that reach a
      // candidate counted by the barrier itself, until exactly k do or no bit is left (ties: the lower
      // pages); then the kept pages in ascending order from one word of flags per 32 pages.
      const int k = min(a.kp, ns);
      const int nk = (ns + kRfThreads - 1) / kRfThreads;   // pages per thread: tid, tid + 256, ..
      constexpr int KR = 4;                            // of them with their keys in registers
      uint32_t key[KR];
#pragma unroll
      for (int u = 0; u < KR; ++u) {
        const int p = tid + u * kRfThreads;
        key[u] = p < ns ? f32_key(sc[p]) : 0u;         // a pad never reaches a candidate (they are >= 1)
      }
      auto key_of = [&](int u) {
        const int p = tid + u * kRfThreads;
        return p < ns ? f32_key(sc[p]) : 0u;
      };
      uint32_t thr = 1;                                // kept: keys at or above it (ge),
      bool ge = true;
      int need = 0;                                    // or above it and the first `need` equal to it
      if (k < ns && ns <= kRankPages) {                // few: the pages ahead of each one counted
        uint32_t* kp_ = reinterpret_cast<uint32_t*>(sc);
        if (tid < ((ns + 3) & ~3)) kp_[tid] = key[0];  // (its own score; 0 behind the last)
        __syncthreads();
        int ahead = 0;                                 // before p: keys >= its own, after it: > its own
        if (tid < ns) {
          const uint32_t own = key[0], before = own - 1u;
#pragma unroll 4
          for (int j = 0; j < ns; j += 4) {
            const uint4 x = *reinterpret_cast<const uint4*>(kp_ + j);
            ahead += (x.x > (j < tid ? before : own)) + (x.y > (j + 1 < tid ? before : own)) +
                     (x.z > (j + 2 < tid ? before : own)) + (x.w > (j + 3 < tid ? before : own));
          }
        }
        key[0] = tid < ns && ahead < k ? 1u : 0u;      // (thr = 1: these are kept)
      } else if (k < ns) {
        uint32_t mx = 0, mn = 0xffffffffu;
        for (int u = 0; u < nk; ++u) {
          const uint32_t x = key_of(u);
          mx = max(mx, x);
          if (x != 0u) mn = min(mn, x);
        }
        mx = __reduce_max_sync(0xffffffffu, mx);
        mn = __reduce_min_sync(0xffffffffu, mn);
        if (lane == 0) {
          red[2 * warp] = mx;
          red[2 * warp + 1] = mn;
        }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kRfWarps; ++w) {
          mx = max(mx, red[2 * w]);
          mn = min(mn, red[2 * w + 1]);
        }
        ge = false;
        thr = mx;                                      // all keys equal: the first k
        need = k;
        int par = 0;
        if (mx != mn) {
          int above = 0;                               // keys above the prefix's range
          uint32_t bit = 0x80000000u >> __clz((int)(mx ^ mn));
          thr = mx & ~(2u * bit - 1u);                 // (bit 31: 2 * bit wraps to 0, thr to 0)
          // two bits a round while three counts fit a word; the last round may have one bit (lo = 0: its
          // first candidate is thr itself)
          for (; nk > 1 && ns < 1024 && bit != 0u && !ge; bit >>= 2) {
            const uint32_t lo = bit >> 1, t1 = thr | lo, t2 = thr | bit, t3 = t2 | lo;
            uint32_t c = 0;
#pragma unroll
            for (int u = 0; u < KR; ++u)
              c += (key[u] >= t1 ? 1u : 0u) + (key[u] >= t2 ? 1u << 10 : 0u) + (key[u] >= t3 ? 1u << 20 : 0u);
            c = __reduce_add_sync(0xffffffffu, c);
            if (lane == 0) cnt[par][warp] = (int)c;
            __syncthreads();
            const int4 x = *reinterpret_cast<const int4*>(cnt[par]), y = *reinterpret_cast<const int4*>(cnt[par] + 4);
            c = (uint32_t)(((x.x + x.y) + (x.z + x.w)) + ((y.x + y.y) + (y.z + y.w)));
            par ^= 1;
            const int c1 = (int)(c & 1023u), c2 = (int)((c >> 10) & 1023u), c3 = (int)(c >> 20);
            if (c3 >= k) {
              thr = t3;
              ge = c3 == k;
            } else if (c2 >= k) {
              thr = t2;
              above = c3;
              ge = c2 == k;
            } else if (c1 >= k) {
              thr = t1;
              above = c2;
              ge = c1 == k;
            } else {
              above = c1;
            }
          }
          if (ge) bit = 0u;
          for (; bit != 0u; bit >>= 1) {
            const uint32_t t = thr | bit;
            int c;
            if (nk == 1) {                             // counted by the barrier itself
              c = __syncthreads_count(key[0] >= t);
            } else {
              c = 0;
#pragma unroll
              for (int u = 0; u < KR; ++u) c += key[u] >= t ? 1 : 0;
              for (int u = KR; u < nk; ++u) c += key_of(u) >= t ? 1 : 0;
              c = __reduce_add_sync(0xffffffffu, c);
              if (lane == 0) cnt[par][warp] = c;
              __syncthreads();
              const int4 x = *reinterpret_cast<const int4*>(cnt[par]), y = *reinterpret_cast<const int4*>(cnt[par] + 4);
              c = ((x.x + x.y) + (x.z + x.w)) + ((y.x + y.y) + (y.z + y.w));
              par ^= 1;
            }
            if (c >= k) {
              thr = t;
              if (c == k) {
                ge = true;
                break;
              }
            } else {
              above = c;
            }
          }
          need = ge ? 0 : k - above;
        }
      }
      const int words = (ns + 31) / 32;                // flags of 32 pages each: kept for sure / equal to thr
      for (int u = 0; u < nk; ++u) {
        const uint32_t x = ns <= kRankPages ? key[0] : key_of(u);
        const uint32_t fg = __ballot_sync(0xffffffffu, ge ? x >= thr : x > thr);
        const uint32_t fe = __ballot_sync(0xffffffffu, !ge && x == thr);
        const int w = warp + u * kRfWarps;
        if (lane == 0 && w < words) {
          flags[2 * w] = fg;
          flags[2 * w + 1] = fe;
        }
      }
      __syncthreads();
      {
        // every warp: kept and equal counts before each word (lane = word), then its own words' pages
        int base_g = 0, base_e = 0;
        for (int w0 = 0; w0 < words; w0 += 32) {
          const int w = w0 + lane;
          const uint2 f = w < words ? *reinterpret_cast<const uint2*>(flags + 2 * w) : make_uint2(0u, 0u);
          const int mine = __popc(f.x) | (__popc(f.y) << 16);
          int incl = mine;
#pragma unroll
          for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
          }
          const int excl = incl - mine;
          for (int v = warp; v < min(32, words - w0); v += kRfWarps) {   // word w0 + v, lane = page
            const int ex = __shfl_sync(0xffffffffu, excl, v);
            const uint32_t fg = __shfl_sync(0xffffffffu, f.x, v), fe = __shfl_sync(0xffffffffu, f.y, v);
            const unsigned lt = (1u << lane) - 1u;
            const int gt = base_g + (ex & 0xffff) + __popc(fg & lt), eq = base_e + (ex >> 16) + __popc(fe & lt);
            if (((fg >> lane) & 1u) || (((fe >> lane) & 1u) && eq < need)) sel[gt + min(eq, need)] = (w0 + v) * 32 + lane;
          }
          const int all = __shfl_sync(0xffffffffu, incl, 31);
          base_g += all & 0xffff;
          base_e += all >> 16;
        }
      }
      __syncthreads();
      n_att = k;
      if (rank == 0 && a.page_idx != nullptr)
        for (int e = tid; e < a.kp; e += kRfThreads) a.page_idx[bh * a.kp + e] = e < n_att ? sel[e] : -1;
      // ---- 4. attention: chosen page i goes to CTA i % CL, warp (i / CL) % kRfWarps
      i = rank + CL * warp;
      step = CL * kRfWarps;
      end = n_att;
    }
    int valid = kPage;
    if (pass == 0) {
      valid = tail_valid;
      if (i < end) load_tail();
    } else {
      const int page = i < end ? sel[i] : 0;
      load_k(page, i < end);                           // (no page: zeros, so that nothing is kept across passes)
      load_v(page, i < end);
      prefetch(i + step);
      prefetch(i + 2 * step);
    }
#pragma unroll 1
    while (i < end) {
      float s0[4] = {0.f, 0.f, 0.f, 0.f}, s1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int j = 0; j < KJ; ++j) {
        const uint4 q = real ? qrow[4 * j] : make_uint4(0u, 0u, 0u, 0u);
        mma16816(s0, kx[0][j].x, kx[1][j].x, kx[0][j].y, kx[1][j].y, q.x, q.y);
        mma16816(s1, kx[0][j].z, kx[1][j].z, kx[0][j].w, kx[1][j].w, q.z, q.w);
      }
      i += step;
      const bool more = i < end;
      const int page = more ? sel[i] : 0;
      prefetch(i + 2 * step);
      // online softmax in the log2 domain: x[e][u] is head 2r + e, token g + 8u
      float x[2][2], p[2][2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        x[e][0] = g < valid ? (s0[e] + s1[e]) * a.scale_log2 : -INFINITY;
        x[e][1] = g + 8 < valid ? (s0[2 + e] + s1[2 + e]) * a.scale_log2 : -INFINITY;
      }
      valid = kPage;
      // the running maxima move only when a score exceeds them
      if (__any_sync(0xffffffffu, fmaxf(x[0][0], x[0][1]) > m_run[0] || fmaxf(x[1][0], x[1][1]) > m_run[1])) {
        float alpha[2] = {1.f, 1.f};
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float mx = fmaxf(x[e][0], x[e][1]);
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
          const float m_new = fmaxf(m_run[e], mx);
          if (m_new != -INFINITY) alpha[e] = exp2f(m_run[e] - m_new);
          l_part[e] *= alpha[e];
          m_run[e] = m_new;
        }
#pragma unroll
        for (int j = 0; j < D / 16; ++j) {
          o[j][0] *= alpha[0];
          o[j][1] *= alpha[1];
          o[j][2] *= alpha[0];
          o[j][3] *= alpha[1];
        }
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        // 2^8 times the probabilities relative to the maximum, and l with them: fp16 then rounds those down
        // to 2^-22 of the maximum as normal numbers (a warp meets many pages)
        const float mr = m_run[e] - 8.f;
        p[e][0] = m_run[e] != -INFINITY ? exp2f(x[e][0] - mr) : 0.f;
        p[e][1] = m_run[e] != -INFINITY ? exp2f(x[e][1] - mr) : 0.f;
        l_part[e] += p[e][0] + p[e][1];
      }
      // P^T as the (tokens x heads) operand, two 8x8 matrices transposed in registers, in fp16 and its
      // fp16 remainder: a warp takes up to dozens of pages against one maximum, where a warp of one or two
      // pages had its heaviest tokens' probabilities near 1 and so exact
      const uint32_t h0 = pack_half2(p[0][0], p[1][0]), h1 = pack_half2(p[0][1], p[1][1]);
      const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&h0));
      const float2 f1 = __half22float2(*reinterpret_cast<const __half2*>(&h1));
      const uint32_t b0 = movm_trans(h0), b1 = movm_trans(h1);
      const uint32_t c0 = movm_trans(pack_half2(p[0][0] - f0.x, p[1][0] - f0.y));
      const uint32_t c1 = movm_trans(pack_half2(p[0][1] - f1.x, p[1][1] - f1.y));
      // PV: tile j has rows g and g + 8 = dims 8g + j and 64 + 8g + j (D = 64: 8g + j and 8g + 4 + j)
#pragma unroll
      for (int j0 = 0; j0 < D / 16; j0 += 2) {         // two tiles at a time: their products do not wait
        const int w0 = j0 >> 1, w1 = VH == 2 ? w0 : w0 + 2;   // 4-byte words of the lane's pieces
        uint32_t av[2][4];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const uint32_t sel2 = e ? 0x7632 : 0x5410;
          av[e][0] = __byte_perm((&vx[0][0].x)[w0], (&vx[1][0].x)[w0], sel2);
          av[e][1] = __byte_perm((&vx[0][VH - 1].x)[w1], (&vx[1][VH - 1].x)[w1], sel2);
          av[e][2] = __byte_perm((&vx[2][0].x)[w0], (&vx[3][0].x)[w0], sel2);
          av[e][3] = __byte_perm((&vx[2][VH - 1].x)[w1], (&vx[3][VH - 1].x)[w1], sel2);
          mma16816(o[j0 + e], av[e][0], av[e][1], av[e][2], av[e][3], b0, b1);
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) mma16816(o[j0 + e], av[e][0], av[e][1], av[e][2], av[e][3], c0, c1);
      }
      load_k(page, more);
      load_v(page, more);
    }
  }

  // ---- 5. merge: warps -> CTA partial -> CTA 0
  float* wm = reinterpret_cast<float*>(smem + L.wpart);   // [warp][G] m, then l, then o [warp][G][D]
  float* wl = wm + kRfWarps * G;
  float* wo = wl + kRfWarps * G;                          // (16-byte aligned: 2 * 8 warps * G floats before it)
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    l_part[e] += __shfl_xor_sync(0xffffffffu, l_part[e], 4);
    l_part[e] += __shfl_xor_sync(0xffffffffu, l_part[e], 8);
    l_part[e] += __shfl_xor_sync(0xffffffffu, l_part[e], 16);
    const int h = 2 * r + e;
    if (h < G) {
      if (g == 0) {
        wm[warp * G + h] = m_run[e];
        wl[warp * G + h] = l_part[e];
      }
#pragma unroll
      for (int j = 0; j < D / 16; ++j) {
        wo[(warp * G + h) * D + 8 * g + j] = o[j][e];
        wo[(warp * G + h) * D + 8 * g + j + (VH == 2 ? 64 : 4)] = o[j][2 + e];
      }
    }
  }
  __syncthreads();
  float* cpo = reinterpret_cast<float*>(smem + L.cpart);  // CTA 0: o [CL][G][D], then (m, l) [CL][G]
  float2* cpm = reinterpret_cast<float2*>(cpo + CL * G * D);
  for (int e = tid; e < G * (D / 4); e += kRfThreads) {    // four dims of a head
    const int row = e / (D / 4), d = e % (D / 4) * 4;
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < kRfWarps; ++w) M = fmaxf(M, wm[w * G + row]);
    float Lsum = 0.f;
    float4 O = make_float4(0.f, 0.f, 0.f, 0.f);
    if (M != -INFINITY) {
#pragma unroll
      for (int w = 0; w < kRfWarps; ++w) {
        const float f = exp2f(wm[w * G + row] - M);
        const float4 x = *reinterpret_cast<const float4*>(wo + (w * G + row) * D + d);
        Lsum += wl[w * G + row] * f;
        O.x += x.x * f;
        O.y += x.y * f;
        O.z += x.z * f;
        O.w += x.w * f;
      }
    }
    if constexpr (CL > 1) {
      const uint32_t b1 = cluster_addr(&bar[1], 0);
      st_async4(cluster_addr(cpo + (rank * G + row) * D + d, 0), O, b1);
      if (d == 0) {
        const uint32_t at = cluster_addr(cpm + rank * G + row, 0);
        st_async(at, M, b1);
        st_async(at + 4u, Lsum, b1);
      }
    } else {
      const float inv = Lsum > 0.f ? 1.f / Lsum : 0.f;
      store_out4(a.out + ((int64_t)b * a.Hq + (int64_t)kvh * G + row) * D + d, O.x * inv, O.y * inv, O.z * inv, O.w * inv);
    }
  }
  if constexpr (CL > 1) {
    if (rank == 0) {
      wait_received(&bar[1]);
      for (int e = tid; e < G * (D / 2); e += kRfThreads) {
        const int row = e / (D / 2), d = e % (D / 2) * 2;
        float M = -INFINITY;
#pragma unroll
        for (int c = 0; c < CL; ++c) M = fmaxf(M, cpm[c * G + row].x);
        float Lsum = 0.f;
        float2 O = make_float2(0.f, 0.f);
        if (M != -INFINITY) {
#pragma unroll
          for (int c = 0; c < CL; ++c) {
            const float2 ml = cpm[c * G + row];
            const float2 x = *reinterpret_cast<const float2*>(cpo + (c * G + row) * D + d);
            const float f = exp2f(ml.x - M);
            Lsum += ml.y * f;
            O.x += x.x * f;
            O.y += x.y * f;
          }
        }
        const float inv = Lsum > 0.f ? 1.f / Lsum : 0.f;
        store_out2(a.out + ((int64_t)b * a.Hq + (int64_t)kvh * G + row) * D + d, O.x * inv, O.y * inv);
      }
    }
  }
  if constexpr (CL > 1) asm volatile("barrier.cluster.wait.aligned;\n" ::: "memory");
  if (!append) return;
  // the appended token filled its page: the page's per-dim min and max (its other rows from the cache)
  if (tail_warp && room && n % kPage == 0) {
    for (int d = lane; d < D; d += 32) {
      __half x[kPage];
#pragma unroll
      for (int row = 0; row < kPage - 1; ++row) x[row] = a.k[(bh * a.T_cap + (int64_t)ns * kPage + row) * D + d];
      x[kPage - 1] = a.k_new[bh * D + d];
      __half lo = x[0], hi = x[0];
#pragma unroll
      for (int row = 1; row < kPage; ++row) {
        lo = __hlt(x[row], lo) ? x[row] : lo;
        hi = __hgt(x[row], hi) ? x[row] : hi;
      }
      a.kmin[(bh * D + d) * a.npc + ns] = lo;
      a.kmax[(bh * D + d) * a.npc + ns] = hi;
    }
  }
  // every thread of this CTA read T_len before this point; the last CTA of batch entry b (all
  // CL CTAs of its Hkv clusters) stores the new length and clears the count
  __syncthreads();
  if (tid == 0) {
    const unsigned old = atomicAdd(reinterpret_cast<unsigned*>(a.T_len) + b, 1u << 24);
    if ((int)(old >> 24) == CL * a.Hkv - 1) a.T_len[b] = n;
    if (!room && rank == 0 && kvh == 0) atomicOr(&g_status_rocket, MKV_FLAG_CACHE_FULL);
  }
}

constexpr int kRfDynMax = (227 - 5) * 1024;   // dynamic shared memory beside the kernel's 4.8 KB of static

int rf_row(int64_t npc, int cl) { return ((int)((npc + cl - 1) / cl) + 8 + 7) / 8 * 8; }   // halves per bounds row
size_t rf_smem(const RfArgs& a, int D, int cl) {
  return (size_t)RfLayout(D, a.G, a.npc, a.kp, a.rd, rf_row(a.npc, cl), cl).bytes;
}

template <int D, int CL>
cudaError_t launch_rf_t(RfArgs a, int units, cudaStream_t st) {
  a.rs = rf_row(a.npc, CL);
  const size_t smem = rf_smem(a, D, CL);
  cudaError_t e = allow_all_smem<rocket_fused_kernel<D, CL>>();
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CL;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CL, units);
  cfg.blockDim = dim3(kRfThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = CL > 1 ? 1 : 0;
  e = cudaLaunchKernelEx(&cfg, rocket_fused_kernel<D, CL>, a);
  return e != cudaSuccess ? e : cudaPeekAtLastError();
}

// CTAs per (batch, kv-head).  More of them shorten a unit's serial parts (page scores, pages per warp);
// fewer leave each SM one CTA and repeat the common prologue less.  Measured, us a launch at CL = 8 / 4 /
// 2 / 1 (32/8 heads, D = 128, 4097 slots and 64 pages; 16341 slots and 256 pages):
//   16 units 12.8 / 13.1 / 16.2 / 19.7; 21.8 / 24.4 / 39.0 / 53.9
//   32 units 14.0 / 13.5 / 16.5 / 20.2; 24.6 / 25.1 / 39.4 / 54.1
//   64 units 26.1 / 17.0 / 17.5 / 20.6; 49.5 / 36.6 / 43.2 / 57.1
//  128 units 49.0 / 32.0 / 23.2 / 22.3; 96.3 / 73.3 / 64.6 / 59.7
// A CTA holds the chosen dims' bounds and the partial scores of its 1 / CL of the pages, so long caches and many
// dims need more CTAs than that (32/8 heads, D = 128, 128 units: 20160 slots fit CL = 1 with 32 dims, 5888
// with 128); eight hold every accepted length.
template <int D>
cudaError_t launch_rf_d(const RfArgs& a, int units, cudaStream_t st) {
  int cl = units <= 16 ? 8 : units <= 64 ? 4 : units <= 112 ? 2 : 1;
  while (cl < kRocketCluster && rf_smem(a, D, cl) > (size_t)kRfDynMax) cl *= 2;
  if (cl == 8) return launch_rf_t<D, 8>(a, units, st);
  if (cl == 4) return launch_rf_t<D, 4>(a, units, st);
  if (cl == 2) return launch_rf_t<D, 2>(a, units, st);
  return launch_rf_t<D, 1>(a, units, st);
}

}  // namespace

// Bytes that bound the accepted cache length: the page scores, the kept flags, every dim's bounds of an eighth
// of the pages and the warps' staged pages (the layout behind the documented limit).  RfLayout for eight CTAs
// needs at most 209104 bytes for a length within it.
size_t rocket_fused_smem(const mkv_config& c, int64_t T_cap) {
  const int D = c.D, G = c.Hq / c.Hkv, kp = c.topk_pages;
  const int64_t npc = T_cap / kPage;
  const int sp = (int)((npc + 7) / 8), rs = (sp + 8 + 7) / 8 * 8;
  const int sc = a16(G * D * 4), kf = a16(sc + (int)((npc + 3) & ~3ll) * 4), part = a16(kf + (int)npc);
  const int sel = a16(part + 8 * sp * 4), bounds = a16(sel + (kp + 1) * 4);
  const int pages = a16(bounds + std::max(2 * D * rs * 2, 8 * G * (D + 2) * 4));
  const int tail = a16(std::max(pages + 8 * 2 * kPage * D * 2, pages + 8 * G * (D + 2) * 4));
  return (size_t)tail + 2 * kPage * D * 2;
}

cudaError_t launch_rocket_fused(const mkv_config& c, const void* q, const mkv_cache& cache, int32_t* page_idx,
                                void* out, const void* k_new, const void* v_new, cudaStream_t st) {
  RfArgs a{};
  a.q = static_cast<const __half*>(q);
  a.k = static_cast<__half*>(cache.k);
  a.v = static_cast<__half*>(cache.v);
  a.kmin = static_cast<__half*>(cache.kmin);
  a.kmax = static_cast<__half*>(cache.kmax);
  a.T_len = cache.T_len;
  a.k_new = static_cast<const __half*>(k_new);
  a.v_new = static_cast<const __half*>(v_new);
  a.T_cap = cache.T_cap;
  a.npc = cache.T_cap / kPage;
  a.Hq = c.Hq;
  a.Hkv = c.Hkv;
  a.G = c.Hq / c.Hkv;
  a.kp = c.topk_pages;
  a.rd = c.topq_dims;
  const float scale = c.softmax_scale > 0.f ? c.softmax_scale : 1.0f / sqrtf((float)c.D);
  a.scale_log2 = scale * kLog2e;
  a.page_idx = page_idx;
  a.out = static_cast<__half*>(out);
  const int units = c.B * c.Hkv;
  return c.D == 128 ? launch_rf_d<128>(a, units, st) : launch_rf_d<64>(a, units, st);
}

cudaError_t take_status_rocket(uint32_t* flags, cudaStream_t st) {
  uint32_t zero = 0, v = 0;
  cudaError_t e = cudaMemcpyFromSymbolAsync(&v, g_status_rocket, sizeof(v), 0, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(g_status_rocket, &zero, sizeof(zero), 0, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  *flags |= v;
  return e;
}

}  // namespace mkv
