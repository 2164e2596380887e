// route_topk.cu -- router logits over the retained pool, top-k and
// renormalised gates (SlimWise Sec. 3.1, Eq. 2 and the renormalisation that
// follows it).
//
// Two forms, chosen by route_tiled: small batches take the cluster kernel that
// follows, larger ones (and large pools) a tiled product and a selecting
// kernel further down.  Both give the same bits.
//
// A thread-block cluster of kClusterCtas CTAs handles TB tokens.  CTA r of
// the cluster evaluates the logits of its slice of the retained experts for
// those tokens and writes each one, through distributed shared memory, into
// the shared memory of the CTA that runs that token's top-k (token tw on CTA
// tw mod 8); after one cluster barrier every top-k reads only its own shared
// memory.  Each CTA thus reads only 1/kClusterCtas of the router rows, and no
// global counter or second kernel is needed to join the slices.
//
// Logits follow the canonical fp32 order: lane l of a warp owns elements
// 128c + 4l + q (q = 0..3) of every 128-wide chunk c, accumulated with fused
// multiply-adds in (c, q) order, then the 32 lane partials are combined by an
// xor butterfly (offsets 16, 8, 4, 2, 1).  Two tokens' sums advance together
// in one packed fma.rn.f32x2 (two independent fp32 fused multiply-adds, each
// rounded as fmaf), which halves the multiply-add instructions of the
// issue-bound logit phase at large batches without changing a bit.  Pruned
// experts are never evaluated: restricting top-k to K' is the Eq. 2 mask
// with tau = -inf, with no separate masking pass.  Top-k is a warp-wide
// arg-max repeated k times on (order-preserving logit bits desc, expert id
// asc): each lane sorts its candidates once, then every round is two warp
// reductions over the lanes' current heads, so ties go to the lowest
// original id whatever the order of K'.
#include <cooperative_groups.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace slimwise {

constexpr int kRouteThreads = 256;
constexpr int kRouteWarps = kRouteThreads / 32;
constexpr int kClusterCtas = 8;
constexpr int kChunkBatch = 8;  // 128-wide chunks whose loads are issued together
constexpr int kPairChunkBatch = 4;  // the same, per row, when a warp takes two rows

// Order-preserving map of an fp32 value to uint32 (-0 folded onto +0).
__device__ __forceinline__ uint32_t logit_order_bits(float z) {
  uint32_t b = __float_as_uint(z);
  if ((b << 1) == 0u) b = 0u;
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float logit_from_order_bits(uint32_t o) {
  uint32_t b = (o & 0x80000000u) ? (o & 0x7FFFFFFFu) : ~o;
  return __uint_as_float(b);
}

// Hidden rows are staged in shared memory either as bf16 (half the space) or
// converted once to fp32 (no per-use conversion).  The product and the
// summation order are the same.  With two or more tokens per cluster the
// tokens are staged in pairs, interleaved element by element: for token pair
// tp, 128-wide chunk c and lane l, the quads ((tp nchunks + c) 2 + half) 32
// + l hold elements h = 128 c + 4 l + 2 half + {0, 1} as (t, h), (t + 1, h),
// (t, h + 1), (t + 1, h + 1), so that one load gives both tokens' values of
// two elements and consecutive lanes read consecutive quads.  A single token
// (TB = 1) is staged as its plain row.
// load_x4: the four consecutive staged elements from element index i.
__device__ __forceinline__ float4 load_x4(const __nv_bfloat16 *xs, size_t i) {
  const uint2 xr = *reinterpret_cast<const uint2 *>(xs + i);
  return make_float4(__uint_as_float(xr.x << 16), __uint_as_float(xr.x & 0xFFFF0000u),
                     __uint_as_float(xr.y << 16), __uint_as_float(xr.y & 0xFFFF0000u));
}
__device__ __forceinline__ float4 load_x4(const float *xs, size_t i) {
  return *reinterpret_cast<const float4 *>(xs + i);
}

// c0 = fma(a0, w, c0) and c1 = fma(a1, w, c1): two independent fused
// multiply-adds in one packed instruction, each rounded once to nearest
// exactly as fmaf, so two tokens' canonical sums advance together.
__device__ __forceinline__ void ffma2_acc(float &c0, float &c1, float a0, float a1, float w) {
  asm("{\n\t.reg .b64 ra, rw, rc;\n\t"
      "mov.b64 ra, {%2, %3};\n\t"
      "mov.b64 rw, {%4, %4};\n\t"
      "mov.b64 rc, {%0, %1};\n\t"
      "fma.rn.f32x2 rc, ra, rw, rc;\n\t"
      "mov.b64 {%0, %1}, rc;\n\t}"
      : "+f"(c0), "+f"(c1)
      : "f"(a0), "f"(a1), "f"(w));
}

// Element index of quad (tp, c, half, lane) of the paired staging.
__device__ __forceinline__ size_t pair_quad(int tp, int nchunks, int c, int half, int lane) {
  return ((((size_t)tp * nchunks + c) * 2 + half) * 32 + lane) * 4;
}

// Chunk c of one router row (lane's four weights w) into every token's sum,
// elements h = 128 c + 4 lane + q in q order.
template <int TB, typename XT>
__device__ __forceinline__ void fma_chunk(const XT *xs, int nchunks, int c, int lane, float4 w,
                                          float (&p)[TB]) {
  if constexpr (TB == 1) {
    const float4 x = load_x4(xs, ((size_t)c * 32 + lane) * 4);
    p[0] = fmaf(x.x, w.x, p[0]);
    p[0] = fmaf(x.y, w.y, p[0]);
    p[0] = fmaf(x.z, w.z, p[0]);
    p[0] = fmaf(x.w, w.w, p[0]);
  } else {
#pragma unroll
    for (int tp = 0; tp < TB / 2; ++tp) {
      const float4 a = load_x4(xs, pair_quad(tp, nchunks, c, 0, lane));
      const float4 b = load_x4(xs, pair_quad(tp, nchunks, c, 1, lane));
      ffma2_acc(p[2 * tp], p[2 * tp + 1], a.x, a.y, w.x);
      ffma2_acc(p[2 * tp], p[2 * tp + 1], a.z, a.w, w.y);
      ffma2_acc(p[2 * tp], p[2 * tp + 1], b.x, b.y, w.z);
      ffma2_acc(p[2 * tp], p[2 * tp + 1], b.z, b.w, w.w);
    }
  }
}

// Two router rows at once: each staged hidden vector feeds both rows' sums.
template <int TB, typename XT>
__device__ __forceinline__ void fma_chunk2(const XT *xs, int nchunks, int c, int lane, float4 w0,
                                           float4 w1, float (&p0)[TB], float (&p1)[TB]) {
  if constexpr (TB == 1) {
    const float4 x = load_x4(xs, ((size_t)c * 32 + lane) * 4);
    p0[0] = fmaf(x.x, w0.x, p0[0]);
    p0[0] = fmaf(x.y, w0.y, p0[0]);
    p0[0] = fmaf(x.z, w0.z, p0[0]);
    p0[0] = fmaf(x.w, w0.w, p0[0]);
    p1[0] = fmaf(x.x, w1.x, p1[0]);
    p1[0] = fmaf(x.y, w1.y, p1[0]);
    p1[0] = fmaf(x.z, w1.z, p1[0]);
    p1[0] = fmaf(x.w, w1.w, p1[0]);
  } else {
#pragma unroll
    for (int tp = 0; tp < TB / 2; ++tp) {
      const float4 a = load_x4(xs, pair_quad(tp, nchunks, c, 0, lane));
      const float4 b = load_x4(xs, pair_quad(tp, nchunks, c, 1, lane));
      ffma2_acc(p0[2 * tp], p0[2 * tp + 1], a.x, a.y, w0.x);
      ffma2_acc(p0[2 * tp], p0[2 * tp + 1], a.z, a.w, w0.y);
      ffma2_acc(p0[2 * tp], p0[2 * tp + 1], b.x, b.y, w0.z);
      ffma2_acc(p0[2 * tp], p0[2 * tp + 1], b.z, b.w, w0.w);
      ffma2_acc(p1[2 * tp], p1[2 * tp + 1], a.x, a.y, w1.x);
      ffma2_acc(p1[2 * tp], p1[2 * tp + 1], a.z, a.w, w1.y);
      ffma2_acc(p1[2 * tp], p1[2 * tp + 1], b.x, b.y, w1.z);
      ffma2_acc(p1[2 * tp], p1[2 * tp + 1], b.z, b.w, w1.w);
    }
  }
}

// Hidden rows are staged as fp32 (no conversion per use) except at TB = 4
// and TB = 16, which stage bf16: at 16 tokens so that two CTAs fit on an SM,
// at 4 because it measured no slower.
template <int TB>
struct StageType {
  using T = float;
};
template <>
struct StageType<4> {
  using T = __nv_bfloat16;
};
template <>
struct StageType<16> {
  using T = __nv_bfloat16;
};


// Shared memory of one CTA: hidden rows (TB x H elements of StageType, in
// token pairs from TB = 2 on; see load_x4), the logits of
// the tokens whose top-k it runs [ceil(TB/8)][m] fp32 (written by every CTA
// of the cluster), retained ids [m] int32.  Rows of tokens past the batch are
// zero, so every token slot computes (and discards) a logit.
// Round j of the top-k: the winner (order bits whi, complemented id wlo) goes
// to lane j.  With no candidate left (fewer than k distinct ids, already
// reported) a valid id stands in.
__device__ __forceinline__ void take_winner(uint32_t whi, uint32_t wlo, int j, int lane,
                                            const int32_t *ids, const Dims &d, float &my_z,
                                            int &my_e) {
  uint32_t wid = 0xFFFFFFFFu - wlo;
  if (whi == 0u || wid >= (uint32_t)d.E) wid = (uint32_t)ids[0];
  if (lane == j) {
    my_z = logit_from_order_bits(whi);
    my_e = (int)wid;
  }
}

// The grid's last CTA reports bad and repeated retained ids and resets the
// error word (and, for a call that groups locally, the counters).  `earlier`:
// this thread's error bits of the kernels before this one.
__device__ __forceinline__ void report_retained(const int32_t *__restrict__ retained, const Dims &d,
                                                const Ws &ws, int earlier = 0) {
  __shared__ uint32_t seen[kMaxExperts / 32];
  __shared__ int bad;
  for (int i = threadIdx.x; i < kMaxExperts / 32; i += blockDim.x) seen[i] = 0;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  if (earlier) atomicOr(&bad, earlier);
  for (int r = threadIdx.x; r < d.m_ret; r += blockDim.x) {
    int e = retained ? retained[r] : r;
    if (e < 0 || e >= d.E) {
      atomicOr(&bad, SLIMWISE_DEVERR_BAD_RETAINED);
    } else {
      uint32_t bit = 1u << (e & 31);
      if (atomicOr(&seen[e >> 5], bit) & bit)
        atomicOr(&bad, SLIMWISE_DEVERR_DUPLICATE_RETAINED);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) ws.ctrl[kCtrlErr] = bad;
  // without a grouping kernel the FFN's counters start here: at most one
  // entry per expert, and the shared expert's
  if (d.local) {
    if (threadIdx.x == 0) ws.ctrl[kCtrlWorkCounter] = 0;
    for (int i = threadIdx.x; i <= d.E; i += blockDim.x) ws.entry_done[i] = 0;
  }
}

// Top-k and gates of token t, by one warp, from its logits z[0, m') over the
// retained ids: NC candidates per lane in registers (m' <= 32 NC), or NC = 0
// for larger pools.
template <int NC>
__device__ __forceinline__ void topk_token(const float *z, const int32_t *ids, const Dims &d,
                                           const Ws &ws, int t, int lane) {
  const int m = d.m_ret, k = d.k;
  float my_z = 0.0f;
  int my_e = 0;
  if constexpr (NC > 0) {
    // this lane's candidates r = lane + 32 i (i < NC) as 64-bit keys
    // (order-preserving logit bits, complemented id; 0 = none), kept sorted
    // descending in registers -- every index below is a compile-time one;
    // all loads are issued before any is used
    float zc[NC];
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      const int r = lane + 32 * i;
      if (r < m) {
        zc[i] = z[r];
      }
    }
    unsigned long long key[NC];
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      const int r = lane + 32 * i;
      key[i] = r < m ? ((unsigned long long)logit_order_bits(zc[i]) << 32) |
                           (unsigned long long)(0xFFFFFFFFu - (uint32_t)ids[r])
                     : 0ull;
#pragma unroll
      for (int j = i; j > 0; --j)
        if (key[j] > key[j - 1]) {
          const unsigned long long tmp = key[j];
          key[j] = key[j - 1];
          key[j - 1] = tmp;
        }
    }
    // k rounds: the warp's largest head key wins and its lane pops it
    for (int j = 0; j < k; ++j) {
      const unsigned long long mine = key[0];
      const uint32_t hi = (uint32_t)(mine >> 32), lo = (uint32_t)mine;
      const uint32_t whi = __reduce_max_sync(0xFFFFFFFFu, hi);
      const uint32_t wlo = __reduce_max_sync(0xFFFFFFFFu, hi == whi ? lo : 0u);
      const unsigned long long win = ((unsigned long long)whi << 32) | wlo;
      // pop every copy of the winner (repeated retained ids give equal keys)
      for (int pops = 0; pops < NC && key[0] == win && win != 0ull; ++pops) {
#pragma unroll
        for (int i = 0; i + 1 < NC; ++i) key[i] = key[i + 1];
        key[NC - 1] = 0ull;
      }
      take_winner(whi, wlo, j, lane, ids, d, my_z, my_e);
    }
  } else {
    // large pools: the lane's candidates sorted in a local array
    unsigned long long key[kMaxExperts / 32];
    int nc = 0;
    for (int r0 = lane; r0 < m; r0 += 128) {
      float zc[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = r0 + 32 * u;
        if (r < m) {
          zc[u] = z[r];
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = r0 + 32 * u;
        if (r < m) {
          const unsigned long long kv = ((unsigned long long)logit_order_bits(zc[u]) << 32) |
                                        (unsigned long long)(0xFFFFFFFFu - (uint32_t)ids[r]);
          int i = nc++;
          while (i > 0 && key[i - 1] < kv) {
            key[i] = key[i - 1];
            --i;
          }
          key[i] = kv;
        }
      }
    }
    int head = 0;
    for (int j = 0; j < k; ++j) {
      const unsigned long long mine = head < nc ? key[head] : 0ull;
      const uint32_t hi = (uint32_t)(mine >> 32), lo = (uint32_t)mine;
      const uint32_t whi = __reduce_max_sync(0xFFFFFFFFu, hi);
      const uint32_t wlo = __reduce_max_sync(0xFFFFFFFFu, hi == whi ? lo : 0u);
      const unsigned long long win = ((unsigned long long)whi << 32) | wlo;
      while (head < nc && key[head] == win) ++head;
      take_winner(whi, wlo, j, lane, ids, d, my_z, my_e);
    }
  }
  // g_j = exp(z_j - z_1) / sum_j' exp(z_j' - z_1), the sum in j order.
  const float z1 = __shfl_sync(0xFFFFFFFFu, my_z, 0);
  const float w = (lane < k) ? expf(my_z - z1) : 0.0f;
  float denom = 0.0f;
  for (int j = 0; j < k; ++j) denom += __shfl_sync(0xFFFFFFFFu, w, j);
  if (lane < k) {
    ws.topk_idx[(size_t)t * k + lane] = my_e;
    ws.topk_gate[(size_t)t * k + lane] = w / denom;
  }
}

// TB tokens per cluster; NC candidates per lane in the register top-k
// (m' <= 32 NC), or NC = 0 for the general top-k of larger pools.
template <int TB, int NC>
// Two CTAs per SM worth of registers, so one wave of CTAs holds 38 clusters.
__global__ void __launch_bounds__(kRouteThreads, 2)
    route_topk_kernel(const __nv_bfloat16 *__restrict__ hidden,
                      const float *__restrict__ router_w,
                      const int32_t *__restrict__ retained, Dims d, Ws ws) {
  using XT = typename StageType<TB>::T;
  extern __shared__ __align__(16) unsigned char smem[];
  cg::cluster_group cluster = cg::this_cluster();
  const int crank = (int)cluster.block_rank();
  const int H = d.H, m = d.m_ret;
  const int slice = (m + kClusterCtas - 1) / kClusterCtas;
  constexpr int kOwn = (TB + kClusterCtas - 1) / kClusterCtas;  // tokens whose top-k a CTA runs
  XT *xs = reinterpret_cast<XT *>(smem);
  float *zs = reinterpret_cast<float *>(smem + (size_t)TB * H * sizeof(XT));  // [kOwn][m]
  int32_t *ids = reinterpret_cast<int32_t *>(zs + (size_t)kOwn * m);

  // Before waiting for the previous kernel on the stream (this CTA may be
  // resident while it finishes): warm L2 with this CTA's router rows.  These
  // are prefetches only -- no value read here is used, and the ids that
  // address them are read past L1 -- so the results do not depend on whether
  // the previous kernel wrote the router rows or the retained ids.
  {
    const int r_lo = crank * slice, r_hi = min(m, r_lo + slice);
    const int lpr = H / 32;  // 128-byte lines per fp32 router row
    for (int i = threadIdx.x; i < (r_hi - r_lo) * lpr; i += blockDim.x) {
      const int r = r_lo + i / lpr;
      const int e = min(max(retained ? __ldcg(retained + r) : r, 0), d.E - 1);
      prefetch_l2(router_w + (size_t)e * H + (size_t)(i % lpr) * 32);
    }
  }
  // The inputs may come from the previous kernel on the stream.
  pdl_wait_primary();
  // Let the next kernel become resident; it waits for this grid to end.
  pdl_launch_dependents();
#ifdef SLIMWISE_TRACE
  const int tr_step = ws.ctrl[kCtrlTraceStep];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    trace_stamp(ws, tr_step, kTrRouteStart);
    reinterpret_cast<uint64_t *>(ws.ctrl + kCtrlWords)[(tr_step & (kTraceSteps - 1)) * kTrSlots + kTrFfnEnd] = 0;
  }
#endif

  const int cluster_id = blockIdx.x / kClusterCtas;
  const int t0 = cluster_id * TB;
  const int nt = min(TB, d.B - t0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // Retained ids, clamped into [0, E) so a bad id cannot fault.
  for (int r = threadIdx.x; r < m; r += blockDim.x) {
    int e = retained ? retained[r] : r;
    ids[r] = min(max(e, 0), d.E - 1);
  }
  if (blockIdx.x == gridDim.x - 1) report_retained(retained, d, ws);

  // Hidden rows of the cluster's tokens (16-byte vectors of 8 bf16), zero
  // past the batch.  Each thread issues TB loads before storing any, so the
  // staging costs one memory round trip per TB * 256 vectors.  With token
  // pairs a thread loads the same vector of both tokens of a pair and writes
  // the four interleaved quads it covers (lanes 2 (v mod 16) and 2 (v mod 16)
  // + 1 of chunk v / 16, both halves).
  const int vecs = H / 8;
  const int nchunks = H / 128;
  auto hidden_vec = [&](int t, int v) {
    return t < nt ? reinterpret_cast<const uint4 *>(hidden + (size_t)(t0 + t) * H)[v]
                  : make_uint4(0u, 0u, 0u, 0u);
  };
  if constexpr (TB == 1) {
    for (int v = threadIdx.x; v < vecs; v += kRouteThreads) {
      const uint4 r = hidden_vec(0, v);
      float4 *dst = reinterpret_cast<float4 *>(xs + 8 * v);
      dst[0] = make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xFFFF0000u),
                           __uint_as_float(r.y << 16), __uint_as_float(r.y & 0xFFFF0000u));
      dst[1] = make_float4(__uint_as_float(r.z << 16), __uint_as_float(r.z & 0xFFFF0000u),
                           __uint_as_float(r.w << 16), __uint_as_float(r.w & 0xFFFF0000u));
    }
  } else {
    constexpr int kPairsPerPass = TB / 2;  // pair-vectors per thread per pass
    const int items = (TB / 2) * vecs;
    for (int i0 = 0; i0 < items; i0 += kPairsPerPass * kRouteThreads) {
      uint4 r0[kPairsPerPass], r1[kPairsPerPass];
#pragma unroll
      for (int u = 0; u < kPairsPerPass; ++u) {
        const int i = i0 + u * kRouteThreads + (int)threadIdx.x;
        const int tp = i / vecs, v = i - tp * vecs;
        const bool in = i < items;
        r0[u] = in ? hidden_vec(2 * tp, v) : make_uint4(0u, 0u, 0u, 0u);
        r1[u] = in ? hidden_vec(2 * tp + 1, v) : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int u = 0; u < kPairsPerPass; ++u) {
        const int i = i0 + u * kRouteThreads + (int)threadIdx.x;
        if (i >= items) break;
        const int tp = i / vecs, v = i - tp * vecs;
        const int c = v >> 4, l0 = 2 * (v & 15);
        // words w of a vector hold elements 2w (low half) and 2w + 1 (high)
        const uint32_t a[4] = {r0[u].x, r0[u].y, r0[u].z, r0[u].w};
        const uint32_t b[4] = {r1[u].x, r1[u].y, r1[u].z, r1[u].w};
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          // elements 2w, 2w + 1: lane l0 + w / 2, half w % 2
          const size_t q = pair_quad(tp, nchunks, c, w & 1, l0 + (w >> 1));
          if constexpr (sizeof(XT) == 2) {
            // (t, 2w) | (t + 1, 2w) << 16, then the same for element 2w + 1
            *reinterpret_cast<uint2 *>(xs + q) =
                make_uint2((a[w] & 0xFFFFu) | (b[w] << 16), (a[w] >> 16) | (b[w] & 0xFFFF0000u));
          } else {
            *reinterpret_cast<float4 *>(xs + q) =
                make_float4(__uint_as_float(a[w] << 16), __uint_as_float(b[w] << 16),
                            __uint_as_float(a[w] & 0xFFFF0000u), __uint_as_float(b[w] & 0xFFFF0000u));
          }
        }
      }
    }
  }
  __syncthreads();

  // Logits of this CTA's slice [r_lo, r_hi) of the retained list.  With at
  // least two rows per warp (at 8 tokens per cluster: two rows per slice), a
  // warp takes its rows in pairs (rows r, r + 1), which halves the
  // shared-memory reads of the staged hidden rows; the sums and their order
  // are those of one row at a time.
  const int r_lo = crank * slice, r_hi = min(m, r_lo + slice);
  // At 8 tokens per cluster the staged rows' shared-memory reads bound the
  // logits, so pairs pay from two rows on (1.6 us at B = 256, m' = 64); at
  // 16 tokens (fewer warps busy) they lost 2 us at B = 512, m' = 32.
  const int npair = ((TB == 8 && r_hi - r_lo >= 2) || r_hi - r_lo >= 2 * kRouteWarps)
                        ? (r_hi - r_lo) / 2 : 0;
  for (int pi = warp; pi < npair; pi += kRouteWarps) {
    const int r = r_lo + 2 * pi;
    const float4 *w0 = reinterpret_cast<const float4 *>(router_w + (size_t)ids[r] * H) + lane;
    const float4 *w1 = reinterpret_cast<const float4 *>(router_w + (size_t)ids[r + 1] * H) + lane;
    float p0[TB], p1[TB];
#pragma unroll
    for (int t = 0; t < TB; ++t) p0[t] = p1[t] = 0.0f;
    for (int c0 = 0; c0 < nchunks; c0 += kPairChunkBatch) {
      float4 v0[kPairChunkBatch], v1[kPairChunkBatch];
#pragma unroll
      for (int u = 0; u < kPairChunkBatch; ++u)
        if (c0 + u < nchunks) {
          v0[u] = __ldg(w0 + 32 * (c0 + u));
          v1[u] = __ldg(w1 + 32 * (c0 + u));
        }
#pragma unroll
      for (int u = 0; u < kPairChunkBatch; ++u)
        if (c0 + u < nchunks)
          fma_chunk2<TB>(xs, nchunks, c0 + u, lane, v0[u], v1[u], p0, p1);
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1)
#pragma unroll
      for (int t = 0; t < TB; ++t) {
        p0[t] = p0[t] + __shfl_xor_sync(0xFFFFFFFFu, p0[t], off);
        p1[t] = p1[t] + __shfl_xor_sync(0xFFFFFFFFu, p1[t], off);
      }
    // lane t sends token t's two logits to the CTA that runs its top-k
#pragma unroll
    for (int t = 0; t < TB; ++t)
      if (lane == t && t < nt) {
        float *dst = cluster.map_shared_rank(zs, t % kClusterCtas) + (size_t)(t / kClusterCtas) * m;
        dst[r] = p0[t];
        dst[r + 1] = p1[t];
      }
  }
  for (int r = r_lo + 2 * npair + warp; r < r_hi; r += kRouteWarps) {
    const float4 *wrow = reinterpret_cast<const float4 *>(router_w + (size_t)ids[r] * H) + lane;
    float p[TB];
#pragma unroll
    for (int t = 0; t < TB; ++t) p[t] = 0.0f;
    for (int c0 = 0; c0 < nchunks; c0 += kChunkBatch) {
      float4 v[kChunkBatch];
#pragma unroll
      for (int u = 0; u < kChunkBatch; ++u)
        if (c0 + u < nchunks) v[u] = __ldg(wrow + 32 * (c0 + u));
#pragma unroll
      for (int u = 0; u < kChunkBatch; ++u)
        if (c0 + u < nchunks) fma_chunk<TB>(xs, nchunks, c0 + u, lane, v[u], p);
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1)
#pragma unroll
      for (int t = 0; t < TB; ++t) p[t] = p[t] + __shfl_xor_sync(0xFFFFFFFFu, p[t], off);
#pragma unroll
    for (int t = 0; t < TB; ++t)
      if (lane == t && t < nt)
        cluster.map_shared_rank(zs, t % kClusterCtas)[(size_t)(t / kClusterCtas) * m + r] = p[t];
  }
  // every logit is in the shared memory of the CTA that needs it; after this
  // barrier no CTA touches another's shared memory, so none waits at the end
  cluster.sync();

  // Top-k and gates: token tw of the cluster is handled by warp tw / 8 of the
  // cluster's CTA tw % 8, so the tokens' top-k run side by side.
  const int tw = warp * kClusterCtas + crank;
  if (tw < nt) topk_token<NC>(zs + (size_t)warp * m, ids, d, ws, t0 + tw, lane);
#ifdef SLIMWISE_TRACE
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    trace_stamp(ws, tr_step, kTrRouteEnd);
    ws.ctrl[kCtrlTraceStep] = tr_step + 1;
  }
#endif
}

// Dynamic shared memory of a routing CTA with TB tokens.
template <int TB>
size_t route_smem_bytes(const Dims &d) {
  return (size_t)TB * d.H * sizeof(typename StageType<TB>::T) +
         (size_t)((TB + kClusterCtas - 1) / kClusterCtas) * d.m_ret * 4 + (size_t)d.m_ret * 4;
}

// What a routing CTA leaves of the opt-in limit for its static shared memory
// (report_retained's, 144 bytes).
constexpr size_t kRouteStaticSmem = 1024;

template <int TB, int NC>
cudaError_t launch_route_tb(const __nv_bfloat16 *hidden, const float *router_w,
                            const int32_t *retained, Dims d, Ws ws, bool pdl, size_t max_smem,
                            cudaStream_t stream) {
  const size_t smem = route_smem_bytes<TB>(d);
  // one value for every call: the attribute is the kernel's, not the launch's,
  // and another thread may be launching it with another size
  cudaError_t err = cudaFuncSetAttribute(
      route_topk_kernel<TB, NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_smem);
  if (err != cudaSuccess) return err;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(((d.B + TB - 1) / TB) * kClusterCtas);
  cfg.blockDim = dim3(kRouteThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kClusterCtas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, route_topk_kernel<TB, NC>, hidden, router_w, retained, d, ws);
}

template <int TB>
cudaError_t launch_route_nc(const __nv_bfloat16 *hidden, const float *router_w,
                            const int32_t *retained, Dims d, Ws ws, bool pdl, size_t max_smem,
                            cudaStream_t stream) {
  auto launch = d.m_ret <= 128   ? launch_route_tb<TB, 4>
                : d.m_ret <= 256 ? launch_route_tb<TB, 8>
                                 : launch_route_tb<TB, 0>;
  return launch(hidden, router_w, retained, d, ws, pdl, max_smem, stream);
}

// --------------------------------------------------------------------------
// Large batches
// --------------------------------------------------------------------------
// A cluster of the kernel above reads the whole router for its 16 tokens and
// spends more issue slots on loads and conversions than on multiply-adds.
// There (route_tiled says where) the logits are a tiled product on the fp32
// units, in the same canonical order, and a second kernel runs the top-k:
//   route_logits_kernel  32 tokens (16 or 8 where those make too few CTAs) x
//                        16 retained experts per CTA, the K range streamed in
//                        128-wide chunks through a 4-stage cp.async ring.  Lane l of every warp holds partial
//                        sum l of its 8 tokens x 16 experts (128 registers),
//                        so 24 shared-memory loads feed 256 packed
//                        multiply-adds a chunk; the butterfly over the lanes
//                        runs as a transposing reduction (each step halves
//                        the values a lane carries: 124 shuffles for 128
//                        logits, not 640).  z goes to global scratch.
//   route_select_kernel  one warp per token over z.
// Bound by the fp32 multiply-adds: 8192 tokens x 256 experts run at 73 % of
// the 32 T/s that a register-only loop reaches here, two CTAs of 4 warps per
// SM (one of 8 warps: 57 %, all of them waiting for each chunk together;
// 16 tokens x 8 experts per warp: 70 %).
constexpr int kTileRow = 16;
constexpr int kTileThreads = 128;
constexpr int kTileStages = 4;
constexpr int kWarpRow = 16;   // experts of one warp
// WT tokens per warp (4 warps: 4 WT per tile).
constexpr int kTileWBytes = kTileRow * 128 * 4;
__host__ __device__ constexpr int tile_x_bytes(int wt) { return 4 * wt * 128 * 2; }
__host__ __device__ constexpr int tile_smem(int wt) { return kTileStages * (tile_x_bytes(wt) + kTileWBytes); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, uint32_t bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes)
               : "memory");
}

// One step of the transposing reduction: of 2 n values a lane keeps n, those
// of its half, each added to its partner's.
template <int kOff, int kN, int kSize>
__device__ __forceinline__ void reduce_step(float (&a)[kSize], int lane) {
  const bool upper = (lane & kOff) != 0;
#pragma unroll
  for (int i = 0; i < kN; ++i) {
    const float give = upper ? a[i] : a[i + kN], keep = upper ? a[i + kN] : a[i];
    a[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, kOff);
  }
}

template <int WT>
__global__ void __launch_bounds__(kTileThreads, WT == 8 ? 2 : 3)
    route_logits_kernel(const __nv_bfloat16 *__restrict__ hidden,
                        const float *__restrict__ router_w,
                        const int32_t *__restrict__ retained, Dims d, Ws ws,
                        float *__restrict__ z) {
  extern __shared__ __align__(16) unsigned char smem[];
  pdl_wait_primary();
  pdl_launch_dependents();
#ifdef SLIMWISE_TRACE
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
    const int tr_step = ws.ctrl[kCtrlTraceStep];
    trace_stamp(ws, tr_step, kTrRouteStart);
    reinterpret_cast<uint64_t *>(ws.ctrl + kCtrlWords)[(tr_step & (kTraceSteps - 1)) * kTrSlots + kTrFfnEnd] = 0;
  }
#endif
  const int H = d.H, m = d.m_ret, nchunks = H / 128;
  constexpr int kTileTok = 4 * WT, kTileXBytes = tile_x_bytes(WT);
  constexpr int kXLoads = kTileTok * 16 / kTileThreads;  // WT / 2
  const int t0 = blockIdx.x * kTileTok, r0 = blockIdx.y * kTileRow;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t xs = smem_u32(smem), wsm = xs + kTileStages * kTileXBytes;

  // this thread's 16-byte vectors of a chunk: WT / 2 of the hidden rows (rows
  // tid / 16 + 8 u; tokens past the batch are zero) and four of the router
  // rows (rows warp + 4 u; rows past the pool repeat its last one and are
  // dropped at the end)
  const int xrow = tid >> 4, xcol = tid & 15;
  const __nv_bfloat16 *xsrc[kXLoads];
  const float *wsrc[4];
  uint32_t xbytes[kXLoads];
#pragma unroll
  for (int u = 0; u < kXLoads; ++u) {
    const int t = t0 + xrow + 8 * u;
    xbytes[u] = t < d.B ? 16u : 0u;
    xsrc[u] = hidden + (size_t)(t < d.B ? t : 0) * H + xcol * 8;
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = min(r0 + warp + 4 * u, m - 1);
    const int e = min(max(retained ? __ldg(retained + r) : r, 0), d.E - 1);
    wsrc[u] = router_w + (size_t)e * H + lane * 4;
  }
  auto load_chunk = [&](int c) {
    const int st = c % kTileStages;
    const uint32_t xd = xs + st * kTileXBytes + xrow * 256 + xcol * 16;
    const uint32_t wd = wsm + st * kTileWBytes + warp * 512 + lane * 16;
#pragma unroll
    for (int u = 0; u < kXLoads; ++u) cp_async16(xd + u * 8 * 256, xsrc[u] + c * 128, xbytes[u]);
#pragma unroll
    for (int u = 0; u < 4; ++u) cp_async16(wd + u * 4 * 512, wsrc[u] + c * 128, 16u);
  };
#pragma unroll
  for (int c = 0; c < kTileStages - 1; ++c) {
    if (c < nchunks) load_chunk(c);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }

  float acc[kWarpRow][WT];
#pragma unroll
  for (int r = 0; r < kWarpRow; ++r)
#pragma unroll
    for (int t = 0; t < WT; ++t) acc[r][t] = 0.0f;
  const unsigned char *xw = smem + (size_t)warp * WT * 256 + lane * 8;
  const unsigned char *ww = smem + kTileStages * kTileXBytes + lane * 16;
  for (int c = 0; c < nchunks; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kTileStages - 2) : "memory");
    __syncthreads();  // chunk c is here, and chunk c - 1 has been read by all
    if (c + kTileStages - 1 < nchunks) load_chunk(c + kTileStages - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int st = c % kTileStages;
    float x[4][WT];
#pragma unroll
    for (int t = 0; t < WT; ++t) {
      const uint2 v = *reinterpret_cast<const uint2 *>(xw + st * kTileXBytes + t * 256);
      x[0][t] = __uint_as_float(v.x << 16);
      x[1][t] = __uint_as_float(v.x & 0xFFFF0000u);
      x[2][t] = __uint_as_float(v.y << 16);
      x[3][t] = __uint_as_float(v.y & 0xFFFF0000u);
    }
#pragma unroll
    for (int r = 0; r < kWarpRow; ++r) {
      const float4 w = *reinterpret_cast<const float4 *>(ww + st * kTileWBytes + r * 512);
      const float wq[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int t = 0; t < WT; t += 2)
          ffma2_acc(acc[r][t], acc[r][t + 1], x[q][t], x[q][t + 1], wq[q]);
    }
  }

  // the xor butterfly (offsets 16 .. 1) of all 16 WT sums: at each step a lane
  // keeps half of its values and hands the others to its partner; value
  // v = 16 t + r ends on lane v / (WT / 2)
  constexpr int kVals = WT * kWarpRow, kOwn = WT / 2;
  float a[kVals];
#pragma unroll
  for (int v = 0; v < kVals; ++v) a[v] = acc[v % kWarpRow][v / kWarpRow];
  reduce_step<16, kVals / 2>(a, lane);
  reduce_step<8, kVals / 4>(a, lane);
  reduce_step<4, kVals / 8>(a, lane);
  reduce_step<2, kVals / 16>(a, lane);
  reduce_step<1, kVals / 32>(a, lane);
  const int t = t0 + warp * WT + lane * kOwn / kWarpRow, r = r0 + lane * kOwn % kWarpRow;
  if (t < d.B) {
    float *dst = z + (size_t)t * m + r;
    if (kOwn == 4 && (m & 3) == 0 && r + 4 <= m) {
      *reinterpret_cast<float4 *>(dst) = make_float4(a[0], a[1 % kVals], a[2 % kVals], a[3 % kVals]);
    } else {
#pragma unroll
      for (int u = 0; u < kOwn; ++u)
        if (r + u < m) dst[u] = a[u];
    }
  }
}

template <int NC>
__global__ void __launch_bounds__(kRouteThreads)
    route_select_kernel(const int32_t *__restrict__ retained, Dims d, Ws ws,
                        const float *__restrict__ z) {
  __shared__ int32_t ids[kMaxExperts];
  pdl_wait_primary();
  pdl_launch_dependents();
  for (int r = threadIdx.x; r < d.m_ret; r += blockDim.x)
    ids[r] = min(max(retained ? retained[r] : r, 0), d.E - 1);
  if (blockIdx.x == gridDim.x - 1) report_retained(retained, d, ws);
  __syncthreads();
  const int t = blockIdx.x * kRouteWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (t < d.B) topk_token<NC>(z + (size_t)t * d.m_ret, ids, d, ws, t, lane);
#ifdef SLIMWISE_TRACE
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const int tr_step = ws.ctrl[kCtrlTraceStep];
    trace_stamp(ws, tr_step, kTrRouteEnd);
    ws.ctrl[kCtrlTraceStep] = tr_step + 1;
  }
#endif
}

// Which calls take the tiled kernels (where the scratch rows hold the logits).
// Above 256 tokens the cluster kernel's clusters no longer find room all at
// once, and every cluster evaluates the whole pool; below, the second launch
// has to be earned.  Whole layers at H = 2048, cluster kernel / tiled, us:
//   m' = 32    B = 256  64.9 / 65.8    400  70.7 / 70.2    600  85.8 / 79.5
//   m' = 64    B = 256 105.4 / 106.0   304 114.5 / 107.8   500 116.5 / 114.1
//   m' = 128   B = 128 182.0 / 182.8   200 187.6 / 186.5   304 197.5 / 189.4
//   m' = 256   B = 16  101.0 / 101.6    64 206.1 / 204.8   128 239.1 / 237.3
//   m' = 512   B = 4    40.2 / 38.1     32  72.1 / 67.4
//   m' = 1024  B = 1    66.0 / 56.2     16  89.1 / 77.6
// and B = 8192: m' = 128 828 / 727, m' = 256 912 / 747.
inline bool route_tiled(const Dims &d) {
  if ((size_t)d.m_ret * 4 > (size_t)d.k * d.H * 2) return false;
  return d.B > 256 || d.m_ret > 256 ||
         (long long)d.B * d.m_ret >= (d.m_ret > 128 ? 16384 : 24576);
}

cudaError_t launch_route_tiled(const __nv_bfloat16 *hidden, const float *router_w,
                               const int32_t *retained, Dims d, Ws ws, bool pdl, int sms,
                               cudaStream_t stream) {
  // the logits go where the call's expert outputs will be (route_tiled)
  float *z = reinterpret_cast<float *>(ws.y);
  // the smallest tiles that still leave at most one CTA per SM, the largest
  // ones where there are more (m' = 64, tiles of 32, 16 and 8 tokens: B = 256
  // 109.0 / 106.3 / 106.0 us, B = 500 116.5 / 114.1 / 114.2; m' = 128, B = 512
  // 201.2 / 202.5 / 205.0)
  const int row_tiles = (d.m_ret + kTileRow - 1) / kTileRow;
  int wt = 2;
  while (wt < 8 && (d.B + 4 * wt - 1) / (4 * wt) * row_tiles > sms) wt *= 2;
  auto logits = wt == 8 ? route_logits_kernel<8>
                : wt == 4 ? route_logits_kernel<4> : route_logits_kernel<2>;
  cudaError_t err = cudaFuncSetAttribute(logits, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         tile_smem(wt));
  if (err != cudaSuccess) return err;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  cfg.gridDim = dim3((d.B + 4 * wt - 1) / (4 * wt), row_tiles);
  cfg.blockDim = dim3(kTileThreads);
  cfg.dynamicSmemBytes = tile_smem(wt);
  err = cudaLaunchKernelEx(&cfg, logits, hidden, router_w, retained, d, ws, z);
  if (err != cudaSuccess) return err;
  cfg.gridDim = dim3((d.B + kRouteWarps - 1) / kRouteWarps);
  cfg.blockDim = dim3(kRouteThreads);
  cfg.dynamicSmemBytes = 0;
  auto select = d.m_ret <= 128   ? route_select_kernel<4>
                : d.m_ret <= 256 ? route_select_kernel<8>
                                 : route_select_kernel<0>;
  return cudaLaunchKernelEx(&cfg, select, retained, d, ws, (const float *)z);
}

// --------------------------------------------------------------------------
// Large batches on large pools
// --------------------------------------------------------------------------
// Only the k largest logits of a token are used, so there (route_filtered says
// where) the tensor cores bound all of them and the fp32 units evaluate, in the
// canonical order, only those that can be among the k:
//   route_bound_kernel   128 tokens x 128 retained experts per CTA, tcgen05:
//                        the router rows as a sum of two bf16 rows (split when
//                        loaded), fp32 accumulation.  Writes the approximate
//                        logits and the router rows' squared norms to scratch.
//   route_refine_kernel  one warp per token: the k-th largest approximate
//                        logit T (equal ones counted once, which can only lower
//                        it), the canonical logit of every expert whose
//                        approximate one reaches T - 2 b, and the top-k of those.
// b bounds |approximate - canonical| (filter_bound, which says what it assumes
// of the tensor core): k experts have canonical logits of at least T - b, an
// expert left out has less, so the selections, the gates and the order are the
// canonical ones bit for bit.  Where no bound holds (a value that is not finite,
// norms that over- or underflow, fewer than k different logits, a repeated id)
// every logit of the token is evaluated.
// A wait of the bounding kernel that gives up leaves no value (NaN) of its
// tokens' logits and, where it sums them, of its experts' norms, so that no
// token takes a bound from half a norm; the refining kernel reports it.
// The bounding kernel (20 us at 8192 tokens x 128 experts, 33 at 256) waits for
// its loads, the tensor pipe 17-22 % busy; the refining one (43 and 51 us) reads
// k router rows per token from L2 (0.41 and 0.56 GB into the SMs), a few round
// trips a warp with 41 % of the issue slots busy.  More chunks in flight for the
// candidates after the first eight: within 0.5 %.
constexpr int kBoundThreads = 288;          // 8 loading / storing warps, 1 MMA warp
constexpr int kBoundLoaders = 256;
constexpr int kBoundTile = 128;             // tokens, and experts, of a CTA
constexpr int kBoundK = 64;
constexpr int kBoundOperand = kBoundTile * kBoundK * 2;
constexpr int kBoundStages = 4;
constexpr int kBoundParts = 4;              // most shares of K
constexpr int kBoundSmem = kBoundStages * 3 * kBoundOperand + 1024;

// Bound of |approximate - canonical logit| over the product of the norms of the
// hidden and the router row (so of sum |x w|, by Cauchy-Schwarz):
//   2^-17         the part of a weight that neither bf16 term holds (at most
//                 2^-18 of it);
//   (H/8) 2^-21   the tensor core's sum: one step per 16 elements of each term,
//                 allowed 2^-21 of the sum of magnitudes (four units of fp32
//                 truncation) each -- an assumption, since how the unit
//                 rounds its sums is not documented; everything that the
//                 filter claims rests on it;
//   (H/32+6) 2^-23  the canonical sum's own rounding, at least twice over.
// Largest |approximate - exact| seen, of this bound: 0.5 % with normal rows and
// with elements over e^+-6, 4.5 to 6.7 % with rows of one sign (H = 2048 to
// 32768; the tests hold it to 25 %).
__device__ __forceinline__ float filter_bound(int H) {
  return 0x1p-17f + (float)(H / 8) * 0x1p-21f + (float)(H / 32 + 6) * 0x1p-23f;
}

__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c,
                                             uint32_t e) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(e)
               : "memory");
}
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&v);
}

__global__ void __launch_bounds__(kBoundThreads, 1)
    route_bound_kernel(const __nv_bfloat16 *__restrict__ hidden,
                       const float *__restrict__ router_w,
                       const int32_t *__restrict__ retained, Dims d, Ws ws,
                       float *__restrict__ z, float *__restrict__ norm2,
                       int32_t *__restrict__ gave_up, uint64_t timeout_ns, int starve) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bars[2 * kBoundStages + 1];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const uint32_t smem = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kBoundStages + s); };
  const uint32_t done_bar = bar0 + 8u * (2 * kBoundStages);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < kBoundStages; ++s) {
      mbar_init(full_bar(s), kBoundLoaders / 32);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(done_bar, 1);
    abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 8) {
    tmem_alloc(smem_u32(&tmem_slot), kBoundTile);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(&tmem_slot);
  volatile int *abort = &abort_flag;
  pdl_wait_primary();
  pdl_launch_dependents();
#ifdef SLIMWISE_TRACE
  if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) {
    const int tr_step = ws.ctrl[kCtrlTraceStep];
    trace_stamp(ws, tr_step, kTrRouteStart);
    reinterpret_cast<uint64_t *>(ws.ctrl + kCtrlWords)[(tr_step & (kTraceSteps - 1)) * kTrSlots + kTrFfnEnd] = 0;
  }
#endif
  // this CTA's share of K: an even number of blocks (H is a multiple of 128)
  const int H = d.H, m = d.m_ret, nk = H / kBoundK / gridDim.z, k0 = blockIdx.z * nk * kBoundK;
  z += (size_t)blockIdx.z * d.B * m;
  norm2 += (size_t)blockIdx.z * m;
  const int t0 = blockIdx.x * kBoundTile, r0 = blockIdx.y * kBoundTile;

  if (warp < 8) {
    // Each thread carries column block tid % 8 (8 elements) of rows tid / 8 +
    // 32 u of both operands, from global memory through registers (one K block
    // ahead) into the 128-byte swizzled tiles.  Rows past the batch or the
    // pool are zero.
    const int col = tid & 7, row = tid >> 3;
    const __nv_bfloat16 *xsrc[4];
    const float *wsrc[4];
    bool xok[4], wok[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int t = t0 + row + 32 * u, r = r0 + row + 32 * u;
      xok[u] = t < d.B;
      wok[u] = r < m;
      const int rr = wok[u] ? r : 0;
      const int e = min(max(retained ? __ldg(retained + rr) : rr, 0), d.E - 1);
      xsrc[u] = hidden + (size_t)(xok[u] ? t : 0) * H + k0 + col * 8;
      wsrc[u] = router_w + (size_t)e * H + k0 + col * 8;
    }
    struct Block {
      uint4 x[4];
      float4 wa[4], wb[4];
    };
    auto fetch = [&](Block &b, int kc) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        b.x[u] = xok[u] ? __ldg(reinterpret_cast<const uint4 *>(xsrc[u] + kc * kBoundK))
                        : make_uint4(0u, 0u, 0u, 0u);
        const float4 *w = reinterpret_cast<const float4 *>(wsrc[u] + kc * kBoundK);
        b.wa[u] = wok[u] ? __ldg(w) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        b.wb[u] = wok[u] ? __ldg(w + 1) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      }
    };
    float n2[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    auto put = [&](const Block &b, int kc) {
      const int s = kc % kBoundStages;
      const bool got = mbar_wait_bounded(
          empty_bar(s), ((uint32_t)(kc / kBoundStages) & 1u) ^ 1u, abort, timeout_ns);
      if (!__all_sync(0xFFFFFFFFu, got)) {
        *abort = 1;
        return false;
      }
      const uint32_t base = smem + (uint32_t)(s * 3 * kBoundOperand);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int rw = row + 32 * u;
        const uint32_t dst = base + (uint32_t)(rw * 128 + ((col ^ (rw & 7)) * 16));
        const float w[8] = {b.wa[u].x, b.wa[u].y, b.wa[u].z, b.wa[u].w,
                            b.wb[u].x, b.wb[u].y, b.wb[u].z, b.wb[u].w};
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          hi[q] = bf16_pair(w[2 * q], w[2 * q + 1]);
          lo[q] = bf16_pair(w[2 * q] - __uint_as_float(hi[q] << 16),
                            w[2 * q + 1] - __uint_as_float(hi[q] & 0xFFFF0000u));
          n2[u] = fmaf(w[2 * q], w[2 * q], fmaf(w[2 * q + 1], w[2 * q + 1], n2[u]));
        }
        st_shared_v4(dst, b.x[u].x, b.x[u].y, b.x[u].z, b.x[u].w);
        st_shared_v4(dst + kBoundOperand, hi[0], hi[1], hi[2], hi[3]);
        st_shared_v4(dst + 2 * kBoundOperand, lo[0], lo[1], lo[2], lo[3]);
      }
      fence_proxy_async_shared();
      __syncwarp();
      if (lane == 0) mbar_arrive(full_bar(s));
      return true;
    };
    // two K blocks in flight
    Block even, odd;
    fetch(even, 0);
    fetch(odd, 1);
    bool ok = true;
    for (int kc = 0; kc < nk; kc += 2) {
      ok = put(even, kc);
      if (!ok) break;
      if (kc + 2 < nk) fetch(even, kc + 2);
      ok = put(odd, kc + 1);
      if (!ok) break;
      if (kc + 3 < nk) fetch(odd, kc + 3);
    }
    // squared norms of the router rows, once per row (none of rows that this
    // warp has not seen to the end)
    if (blockIdx.x == 0) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float v = n2[u];
#pragma unroll
        for (int off = 1; off < 8; off <<= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
        if (col == 0 && wok[u]) norm2[r0 + row + 32 * u] = ok ? v : __uint_as_float(0x7FC00000u);
      }
    }
    // accumulator rows 32 q .. (tokens), columns 64 h .. (experts)
    if (ok) ok = mbar_wait_bounded(done_bar, 0u, abort, timeout_ns);
    ok = __all_sync(0xFFFFFFFFu, ok && !*abort) != 0;
    if (!ok) *abort = 1;
    tc_fence_after();
    const int q = warp & 3, c_first = (warp >> 2) * 64;
#pragma unroll
    for (int c = 0; c < 64; c += 32) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t v[16];
        tmem_ld_frag(tmem + ((uint32_t)(32 * q + 16 * h) << 16) + (uint32_t)(c_first + c), v);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          // values 2i, 2i + 1: column block i / 2, row half i % 2
          const int t = t0 + 32 * q + 16 * h + 8 * (i & 1) + (lane >> 2);
          const int r = r0 + c_first + c + 8 * (i >> 1) + 2 * (lane & 3);
          // a wait that gave up: no value, so every logit is evaluated
          const float a = ok ? __uint_as_float(v[2 * i]) : __uint_as_float(0x7FC00000u);
          const float b = ok ? __uint_as_float(v[2 * i + 1]) : __uint_as_float(0x7FC00000u);
          if (t < d.B) {
            float *dst = z + (size_t)t * m + r;
            if ((m & 1) == 0 && r + 1 < m) {
              *reinterpret_cast<float2 *>(dst) = make_float2(a, b);
            } else {
              if (r < m) dst[0] = a;
              if (r + 1 < m) dst[1] = b;
            }
          }
        }
      }
    }
    tc_fence_before();
  } else {
    const uint32_t idesc = idesc_bf16_f32(kBoundTile, kBoundTile);
    int issued = 0;
    // tests only: the first CTA multiplies nothing, so the waits of its loading
    // warps run out
    const bool starved = starve && (blockIdx.x | blockIdx.y | blockIdx.z) == 0;
    for (int kc = 0; kc < nk && !starved; ++kc) {
      const int s = kc % kBoundStages;
      if (!__all_sync(0xFFFFFFFFu, mbar_wait_bounded(full_bar(s), (uint32_t)(kc / kBoundStages) & 1u,
                                                     abort, timeout_ns))) {
        *abort = 1;
        __threadfence_block();
        break;
      }
      tc_fence_after();
      const uint32_t a = smem + (uint32_t)(s * 3 * kBoundOperand);
      if (elect_one()) {
#pragma unroll
        for (int term = 1; term <= 2; ++term)
#pragma unroll
          for (int kk = 0; kk < kBoundK / 16; ++kk)
            tc_mma_bf16(tmem, smem_desc_sw128(a + kk * 32),
                        smem_desc_sw128(a + term * kBoundOperand + kk * 32), idesc,
                        (kc > 0 || term > 1 || kk > 0) ? 1u : 0u);
        tc_commit(empty_bar(s));
      }
      __syncwarp();
      ++issued;
    }
    // the accumulator is complete (after a wait that gave up: nothing of this
    // CTA's is in flight any more)
    if (issued > 0) {
      if (elect_one()) tc_commit(done_bar);
      __syncwarp();
      mbar_wait_timeout(done_bar, 0u, 10000000ull);
    }
  }
  __syncthreads();
  if (tid == 0)
    gave_up[(blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = *abort ? 1 : 0;
  if (warp == 8) {
    tc_fence_after();
    tmem_dealloc(tmem, kBoundTile);
  }
}

// Canonical logits (see the head of this file) of N experts for one token, by
// one warp; every lane gets them.
template <int N>
__device__ __forceinline__ void canonical_logits(const __nv_bfloat16 *__restrict__ x,
                                                 const float *const (&w)[N], int H, int lane,
                                                 float (&p)[N]) {
#pragma unroll
  for (int j = 0; j < N; ++j) p[j] = 0.0f;
#pragma unroll 2
  for (int c = 0; c < H / 128; ++c) {
    const int h = 128 * c + 4 * lane;
    const uint2 xv = __ldg(reinterpret_cast<const uint2 *>(x + h));
    const float xf[4] = {__uint_as_float(xv.x << 16), __uint_as_float(xv.x & 0xFFFF0000u),
                         __uint_as_float(xv.y << 16), __uint_as_float(xv.y & 0xFFFF0000u)};
    float4 wv[N];
#pragma unroll
    for (int j = 0; j < N; ++j) wv[j] = __ldg(reinterpret_cast<const float4 *>(w[j] + h));
#pragma unroll
    for (int j = 0; j < N; ++j) {
      p[j] = fmaf(xf[0], wv[j].x, p[j]);
      p[j] = fmaf(xf[1], wv[j].y, p[j]);
      p[j] = fmaf(xf[2], wv[j].z, p[j]);
      p[j] = fmaf(xf[3], wv[j].w, p[j]);
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
#pragma unroll
    for (int j = 0; j < N; ++j) p[j] += __shfl_xor_sync(0xFFFFFFFFu, p[j], off);
}
// ... of the experts cand[0, N), into exact[0, N).
template <int N>
__device__ __forceinline__ void refine(const int32_t *cand, const __nv_bfloat16 *__restrict__ x,
                                       const float *__restrict__ router_w, int H, int lane,
                                       float *exact) {
  const float *w[N];
#pragma unroll
  for (int j = 0; j < N; ++j) w[j] = router_w + (size_t)cand[j] * H;
  float p[N];
  canonical_logits<N>(x, w, H, lane, p);
#pragma unroll
  for (int j = 0; j < N; ++j)
    if (lane == j) exact[j] = p[j];
}

// NC: 32 NC >= m'.  Registers for 4 CTAs on an SM, so that 4001 tokens x 128
// experts are one wave (78 of them: 390.5 -> 395.0 us a layer), or for 3 with the
// larger pool (2048 tokens: 363.2 us, 372.2 with 4).  The top-k runs over the
// candidates alone, one per lane where they are at most 32, and T comes from
// values, not from (value, id) pairs: 8192 tokens x 256 experts 725 -> 715 us.
template <int NC>
__global__ void __launch_bounds__(kRouteThreads, NC == 4 ? 4 : 3)
    route_refine_kernel(const __nv_bfloat16 *__restrict__ hidden,
                        const float *__restrict__ router_w,
                        const int32_t *__restrict__ retained, Dims d, Ws ws,
                        const float *__restrict__ z, const float *__restrict__ norm2, int parts,
                        const int32_t *__restrict__ gave_up, int bound_ctas) {
  __shared__ int32_t ids[32 * NC];
  __shared__ float exact[kRouteWarps][32 * NC];
  __shared__ int32_t cand[kRouteWarps][32 * NC];
  __shared__ uint32_t wmax, seen[kMaxExperts / 32];
  __shared__ int repeated;  // an id is listed twice
  if (threadIdx.x == 0) wmax = 0u, repeated = 0;
  if (threadIdx.x < kMaxExperts / 32) seen[threadIdx.x] = 0u;
  pdl_wait_primary();
  pdl_launch_dependents();
  const int m = d.m_ret, H = d.H, k = d.k;
  const int wi = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.x * kRouteWarps + wi;
  const __nv_bfloat16 *x = hidden + (size_t)min(t, d.B - 1) * H;
  // this lane's approximate logits (the sum of their parts) and the token's
  // squared norm: every load of the parts is issued before any is used
  float part[kBoundParts][NC], zc[NC];
#pragma unroll
  for (int p = 0; p < kBoundParts; ++p)
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      const int r = lane + 32 * i;
      part[p][i] = p < parts && r < m ? z[((size_t)p * d.B + min(t, d.B - 1)) * m + r] : 0.0f;
    }
  float x2 = 0.0f;
#pragma unroll 8
  for (int c = 0; c < H / 128; ++c) {
    const uint2 xv = __ldg(reinterpret_cast<const uint2 *>(x + 128 * c + 4 * lane));
    const float a = __uint_as_float(xv.x << 16), b = __uint_as_float(xv.x & 0xFFFF0000u);
    const float e = __uint_as_float(xv.y << 16), f = __uint_as_float(xv.y & 0xFFFF0000u);
    x2 = fmaf(a, a, fmaf(b, b, fmaf(e, e, fmaf(f, f, x2))));
  }
  for (int r = threadIdx.x; r < m; r += blockDim.x)
    ids[r] = min(max(retained ? retained[r] : r, 0), d.E - 1);
  if (blockIdx.x == gridDim.x - 1) {
    int timeout = 0;  // any bounding CTA's wait
    for (int i = threadIdx.x; i < bound_ctas; i += blockDim.x)
      if (gave_up[i]) timeout = SLIMWISE_DEVERR_PIPELINE_TIMEOUT;
    report_retained(retained, d, ws, timeout);
  }
  __syncthreads();
  // largest squared norm of the router rows, as bits: above every finite value
  // where one is infinite or NaN
  {
    uint32_t v = 0u;
    for (int r = threadIdx.x; r < m; r += blockDim.x) {
      float s = 0.0f;
#pragma unroll
      for (int p = 0; p < kBoundParts; ++p) s += p < parts ? norm2[(size_t)p * m + r] : 0.0f;
      v = max(v, __float_as_uint(s));
      const uint32_t bit = 1u << (ids[r] & 31);
      if (atomicOr(&seen[ids[r] >> 5], bit) & bit) repeated = 1;
    }
    v = __reduce_max_sync(0xFFFFFFFFu, v);
    if (lane == 0) atomicMax(&wmax, v);
  }
  __syncthreads();
  if (t < d.B) {
    bool bad = repeated != 0;
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      zc[i] = part[0][i];
#pragma unroll
      for (int p = 1; p < kBoundParts; ++p) zc[i] += part[p][i];
      bad |= !(fabsf(zc[i]) < __uint_as_float(0x7F800000u));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x2 += __shfl_xor_sync(0xFFFFFFFFu, x2, off);
    // product of the norms (0.2 % up for the sums' rounding and underflow)
    const float w2 = __uint_as_float(wmax);
    const float prod = sqrtf(x2) * sqrtf(w2) * 1.002f;
    bad |= !(x2 > 1e-24f && x2 < 1e36f && w2 > 1e-24f && w2 < 1e36f && prod < 1e36f);
    // T: the k-th largest distinct value, so at most the k-th largest logit
    uint32_t left[NC], win = 0u;  // order bits of the values not taken yet, 0 = none
#pragma unroll
    for (int i = 0; i < NC; ++i) left[i] = lane + 32 * i < m ? logit_order_bits(zc[i]) : 0u;
    for (int j = 0; j < k; ++j) {
      uint32_t best = left[0];
#pragma unroll
      for (int i = 1; i < NC; ++i) best = max(best, left[i]);
      win = __reduce_max_sync(0xFFFFFFFFu, best);
#pragma unroll
      for (int i = 0; i < NC; ++i) left[i] = left[i] == win ? 0u : left[i];
    }
    bad |= win == 0u;
    const bool all = __any_sync(0xFFFFFFFFu, bad) != 0;
    const float least = logit_from_order_bits(win) - 2.02f * filter_bound(H) * prod;
    int n = 0;
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      const int r = lane + 32 * i;
      const bool c = r < m && (all || zc[i] >= least);
      const uint32_t mask = __ballot_sync(0xFFFFFFFFu, c);
      if (c) cand[wi][n + __popc(mask & ((1u << lane) - 1u))] = ids[r];
      n += __popc(mask);
    }
    __syncwarp();
    int j = 0;
    for (; j + 8 <= n; j += 8) refine<8>(cand[wi] + j, x, router_w, H, lane, exact[wi] + j);
    for (; j + 2 <= n; j += 2) refine<2>(cand[wi] + j, x, router_w, H, lane, exact[wi] + j);
    if (j < n) refine<1>(cand[wi] + j, x, router_w, H, lane, exact[wi] + j);
    __syncwarp();
    Dims dn = d;
    dn.m_ret = n;
    if (n <= 32) topk_token<1>(exact[wi], cand[wi], dn, ws, t, lane);
    else topk_token<NC>(exact[wi], cand[wi], dn, ws, t, lane);
  }
#ifdef SLIMWISE_TRACE
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const int tr_step = ws.ctrl[kCtrlTraceStep];
    trace_stamp(ws, tr_step, kTrRouteEnd);
    ws.ctrl[kCtrlTraceStep] = tr_step + 1;
  }
#endif
}

// Which calls take the filtered kernels (where the scratch rows hold `parts`
// approximate logits).  The refining work grows with k, the full product with
// m', and the two kernels' latency (about 20 us) has to be earned.  Whole
// layers at H = 2048, k = 8, full product / filtered, us:
//   m' = 32    B = 8192 594.6 / 610.9     m' = 64   B = 8192 630.9 / 636.5
//   m' = 96    B = 5000 451.4 / 452.5
//   m' = 128   B = 1536 247.4 / 250.0    2048 275.5 / 273.4   2560 304.1 / 297.9
//              3000 328.8 / 320.0   4001 411.6 / 390.6   8192 718.1 / 681.5
//   m' = 192   B = 4096 436.4 / 410.9
//   m' = 256   B =  768 303.3 / 306.2    1024 317.7 / 312.6   1536 358.1 / 347.7
//              2048 389.7 / 363.2   4096 517.5 / 464.6   8192 825.2 / 715.2
// Routing and grouping alone, at the smallest batch of the rule, half as many
// again, twice that batch and 8192, H = 512-8192, m' = 128-256, k = 1-16: 0.28
// to 0.99 of the full product's time, but for H = 8192 at the smallest batch
// with m' = 16 k (113.2 / 116.8, 116.4 / 121.2).
inline bool filtered_fits(const Dims &d, int parts) {
  return (size_t)parts * (d.B + 1) * d.m_ret * 4 <= (size_t)d.B * d.k * d.H * 2;
}
inline bool route_filtered(const Dims &d) {
  const long long bm = (long long)d.B * d.m_ret;
  return d.m_ret >= 128 && d.m_ret >= 16 * d.k && d.m_ret <= 256 && bm >= (1ll << 18) &&
         bm * d.H >= (1ll << 29) && filtered_fits(d, 1);
}

cudaError_t launch_route_filtered(const __nv_bfloat16 *hidden, const float *router_w,
                                  const int32_t *retained, Dims d, Ws ws, bool pdl, int sms,
                                  cudaStream_t stream, uint64_t timeout_ns, int starve) {
  // approximate logits, then the router rows' norms, where the call's expert
  // outputs will be
  float *z = reinterpret_cast<float *>(ws.y);
  // K in 2 or 4 parts while they leave at most one CTA per SM (each writes its
  // own approximate logits): 4001 tokens x 128 experts 410.9 us a layer with
  // one part, 398.6 with two, 392.9 with four, 392.8 with eight
  const int tiles = ((d.B + kBoundTile - 1) / kBoundTile) * ((d.m_ret + kBoundTile - 1) / kBoundTile);
  int parts = 1;
  while (parts < kBoundParts && 2 * parts * tiles <= sms && d.H / 128 % (2 * parts) == 0 &&
         filtered_fits(d, 2 * parts))
    parts *= 2;
  float *norm2 = z + (size_t)parts * d.B * d.m_ret;
  // one word per bounding CTA (at most B / 16 + 8) where the call's activations
  // will be (at least 32 words a token)
  int32_t *gave_up = reinterpret_cast<int32_t *>(ws.act);
  cudaError_t err = cudaFuncSetAttribute(
      route_bound_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBoundSmem);
  if (err != cudaSuccess) return err;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  cfg.gridDim = dim3((d.B + kBoundTile - 1) / kBoundTile, (d.m_ret + kBoundTile - 1) / kBoundTile, parts);
  cfg.blockDim = dim3(kBoundThreads);
  cfg.dynamicSmemBytes = kBoundSmem;
  err = cudaLaunchKernelEx(&cfg, route_bound_kernel, hidden, router_w, retained, d, ws, z, norm2,
                           gave_up, timeout_ns, starve);
  if (err != cudaSuccess) return err;
  cfg.gridDim = dim3((d.B + kRouteWarps - 1) / kRouteWarps);
  cfg.blockDim = dim3(kRouteThreads);
  cfg.dynamicSmemBytes = 0;
  auto refine = d.m_ret <= 128 ? route_refine_kernel<4> : route_refine_kernel<8>;
  return cudaLaunchKernelEx(&cfg, refine, hidden, router_w, retained, d, ws, (const float *)z,
                            (const float *)norm2, parts, (const int32_t *)gave_up, tiles * parts);
}

cudaError_t launch_route_topk(const __nv_bfloat16 *hidden, const float *router_w,
                              const int32_t *retained, Dims d, Ws ws, bool pdl,
                              cudaStream_t stream, uint64_t timeout_ns, int starve_bound) {
  int dev = 0, optin = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  const bool filtered = route_filtered(d);
  if (filtered || route_tiled(d)) {
    int sms = 0;
    err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (err != cudaSuccess) return err;
    return filtered ? launch_route_filtered(hidden, router_w, retained, d, ws, pdl, sms, stream,
                                            timeout_ns, starve_bound)
                    : launch_route_tiled(hidden, router_w, retained, d, ws, pdl, sms, stream);
  }
  err = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (err != cudaSuccess) return err;
  const size_t max_smem = (size_t)optin - kRouteStaticSmem;
  // wide hidden rows: fewer tokens per cluster until they fit in shared memory
  int tb = route_tokens_per_cluster(d.B, d.m_ret);
  auto fits = [&](int t) {
    const size_t need = t == 16 ? route_smem_bytes<16>(d) : t == 8 ? route_smem_bytes<8>(d)
                      : t == 4 ? route_smem_bytes<4>(d) : t == 2 ? route_smem_bytes<2>(d)
                      : route_smem_bytes<1>(d);
    return need <= max_smem;
  };
  while (tb > 1 && !fits(tb)) tb >>= 1;
  auto launch = tb == 1   ? launch_route_nc<1>
                : tb == 2 ? launch_route_nc<2>
                : tb == 4 ? launch_route_nc<4>
                : tb == 8 ? launch_route_nc<8>
                          : launch_route_nc<16>;
  return launch(hidden, router_w, retained, d, ws, pdl, max_smem, stream);
}

}  // namespace slimwise
