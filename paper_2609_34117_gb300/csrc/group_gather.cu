// group_gather.cu -- grouping of the B*k routed (token, slot) pairs by expert
// and gather of the hidden rows into that grouped order.
//
// A decode step must read the weights of the union of experts selected
// across the batch (SlimWise Sec. 2.1, Eq. 1).  This kernel turns the top-k
// selections into:
//   counts[e]  histogram of selections,
//   offsets    exclusive scan of counts (expert ascending),
//   union_ids  selected experts ascending, union size U,
//   perm/pos   grouped order of the slots: (expert asc, token asc),
//   entries    the FFN kernel's work list: one entry per (expert, chunk of
//              at most tok_chunk tokens),
//   xp         hidden rows copied into grouped order, so the FFN kernel can
//              stream each expert's tokens with plain 2-D TMA boxes.
// With a shared expert (Sec. 3.3) it also computes each token's sigmoid gate
// s_t = 1 / (1 + exp(-w_sg . x_t)), the dot product in the canonical order of
// the router logits, and lists the shared expert's work entries (the batch in
// token order, in chunks) ahead of the routed ones.
// Every CTA recomputes the histogram of the whole batch (B*k ids, a few KB
// from L2) so the rank of a slot inside its expert, its token-order prefix
// count, is known without a grid-wide barrier; integer counts make the
// result independent of atomic arrival order.
#include "common.cuh"

namespace slimwise {

// Layers of at most 96 tokens do without this kernel (expert_ffn.cu), except
// for statistics, pair items and routing-only calls.
//
// Tokens per CTA: one up to 64 tokens (only the calls above come here with so
// few), two above.  Fewer tokens per CTA spread the grouped-row copy over more
// SMs (one against two at 4-64 tokens: 0.1-0.2 us of a routing-only call,
// 0.2-0.7 us of a calibration batch or a layer of pair items), but every CTA
// recounts the whole batch's selections, and above 64 tokens the extra CTAs
// cost more (B = 256: 0.9 us, B = 512: 2 us a step); four per CTA was slower at
// every size.
inline int group_tokens_per_cta(int B) { return B <= 64 ? 1 : 2; }
constexpr int kGroupThreads = 512;
// Batches from here on take the tiled kernels below (whole layers, one kernel
// against tiled: m' = 32, B = 512 75.8 / 77.4 us, 640 84.9 / 84.9, 768 92.1 /
// 91.8, 1024 116.9 / 113.9; m' = 128, B = 1024 225.3 / 223.0).
constexpr int kGroupTiledMin = 768;

// Exclusive scans over the experts of the selections cnt[e], of the union flags
// and of the work entries (ceil(cnt / tok_chunk)) into offs, flags and entries
// (totals at [E]), by all warps of the CTA: each takes chunks of 32 experts,
// sums the experts before its chunk by itself and scans its own, so the stage
// is one pass between two block barriers whatever the pool.  (One warp per
// scan, each lane walking E / 32 neighbours, was 0.5 us slower a step at 128
// experts.)
__device__ __forceinline__ void scan_pool(const int *cnt, int E, int tok_chunk, int *offs,
                                          int *flags, int *entries) {
  const int lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  const float inv = 1.0f / (float)tok_chunk;
  auto entries_of = [&](int n) { return entry_count(n, tok_chunk, inv); };
  for (int c = threadIdx.x >> 5; 32 * c < E; c += nwarps) {
    int n0 = 0, f0 = 0, e0 = 0;
    for (int e = lane; e < 32 * c; e += 32) {
      const int n = cnt[e];
      n0 += n;
      f0 += n > 0 ? 1 : 0;
      e0 += entries_of(n);
    }
    n0 = __reduce_add_sync(0xFFFFFFFFu, n0);
    f0 = __reduce_add_sync(0xFFFFFFFFu, f0);
    e0 = __reduce_add_sync(0xFFFFFFFFu, e0);
    const int e = 32 * c + lane;
    const int n = e < E ? cnt[e] : 0, m = entries_of(n);
    const uint32_t in = __ballot_sync(0xFFFFFFFFu, n > 0);
    int sn = n, sm = m;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int on = __shfl_up_sync(0xFFFFFFFFu, sn, off);
      const int om = __shfl_up_sync(0xFFFFFFFFu, sm, off);
      if (lane >= off) {
        sn += on;
        sm += om;
      }
    }
    if (e < E) {
      const int f = f0 + __popc(in & ((1u << lane) - 1u));
      offs[e] = n0 + sn - n;
      flags[e] = f;
      entries[e] = e0 + sm - m;
      if (e == E - 1) {
        offs[E] = n0 + sn;
        flags[E] = f + (n > 0 ? 1 : 0);
        entries[E] = e0 + sm;
      }
    }
  }
}

// The batch-wide results and the FFN work list, each expert written by one of
// the grid's gstride threads.  cnt[e] selections, offs/flag_scan/entry_base
// the exclusive scans (with totals at [E]) of the counts, of the union flags
// and of the work-entry counts.  Entries [0, S) are the shared expert's
// (expert -1, token order); the routed ones follow.
__device__ __forceinline__ void publish_groups(const Dims &d, const Ws &ws, const int *cnt,
                                               const int *offs, const int *flag_scan,
                                               const int *entry_base, int gtid, int gstride) {
  const int E = d.E, B = d.B;
  const int U = flag_scan[E];
  const int n_entries = entry_base[E];
  const int n_se = d.S;
  for (int e = gtid; e < E; e += gstride) {
    const int n_e = cnt[e];
    ws.counts[e] = n_e;
    ws.offsets[e] = offs[e];
    if (n_e > 0) ws.union_ids[flag_scan[e]] = e;
    if (e >= U) ws.union_ids[e] = -1;
    const int per = entry_tokens(n_e, d.tok_chunk);
    for (int c = 0; c < entry_base[e + 1] - entry_base[e]; ++c) {
      const int base = c * per;
      ws.entries[n_se + entry_base[e] + c] = make_int4(e, offs[e] + base, min(per, n_e - base), 0);
    }
  }
  for (int sidx = gtid; sidx < n_se; sidx += gstride)
    ws.entries[sidx] = make_int4(-1, sidx * d.tok_chunk, min(d.tok_chunk, B - sidx * d.tok_chunk), 0);
  for (int i = gtid; i < n_se + n_entries; i += gstride) ws.entry_done[i] = 0;
  if (gtid == 0) {
    const int t1_items = gate_up_tiles(d);
    const int t2_items = down_tiles(d);
    const int t1s_items = shared_gate_up_tiles(d);
    ws.offsets[E] = offs[E];
    ws.ctrl[kCtrlUnionSize] = U;
    ws.ctrl[kCtrlNumEntries] = n_se + n_entries;
    ws.ctrl[kCtrlItems1] = n_entries * t1_items;
    ws.ctrl[kCtrlTotalItems] = n_se * (t1s_items + t2_items) + n_entries * (t1_items + t2_items);
    ws.ctrl[kCtrlWorkCounter] = 0;
  }
}

template <int kGroupTokens>
__global__ void __launch_bounds__(kGroupThreads)
    group_gather_kernel(const __nv_bfloat16 *__restrict__ hidden,
                        const float *__restrict__ w_sg, Dims d, Ws ws, int do_gather) {
  __shared__ int cnt_all[kMaxExperts];
  __shared__ int cnt_before[kMaxExperts];
  __shared__ int offs[kMaxExperts + 1];
  __shared__ int flag_scan[kMaxExperts + 1];
  __shared__ int entry_base[kMaxExperts + 1];
  __shared__ int my_pos[kGroupTokens * kMaxTopK];
  __shared__ int my_ids[kGroupTokens * kMaxTopK];
  __shared__ int bad;

  for (int e = threadIdx.x; e < d.E; e += blockDim.x) {
    cnt_all[e] = 0;
    cnt_before[e] = 0;
  }
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();

  // Wait for the routing kernel's results; then let the FFN kernel's CTAs
  // start their prologue.
  pdl_wait_primary();
  pdl_launch_dependents();
#ifdef SLIMWISE_TRACE
  const int tr_step = ws.ctrl[kCtrlTraceStep] - 1;
  if (blockIdx.x == 0 && threadIdx.x == 0) trace_stamp(ws, tr_step, kTrGroupStart);
#endif

  const int B = d.B, k = d.k, E = d.E, H = d.H;
  const int S = B * k;
  const int t0 = blockIdx.x * kGroupTokens;
  const int t1 = min(B, t0 + kGroupTokens);
  const int nt = t1 - t0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int vecs = H / 8;  // 16-byte vectors per hidden row

  // This CTA's hidden rows go into registers first, so that their loads
  // overlap the histogram below (up to kPre vectors per thread).
  constexpr int kPre = 4;
  const bool early = do_gather && nt * vecs <= kPre * (int)blockDim.x;
  uint4 hv[kPre];
  if (early) {
#pragma unroll
    for (int u = 0; u < kPre; ++u) {
      const int i = tid + u * blockDim.x;
      if (i < nt * vecs)
        hv[u] = __ldg(reinterpret_cast<const uint4 *>(hidden + (size_t)(t0 + i / vecs) * H) + i % vecs);
    }
  }

  const int nslots = nt * k;
  // each thread's selections are loaded together, then counted
  constexpr int kHistBatch = 8;
  for (int s0 = tid; s0 < S; s0 += kHistBatch * blockDim.x) {
    int ev[kHistBatch];
#pragma unroll
    for (int u = 0; u < kHistBatch; ++u) {
      const int s = s0 + u * blockDim.x;
      ev[u] = s < S ? ws.topk_idx[s] : 0;
    }
#pragma unroll
    for (int u = 0; u < kHistBatch; ++u) {
      const int s = s0 + u * blockDim.x;
      if (s < S) {
        int e = ev[u];
        if (e < 0 || e >= E) {  // only possible for caller-given selections
          bad = SLIMWISE_DEVERR_BAD_TOPK;
          e = min(max(e, 0), E - 1);
        }
        atomicAdd(&cnt_all[e], 1);
        if (s < t0 * k) atomicAdd(&cnt_before[e], 1);
        else if (s < t1 * k) my_ids[s - t0 * k] = e;
      }
    }
  }
  __syncthreads();
  // offsets of the experts, the union and the work entries (every CTA has the
  // whole histogram, so each can publish its share of the results)
  scan_pool(cnt_all, E, d.tok_chunk, offs, flag_scan, entry_base);
  __syncthreads();

  // Grouped position of each of this CTA's slots: offset of the expert plus
  // the number of earlier tokens that selected it (tokens before this CTA's
  // range, then earlier tokens of the range).
  for (int i = tid; i < nslots; i += blockDim.x) {
    const int e = my_ids[i];
    int rank = cnt_before[e];
    for (int s = 0; s < (i / k) * k; ++s) rank += (my_ids[s] == e) ? 1 : 0;
    const int s = t0 * k + i, p = offs[e] + rank;
    my_pos[i] = p;
    ws.pos[s] = p;
    ws.perm[p] = s;
  }
  __syncthreads();
  if (early) {
    // each token row, already in registers, goes to its k grouped positions
#pragma unroll
    for (int u = 0; u < kPre; ++u) {
      const int i = tid + u * blockDim.x;
      if (i < nt * vecs) {
        const int tt = i / vecs, vv = i % vecs;
        for (int j = 0; j < k; ++j)
          reinterpret_cast<uint4 *>(ws.xp + (size_t)my_pos[tt * k + j] * H)[vv] = hv[u];
      }
    }
  } else if (do_gather) {
    // wide rows: loaded here, four vectors per thread in flight
    constexpr int kVec = 4;
    for (int i0 = tid; i0 < nt * vecs; i0 += kVec * blockDim.x) {
      uint4 v[kVec];
      int tt[kVec], vv[kVec];
#pragma unroll
      for (int u = 0; u < kVec; ++u) {
        const int i = i0 + u * blockDim.x;
        tt[u] = i / vecs;
        vv[u] = i - tt[u] * vecs;
        if (i < nt * vecs)
          v[u] = __ldg(reinterpret_cast<const uint4 *>(hidden + (size_t)(t0 + tt[u]) * H) + vv[u]);
      }
#pragma unroll
      for (int u = 0; u < kVec; ++u) {
        if (i0 + u * blockDim.x < nt * vecs) {
          for (int j = 0; j < k; ++j)
            reinterpret_cast<uint4 *>(ws.xp + (size_t)my_pos[tt[u] * k + j] * H)[vv[u]] = v[u];
        }
      }
    }
  }
  // shared-expert gate of this CTA's tokens: warp w takes token t0 + w
  if (d.Is > 0 && warp < nt) shared_gate_token(hidden, w_sg, d, ws, t0 + warp, lane);

  publish_groups(d, ws, cnt_all, offs, flag_scan, entry_base, blockIdx.x * blockDim.x + tid,
                 gridDim.x * blockDim.x);
  __syncthreads();
  if (blockIdx.x == 0 && tid == 0 && bad) atomicOr(&ws.ctrl[kCtrlErr], bad);
#ifdef SLIMWISE_TRACE
  if (blockIdx.x == 0 && tid == 0) trace_stamp(ws, tr_step, kTrGroupEnd);
#endif
}

// --------------------------------------------------------------------------
// Large batches
// --------------------------------------------------------------------------
// The kernel above recounts the whole batch in every CTA, work that grows with
// B^2: 42 us at B = 2048 (now 20) and 312 us at B = 8192 (Qwen3.6-shaped
// layer, now 80).  From
// kGroupTiledMin tokens on, two kernels do the same with work linear in B:
//   group_count_kernel  the histogram of each tile of the batch (at most
//                       kGroupTiles tiles of 128 tokens or a multiple), one
//                       CTA per tile;
//   group_place_kernel  a CTA per part of a tile sums the tiles' histograms
//                       (a few hundred KB from L2) into the experts' offsets
//                       and its tile's base in each expert, ranks the tile's
//                       slots by expert with one bit mask per (expert, 32
//                       tokens), and copies its part's hidden rows out.
// The copy (B k H bf16 written) is then what bounds the stage.
constexpr int kGroupTiles = 64;       // most tiles of the batch
constexpr int kGroupTile = 128;       // tokens ranked together
constexpr int kTileWords = kGroupTile / 32;

// Blocks of 128 tokens per tile, and tiles of the batch.
__host__ __device__ inline int group_tile_blocks(int B) {
  return (B + kGroupTile * kGroupTiles - 1) / (kGroupTile * kGroupTiles);
}
__host__ __device__ inline int group_tile_count(int B) {
  const int tile = kGroupTile * group_tile_blocks(B);
  return (B + tile - 1) / tile;
}

__device__ __forceinline__ int checked_id(int e, int E, int *bad) {
  if (e < 0 || e >= E) {  // only possible for caller-given selections
    *bad = SLIMWISE_DEVERR_BAD_TOPK;
    e = min(max(e, 0), E - 1);
  }
  return e;
}

// tile_cnt[tile][e]: selections of expert e by the tile's tokens.
__global__ void __launch_bounds__(kGroupThreads)
    group_count_kernel(Dims d, Ws ws, int32_t *__restrict__ tile_cnt) {
  __shared__ int cnt[kMaxExperts];
  __shared__ int bad;
  for (int e = threadIdx.x; e < d.E; e += blockDim.x) cnt[e] = 0;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  pdl_wait_primary();
  pdl_launch_dependents();
#ifdef SLIMWISE_TRACE
  if (blockIdx.x == 0 && threadIdx.x == 0)
    trace_stamp(ws, ws.ctrl[kCtrlTraceStep] - 1, kTrGroupStart);
#endif
  const int tile = kGroupTile * group_tile_blocks(d.B);
  const int s0 = blockIdx.x * tile * d.k, s1 = min(d.B, (int)(blockIdx.x + 1) * tile) * d.k;
  for (int s = s0 + threadIdx.x; s < s1; s += blockDim.x)
    atomicAdd(&cnt[checked_id(ws.topk_idx[s], d.E, &bad)], 1);
  __syncthreads();
  for (int e = threadIdx.x; e < d.E; e += blockDim.x)
    tile_cnt[(size_t)blockIdx.x * d.E + e] = cnt[e];
  if (threadIdx.x == 0 && bad) atomicOr(&ws.ctrl[kCtrlErr], bad);
}

// blockIdx.x = tile, blockIdx.y = part: tokens [y part, (y + 1) part) of every
// 128-token block of the tile.  Dynamic shared memory: see place_smem.
__global__ void __launch_bounds__(kGroupThreads)
    group_place_kernel(const __nv_bfloat16 *__restrict__ hidden, const float *__restrict__ w_sg,
                       Dims d, Ws ws, const int32_t *__restrict__ tile_cnt, int part,
                       int do_gather) {
  extern __shared__ int gsm[];
  const int B = d.B, k = d.k, E = d.E, H = d.H;
  int *total = gsm;                    // [E] selections in the batch
  int *base = total + E;               // [E] next grouped position of this tile
  int *offs = base + E;                // [E + 1]
  int *flag = offs + E + 1;            // [E + 1] scan of the union flags
  int *chunks = flag + E + 1;          // [E + 1] scan of the work entries
  uint32_t *mask = reinterpret_cast<uint32_t *>(chunks + E + 1);  // [E][kTileWords]
  int *pos_s = reinterpret_cast<int *>(mask + (size_t)E * kTileWords);  // [part][k]

  pdl_wait_primary();
  pdl_launch_dependents();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int T = gridDim.x;
  const int blocks = group_tile_blocks(B);
  const int vecs = H / 8;

  for (int e = tid; e < E; e += blockDim.x) {
    int before = 0, all = 0;
    constexpr int kBatch = 16;
    for (int c0 = 0; c0 < T; c0 += kBatch) {
      int v[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u)
        v[u] = c0 + u < T ? __ldcg(tile_cnt + (size_t)(c0 + u) * E + e) : 0;
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        all += v[u];
        if (c0 + u < (int)blockIdx.x) before += v[u];
      }
    }
    total[e] = all;
    base[e] = before;
  }
  __syncthreads();
  scan_pool(total, E, d.tok_chunk, offs, flag, chunks);
  __syncthreads();
  for (int e = tid; e < E; e += blockDim.x) base[e] += offs[e];

  for (int b = 0; b < blocks; ++b) {
    const int t0 = ((int)blockIdx.x * blocks + b) * kGroupTile;
    if (t0 >= B) break;
    const int nt = min(kGroupTile, B - t0);
    for (int i = tid; i < E * kTileWords; i += blockDim.x) mask[i] = 0u;
    __syncthreads();
    for (int i = tid; i < nt * k; i += blockDim.x) {
      const int e = min(max(ws.topk_idx[(size_t)t0 * k + i], 0), E - 1);
      const int t = i / k;
      atomicOr(&mask[e * kTileWords + (t >> 5)], 1u << (t & 31));
    }
    __syncthreads();
    // this part's tokens [p0, p1) of the block
    const int p0 = (int)blockIdx.y * part, p1 = min(nt, p0 + part);
    for (int i = tid; i < (p1 - p0) * k; i += blockDim.x) {
      const int t = p0 + i / k;
      const int s = (t0 + p0) * k + i;
      const int e = min(max(ws.topk_idx[s], 0), E - 1);
      int p = base[e];
#pragma unroll
      for (int w = 0; w < kTileWords; ++w) {
        const uint32_t m = mask[e * kTileWords + w];
        if (w < (t >> 5)) p += __popc(m);
        else if (w == (t >> 5)) p += __popc(m & ((1u << (t & 31)) - 1u));
      }
      pos_s[i] = p;
      ws.pos[s] = p;
      ws.perm[p] = s;
    }
    __syncthreads();
    if (do_gather) {
      // each hidden row of the part to its k grouped positions: a warp takes 128 vectors of
      // a row, its four loads issued before the stores
      constexpr int kVec = 4;
      const int groups = (vecs + 32 * kVec - 1) / (32 * kVec);
      for (int g = warp; g < (p1 - p0) * groups; g += kGroupThreads / 32) {
        const int tt = g / groups, v0 = (g - tt * groups) * 32 * kVec + lane;
        const uint4 *src = reinterpret_cast<const uint4 *>(hidden + (size_t)(t0 + p0 + tt) * H);
        uint4 v[kVec];
#pragma unroll
        for (int u = 0; u < kVec; ++u)
          if (v0 + 32 * u < vecs) v[u] = __ldg(src + v0 + 32 * u);
        for (int j = 0; j < k; ++j) {
          uint4 *dst = reinterpret_cast<uint4 *>(ws.xp + (size_t)pos_s[tt * k + j] * H);
#pragma unroll
          for (int u = 0; u < kVec; ++u)
            if (v0 + 32 * u < vecs) dst[v0 + 32 * u] = v[u];
        }
      }
      if (d.Is > 0)
        for (int tt = warp; tt < p1 - p0; tt += kGroupThreads / 32)
          shared_gate_token(hidden, w_sg, d, ws, t0 + p0 + tt, lane);
    }
    __syncthreads();
    // the tile's next block continues after this one
    if (b + 1 < blocks) {
      for (int e = tid; e < E; e += blockDim.x) {
        int n = 0;
#pragma unroll
        for (int w = 0; w < kTileWords; ++w) n += __popc(mask[e * kTileWords + w]);
        base[e] += n;
      }
      __syncthreads();
    }
  }

  const int gtid = ((int)blockIdx.y * T + (int)blockIdx.x) * blockDim.x + tid;
  publish_groups(d, ws, total, offs, flag, chunks, gtid, (int)(gridDim.x * gridDim.y * blockDim.x));
#ifdef SLIMWISE_TRACE
  if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 0)
    trace_stamp(ws, ws.ctrl[kCtrlTraceStep] - 1, kTrGroupEnd);
#endif
}

constexpr int kMaxGroupPart = 16;
// Tokens of a block per CTA of group_place_kernel: enough CTAs for the GPU at
// the smallest batches, fewer recounts of the tile at the largest.
inline int group_part_tokens(int B) { return B <= 1024 ? 4 : B <= 4096 ? 8 : kMaxGroupPart; }

constexpr size_t place_smem(int E, int k, int part) {
  return (size_t)(5 * E + 3 + E * kTileWords + part * k) * 4;
}
// never more than a kernel gets without asking (an attribute of the kernel,
// which calls of other threads would set to other sizes)
static_assert(place_smem(kMaxExperts, kMaxTopK, kMaxGroupPart) <= 48 * 1024, "shared memory");

cudaError_t launch_group_tiled(const __nv_bfloat16 *hidden, const float *w_shared_gate, Dims d,
                               Ws ws, bool pdl, bool gather, cudaStream_t stream) {
  // the tiles' histograms go where the call's expert outputs will be:
  // E / 32 bytes a token at most against k H bf16
  int32_t *tile_cnt = reinterpret_cast<int32_t *>(ws.y);
  const int tiles = group_tile_count(d.B), part = group_part_tokens(d.B);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kGroupThreads);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  cfg.gridDim = dim3(tiles);
  cudaError_t err = cudaLaunchKernelEx(&cfg, group_count_kernel, d, ws, tile_cnt);
  if (err != cudaSuccess) return err;
  cfg.gridDim = dim3(tiles, kGroupTile / part);
  cfg.dynamicSmemBytes = place_smem(d.E, d.k, part);
  return cudaLaunchKernelEx(&cfg, group_place_kernel, hidden, w_shared_gate, d, ws,
                            (const int32_t *)tile_cnt, part, gather ? 1 : 0);
}

cudaError_t launch_group_gather(const __nv_bfloat16 *hidden, const float *w_shared_gate,
                                Dims d, Ws ws, bool pdl, bool gather, cudaStream_t stream) {
  if (d.B >= kGroupTiledMin)
    return launch_group_tiled(hidden, w_shared_gate, d, ws, pdl, gather, stream);
  cudaLaunchConfig_t cfg = {};
  const int tpc = group_tokens_per_cta(d.B);
  cfg.gridDim = dim3((d.B + tpc - 1) / tpc);
  cfg.blockDim = dim3(kGroupThreads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  if (tpc == 1)
    return cudaLaunchKernelEx(&cfg, group_gather_kernel<1>, hidden, w_shared_gate, d, ws,
                              gather ? 1 : 0);
  return cudaLaunchKernelEx(&cfg, group_gather_kernel<2>, hidden, w_shared_gate, d, ws,
                            gather ? 1 : 0);
}

// The results a routing-only call hands out, copied by one launch: eight
// device-to-device copies of a few KB took longer than the routing itself
// (B = 300, m' = 96: 70.5 us a call, 47 with one launch, and 37-40 since the
// binding's calls take raw handles; most of it is host time).
__global__ void __launch_bounds__(256) export_kernel(ExportList x) {
  pdl_wait_primary();
  const int gtid = blockIdx.x * blockDim.x + threadIdx.x, gstride = gridDim.x * blockDim.x;
#pragma unroll
  for (int a = 0; a < kMaxExports; ++a)
    if (x.dst[a])
      for (int i = gtid; i < x.n[a]; i += gstride) x.dst[a][i] = __ldcg(x.src[a] + i);
}

cudaError_t launch_export(const ExportList &x, bool pdl, cudaStream_t stream) {
  int most = 0;
  for (int a = 0; a < kMaxExports; ++a)
    if (x.dst[a] && x.n[a] > most) most = x.n[a];
  if (most == 0) return cudaSuccess;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  const int ctas = (most + 255) / 256;
  cfg.gridDim = dim3(ctas < 1024 ? ctas : 1024);
  cfg.blockDim = dim3(256);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, export_kernel, x);
}

}  // namespace slimwise
