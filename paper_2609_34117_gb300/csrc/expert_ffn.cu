// expert_ffn.cu -- grouped SwiGLU expert FFN over the selected-expert union,
// and the gate-weighted combine of its outputs (a second, small kernel).
//
// Decode reads the weights of every expert in the union of the batch's
// selections once per step (SlimWise Sec. 2.1, Eq. 1) and each expert sees
// few tokens (Sec. 2.1: about B*k/m per step), so the kernel is a weight
// stream: HBM -> (TMA, 128-byte swizzle) -> shared-memory ring ->
// tcgen05.mma with the weights as the M = 128 operand and the expert's
// tokens as the N operand (16..256, padded to 16) -> TMEM accumulators ->
// epilogue warps.
//
// One persistent CTA per SM (320 threads):
//   warp 0   producer: takes work items from a global counter, decodes each
//            once (the others read it from shared memory), waits for a down
//            item's activations, and issues each stage's copies -- the
//            128-row weight tile (two 64-row boxes) and the item's token rows
//            (one box, its height the token count rounded up to 16 rows).
//            The whole warp runs the loop and one elected thread issues, so
//            the copies' operands stay in uniform registers; run by lane 0
//            alone, decode steps were 1.5-4 us slower (B = 96 with the shared
//            expert 141.9 against 137.8 us, an 8-layer stack 815 against 798).
//   warp 1   MMA issuer (the same way) and TMEM owner; double-buffered
//            accumulators so the epilogue of one item overlaps the next.  One
//            commit per stage: a second one costs 70-140 cycles.
//   warps 2-9 two epilogue warpgroups; group g handles the items of
//            accumulator buffer g (every other item).
// Work items, all of gate/up before any of down (so a down item only waits
// for work that has already been handed out):
//   gate/up (entry, i-tile): A = 64 gate rows + the matching 64 up rows of
//            W_gu[e], alternating in groups of 8, K = H; epilogue computes act = SiLU(gate) * up (fp32),
//            stores bf16 act in grouped order and counts the tile done.
//   down    (entry, h-tile): A = 128 rows of W_down[e], K = I, B = act of the
//            entry's tokens (after all its gate/up tiles are done); epilogue
//            rounds the fp32 accumulators to bf16 y in grouped order (like
//            act, an intermediate in the activation type: half the bytes
//            for the combine to read, 2-4 us a step faster at B >= 256).
// The combine kernel runs next on the stream (programmatic dependent launch:
// its CTAs become resident beside this grid's last CTAs): one warp per
// (token, 128-column tile) sums g[t,j] y_j in j order and writes bf16.  With
// the whole GPU's warps on it the combine takes a few microseconds after the
// last expert output, where combining inside this kernel left it to the few
// CTAs that finished the last items.
// Every wait is bounded (1 s unless the caller sets another limit): on
// timeout the CTA records an error bit in the workspace, stops taking work,
// drains its own copies and MMAs, frees TMEM and exits.  The 128 threads of an
// epilogue group take each wait's outcome together (a barrier reduction), so
// a wait that completes just as another thread gives up cannot split the
// group between its named barrier and the exit.
#include "common.cuh"

namespace slimwise {

constexpr int kEpiGroups = 2;    // epilogue warpgroups, one per TMEM accumulator
constexpr int kEpiThreads = 128; // threads of one epilogue warpgroup
constexpr int kFfnThreads = 64 + kEpiGroups * kEpiThreads;
constexpr int kItemRing = 4;
constexpr int kNoItem = 0x7FFFFFFF;  // past every item: no more work
// Transposing buffer of one epilogue warp: up to 32 token rows of 16
// activations, or 16 rows of 32 outputs, padded so that neither the 8-row
// matrix stores nor the 16-byte reads conflict.
constexpr int kActRowBytes = 16 * 2 + 16;
constexpr int kOutRowBytes = 32 * 2 + 16;
constexpr int kXchWarpBytes = 32 * kActRowBytes;
constexpr int kXchBytes = kEpiGroups * (kEpiThreads / 32) * kXchWarpBytes;
static_assert(16 * kOutRowBytes <= kXchWarpBytes, "transposing buffer");

// A work item as the producer hands it to the MMA issuer and the epilogue
// (decoded once, in shared memory).
struct __align__(16) ItemSlot {
  int item;       // its number; past the last one (or an abort): the end
  int entry;
  int tile;
  int form;       // bit 0: down, bit 1: shared expert
  int slot_base;
  int n;          // tokens
  int expert;
  int pad;
};

// A pipeline stage: one 64-wide K sub-tile (one 128-byte swizzle atom) of
// the item's weight rows -- 128, or 256 for a wide item -- then tok_chunk
// token rows of the same K range (half of them in each CTA of a pair).
struct FfnSmem {
  int stages;
  int a_bytes;
  int stage_bytes;
  size_t xch_off, bar_off, misc_off, local_off, total;
};

// Local grouping of the batch in a CTA's shared memory: per expert the mask of
// its tokens [E][words] and, for the j-th selected expert, its id and its first
// grouped position.
__host__ __device__ inline size_t local_group_bytes(int E, int words) {
  return words ? (size_t)E * (words * 4 + 2 * 2) : 0;
}

__host__ __device__ inline FfnSmem ffn_smem_plan(int tok_chunk, int stages, int wide,
                                                  int pair, int E, int words) {
  FfnSmem p;
  p.stages = stages;
  p.a_bytes = kATileBytes * (wide ? 2 : 1);
  p.stage_bytes = p.a_bytes + (pair ? tok_chunk / 2 : tok_chunk) * kBlockK * 2;
  p.xch_off = (size_t)stages * p.stage_bytes;
  p.bar_off = p.xch_off + kXchBytes;
  // full[S], empty[S], acc_full[2], acc_empty[2], item_full[R], item_empty[R],
  // drain, and for a pair mailbox_full[R], mailbox_empty[R]
  p.misc_off = align_up(
      p.bar_off + 8 * (2 * stages + 4 + 2 * kItemRing + 1 + (pair ? 2 * kItemRing : 0)), 16);
  // item ring, tmem base, abort, consumed stages, union size, and for a pair
  // the mailbox[R]
  p.local_off =
      align_up(p.misc_off + kItemRing * sizeof(ItemSlot) + 4 * (4 + (pair ? kItemRing : 0)), 16);
  p.total = p.local_off + local_group_bytes(E, words) + 1024;
  return p;
}

// TMEM accumulators: one per 128 weight rows of an item, N = tok_chunk
// columns each, in two buffers (the epilogue of one item overlaps the MMAs
// of the next): at most 512 columns, so wide items need tok_chunk <= 128.
__host__ __device__ inline int ffn_acc_cols(const Dims &d) { return (d.wide ? 2 : 1) * d.tok_chunk; }

// Claiming ahead pays from this token chunk on: a full-pool layer of 8192
// tokens 849 -> 830 us, 4001 tokens 468 -> 461, 2048 tokens (chunk 176) 302 ->
// 298; nothing at chunks of 16-112, and 3 us lost at B = 1, where CTAs have
// two items each.
constexpr int kAheadMinChunk = 128;

struct Item {
  int down;      // 0: gate/up, 1: down
  int shared;    // 1: the shared expert (token order), 0: a routed expert
  int entry;
  int tile;
  int expert;
  int slot_base;
  int n;         // tokens
};

// The local grouping (local_group_bytes); W mask words per expert.
template <int W>
struct LocalGroup {
  uint32_t *mask;        // [E][W] tokens of each expert
  unsigned short *ids;   // [E] selected experts, ascending
  unsigned short *base;  // [E] first grouped position of each of them
  __device__ __forceinline__ void load(int e, uint32_t (&m)[W]) const {
    static_assert(W == 2 || W == 4, "one 8- or 16-byte mask per expert");
    if constexpr (W == 2) {
      const uint2 v = reinterpret_cast<const uint2 *>(mask)[e];
      m[0] = v.x; m[1] = v.y;
    } else {
      const uint4 v = reinterpret_cast<const uint4 *>(mask)[e];
      m[0] = v.x; m[1] = v.y; m[2] = v.z; m[3] = v.w;
    }
  }
  __device__ __forceinline__ int count(int e) const {
    uint32_t m[W];
    load(e, m);
    int n = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) n += __popc(m[w]);
    return n;
  }
  // rank of token t among expert e's, or -1 when it is not one of them
  __device__ __forceinline__ int rank(int e, int t) const {
    uint32_t m[W];
    load(e, m);
    const uint32_t bit = 1u << (t & 31);
    int n = 0;
    bool in = false;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      if (w == (t >> 5)) in = (m[w] & bit) != 0;
      n += w < (t >> 5) ? __popc(m[w]) : w == (t >> 5) ? __popc(m[w] & (bit - 1u)) : 0;
    }
    return in ? n : -1;
  }
};
template <int W>
__device__ __forceinline__ LocalGroup<W> local_group(void *p, int E) {
  LocalGroup<W> lg;
  lg.mask = reinterpret_cast<uint32_t *>(p);
  lg.ids = reinterpret_cast<unsigned short *>(lg.mask + (size_t)E * W);
  lg.base = lg.ids + E;
  return lg;
}
// The tokens' masks from the selections, by all threads of the CTA (masks
// zeroed before).  Ids are kept inside the pool.
template <int W>
__device__ __forceinline__ void mark_tokens(const LocalGroup<W> &lg, const Dims &d, const Ws &ws) {
  for (int i = threadIdx.x; i < d.B * d.k; i += blockDim.x) {
    const int e = min(max(__ldcg(&ws.topk_idx[i]), 0), d.E - 1), t = i / d.k;
    atomicOr(&lg.mask[e * W + (t >> 5)], 1u << (t & 31));
  }
}
// Chunk c (experts 32 c ..) of the exclusive scan over the experts, by one warp
// of any: `n` tokens of this lane's expert; returns the tokens (<< 16) and the
// selected experts of all experts before it.
template <int W>
__device__ __forceinline__ int scan_experts(const LocalGroup<W> &lg, int E, int c, int lane,
                                            int &n) {
  int before = 0;
  for (int e = lane; e < 32 * c; e += 32) {
    const int m = lg.count(e);
    before += (m << 16) | (m > 0 ? 1 : 0);
  }
  before = __reduce_add_sync(0xFFFFFFFFu, before);
  n = 32 * c + lane < E ? lg.count(32 * c + lane) : 0;
  const int own = (n << 16) | (n > 0 ? 1 : 0);
  int incl = own;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int o = __shfl_up_sync(0xFFFFFFFFu, incl, off);
    if (lane >= off) incl += o;
  }
  return before + incl - own;
}

// Work-item ranges of one launch, in the order they are handed out:
//   [shared gate/up: S*t1s][routed gate/up: r1][shared down: S*t2][routed down]
// Every gate/up item precedes every down item; the shared expert's items go
// first in each phase (they depend on no routing and have the widest entries).
struct ItemPlan {
  int r1;           // routed gate/up items
  int t1, t1s, t2;  // tiles per entry: routed gate/up, shared gate/up, down
  int S;            // shared-expert entries (0: none); routed entries follow them
};

template <bool kShared, bool kLocal, int W>
__device__ __forceinline__ Item decode_item(int item, const ItemPlan &ip, const Ws &ws,
                                            const LocalGroup<W> &lg, int B) {
  Item it;
  it.shared = 0;
  if constexpr (!kShared) {
    if (item < ip.r1) {
      it.down = 0;
      it.entry = item / ip.t1;
      it.tile = item - it.entry * ip.t1;
    } else {
      const int j = item - ip.r1;
      it.down = 1;
      it.entry = j / ip.t2;
      it.tile = j - it.entry * ip.t2;
    }
  } else {
    const int s1 = ip.S * ip.t1s;
    const int g = s1 + ip.r1;
    const int s2 = ip.S * ip.t2;
    int j, t;
    if (item < s1) {
      it.down = 0; it.shared = 1; j = item; t = ip.t1s;
    } else if (item < g) {
      it.down = 0; j = item - s1; t = ip.t1;
    } else if (item < g + s2) {
      it.down = 1; it.shared = 1; j = item - g; t = ip.t2;
    } else {
      it.down = 1; j = item - g - s2; t = ip.t2;
    }
    const int e = j / t;
    it.tile = j - e * t;
    it.entry = it.shared ? e : ip.S + e;
  }
  if constexpr (kLocal) {
    // one entry per selected expert (and one for the shared expert); a
    // gate/up item multiplies every token of the batch, in token order
    it.expert = -1;
    it.slot_base = 0;
    it.n = B;
    if (!it.shared) {
      const int j = it.entry - ip.S;
      it.expert = lg.ids[j];
      it.slot_base = lg.base[j];
      if (it.down) it.n = lg.count(it.expert);
    }
    return it;
  }
  const int4 en = __ldcg(&ws.entries[it.entry]);
  it.expert = en.x;
  it.slot_base = en.y;
  it.n = en.z;
  return it;
}

// out[t, h] = sum_j g[t,j] y[pos(t,j), h] in j order (then the shared
// expert's term) for the 128 h of one tile, by one warp: lane l covers
// h = 4l..4l+3 with one 8-byte load per selection (a y tile row is 256
// contiguous bytes), up to 8 loads in flight per lane; lanes j < k hold
// selection j's grouped position and gate.
template <bool kShared>
__device__ __forceinline__ void combine_token(const Ws &ws, const Dims &d,
                                              __nv_bfloat16 *__restrict__ out, int t, int tile,
                                              int lane, int p, float gj, float sg) {
  const __nv_bfloat16 *ytile = ws.y + tile * kCombineTile + 4 * lane;
  float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  for (int j0 = 0; j0 < d.k; j0 += 8) {
    uint2 v[8];
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) {
      const int pj = __shfl_sync(0xFFFFFFFFu, p, (j0 + jj) & 31);
      if (j0 + jj < d.k)
        v[jj] = __ldcg(reinterpret_cast<const uint2 *>(ytile + (size_t)pj * d.H));
    }
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) {
      const float w = __shfl_sync(0xFFFFFFFFu, gj, (j0 + jj) & 31);
      if (j0 + jj < d.k) {
        acc.x = fmaf(w, __uint_as_float(v[jj].x << 16), acc.x);
        acc.y = fmaf(w, __uint_as_float(v[jj].x & 0xFFFF0000u), acc.y);
        acc.z = fmaf(w, __uint_as_float(v[jj].y << 16), acc.z);
        acc.w = fmaf(w, __uint_as_float(v[jj].y & 0xFFFF0000u), acc.w);
      }
    }
  }
  if constexpr (kShared) {
    // the shared expert's term, after the k routed ones (Sec. 3.3)
    const uint2 vs = __ldcg(reinterpret_cast<const uint2 *>(
        ws.y_s + (size_t)t * d.H + tile * kCombineTile + 4 * lane));
    acc.x = fmaf(sg, __uint_as_float(vs.x << 16), acc.x);
    acc.y = fmaf(sg, __uint_as_float(vs.x & 0xFFFF0000u), acc.y);
    acc.z = fmaf(sg, __uint_as_float(vs.y << 16), acc.z);
    acc.w = fmaf(sg, __uint_as_float(vs.y & 0xFFFF0000u), acc.w);
  }
  const __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x, acc.y);
  const __nv_bfloat162 hi = __floats2bfloat162_rn(acc.z, acc.w);
  *reinterpret_cast<uint2 *>(out + (size_t)t * d.H + tile * kCombineTile + 4 * lane) =
      make_uint2(*reinterpret_cast<const uint32_t *>(&lo),
                 *reinterpret_cast<const uint32_t *>(&hi));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 h2 = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&h2);
}

// SiLU(g) * u = g / (1 + e^-g) * u of accumulator values
__device__ __forceinline__ float swiglu(uint32_t g, uint32_t u) {
  const float gv = __uint_as_float(g), uv = __uint_as_float(u);
  return gv * __frcp_rn(1.0f + __expf(-gv)) * uv;
}

// Epilogue of one warp's 32 accumulator rows, without any exchange between
// warps: the rows of a gate/up tile alternate in groups of 8 gate and 8 up
// rows, so a thread's fragment (tmem_ld_frag) holds both values of an
// activation; the bf16 results go through the warp's transposing buffer into
// token rows and out as 16-byte stores.  Bound by the latency of one pass
// (TMEM load, exponentials, stores); with the rows swapped between warps
// through fp32 buffers and block barriers, and 2-byte output stores, an
// epilogue took about 13,000 cycles at 64-80 tokens, a tail on every launch.
// Measured against that: decode steps 1.0-2.5 us faster (B = 64 full pool
// 182.9 -> 180.5 us, B = 96 with the shared expert 143.9 -> 141.9), an
// 8-layer stack 823 -> 815 us, prefill of 4001 tokens 532 -> 524 us.
// `v0`, `v1`: fragments of the warp's
// first and last 16 rows; `base`: the first token's first element of this
// warp; `left`: tokens left from it on.
//
// 16 kTok16 tokens of 16 activations; row(t): row after `base` of the t-th of
// them, -1 to leave it out.
template <int kTok16, int R, class Row>
__device__ __forceinline__ void store_activations(const uint32_t (&v0)[R], const uint32_t (&v1)[R],
                                                  uint32_t wbuf, int lane, __nv_bfloat16 *base,
                                                  int ld, const Row &row) {
  static_assert(R == 8 * kTok16, "fragment of 16 kTok16 columns");
  const uint32_t dst = wbuf + (uint32_t)(((lane >> 4) * 8 + (lane & 7)) * kActRowBytes +
                                         ((lane >> 3) & 1) * 16);
#pragma unroll
  for (int p = 0; p < kTok16; ++p) {
    uint32_t a[4];  // rows half h of column block 2p + j: a[2j + h]
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int o = 4 * (2 * p + j);
      a[2 * j] = pack_bf16(swiglu(v0[o], v0[o + 2]), swiglu(v0[o + 1], v0[o + 3]));
      a[2 * j + 1] = pack_bf16(swiglu(v1[o], v1[o + 2]), swiglu(v1[o + 1], v1[o + 3]));
    }
    stmatrix_x4_trans(dst + (uint32_t)(p * 16 * kActRowBytes), a[0], a[1], a[2], a[3]);
  }
  __syncwarp();
#pragma unroll
  for (int p = 0; p < kTok16; ++p) {
    const int t = p * 16 + (lane >> 1);
    const uint4 w = ld_shared_v4(wbuf + (uint32_t)(t * kActRowBytes + (lane & 1) * 16));
    const int r = row(t);
    if (r >= 0) *reinterpret_cast<uint4 *>(base + (size_t)r * ld + (lane & 1) * 8) = w;
  }
  __syncwarp();
}

// 16 tokens of 32 outputs, from 8-column block kBlock of the fragments.
template <int kBlock, int R>
__device__ __forceinline__ void store_outputs(const uint32_t (&v0)[R], const uint32_t (&v1)[R],
                                              uint32_t wbuf, int lane, __nv_bfloat16 *base, int ld,
                                              int left) {
  const uint32_t dst = wbuf + (uint32_t)((lane & 7) * kOutRowBytes + (lane >> 3) * 16);
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int o = 4 * (kBlock + j);
    uint32_t a[4];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      a[s] = pack_bf16(__uint_as_float(v0[o + 2 * s]), __uint_as_float(v0[o + 2 * s + 1]));
      a[2 + s] = pack_bf16(__uint_as_float(v1[o + 2 * s]), __uint_as_float(v1[o + 2 * s + 1]));
    }
    stmatrix_x4_trans(dst + (uint32_t)(j * 8 * kOutRowBytes), a[0], a[1], a[2], a[3]);
  }
  __syncwarp();
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const int t = p * 8 + (lane >> 2);
    const uint4 w = ld_shared_v4(wbuf + (uint32_t)(t * kOutRowBytes + (lane & 3) * 16));
    if (t < left) *reinterpret_cast<uint4 *>(base + (size_t)t * ld + (lane & 3) * 8) = w;
  }
  __syncwarp();
}

// Named barrier of epilogue group g (ids 1.., id 0 is __syncthreads).
__device__ __forceinline__ void epi_bar(int g) {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "n"(kEpiThreads) : "memory");
}

// The same barrier, returning whether `v` holds on every thread of group g.
__device__ __forceinline__ bool epi_all(int g, bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.and.pred p, %2, %3, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v), "r"(1 + g), "n"(kEpiThreads)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ int ld_acquire(const int *p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void raise_abort(volatile int *abort, Ws &ws, int bit) {
  *abort = 1;
  atomicOr(&ws.ctrl[kCtrlErr], bit);
}

// At most 128 registers a thread (320 threads: 40 K of the SM's 64 K), so
// that a CTA of the dependent combine kernel (256 threads, 40 registers)
// can become resident beside this one.
//
// kPair: the grid is made of 2-CTA clusters.  A routed work item covers two
// adjacent 128-row weight tiles (as a wide item does); CTA r of the pair
// loads tile r and token rows [r N/2, (r + 1) N/2) of the item's N, and the
// pair's first CTA issues one M = 256 MMA per K step over both CTAs' shared
// memory.  Only that CTA's producer takes items from the global counter; it
// hands each one to the second CTA through a mailbox in the second CTA's
// shared memory, so both CTAs work through the same items in the same order.
// The second CTA's copies complete bytes on the first CTA's stage barriers;
// the MMA commits arrive on the stage and accumulator barriers of both CTAs;
// each CTA's epilogue reads its own TMEM lanes (its 128 weight rows) and
// releases the accumulator to the first CTA's MMA issuer.
//
// kAhead: a CTA claims its next item when the current one starts, and fetches
// its work entry, and looks whether a down item's activations are complete,
// while the current one still streams, so that an item boundary costs none of
// these round trips.  Large token chunks only (kAheadMinChunk): their items
// are many per CTA, and an unstarted item held back at the end of the launch
// is a small share of it.
//
// kLocalWords > 0 (at most kLocalTokens tokens): there is no grouping kernel.  Every CTA
// marks the batch's selections in shared memory (one bit mask of tokens per
// expert), lists the selected experts and their first grouped positions, and
// takes one entry per expert from that list.  A gate/up item multiplies all
// tokens of the batch, in token order, straight from the caller's hidden rows
// (a box of at most 96 rows, 12 KB a stage), and its epilogue stores the rows of the expert's tokens in grouped
// order, so a down item reads its own tokens' activations alone, as elsewhere.
// With the grouping kernel, which costs a launch boundary and the copy of the
// rows, against without, a step: m' = 32 B = 37 55.6 / 52.2 us, m' = 64 B = 1
// 31.8 / 27.8, full pool B = 64 176.9 / 172.4, Qwen3.6-shaped layer with the
// shared expert B = 32 120.8 / 114.4; 64 to 128 tokens, m' = 64: 64 99.4 /
// 95.8, 96 100.2 / 98.1, 112 100.2 / 99.7, 128 100.1 / 101.4 (larger token
// boxes take the ring's place and L2 reads; the line is drawn at 96).  The scan
// of the pool in every CTA does not move it: pools of 512 and 1024 experts at
// H = 512-8192 took 0.72-0.99 of the time with the grouping kernel at 1-96
// tokens.
template <bool kShared, bool kWide, bool kPair, bool kAhead, int kLocalWords>
__global__ void __maxnreg__(128)
    expert_ffn_kernel(const __grid_constant__ FfnMaps maps,
                      const __nv_bfloat16 *__restrict__ hidden,
                      const float *__restrict__ w_shared_gate, Dims d, Ws ws,
                      const int32_t *__restrict__ retained, int stages,
                      int tmem_cols, int static_first, int early_dependents,
                      uint64_t timeout_ns,
                      int starve_first_down) {
  constexpr bool kLocal = kLocalWords > 0;
  static_assert(!(kPair && (kShared || kWide)), "pair items are routed 128-row tiles");
  static_assert(!(kAhead && kPair), "a pair's items are handed from CTA to CTA");
  static_assert(!(kLocal && (kWide || kPair || kAhead)), "small batches take plain items");
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const FfnSmem plan =
      ffn_smem_plan(d.tok_chunk, stages, d.wide, kPair ? 1 : 0, d.E, kLocalWords);
  const uint32_t smem_base = smem_u32(smem);
  const uint32_t bar0 = smem_base + (uint32_t)plan.bar_off;
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (stages + s); };
  auto accf_bar = [&](int b) { return bar0 + 8u * (2 * stages + b); };
  auto acce_bar = [&](int b) { return bar0 + 8u * (2 * stages + 2 + b); };
  auto itf_bar = [&](int r) { return bar0 + 8u * (2 * stages + 4 + r); };
  auto ite_bar = [&](int r) { return bar0 + 8u * (2 * stages + 4 + kItemRing + r); };
  const uint32_t drain_bar = bar0 + 8u * (2 * stages + 4 + 2 * kItemRing);
  // pair mailbox: full barriers live in the second CTA, empty ones in the first
  auto mbf_bar = [&](int r) { return bar0 + 8u * (2 * stages + 5 + 2 * kItemRing + r); };
  auto mbe_bar = [&](int r) { return bar0 + 8u * (2 * stages + 5 + 3 * kItemRing + r); };
  ItemSlot *ring = reinterpret_cast<ItemSlot *>(smem + plan.misc_off);  // [kItemRing]
  int *misc = reinterpret_cast<int *>(ring + kItemRing);
  volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(misc);
  volatile int *abort = misc + 1;
  volatile int *consumed = misc + 2;                 // stages the MMA finished with
  int *n_union = misc + 3;                           // selected experts, local grouping only
  volatile int *mbox = misc + 4;                     // [kItemRing], pair only
  const auto lg = local_group<kLocal ? kLocalWords : 2>(smem + plan.local_off, d.E);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t crank = kPair ? cluster_ctarank() : 0u;  // CTA of the pair
  const bool lead = crank == 0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf_bar(b), 1);
      // a pair's accumulator is released by one thread of each CTA's group
      mbar_init(acce_bar(b), kPair ? 2 : kEpiThreads);
    }
    for (int r = 0; r < kItemRing; ++r) {
      mbar_init(itf_bar(r), 1);
      mbar_init(ite_bar(r), 1 + kEpiGroups * kEpiThreads);
      if constexpr (kPair) {
        mbar_init(mbf_bar(r), 1);
        mbar_init(mbe_bar(r), 1);
      }
    }
    mbar_init(drain_bar, 1);
    *abort = 0;
    *consumed = 0;
    mbar_fence_init();
  }
  if constexpr (kLocal)
    for (int i = threadIdx.x; i < d.E * kLocalWords; i += blockDim.x) lg.mask[i] = 0u;
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&maps.w_gu);
    tma_prefetch_desc(&maps.w_down);
    if constexpr (kLocal || kShared) tma_prefetch_desc(&maps.hid);
    for (int m = 0; m < kTokBoxSizes && kTokBox * (m + 1) <= d.tok_chunk; ++m) {
      if constexpr (!kLocal) tma_prefetch_desc(&maps.xp[m]);
      tma_prefetch_desc(&maps.act[m]);
      if constexpr (kShared) {
        tma_prefetch_desc(&maps.act_s[m]);
      }
    }
    if constexpr (kShared) {
      tma_prefetch_desc(&maps.w_gu_s);
      tma_prefetch_desc(&maps.w_down_s);
    }
  }
  if (warp == 1) {
    if constexpr (kPair) {
      tmem_alloc_pair(smem_u32((const void *)tmem_slot), (uint32_t)tmem_cols);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(smem_u32((const void *)tmem_slot), (uint32_t)tmem_cols);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  // both CTAs' barriers are initialised before either arrives on the other's
  if constexpr (kPair) cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // the pair MMA writes both CTAs' accumulators at the first CTA's address:
  // the second CTA checks that its allocation is the same, else it takes no
  // work (its partner's waits then run out)
  if constexpr (kPair) {
    if (threadIdx.x == 0 && !lead &&
        ld_shared_cluster(mapa_shared(smem_u32((const void *)tmem_slot), 0u)) != tmem_base)
      raise_abort(abort, ws, SLIMWISE_DEVERR_TMEM_PAIR);
  }

  // While the routing or grouping kernel runs (this grid may already be
  // resident), warm L2 with this CTA's likely first work item: the gate/up tile that item
  // number blockIdx.x (for a pair, the cluster's number) has when each
  // retained expert is selected and takes one entry.  The work list runs in
  // ascending expert order, so entry j is then the j-th retained expert
  // (retained ids listed in ascending order), which holds for nearly every
  // pool once B k >= 2 m'.  The guess uses only this call's inputs, so it is
  // as good for a stack of different layers as for one layer called again
  // (guessing from the previous call's work list cost a 10-layer skewed stack
  // 3.8 %).  Without it steps of 16 to 256 tokens are 2-5 us slower (m' = 64
  // B = 256 103.4 / 108.8 us).  A wide item warms only its first 64 gate and 64 up rows: all of
  // them would be 152 MB, more than L2 holds; each CTA of a pair warms its
  // own 64 gate and 64 up rows.  Prefetches only, every index bounded, so a
  // wrong guess costs bandwidth, never correctness.
  const int item0 = kPair ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
  if constexpr (!kShared) {
    if (warp == 0 && lane == 0 && d.B * d.k >= 2 * d.m_ret) {
      const int t1g = gate_up_tiles(d);
      const int entry = item0 / t1g;
      if (entry < d.m_ret) {
        const int e = retained ? __ldcg(retained + entry) : entry;
        if (e >= 0 && e < d.E) {
          const int u0 = ((item0 - entry * t1g) * item_tiles(d) + (int)crank) * kTileUnits;
          for (int kc = 0; kc < d.H / kBlockK; ++kc) {
            tma_prefetch_w(&maps.w_gu, kc * kBlockK, u0, e);
            tma_prefetch_w(&maps.w_gu, kc * kBlockK, u0 + kTileUnits / 2, e);
          }
        }
      }
    }
  }

  // Everything below reads the routing and grouping kernels' results.
  pdl_wait_primary();
  // Above 64 tokens the combine kernel that follows may become resident now
  // (it waits for this grid to finish): measured 2-4 us faster per step at
  // B = 128-512, 0.5 us slower at B = 64, where the trigger stays at the end
  // of the work (launch_expert_ffn: and where a combine that groups locally
  // finds no room yet).
  if (early_dependents) pdl_launch_dependents();
#ifdef SLIMWISE_TRACE
  const int tr_step = ws.ctrl[kCtrlTraceStep] - 1;
  if (kLocal && blockIdx.x == 0 && threadIdx.x == 0) trace_stamp(ws, tr_step, kTrGroupStart);
#endif
  if constexpr (kLocal) {
    mark_tokens(lg, d, ws);
    __syncthreads();
    for (int c = warp; 32 * c < d.E; c += blockDim.x / 32) {
      int n;
      const int before = scan_experts(lg, d.E, c, lane, n);
      const int e = 32 * c + lane, j = before & 0xFFFF;
      if (n > 0) {
        lg.ids[j] = (unsigned short)e;
        lg.base[j] = (unsigned short)(before >> 16);
      }
      if (e == d.E - 1) *n_union = j + (n > 0 ? 1 : 0);
    }
    __syncthreads();
  }
#ifdef SLIMWISE_TRACE
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (kLocal) trace_stamp(ws, tr_step, kTrGroupEnd);
    trace_stamp(ws, tr_step, kTrFfnStart);
  }
#endif

  const int t1 = gate_up_tiles(d);
  const int t2 = down_tiles(d);
  ItemPlan ip;
  ip.t1 = t1;
  ip.t1s = kShared ? shared_gate_up_tiles(d) : 0;
  ip.t2 = t2;
  ip.S = kShared ? d.S : 0;
  int total;
  if constexpr (kLocal) {
    ip.r1 = *n_union * t1;
    total = ip.S * (ip.t1s + t2) + *n_union * (t1 + t2);
  } else {
    ip.r1 = __ldcg(&ws.ctrl[kCtrlItems1]);
    total = __ldcg(&ws.ctrl[kCtrlTotalItems]);
  }
  const int nb_cols = ffn_acc_cols(d);  // TMEM columns per accumulator buffer
  constexpr int wmul = kWide ? 2 : 1;   // 128-row halves of a routed item in this CTA
  // 128-row tiles of a routed item (across the pair): its gate/up items count
  // as many finished tiles towards the entry's down items
  constexpr int tiles_per_item = (kWide || kPair) ? 2 : 1;


  if (warp == 0) {
    // ------------------------------------------------------------ producer
    // The whole warp runs the loop (see elect_one); what depends on memory is
    // read once per item and broadcast, so everything the copies take is
    // uniform over the warp.
    const uint64_t pol_w = l2_policy_evict_first();
    const uint64_t pol_x = l2_policy_evict_last();
    int stage = 0;
    uint32_t phase = 0;
    int slot = 0;
    uint32_t rphase = 0;
    int issued = 0;
    // With every CTA of the grid resident (one per SM), CTA i's first item
    // is item i (for pairs, cluster i's) and later ones come from the
    // counter past the grid: the first item costs no atomic round trip after
    // the dependency wait.
    const int n_first = static_first ? (int)(kPair ? gridDim.x >> 1 : gridDim.x) : 0;
    bool first = static_first != 0;
    // a bounded wait of the warp: whether it completed on every lane
    auto all_ok = [&](bool ok) {
      if (!ok && !*abort) raise_abort(abort, ws, SLIMWISE_DEVERR_PIPELINE_TIMEOUT);
      return __all_sync(0xFFFFFFFFu, ok) != 0;
    };
    // work entry of an item, uniform over the warp
    auto fetch = [&](int i) {
      Item r = {};
      if (i < total) r = decode_item<kShared, kLocal>(i, ip, ws, lg, d.B);
      r.expert = __shfl_sync(0xFFFFFFFFu, r.expert, 0);
      r.slot_base = __shfl_sync(0xFFFFFFFFu, r.slot_base, 0);
      r.n = __shfl_sync(0xFFFFFFFFu, r.n, 0);
      return r;
    };
    // gate/up tiles an entry's down items wait for
    auto tiles_needed = [&](const Item &i) {
      return ((kShared && i.shared) ? ip.t1s : t1) * (kPair ? 2 : 1);
    };
    // kAhead: the next item (claimed: on lane 0 until it is fetched), its
    // entry, and whether its activations were seen complete
    int next = 0;
    Item next_it = {};
    bool next_ready = false;
    for (bool started = false;; started = true) {
      int item = 0;
      if (kAhead && started) {
        item = __any_sync(0xFFFFFFFFu, *abort != 0) ? kNoItem : next;
      } else if (!kPair || lead) {
        if (lane == 0) {
          item = first ? item0 : n_first + atomicAdd(&ws.ctrl[kCtrlWorkCounter], 1);
          if (*abort) item = kNoItem;
        }
        first = false;
        if constexpr (kPair) {
          // hand the item to the second CTA; an item past the end (or the
          // abort sentinel) ends its loop too
          if (!all_ok(mbar_wait_cluster_bounded(mbe_bar(slot), rphase ^ 1u, nullptr, timeout_ns)))
            break;
          if (lane == 0) {
            st_shared_cluster(mapa_shared(smem_u32((const void *)(mbox + slot)), 1u), item);
            mbar_arrive_cluster(mapa_shared(mbf_bar(slot), 1u));
          }
        }
      } else {
        // the second CTA of a pair: the item its first CTA took
        if (!all_ok(mbar_wait_cluster_bounded(mbf_bar(slot), rphase, abort, timeout_ns))) break;
        if (lane == 0) {
          item = mbox[slot];
          mbar_arrive_cluster(mapa_shared(mbe_bar(slot), 0u));
          if (*abort) item = kNoItem;
        }
      }
      item = __shfl_sync(0xFFFFFFFFu, item, 0);
      if (!all_ok(mbar_wait_bounded(ite_bar(slot), rphase ^ 1u, abort, timeout_ns))) break;
      const Item it = (kAhead && started) ? next_it : fetch(item);
      const bool ready = kAhead && started && next_ready;
      if (lane == 0) {
        ItemSlot sl = {};
        sl.item = item;
        sl.entry = it.entry;
        sl.tile = it.tile;
        sl.form = it.down | (it.shared << 1);
        sl.slot_base = it.slot_base;
        sl.n = it.n;
        sl.expert = it.expert;
        ring[slot] = sl;
        mbar_arrive(itf_bar(slot));
      }
      if (++slot == kItemRing) {
        slot = 0;
        rphase ^= 1u;
      }
      if (item >= total) {
        // no work left for this CTA: the next kernel on the stream may start
        // its launch (it waits for this grid's completion before reading)
        pdl_launch_dependents();
        break;
      }
      // the item's token rows: one box of the tokens rounded up to 16
      // rows (rows past the entry are loaded but not multiplied); each CTA
      // of a pair loads half of them, from 8 n16 rows further for the second
      const int n16 = (it.n + 15) >> 4;
      const int box_m = token_box_for(n16);
      const int tok_row = (kLocal && !it.down ? 0 : it.slot_base) +
                          (kPair ? (int)crank * n16 * (kTokBox / 2) : 0);
      // weight rows: per 128-row half of the item, two boxes of 4 units (64
      // rows) -- gate and up rows in alternating groups of 8, or 128
      // consecutive down rows; a pair's CTA r loads half r
      const int halves = (kShared && it.shared) ? 1 : wmul;
      const int unit0 = (it.tile * tiles_per_item + (kPair ? (int)crank : 0)) * kTileUnits;
      int nk, expert;
      const void *amap;
      const void *bmap;
      if (kShared && it.shared) {
        // the shared expert: its own weights, tokens in batch order
        nk = it.down ? d.Is / kBlockK : d.H / kBlockK;
        amap = it.down ? (const void *)&maps.w_down_s : (const void *)&maps.w_gu_s;
        bmap = (const void *)&maps.act_s[box_m];
        expert = 0;
      } else {
        nk = it.down ? d.I / kBlockK : d.H / kBlockK;
        amap = it.down ? (const void *)&maps.w_down : (const void *)&maps.w_gu;
        bmap = it.down ? (const void *)&maps.act[box_m] : (const void *)&maps.xp[box_m];
        expert = it.expert;
      }
      // the batch in token order, straight from the caller's hidden rows: boxes
      // of tok_chunk rows
      const bool from_hidden = !it.down && (kLocal || (kShared && it.shared));
      if (from_hidden) bmap = (const void *)&maps.hid;
      if (kAhead && lane == 0) next = n_first + atomicAdd(&ws.ctrl[kCtrlWorkCounter], 1);
      if (it.down && !ready) {
        // the entry's activations must be complete: all its gate/up tiles
        const int *done = &ws.entry_done[it.entry];
        int need = tiles_needed(it);
        // test only: the first routed down item waits for one gate/up tile
        // more than exist, so its wait runs out (the timeout path)
        if (starve_first_down && item == ip.S * ip.t1s + ip.r1) ++need;
        bool ok = __all_sync(0xFFFFFFFFu, ld_acquire(done) >= need) != 0;
        if (!ok) {
          const uint64_t t0 = global_timer_ns();
          while (!(ok = __all_sync(0xFFFFFFFFu, ld_acquire(done) >= need) != 0)) {
            bool give_up = *abort != 0;
            if (!give_up && global_timer_ns() - t0 > timeout_ns) {
              raise_abort(abort, ws, SLIMWISE_DEVERR_DEPENDENCY_TIMEOUT);
              give_up = true;
            }
            if (__any_sync(0xFFFFFFFFu, give_up)) break;
            __nanosleep(128);
          }
        }
        if (!ok) break;
        fence_proxy_async_global();
      }
      // bytes the stage barrier expects: for a pair, both CTAs' copies
      const uint32_t stage_tx =
          kPair ? (uint32_t)(2 * kATileBytes + n16 * kTokBox * kBlockK * 2)
                : (uint32_t)(halves * kATileBytes +
                             (from_hidden ? d.tok_chunk : n16 * kTokBox) * kBlockK * 2);
      bool ok = true;
      for (int kc = 0; kc < nk; ++kc) {
        if (kAhead && kc == (2 * nk) / 3) {
          next = __shfl_sync(0xFFFFFFFFu, next, 0);
          next_it = fetch(next);
          next_ready = false;
          if (next < total && next_it.down && !starve_first_down) {
            next_ready = __all_sync(0xFFFFFFFFu, ld_acquire(&ws.entry_done[next_it.entry]) >=
                                                     tiles_needed(next_it)) != 0;
            if (next_ready) fence_proxy_async_global();
          }
        }
        if (!all_ok(mbar_wait_bounded(empty_bar(stage), phase ^ 1u, abort, timeout_ns))) {
          ok = false;
          break;
        }
        const int x = kc * kBlockK;
        const uint32_t a = smem_base + (uint32_t)(stage * plan.stage_bytes);
        if (elect_one()) {
          if (kPair && !lead) {
            const uint32_t lb = mapa_shared(full_bar(stage), 0u);
            tma_load_w_pair(a, amap, lb, x, unit0, expert, pol_w);
            tma_load_w_pair(a + kATileBytes / 2, amap, lb, x, unit0 + kTileUnits / 2, expert, pol_w);
            tma_load_2d_pair(a + (uint32_t)plan.a_bytes, bmap, lb, x, tok_row, pol_x);
          } else {
            mbar_arrive_expect_tx(full_bar(stage), stage_tx);
            for (int h = 0; h < halves; ++h) {
              const uint32_t ah = a + (uint32_t)(h * kATileBytes);
              const int u = unit0 + h * kTileUnits;
              tma_load_w(ah, amap, full_bar(stage), x, u, expert, pol_w);
              tma_load_w(ah + kATileBytes / 2, amap, full_bar(stage), x, u + kTileUnits / 2, expert,
                         pol_w);
            }
            tma_load_2d(a + (uint32_t)plan.a_bytes, bmap, full_bar(stage), x, tok_row, pol_x);
          }
        }
        __syncwarp();
        ++issued;
        if (++stage == stages) {
          stage = 0;
          phase ^= 1u;
        }
      }
      if (!ok) break;
    }
    if (lane == 0) {
      if (kPair && !lead) {
        // The second CTA's stages complete on the first CTA's barriers; the
        // first CTA's MMAs read them and their commits arrive here.  Wait
        // (bounded) until every stage still in the ring has been released,
        // so that no copy, read or arrival is left on this CTA's shared
        // memory when it exits.
        const int from = issued > stages ? issued - stages : 0;
        for (int s = from; s < issued; ++s)
          mbar_wait_timeout(empty_bar(s % stages), (uint32_t)((s / stages) & 1), 10000000ull);
      } else if (*abort) {
        // let this CTA's copies in flight land before shared memory goes away
        for (int s = *consumed; s < issued; ++s)
          mbar_wait_timeout(full_bar(s % stages), (uint32_t)((s / stages) & 1), 10000000ull);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    // the whole warp runs the loop here too
    int stage = 0;
    uint32_t phase = 0;
    int slot = 0;
    uint32_t rphase = 0;
    int n_consumed = 0;
    auto all_ok = [&](bool ok) {
      if (!ok && !*abort) raise_abort(abort, ws, SLIMWISE_DEVERR_PIPELINE_TIMEOUT);
      return __all_sync(0xFFFFFFFFu, ok) != 0;
    };
    for (int local = 0;; ++local) {
      if (!all_ok(mbar_wait_bounded(itf_bar(slot), rphase, abort, timeout_ns))) break;
      const int item = __shfl_sync(0xFFFFFFFFu, ring[slot].item, 0);
      const int form = __shfl_sync(0xFFFFFFFFu, ring[slot].form, 0);
      const int n16 = (__shfl_sync(0xFFFFFFFFu, ring[slot].n, 0) + 15) >> 4;
      if (lane == 0) mbar_arrive(ite_bar(slot));
      if (++slot == kItemRing) {
        slot = 0;
        rphase ^= 1u;
      }
      if (item >= total) break;
      // the second CTA of a pair issues no MMA: it only keeps its item ring
      // moving
      if (kPair && !lead) continue;
      const bool down = (form & 1) != 0, shared = (form & 2) != 0;
      const int b = local & 1;
      const uint32_t use = (uint32_t)(local >> 1);
      const bool freed =
          kPair ? mbar_wait_cluster_bounded(acce_bar(b), (use & 1u) ^ 1u, abort, timeout_ns)
                : mbar_wait_bounded(acce_bar(b), (use & 1u) ^ 1u, abort, timeout_ns);
      if (!all_ok(freed)) break;
      tc_fence_after();
      // half h of the item: A = the stage's weight rows [128 h, 128 h + 128),
      // D = columns [h tok_chunk, ...) of the buffer; B = the token rows.
      // A pair runs one M = 256 MMA: A rows 128-255 and B rows N/2.. are the
      // second CTA's, at the same shared-memory offsets.
      const uint32_t d_tmem = tmem_base + (uint32_t)(b * nb_cols);
      const uint32_t idesc = idesc_bf16_f32(kPair ? 2 * kTileRows : kTileRows, n16 * kTokBox);
      const int halves = (kShared && shared) ? 1 : wmul;
      const int inner = (kShared && shared) ? d.Is : d.I;
      const int nk = down ? inner / kBlockK : d.H / kBlockK;
      bool ok = true;
      for (int kc = 0; kc < nk; ++kc) {
        if (!all_ok(mbar_wait_bounded(full_bar(stage), phase, abort, timeout_ns))) {
          ok = false;
          break;
        }
        tc_fence_after();
#ifdef SLIMWISE_TRACE
        if (blockIdx.x == 0 && lane == 0 && n_consumed == 0) trace_stamp(ws, tr_step, kTrFfnFirstData);
#endif
        const uint32_t a = smem_base + (uint32_t)(stage * plan.stage_bytes);
        const uint32_t bs = a + (uint32_t)plan.a_bytes;
        ++n_consumed;
        if (elect_one()) {
          if constexpr (kPair) {
#pragma unroll
            for (int kk = 0; kk < kBlockK / 16; ++kk)
              tc_mma_bf16_pair(d_tmem, smem_desc_sw128(a + kk * 32), smem_desc_sw128(bs + kk * 32),
                               idesc, (kc | kk) != 0 ? 1u : 0u);
            tc_commit_pair(empty_bar(stage), (uint16_t)3);
          } else {
            for (int h = 0; h < halves; ++h) {
              const uint32_t as = a + (uint32_t)(h * kATileBytes);
#pragma unroll
              for (int kk = 0; kk < kBlockK / 16; ++kk)
                tc_mma_bf16(d_tmem + (uint32_t)(h * d.tok_chunk), smem_desc_sw128(as + kk * 32),
                            smem_desc_sw128(bs + kk * 32), idesc, (kc | kk) != 0 ? 1u : 0u);
            }
            tc_commit(empty_bar(stage));
          }
          *consumed = n_consumed;
        }
        __syncwarp();
        if (++stage == stages) {
          stage = 0;
          phase ^= 1u;
        }
      }
      if (!ok) break;
      if (elect_one()) {
        if constexpr (kPair) tc_commit_pair(accf_bar(b), (uint16_t)3);
        else tc_commit(accf_bar(b));
      }
      __syncwarp();
    }
    if (__any_sync(0xFFFFFFFFu, *abort != 0) && n_consumed > 0) {
      if (elect_one()) {
        if constexpr (kPair) tc_commit_pair(drain_bar, (uint16_t)1);
        else tc_commit(drain_bar);
      }
      mbar_wait_timeout(drain_bar, 0, 10000000ull);
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------ epilogue
    // Two warpgroups; group g owns TMEM accumulator buffer g, i.e. the items
    // with local index = g (mod 2), so one group's epilogue overlaps the
    // other's and the MMA of the next item.
    const int g = (warp - 2) >> 2;      // epilogue group
    const int q = warp & 3;             // TMEM lane quarter of this warp
    const int et = (threadIdx.x - 64) & (kEpiThreads - 1);
    const uint32_t wbuf = smem_base + (uint32_t)(plan.xch_off + (warp - 2) * kXchWarpBytes);
    // the shared expert's gates, where no grouping kernel computes them: one
    // token per CTA, before its first accumulators are ready
    if (kLocal && kShared && warp == 9)
      for (int t = blockIdx.x; t < d.B; t += gridDim.x)
        shared_gate_token(hidden, w_shared_gate, d, ws, t, lane);
    int slot = 0;
    uint32_t rphase = 0;
    for (int local = 0;; ++local) {
      bool got = mbar_wait_bounded(itf_bar(slot), rphase, abort, timeout_ns);
      if (!got && !*abort) raise_abort(abort, ws, SLIMWISE_DEVERR_PIPELINE_TIMEOUT);
      if (!epi_all(g, got)) break;
      const ItemSlot it = ring[slot];
      mbar_arrive(ite_bar(slot));
      if (++slot == kItemRing) {
        slot = 0;
        rphase ^= 1u;
      }
      if (it.item >= total) break;
      const int b = local & 1;
      if (b != g) continue;
      const bool down = (it.form & 1) != 0, shared = kShared && (it.form & 2) != 0;
      const uint32_t use = (uint32_t)(local >> 1);
      const int halves = shared ? 1 : wmul;
      got = mbar_wait_bounded(accf_bar(b), use & 1u, abort, timeout_ns);
      if (!got && !*abort) raise_abort(abort, ws, SLIMWISE_DEVERR_PIPELINE_TIMEOUT);
      if (!epi_all(g, got)) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * nb_cols);
      const int cols = ((it.n + 15) >> 4) * kTokBox;  // accumulator columns
      // 128-row tile of the item that TMEM half hh holds: half hh of a wide
      // item, the CTA's own half of a pair item
      const int tile0 = it.tile * tiles_per_item + (kPair ? (int)crank : 0);
      // the accumulator is free once its last columns have been loaded
      auto release = [&]() {
        tc_fence_before();
        if constexpr (!kPair) mbar_arrive(acce_bar(b));
      };
      for (int hh = 0; hh < halves; ++hh) {
        const uint32_t th = taddr + (uint32_t)(hh * d.tok_chunk);
        // routed rows in grouped order, shared ones in token order
        __nv_bfloat16 *base;
        int ld;
        if (!down) {
          ld = shared ? d.Is : d.I;
          base = (shared ? ws.act_s : ws.act) + (size_t)it.slot_base * ld +
                 (tile0 + hh) * kGateRows + 16 * q;
        } else {
          ld = d.H;
          base = (shared ? ws.y_s : ws.y) + (size_t)it.slot_base * ld + (tile0 + hh) * kTileRows +
                 32 * q;
        }
        int c = 0;
        // row, after `base`, of the activations of accumulator column c + t
        auto row_of = [&](int t) {
          if (kLocal && !shared) return c + t < d.B ? lg.rank(it.expert, c + t) : -1;
          return c + t < it.n ? c + t : -1;
        };
        for (; c + 32 <= cols; c += 32) {
          uint32_t v0[16], v1[16];
          tmem_ld_frag(th + c, v0);
          tmem_ld_frag(th + c + (16u << 16), v1);
          tmem_ld_wait();
          if (hh == halves - 1 && c + 32 == cols) release();
          if (down) {
            store_outputs<0>(v0, v1, wbuf, lane, base + (size_t)c * ld, ld, it.n - c);
            store_outputs<2>(v0, v1, wbuf, lane, base + (size_t)(c + 16) * ld, ld, it.n - c - 16);
          } else {
            store_activations<2>(v0, v1, wbuf, lane, base, ld, row_of);
          }
        }
        if (c < cols) {  // 16 columns left
          uint32_t v0[8], v1[8];
          tmem_ld_frag(th + c, v0);
          tmem_ld_frag(th + c + (16u << 16), v1);
          tmem_ld_wait();
          if (hh == halves - 1) release();
          if (down) store_outputs<0>(v0, v1, wbuf, lane, base + (size_t)c * ld, ld, it.n - c);
          else store_activations<1>(v0, v1, wbuf, lane, base, ld, row_of);
        }
      }
      if (!down) {
        // publish the activations to the TMA (async proxy) readers of any CTA
        fence_proxy_async_global();
        __threadfence();
        epi_bar(g);
        if (et == 0) {
          if constexpr (kPair) mbar_arrive_cluster(mapa_shared(acce_bar(b), 0u));
          atomicAdd(&ws.entry_done[it.entry], 1);
        }
      } else if constexpr (kPair) {
        // the expert outputs are all a down item writes: the combine kernel
        // that follows this grid sums them
        epi_bar(g);
        if (et == 0) mbar_arrive_cluster(mapa_shared(acce_bar(b), 0u));
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  // neither CTA of a pair leaves (or frees TMEM) while the other may still
  // use its shared memory, barriers or TMEM
  if constexpr (kPair) cluster_sync_all();
#ifdef SLIMWISE_TRACE
  if (threadIdx.x == 0) {
    uint64_t t = global_timer_ns();
    atomicMax(reinterpret_cast<unsigned long long *>(ws.ctrl + kCtrlWords) +
                  (tr_step & (kTraceSteps - 1)) * kTrSlots + kTrFfnEnd,
              (unsigned long long)t);
  }
#endif
  if (warp == 1) {
    tc_fence_after();
    if constexpr (kPair) tmem_dealloc_pair(tmem_base, (uint32_t)tmem_cols);
    else tmem_dealloc(tmem_base, (uint32_t)tmem_cols);
  }
}

// The combine of every (token, 128-column tile) after the FFN grid has
// finished: one warp per pair, the same arithmetic and order as the fused
// combine (combine_token).  Launched as the FFN's programmatic dependent, so
// its CTAs become resident beside the FFN's last CTAs and start as soon as
// the FFN's expert outputs are complete.
constexpr int kCombineThreads = 256;

template <bool kShared, int kLocalWords>
__global__ void __launch_bounds__(kCombineThreads)
    combine_kernel(Dims d, Ws ws, __nv_bfloat16 *__restrict__ out) {
  constexpr bool kLocal = kLocalWords > 0;
  extern __shared__ __align__(16) uint32_t masks[];  // kLocal: [E][kLocalWords], then base [E]
  const int t2 = d.H / kCombineTile;
  const int lane = threadIdx.x & 31;
  const int wpc = kCombineThreads / 32;
  const int pairs = d.B * t2;
  // One pair per warp (the grid covers them all).  Its grouped positions and
  // gates were written by the routing and grouping kernels, which finished
  // before the expert FFN started its work, so they are read before waiting
  // for the FFN; only the expert outputs need the wait.  Without a grouping
  // kernel the positions are worked out here, from the selections: an
  // expert's first position is the number of tokens of the experts before it.
  const int pr = blockIdx.x * wpc + (threadIdx.x >> 5);
  const int t = pr / t2;
  int p = 0;
  float gj = 0.0f, sg = 0.0f;
  if constexpr (kLocal) {
    LocalGroup<kLocal ? kLocalWords : 2> lg;
    lg.mask = masks;
    lg.ids = nullptr;
    lg.base = reinterpret_cast<unsigned short *>(masks + d.E * kLocalWords);  // by expert id
    for (int i = threadIdx.x; i < d.E * kLocalWords; i += blockDim.x) masks[i] = 0u;
    __syncthreads();
    mark_tokens(lg, d, ws);
    __syncthreads();
    for (int c = threadIdx.x >> 5; 32 * c < d.E; c += wpc) {
      int n;
      const int before = scan_experts(lg, d.E, c, lane, n);
      if (32 * c + lane < d.E) lg.base[32 * c + lane] = (unsigned short)(before >> 16);
    }
    __syncthreads();
    if (pr < pairs && lane < d.k) {
      const int e = min(max(__ldcg(&ws.topk_idx[(size_t)t * d.k + lane]), 0), d.E - 1);
      gj = __ldcg(&ws.topk_gate[(size_t)t * d.k + lane]);
      p = lg.base[e] + lg.rank(e, t);
    }
  } else if (pr < pairs) {
    if (lane < d.k) {
      p = __ldcg(&ws.pos[(size_t)t * d.k + lane]);
      gj = __ldcg(&ws.topk_gate[(size_t)t * d.k + lane]);
    }
    if constexpr (kShared) sg = __ldcg(&ws.shared_gate[t]);
  }
  pdl_wait_primary();
  // The next call's routing is not signalled early: its CTAs would compete
  // for SMs with this grid's (and, with 8-token routing clusters, wait for
  // whole GPCs), which cost up to 7 us at B = 288, m' = 32.  It starts when
  // this grid ends.
  if (pr < pairs) {
    if constexpr (kShared && kLocal) sg = __ldcg(&ws.shared_gate[t]);  // written by the FFN
    combine_token<kShared>(ws, d, out, t, pr - t * t2, lane, p, gj, sg);
  }
}

// Dynamic shared memory of a combine CTA: the local grouping's masks and bases.
size_t combine_smem_bytes(const Dims &d) {
  return d.local ? (size_t)d.E * (local_words(d) * 4 + 2) : 0;
}

cudaError_t launch_combine(Dims d, Ws ws, __nv_bfloat16 *out, bool pdl, cudaStream_t stream) {
  const int pairs = d.B * (d.H / kCombineTile);
  const int wpc = kCombineThreads / 32;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((pairs + wpc - 1) / wpc);
  cfg.blockDim = dim3(kCombineThreads);
  const int words = local_words(d);
  cfg.dynamicSmemBytes = combine_smem_bytes(d);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  auto kernel = d.Is > 0 ? (words == 2   ? combine_kernel<true, 2>
                            : words == 4 ? combine_kernel<true, 4>
                                         : combine_kernel<true, 0>)
                         : (words == 2   ? combine_kernel<false, 2>
                            : words == 4 ? combine_kernel<false, 4>
                                         : combine_kernel<false, 0>);
  return cudaLaunchKernelEx(&cfg, kernel, d, ws, out);
}

int ffn_stages_for(const Dims &d, size_t smem_limit) {
  const int words = local_words(d);
  int s = 12;
  while (s > 2 && ffn_smem_plan(d.tok_chunk, s, d.wide, d.pair, d.E, words).total + 1024 > smem_limit) --s;
  return s;
}

// Clusters of two FFN CTAs that can be resident at once (the pairs' SMs must
// share a GPC), kept per kernel, device and shared-memory size.
cudaError_t pair_clusters_resident(const void *kernel, size_t smem, int dev, int *n) {
  thread_local const void *last_kernel = nullptr;
  thread_local int last_dev = -1;
  thread_local size_t last_smem = 0;
  thread_local int last_n = 0;
  if (kernel == last_kernel && dev == last_dev && smem == last_smem) {
    *n = last_n;
    return cudaSuccess;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2);
  cfg.blockDim = dim3(kFfnThreads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int c = 0;
  cudaError_t err = cudaOccupancyMaxActiveClusters(&c, kernel, &cfg);
  if (err != cudaSuccess) return err;
  if (c < 1) return cudaErrorInvalidConfiguration;
  last_kernel = kernel;
  last_dev = dev;
  last_smem = smem;
  last_n = c;
  *n = c;
  return cudaSuccess;
}

cudaError_t launch_expert_ffn(const FfnMaps &maps, const __nv_bfloat16 *hidden,
                              const float *w_shared_gate, Dims d, Ws ws,
                              const int32_t *retained, int grid, bool pdl,
                              cudaStream_t stream, uint64_t timeout_ns,
                              int starve_first_down) {
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  int optin = 0, sms = 0;
  err = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (err != cudaSuccess) return err;
  err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (err != cudaSuccess) return err;
  // the token maps exist for boxes of 16 (m + 1) <= tok_chunk rows, and an
  // entry's box covers at most tok_chunk rows: tok_chunk must be a multiple
  // of 16 in [16, 256]
  if (d.tok_chunk < kTokBox || d.tok_chunk > kMaxTokTile || d.tok_chunk % kTokBox != 0)
    return cudaErrorInvalidValue;
  // every byte the block may opt into goes to pipeline stages, whether or not
  // that leaves room for a CTA of the dependent combine kernel (whose shared
  // memory is the local grouping's): a stage less for its sake cost 0.4-1.4 us
  // at 65-80 tokens (Qwen-class, m' = 64 and 128)
  const int stages = ffn_stages_for(d, (size_t)optin);
  const size_t smem =
      ffn_smem_plan(d.tok_chunk, stages, d.wide, d.pair, d.E, local_words(d)).total + 1024;
  if (smem > (size_t)optin) return cudaErrorInvalidConfiguration;
  // wide items only without a shared expert, on whole 256-row tiles, with
  // both accumulators of two buffers in the 512 TMEM columns
  if (d.wide && (d.Is > 0 || d.I % (2 * kGateRows) != 0 || d.H % (2 * kTileRows) != 0 ||
                 d.tok_chunk > 128))
    return cudaErrorInvalidValue;
  // pair items likewise, and never together with wide ones
  if (d.pair && (d.wide || d.Is > 0 || d.I % (2 * kGateRows) != 0 || d.H % (2 * kTileRows) != 0))
    return cudaErrorInvalidValue;
  const bool ahead = d.tok_chunk >= kAheadMinChunk;
  const int words = local_words(d);
  auto kernel = d.Is > 0 ? (words == 2  ? expert_ffn_kernel<true, false, false, false, 2>
                            : words == 4 ? expert_ffn_kernel<true, false, false, false, 4>
                            : ahead      ? expert_ffn_kernel<true, false, false, true, 0>
                                         : expert_ffn_kernel<true, false, false, false, 0>)
                : words == 2 ? expert_ffn_kernel<false, false, false, false, 2>
                : words == 4 ? expert_ffn_kernel<false, false, false, false, 4>
                : d.pair     ? expert_ffn_kernel<false, false, true, false, 0>
                : d.wide     ? expert_ffn_kernel<false, true, false, false, 0>
                : ahead      ? expert_ffn_kernel<false, false, false, true, 0>
                             : expert_ffn_kernel<false, false, false, false, 0>;
  // one value for every call: the attribute is the kernel's, not the launch's,
  // and another thread may be launching it with another size
  err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (err != cudaSuccess) return err;
  int tmem_cols = 32;
  while (tmem_cols < 2 * ffn_acc_cols(d)) tmem_cols <<= 1;

  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kFfnThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  int na = 0;
  if (pdl) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  // items are assigned statically to first CTAs only if all of them are
  // resident at once (a down item may wait on another CTA's first item)
  int resident = sms;
  if (d.pair) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = 2;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = 1;
    ++na;
    int clusters = 0;
    err = pair_clusters_resident((const void *)kernel, smem, dev, &clusters);
    if (err != cudaSuccess) return err;
    resident = 2 * clusters;
    // whole pairs, no more than fit at once
    grid &= ~1;
    if (grid > resident) grid = resident;
    if (grid < 2) grid = 2;
    cfg.gridDim = dim3(grid);
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  const int static_first = grid <= resident ? 1 : 0;
  // The combine is signalled early above 64 tokens, but a locally grouping one
  // only where its CTAs find room beside these: signalled without room (65-80
  // tokens) it was later than after the last item.  Early / after, us: H = 512,
  // 1024 experts 45.1 / 35.1 (m' = 256), H = 2048, 1024 experts 100.1 / 91.8,
  // Qwen-class m' = 128 172.9 / 171.7, m' = 32 54.8 / 54.2.  Where there is
  // room (81-96 tokens) early is the better for short rows (H = 512, 1024
  // experts 32.6 / 35.8), within 0.4 us with up to 256 experts, and the worse
  // with 1024 experts at H = 2048 (101.7 / 95.6).
  int early_dependents = d.B > 64 ? 1 : 0;
  if (early_dependents && d.local) {
    int sm_smem = 0, reserved = 0;  // an SM's, and what each CTA takes besides its own
    err = cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (err != cudaSuccess) return err;
    err = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    if (err != cudaSuccess) return err;
    if (smem + combine_smem_bytes(d) + 2 * (size_t)reserved > (size_t)sm_smem) early_dependents = 0;
  }
  return cudaLaunchKernelEx(&cfg, kernel, maps, hidden, w_shared_gate, d, ws, retained, stages,
                            tmem_cols, static_first, early_dependents, timeout_ns, starve_first_down);
}

}  // namespace slimwise
