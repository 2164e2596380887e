// compact_layer.cu -- the compact (pruned) checkpoint of one MoE layer.
//
// A decode instance that serves from the pruned pool K' needs only the m'
// retained experts' weights and router rows (SlimWise Sec. 3.1: the Eq. 2
// router mask and a checkpoint holding only K' are two forms of the same
// layer).  These kernels build that form on the device from the full layer:
//   compact_ids_kernel   the retained ids in ascending order (one CTA; the
//                        rank of an id is the number of smaller ids), so
//                        top-k ties in the compact numbering still go to the
//                        lowest original id;
//   compact_copy_kernel  for compact expert j = original expert ids[j]: its
//                        [2I, H] gate/up rows, [H, I] down rows and router
//                        row, one 16 KB block per CTA, with streaming
//                        (evict-first) loads and stores -- a pure copy, bound
//                        by HBM at 2 x (m' x expert bytes).  One contiguous
//                        block per CTA and no loop keeps the memory system
//                        fed by whole CTAs coming and going: 64 Qwen-class
//                        experts (1.2 GB both ways) 208 -> 178 us; four CTAs per SM
//                        striding over the experts reached 5.9 TB/s, a ring
//                        of bulk copies through shared memory 6.4-6.8.
// A repeated or out-of-range id sets every entry of ids to -1, and then the
// copy kernel writes nothing.
#include "common.cuh"

namespace slimwise {

constexpr int kIdsThreads = 1024;   // >= kMaxExperts: one id per thread
constexpr int kCopyThreads = 256;
constexpr int kCopyVecs = 4;        // 16-byte vectors per thread
constexpr int kCopyBlock = kCopyThreads * kCopyVecs;  // vectors per CTA (16 KB)

__global__ void __launch_bounds__(kIdsThreads)
    compact_ids_kernel(const int32_t *__restrict__ retained, int m, int E,
                       int32_t *__restrict__ ids_c) {
  __shared__ int ids[kMaxExperts];
  __shared__ int bad;
  pdl_launch_dependents();
  const int i = threadIdx.x;
  if (i == 0) bad = 0;
  if (i < m) ids[i] = retained[i];
  __syncthreads();
  int rank = 0, same = 0;
  if (i < m) {
    const int e = ids[i];
    for (int j = 0; j < m; ++j) {
      rank += ids[j] < e ? 1 : 0;
      same += ids[j] == e ? 1 : 0;
    }
    if (e < 0 || e >= E || same != 1) bad = 1;
  }
  __syncthreads();
  if (i < m) {
    if (bad) ids_c[i] = -1;
    else ids_c[rank] = ids[i];
  }
}

// blockIdx.y = compact expert j; the CTAs of row j take its blocks in turn:
// gate/up, down, router row (a multiple of 32 vectors, the others of 1024).
__global__ void __launch_bounds__(kCopyThreads)
    compact_copy_kernel(const uint4 *__restrict__ w_gu, const uint4 *__restrict__ w_d,
                        const uint4 *__restrict__ wr, const int32_t *__restrict__ ids_c,
                        size_t gu_vecs, size_t d_vecs, size_t wr_vecs, uint4 *__restrict__ gu_c,
                        uint4 *__restrict__ d_c, uint4 *__restrict__ wr_c) {
  pdl_wait_primary();
  const size_t j = blockIdx.y;
  const int e = __ldcg(ids_c + j);
  if (e < 0) return;  // repeated or out-of-range ids: nothing is copied
  size_t i = (size_t)blockIdx.x * kCopyBlock, n = gu_vecs;
  const uint4 *src = w_gu;
  uint4 *dst = gu_c;
  if (i >= gu_vecs + d_vecs) {
    i -= gu_vecs + d_vecs;
    n = wr_vecs;
    src = wr;
    dst = wr_c;
  } else if (i >= gu_vecs) {
    i -= gu_vecs;
    n = d_vecs;
    src = w_d;
    dst = d_c;
  }
  i += threadIdx.x;
  src += (size_t)e * n;
  dst += j * n;
  uint4 v[kCopyVecs];
#pragma unroll
  for (int u = 0; u < kCopyVecs; ++u)
    if (i + u * kCopyThreads < n) v[u] = __ldcs(src + i + u * kCopyThreads);
#pragma unroll
  for (int u = 0; u < kCopyVecs; ++u)
    if (i + u * kCopyThreads < n) __stcs(dst + i + u * kCopyThreads, v[u]);
}

cudaError_t launch_compact_layer(const void *w_gate_up, const void *w_down, const float *router_w,
                                 const int32_t *retained, int m, int E, int H, int I,
                                 void *w_gate_up_c, void *w_down_c, float *router_w_c,
                                 int32_t *ids_c, cudaStream_t stream) {
  compact_ids_kernel<<<1, kIdsThreads, 0, stream>>>(retained, m, E, ids_c);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  // bytes per expert: 2I x H and H x I bf16, H fp32 -- multiples of 16
  // bytes, since H is a multiple of 128 and I of 64
  const size_t gu_vecs = (size_t)2 * I * H * 2 / 16;
  const size_t d_vecs = (size_t)H * I * 2 / 16;
  const size_t wr_vecs = (size_t)H * 4 / 16;
  // gate/up and down are whole blocks
  static_assert(2 * 64 * 128 / 8 % kCopyBlock == 0 && 64 * 128 / 8 % kCopyBlock == 0, "blocks");
  const dim3 grid((unsigned)(gu_vecs / kCopyBlock + d_vecs / kCopyBlock +
                             (wr_vecs + kCopyBlock - 1) / kCopyBlock),
                  (unsigned)m);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kCopyThreads);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, compact_copy_kernel, static_cast<const uint4 *>(w_gate_up),
                            static_cast<const uint4 *>(w_down),
                            reinterpret_cast<const uint4 *>(router_w), (const int32_t *)ids_c,
                            gu_vecs, d_vecs, wr_vecs, static_cast<uint4 *>(w_gate_up_c),
                            static_cast<uint4 *>(w_down_c), reinterpret_cast<uint4 *>(router_w_c));
}

}  // namespace slimwise
