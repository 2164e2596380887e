// expert_stats.cu -- expert-importance statistics of a calibration pass and
// the retained set they select (SlimWise Sec. 2.3 and Sec. 3.1).
//
// The statistics are taken from a full-pool layer call: its workspace holds,
// for every (token, selection) slot in grouped order (expert ascending, token
// ascending), the selected expert's output row y (accumulated in fp32, stored
// as bf16) and, through perm, the slot's gate.  For each expert e and each token t routed to it:
//   stats[e][0] += 1             tokens routed to e
//   stats[e][1] += g_te          routing mass
//   stats[e][2] += ||y||_2       expert activation norm (EAN)
//   stats[e][3] += g_te ||y||_2  REAP numerator (score = stats[3] / stats[0])
// Two kernels: row_norms_kernel reads y once, one warp per row, so that the
// whole GPU streams it however the rows spread over experts;
// expert_sums_kernel then adds each expert's rows up, one CTA per expert.
// Bound by the read of y (B k H bf16).  Against one warp walking each
// expert's rows in turn (a memory round trip per row on E / 8 CTAs), the pass
// over a Qwen-class calibration batch of 2048 tokens went from 396 us to
// 13 us, and a popular expert's rows no longer set the time.
//
// Every expert's sums are taken in fp64 in one fixed order: thread i adds its
// rows i, i + 128, ... in token order, then the 128 partial sums meet in a
// butterfly over each warp's lanes and a sum over the warps in turn.  They
// accumulate in fp64 across calibration batches.
#include "common.cuh"

namespace slimwise {

constexpr int kNormWarps = 8;
constexpr int kSumThreads = 128;

// norm2[p] = ||y_p||^2 of grouped row p: lane l sums its 8-wide columns
// 256c + 8l .. +7 by fmaf in column order, then an xor butterfly.  A lane's
// loads of 8 steps (a whole row at H = 2048) are issued before any is used.
__global__ void __launch_bounds__(kNormWarps * 32)
    row_norms_kernel(Dims d, Ws ws, float *__restrict__ norm2, int slots) {
  pdl_wait_primary();
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31;
  const int p = blockIdx.x * kNormWarps + (threadIdx.x >> 5);
  if (p >= slots) return;
  const uint4 *row = reinterpret_cast<const uint4 *>(ws.y + (size_t)p * d.H);
  const int vecs = d.H / 8;
  constexpr int kBatch = 8;
  float s = 0.0f;
  for (int c0 = lane; c0 < vecs; c0 += 32 * kBatch) {
    uint4 v[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
      if (c0 + 32 * u < vecs) v[u] = __ldcg(row + c0 + 32 * u);
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      if (c0 + 32 * u < vecs) {
        const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float a = __uint_as_float(w[q] << 16), b = __uint_as_float(w[q] & 0xFFFF0000u);
          s = fmaf(a, a, s);
          s = fmaf(b, b, s);
        }
      }
    }
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
  if (lane == 0) norm2[p] = s;
}

__global__ void __launch_bounds__(kSumThreads)
    expert_sums_kernel(Ws ws, const float *__restrict__ norm2, double *__restrict__ stats,
                       int slots) {
  __shared__ double part[kSumThreads / 32][3];
  pdl_wait_primary();
  const int e = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int p0 = __ldcg(&ws.offsets[e]), p1 = __ldcg(&ws.offsets[e + 1]);
  double mass = 0.0, ean = 0.0, reap = 0.0;
  for (int p = p0 + threadIdx.x; p < p1; p += kSumThreads) {
    const double nrm = sqrt((double)__ldcg(norm2 + p));
    // (a position that no slot took, after a token with repeated selections,
    // holds anything: kept inside the batch)
    const uint32_t s = min((uint32_t)__ldcg(&ws.perm[p]), (uint32_t)slots - 1u);
    const double g = (double)__ldcg(&ws.topk_gate[s]);
    mass += g;
    ean += nrm;
    reap += g * nrm;
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    mass += __shfl_xor_sync(0xFFFFFFFFu, mass, off);
    ean += __shfl_xor_sync(0xFFFFFFFFu, ean, off);
    reap += __shfl_xor_sync(0xFFFFFFFFu, reap, off);
  }
  if (lane == 0) {
    part[warp][0] = mass;
    part[warp][1] = ean;
    part[warp][2] = reap;
  }
  __syncthreads();
  // one thread per statistic of the expert
  if (threadIdx.x < 4) {
    double v = 0.0;
    if (threadIdx.x == 0) v = (double)(p1 - p0);
    else
      for (int w = 0; w < kSumThreads / 32; ++w) v += part[w][threadIdx.x - 1];
    stats[(size_t)e * 4 + threadIdx.x] += v;
  }
}

// The squared norms go where the call's activations were (the FFN is done
// with them): 4 bytes a row against at least 128.
cudaError_t launch_expert_stats(Dims d, Ws ws, double *stats, cudaStream_t stream) {
  float *norm2 = reinterpret_cast<float *>(ws.act);
  const int slots = d.B * d.k;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((slots + kNormWarps - 1) / kNormWarps);
  cfg.blockDim = dim3(kNormWarps * 32);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t err = cudaLaunchKernelEx(&cfg, row_norms_kernel, d, ws, norm2, slots);
  if (err != cudaSuccess) return err;
  cfg.gridDim = dim3(d.E);
  cfg.blockDim = dim3(kSumThreads);
  return cudaLaunchKernelEx(&cfg, expert_sums_kernel, ws, (const float *)norm2, stats, slots);
}

// Retained set: the m' experts of highest score, ties to the lowest id, ids
// ascending.  Scores: 0 routing mass, 1 EAN, 2 REAP (numerator / count, 0 for
// an expert no token chose).  One CTA; each thread ranks its expert against
// all others, then a block scan compacts the kept ids.  Scores are ranked as
// order-preserving 64-bit integers: comparing the doubles themselves on
// GB300's few fp64 units took 13.5 us for 128 experts, 3.7 us so.
__device__ __forceinline__ double expert_score(const double *st, int criterion) {
  if (criterion == 0) return st[1];
  if (criterion == 1) return st[2];
  return st[0] > 0.0 ? st[3] / st[0] : 0.0;
}

// Order-preserving map of a double (-0 folded onto +0).  A NaN compares false
// with everything: it outranks no expert (0 is below every number's key) and
// none outranks it (the caller gives it rank 0).
__device__ __forceinline__ unsigned long long score_key(double v) {
  unsigned long long b = (unsigned long long)__double_as_longlong(v);
  if ((b << 1) == 0ull) b = 0ull;
  if ((b & 0x7FFFFFFFFFFFFFFFull) > 0x7FF0000000000000ull) return 0ull;
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

__global__ void __launch_bounds__(kMaxExperts)
    select_retained_kernel(const double *__restrict__ stats, int E, int m_prime,
                           int criterion, int32_t *__restrict__ ids) {
  __shared__ unsigned long long score[kMaxExperts];
  __shared__ int warp_sum[kMaxExperts / 32];
  const int e = threadIdx.x;
  if (e < E) score[e] = score_key(expert_score(stats + (size_t)e * 4, criterion));
  __syncthreads();
  int keep = 0;
  if (e < E) {
    const unsigned long long se = score[e];
    int rank = 0;
    if (se != 0ull)
      for (int f = 0; f < E; ++f) {
        const unsigned long long sf = score[f];
        rank += (sf > se || (sf == se && f < e)) ? 1 : 0;
      }
    keep = rank < m_prime ? 1 : 0;
  }
  // exclusive scan of keep over the block: warp inclusive scans, then warp totals
  const int lane = e & 31, w = e >> 5;
  int incl = keep;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int o = __shfl_up_sync(0xFFFFFFFFu, incl, off);
    if (lane >= off) incl += o;
  }
  if (lane == 31) warp_sum[w] = incl;
  __syncthreads();
  if (w == 0) {
    const int nw = blockDim.x / 32;
    int v = lane < nw ? warp_sum[lane] : 0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int o = __shfl_up_sync(0xFFFFFFFFu, v, off);
      if (lane >= off) v += o;
    }
    if (lane < nw) warp_sum[lane] = v;  // inclusive totals
  }
  __syncthreads();
  const int before = (w > 0 ? warp_sum[w - 1] : 0) + incl - keep;
  // NaN scores can keep more than m': the lowest ids are written
  if (keep && before < m_prime) ids[before] = e;
}

cudaError_t launch_select_retained(const double *stats, int E, int m_prime, int criterion,
                                   int32_t *ids, cudaStream_t stream) {
  const int threads = (E + 31) / 32 * 32;
  select_retained_kernel<<<1, threads, 0, stream>>>(stats, E, m_prime, criterion, ids);
  return cudaGetLastError();
}

}  // namespace slimwise
