// Dispatch of a forward over 32-token chunks:
//   dispatch_bits_kernel   (more than 512 tokens) the chunk's token bitmap per expert
//                          (bits[c][e]: bit l for token 32c + l), one CTA per chunk
//   dispatch_place_kernel  every CTA finds, per expert, its pairs and those of the chunks
//                          before its own (from the bitmaps, or from all ids itself), and by a
//                          scan over the experts their rows' offsets; each (token, slot) of its
//                          chunk goes to row offset[e] + pairs before the chunk + the popcount
//                          of bits[c][e] below its token. The first CTA writes the offsets, the
//                          unique list and U. In the fused layer call it also copies the x rows
//                          into dispatch order (16 CTAs per chunk)
// No launch waits for the last CTA of another (a ticket and a second phase in one CTA took 3 us):
// the counts are cheap enough to be made in every CTA.
// Every sum is of integers, and each expert's rows are ordered by token, the canonical
// dispatch form. An id outside [0, E) or an expert twice in one token is recorded as a fault;
// the outputs are then unspecified: every pos is in range, some entries of rows are not written.
#include "block_reduce.cuh"
#include "dmoe_internal.cuh"
#include "trace_log.cuh"

namespace dmoe {
namespace {

constexpr int kDispThreads = 256;
constexpr int kDispPerThread = (32 * kMaxTopK + kDispThreads - 1) / kDispThreads;
// Forwards of up to this many tokens take one launch: every CTA counts all T k ids itself (8 KB
// at 256 tokens and k = 8), instead of reading bitmaps that a launch before it has written
// (256 tokens: 9.4 us in two launches, 5.1 in one; with bitmaps, T / 32 words per expert are
// read instead, the shorter way for large T).
constexpr int kOneLaunchTokens = 512;

// The id's bit in the chunk's bitmaps (token l of the chunk). `check`: record ids out of range
// and experts that a token has twice.
__device__ __forceinline__ void add_bit(uint32_t* bits, int e, int l, int E, bool check,
                                        DevErrRecord* err, int i) {
  if (e < 0 || e >= E) {
    if (check) record_error(err, kErrExpertId, kAtDispatch, i);
    return;
  }
  if ((atomicOr(&bits[e], 1u << l) & (1u << l)) != 0u && check)
    record_error(err, kErrDupExpert, kAtDispatch, i);
}

// Large forwards: the chunk's token bitmap per expert.
__global__ void __launch_bounds__(kDispThreads)
dispatch_bits_kernel(const int32_t* __restrict__ topk_idx, int T, int E, int k,
                     uint32_t* __restrict__ gbits, DevErrRecord* err) {
  __shared__ uint32_t bits[kMaxExperts];
  const int c = blockIdx.x, tid = threadIdx.x;
  const int t0 = c * 32, ntok = T - t0 < 32 ? T - t0 : 32, np = ntok * k;
  // the next launch reads the routing too: it may start once every CTA is past this wait
  pdl_wait();
  pdl_launch_dependents();
  KLOG(DMOE_KERNEL_DISPATCH, 0);
  int ids[kDispPerThread];
#pragma unroll
  for (int j = 0; j < kDispPerThread; ++j) {
    const int p = tid + j * kDispThreads;
    ids[j] = p < np ? topk_idx[t0 * k + p] : 0;
  }
  for (int e = tid; e < E; e += kDispThreads) bits[e] = 0u;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kDispPerThread; ++j) {
    const int p = tid + j * kDispThreads;
    if (p < np) add_bit(bits, ids[j], p / k, E, true, err, t0 * k + p);
  }
  __syncthreads();
  for (int e = tid; e < E; e += kDispThreads) gbits[(size_t)c * E + e] = bits[e];
  KLOG(DMOE_KERNEL_DISPATCH, 1);
}

// Placement of chunk blockIdx.x; with xperm, blockIdx.y takes its share of the chunk's
// (token, slot) pairs and also copies their x rows into dispatch order (kGatherRows rows
// in flight per thread). Every CTA finds the experts' row offsets and the rows of the chunks
// before its own: from the chunks' bitmaps, or (kOneLaunch) from all ids.
constexpr int kPlaceSplit = 16;    // CTAs per chunk when the rows are copied too
constexpr int kGatherRows = 8;
template <bool kOneLaunch>
__global__ void __launch_bounds__(kDispThreads)
dispatch_place_kernel(const int32_t* __restrict__ topk_idx, int T, int E, int k,
                      const uint32_t* __restrict__ gbits, int32_t* __restrict__ n_unique,
                      int32_t* __restrict__ unique_ids, int32_t* __restrict__ offsets,
                      int32_t* __restrict__ rows, int32_t* __restrict__ pos,
                      const __nv_bfloat16* __restrict__ x, __nv_bfloat16* __restrict__ xperm,
                      int d, int32_t* zero, int n_zero, DevErrRecord* err) {
  __shared__ uint32_t bits[kMaxExperts];
  __shared__ int base[kMaxExperts];
  __shared__ int iscr[32];
  __shared__ int s_r[32 * kMaxTopK], s_t[32 * kMaxTopK];
  const int c = blockIdx.x, tid = threadIdx.x, nchunks = gridDim.x;
  const int t0 = c * 32, ntok = T - t0 < 32 ? T - t0 : 32, np = ntok * k;
  const int pairs = T * k;
  const bool first = c == 0 && blockIdx.y == 0;
  // this CTA's pairs of the chunk
  const int per = (np + gridDim.y - 1) / gridDim.y;
  const int p0 = blockIdx.y * per, p1 = p0 + per < np ? p0 + per : np;
  pdl_wait();
  // The next launch may start; the first CTA lets it only once the unique list is written (the
  // expert launch reads it before its own dependency wait).
  if (!first) pdl_launch_dependents();
  KLOG(7, 0);
  int ids[kDispPerThread];
#pragma unroll
  for (int j = 0; j < kDispPerThread; ++j) {
    const int p = p0 + tid + j * kDispThreads;
    ids[j] = p < p1 ? __ldcg(topk_idx + t0 * k + p) : 0;
  }
  // pairs per expert, and those in the chunks before this one
  int cnt = 0, before = 0;
  if (kOneLaunch) {
    base[tid] = 0;
    bits[tid] = 0u;
    __syncthreads();
    const bool check = blockIdx.y == 0;
    for (int i0 = 0; i0 < pairs; i0 += 8 * kDispThreads) {
      int e[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int i = i0 + tid + j * kDispThreads;
        e[j] = i < pairs ? __ldcg(topk_idx + i) : -1;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int i = i0 + tid + j * kDispThreads, p = i - t0 * k;
        if (p >= 0 && p < np) add_bit(bits, e[j], p / k, E, check, err, i);
        // (at most 512 * 16 pairs: both counts fit one word)
        if (e[j] >= 0 && e[j] < E) atomicAdd(&base[e[j]], p < 0 ? 0x10001 : 1);
      }
    }
    __syncthreads();
    cnt = base[tid] & 0xffff;
    before = base[tid] >> 16;
  } else if (tid < E) {
    bits[tid] = __ldcg(gbits + (size_t)c * E + tid);
    for (int c0 = 0; c0 < nchunks; c0 += 32) {
      uint32_t w[32];   // one round of loads per 32 chunks
#pragma unroll
      for (int j = 0; j < 32; ++j)
        w[j] = c0 + j < nchunks ? __ldcg(gbits + (size_t)(c0 + j) * E + tid) : 0u;
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const int n = __popc(w[j]);
        cnt += n;
        before += c0 + j < c ? n : 0;
      }
    }
  }
  // rows before each expert's (at most 65536: 20 bits) and the experts with rows before it, in
  // one scan
  static_assert(kMaxTokens * kMaxTopK < (1 << 20) && kMaxExperts < (1 << 11), "packed scan");
  int total = 0;
  const int present = cnt > 0 ? 1 : 0;
  const int scan = block_exclusive_scan_i(cnt | present << 20, iscr, &total);
  const int off = scan & 0xfffff;
  base[tid] = off + before;
  if (first) {
    const int upos = scan >> 20, n_u = total >> 20, total_pairs = total & 0xfffff;
    if (present) {
      unique_ids[upos] = tid;
      offsets[upos] = off;
    }
    for (int u = n_u + tid; u < E; u += kDispThreads) unique_ids[u] = -1;
    for (int u = n_u + tid; u <= E; u += kDispThreads) offsets[u] = pairs;
    if (tid == 0) {
      n_unique[0] = n_u;
      if (total_pairs != pairs) record_error(err, kErrBadDispatch, kAtDispatch, total_pairs);
    }
    __threadfence();
    __syncthreads();
    pdl_launch_dependents();
    if (zero != nullptr)
      for (int i = tid; i < n_zero; i += kDispThreads) zero[i] = 0;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kDispPerThread; ++j) {
    const int p = p0 + tid + j * kDispThreads;
    const int e = ids[j];
    int r = -1;
    if (p < p1 && e >= 0 && e < E) {
      const int i = t0 * k + p, l = (i / k) & 31;
      r = base[e] + __popc(bits[e] & ((1u << l) - 1u));
      if (r >= 0 && r < pairs) {
        rows[r] = i;
        pos[i] = r;
      } else {
        r = -1;
      }
    }
    // (a bad id has no row; its place is one that the combine can read. Checked there instead, it
    // took the combine of 2048 tokens 2 us longer)
    if (r < 0 && p < p1) pos[t0 * k + p] = 0;
    if (xperm != nullptr && p < p1) {
      s_r[p - p0] = r;
      s_t[p - p0] = t0 + p / k;
    }
  }
  if (xperm != nullptr) {
    __syncthreads();
    const int n = p1 - p0, vec = d / 8;   // rows, 16-byte pieces per row
    const uint4* src = reinterpret_cast<const uint4*>(x);
    uint4* dst = reinterpret_cast<uint4*>(xperm);
    for (int q0 = 0; q0 < n; q0 += kGatherRows)
      for (int i = tid; i < vec; i += kDispThreads) {
        uint4 v[kGatherRows];
#pragma unroll
        for (int q = 0; q < kGatherRows; ++q)
          if (q0 + q < n && s_r[q0 + q] >= 0) v[q] = src[(size_t)s_t[q0 + q] * vec + i];
#pragma unroll
        for (int q = 0; q < kGatherRows; ++q)
          if (q0 + q < n && s_r[q0 + q] >= 0) dst[(size_t)s_r[q0 + q] * vec + i] = v[q];
      }
  }
  KLOG(7, 1);
}

}  // namespace

int dispatch_launches(int T) { return T <= kOneLaunchTokens ? 1 : 2; }

cudaError_t launch_dispatch(const DispatchArgs& a, cudaStream_t s) {
  if (a.bits == nullptr || a.k > kMaxTopK || a.E > kMaxExperts ||
      (a.xperm != nullptr && (a.x == nullptr || a.d % 8)))
    return cudaErrorInvalidValue;
  const int nchunks = (a.T + 31) / 32;
  const bool one = dispatch_launches(a.T) == 1;
  static std::atomic<uint32_t> carveout[2];
  cudaError_t e = one ? max_shared_carveout(dispatch_place_kernel<true>, carveout[1])
                      : max_shared_carveout(dispatch_place_kernel<false>, carveout[0]);
  if (e != cudaSuccess) return e;
  prof_begin(DMOE_KERNEL_DISPATCH, s);
  if (!one)
    e = launch_ex(dispatch_bits_kernel, dim3(nchunks), dim3(kDispThreads), 0, s, true, a.topk_idx,
                  a.T, a.E, a.k, a.bits, a.err);
  if (e == cudaSuccess)
    e = launch_ex(one ? dispatch_place_kernel<true> : dispatch_place_kernel<false>,
                  dim3(nchunks, a.xperm != nullptr ? kPlaceSplit : 1), dim3(kDispThreads), 0, s,
                  true, a.topk_idx, a.T, a.E, a.k, static_cast<const uint32_t*>(a.bits),
                  a.n_unique, a.unique_ids, a.offsets, a.rows, a.pos, a.x, a.xperm, a.d, a.zero,
                  a.n_zero, a.err);
  prof_end(DMOE_KERNEL_DISPATCH, s);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace dmoe

#ifdef DMOE_TRACE
DMOE_KLOG_EXPORT(dmoe_debug_klog_dispatch)
#endif
