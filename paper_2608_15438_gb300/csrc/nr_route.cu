// K2 route: binarisation (Eq. 10), deviation scores (Sec. 3.2.3) and the
// probe list of Algorithm 1: one block per query by threshold enumeration
// (nrq::route_block) without the R_max filter, else one warp per query
// (nrq::route_warp).
#include <cuda_runtime.h>
#include <stdint.h>

#include "nr_internal.cuh"
#include "nrq_route.cuh"

namespace {

__global__ void route_kernel(nrq::RouteParams rp, const float *__restrict__ logits, int64_t nq,
                             uint32_t *__restrict__ codes, int32_t *__restrict__ nprobe) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  const int64_t q = (int64_t)blockIdx.x * wpb + warp;
  if (q >= nq) return;  // uniform per warp
  unsigned char *heap = smem + (size_t)warp * nrq::route_heap_bytes(rp.Q);
  uint32_t *out = codes + (size_t)q * rp.P;
  const int n = nrq::route_warp(rp, logits + q * rp.b, heap, out);
  for (int t = n + lane; t < rp.P; t += 32) out[t] = 0xffffffffu;
  if (lane == 0) nprobe[q] = n;
}

// One block of NT threads per query: the threshold enumeration (route_block) of
// N flip sets and, where a non-empty budget needs more, of N2 (0: the heap).
// RETRY: the block has the shared memory for N2 and goes on itself; else the
// query is left to route_more_kernel (nprobe -1).
// logits are not __restrict__: an early launch begins while the encoder still
// writes them, and loads of such data may not take the read-only path.
template <int NT, bool RETRY>
__global__ void __launch_bounds__(NT) route_block_kernel(nrq::RouteParams rp, const float *logits,
                                                         int64_t nq, uint32_t *codes,
                                                         int32_t *nprobe, int N, int N2) {
  extern __shared__ __align__(16) unsigned char smem[];
  nr_let_next();
  nr_after_previous();
  const int64_t q = blockIdx.x;
  if (q >= nq) return;
  uint32_t *out = codes + (size_t)q * rp.P;
  int n;
  if constexpr (RETRY) {
    for (bool more = true;; more = false) {
      n = nrq::route_block<NT>(rp, logits + q * rp.b, smem, out, more ? N : N2, more);
      if (n >= 0) break;
      __syncthreads();
    }
  } else {
    n = nrq::route_block<NT>(rp, logits + q * rp.b, smem, out, N, N2 > 0);
  }
  if (threadIdx.x == 0) nprobe[q] = n;
  if (n < 0) return;
  for (int t = n + (int)threadIdx.x; t < rp.P; t += NT) out[t] = 0xffffffffu;
}

// The queries that route_block_kernel left, one block an SM.
__global__ void __launch_bounds__(nrq::kRouteFewThreads) route_more_kernel(
    nrq::RouteParams rp, const float *__restrict__ logits, int64_t nq, uint32_t *__restrict__ codes,
    int32_t *__restrict__ nprobe, int N) {
  extern __shared__ __align__(16) unsigned char smem[];
  for (int64_t q = blockIdx.x; q < nq; q += gridDim.x) {
    if (nprobe[q] >= 0) continue;  // uniform: only this block writes it
    uint32_t *out = codes + (size_t)q * rp.P;
    const int n = nrq::route_block<nrq::kRouteFewThreads>(rp, logits + q * rp.b, smem, out, N, false);
    for (int t = n + (int)threadIdx.x; t < rp.P; t += nrq::kRouteFewThreads) out[t] = 0xffffffffu;
    __syncthreads();  // every thread has read nprobe[q] and the block's results
    if (threadIdx.x == 0) nprobe[q] = n;
  }
}

}  // namespace

nrq::RouteParams nr_route_params(const nr_index *ix, int P) {
  const nr_params &p = ix->params;
  nrq::RouteParams rp;
  rp.tau = ix->tau;
  rp.b = ix->b;
  rp.bsel = (p.l_sel > 0 && p.l_sel < ix->b) ? p.l_sel : ix->b;
  rp.rmax = p.r_max;
  rp.smax = p.s_max;
  rp.P = P;
  rp.bkt_off = ix->bkt_off;
  rp.nonempty = p.nonempty_budget;
  rp.Q = p.nonempty_budget ? NR_NONEMPTY_SCAN * P : P;
  return rp;
}

size_t nr_route_heap_bytes(int Q) { return nrq::route_heap_bytes(Q); }

cudaError_t nr_launch_route(nr_index *ix, const float *d_logits, int64_t nq, int P,
                            uint32_t *d_codes, int32_t *d_nprobe, cudaStream_t s, bool early) {
  if (nq <= 0) return cudaSuccess;
  const nrq::RouteParams rpb = nr_route_params(ix, P);  // before the launch configuration
  if (ix->params.r_max <= 0) {  // threshold enumeration
    // Few queries leave SMs to themselves: wider blocks take the walk's and the
    // ranking's strides together (the stage of one query at P = 1024 22 -> 18 us,
    // four 1536-value ones 20 -> 16; at P = 64 14 both; past one block an SM the
    // narrow ones overlap).
    const bool few = nq <= ix->num_sms;
    // Non-empty budgets: 2 P flip sets first, which three blocks an SM hold at P
    // = 1024; where less than half of the buckets are occupied, all 4 P that may
    // be examined, by the same block or, with many queries, a second kernel (100
    // queries at P = 1024, 1e7 rows: 61 us, 3,220 by the heap, one flip set after
    // another; 3,000 queries 808 and 13,280).
    const int N = nrq::route_enum_target(P, rpb.nonempty, rpb.Q);
    const int N2 = nrq::route_enum_more(P, rpb.nonempty, rpb.Q);
    const size_t smem2 = N2 > 0 ? nrq::route_block_bytes(N2, rpb.nonempty, rpb.Q) : 0;
    const size_t smem = few && N2 > 0 ? smem2 : nrq::route_block_bytes(N, rpb.nonempty, rpb.Q);
    constexpr int kFew = nrq::kRouteFewThreads, kMany = nrq::kRouteThreads;
    const auto kern = !few ? route_block_kernel<kMany, false>
                           : N2 > 0 ? route_block_kernel<kFew, true> : route_block_kernel<kFew, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = nr_launch_kernel(kern, (unsigned)nq, few ? kFew : kMany, smem, s, early && few, rpb, d_logits, nq, d_codes,
                         d_nprobe, N, N2);
    ix->launches += 1;
    if (few || N2 == 0 || e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(route_more_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem2);
    if (e != cudaSuccess) return e;
    route_more_kernel<<<(unsigned)ix->num_sms, nrq::kRouteFewThreads, smem2, s>>>(rpb, d_logits, nq, d_codes,
                                                                                 d_nprobe, N2);
    ix->launches += 1;
    return cudaGetLastError();
  }
  const size_t per_warp = nr_route_heap_bytes(rpb.Q);
  // warps per block: the choice that packs the most warps into an SM's
  // shared memory (the heap is the limit at large probe budgets)
  const size_t sm_bytes = (size_t)227 * 1024;
  int wpb = 1, best = 0;
  for (int w = 4; w >= 1; w >>= 1) {
    const size_t blk = per_warp * (size_t)w;
    if (blk > sm_bytes) continue;
    int blocks = (int)(sm_bytes / (blk + 1024));
    if (blocks > 32) blocks = 32;
    const int warps = blocks * w > 64 ? 64 : blocks * w;
    if (warps > best) {
      best = warps;
      wpb = w;
    }
  }
  const size_t smem = per_warp * (size_t)wpb;
  cudaError_t e = cudaFuncSetAttribute(route_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t grid = (nq + wpb - 1) / wpb;
  const nrq::RouteParams rp = nr_route_params(ix, P);  // before the launch configuration
  route_kernel<<<(unsigned)grid, 32 * wpb, smem, s>>>(rp, d_logits, nq,
                                                       d_codes, d_nprobe);
  ix->launches += 1;
  return cudaGetLastError();
}
