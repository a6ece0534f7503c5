// K4 refine (Sec. 3.4, Algorithm 2's T_low rule; uint8 distances kept as
// integers, Sec. 4.1.1), by persistent CTAs that pull work from an atomic
// counter and run nrq::refine_span on the segments K3 wrote to global memory.
// Many queries: a CTA refines a query's whole candidate stream (refine_kernel).
// Few: a plan cuts the streams into spans, which CTAs refine side by side and
// commit in stream order (refine_spans_kernel).
//
// Bound by HBM at large batches, less what queries share in L2, and by latency
// at small ones: one block a query left a single query to one SM (one uint8
// query of 61,900 candidates 523 us, four fp32 queries of 154 MB each 7.8 ms;
// cut into spans 41 us and 0.16 ms, with the commits).
//
// Launch shapes measured on GB300: the scan is limited by the bytes in flight
// per SM, so tiles are small (128 uint8 rows, 32-64 fp32 rows). uint8, D = 128:
// 3 stages and 4 CTAs an SM hold 8 tiles in flight, 2 stages and 6 CTAs 6 but
// more warps (see bound_by_stream; 4 stages and 3 CTAs, 6 and 2 were slower
// than both). fp32, D = 96: 2 stages of 64 rows and 4 CTAs of two warps (4,473
// us a batch of 10,000; 32 rows and 9 CTAs 4,805, 3 stages and 6 CTAs 4,905:
// fewer queries side by side share more, but a row's chain is serial and needs
// the warps).
// Tiles held in registers (eight lanes a 128-byte row, no shared memory) had
// fewer bytes in flight: 14.8 ms for 9.1.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "nr_internal.cuh"
#include "nrq_refine.cuh"

namespace {

constexpr int kPlanThreads = 1024;
constexpr int kOrderBins = 1024;

// How streams are cut.
struct SpanRule {
  int R;
  int align;                // rounds of a span: a multiple of this (whole tiles)
  int rounds_most;          // its rounds when there are items enough
  unsigned int items_want;  // items that keep every CTA busy
  unsigned int items_cap;   // items there is room for (nq: whole streams only)
};

struct PlanArgs {
  const uint32_t *slen;
  int64_t nq;
  SpanRule rule;
  nrq::RefinePlan *plan;
  uint32_t *pre;        // [nq + 1] first item of the i-th query (not of whole streams)
  int32_t *perm;        // processing order of whole streams
  const uint32_t *codes;    // [nq x P] probe codes, the base code first
  int P, b;
  int64_t last;         // whole streams kept for the end, longest first
};

// inclusive prefix of v over the block's threads; *all = the sum
__device__ __forceinline__ uint64_t plan_scan(uint64_t v, uint64_t *wsum, uint64_t *all) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint64_t x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(nrq::kFull, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  uint64_t t = wsum[lane];  // kPlanThreads / 32 = 32 warps
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(nrq::kFull, t, o);
    if (lane >= o) t += y;
  }
  *all = __shfl_sync(nrq::kFull, t, 31);
  const uint64_t before = __shfl_sync(nrq::kFull, t, w > 0 ? w - 1 : 0);
  return x + (w > 0 ? before : 0);
}

// Rows of a span (0xffffffff: whole streams) when the streams have `all` rounds
// in total: rounds that leave the items wanted and fit the room for them, whole
// tiles.
__device__ __forceinline__ uint32_t span_length(uint64_t all, int64_t nq, const SpanRule &r) {
  uint64_t S = min((uint64_t)r.rounds_most, all / r.items_want);
  const uint64_t room = r.items_cap - (uint64_t)nq;
  S = max(S, (all + room - 1) / room);
  S = max((S + r.align - 1) / r.align, (uint64_t)1) * r.align;
  const uint64_t rows = S * (uint64_t)r.R;
  return rows < 0xffffffffull ? (uint32_t)rows : 0xffffffffu;
}
// Items of a stream of n rows.
__device__ __forceinline__ uint32_t spans_of(uint32_t n, uint32_t span) {
  return max(1u, (uint32_t)(((uint64_t)n + span - 1) / span));
}

// One CTA: the rounds of a span and the items of every query, bound by latency
// (5 us for 1 to 1,000 queries).
// Whole streams (items_cap = nq): the queries with the `last` shortest streams
// go at the end, longest first (1024 buckets scaled to the longest stream), so
// that the persistent CTAs finish together; the others go by the top bits of
// their base code, since queries of nearby codes have many clusters in common
// and those that run at the same time read them from L2 (last = nq: longest
// first throughout; see nearby_first for both). Order inside a bucket is
// arbitrary; no order affects any result. Streams cut into spans keep the
// batch's order: their items are short.
__global__ void __launch_bounds__(kPlanThreads) plan_kernel(PlanArgs a) {
  __shared__ uint64_t wsum[32];
  __shared__ unsigned int hist[kOrderBins], hcode[kOrderBins];
  __shared__ unsigned int smax, cut;
  const int tid = threadIdx.x;
  const int64_t nq = a.nq;
  const bool whole = a.rule.items_cap <= nq;
  const int64_t per = (nq + kPlanThreads - 1) / kPlanThreads;
  const int64_t lo = min(nq, tid * per), hi = min(nq, lo + per);
  uint64_t rounds = 0;
  if (tid == 0) smax = 1;
  hist[tid] = 0;
  static_assert(kOrderBins == kPlanThreads, "a bucket per thread");
  if (!whole)
    for (int64_t i = lo; i < hi; ++i) rounds += (a.slen[i] + (uint64_t)a.rule.R - 1) / a.rule.R;
  uint64_t all;
  plan_scan(rounds, wsum, &all);  // starts with a barrier
  const uint32_t span = whole ? 0xffffffffu : span_length(all, nq, a.rule);
  if (whole) {
    unsigned int m = 1;
    for (int64_t q = tid; q < nq; q += kPlanThreads) m = max(m, a.slen[q]);
    m = __reduce_max_sync(nrq::kFull, m);
    if ((tid & 31) == 0) atomicMax(&smax, m);
    __syncthreads();
    const uint64_t top = (uint64_t)smax + 1;
    auto bin = [&](int64_t q) { return kOrderBins - 1 - (int)((uint64_t)a.slen[q] * kOrderBins / top); };
    for (int64_t q = tid; q < nq; q += kPlanThreads) atomicAdd(&hist[bin(q)], 1u);
    __syncthreads();
    const unsigned int mine = hist[tid];
    const unsigned int at = (unsigned int)(plan_scan(mine, wsum, &all) - mine);
    // the buckets before the shortest `last` queries' first: by base code
    if (tid == 0) cut = 0;
    __syncthreads();
    if ((int64_t)at + mine <= nq - a.last) atomicMax(&cut, (unsigned int)tid + 1u);
    hist[tid] = at;
    __syncthreads();
    const int nc = (int)cut;
    const int shift = a.b > 10 ? a.b - 10 : 0;  // 1024 ranges of codes
    hcode[tid] = 0;
    __syncthreads();
    if (nc > 0)
      for (int64_t q = tid; q < nq; q += kPlanThreads)
        if (bin(q) < nc) atomicAdd(&hcode[a.codes[q * a.P] >> shift & (kOrderBins - 1)], 1u);
    __syncthreads();
    const unsigned int mc = hcode[tid];
    const unsigned int ac = (unsigned int)(plan_scan(mc, wsum, &all) - mc);
    hcode[tid] = ac;
    __syncthreads();
    for (int64_t q = tid; q < nq; q += kPlanThreads) {
      const int z = bin(q);
      unsigned int *h = z < nc ? &hcode[a.codes[q * a.P] >> shift & (kOrderBins - 1)] : &hist[z];
      a.perm[atomicAdd(h, 1u)] = (int32_t)q;
    }
    all = (uint64_t)nq;
  } else {
    uint64_t items = 0;
    for (int64_t i = lo; i < hi; ++i) items += spans_of(a.slen[i], span);
    const uint64_t incl = plan_scan(items, wsum, &all);
    uint32_t at = (uint32_t)(incl - items);
    for (int64_t i = lo; i < hi; ++i) {
      a.pre[i] = at;
      at += spans_of(a.slen[i], span);
    }
    if (tid == 0) a.pre[nq] = (uint32_t)all;
  }
  if (tid == 0) {
    a.plan->ticket = 0u;
    a.plan->nitems = (unsigned int)all;
    a.plan->span_rows = span;
    a.plan->pool_used = 0ull;
  }
}

// Batches up to this size need no plan kernel: a block's first warp works out
// the spans while the others start (one uint8 query: 5 us less, and a launch).
constexpr int kOwnPlan = 128;

struct RefineArgs {
  nrq::RefineParams rf;
  const uint8_t *q;  // [nq x row_bytes]
  int64_t nq;
  int64_t row_bytes;
  int Lmax;
  // queries of a group: the first spans of a group's queries come before the
  // rest of them, so that most later spans start with a committed threshold
  int group;
  const nr_seg *seg;
  const int32_t *nL;
  const uint32_t *slen;
  int64_t *out_ids;
  float *out_d;
  int64_t *stats;
  nrq::RefinePlan *plan;
  const uint32_t *pre;       // [nq + 1] first item of a query (not with own_plan)
  bool own_plan;             // every block works the plan out itself (at most kOwnPlan queries)
  SpanRule rule;
  const int32_t *perm;       // order of whole streams; they use nothing below
  nrq::RefineQState *state;  // [nq]
  uint32_t *ready;           // [items] 0: not finished, 1: nothing logged, 2: logged, or kSpanRedo
  nrq::SpanHeader *hdr;      // [items]
  uint64_t *heap;            // [nq x k] committed top-k
  nrq::SpanEntry *pool;
  uint32_t pool_cap;
};

// The item of ticket t: its query i and its span, by a whole warp. Tickets go
// group by group: the first spans of the group's queries, then the other spans
// query by query.
template <class F>
__device__ __forceinline__ void item_of(const RefineArgs &a, F pre, uint32_t t, int &i, uint32_t &span) {
  const int nq = (int)a.nq;
  const int g0 = nrq::warp_last_le(0, nq, t, pre) / a.group * a.group;
  const int ng = min(a.group, nq - g0);
  const uint32_t first = pre(g0), o = t - first;
  if (o < (uint32_t)ng) {
    i = g0 + (int)o;
    span = 0;
    return;
  }
  const uint32_t x = o - (uint32_t)ng;  // among the later spans of the group
  i = nrq::warp_last_le(g0, g0 + ng, x,
                        [&](int y) { return pre(y) - first - (uint32_t)(y - g0); });
  span = 1u + x - (pre(i) - first - (uint32_t)(i - g0));
}

// Looks of about a microsecond each.
constexpr int kPolls = 64;

// sctl words of the kernel (1..3 are refine_span's)
enum { kCtlQuery = 4, kCtlItem, kCtlSpan, kCtlSpans, kCtlRun, kCtlHn, kCtlRounds, kCtlLow, kCtlNext };

// The answer of query q (a stream of n rows) from the top-k in r, sorted by
// (distance, id), padded. Whole block of TR threads.
template <int DT, int TR>
__device__ __forceinline__ void write_answer(const RefineArgs &a, const nrq::RefineSmem &m,
                                             const nrq::SpanRun &r, int64_t q, uint32_t n) {
  const int tid = threadIdx.x, k = a.rf.k;
  const uint64_t *H = m.hkey + r.cur * k;
  for (int i = tid; i < k; i += TR) {
    int64_t id = -1;
    float d = __int_as_float(0x7f800000);
    if (i < r.hn) {
      const uint64_t kk = H[i];
      id = (int64_t)(uint32_t)kk;
      const uint32_t db = (uint32_t)(kk >> 32);
      d = DT == 0 ? (float)db : __uint_as_float(db);
    }
    a.out_ids[q * k + i] = id;
    a.out_d[q * k + i] = d;
  }
  if (tid == 0 && a.stats) {
    const uint64_t rows = (uint64_t)r.rounds * (uint64_t)a.rf.R;
    a.stats[q * NR_QSTATS] = (int64_t)(rows < n ? rows : n);  // rows of completed rounds
    a.stats[q * NR_QSTATS + 1] = r.rounds;
  }
}

// Whole streams, a block each, in the order of perm. A kernel of its own: what
// spans need (the log, the commit, the plan) costs registers and 2 KB of shared
// memory, a block an SM less at some row sizes, and instructions in every tile.
// In one kernel with the spans, and here: 10,000 uint8 queries, P 64, k 100
// 5,479 and 3,475 us, k 10 1,370 and 1,113; 2,000 of fp32 rows, D = 64, 1,988
// and 1,642, D = 272 6,020 and 4,886 (each with the order and shape it takes).
template <int DT, int TR, int CPR, int KCC, int ST, int MINB>
__global__ void __launch_bounds__(TR, MINB) refine_kernel(RefineArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x;
  const nrq::RefineSmem m = nrq::refine_carve<DT, TR, CPR, KCC, ST, false>(smem, a.row_bytes, a.rf.k);
  volatile int *ctl = m.sctl;
  for (bool first = true;; first = false) {
    if (tid == 0) {
      const uint32_t t = first ? blockIdx.x : gridDim.x + atomicAdd(&a.plan->ticket, 1u);
      ctl[kCtlQuery] = t < (uint32_t)a.nq ? a.perm[t] : -1;
    }
    __syncthreads();
    const int64_t q = ctl[kCtlQuery];
    if (q < 0) return;
    for (int c = tid; c * 16 < a.row_bytes; c += TR)
      reinterpret_cast<uint4 *>(m.sq)[c] = reinterpret_cast<const uint4 *>(a.q + q * a.row_bytes)[c];
    const uint32_t n = a.slen[q];
    nrq::SpanRun r = {0, 0, 0, 0, false};
    nrq::SpanLog lg;  // not used: nothing is logged
    nrq::refine_span<DT, TR, CPR, KCC, ST>(a.rf, m, 0u, n, a.nL[q], a.seg + (size_t)q * a.Lmax, true, r, lg);
    write_answer<DT, TR>(a, m, r, q, n);
    __syncthreads();  // m and ctl are free for the next query
  }
}

// Streams cut into spans.
template <int DT, int TR, int CPR, int KCC, int ST, int MINB>
__global__ void __launch_bounds__(TR, MINB) refine_spans_kernel(RefineArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  nr_after_previous();
  const int tid = threadIdx.x, lane = tid & 31;
  const int k = a.rf.k;
  const nrq::RefineSmem m = nrq::refine_carve<DT, TR, CPR, KCC, ST, true>(smem, a.row_bytes, k);
  volatile int *ctl = m.sctl;
  uint32_t *spre = m.plan;  // [kOwnPlan + 1], then the span's rows
  if (a.own_plan && tid < 32) {
    constexpr int per = kOwnPlan / 32;
    uint32_t n[per], rounds = 0, items = 0;
#pragma unroll
    for (int e = 0; e < per; ++e) {
      const int i = lane * per + e;
      n[e] = i < a.nq ? a.slen[i] : 0u;
      rounds += (uint32_t)(((uint64_t)n[e] + a.rule.R - 1) / a.rule.R);
    }
    uint64_t all = rounds;
    for (int o = 16; o > 0; o >>= 1) all += __shfl_xor_sync(nrq::kFull, all, o);
    const uint32_t span = span_length(all, a.nq, a.rule);
#pragma unroll
    for (int e = 0; e < per; ++e)
      if (lane * per + e < a.nq) items += spans_of(n[e], span);
    uint32_t at = items;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(nrq::kFull, at, o);
      if (lane >= o) at += v;
    }
    at -= items;
#pragma unroll
    for (int e = 0; e < per; ++e) {
      spre[lane * per + e] = at;
      if (lane * per + e < a.nq) at += spans_of(n[e], span);
    }
    if (lane == 31) spre[kOwnPlan] = at;  // (queries past the batch have no items)
    if (lane == 0) spre[kOwnPlan + 1] = span;
  }
  if (a.own_plan) __syncthreads();
  const uint32_t nitems = a.own_plan ? spre[kOwnPlan] : a.plan->nitems;
  const uint32_t span_rows = a.own_plan ? spre[kOwnPlan + 1] : a.plan->span_rows;
  auto pre = [&](int i) { return a.own_plan ? spre[i] : __ldg(&a.pre[i]); };
  // spans a commit stages at once: what fits the stages beside its view (rows
  // of 16 bytes at least)
  constexpr int kRoom = (int)nrq::refine_stage_bytes<TR, KCC, ST>(CPR > 0 ? CPR * 16 : 16) - TR * 16 - 256;
  constexpr int kFit = kRoom / (nrq::kStagedEntries * 16);
  constexpr int kSlots = kFit < 0 ? 0 : kFit < 32 ? kFit : 32;
  constexpr int kWarpFit = (int)nrq::refine_stage_bytes<TR, KCC, ST>(CPR > 0 ? CPR * 16 : 16) / 512;
  constexpr int kWarpSlots = kWarpFit < 32 ? kWarpFit : 32;
  for (bool first = true;; first = false) {
    if (tid < 32) {  // the next item whose query has not stopped
      int q = -1;
      uint32_t sp = 0, base = 0, spans = 1;
      for (uint32_t t = blockIdx.x;; first = false) {
        if (!first) {
          if (lane == 0) t = gridDim.x + atomicAdd(&a.plan->ticket, 1u);
          t = __shfl_sync(nrq::kFull, t, 0);
        }
        if (t >= nitems) break;
        int i;
        item_of(a, pre, t, i, sp);
        if (sp > 0 && __ldcg(&a.state[i].done)) continue;
        q = i;
        base = pre(i);
        spans = pre(i + 1) - base;
        break;
      }
      if (lane == 0) {
        ctl[kCtlQuery] = q;
        ctl[kCtlItem] = (int)base;
        ctl[kCtlSpan] = (int)sp;
        ctl[kCtlSpans] = (int)spans;
      }
    }
    __syncthreads();
    const int64_t q = ctl[kCtlQuery];
    if (q < 0) break;
    uint32_t sp = (uint32_t)ctl[kCtlSpan];
    for (int c = tid; c * 16 < a.row_bytes; c += TR)
      reinterpret_cast<uint4 *>(m.sq)[c] = reinterpret_cast<const uint4 *>(a.q + q * a.row_bytes)[c];
    const uint32_t n = a.slen[q];
    nrq::RefineQState *st = a.state + q;
    bool held = sp == 0;  // this block owns the query's top-k
    nrq::SpanRun r = {0, 0, 0, 0, false};
    for (;;) {
      const uint32_t p0 = sp * span_rows;
      const uint32_t p1 = n - p0 > span_rows ? p0 + span_rows : n;
      nrq::SpanLog lg;
      lg.nthr = &st->nthr;
      lg.pool_used = &a.plan->pool_used;
      lg.pool = a.pool;
      lg.pool_cap = a.pool_cap;
      nrq::refine_span<DT, TR, CPR, KCC, ST>(a.rf, m, p0, p1, a.nL[q], a.seg + (size_t)q * a.Lmax, held, r,
                                             lg);
      const uint32_t base = (uint32_t)ctl[kCtlItem], spans = (uint32_t)ctl[kCtlSpans];
      uint32_t next = sp + 1;  // the next span to commit, when held
      bool redo = false;
      if (!held && tid < 32) {  // publish the log
        nrq::log_flush(m, lg);
        __syncwarp();
        if (lane == 0) {
          a.hdr[base + sp].minkey = r.hn > 0 ? m.hkey[r.cur * k] : nrq::kEmpty;
          a.hdr[base + sp].off = (uint32_t)lg.first;
          __threadfence();
          atomicExch(&a.ready[base + sp], lg.full ? nrq::kSpanRedo : lg.first != nrq::kEmpty ? 2u : 1u);
          __threadfence();
        }
      }
      for (;;) {
        if (!held) {
          // the thread that takes the lock orders what its last holder wrote
          // before the barrier, which hands that on to the block
          bool took = false;
          if (tid == 0 && atomicCAS(&st->lock, 1, 2) == 1) {
            __threadfence();
            took = true;
          }
          if (!__syncthreads_or(took)) break;
          held = true;
          r.cur = 0;
          r.hn = __ldcg(&st->hn);
          r.rounds = __ldcg(&st->rounds);
          r.low = __ldcg(&st->low);
          r.stop = false;
          next = (uint32_t)__ldcg(&st->next);
          for (int i = tid; i < r.hn; i += TR) {
            m.hkey[i] = __ldcg(&a.heap[q * k + i]);
            m.htag[i] = 0;
          }
          __syncthreads();
        }
        if (!r.stop && next < spans) {  // commit the finished spans that follow
          // With no item left for this block it waits a little for spans in
          // flight (at most kPolls looks) instead of handing the top-k over to
          // the block that finishes one.
          const bool idle = __syncthreads_or(tid == 0 && gridDim.x + __ldcg(&a.plan->ticket) >= nitems);
          // By the block, or for a small top-k by its first warp, whose turns
          // are shorter (k = 100, 16 queries: 139 us a refinement by the
          // block, 195 by a warp).
          const int polls = idle ? kPolls : 0;
          if (k <= 32) {
            if (tid < 32) {
              redo = nrq::commit_warp<kWarpSlots>(a.rf, m, r, a.pool, a.pool_cap, a.ready + base,
                                                   a.hdr + base, next, spans, n, span_rows, polls);
              if (lane == 0) {
                ctl[kCtlRun] = r.cur | (r.stop ? 2 : 0) | (redo ? 4 : 0);
                ctl[kCtlHn] = r.hn;
                ctl[kCtlRounds] = r.rounds;
                ctl[kCtlLow] = r.low;
                ctl[kCtlNext] = (int)next;
              }
            }
            __syncthreads();
            r.cur = ctl[kCtlRun] & 1;
            r.stop = (ctl[kCtlRun] & 2) != 0;
            redo = (ctl[kCtlRun] & 4) != 0;
            r.hn = ctl[kCtlHn];
            r.rounds = ctl[kCtlRounds];
            r.low = ctl[kCtlLow];
            next = (uint32_t)ctl[kCtlNext];
          } else {
            redo = nrq::commit_block<TR, kSlots>(a.rf, m, r, a.pool, a.pool_cap, a.ready + base,
                                                 a.hdr + base, next, spans, n, span_rows, polls);
          }
        }
        if (r.stop || next == spans) {
          write_answer<DT, TR>(a, m, r, q, n);
          if (tid == 0 && spans > 1) atomicExch(&st->done, 1);
          redo = false;
          break;  // the lock stays taken: there is nothing more to commit
        }
        if (redo) break;
        // hand the top-k back
        const uint64_t *H = m.hkey + r.cur * k;
        for (int i = tid; i < r.hn; i += TR) a.heap[q * k + i] = H[i];
        if (tid == 0) {
          st->hn = r.hn;
          st->rounds = r.rounds;
          st->low = r.low;
          st->next = (int)next;
          if (r.hn == k) *reinterpret_cast<volatile unsigned long long *>(&st->nthr) = ~H[k - 1];
        }
        __syncthreads();
        held = false;
        bool again = false;
        if (tid == 0) {
          __threadfence();
          atomicExch(&st->lock, 1);
          __threadfence();
          // a span finished meanwhile was left by its block to this one
          again = nrq::ld_acquire(&a.ready[base + next]) != 0u;
        }
        if (!__syncthreads_or(again)) break;
      }
      if (!redo) break;
      sp = next;  // its block had no room for the log: refined here on the query's top-k
    }
    __syncthreads();  // m and ctl are free for the next item
  }
}

// Resident blocks of `kern` (blocks of TR threads with smem bytes), or 0 and
// the error. (The attribute is what the launch takes and no more: with all there
// is, less is left for L1, and 1,300 fp32 queries, D = 272, took 3,294 us for
// 3,135.)
template <class K>
int64_t resident(const nr_index *ix, K kern, int TR, size_t smem, cudaError_t *e) {
  int per_sm = 0;
  *e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (*e == cudaSuccess) *e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, TR, smem);
  if (*e == cudaSuccess && per_sm < 1) *e = cudaErrorInvalidConfiguration;
  return *e == cudaSuccess ? (int64_t)per_sm * ix->num_sms : 0;
}
// Those of them that the parameters allow.
int64_t allowed(const nr_index *ix, int64_t blocks) {
  const int64_t most = (int64_t)ix->params.refine_ctas * ix->num_sms;
  return most > 0 && blocks > most ? most : blocks;
}

cudaError_t launch_plan(nr_index *ix, const PlanArgs &pa, cudaStream_t s) {
  plan_kernel<<<1, kPlanThreads, 0, s>>>(pa);
  ix->launches += 1;
  return cudaGetLastError();
}

// Whether a batch keeps its streams whole (a block a query) when `blocks` blocks
// are resident. Few queries leave most blocks idle; many keep them busy, and
// cutting their streams only adds work per span (about 7 us each: the item, the
// segment search, the first tile's latency, the commit) and, with an early stop,
// rows read beyond it: the more, the smaller the part of a stream that t_low
// rounds are. The line, in sixteenths of the blocks, lies where both sides
// measured the same (k = 10, `blocks` as the kernel has them for each row size):
// no early stop 18 to 30 (uint8 x 128 18-21, fp32 x 96 21, other rows 20-30; k =
// 100 12); t_low rounds as long as the stream 14 to 24, a quarter of it uint8 5 to
// 11 and fp32 6 to 15, a sixteenth 2 to 8 and 4 to 8. us, cut and whole: u8-10m P
// = C = 256, no early stop: 400 queries 342 / 433, 600 461 / 499, 1,000 721 / 628;
// t_low 16: 200 236 / 259, 300 297 / 269; f32-10m P 512, no early stop: 600 592 /
// 688, 1,000 924 / 870; t_low 4: 150 204 / 220, 200 263 / 246; u8-30m P = C =
// 1024, t_low 80: 150 435 / 492, 300 781 / 585; 768-value fp32 rows, no early
// stop: 600 3,318 / 3,565, t_low 4: 100 597 / 638, 200 1,148 / 721.
constexpr int kCutMost = 18;  // sixteenths, at most
bool whole_streams(const nr_index *ix, int64_t nq, int k, int C, int64_t blocks) {
  const int64_t stop = (int64_t)ix->params.t_low * ix->params.round_size;  // rows
  const int64_t rows = (int64_t)C * (ix->t > 0 ? ix->t : 64);              // of a stream, some
  const int64_t least = ix->dtype == 0 ? rows + 16 * stop : 2 * rows + 24 * stop;  // the line x rows
  const int64_t most = k > 32 ? 12 : kCutMost;
  return nq * 16 >= blocks * most || (stop > 0 && (double)nq * 16 * rows >= (double)blocks * least);
}

// Of whole streams: whether nearby queries go side by side (see plan_kernel).
// Only where the rows read bound the tile (the generic ones are bound by their
// instructions: 2,000 fp32 queries, D = 64, 1,640 us longest first, 1,907 by
// code), and with queries enough to share (long rows, D = 288: 2,000 queries
// 4,565 and 4,868 us, 8,000 16,978 and 14,980; f32-10m, P = 512: 3,000 2,435 and
// 2,454, 10,000 7,858 and 7,134).
bool nearby_first(const RefineArgs &a, bool bound_by_rows) { return bound_by_rows && a.nq >= 4096; }

template <int DT, int TR, int CPR, int KCC, int ST, int MINB>
cudaError_t launch_whole(nr_index *ix, RefineArgs a, PlanArgs pa, cudaStream_t s) {
  const size_t smem = nrq::refine_smem_bytes<DT, TR, CPR, KCC, ST, false>(a.row_bytes, a.rf.k);
  auto kern = refine_kernel<DT, TR, CPR, KCC, ST, MINB>;
  cudaError_t e;
  const int64_t grid = std::min(allowed(ix, resident(ix, kern, TR, smem, &e)), a.nq);
  if (e != cudaSuccess) return e;
  pa.last = nearby_first(a, CPR > 0 || KCC > 0) ? grid : a.nq;
  if ((e = launch_plan(ix, pa, s)) != cudaSuccess) return e;
  kern<<<(unsigned)grid, TR, smem, s>>>(a);
  ix->launches += 1;
  return cudaGetLastError();
}

// Of uint8 rows of 128 bytes, whole streams: whether the stream's bytes bound a
// block (three stages, four blocks an SM: more rows in flight) or its merges
// (two stages, six blocks). Long streams and a small top-k the one, short ones,
// a larger top-k and many queries that share rows the other. us, three stages
// and two: u8-30m P = C = 1024, t_low 80, 10,000 queries: k 10 10,019 / 10,528,
// k 100 13,720 / 12,885; u8-10m P = C = 256, no early stop, k 10: 900 queries
// 607 / 702, 3,000 1,478 / 1,567, 10,000 4,507 / 4,061; k 100, 10,000 6,541 /
// 5,431; P 64, C 128, t_low 4: 2,000 330 / 312, 10,000 1,290 / 1,113.
bool bound_by_stream(const RefineArgs &a, int C) {
  return a.rf.k <= 32 && (C >= 1024 || (C >= 256 && a.nq < 4096 && (a.rf.t_low == 0 || a.rf.t_low >= 8)));
}

template <int DT, int TR, int CPR, int KCC, int ST, int MINB>
cudaError_t launch_spans(nr_index *ix, RefineArgs a, PlanArgs pa, int64_t grid, cudaStream_t s, bool early) {
  const size_t smem = nrq::refine_smem_bytes<DT, TR, CPR, KCC, ST, true>(a.row_bytes, a.rf.k);
  auto kern = refine_spans_kernel<DT, TR, CPR, KCC, ST, MINB>;
  // (another thread's call may have set another size since `resident`)
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  pa.rule.align = a.rf.R < TR ? TR / a.rf.R : 1;
  // Two uint8 items a block, four of the slower fp32 ones (u8-10m k 100, 100
  // queries: 471 us at two, 506 at four; long fp32 rows, 30 queries: 1,144 and
  // 1,075). Three for two blocks where a large top-k makes the commits the longer
  // part, which follow one another in a query: us a search at two items and at one
  // and a half, u8-30m k 100, P 92, C 64, t_low 16: 70 queries 285 / 272; P = C =
  // 256, no early stop: 16 351 / 359, 30 381 / 364, 250 587 / 575; P = C = 1024,
  // t_low 80: 16 408 / 389, 150 568 / 540; u8-10m P = C = 256: 20 307 / 320, 200 446
  // / 436; k 256, P 64, C 512: 20 481 / 444, 80 436 / 411. (k 50: 46 queries of P 92
  // 206 / 195 at four for three, of P = C = 256 281 / 289, of 1024 329 / 336.)
  pa.rule.items_want = (unsigned int)((DT == 0 ? (a.rf.k > 64 ? 3 : 4) : 8) * grid / 2);
  a.group = (int)grid;
  a.rule = pa.rule;
  a.own_plan = a.nq <= kOwnPlan;
  if (!a.own_plan && (e = launch_plan(ix, pa, s)) != cudaSuccess) return e;
  e = nr_launch_kernel(kern, (unsigned)grid, TR, smem, s, early && a.own_plan, a);
  ix->launches += 1;
  return e;
}

// A row size's tile: rows of a tile, chunks of a row (0: any), chunks of a piece
// (0: whole rows), stages, blocks an SM at least.
template <int DT_, int TR_, int CPR_, int KCC_, int ST_, int MINB_>
struct Shape {
  static constexpr int DT = DT_, TR = TR_, CPR = CPR_, KCC = KCC_, ST = ST_, MINB = MINB_;
};
template <class F>
cudaError_t by_shape(const nr_index *ix, F f) {
  const int64_t rb = ix->row_bytes;
  if (ix->dtype == 0) {
    if (rb == 128) return f(Shape<0, 128, 8, 0, 3, 4>());  // uint8, D = 128
    if (rb <= 512) return f(Shape<0, 128, 0, 0, 2, 4>());
    return f(Shape<0, 64, 0, 0, 2, 4>());
  }
  if (rb > 1024) {  // fp32, D above 256: rows staged in pieces
    if (rb % 256 == 0) return f(Shape<1, 128, 0, 16, 2, 3>());
    if (rb % 128 == 0) return f(Shape<1, 128, 0, 8, 2, 3>());
    return f(Shape<1, 128, 0, 4, 2, 3>());  // rb % 64 == 0 (load check)
  }
  if (rb == 384) return f(Shape<1, 64, 24, 0, 2, 4>());  // fp32, D = 96
  if (rb <= 512) return f(Shape<1, 64, 0, 0, 2, 4>());
  return f(Shape<1, 32, 0, 0, 2, 4>());
}

nrq::RefineParams refine_params(const nr_index *ix, int k) {
  const nr_params &p = ix->params;
  nrq::RefineParams rf;
  rf.vec = static_cast<const uint8_t *>(ix->vec);
  rf.ids = ix->ids;
  rf.cpr = (int)(ix->row_bytes / 16);
  rf.swz_mask = (rf.cpr % 8 == 0) ? 7 : (rf.cpr % 4 == 0) ? 3 : (rf.cpr % 2 == 0) ? 1 : 0;
  rf.k = k;
  rf.R = p.round_size;
  rf.t_low = p.t_low;
  rf.u_min = p.u_min;
  rf.f_min = p.f_min;
  rf.r_min = p.r_min;
  const double f = (double)p.alpha_front * (double)k;
  int nf = (int)f;
  if ((double)nf < f) nf += 1;  // ceil
  if (nf < 0) nf = 0;
  if (nf > k) nf = k;
  rf.nfront = nf;
  return rf;
}

size_t up256(size_t v) { return (v + 255) & ~(size_t)255; }

// Scratch of a refine launch. Whole streams: [their order][plan]. Cut ones:
// [item prefix][plan, query states, ready flags (zeroed together)][span
// headers][committed top-k][log entries]
struct RefineScratch {
  size_t plan, perm, pre, state, ready, zero_end, hdr, heap, pool, total;
};
RefineScratch refine_scratch(int64_t nq, int k, int64_t items, int64_t entries) {
  RefineScratch l = {};
  size_t o = 0;
  if (items > nq) {
    l.pre = o;   o = up256(o + ((size_t)nq + 1) * 4);
    l.plan = o;  o = up256(o + sizeof(nrq::RefinePlan));
    l.state = o; o += (size_t)nq * sizeof(nrq::RefineQState);
    l.ready = o; o += (size_t)items * 4;
    l.zero_end = o = up256(o);
    l.hdr = o;   o = up256(o + (size_t)items * sizeof(nrq::SpanHeader));
    l.heap = o;  o = up256(o + (size_t)nq * k * 8);
    l.pool = o;  o = up256(o + (size_t)entries * sizeof(nrq::SpanEntry));
  } else {
    l.perm = o; o = up256(o + (size_t)nq * 4);
    l.plan = o; o = up256(o + sizeof(nrq::RefinePlan));
  }
  l.total = o;
  return l;
}

// Items and log entries a batch of nq queries has room for.
int64_t span_items(int64_t nq) { return nq + std::min<int64_t>(1 << 20, std::max<int64_t>(4096, nq * 64)); }
int64_t span_entries(int64_t nq, int k) {
  return std::min<int64_t>(16 << 20, (int64_t)k * std::max<int64_t>(4096, nq * 32));
}

RefineScratch refine_scratch(int64_t nq, int k, bool cut) {
  return cut ? refine_scratch(nq, k, span_items(nq), span_entries(nq, k)) : refine_scratch(nq, k, nq, 0);
}

}  // namespace

cudaError_t nr_refine_room_of(const nr_index *ix, int k, nr_refine_room *room) {
  return by_shape(ix, [&](auto sh) {
    using S = decltype(sh);
    cudaError_t e;
    const int64_t blocks = resident(ix, refine_spans_kernel<S::DT, S::TR, S::CPR, S::KCC, S::ST, S::MINB>, S::TR,
                       nrq::refine_smem_bytes<S::DT, S::TR, S::CPR, S::KCC, S::ST, true>(ix->row_bytes, k), &e);
    *room = {allowed(ix, blocks), blocks * kCutMost / 16};
    return e;
  });
}

bool nr_refine_cuts(const nr_index *ix, int64_t nq, int k, int C, const nr_refine_room &room) {
  return !whole_streams(ix, nq, k, C, room.blocks);
}

size_t nr_refine_scratch_bytes(int64_t nq, int k, bool cut) { return refine_scratch(nq, k, cut).total; }

nr_zero nr_refine_zero(int64_t nq, int k, bool cut, void *scratch) {
  if (!cut) return {nullptr, 0};
  const RefineScratch l = refine_scratch(nq, k, cut);
  return {static_cast<char *>(scratch) + l.plan, (l.zero_end - l.plan) / 16};
}

cudaError_t nr_launch_refine(nr_index *ix, const void *d_q, int64_t nq, int k, int Lmax,
                             const nr_seg *d_seg, const int32_t *d_nL, const uint32_t *d_slen,
                             const uint32_t *d_codes, int P, int64_t *d_ids, float *d_dists,
                             int64_t *d_stats, bool cut, int64_t blocks, void *d_scratch, cudaStream_t s,
                             bool early) {
  if (nq <= 0) return cudaSuccess;
  char *w = static_cast<char *>(d_scratch);
  const RefineScratch l = refine_scratch(nq, k, cut);
  RefineArgs a;
  a.rf = refine_params(ix, k);
  a.q = static_cast<const uint8_t *>(d_q);
  a.nq = nq;
  a.row_bytes = ix->row_bytes;
  a.Lmax = Lmax;
  a.seg = d_seg;
  a.nL = d_nL;
  a.slen = d_slen;
  a.out_ids = d_ids;
  a.out_d = d_dists;
  a.stats = d_stats;
  a.plan = reinterpret_cast<nrq::RefinePlan *>(w + l.plan);
  a.pre = reinterpret_cast<uint32_t *>(w + l.pre);
  a.perm = reinterpret_cast<int32_t *>(w + l.perm);
  a.state = reinterpret_cast<nrq::RefineQState *>(w + l.state);
  a.ready = reinterpret_cast<uint32_t *>(w + l.ready);
  a.hdr = reinterpret_cast<nrq::SpanHeader *>(w + l.hdr);
  a.heap = reinterpret_cast<uint64_t *>(w + l.heap);
  a.pool = reinterpret_cast<nrq::SpanEntry *>(w + l.pool);
  a.pool_cap = cut ? (uint32_t)span_entries(nq, k) : 0u;
  PlanArgs pa;
  pa.slen = d_slen;
  pa.codes = d_codes;
  pa.P = P;
  pa.b = ix->b;
  pa.last = nq;
  pa.nq = nq;
  pa.rule = {a.rf.R, 1, std::max(1, 8192 / a.rf.R), 1u, (unsigned int)(cut ? span_items(nq) : nq)};
  pa.plan = a.plan;
  pa.pre = reinterpret_cast<uint32_t *>(w + l.pre);
  pa.perm = reinterpret_cast<int32_t *>(w + l.perm);
  return by_shape(ix, [&](auto sh) {
    using S = decltype(sh);
    if (cut) return launch_spans<S::DT, S::TR, S::CPR, S::KCC, S::ST, S::MINB>(ix, a, pa, blocks, s, early);
    if constexpr (S::CPR == 8)
      if (!bound_by_stream(a, Lmax - P)) return launch_whole<S::DT, S::TR, S::CPR, S::KCC, 2, 6>(ix, a, pa, s);
    return launch_whole<S::DT, S::TR, S::CPR, S::KCC, S::ST, S::MINB>(ix, a, pa, s);
  });
}
