// refine_span: one block refines a span of a query's candidate stream exactly,
// with the round-based early stop (Sec. 3.4, Algorithm 2's T_low rule), and
// the in-order commit that joins the spans of a query refined by several
// blocks.
#pragma once

#include "nrq_common.cuh"

namespace nrq {

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// ============================================================== refine
// Candidate stream = rows of the kept clusters in list order, a list of
// contiguous segments. Tiles of TR rows (one row per thread) are gathered by
// 16-byte cp.async copies (each warp copies and later reads only its own 32
// rows, so stage reuse needs no block barrier) into a ring of ST shared-memory
// stages whose 16-byte chunks are XOR-swizzled by row, so one-row-per-thread
// reads are bank-conflict free. fp32 rows too long for whole-row stages (KCC > 0,
// D above 256) are staged in pieces of KCC 16-byte chunks of every row, each
// thread carrying its row's distance from piece to piece.
// Distances: uint8 rows: per-byte |x - q| (__vabsdiffu4) squared and summed by
// __dp4a in int32 (exact); fp32 rows: the sequential fmaf chain over j, so a
// distance is bit-identical to a sequential CPU evaluation.
// Top-k: keys (distance bits << 32 | id) are unique; rows at or below the
// current k-th key are merged by rank, each member tagged with the round it
// entered. After round t: updates = members entered in round t, front
// updates = those within the first nfront slots.
//
// A query's stream is cut into spans of S whole rounds, refined by different
// blocks at once (the plan kernel chooses S). The block of span 0 refines it
// on the query's own top-k. A block of a later span does not know the top-k
// that its rounds start from: it refines its span on an empty top-k of its
// own and logs, per round, the members that entered (a row outside that local
// top-k has k smaller rows before it in its own span, and a row at or above
// the k-th key of the spans committed so far has k smaller ones there, so
// neither can enter the query's). The spans are then committed in stream
// order: each round's logged members are merged into the query's top-k and
// the stop rule is evaluated round by round, which gives the top-k, the
// rounds and the stop of one block refining the whole stream. Whichever block
// finishes the next span to commit takes the query's lock and commits every
// consecutive finished span; a block that does not get the lock moves on (the
// holder looks again after it unlocks), so none depends on another's progress: a
// holder with nothing else to do looks at most a fixed number of times for a
// span in flight (polls) and then hands the top-k over.
struct RefineParams {
  const uint8_t *vec;
  const uint32_t *ids;
  int cpr;       // 16-byte chunks per row (runtime value when CPR = 0)
  int swz_mask;  // XOR mask of the chunk index (runtime value when CPR = 0)
  int k, R;      // top-k size; round size (power of two)
  int t_low, u_min, f_min, r_min, nfront;
};

// What the plan kernel leaves for the refinement: work counters and the spans.
struct RefinePlan {
  unsigned int ticket;            // items handed out beyond each block's first
  unsigned int nitems;            // spans of all queries
  uint32_t span_rows;             // rows of a span (S R)
  unsigned int pad;
  unsigned long long pool_used;   // log entries reserved
};

// A query's committed state, zeroed before the launch. lock: 0 = span 0 not
// committed yet (its block owns the state), 1 = free, 2 = held.
struct RefineQState {
  int lock, next, done, hn, rounds, low;
  unsigned long long nthr;  // ~(k-th key) of a full top-k, 0 before
};
struct SpanHeader {  // of a logged span
  uint64_t minkey;   // its smallest key
  uint32_t off, pad; // its first block of log entries
};
// The log: the members that entered a span's local top-k in its rounds, in
// round order, in blocks of 1 + count entries: first (next block of the span or
// kEmpty, count), then (key, round within the span) per member.
struct SpanEntry {
  uint64_t key;
  uint32_t round, pad;
};
constexpr int kLogBlock = 128;  // members of a block at most
constexpr uint32_t kSpanRedo = 0xffffffffu;  // ready value: not logged (the pool was full)

// Rows that the stages hold as they are (see refine_span).
template <int DT, int CPR>
constexpr bool kRow128 = DT == 0 && CPR == 8;

// Bytes of the stages: ST tiles.
template <int TR, int KCC, int ST>
__host__ __device__ constexpr size_t refine_stage_bytes(int64_t row_bytes) {
  return (size_t)ST * TR * (KCC > 0 ? KCC * 16 : row_bytes);
}

// Shared memory of refine_span.
struct RefineSmem {
  unsigned char *stage;  // refine_stage_bytes (16-byte aligned)
  unsigned char *sq;     // the query row (row_bytes)
  uint32_t *srow;        // ST x TR: rows of the open tiles (kRow128: held in registers)
  uint64_t *hkey;        // 2 x k
  uint64_t *skey;        // 2 x TR
  int *htag;             // 2 x k
  int *sctl;             // 16 ints: [1..3] survivor counters, [4..15] the kernel's
  // only where streams are cut (CUT):
  uint64_t *logk;        // kLogBlock: members logged and not yet written, and
  uint32_t *logr;        // their rounds
  uint32_t *plan;        // 132: the kernel's
};

// Carve RefineSmem from base (16-byte aligned).
template <int DT, int TR, int CPR, int KCC, int ST, bool CUT>
__device__ __forceinline__ RefineSmem refine_carve(unsigned char *base, int64_t row_bytes, int k) {
  RefineSmem m;
  m.stage = base;
  m.sq = base + refine_stage_bytes<TR, KCC, ST>(row_bytes);
  m.srow = reinterpret_cast<uint32_t *>(m.sq + row_bytes);
  m.hkey = reinterpret_cast<uint64_t *>(m.srow + (kRow128<DT, CPR> ? 0 : ST * TR));
  m.skey = m.hkey + 2 * k;
  m.logk = m.skey + 2 * TR;
  m.htag = reinterpret_cast<int *>(m.logk + (CUT ? kLogBlock : 0));
  m.sctl = m.htag + 2 * k;
  m.logr = reinterpret_cast<uint32_t *>(m.sctl + 16);
  m.plan = m.logr + kLogBlock;
  return m;
}
template <int DT, int TR, int CPR, int KCC, int ST, bool CUT>
__host__ __device__ inline size_t refine_smem_bytes(int64_t row_bytes, int k) {
  return refine_stage_bytes<TR, KCC, ST>(row_bytes) + (size_t)row_bytes +
         (kRow128<DT, CPR> ? 0 : (size_t)ST * TR * 4) + (size_t)2 * k * 8 + (size_t)2 * TR * 8 +
         (size_t)2 * k * 4 + 16 * 4 + (CUT ? (size_t)kLogBlock * 12 + 132 * 4 : 0);
}

// Top-k state of a block (uniform in the block): which buffer, members,
// rounds done, consecutive low-quality rounds, stopped.
struct SpanRun {
  int cur, hn, rounds, low;
  bool stop;
};

// The stop rule after round `roundno` with newc members entered in it, frontc
// of them in the front slots.
__device__ __forceinline__ void round_done(const RefineParams &a, SpanRun &r, int roundno, int newc,
                                           int frontc) {
  r.rounds = roundno;
  r.low = newc < a.u_min && frontc < a.f_min ? r.low + 1 : 0;
  r.stop = a.t_low > 0 && r.hn == a.k && roundno >= a.r_min && r.low >= a.t_low;
}
// The same after m rounds that changed nothing.
__device__ __forceinline__ void rounds_unchanged(const RefineParams &a, SpanRun &r, int m) {
  if (m <= 0) return;
  const bool lowq = 0 < a.u_min && 0 < a.f_min;
  if (a.t_low > 0 && r.hn == a.k && lowq) {
    const int j = max(1, max(a.r_min - r.rounds, a.t_low - r.low));  // the round that stops
    if (j <= m) {
      r.rounds += j;
      r.low += j;
      r.stop = true;
      return;
    }
  }
  r.rounds += m;
  r.low = lowq ? r.low + m : 0;
}

// The members that entered the top-k in round `roundno` (all of them, those in
// the front slots), counted by a warp.
__device__ __forceinline__ void count_new(const RefineSmem &m, const SpanRun &r, int k, int nfront,
                                          int roundno, int &newc, int &frontc) {
  newc = frontc = 0;
  for (int i = threadIdx.x & 31; i < r.hn; i += 32) {
    const bool nw = m.htag[r.cur * k + i] == roundno;
    newc += nw ? 1 : 0;
    frontc += (nw && i < nfront) ? 1 : 0;
  }
  newc = __reduce_add_sync(kFull, newc);
  frontc = __reduce_add_sync(kFull, frontc);
}

// Last index in [lo, hi) with f(index) <= x, by a whole warp, 32 probes a
// step; f nondecreasing, f(lo) <= x.
template <class F>
__device__ __forceinline__ int warp_last_le(int lo, int hi, uint32_t x, F f) {
  const int lane = threadIdx.x & 31;
  while (hi - lo > 1) {
    const int step = (hi - lo + 31) / 32, i = lo + lane * step;
    const unsigned b = __ballot_sync(kFull, i < hi && f(i) <= x);
    lo += (__popc(b) - 1) * step;
    hi = min(hi, lo + step);
  }
  return lo;
}

// Where a span that is not refined on the query's own top-k is logged.
struct SpanLog {
  const unsigned long long *nthr;  // the query's committed threshold
  unsigned long long *pool_used;
  SpanEntry *pool;
  uint32_t pool_cap;
  // out (warp 0): the first block written and the last, whether the pool was
  // full, and the members waiting in shared memory
  uint64_t first, last;
  bool full;
  int waiting;
};

// Writes the members waiting in shared memory as a block of the span's log, by
// warp 0.
__device__ __forceinline__ void log_flush(const RefineSmem &m, SpanLog &lg) {
  const int lane = threadIdx.x & 31, n = lg.waiting;
  if (n == 0 || lg.full) return;
  unsigned long long at = 0;
  if (lane == 0) at = atomicAdd(lg.pool_used, (unsigned long long)n + 1ull);
  at = __shfl_sync(kFull, at, 0);
  lg.full = at + (unsigned)n + 1u > lg.pool_cap;
  if (lg.full) return;
  ulonglong2 *g = reinterpret_cast<ulonglong2 *>(lg.pool + at);
  if (lane == 0) {
    g[0] = make_ulonglong2(kEmpty, (unsigned long long)n);
    if (lg.first != kEmpty) lg.pool[lg.last].key = at;
  }
  for (int e = lane; e < n; e += 32) g[1 + e] = make_ulonglong2(m.logk[e], (unsigned long long)m.logr[e]);
  if (lg.first == kEmpty) lg.first = at;
  lg.last = at;
  lg.waiting = 0;
  __syncwarp();
}

// Merges the ns keys of sk into the top-k, tagged with round `roundno`: merged
// order by key; on equal keys (possible only when an index stores a row twice)
// the members before the new ones, and those by slot, so ranks are unique.
// Whole block; the keys are visible to it, and the result is on return.
template <int TR>
__device__ __forceinline__ void block_merge(const RefineSmem &m, SpanRun &r, int k, const uint64_t *sk_buf,
                                            int ns, int roundno) {
  const int tid = threadIdx.x;
  const int nxt = r.cur ^ 1;
  const uint64_t *H = m.hkey + r.cur * k;
  for (int i = tid; i < ns; i += TR) {
    const uint64_t sk = sk_buf[i];
    int lo = 0, hi = r.hn;  // # of H at or below sk
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (H[mid] <= sk) lo = mid + 1; else hi = mid;
    }
    int rk = lo;
    for (int j = 0; j < ns; ++j) rk += (sk_buf[j] < sk || (sk_buf[j] == sk && j < i)) ? 1 : 0;
    if (rk < k) {
      m.hkey[nxt * k + rk] = sk;
      m.htag[nxt * k + rk] = roundno;
    }
  }
  for (int j = tid; j < r.hn; j += TR) {
    const uint64_t hk = H[j];
    int rk = j;
    for (int i = 0; i < ns; ++i) rk += sk_buf[i] < hk ? 1 : 0;
    if (rk < k) {
      m.hkey[nxt * k + rk] = hk;
      m.htag[nxt * k + rk] = m.htag[r.cur * k + j];
    }
  }
  __syncthreads();
  r.cur = nxt;
  r.hn = r.hn + ns < k ? r.hn + ns : k;
}

// Positions [p0, p1) of a query's stream of nl segments, p0 a whole number of
// rounds and of tiles, p1 the stream's end or a whole number of rounds. The
// caller has written the query row into m.sq (block-visible after this
// function's first barrier). direct: r is the query's top-k, and the stop rule
// ends the span; else r is the span's own, empty at first, and the members
// that enter are logged. Whole block (TR threads) calls; ends with a barrier.
template <int DT, int TR, int CPR, int KCC, int ST>
__device__ __forceinline__ void refine_span(const RefineParams &a, const RefineSmem &m, uint32_t p0,
                                            uint32_t p1, int nl, const nr_seg *segs, bool direct,
                                            SpanRun &r, SpanLog &lg) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = a.k;
  const int chunk = a.R < TR ? a.R : TR;
  const uint32_t ntiles = (uint32_t)(((uint64_t)(p1 - p0) + TR - 1) / TR);
  if (tid == 0) m.sctl[1] = m.sctl[2] = m.sctl[3] = 0;
  __syncthreads();  // the caller's copy of the query row into m.sq is visible after this

  // The warp's window of 32 segments, one a lane: where it begins in the
  // stream and the stored row less that (positions past the list: none).
  // Positions only grow, so a window serves many tiles.
  int wseg = 0;
  uint32_t wpos = 0xffffffffu, wdelta = 0;
  auto window = [&](int at) {
    wseg = at;
    const nr_seg sg = segs[min(at + lane, nl - 1)];
    wpos = at + lane < nl ? sg.pos : 0xffffffffu;
    wdelta = sg.row0 - sg.pos;
  };
  if (p0 < p1)
    window(p0 == 0 ? 0
                   : warp_last_le(0, nl, min(p0 + (uint32_t)warp * 32u, p1 - 1u),
                                  [&](int i) { return segs[i].pos; }));
  // the stored row of this thread in tile t (row 0 past the span); whole warp
  auto row_of = [&](uint32_t t) {
    const uint32_t first = p0 + t * TR + warp * 32u, p = first + lane;
    if (first >= p1) return 0u;
    const uint32_t last = min(first + 31u, p1 - 1u);
    int head;       // segments of the window that begin at or before the first row
    uint32_t tail;  // where its last one begins
    for (;;) {
      head = __popc(__ballot_sync(kFull, wpos <= first));
      tail = __shfl_sync(kFull, wpos, 31);
      if (tail > last || head <= 1) break;
      window(wseg + head - 1);
    }
    // a bit for each row of the warp that begins a segment after the first's
    const bool starts = wpos > first && wpos <= last;
    const unsigned bits = __reduce_or_sync(kFull, starts ? 1u << (wpos - first) : 0u);
    // the bits name the segments if no two begin at one row, neither in the
    // window nor just past one that ends among these rows (31 of one row and one
    // without rows as its last: the row at `last` is the segment's after it)
    const bool one_each = __popc(__ballot_sync(kFull, starts)) == __popc(bits);
    auto by_bits = [&]() {
      const int i = head - 1 + __popc(bits & (0xffffffffu >> (31 - lane)));
      const uint32_t row = __shfl_sync(kFull, wdelta, i) + p;
      return p < p1 ? row : 0u;
    };
    if (one_each && tail > last) return by_bits();
    if (one_each && (wseg + 32 >= nl || segs[wseg + 32].pos > last)) return by_bits();
    // segments without rows share their place with the next: the last one counts
    int i = wseg;
    while (i + 1 < nl && segs[i + 1].pos <= min(p, last)) ++i;
    return p < p1 ? segs[i].row0 + (p - segs[i].pos) : 0u;
  };

  int ci = 0;
  bool changed = false;  // the top-k in this round
  const uint32_t rmask_round = (uint32_t)a.R - 1u;  // R is a power of two
  lg.first = kEmpty;
  lg.full = false;
  lg.waiting = 0;
  // The committed threshold of the query, as the load of the previous tile
  // found it: a stale one only keeps more rows than it need, and waiting for
  // the load here would add an L2 latency to every tile.
  unsigned long long nthr = direct ? 0ull : __ldcg(lg.nthr);
  // Merges a tile (dkey: this thread's distance, row: its stored row) chunk by
  // chunk; a round ends every R stream positions. One block barrier per chunk
  // (two when the top-k changes): survivor counters rotate over three slots
  // and survivor buffers over two, and every warp evaluates the stop rule
  // itself from the shared top-k.
  auto merge = [&](uint32_t t, uint32_t dkey, uint32_t row, uint64_t ext) {
    const uint32_t p = p0 + t * TR + tid;
    for (int cs = 0; cs < TR && !r.stop; cs += chunk, ++ci) {
      const uint32_t cstart = p0 + t * TR + cs;
      if (cstart >= p1) break;
      int *cnt = &m.sctl[1 + ci % 3];
      uint64_t *sk_buf = m.skey + (ci & 1) * TR;
      uint64_t thr = r.hn == k ? m.hkey[r.cur * k + k - 1] : kEmpty;
      if (ext < thr) thr = ext;
      const uint32_t thr_hi = (uint32_t)(thr >> 32);
      if (tid >= cs && tid < cs + chunk && p < p1 && dkey <= thr_hi) {
        const uint32_t id = __ldg(&a.ids[row]);
        const uint64_t key = ((uint64_t)dkey << 32) | id;
        if (key < thr) sk_buf[atomicAdd(cnt, 1)] = key;
      }
      if (tid == 0) m.sctl[1 + (ci + 1) % 3] = 0;  // counter of the next chunk
      __syncthreads();
      const int ns = *cnt;
      const int roundno = r.rounds + 1;
      if (ns > 0) {
        block_merge<TR>(m, r, k, sk_buf, ns, roundno);
        changed = true;
      }
      const uint32_t cend = p1 - cstart > (uint32_t)chunk ? cstart + chunk : p1;
      if ((cend & rmask_round) == 0 || cend >= p1) {  // round complete
        int newc = 0, frontc = 0;
        if (changed) count_new(m, r, k, a.nfront, roundno, newc, frontc);
        changed = false;
        if (direct) {
          round_done(a, r, roundno, newc, frontc);
        } else {
          r.rounds = roundno;
          if (warp == 0 && newc > 0)  // log the members that entered
            for (int i0 = 0; i0 < r.hn; i0 += 32) {
              const bool nw = i0 + lane < r.hn && m.htag[r.cur * k + i0 + lane] == roundno;
              const unsigned b = __ballot_sync(kFull, nw);
              if (lg.waiting + __popc(b) > kLogBlock) log_flush(m, lg);
              if (lg.full) break;
              if (nw) {
                const int e = lg.waiting + __popc(b & ((1u << lane) - 1u));
                m.logk[e] = m.hkey[r.cur * k + i0 + lane];
                m.logr[e] = (uint32_t)(roundno - 1);
              }
              lg.waiting += __popc(b);
              __syncwarp();
            }
        }
      }
    }
  };

  if constexpr (kRow128<DT, CPR>) {
    // uint8 rows of 128 bytes lie in the stages as they are (eight lanes copy
    // a row, so a copy's place is the lane's plus a constant); thread i reads
    // its row's pieces in the order c ^ (i & 7), without bank conflicts, and
    // holds the query's pieces in registers in that order. With the segment
    // window this takes 373 warp instructions per 32 rows where swizzled
    // stages and a search per tile took 523: 4-15% of a batch of 300 to 1,300
    // queries (1,000 queries x 30,000 rows 672 -> 625 us); at 10,000 queries
    // HBM binds either way.
    uint4 w[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) w[c] = reinterpret_cast<const uint4 *>(m.sq)[c ^ (lane & 7)];
    const uint8_t *piece = a.vec + (lane & 7) * 16;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(m.stage) + (uint32_t)(warp * 4096 + lane * 16);
    const uint32_t mine = (uint32_t)(tid * 128 + (lane & 7) * 16);
    uint32_t rows[ST];  // of the tiles in flight, the oldest first
    auto issue = [&](uint32_t t, uint32_t st) {
#pragma unroll
      for (int i = 0; i + 1 < ST; ++i) rows[i] = rows[i + 1];
      if (t < ntiles) {
        const uint32_t row = rows[ST - 1] = row_of(t);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint32_t gr = __shfl_sync(kFull, row, i * 4 + (lane >> 3));
          cp_async16(dst + st * (TR * 128u) + i * 512u, piece + (size_t)gr * 128);
        }
      }
      cp_async_commit();
    };
#pragma unroll
    for (int i = 0; i < ST; ++i) rows[i] = 0;
#pragma unroll
    for (int i = 0; i + 1 < ST; ++i) issue(i, i);
    uint32_t st = 0, into = ST - 1;  // the stages of tile t and of the one being issued
    for (uint32_t t = 0; t < ntiles && !r.stop; ++t) {
      issue(t + ST - 1, into);
      const uint64_t ext = ~nthr;
      if (!direct) nthr = __ldcg(lg.nthr);
      cp_async_wait<ST - 1>();
      __syncwarp();
      const uint32_t at = mine + st * (TR * 128u);
      into = st;
      st = st + 1 == ST ? 0 : st + 1;
      unsigned a0 = 0, a1 = 0, a2 = 0, a3 = 0;  // integer sums: any order is exact
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const uint4 v = *reinterpret_cast<const uint4 *>(m.stage + (at ^ (c * 16u)));
        unsigned d;
        d = __vabsdiffu4(v.x, w[c].x); a0 = __dp4a(d, d, a0);
        d = __vabsdiffu4(v.y, w[c].y); a1 = __dp4a(d, d, a1);
        d = __vabsdiffu4(v.z, w[c].z); a2 = __dp4a(d, d, a2);
        d = __vabsdiffu4(v.w, w[c].w); a3 = __dp4a(d, d, a3);
      }
      merge(t, (a0 + a1) + (a2 + a3), rows[0], ext);
    }
    cp_async_wait<0>();
  } else {
    const int cpr = CPR > 0 ? CPR : a.cpr;
    constexpr int swz_c = KCC > 0 ? KCC : CPR;
    constexpr bool kLanes8 = swz_c > 0 && swz_c % 8 == 0;
    const int swz = swz_c > 0 ? ((swz_c % 8 == 0) ? 7 : (swz_c % 4 == 0) ? 3 : (swz_c % 2 == 0) ? 1 : 0)
                              : a.swz_mask;
    const int64_t RB = (int64_t)cpr * 16;
    const int pc = KCC > 0 ? KCC : cpr;       // chunks of a row in a stage
    const uint32_t PB = (uint32_t)pc * 16u;   // bytes of a row in a stage
    const uint32_t nk = KCC > 0 ? (uint32_t)(cpr / KCC) : 1u;  // pieces per row
    const uint32_t nitems = ntiles * nk;
    const uint32_t stage_s = (uint32_t)__cvta_generic_to_shared(m.stage);
    uint32_t grow = 0;  // this thread's row in the tile being issued
    auto issue = [&](uint32_t it, uint32_t st) {
      if (it < nitems) {
        const uint32_t t = KCC > 0 ? it / nk : it;
        const uint32_t kk = KCC > 0 ? it - t * nk : 0u;
        if (KCC == 0 || kk == 0) {  // a new tile
          grow = row_of(t);
          m.srow[(t % ST) * TR + tid] = grow;
        }
        const uint32_t sbase = stage_s + st * (uint32_t)(TR * PB);
        if constexpr (kLanes8) {
          // eight lanes a row, every eighth chunk a lane: the swizzle moves a
          // chunk among its eight, so a copy's place is one of two offsets of
          // the lane (by the parity of its four rows) plus a constant. 10,000
          // fp32 queries (D = 96) 5,451 -> 5,130 us, four 1536-value ones 190
          // -> 166 against a chunk index divided and swizzled per copy.
          const uint32_t x = (uint32_t)(lane & 7), y = (uint32_t)(lane >> 3);
          const uint32_t even = sbase + (warp * 32 + y) * PB + ((x ^ y) << 4);
          const uint32_t odd = sbase + (warp * 32 + y) * PB + ((x ^ (y + 4)) << 4);
          const uint8_t *piece = a.vec + (size_t)kk * PB + x * 16;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint8_t *src = piece + (size_t)__shfl_sync(kFull, grow, i * 4 + (lane >> 3)) * RB;
#pragma unroll
            for (int j = 0; j < swz_c / 8; ++j)
              cp_async16((i & 1 ? odd : even) + i * 4 * PB + j * 128, src + j * 128);
          }
        } else {
          const uint32_t wbase = p0 + t * TR + warp * 32;
#pragma unroll 4
          for (int f = lane; f < 32 * pc; f += 32) {
            const int rr = f / pc;
            const int c = f - rr * pc;
            const uint32_t gr = __shfl_sync(kFull, grow, rr);
            if (wbase + rr < p1) {
              const int row = warp * 32 + rr;
              const uint32_t dst = sbase + (uint32_t)(row * PB) + (uint32_t)((c ^ (row & swz)) << 4);
              cp_async16(dst, a.vec + (size_t)gr * RB + (size_t)kk * PB + ((size_t)c << 4));
            }
          }
        }
      }
      cp_async_commit();
    };
#pragma unroll
    for (int i = 0; i + 1 < ST; ++i) issue(i, i);
    uint32_t st = 0, into = ST - 1;  // the stages of item it and of the one being issued
    float acc = 0.0f;  // a long row's distance so far
    for (uint32_t it = 0; it < nitems && !r.stop; ++it) {
      issue(it + ST - 1, into);
      const uint64_t ext = ~nthr;
      if (!direct) nthr = __ldcg(lg.nthr);
      cp_async_wait<ST - 1>();
      __syncwarp();
      const uint32_t t = KCC > 0 ? it / nk : it;
      const uint32_t kk = KCC > 0 ? it - t * nk : 0u;
      uint32_t dkey = 0xffffffffu;
      if (p0 + t * TR + tid < p1) {
        const unsigned char *row = m.stage + (size_t)st * TR * PB + (size_t)tid * PB;
        if (DT == 0) {
          unsigned a0 = 0, a1 = 0, a2 = 0, a3 = 0;  // integer sums: any order is exact
#pragma unroll 8
          for (int c = 0; c < cpr; ++c) {
            const uint4 v = *reinterpret_cast<const uint4 *>(row + ((c ^ (tid & swz)) << 4));
            const uint4 w = reinterpret_cast<const uint4 *>(m.sq)[c];
            unsigned d;
            d = __vabsdiffu4(v.x, w.x); a0 = __dp4a(d, d, a0);
            d = __vabsdiffu4(v.y, w.y); a1 = __dp4a(d, d, a1);
            d = __vabsdiffu4(v.z, w.z); a2 = __dp4a(d, d, a2);
            d = __vabsdiffu4(v.w, w.w); a3 = __dp4a(d, d, a3);
          }
          dkey = (a0 + a1) + (a2 + a3);
        } else {
          const float4 *q4 = reinterpret_cast<const float4 *>(m.sq + (size_t)kk * PB);
          if (KCC == 0) acc = 0.0f;  // sequential over j: the order fixes the rounding
#pragma unroll 8
          for (int c = 0; c < pc; ++c) {
            const float4 v = *reinterpret_cast<const float4 *>(row + ((c ^ (tid & swz)) << 4));
            const float4 w = q4[c];
            float d;
            d = __fsub_rn(v.x, w.x); acc = __fmaf_rn(d, d, acc);
            d = __fsub_rn(v.y, w.y); acc = __fmaf_rn(d, d, acc);
            d = __fsub_rn(v.z, w.z); acc = __fmaf_rn(d, d, acc);
            d = __fsub_rn(v.w, w.w); acc = __fmaf_rn(d, d, acc);
          }
          dkey = __float_as_uint(acc);
        }
      }
      into = st;
      st = st + 1 == ST ? 0 : st + 1;
      if (KCC > 0) {
        if (kk + 1 < nk) {  // the row is not complete yet
          __syncwarp();     // the piece is read before the next copies reuse its stage
          continue;
        }
        acc = 0.0f;
      }
      merge(t, dkey, m.srow[(t % ST) * TR + tid], ext);
    }
    cp_async_wait<0>();
  }
  __syncthreads();
}

// The commit stages the first entries of the spans that can change the top-k in
// the tiles' stages, which are free between spans.
constexpr int kStagedEntries = 64;

struct CommitView {  // over the stages
  uint64_t *min;     // [TR] smallest key of the batch's spans (kEmpty: nothing logged)
  uint32_t *off;     // [TR] first block
  uint32_t *slot;    // [TR] staged at, or 0xffffffff
  uint32_t *want;    // [slots] the span of a slot
  uint4 *entry;      // [slots][kStagedEntries]
};

// Commits the finished spans from `next` on, in stream order, to the query's
// top-k: until one is not finished, was not logged (returns true), or the stop.
// Whole block of TR threads. Spans are looked at TR at a time: those whose smallest key is
// below the k-th have their first entries staged together, so a batch costs two
// memory latencies and not one a span, and a round's members are merged by the
// whole block. polls: how often to look again for one that is not finished.
template <int TR, int SLOTS>
__device__ __forceinline__ bool commit_block(const RefineParams &a, const RefineSmem &m, SpanRun &r,
                                             const SpanEntry *pool, uint32_t cap,
                                             const uint32_t *ready, const SpanHeader *hdr,
                                             uint32_t &next, uint32_t spans, uint32_t n,
                                             uint32_t span_rows, int polls) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k = a.k;
  CommitView c;
  c.min = reinterpret_cast<uint64_t *>(m.stage);
  c.off = reinterpret_cast<uint32_t *>(c.min + TR);
  c.slot = c.off + TR;
  c.want = c.slot + TR;
  c.entry = reinterpret_cast<uint4 *>(c.want + 64);
  int *ctl = m.sctl + 1;  // [0] the first span not to commit; then counters
  const int rounds_span = (int)((span_rows + (uint32_t)a.R - 1u) / (uint32_t)a.R);
  const int rounds_last = (int)((n - (spans - 1u) * span_rows + (uint32_t)a.R - 1u) / (uint32_t)a.R);
  auto kth = [&]() { return r.hn == k ? m.hkey[r.cur * k + k - 1] : kEmpty; };
  while (next < spans) {
    const uint32_t x = next + tid;
    const uint32_t rdy = x < spans ? ld_acquire(&ready[x]) : 0u;
    if (tid == 0) ctl[0] = TR;
    const bool logged = rdy > 1u && rdy != kSpanRedo;
    uint4 h = make_uint4(0xffffffffu, 0xffffffffu, 0u, 0u);
    if (logged) h = __ldcg(reinterpret_cast<const uint4 *>(hdr + x));
    __syncthreads();
    if (rdy == 0u || rdy == kSpanRedo) atomicMin(&ctl[0], tid);
    c.min[tid] = ((uint64_t)h.y << 32) | h.x;
    c.off[tid] = h.z;
    c.slot[tid] = 0xffffffffu;
    __syncthreads();
    const int nb = ctl[0];  // finished spans of this batch
    const bool redo = __syncthreads_or(tid == nb && rdy == kSpanRedo);
    if (nb == 0 && polls > 0 && !redo) {
      --polls;
      continue;
    }
    {  // stage, the earliest first
      const uint64_t top = kth();
      // wanted spans, counted by every thread: a word of ctl would be cleared
      // below while other warps may not have read it yet
      int nw = 0;
      for (int i0 = 0, at = 0; i0 < nb && at < SLOTS; i0 += 32) {
        const unsigned b = __ballot_sync(kFull, i0 + lane < nb && c.min[min(i0 + lane, TR - 1)] < top);
        if (warp == 0 && ((b >> lane) & 1u)) {
          const int sl = at + __popc(b & ((1u << lane) - 1u));
          if (sl < SLOTS) {
            c.slot[i0 + lane] = sl;
            c.want[sl] = i0 + lane;
          }
        }
        at += __popc(b);
        nw = min(at, SLOTS);
      }
      __syncthreads();
      for (int e = tid; e < nw * kStagedEntries; e += TR) {
        const uint32_t at = c.off[c.want[e / kStagedEntries]] + (uint32_t)(e % kStagedEntries);
        if (at < cap) cp_async16((uint32_t)__cvta_generic_to_shared(c.entry + e), pool + at);
      }
      cp_async_commit();
      cp_async_wait<0>();
      if (tid == 0) ctl[0] = ctl[1] = ctl[2] = 0;  // survivor counters, as refine_span's
      __syncthreads();
    }
    int at = 0, ci = 0;  // spans of the batch committed; merges (counters rotate)
    while (at < nb && !r.stop) {
      int j = nb;  // the next span that can change the top-k
      const uint64_t top = kth();
      for (int i0 = at & ~31; i0 < nb; i0 += 32) {
        const int i = i0 + lane;
        const unsigned b = __ballot_sync(kFull, i >= at && i < nb && c.min[min(i, TR - 1)] < top);
        if (b) {
          j = i0 + __ffs(b) - 1;
          break;
        }
      }
      const bool last = j == nb && next + nb == spans;  // the stream's last span may be short
      rounds_unchanged(a, r, (j - at - (last ? 1 : 0)) * rounds_span + (last ? rounds_last : 0));
      at = j;
      if (r.stop || j == nb) break;
      // span j: its members round by round
      const uint32_t sl = c.slot[j];
      int open = -1;  // the round being merged
      auto close = [&]() {
        int newc, frontc;
        count_new(m, r, k, a.nfront, r.rounds + 1, newc, frontc);
        round_done(a, r, r.rounds + 1, newc, frontc);
      };
      bool staged = sl != 0xffffffffu;
      for (uint64_t blk = c.off[j]; blk != kEmpty && !r.stop;) {
        const uint4 head = staged ? c.entry[sl * kStagedEntries] : __ldcg(reinterpret_cast<const uint4 *>(pool + blk));
        const int cnt = (int)head.z;
        for (int e0 = 0; e0 < cnt && !r.stop; e0 += TR) {
          const int e = e0 + tid;
          uint4 v = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0u);
          if (e < cnt)
            v = staged && e + 1 < kStagedEntries
                    ? c.entry[sl * kStagedEntries + 1 + e]
                    : __ldcg(reinterpret_cast<const uint4 *>(pool + blk + 1 + e));
          const uint64_t key = ((uint64_t)v.y << 32) | v.x;
          const int nch = min(TR, cnt - e0);
          for (int i = 0; i < nch && !r.stop;) {
            // the round of entry i, which opens if it is not open
            int *cn = &ctl[ci % 3];
            int *rd = reinterpret_cast<int *>(c.want);  // a word per turn
            if (tid == i) rd[ci & 1] = (int)v.z;
            if (tid == 0) ctl[(ci + 1) % 3] = 0;
            __syncthreads();
            const int round = rd[ci & 1];
            if (round != open) {
              if (open >= 0) close();
              if (!r.stop) rounds_unchanged(a, r, round - open - 1);
              if (r.stop) break;
              open = round;
            }
            const bool in = tid >= i && tid < nch && (int)v.z == round;
            uint64_t *sk = m.skey + (ci & 1) * TR;
            if (in && key < kth()) sk[atomicAdd(cn, 1)] = key;
            const int of = __syncthreads_count(in);
            const int ns = *cn;
            if (ns > 0) block_merge<TR>(m, r, k, sk, ns, r.rounds + 1);
            i += of;
            ++ci;
          }
        }
        blk = ((uint64_t)head.y << 32) | head.x;
        staged = false;
      }
      if (!r.stop) close();
      if (!r.stop) rounds_unchanged(a, r, (next + j + 1 == spans ? rounds_last : rounds_span) - open - 1);
      at = j + 1;
    }
    next += (uint32_t)at;
    __syncthreads();  // the view is free
    if (r.stop) return false;
    if (redo) return true;
    if (nb < TR && polls == 0) return false;  // the next one is not finished
  }
  return false;
}

// The same for k <= 32 by one warp, the top-k in its registers (a member a
// lane): a member is merged by a vote and a shift. One query of 242 spans and
// k = 10: 49 us a refinement with the top-k in shared memory, 53 by the block,
// 41 so (37 queries 108, 110, 78).
template <int SLOTS>
__device__ __forceinline__ bool commit_warp(const RefineParams &a, const RefineSmem &m, SpanRun &r,
                                            const SpanEntry *pool, uint32_t cap,
                                            const uint32_t *ready, const SpanHeader *hdr,
                                            uint32_t &next, uint32_t spans, uint32_t n,
                                            uint32_t span_rows, int polls) {
  constexpr int kEntries = 32;  // staged of a span: its block's first entry and 31 members
  const int lane = threadIdx.x & 31, k = a.k;
  uint4 *stage = reinterpret_cast<uint4 *>(m.stage);
  uint64_t hk = lane < r.hn ? m.hkey[r.cur * k + lane] : kEmpty;  // kEmpty past the members
  int ht = 0;                                                     // the round it entered
  const int rounds_span = (int)((span_rows + (uint32_t)a.R - 1u) / (uint32_t)a.R);
  const int rounds_last = (int)((n - (spans - 1u) * span_rows + (uint32_t)a.R - 1u) / (uint32_t)a.R);
  // kEmpty while there is room; by the whole warp (not behind a lane's condition)
  auto kth = [&]() { return __shfl_sync(kFull, hk, k - 1); };
  int open = -1;  // of the span being committed: the round being merged
  auto close = [&]() {
    const int roundno = r.rounds + 1;
    const unsigned nw = __ballot_sync(kFull, lane < r.hn && ht == roundno);
    round_done(a, r, roundno, __popc(nw), __popc(a.nfront < 32 ? nw & ((1u << a.nfront) - 1u) : nw));
  };
  // merges the members of the lanes in `left` (rounds in lane order)
  auto take = [&](uint64_t key, int rd, unsigned left) {
    while (left && !r.stop) {
      const int round = __shfl_sync(kFull, rd, __ffs(left) - 1);
      const unsigned group = __ballot_sync(kFull, rd == round) & left;
      left &= ~group;
      if (round != open) {
        if (open >= 0) close();
        if (!r.stop) rounds_unchanged(a, r, round - open - 1);
        if (r.stop) return;
        open = round;
      }
      const int roundno = r.rounds + 1;
      const uint64_t top = kth();
      unsigned g = __ballot_sync(kFull, key < top) & group;
      for (; g; g &= g - 1) {
        const uint64_t x = __shfl_sync(kFull, key, __ffs(g) - 1);
        const int at = __popc(__ballot_sync(kFull, hk <= x && lane < r.hn));
        const uint64_t uk = __shfl_up_sync(kFull, hk, 1);
        const int ut = __shfl_up_sync(kFull, ht, 1);
        if (lane >= at) {
          hk = lane == at ? x : uk;
          ht = lane == at ? roundno : ut;
        }
        r.hn = min(k, r.hn + 1);
        if (lane >= k) hk = kEmpty;
      }
    }
  };
  bool redo = false;
  while (next < spans && !r.stop) {
    const uint32_t x = next + lane;
    const uint32_t rdy = x < spans ? ld_acquire(&ready[x]) : 0u;
    const bool logged = rdy > 1u && rdy != kSpanRedo;
    uint4 h = make_uint4(0xffffffffu, 0xffffffffu, 0u, 0u);  // smallest key, first block
    if (logged) h = __ldcg(reinterpret_cast<const uint4 *>(hdr + x));
    const uint64_t mk = ((uint64_t)h.y << 32) | h.x;
    // each lane has acquired its own span's flag; the lanes copy one another's
    // logs below, and votes and shuffles order no memory
    __syncwarp();
    const unsigned idle = __ballot_sync(kFull, rdy == 0u || rdy == kSpanRedo);
    const int nb = idle ? __ffs(idle) - 1 : 32;  // finished spans of this batch
    redo = nb < 32 && __shfl_sync(kFull, rdy, nb & 31) == kSpanRedo;
    if (nb == 0 && polls > 0 && !redo) {
      --polls;
      continue;
    }
    const uint64_t top = kth();
    const unsigned want = __ballot_sync(kFull, lane < nb && mk < top);  // can change the top-k
    const int slot = __popc(want & ((1u << lane) - 1u));
    int sl = 0;
    for (unsigned b = want; b && sl < SLOTS; b &= b - 1, ++sl) {
      const uint32_t at = __shfl_sync(kFull, h.z, __ffs(b) - 1) + (uint32_t)lane;
      if (at < cap) cp_async16((uint32_t)__cvta_generic_to_shared(stage + sl * kEntries + lane), pool + at);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncwarp();
    int at = 0;  // spans of the batch committed
    while (at < nb) {
      const uint64_t now = kth();
      const unsigned b = want & __ballot_sync(kFull, mk < now) & (kFull << at);
      const int j = b ? __ffs(b) - 1 : nb;  // the next one that can change it
      const bool last = j == nb && next + nb == spans;  // the stream's last span may be short
      rounds_unchanged(a, r, (j - at - (last ? 1 : 0)) * rounds_span + (last ? rounds_last : 0));
      at = j;
      if (r.stop || j == nb) break;
      const int sj = __shfl_sync(kFull, slot, j);
      bool staged = sj < SLOTS;
      open = -1;
      for (uint64_t blk = __shfl_sync(kFull, h.z, j); blk != kEmpty && !r.stop;) {
        // lane 0: the block's first entry; the members after it
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (staged) v = stage[sj * kEntries + lane];
        else if (blk + lane < cap) v = __ldcg(reinterpret_cast<const uint4 *>(pool + blk + lane));
        const uint64_t key = ((uint64_t)v.y << 32) | v.x;
        const uint64_t after = __shfl_sync(kFull, key, 0);
        const int cnt = (int)__shfl_sync(kFull, v.z, 0);
        take(key, (int)v.z, __ballot_sync(kFull, lane >= 1 && lane <= cnt));
        for (int e0 = kEntries; e0 <= cnt && !r.stop; e0 += 32) {
          const int e = e0 + lane;
          if (e <= cnt) v = __ldcg(reinterpret_cast<const uint4 *>(pool + blk + e));
          take(((uint64_t)v.y << 32) | v.x, (int)v.z, __ballot_sync(kFull, e <= cnt));
        }
        blk = after;
        staged = false;
      }
      if (!r.stop) close();
      if (!r.stop) rounds_unchanged(a, r, (next + j + 1 == spans ? rounds_last : rounds_span) - open - 1);
      at = j + 1;
      if (r.stop) break;
    }
    next += (uint32_t)at;
    __syncwarp();  // the stages are free
    if (r.stop || redo || (nb < 32 && polls == 0)) break;
  }
  if (lane < r.hn) {
    m.hkey[r.cur * k + lane] = hk;
    m.htag[r.cur * k + lane] = 0;
  }
  __syncwarp();
  return redo && !r.stop;
}

}  // namespace nrq
