// Input staging and rough-graph construction.
//
//  k_sort         per event, a stable counting sort of the hits by plane: the
//                 sorted order is (event, plane, input index), so the
//                 candidates of a hit on plane p (planes p+1 and p+2) form one
//                 contiguous range.
//  k_graph_event  per event, the rough graph of Sec. "Hit Embedding and Rough
//                 Graph Construction" in CSR form and its in-edge index (see
//                 the kernel's comment): degrees, offsets (block scan plus a
//                 look-back over the earlier events), fill, in-edge lists.
//  k_scan_*       exclusive scan in two kernels (block sums, with the last
//                 block scanning them; then block scans plus the block offset),
//                 used by the triplet stage.
#include <cooperative_groups.h>

#include <algorithm>

#include "internal.cuh"

namespace gnntrk {

namespace cg = cooperative_groups;

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kSortThreads = 256;
constexpr int kScanThreads = 512;
constexpr int kMidHits = 1280;  // see GraphShape
constexpr int kScanPer = 8;
constexpr int kScanChunk = kScanThreads * kScanPer;

__device__ __forceinline__ bool input_bad(const Ws& w) {
  return (*(volatile int32_t*)&w.counters[C_STATUS] & ST_INPUT) != 0;
}

// ---------------------------------------------------------------------------
// stable plane sort, one block per event
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kSortThreads) k_sort(Batch b, Ws w, const int64_t* offsets, int P) {
  __shared__ int cnt[kMaxPlanes];
  __shared__ int base[kMaxPlanes];
  __shared__ int wcnt[kSortThreads / 32][kMaxPlanes];
  __shared__ int ctot[kMaxPlanes];
  __shared__ int bad;
  const int ev = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_begin();
  const int64_t o0 = offsets[ev], o1 = offsets[ev + 1];
  if (w.rs_counts != nullptr && ev == 0)
    for (int i = tid; i < 6 * (kMaxIters + 2); i += kSortThreads) w.rs_counts[i] = 0;
  if (tid == 0) {
    w.ev_off[ev] = o0;
    if (ev == b.n_events - 1) w.ev_off[ev + 1] = o1;
    w.graph_desc[ev] = 0;
    if (w.rs_desc != nullptr) w.rs_desc[ev] = 0;
    if (o1 - o0 > kMidHits) w.counters[C_LARGE_EVENT] = 1;
    int f = 0;
    if (o0 < 0 || o1 < o0 || o1 > b.n_hits) f = 1;
    if (ev == 0 && o0 != 0) f = 1;
    if (ev == b.n_events - 1 && o1 != b.n_hits) f = 1;
    if (f) set_status(w.counters, ST_INPUT);
    bad = f;
  }
  for (int i = tid; i < P; i += kSortThreads) cnt[i] = 0;
  for (int i = tid; i < (kSortThreads / 32) * kMaxPlanes; i += kSortThreads)
    (&wcnt[0][0])[i] = 0;
  __syncthreads();
  if (bad) return;
  const int lo = int(o0), hi = int(o1);

  for (int i = lo + tid; i < hi; i += kSortThreads) {
    int p = b.plane[i];
    if (p >= P) {
      set_status(w.counters, ST_INPUT);
      p = P - 1;
    }
    atomicAdd(&cnt[p], 1);
  }
  __syncthreads();
  if (tid == 0) {
    int run = 0;
    int32_t* po = w.plane_off + size_t(ev) * (P + 1);
    for (int p = 0; p < P; ++p) {
      base[p] = run;
      po[p] = lo + run;
      run += cnt[p];
    }
    po[P] = hi;
  }
  __syncthreads();

  for (int c0 = lo; c0 < hi; c0 += kSortThreads) {
    const int i = c0 + tid;
    const bool valid = i < hi;
    const int p = valid ? min(int(b.plane[i]), P - 1) : P;
    const unsigned peers = __match_any_sync(kFull, p);
    const int rank = __popc(peers & ((1u << lane) - 1u));
    if (valid && rank == 0) wcnt[warp][p] = __popc(peers);
    __syncthreads();
    if (tid < P) {
      int run = 0;
      for (int k = 0; k < kSortThreads / 32; ++k) {
        int t = wcnt[k][tid];
        wcnt[k][tid] = run;
        run += t;
      }
      ctot[tid] = run;
    }
    __syncthreads();
    if (valid) {
      const int d = lo + base[p] + wcnt[warp][p] + rank;
      w.perm[d] = i;
      w.node_event[d] = ev;
      w.pos[d] = make_float4(b.x[i], b.y[i], b.z[i], 0.0f);
      w.in_cnt[d] = 0;
      w.deg[d] = 0;
    }
    __syncthreads();
    if (tid < P) base[tid] += ctot[tid];
    for (int k = tid; k < (kSortThreads / 32) * kMaxPlanes; k += kSortThreads)
      (&wcnt[0][0])[k] = 0;
    __syncthreads();
  }
  for (int i = lo + tid; i < hi; i += kSortThreads) w.parent[i] = i;
}

// ---------------------------------------------------------------------------
// radius search helpers
// ---------------------------------------------------------------------------
template <int D>
__device__ __forceinline__ float dist2(const float (&q)[D], const float* c) {
  float cv[D];
  if constexpr (D % 4 == 0) {  // 16-byte loads (rows are 16-byte aligned)
#pragma unroll
    for (int d = 0; d < D; d += 4) {
      const float4 v = *reinterpret_cast<const float4*>(c + d);
      cv[d] = v.x;
      cv[d + 1] = v.y;
      cv[d + 2] = v.z;
      cv[d + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int d = 0; d < D; ++d) cv[d] = c[d];
  }
  float s = 0.0f;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const float t = q[d] - cv[d];
    s = fmaf(t, t, s);
  }
  return s;
}

template <int D>
__device__ __forceinline__ void load_row(const float* r, float (&q)[D]) {
  if constexpr (D % 4 == 0) {
#pragma unroll
    for (int d = 0; d < D; d += 4) {
      const float4 v = *reinterpret_cast<const float4*>(r + d);
      q[d] = v.x;
      q[d + 1] = v.y;
      q[d + 2] = v.z;
      q[d + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int d = 0; d < D; ++d) q[d] = r[d];
  }
}

// Candidate rows of an event, by event-local index c. Both forms give d^2 =
// sum_d (q_d - c_d)^2 accumulated by fmaf in increasing d, bit for bit:
//  CandRows  rows of D floats (global memory, events too large to stage);
//  CandNegT  the event staged in shared memory transposed and negated,
//            t[d * ns + c] = -e_c[d], so that four candidates c .. c + 3 of one
//            dimension are one 16-byte load and q_d + (-c_d) (exactly q_d - c_d)
//            runs as a packed FP32 add, two candidates per instruction.
template <int D>
struct CandRows {
  const float* e;
  __device__ __forceinline__ float d2(const float (&q)[D], int c) const {
    return dist2<D>(q, e + size_t(c) * D);
  }
  __device__ __forceinline__ void row(int c, float (&q)[D]) const { load_row<D>(e + size_t(c) * D, q); }
};

template <int D>
struct CandNegT {
  const float* t;
  int ns;
  __device__ __forceinline__ float d2(const float (&q)[D], int c) const {
    float s = 0.0f;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const float u = q[d] + t[d * ns + c];
      s = fmaf(u, u, s);
    }
    return s;
  }
  // d^2 of the candidates c .. c + 3 (c a multiple of 4)
  __device__ __forceinline__ float4 d2_quad(const float (&q)[D], int c) const {
    float2 s = make_float2(0.0f, 0.0f), z = s;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const float4 nc = *reinterpret_cast<const float4*>(t + d * ns + c);
      const float2 u = __fadd2_rn(make_float2(q[d], q[d]), make_float2(nc.x, nc.y));
      const float2 v = __fadd2_rn(make_float2(q[d], q[d]), make_float2(nc.z, nc.w));
      s = __ffma2_rn(u, u, s);
      z = __ffma2_rn(v, v, z);
    }
    return make_float4(s.x, s.y, z.x, z.y);
  }
  __device__ __forceinline__ void row(int c, float (&q)[D]) const {
#pragma unroll
    for (int d = 0; d < D; ++d) q[d] = -t[d * ns + c];
  }
};

// number of candidates [c0, c0 + nc) inside the radius whose key (d^2 as
// ordered bits) is < bound (<= bound when inclusive)
template <int D, class Cand>
__device__ int count_below(const Cand& cd, const float (&q)[D], int c0, int nc, float r2,
                           unsigned bound, bool inclusive) {
  const int lane = threadIdx.x & 31;
  int n = 0;
  for (int base = 0; base < nc; base += 32) {
    const int c = base + lane;
    bool ok = false;
    if (c < nc) {
      const float s = cd.d2(q, c0 + c);
      const unsigned key = __float_as_uint(s);
      ok = s < r2 && (inclusive ? key <= bound : key < bound);
    }
    n += __popc(__ballot_sync(kFull, ok));
  }
  return n;
}

// The edges of one hit with more than k_max candidates inside the radius,
// written by its warp: the k_max smallest keys (d^2 as ordered bits), ties
// broken by candidate position, in ascending candidate order. T is the
// k_max-th smallest key (bisection over the key bits); keys < T are kept,
// then the first keys == T. Candidates are [c0, c0 + nc), event-local;
// positions are written as pos0 + local index.
template <int D, class Cand>
__device__ void fill_capped(const Ws& w, const Cand& cd, const float (&qe)[D], int c0, int nc,
                            float r2, int k_max, int64_t out0, int src_pos, int pos0) {
  const int lane = threadIdx.x & 31;
  unsigned lo = 0, hi = __float_as_uint(r2);
  for (int it = 0; it < 40 && lo < hi; ++it) {
    const unsigned mid = lo + (hi - lo) / 2;
    if (count_below<D>(cd, qe, c0, nc, r2, mid, true) >= k_max)
      hi = mid;
    else
      lo = mid + 1;
  }
  const unsigned T = lo;
  const int need_eq = k_max - count_below<D>(cd, qe, c0, nc, r2, T, false);
  int written = 0, eq_seen = 0;
  for (int base = 0; base < nc; base += 32) {
    const int c = base + lane;
    bool ok = false, eq = false;
    float s = 0.0f;
    if (c < nc) {
      s = cd.d2(qe, c0 + c);
      if (s < r2) {
        const unsigned key = __float_as_uint(s);
        eq = key == T;
        ok = key < T;
      }
    }
    const unsigned eqm = __ballot_sync(kFull, eq);
    const int eq_rank = eq_seen + __popc(eqm & ((1u << lane) - 1u));
    if (eq && eq_rank < need_eq) ok = true;
    eq_seen += __popc(eqm);
    const unsigned m = __ballot_sync(kFull, ok);
    if (ok) {
      const int64_t e = out0 + written + __popc(m & ((1u << lane) - 1u));
      if (e < w.e_cap) {
        w.col[e] = pos0 + c0 + c;
        w.src[e] = src_pos;
        w.d2[e] = s;
      }
    }
    written += __popc(m);
  }
}

// The k_max edges of a hit over k_max as its mask (the same selection as
// fill_capped), rewritten by its warp: mrow[k] bit b is candidate
// cA + 32 k + b, candidates [c0, c1).
template <int D, class Cand>
__device__ void select_capped(const Cand& cd, const float (&qe)[D], int c0, int c1, int cA,
                              float r2, int k_max, uint32_t* mrow) {
  const int lane = threadIdx.x & 31;
  const int nc = c1 - c0;
  unsigned lo = 0, hi = __float_as_uint(r2);
  for (int it = 0; it < 40 && lo < hi; ++it) {
    const unsigned mid = lo + (hi - lo) / 2;
    if (count_below<D>(cd, qe, c0, nc, r2, mid, true) >= k_max)
      hi = mid;
    else
      lo = mid + 1;
  }
  const unsigned T = lo;
  const int need_eq = k_max - count_below<D>(cd, qe, c0, nc, r2, T, false);
  int eq_seen = 0;
  for (int k = 0; cA + 32 * k < c1; ++k) {
    const int c = cA + 32 * k + lane;
    bool keep = false, eq = false;
    if (c >= c0 && c < c1) {
      const float s = cd.d2(qe, c);
      if (s < r2) {
        const unsigned key = __float_as_uint(s);
        eq = key == T;
        keep = key < T;
      }
    }
    const unsigned eqm = __ballot_sync(kFull, eq);
    if (eq && eq_seen + __popc(eqm & ((1u << lane) - 1u)) < need_eq) keep = true;
    eq_seen += __popc(eqm);
    const unsigned m = __ballot_sync(kFull, keep);
    if (lane == 0) mrow[k] = m;
  }
}

// ---------------------------------------------------------------------------
// rough graph and in-edge index, one block per event
// ---------------------------------------------------------------------------
// Rough graph of Sec. "Hit Embedding and Rough Graph Construction": hit i on
// plane p joins hit j on plane p+1 or p+2 when d^2(i, j) = |e_i - e_j|^2 <
// d^2_max, keeping at most k_max per i (the k_max smallest by (d^2, sorted
// position)); the edges of a hit are stored in ascending target order, the
// hits in sorted order (CSR). Then the in-edge index: each hit's in-edges in
// ascending edge id, so that message sums run in a fixed order.
//
// Events go to blocks in index order by a ticket (counters[C_GRAPH_TICKET]),
// and each event takes its global edge offset (the edges of all earlier
// events) from a look-back over the totals its predecessors publish: an event
// publishes its own edge count as soon as its degrees are known and its
// inclusive prefix after its look-back, so a block only waits for blocks that
// took their tickets before it and are therefore running. Per event, all in
// shared memory when it fits (GraphPlan):
//   1. masks: an item is 32 query hits of one plane (a lane each, so that the
//      lanes read the same candidate rows, broadcast) x 32 candidates, one
//      mask word per hit; degrees are the popcounts; a hit over k_max keeps its
//      k_max selected candidates;
//   2. CSR offsets: block scan, the event's count published;
//   3. targets: a thread per hit lists its mask's bits as 16-bit targets and
//      counts the in-edges of each;
//   4. in-edge lists: a scan of the counts, placement by cursors, a thread per
//      edge; an entry's place is the number of smaller entries in its list;
//   5. after the look-back: the edges (a thread per edge, d^2 again from the
//      staged rows), the lists and the row pointers, all in coalesced stores.
// An event too large for that falls back step by step: without the lists the
// hits write their mask's edges one by one and the in-edge index is built over
// global memory (csc_general); without the masks the candidates are tested
// again in the fill; without the staged rows they are read from global memory.
//
// What bounds it: the distance tests (an event of 1689 hits in 4 dimensions and
// 10.1 k edges: 44 of about 102 thousand cycles, 117 of 228 at 2195 hits in 8
// dimensions), then the latency of the short steps. Before, each lane stored
// its hit's edges to scattered places (68 of 275 thousand cycles; 326 of 655),
// and the in-edge lists of an event over 14 k list words were sorted in global
// memory (155 thousand cycles).

// One block of 1024 threads per SM with all of its shared memory: every event
// of up to about 2.5 k hits then stays in shared memory, and the threads of one
// event finish its short steps sooner than those of two events side by side.
// Per call (two blocks of 512 threads with half the memory each; before the
// lists were built in shared memory): 1000 events of 1685 hits 433 us (568;
// 626), 400 events of 2185 hits and 13 k edges 248 us (648; 622), one event of
// 2146 hits in 8 dimensions 116 us (299; 287).
//
// Batches of thousands of small events spend those blocks' time at barriers. Such a
// call takes two blocks of 512 threads per SM if no event has more than kMidHits hits,
// which the sort finds out. Graph kernel in us with one / two blocks per SM (and with
// the two blocks of before): 40 000 events of 11 hits 2366 / 1030 (1357), 5000 of 56
// hits 316 / 164 (218), 1000 of 450 hits 93 / 65 (85). The line is where half the shared
// memory no longer holds an event in 8 dimensions: 1000 events of 1340 hits 351 / 349
// (402); two events of 4400 hits among 600 of 32: 205 / 768 (476).
template <int NT_, int PER_SM_, int KB>
struct GraphShape {
  static constexpr int NT = NT_, WARPS = NT_ / 32, PER_SM = PER_SM_;
  static constexpr int INTS = KB * 1024 / 4;  // shared memory of an event's arrays
};
using GraphWide = GraphShape<1024, 1, 224>;
using GraphMid = GraphShape<512, 2, 110>;
// calls whose largest event decides (a launch more: of the two one ends at once, about
// 2 us): a few thousand events at least, of half that size on average
inline bool by_largest_event(int n_events, int n_hits, int sms) {
  return n_events >= 16 * sms && n_hits <= int64_t(n_events) * (kMidHits / 2);
}
enum GraphWhen : int { G_ALWAYS = 0, G_ALL_SMALL = 1, G_SOME_LARGE = 2 };
constexpr unsigned long long kDescAgg = 1ull << 62;  // the event's own edge count
constexpr unsigned long long kDescInc = 2ull << 62;  // edges up to and including the event
constexpr unsigned long long kDescVal = (1ull << 62) - 1;
constexpr int kLookbackSpins = 1 << 22;  // x >= 100 ns sleeps: a bound of about half a second

// The look-back walks back over windows of 32 predecessors until one has
// published its inclusive prefix, summing the counts of the others. A wait
// that runs out sets ST_TIMEOUT and returns what was summed (the event then
// publishes no inclusive prefix; later events sum its count instead).

// (lane 0) publishes the event's edge count: event 0's is its inclusive prefix
__device__ __forceinline__ void graph_publish(unsigned long long* desc, int ev, long long agg) {
  atomicExch(desc + ev, (ev == 0 ? +kDescInc : +kDescAgg) | static_cast<unsigned long long>(agg));
}

// Warp 0, after graph_publish: the edges of all earlier events, then the
// event's inclusive prefix published.
__device__ long long graph_wait(unsigned long long* desc, int ev, long long agg,
                                int32_t* counters) {
  const int lane = threadIdx.x & 31;
  long long excl = 0;
  int spins = 0;
  for (int top = ev - 1; top >= 0; top -= 32) {
    const int i = top - lane;
    unsigned long long d = i >= 0 ? *reinterpret_cast<volatile unsigned long long*>(desc + i)
                                  : +kDescInc;  // before event 0: an inclusive prefix of 0
    while (__any_sync(kFull, (d >> 62) == 0)) {
      if (++spins > kLookbackSpins) {
        if (lane == 0) set_status(counters, ST_TIMEOUT);
        return excl;
      }
      __nanosleep(100);
      if ((d >> 62) == 0) d = *reinterpret_cast<volatile unsigned long long*>(desc + i);
    }
    const unsigned inc = __ballot_sync(kFull, (d >> 62) == 2);
    const int stop = inc ? __ffs(inc) - 1 : 31;  // the nearest inclusive prefix
    long long v = lane <= stop ? static_cast<long long>(d & kDescVal) : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    excl += v;
    if (inc) break;
  }
  if (lane == 0 && ev > 0)
    atomicExch(desc + ev, kDescInc | static_cast<unsigned long long>(excl + agg));
  return excl;
}

// exclusive scan of min(in[i], clamp) over i < n into out (both may be
// shared or global memory); every thread gets the total
template <class S>
__device__ int block_scan(const int32_t* in, int32_t* out, int n, int clamp, int* wsum) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = (n + S::NT - 1) / S::NT;
  const int a = min(n, tid * per), z = min(n, a + per);
  int sum = 0;
  for (int i = a; i < z; ++i) sum += min(in[i], clamp);
  int x = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(kFull, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  int before = 0, total = 0;
#pragma unroll
  for (int k = 0; k < S::WARPS; ++k) {
    const int t = wsum[k];
    if (k < warp) before += t;
    total += t;
  }
  int run = before + x - sum;
  for (int i = a; i < z; ++i) {
    const int c = min(in[i], clamp);
    out[i] = run;
    run += c;
  }
  __syncthreads();  // out complete, wsum free
  return total;
}

__device__ __forceinline__ int clamp31(long long v) {
  return int(v > 0x7fffffffLL ? 0x7fffffffLL : v);
}

// Per-plane layout of an event, computed by warp 0: plane p's query hits are cut
// into chunks of up to 32 (chunk[p] chunks before plane p), each of its hits
// owns nw[p] mask words from words[p] on, and its mask items (chunk x word)
// start at items[p]. All arrays end with the total at [P - 1] (the last plane
// holds no query hits).
struct GraphPlanes {
  int po[kMaxPlanes + 1];  // event-local plane offsets
  int chunk[kMaxPlanes + 1], items[kMaxPlanes + 1], words[kMaxPlanes + 1], nw[kMaxPlanes + 1];
};

// first candidate of a mask: the first hit of plane p + 1, rounded down to a quad
__device__ __forceinline__ int mask_first(int c0) { return c0 & ~3; }

__device__ __forceinline__ void graph_planes(GraphPlanes& g, int P) {  // warp 0
  const int lane = threadIdx.x & 31;
  int carry[3] = {0, 0, 0};
  for (int p0 = 0; p0 < P; p0 += 32) {
    const int p = p0 + lane;
    int v[3] = {0, 0, 0}, nw = 0;
    if (p + 1 < P) {
      const int np = g.po[p + 1] - g.po[p], c0 = g.po[p + 1], c1 = g.po[min(p + 3, P)];
      nw = np > 0 && c1 > c0 ? (c1 - mask_first(c0) + 31) / 32 : 0;
      v[0] = (np + 31) / 32;
      v[1] = v[0] * nw;
      v[2] = np * nw;
    }
    int x[3] = {v[0], v[1], v[2]};
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const int y = __shfl_up_sync(kFull, x[i], o);
        if (lane >= o) x[i] += y;
      }
    if (p < P) {
      g.chunk[p] = carry[0] + x[0] - v[0];
      g.items[p] = carry[1] + x[1] - v[1];
      g.words[p] = carry[2] + x[2] - v[2];
      g.nw[p] = nw;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) carry[i] += __shfl_sync(kFull, x[i], 31);
  }
}

// the plane p with first[p] <= t < first[p + 1] (warp-uniform t below the total)
__device__ __forceinline__ int plane_of(const int* first, int P, int t) {
  const int lane = threadIdx.x & 31;
  int p = 0;
  for (int p0 = 1; p0 < P; p0 += 32)
    p += __popc(__ballot_sync(kFull, p0 + lane < P && first[p0 + lane] <= t));
  return p;
}

struct GraphItem {
  int q0, q1, c0, c1;  // its hits [q0, q1) and their candidates [c0, c1), event-local
};

__device__ __forceinline__ GraphItem graph_item(const GraphPlanes& g, int P, int t) {
  const int p = plane_of(g.chunk, P, t);
  return GraphItem{g.po[p] + (t - g.chunk[p]) * 32, g.po[p + 1], g.po[p + 1], g.po[min(p + 3, P)]};
}

// mask words of query hit q on plane p
__device__ __forceinline__ int mask_word(const GraphPlanes& g, int p, int q) {
  return g.words[p] + (q - g.po[p]) * g.nw[p];
}

// 1. mask words: bit b of word k of a hit is candidate mask_first + 32 k + b; this
// block's share of the items, rank of `ranks` blocks
template <class S, int D>
__device__ void graph_masks(const CandNegT<D>& cd, const GraphPlanes& g, int P, float r2,
                            uint32_t* mask, int rank, int ranks) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n_items = g.items[P - 1];
  for (int t = warp * ranks + rank; t < n_items; t += S::WARPS * ranks) {
    const int p = plane_of(g.items, P, t);
    const int nw = g.nw[p], chunk = (t - g.items[p]) / nw, k = t - g.items[p] - chunk * nw;
    const int q = g.po[p] + 32 * chunk + lane, c0 = g.po[p + 1], c1 = g.po[min(p + 3, P)];
    const bool valid = q < c0;
    float qe[D];
    cd.row(valid ? q : g.po[p], qe);
    const int wb = mask_first(c0) + 32 * k;
    unsigned m = 0;
#pragma unroll
    for (int c = 0; c < 32; c += 4) {  // (past c1: staged pad or other rows, masked off)
      const float4 s = cd.d2_quad(qe, wb + c);
      m |= (s.x < r2 ? 1u << c : 0u) | (s.y < r2 ? 2u << c : 0u) | (s.z < r2 ? 4u << c : 0u) |
           (s.w < r2 ? 8u << c : 0u);
    }
    if (wb < c0) m &= ~0u << (c0 - wb);
    if (c1 - wb < 32) m &= (1u << (c1 - wb)) - 1u;
    if (valid) mask[mask_word(g, p, q) + k] = m;
  }
}

// 1. degrees (uncapped) of the event's query hits, without masks
template <class S, int D, class Cand>
__device__ void graph_degrees(const Cand& cd, const GraphPlanes& g, int P, float r2, int32_t* deg) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int t = warp; t < g.chunk[P - 1]; t += S::WARPS) {
    const GraphItem it = graph_item(g, P, t);
    const int q = it.q0 + lane;
    const bool valid = q < it.q1;
    float qe[D];
    cd.row(valid ? q : it.q0, qe);
    int cnt = 0;
    for (int c = it.c0; c < it.c1; ++c) cnt += cd.d2(qe, c) < r2;
    if (valid) deg[q] = cnt;
  }
}

// 3. fill from the candidate masks (which hold exactly each hit's edges,
// capped hits reduced to their selection): one lane per query hit walks the
// set bits of its mask in ascending order, recomputes d^2 there from the
// staged rows and writes its edges at base + off[q].
template <class S, int D>
__device__ void graph_fill_masks(const Ws& w, const CandNegT<D>& cd, const GraphPlanes& g, int P,
                                 const int32_t* off, const uint32_t* mask, long long base, int v0) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int t = warp; t < g.chunk[P - 1]; t += S::WARPS) {
    const int p = plane_of(g.chunk, P, t);
    const int q = g.po[p] + (t - g.chunk[p]) * 32 + lane;
    if (q >= g.po[p + 1]) continue;
    float qe[D];
    cd.row(q, qe);
    int64_t e = base + off[q];
    const int cA = mask_first(g.po[p + 1]);
    for (int k = 0; k < g.nw[p]; ++k) {
      unsigned m = mask[mask_word(g, p, q) + k];
      while (m) {
        const int c = cA + 32 * k + __ffs(m) - 1;
        m &= m - 1;
        if (e < w.e_cap) {
          w.col[e] = v0 + c;
          w.src[e] = v0 + q;
          w.d2[e] = cd.d2(qe, c);
        }
        ++e;
      }
    }
  }
}

// 3. fill without masks: one lane per query hit tests its candidates again in
// ascending order and writes its edges at base + off[q]; a hit over k_max is
// filled by its warp (fill_capped).
template <class S, int D, class Cand>
__device__ void graph_fill(const Ws& w, const Cand& cd, const GraphPlanes& g, int P, float r2,
                           int k_max, const int32_t* deg, const int32_t* off, long long base,
                           int v0) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int t = warp; t < g.chunk[P - 1]; t += S::WARPS) {
    const GraphItem it = graph_item(g, P, t);
    const int q = it.q0 + lane;
    const bool valid = q < it.q1;
    const int cnt = valid ? deg[q] : 0;
    if (valid && cnt > 0 && cnt <= k_max) {
      float qe[D];
      cd.row(q, qe);
      int64_t e = base + off[q];
      for (int c = it.c0; c < it.c1; ++c) {
        const float s = cd.d2(qe, c);
        if (s < r2) {
          if (e < w.e_cap) {
            w.col[e] = v0 + c;
            w.src[e] = v0 + q;
            w.d2[e] = s;
          }
          ++e;
        }
      }
    }
    unsigned capped = __ballot_sync(kFull, cnt > k_max);
    while (capped) {
      const int qq = it.q0 + __ffs(capped) - 1;
      capped &= capped - 1;
      float qe[D];
      cd.row(qq, qe);
      fill_capped<D>(w, cd, qe, it.c0, it.c1 - it.c0, r2, k_max, base + off[qq], v0 + qq, v0);
    }
  }
}

// In-edge index of the event's stored edges [e0, e1) (read back from col):
// in-degrees by shared-memory atomics, a block scan, placement by cursors,
// then each target's list in ascending edge id. When the counts, list starts,
// lists and list targets all fit in shared memory, each list is ranked into
// in_edge (an entry's place is the number of smaller entries in its list);
// else the lists are placed in the event's slice of in_edge and sorted there
// (counts in in_cnt for events of more hits than fit).
template <class S>
__device__ void csc_general(const Ws& w, int n, int v0, int v1, int e0, int e1, int32_t* sm_i,
                            int* wsum) {
  const int tid = threadIdx.x;
  const int ne = e1 - e0;
  const bool full = 2 * int64_t(n) + 2 * int64_t(ne) <= S::INTS;
  const bool c_smem = n <= S::INTS;
  int32_t* C = c_smem ? sm_i : w.in_cnt + v0;
  int32_t* St = sm_i + n;               // (full only) list starts, event-local
  int32_t* L = full ? sm_i + 2 * n : w.in_edge + e0;
  int32_t* Tg = sm_i + 2 * n + ne;      // (full only) target of each list entry
  for (int i = tid; i < n; i += S::NT) C[i] = 0;
  __syncthreads();
  for (int e = e0 + tid; e < e1; e += S::NT) atomicAdd(&C[w.col[e] - v0], 1);
  __syncthreads();
  if (full) {
    block_scan<S>(C, St, n, 0x7fffffff, wsum);
    for (int i = tid; i < n; i += S::NT) {
      C[i] = St[i];  // cursor
      w.in_ptr[v0 + i] = e0 + St[i];
    }
  } else {
    // in place: C becomes the cursors, in_ptr the starts
    const int lane = tid & 31, warp = tid >> 5;
    const int per = (n + S::NT - 1) / S::NT;
    const int a = min(n, tid * per), z = min(n, a + per);
    int sum = 0;
    for (int i = a; i < z; ++i) sum += C[i];
    int x = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(kFull, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    int before = 0;
    for (int k = 0; k < warp; ++k) before += wsum[k];
    int run = before + x - sum;
    for (int i = a; i < z; ++i) {
      const int c = C[i];
      C[i] = run;
      w.in_ptr[v0 + i] = e0 + run;
      run += c;
    }
  }
  if (tid == 0) w.in_ptr[v1] = e1;  // the next event writes the same value
  __syncthreads();
  for (int e = e0 + tid; e < e1; e += S::NT) {
    const int t = w.col[e] - v0;
    const int k = atomicAdd(&C[t], 1);
    L[k] = e;
    if (full) Tg[k] = t;
  }
  __syncthreads();
  // C[i] is now the end of target i's list (event-local position)
  if (full) {
    for (int k = tid; k < ne; k += S::NT) {
      const int e = L[k], t = Tg[k];
      const int lo = St[t], hi = C[t];
      int rank = 0;
      for (int m = lo; m < hi; ++m) rank += L[m] < e;
      w.in_edge[e0 + lo + rank] = e;
    }
  } else {
    for (int i = tid; i < n; i += S::NT) {
      const int lo = w.in_ptr[v0 + i] - e0, hi = C[i];
      for (int j = lo + 1; j < hi; ++j) {
        const int key = L[j];
        int k = j - 1;
        while (k >= lo && L[k] > key) {
          L[k + 1] = L[k];
          --k;
        }
        L[k + 1] = key;
      }
    }
  }
}

// Shared-memory layout of an event (in ints): [off n + 1][cnt n][start n][mask
// words][rows D x ns + pad][targets, 16 bit][sources, 16 bit]. cnt: degrees, then
// in-degrees, then cursors; start: starts of the in-edge lists; the lists (16
// bit) take the mask words' place once the targets are listed. ns: a multiple
// of 4 (quads). Without room for the sources an edge's source is found by
// bisection of the offsets.
struct GraphPlan {
  int n, ns, words, ne;
  int cnt, start, mask, rows, targets;  // offsets; off at 0
  int lists, sources;                   // the in-edge lists, the edges' sources (16 bit)
  int64_t ints_rows, ints_masks, ints_all;
  bool with_sources;                    // the sources fit too

  template <int D>
  __device__ __forceinline__ void rows_and_masks(int n_, int words_) {
    n = n_;
    ns = (n + 3) & ~3;
    words = words_;
    cnt = n + 1;
    start = cnt + n;
    mask = start + n;
    ints_rows = 3 * int64_t(n) + 1 + int64_t(D) * ns + 40;  // without masks
    ints_masks = ints_rows + words;
  }
  // (after ints_masks was found to fit)
  template <int D>
  __device__ __forceinline__ void place_rows(bool masks) {
    rows = (mask + (masks ? words : 0) + 3) & ~3;
  }
  template <class S, int D>
  __device__ __forceinline__ void edges(int ne_) {
    ne = ne_;
    const int half = (ne + 1) / 2;
    targets = rows + D * ns + 36;  // (36: a mask word reads up to 35 past the last row)
    lists = half <= words ? mask : targets + half;
    sources = half <= words ? targets + half : lists + half;
    ints_all = sources;
    with_sources = int64_t(sources) + half <= S::INTS;
  }
};

// CLUSTER: the blocks of a cluster share an event's mask items (the bulk of its
// arithmetic) and write their words into the first block's shared memory, which
// alone does the rest.
template <class S, int D, bool CLUSTER>
__global__ void __launch_bounds__(S::NT, S::PER_SM) k_graph_event(Batch b, Ws w, GraphParams g, GraphWhen when) {
  extern __shared__ __align__(16) float sm_graph[];
  __shared__ GraphPlanes pl;
  __shared__ int wsum[S::WARPS];
  __shared__ int ticket_s;
  __shared__ long long base_s;
  const cg::cluster_group cluster = cg::this_cluster();
  // (no access to another block's shared memory before every block runs; in the time of
  // the kernel before)
  if constexpr (CLUSTER) cluster.sync();
  pdl_begin();
  // (both written by an earlier kernel: uniform over the grid)
  if (input_bad(w)) return;
  if (when != G_ALWAYS && (w.counters[C_LARGE_EVENT] != 0) != (when == G_SOME_LARGE)) return;
  constexpr int NT = S::NT;
  const int rank = CLUSTER ? int(cluster.block_rank()) : 0;
  const int ranks = CLUSTER ? int(cluster.num_blocks()) : 1;
  const int P = g.n_planes;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float r2 = g.radius2;
  const int k_max = g.k_max;
  int32_t* sm_i = reinterpret_cast<int32_t*>(sm_graph);
  for (;;) {
    if (tid == 0 && rank == 0) {
      const int t = atomicAdd(&w.counters[C_GRAPH_TICKET], 1);
      for (int r = 0; r < ranks; ++r) *(CLUSTER ? cluster.map_shared_rank(&ticket_s, r) : &ticket_s) = t;
    }
    if constexpr (CLUSTER)
      cluster.sync();
    else
      __syncthreads();
    const int ev = ticket_s;
    if (ev >= b.n_events) return;
    const int v0 = int(w.ev_off[ev]), v1 = int(w.ev_off[ev + 1]);
    const int n = v1 - v0;
    const int32_t* po = w.plane_off + size_t(ev) * (P + 1);
    if (warp == 0) {
      for (int i = lane; i <= P; i += 32) pl.po[i] = po[i] - v0;
      __syncwarp();
      graph_planes(pl, P);
    }
    __syncthreads();  // the layout below depends on the planes
    GraphPlan L{};
    L.rows_and_masks<D>(n, pl.words[P - 1]);
    const bool staged = L.ints_rows <= S::INTS;
    // The masks, where the shared memory has no room for them, lie in the event's
    // part of the edge states, which the encoder writes later (32 words per hit at
    // least). Testing every candidate again in the fill instead took 446 / 856
    // us for one event of 3.4 k / 4.6 k hits, against 249 / 564.
    const bool masks_s = staged && L.ints_masks <= S::INTS;
    const bool masks = masks_s || (staged && L.words <= 32 * int64_t(n) && w.e_cap >= w.h_cap);
    if (!masks_s) L.words = 0;
    L.place_rows<D>(masks_s);
    int32_t* off = staged ? sm_i : w.in_cnt + v0;
    int32_t* deg = staged ? sm_i + L.cnt : w.deg + v0;
    uint32_t* mask = masks_s ? reinterpret_cast<uint32_t*>(sm_i + L.mask)
                             : reinterpret_cast<uint32_t*>(w.estate) + 32 * size_t(v0);
    float* tT = sm_graph + L.rows;
    if (staged) {
      for (int k = tid; k < n * D; k += NT) {
        const int i = k / D, d = k - i * D;
        tT[d * L.ns + i] = -w.emb[size_t(v0) * D + k];
      }
    }
    __syncthreads();
    const CandNegT<D> cst{tT, L.ns};
    const CandRows<D> cgl{w.emb + size_t(v0) * D};

    // 1. degrees (uncapped); with masks, a hit over k_max keeps only its
    //    k_max selected candidates in its mask (the masks then hold exactly
    //    the edges)
    if constexpr (CLUSTER) {
      if (masks) graph_masks<S, D>(cst, pl, P, r2, masks_s ? cluster.map_shared_rank(mask, 0) : mask, rank, ranks);
      // (without masks too: every block has read its ticket, so the first may write the
      // next one)
      cluster.sync();
    } else if (masks) {
      graph_masks<S, D>(cst, pl, P, r2, mask, 0, 1);
      __syncthreads();
    }
    if (rank > 0) continue;  // (the next ticket comes when the first block is done)
    if (masks) {
      for (int t = warp; t < pl.chunk[P - 1]; t += S::WARPS) {
        const int p = plane_of(pl.chunk, P, t);
        const int q0 = pl.po[p] + (t - pl.chunk[p]) * 32, q = q0 + lane;
        const int c0 = pl.po[p + 1], c1 = pl.po[min(p + 3, P)];
        int cnt = 0;
        if (q < c0) {
          for (int k = 0; k < pl.nw[p]; ++k) cnt += __popc(mask[mask_word(pl, p, q) + k]);
          deg[q] = cnt;
        }
        unsigned capped = __ballot_sync(kFull, cnt > k_max);
        while (capped) {
          const int qq = q0 + __ffs(capped) - 1;
          capped &= capped - 1;
          float qe[D];
          cst.row(qq, qe);
          select_capped<D>(cst, qe, c0, c1, mask_first(c0), r2, k_max, mask + mask_word(pl, p, qq));
        }
      }
    } else if (staged) {
      graph_degrees<S, D>(cst, pl, P, r2, deg);
    } else {
      graph_degrees<S, D>(cgl, pl, P, r2, deg);
    }
    for (int q = pl.po[P - 1] + tid; q < n; q += NT) deg[q] = 0;  // no candidates
    __syncthreads();

    // 2. offsets: event-local exclusive scan of min(deg, k_max), the event's
    //    count published
    const int total = block_scan<S>(deg, off, n, k_max, wsum);
    if (tid == 0) graph_publish(w.graph_desc, ev, total);
    L.edges<S, D>(total);
    const bool lists = masks && L.ints_all <= S::INTS && n <= 65535 && total <= 65535;
    uint16_t* tgt = reinterpret_cast<uint16_t*>(sm_i + L.targets);
    uint16_t* list = reinterpret_cast<uint16_t*>(sm_i + L.lists);
    uint16_t* srcs = reinterpret_cast<uint16_t*>(sm_i + L.sources);
    int32_t* start = sm_i + L.start;
    if (lists) {
      // 3. targets and in-degrees
      if (tid == 0) off[n] = total;
      for (int i = tid; i < n; i += NT) deg[i] = 0;
      __syncthreads();
      for (int t = warp; t < pl.chunk[P - 1]; t += S::WARPS) {
        const int p = plane_of(pl.chunk, P, t);
        const int q = pl.po[p] + (t - pl.chunk[p]) * 32 + lane;
        if (q >= pl.po[p + 1]) continue;
        int e = off[q];
        const int cA = mask_first(pl.po[p + 1]), w0 = mask_word(pl, p, q);
        for (int k = 0; k < pl.nw[p]; ++k) {
          unsigned m = mask[w0 + k];
          while (m) {
            const int c = cA + 32 * k + __ffs(m) - 1;
            m &= m - 1;
            tgt[e] = uint16_t(c);
            if (L.with_sources) srcs[e] = uint16_t(q);
            ++e;
            atomicAdd(&deg[c], 1);
          }
        }
      }
      __syncthreads();
      // 4. in-edge lists
      block_scan<S>(deg, start, n, 0x7fffffff, wsum);
      for (int i = tid; i < n; i += NT) deg[i] = start[i];
      __syncthreads();
      for (int k = tid; k < total; k += NT) list[atomicAdd(&deg[tgt[k]], 1)] = uint16_t(k);
      __syncthreads();  // deg[i]: the end of target i's list
    }

    // 5. the event's base, then the stores
    if (warp == 0) {
      const long long ex = graph_wait(w.graph_desc, ev, total, w.counters);
      if (lane == 0) base_s = ex;
    }
    __syncthreads();
    const long long base = base_s;
    for (int i = tid; i < n; i += NT) w.row_ptr[v0 + i] = clamp31(base + off[i]);
    if (ev == b.n_events - 1 && tid == 0) {
      const long long all = base + total;
      w.row_ptr[v1] = clamp31(all);
      w.counters[C_EDGES] = clamp31(all);
      if (all > w.e_cap || all > 0x7fffffffLL) set_status(w.counters, ST_CAPACITY);
    }
    const int e0 = int(base < w.e_cap ? base : w.e_cap);
    const int e1 = int(base + total < w.e_cap ? base + total : w.e_cap);
    const bool fits = base + total <= w.e_cap;
    if (lists) {
      for (int k = tid; k < total; k += NT) {
        if (!fits && base + k >= w.e_cap) break;
        int lo = 0;
        if (L.with_sources) {
          lo = srcs[k];
        } else {
          int hi = n;  // off[lo] <= k < off[hi]
          while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (off[mid] <= k)
              lo = mid;
            else
              hi = mid;
          }
        }
        const int c = tgt[k];
        float qe[D];
        cst.row(lo, qe);
        w.col[base + k] = v0 + c;
        w.src[base + k] = v0 + lo;
        w.d2[base + k] = cst.d2(qe, c);
      }
    } else if (masks) {
      graph_fill_masks<S, D>(w, cst, pl, P, off, mask, base, v0);
    } else if (staged) {
      graph_fill<S, D>(w, cst, pl, P, r2, k_max, deg, off, base, v0);
    } else {
      graph_fill<S, D>(w, cgl, pl, P, r2, k_max, deg, off, base, v0);
    }
    if (lists && fits) {
      for (int i = tid; i < total; i += NT) {
        const int k = list[i], t = tgt[k];
        const int lo = start[t], hi = deg[t];
        int rank = 0;
        for (int m = lo; m < hi; ++m) rank += list[m] < k;
        w.in_edge[e0 + lo + rank] = e0 + k;
      }
      for (int i = tid; i < n; i += NT) w.in_ptr[v0 + i] = e0 + start[i];
      if (tid == 0) w.in_ptr[v1] = e1;  // the next event writes the same value
    } else {  // (an event that overflows the workspace: its lists end there)
      __syncthreads();  // edges written; shared memory free
      csc_general<S>(w, n, v0, v1, e0, e1, sm_i, wsum);
    }
    __syncthreads();  // shared memory and ticket_s are reused by the next event
  }
}

int num_sms() {
  // queried once per process (thread-safe initialisation of a local static)
  static const int n = [] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 1;
  }();
  return n;
}

// Blocks per event: while the events leave SMs idle, clusters of 2, 4 or 8 blocks
// share an event's mask items (one event of 2146 hits in 8 dimensions: 112 of
// 215 thousand cycles in one block; 75 events of 1671 hits: 44 of 83 thousand).
// A block takes a whole SM, and clusters are placed within groups of SMs, so
// the lines leave room: 8 blocks up to 12 events, 4 up to 30, 2 up to 76.
template <class S, int D, bool CLUSTER>
void graph_shape(const Batch& b, const Ws& w, const GraphParams& g, int ranks, GraphWhen when, cudaStream_t s) {
  // set once per instantiation (thread-safe initialisation of a local static)
  static const bool attr = [] {
    cudaFuncSetAttribute(k_graph_event<S, D, CLUSTER>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         S::INTS * 4);
    return true;
  }();
  (void)attr;
  launch_pdl(true, k_graph_event<S, D, CLUSTER>, std::min(b.n_events, num_sms() * S::PER_SM) * ranks, S::NT,
             S::INTS * 4, s, ranks, b, w, g, when);
}

template <int D>
int graph_d(const Batch& b, const Ws& w, const GraphParams& g, cudaStream_t s) {
  const int sms = num_sms(), n = b.n_events;
  const int ranks = 12 * n <= sms ? 8 : 5 * n <= sms ? 4 : 2 * n <= sms ? 2 : 1;
  if (ranks > 1) {
    graph_shape<GraphWide, D, true>(b, w, g, ranks, G_ALWAYS, s);
    return 1;
  }
  const bool by_largest = by_largest_event(n, b.n_hits, sms);
  if (by_largest) graph_shape<GraphMid, D, false>(b, w, g, 1, G_ALL_SMALL, s);
  graph_shape<GraphWide, D, false>(b, w, g, 1, by_largest ? G_SOME_LARGE : G_ALWAYS, s);
  return by_largest ? 2 : 1;
}

// ---------------------------------------------------------------------------
// scan
// ---------------------------------------------------------------------------
__device__ __forceinline__ int block_exclusive_scan(int v, int* warp_s, int& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_s[warp] = x;
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    int t = lane < nw ? warp_s[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, t, o);
      if (lane >= o) t += y;
    }
    if (lane < nw) warp_s[lane] = t;
  }
  __syncthreads();
  total = warp_s[(blockDim.x >> 5) - 1];
  const int r = x - v + (warp > 0 ? warp_s[warp - 1] : 0);
  __syncthreads();
  return r;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const int32_t* in, int n,
                                                              int clamp_max, int32_t* blocks,
                                                              int32_t* counters, int total_slot,
                                                              int64_t cap) {
  __shared__ int warp_s[32];
  __shared__ int is_last;
  pdl_begin();
  if ((*(volatile int32_t*)&counters[C_STATUS]) & ST_INPUT) return;
  const int base = blockIdx.x * kScanChunk;
  int v = 0;
  for (int k = 0; k < kScanPer; ++k) {
    const int i = base + k * kScanThreads + threadIdx.x;
    if (i < n) v += min(in[i], clamp_max);
  }
  int total;
  block_exclusive_scan(v, warp_s, total);
  if (threadIdx.x == 0) {
    blocks[blockIdx.x] = total;
    __threadfence();
    const int t = atomicAdd(&counters[C_TICKET], 1);
    is_last = t == int(gridDim.x) - 1;
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  // the last block scans the block sums
  long long run = 0;
  for (int c = 0; c < int(gridDim.x); c += kScanThreads) {
    const int i = c + threadIdx.x;
    const int x = i < int(gridDim.x) ? ((volatile int32_t*)blocks)[i] : 0;
    int tot;
    const int ex = block_exclusive_scan(x, warp_s, tot);
    if (i < int(gridDim.x)) blocks[i] = int(run + ex);
    run += tot;
  }
  if (threadIdx.x == 0) {
    if (run > cap || run > 0x7fffffffLL) set_status(counters, ST_CAPACITY);
    counters[total_slot] = int(run > 0x7fffffffLL ? 0x7fffffffLL : run);
    counters[C_TICKET] = 0;
  }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_apply(const int32_t* in, int32_t* out,
                                                             int n, int clamp_max,
                                                             const int32_t* blocks,
                                                             const int32_t* counters,
                                                             int total_slot) {
  __shared__ int warp_s[32];
  pdl_begin();
  if ((*(volatile const int32_t*)&counters[C_STATUS]) & ST_INPUT) return;
  const int base = blockIdx.x * kScanChunk + threadIdx.x * kScanPer;
  int v[kScanPer];
  int sum = 0;
#pragma unroll
  for (int k = 0; k < kScanPer; ++k) {
    const int i = base + k;
    v[k] = i < n ? min(in[i], clamp_max) : 0;
    sum += v[k];
  }
  int total;
  int run = block_exclusive_scan(sum, warp_s, total) + blocks[blockIdx.x];
#pragma unroll
  for (int k = 0; k < kScanPer; ++k) {
    const int i = base + k;
    if (i < n) out[i] = run;
    run += v[k];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[n] = counters[total_slot];
}


}  // namespace

void launch_sort(const Batch& b, const Ws& w, const int64_t* offsets, int n_planes, cudaStream_t s) {
  if (b.n_events <= 0) return;
  launch_pdl(true, k_sort, b.n_events, kSortThreads, 0, s, 1, b, w, offsets, n_planes);
}

void launch_scan(const int32_t* in, int32_t* out, int n, int clamp_max, int32_t* counters,
                 int total_slot, int64_t cap, int32_t* blocks, cudaStream_t s) {
  const int nb = div_up(n > 0 ? n : 1, kScanChunk);
  launch_pdl(false, k_scan_reduce, nb, kScanThreads, 0, s, 1, in, n, clamp_max, blocks, counters,
             total_slot, cap);
  launch_pdl(false, k_scan_apply, nb, kScanThreads, 0, s, 1, in, out, n, clamp_max, blocks, counters,
             total_slot);
}

int launch_graph(const Batch& b, const Ws& w, const GraphParams& g, int D, cudaStream_t s) {
  if (b.n_events <= 0) return 0;
  switch (D) {
    case 1: return graph_d<1>(b, w, g, s);
    case 2: return graph_d<2>(b, w, g, s);
    case 3: return graph_d<3>(b, w, g, s);
    case 4: return graph_d<4>(b, w, g, s);
    case 5: return graph_d<5>(b, w, g, s);
    case 6: return graph_d<6>(b, w, g, s);
    case 7: return graph_d<7>(b, w, g, s);
    case 8: return graph_d<8>(b, w, g, s);
    case 16: return graph_d<16>(b, w, g, s);
    default: return 0;
  }
}

int device_sms() { return num_sms(); }

}  // namespace gnntrk
