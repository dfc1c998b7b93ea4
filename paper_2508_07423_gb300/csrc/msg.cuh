// Messages of a node step, m_v = [sum of e over v's out edges, sum over its in
// edges]: each sum in increasing list order starting from zero, FP32, whatever
// the type of the edge rows.
//
// A group of LANES lanes sums one hit, 16 bytes of a row per lane. What bounds it
// is the latency of a hit's chain of loads: list bounds -> in-edge ids -> rows,
// once per list before. The chain is spread over the group's loop: while the
// rows of one hit are in flight (up to U of a list at a time), the ids of the
// next hit, the bounds of the one after it and the row id of the third are,
// too, so that a list waits for its rows only. Rows past a list's end are not
// loaded.
//
// Four launches of a call, before -> now (32 warps per SM, U = 4): BF16, 1.68 M
// hits with 1.9 edges each 657 -> 481 us, 0.87 M hits at hidden 128 with 2.1 edges
// 1524 -> 1180 us, 1.68 M hits with 6.0 edges 1210 -> 1182 us (3.9 TB/s of
// rows); FP32, 0.67 M hits with 6.0 edges 785 -> 736 us, 0.22 M hits at hidden 64
// with 8.0 edges (8 launches) 1475 -> 1107 us. Both lists' rows in flight
// together (80 registers, 24 warps) measured 592, 1292, 1531, 960 and 1359 us; U =
// 8 at the same registers 740, 1564, 1392, 864 and 1311 us. HBM is not the limit: 33 %
// (BF16, hidden 32), 40 % (FP8, 128) and 42 % (FP32, 32) of its rate; the stalls are
// waits for loads, 45-47 % of the warps active.
#pragma once

#include "internal.cuh"

namespace gnntrk {

// R: LANES, Chunk (16 bytes), Acc (add(chunk), finish() by the whole warp); load(w, edge, q), store(w, row,
// side, q, acc)
template <class R>
__device__ __forceinline__ void message_sums(const Ws& w, Sel sel, int lo, int hi) {
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int L = R::LANES, U = 4, NI = (U + L - 1) / L;
  const int E = clamp_edges(w.counters, w.e_cap);
  const int lane = threadIdx.x & 31, q = lane % L, g0 = lane - q;
  const int groups = gridDim.x * (blockDim.x / L);
  auto row_at = [&](int pos) { return pos < hi ? sel_row(sel, pos) : -1; };
  // lane 0, 1 of a group: the out list's bounds; lane 2, 3: the in list's
  auto bounds = [&](int row) {
    if (row < 0 || q >= 4) return 0;
    return q < 2 ? min(w.row_ptr[row + q], E) : w.in_ptr[row + q - 2];
  };
  // lane q: in-edge ids q, q + L, ... of the first U
  auto ids = [&](int bnd, int (&id)[NI]) {
    const int a = __shfl_sync(kAll, bnd, g0 + 2), n = __shfl_sync(kAll, bnd, g0 + 3) - a;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int k = q + L * i;
      id[i] = k < U && k < n ? w.in_edge[a + k] : 0;
    }
  };
  int pos = lo + blockIdx.x * (blockDim.x / L) + threadIdx.x / L;
  int row = row_at(pos), row1 = row_at(pos + groups), row2 = row_at(pos + 2 * groups);
  int bnd = bounds(row), bnd1 = bounds(row1);
  int id[NI];
  ids(bnd, id);
  // (warp-uniform: the warp's first group has its smallest position)
  for (int first = pos - g0 / L; first < hi; first += groups, pos += groups) {
    const int oa = __shfl_sync(kAll, bnd, g0), on = __shfl_sync(kAll, bnd, g0 + 1) - oa;
    const int ia = __shfl_sync(kAll, bnd, g0 + 2), in = __shfl_sync(kAll, bnd, g0 + 3) - ia;
    typename R::Chunk v[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (u < on) v[u] = R::load(w, oa + u, q);
    int id1[NI];
    ids(bnd1, id1);
    const int bnd2 = bounds(row2), row3 = row_at(pos + 3 * groups);
    typename R::Acc s;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (u < on) s.add(v[u]);
    for (int t = U; t < on; t += U) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (t + u < on) v[u] = R::load(w, oa + t + u, q);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (t + u < on) s.add(v[u]);
    }
    s.finish();
    if (row >= 0) R::store(w, row, 0, q, s);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = __shfl_sync(kAll, id[u / L], g0 + u % L);
      if (u < in) v[u] = R::load(w, e, q);
    }
    s = typename R::Acc();
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (u < in) s.add(v[u]);
    for (int t = U; t < in; t += U) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (t + u < in) v[u] = R::load(w, w.in_edge[ia + t + u], q);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (t + u < in) s.add(v[u]);
    }
    s.finish();
    if (row >= 0) R::store(w, row, 1, q, s);
    row = row1;
    row1 = row2;
    row2 = row3;
    bnd = bnd1;
    bnd1 = bnd2;
#pragma unroll
    for (int i = 0; i < NI; ++i) id[i] = id1[i];
  }
}

}  // namespace gnntrk
