// topk.cuh -- fixed-length top lists kept in registers by the sweeps that
// report each row's K largest logits (K <= 16).
#pragma once

namespace olive {

constexpr int kTopMax = 16;  // list length kept per row

// Inserts (cv, ci) into a list sorted by value descending, then id ascending;
// the last entry falls off.  For a sweep that visits ids in ascending order
// within the list's lifetime: the new id is larger than every id already
// listed, so among equal values it belongs last, and the value alone decides
// its place (no id comparisons).  Every entry below that place moves by one:
// all are compared with the new value, and none with its neighbour, which an
// equal value would let past.
__device__ __forceinline__ void topk_insert_asc(float (&tv)[kTopMax], int (&ti)[kTopMax], float cv,
                                                int ci) {
#pragma unroll
  for (int j = kTopMax - 1; j > 0; --j) {
    const bool at = cv > tv[j], above = cv > tv[j - 1];
    ti[j] = above ? ti[j - 1] : at ? ci : ti[j];
    tv[j] = above ? tv[j - 1] : at ? cv : tv[j];
  }
  if (cv > tv[0]) {
    tv[0] = cv;
    ti[0] = ci;
  }
}

// The same with a payload value carried along with each entry.
__device__ __forceinline__ void topk_insert3_asc(float (&tv)[kTopMax], int (&ti)[kTopMax],
                                                 float (&tx)[kTopMax], float cv, int ci, float cx) {
#pragma unroll
  for (int j = kTopMax - 1; j > 0; --j) {
    const bool at = cv > tv[j], above = cv > tv[j - 1];
    tx[j] = above ? tx[j - 1] : at ? cx : tx[j];
    ti[j] = above ? ti[j - 1] : at ? ci : ti[j];
    tv[j] = above ? tv[j - 1] : at ? cv : tv[j];
  }
  if (cv > tv[0]) {
    tv[0] = cv;
    ti[0] = ci;
    tx[0] = cx;
  }
}

// An entry of a sorted list of 16 that a half warp holds, entry j in its lane j:
// value, id, and where it came from (list * 16 + entry).
struct TopEntry {
  float v;
  int id, from;
};
__device__ __forceinline__ bool top_before(float av, int ai, float bv, int bi) {
  return av > bv || (av == bv && ai < bi);
}
// Sorts a bitonic sequence of 16 (the larger halves of two sorted lists, one of
// them reversed), best first, in every half warp.
__device__ __forceinline__ void top_sort16(TopEntry& e, int lane) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    const float v = __shfl_xor_sync(0xffffffffu, e.v, o);
    const int id = __shfl_xor_sync(0xffffffffu, e.id, o);
    const int from = __shfl_xor_sync(0xffffffffu, e.from, o);
    if (lane & o ? top_before(e.v, e.id, v, id) : top_before(v, id, e.v, e.id)) e = TopEntry{v, id, from};
  }
}

// Every lane of a warp: the 16 largest entries of row r over nsv lists of
// kTopMax entries each, sorted by value descending, then id ascending (list s
// at (s ld + r) kTopMax of tv, ti).  Lane j < 16 ends with the j-th entry and
// the place `at` it came from.  The half warps take every other list: a list
// comes in reversed, the better of each pair of entries are the 16 best of both,
// four exchanges sort them, and a list of which no entry gets in costs its two
// loads and one vote; eight lists' loads are in flight.  (The best of the
// lists' heads taken 16 times over the warp, five exchanges and a dependent load
// each, cost as much for one list as for 64: the top-16 call took 650 us for
// 131072 rows, d = 64, V = 512, and takes 278.  One thread a row, inserting up to
// 64 lists of 16 one entry after the other, took 294 there and 130 us of its own
// for 2048 rows.)
__device__ __forceinline__ void warp_top_merge(const float* __restrict__ tv,
                                               const int32_t* __restrict__ ti, int nsv, size_t ld,
                                               int r, int lane, float& v_out, int& i_out,
                                               size_t& at_out) {
  constexpr int kAhead = 4;  // lists a half warp loads at a time
  const int half = lane >> 4, sub = lane & 15;
  TopEntry e{-INFINITY, INT_MAX, 0};
  for (int s0 = 0; s0 < nsv; s0 += 2 * kAhead) {
    float v[kAhead];
    int id[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int s = s0 + 2 * u + half;
      const size_t o = (static_cast<size_t>(s) * ld + r) * kTopMax + (kTopMax - 1 - sub);
      v[u] = s < nsv ? __ldg(tv + o) : -INFINITY;
      id[u] = s < nsv ? __ldg(ti + o) : INT_MAX;
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const bool in = top_before(v[u], id[u], e.v, e.id);
      if (!__any_sync(0xffffffffu, in)) continue;
      if (in) e = TopEntry{v[u], id[u], (s0 + 2 * u + half) * kTopMax + kTopMax - 1 - sub};
      top_sort16(e, lane);
    }
  }
  if (nsv > 1) {  // the two halves' lists: the other one's, reversed
    const float v = __shfl_xor_sync(0xffffffffu, e.v, 31);
    const int id = __shfl_xor_sync(0xffffffffu, e.id, 31);
    const int from = __shfl_xor_sync(0xffffffffu, e.from, 31);
    if (top_before(v, id, e.v, e.id)) e = TopEntry{v, id, from};
    top_sort16(e, lane);
  }
  v_out = e.v;
  i_out = e.id;
  at_out = (static_cast<size_t>(e.from / kTopMax) * ld + r) * kTopMax + e.from % kTopMax;
}

}  // namespace olive
