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

// Every lane of a warp: the K largest entries of row r over nsv lists of
// kTopMax entries each, sorted by value descending, then id ascending (list s
// at (s ld + r) kTopMax of tv, ti).  Lane j < K ends with the j-th entry and
// the place `at` it came from.  Beyond a batch of lists, those that cannot
// contribute go first: each lane takes the best head of every 32nd list, K
// entries reach the K-th best of those 32, and a list whose head does not is
// left out.  The half warps take every other list of the rest: a list comes in
// reversed, the better of each pair of entries are the 16 best of both, and four
// exchanges sort them; a batch's loads are in flight together.  (The best of the
// lists' heads taken K times over the warp, five exchanges and a dependent load
// each, cost as much for one list as for 64: the top-16 call took 650 us for
// 131072 rows, d = 64, V = 512, and takes 284; all of 160 lists taken in cost a
// top-1 call of 60 rows 40 us.  One thread a row, inserting up to 64 lists of 16
// one entry after the other, took 294 there and 130 us of its own for 2048 rows.)
__device__ __forceinline__ void warp_top_merge(const float* __restrict__ tv,
                                               const int32_t* __restrict__ ti, int nsv, size_t ld,
                                               int r, int K, int lane, float& v_out, int& i_out,
                                               size_t& at_out) {
  constexpr int kAhead = 4;  // lists a half warp loads at a time
  const int half = lane >> 4, sub = lane & 15;
  auto place = [&](int s) { return (static_cast<size_t>(s) * ld + r) * kTopMax; };
  int group = 0;       // of 32 lists
  unsigned left = 0u;  // those of the group still to take
  float bound = -INFINITY;
  if (nsv <= 2 * kAhead) {
    left = (1u << nsv) - 1u;
  } else {
    float head = -INFINITY;
    for (int s = lane; s < nsv; s += 32) head = fmaxf(head, __ldg(tv + place(s)));
    int rank = 0;
#pragma unroll
    for (int q = 0; q < 32; ++q) {
      const float o = __shfl_sync(0xffffffffu, head, q);
      rank += o > head || (o == head && q < lane);
    }
    bound = __shfl_sync(0xffffffffu, head, __ffs(__ballot_sync(0xffffffffu, rank == K - 1)) - 1);
    group = -1;
  }
  // the next list (the same in every lane), -1 after the last
  auto next = [&]() -> int {
    while (!left) {
      if (32 * (group + 1) >= nsv) return -1;
      ++group;
      const int s = 32 * group + lane;
      left = __ballot_sync(0xffffffffu, s < nsv && __ldg(tv + place(s)) >= bound);
    }
    const int s = 32 * group + __ffs(left) - 1;
    left &= left - 1u;
    return s;
  };
  TopEntry e{-INFINITY, INT_MAX, 0};
  for (bool more = true; more;) {
    int list[kAhead], id[kAhead];
    float v[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int s0 = next(), s1 = next();
      more = s1 >= 0;
      list[u] = half ? s1 : s0;
      const size_t o = place(list[u]) + (kTopMax - 1 - sub);
      v[u] = list[u] >= 0 ? __ldg(tv + o) : -INFINITY;
      id[u] = list[u] >= 0 ? __ldg(ti + o) : INT_MAX;
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const bool in = top_before(v[u], id[u], e.v, e.id);
      if (!__any_sync(0xffffffffu, in)) continue;
      if (in) e = TopEntry{v[u], id[u], list[u] * kTopMax + kTopMax - 1 - sub};
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
