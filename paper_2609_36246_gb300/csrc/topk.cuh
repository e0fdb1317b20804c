// topk.cuh -- fixed-length top lists kept in registers by the sweeps that
// report each row's K largest logits (K <= 16).
#pragma once

namespace olive {

constexpr int kTopMax = 16;  // list length kept per row

// Inserts (cv, ci) into a list sorted by value descending, then id ascending;
// the last entry falls off.  For a sweep that visits ids in ascending order
// within the list's lifetime: the new id is larger than every id already
// listed, so among equal values it belongs last, and the value alone decides
// its place (no id comparisons).
__device__ __forceinline__ void topk_insert_asc(float (&tv)[kTopMax], int (&ti)[kTopMax], float cv,
                                                int ci) {
#pragma unroll
  for (int j = 0; j < kTopMax; ++j) {
    const bool before = cv > tv[j];
    const float v = tv[j];
    const int i = ti[j];
    tv[j] = before ? cv : v;
    ti[j] = before ? ci : i;
    cv = before ? v : cv;
    ci = before ? i : ci;
  }
}

// The same with a payload value carried along with each entry.
__device__ __forceinline__ void topk_insert3_asc(float (&tv)[kTopMax], int (&ti)[kTopMax],
                                                 float (&tx)[kTopMax], float cv, int ci, float cx) {
#pragma unroll
  for (int j = 0; j < kTopMax; ++j) {
    const bool before = cv > tv[j];
    const float v = tv[j];
    const int i = ti[j];
    const float x = tx[j];
    tv[j] = before ? cv : v;
    ti[j] = before ? ci : i;
    tx[j] = before ? cx : x;
    cv = before ? v : cv;
    ci = before ? i : ci;
    cx = before ? x : cx;
  }
}

// Every lane of a warp: the K largest entries of row r over nsv lists of
// kTopMax entries each, sorted by value descending, then id ascending (list s
// at (s ld + r) kTopMax of tv, ti).  Lane j < K ends with the j-th entry and
// the place `at` it came from.  A lane keeps the best head of every 32nd list;
// the warp takes the best of the 32 heads K times, and only the lane it came
// from looks at its lists again.  (One thread a row inserted up to 64 lists of
// 16 one entry after the other: 130 us for 2048 rows, 296 us for 2900 rows of
// the OPD sweep's two lists.)
__device__ __forceinline__ void warp_top_merge(const float* __restrict__ tv,
                                               const int32_t* __restrict__ ti, int nsv, size_t ld,
                                               int r, int K, int lane, float& v_out, int& i_out,
                                               size_t& at_out) {
  uint64_t heads = 0;  // entries taken from each of this lane's lists, 5 bits each (at most 10 lists)
  float v;
  int id, list;
  size_t at;
  auto look = [&]() {
    v = -INFINITY;
    id = INT_MAX;
    at = 0;
    list = 0;
    for (int s = lane, q = 0; s < nsv; s += 32, ++q) {
      const int h = static_cast<int>(heads >> (5 * q)) & 31;
      if (h >= kTopMax) continue;
      const size_t o = (static_cast<size_t>(s) * ld + r) * kTopMax + h;
      const float cv = __ldg(tv + o);
      const int ci = __ldg(ti + o);
      if (cv > v || (cv == v && ci < id)) {
        v = cv;
        id = ci;
        at = o;
        list = q;
      }
    }
  };
  look();
  v_out = -INFINITY;
  i_out = INT_MAX;
  at_out = 0;
  for (int j = 0; j < K; ++j) {
    float bv = v;
    int bi = id, bl = lane;
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      const int ol = __shfl_xor_sync(0xffffffffu, bl, o);
      if (ov > bv || (ov == bv && (oi < bi || (oi == bi && ol < bl)))) {
        bv = ov;
        bi = oi;
        bl = ol;
      }
    }
    const unsigned long long ba = __shfl_sync(0xffffffffu, static_cast<unsigned long long>(at), bl);
    if (lane == j) {
      v_out = bv;
      i_out = bi;
      at_out = static_cast<size_t>(ba);
    }
    if (lane == bl && id != INT_MAX) {
      heads += 1ull << (5 * list);
      look();
    }
    __syncwarp();
  }
}

}  // namespace olive
