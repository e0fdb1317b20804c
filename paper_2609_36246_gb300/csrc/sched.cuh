// sched.cuh -- device-side work decomposition shared by the kernels that
// reduce a row over vocabulary tiles (forward log-sum-exp, divergence).
//
// The row count N_mask lives on the device, so every CTA (and the finalize
// kernels) derive the same decomposition from it: rt row tiles of 128 rows,
// vt vocabulary tiles, split into sv contiguous segments of seg tiles.  A
// unit is one (row tile, segment); its partial (max, sum) per row is merged by
// the finalize kernel.  sv is chosen to minimise the critical path
// ceil(units / ctas) * seg, which removes most of the wave-quantisation loss
// when rt is small compared with the SM count.  One or two row tiles may be cut
// into more than kSvMax segments, as many as fill the SMs: with 64, 96 rows of
// d = 4096 ran on 60 SMs (276 us over V = 151936).
#pragma once

#include <climits>
#include <cuda_bf16.h>

#include "internal.h"

namespace olive {

struct Split {
  int n;     // valid rows
  int rt;    // row tiles
  int vt;    // vocabulary tiles
  int sv;    // segments
  int seg;   // tiles per segment
  int units; // rt * sv
};

// Segments a row tile may be cut into when there are rt of them; `parts` is
// the least number of (row tile, segment) partials the workspace holds.
__device__ inline int split_cap(int rt, int parts) {
  return rt > 0 ? max(kSvMax, parts / rt) : kSvMax;
}

// Every lane of a warp: the decomposition of n rows over vt vocabulary tiles
// for `ctas` CTAs, at most sv_cap segments (a lane tries every 32nd count; on
// one thread the search took several microseconds of each kernel that needs
// it).
__device__ inline Split choose_split(int n, int vt, int ctas, int sv_cap) {
  Split s;
  s.n = n;
  s.rt = (n + 127) / 128;
  s.vt = vt;
  int best_sv = 1;
  long long best_cost = LLONG_MAX;
  const int max_sv = min(vt, sv_cap);
  for (int sv = static_cast<int>(threadIdx.x & 31) + 1; sv <= max_sv; sv += 32) {
    const int seg = (vt + sv - 1) / sv;
    if ((vt + seg - 1) / seg != sv) continue;
    const uint32_t units = static_cast<uint32_t>(s.rt) * static_cast<uint32_t>(sv);
    const uint32_t waves = (units + static_cast<uint32_t>(ctas) - 1) / static_cast<uint32_t>(ctas);
    // a unit also pays a pipeline fill and a partial write: ~1/8 tile
    const long long cost = static_cast<long long>(waves) * (8LL * seg + 1);
    if (cost < best_cost) {
      best_cost = cost;
      best_sv = sv;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const long long c = __shfl_xor_sync(0xffffffffu, best_cost, o);
    const int v = __shfl_xor_sync(0xffffffffu, best_sv, o);
    if (c < best_cost || (c == best_cost && v < best_sv)) {
      best_cost = c;
      best_sv = v;
    }
  }
  s.sv = best_sv;
  s.seg = (vt + best_sv - 1) / best_sv;
  s.units = s.rt * s.sv;
  return s;
}

// Slabs of the G buffer: n masked rows are cut into n_slabs equal slabs of
// at most tc rows (rps rows each, a multiple of 128); slab s covers compacted
// rows [row0, row0 + in_s).  Shared by every kernel that works on one slab.
struct SlabPlan {
  int n_slabs, rps;
  __host__ __device__ SlabPlan(int n, int tc) {
    n_slabs = n > 0 ? (n + tc - 1) / tc : 1;
    const int per = (n + n_slabs - 1) / n_slabs;
    rps = (per + 127) / 128 * 128;
  }
  __host__ __device__ int rows_in(int n, int s) const {
    const int r = n - s * rps;
    return r < 0 ? 0 : (r > rps ? rps : r);
  }
};

__device__ inline int read_n_rows(const int32_t* n_rows, int T, int32_t* dev_status) {
  int n = *n_rows;
  if (n < 0 || n > T) {
    if (dev_status) atomicOr(dev_status, 1 << OLIVE_ERR_OFFSETS);
    n = n < 0 ? 0 : T;
  }
  return n;
}

// Rows beyond which a merge of the sweeps' partials gives a row no more lanes than
// it has segments (merge_lanes): a warp a row is quicker at few rows, which are
// cut into many segments, and its code is shorter.
constexpr int kManyRows = 1024;
// Lanes of a warp that share a row's sv segments: a power of two, one segment
// each where 32 are enough.
__device__ __forceinline__ int merge_lanes(int sv) {
  int l = 1;
  while (l < sv && l < 32) l *= 2;
  return l;
}

// (m, s) + (m2, s2): a base-2 maximum and the sum of 2^(x - m); an empty side
// (m = -inf) adds nothing.  w receives the factors applied to each side.
__device__ __forceinline__ void merge_ms(float& m, float& s, float m2, float s2, float* w = nullptr) {
  const float mn = fmaxf(m, m2);
  const float f1 = m == -INFINITY ? 0.f : exp2f(m - mn);
  const float f2 = m2 == -INFINITY ? 0.f : exp2f(m2 - mn);
  s = s * f1 + s2 * f2;
  m = mn;
  if (w) {
    w[0] = f1;
    w[1] = f2;
  }
}

}  // namespace olive
