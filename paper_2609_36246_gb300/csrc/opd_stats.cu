// opd_stats.cu -- OPD's per-token quantities from one sweep over the
// vocabulary with both LM heads (Section 1: OPD scores each student token
// against the teacher; Appendix A, Table opd-config: top-16 log-probs;
// Section 4.1: the top-K overlap ratio).  Per masked row t:
//   kl[t]            full-vocabulary KL (reverse or forward, as
//                    olive_token_divergence)
//   s_lse, t_lse     log-sum-exp of both heads
//   s_entropy        -sum_v p_s log p_s
//   s_topk_*         the student's K most probable tokens and their log-probs
//   t_logp_s[t, j]   the teacher's log-prob at the student's j-th token
//   overlap[t]       |top_K(p_s) intersect top_K(p_t)| / K
//   kl_topk[t]       sum_j p_s(v_j) (log p_s(v_j) - log p_t(v_j)), the top-K
//                    truncated reverse KL
// Every 128 x 256 tile runs the student and teacher products into the two
// halves of one 512-column TMEM accumulator (as the divergence forward), so
// the epilogue cannot overlap the next tile's MMAs.  What of it needs the
// student's logits alone (maximum, sum, entropy, top list) therefore runs while
// the teacher's MMAs do (first()), and what is left (the teacher's sum and
// list, the KL sum, the teacher logits of new student entries) hands the
// accumulator back once its last 32 columns are in registers: 5.70 -> 5.43 ms
// for a call of 2900 rows, d_s = 4096, d_t = 5120, V = 151936, whose
// operations take 4.22 ms at the peak rate.  Eight epilogue warps shorten
// the rest: the two warps of a TMEM lane quadrant take the two 128-column
// halves of every tile.  Each epilogue thread owns a (row, half) and keeps, in
// base-2 units x = z inv_tau log2 e, the online (m_s, s_s, E_s = sum e_s x_s,
// m_t, s_t, A) and two 16-entry top lists of raw logits (the student's carries
// the teacher logit of each entry).
// Per 32-column chunk each thread first marks, in a 32-bit mask per list, the
// columns that beat the list's last entry (after the first tiles of a segment
// few do), then walks the mask in a rolled loop: the value is picked from the
// chunk's registers by a 5-level select tree and the insertion network runs
// once per candidate, so the network exists in one copy (a copy per column
// overflows the instruction cache).  Each half writes its own partial, as
// segment 2 sg + half of the row's vocabulary segment sg; opd_finalize_kernel
// merges them, one warp a row.
#include <algorithm>
#include <climits>
#include <cmath>

#include "gemm_core.cuh"
#include "sched.cuh"
#include "topk.cuh"

namespace olive {
namespace {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

// a[k] for a lane-varying k in [0, 32) without local memory: a select tree
__device__ __forceinline__ uint32_t pick32(const uint32_t (&a)[32], int k) {
  uint32_t l0[16], l1[8], l2[4], l3[2];
#pragma unroll
  for (int i = 0; i < 16; ++i) l0[i] = (k & 1) ? a[2 * i + 1] : a[2 * i];
#pragma unroll
  for (int i = 0; i < 8; ++i) l1[i] = (k & 2) ? l0[2 * i + 1] : l0[2 * i];
#pragma unroll
  for (int i = 0; i < 4; ++i) l2[i] = (k & 4) ? l1[2 * i + 1] : l1[2 * i];
#pragma unroll
  for (int i = 0; i < 2; ++i) l3[i] = (k & 8) ? l2[2 * i + 1] : l2[2 * i];
  return (k & 16) ? l3[1] : l3[0];
}

struct OpdKern {
  static constexpr int kBN = 256;
  static constexpr bool kAMn = false;
  static constexpr bool kBMn = false;
  static constexpr bool kDual = true;
  static constexpr bool kFirst = true;
  static constexpr int kStages = 4;
  static constexpr int kAccBufs = 1;
  static constexpr int kEpiWarps = 8;
  // each (row, half)'s 16th values so far and the unit they belong to
  // and, per thread, the tile's student candidates, a word a chunk
  static constexpr int kEpiSmem = 2 * 2 * 128 * 8 + 4 * 256 * 4;
  // segments per row tile (each writes two halves)
  static __device__ int seg_cap(int n) { return split_cap((n + 127) / 128, kMinPartsOpd) / 2; }

  struct Params {
    int32_t* dev_status;
    uint64_t wait_limit_ns;
    const int32_t* n_rows;
    int32_t T, V, d_s, d_t;
    int32_t ctas, group_rows, reverse;
    float scale2;
    size_t plane;      // floats of one of the partial arrays
    float* part;       // [6][plane], [2 segment + half][rt 128] each: m_s, s_s, E_s, m_t, s_t, A
    float* part_sv;    // [2 segment + half][rt 128][16] student top raw logits
    int32_t* part_si;  // their ids
    float* part_sx;    // the teacher's raw logits at those ids
    float* part_tv;    // teacher top raw logits
    int32_t* part_ti;  // their ids
  };
  struct Sched {
    Split sp;
  };
  static __device__ Sched make_sched(const Params& p) {
    Sched s;
    const int n = read_n_rows(p.n_rows, p.T, p.dev_status);
    s.sp = choose_split(n, (p.V + kBN - 1) / kBN, p.ctas, seg_cap(n));
    return s;
  }
  static __device__ int num_units(const Params&, const Sched& s) { return s.sp.units; }
  static __device__ void unit_pos(const Params& p, const Sched& s, int u, int& i, int& sg) {
    const Raster r{s.sp.rt, s.sp.sv, p.group_rows};
    r.tile(u, i, sg);
  }
  static __device__ int unit_len(const Params& p, const Sched& s, int u) {
    int i, sg;
    unit_pos(p, s, u, i, sg);
    return min(s.sp.seg, s.sp.vt - sg * s.sp.seg);
  }
  static __device__ TileC tile(const Params& p, const Sched& s, int u, int t) {
    int i, sg;
    unit_pos(p, s, u, i, sg);
    TileC c;
    c.m0 = i * kBM;
    c.n0 = (sg * s.sp.seg + t) * kBN;
    c.ka0 = 0;
    c.kb0 = 0;
    c.nk = (p.d_s + kBK - 1) / kBK;
    c.nk2 = (p.d_t + kBK - 1) / kBK;
    return c;
  }

  struct Epi {
    int r, sg, half, unit;
    // shared by the epilogue threads: the student lists' and the teacher lists'
    // bounds [half][row][2], value bits and unit number in one 64-bit word, then
    // the candidate words [4][thread]
    uint8_t* shared;
    float bound_s, bound_t;
    float ms, ss, es, mt, st, A;
    float sv[kTopMax], sx[kTopMax], tv[kTopMax];
    int si[kTopMax], ti[kTopMax];

    __device__ void init(uint8_t* smem, int prt) {
      half = prt;
      shared = smem;
      bound(half, 0) = bound(half, 1) = ~0ull;
    }
    __device__ void begin(const Params& p, const Sched& s, int u, int row) {
      int i;
      unit_pos(p, s, u, i, sg);
      unit = u;
      bound_s = bound_t = -INFINITY;
      r = i * kBM + row;
      ms = mt = -INFINITY;
      ss = es = st = A = 0.f;
#pragma unroll
      for (int j = 0; j < kTopMax; ++j) {
        sv[j] = tv[j] = sx[j] = -INFINITY;
        si[j] = ti[j] = INT_MAX;
      }
    }

    __device__ __forceinline__ volatile unsigned long long& bound(int h, int list) const {
      return reinterpret_cast<volatile unsigned long long*>(shared)[256 * h + 2 * (threadIdx.x & 127) + list];
    }
    __device__ __forceinline__ volatile uint32_t& fresh(int chunk) const {
      return reinterpret_cast<volatile uint32_t*>(shared)[1024 + 256 * chunk + threadIdx.x];
    }

    // columns of v that beat both the list's last entry and the halves' bound
    template <bool kFull>
    static __device__ __forceinline__ uint32_t candidates(const uint32_t (&v)[32], int nvalid, float top,
                                                          float last, float bound) {
      uint32_t cand = 0u;
      // a unit visits its ids in ascending order, so a new id is larger than
      // every listed one: values alone decide the candidates and their places
      if (top > last && top >= bound) {
#pragma unroll
        for (int k = 0; k < 32; ++k) {
          const float x = __uint_as_float(v[k]);
          if ((kFull || k < nvalid) && x > last && x >= bound) cand |= 1u << k;
        }
      }
      return cand;
    }

    // Student's half of a 32-column chunk: sum and entropy numerator; returns
    // the candidates.  kFull: all 32 columns are below V.
    template <bool kFull>
    __device__ __forceinline__ uint32_t chunk_s(const Params& p, const uint32_t (&a)[32], int col0) {
      const int nvalid = kFull ? 32 : p.V - col0;
      // raw maximum (the scale is positive), then one fma an exponent
      float cs = -INFINITY;
#pragma unroll
      for (int k = 0; k < 32; ++k)
        if (k < nvalid) cs = fmaxf(cs, __uint_as_float(a[k]));
      const float msn = fmaxf(ms, cs * p.scale2);
      float e_s = 0.f, e_e = 0.f;
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        const bool ok = k < nvalid;
        const float zs = __uint_as_float(a[k]);
        const float qs = ok ? fast_exp2(fmaf(zs, p.scale2, -msn)) : 0.f;
        e_s += qs;
        e_e = ok ? fmaf(qs, zs, e_e) : e_e;
      }
      const float rs = fast_exp2(ms - msn);
      ss = ss * rs + e_s;
      es = es * rs + e_e * p.scale2;
      ms = msn;
      return candidates<kFull>(a, nvalid, cs, sv[kTopMax - 1], bound_s);
    }

    // Teacher's half: sum and A (the student's maximum is this tile's already)
    template <bool kFull>
    __device__ __forceinline__ uint32_t chunk_t(const Params& p, const uint32_t (&a)[32],
                                                const uint32_t (&b)[32], int col0) {
      const int nvalid = kFull ? 32 : p.V - col0;
      float ct = -INFINITY;
#pragma unroll
      for (int k = 0; k < 32; ++k)
        if (k < nvalid) ct = fmaxf(ct, __uint_as_float(b[k]));
      const float mtn = fmaxf(mt, ct * p.scale2);
      float e_t = 0.f, e_a = 0.f;
      if (p.reverse) {
#pragma unroll
        for (int k = 0; k < 32; ++k) {
          const bool ok = k < nvalid;
          const float zs = __uint_as_float(a[k]), zt = __uint_as_float(b[k]);
          const float qs = ok ? fast_exp2(fmaf(zs, p.scale2, -ms)) : 0.f;
          e_t += ok ? fast_exp2(fmaf(zt, p.scale2, -mtn)) : 0.f;
          e_a = ok ? fmaf(qs, zs - zt, e_a) : e_a;
        }
      } else {
#pragma unroll
        for (int k = 0; k < 32; ++k) {
          const bool ok = k < nvalid;
          const float zs = __uint_as_float(a[k]), zt = __uint_as_float(b[k]);
          const float qt = ok ? fast_exp2(fmaf(zt, p.scale2, -mtn)) : 0.f;
          e_t += qt;
          e_a = ok ? fmaf(-qt, zs - zt, e_a) : e_a;
        }
      }
      const float rt = fast_exp2(mt - mtn);
      st = st * rt + e_t;
      A = A * (p.reverse ? 1.f : rt) + e_a * p.scale2;
      mt = mtn;
      return candidates<kFull>(b, nvalid, ct, tv[kTopMax - 1], bound_t);
    }

    // The student's part of a tile, while the teacher's MMAs run.  New list
    // entries get their teacher logits in tile(), which finds them by the
    // masks in `fresh`.
    __device__ void first(const Params& p, const TileC& tc, uint32_t taddr) {
      // The other half of the row lists 16 logits no smaller than its 16th, so
      // what is below that cannot be among the row's 16 largest: fewer
      // insertions, which are what this epilogue spends most of its time on.
      // (The two halves are not in step: a bound counts only if it carries this
      // unit's number, and a stale one is merely lower.)
      const unsigned long long ps = bound(1 - half, 0);
      if (ps >> 32 == static_cast<uint32_t>(unit)) bound_s = __uint_as_float(static_cast<uint32_t>(ps));
      const int lo = half * (kBN / 2);
      const int hi = min(lo + kBN / 2, p.V - tc.n0);
      const float before = ms;
#pragma unroll 1
      for (int c = lo; c < hi; c += 32) {
        const int col0 = tc.n0 + c;
        uint32_t a[32];
        tmem_ld_32x32b_x32(taddr + c, a);
        tmem_ld_wait();
        uint32_t cand = c + 32 <= p.V - tc.n0 ? chunk_s<true>(p, a, col0) : chunk_s<false>(p, a, col0);
        fresh((c - lo) / 32) = cand;
#pragma unroll 1
        while (cand) {
          const int k = __ffs(cand) - 1;
          cand &= cand - 1u;
          const float v = __uint_as_float(pick32(a, k));
          if (v > sv[kTopMax - 1]) topk_insert3_asc(sv, si, sx, v, col0 + k, 0.f);
        }
      }
      if (p.reverse && hi > lo) A *= fast_exp2(before - ms);
      bound(half, 0) = static_cast<unsigned long long>(static_cast<uint32_t>(unit)) << 32 |
               __float_as_uint(sv[kTopMax - 1]);
    }

    template <class Release>
    __device__ void tile(const Params& p, const Sched&, int, int, const TileC& tc, uint32_t taddr,
                         const Release& release) {
      const unsigned long long pt = bound(1 - half, 1);
      if (pt >> 32 == static_cast<uint32_t>(unit)) bound_t = __uint_as_float(static_cast<uint32_t>(pt));
      const int lo = half * (kBN / 2);
      const int hi = min(lo + kBN / 2, p.V - tc.n0);
      if (hi <= lo) release();
#pragma unroll 1
      for (int c = lo; c < hi; c += 32) {
        const int col0 = tc.n0 + c;
        uint32_t a[32], b[32];
        tmem_ld_32x32b_x32(taddr + c, a);
        tmem_ld_32x32b_x32(taddr + kBN + c, b);
        tmem_ld_wait();
        if (c + 32 >= hi) release();
        uint32_t cand = c + 32 <= p.V - tc.n0 ? chunk_t<true>(p, a, b, col0) : chunk_t<false>(p, a, b, col0);
        uint32_t listed = fresh((c - lo) / 32);
#pragma unroll 1
        while (listed) {
          const int k = __ffs(listed) - 1;
          listed &= listed - 1u;
          const float x = __uint_as_float(pick32(b, k));
#pragma unroll
          for (int j = 0; j < kTopMax; ++j)
            if (si[j] == col0 + k) sx[j] = x;
        }
#pragma unroll 1
        while (cand) {
          const int k = __ffs(cand) - 1;
          cand &= cand - 1u;
          const float w = __uint_as_float(pick32(b, k));
          if (w > tv[kTopMax - 1]) topk_insert_asc(tv, ti, w, col0 + k);
        }
      }
      bound(half, 1) = static_cast<unsigned long long>(static_cast<uint32_t>(unit)) << 32 |
               __float_as_uint(tv[kTopMax - 1]);
    }

    __device__ void end(const Params& p, const Sched& s, int) {
      if (r >= s.sp.n) return;
      const size_t plane = p.plane;
      const size_t o = static_cast<size_t>(2 * sg + half) * s.sp.rt * kBM + r;
      p.part[0 * plane + o] = ms;
      p.part[1 * plane + o] = ss;
      p.part[2 * plane + o] = es;
      p.part[3 * plane + o] = mt;
      p.part[4 * plane + o] = st;
      p.part[5 * plane + o] = A;
      float4* v4 = reinterpret_cast<float4*>(p.part_sv + o * kTopMax);
      float4* x4 = reinterpret_cast<float4*>(p.part_sx + o * kTopMax);
      float4* w4 = reinterpret_cast<float4*>(p.part_tv + o * kTopMax);
      int4* i4 = reinterpret_cast<int4*>(p.part_si + o * kTopMax);
      int4* j4 = reinterpret_cast<int4*>(p.part_ti + o * kTopMax);
#pragma unroll
      for (int q = 0; q < kTopMax / 4; ++q) {
        v4[q] = make_float4(sv[4 * q], sv[4 * q + 1], sv[4 * q + 2], sv[4 * q + 3]);
        x4[q] = make_float4(sx[4 * q], sx[4 * q + 1], sx[4 * q + 2], sx[4 * q + 3]);
        w4[q] = make_float4(tv[4 * q], tv[4 * q + 1], tv[4 * q + 2], tv[4 * q + 3]);
        i4[q] = make_int4(si[4 * q], si[4 * q + 1], si[4 * q + 2], si[4 * q + 3]);
        j4[q] = make_int4(ti[4 * q], ti[4 * q + 1], ti[4 * q + 2], ti[4 * q + 3]);
      }
    }
  };
};

struct OpdOut {
  float *kl, *s_lse, *t_lse, *s_entropy, *s_topk_logp, *t_logp_s, *overlap, *kl_topk;
  int32_t* s_topk_ids;
};

__global__ void __launch_bounds__(128)
    opd_finalize_kernel(const int32_t* __restrict__ n_rows, const int32_t* __restrict__ rows, int T,
                        int vt, int ctas, size_t plane, int reverse, int K, float inv_tau,
                        const float* __restrict__ part, const float* __restrict__ part_sv,
                        const int32_t* __restrict__ part_si, const float* __restrict__ part_sx,
                        const float* __restrict__ part_tv, const int32_t* __restrict__ part_ti,
                        OpdOut out) {
  const int n = read_n_rows(n_rows, T, nullptr);
  const Split sp = choose_split(n, vt, ctas, OpdKern::seg_cap(n));
  const int nsv = 2 * sp.sv;  // two halves per vocabulary segment
  const size_t ld = static_cast<size_t>(sp.rt) * 128;
  const int lane = threadIdx.x & 31;
  const int warps = gridDim.x * 4;
  for (int r = blockIdx.x * 4 + (threadIdx.x >> 5); r < n; r += warps) {
    const int t = rows[r];
    if (t < 0 || t >= T) continue;  // reported by prepare_kernel
    float Ms = -INFINITY, Mt = -INFINITY, Ss = 0.f, Es = 0.f, St = 0.f, A = 0.f;
    float fs[2], ft[2];
    for (int s = lane; s < nsv; s += 32) {
      const size_t o = s * ld + r;
      merge_ms(Ms, Ss, part[0 * plane + o], part[1 * plane + o], fs);
      merge_ms(Mt, St, part[3 * plane + o], part[4 * plane + o], ft);
      Es = Es * fs[0] + part[2 * plane + o] * fs[1];
      A = reverse ? A * fs[0] + part[5 * plane + o] * fs[1] : A * ft[0] + part[5 * plane + o] * ft[1];
    }
    for (int o = merge_lanes(nsv) / 2; o > 0; o >>= 1) {
      const float ms2 = __shfl_xor_sync(0xffffffffu, Ms, o), ss2 = __shfl_xor_sync(0xffffffffu, Ss, o);
      const float mt2 = __shfl_xor_sync(0xffffffffu, Mt, o), st2 = __shfl_xor_sync(0xffffffffu, St, o);
      const float es2 = __shfl_xor_sync(0xffffffffu, Es, o), a2 = __shfl_xor_sync(0xffffffffu, A, o);
      merge_ms(Ms, Ss, ms2, ss2, fs);
      merge_ms(Mt, St, mt2, st2, ft);
      Es = Es * fs[0] + es2 * fs[1];
      A = reverse ? A * fs[0] + a2 * fs[1] : A * ft[0] + a2 * ft[1];
    }
    const float l2s = Ms + log2f(Ss);  // (lane 0's)
    const float l2t = Mt + log2f(St);
    const float ls = __shfl_sync(0xffffffffu, l2s * kLn2, 0), lt = __shfl_sync(0xffffffffu, l2t * kLn2, 0);
    if (lane == 0) {
      // KL = ln2 A / S_p - lse_p + lse_q
      if (out.kl) out.kl[t] = reverse ? kLn2 * (A / Ss) - ls + lt : kLn2 * (A / St) - lt + ls;
      if (out.s_lse) out.s_lse[t] = ls;
      if (out.t_lse) out.t_lse[t] = lt;
      if (out.s_entropy) out.s_entropy[t] = kLn2 * (l2s - Es / Ss);
    }
    float sv, tv;
    int si, ti;
    size_t at;
    warp_top_merge(part_tv, part_ti, nsv, ld, r, K, lane, tv, ti, at);
    warp_top_merge(part_sv, part_si, nsv, ld, r, K, lane, sv, si, at);
    bool hit = false;
    for (int q = 0; q < K; ++q) hit |= __shfl_sync(0xffffffffu, ti, q) == si;
    const int common = __popc(__ballot_sync(0xffffffffu, lane < K && hit));
    float term = 0.f;
    if (lane < K) {
      const float lps = sv * inv_tau - ls;
      const float lpt = (si == INT_MAX ? -INFINITY : part_sx[at]) * inv_tau - lt;
      term = expf(lps) * (lps - lpt);
      const size_t oj = static_cast<size_t>(t) * K + lane;
      if (out.s_topk_logp) out.s_topk_logp[oj] = lps;
      if (out.s_topk_ids) out.s_topk_ids[oj] = si;
      if (out.t_logp_s) out.t_logp_s[oj] = lpt;
    }
    for (int o = 16; o > 0; o >>= 1) term += __shfl_xor_sync(0xffffffffu, term, o);
    if (lane == 0) {
      if (out.overlap) out.overlap[t] = static_cast<float>(common) / static_cast<float>(K);
      if (out.kl_topk) out.kl_topk[t] = term;
    }
  }
}

}  // namespace

olive_status launch_opd_stats(const Ctx& c, const void* h_s, const void* W_s, int32_t d_s,
                              const void* h_t, const void* W_t, int32_t d_t, const int32_t* rows,
                              const int32_t* n_rows, int32_t T, int32_t V, float inv_tau,
                              int direction, int32_t K, float* kl, float* s_lse, float* t_lse,
                              float* s_entropy, float* s_topk_logp, int32_t* s_topk_ids,
                              float* t_logp_s, float* overlap, float* kl_topk, void* ws,
                              int32_t* dev_status) {
  const int64_t Tpad = align_up(static_cast<size_t>(T), kRowAlign);
  const OpdWs w = carve_opd(ws, T, d_s, d_t);
  const size_t tb = sizeof(float) * T, tkb = sizeof(float) * T * static_cast<size_t>(K);
  Prepare q;
  q.gather(h_s, d_s, w.hcs);
  q.gather(h_t, d_t, w.hct);
  for (float* z : {kl, s_lse, t_lse, s_entropy, overlap, kl_topk}) q.fill(z, tb);
  q.fill(s_topk_logp, tkb);
  q.fill(t_logp_s, tkb);
  q.fill(s_topk_ids, tkb, 0xff);
  olive_status st;
  if ((st = launch_prepare(c, q, rows, n_rows, T, dev_status)) != OLIVE_OK) return st;

  CUtensorMap mHs, mWs, mHt, mWt;
  if (!encode_bf16_2d(&mHs, w.hcs, d_s, Tpad, 2ull * d_s, 64, 128) ||
      !encode_bf16_2d(&mWs, W_s, d_s, V, 2ull * d_s, 64, OpdKern::kBN) ||
      !encode_bf16_2d(&mHt, w.hct, d_t, Tpad, 2ull * d_t, 64, 128) ||
      !encode_bf16_2d(&mWt, W_t, d_t, V, 2ull * d_t, 64, OpdKern::kBN))
    return OLIVE_ERR_CUDA;

  OpdKern::Params p = {};
  p.dev_status = dev_status;
  p.wait_limit_ns = c.wait_limit_ns;
  p.n_rows = n_rows;
  p.T = T;
  p.V = V;
  p.d_s = d_s;
  p.d_t = d_t;
  p.ctas = c.num_sms;
  p.group_rows = 16;
  p.plane = part_rows(Tpad, kMinPartsOpd);
  p.reverse = direction == OLIVE_KL_REVERSE;
  p.scale2 = inv_tau * kLog2e;
  p.part = w.part;
  p.part_sv = w.part_sv;
  p.part_si = w.part_si;
  p.part_sx = w.part_sx;
  p.part_tv = w.part_tv;
  p.part_ti = w.part_ti;
  const int smem = core_smem_bytes<OpdKern>();
  static std::atomic<int> done[kMaxDevices];
  if (!set_smem_once(reinterpret_cast<const void*>(gemm_persistent<OpdKern>), smem, c.device, done))
    return OLIVE_ERR_CUDA;
  gemm_persistent<OpdKern><<<c.num_sms, core_threads<OpdKern>(), smem, c.stream>>>(mHs, mWs, mHt, mWt, p);
  if (cudaGetLastError() != cudaSuccess) return OLIVE_ERR_CUDA;

  const int vt = (V + OpdKern::kBN - 1) / OpdKern::kBN;
  const OpdOut out{kl, s_lse, t_lse, s_entropy, s_topk_logp, t_logp_s, overlap, kl_topk, s_topk_ids};
  const int blocks = static_cast<int>(std::min<int64_t>(ceil_div(T, 4), c.num_sms * 16));
  opd_finalize_kernel<<<blocks, 128, 0, c.stream>>>(
      n_rows, rows, T, vt, c.num_sms, p.plane, p.reverse, K, inv_tau, w.part, w.part_sv, w.part_si,
      w.part_sx, w.part_tv, w.part_ti, out);
  return cudaGetLastError() == cudaSuccess ? OLIVE_OK : OLIVE_ERR_CUDA;
}

}  // namespace olive
