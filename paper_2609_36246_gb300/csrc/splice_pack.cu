// splice_pack.cu -- builds the packed student-update batch of Section 3.1:
// every sequence is prefix_s (prompt x and student prefix y_{1:k}) followed by
// the teacher continuation y~_{1:l}; row t predicts packed token t+1 of the
// same sequence, and only rows whose target is a continuation token carry a
// term of Eq. (osd-ce).
//
// Integer work only.  Up to kOwnSeqs sequences it is one launch: every block
// reads the offsets, validates and scans them into shared memory for itself
// (a few microseconds that all blocks spend side by side, where a scan kernel
// before the fill cost 5 us and a launch: 18.5 -> 13 us of kernels at 256
// sequences, 1.29 M positions), block 0 writes cu_seqlens, cut_offsets and
// n_rows (= sum_s C_s), and the block fills tiles of 1024 packed positions:
// it finds the sequences of the tile's ends by binary search in shared memory
// and each position's between those.  A row t < T is
// masked when its target is a continuation token; the j-th continuation token
// of sequence s is predicted by row cut_s - 1 + j, so rows[cont_off[s] + j] = t
// comes out ascending with no scan over the mask.  Malformed input clears
// every output.  Beyond kOwnSeqs sequences a scan kernel of one block writes
// the offsets first and the fill reads them from global memory.
//
// Multi-turn variant (Section 3.2: the loss covers only the teacher's
// actions; student turns and environment observations stay as context): a
// flag per continuation token selects the rows, so the row list needs a scan
// over the packed stream: a launch that counts the masked rows of every
// 2048-position chunk and one that adds up the counts before its chunk (one
// block does that beforehand where there are more than kOwnChunks) and fills,
// both with their own scan of the offsets as above (four kernels and 30 us
// before, two and 24 us now, at 64 sequences, 545 k positions).
#include <algorithm>

#include "internal.h"

namespace olive {
namespace {

constexpr int kScanThreads = 1024;

__device__ __forceinline__ long long block_excl_scan(long long v, long long* total, long long* sh) {
  // inclusive scan of one value per thread, 1024 threads
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  long long x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sh[warp] = x;
  __syncthreads();
  if (warp == 0) {
    long long w = sh[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    sh[lane] = w;
  }
  __syncthreads();
  const long long before = (warp > 0 ? sh[warp - 1] : 0) + x - v;
  *total = sh[31];
  __syncthreads();
  return before;
}

__global__ void __launch_bounds__(kScanThreads)
    splice_scan_kernel(const int32_t* __restrict__ prefix_off, const int32_t* __restrict__ cont_off,
                       int S, int T_cap, int32_t* __restrict__ cu, int32_t* __restrict__ cut,
                       int32_t* __restrict__ n_rows, int32_t* dev_status) {
  __shared__ long long sh[32];
  __shared__ int bad;
  if (threadIdx.x == 0) bad = (prefix_off[0] != 0 || cont_off[0] != 0) ? 1 : 0;
  __syncthreads();
  // pass 1: validate lengths and totals
  long long tot_len = 0, tot_c = 0;
  for (int b = 0; b < S; b += kScanThreads) {
    const int s = b + threadIdx.x;
    long long L = 0, C = 0;
    if (s < S) {
      const long long P = static_cast<long long>(prefix_off[s + 1]) - prefix_off[s];
      C = static_cast<long long>(cont_off[s + 1]) - cont_off[s];
      if (P < 1 || C < 0) bad = 1;
      L = P + C;
    }
    long long t1, t2;
    block_excl_scan(L, &t1, sh);
    block_excl_scan(C, &t2, sh);
    tot_len += t1;
    tot_c += t2;
  }
  __syncthreads();
  if (tot_len > T_cap) bad = 1;
  __syncthreads();
  if (bad) {
    for (int s = threadIdx.x; s <= S; s += kScanThreads) {
      cu[s] = 0;
      if (s < S) cut[s] = 0;
    }
    if (threadIdx.x == 0) {
      *n_rows = 0;
      atomicOr(dev_status, 1 << OLIVE_ERR_OFFSETS);
    }
    return;
  }
  // pass 2: exclusive scan of L_s = P_s + C_s
  long long carry = 0;
  for (int b = 0; b < S; b += kScanThreads) {
    const int s = b + threadIdx.x;
    long long L = 0, P = 0;
    if (s < S) {
      P = static_cast<long long>(prefix_off[s + 1]) - prefix_off[s];
      L = P + (static_cast<long long>(cont_off[s + 1]) - cont_off[s]);
    }
    long long tot;
    const long long before = block_excl_scan(L, &tot, sh);
    if (s < S) {
      cu[s] = static_cast<int32_t>(carry + before);
      cut[s] = static_cast<int32_t>(carry + before + P);
    }
    carry += tot;
  }
  if (threadIdx.x == 0) {
    cu[S] = static_cast<int32_t>(carry);
    *n_rows = static_cast<int32_t>(tot_c);
  }
}

constexpr int kOwnSeqs = 2048;    // sequences a block scans for itself
constexpr int kOwnChunks = 4096;  // chunk counts a block adds up for itself
constexpr int kFillThreads = 256;
constexpr int kTile = 1024;       // packed positions a block fills at a time
constexpr int kChunk = 2048;      // packed positions per block (masked variant)
constexpr int kPer = kChunk / kFillThreads;

// The batch's offsets as a block sees them: its own copies in shared memory
// (kOwn) or the arrays in global memory.
struct Batch {
  const int32_t *cu, *poff, *coff;
  int S, T;
};

struct BatchSmem {
  int32_t cu[kOwnSeqs + 1], poff[kOwnSeqs + 1], coff[kOwnSeqs + 1];
  long long scan[32];
  int bad;
};

// a block's shared copies, or nothing
template <bool kOwn>
struct SmemFor {
  BatchSmem batch;
};
template <>
struct SmemFor<false> {};

// Validates and scans the offsets into `sh`; block 0 writes the outputs that
// belong to them.  Every thread of the block calls it (kFillThreads threads).
__device__ Batch own_batch(BatchSmem& sh, const int32_t* __restrict__ prefix_off,
                           const int32_t* __restrict__ cont_off, int S, int T_cap,
                           int32_t* __restrict__ cu, int32_t* __restrict__ cut,
                           int32_t* __restrict__ n_rows, int32_t* dev_status) {
  const int tid = threadIdx.x;
  if (tid == 0) sh.bad = 0;
  __syncthreads();
  for (int s = tid; s <= S; s += kFillThreads) {
    sh.poff[s] = prefix_off[s];
    sh.coff[s] = cont_off[s];
  }
  __syncthreads();
  if (tid == 0 && (sh.poff[0] != 0 || sh.coff[0] != 0)) sh.bad = 1;
  // a thread takes `per` sequences in a row
  const int per = (S + kFillThreads - 1) / kFillThreads;
  const int s0 = tid * per, s1 = min(S, s0 + per);
  long long len = 0;
  bool bad = false;
  for (int s = s0; s < s1; ++s) {
    const long long P = static_cast<long long>(sh.poff[s + 1]) - sh.poff[s];
    const long long C = static_cast<long long>(sh.coff[s + 1]) - sh.coff[s];
    if (P < 1 || C < 0) bad = true;
    len += P + C;
  }
  // inclusive scan over the threads' lengths
  const int lane = tid & 31, warp = tid >> 5;
  long long x = len;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sh.scan[warp] = x;
  if (bad) sh.bad = 1;
  __syncthreads();
  long long before = x - len, total = 0;
#pragma unroll
  for (int w = 0; w < kFillThreads / 32; ++w) {
    if (w < warp) before += sh.scan[w];
    total += sh.scan[w];
  }
  const bool ok = !sh.bad && total <= T_cap;
  for (int s = s0; s < s1; ++s) {
    sh.cu[s] = ok ? static_cast<int32_t>(before) : 0;
    before += static_cast<long long>(sh.poff[s + 1]) - sh.poff[s] + sh.coff[s + 1] - sh.coff[s];
  }
  if (tid == 0) sh.cu[S] = ok ? static_cast<int32_t>(total) : 0;
  __syncthreads();
  if (blockIdx.x == 0) {
    for (int s = tid; s <= S; s += kFillThreads) {
      cu[s] = sh.cu[s];
      if (s < S) cut[s] = ok ? sh.cu[s] + (sh.poff[s + 1] - sh.poff[s]) : 0;
    }
    if (tid == 0) {
      if (n_rows) *n_rows = ok ? sh.coff[S] : 0;
      if (!ok) atomicOr(dev_status, 1 << OLIVE_ERR_OFFSETS);
    }
  }
  return Batch{sh.cu, sh.poff, sh.coff, S, ok ? static_cast<int>(total) : 0};
}

// sequence s in [lo, hi) with cu[s] <= t < cu[s + 1], given cu[lo] <= t < cu[hi]
__device__ __forceinline__ int find_seq(const Batch& b, int t, int lo, int hi) {
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (b.cu[mid] <= t) lo = mid; else hi = mid;
  }
  return lo;
}

// the sequences [lo, hi) that positions [t, e) of the stream (t < T) meet
__device__ __forceinline__ void seq_range(const Batch& b, int t, long long e, int& lo, int& hi) {
  lo = find_seq(b, t, 0, b.S);
  const int last = static_cast<int>(e < b.T ? e : b.T) - 1;
  hi = find_seq(b, last, lo, b.S) + 1;
}

struct PosInfo {
  int id, tgt;
  int j;  // index into cont_ids of the target, -1 when it is no continuation token
};

// Id and target of packed position t < T, in one of the sequences [lo, hi).
__device__ __forceinline__ PosInfo position_info(const Batch& b, int t, int lo, int hi,
                                                 const int32_t* __restrict__ prefix_ids,
                                                 const int32_t* __restrict__ cont_ids) {
  const int s = find_seq(b, t, lo, hi);
  const int i = t - b.cu[s];
  const int L = b.cu[s + 1] - b.cu[s];
  const int p0 = b.poff[s], c0 = b.coff[s];
  const int P = b.poff[s + 1] - p0;
  PosInfo r;
  r.id = i < P ? prefix_ids[p0 + i] : cont_ids[c0 + (i - P)];
  r.tgt = -1;
  r.j = -1;
  if (i + 1 < L) {
    if (i + 1 >= P) r.j = c0 + (i + 1 - P);
    r.tgt = r.j >= 0 ? cont_ids[r.j] : prefix_ids[p0 + i + 1];
  }
  return r;
}

template <bool kOwn>
__global__ void __launch_bounds__(kFillThreads)
    splice_fill_kernel(const int32_t* __restrict__ prefix_ids, const int32_t* __restrict__ prefix_off,
                       const int32_t* __restrict__ cont_ids, const int32_t* __restrict__ cont_off,
                       int S, int V, int T_cap, int32_t* __restrict__ cu, int32_t* __restrict__ cut,
                       int32_t* __restrict__ n_rows, int32_t* __restrict__ ids,
                       int32_t* __restrict__ targets, uint8_t* __restrict__ loss_mask,
                       int32_t* __restrict__ rows, int32_t* dev_status) {
  __shared__ SmemFor<kOwn> sh;
  Batch b;
  int nr;
  if constexpr (kOwn) {
    b = own_batch(sh.batch, prefix_off, cont_off, S, T_cap, cu, cut, n_rows, dev_status);
    nr = b.T > 0 ? b.coff[S] : 0;
  } else {
    b = Batch{cu, prefix_off, cont_off, S, cu[S]};
    nr = *n_rows;
  }
  bool range_bad = false;
  for (long long t0 = static_cast<long long>(blockIdx.x) * kTile; t0 < T_cap;
       t0 += static_cast<long long>(gridDim.x) * kTile) {
    int lo = 0, hi = 0;
    if (t0 < b.T) seq_range(b, static_cast<int>(t0), t0 + kTile, lo, hi);
#pragma unroll
    for (int q = 0; q < kTile / kFillThreads; ++q) {
      const long long tl = t0 + q * kFillThreads + threadIdx.x;
      if (tl >= T_cap) break;
      const int t = static_cast<int>(tl);
      if (t >= nr) rows[t] = -1;
      PosInfo r{0, -1, -1};
      if (t < b.T) {
        r = position_info(b, t, lo, hi, prefix_ids, cont_ids);
        if (r.id < 0 || r.id >= V) range_bad = true;
        if (r.j >= 0) rows[r.j] = t;
      }
      ids[t] = r.id;
      targets[t] = r.tgt;
      loss_mask[t] = r.j >= 0 ? 1 : 0;
    }
  }
  if (range_bad) atomicOr(dev_status, 1 << OLIVE_ERR_TOKEN_RANGE);
}

__device__ __forceinline__ int block_excl_scan_int(int v, int* total, int* sh) {
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sh[warp] = x;
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    int w = lane < nw ? sh[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    sh[lane] = w;
  }
  __syncthreads();
  const int before = (warp > 0 ? sh[warp - 1] : 0) + x - v;
  *total = sh[(blockDim.x >> 5) - 1];
  __syncthreads();
  return before;
}

// sum of one int per thread of the block (kFillThreads threads)
__device__ __forceinline__ int block_sum(int v, int* sh) {
  v = __reduce_add_sync(0xffffffffu, v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  int total = 0;
#pragma unroll
  for (int w = 0; w < kFillThreads / 32; ++w) total += sh[w];
  return total;
}

template <bool kOwn>
__global__ void __launch_bounds__(kFillThreads)
    turns_count_kernel(const int32_t* __restrict__ prefix_off, const int32_t* __restrict__ cont_off,
                       const uint8_t* __restrict__ cont_loss, int S, int T_cap,
                       int32_t* __restrict__ cu, int32_t* __restrict__ cut,
                       int32_t* __restrict__ chunk_count, int32_t* dev_status) {
  __shared__ SmemFor<kOwn> sh;
  __shared__ int part[32];
  Batch b;
  if constexpr (kOwn)
    b = own_batch(sh.batch, prefix_off, cont_off, S, T_cap, cu, cut, nullptr, dev_status);
  else
    b = Batch{cu, prefix_off, cont_off, S, cu[S]};
  const long long t0 = static_cast<long long>(blockIdx.x) * kChunk;
  int c = 0;
  if (t0 < b.T) {
    int lo, hi;
    seq_range(b, static_cast<int>(t0), t0 + kChunk, lo, hi);
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const long long t = t0 + q * kFillThreads + threadIdx.x;
      if (t >= b.T) break;
      const int s = find_seq(b, static_cast<int>(t), lo, hi);
      const int j = static_cast<int>(t) + 1 - b.cu[s] - (b.poff[s + 1] - b.poff[s]);
      if (t + 1 < b.cu[s + 1] && j >= 0) c += cont_loss[b.coff[s] + j] != 0;
    }
  }
  const int total = block_sum(c, part);
  if (threadIdx.x == 0) chunk_count[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanThreads)
    turns_offsets_kernel(int32_t* __restrict__ chunk_count, int n_chunks, int32_t* __restrict__ n_rows) {
  __shared__ int sh[32];
  int carry = 0;
  for (int b = 0; b < n_chunks; b += kScanThreads) {
    const int k = b + threadIdx.x;
    const int v = k < n_chunks ? chunk_count[k] : 0;
    int total;
    const int before = block_excl_scan_int(v, &total, sh);
    if (k < n_chunks) chunk_count[k] = carry + before;
    carry += total;
  }
  if (threadIdx.x == 0) *n_rows = carry;
}

// kSum: chunk_at holds the counts, which the block adds up itself (and the
// last block writes n_rows); else it holds the chunks' offsets.
template <bool kOwn, bool kSum>
__global__ void __launch_bounds__(kFillThreads)
    turns_fill_kernel(const int32_t* __restrict__ prefix_ids, const int32_t* __restrict__ prefix_off,
                      const int32_t* __restrict__ cont_ids, const int32_t* __restrict__ cont_off,
                      const uint8_t* __restrict__ cont_loss, int S, int V, int T_cap,
                      int32_t* __restrict__ cu, int32_t* __restrict__ cut,
                      const int32_t* __restrict__ chunk_at, int32_t* __restrict__ n_rows,
                      int32_t* __restrict__ ids, int32_t* __restrict__ targets,
                      uint8_t* __restrict__ loss_mask, int32_t* __restrict__ rows,
                      int32_t* dev_status) {
  __shared__ SmemFor<kOwn> sh;
  __shared__ int part[32];
  __shared__ int counts[kPer][kFillThreads / 32];
  Batch b;
  if constexpr (kOwn)
    b = own_batch(sh.batch, prefix_off, cont_off, S, T_cap, cu, cut, nullptr, dev_status);
  else
    b = Batch{cu, prefix_off, cont_off, S, cu[S]};
  int at, nr;
  if (kSum) {
    int head = 0, all = 0;
    for (int k = threadIdx.x; k < static_cast<int>(gridDim.x); k += kFillThreads) {
      const int v = chunk_at[k];
      all += v;
      if (k < static_cast<int>(blockIdx.x)) head += v;
    }
    at = block_sum(head, part);
    nr = block_sum(all, part);
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *n_rows = nr;
  } else {
    at = chunk_at[blockIdx.x];
    nr = *n_rows;
  }
  const long long t0 = static_cast<long long>(blockIdx.x) * kChunk;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int lo = 0, hi = 0;
  if (t0 < b.T) seq_range(b, static_cast<int>(t0), t0 + kChunk, lo, hi);
  bool range_bad = false;
  uint32_t marks[kPer];  // the warp's masked positions of each stride
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const long long tl = t0 + q * kFillThreads + threadIdx.x;
    bool masked = false;
    if (tl < T_cap) {
      const int t = static_cast<int>(tl);
      if (t >= nr) rows[t] = -1;
      PosInfo r{0, -1, -1};
      if (t < b.T) {
        r = position_info(b, t, lo, hi, prefix_ids, cont_ids);
        if (r.id < 0 || r.id >= V) range_bad = true;
        masked = r.j >= 0 && cont_loss[r.j] != 0;
      }
      ids[t] = r.id;
      targets[t] = r.tgt;
      loss_mask[t] = masked ? 1 : 0;
    }
    marks[q] = __ballot_sync(0xffffffffu, masked);
    if (lane == 0) counts[q][warp] = __popc(marks[q]);
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    int mine = at;
#pragma unroll
    for (int w = 0; w < kFillThreads / 32; ++w) {
      if (w < warp) mine += counts[q][w];
      at += counts[q][w];
    }
    if (marks[q] >> lane & 1u)
      rows[mine + __popc(marks[q] & ((1u << lane) - 1u))] =
          static_cast<int>(t0) + q * kFillThreads + static_cast<int>(threadIdx.x);
  }
  if (range_bad) atomicOr(dev_status, 1 << OLIVE_ERR_TOKEN_RANGE);
}

}  // namespace

olive_status launch_splice_pack(const Ctx& c, const int32_t* prefix_ids, const int32_t* prefix_off,
                                const int32_t* cont_ids, const int32_t* cont_off, int32_t S,
                                int32_t V, int32_t T_cap, int32_t* ids, int32_t* targets,
                                uint8_t* loss_mask, int32_t* cu_seqlens, int32_t* cut_offsets,
                                int32_t* rows, int32_t* n_rows, int32_t* dev_status) {
  // at most 8 blocks an SM: each scans the offsets once
  const int blocks = static_cast<int>(std::min<int64_t>(ceil_div(T_cap, kTile), c.num_sms * 8LL));
  if (S <= kOwnSeqs) {
    splice_fill_kernel<true><<<blocks, kFillThreads, 0, c.stream>>>(
        prefix_ids, prefix_off, cont_ids, cont_off, S, V, T_cap, cu_seqlens, cut_offsets, n_rows, ids,
        targets, loss_mask, rows, dev_status);
    return cudaGetLastError() == cudaSuccess ? OLIVE_OK : OLIVE_ERR_CUDA;
  }
  splice_scan_kernel<<<1, kScanThreads, 0, c.stream>>>(prefix_off, cont_off, S, T_cap, cu_seqlens,
                                                       cut_offsets, n_rows, dev_status);
  if (cudaGetLastError() != cudaSuccess) return OLIVE_ERR_CUDA;
  splice_fill_kernel<false><<<blocks, kFillThreads, 0, c.stream>>>(
      prefix_ids, prefix_off, cont_ids, cont_off, S, V, T_cap, cu_seqlens, cut_offsets, n_rows, ids,
      targets, loss_mask, rows, dev_status);
  return cudaGetLastError() == cudaSuccess ? OLIVE_OK : OLIVE_ERR_CUDA;
}

}  // namespace olive

namespace olive {

size_t splice_masked_ws_bytes(int64_t T_cap) {
  return align_up(sizeof(int32_t) * static_cast<size_t>(ceil_div(T_cap, kChunk)), kWsAlign);
}

olive_status launch_splice_pack_masked(const Ctx& c, const int32_t* prefix_ids,
                                       const int32_t* prefix_off, const int32_t* cont_ids,
                                       const int32_t* cont_off, const uint8_t* cont_loss, int32_t S,
                                       int32_t V, int32_t T_cap, int32_t* ids, int32_t* targets,
                                       uint8_t* loss_mask, int32_t* cu_seqlens,
                                       int32_t* cut_offsets, int32_t* rows, int32_t* n_rows,
                                       void* ws, int32_t* dev_status) {
  int32_t* chunk = static_cast<int32_t*>(ws);
  const int n_chunks = static_cast<int>(ceil_div(T_cap, kChunk));
  const bool own = S <= kOwnSeqs, sum = n_chunks <= kOwnChunks;
  if (!own) {
    splice_scan_kernel<<<1, kScanThreads, 0, c.stream>>>(prefix_off, cont_off, S, T_cap, cu_seqlens,
                                                         cut_offsets, n_rows, dev_status);
    if (cudaGetLastError() != cudaSuccess) return OLIVE_ERR_CUDA;
  }
  auto count = own ? turns_count_kernel<true> : turns_count_kernel<false>;
  count<<<n_chunks, kFillThreads, 0, c.stream>>>(prefix_off, cont_off, cont_loss, S, T_cap, cu_seqlens,
                                                 cut_offsets, chunk, dev_status);
  if (cudaGetLastError() != cudaSuccess) return OLIVE_ERR_CUDA;
  if (!sum) {
    turns_offsets_kernel<<<1, kScanThreads, 0, c.stream>>>(chunk, n_chunks, n_rows);
    if (cudaGetLastError() != cudaSuccess) return OLIVE_ERR_CUDA;
  }
  auto fill = own ? (sum ? turns_fill_kernel<true, true> : turns_fill_kernel<true, false>)
                  : (sum ? turns_fill_kernel<false, true> : turns_fill_kernel<false, false>);
  fill<<<n_chunks, kFillThreads, 0, c.stream>>>(prefix_ids, prefix_off, cont_ids, cont_off, cont_loss, S,
                                                V, T_cap, cu_seqlens, cut_offsets, chunk, n_rows, ids,
                                                targets, loss_mask, rows, dev_status);
  return cudaGetLastError() == cudaSuccess ? OLIVE_OK : OLIVE_ERR_CUDA;
}

}  // namespace olive
