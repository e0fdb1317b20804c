// lmhead_group.cu -- the training step of the Eq. (osd-ce) loss (Section 3.1)
// with its logit gradient formed and consumed on chip.
//
// With z = inv_tau H[rows] W^T, lse per row and G = coef (softmax(z) -
// onehot(y)) (coef = g inv_tau, / N_mask for OLIVE_REDUCE_MEAN):
//   dH = G . W       reduces over the vocabulary  (K = V)
//   dW = G^T . hc    reduces over the masked rows (K = N_mask)
// Either output tile is [128, d] fp32 for a 128-row M tile: 2 MB at d = 4096,
// eight SMs' worth of tensor memory, so one SM cannot hold it.  The CTAs are
// therefore split into GROUPS of g >= ceil(d / 256) members.  Member m owns
// the output columns [c0, c0 + cw) of d (cw <= 256) and keeps their 128 x cw
// fp32 accumulator in TMEM for a whole OUTER tile, while the members take
// turns computing the 128 x 256 logit tiles (Z jobs, K = d) that every member
// needs.  The member that computed a Z tile turns it into a bf16 EXCHANGE
// tile and stores it in its group's ring of R slots of 64 KB; every member
// bulk-copies each exchange tile, 64 K-columns at a time, into shared memory
// as the A operand of its accumulating MMA.  The ring has a fixed size (R
// slots per group, a few tens of MB in all, independent of T and V), each
// slot is rewritten once all g members have read it, and no slot outlives R
// exchange tiles: the logits and G are never stored as a [rows, V] array.
// (The ring is read from the L2; its lines are written back to DRAM when the
// L2 evicts them, about one write of each tile, the size of the exchange.)
//
//   Pass A (outer = 128 masked rows, inner = 256-column vocabulary tile):
//     exchange tile P'[r, v] = 2^(x - R_r), x = z log2(e), R_r a per-row
//     reference (the maximum of the row's first vocabulary tile, from the
//     GM_REF launch, or the row's lse when it is given); the members
//     accumulate acc = P' . W[:, chunk] and keep per-row partial sums of
//     2^(x - R) over their own Z jobs, merged at the end of the outer tile
//     into lse2 = R + log2(sum) (a group barrier through a global counter).
//     The epilogue then applies the softmax-minus-onehot scaling:
//       dH[r, chunk] = coef (2^(R - lse2) acc - W[y_r, chunk]).
//     A row whose maximum exceeds R by more than kRefMax (2^x - R would leave
//     the range the bf16 operand and the fp32 sums are safe in) puts its row
//     tile on a redo list; a second launch recomputes those tiles with R = the
//     rows' maxima from the first launch.
//   Pass B (outer = 128 vocabulary rows, inner = 256 masked rows): exchange
//     tile G^T[v, r] = coef_r (2^(x - lse2_r) - [v == y_r]) from pass A's
//     lse (transposed logit tile z^T = W hc^T, so a TMEM lane is a vocabulary
//     row); member m accumulates dW[v, chunk] = G^T . hc[:, chunk] and stores
//     it when the outer tile ends (every dW element has one owner: no atomics).
//
//   Divergence mode (GM_KL: the gradient of OPD's per-token KL, Section 1,
//   after the value sweep of lmhead_kl.cu has given KL and both heads' lse):
//     the pass A layout with two products per Z job, the student's (K = d_s)
//     and then the teacher's (K = d_t) logits of a 256-column vocabulary tile
//     in the Z accumulator, half of the previous round's accumulation between
//     them; the epilogue holds the student's logits in registers (128 a
//     thread) until the teacher's arrive and forms the exact G (reverse: g inv_tau p_s ((z_s - z_t) - (lse_s - lse_t) - KL),
//     forward: g inv_tau (p_s - p_t)) and the members accumulate
//     d_h_s = G . W_s.
//
// Each pass executes two products per logit (the Z tile and its share of the
// accumulation), so the training step executes 4 GEMM units of 2 N_mask d V
// flops for the 3 it counts.
//
// CTA pairs: the kernel runs as clusters of two CTAs.  Pair m of pair-group
// pg is member m of group 2 pg (its even CTA) and of group 2 pg + 1 (its odd
// CTA); the two groups walk the same inner tiles at the same time, so every
// MMA is a tcgen05.mma.cta_group::2 issued by the even CTA (M = 256: each CTA
// holds 128 rows of A -- its own hc, W or exchange rows -- and half of B's N
// columns, and receives its 128 accumulator rows in its own TMEM).  Each CTA
// loads 32 KB per 64-deep K step instead of 48 KB, and six stages fit.  The
// group size g is chosen between ceil(d / 256) and ~1.25 times that to fill
// the SMs with pair-groups of 2 g CTAs (d = 4096 on 152 SMs: g = 19, members
// of 224 columns, four pair-groups).  When the even group has one more outer
// tile than the odd one, the odd CTAs run a phantom tile whose rows are
// invalid and never stored.
//
// Schedule inside a group (every member derives it from N_mask on the
// device): the exchange tiles of the group's outer tiles form one sequence
// e = 0 .. E-1 (e = i ni + k for the group's i-th outer tile and inner tile
// k), cut into rounds of g tiles; tile e is computed by member e mod g and
// lives in ring slot e mod R (R = 3 g).  Each pair's tensor pipe runs, per
// round r: its Z job of round r, then the accumulation of all g tiles of
// round r - 1, so the epilogue of a Z tile (and the other members'
// epilogues) overlaps the accumulation MMAs, and a single 256-column Z
// accumulator suffices next to the (<= 256)-column output accumulator (512
// TMEM columns).  Waits between members go through global release/acquire
// counters: a slot's `ready` count (tile written) and `cons` count (tile
// copied by all g members); the producer warp checks a whole round's ready
// flags at once and a signal warp posts the cons counts.  Eight
// epilogue warps, two per TMEM lane quadrant with half of a tile's columns
// each, stage their bf16 values in shared memory and move them to the ring
// with 4 KB bulk stores, one `ready` count a warp; a finished output
// accumulator is taken into registers (up to 128 a thread) and handed back
// before it is converted and stored.  With four warps that stored 16-byte
// pieces from registers and held the accumulator until its rows were stored,
// the training step took 3.93 against 3.73 ms (1024 masked rows, d = 4096,
// V = 151936: outer tiles of pass B last 4 inner tiles; 3.4 ms now) and
// forward call + backward call 4.48 against 4.04 ms (1677 rows, d = 2560,
// V = 100003, fp32 gradients; 3.07 ms now); the divergence with two N = 128
// products side by side in the Z accumulator (60 % of the tensor rate) took
// 21.8 against 18.6 ms (4096 rows, d_s = 4096, d_t = 5120; 17.4 ms now).
// What bounds it now: the tensor pipe and, from some thousand rows on, the
// power cap (16384 rows: pipe 90 % active in pass A, 87 % in pass B); at a few
// hundred rows the rounds' exchange latency.
//
// Why the waits end: every CTA is resident at once (the grid is one CTA per SM;
// the host checks that the GPU holds all its clusters), and each wait is for
// work that does not wait for the waiter.
//   - Within a pair-group a wait for an exchange tile (`ready`) or its slot
//     (`cons`) is for work of an earlier round.
//   - Pass A's merge of an outer tile's sums waits for the posts of all members
//     that hold a part of it.  A member posts, takes its output accumulator out
//     and hands it back before it waits, and its Z tile of the round is
//     published by then, so the members of its own pair-group reach their posts
//     of the same round without it.
//   - Where a row pair of the tail is split between pair-groups, only the last
//     member to arrive for its columns waits, for the posts of the row pair's
//     other runs.  A run goes through its row pairs in ascending order, so what
//     can keep it from its post is a wait on the row pair before, which in turn
//     waits on runs of that one only: the chain ends at the tail's first row
//     pair.  Passes B and the divergence add partials up without waiting.
// Each is bounded all the same (OLIVE_ERR_TIMEOUT on expiry).
//
// A pacing hint keeps the groups within a round of one another, so that one
// DRAM fetch of an inner operand tile (W in pass A, hc in pass B) can serve
// every group from the L2 (how often it does depends on what else the L2
// holds: the call reads the streamed operand several times over).
#include <algorithm>
#include <atomic>
#include <cmath>

#include "sched.cuh"
#include "sm103.cuh"

namespace olive {
namespace {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr int kBM = 128;
constexpr int kBK = 64;
constexpr int kZN = 256;             // logit tile 128 x 256
constexpr int kStages = 6;
constexpr int kSA = kBM * kBK * 2;   // A operand of a stage: this CTA's 128 rows x 64
constexpr int kSB = kBM * kBK * 2;   // B operand: this CTA's half of N (<= 128) x 64
constexpr int kStageBytes = kSA + kSB;
constexpr int kXSlice = kSA;         // one 128 x 64 K-slice of an exchange tile
constexpr int kXTile = 4 * kXSlice;  // 128 x 256 bf16 (64 KB)
constexpr int kTailVecs = 32 * 256;  // float4 of a 128 x 256 fp32 accumulator
constexpr int kWarpSlice = kXSlice / 4;  // an epilogue warp's 32 rows of a slice (4 KB, contiguous)
constexpr int kEpiWarps = 8;         // two per TMEM lane quadrant, half of a tile's columns each
constexpr int kEpi = 32 * kEpiWarps; // epilogue threads: two per accumulator row
constexpr int kProducerWarp = kEpiWarps;
constexpr int kMmaWarp = kEpiWarps + 1;
constexpr int kSignalWarp = kEpiWarps + 2;  // posts the members' "tile copied" counts
constexpr int kLossWarp = kEpiWarps + 3;
constexpr int kThreads = 32 * (kEpiWarps + 4);  // three whole warpgroups
constexpr int kPieceMax = 4;  // K steps (~2000 cycles) of a Z product at an outer tile's boundary
// Registers a thread: 168 at launch (65536 / 384 threads); the warpgroup of
// the producer, MMA and signal warps hands most of its share to the two of
// the epilogue, whose 128 held accumulator values otherwise spill (the L1 left
// beside 227 KB of shared memory is too small for 384 stacks: spilled, a
// 32-column block took ~5500 cycles).  2 x 216 + 72 = 3 x 168.
constexpr int kEpiRegs = 216;
constexpr int kOtherRegs = 72;
constexpr int kStatusTimeoutBit = 1 << OLIVE_ERR_TIMEOUT;
constexpr float kRefMax = 64.f;
constexpr int kMetaBytes = kZN * 8;  // pass B: lse2 and target of the tile's 256 rows
// Pacing across groups: every group walks the same sequence of inner tiles
// (vocabulary tiles of W in pass A, row pairs of hc in pass B), so while the
// groups stay within kPaceLag rounds of one another one DRAM fetch of a tile
// serves all of them from the L2; a group that runs ahead waits, at most
// kPaceLimitNs per round (a hint: giving up only costs bandwidth).
constexpr int kPaceLag = 1;
constexpr uint64_t kPaceLimitNs = 2000000;
constexpr uint32_t kPaceDone = 0x40000000u;

enum GMode : int { GM_REF = 0, GM_A = 1, GM_B = 2, GM_KL = 3 };

// GM_REF / GM_A: za = hc {64 x 128}, zb = W {64 x 128}, xb = W {64 x 64}
// GM_B:          za = W {64 x 128},  zb = hc {64 x 128}, xb = hc {64 x 64}
// xa: the ring, [slices x 128 rows] of 64 bf16, unswizzled {64 x 128} boxes
// (a slice is stored already swizzled, so the copy is linear)
// GM_KL:         za = hc_s {64 x 128}, zb = W_s {64 x 128}, za2 = hc_t {64 x 128},
//                zb2 = W_t {64 x 128}, xb = W_s {64 x 64}
struct GroupMaps {
  CUtensorMap za, zb, xb, xa, za2, zb2;
};

struct GroupParams {
  int32_t* dev_status;
  uint64_t wait_limit_ns;
  const int32_t* n_rows;
  const int32_t* rows;
  const int32_t* targets;
  const __nv_bfloat16* W;   // GM_A: the rows W[y] of the onehot term
  int32_t T, d, V;
  int32_t mode;
  int32_t g, ngroups, R;    // members per group, groups, ring slots per group
  int32_t chunk;            // output columns per member (multiple of 16, <= 256)
  int32_t c_base, c_end;    // output columns [c_base, c_end) of this launch
  int32_t reduction;
  float inv_tau, scale2;    // 1 / tau, log2(e) / tau
  const float* grad_loss;   // device scalar g
  int32_t lse_known;        // GM_A: R = lse2 from lse_in (backward of a given forward)
  int32_t redo;             // GM_A: outer tiles from redo_list, R = rmax
  int32_t write_fwd;        // GM_A: write lse, logp, nll
  const float* lse_in;      // [T] natural lse per packed row (GM_A lse_known, GM_B)
  float* rref;              // [Tpad] base-2 reference per compact row (GM_REF writes)
  float* rmax;              // [Tpad] base-2 row maximum (GM_A writes for redo rows)
  // per member, two rows of [Tpad] for the two column halves of its Z tiles
  float* part_s;            // [2 g][Tpad] sums of 2^(x - R): the second's; the first's are 0
  float* part_m;            // [2 g][Tpad] the logits' maxima (base 2)
  float* zy;                // [Tpad] target logit z_y (natural units)
  float* pyb;               // [Tpad] P'_y as rounded to bf16 in the exchange tile
  float* logp;              // [T]
  float* lse;               // [T]
  float* nll;               // [Tpad] per-row loss terms
  float* loss;              // GM_B: their sum (or mean), null when not asked for
  uint32_t* redo_list;      // [1 + rt]: count, then row tiles
  uint32_t* outer_ctr;      // [rt] pass A group barrier (one array per GM_A launch)
  __nv_bfloat16* ring;      // [ngroups][R][128 x 256] exchange tiles (swizzled images)
  uint32_t* ready;          // [ngroups][R]
  uint32_t* cons;           // [ngroups][R]
  uint32_t* pace;           // [ngroups] rounds each group has begun (a pacing hint)
  // split row pairs (see GSched): partial accumulators [slot][2][g] of
  // kTailVecs float4 (in the order of the epilogue's threads), GM_A's partial
  // sums (as in part_s) and maxima [slot][2 g][2 x 128], and how many runs have left their
  // partial per row tile and member
  float* tail_acc;
  float *tail_s, *tail_m;
  uint32_t* tail_ctr;
  int32_t tail_parts, tail_slots;  // (debug checks)
  void* out;                // GM_A: d_hidden [T, d]; GM_B: d_W [V, d]
  int32_t out_dtype;
  int64_t ring_tiles;       // exchange tiles the ring holds (debug checks)
  int32_t part_groups;      // rows of part_s / part_m (debug checks)
  // GM_KL (divergence gradient): per compact row the lse of both heads from the
  // value sweep, per packed row the KL and the weights g_t
  int32_t d2;               // teacher width
  int32_t reverse;          // KL direction
  const float* lse_sc;      // [Tpad] student lse (natural)
  const float* lse_tc;      // [Tpad] teacher lse (natural)
  const float* kl;          // [T]
  const float* grad_kl;     // [T]
};

// Per-CTA schedule, the same in every CTA of a group.
//
// Outer tiles go in pairs (a row pair: tile 2 rp for the even CTAs, 2 rp + 1
// for the odd ones).  Pair-group pg takes the row pairs pg, pg + npg, ... as
// far as every pair-group gets one; the last r = nrp mod npg pairs are the
// tail.  Left whole, they keep r pair-groups busy for ni inner tiles while the
// others idle, which is all of pass A at up to 256 rows.  So the tail's r * ni
// inner tiles are laid end to end and cut into nt runs of equal length, one a
// pair-group; a run covers the end of one row pair, the start of the next, or
// a part of one.  Each run leaves its partial fp32 accumulator (and pass A's
// row sums) in the workspace, in slot c + t for run c and row pair t of the
// tail (c + t grows along the line, so slots are distinct and fewer than
// 2 npg), and the last member to arrive for its columns adds the partials up
// in run order, the same order every time.
// A run costs its length and every partial of a row pair about 1.2 us to add,
// a quarter of an inner tile's time at the least, so runs are at least
// sqrt(ni / 4) long and the tail stays whole where that cost is not below ni.
// Pass A, whole -> split: 365 rows, d = 2048, V = 151936 (2 row pairs for 8
// pair-groups) 1580 -> 545 us (457 now); 1677 rows, d = 2560, V = 100003
// (7 for 6) 1910 -> 1275 us (1046 now); 300 rows, d = 256, V = 4096 (2 row
// pairs of 16 tiles) 126 -> 30 us.
struct GSched {
  int n;      // masked rows
  int rank;   // 0: the pair's even CTA (issues the MMAs), 1: its peer
  int ph;     // outer index standing for "no outer tile" (past the last)
  int no;     // outer tiles in all
  int ni;     // inner tiles per outer tile
  int nk;     // 64-wide K steps of a Z job
  int q, m;   // group, member
  int pg, npg;  // pair-group, pair-groups
  int rp0;    // first row pair of the tail
  int tail0;  // the group's first exchange tile in the tail
  int x0;     // its place on the tail's line of inner tiles
  int nt;     // runs the tail is cut into (0: left whole)
  int xs;     // inner tiles in the tail
  int E;      // exchange tiles of this group
  int c0, cw; // output columns of this member
  int nbox;   // 64-column boxes of this CTA's half of the accumulation's B
  int nacc;   // N of the accumulation MMA (cw rounded up to 16)
  int b0;     // first column of this CTA's half of B
  int kcount; // inner extent: V (pass A) or n (pass B)
  int nk2;    // 64-wide K steps of a Z job's second product (GM_KL: the teacher)
  float coef;
};

// start of run c of the tail's line
__device__ __forceinline__ int run_start(const GSched& s, int c) {
  return static_cast<int>(static_cast<int64_t>(s.xs) * c / s.nt);
}
// the run that holds place x
__device__ __forceinline__ int run_of(const GSched& s, int x) {
  return static_cast<int>((static_cast<int64_t>(x + 1) * s.nt - 1) / s.xs);
}

// CTAs come in pairs (clusters of 2): pair-group pg of g pairs runs groups
// 2 pg (even CTAs) and 2 pg + 1 (odd CTAs) in lockstep, pair m being member m
// of both; the two groups walk the same inner tiles at the same time, so
// each pair's MMAs share the B operand (W or hc tiles), half from each CTA.
__device__ GSched make_gsched(const GroupParams& p) {
  GSched s;
  s.n = read_n_rows(p.n_rows, p.T, p.dev_status);
  s.rank = static_cast<int>(cluster_rank());
  const int rt = (s.n + kBM - 1) / kBM;
  if (p.mode == GM_B) {
    s.no = (p.V + kBM - 1) / kBM;
    s.ph = s.no;
    s.ni = (s.n + kZN - 1) / kZN;
    s.kcount = s.n;
  } else {
    s.no = (p.mode == GM_A && p.redo) ? static_cast<int>(min(p.redo_list[0], static_cast<uint32_t>(rt))) : rt;
    s.ph = rt;
    s.ni = p.mode == GM_REF ? 1 : (p.V + kZN - 1) / kZN;
    s.kcount = p.V;
  }
  s.nk = (p.d + kBK - 1) / kBK;
  s.nk2 = p.mode == GM_KL ? (p.d2 + kBK - 1) / kBK : 0;
  const int pair = blockIdx.x >> 1;
  s.m = pair % p.g;
  const int pg = pair / p.g;
  s.q = 2 * pg + s.rank;
  // when the number of outer tiles is odd, the odd CTAs' half of the last row
  // pair is a phantom whose rows are invalid
  s.pg = pg;
  s.npg = p.ngroups / 2;
  const int nrp = (s.no + 1) / 2;
  const int nfull = nrp / s.npg;
  const int r = nrp - nfull * s.npg;
  s.rp0 = nfull * s.npg;
  s.tail0 = nfull * s.ni;
  s.xs = r * s.ni;
  s.nt = 0;
  if (p.tail_acc && r > 0) {
    int least = 2;
    while (4 * least * least < s.ni) ++least;
    const int nt = min(s.npg, s.xs / least);
    if (nt > r) {
      const int len = (s.xs + nt - 1) / nt;
      if (len + (s.ni + len - 1) / len / 4 + 2 < s.ni) s.nt = nt;
    }
  }
  if (s.nt > 0) {
    s.x0 = pg < s.nt ? run_start(s, pg) : 0;
    s.E = s.tail0 + (pg < s.nt ? run_start(s, pg + 1) - s.x0 : 0);
  } else {
    s.x0 = pg * s.ni;
    s.E = s.tail0 + (pg < r ? s.ni : 0);
  }
  s.c0 = p.c_base + s.m * p.chunk;
  s.cw = min(p.chunk, p.c_end - s.c0);
  if (s.cw < 0) s.cw = 0;
  s.nacc = (s.cw + 15) / 16 * 16;
  if (s.nacc < 16) s.nacc = 16;
  s.b0 = s.c0 + s.rank * (s.nacc / 2);
  s.nbox = (s.nacc / 2 + 63) / 64;
  s.coef = 0.f;
  if (p.grad_loss) {
    float gl = *p.grad_loss;
    if (p.reduction == OLIVE_REDUCE_MEAN && s.n > 0) gl = gl / static_cast<float>(s.n);
    s.coef = gl * p.inv_tau;
  }
  return s;
}

// row pair and inner tile of the group's exchange tile e
struct Pos {
  int rp, k;
};
__device__ __forceinline__ Pos locate(const GSched& s, int e) {
  const bool tail = e >= s.tail0;
  const int x = tail ? s.x0 + e - s.tail0 : e;
  const int i = x / s.ni;
  return Pos{tail ? s.rp0 + i : s.pg + i * s.npg, x - i * s.ni};
}
// Walks a group's exchange tiles in order without a division a tile.  What the
// producer and MMA warps do between two instructions of theirs shows in the
// tensor pipe, which has little of a queue: pass A at 1024 rows, d = 4096,
// V = 151936 took 657 cycles a K step (480 at the tensor pipe's peak) with
// locate(), a remainder and whole descriptors built at every tile and MMA, 633
// with this and additions, and 511 with the roles' loops run by whole warps
// (mbar_wait_warp).
struct TileWalk {
  int e, k, slot;
  int ni, tail0, ktail, R;
  __device__ __forceinline__ TileWalk(const GSched& s, int ring_slots) {
    e = 0;
    slot = 0;
    ni = s.ni;
    R = ring_slots;
    tail0 = s.tail0;
    ktail = s.nt > 0 ? s.x0 % s.ni : 0;
    k = tail0 == 0 ? ktail : 0;
  }
  __device__ __forceinline__ void next() {
    ++e;
    k = k + 1 == ni ? 0 : k + 1;
    if (e == tail0) k = ktail;
    slot = slot + 1 == R ? 0 : slot + 1;
  }
};
// does tile e open / close its outer tile's part in this group?
__device__ __forceinline__ bool opens(const GSched& s, int e, int k) { return k == 0 || e == s.tail0; }
__device__ __forceinline__ bool closes(const GSched& s, int e, int k) {
  return k == s.ni - 1 || e == s.E - 1;
}
// index of this CTA's outer tile of a row pair (s.ph for a phantom)
__device__ __forceinline__ bool phantom(const GSched& s, int rp) { return 2 * rp + s.rank >= s.no; }
__device__ __forceinline__ int outer_of(const GroupParams& p, const GSched& s, int rp) {
  const int k = 2 * rp + s.rank;
  if (k >= s.no) return s.ph;
  return (p.mode == GM_A && p.redo) ? static_cast<int>(p.redo_list[1 + k]) : k;
}
__device__ __forceinline__ int kvalid_of(const GSched& s, int k) {
  return min(kZN, s.kcount - k * kZN);
}
// 64-wide K slices of inner tile k that hold valid columns
__device__ __forceinline__ int slices_of(const GSched& s, int k) {
  return (kvalid_of(s, k) + kBK - 1) / kBK;
}
// does member m compute a Z job of the outer tile part that tile e (at inner
// tile k) closes?
__device__ __forceinline__ bool member_has_job(const GSched& s, int g, int e, int k) {
  const int lo = e >= s.tail0 ? max(e - k, s.tail0) : e - k;
  return lo + (((s.m - lo) % g) + g) % g <= e;
}

// Order of a round's work, the same for the producer, MMA and epilogue warps of
// a pair.  The round accumulates tiles [e_lo, e_end); where one of them opens
// an outer tile, its MMAs must wait until the epilogue has taken the previous
// outer tile's accumulator.  So the Z product is cut: its first `head` K steps
// start the round, `piece` more run at every such boundary while the
// accumulator changes hands, the rest at the last one, and the Z epilogue comes
// after the outer tiles that close before it (first in the round, it held all
// of them up).  The tail of the round covers the Z epilogue, the head (at least
// half of the product) the latency of the exchange.  Only pass B is cut so: the
// outer tiles of the others are as long as the vocabulary.
//
// A round is `count` + 1 steps of the same two parts, so that each part's code
// stands once in each role (a call of a few microseconds waits for much of its
// code to come from memory): K steps [z0, z1) of a Z product, then tiles up to
// `until`.  The divergence's two products are its two steps: half of the
// previous round's tiles are accumulated between them, which is when the
// epilogue takes the student's logits into registers, and no later than before
// a tile that opens an outer tile (that needs the accumulator which the
// epilogue hands back only after it has had the teacher's logits).
struct Round {
  int count;        // steps after the first
  int first, last;  // tiles that the second and the last step open with
  int head, piece;  // K steps of the Z product in the first step, and in the others
};
struct Step {
  int z0, z1, steps;  // K steps of the product of `steps`
  bool second;        // GM_KL: the teacher's product
  int until;          // then the tiles before this one
};
template <int kMode>
__device__ __forceinline__ Round plan_round(const GSched& s, int e_lo, int e_end) {
  Round rd{0, e_lo, e_lo, s.nk, 0};
  if (kMode == GM_KL) {
    rd.count = 1;
    rd.first = e_lo == e_end ? e_end : min(e_lo + (e_end - e_lo + 1) / 2, e_lo + s.ni - locate(s, e_lo).k);
    return rd;
  }
  if (kMode != GM_B || e_end - e_lo < 2) return rd;
  rd.first = e_lo + s.ni - locate(s, e_lo).k;
  // (tiles past the start of a split tail open at other distances)
  const int end = e_lo < s.tail0 ? min(e_end, s.tail0 + 1) : e_end;
  if (rd.first >= end) return rd;
  rd.count = (end - 1 - rd.first) / s.ni + 1;
  rd.last = rd.first + (rd.count - 1) * s.ni;
  rd.piece = max(1, min(kPieceMax, s.nk / 2 / rd.count));
  rd.head = max(1, s.nk - rd.count * rd.piece);
  return rd;
}
template <int kMode>
__device__ __forceinline__ Step round_step(const GSched& s, const Round& rd, int b, int e_end) {
  Step st;
  st.until = b == rd.count ? e_end : rd.first + b * s.ni;
  st.second = kMode == GM_KL && b == 1;
  if (kMode == GM_KL) {
    st.z0 = 0;
    st.z1 = st.steps = b == 0 ? s.nk : s.nk2;
  } else {
    st.steps = s.nk;
    st.z0 = b == 0 ? 0 : min(s.nk, rd.head + (b - 1) * rd.piece);
    st.z1 = b == rd.count ? s.nk : min(s.nk, rd.head + b * rd.piece);
  }
  return st;
}

// byte offset of row r (a multiple of 8) of K-slice sl in an exchange tile.
// The image is the 128-byte-swizzled K-major layout a TMA load of a 64 x 128
// box produces (row r at r * 128, its 16-byte chunk c at position c ^ (r & 7)),
// so a linear copy of a slice to a 1024-byte-aligned stage is a valid UMMA
// operand.
__device__ __forceinline__ uint32_t img_off(int r, int sl) {
  return static_cast<uint32_t>(sl * kXSlice + r * 128);
}

// 32 fp32 values (the slice's first or last 32 columns) -> four 16-byte
// chunks of this lane's row in the warp's staging copy of a slice: 32 rows of
// 128 bytes in the same swizzled order as the exchange image (img_off), so
// one 4 KB bulk store moves them.  A quarter warp's 8 lanes hit 8 different
// 16-byte columns: no bank conflicts.
__device__ __forceinline__ void stage32(uint32_t stage, int lane, int h, const float (&v)[32]) {
  const uint32_t row = stage + static_cast<uint32_t>((lane >> 3) * 1024 + (lane & 7) * 128);
#pragma unroll
  for (int q = 0; q < 4; ++q)
    st_shared_v4(row + ((((h & 1) * 4 + q) ^ (lane & 7)) << 4),
                 make_uint4(pack_bf16x2(v[8 * q], v[8 * q + 1]), pack_bf16x2(v[8 * q + 2], v[8 * q + 3]),
                            pack_bf16x2(v[8 * q + 4], v[8 * q + 5]), pack_bf16x2(v[8 * q + 6], v[8 * q + 7])));
}

// per-row values of pass A (and GM_REF) for compact row rc
struct RowA {
  bool valid;   // rc < n and rows[rc] in [0, T)
  int t, y;     // packed row, target (-1 when none)
  float R;      // reference (base 2)
};

__device__ __forceinline__ RowA load_row_a(const GroupParams& p, const GSched& s, int rc) {
  RowA a;
  a.valid = false;
  a.t = -1;
  a.y = -1;
  a.R = 0.f;
  if (rc < s.n) {
    const int t = p.rows[rc];
    if (t >= 0 && t < p.T) {
      a.valid = true;
      a.t = t;
      a.y = p.targets[t];
      if (p.mode == GM_A) {
        if (p.lse_known) a.R = p.lse_in[t] * kLog2e;
        else if (p.redo) a.R = p.rmax[rc];
        else a.R = p.rref[rc];
      }
    }
  }
  return a;
}

// All lanes of a warp: wait until the exchange tiles [e_lo, e_end) of a
// round are written (every epilogue warp of their member has posted
// ready[e mod R] e / R + 1 times), lane i checking tiles i, i+32,
// ...  Returns the warp's common decision (false: limit ran out or abort).
__device__ bool wait_round_ready(const uint32_t* ready, int R, int e_lo, int e_end, int lane,
                                 const WaitCtl& ctl) {
  const uint64_t t0 = global_timer_ns();
  while (true) {
    bool mine = true;
    for (int e = e_lo + lane; e < e_end; e += 32)
      mine = mine && ld_acquire(ready + e % R) >= static_cast<uint32_t>(kEpiWarps * (e / R + 1));
    if (__all_sync(0xffffffffu, mine)) return true;
    bool stop = *ctl.abort != 0;
    if (!stop && global_timer_ns() - t0 > ctl.limit_ns) {
      if (lane == 0) *ctl.abort = 1;
      stop = true;
    }
    if (__any_sync(0xffffffffu, stop)) return false;
    nanosleep_ns(64);
  }
}

// All lanes of a warp: wait (at most kPaceLimitNs) until every group has
// begun round `need` (pace[q] >= need), lane i checking groups i, i+32, ...
__device__ void pace_wait(const uint32_t* pace, int ngroups, int need, int lane) {
  if (need <= 0) return;
  const uint64_t t0 = global_timer_ns();
  while (true) {
    bool mine = true;
    for (int q = lane; q < ngroups; q += 32)
      mine = mine && *reinterpret_cast<const volatile uint32_t*>(pace + q) >= static_cast<uint32_t>(need);
    if (__all_sync(0xffffffffu, mine)) return;
    if (global_timer_ns() - t0 > kPaceLimitNs) return;
    nanosleep_ns(128);
  }
}

template <int kMode>
__global__ void __launch_bounds__(kThreads, 1)
    lmhead_group_kernel(const __grid_constant__ GroupMaps maps, const GroupParams p) {
  // the redo launch mostly has nothing to do: it leaves before any barrier or
  // TMEM is set up (the same decision in every CTA)
  if (kMode == GM_A && p.redo && p.redo_list[0] == 0) return;

  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = smem_u32(smem_raw);
  uint8_t* gbase = smem_raw;

  // the same layout in both CTAs of a pair: the MMA reads both at these offsets
  const uint32_t stages = base;
  const uint32_t stage_out = base + kStages * kStageBytes;  // the epilogue warps' staging
  const uint32_t bar0 = stage_out + kEpiWarps * kWarpSlice;
  auto full_bar = [&](int st) { return bar0 + 8u * st; };
  auto empty_bar = [&](int st) { return bar0 + 8u * (kStages + st); };
  const uint32_t zfull = bar0 + 8u * (2 * kStages);
  const uint32_t zempty = zfull + 8;
  const uint32_t ofull = zfull + 16;
  const uint32_t oempty = zfull + 24;
  const uint32_t drain = zfull + 32;
  uint8_t* misc = gbase + kStages * kStageBytes + kEpiWarps * kWarpSlice + 8 * (2 * kStages + 5);
  static_assert(16 + sizeof(GSched) <= 128, "schedule area");
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 4);
  volatile uint32_t* copied = reinterpret_cast<volatile uint32_t*>(misc + 8);  // tiles copied
  GSched* sched_smem = reinterpret_cast<GSched*>(misc + 16);
  float* meta_l = reinterpret_cast<float*>(misc + 128);                 // [256] lse2 (GM_B)
  int* meta_y = reinterpret_cast<int*>(misc + 128 + kMetaBytes / 2);    // [256] targets (GM_B)

  const int warp = warp_uniform(static_cast<int>(threadIdx.x >> 5));
  const int lane = threadIdx.x & 31;
  const uint32_t rank = warp_uniform(cluster_rank());

  if (threadIdx.x == 0) {
    for (int st = 0; st < kStages; ++st) {
      mbar_init(full_bar(st), 1);   // the even CTA's producer (both CTAs' bytes)
      mbar_init(empty_bar(st), 1);  // the even CTA's MMA commit (multicast)
    }
    mbar_init(zfull, 1);
    mbar_init(zempty, 2 * kEpiWarps);  // the epilogue warps of both CTAs
    mbar_init(ofull, 1);
    mbar_init(oempty, 2 * kEpiWarps);
    mbar_init(drain, 1);
    *abort_flag = 0;
    *copied = 0;
    *sched_smem = make_gsched(p);
    fence_mbar_init();
  }
  if (warp == kProducerWarp && lane == 0) {
    tma_prefetch_desc(&maps.za);
    tma_prefetch_desc(&maps.zb);
    tma_prefetch_desc(&maps.xb);
    tma_prefetch_desc(&maps.xa);
  }
  if (warp == kMmaWarp) {
    tmem_alloc_pair(smem_u32(tmem_slot), 512);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  // barriers of both CTAs initialised and TMEM allocated before any CTA
  // touches its peer's
  cluster_sync_all();
  tc_fence_after();

  const uint32_t tmem_base = *tmem_slot;
  // (each role copies it to registers: shared memory is busy with the MMAs'
  // operands, and the epilogue's reads of it cost pass B 3 %)
  const GSched& s = *sched_smem;
  const WaitCtl ctl{abort_flag, p.wait_limit_ns};
  const int g = p.g;
  constexpr bool consume = kMode != GM_REF;
  const int nr = (s.E + g - 1) / g;  // rounds
  const size_t ring0 = static_cast<size_t>(s.q) * p.R;

  if (warp >= kEpiWarps) {
    regs_dec<kOtherRegs>();
    if (warp == kProducerWarp) {
      // one lane issues every copy (this CTA's 128 rows of A and its half of B;
      // completion counted on the even CTA's full barrier, whose producer
      // announces both CTAs' bytes: the odd CTA's copies may land first, the
      // transaction count then dips below zero within the phase, which mbarriers
      // allow; no phase can mix with the next, since a CTA refills a stage only
      // after the MMAs that read it have committed); the lanes share the check
      // of the `ready` flags of a round's g exchange tiles
      const GSched s = warp_uniform_copy(sched_smem);
      const bool leader = elect_one();
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      TileWalk at(s, p.R);
      const int xrow = s.q * p.R * 4;  // the group's first slice in the ring
      const bool paced = consume && p.ngroups > 2;
      // the streamed operand of a Z job (W rows in pass A, hc rows in pass B)
      // is read again by the accumulation a round later: keep it in the L2
      // ahead of other lines (ncu at 16384 rows: DRAM reads 196 -> 149 GB per
      // call, time level)
      const uint64_t keep = l2_policy_evict_last();
      for (int r = 0; ok && r <= nr; ++r) {
        const int j = r * g + s.m;
        if (paced && r < nr) {
          pace_wait(p.pace, p.ngroups, r - kPaceLag, lane);
          if (s.m == 0 && lane == 0)
            *reinterpret_cast<volatile uint32_t*>(p.pace + s.q) = static_cast<uint32_t>(r + 1);
        }
        const bool job = r < nr && j < s.E;
        // a Z product: za x zb, or GM_KL's teacher za2 x zb2; the B rows are this
        // CTA's half of the 256-wide vocabulary (or row) tile
        auto load_z = [&](bool second, int ks0, int ks1) {
          const Pos z = locate(s, j);
          const int o = warp_uniform(outer_of(p, s, z.rp));
          const int k = z.k;
          for (int ks = ks0; ok && ks < ks1; ++ks) {
            if (!mbar_wait_warp(empty_bar(stage), phase ^ 1u, ctl)) { ok = false; break; }
            const uint32_t sA = stages + stage * kStageBytes;
            const uint32_t fb = map_shared(full_bar(stage), 0);
            // (a skipped copy leaves its stage short: the MMA's wait then runs
            // out and the call reports OLIVE_ERR_TIMEOUT as well)
            const bool in = OLIVE_DCHECK(p.dev_status, o >= 0 && o <= s.ph && k >= 0 && k < s.ni);
            if (leader) {
              if (rank == 0) mbar_arrive_expect_tx(full_bar(stage), 2 * kStageBytes);
              if (in) {
                tma_load_2d_pair(sA, second ? &maps.za2 : &maps.za, fb, ks * kBK, o * kBM);
                tma_load_2d_pair_hint(sA + kSA, second ? &maps.zb2 : &maps.zb, fb, ks * kBK,
                                      k * kZN + static_cast<int>(rank) * (kZN / 2), keep);
              }
            }
            if (++stage == kStages) { stage = 0; phase ^= 1u; }
          }
        };
        auto load_tiles = [&](int e_to) {
          for (; ok && at.e < e_to; at.next()) {
            const int slot = at.slot;
            const int k = at.k;
            const int nsl = slices_of(s, k);
            for (int sl = 0; sl < nsl; ++sl) {
              if (!mbar_wait_warp(empty_bar(stage), phase ^ 1u, ctl)) { ok = false; break; }
              const uint32_t sA = stages + stage * kStageBytes;
              const uint32_t fb = map_shared(full_bar(stage), 0);
              // TMA x coordinates must be 16-byte aligned (8 bf16)
              const bool in = OLIVE_DCHECK(p.dev_status, static_cast<int64_t>(ring0 + slot) < p.ring_tiles &&
                                                             s.b0 % 8 == 0 && s.b0 >= 0 && s.b0 < p.d + 64);
              if (leader) {
                if (rank == 0) mbar_arrive_expect_tx(full_bar(stage), 2 * (kXSlice + s.nbox * 8192));
                if (in) {
                  tma_load_2d_pair(sA, &maps.xa, fb, 0, (xrow + slot * 4 + sl) * kBM);
                  tma_load_2d_pair(sA + kSA, &maps.xb, fb, s.b0, k * kZN + sl * kBK);
                  if (s.nbox > 1)
                    tma_load_2d_pair(sA + kSA + 8192, &maps.xb, fb, s.b0 + 64, k * kZN + sl * kBK);
                }
              }
              if (++stage == kStages) { stage = 0; phase ^= 1u; }
            }
          }
        };
        const int e_lo = r > 0 ? (r - 1) * g : 0;
        const int e_end = r > 0 ? min(r * g, s.E) : 0;
        const Round rd = plan_round<kMode>(s, e_lo, e_end);
        for (int b = 0; ok && b <= rd.count; ++b) {
          const Step st = round_step<kMode>(s, rd, b, e_end);
          if (job) load_z(st.second, st.z0, st.z1);
          if (!ok || !consume) break;
          if (b == 0 && r > 0) {
            ok = wait_round_ready(p.ready + ring0, p.R, e_lo, e_end, lane, ctl);
            if (!ok) break;
            __syncwarp();
            fence_proxy_async_global();
          }
          load_tiles(st.until);
        }
      }
      if (paced && s.m == 0 && lane == 0) *reinterpret_cast<volatile uint32_t*>(p.pace + s.q) = kPaceDone;
      if (!ok && lane == 0) {
        // let copies already issued land before the CTA retires
        const uint64_t t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 50000) nanosleep_ns(1000);
      }
      __syncwarp();
    } else if (warp == kSignalWarp) {
      // for every exchange tile, in order, once the pair's MMA thread has seen
      // all its slices land: one release increment of the slot's `cons` count
      if (lane == 0 && consume) {
        uint32_t sent = 0;
        const uint32_t total = static_cast<uint32_t>(s.E);
        uint64_t last = global_timer_ns();
        while (sent < total) {
          const uint32_t c = *copied;
          if (c > sent) {
            for (; sent < c; ++sent) red_release_add(p.cons + ring0 + sent % p.R, 1u);
            last = global_timer_ns();
            continue;
          }
          if (*abort_flag) break;
          nanosleep_ns(100);
          if (global_timer_ns() - last > p.wait_limit_ns) {
            *abort_flag = 1;
            break;
          }
        }
      }
      __syncwarp();
    } else if (warp == kLossWarp) {
      // a warp that has nothing else to do, in one CTA: the loss from pass A's
      // per-row terms, in a fixed order (a launch of its own took 5 us and a
      // gap at the end of every step)
      if (kMode == GM_B && p.loss && blockIdx.x == gridDim.x - 1) {
        double acc = 0.0;
        for (int rc = lane; rc < s.n; rc += 32) acc += static_cast<double>(p.nll[rc]);
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (p.reduction == OLIVE_REDUCE_MEAN) acc = s.n > 0 ? acc / s.n : 0.0;
        if (lane == 0) *p.loss = static_cast<float>(acc);
      }
    } else if (warp == kMmaWarp) {
      // a lane of the even CTA's MMA warp issues the pair's MMAs (M = 256: 128
      // rows in each CTA's TMEM); the odd CTA's only holds its TMEM allocation
      if (rank == 0) {
        const GSched s = warp_uniform_copy(sched_smem);
        const bool leader = elect_one();
        const uint32_t zacc = warp_uniform(tmem_base);
        const uint32_t oacc = zacc + 256;
        const uint32_t idz = idesc_bf16(2 * kBM, kZN, false, false);
        const uint32_t idx = idesc_bf16(2 * kBM, s.nacc, false, true);
        const uint32_t copied_peer = map_shared(smem_u32(const_cast<uint32_t*>(copied)), 1);
        // a stage's operand descriptors are these plus its offset in 16-byte
        // units: the issuing thread then adds twice an MMA
        const uint64_t dA = sdesc_sw128(stages, 16, 1024);
        const uint64_t dBk = sdesc_sw128(stages + kSA, 16, 1024);     // B K-major (Z)
        const uint64_t dBm = sdesc_sw128(stages + kSA, 8192, 1024);   // B MN-major (accumulation)
        int stage = 0;
        uint32_t phase = 0, zph = 0, oph = 0;
        bool ok = true;
        TileWalk at(s, p.R);
        for (int r = 0; ok && r <= nr; ++r) {
          const int j = r * g + s.m;
          const bool job = r < nr && j < s.E;
          // K steps [ks0, ks1) of a Z product of `steps`
          auto z_product = [&](int ks0, int ks1, int steps) {
            if (ks0 == 0) {
              if (!mbar_wait_warp(zempty, zph ^ 1u, ctl)) { ok = false; return; }
              tc_fence_after();
            }
            for (int ks = ks0; ks < ks1; ++ks) {
              if (!mbar_wait_warp(full_bar(stage), phase, ctl)) { ok = false; return; }
              tc_fence_after();
              const uint32_t so = static_cast<uint32_t>(stage) * (kStageBytes >> 4);
              const uint32_t acc0 = ks > 0 ? 1u : 0u;
              if (leader) {
#pragma unroll
                for (int kk = 0; kk < kBK / 16; ++kk)
                  umma_bf16_pair(zacc, dA + (so + kk * 2), dBk + (so + kk * 2), idz, kk > 0 ? 1u : acc0);
                umma_commit_pair(empty_bar(stage));
              }
              if (++stage == kStages) { stage = 0; phase ^= 1u; }
            }
            if (ks1 == steps) {
              if (leader) umma_commit_pair(zfull);
              zph ^= 1u;
            }
          };
          auto accumulate = [&](int e_to) {
            for (; ok && at.e < e_to; at.next()) {
              const int e = at.e, k = at.k;
              const bool first = opens(s, e, k);
              if (first) {
                if (!mbar_wait_warp(oempty, oph ^ 1u, ctl)) { ok = false; break; }
                tc_fence_after();
              }
              const int nsl = slices_of(s, k);
              for (int sl = 0; sl < nsl; ++sl) {
                if (!mbar_wait_warp(full_bar(stage), phase, ctl)) { ok = false; break; }
                tc_fence_after();
                const uint32_t so = static_cast<uint32_t>(stage) * (kStageBytes >> 4);
                const uint32_t acc0 = !first || sl > 0 ? 1u : 0u;
                if (leader) {
#pragma unroll
                  for (int kk = 0; kk < kBK / 16; ++kk)
                    umma_bf16_pair(oacc, dA + (so + kk * 2), dBm + (so + kk * 128), idx, kk > 0 ? 1u : acc0);
                  umma_commit_pair(empty_bar(stage));
                }
                if (++stage == kStages) { stage = 0; phase ^= 1u; }
              }
              if (!ok) break;
              // every slice of tile e has landed in both CTAs: their signal warps
              // tell the two groups (a slot may be rewritten once all of its
              // group's members have said so)
              if (leader) {
                *copied = static_cast<uint32_t>(e + 1);
                st_shared_cluster(copied_peer, static_cast<uint32_t>(e + 1));
              }
              if (closes(s, e, k)) {
                if (leader) umma_commit_pair(ofull);
                oph ^= 1u;
              }
            }
          };
          const int e_lo = r > 0 ? (r - 1) * g : 0;
          const int e_end = r > 0 ? min(r * g, s.E) : 0;
          const Round rd = plan_round<kMode>(s, e_lo, e_end);
          for (int b = 0; ok && b <= rd.count; ++b) {
            const Step st = round_step<kMode>(s, rd, b, e_end);
            if (job && st.z1 > st.z0) z_product(st.z0, st.z1, st.steps);
            if (ok && consume) accumulate(st.until);
          }
        }
        // arrives once every MMA issued above has completed (bounded wait that
        // ignores the abort flag: it only waits for work already in flight)
        if (leader) umma_commit_pair(drain);
        volatile int keep_waiting = 0;
        const uint64_t floor_ns = 200ull * 1000 * 1000;
        const WaitCtl own{&keep_waiting, p.wait_limit_ns > floor_ns ? p.wait_limit_ns : floor_ns};
        mbar_wait_warp(drain, 0, own);
      }
      __syncwarp();
    }
  } else {
    regs_inc<kEpiRegs>();
    // epilogue warps 0..7: the two warps of a TMEM lane quadrant share its 32
    // accumulator rows (thread = row), `half` choosing the columns: the first
    // or last 128 of a Z tile, the first or last 32-column blocks of the
    // member's output chunk
    const GSched s = *sched_smem;
    const int half = warp >> 2;
    const int row = (warp & 3) * 32 + lane;
    const uint32_t lane_addr = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    uint8_t* ring_bytes = reinterpret_cast<uint8_t*>(p.ring);
    // the even CTA's MMA thread waits until both CTAs' epilogues are done with
    // an accumulator: one arrival per epilogue warp on its barriers
    const uint32_t zempty_lead = map_shared(zempty, 0);
    const uint32_t oempty_lead = map_shared(oempty, 0);
    const uint32_t zaddr = lane_addr;
    const uint32_t staging = stage_out + warp * kWarpSlice;
    // this thread's output columns [ob, oe) of the chunk
    const int oblocks = (s.cw + 31) / 32;
    const int ob = half ? (oblocks + 1) / 2 * 32 : 0;
    const int oe = half ? s.cw : min(s.cw, (oblocks + 1) / 2 * 32);
    const uint32_t oaddr = lane_addr + 256 + ob;
    uint32_t zph = 0, oph = 0;
    bool ok = true;
    const size_t Tpad = static_cast<size_t>((p.T + kBM - 1) / kBM) * kBM;

    // The finished output accumulator: every value into registers first, then
    // the accumulator is handed back, so that the next outer tile's MMAs run
    // while this one is scaled, converted and stored.  (Holding it until the
    // stores were issued left the tensor pipe idle for most of every outer
    // tile's epilogue, which shows where outer tiles are short: pass B at few
    // masked rows.)
    // (acc is declared where it is used: held across the loop it would cost
    // its 128 registers everywhere)
    auto take_output = [&](float(&acc)[4][32]) -> bool {
      if (!named_bar_and(1, kEpi, mbar_wait(ofull, oph, ctl))) return false;
      oph ^= 1u;
      tc_fence_after();
#pragma unroll
      for (int b = 0; b < 4; ++b)  // (columns past oe are read and not stored)
        tmem_ld_32x32b_x32(oaddr + 32 * b, reinterpret_cast<uint32_t(&)[32]>(acc[b]));
      tmem_ld_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(oempty_lead);
      return true;
    };
    // acc -> output row t (a packed or vocabulary row; -1: none).  128 bytes
    // of each of the warp's 32 rows at a time (64 bf16 or 32 fp32 columns) go
    // through the staging area, so that a store instruction writes four whole
    // lines; from the registers it would write half sectors of 32 lines, and
    // a 128 x 224 tile took 5 us.
    auto store_output = [&](int t, const float(&acc)[4][32]) {
      const bool wide = p.out_dtype == OLIVE_DTYPE_F32;
      const int per = wide ? 32 : 64;  // columns of a step, 8 chunks of 16 bytes
      const uint32_t mine = staging + lane * 128;
      auto flush = [&](int c) {
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int rr = u * 4 + (lane >> 3);
          const int tr = __shfl_sync(0xffffffffu, t, rr);
          const uint4 v = ld_shared_v4(staging + rr * 128 + (((lane & 7) ^ (rr & 7)) << 4));
          const int col = c + (lane & 7) * (per / 8);
          if (tr >= 0 && col < oe && OLIVE_DCHECK(p.dev_status, s.c0 + col + per / 8 <= p.d)) {
            const size_t at = static_cast<size_t>(tr) * p.d + s.c0 + col;
            *reinterpret_cast<uint4*>(static_cast<uint8_t*>(p.out) + (wide ? 4 : 2) * at) = v;
          }
        }
        __syncwarp();
      };
      if (wide) {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          if (ob + 32 * b >= oe) continue;
#pragma unroll
          for (int q = 0; q < 8; ++q)
            st_shared_v4(mine + ((q ^ (lane & 7)) << 4),
                         make_uint4(__float_as_uint(acc[b][4 * q]), __float_as_uint(acc[b][4 * q + 1]),
                                    __float_as_uint(acc[b][4 * q + 2]), __float_as_uint(acc[b][4 * q + 3])));
          flush(ob + 32 * b);
        }
      } else {
#pragma unroll
        for (int b = 0; b < 4; b += 2) {
          if (ob + 32 * b >= oe) continue;
          stage32(staging, lane, 0, acc[b]);
          stage32(staging, lane, 1, acc[b + 1]);
          flush(ob + 32 * b);
        }
      }
    };

    // pass A: this thread's sum and maximum of the row, for the part of the
    // outer tile that exchange tile e belongs to
    auto tail_row = [&](int slot, int mm) -> size_t {
      return (static_cast<size_t>(slot) * 2 * g + mm) * 2 * kBM + s.rank * kBM + row;
    };
    auto put_sums = [&](int e, int rp, int o, float sum, float mx) {
      const bool tail = s.nt > 0 && e >= s.tail0;
      const size_t i = tail ? tail_row(s.pg + rp - s.rp0, 2 * s.m + half)
                            : static_cast<size_t>(2 * s.m + half) * Tpad + o * kBM + row;
      if (!OLIVE_DCHECK(p.dev_status, tail ? s.pg + rp - s.rp0 < p.tail_slots
                                           : 2 * s.m + half < p.part_groups && o * kBM + row < static_cast<int>(Tpad)))
        return;
      (tail ? p.tail_s : p.part_s)[i] = sum;
      (tail ? p.tail_m : p.part_m)[i] = mx;
    };

    if (kMode == GM_B && s.ni == 0) {
      // no masked rows: dW is zero on this member's columns of its outer tiles
      const int vecs = s.cw * (p.out_dtype == OLIVE_DTYPE_F32 ? 4 : 2) / 16;
      for (int rp = s.pg; 2 * rp < s.no; rp += s.npg) {
        const int v = outer_of(p, s, rp) * kBM + row;
        if (v >= p.V) continue;
        uint4* o = reinterpret_cast<uint4*>(static_cast<uint8_t*>(p.out) +
                                            (p.out_dtype == OLIVE_DTYPE_F32 ? 4 : 2) *
                                                (static_cast<size_t>(v) * p.d + s.c0));
        for (int c = half; c < vecs; c += 2) o[c] = make_uint4(0, 0, 0, 0);
      }
    }

    int cur_rp = -1;            // pass A: the row pair of the running partials
    RowA ra{false, -1, -1, 0.f};
    float run_m = -INFINITY;  // of x - R
    const float s_coef = s.coef;
    for (int r = 0; ok && r <= nr; ++r) {
      const int j = r * g + s.m;
      const int e_lo = r > 0 ? (r - 1) * g : 0;
      const int e_end = r > 0 ? min(r * g, s.E) : 0;
      const Round rd = plan_round<kMode>(s, e_lo, e_end);
      // the outer tiles that close before the round's last boundary, then the Z
      // tile, then the others
      for (int part = kMode == GM_B && rd.count > 0 ? 0 : 1; ok && part < 2; ++part) {
        if (part == 1 && r < nr && j < s.E) {
          // ---------------------------------------------------- Z epilogue
          const Pos at = locate(s, j);
          const int k = at.k;
          const int o = outer_of(p, s, at.rp);
          const int slot = j % p.R;
          const int kv = kvalid_of(s, k);
          // 32-column blocks to read: every block of the slices the members
          // copy, so columns >= kv are written as zeros, never left stale
          const int hlast = 2 * slices_of(s, k);
          const int hbeg = half * (kZN / 64);
          const int hend = min(hlast, hbeg + kZN / 64);
          // the slot's previous tile must have been copied by every member
          bool go = true;
          if (consume && lane == 0) {
            go = wait_counter(p.cons + ring0 + slot, static_cast<uint32_t>(g * (j / p.R)), ctl);
            fence_proxy_async_global();
          }
          if (kMode == GM_B) {
            // lse2 and target of the tile's 256 masked rows (+inf / -1 beyond n)
            for (int c = threadIdx.x; c < kZN; c += kEpi) {
              const int rc = k * kZN + c;
              float l2 = INFINITY;
              int yy = -1;
              if (rc < s.n) {
                const int t = p.rows[rc];
                if (t >= 0 && t < p.T) {
                  l2 = p.lse_in[t] * kLog2e;
                  yy = p.targets[t];
                }
              }
              meta_l[c] = l2;
              meta_y[c] = yy;
            }
          }
          if (!named_bar_and(1, kEpi, go && mbar_wait(zfull, zph, ctl))) { ok = false; break; }
          zph ^= 1u;
          tc_fence_after();
          float pv_all[4][32];  // pass A: 2^(x - R) of this thread's columns
          bool fresh = false;   // pass A: the member's first tile of the outer tile
          uint8_t* img = ring_bytes + (ring0 + slot) * static_cast<size_t>(kXTile);
          if (!OLIVE_DCHECK(p.dev_status, !consume || static_cast<int64_t>(ring0 + slot) < p.ring_tiles))
            img = nullptr;
          // Two 32-column blocks at a time make a slice of this warp's 32 rows,
          // staged in shared memory and moved to the ring by one bulk store
          // (4 KB of whole lines).  `put` stages a block once the previous
          // slice's copy has read the staging area, and starts the copy after
          // the second block.  (Storing the 16-byte chunks straight from the
          // registers writes half sectors of 32 different lines per
          // instruction, and needed a device-wide fence by every thread of the
          // epilogue per tile; the bulk stores need one by each warp's lane 0.)
          auto put = [&](int h, const float (&v)[32]) {
            if (!(h & 1)) {
              if (lane == 0) bulk_wait_read();
              __syncwarp();
            }
            stage32(staging, lane, h, v);
            if (h & 1) {
              fence_proxy_async_shared();
              __syncwarp();
              if (lane == 0 && img) {
                bulk_store(img + img_off((warp & 3) * 32, h >> 1), staging, kWarpSlice);
                bulk_commit();
              }
            }
          };
          // the accumulator goes back to the MMA thread once its last block is
          // in registers
          auto drained = [&](int h) {
            if (h + 1 < hend) return;
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(zempty_lead);
          };
          if (kMode != GM_KL && hbeg >= hend) drained(hend);  // no valid column in this half
          if (kMode == GM_B) {
            const int v = o * kBM + row;
            // does any of this half's columns have its target in the outer tile?
            bool hit = false;
#pragma unroll
            for (int q = 0; q < 4; ++q)
              hit = hit || static_cast<uint32_t>(meta_y[half * 128 + q * 32 + lane] - o * kBM) < kBM;
            hit = __any_sync(0xffffffffu, hit);
#pragma unroll 1
            for (int h = hbeg; h < hend; ++h) {
              uint32_t a[32];
              tmem_ld_32x32b_x32(zaddr + h * 32, a);
              tmem_ld_wait();
              drained(h);
              float gv[32];
#pragma unroll
              for (int c = 0; c < 32; ++c)
                gv[c] = s_coef * fast_exp2(fmaf(__uint_as_float(a[c]), p.scale2, -meta_l[h * 32 + c]));
              if (hit) {
                // the target entry p - 1 from expm1, exact where p is near 1
#pragma unroll 1
                for (int c = 0; c < 32; ++c) {
                  if (meta_y[h * 32 + c] != v) continue;
                  float z = 0.f;
#pragma unroll
                  for (int q = 0; q < 32; ++q) z = q == c ? __uint_as_float(a[q]) : z;
                  z = s_coef * expm1f(fmaf(z, p.scale2, -meta_l[h * 32 + c]) * kLn2);
#pragma unroll
                  for (int q = 0; q < 32; ++q) gv[q] = q == c ? z : gv[q];
                }
              }
              if (h * 32 + 32 > kv) {
                // rows beyond the last one may hold anything, NaN too
#pragma unroll
                for (int c = 0; c < 32; ++c) gv[c] = h * 32 + c < kv ? gv[c] : 0.f;
              }
              put(h, gv);
            }
          } else if (kMode == GM_KL) {
            // G of the divergence for this 128 x 256 tile from both heads' fp32
            // logits and the row's lse of each head and KL from the value sweep:
            // reverse g inv_tau p_s (log p_s - log p_t - KL), forward
            // g inv_tau (p_s - p_t).  The student's logits arrive first and wait
            // in registers for the teacher's.
            float zs_all[4][32];
#pragma unroll
            for (int b = 0; b < 4; ++b)
              tmem_ld_32x32b_x32(zaddr + (hbeg + b) * 32, reinterpret_cast<uint32_t(&)[32]>(zs_all[b]));
            tmem_ld_wait();
            drained(hend - 1);
            const int rc = o * kBM + row;
            bool valid = false;
            float ls0 = 0.f, lt0 = 0.f, klv = 0.f, cf = 0.f;
            if (rc < s.n) {
              const int t = p.rows[rc];
              if (t >= 0 && t < p.T) {
                valid = true;
                ls0 = p.lse_sc[rc];
                lt0 = p.lse_tc[rc];
                klv = p.kl[t];
                cf = p.grad_kl[t] * p.inv_tau;
              }
            }
            if (!named_bar_and(1, kEpi, mbar_wait(zfull, zph, ctl))) { ok = false; break; }
            zph ^= 1u;
            tc_fence_after();
            if (hbeg >= hend) drained(hend);
            // log p_s - log p_t as (z_s - z_t) - (lse_s - lse_t): a teacher
            // shifted by a constant per row cancels before the large terms meet
            const float dl = ls0 - lt0;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              const int h = hbeg + b;
              if (h >= hend) break;
              float(&gv)[32] = zs_all[b];
#pragma unroll
              for (int u = 0; u < 32; u += 16) {
                uint32_t zt_b[16];
                tmem_ld_32x32b_x16(zaddr + h * 32 + u, zt_b);
                tmem_ld_wait();
                if (u) drained(h);
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                  const float zs = gv[u + c] * p.inv_tau;
                  const float zt = __uint_as_float(zt_b[c]) * p.inv_tau;
                  const float ps = fast_exp2((zs - ls0) * kLog2e);
                  gv[u + c] = cf * (p.reverse ? ps * (((zs - zt) - dl) - klv)
                                              : ps - fast_exp2((zt - lt0) * kLog2e));
                }
              }
              if (!valid || h * 32 + 32 > kv) {
#pragma unroll
                for (int c = 0; c < 32; ++c) gv[c] = valid && h * 32 + c < kv ? gv[c] : 0.f;
              }
              put(h, gv);
            }
          } else {
            fresh = at.rp != cur_rp;
            if (fresh) {
              cur_rp = at.rp;
              ra = load_row_a(p, s, o * kBM + row);
              run_m = -INFINITY;
            }
            const int v0 = k * kZN;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              const int h = hbeg + b;
              if (h >= hend) {
#pragma unroll
                for (int c = 0; c < 32; ++c) pv_all[b][c] = 0.f;
                continue;
              }
              uint32_t a[32];
              tmem_ld_32x32b_x32(zaddr + h * 32, a);
              tmem_ld_wait();
              drained(h);
              float(&pv)[32] = pv_all[b];
              // (two running maxima of x - R: shorter chains)
              float m1 = -INFINITY;
              if (h * 32 + 32 <= kv) {
#pragma unroll
                for (int c = 0; c < 32; c += 2) {
                  const float x0 = fmaf(__uint_as_float(a[c]), p.scale2, -ra.R);
                  const float x1 = fmaf(__uint_as_float(a[c + 1]), p.scale2, -ra.R);
                  run_m = fmaxf(run_m, x0);
                  m1 = fmaxf(m1, x1);
                  pv[c] = fast_exp2(x0);
                  pv[c + 1] = fast_exp2(x1);
                }
              } else {
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                  const bool in = h * 32 + c < kv;
                  const float x0 = fmaf(__uint_as_float(a[c]), p.scale2, -ra.R);
                  m1 = in ? fmaxf(m1, x0) : m1;
                  pv[c] = in ? fast_exp2(x0) : 0.f;
                }
              }
              run_m = fmaxf(run_m, m1);
              const int yo = ra.y - (v0 + h * 32);
              if (kMode == GM_A && yo >= 0 && yo < 32) {
                // the target's exact logit and the bf16 value of P'_y the MMA
                // sees: the epilogue replaces that term by p_y - 1 from the
                // logit, so rows with p_y near 1 keep their accuracy
#pragma unroll
                for (int c = 0; c < 32; ++c)
                  if (c == yo) {
                    p.zy[o * kBM + row] = __uint_as_float(a[c]) * p.inv_tau;
                    p.pyb[o * kBM + row] = __bfloat162float(__float2bfloat16_rn(pv[c]));
                  }
              }
              if (kMode == GM_A) put(h, pv);
            }
          }
          if (kMode == GM_REF) {
            // the row's two column halves meet in shared memory
            if (half) meta_l[row] = run_m;
            named_bar_sync(1, kEpi);
            const float ref = fmaxf(run_m, meta_l[row]);
            // (a tile of -inf logits alone is no reference: 0 finds the row's maximum,
            // which the redo launch takes where it is out of range)
            if (!half && o * kBM + row < s.n) p.rref[o * kBM + row] = ref == -INFINITY ? 0.f : ref;
            named_bar_sync(1, kEpi);
          } else {
            // publish the warp's part of the tile once its copies are complete
            if (lane == 0) {
              bulk_wait();
              fence_proxy_async_global();
              red_release_add(p.ready + ring0 + slot, 1u);
            }
            __syncwarp();
            // the row metadata of this tile is read: the next one's may be written
            if (kMode == GM_B) named_bar_sync(1, kEpi);
            if (kMode == GM_A) {
              // The row's sum over this member's tiles is one chain in column
              // order, which the first half's thread hands to the second's in
              // shared memory.  (One sum a half rounds less where a large term
              // stands early, but by other amounts than the target's logit does,
              // and the mean loss, in which the two nearly cancel, was 1.5 to 1.7
              // times as far from 64 bits.)
              if (half) named_bar_sync(2, kEpi);
              float sum = !half && fresh ? 0.f : meta_l[row];
#pragma unroll
              for (int b = 0; b < 4; ++b)
#pragma unroll
                for (int c = 0; c < 32; ++c) sum += pv_all[b][c];
              meta_l[row] = sum;
              if (!half) named_bar_arrive(2, kEpi);
              if (ra.valid) put_sums(j, at.rp, o, half ? sum : 0.f, run_m + ra.R);
            }
          }
        }
        if constexpr (!consume) break;
        if (r == 0) continue;
        // ------------------------------------------- outer tiles completed
        for (int e = part == 0 ? e_lo : rd.last; ok && e < (part == 0 ? rd.last : e_end); ++e) {
          const Pos at = locate(s, e);
          if (!closes(s, e, at.k)) continue;
          const int o = outer_of(p, s, at.rp);
          const bool split = s.nt > 0 && e >= s.tail0;
          // the runs [run_lo, run_hi] of the tail that hold a part of this row pair
          const int t = at.rp - s.rp0;
          const int run_lo = split ? run_of(s, t * s.ni) : 0;
          const int run_hi = split ? run_of(s, (t + 1) * s.ni - 1) : 0;
          const int rc = o * kBM + row;
          RowA rw{false, -1, -1, 0.f};
          const bool whole = !phantom(s, at.rp) && OLIVE_DCHECK(p.dev_status, o >= 0 && o <= s.ph);
          if (kMode == GM_A && whole) {
            // every member's sums (and the target's z_y, P'_y from the member
            // that met it) are published before any member reads them
            rw = load_row_a(p, s, rc);
            if (rw.valid && !member_has_job(s, g, e, at.k)) put_sums(e, at.rp, o, 0.f, -INFINITY);
            __threadfence();
            named_bar_sync(1, kEpi);
            if (threadIdx.x == 0) red_release_add(p.outer_ctr + o, 1u);
          }
          float acc[4][32];
          if (!take_output(acc)) { ok = false; break; }
          if (split) {
            if (!whole) continue;  // a phantom: its rows are never stored
            // the layout is the threads' own (16 bytes of every thread side by
            // side), so stores and loads are whole lines
            auto part = [&](int run) {
              return reinterpret_cast<float4*>(p.tail_acc) +
                     (static_cast<size_t>((run + t) * 2 + s.rank) * g + s.m) * kTailVecs + threadIdx.x;
            };
            if (!OLIVE_DCHECK(p.dev_status, ((run_hi + t) * 2 + s.rank) * g + s.m < p.tail_parts)) {
              ok = false;
              break;
            }
            float4* out = part(s.pg);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              if (ob + 32 * b >= oe) continue;
#pragma unroll
              for (int q = 0; q < 8; ++q)
                out[(8 * b + q) * kEpi] =
                    make_float4(acc[b][4 * q], acc[b][4 * q + 1], acc[b][4 * q + 2], acc[b][4 * q + 3]);
            }
            __threadfence();
            named_bar_sync(1, kEpi);
            bool last = true;
            if (threadIdx.x == 0) {
              last = atomicAdd(p.tail_ctr + (2 * t + s.rank) * g + s.m, 1u) ==
                     static_cast<uint32_t>(run_hi - run_lo);
              __threadfence();
            }
            if (!named_bar_and(1, kEpi, last)) continue;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
#pragma unroll
              for (int c = 0; c < 32; ++c) acc[b][c] = 0.f;
            }
            for (int c = run_lo; c <= run_hi; ++c) {
              const float4* in = part(c);
#pragma unroll
              for (int b = 0; b < 4; ++b) {
                if (ob + 32 * b >= oe) continue;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                  const float4 v = __ldcg(in + (8 * b + q) * kEpi);
                  acc[b][4 * q] += v.x;
                  acc[b][4 * q + 1] += v.y;
                  acc[b][4 * q + 2] += v.z;
                  acc[b][4 * q + 3] += v.w;
                }
              }
            }
          }
          if (kMode == GM_B) {
            store_output(rc < p.V ? rc : -1, acc);
            continue;
          }
          if (kMode == GM_KL) {
            // the divergence gradient: G carried g inv_tau, so d_h_s is the sum
            const int tr = rc < s.n ? p.rows[rc] : -1;
            store_output(tr < p.T ? tr : -1, acc);
            continue;
          }
          // pass A: merge the members' sums, then dH
          if (whole) {
            const uint32_t posts = static_cast<uint32_t>(g * (run_hi - run_lo + 1));
            const bool seen = threadIdx.x == 0 ? wait_counter(p.outer_ctr + o, posts, ctl) : true;
            if (!named_bar_and(1, kEpi, seen)) { ok = false; break; }
          }
          float lse2 = rw.R, mx = -INFINITY;
          if (!p.lse_known && rw.valid) {
            float sum = 0.f;
            // (a split row pair's slots stand one after the other)
            const size_t from = split ? tail_row(run_lo + t, 0) : rc;
            const size_t stride = split ? 2 * kBM : Tpad;
            const float* ps = (split ? p.tail_s : p.part_s) + from;
            const float* pm = (split ? p.tail_m : p.part_m) + from;
            const int count = 2 * g * (run_hi - run_lo + 1);
#pragma unroll 8
            for (int e2 = 0; e2 < count; ++e2) {
              sum += __ldcg(ps + e2 * stride);
              mx = fmaxf(mx, __ldcg(pm + e2 * stride));
            }
            lse2 = rw.R + log2f(sum);
          }
          // (the redo launch, with R = the rows' maxima, never flags)
          const bool row_ok = !rw.valid || p.lse_known || p.redo ||
                              (mx - rw.R <= kRefMax && isfinite(lse2));
          const bool tile_ok = named_bar_and(1, kEpi, row_ok);
          if (!tile_ok) {
            // the reference was too low for some row: the redo launch
            // recomputes this row tile with R = the rows' maxima
            if (s.m == 0) {
              if (rw.valid && !half) p.rmax[rc] = mx;
              if (threadIdx.x == 0) {
                const uint32_t at = atomicAdd(p.redo_list, 1u);
                p.redo_list[1 + at] = static_cast<uint32_t>(o);
              }
            }
          } else {
            const bool has_y = rw.valid && rw.y >= 0 && rw.y < p.V;
            if (s.m == 0 && rw.valid && !half) {
              if (!has_y) atomicOr(p.dev_status, 1 << OLIVE_ERR_TOKEN_RANGE);
              if (p.write_fwd) {
                const float l = lse2 * kLn2;
                const float lp = has_y ? __ldcg(p.zy + rc) - l : NAN;
                p.lse[rw.t] = l;
                p.logp[rw.t] = lp;
                p.nll[rc] = -lp;
              }
            } else if (s.m == 0 && p.write_fwd && !half && rc < s.n) {
              p.nll[rc] = 0.f;  // an index outside the batch: reported, and no term of the loss
            }
            const float scale = fast_exp2(rw.R - lse2);
            // dH = coef (scale acc - W[y]) with the target's term taken out of
            // acc (scale P'_y, P'_y as the MMA saw it) and put back as p_y W[y]:
            // together coef (scale acc + corr W[y]), corr = (p_y - 1) - scale P'_y
            float corr = 0.f;
            if (has_y) {
              const float lnat = p.lse_known ? p.lse_in[rw.t] : lse2 * kLn2;
              corr = expm1f(__ldcg(p.zy + rc) - lnat) - scale * __ldcg(p.pyb + rc);
            }
            const uint4* wy =
                has_y ? reinterpret_cast<const uint4*>(p.W + static_cast<size_t>(rw.y) * p.d + s.c0) : nullptr;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              const int c = ob + 32 * b;
              if (c >= oe) continue;
              const int nv = min(32, oe - c);
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                uint4 w4 = make_uint4(0, 0, 0, 0);
                if (wy && 8 * q < nv) w4 = __ldg(wy + c / 8 + q);
                const __nv_bfloat162* w2 = reinterpret_cast<const __nv_bfloat162*>(&w4);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                  const float2 wf = __bfloat1622float2(w2[u]);
                  float& a0 = acc[b][8 * q + 2 * u];
                  float& a1 = acc[b][8 * q + 2 * u + 1];
                  a0 = s.coef * fmaf(scale, a0, corr * wf.x);
                  a1 = s.coef * fmaf(scale, a1, corr * wf.y);
                }
              }
            }
            store_output(rw.valid ? rw.t : -1, acc);
          }
        }
      }
    }
  }

  tc_fence_before();
  // the pair's MMAs (all complete: the even CTA waited for them) and every
  // access to the peer's barriers are over before either CTA frees its TMEM
  cluster_sync_all();
  if (threadIdx.x == 0 && *abort_flag) atomicOr(p.dev_status, kStatusTimeoutBit);
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

constexpr int kGroupSmem =
    kStages * kStageBytes + kEpiWarps * kWarpSlice + 8 * (2 * kStages + 5) + 128 + kMetaBytes;
static_assert(kGroupSmem <= 227 * 1024, "shared memory budget");

int ring_slots_for(int g) { return 3 * g > 4 ? 3 * g : 4; }

// fewest members a group of `cols` output columns can have, and the most the
// shape search below may pick
int g_min_for(int cols) { return cols > kZN ? (cols + kZN - 1) / kZN : 1; }
int g_hi_for(int cols) { return g_min_for(cols) + g_min_for(cols) / 4 + 1; }

// Groups of g members, run as pair-groups of 2 g CTAs.  g is the member count
// between ceil(cols / 256) and ~1.25 times that which puts the most CTAs to
// work (d = 4096 at 152 SMs: g = 19, four pair-groups fill all 152), the
// smaller g on ties; members hold ceil(cols / g) columns rounded up to 16.
struct GroupShape {
  int g, chunk, ngroups, R;
};

GroupShape group_shape(int cols, int sms) {
  GroupShape gs{0, 0, 0, 0};
  int best_used = 0;
  for (int g = g_min_for(cols); g <= g_hi_for(cols); ++g) {
    const int used = 2 * g * (sms / (2 * g));
    if (used > best_used) {
      best_used = used;
      gs.g = g;
    }
  }
  if (gs.g == 0) return gs;
  gs.chunk = ((cols + gs.g - 1) / gs.g + 15) / 16 * 16;
  gs.ngroups = 2 * (sms / (2 * gs.g));
  gs.R = ring_slots_for(gs.g);
  return gs;
}

// Launches one mode of the kernel on `ctas` CTAs.
template <int kMode>
olive_status launch_mode(const Ctx& c, int sms, int ctas, const GroupMaps& maps, const GroupParams& p) {
  static std::atomic<int> done[kMaxDevices];
  if (!set_smem_once(reinterpret_cast<const void*>(lmhead_group_kernel<kMode>), kGroupSmem, c.device, done))
    return OLIVE_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kGroupSmem;
  cfg.stream = c.stream;
  // clusters of two CTAs (the MMA pairs).  Members of a group wait on one
  // another, so every CTA must be resident at once: the grid is at most one
  // CTA per SM, and the first launch on each device checks that the GPU holds
  // all of its clusters together (cudaOccupancyMaxActiveClusters), else the
  // call is refused.  The launch is not marked cooperative: profilers (ncu)
  // cannot launch cooperative grids of clusters, and a grid that fits starts
  // whole on an idle GPU; if another stream's kernel holds SMs, the waits are
  // bounded and report OLIVE_ERR_TIMEOUT.
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  static std::atomic<int> fits[kMaxDevices];  // clusters the device holds at once, + 1
  const bool cached = c.device >= 0 && c.device < kMaxDevices;
  int held = cached ? fits[c.device].load(std::memory_order_acquire) - 1 : -1;
  if (held < 0) {
    cudaLaunchConfig_t q = cfg;
    q.gridDim = dim3(2 * (sms / 2));
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, lmhead_group_kernel<kMode>, &q) != cudaSuccess) {
      cudaGetLastError();
      return OLIVE_ERR_CUDA;
    }
    held = n;
    if (cached) fits[c.device].store(n + 1, std::memory_order_release);
  }
  if (static_cast<int>(cfg.gridDim.x) > 2 * held) return OLIVE_ERR_UNSUPPORTED_DEVICE;
  if (cudaLaunchKernelEx(&cfg, lmhead_group_kernel<kMode>, maps, p) != cudaSuccess) {
    cudaGetLastError();
    return OLIVE_ERR_CUDA;
  }
  return OLIVE_OK;
}

// output columns one sweep covers: the widest whose fewest members still
// form one pair-group
int sweep_cols_for(int sms) { return (sms / 2) * kZN; }

}  // namespace

// the widest group a launch may form for width d (ring and partials are
// sized for it)
int group_g_max(int64_t d) {
  const int64_t cap = static_cast<int64_t>(sweep_cols_for(kGroupMaxSms));
  return g_hi_for(static_cast<int>(d < cap ? d : cap));
}

int ring_slots(int g) { return ring_slots_for(g); }

// groups a launch forms at most (an even number): as many pair-groups as the
// SMs hold, and no more than a pass has (row pair, inner tile) places, the
// same number in both passes
int group_count_max(int64_t T, int64_t d, int64_t V) {
  const int64_t cap = static_cast<int64_t>(sweep_cols_for(kGroupMaxSms));
  const int gmin = g_min_for(static_cast<int>(d < cap ? d : cap));
  return static_cast<int>(2 * std::min<int64_t>(kGroupMaxSms / (2 * gmin),
                                                ceil_div(T, 2 * kBM) * ceil_div(V, 2 * kBM)));
}

// partial accumulators of split row pairs: slots, and 128 x 256 tiles in all
// (two a member of every slot; the grid's members are one a CTA)
int group_tail_slots(int64_t T, int64_t d, int64_t V) { return group_count_max(T, d, V); }
int64_t group_tail_parts(int64_t T, int64_t d, int64_t V) {
  return std::min<int64_t>(2ll * group_tail_slots(T, d, V) * group_g_max(d), 2 * kGroupMaxSms);
}
size_t group_tail_bytes(int64_t T, int64_t d, int64_t V) {
  return static_cast<size_t>(group_tail_parts(T, d, V)) * kTailVecs * sizeof(float4);
}
// GM_A's sums (and as many maxima) of those slots, in floats
size_t group_tail_sums(int64_t T, int64_t d, int64_t V) {
  return static_cast<size_t>(group_tail_slots(T, d, V)) * 2 * group_g_max(d) * 2 * kBM;
}

size_t group_ring_words(int64_t T, int64_t d, int64_t V) {
  return static_cast<size_t>(group_count_max(T, d, V)) * ring_slots_for(group_g_max(d));
}

size_t group_ring_bytes(int64_t T, int64_t d, int64_t V) { return group_ring_words(T, d, V) * kXTile; }

// counter words of one launch: ready and cons per ring slot, pace per group,
// arrivals per split row tile and member (at most one a CTA)
size_t group_ctr_words(int64_t T, int64_t d, int64_t V) {
  return 2 * group_ring_words(T, d, V) + static_cast<size_t>(group_count_max(T, d, V)) + kGroupMaxSms;
}

int group_sweep_cols(int sms) { return sweep_cols_for(sms < kGroupMaxSms ? sms : kGroupMaxSms); }

namespace {

// The tensor maps of a mode's operands (GM_REF and GM_A share theirs, so a call
// encodes them once: half a microsecond of host time a map).
bool make_maps(GroupMaps* maps, int mode, const void* hc, const void* W, int32_t T, int32_t d, int32_t V,
               const GroupArgs& a) {
  const int64_t Tpad = align_up(static_cast<size_t>(T), kRowAlign);
  const bool rowsA = mode != GM_B;
  const void* zaBase = rowsA ? hc : W;
  const void* zbBase = rowsA ? W : hc;
  const uint64_t zaRows = rowsA ? Tpad : V;
  const uint64_t zbRows = rowsA ? V : Tpad;
  // the ring viewed as rows of 64 bf16 (one 128-byte row of a slice image)
  const uint64_t ring_rows = group_ring_bytes(T, d, V) / 128;
  // inner tiles of 256 vocabulary entries (rows in pass B); each CTA of a pair
  // loads half of them as its B rows
  if (!encode_bf16_2d(&maps->za, zaBase, d, zaRows, 2ull * d, 64, 128) ||
      !encode_bf16_2d(&maps->zb, zbBase, d, zbRows, 2ull * d, 64, kZN / 2) ||
      !encode_bf16_2d(&maps->xb, zbBase, d, zbRows, 2ull * d, 64, 64) ||
      !encode_bf16_2d_plain(&maps->xa, a.ring, 64, ring_rows, 128, 64, 128))
    return false;
  if (mode == GM_KL) {
    if (!encode_bf16_2d(&maps->za2, a.hc2, a.d2, Tpad, 2ull * a.d2, 64, 128) ||
        !encode_bf16_2d(&maps->zb2, a.W2, a.d2, V, 2ull * a.d2, 64, kZN / 2))
      return false;
  } else {
    maps->za2 = maps->za;
    maps->zb2 = maps->zb;
  }
  return true;
}

// mode 0: reference maxima, 1: pass A (lse, logp, dH), 2: pass B (dW), 3:
// divergence gradient (d_hidden = G . W with G from both heads); maps_in: the
// mode's tensor maps, null to make them here
olive_status launch_group(const Ctx& c, int mode, const void* hc, const void* W, int32_t T,
                          int32_t d, int32_t V, const GroupArgs& a, int c_base, int c_end,
                          uint32_t* ring_ctr, const GroupMaps* maps_in = nullptr) {
  const int sms = c.num_sms < kGroupMaxSms ? c.num_sms : kGroupMaxSms;
  GroupShape gs;
  if (mode == GM_REF) {
    gs.g = 1;
    gs.chunk = kZN;
    gs.ngroups = sms / 2 * 2;
    gs.R = 1;
  } else {
    gs = group_shape(c_end - c_base, sms);
    gs.ngroups = std::min(gs.ngroups, group_count_max(T, d, V));
    if (gs.ngroups < 2 || gs.g * gs.ngroups > sms) return OLIVE_ERR_SHAPE;
  }
  GroupMaps own;
  if (!maps_in) {
    if (!make_maps(&own, mode, hc, W, T, d, V, a)) return OLIVE_ERR_CUDA;
    maps_in = &own;
  }
  const GroupMaps& maps = *maps_in;

  GroupParams p = {};
  p.dev_status = a.dev_status;
  p.wait_limit_ns = c.wait_limit_ns;
  p.n_rows = a.n_rows;
  p.rows = a.rows;
  p.targets = a.targets;
  p.W = static_cast<const __nv_bfloat16*>(W);
  p.T = T;
  p.d = d;
  p.V = V;
  p.mode = mode;
  p.g = gs.g;
  p.ngroups = gs.ngroups;
  p.R = gs.R;
  p.chunk = gs.chunk;
  p.c_base = c_base;
  p.c_end = c_end;
  p.reduction = a.reduction;
  p.inv_tau = a.inv_tau;
  p.scale2 = a.inv_tau * kLog2e;
  p.grad_loss = a.grad_loss;
  p.lse_known = a.lse_known;
  p.redo = a.redo;
  p.write_fwd = a.write_fwd;
  p.lse_in = a.lse_in;
  p.rref = a.rref;
  p.rmax = a.rmax;
  p.part_s = a.part_s;
  p.part_m = a.part_m;
  p.zy = a.zy;
  p.pyb = a.pyb;
  p.logp = a.logp;
  p.lse = a.lse;
  p.nll = a.nll;
  p.loss = a.loss;
  p.redo_list = a.redo_list;
  p.outer_ctr = a.outer_ctr + (mode == GM_A && a.redo ? (T + kBM - 1) / kBM : 0);
  p.ring = static_cast<__nv_bfloat16*>(a.ring);
  p.ready = ring_ctr;
  p.cons = ring_ctr ? ring_ctr + static_cast<size_t>(gs.ngroups) * gs.R : nullptr;
  p.pace = ring_ctr ? ring_ctr + 2 * static_cast<size_t>(gs.ngroups) * gs.R : nullptr;
  p.tail_ctr = ring_ctr ? p.pace + gs.ngroups : nullptr;
  p.tail_acc = mode == GM_REF ? nullptr : a.tail_acc;
  p.tail_s = a.tail_s;
  p.tail_m = a.tail_m;
  p.tail_parts = static_cast<int32_t>(group_tail_parts(T, d, V));
  p.tail_slots = group_tail_slots(T, d, V);
  p.out = mode == GM_B ? a.d_W : a.d_hidden;  // GM_KL: d_h_s
  p.out_dtype = a.out_dtype;
  p.ring_tiles = static_cast<int64_t>(group_ring_words(T, d, V));
  p.part_groups = 2 * group_g_max(d);
  p.d2 = a.d2;
  p.reverse = a.reverse;
  p.lse_sc = a.lse_sc;
  p.lse_tc = a.lse_tc;
  p.kl = a.kl;
  p.grad_kl = a.grad_kl;

  const int ctas = gs.ngroups * gs.g;
  switch (mode) {
    case GM_REF: return launch_mode<GM_REF>(c, sms, ctas, maps, p);
    case GM_A: return launch_mode<GM_A>(c, sms, ctas, maps, p);
    case GM_B: return launch_mode<GM_B>(c, sms, ctas, maps, p);
    default: return launch_mode<GM_KL>(c, sms, ctas, maps, p);
  }
}

}  // namespace
}  // namespace olive

namespace olive {

olive_status launch_loss_group(const Ctx& c, const void* hidden, const void* W,
                               const int32_t* targets, const int32_t* rows, const int32_t* n_rows,
                               int32_t T, int32_t d, int32_t V, float inv_tau, int reduction,
                               const float* grad_loss, const float* lse_given, float* logp,
                               float* lse, float* loss, void* d_hidden, void* d_W, int grad_dtype,
                               void* ws, int32_t* dev_status) {
  const bool fwd = lse_given == nullptr;
  const GroupWs w = carve_group(ws, T, d, V);
  const size_t elt = grad_dtype == OLIVE_DTYPE_BF16 ? 2 : 4;
  Prepare q;
  q.gather(hidden, d, w.hc);
  q.fill(d_hidden, elt * T * static_cast<size_t>(d));
  q.fill(w.outer, 4 * w.ctr_words);
  if (fwd) {
    q.fill(logp, sizeof(float) * T);
    q.fill(lse, sizeof(float) * T);
  }
  olive_status st = launch_prepare(c, q, rows, n_rows, T, dev_status);
  if (st != OLIVE_OK) return st;

  GroupArgs a = {};
  a.dev_status = dev_status;
  a.n_rows = n_rows;
  a.rows = rows;
  a.targets = targets;
  a.reduction = reduction;
  a.inv_tau = inv_tau;
  a.grad_loss = grad_loss;
  a.lse_in = fwd ? lse : lse_given;
  a.rref = w.rref;
  a.rmax = w.rmax;
  a.part_s = w.part_s;
  a.part_m = w.part_m;
  a.zy = w.zy;
  a.pyb = w.pyb;
  a.logp = logp;
  a.lse = lse;
  a.nll = w.nll;
  a.redo_list = w.redo;
  a.outer_ctr = w.outer;
  a.ring = w.ring;
  a.tail_acc = w.tail_acc;
  a.tail_s = w.tail_s;
  a.tail_m = w.tail_m;
  a.d_hidden = d_hidden;
  a.d_W = d_W;
  a.out_dtype = grad_dtype;

  GroupMaps ma, mb;
  if (!make_maps(&ma, GM_A, w.hc, W, T, d, V, a) || !make_maps(&mb, GM_B, w.hc, W, T, d, V, a))
    return OLIVE_ERR_CUDA;
  if (fwd && (st = launch_group(c, GM_REF, w.hc, W, T, d, V, a, 0, d, nullptr, &ma)) != OLIVE_OK)
    return st;
  // one sweep of both passes per range of output columns the SMs can hold
  // (every d up to 19456 at 152 SMs takes one)
  const int cols = group_sweep_cols(c.num_sms);
  const size_t rw = group_ctr_words(T, d, V);
  for (int cb = 0; cb < d; cb += cols) {
    const int ce = d - cb < cols ? d : cb + cols;
    if (cb > 0 && cudaMemsetAsync(w.outer, 0, 4 * w.ctr_words, c.stream) != cudaSuccess)
      return OLIVE_ERR_CUDA;
    a.lse_known = (!fwd || cb > 0) ? 1 : 0;
    a.write_fwd = (fwd && cb == 0) ? 1 : 0;
    a.redo = 0;
    if ((st = launch_group(c, GM_A, w.hc, W, T, d, V, a, cb, ce, w.ring_ctr, &ma)) != OLIVE_OK)
      return st;
    if (fwd && cb == 0) {
      a.redo = 1;
      if ((st = launch_group(c, GM_A, w.hc, W, T, d, V, a, cb, ce, w.ring_ctr + rw, &ma)) != OLIVE_OK)
        return st;
      a.redo = 0;
    }
    a.loss = fwd && cb == 0 ? loss : nullptr;
    if ((st = launch_group(c, GM_B, w.hc, W, T, d, V, a, cb, ce, w.ring_ctr + 2 * rw, &mb)) != OLIVE_OK)
      return st;
  }
  return OLIVE_OK;
}

}  // namespace olive

namespace olive {

olive_status launch_kl_group_grad(const Ctx& c, const void* hcs, const void* hct, const void* W_s,
                                  int32_t d_s, const void* W_t, int32_t d_t, const int32_t* rows,
                                  const int32_t* n_rows, int32_t T, int32_t V, float inv_tau,
                                  int reverse, const float* kl, const float* lse_s,
                                  const float* lse_t, const float* grad_kl, void* d_h_s,
                                  int grad_dtype, void* ring, float* tail_acc, uint32_t* ctr,
                                  size_t ctr_words, int32_t* dev_status) {
  const int64_t rt = align_up(static_cast<size_t>(T), kRowAlign) / kRowAlign;
  GroupArgs a = {};
  a.dev_status = dev_status;
  a.n_rows = n_rows;
  a.rows = rows;
  a.inv_tau = inv_tau;
  a.ring = ring;
  a.tail_acc = tail_acc;
  a.d_hidden = d_h_s;
  a.out_dtype = grad_dtype;
  a.hc2 = hct;
  a.W2 = W_t;
  a.d2 = d_t;
  a.reverse = reverse;
  a.lse_sc = lse_s;
  a.lse_tc = lse_t;
  a.kl = kl;
  a.grad_kl = grad_kl;
  uint32_t* ring_ctr = ctr + 3 * rt + 1;
  const int cols = group_sweep_cols(c.num_sms);
  for (int cb = 0; cb < d_s; cb += cols) {
    const int ce = d_s - cb < cols ? d_s : cb + cols;
    if (cb > 0 && cudaMemsetAsync(ctr, 0, 4 * ctr_words, c.stream) != cudaSuccess) return OLIVE_ERR_CUDA;
    const olive_status st = launch_group(c, GM_KL, hcs, W_s, T, d_s, V, a, cb, ce, ring_ctr);
    if (st != OLIVE_OK) return st;
  }
  return OLIVE_OK;
}

}  // namespace olive
