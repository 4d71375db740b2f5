// ee_tree_verify_attn: tree-masked attention of every draft node over the
// paged KV cache plus the tree's own K/V, one layer per call (EfficientEdit
// Sec. III-A: a single target forward pass over (prefix, draft) scores every
// draft token; with a tree, each node sees the prefix and its own root path).
// ee_tree_verify_attn_inplace and ee_chain_verify_attn are the same kernel
// with the draft's K/V in the cache after the context (see kKV below).
//
// Work decomposition (split-KV):
//   - For a (sequence, KV head) the query rows are the g = n_q / n_kv heads of
//     the group times the T tree nodes, row r = node * g + head_in_group, so
//     one K/V tile feeds g * T rows (GQA packing).  A CTA owns 128 rows: the
//     M side of a tcgen05 MMA.
//   - A CTA processes segments: contiguous 128-key tile ranges of one row
//     block.  Uniform launches cut each row block's context into S <= 16
//     chunks of `chunk` keys (a multiple of the 16-token page), one CTA each;
//     the last chunk also processes the tree keys (one 128-key tile, masked by
//     the ancestor bitmask).  Balanced launches give each of one CTA per SM an
//     equal share of all row blocks' tiles (a CTA may finish one row block and
//     start the next); choose_split picks between them.
//   - Every role walks the CTA's segments by itself, tiles numbered through over
//     all of them: nothing but the ring barriers separates one segment from the
//     next.  In a balanced launch the K producer, which runs ahead of all others,
//     builds the work list, decodes each segment and publishes it in a ring.
//   - Keys come in 128-key tiles.  Warps 0 and 2 stream K and V tiles with TMA
//     (one 16-row box per page and 64-dim half, all issued by one elected lane
//     from rows that are the same in every lane; the tree's K/V through a 3-D
//     map) into a 3-stage K ring and a 2-stage V ring; page ids are loaded four
//     tiles ahead into registers.
//   - Q lives in shared memory (asynchronous copies in the 128-byte-swizzled
//     K-major layout TMA gives the K tiles: the softmax warps load the first row
//     block, the Q.K^T warp later ones) and is the A operand of S = Q K^T; TMEM
//     holds three S buffers and O (4 x 128 fp32 columns).
//   - Warp 3 issues S = Q K^T up to three tiles ahead (bf16, fp32 accumulators in
//     TMEM), warp 1 O += P V, each from one elected lane; a tile's Q K^T waits
//     for the P V three tiles before, whose P lives in the same TMEM columns.  Two
//     issuing warps, because a warp that waits for one product's operands would
//     hold back the other's.
//   - P.V runs on bf16 operands: P is split into a bf16 head (the fp32 value
//     rounded to nearest bf16) and a bf16 tail (the exact remainder, rounded
//     to nearest bf16), both written over S in TMEM and used as the MMA A
//     operand; V is read straight from shared memory (MN-major).  P is carried
//     to about 2^-17 relative (fp16 would give 2^-11) and V needs no
//     conversion.  Per column pair the split is two packing conversions and two
//     mixed-type subtractions head - p; the MMA negates the tail back.  The tail's
//     MMAs go first: each MMA cuts O's lowest bits off, which is the error of long
//     sums, and before the head's the segment's O is one tile smaller.
//   - Warps 4-11 own one query row per thread (its TMEM lane), two warps per
//     lane quarter splitting each tile's keys: they read S, mask, keep the
//     running max/sum, write P, and rescale O in TMEM only when a row's max
//     grows by more than 2^8 (the stale max keeps every P <= 256, and the final
//     O / l is unchanged).
//   - Every chunk-CTA writes its unnormalised O rows and (max, sum) from TMEM
//     to its own slot of the workspace (fp32, column-chunk major so that a
//     warp's stores are contiguous; the slots stay in L2).  Once all K slots of
//     a row block are written, the softmax warps of piece k merge 32 / K of the
//     32 four-column chunks of all its rows with log-sum-exp weights and write
//     the fp32 output: one launch, no second pass, and L2 moves the partials
//     several times faster than distributed shared memory does.
//     A segment that is a whole row block writes O / l directly.  The CTAs of
//     a row block learn that all slots are written in one of two ways, chosen
//     by the host:
//       cluster: they form a thread-block cluster and meet at one cluster
//         barrier (release / acquire at cluster scope);
//       cooperative: the launch is cooperative (every CTA resident at once);
//         the row block's 64-bit count grows by 720720 = lcm(1..16) per
//         launch: the V producer reads the count early (a multiple of 720720
//         plus some of this launch's arrivals, never all: this CTA's own is
//         missing; a relaxed load whose value is first used at the end), and
//         after the CTA's partial is stored and its threads have met at a
//         barrier one thread adds 720720 / K with a release reduction and waits
//         (acquire) for the next multiple.  One release per CTA orders all its
//         threads' stores, and nothing resets the count at the end of the
//         kernel.  No GPC packing constraint: K can be any value up to 16, so
//         the grid can cover every SM.  Balanced launches count the pieces of
//         each split row block the same way.
//     Every CTA, also one whose chunk is empty for a short sequence, arrives:
//     every wait before the arrival is bounded.
//   - The next kernel in the stream may launch (programmatic dependent launch)
//     once every CTA has drained its pipeline; triggering earlier lets its
//     CTAs hold SMs that a later wave of this grid still needs.
//
// What bounds it (SM cycles at 2.07 GHz).  Long work: the tile period, about
// 2,000.  A tile's MMAs take 1,536 (24 of 128 x 128 x 16) and about 1,700 with
// their operand waits; the softmax warps, two per sub-partition, walk the rest:
// wait for S 140, load and maxima 400, the pair's exchange 165, exponentials,
// split and stores 1,050 to 1,150, sums and arrival 200.  Tensor pipe 69 % active
// (56 heads, 128 nodes, 32,768 keys, one layer: 148 -> 125 us).  A segment switch
// costs 5,700 more.  Short work: latency.  28 heads, 64 nodes, 4,096 keys, 4 tiles
// a CTA: 13.3 us, of which 2.8 until the first scores, 4 x 1 for the tiles, 1.3 to
// store the partial, 0.9 for its release, 0.6 for the count and 2 to merge.
// Shared-memory traffic per 128-key tile: K 64 KB + V 64 KB (TMA write, MMA
// read) + Q 32 KB (MMA read).
#include "ee_common.cuh"
#include "ee_ptx.cuh"

namespace {

using namespace ee;

constexpr int kThreads = 384;                    // 12 warps, roles below
constexpr int kRows = 128;                       // query rows per CTA (MMA M)
constexpr int kKT = 128;                         // keys per tile (MMA N of Q K^T, K of P V)
constexpr int kD = EE_HEAD_DIM;                  // 128
constexpr int kKST = 3;                          // K ring depth
constexpr int kVST = 2;                          // V ring depth
constexpr int kSB = 3;                           // S buffers in TMEM (Q.K^T runs kSB tiles ahead)
constexpr uint32_t kKVHalf = kKT * 128;          // 16 KB: one 64-dim half of a K or V tile
constexpr uint32_t kKVBytes = 2 * kKVHalf;       // 32 KB
// Context pages of one CTA's share at most: 32,768 keys, 256 tiles.  Nothing in shared
// memory needs the limit; it bounds what one accumulator adds up (the error grows with
// its tiles) and, with kMaxCluster chunks, sets the 262,144 positions the calls accept.
// No longer share has been measured.
constexpr int kMaxCtaPages = 2048;
constexpr int kUnitCost = 3;                      // balanced: a unit's weight beyond its tiles (see the work list)
constexpr int kSegRing = 16;                     // published segments (K runs at most 8 ahead of the softmax)
constexpr int kMaskRing = 8;                     // page-validity masks in flight (K runs at most 6 tiles ahead)
constexpr uint32_t kOffK = 0;
constexpr uint32_t kOffV = kOffK + kKST * kKVBytes;
constexpr uint32_t kOffQ = kOffV + kVST * kKVBytes;  // Q block, 128 rows x 128 bf16, SW128 K-major
constexpr uint32_t kOffBar = kOffQ + kKVBytes;
constexpr uint32_t kNumBars = 2 * kKST + 2 * kVST + 3 * kSB + 5 + kSegRing;
constexpr uint32_t kSmemBytes = 1024 + kOffBar + 8 * kNumBars + 64;
constexpr uint32_t kTmemCols = 512;              // S0 [0,128) S1 [128,256) S2 [256,384) O [384,512)
constexpr uint32_t kColO = 384;
constexpr float kRescaleLog2 = 8.0f;
constexpr int kMaxCluster = 8;                   // portable thread-block cluster size
constexpr int kMaxSplits = ee::kAttnMaxSplits;   // chunks per row block (cooperative launch)
constexpr int kMaxBalSeqs = 512;                 // sequences of a balanced launch
// warp roles; softmax warps 4..11, two per TMEM lane quarter
constexpr int kWarpK = 0, kWarpPv = 1, kWarpV = 2, kWarpQk = 3, kWarpSoft0 = 4;
constexpr int kSoftWarps = 8, kSoftThreads = 32 * kSoftWarps;
// registers per thread: at launch (__launch_bounds__(384, 1)), then by role in a uniform launch
constexpr int kRegsLaunch = 168, kRegsSoft = 208, kRegsOther = 88;
static_assert(kSoftThreads * kRegsSoft + 32 * kWarpSoft0 * kRegsOther <= kThreads * kRegsLaunch, "register split");

static_assert(kRows == ee::kAttnRows, "row block size");
static_assert(kThreads == 32 * (kWarpSoft0 + kSoftWarps), "eight softmax warps, two per TMEM lane quarter");
static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
static_assert(ee::kAttnMlOff == kRows * kD * 4, "partial slot: O rows, then (m, l), then counters");

struct AttnParams {
  const __nv_bfloat16* q;
  const int32_t* block_table;
  const int32_t* ctx_len;
  const int32_t* node_off;
  const uint64_t* anc;
  float* out;
  uint8_t* part;               // per-CTA partial slots (ee::kAttnPartBytes each), S > 1 only
  int32_t* err;
  int num_pages, max_pages, max_ctx, n_q, n_kv, g, total_nodes, max_T, chunk, S;
  int coop;                    // 1: cooperative launch, counters; 0: cluster barrier
  int B;                       // sequences (the balanced mode's work list)
  uint32_t g_inv;              // ceil(2^32 / g) for g > 1 (row -> node without a division), 0 for g = 1
  float scale_log2;
};

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// {hi, lo} rounded to nearest bf16 and packed: lo in bits 0-15, hi in 16-31
__device__ __forceinline__ uint32_t bf16x2_rn(float hi, float lo) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}
// three-input maximum (one instruction on sm_100-family GPUs)
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Merge the 16-byte column chunks [c_lo, c_hi) of a row block's rows (query rows
// row0, ..., `rows` of them) from its K partial slots with log-sum-exp weights
// (Sec. III-A: the scores of one row are normalised over all keys it sees) and
// write the fp32 output.  A piece takes 32 / K chunks of every row, not 128 / K
// rows of every chunk: a block with few rows (a root alone has g of them) then
// keeps all its pieces busy.  The softmax threads do it (nthr of them): thread t
// takes row t % rows and the chunks c_lo + t / rows + k * tpr, where tpr = nthr /
// rows threads share a row: the loads of a warp for one chunk are contiguous, and
// up to kOut chunks' loads from all slots (K <= kMax) are issued before the first
// is used.  Rows without keys have (m, l) = (-inf, 0) and weight 0; their O
// words, never written, are not used.
template <int kMax, int kOut>
__device__ __forceinline__ void merge_rows(const AttnParams& p, size_t slot_a, size_t slot_b, int stride, int K,
                                           int row0, int rows, int c_lo, int c_hi, int o, int hk, int tid,
                                           int nthr) {
  // partial s lives in slot slot_a (s = 0) or slot_b + (s - 1) * stride
  auto slot = [&](int s) -> const uint8_t* {
    return p.part + (s == 0 ? slot_a : slot_b + (size_t)(s - 1) * stride) * kAttnPartBytes;
  };
  const int tpr = nthr / rows;                   // >= 1: rows <= 128 <= nthr
  const int cg = tid / rows, j = tid - cg * rows;
  if (cg >= tpr) return;
  float2 ml[kMax];
#pragma unroll
  for (int s = 0; s < kMax; ++s)
    ml[s] = s < K ? __ldcg(reinterpret_cast<const float2*>(slot(s) + kAttnMlOff) + j)
                  : make_float2(-INFINITY, 0.f);
  const int rrow = row0 + j;
  const int nd = rrow / p.g;
  float4* dst = reinterpret_cast<float4*>(p.out + ((size_t)(o + nd) * p.n_q + hk * p.g + (rrow - nd * p.g)) * kD);
  float M = -INFINITY, il = 0.f, w[kMax];
  for (int c0 = c_lo + cg; c0 < c_hi; c0 += kOut * tpr) {
    float4 v[kOut][kMax];
#pragma unroll
    for (int k = 0; k < kOut; ++k) {
      const int c = c0 + k * tpr;
#pragma unroll
      for (int s = 0; s < kMax; ++s)
        v[k][s] = (c < c_hi && s < K)
                      ? __ldcg(reinterpret_cast<const float4*>(slot(s)) + (size_t)c * kRows + j)
                      : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (c0 == c_lo + cg) {   // the weights, while the first chunks are in flight
#pragma unroll
      for (int s = 0; s < kMax; ++s) M = fmaxf(M, ml[s].x);
      float L = 0.f;
#pragma unroll
      for (int s = 0; s < kMax; ++s) {
        w[s] = ml[s].x == -INFINITY ? 0.f : ex2(ml[s].x - M);
        L += w[s] * ml[s].y;
      }
      il = L == 0.f ? 0.f : 1.f / L;   // NaN scores stay NaN
    }
#pragma unroll
    for (int k = 0; k < kOut; ++k) {
      const int c = c0 + k * tpr;
      if (c >= c_hi) break;
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int s = 0; s < kMax; ++s) {
        if (w[s] == 0.f) continue;
        a.x = fmaf(w[s], v[k][s].x, a.x);
        a.y = fmaf(w[s], v[k][s].y, a.y);
        a.z = fmaf(w[s], v[k][s].z, a.z);
        a.w = fmaf(w[s], v[k][s].w, a.w);
      }
      dst[c] = make_float4(a.x * il, a.y * il, a.z * il, a.w * il);
    }
  }
}
// kX: 16 kX loads per thread in flight
template <int kX>
__device__ __forceinline__ void merge_pieces(const AttnParams& p, size_t slot_a, size_t slot_b, int stride, int K,
                                             int k, int row0, int rows, int o, int hk, int tid, int nthr) {
  const int c_lo = kD / 4 * k / K, c_hi = kD / 4 * (k + 1) / K;   // piece k's chunks
  if (K <= 2) merge_rows<2, 8 * kX>(p, slot_a, slot_b, stride, K, row0, rows, c_lo, c_hi, o, hk, tid, nthr);
  else if (K <= 4) merge_rows<4, 4 * kX>(p, slot_a, slot_b, stride, K, row0, rows, c_lo, c_hi, o, hk, tid, nthr);
  else if (K <= 8) merge_rows<8, 2 * kX>(p, slot_a, slot_b, stride, K, row0, rows, c_lo, c_hi, o, hk, tid, nthr);
  else merge_rows<16, kX>(p, slot_a, slot_b, stride, K, row0, rows, c_lo, c_hi, o, hk, tid, nthr);
}

// A row block's partial that this CTA merges with the other pieces of the same
// row block (balanced mode): the unit, the number of pieces K, this CTA's
// piece index k, and where the pieces' slots are (piece 0 at slot0, piece
// s >= 1 at slot1 + 2 (s - 1)).
struct BalPiece {
  int hk, rb, o, R, K, k, slot0, slot1;
  unsigned long long target;   // the count the row block's pieces raise it to
};
// A split row block's pieces meet at a 64-bit count in the trailer of its first
// partial slot: every launch raises it by kCountGen in all (kCountGen / K per
// piece, a release reduction after the piece's partial is stored), so a count a
// piece reads at any time before its own arrival is a multiple of kCountGen
// plus fewer than K arrivals, and the piece waits (acquire) for the next
// multiple.  The count is never reset; ee_workspace_init
// zeroes it.
constexpr unsigned long long kCountGen = 720720;   // lcm(1..16): K <= 16 divides it

// Where the draft's K/V are (template kKV):
//   kKVTree  -- k_tree / v_tree, one extra 128-key tile after the context;
//   kKVInPlace -- in the cache at positions ctx .. ctx + T - 1 (in-place
//     speculative K/V): a sequence's keys are positions [0, ctx + T) of its
//     pages, and a key at p >= ctx is visible to a row when bit p - ctx of the
//     row's ancestor mask is set;
//   kKVChain -- as kKVInPlace for a linear draft of up to EE_MAX_CHAIN tokens:
//     node i sees positions 0 .. ctx + i (causal), and a row block's keys end
//     at its last node's position.
constexpr int kKVTree = 0, kKVInPlace = 1, kKVChain = 2;

// Chain drafts: 128-key tiles of row block r (its last node's position + 1 keys).
__host__ __device__ inline int chain_rb_tiles(int ctx, int T, int g, int r) {
  const int n_hi = min(T - 1, ((r + 1) * kRows - 1) / g);
  return (ctx + n_hi + 1 + kKT - 1) / kKT;
}

// node of query row r, r / g by a multiplication: with g_inv = (2^32 + e) / g and
// e < g it is exact while r * e < 2^32, and r < EE_MAX_CHAIN * g holds that for
// g <= 1024
__device__ __forceinline__ int row_node(const AttnParams& p, int r) {
  if (p.g == 1) return r;
  return p.g <= 1024 ? (int)__umulhi((uint32_t)r, p.g_inv) : r / p.g;
}

// chain_rb_tiles without the division
__device__ __forceinline__ int chain_tiles(const AttnParams& p, int ctx, int T, int r) {
  return (ctx + min(T - 1, row_node(p, (r + 1) * kRows - 1)) + kKT) / kKT;
}

// One segment: a contiguous range of one row block's tiles, run in the order
// rot, rot + 1, ..., n_tiles - 1, 0, ..., rot - 1.  In a balanced launch the K
// producer, which runs ahead of every other role, decodes the CTA's segments and
// publishes them in a ring in shared memory (one mbarrier each): no CTA barrier
// separates one segment from the next, and the decode (about 2,000 cycles of
// dependent integer work) is off the other roles' path.
struct Seg {
  int b, hk, rb, o, T, ctx;    // sequence, KV head, row block, node offset, nodes, context length
  int k_begin, k_end;          // paged keys
  int n_ctx, n_tiles, rot;     // context tiles, all tiles (the tree tile last), first tile
  bool alone;                  // the segment is its whole row block
  int slot;                    // partial slot (alone: unused)
  int y;                       // balanced: where the segment starts in the work list
  int U0, tiles;               // balanced: the unit's start in the work list and its weight
};

// Shared state of a CTA's work: balanced mode, per sequence (node offset, T,
// context length, tiles), the exclusive prefix of the sequences' work in
// tiles, and (range start, range end, W, N, the share ceil(W / N)).
struct WorkList {
  const int4* seq;
  const int* wpre;
  const int* sched;
};

// The segment of the balanced work list that ends at y (this CTA's range is
// walked from its end); tb: tiles the CTA ran before it.  Whole warp.
template <int kKV>
__device__ __forceinline__ void bal_segment(const AttnParams& p, const WorkList& w, int y, int tb, int lane, Seg& s) {
  constexpr bool kIP = kKV != kKVTree;
  constexpr bool kChain = kKV == kKVChain;
  const int g = p.g;
  // The CTA walks its range from the end: its last segment (the head of a
  // row block) first.  Within a segment the tiles run rotated so that the
  // CTA reads tile x of a row block at about its local time x mod P (P =
  // the share): the CTAs holding other row blocks of the same KV head then
  // read the same K/V tiles at about the same time, and L2 serves the
  // repeats (each KV head's tiles are read by all its row blocks).
  const int x_begin = w.sched[0], x_end = w.sched[1], P = w.sched[4];
  int lo = 0, hi = p.B;   // wpre[lo] <= y - 1 < wpre[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (w.wpre[mid] <= y - 1) lo = mid; else hi = mid;
  }
  s.b = lo;
  const int4 sq = w.seq[lo];
  s.o = sq.x;
  s.T = sq.y;
  s.ctx = sq.z;
  int tiles = sq.w;                              // the unit's weight
  int U0;                                        // its start in the work list
  const int base_w = w.wpre[lo];
  const int nrb_b = (int)((unsigned)(s.T * g + kRows - 1) / kRows);
  if constexpr (kChain) {
    // sq.w = tiles of one KV head's row blocks; row block r has chain_rb_tiles
    const int local = y - 1 - base_w;
    s.hk = (int)((unsigned)local / (unsigned)tiles);
    const int rem = local - s.hk * tiles;
    // the row block holding tile rem: a scan of the row blocks' tile counts, four
    // consecutive ones per lane
    int r = nrb_b - 1, cum = 0, tu = 1;
    for (int r0 = 0, base = 0; r0 < nrb_b; r0 += 128) {
      int t[4], sum = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int rr = r0 + 4 * lane + q;
        t[q] = rr < nrb_b ? chain_tiles(p, s.ctx, s.T, rr) + kUnitCost : 0;
        sum += t[q];
      }
      int incl = sum;
#pragma unroll
      for (int dd = 1; dd < 32; dd <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, dd);
        if (lane >= dd) incl += v;
      }
      int excl = base + incl - sum;
      const unsigned hit = __ballot_sync(0xffffffffu, rem >= excl && rem < excl + sum);
      if (hit) {
        const int src = __ffs(hit) - 1;
        int q = 0;      // (the owner lane's)
#pragma unroll
        for (int k = 0; k < 3; ++k)
          if (q == k && rem >= excl + t[k]) {
            excl += t[k];
            q = k + 1;
          }
        const int tq = q == 0 ? t[0] : q == 1 ? t[1] : q == 2 ? t[2] : t[3];
        r = r0 + 4 * src + __shfl_sync(0xffffffffu, q, src);
        cum = __shfl_sync(0xffffffffu, excl, src);
        tu = __shfl_sync(0xffffffffu, tq, src);
        break;
      }
      base += __shfl_sync(0xffffffffu, incl, 31);
    }
    s.rb = r;
    U0 = base_w + s.hk * tiles + cum;
    tiles = tu;
  } else {
    const int u = (int)((unsigned)(y - 1 - base_w) / (unsigned)tiles);
    s.hk = (int)((unsigned)u / (unsigned)nrb_b);
    s.rb = u - s.hk * nrb_b;
    U0 = base_w + u * tiles;
  }
  const int seg0 = max(U0, x_begin);
  // the unit's first kUnitCost places are no tiles
  const int t0 = max(seg0 - U0 - kUnitCost, 0);
  const int len = max(y - U0 - kUnitCost, 0) - t0;
  const int n_tiles_b = tiles - kUnitCost;
  const int n_ctx_b = kIP ? n_tiles_b : n_tiles_b - 1;   // paged tiles of the unit
  s.k_begin = min(t0, n_ctx_b) * kKT;
  const int unit_span =
      kChain ? s.ctx + min(s.T, row_node(p, (s.rb + 1) * kRows - 1) + 1) : (kIP ? s.ctx + s.T : s.ctx);
  s.k_end = t0 < n_ctx_b ? min(unit_span, min(t0 + len, n_ctx_b) * kKT) : s.k_begin;
  s.n_ctx = s.k_end > s.k_begin ? (s.k_end - s.k_begin + kKT - 1) / kKT : 0;
  s.n_tiles = s.n_ctx + (!kIP && len > 0 && t0 + len == n_tiles_b ? 1 : 0);
  int ph = (tb - t0) % P;
  ph += ph < 0 ? P : 0;
  s.rot = ph < len ? ph : 0;
  s.alone = U0 + kUnitCost >= x_begin && U0 + tiles <= x_end;
  s.U0 = U0;
  s.tiles = tiles;
  // a piece starts the CTA's range (slot 2c) or ends it (slot 2c + 1)
  s.slot = 2 * (int)blockIdx.x + (seg0 > x_begin ? 1 : 0);
  s.y = seg0;
}

// The one (row block, chunk) of a CTA of a uniform launch; false when the row
// block has no work (uniform over the row block's CTAs).
template <int kKV>
__device__ __forceinline__ bool uni_segment(const AttnParams& p, bool report, Seg& s) {
  constexpr bool kIP = kKV != kKVTree;
  constexpr bool kChain = kKV == kKVChain;
  constexpr int kMaxT = kChain ? EE_MAX_CHAIN : EE_MAX_TREE;
  s.b = blockIdx.z;
  s.hk = blockIdx.y;
  s.rb = blockIdx.x / p.S;                     // the S chunks of a row block are consecutive
  const int split = blockIdx.x - s.rb * p.S;
  s.o = p.node_off[s.b];
  s.T = p.node_off[s.b + 1] - s.o;
  s.ctx = p.ctx_len[s.b];
  const bool bad_tree = s.T < 1 || s.T > kMaxT || s.T > p.max_T || s.o < 0 || s.o + s.T > p.total_nodes;
  report = report && blockIdx.x == 0 && s.hk == 0;
  if (bad_tree && report) flag_error(p.err, EE_DEVERR_TREE);
  if (bad_tree || s.rb * kRows >= s.T * p.g) return false;
  if (s.ctx < 0 || s.ctx > p.max_ctx) {
    if (report) flag_error(p.err, EE_DEVERR_CTX);
    s.ctx = s.ctx < 0 ? 0 : p.max_ctx;
  }
  // everything above is uniform over the row block's CTAs; from here on every
  // CTA reaches the merge synchronisation
  // paged keys of the row block (chain: up to its last node's position)
  const int span = kChain ? s.ctx + min(s.T, row_node(p, (s.rb + 1) * kRows - 1) + 1) : (kIP ? s.ctx + s.T : s.ctx);
  const int S = attn_splits_for(span, p.chunk);  // chunks this sequence uses, <= p.S
  const bool active = split < S;
  s.k_begin = split * p.chunk;
  s.k_end = active ? min(span, s.k_begin + p.chunk) : s.k_begin;
  s.n_ctx = s.k_end > s.k_begin ? (s.k_end - s.k_begin + kKT - 1) / kKT : 0;
  s.n_tiles = s.n_ctx + (!kIP && active && split == S - 1 ? 1 : 0);
  s.rot = 0;
  s.alone = p.S == 1;
  s.slot = (int)(((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x);
  s.y = 0;
  return true;
}

// Query rows of the segment's row block into shared memory as the A operand of
// Q.K^T: 128 rows x 128 bf16 in two 64-column slabs, 128-byte swizzled K-major
// (the layout TMA gives the K tiles): 16-byte chunk j of row r at slab (j / 8),
// (r / 8) * 1024 + (r % 8) * 128 + ((j % 8) ^ (r % 8)) * 16; rows past R are
// zero.  Rows r0, r0 + kStep, ... (kCount of them; a half-warp copies one
// 256-byte row, so kStep counts rows from one copy of a lane to its next), as
// asynchronous copies, all in flight before the wait.  The (node, head) of a row
// advances by additions: one warp's instruction chain sets the time of the load.
template <int kStep, int kCount>
__device__ __forceinline__ void load_q(const AttnParams& p, const Seg& s, uint32_t sQ, int r0, int lane) {
  const int g = p.g;
  const int j = lane & 15;
  int rq = r0 + (lane >> 4);                     // 0..127
  const int left = s.T * g - s.rb * kRows;       // rows of the block that exist
  const int rr = s.rb * kRows + rq;
  const int nd = row_node(p, rr);
  int h = rr - nd * g;
  const char* base =
      reinterpret_cast<const char*>(p.q + ((size_t)s.o * p.n_q + s.hk * g) * kD + 8 * j);
  // (node, head) as a row number, scaled to bytes in 64 bits: 2048 nodes of more than
  // 8192 heads pass 4 GiB (2^32 rows would be 1 TB)
  uint32_t row = (uint32_t)nd * p.n_q + h;
  const int dn = kStep / g, dh = kStep - dn * g;          // kStep rows = dn nodes and dh heads
  const uint32_t step = (uint32_t)dn * p.n_q + dh, wrap = (uint32_t)(p.n_q - g);
  const uint32_t dst = sQ + (j >> 3) * kKVHalf;
#pragma unroll 8   // (all 64 rows of a later row block: the balanced kernels spill)
  for (int k = 0; k < kCount; ++k) {
    const bool in = rq < left;
    cp_async16(dst + (rq >> 3) * 1024 + (rq & 7) * 128 + (((j & 7) ^ (rq & 7)) << 4),
               base + (size_t)(in ? row : 0u) * (kD * 2), in ? 16u : 0u);
    rq += kStep;
    row += step;
    h += dh;
    if (h >= g) {
      h -= g;
      row += wrap;
    }
  }
  cp_async_wait_all();
  fence_async_smem();   // generic-proxy writes, read by the tensor core
  __syncwarp();
}

// kBal: balanced work list (else one (row block, chunk) per CTA).
template <bool kBal, int kKV>
__global__ void __launch_bounds__(kThreads, 1)
attn_tc_kernel(const __grid_constant__ CUtensorMap tmKc, const __grid_constant__ CUtensorMap tmVc,
               const __grid_constant__ CUtensorMap tmKt, const __grid_constant__ CUtensorMap tmVt,
               const AttnParams p) {
  constexpr bool kIP = kKV != kKVTree;       // draft K/V in the cache
  constexpr bool kChain = kKV == kKVChain;
  constexpr int kMaxT = kChain ? EE_MAX_CHAIN : EE_MAX_TREE;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  __shared__ int s_kissued[kKST], s_vissued[kVST];
  __shared__ uint32_t s_xmax[2][2][kRows];          // [tile parity][half][row]: softmax pair exchange
  __shared__ float s_xl[2][kRows];                  // [half][row]: final row sums
  __shared__ int s_xok[2][4][2];                    // [tile parity][lane quarter][half]: "this half's wait ended well"
  __shared__ uint32_t s_mask[kMaskRing];            // per tile: 16-row blocks with keys in a valid page
  __shared__ int4 s_seq[kBal ? kMaxBalSeqs : 1];
  __shared__ int s_wpre[kBal ? kMaxBalSeqs + 1 : 1];
  __shared__ int s_sched[5];                        // balanced: range start, range end, W, N, ceil(W / N)
  __shared__ Seg s_seg[kBal ? kSegRing : 1];        // balanced: published segments (n_tiles 0: no more)
  __shared__ BalPiece s_pc[2];                      // this CTA's pieces of split row blocks
  __shared__ int s_npc;
  __shared__ int2 s_uni;                            // uniform: the row block's node offset and rows

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t sbase = smem_u32(smem);
  const uint32_t sK = sbase + kOffK, sV = sbase + kOffV, sQ = sbase + kOffQ;
  const uint32_t bar0 = sbase + kOffBar;
  const uint32_t k_full = bar0, k_empty = k_full + 8 * kKST;
  const uint32_t v_full = k_empty + 8 * kKST, v_empty = v_full + 8 * kVST;
  const uint32_t s_full = v_empty + 8 * kVST, p_full = s_full + 8 * kSB, pv_done = p_full + 8 * kSB;
  const uint32_t drain = pv_done + 8 * kSB, q_ready = drain + 16, q_empty = q_ready + 8, o_free = q_empty + 8;
  const uint32_t seg_full = o_free + 8;

  // on-chip set-up first: it touches no global memory, so it overlaps the end
  // of the previous kernel in the stream
  if (threadIdx.x == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmKc)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmVc)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmKt)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmVt)) : "memory");
    s_abort = 0;
    s_npc = 0;
    s_uni = make_int2(0, 0);
    for (int i = 0; i < kKST; ++i) {
      mbar_init(k_full + 8 * i, 1);
      mbar_init(k_empty + 8 * i, 1);
      s_kissued[i] = -1;
    }
    for (int i = 0; i < kVST; ++i) {
      mbar_init(v_full + 8 * i, 1);
      mbar_init(v_empty + 8 * i, 1);
      s_vissued[i] = -1;
    }
    for (int i = 0; i < kSB; ++i) {
      mbar_init(s_full + 8 * i, 2);
      mbar_init(p_full + 8 * i, kSoftWarps);
      mbar_init(pv_done + 8 * i, 1);
    }
    mbar_init(drain, 1);
    mbar_init(drain + 8, 1);
    mbar_init(q_ready, kSoftWarps);
    mbar_init(q_empty, 1);
    mbar_init(o_free, kSoftWarps);
    for (int i = 0; i < kSegRing; ++i) mbar_init(seg_full + 8 * i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (warp == kWarpPv) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&s_tmem)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);

  pdl_wait();   // no global access before the previous kernel's writes are visible
  const int g = p.g;

  // ---- balanced mode: the shared work list ---------------------------------------
  // Work is counted in 128-key tiles: sequence b brings n_kv x nrb_b units (a
  // KV head's row block) of ceil(ctx_b / 128) context tiles + 1 tree tile, and
  // each unit starts with kUnitCost places that are no tiles: a CTA that ends one
  // unit and starts the next waits for the last P V, stores a partial and starts
  // a new pipeline, 5,700 cycles or nearly three tiles more than its neighbours.
  // Units are ordered sequence, KV head, row block; CTA c takes the places
  // [c W / N, (c + 1) W / N) of that order, so a CTA may finish one unit and
  // start the next (at most two of its segments are pieces of split units).
  // N is capped so that every CTA gets at least m = max(2, ceil((t_max +
  // kUnitCost) / 13)) places, which bounds the pieces of any unit by 15.
  // The K producer builds it: lane l takes sequences [per l, per l + per), per = ceil(B / 32).
  if constexpr (kBal) {
    if (warp == kWarpK) {
      const int per = (p.B + 31) >> 5;     // sequences of a lane
      int wsum = 0, asum = 0, tmax = 0;
      for (int k = 0; k < per; ++k) {      // (clamped indices)
        const int bb = min(lane * per + k, p.B - 1);
        s_seq[lane * per + k] = make_int4(p.node_off[bb], p.node_off[bb + 1], p.ctx_len[bb], 0);
      }
      __syncwarp();
      // chain drafts: one KV head's tiles are a sum over its row blocks; for a
      // few sequences the warp sums each one's row blocks 32 at a time (stored
      // in .w), otherwise each lane walks its own sequences' row blocks
      const bool coop = kChain && p.B <= 64;
      if (coop) {
        for (int bb = 0; bb < p.B; ++bb) {
          const int4 sq = s_seq[bb];
          const int Tb = sq.y - sq.x;
          const bool bad = Tb < 1 || Tb > kMaxT || Tb > p.max_T || sq.x < 0 || sq.x + Tb > p.total_nodes;
          const int c = min(max(sq.z, 0), p.max_ctx);
          int acc = 0;
          if (!bad)
            for (int r = lane; r < (Tb * g + kRows - 1) / kRows; r += 32) acc += chain_tiles(p, c, Tb, r) + kUnitCost;
          acc = __reduce_add_sync(0xffffffffu, acc);
          __syncwarp();
          if (lane == 0) s_seq[bb].w = acc;
        }
        __syncwarp();
      }
      for (int k = 0; k < per; ++k) {
        const int bb = lane * per + k;
        if (bb < p.B) {
          int wl = 0;
          const int4 sq = s_seq[bb];
          const int Tb = sq.y - sq.x;
          const bool bad = Tb < 1 || Tb > kMaxT || Tb > p.max_T || sq.x < 0 || sq.x + Tb > p.total_nodes;
          if (bad && blockIdx.x == 0) flag_error(p.err, EE_DEVERR_TREE);
          int c = sq.z;
          if (c < 0 || c > p.max_ctx) {
            if (blockIdx.x == 0) flag_error(p.err, EE_DEVERR_CTX);
            c = c < 0 ? 0 : p.max_ctx;
          }
          // tiles of a unit (chain: of one KV head's row blocks, whose lengths differ)
          const int nrb_b = bad ? 1 : (Tb * g + kRows - 1) / kRows;
          int tiles = (kIP ? (c + (bad ? 1 : Tb) + kKT - 1) / kKT : (c + kKT - 1) / kKT + 1) + kUnitCost;
          int unit_max = tiles;
          if constexpr (kChain) {
            tiles = sq.w;
            if (!coop) {
              tiles = 0;
              for (int r = 0; r < nrb_b && !bad; ++r) tiles += chain_tiles(p, c, Tb, r) + kUnitCost;
            }
            unit_max = bad ? 1 : chain_tiles(p, c, Tb, nrb_b - 1) + kUnitCost;
          }
          if (!bad) {
            wl = p.n_kv * (kChain ? 1 : nrb_b) * tiles;
            asum += wl - p.n_kv * nrb_b * kUnitCost;
            tmax = max(tmax, unit_max);
          }
          s_seq[bb] = make_int4(sq.x, bad ? 0 : Tb, c, tiles);
          s_wpre[bb] = wsum;               // within the lane
          wsum += wl;
        }
      }
      // warp-wide exclusive scan of the lanes' sums (lane order is sequence order)
      int incl = wsum;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += v;
      }
      const int W = __shfl_sync(0xffffffffu, incl, 31);
      const int tmax_all = __reduce_max_sync(0xffffffffu, tmax);
      const int A = __reduce_add_sync(0xffffffffu, asum);   // tiles
      for (int k = 0; k < per; ++k) {
        const int bb = lane * per + k;
        if (bb < p.B) s_wpre[bb] += incl - wsum;
      }
      if (lane == 0) {
        const int m = max(2, (tmax_all + 12) / 13);
        const int N = W > 0 ? min((int)gridDim.x, max(1, A / m)) : 0;
        const bool mine = (int)blockIdx.x < N;
        s_sched[0] = mine ? (int)blockIdx.x * W / N : 0;
        s_sched[1] = mine ? ((int)blockIdx.x + 1) * W / N : 0;
        s_sched[2] = W;
        s_sched[3] = N;
        s_sched[4] = N > 0 ? (W + N - 1) / N : 1;
        s_wpre[p.B] = W;
      }
      __syncwarp();
    }
  }

  const WorkList wlist{s_seq, s_wpre, s_sched};
  // wait outcomes are made warp-uniform: what follows is warp-collective
  auto wait = [&](uint32_t bar, int use) -> bool {
    return __all_sync(0xffffffffu, mbar_wait(bar, (uint32_t)(use & 1), &s_abort));
  };
  // The CTA's segments: `first` starts the walk, `next` moves to the following
  // segment (tiles before it: tb, segments before it: nseg).
  Seg sg;
  int tb = 0, nseg = 0;
  // balanced, the K producer: segment n (ending at y, tb0 tiles before it),
  // decoded and published
  auto publish = [&](int n, int y, int tb0, Seg& o) {
    o.n_tiles = 0;
    while (y > s_sched[0]) {
      bal_segment<kKV>(p, wlist, y, tb0, lane, o);
      if (o.n_tiles > 0) break;   // (else only the unit's first places: no tile)
      y = o.y;
    }
    if (lane == 0) {
      s_seg[kBal ? n % kSegRing : 0] = o;
      mbar_arrive(seg_full + 8 * (n % kSegRing));
    }
    __syncwarp();
  };
  // the other roles: segment nseg, received
  auto receive = [&]() -> bool {
    if (!wait(seg_full + 8 * (nseg % kSegRing), nseg / kSegRing)) return false;
    sg = s_seg[kBal ? nseg % kSegRing : 0];
    return sg.n_tiles > 0;
  };
  if constexpr (kBal) {
    // the first segment meets a CTA barrier: eleven warps polling an mbarrier would
    // take the issue slots the K warp builds and decodes with
    if (warp == kWarpK) publish(0, s_sched[1], 0, sg);
    __syncthreads();
  }
  auto first = [&](bool report) -> bool {
    if constexpr (kBal) {
      if (warp != kWarpK) sg = s_seg[0];
      return sg.n_tiles > 0;
    } else {
      return uni_segment<kKV>(p, report, sg);
    }
  };
  auto next = [&]() -> bool {
    if constexpr (kBal) {
      tb += sg.n_tiles;
      ++nseg;
      return receive();
    } else {
      return false;
    }
  };
  // the same without a wait: segment nseg + 1 is known to be published
  auto next_published = [&]() -> bool {
    if constexpr (kBal) {
      tb += sg.n_tiles;
      ++nseg;
      sg = s_seg[nseg % kSegRing];
      return sg.n_tiles > 0;
    } else {
      return false;
    }
  };

  // Uniform launches: the merge keeps 32 loads a thread in flight, so the softmax
  // warps, which run it, take registers from the others (the shares add up to the
  // launch's).  A balanced launch's producers need theirs: with 88 registers the K
  // warp spills and the tile period grows (33B-shaped layer 129.5 -> 134 us).
  if (warp < kWarpSoft0) {
    if constexpr (!kBal) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsOther));
    if (warp == kWarpK || warp == kWarpV) {
      // ---------------- TMA producers: warp 0 streams K, warp 2 streams V ----------------
      // Ring slots and phases count the CTA's tiles over all its segments.  Lane l
      // holds the page id of 16-row block l % 8 of the (l / 8)-th of four
      // consecutive tiles, loaded four tiles ahead; one elected lane issues the
      // tile's 16 boxes (eight blocks, two 64-dim halves) from warp-uniform rows.
      // Boxes issued by different lanes are serialised one by one: 1100 cycles a
      // tile (and the K stream behind the tensor pipe), against about 300.
      const bool isK = warp == kWarpK;
      const int nst = isK ? kKST : kVST;
      const uint32_t full0 = isK ? k_full : v_full, empty0 = isK ? k_empty : v_empty;
      const uint32_t ring = isK ? sK : sV;
      const CUtensorMap* mc = isK ? &tmKc : &tmVc;
      const CUtensorMap* mt = isK ? &tmKt : &tmVt;
      int* issued = isK ? s_kissued : s_vissued;
      int32_t early = -1;
      unsigned long long u_count = 0;
      if constexpr (!kBal) {
        // the chunk's first page ids (and the row block's count), issued beside the
        // node range and context length so that the round trips overlap
        const int split = (int)(blockIdx.x % p.S);
        const int pg = split * (p.chunk / EE_PAGE) + lane;
        if (pg < p.max_pages) early = ld_nc_pinned(p.block_table + (size_t)blockIdx.z * p.max_pages + pg);
        if (!isK && lane == 0 && p.coop && p.S > 1)
          u_count = ld_relaxed64(reinterpret_cast<const unsigned long long*>(
              p.part +
              (((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x - split) * kAttnPartBytes +
              kAttnCntOff));
      }
      bool more = first(isK && lane == 0);
      if constexpr (!kBal) {
        // the count any time before this CTA's own arrival is a multiple of
        // kCountGen plus the arrivals of this launch so far, never all of them
        if (!isK && lane == 0 && more) {
          s_uni = make_int2(sg.o, sg.T * g);
          s_pc[0].target = (u_count / kCountGen + 1) * kCountGen;
        }
      }
      bool go = true;
      // page ids of tiles 4 c .. 4 c + 3 of the segment's order (INT_MIN: no keys
      // there), one predicated load that nothing waits for before the ids are used
      auto fetch = [&](const Seg& sg, int c) -> int32_t {
        const int t = 4 * c + (lane >> 3);
        const int i = t + sg.rot < sg.n_tiles ? t + sg.rot : t + sg.rot - sg.n_tiles;
        const int pos = sg.k_begin + i * kKT + 16 * (lane & 7);
        const bool need = t < sg.n_tiles && i < sg.n_ctx && pos < sg.k_end;
        if (!kBal && c == 0) return need ? early : INT32_MIN;
        int32_t v = INT32_MIN;
        if (need) v = ld_nc_pinned(p.block_table + (size_t)sg.b * p.max_pages + pos / EE_PAGE);
        return v;
      };
      // balanced, the K producer: the next segment (decoded and published, its first
      // page ids on the way, while this one's tiles wait for ring slots)
      int32_t nx_ids = INT32_MIN;
      while (more && go) {
        int32_t ids = kBal && isK && nseg > 0 ? nx_ids : fetch(sg, 0), ids_next = INT32_MIN;
        for (int t = 0; t < sg.n_tiles; ++t) {
          if ((t & 3) == 0) {
            if (t > 0) ids = ids_next;
            ids_next = fetch(sg, (t >> 2) + 1);
          }
          const int tg = tb + t;
          const int st = tg % nst, use = tg / nst;
          // the tile's eight blocks, the same in every lane: first cache row, -EE_PAGE
          // without a page; need8: the blocks that hold keys
          const int i = t + sg.rot < sg.n_tiles ? t + sg.rot : t + sg.rot - sg.n_tiles;   // the segment's tile
          const int left = sg.k_end - (sg.k_begin + i * kKT);
          const unsigned need8 = i >= sg.n_ctx ? 0u : left >= kKT ? 0xFFu : (1u << ((left + 15) >> 4)) - 1u;
          int row[kKT / 16];
          unsigned okm = 0u;      // bit i: block i has keys in a valid page
          bool bad = false;
#pragma unroll
          for (int q = 0; q < kKT / 16; ++q) {
            const int32_t id = __shfl_sync(0xffffffffu, ids, 8 * (t & 3) + q);
            const bool ok = id >= 0 && id < p.num_pages;
            row[q] = ok ? (id * p.n_kv + sg.hk) * EE_PAGE : -EE_PAGE;
            okm |= ok ? 1u << q : 0u;
            bad |= !ok && (need8 >> q & 1u);
          }
          if (isK && bad && lane == 0) flag_error(p.err, EE_DEVERR_PAGE);
          go = wait(empty0 + 8 * st, use + 1);
          if (!go) break;
          const uint32_t full = full0 + 8 * st;
          const uint32_t dst = ring + st * kKVBytes;
          if (elect_one()) {
            if (isK) s_mask[tg % kMaskRing] = okm;
            mbar_expect_tx(full, 2 * kKVHalf);
            if (i < sg.n_ctx) {
              // every 16-row block is written: blocks without a loaded page are read at
              // row -16, wholly out of range, which the TMA unit fills with zeros (a
              // stale V row would turn 0 * P into NaN)
#pragma unroll
              for (int q = 0; q < kKT / 16; ++q) {
                tma_load_2d(dst + q * 2048, mc, full, 0, row[q]);
                tma_load_2d(dst + kKVHalf + q * 2048, mc, full, 64, row[q]);
              }
            } else {
              tma_load_3d(dst, mt, full, 0, sg.hk, sg.o);
              tma_load_3d(dst + kKVHalf, mt, full, 64, sg.hk, sg.o);
            }
          }
          __syncwarp();
          if (lane == 0) issued[st] = use;
          if constexpr (kBal) {
            if (isK && t == min(kKST - 1, sg.n_tiles - 1)) {
              Seg nx;
              publish(nseg + 1, sg.y, tb + sg.n_tiles, nx);
              nx_ids = fetch(nx, 0);
            }
            // the piece of a split row block, and its count as read before this
            // CTA's own arrival
            if (!isK && t == min(1, sg.n_tiles - 1) && !sg.alone && lane == 0 && s_npc < 2) {
              // the CTAs holding the unit's first and last tiles, piece 0's slot
              const int W = s_sched[2], N = s_sched[3];
              const int c0 = ((sg.U0 + kUnitCost + 1) * N - 1) / W, c1 = ((sg.U0 + sg.tiles) * N - 1) / W;
              const int slot0 = 2 * c0 + (sg.U0 > c0 * W / N ? 1 : 0);
              const unsigned long long c = ld_relaxed64(
                  reinterpret_cast<const unsigned long long*>(p.part + (size_t)slot0 * kAttnPartBytes + kAttnCntOff));
              s_pc[s_npc] = BalPiece{sg.hk, sg.rb, sg.o, sg.T * g, c1 - c0 + 1, (int)blockIdx.x - c0,
                                     slot0, 2 * (c0 + 1), (c / kCountGen + 1) * kCountGen};
              s_npc = s_npc + 1;
            }
          }
        }
        more = kBal && isK ? next_published() : next();
      }
    } else if (warp == kWarpQk) {
      // ---------------- S = Q K^T, up to kSB tiles ahead of P.V ----------------
      // One warp issues Q.K^T and another P.V: while one waits for its operands (a
      // ready mbarrier still costs about 100 cycles to see), the other's MMAs keep
      // the tensor pipe busy.  The whole warp walks the loop and one elected lane
      // issues, every descriptor an offset from a uniform base.
      const uint32_t id_qk = idesc_f16(kRows, kKT, 1, 1, 0);
      const uint64_t dq = smem_desc_sw128(__shfl_sync(0xffffffffu, sQ, 0));
      const uint64_t dk0 = smem_desc_sw128(__shfl_sync(0xffffffffu, sK, 0));
      bool go = true;
      for (bool more = first(false); more && go; more = next()) {
        if (sg.n_tiles == 0) continue;
        if (nseg == 0) {
          go = wait(q_ready, 0);       // the softmax warps load the first row block
        } else {
          // the previous segment's last Q.K^T has read its rows; the load runs while
          // its last kSB tiles are in the softmax
          go = wait(q_empty, nseg - 1);
          if (go) load_q<2, kRows / 2>(p, sg, sQ, 0, lane);
        }
        tc_fence_after();
        for (int t = 0; t < sg.n_tiles && go; ++t) {
          const int tg = tb + t;
          const int st = tg % kKST, sb = tg % kSB;
          if (tg >= kSB) go = wait(pv_done + 8 * sb, tg / kSB - 1);   // S buffer's P consumed
          go = go && wait(k_full + 8 * st, tg / kKST);
          if (!go) break;
          tc_fence_after();
          if (elect_one()) {
            const uint64_t dk = dk0 + (uint64_t)(st * (kKVBytes >> 4));
#pragma unroll
            for (int kk = 0; kk < kD / 16; ++kk) {
              const uint64_t off = ((kk >> 2) * kKVHalf + (kk & 3) * 32) >> 4;
              tc_mma(tmem + sb * kKT, dq + off, dk + off, id_qk, kk > 0 ? 1u : 0u);
            }
            tc_commit(s_full + 8 * sb);
            tc_commit(k_empty + 8 * st);
            if (t == sg.n_tiles - 1) tc_commit(q_empty);
            mbar_arrive(s_full + 8 * sb);   // releases the tile's page mask (acquired with k_full)
          }
          __syncwarp();
        }
      }
    } else if (warp == kWarpPv) {
      // ---------------- O += P V ----------------
      const uint32_t id_pv = idesc_f16(kRows, kD, 1, 1, 1);
      const uint64_t dv0 = smem_desc_sw128_mn(__shfl_sync(0xffffffffu, sV, 0), kKVHalf, 1024);
      bool go = true;
      int filled = 0;    // segments with tiles so far
      for (bool more = first(false); more && go; more = next()) {
        if (sg.n_tiles == 0) continue;
        // the softmax has read the previous segment's O
        if (filled > 0) go = wait(o_free, filled - 1);
        ++filled;
        for (int t = 0; t < sg.n_tiles && go; ++t) {
          const int tg = tb + t;
          const int st = tg % kVST, sb = tg % kSB;
          go = wait(v_full + 8 * st, tg / kVST) && wait(p_full + 8 * sb, tg / kSB);
          if (!go) break;
          tc_fence_after();
          if (elect_one()) {
            const uint32_t pa = tmem + sb * kKT;       // bf16 P head: cols 0..63, tail: 64..127
            const uint64_t dv = dv0 + (uint64_t)(st * (kKVBytes >> 4));
#pragma unroll
            for (int part = 1; part >= 0; --part)    // the tail first
#pragma unroll
              for (int j = 0; j < kKT / 16; ++j)
                tc_mma_ts(tmem + kColO, pa + 64 * part + 8 * j, dv + (uint64_t)(j * (2048 >> 4)),
                          part ? (id_pv | kIdescNegA) : id_pv,
                          (t > 0 || part == 0 || j > 0) ? 1u : 0u);
            tc_commit(pv_done + 8 * sb);
            tc_commit(v_empty + 8 * st);
          }
          __syncwarp();
        }
      }
    }

    // ---- producers and MMA issuers: drain on abort, free TMEM ----------------------
    tc_fence_before();
    __syncthreads();
    pdl_allow_next();   // this grid's pipeline is done: the next kernel may take SMs as they free
    if (s_abort) {
      if (threadIdx.x == 0) {
        flag_error(p.err, EE_DEVERR_TIMEOUT);
        // TMA copies still in flight land before the rings are reused
        for (int st = 0; st < kKST; ++st)
          if (s_kissued[st] >= 0) mbar_wait_plain(k_full + 8 * st, (uint32_t)(s_kissued[st] & 1));
        for (int st = 0; st < kVST; ++st)
          if (s_vissued[st] >= 0) mbar_wait_plain(v_full + 8 * st, (uint32_t)(s_vissued[st] & 1));
      }
      // MMAs still in flight: each issuing warp's elected lane commits and waits
      if ((warp == kWarpPv || warp == kWarpQk) && elect_one()) {
        const uint32_t dr = drain + (warp == kWarpQk ? 8 : 0);
        tc_commit(dr);
        mbar_wait_plain(dr, 0);
      }
      asm volatile("bar.sync 1, %0;" ::"n"(32 * kWarpSoft0) : "memory");
    }
    if (warp == kWarpPv) {
      tc_fence_after();
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(kTmemCols)
                   : "memory");
    }
    if (!kBal && s_uni.y > 0 && p.S > 1 && !p.coop) cluster_sync();   // with the softmax warps' below
    return;
  }
  if constexpr (!kBal) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoft));
  // ---------------- softmax: one query row and half of every tile per thread ----------------
  // Warps w and w + 4 share TMEM lane quarter w & 3 (32 query rows); half hf
  // of the pair takes keys [64 hf, 64 hf + 64) of every tile and O columns
  // [64 hf, 64 hf + 64).  The pair agrees on each tile's row maximum through
  // shared memory at a 64-thread named barrier, so both halves take the same
  // rescale decisions; each keeps the sum over its own keys, and the two sums
  // are added (half 0 first) at the end.  Two warps per sub-partition hide
  // each other's latencies.  Every exit, from the tile loop and from the walk
  // of the segments, happens right after the pair barrier and on a decision both
  // warps share: a bounded wait can end differently in the two (one sees the
  // abort flag, the other its barrier complete), and a warp that left alone
  // would leave its partner at the pair barrier for good.
  const int qd = warp & 3;
  const int hf = (warp - kWarpSoft0) >> 2;
  const uint32_t pair_bar = 2 + qd;
  const int r = qd * 32 + lane;                     // == TMEM lane of this quarter
  const uint32_t tl = tmem + ((uint32_t)(qd * 32) << 16);
  const float sl2 = p.scale_log2;
  bool ok = true;
  bool loaded = false;
  for (bool more = first(false); more && ok; more = next_published()) {
    const int R = sg.T * g;
    const int rr = sg.rb * kRows + r;
    const bool vrow = rr < R;
    const int node = vrow ? row_node(p, rr) : 0;
    if (!loaded) {   // the first row block's Q: each softmax warp copies 16 rows
      load_q<2 * kSoftWarps, kRows / 2 / kSoftWarps>(p, sg, sQ, 2 * (warp - kWarpSoft0), lane);
      if (lane == 0) mbar_arrive(q_ready);
      loaded = true;
    }
    // this half's tree keys (separate tree tile), or the row's whole ancestor
    // mask (in place: tree keys at any offset from a half's first key)
    const uint64_t ancw = (!kChain && vrow) ? p.anc[2 * (size_t)(sg.o + node) + (kIP ? 0 : hf)] : 0ull;
    const uint64_t anc_hi = (kKV == kKVInPlace && vrow) ? p.anc[2 * (size_t)(sg.o + node) + 1] : 0ull;
    // m_used is kept in raw score units (scale > 0, so the max commutes with it)
    float m_used = -INFINITY, l = 0.f;
    // keys below full_end: every row sees all of them (when their pages are valid)
    const int full_end = kIP ? min(sg.k_end, sg.ctx) : sg.k_end;
    // step tg processes the segment's tile tg - tb + rot (mod n_tiles)
    for (int t = 0; t < sg.n_tiles; ++t) {
      const int tg = tb + t;
      const int sb = tg % kSB;    // S buffer of this tile
      const int xb = tg & 1;      // pair-exchange slot
      const bool got = wait(s_full + 8 * sb, tg / kSB);
      uint32_t sr[64];
      float tmax = -INFINITY;
      if (got) {
        tc_fence_after();
        tc_ld32_nowait(tl + sb * kKT + 64 * hf, *reinterpret_cast<uint32_t(*)[32]>(&sr[0]));
        tc_ld32_nowait(tl + sb * kKT + 64 * hf + 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[32]));
        const int i = t + sg.rot < sg.n_tiles ? t + sg.rot : t + sg.rot - sg.n_tiles;
        const unsigned pm = s_mask[tg % kMaskRing];     // bit j: 16-row block j has a valid page
        const int p0 = sg.k_begin + i * kKT;            // the tile's first key
        // a whole tile of context keys in valid pages needs no mask: every row
        // sees all of it (rows past R hold zero queries and are never stored)
        const bool whole = i < sg.n_ctx && pm == 0xFFu && p0 + kKT <= full_end;
        tc_wait_ld32(*reinterpret_cast<uint32_t(*)[32]>(&sr[0]));
        tc_pin32(*reinterpret_cast<uint32_t(*)[32]>(&sr[32]));
        if (!whole) {
          // visibility of this half's 64 keys as one 64-bit word
          uint64_t kw;
          const int h0 = p0 + 64 * hf;
          if (i < sg.n_ctx) {
            const int nv = min(max(sg.k_end - h0, 0), 64);
            uint64_t pgw = 0ull;
#pragma unroll
            for (int pb = 0; pb < 4; ++pb)
              pgw |= ((pm >> (4 * hf + pb)) & 1u) ? (0xFFFFull << (16 * pb)) : 0ull;
            kw = pgw & (nv >= 64 ? ~0ull : ((1ull << nv) - 1ull));
            if constexpr (kChain) {
              // causal: node sees positions up to ctx + node
              const int nvis = min(max(sg.ctx + node + 1 - h0, 0), 64);
              kw &= nvis >= 64 ? ~0ull : ((1ull << nvis) - 1ull);
            } else if constexpr (kIP) {
              // keys below ctx are context; key p >= ctx is tree node p - ctx
              const int nc = min(max(sg.ctx - h0, 0), 64);
              const int sh = h0 - sg.ctx;    // ancestor bit of this half's first key
              uint64_t tm;
              if (sh >= 0)
                tm = sh >= 128 ? 0ull
                     : sh >= 64 ? (anc_hi >> (sh - 64))
                     : sh == 0  ? ancw
                                : ((ancw >> sh) | (anc_hi << (64 - sh)));
              else
                tm = sh <= -64 ? 0ull : (ancw << (-sh));
              kw &= (nc >= 64 ? ~0ull : ((1ull << nc) - 1ull)) | tm;
            }
          } else {
            const int th = min(max(sg.T - 64 * hf, 0), 64);
            kw = ancw & (th >= 64 ? ~0ull : ((1ull << th) - 1ull));
          }
          if (!vrow) kw = 0ull;
#pragma unroll
          for (int c = 0; c < 64; ++c)
            if (!((kw >> c) & 1ull)) sr[c] = __float_as_uint(-INFINITY);
        }
        // 8 independent chains of three-input maxima over the 64 values
        float mx[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) mx[c] = __uint_as_float(sr[c]);
#pragma unroll
        for (int c = 8; c < 56; c += 16)         // values 8 .. 55, two per instruction
#pragma unroll
          for (int k = 0; k < 8; ++k)
            mx[k] = fmax3(mx[k], __uint_as_float(sr[c + k]), __uint_as_float(sr[c + 8 + k]));
#pragma unroll
        for (int k = 0; k < 8; ++k) mx[k] = fmaxf(mx[k], __uint_as_float(sr[56 + k]));   // values 56 .. 63
        tmax = fmax3(fmax3(mx[0], mx[1], mx[2]), fmax3(mx[3], mx[4], mx[5]), fmaxf(mx[6], mx[7]));
      }
      // the pair swaps its halves' maxima; both S halves are in registers before
      // either warp overwrites S with P.  kFail (a NaN no maximum yields: theirs is
      // 0x7fffffff) says that this half's wait failed
      constexpr uint32_t kFail = 0xffffffffu;
      s_xmax[xb][hf][r] = got ? __float_as_uint(tmax) : kFail;
      tc_fence_before();
      asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory");
      tc_fence_after();
      const uint32_t other = s_xmax[xb][hf ^ 1][r];
      if (!__all_sync(0xffffffffu, got && other != kFail)) {
        ok = false;
        break;
      }
      tmax = fmaxf(tmax, __uint_as_float(other));
      const float m_new = fmaxf(m_used, tmax);
      const bool need = (m_new - m_used) * sl2 > kRescaleLog2;   // true when m_used = -inf < m_new
      if (t > 0 && __any_sync(0xffffffffu, need)) {
        // O must hold P.V(tg-1) before this half's columns are rescaled; a failed
        // wait sets the abort flag, and the pair stops at the next barrier
        if (wait(pv_done + 8 * ((tg - 1) % kSB), (tg - 1) / kSB)) {
          tc_fence_after();
          const float f = need ? ex2((m_used - m_new) * sl2) : 1.f;
#pragma unroll 1
          for (int c4 = 0; c4 < 4; ++c4) {
            uint32_t ov[16];
            tc_ld16(tl + kColO + 64 * hf + 16 * c4, ov);
#pragma unroll
            for (int e = 0; e < 16; ++e) ov[e] = __float_as_uint(__uint_as_float(ov[e]) * f);
            tc_st16_nowait(tl + kColO + 64 * hf + 16 * c4, ov);
          }
          tc_wait_st();
        } else {
          ok = false;
        }
      }
      if (need) {
        l *= ex2((m_used - m_new) * sl2);
        m_used = m_new;
      }
      const float nms = m_used == -INFINITY ? 0.f : -m_used * sl2;
      // p = 2^(s*scale_log2 - m); P = head + tail, both bf16: this
      // half's head pairs go to columns 32 hf.. of the S buffer, its tail pairs
      // to 64 + 32 hf..
      // (the scale-and-shift and the running sums take one packed fp32x2
      // instruction per pair of columns)
      const uint64_t sl2x2 = f2_pack(__float_as_uint(sl2), __float_as_uint(sl2));
      const uint64_t nmsx2 = f2_pack(__float_as_uint(nms), __float_as_uint(nms));
      uint64_t ls2[4];
      // two halves of 16 column pairs: each half's head and tail words go
      // out before the next half is computed (fewer live registers)
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        uint32_t hw[16], tw[16];
#pragma unroll
        for (int e2 = 0; e2 < 16; ++e2) {
          const int e = 16 * hh + e2;
          uint32_t y0, y1;
          f2_unpack(f2_fma(f2_pack(sr[2 * e], sr[2 * e + 1]), sl2x2, nmsx2), y0, y1);
          const uint32_t p0 = __float_as_uint(ex2(__uint_as_float(y0)));
          const uint32_t p1 = __float_as_uint(ex2(__uint_as_float(y1)));
          const uint64_t pp = f2_pack(p0, p1);
          ls2[e & 3] = e < 4 ? pp : f2_add(ls2[e & 3], pp);
          // head = p rounded to bf16; the negated tail = head - p (exact in fp32)
          // rounded to bf16, two mixed-type subtractions; the MMA negates it back
          const uint32_t hb = bf16x2_rn(__uint_as_float(p1), __uint_as_float(p0));
          float t0, t1;
          sub_bf16x2(hb, __uint_as_float(p0), __uint_as_float(p1), t0, t1);
          hw[e2] = hb;
          tw[e2] = bf16x2_rn(t1, t0);
        }
        tc_st16_nowait(tl + sb * kKT + 32 * hf + 16 * hh, hw);
        tc_st16_nowait(tl + sb * kKT + 64 + 32 * hf + 16 * hh, tw);
      }
      tc_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_full + 8 * sb);
      {
        uint32_t a0, a1, b0, b1, c0, c1, d0, d1;
        f2_unpack(ls2[0], a0, a1);
        f2_unpack(ls2[1], b0, b1);
        f2_unpack(ls2[2], c0, c1);
        f2_unpack(ls2[3], d0, d1);
        l += ((__uint_as_float(a0) + __uint_as_float(a1)) + (__uint_as_float(b0) + __uint_as_float(b1))) +
             ((__uint_as_float(c0) + __uint_as_float(c1)) + (__uint_as_float(d0) + __uint_as_float(d1)));
      }
    }
    // wait for the last P.V (products complete in order, and this barrier's
    // previous phase, P.V three tiles before, was over before the last S
    // existed); the pair adds its two sums, then each half writes its 64
    // columns out: O / l itself when the segment is a whole row block, else the
    // partial (O, m, l) to the segment's slot
    const int tl_g = tb + sg.n_tiles - 1;
    // (balanced: with the next segment received, or an exit both share)
    const bool have = ok && sg.n_tiles > 0 && wait(pv_done + 8 * (tl_g % kSB), tl_g / kSB) &&
                      (!kBal || wait(seg_full + 8 * ((nseg + 1) % kSegRing), (nseg + 1) / kSegRing));
    s_xl[hf][r] = l;
    if (lane == 0) s_xok[nseg & 1][qd][hf] = have;
    asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory");
    const float l_sum = s_xl[0][r] + s_xl[1][r];
    const bool both = s_xok[nseg & 1][qd][0] && s_xok[nseg & 1][qd][1];
    const bool nan_row = both && vrow && l_sum != l_sum;   // NaN scores: the output is NaN
    const float row_m =
        nan_row ? 0.f : ((both && vrow && m_used != -INFINITY) ? m_used * sl2 : -INFINITY);
    const float row_l = (both && vrow && (m_used != -INFINITY || nan_row)) ? l_sum : 0.f;
    float4* dst;
    size_t dstride;                                   // float4 between column chunks
    float inv = 1.f;
    if (sg.alone) {
      const size_t orow = (size_t)(sg.o + node) * p.n_q + sg.hk * g + (rr - node * g);
      dst = reinterpret_cast<float4*>(p.out + orow * kD);
      dstride = 1;
      inv = row_l == 0.f ? 0.f : 1.f / row_l;
    } else {
      dst = reinterpret_cast<float4*>(p.part + (size_t)sg.slot * kAttnPartBytes) + r;
      dstride = kRows;
    }
    const bool store = sg.alone ? vrow : (row_l > 0.f || nan_row);
    if (sg.n_tiles > 0) {
      tc_fence_after();
      uint32_t ov[64];
      tc_ld32_nowait(tl + kColO + 64 * hf, *reinterpret_cast<uint32_t(*)[32]>(&ov[0]));
      tc_ld32_nowait(tl + kColO + 64 * hf + 32, *reinterpret_cast<uint32_t(*)[32]>(&ov[32]));
      tc_wait_ld32(*reinterpret_cast<uint32_t(*)[32]>(&ov[0]));
      tc_pin32(*reinterpret_cast<uint32_t(*)[32]>(&ov[32]));
      tc_fence_before();   // O is in registers: the next segment's P.V may overwrite it
      __syncwarp();
      if (lane == 0) mbar_arrive(o_free);
      if (store) {
#pragma unroll
        for (int e = 0; e < 16; ++e)
          __stcg(dst + (size_t)(16 * hf + e) * dstride,
                 make_float4(__uint_as_float(ov[4 * e]) * inv, __uint_as_float(ov[4 * e + 1]) * inv,
                             __uint_as_float(ov[4 * e + 2]) * inv, __uint_as_float(ov[4 * e + 3]) * inv));
      }
    }
    if (!sg.alone) {
      if (hf == 0)
        __stcg(reinterpret_cast<float2*>(p.part + (size_t)sg.slot * kAttnPartBytes + kAttnMlOff) + r,
               make_float2(row_m, row_l));
    }
    if (!both) ok = false;
  }

  // ---- merge of split row blocks: the softmax warps' (they hold the registers) ------
  tc_fence_before();
  __syncthreads();
  pdl_allow_next();
  const int tid = threadIdx.x - 32 * kWarpSoft0;
  __shared__ int s_ready[2];
  if constexpr (kBal) {
    // ---- merge of split row blocks (balanced mode) ----------------------------------
    // a CTA's pieces are counted and waited for independently, each by a thread of
    // its own (the launch is cooperative: all CTAs are resident and every count arrives)
    const int npieces = s_npc;     // written before the teardown barrier
    if (npieces == 0) return;
    // two pieces: each group of four warps takes one
    const int nthr = npieces == 2 ? kSoftThreads / 2 : kSoftThreads;
    const int i = tid / nthr;
    const int t = tid - i * nthr;
    const BalPiece q = s_pc[i];
    if (t == 0) {
      // the partials of this CTA's pieces (every thread's stores precede the
      // teardown barrier) are released with the count
      unsigned long long* cnt =
          reinterpret_cast<unsigned long long*>(p.part + (size_t)q.slot0 * kAttnPartBytes + kAttnCntOff);
      red_add_release64(cnt, kCountGen / (unsigned)q.K);
      const bool ready = wait_count64_geq(cnt, q.target);
      if (!ready) flag_error(p.err, EE_DEVERR_TIMEOUT);
      s_ready[i] = ready;
    }
    asm volatile("bar.sync %0, %1;" ::"r"(2 + i), "r"(nthr) : "memory");
    if (s_ready[i])
      merge_pieces<1>(p, (size_t)q.slot0, (size_t)q.slot1, 2, q.K, q.k, q.rb * kRows, min(kRows, q.R - q.rb * kRows),
                      q.o, q.hk, t, nthr);
  } else {
    if (s_uni.y == 0 || p.S == 1) return;   // (y == 0: the row block has no work)
    // ---- merge (uniform modes) -------------------------------------------------------
    // once every slot of the row block is complete and visible, chunk `split`
    // merges its share of the columns
    const int split = (int)(blockIdx.x % p.S);   // == cluster rank in the cluster mode
    const int R = s_uni.y, o = s_uni.x;
    const int rb = blockIdx.x / p.S;
    const size_t cta0 = ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + (size_t)rb * p.S;
    if (p.coop) {
      if (tid == 0) {
        // this CTA's partial (every thread's stores precede the teardown barrier)
        unsigned long long* cnt = reinterpret_cast<unsigned long long*>(p.part + cta0 * kAttnPartBytes + kAttnCntOff);
        red_add_release64(cnt, kCountGen / (unsigned)p.S);
        const bool ready = wait_count64_geq(cnt, s_pc[0].target);
        if (!ready) flag_error(p.err, EE_DEVERR_TIMEOUT);
        s_ready[0] = ready;
      }
    } else {
      cluster_sync();
      if (tid == 0) s_ready[0] = 1;
    }
    asm volatile("bar.sync 2, %0;" ::"n"(kSoftThreads) : "memory");
    if (s_ready[0])
      merge_pieces<2>(p, cta0, cta0 + 1, 1, p.S, split, rb * kRows, min(kRows, R - rb * kRows), o, (int)blockIdx.y, tid,
                      kSoftThreads);
  }
}

// Clusters of `S` CTAs that fit on device `dev` at once (asked once per device
// and size; `dev` is the current device).
int active_clusters(int dev, int S) {
  static std::mutex mu;
  static int cache[kMaxDevices][kMaxCluster + 1] = {};
  std::lock_guard<std::mutex> lock(mu);
  int* cached = &cache[dev][S];
  if (!*cached) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S * 64, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = kSmemBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = S;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, attn_tc_kernel<false, kKVTree>, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      n = std::max(1, kNumSMs / S);
    }
    *cached = n;
  }
  return *cached;
}

// CTAs of one instantiation device `dev` (the current device) holds at once
// (asked once per device; -1 if unknown).
template <bool kBal>
int resident_ctas(int dev) {
  static std::mutex mu;
  static int caps[kMaxDevices] = {};
  std::lock_guard<std::mutex> lock(mu);
  int& cap = caps[dev];
  if (!cap) {
    int sms = 0, per = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, attn_tc_kernel<kBal, kKVTree>, kThreads, kSmemBytes) !=
            cudaSuccess ||
        per < 1) {
      cudaGetLastError();
      cap = -1;
    } else {
      cap = sms * per;
    }
  }
  return cap;
}

// Every instantiation takes the full dynamic shared memory (set once per device;
// `dev` is the current device).
cudaError_t set_attrs(int dev) {
  static std::mutex mu;
  static bool done_dev[kMaxDevices] = {};
  std::lock_guard<std::mutex> lock(mu);
  bool& done = done_dev[dev];
  if (done) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  const void* fns[6] = {(const void*)attn_tc_kernel<false, kKVTree>, (const void*)attn_tc_kernel<true, kKVTree>,
                        (const void*)attn_tc_kernel<false, kKVInPlace>, (const void*)attn_tc_kernel<true, kKVInPlace>,
                        (const void*)attn_tc_kernel<false, kKVChain>, (const void*)attn_tc_kernel<true, kKVChain>};
  for (const void* f : fns)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
  done = e == cudaSuccess;
  return e;
}

// Chunk length for s chunks of `span` paged keys (with tree_tile, the last one
// also carries the 128-key tree tile), the chunks actually used and the
// 128-key tiles of the busiest CTA.
void chunk_for(int span, bool tree_tile, int s, int* chunk, int* used, int* tiles) {
  int c = (span + (tree_tile ? kKT : 0) + s - 1) / s;
  c = (c + EE_PAGE - 1) / EE_PAGE * EE_PAGE;
  c = std::min(c, kMaxCtaPages * EE_PAGE);
  *chunk = c;
  *used = attn_splits_for(span, c);
  const int last = span - (*used - 1) * c;
  *tiles = std::max((c + kKT - 1) / kKT, (last + kKT - 1) / kKT + (tree_tile ? 1 : 0));
}

struct Split {
  int S = 1, chunk = EE_PAGE;
  bool coop = false;
  bool bal = false;            // balanced work list (cooperative, one CTA per SM)
  int ctas = 0;                // balanced: grid size; CTAs sharing the work (at most); tiles per CTA
  int bal_ctas = 0, bal_tiles = 0;
};

// Launch plan: the kind with the least cost.  Cost is in half-tiles of the tile
// period (0.96 us a tile), less a start that every launch has:
//   uniform: 2 + 2 x waves x (tiles of the busiest CTA + 5).  Measured: one wave
//   takes 7.6 (whole row blocks) to 8.7 us + 0.96 us a tile, a further wave about
//   6 us + its tiles;
//     cluster mode: S <= 8, waves from the clusters the GPU holds at once (one
//     slot fewer per wave once a second wave is needed);
//     cooperative mode: one wave by construction, S up to 16 with n_rb x S
//     CTAs no more than the GPU holds.  Ties go to the cooperative mode, and
//     there to the larger S (the smaller one: 0.1 % slower over 98 drawn calls,
//     single ones 12 % slower to 7 % faster);
//   balanced mode: 17 + 2 x share, where every resident CTA takes an equal share
//   of all units' tiles (w_max at most, t_max per unit at most) and of kUnitCost
//   for each unit; measured 13 us + 0.95 us per tile and unit place with all
//   sequences at max_ctx.  The line lies 1 us lower than that says because ragged
//   batches, whose lengths the host does not know, gain from the balance (8
//   sequences of 1,024 to 16,384: 89 us, and 203 us in equal chunks).  Causal
//   drafts: 9 more (a row block's CTA that ends early makes room in the uniform
//   plan, and the units' decode costs more).  It needs 2 partial slots per CTA, a
//   share of at most kMaxCtaPages pages and B <= 512.
// Both sides, us per layer, balanced / uniform: causal 560, 56 heads 30.0 / 24.9;
// causal 4 x 133 after 880 keys 38.5 / 31.8; 16 x 120 nodes after 60 keys, 28
// heads 25.9 / 23.6; 4 x 16,384 keys, 28 heads 61 / 72.
// The relative error against 64 bits grows with the tiles that one CTA adds up in
// its accumulator (about 2.8e-7 a tile).  Where equal chunks would be longer than
// the balanced shares the time therefore does not decide: the balanced launch is
// taken from 1.5 tiles fewer on (4 x 4,096 keys, 56 heads: 46.1 us balanced with
// an error of 6.6e-6; equal chunks would take 38.8 us with 9.4e-6).
Split choose_split(int dev, int span, bool tree_tile, int n_rb, long w_max, int t_max, int B, size_t part_slots,
                   bool chain) {
  Split best;
  if (span <= 0) return best;                      // the tree tile alone: one chunk
  const int min_splits = (span + kMaxCtaPages * EE_PAGE - 1) / (kMaxCtaPages * EE_PAGE);
  long best_cost = -1, best_tiles = 0, best_len = 0;   // (best_len: 2 x waves x (tiles + 3))
  for (int s = std::max(1, min_splits); s <= kMaxCluster; ++s) {
    int chunk, used, tiles;
    chunk_for(span, tree_tile, s, &chunk, &used, &tiles);
    // from the second wave on, clusters start as earlier ones finish, and free
    // SMs scattered over the GPCs can leave a slot unusable: plan such launches
    // with one cluster slot fewer
    if (used > 1 && (size_t)n_rb * used > part_slots) continue;   // one partial slot per CTA
    const long act = active_clusters(dev, used);
    long waves = (n_rb + act - 1) / act;
    if (waves >= 2 && act > 1) waves = (n_rb + act - 2) / (act - 1);
    const long cost = 2 + 2 * waves * (tiles + 5);
    if (best_cost < 0 || cost < best_cost) {
      best_cost = cost;
      best_tiles = tiles;
      best_len = 2 * waves * (tiles + 3);
      best.S = used;
      best.chunk = chunk;
    }
  }
  const int cap = resident_ctas<false>(dev);
  if (cap > 0) {
    for (int s = std::max(2, min_splits); s <= kMaxSplits && (long)s * n_rb <= cap; ++s) {
      int chunk, used, tiles;
      chunk_for(span, tree_tile, s, &chunk, &used, &tiles);
      if (used < 2 || (size_t)n_rb * used > part_slots) continue;
      const long cost = 2 + 2 * (tiles + 5);
      if (cost <= best_cost) {
        best_cost = cost;
        best_tiles = tiles;
        best_len = 2 * (tiles + 3);
        best.S = used;
        best.chunk = chunk;
        best.coop = true;
      }
    }
  }
  const int capb = resident_ctas<true>(dev);
  if (capb > 0 && B <= kMaxBalSeqs && w_max <= (long)(kMaxCtaPages / (kKT / EE_PAGE)) * capb &&
      part_slots >= 2 * (size_t)capb) {
    const long m = std::max(2, (t_max + kUnitCost + 12) / 13);
    const long n_eff = std::min<long>(capb, std::max<long>(1, w_max / m));
    const long share = (w_max + n_eff - 1) / n_eff;
    const long cost = 2 * ((w_max + (long)kUnitCost * n_rb + n_eff - 1) / n_eff) + (chain ? 26 : 17);
    if (best_cost < 0 || cost < best_cost || (best_tiles > share && 2 * share + 9 < best_len)) {
      best_cost = cost;
      best.bal = true;
      best.coop = true;
      best.ctas = capb;
      best.bal_ctas = (int)n_eff;
      best.bal_tiles = (int)share;
    }
  }
  if (best_cost < 0) best.S = 0;   // no plan fits the workspace's partial slots
  return best;
}

// The plan for these sizes: span = paged keys of the longest row block
// (max_ctx, or max_ctx + max_T in place), row blocks, work-list bound.
Split plan_for(int dev, int B, int max_T, int n_q, int n_kv, int max_ctx, int kv, size_t slots) {
  const int g = n_q / n_kv;
  const int nrb = (max_T * g + kRows - 1) / kRows;
  const int span = kv != kKVTree ? max_ctx + max_T : max_ctx;
  const int t_max = kv != kKVTree ? (span + kKT - 1) / kKT : (max_ctx + kKT - 1) / kKT + 1;
  long per_seq = (long)n_kv * nrb * t_max;
  if (kv == kKVChain) {
    per_seq = 0;
    for (int r = 0; r < nrb; ++r) per_seq += chain_rb_tiles(max_ctx, max_T, g, r);
    per_seq *= n_kv;
  }
  return choose_split(dev, span, kv == kKVTree, nrb * n_kv * B, (long)B * per_seq, t_max, B, slots,
                      kv == kKVChain);
}

// Shared by ee_tree_verify_attn (tree K/V from k_tree / v_tree) and
// ee_tree_verify_attn_inplace (tree K/V at cache positions ctx .. ctx + T - 1).
ee_status verify_attn(const ee_bf16* q, const ee_bf16* k_tree, const ee_bf16* v_tree, const ee_bf16* k_cache,
                      const ee_bf16* v_cache, int32_t num_pages, const int32_t* block_table, int32_t max_pages,
                      const int32_t* ctx_len, int32_t max_ctx, const int32_t* node_off, const uint64_t* anc,
                      int32_t B, int32_t total_nodes, int32_t max_T, int32_t n_q, int32_t n_kv, int32_t head_dim,
                      float scale, float* out, void* ws, size_t ws_bytes, ee_stream_t stream, int kv) {
  const bool inplace = kv != kKVTree;
  if (B < 0 || total_nodes < 0 || n_q < 1 || n_kv < 1 || num_pages < 1 || max_pages < 1 ||
      max_ctx < 0 || max_T < 1)
    return EE_ERR_INVALID_ARG;
  if (head_dim != EE_HEAD_DIM || n_q % n_kv != 0 || max_T > (kv == kKVChain ? EE_MAX_CHAIN : EE_MAX_TREE))
    return EE_ERR_UNSUPPORTED;
  // every key position must have a block-table entry: the context, and in
  // place the tree's positions after it
  const int64_t span = (int64_t)max_ctx + (inplace ? max_T : 0);
  if (span > (int64_t)max_pages * EE_PAGE) return EE_ERR_INVALID_ARG;
  if (!(scale > 0.f) || !std::isfinite(scale)) return EE_ERR_INVALID_ARG;
  if (B == 0 || total_nodes == 0) return EE_OK;
  if (!q || (!inplace && (!k_tree || !v_tree)) || !k_cache || !v_cache || !block_table || !ctx_len ||
      !node_off || (kv != kKVChain && !anc) || !out || !ws)
    return EE_ERR_INVALID_ARG;
  if (!aligned(q, 16) || (!inplace && (!aligned(k_tree, 16) || !aligned(v_tree, 16))) ||
      !aligned(k_cache, 16) || !aligned(v_cache, 16) || !aligned(out, 16) || !aligned(anc, 8) ||
      !aligned(ws, 256))
    return EE_ERR_INVALID_ARG;
  if (ws_bytes < kWorkspaceBytes) return EE_ERR_WORKSPACE;
  if ((int64_t)num_pages * n_kv * EE_PAGE >= ((int64_t)1 << 31)) return EE_ERR_UNSUPPORTED;
  // the plans' limits: kMaxCtaPages pages a chunk, 8 chunks in a cluster
  if (span > (int64_t)kMaxCluster * kMaxCtaPages * EE_PAGE) return EE_ERR_UNSUPPORTED;

  int dev = 0;
  {
    const ee_status ds = current_device(&dev);
    if (ds != EE_OK) return ds;
  }
  EE_CUDA_OK(set_attrs(dev));
  // tensor maps: cache [pages * n_kv * 16 rows][128], tree [total][n_kv][128]
  // (in place the tree maps are not read: the cache maps stand in)
  CUtensorMap tmKc, tmVc, tmKt, tmVt;
  {
    const uint64_t dims[2] = {(uint64_t)head_dim, (uint64_t)num_pages * n_kv * EE_PAGE};
    const uint64_t strides[1] = {(uint64_t)head_dim * 2};
    const uint32_t box[2] = {64, EE_PAGE};
    if (!encode_bf16_tmap(&tmKc, k_cache, 2, dims, strides, box)) return EE_ERR_CUDA;
    if (!encode_bf16_tmap(&tmVc, v_cache, 2, dims, strides, box)) return EE_ERR_CUDA;
  }
  if (inplace) {
    tmKt = tmKc;
    tmVt = tmVc;
  } else {
    const uint64_t dims[3] = {(uint64_t)head_dim, (uint64_t)n_kv, (uint64_t)total_nodes};
    const uint64_t strides[2] = {(uint64_t)head_dim * 2, (uint64_t)n_kv * head_dim * 2};
    const uint32_t box[3] = {64, 1, (uint32_t)kKT};
    if (!encode_bf16_tmap(&tmKt, k_tree, 3, dims, strides, box)) return EE_ERR_CUDA;
    if (!encode_bf16_tmap(&tmVt, v_tree, 3, dims, strides, box)) return EE_ERR_CUDA;
  }
  const int g = n_q / n_kv;
  const int nrb = (max_T * g + kRows - 1) / kRows;
  const size_t slots = ws_bytes > kAttnPartOff ? (ws_bytes - kAttnPartOff) / kAttnPartBytes : 0;
  const Split sp = plan_for(dev, B, max_T, n_q, n_kv, max_ctx, kv, slots);
  if (sp.S == 0) return EE_ERR_WORKSPACE;
  const int S = sp.bal ? 1 : sp.S, chunk = sp.chunk;
  // a split launch writes one partial slot per CTA after the zeroed part
  if (!sp.bal && S > 1 && ws_bytes < kAttnPartOff + (size_t)nrb * S * n_kv * B * kAttnPartBytes)
    return EE_ERR_WORKSPACE;

  AttnParams p;
  p.q = reinterpret_cast<const __nv_bfloat16*>(q);
  p.block_table = block_table;
  p.ctx_len = ctx_len;
  p.node_off = node_off;
  p.anc = anc;
  p.out = out;
  p.part = static_cast<uint8_t*>(ws) + kAttnPartOff;
  p.err = err_word(ws);
  p.num_pages = num_pages;
  p.max_pages = max_pages;
  p.max_ctx = max_ctx;
  p.n_q = n_q;
  p.n_kv = n_kv;
  p.g = g;
  p.total_nodes = total_nodes;
  p.max_T = max_T;
  p.chunk = chunk;
  p.S = S;
  p.coop = (S > 1 && sp.coop) || sp.bal ? 1 : 0;
  p.B = B;
  p.g_inv = g > 1 ? (uint32_t)(((1ull << 32) + g - 1) / g) : 0u;
  p.scale_log2 = scale * 1.4426950408889634f;

  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = sp.bal ? dim3(sp.ctas, 1, 1) : dim3(nrb * S, n_kv, B);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (p.coop) {
    attr[1].id = cudaLaunchAttributeCooperative;
    attr[1].val.cooperative = 1;
    cfg.numAttrs = 2;
  } else if (S > 1) {
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = S;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
  }
  decltype(&attn_tc_kernel<false, kKVTree>) fn;
  switch (kv * 2 + (sp.bal ? 1 : 0)) {
    case 0: fn = attn_tc_kernel<false, kKVTree>; break;
    case 1: fn = attn_tc_kernel<true, kKVTree>; break;
    case 2: fn = attn_tc_kernel<false, kKVInPlace>; break;
    case 3: fn = attn_tc_kernel<true, kKVInPlace>; break;
    case 4: fn = attn_tc_kernel<false, kKVChain>; break;
    default: fn = attn_tc_kernel<true, kKVChain>; break;
  }
  EE_CUDA_OK(cudaLaunchKernelEx(&cfg, fn, tmKc, tmVc, tmKt, tmVt, p));
  return EE_OK;
}

}  // namespace

extern "C" ee_status ee_attn_plan(int32_t B, int32_t max_T, int32_t n_q, int32_t n_kv,
                                  int32_t max_ctx, int32_t inplace, int32_t* splits, int32_t* chunk,
                                  int32_t* mode, int32_t* ctas) {
  if (B < 1 || max_T < 1 || inplace < 0 || inplace > 2 ||
      max_T > (inplace == kKVChain ? EE_MAX_CHAIN : EE_MAX_TREE) || n_q < 1 || n_kv < 1 || n_q % n_kv != 0 ||
      max_ctx < 0 || !splits || !chunk || !mode || !ctas)
    return EE_ERR_INVALID_ARG;
  int dev = 0;
  {
    const ee_status ds = current_device(&dev);
    if (ds != EE_OK) return ds;
  }
  EE_CUDA_OK(set_attrs(dev));
  const int nrb = (max_T * (n_q / n_kv) + kRows - 1) / kRows;
  // the partial slots of a workspace sized by ee_workspace_size
  const size_t slots = std::max((size_t)B * n_q * kAttnMaxSplits, 2 * (size_t)kNumSMsMax);
  const Split sp = plan_for(dev, B, max_T, n_q, n_kv, max_ctx, inplace, slots);
  if (sp.S == 0) return EE_ERR_UNSUPPORTED;
  if (sp.bal) {
    *splits = sp.bal_ctas;
    *chunk = sp.bal_tiles * kKT;
    *mode = 3;
    *ctas = sp.ctas;
  } else {
    *splits = sp.S;
    *chunk = sp.chunk;
    *mode = sp.S == 1 ? 0 : (sp.coop ? 2 : 1);
    *ctas = nrb * sp.S * n_kv * B;
  }
  return EE_OK;
}

extern "C" ee_status ee_tree_verify_attn(const ee_bf16* q, const ee_bf16* k_tree,
                                         const ee_bf16* v_tree, const ee_bf16* k_cache,
                                         const ee_bf16* v_cache, int32_t num_pages,
                                         const int32_t* block_table, int32_t max_pages,
                                         const int32_t* ctx_len, int32_t max_ctx,
                                         const int32_t* node_off, const uint64_t* anc, int32_t B,
                                         int32_t total_nodes, int32_t max_T, int32_t n_q,
                                         int32_t n_kv, int32_t head_dim, float scale, float* out,
                                         void* ws, size_t ws_bytes, ee_stream_t stream) {
  return verify_attn(q, k_tree, v_tree, k_cache, v_cache, num_pages, block_table, max_pages, ctx_len, max_ctx,
                     node_off, anc, B, total_nodes, max_T, n_q, n_kv, head_dim, scale, out, ws, ws_bytes, stream,
                     kKVTree);
}

extern "C" ee_status ee_tree_verify_attn_inplace(const ee_bf16* q, const ee_bf16* k_cache,
                                                 const ee_bf16* v_cache, int32_t num_pages,
                                                 const int32_t* block_table, int32_t max_pages,
                                                 const int32_t* ctx_len, int32_t max_ctx,
                                                 const int32_t* node_off, const uint64_t* anc, int32_t B,
                                                 int32_t total_nodes, int32_t max_T, int32_t n_q,
                                                 int32_t n_kv, int32_t head_dim, float scale, float* out,
                                                 void* ws, size_t ws_bytes, ee_stream_t stream) {
  return verify_attn(q, nullptr, nullptr, k_cache, v_cache, num_pages, block_table, max_pages, ctx_len, max_ctx,
                     node_off, anc, B, total_nodes, max_T, n_q, n_kv, head_dim, scale, out, ws, ws_bytes, stream,
                     kKVInPlace);
}

extern "C" ee_status ee_chain_verify_attn(const ee_bf16* q, const ee_bf16* k_cache, const ee_bf16* v_cache,
                                          int32_t num_pages, const int32_t* block_table, int32_t max_pages,
                                          const int32_t* ctx_len, int32_t max_ctx, const int32_t* node_off,
                                          int32_t B, int32_t total_nodes, int32_t max_T, int32_t n_q,
                                          int32_t n_kv, int32_t head_dim, float scale, float* out, void* ws,
                                          size_t ws_bytes, ee_stream_t stream) {
  return verify_attn(q, nullptr, nullptr, k_cache, v_cache, num_pages, block_table, max_pages, ctx_len, max_ctx,
                     node_off, nullptr, B, total_nodes, max_T, n_q, n_kv, head_dim, scale, out, ws, ws_bytes,
                     stream, kKVChain);
}
