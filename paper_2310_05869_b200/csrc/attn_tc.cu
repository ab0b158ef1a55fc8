// Attention tiles on the 5th-generation tensor cores (tcgen05 + TMEM), bf16 inputs.
//
// A work item is a PAIR of query tiles (2 x 128 rows) that are neighbours in the tile order of
// their leaf / recursion node - or one of the two, where the last pairs of a call are split - and a
// CTA walks once over the key tiles (64 keys each) that either of them needs:
//     S_i = Q_i K^T      tcgen05.mma, operands in 128B-swizzled shared memory (d = 64: Q_i from TMEM), S_i in TMEM
//     P_i = exp2(S_i*c + bias - m)   softmax warpgroup i: one thread per query row (TMEM
//                                    lane); P_i is written back over S_i as bf16
//     O_i += P_i V       tcgen05.mma with P_i read from TMEM, V MN-major in shared memory
// which covers the block-diagonal part (Sec. 4), the sampled residual with weight N/m
// (Alg. 2 line 7) and the exact causal leaves (Sec. 3.1) in one loop.  The two query tiles
// of a 256-row block share every key tile, so K and V are fetched once for 256 rows, and
// every warpgroup has two S buffers in TMEM, so the tensor pipe computes the scores of the next
// key tile while the warpgroup exponentiates the current one.  The running
// row maximum is only moved when it grows by more than 2^32 (the accumulators absorb the
// rest), so O is rarely rescaled; outputs are normalised by the sum of the bf16-rounded
// weights that the tensor cores actually used (d = 64: accumulated by the tensor cores
// themselves, in an extra column of O whose B operand is a slab of ones; d = 128: in
// registers), the log-sum-exp by the unrounded sum.  Rows
// of Q, K, V come from their original places: tiles of consecutive rows (causal leaves) as
// one TMA box per 64 columns, tiles of sorted or sampled rows gathered through the sortLSH
// permutations with 16-byte cp.async copies into the same 128B-swizzled operand layout;
// nothing permuted is ever written to HBM.  (The TMA row gather, tile::gather4, was measured
// at about 100 cycles of issue per four rows and warp: too slow for this.)
//
// Warp roles (384 threads): warps 0-3 and 4-7 softmax + epilogue of query tile 0 and 1,
// warps 8 and 9 MMA issue for query tile 0 and 1 (warp 8 also allocates TMEM, all 512
// columns: per query tile two S buffers of 64, then O0, O1 and, d = 64, Q0, Q1), warp 10 prepares work items (row tables of the
// NEXT item while this one computes, TMA boxes of Q), warp 11 streams K / V tiles through
// the stage ring, across item boundaries.  Gathered Q tiles are fetched by the 256 softmax
// threads, for the next item, right before they write the current item's results.
// Every mbarrier wait is bounded: on a timeout the CTA raises the device status word,
// drains its copies, frees its TMEM and returns.
#include <cstdlib>
#include "tc_util.cuh"

namespace hyperattn {
namespace {

// tensor maps of Q, K, V as [G * n rows x d] bf16 tensors, 128-byte swizzle; box = 64 columns x
// 128 rows (Q) or 64 rows (K, V): one slab of an operand tile
struct alignas(64) TmaMaps {
  CUtensorMap q, k, v;
};

constexpr int TK = 64;                  // keys per tile
// Test build only (-DHA_TEST_DROP_ARRIVAL, never in the shipped library): when armed, the K / V streamer of one CTA
// leaves out the copies of one V tile once, so that the wait for that tile runs out and the give-up path can be
// exercised without any fault.
#ifdef HA_TEST_DROP_ARRIVAL
__device__ int g_test_drop_armed;
#endif
constexpr float kRescaleThreshold = 32.f;   // octaves the scores may exceed the reference before it moves
constexpr float kTileSumLimit = 1099511627776.f;   // 2^40: a tile whose weights sum to more has a score > 2^34 above the reference

// Optional per-role cycle counters (compile with -DHA_TC_TIMING; never in the shipped build).
#ifdef HA_TC_TIMING
__device__ unsigned long long g_tc_timing[48];
#define HA_T0(var) const long long var = clock64()
#define HA_TACC(slot, var) atomicAdd(&g_tc_timing[slot], (unsigned long long)(clock64() - var))
#define HA_LDECL(name) long long name = 0
#define HA_LACC(name, var) name += clock64() - var
#define HA_LFLUSH(slot, name) atomicAdd(&g_tc_timing[slot], (unsigned long long)(name))
#else
#define HA_T0(var)
#define HA_TACC(slot, var)
#define HA_LDECL(name)
#define HA_LACC(name, var)
#define HA_LFLUSH(slot, name)
#endif

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// adds the two bf16 numbers of a packed pair to two fp32 sums, as they are
__device__ __forceinline__ void add_bf16_pair(float& lo, float& hi, uint32_t pair) {
  asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %2;\n\tadd.rn.f32.bf16 %0, lo, %0;\n\tadd.rn.f32.bf16 %1, hi, %1;\n\t}"
      : "+f"(lo), "+f"(hi) : "r"(pair));
}

// Tiles with masked columns (a minority: the diagonal tiles of a causal leaf, padding, sampled
// columns that fall into the query tile's own block): the masked scores are overwritten with
// -inf in TMEM before the tile is read, so that the hot loop carries no mask code at all.
// vis: one bit per column, 1 = visible.  All 32 lanes call it together.
__device__ __noinline__ void mask_scores(uint32_t sbase, uint32_t visa, uint32_t visb) {
  uint32_t r[16];
#pragma unroll 1
  for (int gcol = 0; gcol < 4; ++gcol) {
    const uint32_t vis16 = ((gcol < 2 ? visa : visb) >> (16 * (gcol & 1))) & 0xffffu;
    if (__all_sync(0xffffffffu, vis16 == 0xffffu)) continue;      // warp-uniform: TMEM accesses stay convergent
    tmem_ld16_issue(sbase + 16 * gcol, r);
    tmem_ld16_wait(r);
#pragma unroll
    for (int e = 0; e < 16; ++e)
      if (!((vis16 >> e) & 1u)) r[e] = 0xff800000u;
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n"
                 ::"r"(sbase + 16 * gcol), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
                   "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
  }
  tmem_wait_st();
}

// Rare path of the online softmax: multiply the O columns a row has accumulated so far by
// alpha (a power of two, so nothing is re-rounded).  Kept out of line: the hot loop should
// stay small.  All 32 lanes call it together (TMEM accesses are warp-wide).
__device__ __noinline__ void rescale_row(uint32_t o_addr, int ocols, float alpha) {
  uint32_t r[16];
  for (int c = 0; c < ocols; c += 16) {
    tmem_ld16_issue(o_addr + c, r);
    tmem_ld16_wait(r);
#pragma unroll
    for (int e = 0; e < 16; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * alpha);
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n"
                 ::"r"(o_addr + c), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
                   "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
  }
  tmem_wait_st();
}

// One query tile of the pair.  The key tiles it looks at are two runs of the pair's tile
// list: [s1, s1 + n1) and [s2, s2 + n2).
struct QTile {
  int valid;
  int nq;        // valid rows
  int q0;        // dense: first query row (segment-relative)
  int row0;      // dense causal: local index of the tile's first row (relative to the first key)
  int beta;      // node: block (of a second tile that does not exist: -1)
  int spos0;     // node: first sorted position
  int s1, n1, s2, n2;
};

struct PairDesc {
  int mode;            // 0 dense, 1 node
  int seg;
  int causal;          // dense
  int k0, nk;          // dense: key range; node: first key row of the node and N
  int qnode0;          // node: first query row of the node
  size_t slice;        // node: slice offset in perm_q / perm_k / rank_k
  int node;            // node: heap index
  int nq_node, bq;     // node: query rows of the node, rows per group of sorted queries
  int nbA, nbB, nsmp;  // node: key tiles of block A, of block B (0 if shared), of the samples
  float bias_max;      // node, weighted sampling: the largest log2 weight among the samples
  int ntiles;          // key tiles walked
  size_t orow_base; int odelta; int partial;
};

// what every role needs to know about a work item; decoded once, by the item preparer
struct ItemDesc {
  PairDesc t;
  QTile qa, qb;
  int lenA, lenB;      // node: keys of block A, of block B (the streamer's; among the fields that every role reads they cost 1 %)
};

template <int D>
struct Cfg {
  static constexpr int NS = (D == 64) ? 8 : 4;        // K stages and V stages
  static constexpr int kQTile = 128 * D * 2;          // bytes of one 128-row query tile
  static constexpr int kTile = TK * D * 2;            // bytes of one key / value tile
  static constexpr int kOffQ = 0;                     // Q0, Q1
  static constexpr int kOffK = 2 * kQTile;
  static constexpr int kOffV = kOffK + NS * kTile;
  // row tables, two sets (the loaders build the set of the next work item while this one runs)
  static constexpr int kOffIdx = kOffV + NS * kTile;              // int [2][kMaxNodeKeys] key rows
  static constexpr int kOffMask = kOffIdx + 2 * kMaxNodeKeys * 4; // uint32 [2][2][kMaxNodeKeys/32] masked-column bits
  static constexpr int kOffQrow = kOffMask + 4 * (kMaxNodeKeys / 32) * 4;   // int [2][2][128]
  static constexpr int kOffBar = kOffQrow + 4 * 128 * 4;
  static constexpr int kSBufs = 2;                    // S buffers per query tile
  // barriers of the S buffers and of the P buffers of a query tile lie this many slots from those of the other: nothing but the
  // compiled address arithmetic depends on it, and each is the faster one (attention, us, 3 and 2 slots: 32 causal heads x 131072
  // rows, d = 64, 5642 and 5695; 32 x 32768, d = 128, 366 and 355)
  static constexpr int kBarSlots = D == 64 ? 3 : kSBufs;
  // d = 64: the P V product is 80 columns wide - behind the 64 columns of V the B operand
  // continues in a slab of ones, so column 64 of O accumulates the sum of the bf16 weights that
  // normalises the row (the tensor pipe's floor per product does not depend on N up to 128, so
  // the extra columns are free and the softmax warps save one add per weight).  d = 128 would
  // pay for them (N = 144) and keeps the sum in registers.
  static constexpr bool kOnes = D == 64;
  static constexpr int kOCols = kOnes ? 80 : D;       // TMEM columns of one O accumulator
  static constexpr int kNumBar = 21 + 6 * NS + 4 * kBarSlots;
  static constexpr int kOffMisc = kOffBar + 8 * kNumBar;          // tmem slot, abort flag
  // Epilogue staging, one slice of 32 rows x kStageRow bytes per softmax warp: rows leave the
  // warp as whole 64- or 128-byte pieces instead of 16 bytes per lane and row.  d = 64: eight
  // slices of 4 KB.  d = 128 (less shared memory to spare): slices of 2 KB, those of query tile
  // 0 in the item's own key-row table, which nobody reads any more once the item's last K / V
  // tile has been issued - it has been when query tile 0 is done, because that tile walks the
  // last tile of every item (launches do not pair query tiles where it would not) - and which is
  // not rebuilt before the softmax warps release the set.
  static constexpr int kStageRow = (D == 64) ? 128 : 64;
  static constexpr int kStageWarp = 32 * kStageRow;
  static constexpr int kDescBytes = (sizeof(ItemDesc) + 15) / 16 * 16;
  static constexpr int kOffDesc = (kOffMisc + 16 + 15) / 16 * 16;   // ItemDesc [2], one per table set
  static constexpr int kOffStage = (kOffDesc + 2 * kDescBytes + 127) / 128 * 128;
  static constexpr int kOffOnes = (kOffStage + ((D == 64) ? 8 : 4) * kStageWarp + 1023) / 1024 * 1024;   // [TK keys x 128 B] of bf16 1.0
  // float [2][kMaxWeightedSamples]: log2 weight of every sampled column (weighted sampling only)
  static constexpr int kOffBias = kOnes ? kOffOnes + TK * 128 : kOffStage + ((D == 64) ? 8 : 4) * kStageWarp;
  static constexpr int kTotal = kOffBias + 2 * kMaxWeightedSamples * 4;
  static_assert(kTotal <= 232448, "shared memory");
  static_assert(D == 64 || 4 * kStageWarp <= kMaxNodeKeys * 4, "staging of query tile 0 must fit one key-row table");
  static constexpr int kTmemCols = 512;
  static constexpr int kColO = 64 * 2 * kSBufs;       // S buffer b of tile i at 64 (kSBufs i + b); O_i at kColO + kOCols i
  // d = 64 has columns to spare for Q: copied from shared memory once per item, it is the A operand of the scores from there.  Read from
  // shared memory with every key tile (16 KB, beside 8 of K and 10 of V) it keeps the tensor pipe waiting and costs power, which
  // is what bounds the clock here.  (Attention, us, shared memory -> TMEM: 128 causal leaves of 4096 rows 454 -> 440; 32 heads x 65536
  // rows 614 -> 604; 16 causal heads x 32768 673 -> 658.)
  static constexpr bool kQTmem = D == 64;
  static constexpr int kColQ = kColO + 2 * kOCols;    // Q_i at kColQ + i D / 2 (pairs of bf16)
  static_assert(kColQ + (kQTmem ? D : 0) <= 512, "TMEM columns");
};

// only: the pair's query tile that the item consists of, -1: both
__device__ __forceinline__ void decode_pair(const AttnArgs& a, int pair, int only, PairDesc& t, QTile& qa, QTile& qb, int& lenA, int& lenB) {
  const Geometry& g = a.g;
  t.partial = !a.direct;
  qa.valid = 1; qb.valid = 0;
  t.nbA = t.nbB = t.nsmp = lenA = lenB = 0;
  int s, q0n, k0n;
  if (pair < a.n_leaf_pairs) {
    // Leaf after leaf, the pairs of a leaf from the heaviest (last rows, most keys) to the lightest: items are
    // handed out in this order, so the CTAs that run at the same time work on a handful of neighbouring leaves
    // and find each other's K / V tiles in L2, and the list still ends with light items.
    // (The last leaves of a call without node items: all heavy pairs first, see tail_leaves().)
    int rem, rank;
    leaf_of_item(pair, a.n_leaf_pairs, a.pairs_per_leaf, a.tail_leaves, rem, rank);
    const int uu = a.pairs_per_leaf - 1 - rank;
    t.seg = rem / a.leaves_per_seg;
    const int leaf = rem % a.leaves_per_seg;
    t.mode = 0; t.causal = a.dense_causal;
    // a leaf: the rows [k0, k0 + leaf) that exist; a non-causal call that is one block: all n queries against all nk keys
    t.k0 = leaf * g.leaf; t.nk = g.causal ? max(0, min(g.leaf, g.n - t.k0)) : g.nk;
    const int nq_leaf = g.causal ? t.nk : g.n;
    QTile* qs[2] = {&qa, &qb};
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int tt = 2 * uu + i;
      QTile& q = *qs[i];
      q.valid = tt < a.tiles_per_leaf && tt * kTileQ < nq_leaf;
      q.row0 = tt * kTileQ;
      q.q0 = t.k0 + tt * kTileQ;
      q.nq = min(kTileQ, nq_leaf - tt * kTileQ);
      const int lim = t.causal ? min(t.nk, q.row0 + q.nq) : t.nk;
      q.s1 = 0; q.n1 = q.valid ? (lim + TK - 1) / TK : 0; q.s2 = 0; q.n2 = 0;
    }
    t.orow_base = (size_t)t.seg * g.n; t.odelta = 0;
  } else {
    int level = 0;
    while (level + 1 < g.levels && pair >= a.level_pair_start[level + 1]) ++level;
    int idx = pair - a.level_pair_start[level];
    node_rows(g, level, 0, s, q0n, k0n);
    const int nodes_lvl = g.causal ? (1 << level) : 1;
    const int sorted = a.level_sorted[level];
    const int paired = a.level_paired[level];
    const int tiles_node = sorted ? node_blocks(s, g.b) * a.tiles_per_block : ((g.causal ? s : g.n) + kTileQ - 1) / kTileQ;
    const int pairs_node = paired ? (tiles_node + 1) / 2 : tiles_node;
    const int pn = idx % pairs_node; idx /= pairs_node;
    const int j = idx % nodes_lvl;
    t.seg = idx / nodes_lvl;
    node_rows(g, level, j, s, q0n, k0n);
    t.k0 = k0n; t.nk = s; t.qnode0 = q0n; t.causal = 0;
    t.nq_node = node_queries(g, s, q0n);
    t.bq = query_group(g.b, t.nq_node, s);
    t.mode = sorted;
    QTile* qs[2] = {&qa, &qb};
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int tn = paired ? 2 * pn + (only == 1 ? 1 - i : i) : pn;
      QTile& q = *qs[i];
      q.valid = tn < tiles_node && (i == 0 || paired);
      q.row0 = 0;
      if (sorted) {
        q.beta = tn / a.tiles_per_block;
        const int sub = tn % a.tiles_per_block;
        q.spos0 = q.beta * t.bq + sub * kTileQ;
        q.nq = t.bq > 0 ? min(kTileQ, block_len(t.nq_node, t.bq, q.beta) - sub * kTileQ) : 0;
        if (q.nq <= 0) q.valid = 0;                       // the group (a short last one, or one past the node's queries) has no such tile
        // (qb's block stays where the pair is split: the order of the sampled columns is that of the pair)
        if (i == 1 && !q.valid) q.beta = -1;
        if (i == 1 && only >= 0) q.valid = 0;
        q.q0 = 0;
      } else {
        q.q0 = q0n + tn * kTileQ;
        q.nq = min(kTileQ, t.nq_node - tn * kTileQ);
        if (q.nq <= 0) q.valid = 0;
        q.s1 = 0; q.n1 = q.valid ? (s + TK - 1) / TK : 0; q.s2 = 0; q.n2 = 0;
      }
    }
    if (sorted) {
      t.slice = ((size_t)level * g.G + t.seg) * g.nl + (g.causal ? (size_t)j * s : 0);
      t.node = g.causal ? (1 << level) - 1 + j : 0;
      lenA = block_len(s, g.b, qa.beta);
      lenB = qb.valid ? block_len(s, g.b, qb.beta) : 0;
      const int bt = (lenA + TK - 1) / TK, btb = (lenB + TK - 1) / TK;                        // key tiles of a block: its own length
      t.nbA = bt;
      t.nbB = (qb.valid && qb.beta != qa.beta) ? btb : 0;
      t.nsmp = (g.m + TK - 1) / TK;
      // A query tile that does not exist walks no key tiles.  (The short last block may have fewer tiles, and so may every group
      // of a node with fewer queries than keys: then the second tile of a pair, the first of the next group, may exist alone.)
      if (!qa.valid) t.nbA = 0;
      if (!qa.valid && !qb.valid) t.nsmp = 0;
      qa.s1 = 0; qa.n1 = t.nbA; qa.s2 = t.nbA + t.nbB; qa.n2 = qa.valid ? t.nsmp : 0;
      qb.s1 = t.nbB ? t.nbA : 0; qb.n1 = qb.valid ? (t.nbB ? btb : bt) : 0; qb.s2 = t.nbA + t.nbB; qb.n2 = qb.valid ? t.nsmp : 0;
    }
    if (a.direct) { t.orow_base = (size_t)t.seg * g.n; t.odelta = 0; }
    else { t.orow_base = (size_t)g.G * g.n + (size_t)level * g.G * g.nl + (size_t)t.seg * g.nl + (size_t)j * s; t.odelta = -q0n; }
  }
  t.ntiles = max(qa.s1 + qa.n1, max(qa.s2 + qa.n2, max(qb.s1 + qb.n1, qb.s2 + qb.n2)));
}

// Value rows of a key tile with columns that do not exist, which get zeros: their weights are zero, but zero times a NaN or an infinity
// of some other leaf, row or head would not be.  (Their scores are overwritten, whatever K is there.)  All 32 lanes call it together;
// table: the item's key rows from this tile on; null: consecutive rows from `first` on.  Out of line: in line it costs the tiles that
// are whole 1 % of the attention's time (32 heads x 32768 rows, d = 128: 350 us as it is, 354 in line).
template <int D>
__device__ __noinline__ void fill_short(uint32_t stage, const char* base, const int* table, int first, int have, uint32_t bar) {
  constexpr int CPR = D / 8, RPI = 32 / CPR;
  const int lane = threadIdx.x & 31, cc = lane % CPR;
  for (int r = lane / CPR; r < TK; r += RPI) {
    const int row = table ? table[r] : first + min(r, have - 1);
    cp_async16_or_zero(stage + tile_off<TK>(r, cc), base + (size_t)(uint32_t)row * (D * 2) + cc * 16, r < have);
  }
  cp_async_arrive_noinc(bar);
}

// a-th key tile of a query tile -> index in the pair's tile list
__device__ __forceinline__ int tile_of(const QTile& q, int a) { return a < q.n1 ? q.s1 + a : q.s2 + (a - q.n1); }
// GATHER_LATE: the softmax threads fetch the next item's Q tiles after, not before, they write
// the current item's results (see there).
// PRECISE: every softmax weight enters the P V product as a pair of bf16 numbers hi + lo (relative error
// 2^-17 instead of 2^-9): lo is written into the second half of the S buffer and multiplied by V with a
// second set of products.
// RULE, of the sampled columns of sorted nodes: kCapped: their part of the row sum carries the caps of Alg. 2 (lines 6, 7 and 9); kWeighted: every
// column has a weight of its own (columns drawn by value norms).  (One build for
// both, calls, us, -> two: 4 heads of 50000 queries, 131072 keys, by value norms 138.3 -> 129.0, 16 of 32768, d = 128, 306 -> 295, capped, 8 of 16384
// 159.8 -> 149.9.)
// KIND, what the items of the launch are: kFinalNodes: tiles of one sorted node, a call without recursion; kPartialNodes: of sorted nodes of a recursion;
// kDenseItems: leaves, and nodes that are not sorted; kAnyItems: all of these.  What a build does not need is not in the way of the softmax warps: calls,
// us, in a build for everything -> in its own: 32 heads of 4096 rows 55.2 -> 52.9, 12 of 4096 33.6 -> 31.9, 32 of 16384 173.7 -> 167.5, 32 of 131072
// 1289 -> 1229-1253; d = 128, 32 of 32768 516 -> 497-503; by value norms, 50000 queries and 131072 keys, 4 heads 129.2 -> 121.8; leaves alone, 128 of
// 4096 422 -> 413, d = 128, 64 of 4096 313 -> 302.  (kPartialNodes beside kDenseItems: see kTwoLaunches.)
enum SampleRule { kUniform, kCapped, kWeighted };
enum ItemKind { kAnyItems, kFinalNodes, kPartialNodes, kDenseItems };
template <int D, bool GATHER_LATE, bool PRECISE, SampleRule RULE, ItemKind KIND>
__global__ void __launch_bounds__(384, 1) attn_tc_kernel(const __grid_constant__ AttnArgs a, const __grid_constant__ TmaMaps maps, int* status) {
  using C = Cfg<D>;
  constexpr bool CAPPED = RULE == kCapped, WEIGHTED = RULE == kWeighted;
  constexpr bool NODE = KIND == kFinalNodes || KIND == kPartialNodes, DENSE = KIND == kDenseItems;
  extern __shared__ __align__(1024) uint8_t smem[];
  constexpr int MW = kMaxNodeKeys / 32;
  int* s_kidx_all = reinterpret_cast<int*>(smem + C::kOffIdx);              // [2][kMaxNodeKeys]
  uint32_t* s_mask_all = reinterpret_cast<uint32_t*>(smem + C::kOffMask);  // [2][2][MW]
  int* s_qrow_all = reinterpret_cast<int*>(smem + C::kOffQrow);             // [2][2][128]
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + C::kOffMisc);
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem + C::kOffMisc + 4);

  const uint32_t ubase = smem_u32(smem);
  const uint32_t bar0 = ubase + C::kOffBar;
  const uint32_t bar_q = bar0;                                                // Q tiles of the item landed
  const uint32_t bar_qfree = bar0 + 8;                                        // both issuers are done with Q
  auto bar_s = [&](int i, int b) { return bar0 + 168 + 8 * (6 * C::NS + C::kBarSlots * i + b); };          // S_i buffer b written
  auto bar_p = [&](int i, int b) { return bar0 + 168 + 8 * (6 * C::NS + C::kBarSlots * (2 + i) + b); };    // P_i buffer b written
  auto bar_o = [&](int i) { return bar0 + 80 + 8 * i; };                      // O_i of the item complete
  auto bar_ofree = [&](int i) { return bar0 + 112 + 8 * i; };                 // O_i has been read out
  auto bar_tabfull = [&](int set) { return bar0 + 128 + 8 * set; };           // row tables of a set written
  auto bar_tabfree = [&](int set) { return bar0 + 144 + 8 * set; };           // softmax warps are done with a set
  auto bar_kfull = [&](int s) { return bar0 + 168 + 8 * s; };
  auto bar_vfull = [&](int s) { return bar0 + 168 + 8 * (C::NS + s); };
  auto bar_kempty = [&](int i, int s) { return bar0 + 168 + 8 * ((2 + i) * C::NS + s); };     // released by issuer i
  auto bar_vempty = [&](int i, int s) { return bar0 + 168 + 8 * ((4 + i) * C::NS + s); };

  auto is_node = [](const PairDesc& t) { return NODE || (!DENSE && t.mode == 1); };
  auto is_partial = [](const PairDesc& t) { return KIND == kPartialNodes || (KIND != kFinalNodes && t.partial); };
  const Geometry& g = a.g;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);       // (known to be the same for the whole warp)
  HA_T0(t_cta);

  // A CTA of a launch in which some wait already timed out returns at once (nothing allocated
  // yet), so a stuck launch drains quickly instead of timing out tile after tile.  (Read before
  // wait_for_stream(), on purpose: see there.)
  if (tid == 0) *s_abort = *reinterpret_cast<volatile int*>(status);
  __syncthreads();
  if (*s_abort) return;
  __syncthreads();

  // ---- setup: barriers, TMEM ---------------------------------------------------------------------
  if (tid == 0) {
    mbar_init(bar_q, 32 + 256);                         // item preparer + softmax threads
    mbar_init(bar_qfree, 2);
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_o(i), 1);
      mbar_init(bar_ofree(i), 128);
      mbar_init(bar_tabfull(i), 1);
      mbar_init(bar_tabfree(i), 257);                   // 256 softmax threads + the K / V streamer
      for (int b = 0; b < C::kSBufs; ++b) { mbar_init(bar_s(i, b), 1); mbar_init(bar_p(i, b), 128); }
    }
    for (int s = 0; s < C::NS; ++s) {
      mbar_init(bar_kfull(s), 32);
      mbar_init(bar_vfull(s), 32);
      for (int i = 0; i < 2; ++i) { mbar_init(bar_kempty(i, s), 1); mbar_init(bar_vempty(i, s), 1); }
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if constexpr (C::kOnes) {
    constexpr uint32_t one2 = 0x3f803f80u;              // two bf16 ones
    for (int k = tid; k < TK * 128 / 16; k += 384) *reinterpret_cast<uint4*>(smem + C::kOffOnes + 16 * k) = make_uint4(one2, one2, one2, one2);
    fence_async_smem();                                 // the tensor pipe reads the slab through the async proxy
  }
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)), "r"(C::kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *s_tmem, 0);
  wait_for_stream();

  // The CTA is persistent: it takes work items (pairs of query tiles) from the launch's counter
  // until the list is exhausted.  Every role runs the same item loop at its own pace; what
  // they hand to each other across items is described at the barriers above.  All phase
  // counters keep running across items.
  if (warp < 8) {
    // ================= softmax + epilogue of query tile i: thread = query row ==================
    const int i = warp >> 2;
    const int row = tid & 127;
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t colO = C::kColO + C::kOCols * i;
    int ga = 0;                                       // key tiles this warpgroup has processed so far (all items)
    int gbase = 0;                                    // global index (all items) of the item's first key tile
    int vi = 0;                                       // items in which this query tile existed
    bool ok = true;
    int it = 0;
    // Gathered Q tiles (sorted rows) are fetched by the 256 softmax threads together, 16-byte
    // chunks through cp.async: one warp alone is limited by the copies it can keep in flight.
    // Thread -> column chunk cq of rows rq0, rq0 + 256 / CPR, ...; its arrival on the Q barrier
    // is attached to its copies.  (Tiles of consecutive rows are one TMA box, issued by the
    // item preparer; then the arrival here is immediate.)
    auto gather_q = [&](int nit) {
      bool good = wait_fast<19>(bar_tabfull(nit & 1), (nit >> 1) & 1, s_abort, status);
      if (!good) return false;
      const ItemDesc& de = *reinterpret_cast<const ItemDesc*>(smem + C::kOffDesc + (nit & 1) * C::kDescBytes);
      const PairDesc& t = de.t;
      if (t.mode < 0) return true;                        // the end of the work list: nothing to fetch
      if (nit >= 1) good = wait_fast<20>(bar_qfree, (nit - 1) & 1, s_abort, status);
      if (!good) return false;
      const QTile &qa = de.qa, &qb = de.qb;
      if (is_node(t)) {
        constexpr int CPR = D / 8;
        constexpr int RS = 256 / CPR;                       // rows covered by the 256 threads per step
        const int cq = tid % CPR, rq0 = tid / CPR;
        const char* qsrc = reinterpret_cast<const char*>(a.q) + (size_t)t.seg * g.n * (D * 2) + cq * 16;
        const int* rows = s_qrow_all + (nit & 1) * 2 * 128;
#pragma unroll
        for (int ti = 0; ti < 2; ++ti) {
          if (!(ti ? qb.valid : qa.valid)) continue;       // nobody reads the tile of a query tile that does not exist
          int v[128 / RS];
#pragma unroll
          for (int k = 0; k < 128 / RS; ++k) v[k] = rows[ti * 128 + rq0 + k * RS];
#pragma unroll
          for (int k = 0; k < 128 / RS; ++k)               // padding rows: the segment's first row (results never stored)
            cp_async16(ubase + C::kOffQ + ti * C::kQTile + tile_off<128>(rq0 + k * RS, cq), qsrc + (size_t)(uint32_t)max(v[k], 0) * (D * 2));
        }
        cp_async_arrive_noinc(bar_q);
      } else {
        mbar_arrive(bar_q);
      }
      return true;
    };
    HA_LDECL(a_tab); HA_LDECL(a_ws); HA_LDECL(a_cmp); HA_LDECL(a_epi); HA_LDECL(a_gq); HA_LDECL(a_bo); HA_LDECL(a_tiles); HA_LDECL(a_ws0);
    HA_LDECL(a_c1); HA_LDECL(a_c2); HA_LDECL(a_c3); HA_LDECL(a_c4); HA_LDECL(a_e1); HA_LDECL(a_e2); HA_LDECL(a_e3);
    HA_T0(t_role);
    ok = __all_sync(0xffffffffu, gather_q(0));
    for (; ok; ++it) {
      const int set = it & 1;
      const uint32_t* s_mask = s_mask_all + (set * 2 + i) * MW;
      const int* s_qrow = s_qrow_all + (set * 2 + i) * 128;
      // the tables of this item (also for a warpgroup without a tile: it may not run ahead)
      HA_T0(tt);
      ok = __all_sync(0xffffffffu, wait_fast<14>(bar_tabfull(set), (it >> 1) & 1, s_abort, status));
      if (!ok) break;
      HA_LACC(a_tab, tt);
      const ItemDesc& de = *reinterpret_cast<const ItemDesc*>(smem + C::kOffDesc + set * C::kDescBytes);
      const PairDesc t = de.t;
      if (t.mode < 0) break;                              // the work list is exhausted
      const QTile q = i ? de.qb : de.qa;
      const int total = q.n1 + q.n2;
      const float wlog = (is_node(t) && g.m > 0) ? log2f((float)t.nk / (float)g.m) : 0.f;   // log2(N/m): weight of a sampled column
      // key tiles of this item with masked columns for this query tile, one bit per tile (an item has at most 32)
      unsigned tile_masked = 0;
      if (is_node(t)) tile_masked = __ballot_sync(0xffffffffu, lane < t.ntiles && (s_mask[2 * lane] | s_mask[2 * lane + 1]) != 0);
      float m_ref = -INFINITY;
      uint64_t l01 = 0;             // l: unrounded row sum (two partial sums, packed)
      float lra = 0.f, lrb = 0.f;   // lr: sum of the bf16 weights (two partial sums; the mixed-precision add takes the bf16 halves as they are)
      // Alg. 2 with caps (sorted nodes only): the masked row sum (block part) is complete when the first
      // sampled tile starts; from then on every sampled weight enters the row sum as min(weight, (N/m) C_i),
      // C_i = cap_scale m / (N ln N) (masked_i + tau / kappa), while the numerator keeps the weight itself.
      const bool capped_item = CAPPED && is_node(t) && g.m > 0;
      float lblk = 0.f;             // masked row sum in units of 2^m_ref
      bool in_samples = false;
      float capfac = 0.f, lfloor = -INFINITY;     // (N/m) cap_scale m / (N ln N); log2(tau / kappa)
      // weighted sampling (columns drawn by value norms): every sampled column carries its own log2 weight
      const bool weighted_item = WEIGHTED && is_node(t);
      const float* s_bias = reinterpret_cast<const float*>(smem + C::kOffBias) + set * kMaxWeightedSamples;
      if (capped_item) {
        capfac = a.cap_scale / (logf((float)t.nk));
        lfloor = a.ltau[(size_t)t.seg * g.nodes + t.node] - a.log2_kappa;
      }
      for (int na = 0; na < total && ok; ++na) {
        const int j = tile_of(q, na);
        const int gw = ga + na;
        const int buf = gw % C::kSBufs;
        HA_T0(tw);
        ok = __all_sync(0xffffffffu, wait_fast<2>(bar_s(i, buf), (gw / C::kSBufs) & 1, s_abort, status));   // warp-uniform: TMEM ops are .aligned
        if (!ok) break;
        HA_LACC(a_ws, tw);
#ifdef HA_TC_TIMING
        if (na == 0) a_ws0 += clock64() - tw;
#endif
        HA_T0(tc);
        tc_fence_after();
        // mask kind of this (query tile, key tile): uniform over the warpgroup
        const bool table = (tile_masked >> j) & 1u;
        // (weighted sampling: the tile's columns have weights of their own; the largest one stands in where one number is needed)
        const bool weighted_tile = weighted_item && j >= t.nbA + t.nbB;
        const float ubias = (is_node(t) && j >= t.nbA + t.nbB) ? (weighted_tile ? t.bias_max : wlog) : 0.f;
        const bool dense_mask = !is_node(t) && ((j * TK + TK > t.nk) || (t.causal && j * TK + TK - 1 > q.row0));
        // The 64 scores of this row are read from TMEM once; then (1) the row maximum, (2)
        // exponentials, row sums and the bf16 P written over the first half of the S buffer.
        // The reference maximum only moves when the tile exceeds it by more than 2^32, and then
        // by a whole number of octaves, so that what is already accumulated (O and the row
        // sums) is rescaled exactly.
        uint32_t ra[32], rb[32];
        const uint32_t sbase = lane_addr + 64 * (C::kSBufs * i + buf);
        // masked columns become -inf before the tile is read (out of line, in TMEM): they then
        // drop out of the maximum and exponentiate to zero without any test in this loop
        if (table || dense_mask) {
          uint32_t visa, visb;
          if (table) { visa = ~s_mask[j * 2]; visb = ~s_mask[j * 2 + 1]; }
          else {
            const int climit = t.causal ? min(t.nk - 1, q.row0 + row) : t.nk - 1;   // last visible column of this row
            const int rel = climit - j * TK;            // columns 0..rel of the tile are visible
            visa = rel >= 31 ? 0xffffffffu : (rel < 0 ? 0u : ((2u << rel) - 1u));
            visb = rel >= 63 ? 0xffffffffu : (rel < 32 ? 0u : ((2u << (rel - 32)) - 1u));
          }
          mask_scores(sbase, visa, visb);
        }
        // The second half of the scores is requested once the first has arrived and lands while
        // the first is exponentiated.
        tmem_ld32_issue(sbase, ra);
        tmem_ld32_wait(ra);
        tmem_ld32_issue(sbase + 32, rb);
        HA_LACC(a_c1, tc);
        // The row maximum is NOT computed per tile.  Any reference within a few dozen octaves of the
        // true maximum serves (the accumulators are fp32 and the weights keep their relative
        // precision as bf16), so a tile is exponentiated against the reference the row already
        // has, and only when the tile's sum of weights shows that some score lay more than ~2^34
        // above it (or the row has no reference yet: first tile of an item) is the maximum
        // taken, the reference moved by whole octaves, O rescaled exactly, and the tile
        // exponentiated again from the scores still held in registers.
        auto move_reference = [&]() -> bool {
          tmem_ld32_wait(rb);
          float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
          for (int e = 0; e < 32; e += 4) {
            m0 = max3(m0, __uint_as_float(ra[e]), __uint_as_float(ra[e + 1]));
            m1 = max3(m1, __uint_as_float(ra[e + 2]), __uint_as_float(ra[e + 3]));
            m2 = max3(m2, __uint_as_float(rb[e]), __uint_as_float(rb[e + 1]));
            m3 = max3(m3, __uint_as_float(rb[e + 2]), __uint_as_float(rb[e + 3]));
          }
          m0 = fmaxf(m0, m2); m1 = fmaxf(m1, m3);
          const float xm = fmaf(fmaxf(m0, m1), a.scale_log2, ubias);   // scale_log2 > 0: the maximum commutes with it
          const bool grow = xm > m_ref + kRescaleThreshold;
          if (!__any_sync(0xffffffffu, grow)) return true;
          float alpha = 1.f;
          if (grow) {
            // first tile: leave head room for the weight log2(N/m) that the sampled columns will
            // add, so that reaching them does not move the reference again (any reference within
            // 2^32 below the true maximum serves; a higher one only shifts the exponents)
            if (m_ref == -INFINITY) { m_ref = xm + (wlog - ubias); alpha = 0.f; }
            else { const float k = ceilf(xm - m_ref); m_ref += k; alpha = ex2(-k); }
          }
          { const uint64_t al2 = pack_f2(alpha, alpha); l01 = fmul2(l01, al2); lra *= alpha; lrb *= alpha; lblk *= alpha; }
          // O may only be touched between two PV products: the one of the previous tile must
          // have finished (the one of this tile cannot start before this tile's P is published)
          // That product's completion is what releases its V stage to the streamer, so the
          // stage's barrier tells (the issuer has nothing extra to commit for this rare path).  Its
          // phase cannot run ahead of this warpgroup: the next product on the same stage is NS key
          // tiles later and needs this warpgroup's P first.
          if (na > 0) {
            const int gjp = gbase + tile_of(q, na - 1);
            if (!__all_sync(0xffffffffu, wait_fast<3>(bar_vempty(i, gjp % C::NS), (gjp / C::NS) & 1, s_abort, status))) return false;
            tc_fence_after();
            rescale_row(lane_addr + colO, C::kOCols, alpha);
          }
          return true;
        };
        if (__any_sync(0xffffffffu, m_ref == -INFINITY)) {
          ok = move_reference();
          if (!ok) break;
        }
        const bool capped_tile = capped_item && j >= t.nbA + t.nbB;
        if (capped_tile && !in_samples) {            // the block part is complete: its row sum is the masked sum of line 6
          float b0, b1;
          unpack_f2(l01, b0, b1);
          lblk = b0 + b1;
          in_samples = true;
        }
        const uint64_t sc2 = pack_f2(a.scale_log2, a.scale_log2);
        uint64_t lt2;               // this tile's unrounded sum of weights (two partial sums, packed)
        float lrta, lrtb;           // this tile's sum of the bf16 weights (d = 128)
        for (int attempt = 0;; ++attempt) {
          const float off = ubias - (m_ref == -INFINITY ? 0.f : m_ref);
          // packed fp32 arithmetic (two lanes per instruction) for the scaling and the row sums
          const uint64_t off2 = pack_f2(off, off);
          lt2 = 0; lrta = 0.f; lrtb = 0.f;
          auto chunk_exp = [&](const uint32_t (&r)[32], int c) {
            uint32_t p[16], plo[16];
#pragma unroll
            for (int e = 0; e < 32; e += 2) {
              float x0, x1;
              unpack_f2(ffma2(pack_u2(r[e], r[e + 1]), sc2, off2), x0, x1);
              const float p0 = ex2(x0), p1 = ex2(x1);
              lt2 = fadd2(lt2, pack_f2(p0, p1));
              const uint32_t w = pack2(p0, p1);
              if constexpr (!C::kOnes) add_bf16_pair(lrta, lrtb, w);
              p[e >> 1] = w;
              if constexpr (PRECISE) {
                // what the rounding to bf16 left over, as a second bf16 number (an infinite weight leaves NaN here, but it
                // also makes the tile's sum infinite, and the tile is exponentiated again)
                float r0, r1;
                unpack_f2(fadd2(pack_f2(p0, p1), pack_f2(-__uint_as_float(w << 16), -__uint_as_float(w & 0xffff0000u))), r0, r1);
                const uint32_t wl = pack2(r0, r1);
                if constexpr (!C::kOnes) add_bf16_pair(lrta, lrtb, wl);
                plo[e >> 1] = wl;
              }
            }
            tmem_st16(sbase + c * 16, p);
            if constexpr (PRECISE) {
              tmem_st16(sbase + 32 + c * 16, plo);
            }
          };
          // capped tiles: the row sum takes min(weight, cap), the check below and P take the weight itself
          uint64_t ltu2 = 0;
          const float capw = capped_tile ? capfac * (lblk + (m_ref == -INFINITY ? 0.f : ex2(lfloor - m_ref))) : 0.f;
          auto chunk_exp_capped = [&](const uint32_t (&r)[32], int c) {
            uint32_t p[16];
#pragma unroll
            for (int e = 0; e < 32; e += 2) {
              float x0, x1;
              unpack_f2(ffma2(pack_u2(r[e], r[e + 1]), sc2, off2), x0, x1);
              const float p0 = ex2(x0), p1 = ex2(x1);
              ltu2 = fadd2(ltu2, pack_f2(p0, p1));
              lt2 = fadd2(lt2, pack_f2(fminf(p0, capw), fminf(p1, capw)));
              p[e >> 1] = pack2(p0, p1);
            }
            tmem_st16(sbase + c * 16, p);
          };
          // weighted tiles: x = score * scale + (the column's log2 weight - reference)
          const float* bias_tile = s_bias + (j - (t.nbA + t.nbB)) * TK;
          const uint64_t nref2 = pack_f2(off - ubias, off - ubias);
          auto chunk_exp_weighted = [&](const uint32_t (&r)[32], int c) {
            uint32_t p[16];
#pragma unroll
            for (int e = 0; e < 32; e += 2) {
              const float2 bb = *reinterpret_cast<const float2*>(bias_tile + c * 32 + e);
              float x0, x1;
              unpack_f2(ffma2(pack_u2(r[e], r[e + 1]), sc2, fadd2(pack_f2(bb.x, bb.y), nref2)), x0, x1);
              const float p0 = ex2(x0), p1 = ex2(x1);
              lt2 = fadd2(lt2, pack_f2(p0, p1));
              const uint32_t w = pack2(p0, p1);
              if constexpr (!C::kOnes) add_bf16_pair(lrta, lrtb, w);
              p[e >> 1] = w;
            }
            tmem_st16(sbase + c * 16, p);
          };
          HA_T0(tc2);
          if constexpr (PRECISE) tmem_ld32_wait(rb);     // the lo halves overwrite the second half of the scores
          if (CAPPED && capped_tile) chunk_exp_capped(ra, 0); else if (WEIGHTED && weighted_tile) chunk_exp_weighted(ra, 0); else chunk_exp(ra, 0);
          HA_LACC(a_c2, tc2);
          HA_T0(tc3);
          tmem_ld32_wait(rb);
          if (CAPPED && capped_tile) chunk_exp_capped(rb, 1); else if (WEIGHTED && weighted_tile) chunk_exp_weighted(rb, 1); else chunk_exp(rb, 1);
          HA_LACC(a_c3, tc3);
          float lt0, lt1;
          unpack_f2((CAPPED && capped_tile) ? ltu2 : lt2, lt0, lt1);
          // (the negated comparison also catches an infinite sum; one second attempt at most: after the
          // reference has moved every finite score is within range, and non-finite inputs must not loop)
          if (attempt == 1 || !__any_sync(0xffffffffu, !(lt0 + lt1 <= kTileSumLimit))) break;
          ok = move_reference();
          if (!ok) break;
        }
        if (!ok) break;
        HA_T0(tc4);
        l01 = fadd2(l01, lt2);
        lra += lrta; lrb += lrtb;
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(bar_p(i, buf));
        HA_LACC(a_c4, tc4);
        HA_LACC(a_cmp, tc);
#ifdef HA_TC_TIMING
        a_tiles += 1;
#endif
      }
      if (!ok) break;
      // The next item's Q tiles go out before this item's results are written, so that they are
      // there when the results are - except for fp32 partial results of d = 128 (causal
      // recursion): those are twice the bytes to stage and store and queue behind the gather's
      // copies in the load/store unit (measured: 5 % faster with the gather after them, while
      // bf16 results are 5 % slower that way).
      HA_T0(tg);
      if (!GATHER_LATE) {
        ok = __all_sync(0xffffffffu, gather_q(it + 1));
        if (!ok) break;
      }
      HA_LACC(a_gq, tg);
      HA_T0(te);
      // epilogue: normalise, log-sum-exp, rows back to their original places
      if (q.valid) {
        // Everything that does not need O comes first: the last products are still running.  (Nodes 980 -> 962 us,
        // 32 heads x 65536 rows, d = 64.)
        const int qr = s_qrow[row];
        float l0, l1;
        unpack_f2(l01, l0, l1);
        float inv = C::kOnes ? 0.f : 1.f / (lra + lrb);
        float lse = (m_ref + log2f(l0 + l1)) * 0.69314718055994531f;
        if (capped_item) {
          // line 9: d~_i = masked_i + max(d_i, tau / kappa), d_i the sum of the capped sampled weights
          if (!in_samples) lblk = l0 + l1;
          const float fl = m_ref == -INFINITY ? 0.f : ex2(lfloor - m_ref);
          const float dt = lblk + fmaxf((l0 + l1) - lblk, fl);
          inv = 1.f / dt;
          lse = (m_ref + log2f(dt)) * 0.69314718055994531f;
        }
        const size_t orow = t.orow_base + (size_t)(qr + t.odelta);
        {
          // O leaves TMEM in pieces of 16 columns (thread = row), is normalised (and rounded to
          // bf16 for a bf16 result) and staged in shared memory, XOR-swizzled so that neither
          // side has bank conflicts; then LPR lanes per row write kStageRow contiguous bytes of
          // RPI rows per instruction.
          constexpr int RB = C::kStageRow;
          constexpr int LPR = RB / 16, RPI = 32 / LPR, NI = 32 / RPI;
          constexpr int NP = D / 16;
          const bool f32o = is_partial(t) ? !a.part_bf16 : a.out_fp32;
          char* obase = reinterpret_cast<char*>(is_partial(t) ? a.part_o : a.out);
          const long long myoff = qr >= 0 ? (long long)(orow * (size_t)(D * (f32o ? 4 : 2))) : -1;
          long long roff[NI];
#pragma unroll
          for (int k = 0; k < NI; ++k) roff[k] = __shfl_sync(0xffffffffu, myoff, RPI * k + lane / LPR);
          const uint32_t stg = (D == 64) ? ubase + C::kOffStage + warp * C::kStageWarp
                             : (i == 0 ? ubase + C::kOffIdx + set * (kMaxNodeKeys * 4) : ubase + C::kOffStage) + (warp & 3) * C::kStageWarp;
          const int xw = (RB == 128) ? (lane & 7) : ((lane >> 1) & 3);       // swizzle of this thread's own row
          const int crow = lane / LPR, cc = lane % LPR;
          const int lg_pps = f32o ? (RB == 128 ? 1 : 0) : (RB == 128 ? 2 : 1);   // log2(pieces per staging step)
          if (qr >= 0) {
            if (is_partial(t)) a.part_lse[orow] = lse;
            else a.lse[orow] = lse;
          }
          uint32_t r[16];
          HA_LACC(a_e1, te);
          ok = __all_sync(0xffffffffu, wait_fast<5>(bar_o(i), vi & 1, s_abort, status));
          if (!ok) break;
          HA_LACC(a_bo, te);
          tc_fence_after();
          tmem_ld16_issue(lane_addr + colO, r);
          if constexpr (C::kOnes) {                     // the sum of the bf16 weights sits in column D of O
            uint32_t sumw;
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];\n\ttcgen05.wait::ld.sync.aligned;\n"
                         : "=r"(sumw) : "r"(lane_addr + colO + D) : "memory");
            if (!capped_item) inv = 1.f / __uint_as_float(sumw);
          }
#pragma unroll 1
          for (int pc = 0; pc < NP; ++pc) {
            HA_T0(te2);
            tmem_ld16_wait(r);
            float f[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) f[e] = __uint_as_float(r[e]) * inv;
            if (pc + 1 < NP) tmem_ld16_issue(lane_addr + colO + (pc + 1) * 16, r);
            else { tc_fence_before(); mbar_arrive(bar_ofree(i)); }           // O has been read: the next item may overwrite it
            const int pin = pc & ((1 << lg_pps) - 1);
            const uint32_t srow = stg + lane * RB;
            if (f32o) {
#pragma unroll
              for (int c = 0; c < 4; ++c)
                asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(srow + (((pin * 4 + c) ^ xw) << 4)),
                             "f"(f[4 * c]), "f"(f[4 * c + 1]), "f"(f[4 * c + 2]), "f"(f[4 * c + 3]) : "memory");
            } else {
#pragma unroll
              for (int c = 0; c < 2; ++c)
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(srow + (((pin * 2 + c) ^ xw) << 4)),
                             "r"(pack2(f[8 * c], f[8 * c + 1])), "r"(pack2(f[8 * c + 2], f[8 * c + 3])),
                             "r"(pack2(f[8 * c + 4], f[8 * c + 5])), "r"(pack2(f[8 * c + 6], f[8 * c + 7])) : "memory");
            }
            HA_LACC(a_e2, te2);
            if (pin == (1 << lg_pps) - 1) {
              HA_T0(te3);
              __syncwarp();
              const int step = pc >> lg_pps;
#pragma unroll
              for (int k = 0; k < NI; ++k) {
                const int rw = RPI * k + crow;
                const int xr = (RB == 128) ? (rw & 7) : ((rw >> 1) & 3);
                uint4 w;
                asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w)
                             : "r"(stg + rw * RB + ((cc ^ xr) << 4)) : "memory");
                if (roff[k] >= 0) *reinterpret_cast<uint4*>(obase + roff[k] + step * RB + cc * 16) = w;
              }
              __syncwarp();
              HA_LACC(a_e3, te3);
            }
          }
        }
        ++vi;
      }
      if (GATHER_LATE) {
        ok = __all_sync(0xffffffffu, gather_q(it + 1));
        if (!ok) break;
      }
      mbar_arrive(bar_tabfree(set));
      HA_LACC(a_epi, te);
      ga += total;
      gbase += t.ntiles;
    }
#ifdef HA_TC_TIMING
    if (row == 0 && i == 0) {
      HA_LFLUSH(9, a_tab); HA_LFLUSH(0, a_ws); HA_LFLUSH(2, a_cmp); HA_LFLUSH(15, a_epi); HA_LFLUSH(16, a_gq); HA_LFLUSH(17, a_bo);
      HA_LFLUSH(20, a_tiles); HA_TACC(18, t_role); HA_LFLUSH(19, it);
      HA_LFLUSH(40, a_e1); HA_LFLUSH(41, a_e2); HA_LFLUSH(42, a_e3); HA_LFLUSH(24, a_ws0);
      HA_LFLUSH(22, a_c1); HA_LFLUSH(29, a_c2); HA_LFLUSH(30, a_c3); HA_LFLUSH(31, a_c4);
    }
#endif
  } else if (warp < 10) {
    // ================= MMA issue, a warp per query tile (warp 8: tile 0, warp 9: tile 1) ===========
    // Each issuer walks its own key tiles: scores run two tiles ahead of the PV products
    // (S buffers alternate).  A tcgen05.mma occupies the issuer and the tensor pipe for about
    // 45-65 cycles whatever its size, so the two chains are issued by two warps.  An issuer
    // shares its scheduler with two busy softmax warps and has no instruction-level parallelism
    // of its own, so its loop is kept to a minimum of instructions: the whole warp walks it
    // with warp-uniform values and one elected lane issues, so that descriptors are made of
    // uniform registers (a lone lane's have to be moved there one by one: 128 causal leaves of
    // 4096 rows, d = 64, 525 -> 497 us; 32 heads x 32768 rows, d = 128, 400 -> 378); descriptors
    // are two 32-bit words of which only the low one moves; waits are one probe in the common
    // case, everything unusual lives in out-of-line slow paths.
    const int i = warp - 8;
    {
      const bool el = elect_one();
      auto uni = [&](int x) { return __shfl_sync(0xffffffffu, x, 0); };
      constexpr uint32_t idesc_s = (1u << 4) | (1u << 7) | (1u << 10) | (((uint32_t)TK >> 3) << 17) | ((128u >> 4) << 24);
      constexpr uint32_t idesc_o = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | (((uint32_t)C::kOCols >> 3) << 17) | ((128u >> 4) << 24);
      // descriptor: low word = start address >> 4 | (leading byte offset >> 4) << 16,
      // high word = stride byte offset >> 4 | version 1 << 14 | 128-byte swizzle 2 << 29
      constexpr uint32_t desc_hi = (1024u >> 4) | (1u << 14) | (2u << 29);
      const uint32_t dq_lo = ((ubase + C::kOffQ + i * C::kQTile) >> 4) | (1u << 16);
      const uint32_t dk_lo0 = ((ubase + C::kOffK) >> 4) | (1u << 16);
      // V descriptors: the leading byte offset is the distance to the next 64 columns of the B
      // operand - the tile's second slab (d = 128) or the slab of ones (d = 64), whose distance
      // shrinks by one tile per stage
      const uint32_t dv_lo0 = ((ubase + C::kOffV) >> 4) | (((uint32_t)(C::kOnes ? C::kOffOnes - C::kOffV : TK * 128) >> 4) << 16);
      constexpr uint32_t dv_step = (uint32_t)(C::kTile >> 4) - (C::kOnes ? ((uint32_t)(C::kTile >> 4) << 16) : 0u);   // per stage
      const uint32_t ocol = tmem + C::kColO + C::kOCols * i;
      const uint32_t scol = tmem + 64 * C::kSBufs * i;
      const uint32_t qcol = tmem + C::kColQ + (D / 2) * i;
      bool ok = true;
      int gbase = 0;                        // global index (all items) of the item's first key tile
      int knext = 0, vnext = 0;             // next global tile whose K / V stage this issuer has to observe and release
      int ga = 0;                           // key tiles issued so far for this query tile (all items)
      int vi = 0;                           // items in which this query tile existed
      // Tiles this query tile does not look at (the other tile's own block, or everything when
      // the tile does not exist) are released when the walk passes them, but only after they
      // have arrived: a release must never overtake the loader's wait for the previous
      // release of the same stage (the barrier would wrap around unseen).  Releases go through
      // tcgen05.commit, so they also stay behind this thread's earlier MMAs.
      auto skip_k = [&](int gj) {
        for (; knext < gj && ok; ++knext) {
          ok = warp_wait<7>(bar_kfull(knext % C::NS), (knext / C::NS) & 1, s_abort, status);
          if (ok && el) umma_commit(bar_kempty(i, knext % C::NS));
        }
      };
      auto skip_v = [&](int gj) {
        for (; vnext < gj && ok; ++vnext) {
          ok = warp_wait<9>(bar_vfull(vnext % C::NS), (vnext / C::NS) & 1, s_abort, status);
          if (ok && el) umma_commit(bar_vempty(i, vnext % C::NS));
        }
      };
      int it = 0;
      HA_LDECL(b_q); HA_LDECL(b_p); HA_LDECL(b_v); HA_LDECL(b_k);
      HA_T0(tloop);
      for (; ok; ++it) {
        ok = warp_wait<22>(bar_tabfull(it & 1), (it >> 1) & 1, s_abort, status);
        if (!ok) break;
        const ItemDesc& de = *reinterpret_cast<const ItemDesc*>(smem + C::kOffDesc + (it & 1) * C::kDescBytes);
        if (uni(de.t.mode) < 0) break;
        const QTile& qd = i ? de.qb : de.qa;
        QTile q;
        q.s1 = uni(qd.s1); q.n1 = uni(qd.n1); q.s2 = uni(qd.s2); q.n2 = uni(qd.n2);
        const int total = q.n1 + q.n2;
        const int ntiles = uni(de.t.ntiles), exists = uni(qd.valid);
#ifdef HA_TC_TIMING
        if (i == 0) atomicAdd(&g_tc_timing[14], (unsigned long long)ntiles);
#endif
        // Q of this item (an issuer without a tile waits too: it may not run ahead of the others)
        HA_T0(tq);
        ok = warp_wait<6>(bar_q, it & 1, s_abort, status);
        if (!ok) break;
        HA_LACC(b_q, tq);
        fence_async_smem();
        if constexpr (C::kQTmem) {
          // (the scores of the item before have been multiplied: this item's Q was not asked for until then.  Copies and the products
          // issued after them by the same thread run in order.)
          tc_fence_after();
          if (el && total > 0) {
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) tmem_cp_128x256b(qcol + ks * 8, dq_lo + ks * (32 >> 4), desc_hi);
          }
        }
        if (total == 0 && el) mbar_arrive(bar_qfree);
        auto issue_pv = [&](int a2) {
          // ---- O += P V of key tile a2 ----------------------------------------------------------
          const int gj = gbase + tile_of(q, a2);
          const int s = gj % C::NS;
          const int gw = ga + a2;
          if (gj != vnext) skip_v(gj);
          HA_T0(tp);
          ok = ok && warp_wait<8>(bar_p(i, gw % C::kSBufs), (gw / C::kSBufs) & 1, s_abort, status);
          HA_LACC(b_p, tp);
          HA_T0(tv);
          ok = ok && warp_wait<9>(bar_vfull(s), (gj / C::NS) & 1, s_abort, status);
          HA_LACC(b_v, tv);
          // the first product of an item overwrites O: the previous item's O must have been read
          if (a2 == 0 && vi > 0) ok = ok && warp_wait<15>(bar_ofree(i), (vi - 1) & 1, s_abort, status);
          if (!ok) return;
          fence_async_smem();
          tc_fence_after();
          const uint32_t pcol = scol + 64 * (gw % C::kSBufs);
          const uint32_t dv_lo = dv_lo0 + (uint32_t)s * dv_step;
          if (el) {
            mma_ts2(ocol, pcol, dv_lo, desc_hi, idesc_o, a2 > 0);
#pragma unroll
            for (int kk = 1; kk < TK / 16; ++kk) mma_ts2(ocol, pcol + kk * 8, dv_lo + kk * (2048 >> 4), desc_hi, idesc_o, 1);
            if constexpr (PRECISE) {
#pragma unroll
              for (int kk = 0; kk < TK / 16; ++kk) mma_ts2(ocol, pcol + 32 + kk * 8, dv_lo + kk * (2048 >> 4), desc_hi, idesc_o, 1);
            }
            umma_commit(bar_vempty(i, s));
            if (a2 == total - 1) umma_commit(bar_o(i));
          }
          vnext = gj + 1;
        };
        auto issue_s = [&](int r) {
          // ---- S = Q K^T of key tile r into buffer (ga + r) % kSBufs --------------------------------
          const int gj = gbase + tile_of(q, r);
          const int s = gj % C::NS;
          const int gw = ga + r;
          if (gj != knext) skip_k(gj);
          HA_T0(tk);
          ok = ok && warp_wait<7>(bar_kfull(s), (gj / C::NS) & 1, s_abort, status);
          HA_LACC(b_k, tk);
          if (!ok) return;
          fence_async_smem();
          tc_fence_after();
          const uint32_t dcol = scol + 64 * (gw % C::kSBufs);
          const uint32_t dk_lo = dk_lo0 + (uint32_t)s * (C::kTile >> 4);
          if (el) {
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
              const uint32_t dk = dk_lo + (((ks >> 2) * (TK * 128) + (ks & 3) * 32) >> 4);
              if constexpr (C::kQTmem) mma_ts2(dcol, qcol + ks * 8, dk, desc_hi, idesc_s, ks > 0);
              else mma_ss2(dcol, dq_lo + (((ks >> 2) * (128 * 128) + (ks & 3) * 32) >> 4), dk, desc_hi, idesc_s, ks > 0);
            }
            umma_commit(bar_s(i, gw % C::kSBufs));
            umma_commit(bar_kempty(i, s));
            if (r == total - 1) umma_commit(bar_qfree);     // nothing of this item reads Q any more
          }
          knext = gj + 1;
        };
        // The S buffer of tile r held P of tile r - 2, so the product P V of that tile must be
        // issued before the scores of tile r.
        static_assert(C::kSBufs == 2, "scores run two tiles ahead");
        for (int r = 0; r < total + 2 && ok; ++r) {
          if (r >= 2) issue_pv(r - 2);
          if (ok && r < total) issue_s(r);
        }
        if (!ok) break;
        // what is left of the item's tiles (all of them for a query tile that does not exist) is
        // released K, V, K, V ... like the streamer fills them: releasing all K tiles first would
        // wait for a K tile whose stage the streamer cannot reach before a V tile is released
        for (int e = min(knext, vnext) + 1; e <= gbase + ntiles && ok; ++e) { skip_k(e); skip_v(e); }
        gbase += ntiles;
        ga += total;
        vi += exists;
      }
      if (i == 0) { HA_TACC(8, tloop); HA_TACC(12, t_cta); HA_LFLUSH(7, b_q); HA_LFLUSH(4, b_p); HA_LFLUSH(5, b_v); HA_LFLUSH(6, b_k); }
#ifdef HA_TC_TIMING
      if (i == 0) atomicAdd(&g_tc_timing[13], 1ull);
#endif
    }
    __syncwarp();
  } else if (warp == 10) {
    // ================= item preparer: row tables of an item, then its Q tiles ========================
    // Runs one item ahead of the K / V streamer where it can: a table set becomes free when the
    // softmax warps and the streamer are done with the item before the previous one, so the
    // dependent global lookups below overlap with the computation of the item in between.
    bool ok = true;
    int it = 0;
    for (; ok; ++it) {
      HA_T0(tdec);
      // Work items are handed out by a counter in global memory, in list order (heavy first): whichever CTA
      // is free takes the next one.
      int item = 0;
      if (lane == 0) item = atomicAdd(a.sched, 1);
      item = __shfl_sync(0xffffffffu, item, 0);
      const bool end = item >= a.total_pairs + a.split_pairs;
      PairDesc t = {}; QTile qa = {}, qb = {}; int lenA = 0, lenB = 0;
      const int tail = item - (a.total_pairs - a.split_pairs);     // the last pairs: each query tile an item
      const int pair = tail < 0 ? item : item - ((tail + 1) >> 1);
      if (!end) decode_pair(a, pair + (pair >= a.skip_at ? a.skip : 0), tail < 0 ? -1 : tail & 1, t, qa, qb, lenA, lenB);
      else t.mode = -1;                                   // tells every role that the list is exhausted
      if (lane == 0) HA_TACC(26, tdec);
      const int set = it & 1;
      int* s_kidx = s_kidx_all + set * kMaxNodeKeys;
      uint32_t* s_mask = s_mask_all + set * 2 * MW;
      int* s_qrow = s_qrow_all + set * 2 * 128;
      HA_T0(ttab);
      if (it >= 2) {
        ok = wait_fast<16>(bar_tabfree(set), ((it >> 1) - 1) & 1, s_abort, status);
        if (!ok) break;
      }
      if (lane == 0) HA_TACC(21, ttab);
      if (lane == 0) {
        ItemDesc* de = reinterpret_cast<ItemDesc*>(smem + C::kOffDesc + set * C::kDescBytes);
        de->t = t; de->qa = qa; de->qb = qb; de->lenA = lenA; de->lenB = lenB;
      }
      if (end) {
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_tabfull(set));
        break;
      }
      const int segrow = t.seg * g.n;                       // row coordinate of the segment's first query row ...
      const int segrow_k = t.seg * g.nk;                    // ... and of its first key row
      // Key rows as tensor-map row coordinates.  Every global load of a batch is issued before
      // the first one is used; the warp covers 32 consecutive columns per step, so one ballot
      // yields a whole word of the mask tables.  Padding columns point at a valid row (they are
      // masked, and the streamer puts zeros in the place of its values) and are masked for both tiles.
      if (is_node(t)) {
        constexpr int UB = 8;
        const int bcols = t.nbA * TK;
        const int nblk = (t.nbA + t.nbB) * TK;            // columns of the block part (multiple of 64)
        const int ncols = t.ntiles * TK;
        const int32_t* smp = a.samples + ((size_t)t.seg * g.nodes + t.node) * g.m;
        const int32_t* pk = a.perm_k + t.slice;
        const int32_t* sblk = a.smp_blk + ((size_t)t.seg * g.nodes + t.node) * g.m;
        for (int c00 = lane; c00 < nblk; c00 += 32 * UB) {
          int idx[UB];
#pragma unroll
          for (int u = 0; u < UB; ++u) {
            const int c0 = c00 + u * 32;
            idx[u] = -1;
            if (c0 < nblk) {
              const int which = c0 >= bcols;
              const int c = c0 - which * bcols;
              if (c < block_len(t.nk, g.b, which ? qb.beta : qa.beta)) idx[u] = pk[(size_t)(which ? qb.beta : qa.beta) * g.b + c];
            }
          }
#pragma unroll
          for (int u = 0; u < UB; ++u) {
            const int c0 = c00 + u * 32;
            if (c0 - lane < nblk) {                       // warp-uniform (nblk is a multiple of 32)
              const unsigned pad = __ballot_sync(0xffffffffu, idx[u] < 0);
              s_kidx[c0] = segrow_k + (idx[u] < 0 ? 0 : t.k0 + idx[u]);
              if (lane == 0) { s_mask[c0 >> 5] = pad; s_mask[MW + (c0 >> 5)] = pad; }
            }
          }
        }
        // Sampled columns: masked where the sample falls into the tile's own block (the factor
        // (1 - M^H) of Alg. 2 line 7).  The samples are an unordered multiset, so the masked ones
        // (for either query tile) are moved to the end of the sample part: only its last tile(s)
        // then carry mask bits, every other sampled tile takes the softmax warps' fast path.
        // (For a split pair too, so that the columns are added in the same order: whether a call
        // splits its pairs depends on how many heads it has, and a head's result must not.)
        if (nblk < ncols) {
          for (int wd = (nblk >> 5) + lane; wd < (ncols >> 5); wd += 32) { s_mask[wd] = 0; s_mask[MW + wd] = 0; }
          __syncwarp();
          int nfront = 0, nback = 0;                      // unmasked samples placed from the front, masked ones from the back
          float* s_bias = reinterpret_cast<float*>(smem + C::kOffBias) + set * kMaxWeightedSamples;
          const float* swl = WEIGHTED ? a.sample_wlog + ((size_t)t.seg * g.nodes + t.node) * g.m : nullptr;
          float bmax = -INFINITY;
          const unsigned lt_mask = (1u << lane) - 1u;
          for (int c00 = lane; c00 < ncols - nblk; c00 += 32 * UB) {
            int l[UB], blk[UB];
#pragma unroll
            for (int u = 0; u < UB; ++u) {
              const int c = c00 + u * 32;
              l[u] = c < g.m ? smp[c] : -1;
              blk[u] = c < g.m ? sblk[c] : -1;
            }
#pragma unroll
            for (int u = 0; u < UB; ++u) {
              const int c = c00 + u * 32;
              if (c - lane < ncols - nblk) {              // warp-uniform
                const bool valid = l[u] >= 0;
                const bool m0 = !valid || blk[u] == qa.beta;
                const bool m1 = !valid || blk[u] == qb.beta;
                const unsigned bf = __ballot_sync(0xffffffffu, valid && !(m0 || m1));
                const unsigned bb = __ballot_sync(0xffffffffu, valid && (m0 || m1));
                int pos;
                if (!valid) pos = nblk + c;                                             // padding stays where it is (behind all samples)
                else if (!(m0 || m1)) pos = nblk + nfront + __popc(bf & lt_mask);
                else pos = nblk + g.m - 1 - (nback + __popc(bb & lt_mask));
                nfront += __popc(bf); nback += __popc(bb);
                s_kidx[pos] = segrow_k + (valid ? t.k0 + l[u] : 0);
                if (WEIGHTED) {                      // weighted sampling: the column's own log2 weight travels with it
                  const float wl = valid ? swl[c] : 0.f;
                  s_bias[pos - nblk] = wl;
                  if (valid) bmax = fmaxf(bmax, wl);
                }
                if (m0) atomicOr(&s_mask[pos >> 5], 1u << (pos & 31));
                if (m1) atomicOr(&s_mask[MW + (pos >> 5)], 1u << (pos & 31));
              }
            }
          }
          if (WEIGHTED) {
#pragma unroll
            for (int o = 16; o; o >>= 1) bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, o));
            if (lane == 0) reinterpret_cast<ItemDesc*>(smem + C::kOffDesc + set * C::kDescBytes)->t.bias_max = bmax;
          }
        }
      }
      if (lane == 0) HA_TACC(23, ttab);
      // query rows of both tiles: lane l owns rows 4l .. 4l+3
      int qr[2][4];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const QTile& q = i ? qb : qa;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int r = 4 * lane + k;
          qr[i][k] = -1;
          if (q.valid && r < q.nq) qr[i][k] = is_node(t) ? t.qnode0 + a.perm_q[t.slice + q.spos0 + r] : q.q0 + r;
        }
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
        *reinterpret_cast<int4*>(s_qrow + i * 128 + 4 * lane) = make_int4(qr[i][0], qr[i][1], qr[i][2], qr[i][3]);
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_tabfull(set));       // (release: the table writes of all lanes are ordered before it by the warp barrier)
      if (lane == 0) HA_TACC(10, ttab);
      // Sorted query rows are read once in the whole forward pass, so they come from HBM: ask for
      // them now (the softmax threads gather them a whole item later) so that they are found in L2.
      if (is_node(t)) {
        const char* qbase = reinterpret_cast<const char*>(a.q) + (size_t)segrow * (D * 2);
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (qr[i][k] >= 0) {
#pragma unroll
              for (int ln = 0; ln < D * 2 / 128; ++ln)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(qbase + (size_t)qr[i][k] * (D * 2) + ln * 128));
            }
      }
      // ---- Q (the issuers must be done with the previous item's Q) ----------------------------
      HA_T0(tqf);
      if (it >= 1) {
        ok = wait_fast<17>(bar_qfree, (it - 1) & 1, s_abort, status);
        if (!ok) break;
      }
      if (lane == 0) HA_TACC(27, tqf);
      HA_T0(tqi);
      if (!is_node(t)) {
        // consecutive rows: one box per 64 columns and tile (rows past the tile's end are other
        // rows of the tensor or zeros: their results are never stored)
        if (lane == 0) {
          mbar_expect_tx(bar_q, (uint32_t)((qa.valid + qb.valid) * C::kQTile));
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            if (!(i ? qb.valid : qa.valid)) continue;
#pragma unroll
            for (int sl = 0; sl < D / 64; ++sl)
              tma_tile(ubase + C::kOffQ + i * C::kQTile + sl * (128 * 128), &maps.q, sl * 64, segrow + (i ? qb.q0 : qa.q0), bar_q);
          }
        }
        mbar_arrive(bar_q);
      } else {
        mbar_arrive(bar_q);                               // (the softmax threads gather these tiles)
      }
      if (lane == 0) { HA_TACC(25, ttab); HA_TACC(28, tqi); }
    }
    cp_async_commit();
    cp_async_wait_all();
    if (it > 0) mbar_drain(bar_q, (it - 1) & 1);
  } else {
    constexpr int CPR = D / 8;
    // ================= K / V streamer: key tiles of all items through the stage ring ====================
    // Tiles of consecutive rows: lane 0 issues one TMA box per 64 columns.  Gathered tiles: lane ->
    // column chunk cc and the row quads {4 (rq + k R) .. + 3}, R = 32 / CPR; the four row
    // coordinates of a quad come with one shared-memory load, and the swizzled destination of
    // every copy is the lane's base plus a compile-time offset (the swizzle phase (row & 7) of
    // row e of a quad is 4 (rq & 1) + e for every quad of the lane, R being even).
    bool ok = true;
    int gbase = 0;
    int it = 0;
    int k_armed = 0, v_armed = 0;                         // tiles whose K / V copies have been issued (all items)
    constexpr int R = 32 / CPR;                            // row quads covered by the warp per step
    constexpr int QUADS = (TK / 4) / R;                    // steps per tile
    const int cc = lane % CPR, rq = lane / CPR;
    uint32_t doff[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
      doff[e] = (uint32_t)((cc >> 3) * (TK * 128) + (4 * rq + e) * 128 + (((cc & 7) ^ ((4 * rq + e) & 7)) << 4));
    const char* ksrc = reinterpret_cast<const char*>(a.k) + cc * 16;
    const char* vsrc = reinterpret_cast<const char*>(a.v) + cc * 16;
    for (; ok; ++it) {
      const int set = it & 1;
      const int* s_kidx = s_kidx_all + set * kMaxNodeKeys;
      ok = wait_fast<18>(bar_tabfull(set), (it >> 1) & 1, s_abort, status);
      if (!ok) break;
      const ItemDesc& de = *reinterpret_cast<const ItemDesc*>(smem + C::kOffDesc + set * C::kDescBytes);
      const PairDesc t = de.t;
      if (t.mode < 0) break;
      const int lenA = de.lenA, lenB = de.lenB;
      const int segrow = t.seg * g.nk;                      // (keys)
      // does any of the item's key tiles have columns that do not exist?
      const bool shorts = !is_node(t) ? t.nk % TK != 0 : (lenA % TK | lenB % TK | g.m % TK) != 0;
      for (int j = 0; j < t.ntiles && ok; ++j) {
        const int gj = gbase + j;
        const int s = gj % C::NS;
        const int use = gj / C::NS;
        int4 rows[QUADS];
        if (is_node(t)) {
#pragma unroll
          for (int k = 0; k < QUADS; ++k) rows[k] = *reinterpret_cast<const int4*>(s_kidx + j * TK + 4 * (rq + k * R));
        }
        auto fill = [&](uint32_t stage, const CUtensorMap* map, const char* src, uint32_t bar) {
          if (!is_node(t)) {
            // (rows past the end of the key range are masked by the softmax warps)
            if (lane == 0) {
              mbar_expect_tx(bar, C::kTile);
#pragma unroll
              for (int sl = 0; sl < D / 64; ++sl) tma_tile(stage + sl * (TK * 128), map, sl * 64, segrow + t.k0 + j * TK, bar);
            }
            mbar_arrive(bar);
          } else {
#pragma unroll
            for (int k = 0; k < QUADS; ++k) {
              const uint32_t d = stage + k * (4 * R * 128);
              cp_async16(d + doff[0], src + (size_t)(uint32_t)rows[k].x * (D * 2));
              cp_async16(d + doff[1], src + (size_t)(uint32_t)rows[k].y * (D * 2));
              cp_async16(d + doff[2], src + (size_t)(uint32_t)rows[k].z * (D * 2));
              cp_async16(d + doff[3], src + (size_t)(uint32_t)rows[k].w * (D * 2));
            }
            cp_async_arrive_noinc(bar);
          }
        };
        HA_T0(tle);
        if (use > 0) {
          ok = wait_fast<10>(bar_kempty(0, s), (use - 1) & 1, s_abort, status);
          ok = ok && wait_fast<11>(bar_kempty(1, s), (use - 1) & 1, s_abort, status);
          if (!ok) break;
        }
        if (lane == 0) HA_TACC(11, tle);
        HA_T0(tgk);
        fill(ubase + C::kOffK + s * C::kTile, &maps.k, ksrc, bar_kfull(s));
        k_armed = gj + 1;
        if (lane == 0) HA_TACC(3, tgk);
        HA_T0(tle2);
        if (use > 0) {
          ok = wait_fast<12>(bar_vempty(0, s), (use - 1) & 1, s_abort, status);
          ok = ok && wait_fast<13>(bar_vempty(1, s), (use - 1) & 1, s_abort, status);
          if (!ok) break;
        }
        if (lane == 0) HA_TACC(11, tle2);
        HA_T0(tgv);
#ifdef HA_TEST_DROP_ARRIVAL
        {
          int drop = 0;
          if (lane == 0 && gj == 1) drop = atomicExch(&g_test_drop_armed, 0);
          if (__shfl_sync(0xffffffffu, drop, 0)) { v_armed = gj; continue; }     // nothing issued, nothing will arrive
        }
#endif
        const int have = !shorts ? TK                     // columns of the tile that exist
                         : !is_node(t) ? t.nk - j * TK
                         : j < t.nbA ? lenA - j * TK
                         : j < t.nbA + t.nbB ? lenB - (j - t.nbA) * TK : g.m - (j - t.nbA - t.nbB) * TK;
        if (have >= TK) fill(ubase + C::kOffV + s * C::kTile, &maps.v, vsrc, bar_vfull(s));
        else fill_short<D>(ubase + C::kOffV + s * C::kTile, reinterpret_cast<const char*>(a.v), is_node(t) ? s_kidx + j * TK : nullptr,
                           segrow + t.k0 + j * TK, have, bar_vfull(s));
        v_armed = gj + 1;
        if (lane == 0) HA_TACC(1, tgv);
      }
      if (!ok) break;
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_tabfree(set));       // done reading this item's key rows
      gbase += t.ntiles;
    }
    // nothing may be in flight into shared memory when the CTA exits (trivially true unless it is giving up)
    cp_async_commit();
    cp_async_wait_all();
    for (int s = 0; s < C::NS; ++s) {
      if (k_armed > s) mbar_drain(bar_kfull(s), ((k_armed - 1 - s) / C::NS) & 1);   // phase of the last tile that used stage s
      if (v_armed > s) mbar_drain(bar_vfull(s), ((v_armed - 1 - s) / C::NS) & 1);
    }
  }

  // ---- teardown ------------------------------------------------------------------------------------
  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::kTmemCols) : "memory");
  }
}

}  // namespace

#ifdef HA_TEST_DROP_ARRIVAL
extern "C" int hyperattn_test_arm_drop(int on) {
  return cudaMemcpyToSymbol(g_test_drop_armed, &on, sizeof(int)) == cudaSuccess ? 0 : -5;
}
#endif

#ifdef HA_TC_TIMING
extern "C" int hyperattn_debug_tc_timing(unsigned long long* host16, int reset) {
  if (cudaMemcpyFromSymbol(host16, g_tc_timing, sizeof(unsigned long long) * 48) != cudaSuccess) return -5;
  if (reset) { unsigned long long z[48] = {0}; cudaMemcpyToSymbol(g_tc_timing, z, sizeof(z)); }
  return 0;
}
#endif

namespace {

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                   const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// the driver's tensor-map encoder, looked up through the runtime (no link against libcuda)
EncodeTiledFn encode_tiled_fn() {
  static EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) p = nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

}  // namespace

// [rows x d] bf16, row-major; one box = 64 columns x box_rows rows (one slab of an operand tile).
// (Also used by the backward pass's launcher.)
bool encode_rows_map(CUtensorMap* m, const void* base, size_t rows, int d, int box_rows) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)d * 2};
  const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_acc_map(CUtensorMap* m, const void* base, size_t rows, int d) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)d * 4};
  const cuuint32_t box[2] = {32, 32};
  const cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

namespace {

template <int D, bool LATE, bool PRECISE, SampleRule RULE, ItemKind KIND>
cudaError_t run_build(const AttnArgs& b, const TmaMaps& maps, int grid, int* status, cudaStream_t st) {
  const cudaError_t e = allow_smem<attn_tc_kernel<D, LATE, PRECISE, RULE, KIND>>(Cfg<D>::kTotal);
  return e != cudaSuccess ? e : launch(attn_tc_kernel<D, LATE, PRECISE, RULE, KIND>, grid, 384, Cfg<D>::kTotal, st, b, maps, status);
}

// the launch of a part of the list: b.total_pairs pairs, those from b.skip_at on b.skip further on
template <int D, ItemKind KIND>
cudaError_t run_items(const AttnArgs& b, const TmaMaps& maps, int sms, int* status, cudaStream_t st) {
  const int items = b.total_pairs + b.split_pairs, grid = items < sms ? items : sms;     // persistent: one CTA per SM walks the item list
  // (fp32 partial results of d = 128: see the epilogue)
  constexpr bool CAN_BE_LATE = D == 128 && KIND != kFinalNodes;
  const bool late = CAN_BE_LATE && !b.direct && !b.part_bf16;
  if constexpr (KIND != kDenseItems) {
    if (b.capped) return late ? run_build<D, CAN_BE_LATE, false, kCapped, KIND>(b, maps, grid, status, st) : run_build<D, false, false, kCapped, KIND>(b, maps, grid, status, st);
    if (b.sample_wlog) return late ? run_build<D, CAN_BE_LATE, false, kWeighted, KIND>(b, maps, grid, status, st) : run_build<D, false, false, kWeighted, KIND>(b, maps, grid, status, st);
  }
  if (b.precise) return late ? run_build<D, CAN_BE_LATE, true, kUniform, KIND>(b, maps, grid, status, st) : run_build<D, false, true, kUniform, KIND>(b, maps, grid, status, st);
  return late ? run_build<D, CAN_BE_LATE, false, kUniform, KIND>(b, maps, grid, status, st) : run_build<D, false, false, kUniform, KIND>(b, maps, grid, status, st);
}

// pairs of the sorted nodes (the first levels: nodes get smaller from level to level)
void sorted_pairs(const AttnArgs& a, int& first, int& end) {
  int l = 0;
  while (l < a.g.levels && a.level_sorted[l]) ++l;
  first = a.n_leaf_pairs; end = l > 0 ? a.level_pair_start[l] : a.n_leaf_pairs;
}

}  // namespace

// A call with recursion gains by two launches what their own builds are faster by, about 2 %, and loses the end of the first launch and the heavy items at
// the end of the second, 10 to 15 us: from 64 pairs of query tiles for an SM on.  (Calls, us, one launch -> two: 32 heads of 131072 rows, 387 pairs
// for an SM, 6636 -> 6476, d = 128, split weights, 64 of 16384, 69 pairs, 1976 -> 1944; 4 of 100003, 38 pairs, 592 -> 593, 8 of 50000, 32 pairs, 537 -> 542,
// d = 128, 8 of 32768, 17 pairs, 514 -> 530, 16 of 9000, 8 pairs, 138 -> 149.  Capped and weighted columns, 69 pairs, 32 of 32768: caps 1951 -> 1814, value
// norms 1507 -> 1403, d = 128 caps 3002 -> 2915, fp32 results 3303 -> 3254, value norms 2192 -> 2091, fp32 results 2482 -> 2417; 139 pairs, 64 of 32768: caps
// 3809 -> 3534, value norms 3036 -> 2822.)
constexpr int kTwoLaunches = 64;
bool attention_in_two(const AttnArgs& a) {
  int first, end, sms = 0;
  sorted_pairs(a, first, end);
  return end > first && end - first < a.total_pairs && sm_count(&sms) == cudaSuccess && a.total_pairs >= (long long)kTwoLaunches * sms;
}

cudaError_t launch_attention_tc(const AttnArgs& a, int* status, cudaStream_t st) {
  if (a.total_pairs == 0) return cudaSuccess;
  const size_t rows = (size_t)a.g.G * a.g.n, rows_k = (size_t)a.g.G * a.g.nk;
  if (rows > 0x7fffffffull || rows_k > 0x7fffffffull) return cudaErrorInvalidValue;        // row coordinates are 32-bit
  if ((a.capped != 0) + (a.sample_wlog != nullptr) + (a.precise != 0) > 1) return cudaErrorInvalidValue;
  TmaMaps maps;
  if (!encode_rows_map(&maps.q, a.q, rows, a.g.d, 128) || !encode_rows_map(&maps.k, a.k, rows_k, a.g.d, TK) ||
      !encode_rows_map(&maps.v, a.v, rows_k, a.g.d, TK)) return cudaErrorInvalidValue;
  int sms = 0;
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  auto run = [&](const AttnArgs& b, auto kind) {
    constexpr ItemKind KIND = decltype(kind)::value;
    return a.g.d == 64 ? run_items<64, KIND>(b, maps, sms, status, st) : run_items<128, KIND>(b, maps, sms, status, st);
  };
  using any = std::integral_constant<ItemKind, kAnyItems>;
  using final_nodes = std::integral_constant<ItemKind, kFinalNodes>;
  using partial_nodes = std::integral_constant<ItemKind, kPartialNodes>;
  using dense = std::integral_constant<ItemKind, kDenseItems>;
  AttnArgs b = a;
  b.split_pairs = split_pairs(a, sms);
  b.skip_at = b.skip = b.tail_leaves = 0;
  int first, end;
  sorted_pairs(a, first, end);
  if (end == a.total_pairs && first == 0) return run(b, final_nodes{});
  const bool two = attention_in_two(a), no_nodes = first == end;
  if (two) {                                              // the nodes first: their items are light and equal
    b.total_pairs = end - first; b.skip = first;
    e = run(b, partial_nodes{});
    if (e != cudaSuccess) return e;
    b.total_pairs = a.total_pairs - (end - first); b.skip_at = first; b.skip = end - first; b.sched = a.sched + 1;
  }
  if (a.dense_causal && b.total_pairs == a.n_leaf_pairs) b.tail_leaves = tail_leaves(a.n_leaf_pairs / a.pairs_per_leaf, a.pairs_per_leaf, sms);
  return two || no_nodes ? run(b, dense{}) : run(b, any{});
}

}  // namespace hyperattn
