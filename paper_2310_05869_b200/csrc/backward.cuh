// Backward pass of the HyperAttention forward map (the paper times one in Sec. 4.2 without
// writing it down): the derivative of out = rownorm(C o exp(scale Q K^T)) V with the sortLSH
// permutations and the sampled columns - hence the coefficient matrix C of Alg. 2 lines 7
// and 9 and of the causal recursion of Alg. 4 - held fixed.  With P = rownorm(C o A), which
// the forward pass's log-sum-exp gives back as P_ij = C_ij exp(s_ij - lse_i):
//     delta_i = <dO_i, O_i>
//     dV_j   += sum_i P_ij dO_i
//     dS_ij   = P_ij (<dO_i, V_j> - delta_i)
//     dQ_i   += scale sum_j dS_ij K_j,      dK_j += scale sum_i dS_ij Q_i.
// The merge of the causal recursion needs no derivative of its own: the merged output is one
// softmax over everything a row sees, so every tile of every level uses the FINAL lse and delta.
//
// A work item is a tile of 128 KEYS and a run of query tiles (steps): the key tiles of a leaf against the query tiles from the
// diagonal on, a key tile of a sorted block against the block's query tiles, a tile of a node's sampled keys against a chunk of
// the node's query tiles.  dK and dV of the item stay in TMEM over its steps and leave once: by fp32 reductions, or, without
// recursion and for keys that are not sampled, which no other item adds to, as bf16 results (32 heads x 32768 rows, d = 128:
// accumulators that need not be cleared, added to and converted, 1936 -> 1409 us); dQ leaves after every step.  (The other way
// round - query tiles stay, dK and dV leave after every step - is twice the reductions.)
// Per step, all five products on the tcgen05 tensor cores, keys in the TMEM lanes of the first two:
//     S^T  = K Q^T,  dP^T = V dO^T      operands in 128-byte-swizzled shared memory, K-major
//     P^T  -> TMEM (bf16), dS^T -> shared memory (bf16, [key][query])          two warpgroups, 64 query columns each
//     dV  += P^T dO      A from TMEM, B = dO [query][d] MN-major
//     dK  += dS^T Q      A K-major, B = Q MN-major
//     dQ   = dS K        A = the same dS^T tile read MN-major, B = K [key][d] MN-major
// d = 64: a step's two halves of 64 queries are two chains - scores, hand-over, exponentials, hand-over - that P warpgroups 0 and 1 work
// through independently, half a step apart, with S^T, dP^T, P^T, dV, dK and dQ side by side in TMEM; the tensor pipe needs about 2000
// clocks per step, the exponentials 1024.  d = 128 has not the TMEM columns (P^T goes over S^T, dQ over dP^T): one chain, in
// which dQ comes before dK so that it leaves TMEM while dK and the next S^T are multiplied.
// What bounds it, sorted blocks (about 5000 clocks a step): the load and store unit, whose data pipe is busy for 58 % (d = 64) or 52 % (d = 128) of
// the time beside 26 and 29 % of the tensor pipe - gathered copies, dS, statistics, results through shared memory, reductions at 25 bytes per clock
// - and everything else in a chain waits behind it.  Causal leaves (less than 4000 clocks): no unit by itself; the results leave through the TMA
// unit, load and store unit and tensor pipe are level at 44 and 43 %, the exponential unit at 34, and the rest is hand-overs of a chain.  The P
// warps are busy for most of a step, with latencies: a satisfied barrier probe is 100 to 300 clocks here, a read of the statistics about as much.
// So they wait three times a step, not five, ask for 16 columns of S^T or dP^T while they work on the 16 before, and take them as 8 x 8 fragments,
// in which a thread needs the statistics of 16 queries instead of 64 (in turn, us: causal leaves of 4096 rows, 128 heads, d = 64, 1092 -> 1049 ->
// 1033; 65536 rows, 32 heads 1640 -> 1635 -> 1617; 32 heads x 32768 rows, d = 128, 1507 -> 1515 -> 1509; items of one or two steps on tiles that are
// not whole lose 1 to 3 %: 2048 heads of 127 rows, exact, 105.7 -> 108.1).  One chain -> two, us of the whole pass: 131072 rows, 32 heads 3343 ->
// 3022; causal leaves of 4096 rows, 128 heads 1167 -> 1105 (d = 64; two chains at d = 128 are 10 % slower in the leaves).  16 P warps instead of 8
// force 64 registers a thread and are slower (3160 us).
//
// Warp roles (672 threads; with four results warps 544): warps 0-7 P and dS; 8-15 (8-11) dQ, dK and dV to global memory; then a warp each: issue
// of S^T and dP^T (it also allocates TMEM); issue of the gradient products; item descriptors, K and V; Q and the row statistics; dO.
// Every wait is bounded: on a timeout the CTA raises the device status word, drains its copies, frees its TMEM and returns.
#pragma once
#include <type_traits>

#include "tc_util.cuh"

namespace hyperattn {

// tensor maps of Q, K, V, dO as [G n x d] bf16 tensors, 128-byte swizzle, box = 64 columns x 128 rows: tiles of consecutive rows
struct alignas(64) BwdMaps {
  CUtensorMap q, k, v, dout;
  CUtensorMap dq, dk, dv;      // the fp32 accumulators, box = 32 columns x 32 rows: what a results warp stages (direct: dk, dv unused)
};

struct BwdArgs {
  AttnArgs a;                  // geometry, permutations, samples
  const __nv_bfloat16* dout;   // [G, n, D]
  const float2* stat;          // [G, n] (-lse log2 e, -<dO, O>) of the rows
  float *dq, *dk, *dv;         // fp32 accumulators: [G, n, D]; direct: dk and dv [G, m, D], of the samples.  Cleared by row_stat_kernel, but for dk and
                               // dv that the leaves write in a launch before the nodes' (kFirst)
  __nv_bfloat16 *dk16, *dv16;  // direct: dK and dV of the keys without samples
  const int32_t* key_slot;     // direct: [G, n] the sample that stands for a key, -1: none (null: none for any)
  int direct;
  float scale;
  int* sched;                  // work counter of the launch (each launch of a call has its own), zero at launch
  // items: the key tiles of the leaves, then level by level those of the nodes
  int leaf_ktiles, n_leaf_items;
  int level_item_start[kMaxLevels + 1];
  int block_ktiles, smp_ktiles;          // key tiles per sorted block, per sample set
  int chunk;                             // query tiles of a sampled item
  int total_items;
};

namespace {

constexpr int kDescs = 3;              // item descriptors in flight
constexpr int kTileK = 128;            // keys per item, query rows per step
constexpr int kNoRow = (int)0x80000000;   // (rows are numbered below 2^31 - 1)

// what every role needs to know about a work item; made once, by the descriptor warp
struct BwdItem {
  int kind;              // 0 consecutive keys and queries, 1 sorted block, 2 samples; -1: the list is exhausted
  int seg, steps;
  int causal;            // the first step's tile lies on the diagonal
  int nkeys;             // keys of the tile that exist
  int k0;                // kind 0: first key row; else: first key row of the node (segment-relative)
  int q0;                // kind 0: first query row; else: first query row of the node (segment-relative)
  int qend;              // kind 0: end of the query rows
  int tn0;               // else: query tile (in sorted order) of the first step
  int nq_node;
  float wlog;            // log2 of the weight of the tile's columns
  size_t slice;          // slice offset in perm_q / rank_k
  size_t kidx;           // kind 1: the tile's first entry of perm_k; kind 2: of the samples
};

__device__ __forceinline__ bool decode_item(const BwdArgs& b, int item, BwdItem& t) {
  const AttnArgs& a = b.a;
  const Geometry& g = a.g;
  t.causal = 0; t.wlog = 0.f; t.slice = t.kidx = 0; t.tn0 = t.nq_node = t.qend = 0;
  if (item < b.n_leaf_items) {
    // leaf after leaf, heaviest key tile (the first: every query tile sees it) first; the CTAs that run at the same time work on
    // a few neighbouring leaves and find each other's rows - and dQ accumulators - in L2
    // (the last leaves of a call without node items: all heavy tiles first, see tail_leaves())
    int kt, rem;
    leaf_of_item(item, b.n_leaf_items, b.leaf_ktiles, a.tail_leaves, rem, kt);
    t.seg = rem / a.leaves_per_seg;
    const int leaf0 = (rem % a.leaves_per_seg) * g.leaf;
    t.kind = 0;
    t.nkeys = min(kTileK, g.leaf - kt * kTileK);
    t.k0 = leaf0 + kt * kTileK;
    t.causal = a.dense_causal;
    t.q0 = a.dense_causal ? t.k0 : leaf0;
    t.qend = leaf0 + g.leaf;
    t.steps = (t.qend - t.q0 + kTileQ - 1) / kTileQ;
    return true;
  }
  int level = 0;
  while (level + 1 < g.levels && item >= b.level_item_start[level + 1]) ++level;
  int idx = item - b.level_item_start[level];
  int s, q0n, k0n;
  node_rows(g, level, 0, s, q0n, k0n);
  const int nodes_lvl = g.causal ? (1 << level) : 1;
  if (!a.level_sorted[level]) {
    const int kts = (s + kTileK - 1) / kTileK;
    const int kt = idx % kts; idx /= kts;
    t.seg = idx / nodes_lvl;
    node_rows(g, level, idx % nodes_lvl, s, q0n, k0n);
    t.kind = 0;
    t.nkeys = min(kTileK, s - kt * kTileK);
    t.k0 = k0n + kt * kTileK;
    t.q0 = q0n; t.qend = q0n + s;
    t.steps = (s + kTileQ - 1) / kTileQ;
    return true;
  }
  const int blocks = node_blocks(s, g.b), tiles_node = blocks * a.tiles_per_block;
  const int chunks = (tiles_node + b.chunk - 1) / b.chunk;
  const int smp_items = b.smp_ktiles * chunks, per_node = smp_items + blocks * b.block_ktiles;
  int x = idx % per_node; idx /= per_node;
  const int j = idx % nodes_lvl;
  t.seg = idx / nodes_lvl;
  node_rows(g, level, j, s, q0n, k0n);
  t.k0 = k0n; t.q0 = q0n; t.nq_node = s;
  t.slice = ((size_t)level * g.G + t.seg) * g.nl + (g.causal ? (size_t)j * s : 0);
  if (x < smp_items) {
    const int st = x % b.smp_ktiles, node = g.causal ? (1 << level) - 1 + j : 0;
    t.kind = 2;
    t.nkeys = min(kTileK, g.m - st * kTileK);
    t.kidx = ((size_t)t.seg * g.nodes + node) * g.m + st * kTileK;
    t.tn0 = (x / b.smp_ktiles) * b.chunk;
    t.steps = min(b.chunk, tiles_node - t.tn0);
    t.wlog = log2f((float)s / (float)g.m);
  } else {
    x -= smp_items;
    const int kt = x % b.block_ktiles, beta = x / b.block_ktiles, len = block_len(s, g.b, beta);
    t.kind = 1;
    t.nkeys = min(kTileK, len - kt * kTileK);
    t.kidx = t.slice + (size_t)beta * g.b + kt * kTileK;
    t.tn0 = beta * a.tiles_per_block;
    t.steps = (len + kTileQ - 1) / kTileQ;
    if (t.nkeys <= 0) return false;                     // (a short last block has fewer key tiles)
  }
  return true;
}

// query tile of a step: its rows, and where they start (kind 0: row of the segment; else: sorted position of the node)
struct StepRows { int first, nq, beta; };
__device__ __forceinline__ StepRows step_rows(const BwdArgs& b, const BwdItem& t, int s) {
  StepRows r;
  if (t.kind == 0) { r.first = t.q0 + s * kTileQ; r.nq = min(kTileQ, t.qend - r.first); r.beta = -1; return r; }
  const int tn = t.tn0 + s, tpb = b.a.tiles_per_block;
  r.beta = tn / tpb;
  const int sub = tn - r.beta * tpb;
  r.first = r.beta * b.a.g.b + sub * kTileQ;
  r.nq = max(0, min(kTileQ, block_len(t.nq_node, b.a.g.b, r.beta) - sub * kTileQ));
  return r;
}

template <int D, int RW_>
struct Cfg {
  // warps: P and dS (SW of them, 128 / (SW / 4) query columns each), results (RW), issue of scores, of gradients, items, Q, dO; NH: chains
  static constexpr int SW = 8, RW = RW_, NH = D == 64 ? 2 : 1, kThreads = 32 * (SW + RW + 5);
  static constexpr int kTile = 128 * D * 2;           // bytes of a [128 rows x D] tile
  // buffers: K and V (an item each), Q, dO and dS (a step each); d = 128 has room for two only of Q
  static constexpr int NKV = D == 64 ? 2 : 1, NQ = 2, NDO = D == 64 ? 2 : 1, NDS = D == 64 ? 2 : 1;
  static constexpr int kOffK = 0;
  static constexpr int kOffV = kOffK + NKV * kTile;
  static constexpr int kOffQ = kOffV + NKV * kTile;
  static constexpr int kOffDO = kOffQ + NQ * kTile;
  static constexpr int kOffDS = kOffDO + NDO * kTile;
  static constexpr int kOffStage = kOffDS + NDS * 128 * 128 * 2;            // results on their way out: 4 KB per warp
  static constexpr int kOffStat = kOffStage + RW * 4096;                     // float [NQ][-lse2 | -delta][128]
  static constexpr int kOffDesc = kOffStat + NQ * 1024;
  static constexpr int kDescBytes = (sizeof(BwdItem) + 15) / 16 * 16;
  static constexpr int kOffBar = kOffDesc + kDescs * kDescBytes;
  static constexpr int kNumBar = 27 + 2 * kDescs;
  static constexpr int kOffMisc = kOffBar + 8 * kNumBar;
  static constexpr int kTotal = kOffMisc + 16;
  static_assert(kTotal <= 232448, "shared memory");
  // TMEM columns.  d = 64: S^T | dP^T | P^T | dV | dK | dQ.  d = 128: S^T (P^T over it) | dP^T (dQ over it) | dV | dK.
  static constexpr int kColS = 0, kColDP = 128;
  static constexpr int kColP = D == 64 ? 256 : 0;
  static constexpr int kPHalf = D == 64 ? 32 : 64;    // columns from the first 64 queries' P^T to the other 64's
  static constexpr int kColDV = D == 64 ? 320 : 256, kColDK = 384, kColDQ = D == 64 ? 448 : 128;
};

// (-lse log2 e, -<dO, O>) of every row: D / 8 lanes per row, 16 bytes of dO and O each (HBM-bound).
// The same threads clear the accumulators, 32 bytes of each (kv_rows rows of dK and dV), and the work counters of two launches.
template <int D, bool OUT_FP32>
__global__ void __launch_bounds__(256) row_stat_kernel(const uint4* __restrict__ dout, const void* __restrict__ out, const float* __restrict__ lse,
                                                       float2* __restrict__ stat, size_t rows, int* sched, float4* dq, float4* dk, float4* dv,
                                                       size_t kv_rows) {
  constexpr int LPR = D / 8;
  const size_t c = (size_t)blockIdx.x * 256 + threadIdx.x;
  wait_for_stream();
  if (c == 0) sched[0] = sched[1] = 0;
  const size_t row = c / LPR;
  float acc = 0.f;
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  for (size_t i = c; i < kv_rows * LPR; i += (size_t)gridDim.x * 256) { dk[2 * i] = z; dk[2 * i + 1] = z; dv[2 * i] = z; dv[2 * i + 1] = z; }
  if (row < rows) {
    dq[2 * c] = z; dq[2 * c + 1] = z;
    const uint4 x = __ldcs(dout + c);
    const uint32_t xd[4] = {x.x, x.y, x.z, x.w};
    float o[8];
    if (OUT_FP32) {
      const float4 a0 = __ldcs(reinterpret_cast<const float4*>(out) + 2 * c), a1 = __ldcs(reinterpret_cast<const float4*>(out) + 2 * c + 1);
      o[0] = a0.x; o[1] = a0.y; o[2] = a0.z; o[3] = a0.w; o[4] = a1.x; o[5] = a1.y; o[6] = a1.z; o[7] = a1.w;
    } else {
      const uint4 y = __ldcs(reinterpret_cast<const uint4*>(out) + c);
      const uint32_t yd[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) { o[2 * e] = __uint_as_float(yd[e] << 16); o[2 * e + 1] = __uint_as_float(yd[e] & 0xffff0000u); }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      acc = fmaf(o[2 * e], __uint_as_float(xd[e] << 16), acc);
      acc = fmaf(o[2 * e + 1], __uint_as_float(xd[e] & 0xffff0000u), acc);
    }
  }
#pragma unroll
  for (int o = LPR / 2; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (row < rows && c % LPR == 0) stat[row] = make_float2(-lse[row] * 1.4426950408889634f, -acc);
}

// How results leave.  kRows: every row by reductions.  kBoxes: whole tiles of consecutive rows (leaves of the recursion, nodes that are not sorted) as boxes.
// kFirst: as kBoxes, but dK and dV are written, not added: every key row has one item and nothing has been added to it yet.  (A build of its own: as a switch
// in kBoxes it made calls that do not use it 1 to 2 % slower, 11 causal heads of 5512 rows 149.2 -> 152.0 us, 128 leaves 1014 -> 1027.)
// kNodes: as kRows, where all items are tiles of sorted nodes.  (The pass, us, kRows -> kNodes, in the case of recursion also kFirst knowing that it has
// leaves alone: 12 heads of 4096 rows 59.7 -> 58.6, 10 of 20000 194.5 -> 190.4, 32 of 65536 1797 -> 1766, 32 causal of 131072 16199 -> 15871; d =
// 128, 32 of 32768 1665 -> 1657, 8 causal of 32768 1620 -> 1584.)
// RW: results warps.  With eight the block has 21 warps, six of them on one quarter of the SM, which leaves 80 registers a thread; with four it has 17
// and 96.  Whole tiles of consecutive rows need no more than four while they follow one another - a box goes out with a few instructions - and the P
// warps gain from the registers; scattered rows, and dK and dV of items of few steps, keep eight busy.  (Which build a call takes: backward_launches()
// in backward.cu, with figures.  d = 128 always has eight: 64 leaves of 4096 rows 838 us, with four 998.)
template <int D, BwdOut OUT, int RW>
__global__ void __launch_bounds__(Cfg<D, RW>::kThreads, 1) bwd_kernel(const __grid_constant__ BwdArgs b, const __grid_constant__ BwdMaps maps,
                                                                  int* status) {
  using C = Cfg<D, RW>;
  constexpr bool BOXES = OUT == kBoxes || OUT == kFirst;
  // (kFirst: leaves alone)
  auto consecutive = [](const BwdItem& t) { return OUT == kFirst || (OUT != kNodes && t.kind == 0); };
  extern __shared__ __align__(1024) uint8_t smem[];
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + C::kOffMisc);
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem + C::kOffMisc + 4);
  const uint32_t ubase = smem_u32(smem);
  const uint32_t bar0 = ubase + C::kOffBar;
  // g: step, it: item, counted over the CTA's whole work list.  (Pairs of barriers are used in turn by the steps; a waiter that
  // is a step behind never meets a phase twice.)
  // x: half of the step's queries, 64 columns of S^T and dP^T
  auto bar_s = [&](int x) { return bar0 + 8 * (0 + x); };                         // S^T of the half written
  auto bar_dp = [&](int x) { return bar0 + 8 * (2 + x); };                        // dP^T of the half written
  auto bar_h = [&](int x) { return bar0 + 8 * (4 + x); };                         // P and dS of the half written (S^T and dP^T have been read)
  auto bar_pfree = [&](int x) { return bar0 + 8 * (6 + x); };                     // dV of the half multiplied: its P is free
  auto bar_dq = [&](uint32_t g) { return bar0 + 8 * (8 + (g & 1)); };             // dQ of a step in TMEM: all its products are done, its dS is free
  auto bar_qfull = [&](uint32_t g) { return bar0 + 8 * (10 + (g & 1)); };         // Q and the row statistics of a step landed
  auto bar_qfree = [&](uint32_t g) { return bar0 + 8 * (12 + (g & 1)); };
  auto bar_dofull = [&](uint32_t g) { return bar0 + 8 * (14 + g % C::NDO); };     // dO landed
  auto bar_dofree = [&](uint32_t g) { return bar0 + 8 * (16 + (g & 1)); };        // dV multiplied: dO is free
  auto bar_kfull = [&](int it) { return bar0 + 8 * (18 + it % C::NKV); };         // K, V of an item landed
  auto bar_vfull = [&](int it) { return bar0 + 8 * (20 + it % C::NKV); };
  auto bar_kfree = [&](int it) { return bar0 + 8 * (22 + it % C::NKV); };         // dQ of the item multiplied: K and V are free
  // dQ has left TMEM; dK, dV of the item complete; dK, dV have left TMEM
  const uint32_t bar_dqfree = bar0 + 8 * 24, bar_acc = bar0 + 8 * 25, bar_accfree = bar0 + 8 * 26;
  auto bar_dfull = [&](int it) { return bar0 + 8 * (27 + it % kDescs); };         // item descriptor written
  auto bar_dfree = [&](int it) { return bar0 + 8 * (27 + kDescs + it % kDescs); };

  const AttnArgs& a = b.a;
  const Geometry& g_ = a.g;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);       // (known to be the same for the whole warp)

  if (tid == 0) *s_abort = *reinterpret_cast<volatile int*>(status);
  __syncthreads();
  if (*s_abort) return;         // (a launch in which some wait already timed out drains quickly; read early, see wait_for_stream())
  __syncthreads();
  if (tid == 0) {
    mbar_init(bar_dqfree, C::RW); mbar_init(bar_acc, 1); mbar_init(bar_accfree, C::RW);   // (one arrival per warp)
    for (int x = 0; x < 2; ++x) {
      mbar_init(bar_s(x), 2); mbar_init(bar_dp(x), 1); mbar_init(bar_h(x), C::SW / C::NH); mbar_init(bar_pfree(x), 1); mbar_init(bar_dq(x), 1);
      mbar_init(bar_qfull(x), 64); mbar_init(bar_qfree(x), 1); mbar_init(bar_dofree(x), 1);
    }
    for (int x = 0; x < C::NDO; ++x) mbar_init(bar_dofull(x), 32);
    for (int x = 0; x < C::NKV; ++x) { mbar_init(bar_kfull(x), 32); mbar_init(bar_vfull(x), 32); mbar_init(bar_kfree(x), 1); }
    // (P and results warps, two issuers, loaders of Q and dO)
    for (int x = 0; x < kDescs; ++x) { mbar_init(bar_dfull(x), 1); mbar_init(bar_dfree(x), C::SW + C::RW + 4); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == C::SW + C::RW) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *s_tmem, 0);
  wait_for_stream();
  auto desc_of = [&](int it) -> const BwdItem& { return *reinterpret_cast<const BwdItem*>(smem + C::kOffDesc + (it % kDescs) * C::kDescBytes); };
  auto wait_desc = [&](int it) { return wait_fast<1>(bar_dfull(it), (it / kDescs) & 1, s_abort, status); };
  // key row (segment-relative) of key r of an item's tile, r < nkeys
  auto key_row = [&](const BwdItem& t, int r) -> int {
    if (consecutive(t)) return t.k0 + r;
    return t.k0 + __ldg((t.kind == 1 ? a.perm_k : a.samples) + t.kidx + r);
  };
  // query row (segment-relative) of row r of a step, -1: does not exist
  auto query_row = [&](const BwdItem& t, const StepRows& sr, int r) -> int {
    if (r >= sr.nq) return -1;
    return consecutive(t) ? sr.first + r : t.q0 + __ldg(a.perm_q + t.slice + sr.first + r);
  };

  bool ok = true;
  if (warp < C::SW) {
    // ================= P and dS: warp = 32 keys, warpgroup q: query columns W q .. W q + W - 1, in two chunks of CW; a thread has a fragment's
    // share, two queries of every eight for four keys ===================
    constexpr int W = 128 / (C::SW / 4), CW = W / 2;
    static_assert(CW == 32, "a chunk's P is one TMEM store of 16 columns");
    // The thread's share of a unit of 32 keys x 16 queries is that of four 8 x 8 matrices side by side, twice: keys frow + 8 j, queries 8 k +
    // fcol and the next, value 8 (j / 2) + 4 k + 2 (j % 2) (+ 1).  A thread that has a whole key row, 64 queries, needs four times as
    // many of the statistics, and the load and store unit gives a word of them per clock whatever lanes share.
    const int row = tid & 127, frow = (row & ~31) + (lane >> 2), fcol = 2 * (lane & 3), col0 = (warp >> 2) * W, half = C::NH == 2 ? col0 >> 6 : 0;
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t p_addr = lane_addr + C::kColP + C::kPHalf * (col0 >> 6) + (col0 & 63) / 2;
    const uint64_t sc2 = pack_f2(a.scale_log2, a.scale_log2);
    uint32_t g = 0;
    for (int it = 0; ok; ++it) {
      ok = __all_sync(0xffffffffu, wait_desc(it));
      if (!ok) break;
      const BwdItem& t = desc_of(it);
      if (t.kind < 0) break;
      const int kind = t.kind, steps = t.steps, causal = t.causal, nkeys = t.nkeys;
      int kblk[4] = {-2, -2, -2, -2};                   // sampled keys: the sorted blocks the thread's keys lie in (their entries there are masked)
      if (OUT != kFirst && kind == 2) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (frow + 8 * j < nkeys) kblk[j] = __ldg(a.smp_blk + t.kidx + frow + 8 * j);
      }
#pragma unroll 1
      for (int s = 0; s < steps; ++s, ++g) {
        // entries that do not count: keys that do not exist, sampled keys of the query tile's own block, above the diagonal
        const int own = OUT != kFirst && kind == 2 ? (t.tn0 + s) / a.tiles_per_block : -1;
        const bool diag = OUT != kNodes && causal && s == 0;
        int first[4];                                   // rows of the thread: columns below it do not count
        bool masked = diag;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int r = frow + 8 * j;
          const bool dead = r >= nkeys || kblk[j] == own;
          masked = masked || dead;
          first[j] = dead ? 128 : (diag ? r : 0) - col0;
        }
        masked = __any_sync(0xffffffffu, masked);
        // (the issuer of the scores has waited for Q and the row statistics, and says so on the scores' barrier)
        ok = __all_sync(0xffffffffu, wait_fast<3>(bar_s(half), g & 1, s_abort, status));
        if (!ok) break;
        tc_fence_after();
        const float* st = reinterpret_cast<const float*>(smem + C::kOffStat) + (g & 1) * 256 + col0 + fcol;
        const uint32_t uds = ubase + C::kOffDS + (g % C::NDS) * 32768 + (col0 >> 6) * 16384 + row * 128;
        const uint32_t s_addr = lane_addr + C::kColS + col0, dp_addr = lane_addr + C::kColDP + col0;
        // Every TMEM load is under way while the 16 columns before it are worked on.
        uint32_t ra[16], rb[16];
        float p[CW];
        auto load = [&](uint32_t taddr, uint32_t (&r)[16]) { tmem_ld_frag16_issue(taddr, r); };
        auto weights = [&](uint32_t (&r)[16], int c0, int i0) {     // columns c0 .. c0 + 15 of the warpgroup, into p[i0 ..]
          if (masked) {
#pragma unroll
            for (int e = 0; e < 16; ++e)
              if (c0 + 8 * ((e >> 2) & 1) + fcol + (e & 1) < first[2 * (e >> 3) + ((e >> 1) & 1)]) r[e] = 0xff800000u;
          }
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const float2 nl = *reinterpret_cast<const float2*>(st + c0 + 8 * k);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int e = 8 * (j >> 1) + 4 * k + 2 * (j & 1);
              float x0, x1;
              unpack_f2(ffma2(pack_u2(r[e], r[e + 1]), sc2, pack_f2(nl.x, nl.y)), x0, x1);
              p[i0 + e] = ex2(x0); p[i0 + e + 1] = ex2(x1);
            }
          }
        };
        auto grads = [&](const uint32_t (&r)[16], int c0, int i0) {
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const float2 nd = *reinterpret_cast<const float2*>(st + 128 + c0 + 8 * k);
            uint32_t dd[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int e = 8 * (j >> 1) + 4 * k + 2 * (j & 1);
              float d0, d1;
              unpack_f2(fmul2(pack_f2(p[i0 + e], p[i0 + e + 1]), fadd2(pack_u2(r[e], r[e + 1]), pack_f2(nd.x, nd.y))), d0, d1);
              dd[j] = pack2(d0, d1);
            }
            // (no memory clobber: the reads of the statistics may move across; what follows is ordered by the fences below)
            asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(uds + (((((col0 & 63) + c0 + 8 * k) >> 3) ^ (row & 7)) << 4)),
                         "r"(dd[0]), "r"(dd[1]), "r"(dd[2]), "r"(dd[3]));
          }
        };
        load(s_addr, ra);
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
          const int c0 = CW * c;
          tmem_ld16_wait_regs(ra);
          load(s_addr + c0 + 16, rb);
          weights(ra, c0, 0);
          tmem_ld16_wait_regs(rb);
          if (c == 0) {
            ok = wait_fast<4>(bar_dp(half), g & 1, s_abort, status);
            // The gradients of the step before that must be done with before dS and P are written.  d = 64: dV of the half, whose P
            // lies where this one goes - and, multiplied before it, dQ of the step before that, which used this dS buffer.  d = 128:
            // dK, the last product that reads the one dS buffer.
            if (g > 0) ok = ok && wait_fast<6>(D == 64 ? bar_pfree(half) : bar_qfree(g - 1), (D == 64 ? g - 1 : (g - 1) >> 1) & 1, s_abort, status);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
          }
          load(dp_addr + c0, ra);
          weights(rb, c0 + 16, 16);
          tmem_ld16_wait_regs(ra);
          load(dp_addr + c0 + 16, rb);
          grads(ra, c0, 0);
          tmem_ld16_wait_regs(rb);
          if (c == 0) load(s_addr + CW, ra);
          grads(rb, c0 + 16, 16);
          // (d = 128: P goes over scores of this warpgroup that have been read)
          uint32_t pp[CW / 2];
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                const int e = 16 * (k >> 1) + 8 * h + 4 * (k & 1) + 2 * i;
                pp[8 * h + 2 * k + i] = pack2(p[e], p[e + 1]);
              }
          tmem_st_frag16(p_addr + 16 * c, pp);
        }
        if (!ok) break;
        tmem_wait_st();
        tc_fence_before();
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_h(half));
      }
      if (!ok) break;
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_dfree(it));
    }
  } else if (warp < C::SW + C::RW) {
    // ================= results, fp32 reductions into the accumulators: dQ after every step, dK and dV after every item; warpgroup
    // r of RW / 4 takes NC columns ===================
    const int r_ = (warp - C::SW) >> 2, row = tid & 127;
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    constexpr int NC = D * 4 / C::RW;                // columns of a result that this warpgroup takes
    // A reduction instruction whose lanes hit 32 different rows costs the L2 32 half-filled sectors: a warp's 32 rows x 32
    // columns pass through shared memory (chunks XOR-swizzled by row) and go out with eight lanes per row, four rows per instruction.
    const uint32_t stage = ubase + C::kOffStage + (warp - C::SW) * 4096;
    // grow: accumulator row of this thread's lane, < 0: none.  DIRECT: ~row of the bf16 result instead.
    auto out_rows = [&](auto direct, uint32_t taddr, float f, float* base, __nv_bfloat16* base16, int grow, uint32_t bar_done) {
      const int c = lane & 7;
#pragma unroll
      for (int p = 0; p < NC / 32; ++p) {
        uint32_t r[32];
        tmem_ld32_issue(taddr + NC * r_ + 32 * p, r);
        tmem_ld32_wait(r);
        if (p == NC / 32 - 1 && bar_done) {             // it has left TMEM
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_done);
        }
#pragma unroll
        for (int x = 0; x < 8; ++x)
          asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(stage + lane * 128 + ((x ^ (lane & 7)) << 4)),
                       "f"(__uint_as_float(r[4 * x]) * f), "f"(__uint_as_float(r[4 * x + 1]) * f),
                       "f"(__uint_as_float(r[4 * x + 2]) * f), "f"(__uint_as_float(r[4 * x + 3]) * f) : "memory");
        __syncwarp();
#pragma unroll
        for (int q0 = 0; q0 < 8; q0 += 4) {
          float4 v[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int rr = 4 * (q0 + q) + (lane >> 3);
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[q].x), "=f"(v[q].y), "=f"(v[q].z), "=f"(v[q].w)
                         : "r"(stage + rr * 128 + ((c ^ (rr & 7)) << 4)) : "memory");
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int gr = __shfl_sync(0xffffffffu, grow, 4 * (q0 + q) + (lane >> 3));
            float4* dst = reinterpret_cast<float4*>(base + (size_t)gr * D + NC * r_ + 32 * p + 4 * c);
            if (OUT == kFirst && decltype(direct)::value) { if (gr >= 0) *dst = v[q]; }
            else if (gr >= 0) atomicAdd(dst, v[q]);
            else if (decltype(direct)::value && gr != kNoRow)
              *reinterpret_cast<uint2*>(base16 + (size_t)~gr * D + NC * r_ + 32 * p + 4 * c) =
                  make_uint2(pack2(v[q].x, v[q].y), pack2(v[q].z, v[q].w));
          }
        }
        __syncwarp();
      }
    };
    // Whole tiles of consecutive rows: a box per 32 columns, added by the TMA unit (causal leaves, 128 heads x 4096 rows, d = 64, the pass, eight
    // results warps: 999 -> 931 us).  In code of its own: one routine for both slows the scattered rows by 8 %.
    auto staged_read = [&]() {                          // the boxes before have been read out of the staging buffer
      if (lane == 0) bulk_wait_read();
      __syncwarp();
    };
    auto out_boxes = [&](auto first, uint32_t taddr, float f, const CUtensorMap* map, int y, uint32_t bar_done) {
#pragma unroll
      for (int p = 0; p < NC / 32; ++p) {
        uint32_t r[32];
        tmem_ld32_issue(taddr + NC * r_ + 32 * p, r);
        tmem_ld32_wait(r);
        if (p == NC / 32 - 1 && bar_done) {             // it has left TMEM
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_done);
        }
        staged_read();
#pragma unroll
        for (int x = 0; x < 8; ++x)
          asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(stage + lane * 128 + ((x ^ (lane & 7)) << 4)),
                       "f"(__uint_as_float(r[4 * x]) * f), "f"(__uint_as_float(r[4 * x + 1]) * f),
                       "f"(__uint_as_float(r[4 * x + 2]) * f), "f"(__uint_as_float(r[4 * x + 3]) * f) : "memory");
        fence_async_smem();
        __syncwarp();
        if (lane == 0) {
          if (OUT == kFirst && decltype(first)::value) tma_put_tile(map, NC * r_ + 32 * p, y, stage);
          else tma_add_tile(map, NC * r_ + 32 * p, y, stage);
        }
      }
    };
    uint32_t g = 0;
    for (int it = 0; ok; ++it) {
      ok = __all_sync(0xffffffffu, wait_desc(it));
      if (!ok) break;
      const BwdItem& t = desc_of(it);
      if (t.kind < 0) break;
      if (BOXES) staged_read();
      const int seg_row0 = t.seg * g_.n;
      int kr = kNoRow;
      if (row < t.nkeys) {
        kr = seg_row0 + key_row(t, row);
        if (b.direct) {                                 // the key's tile has all of its gradient, or the sample's row collects it
          const int slot = !consecutive(t) && b.key_slot ? __ldg(b.key_slot + kr) : -1;
          kr = slot >= 0 ? t.seg * g_.m + slot : ~kr;
        }
      }
      const int steps = t.steps;
#pragma unroll 1
      for (int s = 0; s < steps; ++s, ++g) {
        const StepRows sr = step_rows(b, t, s);
        const bool box = BOXES && consecutive(t) && sr.nq == kTileQ;
        const int qr = query_row(t, sr, row);
        ok = __all_sync(0xffffffffu, wait_fast<7>(bar_dq(g), (g >> 1) & 1, s_abort, status));
        if (!ok) break;
        tc_fence_after();
        if (box) {
          out_boxes(std::false_type{}, lane_addr + C::kColDQ, b.scale, &maps.dq, seg_row0 + sr.first + (row & ~31), bar_dqfree);
          continue;
        }
        if (BOXES && consecutive(t)) staged_read();
        out_rows(std::false_type{}, lane_addr + C::kColDQ, b.scale, b.dq, nullptr, qr >= 0 ? seg_row0 + qr : kNoRow, bar_dqfree);
      }
      if (!ok) break;
      ok = __all_sync(0xffffffffu, wait_fast<8>(bar_acc, it & 1, s_abort, status));
      if (!ok) break;
      tc_fence_after();
      if (BOXES && consecutive(t) && t.nkeys == kTileK && !b.direct) {
        const int y = seg_row0 + t.k0 + (row & ~31);
        out_boxes(std::true_type{}, lane_addr + C::kColDV, 1.f, &maps.dv, y, 0);
        out_boxes(std::true_type{}, lane_addr + C::kColDK, b.scale, &maps.dk, y, bar_accfree);
      } else {
        if (BOXES && consecutive(t)) staged_read();
        out_rows(std::true_type{}, lane_addr + C::kColDV, 1.f, b.dv, b.dv16, kr, 0);
        out_rows(std::true_type{}, lane_addr + C::kColDK, b.scale, b.dk, b.dk16, kr, bar_accfree);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_dfree(it));
    }
    if (BOXES && lane == 0) bulk_wait_all();                     // (shared memory is read until then)
  } else if (warp < C::SW + C::RW + 2) {
    // ================= MMA issue, a warp for the scores and one for the gradients ==================
    // The whole warp walks through this code together and one elected lane issues: descriptors and addresses are then made of
    // uniform registers, which the instructions take directly (a lone lane's have to be moved there one by one).
    const bool el = elect_one();
    auto uni = [&](int x) { return __shfl_sync(0xffffffffu, x, 0); };
    // descriptors: low word = start >> 4 | (leading byte offset >> 4) << 16, high word = stride 1024 B | version | 128-byte swizzle
    constexpr uint32_t desc_hi = (1024u >> 4) | (1u << 14) | (2u << 29);
    constexpr uint32_t kSlab = 128 * 128;               // bytes of one [128 rows x 64 columns] slab
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);
    constexpr uint32_t idesc_s = idesc | (((128u / C::NH) >> 3) << 17);                                  // K-major x K-major, N = 128 / NH
    constexpr uint32_t idesc_n = idesc | (1u << 16) | (((uint32_t)D >> 3) << 17);                        // K-major (or TMEM) x MN-major, N = D
    constexpr uint32_t idesc_t = idesc | (1u << 15) | (1u << 16) | (((uint32_t)D >> 3) << 17);           // MN-major x MN-major, N = D
    const uint32_t base = ubase >> 4;
    auto kmajor = [&](uint32_t off, int ks) { return base + ((off + (ks >> 2) * kSlab + (ks & 3) * 32) >> 4) + (1u << 16); };
    auto mnmajor = [&](uint32_t off, int kk) { return base + ((off + kk * 2048) >> 4) + ((kSlab >> 4) << 16); };
    uint32_t g = 0;
    if (warp == C::SW + C::RW) {
      // S^T and dP^T of a half, as soon as the half's warps have read the step before
      for (int it = 0; ok; ++it) {
        ok = __all_sync(0xffffffffu, wait_desc(it)) != 0;
        if (!ok || uni(desc_of(it).kind) < 0) break;
        const int steps = uni(desc_of(it).steps);
        const uint32_t k = C::kOffK + (it % C::NKV) * C::kTile, v = C::kOffV + (it % C::NKV) * C::kTile;
        ok = warp_wait<9>(bar_kfull(it), (it / C::NKV) & 1, s_abort, status);
#pragma unroll 1
        for (int s = 0; s < steps && ok; ++s, ++g) {
          const uint32_t q = C::kOffQ + (g & 1) * C::kTile, o = C::kOffDO + (g % C::NDO) * C::kTile;
          ok = warp_wait<10>(bar_qfull(g), (g >> 1) & 1, s_abort, status);
          auto scores = [&](int x) {
            // (d = 128: P lies over the scores)
            if (g > 0) ok = ok && warp_wait<14>(D == 64 ? bar_h(x) : bar_pfree(x), (g - 1) & 1, s_abort, status);
            if (!ok) return;
            if (x == 0) fence_async_smem();
            tc_fence_after();
            if (el) {
#pragma unroll
              for (int ks = 0; ks < D / 16; ++ks)
                mma_ss2(tmem + C::kColS + 64 * x, kmajor(k, ks), kmajor(q + x * 8192, ks), desc_hi, idesc_s, ks > 0);
              umma_commit(bar_s(x));
              mbar_arrive(bar_s(x));                     // (passes on that Q and the row statistics are there)
            }
          };
          auto dprob = [&](int x) {
            if (x == 0) {
              if (s == 0) ok = ok && warp_wait<11>(bar_vfull(it), (it / C::NKV) & 1, s_abort, status);
              ok = ok && warp_wait<13>(bar_dofull(g), (g / C::NDO) & 1, s_abort, status);
              if (D == 128 && g > 0) ok = ok && warp_wait<12>(bar_dqfree, (g - 1) & 1, s_abort, status);   // (dQ lies over dP)
              fence_async_smem();
              if (D == 128) tc_fence_after();
            }
            if (!ok) return;
            if (el) {
#pragma unroll
              for (int ks = 0; ks < D / 16; ++ks)
                mma_ss2(tmem + C::kColDP + 64 * x, kmajor(v, ks), kmajor(o + x * 8192, ks), desc_hi, idesc_s, ks > 0);
              umma_commit(bar_dp(x));
            }
          };
#pragma unroll
          for (int x = 0; x < C::NH; ++x) { scores(x); dprob(x); }
          if (!ok) break;
        }
        if (ok && el) mbar_arrive(bar_dfree(it));
      }
    } else {
      for (int it = 0; ok; ++it) {
        ok = __all_sync(0xffffffffu, wait_desc(it)) != 0;
        if (!ok || uni(desc_of(it).kind) < 0) break;
        const int steps = uni(desc_of(it).steps);
        const uint32_t kt = C::kOffK + (it % C::NKV) * C::kTile;
#pragma unroll 1
        for (int s = 0; s < steps && ok; ++s, ++g) {
          const bool last = s + 1 == steps;
          const uint32_t q = C::kOffQ + (g & 1) * C::kTile, o = C::kOffDO + (g % C::NDO) * C::kTile, ds = C::kOffDS + (g % C::NDS) * (128 * 128 * 2);
          constexpr int KK = 8 / C::NH;                 // 16-query slices of a half
          auto grad_v = [&](int x) {
            ok = warp_wait<14>(bar_h(x), g & 1, s_abort, status);
            if (x == 0 && s == 0 && it > 0) ok = ok && warp_wait<15>(bar_accfree, (it - 1) & 1, s_abort, status);
            if (!ok) return;
            fence_async_smem();
            tc_fence_after();
            if (el) {
#pragma unroll
              for (int kk = x * KK; kk < (x + 1) * KK; ++kk)
                mma_ts2(tmem + C::kColDV, tmem + C::kColP + (kk >> 2) * C::kPHalf + (kk & 3) * 8, mnmajor(o, kk), desc_hi, idesc_n,
                        (s > 0 || kk > 0) ? 1u : 0u);
              umma_commit(bar_pfree(x));
              if (x + 1 == C::NH) umma_commit(bar_dofree(g));
            }
          };
          auto grad_k = [&](int x) {
            if (ok && el) {
#pragma unroll
              for (int kk = x * KK; kk < (x + 1) * KK; ++kk)
                mma_ss2(tmem + C::kColDK, kmajor(ds, kk), mnmajor(q, kk), desc_hi, idesc_n, (s > 0 || kk > 0) ? 1u : 0u);
              if (x + 1 == C::NH) {
                umma_commit(bar_qfree(g));
                if (last) umma_commit(bar_acc);
              }
            }
          };
          auto grad_q = [&]() {
            if (D == 64 && g > 0) ok = ok && warp_wait<12>(bar_dqfree, (g - 1) & 1, s_abort, status);
            if (!ok) return;
            tc_fence_after();
            if (el) {
#pragma unroll
              for (int kk = 0; kk < 8; ++kk) mma_ss2(tmem + C::kColDQ, mnmajor(ds, kk), mnmajor(kt, kk), desc_hi, idesc_t, kk > 0);
              umma_commit(bar_dq(g));
              if (last) umma_commit(bar_kfree(it));
            }
          };
          if (D == 64) {
            grad_v(0); grad_k(0);
            if (!ok) break;
            grad_v(1); grad_k(1);
            grad_q();
          } else {
            grad_v(0);
            grad_q();                                   // (the next dP^T waits until dQ has left)
            grad_k(0);
          }
        }
        if (ok && el) mbar_arrive(bar_dfree(it));
      }
    }
    __syncwarp();
  } else {
    // ================= loaders, a warp each: Q and row statistics; dO; items, K and V ==================
    // Whole tiles of consecutive rows: lane 0 issues TMA boxes.  Others: rows gathered in 16-byte chunks, lane -> chunk cc of row
    // k RPI + crow of instruction k; lane l holds the row numbers of rows l, l + 32, ..., handed round by shuffles.
    // Rows of a short tile that do not exist are zeros: their weights are zero, but zero times a NaN or an infinity of
    // some other leaf, block or head would not be.
    constexpr int CPR = D / 8, RPI = 32 / CPR, NSW = 8 / RPI;
    const int cc = lane % CPR, crow = lane / CPR;
    uint32_t sw[NSW];                                    // byte offset of (row k RPI + crow, chunk cc) in its slab is k RPI 128 + sw[k % NSW]
#pragma unroll
    for (int k = 0; k < NSW; ++k) sw[k] = (uint32_t)(crow * 128 + (((cc & 7) ^ ((k * RPI + crow) & 7)) << 4));
    // (v: a valid row also where none exists.  The short tiles' copies are a rolled loop at d = 128: a second set of 64 in line at every
    // call makes the pass slower also where no tile is short - 32 heads x 32768 rows 1367 -> 1380 us; without the short form 1357.)
    auto gather = [&](int rows, uint32_t dst, const __nv_bfloat16* base, const int (&v)[4], uint32_t bar) {
      const char* src = reinterpret_cast<const char*>(base) + cc * 16;
      const uint32_t d = dst + (cc >> 3) * (128 * 128);
      if (rows == 128) {
#pragma unroll
        for (int k = 0; k < 128 / RPI; ++k) {
          const int rw = __shfl_sync(0xffffffffu, v[k * RPI / 32], (k * RPI & 31) + crow);
          cp_async16(d + k * RPI * 128 + sw[k % NSW], src + (size_t)(uint32_t)rw * (D * 2));
        }
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
#pragma unroll (D == 64 ? 32 / RPI / NSW : 1)
          for (int k0 = 0; k0 < 32 / RPI; k0 += NSW) {
#pragma unroll
            for (int k1 = 0; k1 < NSW; ++k1) {
              const int r = (k0 + k1) * RPI + crow, rw = __shfl_sync(0xffffffffu, v[u], r);
              cp_async16_or_zero(d + (32 * u + (k0 + k1) * RPI) * 128 + sw[k1], src + (size_t)(uint32_t)rw * (D * 2), 32 * u + r < rows);
            }
          }
        }
      }
      cp_async_arrive_noinc(bar);
    };
    auto boxes = [&](uint32_t dst, int rows, const CUtensorMap* map, int y, uint32_t bar) {
      if (lane == 0) {
        mbar_expect_tx(bar, rows * D * 2);
#pragma unroll
        for (int sl = 0; sl < D / 64; ++sl) tma_tile(dst + sl * rows * 128, map, sl * 64, y, bar);
      }
      __syncwarp();
      mbar_arrive(bar);
    };
    if (warp > C::SW + C::RW + 2) {
      const bool is_q = warp == C::SW + C::RW + 3;
      const int nbuf = is_q ? C::NQ : C::NDO;
      // The next step's row numbers are asked for before this step's copies, its statistics after them, across items: under this
      // kernel's load a read takes about 2000 clocks, and in line with the copies two of them made the round of this warp longer than
      // a step.  (131072 rows, d = 64, 32 heads: 3560 -> 3343 us for the whole pass.)
      struct Step {
        int rel[4];                                      // row lane + 32 u of the query tile, relative to base (rows that do not exist: 0)
        int base, nq;                                    // nq: rows that exist
        int y;                                           // whole tiles of consecutive rows: the first (else -1)
        float wlog;
      };
      Step s0, s1;                                       // this step, the next
      float2 n0[4];                                      // statistics of this step
      int have = 0, pit = 0, ps = 0;                     // steps asked for; item and step to ask for next
      bool end = false;
      auto ask = [&](Step& d) {
        const BwdItem& t = desc_of(pit);
        const StepRows sr = step_rows(b, t, ps);
        d.base = t.seg * g_.n + t.q0; d.nq = sr.nq; d.wlog = t.wlog;
        d.y = consecutive(t) && sr.nq == 128 ? t.seg * g_.n + sr.first : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int r = lane + 32 * u;
          d.rel[u] = r < sr.nq ? (consecutive(t) ? sr.first - t.q0 + r : __ldg(a.perm_q + t.slice + sr.first + r)) : 0;
        }
        ++have;
        if (++ps == t.steps) {
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_dfree(pit));
          ps = 0; ++pit;
        }
      };
      // the next step, if its item is known by now
      auto more = [&]() {
        if (end) return false;
        if (ps == 0) {
          if (!__all_sync(0xffffffffu, mbar_test(bar_dfull(pit), (pit / kDescs) & 1))) return false;
          if (desc_of(pit).kind < 0) { end = true; return false; }
        }
        return true;
      };
      auto stats = [&]() {
#pragma unroll
        for (int u = 0; u < 4; ++u) n0[u] = lane + 32 * u < s0.nq ? __ldg(b.stat + s0.base + s0.rel[u]) : make_float2(-INFINITY, 0.f);
      };
      for (uint32_t g = 0; ok; ++g) {
        if (have == 0) {
          if (!end && ps == 0) ok = __all_sync(0xffffffffu, wait_desc(pit));
          if (!ok || !more()) break;
          ask(s0);
          if (is_q) stats();
        }
        if (more()) ask(s1);
        const uint32_t bar = is_q ? bar_qfull(g) : bar_dofull(g);
        const uint32_t dst = ubase + (is_q ? C::kOffQ + (g % C::NQ) * C::kTile : C::kOffDO + (g % C::NDO) * C::kTile);
        if (g >= (uint32_t)nbuf) {
          const uint32_t last = g - nbuf;                // (the step that used the buffer before)
          ok = __all_sync(0xffffffffu, wait_fast<16>(is_q ? bar_qfree(last) : bar_dofree(last), (last >> 1) & 1, s_abort, status));
          if (!ok) break;
        }
        if (is_q) {
          float* st = reinterpret_cast<float*>(smem + C::kOffStat) + (g % C::NQ) * 256;
#pragma unroll
          for (int u = 0; u < 4; ++u) { st[lane + 32 * u] = n0[u].x + s0.wlog; st[128 + lane + 32 * u] = n0[u].y; }
          mbar_arrive(bar);
        }
        if (OUT != kNodes && s0.y >= 0) boxes(dst, 128, is_q ? &maps.q : &maps.dout, s0.y, bar);
        else {
          int v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) v[u] = s0.base + s0.rel[u];
          gather(s0.nq, dst, is_q ? a.q : b.dout, v, bar);
        }
        s0 = s1;
        --have;
        if (is_q && have > 0) stats();
      }
      cp_async_commit();
      cp_async_wait_all();
      // (nothing may be in flight into shared memory when the CTA exits - trivially true unless it is giving up)
      if (!ok)
        for (int x = 0; x < nbuf; ++x) { mbar_drain(is_q ? bar_qfull(x) : bar_dofull(x), 0); mbar_drain(is_q ? bar_qfull(x) : bar_dofull(x), 1); }
    } else {
      // Work items are handed out by a counter in global memory, in list order (heavy first); the first gridDim.x need none.
      int item = blockIdx.x;
      for (int it = 0; ok; ++it) {
        BwdItem t;
        for (;;) {
          if (it > 0 || item < 0) {
            if (lane == 0) item = gridDim.x + atomicAdd(b.sched, 1);
            item = __shfl_sync(0xffffffffu, item, 0);
          }
          if (item >= b.total_items) { t.kind = -1; break; }
          if (decode_item(b, item, t)) break;
          item = -1;
        }
        if (it >= kDescs) {
          ok = __all_sync(0xffffffffu, wait_fast<17>(bar_dfree(it), (it / kDescs - 1) & 1, s_abort, status));
          if (!ok) break;
        }
        if (lane == 0) {
          *reinterpret_cast<BwdItem*>(smem + C::kOffDesc + (it % kDescs) * C::kDescBytes) = t;
          mbar_arrive(bar_dfull(it));
        }
        __syncwarp();
        if (t.kind < 0) break;
        const uint32_t dk = ubase + C::kOffK + (it % C::NKV) * C::kTile, dv = ubase + C::kOffV + (it % C::NKV) * C::kTile;
        const int seg_row0 = t.seg * g_.n;
        const bool box = consecutive(t) && t.nkeys == 128;
        int v[4] = {0, 0, 0, 0};
        if (!box) {
#pragma unroll
          for (int u = 0; u < 4; ++u) v[u] = seg_row0 + key_row(t, min(lane + 32 * u, t.nkeys - 1));
        }
        if (it >= C::NKV) ok = __all_sync(0xffffffffu, wait_fast<18>(bar_kfree(it), (it / C::NKV - 1) & 1, s_abort, status));
        if (!ok) break;
        if (box) boxes(dk, 128, &maps.k, seg_row0 + t.k0, bar_kfull(it));
        else gather(t.nkeys, dk, a.k, v, bar_kfull(it));
        if (box) boxes(dv, 128, &maps.v, seg_row0 + t.k0, bar_vfull(it));
        else gather(t.nkeys, dv, a.v, v, bar_vfull(it));
      }
      cp_async_commit();
      cp_async_wait_all();
      if (!ok) for (int x = 0; x < C::NKV; ++x) for (int y = 0; y < 2; ++y) { mbar_drain(bar_kfull(x), y); mbar_drain(bar_vfull(x), y); }
    }
  }

  // ---- teardown ------------------------------------------------------------------------------------
  tc_fence_before();
  __syncthreads();
  if (warp == C::SW + C::RW) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

}  // namespace
}  // namespace hyperattn
