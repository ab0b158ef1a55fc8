// Backward pass: the launches (the kernel: backward.cuh).
#include "backward.cuh"

namespace hyperattn {

// backward_leaves.cu
cudaError_t launch_bwd_leaves_d64(const BwdArgs& b, const BwdMaps& maps, unsigned grid, int* status, cudaStream_t st);
// backward_nodes.cu
cudaError_t launch_bwd_nodes(const BwdArgs& b, const BwdMaps& maps, unsigned grid, int* status, cudaStream_t st);
// backward_first.cu
cudaError_t launch_bwd_first(const BwdArgs& b, const BwdMaps& maps, int results_warps, unsigned grid, int* status, cudaStream_t st);

namespace {

// fp32 accumulators rounded to bf16, 32 bytes in and 16 out per thread and pass: blockIdx.y 0: dQ, 1 and 2: dK and dV, all rows
// or (direct) the samples' rows, each to the key that it stands for.
struct ToBf16Args {
  const float4* src[3];
  uint4* dst[3];
  size_t count8[3];
  const int32_t *key_slot, *samples;     // direct (else null)
  int n, m, lg_lpr;                      // lg_lpr: log2 of the 16-byte pieces of a row
};
__global__ void __launch_bounds__(256) to_bf16_kernel(const __grid_constant__ ToBf16Args a) {
  wait_for_stream();
  const int y = blockIdx.y;
  const float4* __restrict__ src = a.src[y];
  uint4* __restrict__ dst = a.dst[y];
  for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < a.count8[y]; i += (size_t)gridDim.x * 256) {
    size_t o = i;
    if (y > 0 && a.key_slot) {
      const int slot = (int)(i >> a.lg_lpr), seg = slot / a.m;
      const size_t row = (size_t)seg * a.n + a.samples[slot];
      if (a.key_slot[row] != slot - seg * a.m) continue;                  // (another draw of the same key stands for it)
      o = (row << a.lg_lpr) + (i & ((1u << a.lg_lpr) - 1));
    }
    const float4 x = __ldcs(src + 2 * i), y4 = __ldcs(src + 2 * i + 1);
    __stcs(dst + o, make_uint4(pack2(x.x, x.y), pack2(x.z, x.w), pack2(y4.x, y4.y), pack2(y4.z, y4.w)));
  }
}

}  // namespace

// What pays is whole tiles of 128 consecutive rows (leaves, nodes that are not sorted): their dQ leaves as a box at every step, with a few
// instructions.  What costs: the boxes' code in the results warps at every short tile and at every tile of sorted rows, and, with half of the warps,
// those tiles themselves and the dK and dV of every key tile, behind which the next item waits.  So the rules weigh steps on whole tiles against key
// tiles of consecutive rows (`items`) and all other steps.  The pass, us, without boxes / with boxes / four results warps (* what the rules take).
// d = 64, causal leaves alone: 1024 leaves of 127 rows 57.5* / 59.1 / 63.6, 781 of 256 85.5* / 86.5 / 98.5, 390 of 512 106 / 104* / 115, 195 of 1024
// 150 / 148 / 150*, 130 of 1536 195 / 192 / 185*, 128 of 4096 999 / 931 / 869*; exact, 2048 heads of 127 rows 108* / 111 / 119, 781 of 256 93.6 /
// 92.1* / 100, 32 of 4096 452 / 423 / 386*; 32768 rows, 16 heads, in leaves of 512 (blocks of 64) 1764* / 1793 / 1923, 1024 1336 / 1327* / 1352,
// 2048 1385 / 1356 / 1335*, 4096 1667 / 1602 / 1539*; 64 heads of 1600 rows in leaves of 100 under nodes that are not sorted 179* / 179 / 189; no
// recursion, 32 heads of 4096 rows 131* / 134 / 142.  d = 128, without and with boxes: 1024 leaves of 100 rows 87.8* / 88.3, 781 of 256 162* / 161,
// 390 of 512 197 / 191*, 64 of 4096 945 / 827*; 32 heads of 32768 rows without recursion 1494* / 1514.
static BwdLaunch launch_of(const Geometry& g, bool with_leaves, bool with_nodes) {
  BwdLaunch r = {with_leaves && (g.causal || !g.sorted), with_nodes && g.levels > 0, kRows, 8};
  bool sorted = !r.leaves;                              // all items are tiles of sorted nodes
  long long whole = 0, other = 0, items = 0;            // per segment
  if (r.leaves) {
    const long long leaves = g.npad / g.leaf, kts = (g.leaf + kTileK - 1) / kTileK, full = g.leaf / kTileQ;
    const long long on_full = g.causal ? full * (full + 1) / 2 : kts * full, all = g.causal ? kts * (kts + 1) / 2 : kts * kts;
    whole += leaves * on_full; other += leaves * (all - on_full); items += leaves * kts;
  }
  for (int l = 0; l < g.levels && r.nodes; ++l) {
    int s, q0, k0;
    node_rows(g, l, 0, s, q0, k0);
    const long long nodes = g.causal ? 1 << l : 1;
    if (g.b < s) {
      const long long key_tiles = (g.b + kTileK - 1) / kTileK + (g.m + kTileK - 1) / kTileK;
      other += nodes * node_blocks(s, g.b) * ((g.b + kTileQ - 1) / kTileQ) * key_tiles;
    } else {
      const long long kts = (s + kTileK - 1) / kTileK, full = s / kTileQ;
      sorted = false;
      whole += nodes * kts * full; other += nodes * kts * (kts - full); items += nodes * kts;
    }
  }
  if (whole > 0 && 4 * whole >= 7 * items + other) r.out = kBoxes;
  if (g.d == 64 && whole > 0 && 2 * whole >= 9 * items + other) r.results_warps = 4;     // (kBoxes all the more)
  if (sorted) r.out = kNodes;
  return r;
}

// With recursion every row of dK and dV gets one contribution from its leaf and more from the nodes above it.  The leaves in a launch of their own,
// first, write theirs, so that the accumulators need not be cleared, and leaves and nodes take the build that is best for each.  Against that stand a
// launch and the end of the first one, where SMs run out of items: it pays from 192 MiB of accumulators on, where leaves leave as boxes.  (The pass,
// us, one launch -> two: 32 heads of 131072 rows, d = 64, 16322 -> 16046 and, another time, 16239 -> 15962, 16 of 32768 (256 MiB) 1715 -> 1708 and
// 1719 -> 1700, 8 of 32768, d = 128, (256 MiB) 1680 -> 1609 and 1669 -> 1614; 4 of 65536, d = 64, (128 MiB) 972 -> 984.)
constexpr size_t kSplitBytes = 192u << 20;
int backward_launches(const Geometry& g, BwdLaunch launches[2]) {
  launches[0] = launch_of(g, true, false);
  if (g.L > 0 && (size_t)g.G * g.n * g.d * 8 >= kSplitBytes && launches[0].out == kBoxes) {
    launches[0].out = kFirst;
    launches[1] = launch_of(g, false, true);
    return 2;
  }
  launches[0] = launch_of(g, true, true);
  return 1;
}

// a: the forward schedule (permutations, samples, tile geometry); the accumulators of gr are cleared here, but for what the first launch writes
cudaError_t launch_backward(const AttnArgs& a, const void* out, int out_fp32, const float* lse, const void* dout, float2* stat, int* sched,
                            const BwdGrads& gr, float scale, int* status, cudaStream_t st) {
  const Geometry& g = a.g;
  const size_t rows = (size_t)g.G * g.n;
  if (rows > 0x7fffffffull) return cudaErrorInvalidValue;            // TMA row coordinates are 32-bit
  BwdLaunch launches[2];
  const bool split = backward_launches(g, launches) == 2;
  {
    const unsigned grid = (unsigned)((rows * (g.d / 8) + 255) / 256);
    const uint4* d4 = reinterpret_cast<const uint4*>(dout);
    auto* kernel = g.d == 64 ? (out_fp32 ? row_stat_kernel<64, true> : row_stat_kernel<64, false>)
                             : (out_fp32 ? row_stat_kernel<128, true> : row_stat_kernel<128, false>);
    const cudaError_t e = launch(kernel, grid, 256, 0, st, d4, out, lse, stat, rows, sched, reinterpret_cast<float4*>(gr.dq),
                                 reinterpret_cast<float4*>(gr.dk), reinterpret_cast<float4*>(gr.dv), split ? 0 : gr.kv_elems / g.d);
    if (e != cudaSuccess) return e;
  }
  int sms = 0;
  if (const cudaError_t e = sm_count(&sms); e != cudaSuccess) return e;
  BwdArgs b;
  b.a = a; b.dout = reinterpret_cast<const __nv_bfloat16*>(dout); b.stat = stat; b.scale = scale; b.sched = sched;
  b.dq = gr.dq; b.dk = gr.dk; b.dv = gr.dv;
  b.dk16 = reinterpret_cast<__nv_bfloat16*>(gr.dk16); b.dv16 = reinterpret_cast<__nv_bfloat16*>(gr.dv16);
  b.key_slot = gr.key_slot; b.direct = gr.direct;
  b.leaf_ktiles = a.n_leaf_tiles ? (g.leaf + kTileK - 1) / kTileK : 0;
  b.block_ktiles = (g.b + kTileK - 1) / kTileK;
  b.smp_ktiles = (g.m + kTileK - 1) / kTileK;
  // Sampled items take at most 16 query tiles (their dK and dV leave once per item) and fewer, down to 2, where that leaves less
  // than about six items for an SM.  The pass, us, with 2 / 4 / 8 / 16 / 32 tiles (* what the rule takes): 12 heads x 4096 rows
  // 60* / 66 / 82 / 113 / 160, 32 x 32768 924 / 914 / 900 / 906* / 948 (d = 64); 32 x 4096 231 / 241* / 253 / 285 / 390, 32 x 32768
  // 1736 / 1672 / 1641 / 1637* / 1708 (d = 128); 4 causal heads of 65536 rows 1006 / 1026 / 1040 / 1027-1058* / 1105 (d = 64).
  long long steps = 0;
  for (int l = 0; l < g.levels; ++l) {
    int s, q0, k0;
    node_rows(g, l, 0, s, q0, k0);
    if (a.level_sorted[l])
      steps += (long long)(g.causal ? (1 << l) : 1) * g.G * node_blocks(s, g.b) * a.tiles_per_block * (b.smp_ktiles + b.block_ktiles);
  }
  if (b.leaf_ktiles) steps += (long long)a.leaves_per_seg * g.G * b.leaf_ktiles * (a.dense_causal ? (b.leaf_ktiles + 1) / 2 : b.leaf_ktiles);
  const long long want = steps / (6LL * sms);
  b.chunk = (int)(want < 2 ? 2 : (want > 16 ? 16 : want));
  long long items = b.leaf_ktiles ? (long long)g.G * a.leaves_per_seg * b.leaf_ktiles : 0;
  b.n_leaf_items = (int)items;
  for (int l = 0; l < g.levels; ++l) {
    int s, q0, k0;
    node_rows(g, l, 0, s, q0, k0);
    b.level_item_start[l] = (int)items;
    long long per_node = (s + kTileK - 1) / kTileK;
    if (a.level_sorted[l]) {
      const int blocks = node_blocks(s, g.b), tiles_node = blocks * a.tiles_per_block;
      per_node = (long long)b.smp_ktiles * ((tiles_node + b.chunk - 1) / b.chunk) + (long long)blocks * b.block_ktiles;
    }
    items += per_node * (g.causal ? (1 << l) : 1) * g.G;
    if (items > 0x7fffffffLL) return cudaErrorInvalidValue;
  }
  b.level_item_start[g.levels] = (int)items;
  b.total_items = (int)items;
  if (items == 0) return cudaSuccess;
  b.a.tail_leaves = a.dense_causal && (split || items == b.n_leaf_items) ? tail_leaves(b.n_leaf_items / b.leaf_ktiles, b.leaf_ktiles, sms) : 0;
  BwdMaps maps;
  if (!encode_rows_map(&maps.q, a.q, rows, g.d, 128) || !encode_rows_map(&maps.k, a.k, rows, g.d, 128) ||
      !encode_rows_map(&maps.v, a.v, rows, g.d, 128) || !encode_rows_map(&maps.dout, dout, rows, g.d, 128) ||
      !encode_acc_map(&maps.dq, gr.dq, rows, g.d)) return cudaErrorInvalidValue;
  maps.dk = maps.dv = maps.dq;
  if (!gr.direct && (!encode_acc_map(&maps.dk, gr.dk, rows, g.d) || !encode_acc_map(&maps.dv, gr.dv, rows, g.d))) return cudaErrorInvalidValue;
  auto go = [&](auto dim, auto how, unsigned grid) {
    constexpr int D = decltype(dim)::value;
    constexpr BwdOut OUT = decltype(how)::value;
    using C = Cfg<D, 8>;
    const cudaError_t allowed = allow_smem<bwd_kernel<D, OUT, 8>>(C::kTotal);
    return allowed != cudaSuccess ? allowed : launch(bwd_kernel<D, OUT, 8>, grid, C::kThreads, C::kTotal, st, b, maps, status);
  };
  using d64 = std::integral_constant<int, 64>;
  using d128 = std::integral_constant<int, 128>;
  using rows_out = std::integral_constant<BwdOut, kRows>;
  using boxes_out = std::integral_constant<BwdOut, kBoxes>;
  auto run = [&](const BwdLaunch& l) {
    const unsigned grid = b.total_items < sms ? b.total_items : sms;      // persistent: one CTA per SM
    if (l.out == kNodes) return launch_bwd_nodes(b, maps, grid, status, st);
    if (l.out == kFirst) return launch_bwd_first(b, maps, l.results_warps, grid, status, st);
    if (l.results_warps == 4) return launch_bwd_leaves_d64(b, maps, grid, status, st);
    if (g.d == 64) return l.out == kBoxes ? go(d64{}, boxes_out{}, grid) : go(d64{}, rows_out{}, grid);
    return l.out == kBoxes ? go(d128{}, boxes_out{}, grid) : go(d128{}, rows_out{}, grid);
  };
  if (split) b.total_items = b.n_leaf_items;
  cudaError_t e = run(launches[0]);
  if (e == cudaSuccess && split) {
    b.total_items = (int)items - b.n_leaf_items; b.sched = sched + 1; b.a.tail_leaves = 0;
    for (int l = g.levels; l >= 0; --l) b.level_item_start[l] -= b.n_leaf_items;
    b.n_leaf_items = 0;
    e = run(launches[1]);
  }
  if (e != cudaSuccess || !gr.dq16) return e;
  ToBf16Args c;
  const size_t elems[3] = {rows * g.d, gr.kv_elems, gr.kv_elems};
  const float* src[3] = {gr.dq, gr.dk, gr.dv};
  void* dst[3] = {gr.dq16, gr.dk16, gr.dv16};
  for (int y = 0; y < 3; ++y) {
    c.src[y] = reinterpret_cast<const float4*>(src[y]); c.dst[y] = reinterpret_cast<uint4*>(dst[y]); c.count8[y] = elems[y] / 8;
  }
  c.key_slot = gr.direct ? gr.key_slot : nullptr; c.samples = a.samples; c.n = g.n; c.m = g.m; c.lg_lpr = g.d == 64 ? 3 : 4;
  const size_t blocks = (c.count8[0] + 255) / 256;
  return launch(to_bf16_kernel, dim3((unsigned)(blocks < 16 * (size_t)sms ? blocks : 16 * (size_t)sms), gr.kv_elems ? 3 : 1), 256, 0, st, c);
}

}  // namespace hyperattn
