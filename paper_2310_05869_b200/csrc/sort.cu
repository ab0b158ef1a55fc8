// sortLSH permutations (Alg. 1 line 3) and sampled columns (Alg. 2 line 4).
//
// The argsort is a stable counting sort: bucket ids have at most 256 values, so one pass of
//   per-chunk histogram (done by the hash kernel) -> per-node exclusive scan -> stable scatter
// orders every (level, segment, node, side) slice.  A chunk never straddles a recursion
// node, so the histogram of a chunk is the same at every level of the causal recursion and
// only the scan differs per level.  Ties keep the original row order, which makes the
// permutation unique.
#include "vnorm_common.cuh"

namespace hyperattn {
namespace {

struct SortArgs {
  const uint8_t* ids;     // queries [G, n], then keys [G, nk]
  const uint32_t* hist;   // queries [G, chunks_per_seg, 256], then keys [G, chunks_per_seg_k, 256]
  uint32_t* offs;         // queries [levels, G, chunks per (level, segment), 256], then the same for keys
  int32_t *perm_q, *perm_k, *rank_k;  // [levels, G, nl]
  int32_t* smp_blk;       // [G, nodes, m] sorted block of every sampled key, or null
  int32_t* key_slot;      // [G, nk] one of the samples that drew the key, or -1 (null: not wanted)
  Geometry g;
  int side_mask;          // bit s set: side s is sorted (both, unless a caller wants one side only)
};

// chunk index (within a segment) of the first chunk of node j's query (side 0) or key (side 1) rows
// (chunks that lie beyond the last row have empty histograms and place nothing)
__device__ __forceinline__ int node_first_chunk(const Geometry& g, int level, int j, int side, int& nchunks) {
  if (!g.causal) { nchunks = side_cps(g, side); return 0; }
  int s, q0, k0;
  node_rows(g, level, j, s, q0, k0);
  nchunks = (s / g.unit) * g.chunks_per_unit;
  return ((side == 0 ? q0 : k0) / g.unit) * g.chunks_per_unit;
}
__device__ __forceinline__ size_t side_hist_base(const Geometry& g, int side) { return side ? (size_t)g.G * g.chunks_per_seg * kBuckets : 0; }
__device__ __forceinline__ size_t side_offs_base(const Geometry& g, int side) {
  return side ? (size_t)g.levels * g.G * side_cpl(g, 0) * kBuckets : 0;
}
__device__ __forceinline__ size_t side_ids_base(const Geometry& g, int side) { return side ? (size_t)g.G * g.n : 0; }

struct SampleArgs {
  int32_t* samples;  // [G, nodes, m]
  int32_t* tpos;     // capped row sums only (else null): [G, nodes, m] probe positions of Alg. 2 line 2
  float* ltau;       // capped row sums only: [G, nodes], set to -inf here (the probe pass takes a maximum into it)
  Geometry g;
  uint32_t k0, k1;
  int draw;          // 1: the samples are drawn by this launch
  int* sched;        // zeroed by the launch (null: nothing)
};

// Alg. 2 line 4: m i.i.d. uniform key indices per (segment, node); word w of Philox call c is
// sample 4c + w, mapped to [0, N) by a 64-bit multiply-high.  `block` of `nblocks` blocks.
__device__ __forceinline__ void samples_body(const SampleArgs& a, int block, int nblocks) {
  const Geometry& g = a.g;
  const int calls = (g.m + 3) / 4;
  const size_t total = (size_t)g.G * g.nodes * calls;
  for (size_t i = (size_t)block * blockDim.x + threadIdx.x; i < total; i += (size_t)nblocks * blockDim.x) {
    const int c = (int)(i % calls);
    const int nd = (int)((i / calls) % g.nodes);
    const int seg = (int)(i / ((size_t)calls * g.nodes));
    const int level = g.causal ? 31 - __clz(nd + 1) : 0;
    const uint32_t N = g.causal ? (uint32_t)(g.npad >> (level + 1)) : (uint32_t)g.nk;
    const Philox4 x = philox4x32_10((uint32_t)c, (uint32_t)(g.seg0 + seg), (uint32_t)nd, kDomainSamples, a.k0, a.k1);
    int32_t* dst = a.samples + ((size_t)seg * g.nodes + nd) * g.m;
#pragma unroll
    for (int w = 0; w < 4; ++w)
      if (4 * c + w < g.m) dst[4 * c + w] = (int32_t)__umulhi(x.x[w], N);
    if (a.tpos) {
      // Alg. 2 line 2: the probe rows T, m i.i.d. uniform positions of the node's sorted query order, from a
      // stream of their own (the node may have fewer queries than keys; none: nothing is read later)
      int s, q0, k0;
      node_rows(g, level, g.causal ? nd + 1 - (1 << level) : 0, s, q0, k0);
      const uint32_t NQ = (uint32_t)node_queries(g, s, q0);
      const Philox4 y = philox4x32_10((uint32_t)c, (uint32_t)(g.seg0 + seg), (uint32_t)nd, kDomainRowSubset, a.k0, a.k1);
      int32_t* dt = a.tpos + ((size_t)seg * g.nodes + nd) * g.m;
#pragma unroll
      for (int w = 0; w < 4; ++w)
        if (4 * c + w < g.m) dt[4 * c + w] = (int32_t)__umulhi(y.x[w], NQ);
      if (c == 0) a.ltau[(size_t)seg * g.nodes + nd] = -INFINITY;
    }
  }
}

// One CTA per (side, level, segment, node): thread v of each of NG groups owns bucket v of its share of the node's chunks.  All
// latency: one group reads the chunks in batches one after the other, four groups a quarter each.  The launch carries the sampling as extra
// blocks, or the cumulative sums of the value norms (NG = 4; all are tiny and independent of each other).
template <int NG>
__global__ void __launch_bounds__(256 * NG) sort_scan_kernel(SortArgs a, SampleArgs sa, VnormArgs va, int scan_blocks, int sample_blocks) {
  __shared__ uint32_t s_tot[NG][kBuckets], s_warp[NG][8];
  wait_for_stream();
  if (sa.sched && blockIdx.x == 0 && threadIdx.x == 0) sa.sched[0] = sa.sched[1] = 0;
  if ((int)blockIdx.x >= scan_blocks) {
    const int x = blockIdx.x - scan_blocks;
    if (x < sample_blocks) samples_body(sa, x, sample_blocks);
    else if (NG == 4) {
      const int parts = (va.nk + 4095) / 4096;
      vnorm_scan_body(va, (x - sample_blocks) / parts, (x - sample_blocks) % parts);
    }
    return;
  }
  const Geometry& g = a.g;
  const int v = threadIdx.x & (kBuckets - 1), grp = threadIdx.x / kBuckets, lane = threadIdx.x & 31;
  int cta = blockIdx.x;
  // nodes of all levels are enumerated heap-style: per (side, seg): sum over levels of 2^level
  const int nodes_per = g.causal ? g.nodes : 1;
  const int nd = cta % nodes_per; cta /= nodes_per;
  const int seg = cta % g.G;
  const int side = cta / g.G;
  if (!((a.side_mask >> side) & 1)) return;
  int level = 0, j = nd;
  if (g.causal) { level = 31 - __clz(nd + 1); j = nd + 1 - (1 << level); }
  int nchunks;
  const int first = node_first_chunk(g, level, j, side, nchunks);
  const uint32_t* h = a.hist + level * hist_level_stride(g) + side_hist_base(g, side) + ((size_t)seg * side_cps(g, side) + first) * kBuckets;
  const int lvl_chunk0 = g.causal ? j * nchunks : 0;
  uint32_t* o = a.offs + side_offs_base(g, side) + (((size_t)level * g.G + seg) * side_cpl(g, side) + lvl_chunk0) * kBuckets;
  constexpr int UB = NG == 1 ? 8 : 16;                   // loads in flight
  const int share = (nchunks + NG - 1) / NG, begin = grp * share, end = min(nchunks, begin + share);
  uint32_t t[UB];
  auto load = [&](int c0) {
#pragma unroll
    for (int u = 0; u < UB; ++u) t[u] = c0 + u < end ? h[(size_t)(c0 + u) * kBuckets + v] : 0u;
  };
  // pass 1: bucket totals of the share
  uint32_t mine = 0;
  for (int c0 = begin; c0 < end; c0 += UB) {
    load(c0);
#pragma unroll
    for (int u = 0; u < UB; ++u) mine += t[u];
  }
  s_tot[grp][v] = mine;
  __syncthreads();
  // exclusive scan over v of the node's bucket totals, in every group; run: also what the bucket has in the shares before this one
  uint32_t tot = 0, run = 0;
#pragma unroll
  for (int e = 0; e < NG; ++e) { const uint32_t x = s_tot[e][v]; tot += x; if (e < grp) run += x; }
  uint32_t incl = tot;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t x = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += x;
  }
  if (lane == 31) s_warp[grp][v >> 5] = incl;
  __syncthreads();
  run += incl - tot;
  for (int e = 0; e < (v >> 5); ++e) run += s_warp[grp][e];
  // pass 2: first position of bucket v in every chunk = buckets before v + the same bucket in earlier chunks
  for (int c0 = begin; c0 < end; c0 += UB) {
    if (share > UB) load(c0);                            // (else they are still there)
#pragma unroll
    for (int u = 0; u < UB; ++u) {
      if (c0 + u < end) o[(size_t)(c0 + u) * kBuckets + v] = run;
      run += t[u];
    }
  }
}

// One CTA per (side, level, segment, chunk of the level): stable placement of <= g.chunk rows.  SCAN: the launch takes over
// the scan's work where nodes have few chunks - every CTA adds up the histograms of its node's chunks by itself and extra blocks draw the
// samples - which saves a small call one launch of three.
// Bound by instruction issue.  A row's place among the rows of its warp's range comes from a word per bucket into which the lanes of a group put a bit
// each, and is kept in a register until the ranges before it are counted, so that every row is looked up once.  (Before: a histogram of the ranges,
// then a ballot per id bit and group.  Kernel, us, ballots -> words: 32 heads x 131072 rows 47.9 -> 42.6, 32 causal ones 129 -> 110, 4 causal x 100003
// 19.5 -> 17.1; with the scan's work in it 32 x 32768, d = 128, 17.5 -> 17.4 - five CTAs an SM; four 18.9, six, with spills, 17.4 to 18.3 -, 32 x 4096 5.7 -> 5.5.
// Rows that are all in one bucket set their bits one after another, as the histogram counted them before.)
template <bool SCAN>
__global__ void __launch_bounds__(256, SCAN ? 5 : 6) sort_scatter_kernel(SortArgs a, SampleArgs sa, int place_blocks) {
  // per warp and bucket: lanes of the row group at hand that are in the bucket; rows of the warp's range counted so far, then its first position
  __shared__ __align__(16) uint2 s_bkt[8][kBuckets];
  const Geometry& g = a.g;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (SCAN && (int)blockIdx.x >= place_blocks) {
    wait_for_stream();
    samples_body(sa, blockIdx.x - place_blocks, gridDim.x - place_blocks);
    return;
  }
  int cta = blockIdx.x;
  const int ctas0 = ((a.side_mask & 1) ? g.levels * g.G * side_cpl(g, 0) : 0);
  const int side = (cta >= ctas0 || !(a.side_mask & 1)) ? 1 : 0;
  if (side) cta -= ctas0;
  const int cpl = side_cpl(g, side);
  const int lc = cta % cpl; cta /= cpl;
  const int seg = cta % g.G;
  const int level = cta / g.G;
  // which node and which row range this chunk is
  int s, q0, k0, j = 0, nchunks_node = cpl;
  if (g.causal) {
    s = g.npad >> (level + 1);
    nchunks_node = (s / g.unit) * g.chunks_per_unit;
    j = lc / nchunks_node;
  }
  node_rows(g, level, j, s, q0, k0);
  const int cn = lc - j * nchunks_node;                  // chunk within the node
  const int cpu_s = side_cpu(g, side), unit_s = side_unit(g, side);
  const int u = cn / cpu_s, cu = cn % cpu_s;
  const int local0 = u * unit_s + cu * g.chunk;       // first row, relative to the node
  const int row0 = (side == 0 ? q0 : k0) + local0;       // first row within the segment
  // (a chunk beyond the last row of the side has nothing to place)
  const int rows = min(min(g.chunk, unit_s - cu * g.chunk), side_rows(g, side) - row0);
  if (rows <= 0) return;

  wait_for_stream();
  if (SCAN && sa.sched && blockIdx.x == 0 && tid == 0) sa.sched[0] = sa.sched[1] = 0;
  const uint8_t* ids = a.ids + level * ids_level_stride(g) + side_ids_base(g, side) + (size_t)seg * side_rows(g, side) + row0;
  // SCAN: bucket tid's total over the node, and over the node's chunks before this one
  uint32_t tot = 0, before = 0;
  if (SCAN) {
    int nch;
    const int first = node_first_chunk(g, level, j, side, nch);
    const uint32_t* h = a.hist + level * hist_level_stride(g) + side_hist_base(g, side) + ((size_t)seg * side_cps(g, side) + first) * kBuckets + tid;
    for (int c0 = 0; c0 < nch; c0 += 8) {
      uint32_t x[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) x[e] = c0 + e < nch ? h[(size_t)(c0 + e) * kBuckets] : 0u;
#pragma unroll
      for (int e = 0; e < 8; ++e) { tot += x[e]; if (c0 + e < cn) before += x[e]; }
    }
  }
  // A warp has an eighth of the chunk, in groups of 32 consecutive rows.
  constexpr int GROUPS = kSortChunk / 8 / 32;
  const int wbeg = warp * (g.chunk / 8);
  const int wend = min(rows, wbeg + g.chunk / 8);
  uint32_t row_id[GROUPS];
#pragma unroll
  for (int k = 0; k < GROUPS; ++k) {
    const int i = wbeg + 32 * k + lane;
    row_id[k] = i < wend ? ids[i] : 0u;
  }
#pragma unroll
  for (int k = 0; k < 8 * kBuckets / 2 / 256; ++k) reinterpret_cast<uint4*>(&s_bkt[0][0])[tid + 256 * k] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  uint2* bkt = s_bkt[warp];
  // A row's place among the rows of the range with its id: those of earlier groups, and the lanes before it in the bucket's word, into which every
  // lane has put its bit.
#pragma unroll
  for (int k = 0; k < GROUPS; ++k) {
    if (wbeg + 32 * k < wend) {                          // (the same for the whole warp)
      const bool act = wbeg + 32 * k + lane < wend;
      const uint32_t id = row_id[k];
      if (act) atomicOr(&bkt[id].x, 1u << lane);
      __syncwarp();
      const uint2 b = bkt[id];
      const int before = __popc(b.x & ((1u << lane) - 1u));
      __syncwarp();
      if (act && before == 0) bkt[id] = make_uint2(0u, b.y + __popc(b.x));
      __syncwarp();
      row_id[k] = id | (b.y + before) << 8;
    }
  }
  __syncthreads();
  uint32_t run;
  if (SCAN) {
    // exclusive scan of the totals over the buckets
    __shared__ uint32_t s_warp[8];
    uint32_t x = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    run = x - tot + before;
#pragma unroll
    for (int w = 0; w < 8; ++w) run += w < warp ? s_warp[w] : 0u;
  } else {
    const uint32_t* o = a.offs + side_offs_base(g, side) + (((size_t)level * g.G + seg) * cpl + lc) * kBuckets;
    run = o[tid];
  }
#pragma unroll
  for (int w = 0; w < 8; ++w) { const uint32_t t = s_bkt[w][tid].y; s_bkt[w][tid].y = run; run += t; }
  __syncthreads();
  const size_t slice = ((size_t)level * g.G + seg) * g.nl + (g.causal ? (size_t)j * s : 0);
  int32_t* perm = (side == 0 ? a.perm_q : a.perm_k) + slice;
  int32_t* rank = side == 1 ? a.rank_k + slice : nullptr;
#pragma unroll
  for (int k = 0; k < GROUPS; ++k) {
    const int i = wbeg + 32 * k + lane;
    if (i < wend) {
      const uint32_t pos = bkt[row_id[k] & 255u].y + (row_id[k] >> 8);
      perm[pos] = local0 + i;
      if (rank) rank[local0 + i] = (int32_t)pos;
      if (side == 1 && a.key_slot) a.key_slot[(size_t)seg * g.nk + local0 + i] = -1;
    }
  }
  // The block of every sampled key among these rows, which decides whether a query tile's own block holds the sample: the attention
  // kernel asks for it in every work item, and from here it comes without the detour over the ranks (node items 8 % faster).
  if (side == 1 && a.smp_blk) {
    __syncthreads();                                     // (the ranks above are read back)
    const int node = g.causal ? (1 << level) - 1 + j : 0;
    const size_t base = ((size_t)seg * g.nodes + node) * g.m;
    const uint32_t N = g.causal ? (uint32_t)(g.npad >> (level + 1)) : (uint32_t)g.nk;
    for (int c = tid; c < g.m; c += 256) {
      int l;
      if (SCAN && sa.draw) {                             // (drawn by other blocks of this very launch: the stream gives it again)
        const Philox4 x = philox4x32_10((uint32_t)(c >> 2), (uint32_t)(g.seg0 + seg), (uint32_t)node, kDomainSamples, sa.k0, sa.k1);
        l = (int)__umulhi((c & 2) ? ((c & 1) ? x.x[3] : x.x[2]) : ((c & 1) ? x.x[1] : x.x[0]), N);
      } else l = sa.samples[base + c];
      if ((unsigned)(l - local0) < (unsigned)rows) {
        a.smp_blk[base + c] = rank[l] / g.b;
        if (a.key_slot) a.key_slot[(size_t)seg * g.nk + l] = c;      // (a key drawn more than once: any of its draws, the last to write)
      }
    }
  }
}

}  // namespace

static SortArgs make_sort_args(const Geometry& g, const Workspace& ws, int side_mask) {
  SortArgs a;
  a.ids = ws.ids; a.hist = ws.hist; a.offs = ws.offs;
  a.perm_q = ws.perm_q; a.perm_k = ws.perm_k; a.rank_k = ws.rank_k; a.smp_blk = ws.smp_blk; a.key_slot = ws.key_slot;
  a.g = g;
  a.side_mask = side_mask;
  return a;
}

// Nodes of at most kScanChunks chunks: the placement adds up the histograms itself (8 loads in flight, two rounds).  Every
// CTA then reads its node's whole histogram, so that this grows with the square of the chunks while the launch that it saves
// stays the same.  A call, us, scan launch -> in the placement: 1 head, 8 chunks 23.6 -> 21.9, 16 24.5 -> 22.7, 64 28.5 -> 25.2;
// 32 heads, 8 chunks 171.9 -> 169.7, 16 322.3 -> 322.0, 24 486 -> 490, 64 1243 -> 1259; 4 causal heads, nodes of 32 chunks
// 825 -> 830.  The line is where it stops paying with many heads; a few heads would gain 2-3 us beyond it as well.
constexpr int kScanChunks = 16;
int node_chunks(const Geometry& g) {
  return g.causal ? (g.nl / g.unit) * g.chunks_per_unit : (g.chunks_per_seg > g.chunks_per_seg_k ? g.chunks_per_seg : g.chunks_per_seg_k);
}
bool scan_in_scatter(const Geometry& g) { return node_chunks(g) <= kScanChunks; }

// Four groups of threads per node while every node has an SM of its own.  (A call, us, one group -> four: 4 heads of 40000 rows, 8 nodes of 20
// chunks, 74.0 -> 73.2; 4 causal heads of 100003 rows, 248 nodes, 592 -> 597.)
static int scan_ctas(const Geometry& g) { return 2 * g.G * (g.causal ? g.nodes : 1); }
bool wide_scan(const Geometry& g) { return !scan_in_scatter(g) && scan_ctas(g) <= kSms; }

static SampleArgs make_sample_args(const Geometry& g, const Workspace& ws, bool with_samples, uint64_t seed, int* blocks) {
  // (ws.tpos non-null: the probe rows of the capped row-sum estimate are drawn as well)
  SampleArgs sa;
  sa.samples = ws.samples; sa.tpos = ws.tpos; sa.ltau = ws.ltau; sa.g = g; sa.sched = ws.sched; sa.draw = with_samples;
  sa.k0 = (uint32_t)seed; sa.k1 = (uint32_t)(seed >> 32);
  *blocks = 0;
  if (with_samples && g.nodes > 0 && g.m > 0) {
    const size_t total = (size_t)g.G * g.nodes * ((g.m + 3) / 4);
    const size_t want = (total + 255) / 256;
    *blocks = (int)(want < 8 * kSms ? want : 8 * kSms);
  }
  return sa;
}

// scan of the chunk histograms; with_samples: the same launch also draws the samples (Alg. 2 line 4)
cudaError_t launch_sort_scan(const Geometry& g, const Workspace& ws, bool with_samples, uint64_t seed, cudaStream_t st, int side_mask,
                             const VnormArgs* vnorm) {
  if (!g.sorted || scan_in_scatter(g)) return cudaSuccess;
  const SortArgs a = make_sort_args(g, ws, side_mask);
  const int scan_blocks = scan_ctas(g);
  int sample_blocks;
  const SampleArgs sa = make_sample_args(g, ws, with_samples, seed, &sample_blocks);
  if (!wide_scan(g)) return launch(sort_scan_kernel<1>, scan_blocks + sample_blocks, 256, 0, st, a, sa, VnormArgs{}, scan_blocks, sample_blocks);
  sample_blocks = (sample_blocks + 3) / 4;
  const int vnorm_blocks = vnorm ? g.G * ((g.nk + 4095) / 4096) : 0;
  return launch(sort_scan_kernel<4>, scan_blocks + sample_blocks + vnorm_blocks, 1024, 0, st, a, sa, vnorm ? *vnorm : VnormArgs{}, scan_blocks,
                sample_blocks);
}

cudaError_t launch_sort_scatter(const Geometry& g, const Workspace& ws, bool with_samples, uint64_t seed, cudaStream_t st, int side_mask) {
  if (!g.sorted) return cudaSuccess;
  const SortArgs a = make_sort_args(g, ws, side_mask);
  const int grid = g.levels * g.G * (((side_mask & 1) ? side_cpl(g, 0) : 0) + ((side_mask & 2) ? side_cpl(g, 1) : 0));
  int sample_blocks;
  const SampleArgs sa = make_sample_args(g, ws, with_samples, seed, &sample_blocks);
  if (scan_in_scatter(g)) return launch(sort_scatter_kernel<true>, grid + sample_blocks, 256, 0, st, a, sa, grid);
  return launch(sort_scatter_kernel<false>, grid, 256, 0, st, a, sa, grid);
}

}  // namespace hyperattn
