// Shared declarations of the HyperAttention forward library (sm_100a).
// Notation follows the paper: n rows, d head dimension, b block size, m sampled columns,
// r hash bits, G = B*H independent (batch, head) segments.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <atomic>

namespace hyperattn {

constexpr int kSortChunk = 2048;      // most rows per histogram / scatter chunk
constexpr int kBuckets = 256;         // 2^r with r <= 8
constexpr int kTileQ = 128;           // query rows per attention tile
constexpr int kMaxLevelsMerge = 24;   // deepest causal recursion supported
// SMs of a B200, where a rule must not depend on the device in hand (workspace sizes are asked for without one) or a grid only has
// to be large enough; the grids of the persistent kernels ask the device (sm_count)
constexpr int kSms = 148;

// ---- Philox4x32-10 (Salmon et al., SC'11); identical on host and device -------------
struct Philox4 { uint32_t x[4]; };

__host__ __device__ inline void mulhilo32(uint32_t a, uint32_t b, uint32_t& hi, uint32_t& lo) {
#ifdef __CUDA_ARCH__
  lo = a * b;
  hi = __umulhi(a, b);
#else
  uint64_t p = (uint64_t)a * b;
  lo = (uint32_t)p;
  hi = (uint32_t)(p >> 32);
#endif
}

__host__ __device__ inline Philox4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                                 uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int rnd = 0; rnd < 10; ++rnd) {
    if (rnd > 0) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
    uint32_t hi0, lo0, hi1, lo1;
    mulhilo32(0xD2511F53u, c0, hi0, lo0);
    mulhilo32(0xCD9E8D57u, c2, hi1, lo1);
    uint32_t n0 = hi1 ^ c1 ^ k0, n1 = lo1, n2 = hi0 ^ c3 ^ k1, n3 = lo0;
    c0 = n0; c1 = n1; c2 = n2; c3 = n3;
  }
  Philox4 r; r.x[0] = c0; r.x[1] = c1; r.x[2] = c2; r.x[3] = c3;
  return r;
}
constexpr uint32_t kDomainDirections = 1, kDomainSamples = 2, kDomainRowSubset = 3;

// ---- geometry of one forward call, shared by all stages --------------------------------
// "unit" = the largest row range that never straddles a recursion node: a causal leaf of n0
// rows, or the whole segment.  Units are cut into chunks of `chunk` rows; one
// hash CTA produces the ids and the 256-bin histogram of one chunk, one scatter CTA places it.
struct Geometry {
  int G, n, d;         // n: query rows per segment
  int nk;              // key / value rows per segment (n, unless a non-causal call has another number of keys)
  int npad;            // causal: leaf << L, the length whose halves the recursion cuts (>= n: rows beyond n do
                       // not exist, so the last leaf and the query side of a level's last node may be short);
                       // non-causal: n
  int b, m, r;
  int bq;              // rows per group of sorted queries of a full node: b, or ceil(b n / nk) for unequal sides
  int causal;          // 1: causal with L >= 1 levels or a single causal leaf
  int L;               // number of recursion levels with off-diagonal nodes (0: none)
  int leaf;            // rows per exact leaf (n if L == 0)
  int chunk;           // rows per chunk: at most kSortChunk, a multiple of 256
  int unit;            // rows per unit (query side; both sides of a causal call)
  int chunks_per_unit;
  int chunks_per_seg;  // (npad / unit) * chunks_per_unit
  int unit_k, chunks_per_unit_k, chunks_per_seg_k;   // the same for the key side
  int levels;          // sorted levels: L if causal, else 1 (0 if nothing is sorted)
  int nl;              // sorted rows per (level, segment, side): npad/2 causal, max(n, nk) non-causal
  int nodes;           // off-diagonal nodes per segment (heap-numbered)
  int sorted;          // 1 if any node needs sortLSH (some node has b < its size)
  int seg0;            // index, in the caller's tensor, of this call's first segment (the sampling counters carry it)
  int node_dirs;       // 1: every recursion node hashes with directions of its own: ids and chunk histograms exist
                       // once per level (a row is on one side of exactly one node per level)
};
// ids / histograms of a level start this many elements after those of level 0 (0: one set shared by all levels)
__host__ __device__ inline size_t ids_level_stride(const Geometry& g) { return g.node_dirs ? (size_t)g.G * ((size_t)g.n + g.nk) : 0; }
__host__ __device__ inline size_t hist_level_stride(const Geometry& g) {
  return g.node_dirs ? (size_t)g.G * (g.chunks_per_seg + g.chunks_per_seg_k) * kBuckets : 0;
}

// sorted blocks of a node of s rows: ceil(s / b) of them, the last one with the remaining rows
// (Alg. 1 line 4: row i belongs to block floor(P(i) / b))
__host__ __device__ inline int node_blocks(int s, int b) { return (s + b - 1) / b; }
__host__ __device__ inline int block_len(int s, int b, int beta) { return (s - beta * b) < b ? (s - beta * b) : b; }

// node j of level l: number of keys s, first query row, first key row (non-causal: the whole segment)
__host__ __device__ inline void node_rows(const Geometry& g, int level, int j, int& s, int& q0, int& k0) {
  if (!g.causal) { s = g.nk; q0 = 0; k0 = 0; return; }
  s = g.npad >> (level + 1);
  q0 = (2 * j + 1) * s;
  k0 = 2 * j * s;
}
// query rows of a node whose nominal size is s and whose first query row is q0: s, unless the sequence
// ends inside it (the last node of a causal level) or the call has another number of queries than keys
__host__ __device__ inline int node_queries(const Geometry& g, int s, int q0) {
  if (!g.causal) return g.n;
  const int left = g.n - q0;
  return left < 0 ? 0 : (left < s ? left : s);
}
// rows per group of sorted queries when nq queries meet s keys in groups of b (Alg. 1 line 4 pairs group
// beta of either side; with nq != s the groups cover the same fraction of the sorted order): ceil(b nq / s)
__host__ __device__ inline int query_group(int b, int nq, int s) {
  return (int)(((long long)b * nq + s - 1) / s);
}
// per-side chunk geometry (side 0: queries, side 1: keys)
__host__ __device__ inline int side_rows(const Geometry& g, int side) { return side ? g.nk : g.n; }
__host__ __device__ inline int side_unit(const Geometry& g, int side) { return side ? g.unit_k : g.unit; }
__host__ __device__ inline int side_cpu(const Geometry& g, int side) { return side ? g.chunks_per_unit_k : g.chunks_per_unit; }
__host__ __device__ inline int side_cps(const Geometry& g, int side) { return side ? g.chunks_per_seg_k : g.chunks_per_seg; }
// chunks of one (level, segment) on a side: every node of the level (causal), or the whole side
__host__ __device__ inline int side_cpl(const Geometry& g, int side) { return g.causal ? (g.nl / g.unit) * g.chunks_per_unit : side_cps(g, side); }

// ---- launches -----------------------------------------------------------------------------
// Every kernel of a call is launched with programmatic stream serialisation: its launch is prepared while the kernel before
// it on the stream runs, and its blocks wait in wait_for_stream() until that one has completed and its writes are visible.  So
// nothing that an earlier kernel writes may be read - and nothing written - before it; since every kernel waits, all
// earlier ones have completed by then, not only the last.  The one exception is the device status word, which the tcgen05
// kernels look at first thing, before they allocate anything, so that the launches behind a wait that gave up drain quickly: a
// value from before that moment costs no more than this, the follower's own waits being bounded too.
// (Small calls gain 5-8 us; letting the next kernel's blocks in early with griddepcontrol.launch_dependents costs large calls
// 3-7 %: they take slots from the kernel that still runs.)
__device__ __forceinline__ void wait_for_stream() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st; cfg.attrs = &attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
// dynamic shared memory beyond the default is asked for once per kernel and device, not on every launch
template <auto Kernel>
cudaError_t allow_smem(int bytes) {
  static std::atomic<unsigned long long> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0;
  if (done.load(std::memory_order_relaxed) & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
  return e;
}
inline cudaError_t sm_count(int* sms) {
  static std::atomic<int> known[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 64 && (*sms = known[dev].load(std::memory_order_relaxed)) > 0) return cudaSuccess;
  e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess && dev < 64) known[dev].store(*sms, std::memory_order_relaxed);
  return e;
}

// sampling by value norms (vnorm.cu): what its first two steps read and write
struct VnormArgs {
  const __nv_bfloat16* v;          // [G, nk, d]
  uint32_t* wq;                    // [G, nk] weights of the rows
  unsigned long long* sums;        // [G, blocks] of 256 rows each
  unsigned long long* cum;         // [G, nk + 1] cumulative weights
  int G, nk, blocks;
};

// ---- stage launchers (each enqueues on `st`; returns cudaGetLastError()) ---------------
struct Workspace {
  __nv_bfloat16 *q16, *k16, *v16;  // bf16 staging of fp32 inputs (else null)
  __nv_bfloat16 *q16lo, *k16lo;    // second bf16 term of fp32 Q, K: x ~= x16 + x16lo
  uint8_t* ids;                    // queries [G, n], then keys [G, nk]
  uint32_t* hist;                  // queries [G, chunks_per_seg, 256], then keys [G, chunks_per_seg_k, 256]
  uint32_t* offs;                  // per side: [levels, G, chunks per (level,seg), 256]
  int32_t *perm_q, *perm_k, *rank_k;  // [levels, G, nl]
  int32_t* samples;                // [G, nodes, m]
  int32_t* smp_blk;                // [G, nodes, m] sorted block that the sampled key lies in (null: not wanted)
  int32_t* key_slot;               // [G, nk] one of the samples that drew the key, -1: none did (one node only; null: not wanted)
  int32_t* tpos;                   // capped row sums: [G, nodes, m] probe positions (else null)
  float* ltau;                     // capped row sums: [G, nodes] log2 of the largest unmasked probe row sum
  void* part_o; float* part_lse;   // causal partials: leaf [G,n,(d)] then per level [G,nl,(d)]; rows of fp32 or bf16
  int part_bf16;
  int* sched;                      // work counters of the attention's launches (up to two): zeroed by the first launch of the sort
  int* status;                     // device status word
};

// fp32 inputs of count_q (q) and count_k (k, v) entries to the workspace's bf16 copies
cudaError_t launch_convert(const float* q, const float* k, const float* v, const Workspace& ws, size_t count_q, size_t count_k, cudaStream_t st);
// w_host: the shared direction matrix; w_nodes (device, [nodes, d, r], g.node_dirs only): the nodes' own
// vnorm: bf16 inputs - the launch also weighs the rows of V
// convert_v: fp32 V - the launch also makes the workspace's bf16 copies of Q, K and V (fp32 inputs, convert_in_hash(g))
bool convert_in_hash(const Geometry& g);
cudaError_t launch_hash(const Geometry& g, const void* q, const void* k, int is_fp32, const float* w_host,
                        const Workspace& ws, unsigned long long* near_zero, cudaStream_t st, int side_mask = 3,
                        const float* w_nodes = nullptr, const void* convert_v = nullptr, const VnormArgs* vnorm = nullptr);
// side_mask: bit 0 queries, bit 1 keys (3: both)
// vnorm: the cumulative sums of the value norms as well; only where wide_scan(g)
cudaError_t launch_sort_scan(const Geometry& g, const Workspace& ws, bool with_samples, uint64_t seed, cudaStream_t st, int side_mask = 3,
                             const VnormArgs* vnorm = nullptr);
bool wide_scan(const Geometry& g);
int node_chunks(const Geometry& g);      // chunks of the longest node
bool scan_in_scatter(const Geometry& g);
// (small nodes: the scatter does the scan's work, samples included, and launch_sort_scan launches nothing)
cudaError_t launch_sort_scatter(const Geometry& g, const Workspace& ws, bool with_samples, uint64_t seed, cudaStream_t st, int side_mask = 3);
// side_mask for the hash as well (a side that is left out is neither read nor written)
cudaError_t launch_merge(const Geometry& g, const Workspace& ws, void* out, float* lse, int out_fp32,
                         cudaStream_t st);

}  // namespace hyperattn
