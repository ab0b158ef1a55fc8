// Stage 1 of sortLSH (Def. 1; Alg. 1 line 2): bucket id of every query and key row.
//
//   p_t = <x, w_t>,  bit_t = [p_t > 0],  g = sum_t bit_t 2^t,  id = Gray rank of g.
//
// The kernel streams Q and K once (HBM-bound: d*e bytes in, 1 byte out per row) and also
// leaves a 256-bin histogram per chunk of rows, which is the first pass of the counting
// argsort (Alg. 1 line 3).
//
// bf16 rows: the projection [16 rows x d] . [d x 8] runs on the tensor cores
// (mma.sync m16n8k16, fp32 accumulate).  Each lane fetches its operands with 128-bit loads;
// because a dot product does not care in which order the coordinates are visited, the
// coordinates a lane happens to hold are assigned to MMA k-slots by a fixed permutation and
// the direction matrix is laid out with the same permutation.  The fp32 directions are split
// into three bf16 terms (w = w1 + w2 + w3 exactly), so the products are exact and only the
// fp32 accumulation rounds; signs can differ from an exact evaluation only where |p_t| is
// within ~1e-5 of zero.
#include "vnorm_common.cuh"

namespace hyperattn {
namespace {

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint4 ldg_stream(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&t);
}

// Gray rank: h with h ^ (h >> 1) == g (prefix xor), 8-bit patterns.
__device__ __forceinline__ uint32_t gray_rank8(uint32_t g) {
  g ^= g >> 1; g ^= g >> 2; g ^= g >> 4;
  return g & 0xFFu;
}

// fp32 -> bf16 staging of Q, K, V; for Q and K also the rounding remainder as a second bf16 term
struct ConvertArgs {
  const float4* src[3];
  uint2 *hi[3], *lo[3];
  size_t count4[3];
};

struct HashArgs {
  const void* x[2];       // Q, K  [G, n, d]
  float w[128 * 8];       // [d, r] directions, passed by value (<= 4 KB of kernel parameters)
  uint8_t* ids;           // queries [G, n], then keys [G, nk]
  uint32_t* hist;         // queries [G, chunks_per_seg, 256], then keys [G, chunks_per_seg_k, 256]
  unsigned long long* near_zero;
  int G, r;
  int side_mask;          // bit s set: side s is hashed
  int chunk;              // rows per chunk
  int n[2];               // rows per segment of either side
  int unit[2], chunks_per_unit[2], chunks_per_seg[2];
  // directions of every recursion node's own (causal calls): the grid covers every level; a chunk belongs to
  // node j = unit / (2 u) of its level (u units per half) and is hashed there if it lies on the side's half
  const float* w_nodes;   // [nodes, d, r] or null
  int levels, L, d;
  size_t ids_level_stride, hist_level_stride;
  // fp32 inputs, where this launch also makes the bf16 copies: the CTAs from hash_ctas on
  ConvertArgs conv;
  int hash_ctas;
  VnormArgs vnorm;        // bf16 inputs, columns sampled by value norms: the CTAs from hash_ctas on weigh the rows of V
};

// which chunk a CTA owns: side, segment, first row, number of rows (0: the chunk lies beyond the last row)
struct ChunkPos { int side, seg, chunk, row0, rows, level, node; };
__device__ __forceinline__ ChunkPos chunk_of_cta(const HashArgs& a, int cta) {
  ChunkPos c;
  const int per_level = a.G * (a.chunks_per_seg[0] + a.chunks_per_seg[1]);
  c.level = cta / per_level; cta -= c.level * per_level;
  c.node = 0;
  const int ctas0 = a.G * a.chunks_per_seg[0];
  c.side = cta >= ctas0;
  if (c.side) cta -= ctas0;
  c.chunk = cta % a.chunks_per_seg[c.side];
  c.seg = cta / a.chunks_per_seg[c.side];
  const int unit_idx = c.chunk / a.chunks_per_unit[c.side], cu = c.chunk % a.chunks_per_unit[c.side];
  c.row0 = unit_idx * a.unit[c.side] + cu * a.chunk;
  c.rows = max(0, min(min(a.chunk, a.unit[c.side] - cu * a.chunk), a.n[c.side] - c.row0));
  if (a.w_nodes) {
    // level l: nodes of 2 u units, u = 2^(L - 1 - l); queries live in the second half, keys in the first
    const int u = 1 << (a.L - 1 - c.level);
    const int j = unit_idx / (2 * u);
    const bool second = (unit_idx / u) & 1;
    c.node = (1 << c.level) - 1 + j;
    if (second != (c.side == 0)) c.rows = -1;          // this side of the level does not hold the chunk: nothing to do
  }
  return c;
}
__device__ __forceinline__ size_t ids_base(const HashArgs& a, const ChunkPos& c) {
  return c.level * a.ids_level_stride + (c.side ? (size_t)a.G * a.n[0] : 0) + (size_t)c.seg * a.n[c.side] + c.row0;
}
__device__ __forceinline__ size_t hist_base(const HashArgs& a, const ChunkPos& c) {
  return c.level * a.hist_level_stride +
         ((c.side ? (size_t)a.G * a.chunks_per_seg[0] : 0) + (size_t)c.seg * a.chunks_per_seg[c.side] + c.chunk) * kBuckets;
}

// One CTA = one chunk (<= a.chunk rows of one side of one segment).  Each warp walks over
// groups of 16 rows; the loads of the next group are issued between the MMAs of the current
// one, and the direction fragments live in shared memory (one 8-byte read per MMA) instead
// of 48 registers, so that two to four CTAs fit an SM and ~128 KB of loads are in flight.
// VNORM: further CTAs weigh the rows of V for the sampling by value norms: neither of the two reads by itself keeps the memory busy to its end.
// (With the cumulative sums beside the scan of the histograms, the call, us: 4 heads of 50000 queries, 131072 keys, d = 64, 154 -> 139; 40000
// queries, d = 128, 270 -> 248, but 275 with 64 KB of rows per CTA at a time instead of 32.  The 32 KB are asked for by every CTA of the launch; it
// pays also where the hash alone fills the chip: 32 heads of 131072 rows 1510 -> 1481, of 32768 414 -> 398, 128 of 4096 226 -> 215, 512 of 1024 192
// -> 187, d = 128, 32 of 32768 601 -> 575, 32 of 4096 108 -> 103, 32 causal ones of 16384 1034 -> 982.)
template <int D, bool VNORM>
__global__ void __launch_bounds__(256, D == 64 ? 4 : 3) hash_bf16_kernel(const __grid_constant__ HashArgs a) {
  if (VNORM && (int)blockIdx.x >= a.hash_ctas) {
    extern __shared__ uint4 s_row[];
    wait_for_stream();
    const int x = blockIdx.x - a.hash_ctas;
    vnorm_weights_body<D>(a.vnorm, x / a.vnorm.blocks, x % a.vnorm.blocks, s_row);
    return;
  }
  constexpr int KS = D / 16;             // MMA k-steps
  constexpr int CPL = D / 32;            // 16-byte chunks per lane per row
  __shared__ __align__(16) uint8_t s_ids[kSortChunk];
  __shared__ uint32_t s_hist[kBuckets];
  __shared__ uint2 s_bw[3][KS][32];      // [split][k-step][lane] -> (b0, b1) of that lane

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gid = lane >> 2, tig = lane & 3;
  const ChunkPos cp = chunk_of_cta(a, blockIdx.x);
  const int side = cp.side, seg = cp.seg, row0 = cp.row0, rows = cp.rows;
  if (!((a.side_mask >> side) & 1) || rows < 0) return;
  const float* wsrc = a.w_nodes ? a.w_nodes + (size_t)cp.node * (D * a.r) : a.w;

  s_hist[tid] = 0;
  wait_for_stream();

  const char* base = reinterpret_cast<const char*>(a.x[side]) + ((size_t)seg * a.n[side] + row0) * (D * 2);
  unsigned nz = 0;
  const int groups = (rows + 15) >> 4;
  // The 16-byte chunks of a lane's two rows are asked for again (for the warp's next group) as soon as they have been
  // multiplied: no second set of registers, and no spills at d = 128.
  uint4 xa[CPL], xb[CPL];
  auto load_chunk = [&](int grp, int h) {
    const int ra = grp * 16 + gid, rb = ra + 8;
    const char* pa = base + (size_t)ra * (D * 2) + (tig + 4 * h) * 16;
    xa[h] = ra < rows ? ldg_stream(pa) : make_uint4(0, 0, 0, 0);
    xb[h] = rb < rows ? ldg_stream(pa + 8 * (D * 2)) : make_uint4(0, 0, 0, 0);
  };
#pragma unroll
  for (int h = 0; h < CPL; ++h) load_chunk(warp, h);  // the first rows are on their way while the fragments are built

  // Direction fragments.  k-slot (step s, half h, element e) of lane (gid, tig) holds
  // coordinate 8*(tig + 4*(s>>1)) + 2*(2*(s&1) + h) + e; column gid is direction gid.
  for (int idx = tid; idx < KS * 32; idx += 256) {
    const int s = idx >> 5, l = idx & 31;
    const int lg = l >> 2, lt = l & 3;
    uint32_t packed[3][2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float t1[2], t2[2], t3[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int coord = 8 * (lt + 4 * (s >> 1)) + 2 * (2 * (s & 1) + h) + e;
        const float w = (lg < a.r) ? wsrc[coord * a.r + lg] : 0.f;
        t1[e] = __bfloat162float(__float2bfloat16_rn(w));
        const float r1 = w - t1[e];
        t2[e] = __bfloat162float(__float2bfloat16_rn(r1));
        t3[e] = __bfloat162float(__float2bfloat16_rn(r1 - t2[e]));
      }
      packed[0][h] = pack_bf16(t1[0], t1[1]);
      packed[1][h] = pack_bf16(t2[0], t2[1]);
      packed[2][h] = pack_bf16(t3[0], t3[1]);
    }
#pragma unroll
    for (int sp = 0; sp < 3; ++sp) s_bw[sp][s][l] = make_uint2(packed[sp][0], packed[sp][1]);
  }
  __syncthreads();

  for (int grp = warp; grp < groups; grp += 8) {
    const int ra = grp * 16 + gid, rb = ra + 8;
    float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int s = 0; s < KS; ++s) {
      const uint4 va = xa[s >> 1], vb = xb[s >> 1];
      uint32_t af[4];
      af[0] = (s & 1) ? va.z : va.x;   // row gid,   half 0
      af[1] = (s & 1) ? vb.z : vb.x;   // row gid+8, half 0
      af[2] = (s & 1) ? va.w : va.y;   // row gid,   half 1
      af[3] = (s & 1) ? vb.w : vb.y;   // row gid+8, half 1
      const uint2 w3 = s_bw[2][s][lane], w2 = s_bw[1][s][lane], w1 = s_bw[0][s][lane];
      mma_bf16_16816(lo, af, w3.x, w3.y);
      mma_bf16_16816(lo, af, w2.x, w2.y);
      mma_bf16_16816(hi, af, w1.x, w1.y);
      if (s & 1) load_chunk(grp + 8, s >> 1);         // (rows past the end are not read)
    }
    // lane holds p[row gid][2tig], p[gid][2tig+1], p[gid+8][2tig], p[gid+8][2tig+1]
    float p[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) p[i] = hi[i] + lo[i];
    uint32_t ga = (p[0] > 0.f ? 1u : 0u) << (2 * tig) | (p[1] > 0.f ? 1u : 0u) << (2 * tig + 1);
    uint32_t gb = (p[2] > 0.f ? 1u : 0u) << (2 * tig) | (p[3] > 0.f ? 1u : 0u) << (2 * tig + 1);
    if (a.near_zero) {
      if (2 * tig < a.r) { nz += (ra < rows && fabsf(p[0]) < 1e-4f); nz += (rb < rows && fabsf(p[2]) < 1e-4f); }
      if (2 * tig + 1 < a.r) { nz += (ra < rows && fabsf(p[1]) < 1e-4f); nz += (rb < rows && fabsf(p[3]) < 1e-4f); }
    }
    ga |= __shfl_xor_sync(0xffffffffu, ga, 1); ga |= __shfl_xor_sync(0xffffffffu, ga, 2);
    gb |= __shfl_xor_sync(0xffffffffu, gb, 1); gb |= __shfl_xor_sync(0xffffffffu, gb, 2);
    if (tig == 0 && ra < rows) { const uint32_t id = gray_rank8(ga); s_ids[ra] = (uint8_t)id; atomicAdd(&s_hist[id], 1u); }
    if (tig == 1 && rb < rows) { const uint32_t id = gray_rank8(gb); s_ids[rb] = (uint8_t)id; atomicAdd(&s_hist[id], 1u); }
  }
  if (a.near_zero) {
#pragma unroll
    for (int o = 16; o; o >>= 1) nz += __shfl_xor_sync(0xffffffffu, nz, o);
    if (lane == 0 && nz) atomicAdd(a.near_zero, (unsigned long long)nz);
  }
  __syncthreads();
  uint8_t* dst = a.ids + ids_base(a, cp);
  if ((rows & 15) == 0 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
    for (int i = tid; i < rows / 16; i += 256)
      reinterpret_cast<uint4*>(dst)[i] = reinterpret_cast<const uint4*>(s_ids)[i];
  } else {
    for (int i = tid; i < rows; i += 256) dst[i] = s_ids[i];
  }
  a.hist[hist_base(a, cp) + tid] = s_hist[tid];
}

// four entries as bf16, and their rounding remainders as a second bf16 term
__device__ __forceinline__ void split_bf16(const float4& x, uint2& hi, uint2& lo) {
  const float xs[4] = {x.x, x.y, x.z, x.w};
  float h[4], l[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) { h[e] = __bfloat162float(__float2bfloat16_rn(xs[e])); l[e] = xs[e] - h[e]; }
  hi = make_uint2(pack_bf16(h[0], h[1]), pack_bf16(h[2], h[3]));
  lo = make_uint2(pack_bf16(l[0], l[1]), pack_bf16(l[2], l[3]));
}

// one CTA's share of the copies of array s, U pieces of 16 bytes in flight per thread
template <int U>
__device__ __forceinline__ void convert_body(const ConvertArgs& a, int s, size_t cta, size_t ctas) {
  for (size_t i0 = cta * (256 * U) + threadIdx.x; i0 < a.count4[s]; i0 += ctas * (256 * U)) {
    float4 x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) x[u] = i0 + 256 * u < a.count4[s] ? a.src[s][i0 + 256 * u] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const size_t i = i0 + 256 * u;
      if (i >= a.count4[s]) break;
      uint2 hi, lo;
      split_bf16(x[u], hi, lo);
      a.hi[s][i] = hi;
      if (a.lo[s]) a.lo[s][i] = lo;
    }
  }
}

// fp32 rows: thread = row, plain fp32 FMA in coordinate order, 256 rows at a time through shared memory (cp.async; rows padded by 16
// bytes, so that the lanes' 16-byte reads meet no bank conflict).  Bound by latency and, with many rows, by shared-memory reads: a row's
// coordinates are read once for all directions, a direction's by the whole warp at once.  (1024 rows on both sides, us, d = 64 / 128: eight
// threads per row - a direction each - and loads into registers 11.9 / 22.9, the same with 1024 threads and copies in flight 7.1 / 11.4;
// each of their 16-byte reads takes the shared memory four cycles, whatever lanes share; this form 4.4 / 7.1.)
// The bf16 copies of Q, K and V are made by extra CTAs of this launch, while the others wait for memory (convert_in_hash).
template <int D> constexpr int kHash32Smem = 256 * (D + 4) * 4;
template <int D>
__global__ void __launch_bounds__(256) hash_fp32_kernel(const __grid_constant__ HashArgs a) {
  extern __shared__ __align__(16) float s_x[];           // [256][D + 4]
  __shared__ __align__(16) float s_w[D][8];
  __shared__ uint32_t s_hist[kBuckets];
  const int tid = threadIdx.x;
  if ((int)blockIdx.x >= a.hash_ctas) {
    wait_for_stream();
    for (int x = 0; x < 3; ++x) convert_body<4>(a.conv, x, blockIdx.x - a.hash_ctas, gridDim.x - a.hash_ctas);
    return;
  }
  const ChunkPos cp = chunk_of_cta(a, blockIdx.x);
  const int rows = cp.rows;
  if (!((a.side_mask >> cp.side) & 1) || rows < 0) return;
  const float* wsrc = a.w_nodes ? a.w_nodes + (size_t)cp.node * (D * a.r) : a.w;
  s_hist[tid] = 0;
  wait_for_stream();
  const float* base = reinterpret_cast<const float*>(a.x[cp.side]) + ((size_t)cp.seg * a.n[cp.side] + cp.row0) * D;
  uint8_t* dst = a.ids + ids_base(a, cp);
  unsigned nz = 0;
  for (int row0 = 0; row0 < rows; row0 += 256) {
    const int n = min(256, rows - row0);
#pragma unroll 16
    for (int i = 0; i < D / 4; ++i) {
      const int c = tid + i * 256, row = c / (D / 4), col = c % (D / 4);
      if (row < n)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(s_x + row * (D + 4) + 4 * col)),
                     "l"(base + (size_t)(row0 + row) * D + 4 * col) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (row0 == 0)
      for (int i = tid; i < D * 8; i += 256) s_w[i >> 3][i & 7] = (i & 7) < a.r ? wsrc[(i >> 3) * a.r + (i & 7)] : 0.f;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (tid < n) {
      float p[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) p[t] = 0.f;
#pragma unroll 4
      for (int c = 0; c < D; c += 4) {
        const float4 x4 = *reinterpret_cast<const float4*>(s_x + tid * (D + 4) + c);
        const float x[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float4 wa = *reinterpret_cast<const float4*>(&s_w[c + e][0]), wb = *reinterpret_cast<const float4*>(&s_w[c + e][4]);
          p[0] = fmaf(x[e], wa.x, p[0]); p[1] = fmaf(x[e], wa.y, p[1]); p[2] = fmaf(x[e], wa.z, p[2]); p[3] = fmaf(x[e], wa.w, p[3]);
          p[4] = fmaf(x[e], wb.x, p[4]); p[5] = fmaf(x[e], wb.y, p[5]); p[6] = fmaf(x[e], wb.z, p[6]); p[7] = fmaf(x[e], wb.w, p[7]);
        }
      }
      uint32_t bits = 0;
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        bits |= (p[t] > 0.f ? 1u : 0u) << t;
        nz += t < a.r && fabsf(p[t]) < 1e-4f;
      }
      const uint32_t id = gray_rank8(bits);
      dst[row0 + tid] = (uint8_t)id;
      atomicAdd(&s_hist[id], 1u);
    }
    __syncthreads();
  }
  if (a.near_zero && nz) atomicAdd(a.near_zero, (unsigned long long)nz);
  __syncthreads();                                       // (a chunk without rows)
  a.hist[hist_base(a, cp) + tid] = s_hist[tid];
}

// fp32 -> bf16 staging of Q, K, V (blockIdx.y); for Q and K also the rounding remainder as a second bf16 term
__global__ void __launch_bounds__(256) convert_kernel(const __grid_constant__ ConvertArgs a) {
  wait_for_stream();
  convert_body<1>(a, blockIdx.y, blockIdx.x, gridDim.x);
}

}  // namespace

static ConvertArgs make_convert_args(const void* q, const void* k, const void* v, const Workspace& ws, size_t count_q, size_t count_k) {
  ConvertArgs a;
  const void* src[3] = {q, k, v};
  __nv_bfloat16 *hi[3] = {ws.q16, ws.k16, ws.v16}, *lo[3] = {ws.q16lo, ws.k16lo, nullptr};
  for (int s = 0; s < 3; ++s) {
    a.src[s] = reinterpret_cast<const float4*>(src[s]);
    a.hi[s] = reinterpret_cast<uint2*>(hi[s]); a.lo[s] = reinterpret_cast<uint2*>(lo[s]);
    a.count4[s] = (s ? count_k : count_q) / 4;
  }
  return a;
}
cudaError_t launch_convert(const float* q, const float* k, const float* v, const Workspace& ws, size_t count_q, size_t count_k, cudaStream_t st) {
  const ConvertArgs a = make_convert_args(q, k, v, ws, count_q, count_k);
  const size_t most = a.count4[0] > a.count4[1] ? a.count4[0] : a.count4[1], want = (most + 255) / 256;
  const dim3 grid((unsigned)(want < 16 * kSms ? want : 16 * kSms), 3);
  return launch(convert_kernel, grid, 256, 0, st, a);
}

// 1024 pieces of 16 bytes of each array per CTA
static int convert_ctas(const Geometry& g) {
  const size_t want = ((size_t)g.G * (g.n > g.nk ? g.n : g.nk) * g.d / 4 + 1023) / 1024;
  return want < (1u << 20) ? (int)want : 1 << 20;
}
// Copies of up to two CTAs per SM run beside the hash.  The hash's CTAs take 70 (d = 64) or 135 KB (d = 128) of shared memory each, so
// that three or one fit an SM, and the copies' CTAs, being of the same launch, are as few; beyond the line a launch of their own has
// more threads in flight.  A call, us, own launch -> beside the hash: d = 64, 16 copy CTAs 17.5 -> 16.5, 256 23.1 -> 22.7, 512
// 39.2 -> 37.2 (three CTAs per SM are enough there: the line could lie higher); d = 128, 32 25.0 -> 23.8, 157 27.2 -> 25.2, 512
// 35.2 -> 36.5, 1024 70.7 -> 77.8.
bool convert_in_hash(const Geometry& g) { return g.sorted && !g.node_dirs && convert_ctas(g) <= 2 * kSms; }

cudaError_t launch_hash(const Geometry& g, const void* q, const void* k, int is_fp32, const float* w_host,
                        const Workspace& ws, unsigned long long* near_zero, cudaStream_t st, int side_mask,
                        const float* w_nodes, const void* convert_v, const VnormArgs* vnorm) {
  HashArgs a;
  a.side_mask = side_mask; a.chunk = g.chunk;
  a.w_nodes = g.node_dirs ? w_nodes : nullptr;
  a.levels = g.node_dirs ? g.levels : 1; a.L = g.L; a.d = g.d;
  a.ids_level_stride = ids_level_stride(g); a.hist_level_stride = hist_level_stride(g);
  for (int i = 0; i < g.d * g.r; ++i) a.w[i] = w_host[i];
  a.x[0] = q; a.x[1] = k; a.ids = ws.ids; a.hist = ws.hist; a.near_zero = near_zero;
  a.G = g.G; a.r = g.r;
  for (int s = 0; s < 2; ++s) {
    a.n[s] = side_rows(g, s); a.unit[s] = side_unit(g, s);
    a.chunks_per_unit[s] = side_cpu(g, s); a.chunks_per_seg[s] = side_cps(g, s);
  }
  const int grid = a.levels * g.G * (g.chunks_per_seg + g.chunks_per_seg_k);
  if (is_fp32) {
    const cudaError_t e = g.d == 64 ? allow_smem<hash_fp32_kernel<64>>(kHash32Smem<64>) : allow_smem<hash_fp32_kernel<128>>(kHash32Smem<128>);
    if (e != cudaSuccess) return e;
    a.hash_ctas = grid;
    int copy_ctas = 0;
    if (convert_v) {
      a.conv = make_convert_args(q, k, convert_v, ws, (size_t)g.G * g.n * g.d, (size_t)g.G * g.nk * g.d);
      copy_ctas = convert_ctas(g);
    }
    return launch(g.d == 64 ? hash_fp32_kernel<64> : hash_fp32_kernel<128>, grid + copy_ctas, 256,
                  g.d == 64 ? kHash32Smem<64> : kHash32Smem<128>, st, a);
  }
  if (vnorm) {
    a.hash_ctas = grid;
    a.vnorm = *vnorm;
    const unsigned ctas = (unsigned)grid + (unsigned)vnorm->G * (unsigned)vnorm->blocks;
    return launch(g.d == 64 ? hash_bf16_kernel<64, true> : hash_bf16_kernel<128, true>, ctas, 256, kVnormSmem, st, a);
  }
  return launch(g.d == 64 ? hash_bf16_kernel<64, false> : hash_bf16_kernel<128, false>, grid, 256, 0, st, a);
}

}  // namespace hyperattn
