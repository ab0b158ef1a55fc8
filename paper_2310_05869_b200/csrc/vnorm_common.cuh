// Device bodies of the value-norm sampling (vnorm.cu) that run as extra blocks of other launches: the weights beside the hash (hash.cu), the
// cumulative sums beside the scan of the histograms (sort.cu; else in a launch of their own).
#pragma once
#include "common.cuh"

namespace hyperattn {
namespace {

constexpr float kNormScale = 4096.f;      // 2^12

constexpr int kVnormSmem = 32768;         // of a CTA that weighs rows

// A CTA of 256 threads weighs 256 rows (part `part`) of one segment, 32 KB at a time: the rows come in by whole lines and are read back
// one per thread (the chunks of a row XOR-swizzled, so that neither side has bank conflicts); also the sum of the CTA's weights.
template <int D>
__device__ __forceinline__ void vnorm_weights_body(const VnormArgs& a, int seg, int part, uint4* s_row) {
  constexpr int CPR = D / 8, ROWS = kVnormSmem / (D * 2);
  __shared__ unsigned long long s_warp[8];
  const int tid = threadIdx.x, lane = tid & 31;
  const int row0 = part * 256, rows = min(256, a.nk - row0);
  const size_t first = (size_t)seg * a.nk + row0;
  const uint4* src = reinterpret_cast<const uint4*>(a.v) + first * CPR;
  unsigned long long w = 0;
#pragma unroll
  for (int r0 = 0; r0 < 256; r0 += ROWS) {
    if (r0) __syncthreads();
#pragma unroll
    for (int e = 0; e < ROWS * CPR / 256; ++e) {
      const int c = tid + 256 * e, r = c / CPR, cc = c % CPR;
      if (r0 + r < rows) s_row[r * CPR + (cc ^ (r & 7))] = __ldg(src + r0 * CPR + c);
    }
    __syncthreads();
    const int own = tid - r0;
    if (own >= 0 && own < ROWS && tid < rows) {
      float acc = 0.f;
#pragma unroll
      for (int c = 0; c < CPR; ++c) {
        const uint4 x = s_row[own * CPR + (c ^ (own & 7))];
        const uint32_t words[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float lo = __uint_as_float(words[e] << 16), hi = __uint_as_float(words[e] & 0xffff0000u);
          acc = __fadd_rn(acc, __fmul_rn(lo, lo));        // (coordinate order, no fused multiply-add: the stated arithmetic)
          acc = __fadd_rn(acc, __fmul_rn(hi, hi));
        }
      }
      const uint32_t q = (uint32_t)(acc * kNormScale);    // exact scaling, truncation = floor (acc >= 0)
      a.wq[first + tid] = q;
      w = q;
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
  if (lane == 0) s_warp[tid >> 5] = w;
  __syncthreads();
  if (tid == 0) {
    for (int e = 1; e < 8; ++e) w += s_warp[e];
    a.sums[(size_t)seg * a.blocks + part] = w;
  }
}

// cum[seg][0] = 0, cum[seg][i + 1] = wq[seg][0] + ... + wq[seg][i] (64-bit).  A CTA of 1024 threads does 4096 rows of one segment and adds
// up the sums of the rows before them by itself, so all CTAs run at once (one CTA per segment walking its rows: 94 us for 4 segments of
// 131072 rows, now 5 us).
__device__ __forceinline__ void vnorm_scan_body(const VnormArgs& a, int seg, int part) {
  __shared__ unsigned long long s_warp[32], s_before[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nk = a.nk;
  const uint32_t* w = a.wq + (size_t)seg * nk;
  unsigned long long* c = a.cum + (size_t)seg * (nk + 1);
  const int i = part * 4096 + 4 * tid;
  unsigned long long x[4], before = 0;
#pragma unroll
  for (int e = 0; e < 4; ++e) x[e] = i + e < nk ? w[i + e] : 0ull;
  for (int e = tid; e < part * 16; e += 1024) before += a.sums[(size_t)seg * a.blocks + e];
  x[1] += x[0]; x[2] += x[1]; x[3] += x[2];
  unsigned long long run = x[3];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long t = __shfl_up_sync(0xffffffffu, run, o);
    if (lane >= o) run += t;
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
  if (lane == 31) { s_warp[warp] = run; s_before[warp] = before; }
  __syncthreads();
  // sums of the warps before this one, and of everything before the CTA
  unsigned long long t = s_before[lane] + (lane < warp ? s_warp[lane] : 0ull);
#pragma unroll
  for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  t += run - x[3];
#pragma unroll
  for (int e = 0; e < 4; ++e)
    if (i + e < nk) c[i + e + 1] = t + x[e];
  if (i == 0) c[0] = 0;
}

}  // namespace
}  // namespace hyperattn
