// Sampling the residual's columns by squared row norms of V (Lemma 2) instead of uniformly (Sec. 4):
//   p_l = ||V_l||^2 / ||V||_F^2 over the keys of a (segment, recursion node), m i.i.d. draws, weight
//   1 / (m p_l) per draw (the rows of Lemma 2's sampling matrix S, squared).
// Indices must be reproducible bit for bit, so the distribution is made of integers: the squared norm
// of a row is accumulated in fp32 in coordinate order (bf16 squares are exact in fp32) and cut to a
// multiple of 2^-12; cumulative sums are 64-bit integers; a draw is the first key whose cumulative
// weight exceeds floor(x * total / 2^32), x the Philox word the uniform sampler would have used.
// Three small steps: weights (streams V once; further blocks of the hash launch), per-segment cumulative sums (further blocks of the
// scan of the histograms, or, with few chunks or many nodes, a launch of their own here), draws.
#include "vnorm_common.cuh"

namespace hyperattn {
namespace {

// (Segment = y + gridDim.y * z, its part x: a grid's y ends at 65535, and a call may have 2^20 segments.)
__global__ void __launch_bounds__(1024) vnorm_scan_kernel(VnormArgs a) {
  wait_for_stream();
  const int seg = blockIdx.y + gridDim.y * blockIdx.z;
  if (seg < a.G) vnorm_scan_body(a, seg, blockIdx.x);
}

struct VnormSampleArgs {
  const unsigned long long* cum;   // [G, nk + 1]
  int32_t* samples;                // [G, nodes, m]
  float* wlog;                     // [G, nodes, m] log2 of the weight 1 / (m p) of every draw
  Geometry g;
  uint32_t k0, k1;
};

// LPD lanes per draw: 1, or 32 where draws are few - the search is a chain of dependent reads, and 32 probes at a time
// make it four steps long instead of 17 for 131072 keys.
template <int LPD>
__global__ void __launch_bounds__(256) vnorm_sample_kernel(VnormSampleArgs a) {
  const Geometry& g = a.g;
  wait_for_stream();
  const size_t total_draws = (size_t)g.G * g.nodes * g.m;
  const size_t i = ((size_t)blockIdx.x * 256 + threadIdx.x) / LPD;
  if (i >= total_draws) return;
  const int jd = (int)(i % g.m);
  const int nd = (int)((i / g.m) % g.nodes);
  const int seg = (int)(i / ((size_t)g.m * g.nodes));
  const int level = g.causal ? 31 - __clz(nd + 1) : 0;
  int s, q0, k0;
  node_rows(g, level, g.causal ? nd + 1 - (1 << level) : 0, s, q0, k0);
  const Philox4 x4 = philox4x32_10((uint32_t)(jd >> 2), (uint32_t)(g.seg0 + seg), (uint32_t)nd, kDomainSamples, a.k0, a.k1);
  const uint32_t x = x4.x[jd & 3];
  const unsigned long long* c = a.cum + (size_t)seg * (g.nk + 1) + k0;     // c[l] - c[0]: weight of the node's first l keys
  const int have = min(s, g.nk - k0);                                     // keys of the node that exist
  int idx;
  float wl;
  const unsigned long long base = have > 0 ? c[0] : 0ull;
  const unsigned long long total = have > 0 ? c[have] - base : 0ull;
  if (total == 0ull) {
    idx = (int)__umulhi(x, (uint32_t)s);
    wl = g.m > 0 ? log2f((float)s / (float)g.m) : 0.f;
  } else {
    const unsigned long long target = __umul64hi((unsigned long long)x << 32, total);     // floor(x * total / 2^32)
    int lo = 0, hi = have - 1;                           // smallest l with c[l + 1] - base > target
    if (LPD == 1) {
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (c[mid + 1] - base > target) hi = mid; else lo = mid + 1;
      }
    } else {
      const int lane = threadIdx.x & 31;
      while (lo < hi) {
        const int step = (hi - lo) / 32 + 1;               // probes lo + step - 1, lo + 2 step - 1, ...; those past hi: hi, where it holds
        const int at = min((long long)hi, lo + (long long)(lane + 1) * step - 1);
        const int first = __ffs(__ballot_sync(0xffffffffu, c[at + 1] - base > target)) - 1;
        hi = (int)min((long long)hi, lo + (long long)(first + 1) * step - 1);
        lo += first * step;
      }
    }
    idx = lo;
    const unsigned long long w = c[idx + 1] - c[idx];
    wl = log2f((float)total / ((float)g.m * (float)w));
  }
  if (LPD > 1 && (threadIdx.x & 31)) return;
  a.samples[i] = idx;
  a.wlog[i] = wl;
}

}  // namespace

// (the weights are there: the hash launch has made them)  scan_done: so are their cumulative sums
cudaError_t launch_vnorm_sampling(const Geometry& g, const VnormArgs& v, bool scan_done, int32_t* samples, float* wlog, uint64_t seed,
                                  cudaStream_t st) {
  if (!g.sorted || g.m == 0 || g.nodes == 0) return cudaSuccess;
  const unsigned y = g.G < 65536 ? g.G : 65535, z = ((unsigned)g.G + y - 1) / y;
  cudaError_t e = cudaSuccess;
  if (!scan_done) e = launch(vnorm_scan_kernel, dim3((g.nk + 4095) / 4096, y, z), 1024, 0, st, v);
  if (e != cudaSuccess) return e;
  VnormSampleArgs a;
  a.cum = v.cum; a.samples = samples; a.wlog = wlog; a.g = g; a.k0 = (uint32_t)seed; a.k1 = (uint32_t)(seed >> 32);
  // A call, us, one lane per draw -> 32: 256 draws 111.7 -> 105.7, 1024 160.9 -> 156.8, 4096 477.7 -> 474.3 (131072 keys), 2048
  // 63.6 -> 60.4 (16384 keys); 8192 893.8 -> 894.2 (131072 keys), 67.9 -> 68.6 (4096 keys); 16384 264.2 -> 267.5 (16384 keys),
  // 128.7 -> 132.7 (4096 keys); 65536 616.7 -> 642.7 (16384 keys).
  const size_t draws = (size_t)g.G * g.nodes * g.m;
  if (draws < 16384) return launch(vnorm_sample_kernel<32>, (unsigned)((draws + 7) / 8), 256, 0, st, a);
  return launch(vnorm_sample_kernel<1>, (unsigned)((draws + 255) / 256), 256, 0, st, a);
}

}  // namespace hyperattn
