// tree_merge_partials: attention over a key set that was split in R disjoint ranges (one per GPU of a
// context-split group), from the per-range outputs and log-sum-exps (Section 6, "Limitations and future
// work": longer-context, multi-device serving; the attention is Section 2.4).  For every query row
//   out = sum_r w_r O_r / sum_r w_r,  w_r = exp(lse_r - max_r lse_r),  lse = max + log sum_r w_r.
// Pure streaming: R reads of the partials, one write; one thread per (row, 8 output columns), four ranges' weights and
// payloads requested together.  Eight ranges of 4 x 128 nodes x 32 heads (38 MB, 5.8 us at the copy rate): 11.0 -> 8.4 us,
// two ranges 5.9 -> 4.8; with eight ranges in flight 9.2 and 6.5 (fewer threads fit an SM).
#include "common.cuh"

#include <cuda_bf16.h>

namespace {

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

constexpr int kThreads = 128;
constexpr int kHold = 4;          // ranges whose loads are in flight together

// Index: 32 bits wherever the number of threads fits (five 64-bit divisions per thread took longer than its loads).
template <typename Index>
__global__ void __launch_bounds__(kThreads)
merge_partials_kernel(const uint4* __restrict__ o_parts, const float* __restrict__ lse_parts, int R,
                      int B, int Nmax, int Hq, int d8, uint4* __restrict__ out, float* __restrict__ lse_out) {
  tv::pdl_enter();
  const Index total = (Index)B * Nmax * Hq * d8;
  const Index t = (Index)blockIdx.x * kThreads + threadIdx.x;
  if (t >= total) return;
  const Index row = t / (Index)d8;                    // (b * Nmax + node) * Hq + h
  const int cg = (int)(t - row * (Index)d8);
  const Index bn = row / (Index)Hq;
  const int h = (int)(row - bn * (Index)Hq);
  const int b = (int)(bn / (Index)Nmax);
  const int node = (int)(bn - (Index)b * (Index)Nmax);
  const long long rows = (long long)B * Nmax * Hq;
  const long long lse_idx = ((long long)b * Hq + h) * Nmax + node;
  const float* lp = lse_parts + lse_idx;
  const uint4* op = o_parts + t;
  float m = -INFINITY;                                 // running maximum: more than kHold ranges rescale what they find
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  float tot = 0.f;
  bool nan = false;                                    // a log-sum-exp that is NaN: the row is NaN, unless no range has a key
  for (int r0 = 0; r0 < R; r0 += kHold) {
    float w[kHold];
    uint4 v[kHold];
#pragma unroll
    for (int k = 0; k < kHold; ++k) w[k] = r0 + k < R ? __ldcs(lp + (r0 + k) * rows) : -INFINITY;
#pragma unroll
    for (int k = 0; k < kHold; ++k)
      if (r0 + k < R) v[k] = __ldcs(op + (r0 + k) * rows * d8);
    float mx = m;
#pragma unroll
    for (int k = 0; k < kHold; ++k) {
      mx = fmaxf(mx, w[k]);
      nan |= w[k] != w[k];
    }
    if (mx == -INFINITY) continue;
    const float keep = expf(m - mx);                   // 0 the first time
    m = mx;
    tot *= keep;
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = keep == 0.f ? 0.f : acc[i] * keep;      // (what has no weight left may not be finite)
#pragma unroll
    for (int k = 0; k < kHold; ++k) {
      const float wk = expf(w[k] - mx);
      if (wk != 0.f) {                                 // the payload of an empty range (weight 0) may be anything
        tot += wk;
        const uint32_t e[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          acc[2 * i] = fmaf(wk, bf16_lo(e[i]), acc[2 * i]);
          acc[2 * i + 1] = fmaf(wk, bf16_hi(e[i]), acc[2 * i + 1]);
        }
      }
    }
  }
  if (nan && m > -INFINITY) tot = acc[0] = acc[1] = acc[2] = acc[3] = acc[4] = acc[5] = acc[6] = acc[7] = NAN;
  const float inv = tot > 0.f ? 1.f / tot : 0.f;
  uint4 o;
  o.x = pack_bf16(acc[0] * inv, acc[1] * inv);
  o.y = pack_bf16(acc[2] * inv, acc[3] * inv);
  o.z = pack_bf16(acc[4] * inv, acc[5] * inv);
  o.w = pack_bf16(acc[6] * inv, acc[7] * inv);
  out[t] = o;
  if (lse_out && cg == 0) lse_out[lse_idx] = tot > 0.f ? m + logf(tot) : -INFINITY;
}

}  // namespace

extern "C" int tree_merge_partials(const tv_bf16* o_parts, const float* lse_parts, int R, int B, int Nmax, int Hq, int d,
                                   tv_bf16* out, float* lse, tv_stream stream) {
  TV_REQUIRE(o_parts && lse_parts && out, "tree_merge_partials: NULL pointer");
  TV_REQUIRE(R >= 1 && B >= 0 && Nmax >= 1 && Hq >= 1 && d >= 8 && d % 8 == 0,
             "tree_merge_partials: need R >= 1, B >= 0, Nmax >= 1, Hq >= 1, d a multiple of 8");
  TV_REQUIRE(tv::aligned16(o_parts) && tv::aligned16(out), "tree_merge_partials: tensors must be 16-byte aligned");
  if (B == 0) return TV_OK;
  const long long total = (long long)B * Nmax * Hq * (d / 8);
  TV_REQUIRE((total + kThreads - 1) / kThreads < (1ll << 31), "tree_merge_partials: problem too large for one launch");
  const auto launch = [&](auto kernel) {
    return tv::launch_pdl(kernel, dim3((unsigned)((total + kThreads - 1) / kThreads)), dim3(kThreads), 0, (cudaStream_t)stream,
                          reinterpret_cast<const uint4*>(o_parts), lse_parts, R, B, Nmax, Hq, d / 8,
                          reinterpret_cast<uint4*>(out), lse);
  };
  TV_CUDA_OK(total < (1ll << 31) ? launch(merge_partials_kernel<unsigned>) : launch(merge_partials_kernel<long long>));
  tv::count_launches(1);
  return TV_OK;
}
