// Reading one row of a [rows, V] bf16 tensor in 16-byte vectors whatever V is.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "common.cuh"

namespace tv {

// The row is covered by the aligned 16-byte vectors of memory it lies in: vector i holds entries 8 i - off .. 8 i - off + 7.
// vector() gives the vectors that lie wholly inside the row and -inf for all others; edge() gives the entries that are
// left, at most seven before the first such vector and at most seven behind the last one.  (Putting the outer vectors
// together inside vector() cost registers and kept a thread's loads from being issued together.)  All loads bypass L1: a
// scan that starts ahead of its wait must not meet a line that an earlier launch on this SM has left there.
struct LogitsRow {
  const uint16_t* row;
  int off, V;
  __device__ __forceinline__ LogitsRow(const tv_bf16* logits, long long r, int V_) : row(logits + r * V_), V(V_) {
    off = (int)((reinterpret_cast<uintptr_t>(row) & 15u) >> 1);
  }
  __device__ __forceinline__ uint4 vector(int i) const {
    const int v = 8 * i - off;
    return v >= 0 && v <= V - 8 ? __ldcg(reinterpret_cast<const uint4*>(row + v))
                                : make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u);
  }
  // Entry number t (0..15) of those no whole vector holds, or -1.
  __device__ __forceinline__ int edge(int t) const {
    const int head = min((8 - off) & 7, V);               // entries before the first aligned vector
    const int tail = head + ((V - head) & ~7);            // first entry behind the last one
    const int v = t < 8 ? t : tail + t - 8;
    return t < 8 ? (v < head ? v : -1) : (v < V ? v : -1);
  }
  __device__ __forceinline__ float entry(int v) const { return __uint_as_float((uint32_t)__ldcg(row + v) << 16); }
};

// Streaming the rows through shared memory: a warp requests stage after stage with bulk copies, 24 others reduce them.  A
// stage is one item, 16384 logits of one row; three groups of eight warps take the items in turn, each warp 2048 of them.
// The copies need no registers, so that a whole ring (192 KB of an SM's 227) is on its way, where loads of the reducing
// threads drain at every item's end.  Greedy call, 16 x 60 rows of 153600 (295 MB, 45.1 us at the rate of a copy): 56.6 -> 47.1 us;
// two groups 48.8, one 64.4; five stages 48.6.  8 x 64 rows of 128256: 27.6 -> 23.9 us.  Sampling call: 68.7 -> 63.3 us.
constexpr int kStreamStages = 6;
constexpr int kStreamGroups = 3;
constexpr int kStreamWarps = 8;                                     // of a group
constexpr int kStreamVecs = 8;                                      // 16-byte vectors of a lane
constexpr int kStreamSlice = 32 * kStreamVecs * 8;                  // 2048 logits of a warp
constexpr int kStreamItem = kStreamWarps * kStreamSlice;            // 16384 logits
constexpr int kStreamThreads = 32 * (kStreamGroups * kStreamWarps + 1);
constexpr int kStreamStageBytes = kStreamItem * 2;
constexpr int kStreamSmem = kStreamStages * (kStreamStageBytes + 2 * 8 + 8) + 16;
constexpr unsigned long long kStreamWaitNs = 2000000000ull;

__device__ __forceinline__ unsigned long long stream_now() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ bool stream_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// Bounded; false when the wait was given up here or elsewhere in the CTA.
__device__ __forceinline__ bool stream_wait(uint32_t bar, uint32_t parity, volatile int* gone) {
  bool ok = stream_try(bar, parity);
  if (!ok) {
    const unsigned long long t0 = stream_now();
    while (!(ok = stream_try(bar, parity))) {
      if (*gone || stream_now() - t0 > kStreamWaitNs) {
        *gone = 1;
        break;
      }
    }
  }
  return __all_sync(0xffffffffu, ok);
}
__device__ __forceinline__ void stream_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// reduce(row, item of the row, w, first, r, u, rest, rest_v, stage): called by a converged warp, number w of its group, with
// the vectors of its slice (-inf outside the row's whole vectors); first = number in the row of lane 0's u[0], r the row.
// Lanes 0-15 also get one entry each that no whole vector holds (rest_v: its index in the row, -1 if there is none), in the
// slice that it lies in (own_slice) or in the row's first.  Rows of padded nodes are never read.  n_items = rows * n_chunks.
template <bool own_slice, class F>
__device__ __forceinline__ void stream_rows(const tv_bf16* __restrict__ logits, const int32_t* __restrict__ n_nodes, int Nmax, int V,
                                            int n_chunks, int n_items, int32_t* __restrict__ status, F&& reduce) {
  extern __shared__ __align__(128) uint8_t stream_smem[];
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(stream_smem);
  const uint32_t full = base + kStreamStages * kStreamStageBytes, empty = full + kStreamStages * 8;
  volatile int* items = reinterpret_cast<volatile int*>(stream_smem + kStreamStages * (kStreamStageBytes + 16));
  volatile int* gone = items + 2 * kStreamStages;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kStreamStages; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full + 8 * i) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(empty + 8 * i), "n"(kStreamWarps) : "memory");
    }
    *gone = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  bool ok = true;
  if (warp == kStreamGroups * kStreamWarps) {
    uint64_t policy;      // read once: first in line for eviction from L2
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    unsigned k = 0;                                  // items of this CTA so far
    auto stage_free = [&]() -> bool {
      return k < kStreamStages || stream_wait(empty + 8 * (k % kStreamStages), (k / kStreamStages + 1) & 1u, gone);
    };
    // 32 items of this CTA at a time: which of them belong to a node
    for (long long i0 = blockIdx.x; ok && i0 < n_items; i0 += 32ll * gridDim.x) {
      const long long mine = i0 + (long long)lane * gridDim.x;
      bool active = mine < n_items;
      if (active) {
        const int row = (int)mine / n_chunks, b = row / Nmax;
        active = row - b * Nmax < __ldcg(n_nodes + b);      // (not from an L1 line that an earlier launch on this SM has left)
      }
      unsigned todo = __ballot_sync(0xffffffffu, active);
      while (ok && todo) {
        const int item = (int)(i0 + (long long)(__ffs(todo) - 1) * gridDim.x);
        todo &= todo - 1;
        ok = stage_free();
        if (ok && lane == 0) {
          const int row = item / n_chunks, chunk = item - row * n_chunks, st = k % kStreamStages;
          const LogitsRow r(logits, row, V);
          const int lo = chunk * (kStreamItem / 8);
          const int a = max(lo, r.off ? 1 : 0), z = min(lo + kStreamItem / 8, (V + r.off) / 8);      // whole vectors [a, z)
          items[2 * st] = row;
          items[2 * st + 1] = chunk;
          if (z > a) {
            const uint32_t bytes = (uint32_t)(z - a) * 16u;
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full + 8 * st), "r"(bytes) : "memory");
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
                    base + st * kStreamStageBytes + (a - lo) * 16),
                "l"(r.row + 8 * a - r.off), "r"(bytes), "r"(full + 8 * st), "l"(policy)
                : "memory");
          } else {
            stream_arrive(full + 8 * st);
          }
        }
        __syncwarp();
        ++k;
      }
    }
    for (int g = 0; ok && g < kStreamGroups; ++g, ++k) {      // no more items
      ok = stage_free();
      if (ok && lane == 0) {
        items[2 * (k % kStreamStages)] = -1;
        stream_arrive(full + 8 * (k % kStreamStages));
      }
      __syncwarp();
    }
  } else {
    const int w = warp % kStreamWarps;
    for (unsigned k = warp / kStreamWarps;; k += kStreamGroups) {
      const int st = k % kStreamStages;
      ok = stream_wait(full + 8 * st, (k / kStreamStages) & 1u, gone);
      if (!ok) break;
      const int row = items[2 * st], chunk = items[2 * st + 1];
      if (row < 0) break;
      const LogitsRow r(logits, row, V);
      float rest = -INFINITY;
      int rest_v = -1;
      if (lane < 16 && (own_slice ? chunk == 0 || chunk + 2 >= n_chunks : chunk == 0 && w == 0)) {
        rest_v = r.edge(lane);
        if (own_slice && rest_v >= 0 && (rest_v + r.off) / kStreamSlice != chunk * kStreamWarps + w) rest_v = -1;
        if (rest_v >= 0) rest = r.entry(rest_v);
      }
      const int in_stage = w * (kStreamSlice / 8), first = chunk * (kStreamItem / 8) + in_stage;
      uint4 u[kStreamVecs];
#pragma unroll
      for (int q = 0; q < kStreamVecs; ++q) {
        const int i = in_stage + q * 32 + lane, v = 8 * (first + q * 32 + lane) - r.off;
        u[q] = v >= 0 && v <= V - 8 ? *reinterpret_cast<const uint4*>(stream_smem + st * kStreamStageBytes + i * 16)
                                    : make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u);
      }
      reduce(row, chunk, w, first, r, u, rest, rest_v, st);
      __syncwarp();
      if (lane == 0) stream_arrive(empty + 8 * st);
    }
  }
  if (!ok) {      // a copy that never came: reported, and given time to land before the shared memory is released
    if (lane == 0)
      for (int b = 0; b < (n_items / n_chunks) / Nmax; ++b) atomicOr(status + b, TV_ST_TIMEOUT);
    const unsigned long long t0 = stream_now();
    while (stream_now() - t0 < 200000ull) {
    }
  }
}

// The shared memory of stream_rows is more than a kernel gets unasked: once per kernel and device.
template <auto kernel>
inline cudaError_t stream_configure() {
  static std::atomic<bool> configured[64];
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || (dev >= 0 && dev < 64 && configured[dev].load(std::memory_order_acquire))) return e;
  e = cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel), cudaFuncAttributeMaxDynamicSharedMemorySize, kStreamSmem);
  if (e == cudaSuccess && dev >= 0 && dev < 64) configured[dev].store(true, std::memory_order_release);
  return e;
}

}  // namespace tv
