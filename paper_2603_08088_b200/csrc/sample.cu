// tree_accept_sample: sampling-mode acceptance over the tree (Section 2.2: an acceptance rule "rejection
// sampling style" that keeps the teacher's distribution; Section 3.3: the node scores are what it consumes).
// The rule is speculative sampling for proposals without a draft probability (q = one-hot), walked down the
// tree: at the current node the children are tried in node order, child k with token x is accepted iff
// u_node[k] < p(x) / (1 - mass rejected so far at this node), a rejected token's mass is removed; when no
// child passes, the next token is drawn from what is left of p by inversion of the cumulative sum in
// vocabulary order at u_bonus.  p = softmax(logits / T) of the current node's row.
//
// Phase 1 (row_stats_stream_kernel, row_stats_kernel for few rows) streams logits[B,Nmax,V] once: every warp reduces one
// vocabulary chunk of one row to (max, sum of 2^((l - max) k)), k = log2(e) / T.  Phase 2 (sample_walk_kernel), one CTA per
// sequence: folds the chunk pairs per row, gathers the mass of every node's token in its parent's row, walks the tree with one warp, and
// draws the next token from the last node's row by two scans in vocabulary order: over the masses of its chunks, then
// over the entries of the chunk that holds the target.  All arithmetic in fp32.
#include "common.cuh"
#include "logits.cuh"

#include <cuda_bf16.h>

namespace {

constexpr int kStatThreads = 256;
constexpr int kStatChunk = tv::kStreamSlice;                          // 2048 logits: a warp's share of an item
constexpr int kWalkThreads = 1024;
constexpr int kLanesPerRow = 8;                                       // lanes that fold one row's chunk pairs
constexpr int kMaxNodes = 256;
constexpr float kLog2e = 1.4426950408889634f;

struct RowStat {
  float m;      // maximum of the chunk (raw logit units); -inf for an empty chunk
  float s;      // sum over the chunk of 2^((l - m) * k)
};

__device__ __forceinline__ float bf16_to_float(uint32_t bits16) { return __uint_as_float(bits16 << 16); }

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Unnormalised mass of a vocabulary entry with logit l in a row whose maximum is M: 2^((l - M) k); 0 for NaN
// and -inf (fmaxf returns its other operand for a NaN, and 2^-150 flushes to 0).
__device__ __forceinline__ float mass_of(float l, float M, float k) {
  return ex2_approx(fmaxf((l - M) * k, -150.f));
}

// (m, s) <- (m, s) merged with (mo, so): s = sum of 2^((l - m) k) over a set whose maximum is m.
__device__ __forceinline__ void merge_pair(float& m, float& s, float mo, float so, float k) {
  const float M = fmaxf(m, mo);
  if (M > -INFINITY) {
    s = (m > -INFINITY ? s * ex2_approx((m - M) * k) : 0.f) + (mo > -INFINITY ? so * ex2_approx((mo - M) * k) : 0.f);
    m = M;
  }
}

// (max, sum) of a chunk whose vectors a converged warp holds, with one more entry in some lanes (-inf: none): the maximum
// first (packed bf16), then one exponential per logit.
__device__ __forceinline__ RowStat chunk_stat(const uint4* u, float rest, float k) {
  __nv_bfloat162 mx = *reinterpret_cast<const __nv_bfloat162*>(&u[0].x);
#pragma unroll
  for (int q = 0; q < tv::kStreamVecs; ++q) {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u[q]);
    mx = __hmax2(mx, __hmax2(__hmax2(h[0], h[1]), __hmax2(h[2], h[3])));
  }
  RowStat out;
  out.s = 0.f;
  out.m = fmaxf(fmaxf(__low2float(mx), __high2float(mx)), rest);      // max of a NaN and x is x: only NaNs give a NaN
  if (!(out.m == out.m)) out.m = -INFINITY;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) out.m = fmaxf(out.m, __shfl_xor_sync(0xffffffffu, out.m, off));
  if (out.m > -INFINITY) {
    // (l - m) k in this order, as mass_of has it: the mass of the maximum is 1 and the rounding is that of the difference.  As
    // l k - m k in one FMA the rounding of m k, 2^-24 |m k| of every mass of the chunk, grows without limit as 1 / T.
    const float2 k2 = make_float2(k, k), m2 = make_float2(-out.m, -out.m);
    float2 sum = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < tv::kStreamVecs; ++q) {
      const uint32_t e[4] = {u[q].x, u[q].y, u[q].z, u[q].w};
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        float2 x = __fmul2_rn(__fadd2_rn(make_float2(__uint_as_float(e[t] << 16), __uint_as_float(e[t] & 0xffff0000u)), m2), k2);
        x.x = ex2_approx(fmaxf(x.x, -150.f));
        x.y = ex2_approx(fmaxf(x.y, -150.f));
        sum = __fadd2_rn(sum, x);
      }
    }
    out.s = sum.x + sum.y + mass_of(rest, out.m, k);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) out.s += __shfl_xor_sync(0xffffffffu, out.s, off);
  }
  return out;
}

// Long scans (see stream_rows).  Bounds: the logits once through HBM (295 MB: 45 us), one special-function result per
// logit (147 M: 33 us).
__global__ void __launch_bounds__(tv::kStreamThreads, 1)
row_stats_stream_kernel(const tv_bf16* __restrict__ logits, const int32_t* __restrict__ n_nodes, int Nmax, int V, int n_chunks,
                        int row_items, int n_items, float k, RowStat* __restrict__ stats, int32_t* __restrict__ status) {
  tv::pdl_enter();
  tv::stream_rows<true>(logits, n_nodes, Nmax, V, row_items, n_items, status,
                        [&](int row, int item, int w, int, const tv::LogitsRow&, const uint4* u, float rest, int, int) {
    const int chunk = item * tv::kStreamWarps + w;
    if (chunk >= n_chunks) return;
    const RowStat out = chunk_stat(u, rest, k);
    if ((threadIdx.x & 31) == 0) stats[(size_t)row * n_chunks + chunk] = out;
  });
}

// Short scans: persistent, one warp per (row, chunk) item, no barrier anywhere; a warp requests the vectors of its next item
// before it reduces the ones it holds.
__global__ void __launch_bounds__(kStatThreads, 3)
row_stats_kernel(const tv_bf16* __restrict__ logits, const int32_t* __restrict__ n_nodes, int Nmax, int V,
                 int n_chunks, int n_items, float k, RowStat* __restrict__ stats) {
  tv::pdl_enter();
  const int lane = threadIdx.x & 31;
  const int n_warps = gridDim.x * (kStatThreads / 32);
  auto locate = [&](int item, int& row, int& chunk) -> bool {
    if (item >= n_items) return false;
    row = item / n_chunks;
    chunk = item - row * n_chunks;
    const int b = row / Nmax;
    return row - b * Nmax < n_nodes[b];
  };
  auto fetch = [&](int row, int chunk, uint4* u) {
    const tv::LogitsRow r(logits, row, V);
#pragma unroll
    for (int q = 0; q < tv::kStreamVecs; ++q) u[q] = r.vector((chunk * tv::kStreamVecs + q) * 32 + lane);
  };
  int item = blockIdx.x * (kStatThreads / 32) + (threadIdx.x >> 5);
  int row = 0, chunk = 0;
  bool active = locate(item, row, chunk);
  uint4 u[tv::kStreamVecs];
  if (active) fetch(row, chunk, u);
  while (item < n_items) {
    const int nitem = item + n_warps;
    int nrow = 0, nchunk = 0;
    const bool nactive = locate(nitem, nrow, nchunk);
    uint4 un[tv::kStreamVecs];
    if (nactive) fetch(nrow, nchunk, un);
    if (active) {
      // entries outside the row's whole vectors, in the chunk they lie in
      float rest = -INFINITY;
      if (lane < 16 && (chunk == 0 || chunk >= n_chunks - 2)) {
        const tv::LogitsRow r(logits, row, V);
        const int v = r.edge(lane);
        if (v >= 0 && (v + r.off) / kStatChunk == chunk) rest = r.entry(v);
      }
      const RowStat out = chunk_stat(u, rest, k);
      if (lane == 0) stats[(size_t)row * n_chunks + chunk] = out;
    }
    item = nitem;
    row = nrow;
    chunk = nchunk;
    active = nactive;
#pragma unroll
    for (int q = 0; q < tv::kStreamVecs; ++q) u[q] = un[q];
  }
}

// Inclusive scan over the CTA in thread order; `total` is the sum over all threads.  Two barriers.
__device__ __forceinline__ float block_scan(float v, float* warp_sums, float& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float o = __shfl_up_sync(0xffffffffu, v, off);
    if (lane >= off) v += o;
  }
  if (lane == 31) warp_sums[warp] = v;
  __syncthreads();
  float w = warp_sums[lane];                   // kWalkThreads / 32 = 32 warps
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float o = __shfl_up_sync(0xffffffffu, w, off);
    if (lane >= off) w += o;
  }
  total = __shfl_sync(0xffffffffu, w, 31);
  const float before = __shfl_sync(0xffffffffu, w, (warp + 31) & 31);
  __syncthreads();
  return v + (warp > 0 ? before : 0.f);
}

// One CTA per sequence.  A chain of dependent round trips, so everything that does not depend on the row statistics
// (tree, tokens, uniforms, the token logits) is fetched while row_stats_kernel still runs: that kernel lets this one
// start only after every earlier kernel of the stream has completed, and the loads bypass L1.  The draw reads one chunk
// of the row (4 KB), and the ones with rejected tokens, and not the row up to the crossing (walk and draw took 37 us before).
__global__ void __launch_bounds__(kWalkThreads)
sample_walk_kernel(const tv_bf16* __restrict__ logits, const RowStat* __restrict__ stats, int n_chunks,
                   const int32_t* __restrict__ tokens, const int32_t* __restrict__ parent,
                   const int32_t* __restrict__ n_nodes, const float* __restrict__ u_node,
                   const float* __restrict__ u_bonus, float k, int Nmax, int V, int Dp1,
                   int32_t* __restrict__ accept_len, int32_t* __restrict__ accepted_nodes,
                   int32_t* __restrict__ next_token, int32_t* __restrict__ status) {
  static_assert(kWalkThreads == 1024 && kMaxNodes <= kWalkThreads, "block_scan and the node arrays rely on it");
  __shared__ float sM[kMaxNodes], sZ[kMaxNodes], sE[kMaxNodes], sU[kMaxNodes];   // row max, row sum, token mass, uniform
  __shared__ int sPar[kMaxNodes], sTok[kMaxNodes], sRej[kMaxNodes];
  __shared__ float sKept[kMaxNodes];                              // what is left of the chunk that holds rejected token x
  __shared__ uint32_t sHide[kWalkThreads / 32][kStatChunk / 32];  // per warp: rejected entries of the chunk it sums
  __shared__ float sWarp[kWalkThreads / 32];
  __shared__ int sLast, sNrej, sChunk, sHit, sLastMass;
  __shared__ float sExcl;
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  int n = __ldcg(n_nodes + b);
  n = n < 0 ? 0 : (n > Nmax ? Nmax : n);
  const uint16_t* lg = reinterpret_cast<const uint16_t*>(logits) + (size_t)b * Nmax * V;
  float tok_logit = -INFINITY;
  bool bad = false;
  if (tid < n) {
    const int p = __ldcg(parent + (size_t)b * Nmax + tid), x = __ldcg(tokens + (size_t)b * Nmax + tid);
    const int sp = (p >= 0 && p < n) ? p : 0;            // dummy-root remap (Section 3.2)
    sPar[tid] = sp;
    sTok[tid] = x;
    sU[tid] = __ldcg(u_node + (size_t)b * Nmax + tid);
    if (tid >= 1) {
      bad = x < 0 || x >= V;
      if (!bad) tok_logit = bf16_to_float(__ldcg(lg + (size_t)sp * V + x));
    }
  }
  const float ub = __ldcg(u_bonus + b);
  if (tid == 0) {
    sChunk = sHit = sLastMass = -1;
  }
  tv::pdl_enter();
  const bool any_bad = __syncthreads_or(bad);
  // ---- per-row maximum and sum: kLanesPerRow lanes fold a row's chunk pairs
  for (int i0 = 0; i0 < n; i0 += kWalkThreads / kLanesPerRow) {
    const int i = i0 + tid / kLanesPerRow;
    float M = -INFINITY, Z = 0.f;
    if (i < n) {
      const RowStat* rs = stats + ((size_t)b * Nmax + i) * n_chunks;
#pragma unroll 8
      for (int c = tid % kLanesPerRow; c < n_chunks; c += kLanesPerRow) merge_pair(M, Z, rs[c].m, rs[c].s, k);
    }
#pragma unroll
    for (int off = kLanesPerRow / 2; off > 0; off >>= 1) {
      const float mo = __shfl_xor_sync(0xffffffffu, M, off), so = __shfl_xor_sync(0xffffffffu, Z, off);
      merge_pair(M, Z, mo, so, k);
    }
    if (i < n && tid % kLanesPerRow == 0) {
      sM[i] = M;
      sZ[i] = Z;
    }
  }
  __syncthreads();
  // ---- mass of every node's token in its parent's row (the node score of Section 3.3, exponentiated)
  if (tid < n) sE[tid] = (tid >= 1 && !bad) ? mass_of(tok_logit, sM[sPar[tid]], k) : 0.f;
  __syncthreads();
  // ---- the walk (one warp): the children of a node are found 32 nodes at a time and tried in node order
  if (tid < 32) {
    int c = 0, depth = 0, nrej = 0;
    float rem = n > 0 ? sZ[0] : 0.f;
    for (int j = lane; j < Dp1; j += 32) accepted_nodes[(size_t)b * Dp1 + j] = 0;
    __syncwarp();
    while (depth < Dp1 - 1) {
      int acc = -1;
      for (int base = (c + 1) & ~31; base < n && acc < 0; base += 32) {
        const int kk = base + lane;
        bool child = kk > c && kk < n && sPar[kk] == c;
        if (child) child = sTok[kk] >= 0 && sTok[kk] < V;
        unsigned todo = __ballot_sync(0xffffffffu, child);
        while (todo) {
          const int cand = base + __ffs(todo) - 1;
          todo &= todo - 1;
          const int x = sTok[cand];
          bool dup = false;
          for (int r0 = 0; r0 < nrej; r0 += 32) dup |= __any_sync(0xffffffffu, r0 + lane < nrej && sRej[r0 + lane] == x);
          if (dup) continue;
          const float prob = rem > 0.f ? sE[cand] / rem : 0.f;
          if (sU[cand] < prob) {
            acc = cand;
            break;
          }
          if (lane == 0) sRej[nrej] = x;
          __syncwarp();
          ++nrej;
          rem -= sE[cand];
        }
      }
      if (acc < 0) break;
      ++depth;
      if (lane == 0) accepted_nodes[(size_t)b * Dp1 + depth] = acc;
      c = acc;
      nrej = 0;
      rem = sZ[c];
    }
    if (lane == 0) {
      accept_len[b] = depth;
      sLast = c;
      sNrej = nrej;
      if (any_bad) atomicOr(status + b, TV_ST_BAD_INDEX);
    }
  }
  __syncthreads();
  // ---- next token: the first entry of row c, rejected tokens left out, whose cumulative mass in vocabulary order
  // exceeds the target, u_bonus of what is left.
  if (n == 0) {
    if (tid == 0) next_token[b] = -1;       // no row to draw from
    return;
  }
  const int c = sLast, nrej = sNrej;
  const float M = sM[c];
  const uint16_t* row = lg + (size_t)c * V;
  const tv::LogitsRow lr(logits, (long long)b * Nmax + c, V);
  const int off = lr.off;                                      // chunk q holds entries q * kStatChunk - off ...
  const RowStat* row_stats = stats + ((size_t)b * Nmax + c) * n_chunks;
  RowStat st = {-INFINITY, 0.f};
  if (tid < n_chunks) st = row_stats[tid];
  // A chunk with rejected tokens is summed again without them, by one warp: taking their masses off its sum would leave the
  // rounding of that sum, which is more than all other entries where the rejected ones have nearly all of the mass.
  for (int x = tid >> 5; x < nrej; x += kWalkThreads / 32) {
    const int q = (sRej[x] + off) / kStatChunk;
    bool first = true;                                         // of the rejected tokens in this chunk
    for (int y0 = 0; y0 < x; y0 += 32)
      first &= !__any_sync(0xffffffffu, y0 + lane < x && (sRej[y0 + lane] + off) / kStatChunk == q);
    float sum = 0.f;
    if (first) {
      uint4 u[tv::kStreamVecs];                                // requested before anything else
#pragma unroll
      for (int w = 0; w < tv::kStreamVecs; ++w) u[w] = lr.vector((q * tv::kStreamVecs + w) * 32 + lane);
      const int v = lane < 16 ? lr.edge(lane) : -1, at_v = v + off - q * kStatChunk;
      const bool mine = v >= 0 && at_v >= 0 && at_v < kStatChunk;
      const float rest = mine ? lr.entry(v) : -INFINITY;
      uint32_t* hide = sHide[tid >> 5];
      hide[lane] = hide[lane + 32] = 0u;
      __syncwarp();
      for (int y = x + lane; y < nrej; y += 32) {
        const int at = sRej[y] + off - q * kStatChunk;
        if (at >= 0 && at < kStatChunk) atomicOr(&hide[at >> 5], 1u << (at & 31));
      }
      __syncwarp();
      if (mine && !((hide[at_v >> 5] >> (at_v & 31)) & 1u)) sum = mass_of(rest, M, k);
#pragma unroll
      for (int w = 0; w < tv::kStreamVecs; ++w) {
        const uint32_t hidden = hide[w * 8 + (lane >> 2)] >> ((lane & 3) * 8);
        const uint32_t e[4] = {u[w].x, u[w].y, u[w].z, u[w].w};
#pragma unroll
        for (int t = 0; t < 8; ++t)
          sum += (hidden >> t) & 1u ? 0.f : mass_of(bf16_to_float((t & 1) ? (e[t >> 1] >> 16) : (e[t >> 1] & 0xffffu)), M, k);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      __syncwarp();                                            // (the next round of this warp writes `hide`)
    }
    if (lane == 0) sKept[x] = first ? sum : -1.f;
  }
  __syncthreads();
  auto chunk_mass = [&](int q) -> float {                      // st: the chunk's statistics
    float mass = st.m > -INFINITY ? st.s * ex2_approx(fmaxf((st.m - M) * k, -150.f)) : 0.f;
    for (int x = 0; x < nrej; ++x)
      if ((sRej[x] + off) / kStatChunk == q && sKept[x] >= 0.f) mass = sKept[x];
    return mass;
  };
  // first the chunk: cumulative masses of the chunks (rows of at most kWalkThreads of them take one round)
  float left = 0.f, mass = 0.f, incl = 0.f, total;
  for (int q0 = 0; q0 < n_chunks; q0 += kWalkThreads) {
    const int q = q0 + tid;
    if (q0 > 0 && q < n_chunks) st = row_stats[q];
    mass = q < n_chunks ? chunk_mass(q) : 0.f;
    incl = left + block_scan(mass, sWarp, total);
    left += total;
  }
  const float target = ub * left;
  float carried = 0.f;
  for (int q0 = 0; q0 < n_chunks; q0 += kWalkThreads) {
    const int q = q0 + tid;
    if (n_chunks > kWalkThreads) {
      if (q < n_chunks) st = row_stats[q];
      mass = q < n_chunks ? chunk_mass(q) : 0.f;
      incl = carried + block_scan(mass, sWarp, total);
      carried += total;
    }
    if (mass > 0.f) {
      if (target < incl) atomicMin(reinterpret_cast<unsigned*>(&sChunk), (unsigned)q);      // -1 is the largest unsigned
      atomicMax(&sLastMass, q);
    }
    __syncthreads();
    if (sChunk >= 0) {                                 // uniform: read after the barrier
      if (q == sChunk) sExcl = incl - mass;
      break;
    }
  }
  // rounding can leave the target above the scanned total (u_bonus close to 1): the last chunk with mass then, and the
  // last of its entries that has mass
  const int chunk = sChunk >= 0 ? sChunk : max(sLastMass, 0);
  auto entry_mass = [&](int v) -> float {
    if (v < 0 || v >= V) return 0.f;
    for (int x = 0; x < nrej; ++x)
      if (sRej[x] == v) return 0.f;
    return mass_of(bf16_to_float(row[v]), M, k);
  };
  __syncthreads();
  const float excl = sChunk >= 0 ? sExcl : INFINITY;
  if (tid == 0) sLastMass = -1;
  __syncthreads();
  {
    constexpr int kPer = kStatChunk / kWalkThreads;       // entries per thread, in vocabulary order
    const int v0 = chunk * kStatChunk - off + tid * kPer;
    float vals[kPer], sum = 0.f;
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      vals[t] = entry_mass(v0 + t);
      sum += vals[t];
    }
    float total;
    float cum = excl + (block_scan(sum, sWarp, total) - sum);
    int first = -1, last = -1;
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      cum += vals[t];
      if (vals[t] > 0.f) {
        last = v0 + t;
        if (first < 0 && cum > target) first = v0 + t;
      }
    }
    if (excl == INFINITY) first = -1;
    if (first >= 0) atomicMin(reinterpret_cast<unsigned*>(&sHit), (unsigned)first);
    if (last >= 0) atomicMax(&sLastMass, last);
  }
  __syncthreads();
  if (tid == 0) next_token[b] = sHit >= 0 ? sHit : (sLastMass >= 0 ? sLastMass : V - 1);
}

// A row may start anywhere inside a 16-byte vector, so up to seven entries of it fall into one more vector.
int stat_chunks(int V) { return (int)(((long long)V + 7 + kStatChunk - 1) / kStatChunk); }

}  // namespace

extern "C" size_t tv_sample_workspace_bytes(int B, int Nmax, int V) {
  if (B <= 0 || Nmax <= 0 || V <= 0) return 16;
  return (size_t)B * Nmax * stat_chunks(V) * sizeof(RowStat);
}

extern "C" int tree_accept_sample(const tv_bf16* logits, const int32_t* tokens, const int32_t* parent,
                                  const int32_t* n_nodes, const float* u_node, const float* u_bonus,
                                  float temperature, int B, int Nmax, int V, int Dp1,
                                  int32_t* accept_len, int32_t* accepted_nodes, int32_t* next_token,
                                  void* workspace, size_t workspace_bytes,
                                  int32_t* status, tv_stream stream) {
  TV_REQUIRE(logits && tokens && parent && n_nodes && u_node && u_bonus && accept_len && accepted_nodes && next_token &&
                 workspace && status,
             "tree_accept_sample: NULL pointer");
  TV_REQUIRE(B >= 0 && Nmax >= 1 && Nmax <= kMaxNodes && V >= 1 && Dp1 >= 1,
             "tree_accept_sample: need B >= 0, 1 <= Nmax <= 256, V >= 1, Dp1 >= 1");
  TV_REQUIRE(temperature > 0.f, "tree_accept_sample: temperature must be > 0 (tree_accept is the greedy rule)");
  TV_REQUIRE((long long)B * Nmax <= 65535, "tree_accept_sample: B * Nmax must be <= 65535");
  if (workspace_bytes < tv_sample_workspace_bytes(B, Nmax, V))
    return tv::fail(TV_ERR_WORKSPACE, "tree_accept_sample: workspace of %zu bytes, need %zu", workspace_bytes,
                    tv_sample_workspace_bytes(B, Nmax, V));
  if (B == 0) return TV_OK;
  const int n_chunks = stat_chunks(V);
  const float k = kLog2e / temperature;
  RowStat* stats = static_cast<RowStat*>(workspace);
  cudaStream_t s = (cudaStream_t)stream;
  const int row_items = (n_chunks + tv::kStreamWarps - 1) / tv::kStreamWarps;
  const long long n_slices = (long long)B * Nmax * n_chunks, n_items = (long long)B * Nmax * row_items;
  TV_REQUIRE(n_slices < (1ll << 31) - (1 << 20), "tree_accept_sample: B * Nmax * ceil(V / 2048) must stay below 2^31");
  // The long scan from 24 items an SM on (us a call, short / long: 13.8 items an SM 22.3 / 23.2, 21.6 29.1 / 29.3, 43 47.1 / 46.2,
  // 65 68.7 / 63.3): its 800 threads an SM keep the walk from being scheduled beside it.
  if (n_items >= 24ll * tv::sm_count()) {
    TV_CUDA_OK(tv::stream_configure<row_stats_stream_kernel>());
    TV_CUDA_OK(tv::launch_pdl(row_stats_stream_kernel, dim3(tv::sm_count()), dim3(tv::kStreamThreads), tv::kStreamSmem, s, logits,
                              n_nodes, Nmax, V, n_chunks, row_items, (int)n_items, k, stats, status));
  } else {
    constexpr int kWarps = kStatThreads / 32;
    const int resident = 3 * tv::sm_count();
    const long long want = (n_slices + kWarps - 1) / kWarps;
    TV_CUDA_OK(tv::launch_pdl(row_stats_kernel, dim3((int)(want < resident ? want : resident)), dim3(kStatThreads), 0, s, logits,
                              n_nodes, Nmax, V, n_chunks, (int)n_slices, k, stats));
  }
  TV_CUDA_OK(tv::launch_pdl(sample_walk_kernel, dim3(B), dim3(kWalkThreads), 0, s, logits, stats, n_chunks, tokens, parent,
                            n_nodes, u_node, u_bonus, k, Nmax, V, Dp1, accept_len, accepted_nodes, next_token, status));
  tv::count_launches(2);
  return TV_OK;
}
