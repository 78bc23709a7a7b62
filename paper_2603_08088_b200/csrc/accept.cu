// tree_accept: teacher argmax over the vocabulary (an HBM-bound scan of the
// logits), the accelerator-safe path gather (Section 2.5 / 3.2) and greedy
// acceptance along root-to-leaf rows (Section 2.3).
//
// Phase 1 (argmax_stream_kernel, argmax_scan_kernel for few rows) streams logits[B,Nmax,V] once in items of 16384
// entries of one row and reduces each to a (value, index) pair in scratch.  Phase 2 (accept_kernel), one CTA per
// sequence, folds the item pairs in index order, then remaps, gathers and compares.
// Ties resolve to the lowest index at every level of the reduction.
#include "common.cuh"
#include "logits.cuh"

#include <cuda_bf16.h>

#include <mutex>

namespace {

constexpr int kScanThreads = 256;
constexpr int kChunkElems = tv::kStreamItem;                       // 16384 logits per item of either scan
static_assert(kChunkElems == kScanThreads * tv::kStreamVecs * 8, "a CTA of the short scan holds one item");

struct ArgPair {
  float val;
  int32_t idx;
};

__device__ __forceinline__ float bf16_bits_to_float(uint32_t bits16) {
  return __uint_as_float(bits16 << 16);
}

// (v, i) beats (bv, bi) when it is larger, or equal with a lower index.
__device__ __forceinline__ void take_better(float& bv, int& bi, float v, int i) {
  if (v > bv || (v == bv && i < bi)) {
    bv = v;
    bi = i;
  }
}

__device__ __forceinline__ float vec8_max(const uint4& u) {
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
  __nv_bfloat162 m = __hmax2(__hmax2(h[0], h[1]), __hmax2(h[2], h[3]));
  const float r = fmaxf(__low2float(m), __high2float(m));   // max of a NaN and x is x
  return r == r ? r : -INFINITY;                            // an all-NaN vector can never win
}

// Best entry among a thread's vectors, number first_vec + k stride of the row: lowest index of the largest value.
__device__ __forceinline__ void thread_best(const uint4* u, int first_vec, int stride, int off, int V, float& best, int& best_i) {
  best = -INFINITY;
  best_i = 0x7fffffff;
  int best_vec = 0;
#pragma unroll
  for (int k = 0; k < tv::kStreamVecs; ++k) {      // increasing index order: strict > keeps the first
    const float m = vec8_max(u[k]);
    if (m > best) {
      best = m;
      best_vec = k;
    }
  }
  uint4 w = u[0];
#pragma unroll
  for (int k = 1; k < tv::kStreamVecs; ++k) if (best_vec == k) w = u[k];
  const uint32_t e[4] = {w.x, w.y, w.z, w.w};
  const int first = 8 * (first_vec + best_vec * stride) - off;      // entry of the vector's first half-word
  best = -INFINITY;
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    float f = bf16_bits_to_float((t & 1) ? (e[t >> 1] >> 16) : (e[t >> 1] & 0xffffu));
    f = f == f ? f : -INFINITY;
    if (first >= 0 && first <= V - 8) take_better(best, best_i, f, first + t);
  }
}

// Both scans are persistent, and a row of any V is read in 16-byte vectors (V = 128257, 8 x 64 rows: 107 -> 28 us a call
// against 2-byte loads; V = 128256 took the same 28 us).
// `early` (tree_accept_behind_attn): the kernel in front is a tree_verify_attn launch, which lets this one be scheduled only
// when everything before it has completed, and it does not write what the scan reads.  The scan then runs beside it, on
// the SMs it leaves, and waits for it at the end: whoever waits for the scan has waited for the attention too.  A step of
// the ragged batch (8 x 64 nodes, V = 128256) 90.5 -> 86.4 us, of one sequence with 32 KV heads 27.5 -> 25.9
// (with the short scan).
//
// Short scans: the (row, vocabulary chunk) items are dealt round-robin to a grid of a few CTAs per SM, and a CTA requests
// the vectors of its next item before it reduces the ones it holds.
__global__ void __launch_bounds__(kScanThreads, 3)
argmax_scan_kernel(const tv_bf16* __restrict__ logits, const int32_t* __restrict__ n_nodes,
                   int Nmax, int V, int n_chunks, int n_items, int early, ArgPair* __restrict__ partial) {
  if (early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  else tv::pdl_enter();
  const int tid = threadIdx.x;
  __shared__ float sv[2][kScanThreads / 32];      // two sets, taken in turn: one barrier per item suffices
  __shared__ int si[2][kScanThreads / 32];
  int set = 0;

  // item -> (row, chunk, active); padded rows are never read
  auto locate = [&](int item, int& row, int& chunk) -> bool {
    if (item >= n_items) return false;
    row = item / n_chunks;
    chunk = item - row * n_chunks;
    const int b = row / Nmax;
    return row - b * Nmax < __ldcg(n_nodes + b);      // (not from an L1 line that an earlier launch on this SM has left)
  };
  auto fetch = [&](int row, int chunk, uint4* u) {
    const tv::LogitsRow r(logits, row, V);
    const int v0 = chunk * (kChunkElems / 8);
#pragma unroll
    for (int k = 0; k < tv::kStreamVecs; ++k) u[k] = r.vector(v0 + k * kScanThreads + tid);
  };

  int item = blockIdx.x;
  int row = 0, chunk = 0;
  bool active = locate(item, row, chunk);
  uint4 u[tv::kStreamVecs];
  if (active) fetch(row, chunk, u);
  while (item < n_items) {
    const int nitem = item + gridDim.x;
    int nrow = 0, nchunk = 0;
    const bool nactive = locate(nitem, nrow, nchunk);
    uint4 un[tv::kStreamVecs];
    if (nactive) fetch(nrow, nchunk, un);
    if (active) {
      const tv::LogitsRow r(logits, row, V);
      const int v0 = chunk * (kChunkElems / 8);
      float best;
      int best_i;
      thread_best(u, v0 + tid, kScanThreads, r.off, V, best, best_i);
      // the row's entries outside its whole vectors go with its first chunk
      if (chunk == 0 && tid < 16) {
        const int v = r.edge(tid);
        if (v >= 0) {
          float f = r.entry(v);
          f = f == f ? f : -INFINITY;
          take_better(best, best_i, f, v);
        }
      }
      // warp, then block reduction with the same rule
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, best, off);
        const int oi = __shfl_xor_sync(0xffffffffu, best_i, off);
        take_better(best, best_i, ov, oi);
      }
      if ((tid & 31) == 0) {
        sv[set][tid >> 5] = best;
        si[set][tid >> 5] = best_i;
      }
      __syncthreads();
      if (tid == 0) {
        for (int w = 1; w < kScanThreads / 32; ++w) take_better(best, best_i, sv[set][w], si[set][w]);
        ArgPair out;
        out.val = best;
        out.idx = best_i;
        partial[(size_t)row * n_chunks + chunk] = out;
      }
      set ^= 1;              // the next item writes the other set; this one is rewritten only after the next barrier
    }
    item = nitem;
    row = nrow;
    chunk = nchunk;
    active = nactive;
#pragma unroll
    for (int k = 0; k < tv::kStreamVecs; ++k) u[k] = un[k];
  }
  if (early) tv::pdl_wait_only();
}

// Long scans (see stream_rows).  The eight warps of an item leave their pairs as one 64-bit key - the value, then the
// complement of the index - in a maximum in shared memory; the last of them writes the item's pair.
__global__ void __launch_bounds__(tv::kStreamThreads, 1)
argmax_stream_kernel(const tv_bf16* __restrict__ logits, const int32_t* __restrict__ n_nodes,
                   int Nmax, int V, int n_chunks, int n_items, int early, ArgPair* __restrict__ partial,
                   int32_t* __restrict__ status) {
  if (early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  else tv::pdl_enter();
  const int lane = threadIdx.x & 31;
  __shared__ unsigned long long s_key[tv::kStreamStages];
  __shared__ unsigned s_count[tv::kStreamStages];
  if (threadIdx.x < tv::kStreamStages) {
    s_key[threadIdx.x] = 0;
    s_count[threadIdx.x] = 0;
  }                                        // (stream_rows starts with a barrier)
  tv::stream_rows<false>(logits, n_nodes, Nmax, V, n_chunks, n_items, status,
                         [&](int row, int chunk, int, int first_vec, const tv::LogitsRow& r, const uint4* u, float rest, int rest_v,
                             int stage) {
    float best;
    int best_i;
    thread_best(u, first_vec + lane, 32, r.off, V, best, best_i);
    // the row's entries outside its whole vectors go with its first slice
    if (rest_v >= 0) take_better(best, best_i, rest == rest ? rest : -INFINITY, rest_v);
    // the warp's best, then the item's: a float as an unsigned number in the same order (+ 0: one key for both zeros)
    const uint32_t bits = __float_as_uint(best + 0.f);
    const uint32_t key = bits & 0x80000000u ? ~bits : bits | 0x80000000u;
    const uint32_t top = __reduce_max_sync(0xffffffffu, key);
    const uint32_t low = __reduce_min_sync(0xffffffffu, key == top ? (uint32_t)best_i : 0x7fffffffu);
    if (lane == 0) {
      atomicMax(&s_key[stage], (unsigned long long)top << 32 | (uint32_t)~low);
      __threadfence_block();
      if (atomicAdd(&s_count[stage], 1u) == tv::kStreamWarps - 1) {
        __threadfence_block();
        const unsigned long long all = *reinterpret_cast<volatile unsigned long long*>(&s_key[stage]);
        const uint32_t t = (uint32_t)(all >> 32);
        ArgPair out;
        out.val = __uint_as_float(t & 0x80000000u ? t & 0x7fffffffu : ~t);
        out.idx = (int32_t)~(uint32_t)all;
        partial[(size_t)row * n_chunks + chunk] = out;
        s_key[stage] = 0;
        s_count[stage] = 0;
      }
    }
  });
  if (early) tv::pdl_wait_only();
}

// One CTA per sequence: a chain of look-ups on a few KB.  The tree's tokens and the candidate rows do not depend on the
// scan, so they are brought into shared memory (`staged`: they fit) while the scan still runs: the scan lets this kernel
// start only after every earlier kernel of the stream has completed, and the loads bypass L1.  Scan and this kernel, one
// sequence of 60 nodes, V = 32000: 5.8 -> 4.9 us.
constexpr int kAcceptThreads = 512;
constexpr int kLanesPerNode = 4;               // lanes that fold the chunk pairs of one node

__global__ void __launch_bounds__(kAcceptThreads)
accept_kernel(const ArgPair* __restrict__ partial, int n_chunks,
              const int32_t* __restrict__ tokens, const int32_t* __restrict__ retrieve,
              const int32_t* __restrict__ n_nodes,
              int Nmax, int P, int Dp1, int staged,
              int32_t* __restrict__ argmax_tok, int32_t* __restrict__ safe_idx,
              int32_t* __restrict__ candidates, int32_t* __restrict__ accept_len,
              int32_t* __restrict__ best_path, int32_t* __restrict__ accepted_nodes,
              int32_t* __restrict__ next_token, int32_t* __restrict__ status) {
  extern __shared__ int32_t am[];          // [Nmax] teacher argmax of this sequence, then (staged) tokens and rows
  __shared__ unsigned long long best_key;  // (accepted length << 32) | ~row : max = longest, then lowest row
  const int b = blockIdx.x;
  const int tid = threadIdx.x;
  int n = __ldcg(n_nodes + b);
  n = n < 0 ? 0 : (n > Nmax ? Nmax : n);
  const int32_t* rows = retrieve + (size_t)b * P * Dp1;
  const int32_t* tok_b = tokens + (size_t)b * Nmax;
  if (staged) {
    int32_t* s_tok = am + Nmax;
    int32_t* s_rows = s_tok + Nmax;
    for (int i = tid; i < Nmax; i += kAcceptThreads) s_tok[i] = __ldcg(tok_b + i);
#pragma unroll 8
    for (int i = tid; i < P * Dp1; i += kAcceptThreads) s_rows[i] = __ldcg(rows + i);
    rows = s_rows;
    tok_b = s_tok;
  }
  if (tid == 0) best_key = 0xffffffffull;  // length 0, row 0
  tv::pdl_enter();
  for (int i0 = 0; i0 < Nmax; i0 += kAcceptThreads / kLanesPerNode) {
    const int i = i0 + tid / kLanesPerNode;
    float bv = -INFINITY;
    int bi = 0x7fffffff;
    if (i < n) {
      const ArgPair* pp = partial + ((size_t)b * Nmax + i) * n_chunks;
#pragma unroll 4
      for (int c = tid % kLanesPerNode; c < n_chunks; c += kLanesPerNode) take_better(bv, bi, pp[c].val, pp[c].idx);
    }
#pragma unroll
    for (int off = kLanesPerNode / 2; off > 0; off >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, bv, off);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
      take_better(bv, bi, ov, oi);
    }
    if (i < Nmax && tid % kLanesPerNode == 0) {
      const int tok = i < n ? bi : -1;
      am[i] = tok;
      argmax_tok[(size_t)b * Nmax + i] = tok;
    }
  }
  __syncthreads();

  bool bad_index = false;
  for (int p0 = 0; p0 < P; p0 += kAcceptThreads) {
    const int p = p0 + tid;
    int a = -1;
    if (p < P) {
      a = 0;
      bool chain = true;
      bool prev_ok = false;
      int prev_safe = 0;
      for (int j = 0; j < Dp1; ++j) {
        const int r = rows[p * Dp1 + j];
        const bool ok = r >= 0 && r < n;
        bad_index |= r < -1 || r >= n;
        const int s = ok ? r : 0;            // remap BEFORE the gather: s is always in [0, Nmax)
        const int cand = tok_b[s];
        if (safe_idx) safe_idx[((size_t)b * P + p) * Dp1 + j] = s;
        if (candidates) candidates[((size_t)b * P + p) * Dp1 + j] = cand;
        if (j > 0 && chain) {
          if (ok && prev_ok && cand == am[prev_safe]) a = j;
          else chain = false;
        }
        prev_ok = ok;
        prev_safe = s;
      }
    }
    // longest first, then the lowest row: one atomic per warp
    const int wa = __reduce_max_sync(0xffffffffu, a);
    const unsigned wp = __reduce_min_sync(0xffffffffu, a == wa ? (unsigned)p : 0xffffffffu);
    if ((tid & 31) == 0 && wa >= 0)
      atomicMax(&best_key, ((unsigned long long)wa << 32) | (unsigned long long)(0xffffffffu - wp));
  }
  const bool any_bad = __syncthreads_or(bad_index);
  const int A = (int)(best_key >> 32);
  const int pstar = (int)(0xffffffffu - (unsigned)(best_key & 0xffffffffull));
  for (int j = tid; j < Dp1; j += kAcceptThreads) {
    int node = 0;
    if (j <= A && P > 0) {
      const int r = rows[pstar * Dp1 + j];
      node = (r >= 0 && r < n) ? r : 0;
    }
    accepted_nodes[(size_t)b * Dp1 + j] = node;
    if (j == A) next_token[b] = am[node];
  }
  if (tid == 0) {
    accept_len[b] = A;
    best_path[b] = pstar;
    if (any_bad) atomicOr(&status[b], TV_ST_BAD_INDEX);
  }
}

// One thread per (sequence, node): score of the node's proposed token in the logits of its parent's slot.
__global__ void node_scores_kernel(const tv_bf16* __restrict__ logits, const int32_t* __restrict__ tokens,
                                   const int32_t* __restrict__ parent, const int32_t* __restrict__ n_nodes,
                                   int B, int Nmax, int V, float* __restrict__ scores, int32_t* __restrict__ status) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= B * Nmax) return;
  const int b = idx / Nmax, k = idx - b * Nmax;
  int n = n_nodes[b];
  n = n < 0 ? 0 : (n > Nmax ? Nmax : n);
  float val = 0.f;
  if (k >= 1 && k < n) {
    const int p = parent[idx];
    const int sp = (p >= 0 && p < n) ? p : 0;          // dummy-root remap before the gather
    const int t = tokens[idx];
    const bool ok = t >= 0 && t < V;
    const int st = ok ? t : 0;                          // in-range vocabulary index
    const float g = bf16_bits_to_float(logits[((size_t)b * Nmax + sp) * V + st]);
    val = ok ? g : -INFINITY;
    if (!ok) atomicOr(&status[b], TV_ST_BAD_INDEX);
  }
  scores[idx] = val;
}

// CTAs of the short scan: three per SM (what its registers allow).
int scan_ctas() { return 3 * tv::sm_count(); }

int scan_chunks(int V) { return (V + kChunkElems - 1) / kChunkElems; }

// Scratch of tree_accept_noalloc: a fixed device array that lives in the library image, so that callers
// who may not allocate device memory can still run the accept step.  Every GPU that loads the library
// holds these 256 KiB until the process exits.
constexpr size_t kStaticPairs = 32768;                       // (row, vocabulary chunk) pairs
static __device__ __align__(256) unsigned char g_accept_scratch[kStaticPairs * sizeof(ArgPair)];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mutex;
void* g_scratch_ptr[kMaxDevices] = {nullptr};

// Device address of g_accept_scratch on the current device.  In host code the symbol's name is only a
// stand-in, not an address a kernel can use; the runtime hands out the real one, once per device.
int static_scratch(void** out) {
  int dev = -1;
  TV_CUDA_OK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices)
    return tv::fail(TV_ERR_INVALID_ARG, "tree_accept_noalloc: device ordinal %d is not supported", dev);
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    TV_CUDA_OK(cudaGetSymbolAddress(&p, g_accept_scratch));
    g_scratch_ptr[dev] = p;
  }
  *out = g_scratch_ptr[dev];
  return TV_OK;
}

int accept_entry(const tv_bf16* logits, const int32_t* tokens, const int32_t* retrieve_indices, const int32_t* n_nodes,
                 int B, int Nmax, int V, int P, int Dp1, int32_t* argmax_tok, int32_t* safe_idx, int32_t* candidates,
                 int32_t* accept_len, int32_t* best_path, int32_t* accepted_nodes, int32_t* next_token,
                 void* workspace, size_t workspace_bytes, int32_t* status, bool behind_attn, tv_stream stream) {
  TV_REQUIRE(logits && tokens && n_nodes && argmax_tok && accept_len && best_path && accepted_nodes &&
                 next_token && status && workspace,
             "tree_accept: NULL required pointer");
  TV_REQUIRE(B >= 0 && Nmax >= 1 && Nmax <= 8192 && V >= 1 && P >= 0 && Dp1 >= 1,
             "tree_accept: need B >= 0, 1 <= Nmax <= 8192, V >= 1, P >= 0, Dp1 >= 1");
  TV_REQUIRE(P == 0 || retrieve_indices, "tree_accept: retrieve_indices is NULL with P > 0");
  TV_REQUIRE(B * (long long)Nmax <= 65535, "tree_accept: B*Nmax exceeds 65535 rows");
  TV_REQUIRE((reinterpret_cast<uintptr_t>(workspace) & 7u) == 0, "tree_accept: workspace must be 8-byte aligned");
  if (workspace_bytes < tv_accept_workspace_bytes(B, Nmax, V))
    return tv::fail(TV_ERR_WORKSPACE, "tree_accept: workspace of %zu bytes, need %zu", workspace_bytes,
                    tv_accept_workspace_bytes(B, Nmax, V));
  if (B == 0) return TV_OK;
  const int n_chunks = scan_chunks(V);
  ArgPair* partial = static_cast<ArgPair*>(workspace);
  cudaStream_t s = (cudaStream_t)stream;
  const long long n_items = (long long)B * Nmax * n_chunks;
  TV_REQUIRE(n_items < (1ll << 31), "tree_accept: B * Nmax * ceil(V / 16384) must stay below 2^31");
  // The long scan from six items an SM on (us a call, short / long: 4.9 items an SM 9.0 / 8.8, 6.5 10.0 / 10.0, 10.8 13.5 /
  // 12.3, 21.6 22.4 / 19.2, 43 38.8 / 32.1; below, its rings take longer to set up: 1.6 items 6.0 / 7.0).
  if (n_items >= 6ll * tv::sm_count()) {
    TV_CUDA_OK(tv::stream_configure<argmax_stream_kernel>());
    TV_CUDA_OK(tv::launch_pdl(argmax_stream_kernel, dim3(tv::sm_count()), dim3(tv::kStreamThreads), tv::kStreamSmem, s, logits,
                              n_nodes, Nmax, V, n_chunks, (int)n_items, behind_attn ? 1 : 0, partial, status));
  } else {
    const int scan_grid = (int)(n_items < (long long)scan_ctas() ? n_items : scan_ctas());
    TV_CUDA_OK(tv::launch_pdl(argmax_scan_kernel, dim3(scan_grid), dim3(kScanThreads), 0, s, logits, n_nodes, Nmax, V,
                              n_chunks, (int)n_items, behind_attn ? 1 : 0, partial));
  }
  const long long staged_ints = 2ll * Nmax + (long long)P * Dp1;
  const int staged = staged_ints * 4 <= 47 * 1024 ? 1 : 0;        // what a CTA may have without asking for more
  const size_t smem = (staged ? (size_t)staged_ints : (size_t)Nmax) * sizeof(int32_t);
  TV_CUDA_OK(tv::launch_pdl(accept_kernel, dim3(B), dim3(kAcceptThreads), smem, s, partial, n_chunks, tokens, retrieve_indices,
                            n_nodes, Nmax, P, Dp1, staged, argmax_tok, safe_idx, candidates, accept_len, best_path,
                            accepted_nodes, next_token, status));
  tv::count_launches(2);
  return TV_OK;
}

}  // namespace

extern "C" size_t tv_accept_workspace_bytes(int B, int Nmax, int V) {
  if (B <= 0 || Nmax <= 0 || V <= 0) return 16;
  return (size_t)B * Nmax * scan_chunks(V) * sizeof(ArgPair);
}

extern "C" int tree_accept(const tv_bf16* logits, const int32_t* tokens,
                           const int32_t* retrieve_indices, const int32_t* n_nodes,
                           int B, int Nmax, int V, int P, int Dp1,
                           int32_t* argmax_tok, int32_t* safe_idx, int32_t* candidates,
                           int32_t* accept_len, int32_t* best_path, int32_t* accepted_nodes,
                           int32_t* next_token,
                           void* workspace, size_t workspace_bytes,
                           int32_t* status, tv_stream stream) {
  return accept_entry(logits, tokens, retrieve_indices, n_nodes, B, Nmax, V, P, Dp1, argmax_tok, safe_idx, candidates, accept_len,
                      best_path, accepted_nodes, next_token, workspace, workspace_bytes, status, false, stream);
}

extern "C" int tree_accept_behind_attn(const tv_bf16* logits, const int32_t* tokens,
                                       const int32_t* retrieve_indices, const int32_t* n_nodes,
                                       int B, int Nmax, int V, int P, int Dp1,
                                       int32_t* argmax_tok, int32_t* safe_idx, int32_t* candidates,
                                       int32_t* accept_len, int32_t* best_path, int32_t* accepted_nodes,
                                       int32_t* next_token,
                                       void* workspace, size_t workspace_bytes,
                                       int32_t* status, tv_stream stream) {
  return accept_entry(logits, tokens, retrieve_indices, n_nodes, B, Nmax, V, P, Dp1, argmax_tok, safe_idx, candidates, accept_len,
                      best_path, accepted_nodes, next_token, workspace, workspace_bytes, status, true, stream);
}

extern "C" size_t tv_accept_noalloc_max_bytes(void) { return kStaticPairs * sizeof(ArgPair); }

extern "C" int tree_accept_noalloc(const tv_bf16* logits, const int32_t* tokens,
                                   const int32_t* retrieve_indices, const int32_t* n_nodes,
                                   int B, int Nmax, int V, int P, int Dp1,
                                   int32_t* argmax_tok, int32_t* safe_idx, int32_t* candidates,
                                   int32_t* accept_len, int32_t* best_path, int32_t* accepted_nodes,
                                   int32_t* next_token, int32_t* status, tv_stream stream) {
  TV_REQUIRE(B >= 0 && Nmax >= 1 && V >= 1, "tree_accept_noalloc: need B >= 0, Nmax >= 1, V >= 1");
  const size_t need = tv_accept_workspace_bytes(B, Nmax, V);
  if (need > kStaticPairs * sizeof(ArgPair))
    return tv::fail(TV_ERR_WORKSPACE,
                    "tree_accept_noalloc: B*Nmax*ceil(V/%d) = %zu scratch entries, the built-in scratch holds %zu; "
                    "use tree_accept with a caller workspace",
                    kChunkElems, need / sizeof(ArgPair), kStaticPairs);
  void* scratch = nullptr;
  const int rc = static_scratch(&scratch);
  if (rc != TV_OK) return rc;
  return tree_accept(logits, tokens, retrieve_indices, n_nodes, B, Nmax, V, P, Dp1, argmax_tok, safe_idx, candidates,
                     accept_len, best_path, accepted_nodes, next_token, scratch, kStaticPairs * sizeof(ArgPair),
                     status, stream);
}

extern "C" int tree_node_scores(const tv_bf16* logits, const int32_t* tokens, const int32_t* parent,
                                const int32_t* n_nodes, int B, int Nmax, int V, float* scores,
                                int32_t* status, tv_stream stream) {
  TV_REQUIRE(logits && tokens && parent && n_nodes && scores && status, "tree_node_scores: NULL pointer");
  TV_REQUIRE(B >= 0 && Nmax >= 1 && V >= 1, "tree_node_scores: need B >= 0, Nmax >= 1, V >= 1");
  if (B == 0) return TV_OK;
  const int total = B * Nmax;
  node_scores_kernel<<<(total + 127) / 128, 128, 0, (cudaStream_t)stream>>>(logits, tokens, parent, n_nodes, B, Nmax, V,
                                                                             scores, status);
  TV_CUDA_OK(cudaGetLastError());
  tv::count_launches(1);
  return TV_OK;
}
