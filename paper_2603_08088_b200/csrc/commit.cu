// kv_commit, kv_commit_inplace, kv_commit_paged: path-index commit (Section 3.1).  The committed prefix is never
// moved; the accepted nodes' K/V rows are gathered behind it, for every layer and KV head, and prefix_len advances.
//
// One warp moves up to 128 pieces of 16 bytes of a (layer, K or V, node) row over all heads, four a lane (a head row of d bf16 is d/8 adjacent
// lanes, coalesced on both sides); a sequence has as many CTAs as its rows keep busy.  Every CTA reads the sequence's scalars and its node list
// and decides alike whether the sequence commits.  Where one CTA per sequence is enough (see launch_commit) it also
// advances prefix_len; otherwise a second launch does, so that no copying CTA can observe the updated length.
// (One launch with a thread-block cluster per sequence instead was 1.9 times slower on 16 sequences of 32 layers: 6.2
// -> 11.9 us; clusters start late when many of them are needed.)  Before / now, us a call: one layer of 32 heads, seven
// rows 10.6 / 3.7; one sequence of 32 layers 5.1 / 4.2; in-cache, 16 sequences of 32 layers 8.7 / 7.1; paged, 8 of 8
// layers 5.6 / 5.0; 16 sequences of 32 layers 6.3 / 6.7.
#include "common.cuh"

namespace {

constexpr int kThreads = 256;                 // of a CTA when a sequence has several
constexpr int kMaxThreads = 512;              // ... when it has one
constexpr int kPerLane = 4;                   // 16-byte pieces of a row in flight per lane
constexpr int kHeld = 4;                      // in-cache layout: pieces a thread holds
constexpr int kMaxDp1 = 2048;                 // longest path of the in-cache layout (the others: 1024)
constexpr int kPageRows = 128;
constexpr int kMaxPages = 1024 / kPageRows + 1;      // pages under a segment of at most 1024 rows
constexpr int kMaxCtas = 4096;                // CTAs of a launch beyond which more of them cannot help

struct Commit {
  uint4* k_cache;
  uint4* v_cache;
  const uint4* k_tree;                        // unused in the in-cache layout
  const uint4* v_tree;
  const int32_t* block_table;                 // paged layout only
  const int32_t* accepted_nodes;
  const int32_t* accept_len;
  int32_t* prefix_len;
  int32_t* status;
  int L, Nmax, Hkv, dvec, Scap, Dp1, n_pages, max_blocks;
  int64_t cache_layer, tree_layer;            // 16-byte pieces between two layers
};

enum Layout { kContiguous, kInCache, kPaged };

// COPY: move the accepted rows.  FINISH: advance prefix_len, raise status bits.
template <Layout LAYOUT, bool COPY, bool FINISH>
__global__ void __launch_bounds__(kMaxThreads)
commit_kernel(const Commit c, int ctas_per_seq) {
  // A kernel that writes prefix_len, which a tree_verify_attn launch directly behind it may read before its own wait,
  // releases nothing early: the next launch must not start until this grid is complete.
  if (FINISH) tv::pdl_wait_only();
  else tv::pdl_enter();
  __shared__ int s_nodes[LAYOUT == kInCache ? kMaxDp1 : 1024];
  __shared__ int s_pages[LAYOUT == kPaged ? kMaxPages : 1];
  const unsigned ranks = ctas_per_seq, rank = blockIdx.x % ranks;
  const int b = blockIdx.x / ranks, tid = threadIdx.x, nt = blockDim.x;
  const int A = c.accept_len[b];
  const int S = c.prefix_len[b];
  const int st = c.status[b];
  for (int j = tid; j < c.Dp1; j += nt) s_nodes[j] = c.accepted_nodes[(size_t)b * c.Dp1 + j];
  const int cap = LAYOUT == kPaged ? c.max_blocks * kPageRows : c.Scap;
  const bool skip = (st & tv::kFatalStatus) != 0;               // nothing new to report
  const bool len_ok = A >= 0 && A < c.Dp1;
  const bool fits = len_ok && S >= 0 && S <= cap - (A + 1);
  __syncthreads();
  bool bad_node = false, bad_source = false, bad_page = false;
  if (len_ok)
    for (int j = tid; j <= A; j += nt) {
      const int node = s_nodes[j];
      bad_node |= node < 0 || node >= c.Nmax;
      if (LAYOUT == kInCache) bad_source |= S + (long long)node >= c.Scap;      // a source row outside the cache
    }
  if (LAYOUT == kPaged && fits)
    for (int t = tid; t <= (S + A) / kPageRows - S / kPageRows; t += nt) {
      const int pg = c.block_table[(size_t)b * c.max_blocks + S / kPageRows + t];
      bad_page |= pg < 0 || pg >= c.n_pages;
      s_pages[t] = pg;
    }
  int report = 0;                                               // status bits to raise; 0: commit
  if (!len_ok || __syncthreads_or(bad_node)) report = TV_ST_BAD_INDEX;
  else if (!fits || (LAYOUT == kInCache && __syncthreads_or(bad_source))) report = TV_ST_CAPACITY;
  else if (LAYOUT == kPaged && __syncthreads_or(bad_page)) report = TV_ST_BAD_INDEX;
  if (FINISH && tid == 0 && !skip) {                            // (every thread has read the scalars before a barrier)
    if (report == 0) c.prefix_len[b] = S + A + 1;
    else c.status[b] = st | report;
  }
  if (!COPY || skip || report != 0) return;
  const int dvec = c.dvec;
  if (LAYOUT == kInCache) {
    // Row S + j takes the OLD row S + accepted_nodes[j]: source and destination ranges overlap (a row can be the
    // source of one slot and the destination of another), so a CTA owns all rows of a (layer, K or V, head) slab,
    // holds every piece it needs in registers and writes only behind a barrier.
    const int per_head = (A + 1) * dvec;                        // <= kHeld * nt (launch_commit)
    const int hpc = kHeld * nt / per_head;           // slabs a CTA holds at once
    const long long slabs = 2ll * c.L * c.Hkv;
    for (long long s0 = (long long)rank * hpc; s0 < slabs; s0 += (long long)ranks * hpc) {
      uint4 held[kHeld];
      uint4* dst[kHeld];
#pragma unroll
      for (int i = 0; i < kHeld; ++i) {
        const int t = tid + i * nt;
        const int h = t / per_head, u = t - h * per_head;
        const int j = u / dvec, w = u - j * dvec;
        const long long slab = s0 + h;
        dst[i] = nullptr;
        if (h < hpc && slab < slabs) {
          const int l = (int)(slab / (2 * c.Hkv)), r = (int)(slab - (long long)l * 2 * c.Hkv);
          const int kv = r >= c.Hkv, head = kv ? r - c.Hkv : r;
          uint4* base = (kv ? c.v_cache : c.k_cache) + (size_t)l * c.cache_layer +
                        (((size_t)b * c.Hkv + head) * c.Scap + S) * (size_t)dvec;
          held[i] = base[(size_t)s_nodes[j] * dvec + w];
          if (s_nodes[j] != j) dst[i] = base + (size_t)j * dvec + w;
        }
      }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < kHeld; ++i)
        if (dst[i]) *dst[i] = held[i];
    }
  } else {
    const int per = c.Hkv * dvec;                               // pieces of one node's row over all heads
    const int warps = nt >> 5, lane = tid & 31;
    const int rounds = (per + 32 * kPerLane - 1) / (32 * kPerLane);
    const long long units = 2ll * c.L * (A + 1) * rounds;
    for (long long r = (long long)rank * warps + (tid >> 5); r < units; r += (long long)ranks * warps) {
      const int in_layer = 2 * (A + 1) * rounds;
      const int l = (int)(r / in_layer), in = (int)(r - (long long)l * in_layer);
      const int u = in / rounds, w0 = (in - u * rounds) * 32 * kPerLane + lane;
      const bool kv = u > A;
      const int j = kv ? u - (A + 1) : u, row = S + j;
      const uint4* src = (kv ? c.v_tree : c.k_tree) + (size_t)l * c.tree_layer + ((size_t)b * c.Nmax + s_nodes[j]) * per;
      const size_t at = LAYOUT == kPaged ? (size_t)s_pages[row / kPageRows - S / kPageRows] * c.Hkv * kPageRows + row % kPageRows
                                         : (size_t)b * c.Hkv * c.Scap + row;      // row of head 0
      const size_t head_rows = LAYOUT == kPaged ? kPageRows : c.Scap;
      uint4* dst = (kv ? c.v_cache : c.k_cache) + (size_t)l * c.cache_layer + at * dvec;
      uint4 val[kPerLane];
#pragma unroll
      for (int i = 0; i < kPerLane; ++i)
        if (w0 + 32 * i < per) val[i] = src[w0 + 32 * i];
#pragma unroll
      for (int i = 0; i < kPerLane; ++i) {
        const int w = w0 + 32 * i;
        if (w < per) {
          const int h = w / dvec;
          dst[(size_t)h * head_rows * dvec + (w - h * dvec)] = val[i];
        }
      }
    }
  }
}

// CTAs per sequence: what the longest path of the call keeps busy for one round.  One larger CTA and one launch where
// the call is small (one layer, eight heads of 128, paths of eight: 4.1 -> 2.8 us), two launches where it is not.
template <Layout LAYOUT>
cudaError_t launch_commit(const Commit& c, int B, cudaStream_t s) {
  const long long pieces = 2ll * c.L * c.Hkv * c.dvec * c.Dp1;
  if (pieces <= kMaxThreads * kPerLane || kMaxCtas / B <= 1) {
    tv::count_launches(1);
    return tv::launch_pdl(commit_kernel<LAYOUT, true, true>, dim3(B), dim3(kMaxThreads), 0, s, c, 1);
  }
  int threads = kThreads;
  long long ctas;
  if (LAYOUT == kInCache) {
    if (c.Dp1 * c.dvec > kHeld * kThreads) threads = kMaxThreads;       // one head's longest segment has to fit a CTA
    ctas = (pieces * 5 / 8 + threads * kHeld - 1) / (threads * kHeld);  // most paths are shorter than the longest
  } else {
    const int rounds = (c.Hkv * c.dvec + 32 * kPerLane - 1) / (32 * kPerLane), warps = kThreads / 32;
    ctas = (2ll * c.L * c.Dp1 * rounds + warps - 1) / warps;
    if (ctas * B > 8ll * tv::sm_count()) ctas = (ctas * 5 + 7) / 8;     // more than one wave: most paths are shorter
  }
  if (ctas > kMaxCtas / B) ctas = kMaxCtas / B;
  tv::count_launches(2);
  const cudaError_t e = tv::launch_pdl(commit_kernel<LAYOUT, true, false>, dim3((unsigned)ctas * B), dim3(threads), 0, s, c,
                                       (int)ctas);
  if (e != cudaSuccess) return e;
  return tv::launch_pdl(commit_kernel<LAYOUT, false, true>, dim3(B), dim3(kThreads), 0, s, c, 1);
}

}  // namespace

extern "C" int kv_commit_paged(tv_bf16* k_pages, tv_bf16* v_pages, const int32_t* block_table,
                               const tv_bf16* k_tree, const tv_bf16* v_tree,
                               const int32_t* accepted_nodes, const int32_t* accept_len,
                               int32_t* prefix_len,
                               int L, int B, int Nmax, int Hkv, int d, int n_pages, int max_blocks, int Dp1,
                               int64_t page_layer_stride, int64_t tree_layer_stride,
                               int32_t* status, tv_stream stream) {
  TV_REQUIRE(k_pages && v_pages && block_table && k_tree && v_tree && accepted_nodes && accept_len && prefix_len && status,
             "kv_commit_paged: NULL pointer");
  TV_REQUIRE(L >= 0 && B >= 0 && Nmax >= 1 && Hkv >= 1 && d >= 8 && n_pages >= 1 && max_blocks >= 1 && Dp1 >= 1,
             "kv_commit_paged: bad dimension");
  TV_REQUIRE(max_blocks <= (1 << 20), "kv_commit_paged: max_blocks must be <= 2^20");
  TV_REQUIRE(d % 8 == 0, "kv_commit_paged: d must be a multiple of 8 (16-byte rows)");
  TV_REQUIRE(page_layer_stride % 8 == 0 && tree_layer_stride % 8 == 0, "kv_commit_paged: layer strides must be multiples of 8 elements");
  TV_REQUIRE(tv::aligned16(k_pages) && tv::aligned16(v_pages) && tv::aligned16(k_tree) && tv::aligned16(v_tree),
             "kv_commit_paged: tensors must be 16-byte aligned");
  TV_REQUIRE(L <= 65535 && Dp1 <= 1024, "kv_commit_paged: L must be <= 65535 and Dp1 <= 1024");
  if (L == 0 || B == 0) return TV_OK;
  Commit c{};
  c.k_cache = reinterpret_cast<uint4*>(k_pages);
  c.v_cache = reinterpret_cast<uint4*>(v_pages);
  c.k_tree = reinterpret_cast<const uint4*>(k_tree);
  c.v_tree = reinterpret_cast<const uint4*>(v_tree);
  c.block_table = block_table;
  c.accepted_nodes = accepted_nodes;
  c.accept_len = accept_len;
  c.prefix_len = prefix_len;
  c.status = status;
  c.L = L; c.Nmax = Nmax; c.Hkv = Hkv; c.dvec = d / 8; c.Dp1 = Dp1; c.n_pages = n_pages; c.max_blocks = max_blocks;
  c.cache_layer = page_layer_stride / 8;
  c.tree_layer = tree_layer_stride / 8;
  TV_CUDA_OK(launch_commit<kPaged>(c, B, (cudaStream_t)stream));
  return TV_OK;
}

extern "C" int kv_commit_inplace(tv_bf16* k_cache, tv_bf16* v_cache,
                                 const int32_t* accepted_nodes, const int32_t* accept_len,
                                 int32_t* prefix_len,
                                 int L, int B, int Nmax, int Hkv, int d, int Scap, int Dp1,
                                 int64_t cache_layer_stride,
                                 int32_t* status, tv_stream stream) {
  TV_REQUIRE(k_cache && v_cache && accepted_nodes && accept_len && prefix_len && status, "kv_commit_inplace: NULL pointer");
  TV_REQUIRE(L >= 0 && B >= 0 && Nmax >= 1 && Hkv >= 1 && d >= 8 && Scap >= 1 && Dp1 >= 1,
             "kv_commit_inplace: bad dimension");
  TV_REQUIRE(d % 8 == 0, "kv_commit_inplace: d must be a multiple of 8 (16-byte rows)");
  TV_REQUIRE(cache_layer_stride % 8 == 0, "kv_commit_inplace: the layer stride must be a multiple of 8 elements");
  TV_REQUIRE(tv::aligned16(k_cache) && tv::aligned16(v_cache), "kv_commit_inplace: tensors must be 16-byte aligned");
  TV_REQUIRE(B <= 65535 && L <= 65535 && Hkv <= 32767, "kv_commit_inplace: B and L must be <= 65535, Hkv <= 32767");
  TV_REQUIRE((long long)Dp1 * (d / 8) <= kMaxDp1,
             "kv_commit_inplace: Dp1 * d / 8 must be <= 2048 (the accepted segment of a head is staged in registers)");
  if (L == 0 || B == 0) return TV_OK;
  Commit c{};
  c.k_cache = reinterpret_cast<uint4*>(k_cache);
  c.v_cache = reinterpret_cast<uint4*>(v_cache);
  c.accepted_nodes = accepted_nodes;
  c.accept_len = accept_len;
  c.prefix_len = prefix_len;
  c.status = status;
  c.L = L; c.Nmax = Nmax; c.Hkv = Hkv; c.dvec = d / 8; c.Scap = Scap; c.Dp1 = Dp1;
  c.cache_layer = cache_layer_stride / 8;
  TV_CUDA_OK(launch_commit<kInCache>(c, B, (cudaStream_t)stream));
  return TV_OK;
}

extern "C" int kv_commit(tv_bf16* k_cache, tv_bf16* v_cache,
                         const tv_bf16* k_tree, const tv_bf16* v_tree,
                         const int32_t* accepted_nodes, const int32_t* accept_len,
                         int32_t* prefix_len,
                         int L, int B, int Nmax, int Hkv, int d, int Scap, int Dp1,
                         int64_t cache_layer_stride, int64_t tree_layer_stride,
                         int32_t* status, tv_stream stream) {
  TV_REQUIRE(k_cache && v_cache && k_tree && v_tree && accepted_nodes && accept_len && prefix_len && status,
             "kv_commit: NULL pointer");
  TV_REQUIRE(L >= 0 && B >= 0 && Nmax >= 1 && Hkv >= 1 && d >= 8 && Scap >= 1 && Dp1 >= 1,
             "kv_commit: bad dimension");
  TV_REQUIRE(d % 8 == 0, "kv_commit: d must be a multiple of 8 (16-byte rows)");
  TV_REQUIRE(cache_layer_stride % 8 == 0 && tree_layer_stride % 8 == 0, "kv_commit: layer strides must be multiples of 8 elements");
  TV_REQUIRE(tv::aligned16(k_cache) && tv::aligned16(v_cache) && tv::aligned16(k_tree) && tv::aligned16(v_tree),
             "kv_commit: tensors must be 16-byte aligned");
  TV_REQUIRE(L <= 65535, "kv_commit: L must be <= 65535");
  TV_REQUIRE(Dp1 <= 1024, "kv_commit: Dp1 must be <= 1024");
  if (L == 0 || B == 0) return TV_OK;
  Commit c{};
  c.k_cache = reinterpret_cast<uint4*>(k_cache);
  c.v_cache = reinterpret_cast<uint4*>(v_cache);
  c.k_tree = reinterpret_cast<const uint4*>(k_tree);
  c.v_tree = reinterpret_cast<const uint4*>(v_tree);
  c.accepted_nodes = accepted_nodes;
  c.accept_len = accept_len;
  c.prefix_len = prefix_len;
  c.status = status;
  c.L = L; c.Nmax = Nmax; c.Hkv = Hkv; c.dvec = d / 8; c.Scap = Scap; c.Dp1 = Dp1;
  c.cache_layer = cache_layer_stride / 8;
  c.tree_layer = tree_layer_stride / 8;
  TV_CUDA_OK(launch_commit<kContiguous>(c, B, (cudaStream_t)stream));
  return TV_OK;
}
