// tv_verify_step_host: one verification step driven from host buffers.
// Copies the per-step inputs into a caller-provided device staging area,
// enqueues the four calls of the step in the paper's order (tensorise + mask,
// attention per layer, gather + accept, commit; Section 3), copies the
// per-step results back and waits for the stream.  The KV cache and
// prefix_len are resident device state and are not copied.
//
// The step is bound by the host link (hundreds of MB each way), so the copies
// are pipelined against the kernels: an input stream feeds Q and the tree K/V
// stage by stage and the logits last, the caller's stream runs the layers of a
// stage in one launch as soon as their inputs have landed, and an output stream
// returns their results as soon as they are complete, while later ones are still
// coming in (the link is full duplex).  A stage is as many layers as it takes to
// move kStageBytes: with one layer a stage throughout, a small model's step was
// bound by some ninety driver calls of 2 us each (8 layers of 0.2 MB: 331 us, now 196).
#include "common.cuh"

#include <cstring>
#include <mutex>
#include <vector>

namespace {

struct Staging {
  size_t parent, n_nodes, tokens, retrieve, q, k_tree, v_tree, logits, out, anc_bits, status, argmax,
      accept_len, best_path, accepted, next_token, n_paths, attn_ws, accept_ws, total;
  size_t attn_ws_bytes, accept_ws_bytes;
};

// Inputs of a stage: 2 MB are 36 us on the link, several times what the calls of a stage cost the host.
constexpr size_t kStageBytes = size_t(2) << 20;

size_t up256(size_t x) { return (x + 255) & ~size_t(255); }

Staging layout(int L, int B, int Nmax, int Hq, int Hkv, int d, int Scap, int V, int P, int Dp1) {
  Staging s{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    size_t at = off;
    off += up256(bytes ? bytes : 1);
    return at;
  };
  const size_t W = (Nmax + 31) / 32;
  s.parent = take(sizeof(int32_t) * B * Nmax);
  s.n_nodes = take(sizeof(int32_t) * B);
  s.tokens = take(sizeof(int32_t) * B * Nmax);
  s.retrieve = take(sizeof(int32_t) * B * P * Dp1);
  s.q = take(sizeof(tv_bf16) * (size_t)L * B * Nmax * Hq * d);
  s.k_tree = take(sizeof(tv_bf16) * (size_t)L * B * Nmax * Hkv * d);
  s.v_tree = take(sizeof(tv_bf16) * (size_t)L * B * Nmax * Hkv * d);
  s.logits = take(sizeof(tv_bf16) * (size_t)B * Nmax * V);
  s.out = take(sizeof(tv_bf16) * (size_t)L * B * Nmax * Hq * d);
  s.anc_bits = take(sizeof(uint32_t) * B * Nmax * W);
  s.argmax = take(sizeof(int32_t) * B * Nmax);
  s.best_path = take(sizeof(int32_t) * B);
  s.accept_len = take(sizeof(int32_t) * B);       // the small results lie together, like the small inputs above
  s.accepted = take(sizeof(int32_t) * B * Dp1);
  s.next_token = take(sizeof(int32_t) * B);
  s.status = take(sizeof(int32_t) * B);
  s.n_paths = take(sizeof(int32_t) * B);
  s.attn_ws_bytes = tv_attn_workspace_bytes(B, Nmax, Hq, Hkv, d, Scap);
  s.attn_ws = take(s.attn_ws_bytes);
  s.accept_ws_bytes = tv_accept_workspace_bytes(B, Nmax, V);
  s.accept_ws = take(s.accept_ws_bytes);
  s.total = off;
  return s;
}

// The small arrays of a step cross the link together: a copy of its own costs each of them some 6 us in front of the step
// or behind it (8 + 20 us of a small model's step).  The results come back in one copy to a pinned block.  The inputs may
// still be written by work that is queued on the caller's stream (a drafter's copies to the host, say), so the host must
// not read them when the call is made: a kernel on that stream reads them where they are, if they are pinned.
constexpr size_t kBlockBytes = 64 << 10;

struct SmallInputs {
  const int32_t* src[4];
  int32_t* dst[4];
  int count[4];
};

constexpr int kFetchThreads = 256;

// Bound by one round trip over the host link: every thread has one load in flight, 64 KB take 64 CTAs.
__global__ void __launch_bounds__(kFetchThreads)
fetch_small_kernel(const SmallInputs a) {
  tv::pdl_enter();
  int i = blockIdx.x * kFetchThreads + threadIdx.x;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (i >= 0 && i < a.count[k]) a.dst[k][i] = __ldcv(a.src[k] + i);
    i -= a.count[k];
  }
}

// Address under which kernels of this device read `bytes` of pinned host memory, or nullptr.
const int32_t* mapped(const int32_t* host, size_t bytes) {
  if ((reinterpret_cast<uintptr_t>(host) & 3u) != 0) return nullptr;
  const char* ends[2] = {reinterpret_cast<const char*>(host), reinterpret_cast<const char*>(host) + bytes - 1};
  cudaPointerAttributes attr[2];
  for (int i = 0; i < 2; ++i) {
    if (cudaPointerGetAttributes(&attr[i], ends[i]) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    if (attr[i].type != cudaMemoryTypeHost || !attr[i].devicePointer) return nullptr;
  }
  const char* first = static_cast<const char*>(attr[0].devicePointer);
  if (static_cast<const char*>(attr[1].devicePointer) != first + bytes - 1) return nullptr;
  return reinterpret_cast<const int32_t*>(first);
}

// Per-device copy streams, a growing pool of timing-free events and a pinned block, created on first use and kept.  A
// step holds `busy` while it uses them (the call is synchronous).
struct Pipes {
  std::mutex busy;
  cudaStream_t in = nullptr, out = nullptr;
  char* block_out = nullptr;
  std::vector<cudaEvent_t> events;
};

cudaError_t get_pipes(int n_events, Pipes** result, std::unique_lock<std::mutex>* held) {
  static Pipes pipes[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  Pipes& p = pipes[dev];
  *held = std::unique_lock<std::mutex>(p.busy);
  if (!p.in) {
    if ((e = cudaStreamCreateWithFlags(&p.in, cudaStreamNonBlocking)) != cudaSuccess) return e;
    if ((e = cudaStreamCreateWithFlags(&p.out, cudaStreamNonBlocking)) != cudaSuccess) return e;
  }
  if (!p.block_out) {
    if ((e = cudaHostAlloc(reinterpret_cast<void**>(&p.block_out), kBlockBytes, cudaHostAllocDefault)) != cudaSuccess) return e;
  }
  while ((int)p.events.size() < n_events) {
    cudaEvent_t ev;
    if ((e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming)) != cudaSuccess) return e;
    p.events.push_back(ev);
  }
  *result = &p;
  return cudaSuccess;
}

}  // namespace

extern "C" size_t tv_step_staging_bytes(int L, int B, int Nmax, int Hq, int Hkv, int d, int Scap, int V,
                                        int P, int Dp1) {
  if (L < 0 || B < 0 || Nmax < 1 || Hq < 1 || Hkv < 1 || d < 1 || V < 1 || P < 0 || Dp1 < 1) return 0;
  return layout(L, B, Nmax, Hq, Hkv, d, Scap, V, P, Dp1).total;
}

extern "C" int tv_verify_step_host(const tv_step_host_args* a) {
  TV_REQUIRE(a, "tv_verify_step_host: NULL args");
  TV_REQUIRE(a->parent && a->n_nodes && a->tokens && a->q && a->k_tree && a->v_tree && a->logits && a->out &&
                 a->accept_len && a->accepted_nodes && a->next_token && a->status && a->k_cache && a->v_cache &&
                 a->prefix_len && a->staging,
             "tv_verify_step_host: NULL pointer");
  TV_REQUIRE(a->L >= 1 && a->B >= 1 && a->Nmax >= 1 && a->V >= 1 && a->P >= 1 && a->Dp1 >= 1 && a->Dp1 <= a->Nmax,
             "tv_verify_step_host: bad dimension");
  TV_REQUIRE((reinterpret_cast<uintptr_t>(a->staging) & 255u) == 0, "tv_verify_step_host: staging must be 256-byte aligned");
  // Everything the four calls below would refuse is refused here, before the first copy is queued: a call that
  // returns an error has then never touched the host buffers or the staging area.
  TV_REQUIRE(a->B <= 512 && a->Nmax <= 256 && (long long)a->B * a->Nmax <= 65535,
             "tv_verify_step_host: need B <= 512, Nmax <= 256, B * Nmax <= 65535");
  TV_REQUIRE(a->d == 64 || a->d == 128, "tv_verify_step_host: d must be 64 or 128");
  TV_REQUIRE(a->Hq >= 1 && a->Hkv >= 1 && a->Hq % a->Hkv == 0 && a->Hq / a->Hkv <= 128,
             "tv_verify_step_host: need Hq %% Hkv == 0 and Hq / Hkv <= 128");
  TV_REQUIRE(a->Scap >= 1 && a->scale > 0.f && a->L <= 65535 && a->Dp1 <= 1024,
             "tv_verify_step_host: need Scap >= 1, scale > 0, L <= 65535, Dp1 <= 1024");
  TV_REQUIRE((long long)a->B * a->Hkv * ((a->Scap + 127) / 128 + 8) < (1ll << 31),
             "tv_verify_step_host: B * Hkv * Scap is too large for the attention's tile scheduler");
  TV_REQUIRE(tv::aligned16(a->k_cache) && tv::aligned16(a->v_cache), "tv_verify_step_host: the caches must be 16-byte aligned");
  const int L = a->L, B = a->B, Nmax = a->Nmax, Hq = a->Hq, Hkv = a->Hkv, d = a->d, Scap = a->Scap, V = a->V,
            P = a->P, Dp1 = a->Dp1;
  const Staging s = layout(L, B, Nmax, Hq, Hkv, d, Scap, V, P, Dp1);
  if (a->staging_bytes < s.total)
    return tv::fail(TV_ERR_WORKSPACE, "tv_verify_step_host: staging of %zu bytes, need %zu", a->staging_bytes, s.total);
  char* base = static_cast<char*>(a->staging);
  cudaStream_t st = (cudaStream_t)a->stream;
  auto dptr = [&](size_t off) { return base + off; };
  const size_t q_layer = (size_t)B * Nmax * Hq * d, t_layer = (size_t)B * Nmax * Hkv * d, c_layer = (size_t)B * Hkv * Scap * d;
  const size_t layer_bytes = sizeof(tv_bf16) * (q_layer + 2 * t_layer);
  const size_t by_bytes = (kStageBytes + layer_bytes - 1) / layer_bytes;
  const int per_stage = by_bytes < (size_t)L ? (int)by_bytes : L;
  // events: 0 entry, 1 small inputs in, 2 logits in, 3 step done, 4 results out, 5 + l inputs of the stage of layer l in,
  // 5 + L + l stage computed.
  Pipes* pp = nullptr;
  std::unique_lock<std::mutex> held;
  TV_CUDA_OK(get_pipes(5 + 2 * L, &pp, &held));
  cudaStream_t s_in = pp->in, s_out = pp->out;
  cudaEvent_t* ev = pp->events.data();
  // From here on copies are in flight on the two private streams: if anything fails further down, the three
  // streams are drained before the error is returned, so that the caller may free or reuse its buffers at once.
  auto body = [&]() -> int {
  // work already queued on the caller's stream may still use the staging area and the host buffers
  TV_CUDA_OK(cudaEventRecord(ev[0], st));
  TV_CUDA_OK(cudaStreamWaitEvent(s_in, ev[0], 0));
  TV_CUDA_OK(cudaStreamWaitEvent(s_out, ev[0], 0));
  tv_bf16* d_q = reinterpret_cast<tv_bf16*>(dptr(s.q));
  tv_bf16* d_kt = reinterpret_cast<tv_bf16*>(dptr(s.k_tree));
  tv_bf16* d_vt = reinterpret_cast<tv_bf16*>(dptr(s.v_tree));
  tv_bf16* d_out = reinterpret_cast<tv_bf16*>(dptr(s.out));
  struct Part {
    void* host;
    size_t at, bytes;
  };
  const Part in[4] = {{const_cast<int32_t*>(a->parent), s.parent, sizeof(int32_t) * B * Nmax},
                      {const_cast<int32_t*>(a->n_nodes), s.n_nodes, sizeof(int32_t) * B},
                      {const_cast<int32_t*>(a->tokens), s.tokens, sizeof(int32_t) * B * Nmax},
                      {const_cast<int32_t*>(a->retrieve_indices), s.retrieve, a->retrieve_indices ? sizeof(int32_t) * B * P * Dp1 : 0}};
  SmallInputs small{};
  size_t in_bytes = 0;
  bool fetch = true;
  for (int k = 0; k < 4; ++k) {
    in_bytes += in[k].bytes;
    if (!in[k].bytes || !fetch) continue;
    small.src[k] = in_bytes <= kBlockBytes ? mapped(static_cast<const int32_t*>(in[k].host), in[k].bytes) : nullptr;
    small.dst[k] = reinterpret_cast<int32_t*>(dptr(in[k].at));
    small.count[k] = (int)(in[k].bytes / sizeof(int32_t));
    fetch = small.src[k] != nullptr;
  }
  if (fetch) {
    const unsigned ctas = (unsigned)((in_bytes / sizeof(int32_t) + kFetchThreads - 1) / kFetchThreads);
    TV_CUDA_OK(tv::launch_pdl(fetch_small_kernel, dim3(ctas), dim3(kFetchThreads), 0, st, small));
    tv::count_launches(1);
  } else {
    for (const Part& p : in)
      if (p.bytes) TV_CUDA_OK(cudaMemcpyAsync(dptr(p.at), p.host, p.bytes, cudaMemcpyHostToDevice, s_in));
    TV_CUDA_OK(cudaEventRecord(ev[1], s_in));
    TV_CUDA_OK(cudaStreamWaitEvent(st, ev[1], 0));
  }
  for (int l = 0; l < L; l += per_stage) {
    const size_t n = (size_t)(L - l < per_stage ? L - l : per_stage);
    TV_CUDA_OK(cudaMemcpyAsync(d_q + l * q_layer, a->q + l * q_layer, sizeof(tv_bf16) * n * q_layer, cudaMemcpyHostToDevice, s_in));
    TV_CUDA_OK(cudaMemcpyAsync(d_kt + l * t_layer, a->k_tree + l * t_layer, sizeof(tv_bf16) * n * t_layer, cudaMemcpyHostToDevice, s_in));
    TV_CUDA_OK(cudaMemcpyAsync(d_vt + l * t_layer, a->v_tree + l * t_layer, sizeof(tv_bf16) * n * t_layer, cudaMemcpyHostToDevice, s_in));
    TV_CUDA_OK(cudaEventRecord(ev[5 + l], s_in));
  }
  TV_CUDA_OK(cudaMemcpyAsync(dptr(s.logits), a->logits, sizeof(tv_bf16) * (size_t)B * Nmax * V, cudaMemcpyHostToDevice, s_in));
  TV_CUDA_OK(cudaEventRecord(ev[2], s_in));

  int32_t* d_n_nodes = reinterpret_cast<int32_t*>(dptr(s.n_nodes));
  int32_t* d_status = reinterpret_cast<int32_t*>(dptr(s.status));
  int32_t* d_retrieve = reinterpret_cast<int32_t*>(dptr(s.retrieve));
  uint32_t* d_bits = reinterpret_cast<uint32_t*>(dptr(s.anc_bits));
  int rc = tree_build_mask(reinterpret_cast<int32_t*>(dptr(s.parent)), d_n_nodes, B, Nmax, Dp1 - 1, P, d_bits,
                           nullptr, nullptr, nullptr, a->retrieve_indices ? nullptr : d_retrieve,
                           reinterpret_cast<int32_t*>(dptr(s.n_paths)), d_status, a->stream);
  if (rc != TV_OK) return rc;
  for (int l = 0; l < L; l += per_stage) {
    const int n = L - l < per_stage ? L - l : per_stage;
    TV_CUDA_OK(cudaStreamWaitEvent(st, ev[5 + l], 0));
    // (the kernel in front, the mask or the stage before, leaves prefix_len and the cache alone)
    rc = tree_verify_attn_layers(d_q + l * q_layer, a->k_cache + l * c_layer, a->v_cache + l * c_layer, d_kt + l * t_layer,
                                 d_vt + l * t_layer, a->prefix_len, d_n_nodes, d_bits, n, B, Nmax, Hq, Hkv, d, Scap, a->scale,
                                 (int64_t)q_layer, (int64_t)c_layer, (int64_t)t_layer, d_out + l * q_layer, (int64_t)q_layer,
                                 nullptr, dptr(s.attn_ws), s.attn_ws_bytes, d_status, TV_ATTN_STABLE_INPUTS, a->stream);
    if (rc != TV_OK) return rc;
    TV_CUDA_OK(cudaEventRecord(ev[5 + L + l], st));
    TV_CUDA_OK(cudaStreamWaitEvent(s_out, ev[5 + L + l], 0));
    TV_CUDA_OK(cudaMemcpyAsync(a->out + l * q_layer, d_out + l * q_layer, sizeof(tv_bf16) * n * q_layer, cudaMemcpyDeviceToHost, s_out));
  }
  int32_t* d_alen = reinterpret_cast<int32_t*>(dptr(s.accept_len));
  int32_t* d_acc = reinterpret_cast<int32_t*>(dptr(s.accepted));
  int32_t* d_next = reinterpret_cast<int32_t*>(dptr(s.next_token));
  TV_CUDA_OK(cudaStreamWaitEvent(st, ev[2], 0));
  rc = tree_accept(reinterpret_cast<tv_bf16*>(dptr(s.logits)), reinterpret_cast<int32_t*>(dptr(s.tokens)),
                   d_retrieve, d_n_nodes, B, Nmax, V, P, Dp1, reinterpret_cast<int32_t*>(dptr(s.argmax)),
                   nullptr, nullptr, d_alen, reinterpret_cast<int32_t*>(dptr(s.best_path)), d_acc, d_next,
                   dptr(s.accept_ws), s.accept_ws_bytes, d_status, a->stream);
  if (rc != TV_OK) return rc;
  rc = kv_commit(a->k_cache, a->v_cache, d_kt, d_vt, d_acc, d_alen, a->prefix_len, L, B, Nmax, Hkv, d, Scap, Dp1,
                 (int64_t)c_layer, (int64_t)t_layer, d_status, a->stream);
  if (rc != TV_OK) return rc;
  TV_CUDA_OK(cudaEventRecord(ev[3], st));
  TV_CUDA_OK(cudaStreamWaitEvent(s_out, ev[3], 0));
  const Part res[4] = {{a->accept_len, s.accept_len, sizeof(int32_t) * B},
                       {a->accepted_nodes, s.accepted, sizeof(int32_t) * B * Dp1},
                       {a->next_token, s.next_token, sizeof(int32_t) * B},
                       {a->status, s.status, sizeof(int32_t) * B}};
  const size_t res_bytes = res[3].at + res[3].bytes - res[0].at;
  const bool together = res_bytes <= kBlockBytes;
  if (together) TV_CUDA_OK(cudaMemcpyAsync(pp->block_out, dptr(res[0].at), res_bytes, cudaMemcpyDeviceToHost, s_out));
  else
    for (const Part& p : res) TV_CUDA_OK(cudaMemcpyAsync(p.host, dptr(p.at), p.bytes, cudaMemcpyDeviceToHost, s_out));
  TV_CUDA_OK(cudaEventRecord(ev[4], s_out));
  TV_CUDA_OK(cudaStreamWaitEvent(st, ev[4], 0));
  TV_CUDA_OK(cudaStreamSynchronize(st));
  if (together)
    for (const Part& p : res) memcpy(p.host, pp->block_out + (p.at - res[0].at), p.bytes);
  return TV_OK;
  };
  const int rc_step = body();
  if (rc_step != TV_OK) {
    cudaStreamSynchronize(s_in);
    cudaStreamSynchronize(s_out);
    cudaStreamSynchronize(st);
  }
  return rc_step;
}
