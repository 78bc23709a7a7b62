// tree_verify_attn: GQA tree attention for sm_100a (Sections 2.3, 2.4, 3.3).
//
// Packing.  For one sequence b and KV head hk, the G = Hq/Hkv query heads of
// every tree node share the same K/V, so (node, group member) pairs are packed
// into dense MMA rows r = node_local * G + g.  A row tile holds 128 rows =
// 128/G nodes; a CTA owns MT (1 or 2) row tiles and streams 128-key tiles of
// the committed prefix, then one tile of the tree's own keys.
//
// Pipeline (one CTA per SM, 12 warps):
//   warp 0      TMA producer: Q tiles once per work item, then K and V tiles
//               through a shared-memory ring of 5 or 10 slots (128-byte swizzled
//               boxes).
//   warp 1      tcgen05.mma issuer (one thread): S = Q K^T for a whole 128-key
//               tile (N = 128; 64-key MMAs re-read Q from shared memory twice as
//               often and run at 2/3 of the rate), O += P V with P read from
//               TMEM; completion goes to mbarriers with tcgen05.commit.  With
//               two row tiles it serves them in turn, so the softmax of one row
//               tile runs while the tensor pipe works for the other.
//   warp 2      raises the flag of the CTA's partials, where another CTA merges them
//   warp 3      of the first CTA: lets the launch with an odd last row tile start (see beside)
//   warps 4-7   two softmax warpgroups, one thread per row, online softmax with
//   warps 8-11  lazy rescale, one for each row tile.  With one row tile and
//               64-wide heads (KS) one takes the even and one the odd key tiles of
//               an item, each with an O of its own (combined in the epilogue);
//               with 128-wide heads, whose K/V stream sets the pace, the second
//               one idles.  The ancestor bitmask of the row is applied only
//               on the tree tile(s), the prefix length only on the ragged
//               last prefix tile.
// TMEM: S0 (128 columns) | P0 P1 (bf16, 64 columns each) | O0 O1 (D columns each),
// and S1 where O1 leaves room for it (see SmemLayout).  With one warpgroup the S and
// P buffers alternate by key tile.
//
// Code size matters here: instruction fetches compete with the K/V stream for
// L2 and HBM, and code that runs once per work item (set-up, epilogue, merge)
// is fetched cold every time.  Cold paths are therefore written as loops, not
// unrolled, and the timeline marks are compiled out unless -DTV_TRACE is given.
//
// Work split.  All key tiles of all (layer, b, hk) units of the launch - one
// layer, or all layers of a step - form one linear space that
// is cut evenly over the CTA groups (a group = the CTAs that hold the row
// tiles of the same unit and walk the same keys together, so the second reader
// hits L2).  A unit cut in pieces leaves partials (normalised O in bf16, m, l) in the
// workspace; the CTA that holds the unit's first piece merges them.  Groups run
// downwards over the block index, so a merging CTA waits only for CTAs with a lower
// block index, which were started before it.  Flags hold the epoch of the call, so the
// workspace needs no initialisation.
//
// Few units (CL = true).  A unit is shared by a thread-block cluster instead: its CTAs
// take equal shares of the unit's key tiles, leave their partials in their own shared
// memory and, behind a cluster barrier, each merges a share of the rows through
// distributed shared memory.  No tile table, no workspace, no flags; see cluster_size.
//
// Every wait on an mbarrier is bounded: on expiry the CTA raises
// TV_ST_TIMEOUT for all sequences, all roles leave their loops, outstanding
// copies are given time to land, TMEM is freed and the kernel returns.  The two
// barriers of a cluster have no limit of their own: every role of every CTA
// reaches them, because every wait in front of them ends.
#include "common.cuh"
#include "row_tiles.h"
#include "treeverify_debug.h"

#include <cuda.h>
#include <cuda_bf16.h>

#include <atomic>
#include <chrono>
#include <type_traits>

namespace {

constexpr int kTileN = 128;        // keys per tile
constexpr int kTileM = 128;        // rows per row tile
constexpr int kThreads = 384;
constexpr int kMaxB = 512;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kRescaleThreshold = 8.0f;            // in log2 units
constexpr unsigned long long kWaitLimitNs = 2000000000ull;
// Virtual tiles charged per unit by the scheduler: what a CTA pays for one more item (epilogue, masked tiles, refill) is
// some 5 us, three to four tiles' time.  Eight shapes, one and 32 layers a launch: 4 is 1 to 2 % faster than 1 and 5 on most; 3 is
// level with 4.  Of 72 shapes 2 is 1 to 4 % faster than 4 on 33 (one row tile above all) and slower on 9, where every unit, or every
// second, is cut once: us a launch, 2 / 4, 128-wide heads, 8 sequences of 4096 41.7 / 39.8, 32 of 1024 45.2 / 43.9, 4 of 4096 with
// 128 nodes 41.7 / 40.8, of 4000 ... 4096 58.1 / 56.2, 32 of 650 ... 4550 with one row tile 65.3 / 63.0; 8 of 1024 ... 8192 47.8 / 46.1.
#ifndef TV_SETUP_COST
#define TV_SETUP_COST 4
#endif
constexpr int kSetupCost = TV_SETUP_COST;
// K/V tiles that a CTA asks for in L2 while the kernel in front is still running.  16 sequences of 512 to 4096, layer after
// layer: 48.6 us a launch with none, 47.7 with 2, 47.9 with 4, 48.6 with 8 (they take their bandwidth from that kernel's tail).
#ifndef TV_PREFETCH_TILES
#define TV_PREFETCH_TILES 2
#endif
constexpr int kPrefetchTiles = TV_PREFETCH_TILES;
constexpr int kMaxGroups = 160;
// do not spread a small problem over more CTA groups than this allows.  Few short units outside the cluster kernel's range, us a
// call for 6 / 8: 16 sequences of 150 to 600 with 8 KV heads, 60 nodes 22.3 / 25.4, two of 2300 in a cache of 32768 25.6 / 28.3,
// four of 1000, 17 nodes 17.9 / 19.3.
#ifndef TV_MIN_VT
#define TV_MIN_VT 6
#endif
constexpr int kMinVirtualTilesPerGroup = TV_MIN_VT;
// Virtual tiles of a unit up to which equal units stay whole, on one group each.  us a call, cut / whole, 8 KV heads: 8 sequences
// of 65 nodes, prefixes of 300 19.9 / 16.6, 600 22.8 / 19.4, 1000 26.8 / 23.9, 2300 41.0 / 39.1; 10 of 20 nodes 15.7 / 12.9, 17.5 /
// 14.6, 20.4 / 17.8, 26.7 / 29.2; 12 of 40 nodes with 64-wide heads 15.2 / 14.2, 19.2 / 17.1, 23.5 / 21.6, 34.4 / 36.8.
constexpr int kMaxWholeUnit = 13;
// An odd last row tile has a launch of its own where the capacity of the cache allows this many key tiles per SM, and the lengths
// reach those of odd_row_tile.  In a smaller cache the short calls would lose what the long ones gain, to a second launch that
// finds nothing to do: 65 nodes, 8 sequences, us a call, one launch / two, in a cache of 28 key tiles per SM with lengths of 4
// 31.1 / 33.7, 10 50.7 / 53.2, 14 64.0 / 60.5, in one of 33 with 22 98.6 / 91.1.
constexpr int kSplitTilesPerSm = 60;
constexpr int kMaxCluster = 8;     // CTAs that share a unit (16 is not portable; few clusters of 16 fit the GPU at once: 21.7 us
                                   // instead of 10.8 us a launch for eight units of 12 key tiles)
constexpr int kTraceCap = 256;     // events per (CTA, role) kept by the optional trace

// ---------------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait.  Returns false if the wait was abandoned (timeout here or abort raised elsewhere).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          unsigned long long limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = globaltimer_ns();
  uint32_t spins = 0;
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((++spins & 255u) == 0) {
      if (*abort_flag) return false;
      if (globaltimer_ns() - t0 > limit_ns) {
        *abort_flag = 1;
        return false;
      }
    }
  }
}
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// Programmatic dependent launch.  gdc_wait: every kernel launched before this one in the stream has finished and
// its writes are visible.  gdc_launch_dependents: the next kernel in the stream may be scheduled once every CTA of
// this grid has got here or has exited.
__device__ __forceinline__ void gdc_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void gdc_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Asks for a tile of a tensor in L2.
__device__ __forceinline__ void tma_prefetch_4d(const CUtensorMap* map, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.prefetch.tensor.4d.L2.global.tile [%0, {%1, %2, %3, %4}];" ::"l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
               : "memory");
}
__device__ __forceinline__ void tma_prefetch_5d(const CUtensorMap* map, int c0, int c1, int c2, int c3, int c4) {
  asm volatile("cp.async.bulk.prefetch.tensor.5d.L2.global.tile [%0, {%1, %2, %3, %4, %5}];" ::"l"(map), "r"(c0), "r"(c1), "r"(c2),
               "r"(c3), "r"(c4)
               : "memory");
}
// One lane of a converged warp (the compiler keeps what it guards in the uniform datapath).
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
  return pred != 0;
}
// 32 bytes per thread in one store (a whole sector); the address must be 32-byte aligned.
__device__ __forceinline__ void st_global_32B(void* p, uint4 a, uint4 b) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w),
               "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w) : "memory");
}
// Thread-block clusters: barrier over all threads, and reads of another CTA's shared memory (32-bit cluster addresses).
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The same without ordering any memory access: for a barrier that only keeps a CTA's shared memory alive.
__device__ __forceinline__ void cluster_sync_relaxed() {
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_size_x() {
  uint32_t n;
  asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(n));
  return n;
}
__device__ __forceinline__ uint32_t peer_smem(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ float2 ld_peer_8B(uint32_t addr) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ uint4 ld_peer_16B(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared::cluster.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Tiled TMA loads.  The one for the cache carries an L2 eviction-priority hint: the committed K/V prefix is read once per
// launch, and letting it leave L2 first keeps Q, the partials and the kernel's own code resident.
// (The outermost coordinate of every tensor is the layer.)
__device__ __forceinline__ void tma_load_4d_hint(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2,
                                                 int c3, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5, %6}], [%2], %7;"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2,
                                            int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
      : "memory");
}

// Shared-memory matrix descriptor, 128-byte swizzle, descriptor version 1 (sm_100).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((addr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>((lbo_bytes >> 4) & 0x3FFFu) << 16;
  d |= static_cast<uint64_t>((sbo_bytes >> 4) & 0x3FFFu) << 32;
  d |= 1ull << 46;
  d |= 2ull << 61;
  return d;
}
// Instruction descriptor, kind::f16: bf16 x bf16 -> fp32, M = 128, A K-major.
__host__ __device__ constexpr uint32_t instr_desc(int n, bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) | (static_cast<uint32_t>(n >> 3) << 17) |
         (static_cast<uint32_t>(kTileM >> 4) << 24);
}
// tcgen05.mma, kind::f16, one CTA.  The 64-bit shared-memory descriptors are given as (low, high) words: the
// high word of every descriptor used here is one constant, so the issuing thread only adds an offset to a
// low word per MMA.
__device__ __forceinline__ void mma_ss_lohi(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc,
                                            uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "mov.b64 da, {%1, %3};\n\t"
      "mov.b64 db, {%2, %3};\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}"
      ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void mma_ts_lohi(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t hi, uint32_t idesc,
                                            uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t"
      "mov.b64 db, {%2, %3};\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(hi), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]),
        "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]),
        "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
      : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Optional timeline for tuning: role r of this CTA appends (tag, time since kernel start of CTA 0).
struct Tracer {
  unsigned long long* base;
  int n;
  __device__ __forceinline__ void init(unsigned long long* trace, int role) {
    base = trace ? trace + ((size_t)blockIdx.x * 4 + role) * kTraceCap : nullptr;
    n = 0;
  }
  __device__ __forceinline__ void mark(uint32_t tag) {
#ifndef TV_TRACE
    (void)tag;        // compiled out: even switched off, the marks cost several per cent of the kernel's time
    return;
#endif
    if (base && n < kTraceCap) base[n++] = ((unsigned long long)tag << 48) | (globaltimer_ns() & 0xffffffffffffull);
  }
};

// Packed fp32 pair arithmetic (one issue slot for two lanes of work).
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 fadd2(float2 a, float2 b) { return __fadd2_rn(a, b); }
// Three-operand maximum (one instruction on sm_100); a NaN operand is ignored.
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// Flags between CTAs.  Whoever sees the released value also sees what this thread wrote before, and what threads that it
// has synchronised with wrote before.
__device__ __forceinline__ void st_release(unsigned long long* p, unsigned long long v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// ---------------------------------------------------------------- kernel parameters
struct AttnParams {
  const int32_t* prefix_len;
  const int32_t* n_nodes;
  const uint32_t* anc_bits;
  tv_bf16* out;
  float* lse;
  int32_t* status;
  tv_bf16* part_o;               // [slots][D/8][MT*128][8] bf16 normalised outputs, column-group major
  float* part_ml;                // [slots][2][MT*128]  (m in log2 units, then l); one slot per CTA
  unsigned long long* flags;     // [slots]: the epoch of the call once the partial in that slot is complete
  unsigned long long epoch;      // tag of this call
  int B, Nmax, Hq, Hkv, Scap, G, NPT, NP, W, groups;
  int tile0;                     // first row tile of this launch
  int split_tiles;               // > 0: one of a pair of launches.  From this many key tiles on (all units of the launch, by the lengths
                                 // on the device) the odd last row tile belongs to the second one; below, that one has no work
  int behind_tiles;              // from this many on the second one runs behind the first one, below it runs beside it
  int split_NP, beside_groups, behind_groups;      // NP of this launch where the last row tile is split off, its groups in either case
  int slot0;                     // its first slot where it runs beside the other
  int TT;                        // key tiles of the tree's own K/V: ceil(Nmax / 128), 1 or 2
  uint32_t q_box_bytes;          // bytes of one Q box {64, G, NPT}: 16 KB when G divides 128
  unsigned long long* trace;     // optional event trace [cta][role 0..3][kTraceCap] of (tag << 48 | ns), or NULL
  int tree_in_cache;             // the tree's K/V rows live in the cache behind the prefix (rows S_b + node)
  const int32_t* block_table;    // paged cache: page of key tile j of sequence b at [b * max_blocks + j]; else nullptr
  int max_blocks, n_pages;
  int out_al32;                  // out is 32-byte aligned: rows can be written 32 bytes per thread and store
  float scale_log2e;             // scale * log2(e)
  float scale;
  unsigned long long* passed;    // a pair of launches: holds passed_tag once the first one has seen everything in front of the
  unsigned long long passed_tag; // pair complete, until the second one ends; else nullptr
  int early;                     // the caller promises that the kernel in front leaves prefix_len, n_nodes, the block
                                 // table and the committed rows alone: they are read before the grid-dependency wait
  unsigned long long wait_limit_ns;   // limit of every bounded wait
  int debug;                     // bit 0: the producer issues no copy at all; bit 1: pieces of cut units store their
                                 // partials but never announce them (both exercise the expiry of a bounded wait);
                                 // bit 3: the guessed table is built from lengths one tile too long;
                                 // bit 4 (host): the cluster kernel is not left out;
                                 // bit 5: the flag that lets two launches run at the same time is not raised;
                                 // bit 2: the K/V stream alone - the issuing warp only hands every slot back as
                                 // soon as it is full, no MMA, no softmax, no output (what the memory side can do)
  int L;                         // layers in this launch: their units form one tile space, layer after layer
  long long out_layer_stride;    // elements between the outputs of two layers (lse is dense, [L,B,Hq,Nmax])
};

struct Item {
  int b, hk, j0, j1, len, S, n, layer;
};

// Shared bookkeeping of the linear tile space: cum[b] = sum of len over b' < b, len_b = ceil(S_b/128) + 1.
// The schedule works in a "virtual" tile space: every (sequence, KV head) unit is charged kSetupCost
// virtual tiles in front of its real key tiles, the price of starting a unit (Q load, pipeline refill,
// epilogue).  Cutting that space evenly gives CTAs that start more units fewer real tiles, and a cut that
// falls into a unit's setup region snaps to the unit boundary, which saves a split.
struct Sched {
  const int* cum;    // cum[b] = sum over b' < b of (len_b' + kSetupCost)
  const int* gs;     // gs[k] = first virtual tile of CTA group k, gs[groups] = total
  int B, Hkv;
  int total;         // layers * Hkv * cum[B]; the host refuses problems whose tile count does not fit 31 bits
  int per_layer;     // Hkv * cum[B]: the units of a layer tile one such stretch, layer after layer
  __device__ __forceinline__ int group_start(int k, int) const { return gs[k]; }
  __device__ __forceinline__ int find_b(int g) const {
    int lo = 0, hi = B - 1;   // largest b with Hkv*cum[b] <= g
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (Hkv * cum[mid] <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
  }
};

template <int D, int MT>
struct SmemLayout {
  static constexpr int kHalf = 64 * 128 * 2;               // one 64-column, 128-row swizzled box: 16 KB
  static constexpr int kTileBytes = (D / 64) * kHalf;      // a 128 x D bf16 tile
  static constexpr int kSlots = D == 64 ? 10 : 5;             // K/V ring slots
  static constexpr int kQ = 0;
  static constexpr int kRing = MT * kTileBytes;
  static constexpr int kBars = kRing + kSlots * kTileBytes;
  // barrier indices (8 bytes each)
  static constexpr int Q_FULL = 0, Q_EMPTY = 1, KV_FULL = 2, KV_EMPTY = 2 + kSlots, S_FULL = 2 + 2 * kSlots,
                       S_FREE = S_FULL + 2, P_READY = S_FREE + 2, O_DONE = P_READY + 2, ITEM_DONE = O_DONE + 1,
                       EPI = ITEM_DONE + 2, ITEM_READ = EPI + 1, PIECE = ITEM_READ + 1, NBARS = PIECE + 1;
  // Tensor memory columns.  One S buffer for two row tiles of 128-wide heads (there is no room for a second one
  // beside P0 P1 O0 O1), two buffers otherwise.
  static constexpr int kTmemS0 = 0, kTmemP0 = 128, kTmemO0 = 256;
  static constexpr int kTmemS1 = (D == 128 && MT == 2) ? kTmemS0 : 384;
  static constexpr int kMisc = kBars + NBARS * 8;          // tmem ptr, abort flag, announcement (see PIECE)
  static constexpr int kItems = kMisc + 16;                // the producer's current and next item (see publish)
  static constexpr int kCum = kItems + 3 * 32 + 16;
  static constexpr int kGs = kCum + (kMaxB + 1) * 4;
  static constexpr int kXch = (kGs + (kMaxGroups + 1) * 4 + 7) & ~7;      // KS: (m, l) of both warpgroups' rows
  static constexpr bool kKeySplit = MT == 1 && D == 64;
  static constexpr int kTotal = kKeySplit ? kXch + 256 * 8 : kGs + (kMaxGroups + 1) * 4;
  static_assert(kTotal <= 232448, "shared memory of a CTA");
  static constexpr int kMl = kCum;                         // cluster kernel: (m, l) of every row, in place of the tile table
  static_assert(kMl + MT * 128 * 8 <= kTotal && kMl % 8 == 0, "(m, l) pairs fit the room of the tile table");
  static_assert(MT * 128 * D * 4 <= kSlots * kTileBytes, "fp32 partials of the cluster kernel fit the K/V ring");
};

// ---------------------------------------------------------------- the kernel
template <int D, int MT, bool CL>
__global__ void __launch_bounds__(kThreads, 1)
tree_attn_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_kc,
                 const __grid_constant__ CUtensorMap map_vc, const __grid_constant__ CUtensorMap map_kt,
                 const __grid_constant__ CUtensorMap map_vt, const AttnParams prm) {
  using L = SmemLayout<D, MT>;
  // One row tile.  KS: the two softmax warpgroups share the keys of an item, tile by tile.  A 64-wide head's key tile is
  // 32 KB, 0.7 us of the HBM rate, and one warpgroup needs 1 us for it (16 sequences of 8000, G = 4, 24 nodes: 72.7 ->
  // 59.5 us a launch).  ONE: a 128-wide head's tile takes 1.5 us to arrive; there the second tile in hand only takes ring
  // slots away from the stream (16 sequences of 1000, 17 nodes: 22.5 -> 25.7 us), and one warpgroup does it all.
  constexpr bool KS = L::kKeySplit, ONE = MT == 1 && !KS;
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t sbase = smem_u32(smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bars = sbase + L::kBars;
  auto bar = [&](int i) { return bars + 8u * i; };
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::kMisc + 4);
  Item* items = reinterpret_cast<Item*>(smem + L::kItems);
  volatile unsigned long long* announce = reinterpret_cast<volatile unsigned long long*>(smem + L::kMisc + 8);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + L::kMisc);
  int* cum = reinterpret_cast<int*>(smem + L::kCum);
  int* gs = reinterpret_cast<int*>(smem + L::kGs);
  const unsigned long long wait_limit = prm.wait_limit_ns;

  // What happens to an odd last row tile, from the key tiles of one KV head over all sequences: 0 it stays with the others, 1 it
  // has a launch beside them, 2 behind them.
  auto odd_mode = [&](int tiles) -> int {
    const unsigned all = (unsigned)(prm.Hkv * tiles) * (unsigned)prm.L;
    return all < (unsigned)prm.split_tiles ? 0 : (all < (unsigned)prm.behind_tiles ? 1 : 2);
  };
  // The second launch of a pair.  It is scheduled when every CTA of the first one is behind its grid-dependency wait.  What that makes
  // complete is visible to the first launch; the flag that it released there and every thread here acquires hands it on.  Who does
  // not find the flag waits for the first launch like any other kernel.  Beside the first one it reads nothing that one writes, and
  // waits for it only where it ends; behind it it waits like any other.
  constexpr bool MAY_BE_SECOND = MT == 1 && !CL;
  bool beside = false;
  // Who waits for this launch waits for the first one.  All CTAs with work stay for that: where only one did, the next
  // attention spread over the SMs as they came free (65 nodes, layer after layer: 63.5 -> 79 us, 8 layers a launch 290 -> 349).
  auto end_pair = [&]() {
    gdc_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0) *reinterpret_cast<volatile unsigned long long*>(prm.passed) = 0ull;      // (a graph comes with the tag again)
  };
  if (MAY_BE_SECOND && prm.split_tiles > 0) {
    if (ld_acquire(prm.passed) != prm.passed_tag) gdc_wait();
    int tiles = 0;
#pragma unroll 1
    for (int b = lane; b < prm.B; b += 32) {
      const int S = __ldcg(prm.prefix_len + b);
      tiles += ((S < 0 ? 0 : (S > prm.Scap ? prm.Scap : S)) + kTileN - 1) / kTileN + prm.TT;
    }
    const int mode = odd_mode(__reduce_add_sync(0xffffffffu, tiles));
    beside = mode == 1;
    if (mode == 0 || (beside && blockIdx.x >= prm.beside_groups)) {      // no work for this CTA
      if (threadIdx.x == 0) gdc_launch_dependents();
      if (blockIdx.x == 0) end_pair();      // one CTA is enough to wait; the others leave their SMs (short calls 44.5 -> 43.4 us)
      return;
    }
  }

  unsigned long long* const trace = prm.trace && beside ? prm.trace + (size_t)prm.slot0 * 2 * kTraceCap : prm.trace;

  // ---- setup: schedule table, barriers, TMEM
  if (threadIdx.x == 64) {     // fetch the five TMA descriptors while the rest of the set-up runs
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_q) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_kc) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_vc) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_kt) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_vt) : "memory");
  }
  if (threadIdx.x == 32) {
    mbar_init(bar(L::Q_FULL), 1);
    mbar_init(bar(L::Q_EMPTY), 1);
#pragma unroll 1
    for (int s = 0; s < L::kSlots; ++s) {
      mbar_init(bar(L::KV_FULL + s), 1);
      mbar_init(bar(L::KV_EMPTY + s), 1);
    }
    for (int s = 0; s < 2; ++s) {                // index = softmax warpgroup, or parity of the key tile with one warpgroup
      mbar_init(bar(L::S_FULL + s), 1);
      mbar_init(bar(L::S_FREE + s), 4);
      mbar_init(bar(L::P_READY + s), 4);
      mbar_init(bar(L::ITEM_DONE + s), 1);
    }
    mbar_init(bar(L::O_DONE), 1);
    mbar_init(bar(L::EPI), ONE ? 128 : 256);
    mbar_init(bar(L::ITEM_READ), ONE ? 4 : 8);
    mbar_init(bar(L::PIECE), ONE ? 4 : 8);
    *announce = 0;
    *abort_flag = ((sbase & 1023u) != 0) ? 1 : 0;   // swizzled tiles need a 1024-byte aligned base
    fence_barrier_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32((const void*)tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  // Without the caller's promise nothing of the problem counts before every earlier kernel has finished (a kernel in front may
  // still be writing prefix_len, and lines of it cached by an earlier launch on this SM are only dropped by the wait).  This
  // kernel is resident long before that, on SMs that the one in front has left, so it goes by what prefix_len says now, builds
  // the table, asks for the first K/V tiles of its range in L2, and after the wait compares: only if a length has
  // changed the table is built again (layers behind one another as above: 50.1 -> 47.8 us a launch, the first S is there 3.5 us
  // after the wait and not 5; a member of a context split 41.2 -> 40.7; 64-wide heads, one row tile, 16 sequences of 8000,
  // 24 nodes: 62.8 -> 63.6).  What is asked for in L2 is right whoever writes it until the wait.  The cluster
  // kernel has no table to build: its roles wait where they read.
  bool guess = !CL && !prm.early;
  Sched sch{cum, gs, prm.B, prm.Hkv, 0, 0};
  int groups = 1, group = 0, g_begin = 0, g_end = 1;

  // Walks the items of this CTA's range (producer warp).  It publishes every item to the other roles through shared
  // memory, in front of the arrival on Q_FULL that they wait for; entries are used in turn, and an item is published only
  // when the softmax warps have read the one before (a parity wait cannot tell phases two apart).  (Walking in every role
  // cost each of them a division, a search and two L2 round trips per item: about 1.5 us between the epilogue of an item and its
  // successor's first tile.)  locate: from the table alone, all but S and n.
  auto locate = [&](int& g, Item& it) -> bool {
    while (g < g_end) {
      const int layer = (int)((unsigned)g / (unsigned)sch.per_layer);
      const int gl = g - layer * sch.per_layer;                   // place inside the layer
      const int b = sch.find_b(gl);
      const int lenv = cum[b + 1] - cum[b];                       // setup region + real tiles
      const unsigned local = (unsigned)(gl - prm.Hkv * cum[b]);
      const int hk = (int)(local / (unsigned)lenv);
      const int r0 = (int)(local - (unsigned)hk * (unsigned)lenv);
      const int room = g_end - g;
      const int r1 = (lenv - r0) < room ? lenv : r0 + room;
      g += r1 - r0;
      const int j0 = r0 > kSetupCost ? r0 - kSetupCost : 0;
      const int j1 = r1 > kSetupCost ? r1 - kSetupCost : 0;
      if (j1 <= j0) continue;                                     // only setup tiles of this unit fall in the range
      it.b = b;
      it.hk = hk;
      it.layer = layer;
      it.j0 = j0;
      it.j1 = j1;
      it.len = lenv - kSetupCost;
      return true;
    }
    return false;
  };
  // one warp: Q and the first prefix tiles of this CTA's first item, a box per lane and turn, in the order of their use
  // (items[2]: that item; at[0]: it is there; at[1]: where the search goes on, for the second launch of a pair its first slot; at[2]: CTA
  // groups; at[3]: CTAs of a group)
  volatile int* at = reinterpret_cast<volatile int*>(items + 3);
  auto prefetch_first = [&]() {
    Item first;
    int g_first = g_begin;
    const bool have = locate(g_first, first);
    if (lane == 0) {
      at[0] = have;
      at[1] = g_first;
      items[2] = first;
    }
    __syncwarp();
    if (!have) return;
    constexpr int kBoxes = 2 * (D / 64), kQBoxes = MT * (D / 64);
    const int tiles = min(min(first.j1, first.len - prm.TT) - first.j0, kPrefetchTiles);
    for (int x = lane; x < kQBoxes + tiles * kBoxes; x += 32) {
      if (x < kQBoxes) {
        const int tile = prm.tile0 + (int)(blockIdx.x % (MT == 2 ? at[3] : prm.NP)) * MT + x / (D / 64);
        tma_prefetch_5d(&map_q, x % (D / 64) * 64, first.hk * prm.G, tile * prm.NPT, first.b, first.layer);
        continue;
      }
      const int y = x - kQBoxes, j = first.j0 + y / kBoxes, kv = y % kBoxes / (D / 64), h = y % (D / 64);
      int row0 = j * kTileN, slab = first.b * prm.Hkv + first.hk;
      if (prm.block_table) {
        const int pg = __ldcg(prm.block_table + (size_t)first.b * prm.max_blocks + j);
        if ((unsigned)pg >= (unsigned)prm.n_pages) continue;
        row0 = 0;
        slab = pg * prm.Hkv + first.hk;
      }
      tma_prefetch_4d(kv ? &map_vc : &map_kc, h * 64, row0, slab, first.layer);
    }
    __syncwarp();
  };

  while (!CL) {
    if (warp == 0) {
      int run = 0, first_len = 0;
      bool same = true;      // every unit has the key tiles of the first
      // Under the caller's promise this warp reads lengths, node counts and pages before the wait: the fence drops what an
      // earlier launch on this SM has left of them in L1.  (Loads past L1 in the item walk, which goes on behind the wait,
      // cost 16 sequences of 600 to 1000 1 to 3 %.)
      if (prm.early) __threadfence();
#pragma unroll 1
      for (int base = 0; base < prm.B; base += 32) {
        const int b = base + lane;
        int len = 0;
        if (b < prm.B) {
          int S = !guess ? prm.prefix_len[b] : __ldcg(prm.prefix_len + b) + (prm.debug & 8 ? kTileN : 0);
          S = S < 0 ? 0 : (S > prm.Scap ? prm.Scap : S);
          len = (S + kTileN - 1) / kTileN + prm.TT + kSetupCost;
        }
        int inc = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += t;
        }
        if (b < prm.B) cum[b] = run + inc - len;
        run += __shfl_sync(0xffffffffu, inc, 31);
        if (base == 0) first_len = __shfl_sync(0xffffffffu, len, 0);
        same = same && (b >= prm.B || len == first_len);
      }
      same = __all_sync(0xffffffffu, same);
      if (lane == 0) {
        cum[prm.B] = run;
        // Small problems use fewer CTA groups, so that a unit is cut into few pieces (each piece costs a partial
        // write and a merge) and every group still gets a worthwhile share of tiles.
        const int units = prm.B * prm.Hkv * prm.L;
        const int mode = prm.split_tiles > 0 ? odd_mode(run - prm.B * kSetupCost) : 0;
        const int np = mode ? prm.split_NP : prm.NP;
        const int max_groups = mode == 0 ? prm.groups : (mode == 1 ? prm.beside_groups : prm.behind_groups);
        const int want = (int)((unsigned)(prm.Hkv * run) * (unsigned)prm.L / (unsigned)kMinVirtualTilesPerGroup);
        int n = want < 1 ? 1 : (want < max_groups ? want : max_groups);
        // A group count just above a multiple of the unit count is rounded down to it: with units of equal length
        // (one sequence, all heads) every unit is then cut into the same number of equal pieces and no cut falls
        // just behind a unit boundary.  Not worth more than 1/16 of the groups, but for short units of equal length:
        // those stay whole, one a group, because a cut and its merge cost more than the idle groups.
        const int over = n % units;
        if (n > units && (over * 16 <= n || (n < 2 * units && same && first_len <= kMaxWholeUnit))) n -= over;
        if (MAY_BE_SECOND) at[1] = mode == 1 ? prm.slot0 : 0;      // (a launch of a pair builds its table once, the second one)
        at[2] = n;
        at[3] = np;
      }
    }
    __syncthreads();
    const unsigned total = (unsigned)(prm.Hkv * cum[prm.B]) * (unsigned)prm.L;
    const int np = at[3];
    groups = at[2];
    // gs[k] = floor(total * k / groups) in 32-bit arithmetic: total = q * groups + r
    const unsigned q = total / (unsigned)groups, r = total % (unsigned)groups;
#pragma unroll 1
    for (int k = threadIdx.x; k <= kMaxGroups; k += kThreads)
      gs[k] = k <= groups ? (int)(k * q + (k * r) / (unsigned)groups) : (int)total;
    __syncthreads();
    sch.per_layer = prm.Hkv * cum[prm.B];
    sch.total = sch.per_layer * prm.L;
    // Downwards over the block index (see "Work split"); groups past the last used one get an empty range, and the CTAs
    // that are started first (on SMs the kernel in front does not use) get work.
    const int place = (int)(blockIdx.x / np);
    group = place < groups ? groups - 1 - place : place;
    g_begin = sch.group_start(group, groups);
    g_end = sch.group_start(group + 1, groups);
    if (!guess) break;
    if (warp == 0) prefetch_first();
    gdc_wait();
    bool changed = false;
    if (warp == 0 && at[0]) {
      const int b = items[2].b;
      const int S = prm.prefix_len[b], n = prm.n_nodes[b];
      __syncwarp();
      if (lane == 0) {
        items[2].S = S < 0 ? 0 : (S > prm.Scap ? prm.Scap : S);
        items[2].n = n < 0 ? 0 : (n > prm.Nmax ? prm.Nmax : n);
      }
    }
#pragma unroll 1
    for (int b = threadIdx.x; b < prm.B; b += kThreads) {
      int S = prm.prefix_len[b];
      S = S < 0 ? 0 : (S > prm.Scap ? prm.Scap : S);
      changed |= (S + kTileN - 1) / kTileN + prm.TT + kSetupCost != cum[b + 1] - cum[b];
    }
    guess = false;
    if (!__syncthreads_or(changed)) break;
    if (threadIdx.x == 0) at[0] = 0;
  }
  if (CL) __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  const int unit = CL ? (int)(blockIdx.x / cluster_size_x()) : 0;      // cluster kernel: (layer, sequence, KV head, pair)
  const int pair = CL ? unit % prm.NP : (int)(blockIdx.x % (MT == 2 ? at[3] : prm.NP));
  auto next_item = [&](int& g, Item& it) -> bool {
    if (CL) {                      // one item: this CTA's share of the key tiles of its cluster's unit (may be empty)
      if (g > 0) return false;
      g = 1;
      const int u = unit / prm.NP;
      it.hk = u % prm.Hkv;
      it.b = u / prm.Hkv % prm.B;
      it.layer = u / prm.Hkv / prm.B;
      const int S = __ldcg(prm.prefix_len + it.b), n = __ldcg(prm.n_nodes + it.b);      // (perhaps ahead of the wait: past L1)
      it.S = S < 0 ? 0 : (S > prm.Scap ? prm.Scap : S);
      it.n = n < 0 ? 0 : (n > prm.Nmax ? prm.Nmax : n);
      it.len = (it.S + kTileN - 1) / kTileN + prm.TT;
      const int size = (int)cluster_size_x(), rank = (int)(blockIdx.x % size);
      // (rounded up: where the shares are not equal the last CTA, whose tiles are the masked ones, has a smaller one; rounded down /
      // up, us a layer: two sequences of 3000 22.0 / 20.4, four of 500 ... 2000 19.6 / 18.1, one of 4000 15.6 / 14.6, of 1392 10.05 / 9.8,
      // the same with 60 nodes 15.55 / 15.7)
      it.j0 = (it.len * rank + size - 1) / size;
      it.j1 = (it.len * (rank + 1) + size - 1) / size;
      return it.j1 > it.j0;
    }
    if (!locate(g, it)) return false;
    const int S = prm.prefix_len[it.b], n = prm.n_nodes[it.b];
    it.S = S < 0 ? 0 : (S > prm.Scap ? prm.Scap : S);
    it.n = n < 0 ? 0 : (n > prm.Nmax ? prm.Nmax : n);
    return true;
  };

  constexpr uint32_t kIdescQK = instr_desc(kTileN, false);
  constexpr uint32_t kIdescPV = instr_desc(D, true);

  if (warp == 0) {
    // =========================================================== TMA producer
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    if (!*abort_flag && !(prm.debug & 1)) {        // the whole warp walks the items; one elected lane issues the copies
      int g = g_begin;
      Item it;
      uint32_t item_idx = 0, fill = 0;
      bool ok = true;
      Tracer tr;
      tr.init(lane == 0 ? trace : nullptr, 0);
      tr.mark(0);
      uint64_t kv_policy;      // the committed prefix is streamed once: first in line for eviction from L2
      asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(kv_policy));
      // Overlap with the kernel in front (programmatic dependent launch).  With the caller's promise (prm.early)
      // that this kernel leaves prefix_len, n_nodes, the block table and the committed rows alone, the first
      // prefix tiles are requested at once; Q and the tree's K/V - what a preceding kernel may still be
      // producing - wait for that kernel to finish.  Only then may the next kernel be scheduled, so that at
      // most two launches are in flight - three behind a pair that runs at the same time, whose second one lets the next
      // kernel go while the first may still be writing out, lse, status and the workspace.
      // status[] may still be written by the kernel in front (tree_build_mask stores it last), so a flag found
      // before the wait is kept here and raised after it.
      bool synced = false;
      int bad_page_b = -1;
      auto sync_with_predecessor = [&]() {
        if (!beside) gdc_wait();
        if (elect_one()) gdc_launch_dependents();
        if (bad_page_b >= 0 && lane == 0) atomicOr(prm.status + bad_page_b, TV_ST_BAD_INDEX);
        bad_page_b = -1;
        __syncwarp();
        synced = true;
      };
      auto publish = [&](const Item& x) {
        if (item_idx > 0 && !(prm.debug & 4)) ok = mbar_wait(bar(L::ITEM_READ), (item_idx - 1) & 1, abort_flag, wait_limit);
        if (ok && elect_one()) items[(item_idx & 1)] = x;
        __syncwarp();
      };
      auto load_q = [&]() {
        publish(it);
        if (ok && elect_one()) {
          mbar_expect_tx(bar(L::Q_FULL), MT * (D / 64) * prm.q_box_bytes);
#pragma unroll
          for (int t = 0; t < MT; ++t)
#pragma unroll
            for (int h = 0; h < D / 64; ++h)
              tma_load_5d(sbase + L::kQ + t * L::kTileBytes + h * L::kHalf, &map_q, bar(L::Q_FULL), h * 64,
                          it.hk * prm.G, (prm.tile0 + pair * MT + t) * prm.NPT, it.b, it.layer);
        }
        __syncwarp();
      };
      if (!prm.early || beside) sync_with_predecessor();
      bool have_first = !CL && !prm.early && at[0];
      if (have_first) {
        g = at[1];
        it = items[2];
      }
      while (ok && (have_first || next_item(g, it))) {
        have_first = false;
        ok = mbar_wait(bar(L::Q_EMPTY), (item_idx & 1) ^ 1, abort_flag, wait_limit);
        if (!ok) break;
        tr.mark(0x1000u | item_idx);
        bool q_pending = !synced;          // first item: Q goes out after the first prefix tiles
        if (!q_pending) load_q();
        if (!ok) break;
        // paged cache: the page of a prefix key tile comes from the block table, fetched one tile ahead of its use
        auto page_of = [&](int jj) -> int {
          if (!prm.block_table || jj >= it.len - prm.TT || jj >= it.j1) return 0;
          const int32_t* entry = prm.block_table + (size_t)it.b * prm.max_blocks + jj;
          int pg = CL ? __ldcg(entry) : *entry;
          if ((unsigned)pg >= (unsigned)prm.n_pages) {       // reported; the tile then reads page 0
            if (!synced) bad_page_b = it.b;                  // (only the first item can get here before the wait)
            else if (lane == 0) atomicOr(prm.status + it.b, TV_ST_BAD_INDEX);
            pg = 0;
          }
          return pg;
        };
        int page_next = page_of(it.j0);
        for (int j = it.j0; j < it.j1 && ok; ++j) {
          const int tt = j - (it.len - prm.TT);      // >= 0: index of the tree key tile
          const bool tree = tt >= 0;
          const int page = page_next;
          page_next = page_of(j + 1);
          const int row0 = prm.block_table ? 0 : j * kTileN;                                // of the tile in its slab
          const int slab = (prm.block_table ? page : it.b) * prm.Hkv + it.hk;               // (page or sequence, KV head)
#pragma unroll
          for (int kv = 0; kv < 2; ++kv) {
            const uint32_t slot = fill % L::kSlots, round = fill / L::kSlots;
            if (q_pending && (tree || fill >= (uint32_t)L::kSlots)) {      // before the first wait for a ring slot
              sync_with_predecessor();
              load_q();
              q_pending = false;
            }
            ok = mbar_wait(bar(L::KV_EMPTY + slot), (round & 1) ^ 1, abort_flag, wait_limit);
            if (!ok) break;
            tr.mark(0x2000u | (fill & 0xfffu));
            const uint32_t dst = sbase + L::kRing + slot * L::kTileBytes;
            if (elect_one()) {
              mbar_expect_tx(bar(L::KV_FULL + slot), L::kTileBytes);
#pragma unroll
              for (int h = 0; h < D / 64; ++h) {
                if (tree && prm.tree_in_cache)
                  tma_load_4d_hint(dst + h * L::kHalf, kv ? &map_vc : &map_kc, bar(L::KV_FULL + slot), h * 64,
                                   it.S + tt * kTileN, it.b * prm.Hkv + it.hk, it.layer, kv_policy);
                else if (tree)
                  tma_load_5d(dst + h * L::kHalf, kv ? &map_vt : &map_kt, bar(L::KV_FULL + slot), h * 64, it.hk, tt * kTileN, it.b,
                              it.layer);
                else
                  tma_load_4d_hint(dst + h * L::kHalf, kv ? &map_vc : &map_kc, bar(L::KV_FULL + slot), h * 64, row0, slab,
                                   it.layer, kv_policy);
              }
            }
            __syncwarp();
            ++fill;
          }
        }
        if (ok && q_pending) {
          sync_with_predecessor();
          load_q();
        }
        ++item_idx;
      }
      if (ok) ok = mbar_wait(bar(L::Q_EMPTY), (item_idx & 1) ^ 1, abort_flag, wait_limit);
      if (ok) {                            // no more items
        publish(Item{});
        if (ok && elect_one()) mbar_arrive(bar(L::Q_FULL));
      }
      if (!synced) sync_with_predecessor();        // a CTA without work still has to let the next kernel go
    } else {
      if (!beside) gdc_wait();
      if (elect_one()) gdc_launch_dependents();
    }
    if (CL) {
      __syncwarp();
      cluster_sync();
      cluster_sync_relaxed();
    }
  } else if (warp == 1) {
    // =========================================================== MMA issuer
    // One thread issues every MMA of the CTA.  S of a key tile is a full 128-key tile (N = 128: with 64-key
    // MMAs the Q operand is re-read from shared memory twice as often and the pipe runs at 2/3 of its rate).
    // A softmax warpgroup takes S into registers at once and P has columns of its own, so an S buffer is free again
    // a few hundred cycles after it was filled and the next S is ready before its warpgroup asks for it: the chain
    // hand-over -> PV -> QK^T -> wake-up of a row tile runs beside that row tile's softmax instead of in front of it
    // (32-layer shape: 1342 -> 1312 us a launch, power-capped 1583 -> 1540 us, against P overlaying its S).
    //   two row tiles:  S_0(j+1), O_0 += P_0(j) V(j), S_1(j+1), O_1 += P_1(j) V(j): each S as soon as the other row
    //     tile's S has been taken out of the buffer, each PV as soon as its P is there;
    //   KS:  S(j+2), O_w += P(j) V(j), w = j mod 2 the warpgroup of key tile j;
    //   one warpgroup (buffers alternate by key tile):  S(j+1), O += P(j) V(j).
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    if (!*abort_flag) {      // the whole warp walks the items; one elected lane issues
      uint32_t item_idx = 0, fill = 0, tj = 0;
      uint32_t done[2] = {0, 0};             // KS: key tiles of each warpgroup in earlier items
      bool ok = true;
      Tracer tr;
      tr.init(lane == 0 ? trace : nullptr, 1);
      tr.mark(0);
      // descriptor words: low = start address >> 4 | LBO field, high = SBO 1024 B | version 1 | 128-byte swizzle
      const uint32_t desc_hi = (uint32_t)(smem_desc(0, 0, 1024) >> 32);
      const uint32_t q_lo = (uint32_t)smem_desc(sbase + L::kQ, 16, 1024);   // K-major: LBO unused
      const uint32_t k_lo = (uint32_t)smem_desc(sbase + L::kRing, 16, 1024);
      const uint32_t v_lo = (uint32_t)smem_desc(sbase + L::kRing, L::kHalf, 1024);  // MN-major: LBO = next 64 columns
      constexpr int kHalf16 = L::kHalf >> 4, kTile16 = L::kTileBytes >> 4;
      // S = Q_t K^T for the 128 keys of the K tile in `slot`; idx: row tile, or parity of the key tile
      auto issue_qk = [&](int t, int idx, uint32_t slot) {
        const uint32_t qa = q_lo + t * kTile16, ka = k_lo + slot * kTile16;
        const uint32_t s_col = tmem + (idx ? L::kTmemS1 : L::kTmemS0);
        if (elect_one()) {
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks) {
            const uint32_t off = (ks / 4) * kHalf16 + (ks % 4) * 2;        // 16 columns = 32 bytes inside a swizzled row
            mma_ss_lohi(s_col, qa + off, ka + off, desc_hi, kIdescQK, ks > 0);
          }
          mma_commit(bar(L::S_FULL + idx));
        }
        __syncwarp();
      };
      // O_t += P V for the 128 keys of the V tile in `slot`.  The completion of a PV is known from the S that is
      // committed behind it (a commit of its own stalls the pipe for some 45 cycles), except where none follows.
      auto issue_pv = [&](int t, int idx, uint32_t slot, bool first_tile) {
        const uint32_t va = v_lo + slot * kTile16;
        if (elect_one()) {
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)            // 16 keys = 16 rows of 128 bytes = 8 packed P columns
            mma_ts_lohi(tmem + L::kTmemO0 + t * D, tmem + L::kTmemP0 + idx * 64 + ks * 8, va + ks * 128, desc_hi, kIdescPV,
                        (!first_tile || ks > 0) ? 1u : 0u);
          if (ONE) mma_commit(bar(L::O_DONE));
        }
        __syncwarp();
      };
      while (true) {
        ok = mbar_wait(bar(L::Q_FULL), item_idx & 1, abort_flag, wait_limit);
        if (!ok) break;
        const int nt = items[item_idx & 1].j1 - items[item_idx & 1].j0;
        if (nt == 0) break;
        tr.mark(0x1000u | item_idx);
        if (prm.debug & 4) {       // stream only: every tile of the item is released as soon as it has landed
#pragma unroll 1
          for (int f = 0; f < 2 * nt && ok; ++f) {
            const uint32_t ff = fill + f;
            ok = mbar_wait(bar(L::KV_FULL + ff % L::kSlots), (ff / L::kSlots) & 1, abort_flag, wait_limit);
            if (ok && elect_one()) mbar_arrive(bar(L::KV_EMPTY + ff % L::kSlots));
            __syncwarp();
          }
          if (elect_one()) mbar_arrive(bar(L::Q_EMPTY));
          __syncwarp();
          fill += 2 * nt;
          ++item_idx;
          continue;
        }
        if (KS) {
          auto phase = [&](int i) -> uint32_t { return (done[i & 1] + (i >> 1)) & 1u; };      // of key tile i's barriers
          auto next_s = [&](int i) {       // S of key tile i, i < nt; its buffer was last filled for tile i - 1 (or i - 2)
            const uint32_t f = fill + 2 * i, slot = f % L::kSlots;
            ok = mbar_wait(bar(L::KV_FULL + slot), (f / L::kSlots) & 1, abort_flag, wait_limit);
            const int before = L::kTmemS1 == L::kTmemS0 ? i - 1 : i - 2;
            if (ok && before >= 0) ok = mbar_wait(bar(L::S_FREE + (before & 1)), phase(before), abort_flag, wait_limit);
            if (!ok) return;
            tc_fence_after();
            issue_qk(0, i & 1, slot);
            if (elect_one()) {
              mma_commit(bar(L::KV_EMPTY + slot));
              if (i + 1 == nt) mma_commit(bar(L::Q_EMPTY));
            }
            __syncwarp();
          };
          // The S buffers are free: the P of every earlier key tile has been waited for, hence its S was taken.
          next_s(0);
          if (ok && nt > 1) next_s(1);
#pragma unroll 1
          for (int i = 0; i < nt && ok; ++i) {
            if (i + 2 < nt) next_s(i + 2);
            const uint32_t f = fill + 2 * i + 1, slot = f % L::kSlots;
            if (ok) ok = mbar_wait(bar(L::P_READY + (i & 1)), phase(i), abort_flag, wait_limit);
            if (ok) ok = mbar_wait(bar(L::KV_FULL + slot), (f / L::kSlots) & 1, abort_flag, wait_limit);
            if (!ok) break;
            tc_fence_after();
            tr.mark(0x4000u | (i & 0xfffu));
            issue_pv(i & 1, i & 1, slot, i < 2);
            if (elect_one()) {
              if (i + 3 == nt) mma_commit(bar(L::O_DONE));      // no S follows the PV behind the last key tile's predecessor
              if (i + 1 == nt) mma_commit(bar(L::ITEM_DONE));
              mma_commit(bar(L::KV_EMPTY + slot));
            }
            __syncwarp();
          }
          done[0] += (nt + 1) / 2;
          done[1] += nt / 2;
          fill += 2 * nt;
          ++item_idx;
          if (!ok) break;
          continue;
        }
        {
          // The S buffers are free: the P of every earlier key tile has been waited for, hence its S was taken.
          const uint32_t slot = fill % L::kSlots;
          ok = mbar_wait(bar(L::KV_FULL + slot), (fill / L::kSlots) & 1, abort_flag, wait_limit);
          if (!ok) break;
          tc_fence_after();
          if (ONE) {
            issue_qk(0, tj & 1, slot);
          } else {
            issue_qk(0, 0, slot);
            if (L::kTmemS1 == L::kTmemS0) ok = mbar_wait(bar(L::S_FREE + 0), tj & 1, abort_flag, wait_limit);
            if (!ok) break;
            tc_fence_after();
            issue_qk(1, 1, slot);
          }
          if (elect_one()) mma_commit(bar(L::KV_EMPTY + slot));
          if (nt == 1 && elect_one()) mma_commit(bar(L::Q_EMPTY));
        }
        for (int jt = 0; jt < nt && ok; ++jt, ++tj) {
          const uint32_t fv = fill + 2 * jt + 1, vslot = fv % L::kSlots;
          const uint32_t fk = fv + 1, kslot = fk % L::kSlots;
          const bool more = jt + 1 < nt;
          if (ONE) {
            const int buf = tj & 1;
            if (more) {
              ok = mbar_wait(bar(L::KV_FULL + kslot), (fk / L::kSlots) & 1, abort_flag, wait_limit);
              if (!ok) break;
              tc_fence_after();
              issue_qk(0, buf ^ 1, kslot);       // the P of the key tile before has been waited for: its S was taken
            }
            ok = mbar_wait(bar(L::P_READY + buf), (tj >> 1) & 1, abort_flag, wait_limit);
            if (ok) ok = mbar_wait(bar(L::KV_FULL + vslot), (fv / L::kSlots) & 1, abort_flag, wait_limit);
            if (!ok) break;
            tc_fence_after();
            issue_pv(0, buf, vslot, jt == 0);
            if (elect_one()) {
              if (!more) mma_commit(bar(L::ITEM_DONE));
              mma_commit(bar(L::KV_EMPTY + vslot));
              if (more) mma_commit(bar(L::KV_EMPTY + kslot));
              if (jt + 2 == nt) mma_commit(bar(L::Q_EMPTY));
            }
          } else {
#pragma unroll
            for (int t = 0; t < 2; ++t) {
              // S_t(j+1): the buffer was last filled for the other row tile (or, with two buffers, for S_t(j))
              if (more) {
                if (t == 0) {
                  ok = mbar_wait(bar(L::KV_FULL + kslot), (fk / L::kSlots) & 1, abort_flag, wait_limit);
                  if (!ok) break;
                }
                if (L::kTmemS1 == L::kTmemS0)
                  ok = mbar_wait(bar(L::S_FREE + (t ^ 1)), (t == 0 ? tj : tj + 1) & 1, abort_flag, wait_limit);
                else
                  ok = mbar_wait(bar(L::S_FREE + t), tj & 1, abort_flag, wait_limit);
                if (!ok) break;
                tc_fence_after();
                issue_qk(t, t, kslot);
                if (t == 1 && elect_one()) {
                  mma_commit(bar(L::KV_EMPTY + kslot));
                  if (jt + 2 == nt) mma_commit(bar(L::Q_EMPTY));
                }
                __syncwarp();
              }
              tr.mark(0x2000u | ((2 * tj + t) & 0xfffu));
              ok = mbar_wait(bar(L::P_READY + t), tj & 1, abort_flag, wait_limit);
              if (ok && t == 0) ok = mbar_wait(bar(L::KV_FULL + vslot), (fv / L::kSlots) & 1, abort_flag, wait_limit);
              if (!ok) break;
              tc_fence_after();
              tr.mark(0x4000u | ((2 * tj + t) & 0xfffu));
              issue_pv(t, t, vslot, jt == 0);
              if (!more && elect_one()) mma_commit(bar(L::ITEM_DONE + t));      // all MMAs of the item's row tile are done
            }
            if (!ok) break;
            // row tile 1 of the last key tile: no S follows its PV of the key tile before, so that is committed here
            if (elect_one()) {
              if (jt + 2 == nt) mma_commit(bar(L::O_DONE));
              mma_commit(bar(L::KV_EMPTY + vslot));
            }
          }
          __syncwarp();
        }
        fill += 2 * nt;
        ++item_idx;
      }
    }
    if (CL) {
      __syncwarp();
      cluster_sync();
      cluster_sync_relaxed();
    }
  } else if (warp >= 4) {
    // =========================================================== softmax / epilogue warpgroups
    // Register budget: the CTA starts with 168 registers per thread; warps 0-3 give up 96 each (168 -> 72) and
    // warps 4-11 take 48 each (168 -> 216).  4 x 96 = 8 x 48: the increase below can only complete once the
    // other warpgroup has released enough, so any other split has to keep 4 (168 - low) >= 8 (high - 168) or the
    // kernel never gets past this instruction.
    asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
    const int wg = (warp - 4) >> 2;                  // its row tile, or parity of its key tiles
    const int row = ((warp & 3) << 5) | lane;        // TMEM lane = row inside the tile
    const uint32_t lane_addr = (uint32_t)((warp & 3) << 5) << 16;
    // anc_bits, the workspace and the outputs may belong to the kernel in front until it is done
    if (!beside) gdc_wait();
    // in-cache layout: a tree that does not fit behind its prefix is reported, not read past the capacity (rows
    // past Scap arrive as zeros and the sequence's output is unspecified).  Raised after the wait: status[] may
    // be written by the kernel in front until then.
    if (prm.tree_in_cache && blockIdx.x == 0)
#pragma unroll 1
      for (int b = threadIdx.x - 128; b < prm.B; b += kThreads - 128) {
        int S = prm.prefix_len[b];
        S = S < 0 ? 0 : (S > prm.Scap ? prm.Scap : S);
        if (S + prm.n_nodes[b] > prm.Scap) atomicOr(prm.status + b, TV_ST_CAPACITY);
      }
    float m_fin = -INFINITY, l_fin = 0.f;            // cluster kernel: (m, l) of the row; no key tile: weight 0
    if (!(ONE && wg) && !*abort_flag && !(prm.debug & 4)) {
      uint32_t fill = 0, tj = 0, epi_phase = 0, item_cnt = 0;   // tj: key tiles of this warpgroup so far (all items)
      uint32_t to = 0;                                          // KS: those of the other one in earlier items
      uint32_t od_phase = 0;                                    // completions of O_DONE so far
      bool ok = true;
      Tracer tr;
      tr.init((threadIdx.x & 127) == 0 ? trace : nullptr, 2 + wg);
      tr.mark(0);
      // Rendezvous of the softmax warpgroups through an mbarrier, so that it is bounded like every other wait.
      // All 32 lanes wait together and agree on the outcome, so that the warp-wide TMEM instructions
      // below are never executed by a part of a warp.  The waits that every key tile has do not vote (LAZY): a lane whose
      // wait was abandoned notes it, goes on with whatever tensor memory holds, hands nothing on, and the vote on the row
      // maxima of the next tile, or the one behind the last tile, takes the whole warp out.  The lanes leave such a wait one by
      // one; the tensor-memory instruction behind it is the same for all of them whatever the wait returned (.aligned), and
      // waits until the last of them has come (.sync), so no barrier stands in front of it: one after each wait costs as much as
      // the votes and more (dependent layers of 16 sequences 509 -> 530 us, long context 261 -> 272).  (32-layer shape
      // 1254 -> 1240 us a launch, long context 226.7 -> 224.1, 4 sequences of 4096 41.3 -> 40.9.  The cluster kernel, a tile or two
      // per CTA, keeps the votes: 32 layers of one sequence 10.0 us a layer with them, 10.2 without.)
      constexpr bool LAZY = !CL;
      bool lane_ok = true;
      auto wwait = [&](uint32_t b_, uint32_t parity) -> bool {
        return __all_sync(0xffffffffu, mbar_wait(b_, parity, abort_flag, wait_limit));
      };
      auto tile_wait = [&](uint32_t b_, uint32_t parity) -> bool {
        return LAZY ? mbar_wait(b_, parity, abort_flag, wait_limit) : wwait(b_, parity);
      };
      auto leave = [&](bool waited) -> bool {      // true: leave the tile loop now
        if (LAZY) lane_ok = lane_ok && waited;
        else ok = waited;
        return !LAZY && !waited;
      };
      auto epi_sync = [&]() -> bool {
        mbar_arrive(bar(L::EPI));
        const bool r = wwait(bar(L::EPI), epi_phase & 1);
        ++epi_phase;
        return r;
      };
      while (true) {
        ok = wwait(bar(L::Q_FULL), item_cnt & 1);
        if (!ok) break;
        const Item it = items[item_cnt & 1];
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(bar(L::ITEM_READ));
          if (!CL && item_cnt == 0 && it.j0 == 0) mbar_arrive(bar(L::PIECE));      // nothing to announce
        }
        const int nt = it.j1 - it.j0;
        if (nt == 0) break;
        const int node = (prm.tile0 + pair * MT + (MT == 1 ? 0 : wg)) * prm.NPT + row / prm.G;
        const int gm = row % prm.G;
        const bool row_exists = row < prm.NPT * prm.G && node < prm.Nmax;
        const bool row_active = row_exists && node < it.n;
        // One row tile: a warp without an active row takes part in the barriers only.  (With two row tiles the test costs
        // the loop more than it saves: 32-layer shape 1296 -> 1314 us.)
        const bool warp_active = MT == 2 || __any_sync(0xffffffffu, row_active);
        // the row's ancestor words are wanted on the last tile(s): fetched into L1 now, not a round trip in front of that tile
        if (row_active) {
          const uint32_t* words = prm.anc_bits + ((size_t)it.b * prm.Nmax + node) * prm.W;
          asm volatile("prefetch.global.L1 [%0];" ::"l"(words));
          asm volatile("prefetch.global.L1 [%0];" ::"l"(words + prm.W - 1));
        }
        float m_used = -INFINITY;      // running reference maximum, in log2 units (score * scale * log2e)
        float l_sum = 0.f;
        const uint32_t o_addr_loop = tmem + lane_addr + L::kTmemO0 + wg * D;
        // key tiles below this index are full tiles of the committed prefix (no mask of any kind)
        const int j_full = min(it.S / kTileN, it.len - prm.TT);
        for (int jt = KS ? wg : 0; jt < nt && (LAZY || ok); jt += KS ? 2 : 1, ++tj) {
          const int j = it.j0 + jt;
          const bool masked = j >= j_full;
          uint32_t vis[4] = {0u, 0u, 0u, 0u};      // masked tiles: visible keys of this row
          if (masked) {
            const int tt = j - (it.len - prm.TT);      // >= 0: index of the tree key tile
            const bool tree = tt >= 0;
            const int valid_keys = tree ? max(0, min(kTileN, it.n - tt * kTileN)) : min(kTileN, it.S - j * kTileN);
            if (tree) {      // ancestor words of the node; none for a row without a node
              const uint32_t* words = prm.anc_bits + ((size_t)it.b * prm.Nmax + node) * prm.W + tt * 4;
#pragma unroll
              for (int w = 0; w < 4; ++w)
                if (row_active && tt * 4 + w < prm.W) vis[w] = words[w];
            } else {
#pragma unroll
              for (int w = 0; w < 4; ++w) {
                const int left = valid_keys - 32 * w;
                vis[w] = left >= 32 ? 0xffffffffu : (left > 0 ? (1u << left) - 1u : 0u);
              }
            }
            // ---- V rows past the valid keys may hold anything (stale cache rows, padded tree slots): zero
            // them so that 0 * NaN never reaches O.  Idempotent, so both warpgroups may do it.  Rows that lie
            // outside the tensor arrive as zeros from the copy itself: a tree tile whose tree is full (the
            // usual case) needs nothing.
            if (valid_keys < kTileN && !(tree && !prm.tree_in_cache && tt * kTileN + valid_keys >= prm.Nmax)) {
              const uint32_t f = fill + 2 * jt + 1, slot = f % L::kSlots;
              ok = wwait(bar(L::KV_FULL + slot), (f / L::kSlots) & 1);
              if (!ok) break;
              if (row >= valid_keys) {
                uint8_t* vrow = smem + L::kRing + slot * L::kTileBytes + row * 128;
#pragma unroll
                for (int h = 0; h < D / 64; ++h)
#pragma unroll
                  for (int c = 0; c < 8; ++c)
                    *reinterpret_cast<uint4*>(vrow + h * L::kHalf + c * 16) = make_uint4(0, 0, 0, 0);
              }
              fence_proxy_async_smem();
            }
          }
          // Completion of the PV of this warpgroup's key tile before this one (for its first key tile of an item: nothing to
          // wait for).  The pipe works in issue order.  Two row tiles: S_1(j) is issued behind O_0 += P_0(j-1) V, S_0(j+1)
          // behind O_1 += P_1(j-1) V; KS: S(j+1) behind O += P(j-2) V.  Where no such S follows, that PV has a commit of its
          // own (once per item).  One warpgroup: each PV has one.
          auto previous_pv_done = [&]() -> bool {
            if (KS) {
              if (jt < 2) return true;
              return jt + 1 < nt ? tile_wait(bar(L::S_FULL + (wg ^ 1)), (to + ((jt + 1) >> 1)) & 1u) : tile_wait(bar(L::O_DONE), od_phase & 1u);
            }
            if (jt == 0) return true;
            if (ONE) return tile_wait(bar(L::O_DONE), (tj - 1) & 1u);
            if (wg == 0) return tile_wait(bar(L::S_FULL + 1), tj & 1u);
            return jt + 1 < nt ? tile_wait(bar(L::S_FULL + 0), (tj + 1) & 1u) : tile_wait(bar(L::O_DONE), od_phase & 1u);
          };
          // S and P of this key tile: index = warpgroup, or parity of the key tile when there is one
          const int idx = ONE ? (int)(tj & 1u) : wg;
          tr.mark(0x0800u | (tj & 0x7ffu));
          if (leave(tile_wait(bar(L::S_FULL + idx), (ONE ? tj >> 1 : tj) & 1u))) break;
          tc_fence_after();
          tr.mark(0x1000u | (tj & 0xfffu));
          if (MT == 1 && !warp_active) {      // nothing of S is looked at; P and O keep whatever tensor memory holds there
            if (KS) {
              if (lane == 0) mbar_arrive(bar(L::S_FREE + wg));
              if (leave(previous_pv_done())) break;        // or this warp could arrive for P twice in one phase
            }
            if (LAZY) ok = __all_sync(0xffffffffu, lane_ok);
            if (!ok) break;
            if (lane == 0) mbar_arrive(bar(L::P_READY + idx));
            continue;
          }
          // ---- all 128 scores of the row into registers; the S buffer is free for the next S from here on
          uint32_t sall[128];
          {
            const uint32_t s_base = tmem + lane_addr + (idx ? L::kTmemS1 : L::kTmemS0);
            tmem_ld32(s_base, sall);
            tmem_ld32(s_base + 32, sall + 32);
            tmem_ld32(s_base + 64, sall + 64);
            tmem_ld32(s_base + 96, sall + 96);
            tmem_wait_ld();
            if (!ONE) {
              tc_fence_before();
              __syncwarp();
              if (lane == 0 && lane_ok) mbar_arrive(bar(L::S_FREE + wg));
            }
          }
          float* sa = reinterpret_cast<float*>(sall);
          if (masked) {
#pragma unroll
            for (int c = 0; c < 128; ++c)
              if (!((vis[c >> 5] >> (c & 31)) & 1u)) sa[c] = -INFINITY;
          }
          // ---- lazy rescale: the reference maximum moves only when it would grow by more than the threshold.  The
          // TMEM accesses are warp-wide (.sync.aligned), so the warp rescales as soon as one of its rows has to;
          // rows that keep their reference multiply by 1.
          {
            float mx[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) mx[c] = fmaxf(sa[c], sa[c + 4]);
#pragma unroll
            for (int c = 8; c < 128; c += 8)
#pragma unroll
              for (int k = 0; k < 4; ++k) mx[k] = fmax3(mx[k], sa[c + 2 * k], sa[c + 2 * k + 1]);
            const float mx2 = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * prm.scale_log2e;
            const bool moves = mx2 > m_used + kRescaleThreshold || (m_used == -INFINITY && mx2 > -INFINITY);
            if (__any_sync(0xffffffffu, moves || !lane_ok)) {
              if (LAZY) ok = __all_sync(0xffffffffu, lane_ok);
              if (!ok) break;
              const float alpha = (moves && m_used > -INFINITY) ? fast_exp2(m_used - mx2) : 1.f;
              if (moves) m_used = mx2;
              l_sum *= alpha;
              if (jt > (KS ? 1 : 0)) {
                if (leave(previous_pv_done())) break;
                tc_fence_after();
                // one 16-column group at a time: this runs while all 128 scores are held in registers
#pragma unroll 1
                for (int q = 0; q < D / 16; ++q) {
                  uint32_t o[16];
                  tmem_ld16(o_addr_loop + q * 16, o);
                  tmem_wait_ld();
#pragma unroll
                  for (int c = 0; c < 16; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * alpha);
                  tmem_st16(o_addr_loop + q * 16, o);
                }
              }
            }
          }
          // ---- P = exp2(s * c - m), row sum in fp32, P rounded to bf16.  All of it on the special-function unit: three pairs in
          // sixteen as a cubic on the FMA pipe were level in short runs and cost 1 % where the power limit sets the clock
          // (32-layer shape, seconds on end, on one board 1503 -> 1484 us a launch, on another 1462 -> 1441).
          uint32_t pkk[64];
          {
            const float2 c2 = make_float2(prm.scale_log2e, prm.scale_log2e);
            const float neg_m = (m_used == -INFINITY) ? 0.f : -m_used;       // no visible key yet: every P is 0
            const float2 nm2 = make_float2(neg_m, neg_m);
            float2 sum = make_float2(0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 64; ++i) {
              const float2 x = ffma2(make_float2(sa[2 * i], sa[2 * i + 1]), c2, nm2);
              const float2 pv = make_float2(fast_exp2(x.x), fast_exp2(x.y));
              sum = fadd2(sum, pv);
              pkk[i] = pack_bf16(pv.x, pv.y);
            }
            l_sum += sum.x + sum.y;
          }
          // ---- P into its columns once the PV that read them last is done; with one warpgroup (two P buffers in turn) that
          // was issued in front of the S this tile has waited for
          if (!ONE) {
            if (leave(previous_pv_done())) break;
            tc_fence_after();
          }
          {
            const uint32_t p_base = tmem + lane_addr + L::kTmemP0 + idx * 64;
            tmem_st32(p_base, pkk);
            tmem_st32(p_base + 32, pkk + 32);
          }
          tmem_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0 && lane_ok) mbar_arrive(bar(L::P_READY + idx));
          tr.mark(0x2000u | (tj & 0xfffu));
        }
        if (nt > (KS ? 2 : 1)) ++od_phase;
        to += (nt + wg) / 2;
        if (LAZY) ok = __all_sync(0xffffffffu, ok && lane_ok);
        if (!ok) break;
        // ---- epilogue of the item: wait for the last PV into this O buffer
        {
          // Wait for every MMA of the item.  This barrier completes once per item, so its phase is never
          // more than one away from the one waited for (a parity wait cannot tell phases two apart, which
          // is why the per-PV barrier O_DONE is not used here: both last PVs may or may not be done yet).
          // (Cluster kernel: of both row tiles, whose V the partials overwrite; the pipe works in issue order.)
          ok = wwait(bar(L::ITEM_DONE + (MT == 1 ? 0 : (CL ? 1 : wg))), item_cnt & 1);
          ++item_cnt;
          if (!ok) break;
          tc_fence_after();
          tr.mark(0x5000u);
          // KS: the two warpgroups have half of the keys each.  They exchange (m, l), and each of them finishes half
          // of the columns: O = e_0 O_0 + e_1 O_1 with e_w = 2^(m_w - max m); a warpgroup without keys has weight 0 (its O was
          // not written).
          float e_0 = 1.f, e_1 = 0.f;
          if (KS) {
            float2* xch = reinterpret_cast<float2*>(smem + L::kXch);
            xch[wg * 128 + row] = make_float2(m_used, l_sum);
            ok = epi_sync();
            if (!ok) break;
            const float2 a = xch[row], b = xch[128 + row];
            m_used = fmaxf(a.x, b.x);
            e_0 = a.x > -INFINITY ? fast_exp2(a.x - m_used) : a.y * 0.f;      // (0, or NaN for a row of NaN scores)
            e_1 = b.x > -INFINITY ? fast_exp2(b.x - m_used) : b.y * 0.f;
            l_sum = e_0 * a.y + e_1 * b.y;
          }
          constexpr int kGroups = KS ? D / 64 : D / 32;                // groups of 32 columns that this warpgroup finishes,
          const int q0 = KS ? wg * kGroups : 0;                        // from this one on
          const uint32_t o_addr = MT == 1 ? tmem + lane_addr + L::kTmemO0 : o_addr_loop;
          auto load_own = [&](int q, uint32_t* o) {
            tmem_ld32(o_addr + q * 32, o);
            if (KS) {
              uint32_t o1[32];
              tmem_ld32(o_addr + D + q * 32, o1);
              tmem_wait_ld();
#pragma unroll
              for (int c = 0; c < 32; ++c) {
                const float x = e_0 != 0.f ? e_0 * __uint_as_float(o[c]) : 0.f;
                o[c] = __float_as_uint(e_1 != 0.f ? fmaf(e_1, __uint_as_float(o1[c]), x) : x);
              }
            } else {
              tmem_wait_ld();
            }
          };
          const bool whole = (it.j0 == 0 && it.j1 == it.len);
          const int h = it.hk * prm.G + gm;
          tv_bf16* orow = prm.out + (size_t)it.layer * prm.out_layer_stride + (((size_t)it.b * prm.Nmax + node) * prm.Hq + h) * D;
          float* lse_p = prm.lse ? prm.lse + (((size_t)it.layer * prm.B + it.b) * prm.Hq + h) * prm.Nmax + node : nullptr;
          // Normalised bf16 output of this row, 32 columns at a time (one copy of the loop for every use: the
          // epilogue is cold code, fetched while the other CTAs still stream K/V).
          auto store_rows = [&](uint4* dst, size_t stride_u4, float inv, bool do_store, bool zero) {
#pragma unroll 1
            for (int q = q0; q < q0 + kGroups; ++q) {
              uint32_t o[32];
              load_own(q, o);
              if (do_store) {
                uint4 v[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                  v[c].x = pack_bf16(__uint_as_float(o[8 * c + 0]) * inv, __uint_as_float(o[8 * c + 1]) * inv);
                  v[c].y = pack_bf16(__uint_as_float(o[8 * c + 2]) * inv, __uint_as_float(o[8 * c + 3]) * inv);
                  v[c].z = pack_bf16(__uint_as_float(o[8 * c + 4]) * inv, __uint_as_float(o[8 * c + 5]) * inv);
                  v[c].w = pack_bf16(__uint_as_float(o[8 * c + 6]) * inv, __uint_as_float(o[8 * c + 7]) * inv);
                  if (zero) v[c] = make_uint4(0, 0, 0, 0);       // rows of padded nodes: O may hold anything
                }
                if (stride_u4 == 1 && prm.out_al32) {     // a row of the output: whole 32-byte sectors per store
                  st_global_32B(dst + q * 4, v[0], v[1]);
                  st_global_32B(dst + q * 4 + 2, v[2], v[3]);
                } else {
#pragma unroll
                  for (int c = 0; c < 4; ++c) dst[(size_t)(q * 4 + c) * stride_u4] = v[c];
                }
              }
            }
          };
          if (CL) {
            // ---- the partial of this CTA: O as it is, fp32 rows over the K/V ring (every MMA of the item is done, and a CTA
            // has one item), 16-byte pieces of a row swizzled by the row so that neither the writes nor the reads collide;
            // (m, l) beside them
            uint8_t* mine = smem + L::kRing + ((MT == 1 ? 0 : wg) * 128 + row) * (D * 4);
#pragma unroll 1
            for (int q = q0; q < q0 + kGroups; ++q) {
              uint32_t o[32];
              load_own(q, o);
#pragma unroll
              for (int c = 0; c < 8; ++c)
                *reinterpret_cast<uint4*>(mine + (((q * 8 + c) ^ (row & 7)) * 16)) =
                    make_uint4(o[4 * c], o[4 * c + 1], o[4 * c + 2], o[4 * c + 3]);
            }
            m_fin = m_used;
            l_fin = l_sum;
            tc_fence_before();
          } else if (whole) {
            const float inv = (row_active && m_used > -INFINITY) ? 1.f / l_sum : 0.f;
            store_rows(reinterpret_cast<uint4*>(orow), 1, inv, row_exists, !row_active);
            if (row_exists && lse_p && !(KS && wg))
              *lse_p = (row_active && m_used > -INFINITY) ? (m_used + log2f(l_sum)) / kLog2e : -INFINITY;
            tc_fence_before();
          } else {
            // ---- a piece of a unit.  The first piece (the one with the unit's first key tile, always the last thing
            // its CTA does) merges; every other piece leaves its normalised output O/l (bf16) and (m, l) in its CTA's
            // slot and raises its flag.  The merger waits (bounded) for the flags and combines
            // out = sum_p w_p O_p / sum_p w_p with w_p = l_p 2^(m_p - max m).  Every piece enters the sum as its
            // bf16-rounded normalised output, the merger's own included, in piece order with one fused multiply-add
            // per piece.  What bounds this is dependent round trips to L2 (some 2 K cycles each under load): a fixed
            // merger needs no ticket, its pieces are usually ready long before, and two pieces' whole rows are requested
            // at once beside their (m, l) (one piece at a time: 4 sequences of 4096, 128 nodes 42.6 -> 41.7 us, 32 of 1024
            // 50.6 -> 50.1 us a launch; three do not fit the registers).  The sum stays in tensor memory between two pairs.
            // The code is cold, so the columns go in two equal turns, each in the first half of the registers (unrolled
            // over all of them: +1 %, over a quarter of them: +1 %).
            // Partial outputs are stored column-group major, [slot][D/8][MT*128 rows][8 bf16]: a warp writes
            // and reads 512 contiguous bytes per instruction.
            constexpr int kRows = MT * 128;
            const int rr = (MT == 1 ? 0 : wg * 128) + row;
            // The unit's real tiles occupy [real0, uend) of the virtual tile space.  CTA groups k_first..k_last
            // hold them, one piece each (a group between the two lies wholly inside the unit), and this CTA's
            // group is one of them: two short walks over the cut table find both ends.
            const int np = at[3], place = (int)(blockIdx.x / np), groups = at[2];      // (read here: registers are short in the loop)
            const int group = place < groups ? groups - 1 - place : place;
            const int slot0 = MAY_BE_SECOND && prm.split_tiles > 0 ? at[1] : 0;
            const int real0 = it.layer * (prm.Hkv * cum[prm.B]) + prm.Hkv * cum[it.b] + it.hk * (it.len + kSetupCost) + kSetupCost;
            const int uend = real0 + it.len;
            int k_first = group, k_last = group;
            while (gs[k_first] > real0) --k_first;
            while (gs[k_last + 1] < uend) ++k_last;
            const int n_other = k_last - k_first;
            const float inv_own = (row_active && m_used > -INFINITY) ? 1.f / l_sum : 0.f;
            if (group != k_first) {
              const size_t slot = (size_t)slot0 + (size_t)group * np + pair;
              uint4* po = reinterpret_cast<uint4*>(prm.part_o) + slot * (D / 8) * kRows;
              float* pml = prm.part_ml + slot * 2 * kRows;
              if (row_active && !(KS && wg)) {
                pml[rr] = m_used;
                pml[kRows + rr] = l_sum;
              }
              store_rows(po + rr, kRows, inv_own, row_active, false);
              tc_fence_before();
              // Warp 2 announces the piece: the release behind these stores (a round trip to L2) and the wait for the other
              // warps' stores are not in front of this warp's next item (32 sequences of 1024, one layer: 51.3 -> 50.6 us; 4 of
              // 4096, 128 nodes: 43.5 -> 42.6 us).
              if (threadIdx.x == 128 && !(prm.debug & 2))      // (debug bit 1: the piece is never announced)
                *announce = reinterpret_cast<unsigned long long>(prm.flags + slot);
              tr.mark(0x6000u);
              __syncwarp();
              if (lane == 0) mbar_arrive(bar(L::PIECE));
            } else {
              if (warp == 4) {
                // Wait until the other pieces have published their partials, a lane for each.  A flag per slot, written once
                // with a release and polled with an acquire: with a counter for all later pieces (a read, a compare-and-swap, a
                // full fence on either side) the last partial was seen 3 us after its last store, now 2 (us a launch, 8 KV heads:
                // 8 sequences of 1024 ... 8192 46.9 -> 45.7, 4 of 500 ... 16000 50.7 -> 48.4; 64-wide heads, one row tile, 16 of
                // 8000 59.8 -> 55.9).
#pragma unroll 1
                for (int i = 1 + lane; i <= n_other; i += 32) {
                  unsigned long long* flag = prm.flags + slot0 + (size_t)(k_first + i) * np + pair;
                  const unsigned long long t0 = globaltimer_ns();
                  while (ld_acquire(flag) != prm.epoch) {
                    if (*abort_flag || globaltimer_ns() - t0 > wait_limit) {
                      *abort_flag = 1;
                      break;
                    }
                  }
                  // nobody touches the flag again in this launch.  Clearing it lets the same launch be replayed with the
                  // same epoch (a captured CUDA graph) and find it unused.
                  *reinterpret_cast<volatile unsigned long long*>(flag) = 0ull;
                }
                __syncwarp();
              }
              ok = epi_sync();
              if (!ok || *abort_flag) { ok = false; break; }
              tr.mark(0x7001u);
              // Loads are issued by every thread (row rr always lies inside a slot; rows that are not active read stale
              // bytes and are masked by selects): no thread-divergent branch sits between the warp-wide TMEM ops.
              // (64-wide heads with many pieces a unit: 32-bit slots 48.3 -> 47.8 us a call; the others keep 64 bits, level or 1 %)
              using Slot = std::conditional_t<D == 64, uint32_t, size_t>;
              auto slot_of = [&](int i) -> Slot { return (Slot)slot0 + (Slot)(k_first + i) * (Slot)np + (Slot)pair; };       // i-th other piece, i >= 1
              auto ml_of = [&](int i) -> const float* { return prm.part_ml + slot_of(i) * 2 * kRows + rr; };
              auto o_of = [&](int i) -> const uint4* { return reinterpret_cast<const uint4*>(prm.part_o) + slot_of(i) * (D / 8) * kRows + rr; };
              // two pieces at a time: (m, l) of the row and the columns of this warpgroup
              float m_a = 0.f, l_a = 0.f, m_b = 0.f, l_b = 0.f;
              constexpr int kTurn = kGroups > 2 ? 2 : kGroups;      // groups of 32 columns in a turn
              uint4 va[kGroups * 4], vb[kGroups * 4];
              auto fetch = [&](int i) {
                m_a = __ldcg(ml_of(i));
                l_a = __ldcg(ml_of(i) + kRows);
                const uint4* a_o = o_of(i) + (size_t)q0 * 4 * kRows;
#pragma unroll
                for (int c = 0; c < kGroups * 4; ++c) va[c] = __ldcg(a_o + (size_t)c * kRows);
                m_b = -INFINITY;
                l_b = 0.f;
                if (i < n_other) {
                  m_b = __ldcg(ml_of(i + 1));
                  l_b = __ldcg(ml_of(i + 1) + kRows);
                  const uint4* b_o = o_of(i + 1) + (size_t)q0 * 4 * kRows;
#pragma unroll
                  for (int c = 0; c < kGroups * 4; ++c) vb[c] = __ldcg(b_o + (size_t)c * kRows);
                } else {
#pragma unroll
                  for (int c = 0; c < kGroups * 4; ++c) vb[c] = make_uint4(0, 0, 0, 0);
                }
              };
              fetch(1);
              float mm = fmaxf(m_used, fmaxf(m_a, m_b));
#pragma unroll 4
              for (int i = 3; i <= n_other; ++i) mm = fmaxf(mm, __ldcg(ml_of(i)));
              const float mref = mm == -INFINITY ? 0.f : mm;
              const float w_own = l_sum * fast_exp2(m_used - mref);
              float w_a = l_a * fast_exp2(m_a - mref), w_b = l_b * fast_exp2(m_b - mref), lt = w_own + w_a + w_b;
#pragma unroll 4
              for (int i = 3; i <= n_other; ++i) lt += __ldcg(ml_of(i) + kRows) * fast_exp2(__ldcg(ml_of(i)) - mref);
              const bool any_key = row_active && (mm > -INFINITY || lt != lt);      // (a row of NaN scores stays NaN)
              const float inv = any_key ? 1.f / lt : 0.f;
              const float2 own2 = make_float2(w_own, w_own), inv_own2 = make_float2(inv_own, inv_own), inv2 = make_float2(inv, inv);
#pragma unroll 1
              for (int i = 1; i <= n_other; i += 2) {
                const float2 wa2 = make_float2(w_a, w_a), wb2 = make_float2(w_b, w_b);
                const bool more = i + 2 <= n_other;
#pragma unroll 1
                for (int xo = 0; xo < kGroups; xo += kTurn) {
#pragma unroll
                  for (int x = 0; x < kTurn; ++x) {
                    const int q = q0 + xo + x;
                    uint32_t o[32];
                    if (i == 1) {
                      load_own(q, o);
                    } else {
                      tmem_ld32(o_addr + q * 32, o);
                      tmem_wait_ld();
                    }
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                      float2 acc = make_float2(__uint_as_float(o[2 * c]), __uint_as_float(o[2 * c + 1]));
                      if (i == 1) {
                        const float2 t = __fmul2_rn(acc, inv_own2);
                        const uint32_t own = pack_bf16(t.x, t.y);
                        acc = __fmul2_rn(own2, make_float2(__uint_as_float(own << 16), __uint_as_float(own & 0xffff0000u)));
                      }
                      const uint4 aa = va[x * 4 + (c >> 2)], bb = vb[x * 4 + (c >> 2)];
                      const uint32_t pa = (c & 3) == 0 ? aa.x : ((c & 3) == 1 ? aa.y : ((c & 3) == 2 ? aa.z : aa.w));
                      const uint32_t pb = (c & 3) == 0 ? bb.x : ((c & 3) == 1 ? bb.y : ((c & 3) == 2 ? bb.z : bb.w));
                      acc = ffma2(wa2, make_float2(__uint_as_float(pa << 16), __uint_as_float(pa & 0xffff0000u)), acc);
                      acc = ffma2(wb2, make_float2(__uint_as_float(pb << 16), __uint_as_float(pb & 0xffff0000u)), acc);
                      o[2 * c] = __float_as_uint(acc.x);
                      o[2 * c + 1] = __float_as_uint(acc.y);
                    }
                    if (more) {
                      tmem_st32(o_addr + q * 32, o);
                    } else if (row_exists) {
                      uint4 r[4];
#pragma unroll
                      for (int c = 0; c < 4; ++c) {
                        uint32_t pk4[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                          const float2 t = __fmul2_rn(make_float2(__uint_as_float(o[8 * c + 2 * e]), __uint_as_float(o[8 * c + 2 * e + 1])), inv2);
                          pk4[e] = any_key ? pack_bf16(t.x, t.y) : 0u;
                        }
                        r[c] = make_uint4(pk4[0], pk4[1], pk4[2], pk4[3]);
                      }
                      if (prm.out_al32) {
                        st_global_32B(orow + q * 32, r[0], r[1]);
                        st_global_32B(orow + q * 32 + 16, r[2], r[3]);
                      } else {
#pragma unroll
                        for (int c = 0; c < 4; ++c) *reinterpret_cast<uint4*>(orow + q * 32 + c * 8) = r[c];
                      }
                    }
                  }
                  if (kTurn < kGroups) {
#pragma unroll
                    for (int c = 0; c + 4 * kTurn < kGroups * 4; ++c) {
                      va[c] = va[c + 4 * kTurn];
                      vb[c] = vb[c + 4 * kTurn];
                    }
                  }
                }
                if (more) {
                  tmem_wait_st();
                  fetch(i + 2);
                  w_a = l_a * fast_exp2(m_a - mref);
                  w_b = l_b * fast_exp2(m_b - mref);
                }
              }
              if (row_exists && lse_p && !(KS && wg)) *lse_p = any_key && mm > -INFINITY ? (mm + log2f(lt)) / kLog2e : -INFINITY;
              tc_fence_before();
            }
          }
        }
        if (KS) {      // both warpgroups have read both O: the next item may write them
          ok = epi_sync();
          if (!ok) break;
        }
        tr.mark(0x8000u);
        fill += 2 * nt;
      }
    }
    if (CL) {
      // ---- merge of the cluster's partials: each CTA takes a share of the rows, 16 bytes of a row per thread; out =
      // sum_p w_p O_p / sum_p w_p l_p, w_p = 2^(m_p - max m), in rank order, all in fp32.  A piece without keys has weight 0
      // (its rows were not written and are not used).  With normalised bf16 partials outputs were further from 64 bits than
      // those of units in one piece: relative error 2.70e-3 to 2.87e-3, now 2.12e-3 to 2.34e-3.  A layer of one sequence, 8 KV
      // heads, 1392 rows: 17 nodes 10.1 us as before, 60 nodes 14.2 -> 15.3 (what is read from other CTAs sets the pace there; the
      // two halves of a row go to the columns c and D/2 + c, so that eight lanes never meet in a bank).
      if (MT == 2 || wg == 0) *reinterpret_cast<float2*>(smem + L::kMl + (wg * 128 + row) * 8) = make_float2(m_fin, l_fin);
      const int size = (int)cluster_size_x(), rank = (int)(blockIdx.x % size);
      const int u = unit / prm.NP, hk = u % prm.Hkv, b = u / prm.Hkv % prm.B, layer = u / prm.Hkv / prm.B;
      int n = prm.n_nodes[b];                                      // (on its way while the barrier is waited for)
      __syncwarp();
      cluster_sync();
      if (!*abort_flag && !(prm.debug & 4)) {
        constexpr int kVecs = D / 8;
        n = n < 0 ? 0 : (n > prm.Nmax ? prm.Nmax : n);
        const int node0 = (prm.tile0 + pair * MT) * prm.NPT;
        const int nodes = max(0, min(MT * prm.NPT, prm.Nmax - node0));      // nodes of this pair of row tiles
        const int total = nodes * prm.G * kVecs;
        const int share = (total + size - 1) / size, x_end = min(total, (rank + 1) * share);
        for (int x = rank * share + (int)threadIdx.x - 128; x < x_end; x += 256) {
          const int r = x / kVecs, c = x - r * kVecs;              // row among the existing ones, piece of the row
          const int node_l = r / prm.G, gm = r - node_l * prm.G;
          const int t = MT == 2 && node_l >= prm.NPT ? 1 : 0, in_tile = (node_l - t * prm.NPT) * prm.G + gm;
          const uint32_t ml = sbase + L::kMl + (t * 128 + in_tile) * 8;
          const uint32_t at_lo = sbase + L::kRing + (t * 128 + in_tile) * (D * 4) + ((c ^ (in_tile & 7)) * 16), at_hi = at_lo + kVecs * 16;
          float pm[kMaxCluster], l[kMaxCluster];
          uint4 v[kMaxCluster], u[kMaxCluster];
#pragma unroll
          for (int k = 0; k < kMaxCluster; ++k)
            if (k < size) {
              const float2 p = ld_peer_8B(peer_smem(ml, k));
              pm[k] = p.x;
              l[k] = p.y;
              v[k] = ld_peer_16B(peer_smem(at_lo, k));
              u[k] = ld_peer_16B(peer_smem(at_hi, k));
            }
          float mm = -INFINITY;
#pragma unroll
          for (int k = 0; k < kMaxCluster; ++k)
            if (k < size) mm = fmaxf(mm, pm[k]);
          float lt = 0.f, acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int k = 0; k < kMaxCluster; ++k)
            if (k < size) {
              if (pm[k] > -INFINITY || l[k] != l[k]) {      // (a row of NaN scores stays NaN)
                const float wk = fast_exp2(pm[k] - mm);
                lt = fmaf(wk, l[k], lt);
                const uint32_t e[8] = {v[k].x, v[k].y, v[k].z, v[k].w, u[k].x, u[k].y, u[k].z, u[k].w};
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[i] = fmaf(wk, __uint_as_float(e[i]), acc[i]);
              }
            }
          const int node = node0 + node_l, h = hk * prm.G + gm;
          const bool any_key = node < n && (mm > -INFINITY || lt != lt);
          const float inv = any_key ? 1.f / lt : 0.f;
          uint2 lo = make_uint2(pack_bf16(acc[0] * inv, acc[1] * inv), pack_bf16(acc[2] * inv, acc[3] * inv));
          uint2 hi = make_uint2(pack_bf16(acc[4] * inv, acc[5] * inv), pack_bf16(acc[6] * inv, acc[7] * inv));
          if (!any_key) lo = hi = make_uint2(0, 0);
          tv_bf16* dst = prm.out + (size_t)layer * prm.out_layer_stride + (((size_t)b * prm.Nmax + node) * prm.Hq + h) * D + c * 4;
          *reinterpret_cast<uint2*>(dst) = lo;
          *reinterpret_cast<uint2*>(dst + D / 2) = hi;
          if (c == 0 && prm.lse)
            prm.lse[(((size_t)layer * prm.B + b) * prm.Hq + h) * prm.Nmax + node] =
                any_key && mm > -INFINITY ? (mm + log2f(lt)) / kLog2e : -INFINITY;
        }
      }
      __syncwarp();
      cluster_sync_relaxed();    // nobody leaves while its shared memory may still be read
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    // (in front of gdc_launch_dependents in warp 0, where nothing could miss it, the release and its code cost 0.2 to 0.9 us a launch)
    if (MT == 2 && !CL && threadIdx.x == 96 && prm.passed && blockIdx.x == 0 && !(prm.debug & 32)) {
      gdc_wait();
      st_release(prm.passed, prm.passed_tag);
    }
    // Only the first item of a CTA can be a piece whose partials another CTA merges.  Warp 2 waits for every softmax warp to
    // have stored its part (or to have seen that there is none), and then raises the flag.
    if (!CL && warp == 2 && !*abort_flag && !(prm.debug & 4) && mbar_wait(bar(L::PIECE), 0, abort_flag, wait_limit) && lane == 0 &&
        *announce != 0)
      st_release(reinterpret_cast<unsigned long long*>(*announce), prm.epoch);
    if (CL) {
      cluster_sync();
      cluster_sync_relaxed();
    }
  }

  // ---- teardown
  if (MAY_BE_SECOND && prm.split_tiles > 0) end_pair();
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // give copies that may still be in flight time to land before the shared memory is released
    const unsigned long long t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) {
    }
    if (threadIdx.x == 0)
#pragma unroll 1
      for (int b = 0; b < prm.B; ++b) atomicOr(&prm.status[b], TV_ST_TIMEOUT);
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

bool encode_map(CUtensorMap* m, const void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides_bytes,
                const cuuint32_t* box) {
  cuuint32_t ones[5] = {1, 1, 1, 1, 1};
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), dims, strides_bytes, box, ones,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct Geometry {
  int G, NPT, n_row_tiles, MT, NP, sms, groups, grid;
  size_t ml_off, flags_off, o_off, layers_off, per_layer, total;
};

constexpr int kWorkspaceLayers = 32;    // layers in one launch with the workspace of tv_attn_workspace_bytes

Geometry geometry(int B, int Nmax, int Hq, int Hkv, int d, bool query_device) {
  Geometry g{};
  g.G = Hq / Hkv;
  g.NPT = kTileM / g.G;
  g.n_row_tiles = (Nmax + g.NPT - 1) / g.NPT;
  g.MT = g.n_row_tiles > 1 ? 2 : 1;
  g.NP = (g.n_row_tiles + g.MT - 1) / g.MT;
  g.sms = query_device ? tv::sm_count() : 148;
  g.groups = g.sms / g.NP > 0 ? g.sms / g.NP : 1;
  g.grid = g.groups * g.NP;
  // workspace: (m,l) pairs and partial O, both with 160 slots (one per CTA) whatever the device, the flags of all slots in the O room
  // of the first one: the pieces of CTA group 0 are all the first of their unit, which leave no partial; then a
  // stretch per layer, none of which is used: how many there are bounds the layers that share a launch
  constexpr size_t kSlotsMax = 160;
  static_assert(kSlotsMax == kMaxGroups && (2 * kSlotsMax + 1) * sizeof(unsigned long long) <= 128 * 64 * sizeof(tv_bf16),
                "the flags, two for a slot of two row tiles, and the one between two launches fit a slot of one row tile, 64-wide");
  const size_t ml_bytes = (size_t)g.MT * 128 * 2 * sizeof(float);
  g.ml_off = 0;
  g.o_off = (kSlotsMax * ml_bytes + 255) & ~size_t(255);
  g.flags_off = g.o_off;
  g.layers_off = (g.o_off + kSlotsMax * g.MT * 128 * d * sizeof(tv_bf16) + 255) & ~size_t(255);
  g.per_layer = ((size_t)B * Hkv * g.NP * 2 * sizeof(unsigned long long) + 255) & ~size_t(255);
  g.total = g.layers_off + kWorkspaceLayers * g.per_layer;
  return g;
}

std::atomic<unsigned long long*> g_trace{nullptr};

// Tag of a call in its workspace flags (never repeated within a process, never 0): the only state the
// library keeps for this entry point besides the cached driver entry point and device attributes.
unsigned long long next_epoch() {
  static std::atomic<unsigned long long> ctr{
      (unsigned long long)std::chrono::steady_clock::now().time_since_epoch().count() * 2654435761ull};
  return ctr.fetch_add(1, std::memory_order_relaxed) | 1ull << 63;
}

// Allows the kernel its shared memory, once per device.
template <int D, int MT, bool CL>
cudaError_t configure(int dev) {
  static std::atomic<bool> configured[64];
  if (dev >= 0 && dev < 64 && configured[dev].load(std::memory_order_acquire)) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(tree_attn_kernel<D, MT, CL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             SmemLayout<D, MT>::kTotal);
  if (e == cudaSuccess && dev >= 0 && dev < 64) configured[dev].store(true, std::memory_order_release);
  return e;
}

struct LaunchConfig {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  LaunchConfig(unsigned grid, unsigned cluster, size_t smem, cudaStream_t s) {
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    // Programmatic stream serialisation: this launch may be scheduled while the kernel in front is still
    // running (if that kernel allows it); the kernel itself waits before it touches anything that kernel writes.
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
  }
};

// Clusters of 2, 4 and 8 CTAs that the device runs at the same time (asked once per device and size; 0: none).
template <int D, int MT>
int clusters_at_once(int dev, int log2_size) {
  static std::atomic<int> known[64][4];          // value + 1
  if (dev < 0 || dev >= 64) return 0;
  int v = known[dev][log2_size].load(std::memory_order_relaxed);
  if (v == 0) {
    int n = 0;
    const unsigned size = 1u << log2_size;
    LaunchConfig lc(size, size, SmemLayout<D, MT>::kTotal, nullptr);
    if (configure<D, MT, true>(dev) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, tree_attn_kernel<D, MT, true>, &lc.cfg) != cudaSuccess)
      n = 0;
    v = n + 1;
    known[dev][log2_size].store(v, std::memory_order_relaxed);
  }
  return v - 1;
}

// CTAs per unit for the cluster kernel, 1: the even cut over all CTAs.  `units`: (layer, sequence, KV head, row-tile pair);
// `tiles`: key tiles of the longest unit the call can have (the lengths themselves are on the device).  The largest
// cluster for which all units run at once; then the rule weighs a CTA's share of the tiles against the share of the even
// cut plus what that pays beyond its tiles: flags and partials through L2 (about six tiles' time) and the serial merge of
// a unit's pieces (about one tile's each).  Measured (32 query heads, d = 128; cluster / even cut, us a launch): 8 KV
// heads, 17 nodes, one sequence of 200: 8.9 / 15.6, 1392: 10.9 / 18.3, 8192: 18.3 / 31.1, 32768: 44 / 54; 60 nodes, 65536:
// 110 / 89; 32 KV heads, 60 nodes, 2048: 14.2 / 20.6, 32768: 85 / 90.  Several sequences may differ in length, which only
// the even cut can level: they take the cluster kernel only while a share is short (4 sequences of 2048 ... 256: 13.9 /
// 20.1, of 4096 ... 512: 18.5 / 24.4; four equal ones of 4096: 19.0 / 25.0).
template <int D, int MT>
int cluster_size(long long units, int B, int tiles, int sms) {
  if (units * 2 > sms) return 1;
  int dev = 0;
  cudaGetDevice(&dev);
  for (int lg = 3; lg >= 1; --lg) {
    const int size = 1 << lg;
    if (units * size > sms || (size > 2 && size / 2 >= tiles) || clusters_at_once<D, MT>(dev, lg) < units) continue;
    const int share = (tiles + size - 1) / size;
    if (B > 1) return share <= 12 ? size : 1;
    return share <= units * tiles / sms + 6 + sms / units ? size : 1;
  }
  return 1;
}

// cluster = 1: the even cut
template <int D, int MT, bool CL>
cudaError_t launch_kernel(unsigned grid, unsigned cluster, const CUtensorMap* maps, const AttnParams& prm, cudaStream_t s) {
  int dev = 0;
  cudaGetDevice(&dev);
  const cudaError_t e = configure<D, MT, CL>(dev);
  if (e != cudaSuccess) return e;
  LaunchConfig lc(grid, cluster, SmemLayout<D, MT>::kTotal, s);
  return cudaLaunchKernelEx(&lc.cfg, tree_attn_kernel<D, MT, CL>, maps[0], maps[1], maps[2], maps[3], maps[4], prm);
}

template <int D, int MT>
cudaError_t launch(const Geometry& g, const CUtensorMap* maps, AttnParams prm, cudaStream_t s) {
  const long long units = (long long)prm.L * prm.B * prm.Hkv;
  const int tiles = (prm.Scap + kTileN - 1) / kTileN + prm.TT;
  // (the test entries exercise the waits of the even cut, or with bit 4 those of the kernel that the call takes)
  const int cluster = prm.debug && !(prm.debug & 16) ? 1 : cluster_size<D, MT>(units * prm.NP, prm.B, tiles, g.sms);
  tv::count_launches(1);
  if (cluster > 1) return launch_kernel<D, MT, true>((unsigned)(units * prm.NP * cluster), (unsigned)cluster, maps, prm, s);
  // An odd number of row tiles leaves the last CTA of a group with an empty one, as expensive as a full one in the time
  // its group takes.  Where the work is long the last row tile gets a launch of its own, one row tile per CTA, beside the one with
  // the others or behind it (see odd_row_tile).  Only the capacity of the cache is known here: where it allows
  // long work both launches are made, and both go by the lengths on the device (short work: the front launch takes all row tiles,
  // the other finds nothing to do, some 2 us).
  if (MT == 2 && g.n_row_tiles % 2 == 1 && units * tiles >= (long long)kSplitTilesPerSm * g.sms) {
    const tv::OddRowTile odd = tv::odd_row_tile(g.sms, g.n_row_tiles, D);
    if (odd.behind_groups > 0) {
      prm.split_tiles = odd.split_from * g.sms;
      prm.behind_tiles = odd.behind_from * g.sms;
      prm.passed = prm.flags + 2 * kMaxGroups;
      prm.passed_tag = prm.epoch;
      AttnParams front = prm;
      front.split_NP = g.n_row_tiles / 2;
      front.beside_groups = odd.beside_groups;
      front.behind_groups = odd.behind_groups;
      const int ctas = front.behind_groups * front.split_NP;      // (never fewer than beside the other launch)
      const cudaError_t e = launch_kernel<D, MT, false>((unsigned)(ctas > g.grid ? ctas : g.grid), 1, maps, front, s);
      if (e != cudaSuccess) return e;
      tv::count_launches(1);
      prm.tile0 = g.n_row_tiles - 1;
      prm.NP = prm.split_NP = 1;
      prm.beside_groups = odd.odd_groups;
      prm.behind_groups = g.sms;
      prm.slot0 = 2 * odd.beside_groups * front.split_NP;         // behind those of the first launch, which are twice as long
      prm.early = 1;          // behind a launch of this very call the inputs are stable
      prm.epoch = next_epoch();
      return launch_kernel<D, 1, false>((unsigned)g.sms, 1, maps, prm, s);
    }
  }
  return launch_kernel<D, MT, false>((unsigned)g.grid, 1, maps, prm, s);
}

struct AttnOptions {
  bool early = false;                              // TV_ATTN_STABLE_INPUTS was promised
  unsigned long long wait_limit_ns = kWaitLimitNs;
  int debug = 0;
};

// Layer strides of a call (elements); a single-layer call has L = 1 and strides that are never used.
struct LayerStrides {
  int64_t q = 0, cache = 0, tree = 0, out = 0;
};

// One launch over L layers.  Both layouts of the committed cache: contiguous [L,B,Hkv,Scap,d]
// (block_table == nullptr) or, for one layer, pages [n_pages,Hkv,128,d] named by block_table[B,max_blocks]
// (then Scap = 128 * max_blocks).  The layer is the outermost coordinate of every tensor map.
int attn_launch(const tv_bf16* q, const tv_bf16* k_cache, const tv_bf16* v_cache,
                const int32_t* block_table, int n_pages, int max_blocks,
                const tv_bf16* k_tree, const tv_bf16* v_tree, bool in_cache,
                const int32_t* prefix_len, const int32_t* n_nodes, const uint32_t* anc_bits,
                int L, const LayerStrides& ls, int B, int Nmax, int Hq, int Hkv, int d, int Scap, float scale,
                tv_bf16* out, float* lse, void* workspace, int32_t* status, const AttnOptions& opt, cudaStream_t s) {
  const Geometry g = geometry(B, Nmax, Hq, Hkv, d, true);
  CUtensorMap maps[5];
  {
    const cuuint64_t e = 2;
    const cuuint64_t layers = (cuuint64_t)L;
    // a stride of a dimension of extent 1 is never used, but has to be a valid one
    const cuuint64_t q_ls = L > 1 ? (cuuint64_t)ls.q * e : (cuuint64_t)B * Nmax * Hq * d * e;
    const cuuint64_t t_ls = L > 1 ? (cuuint64_t)ls.tree * e : (cuuint64_t)B * Nmax * Hkv * d * e;
    cuuint64_t qd[5] = {(cuuint64_t)d, (cuuint64_t)Hq, (cuuint64_t)Nmax, (cuuint64_t)B, layers};
    cuuint64_t qs[4] = {(cuuint64_t)d * e, (cuuint64_t)Hq * d * e, (cuuint64_t)Nmax * Hq * d * e, q_ls};
    cuuint32_t qb[5] = {64, (cuuint32_t)g.G, (cuuint32_t)g.NPT, 1, 1};
    // rows of one (sequence, KV head) slab, or of one (page, KV head) slab of 128 rows
    const cuuint64_t slab_rows = block_table ? (cuuint64_t)kTileN : (cuuint64_t)Scap;
    const cuuint64_t slabs = block_table ? (cuuint64_t)n_pages * Hkv : (cuuint64_t)B * Hkv;
    const cuuint64_t c_ls = L > 1 ? (cuuint64_t)ls.cache * e : slabs * slab_rows * d * e;
    cuuint64_t cd[4] = {(cuuint64_t)d, slab_rows, slabs, layers};
    cuuint64_t cs[3] = {(cuuint64_t)d * e, slab_rows * d * e, c_ls};
    cuuint32_t cb[4] = {64, kTileN, 1, 1};
    cuuint64_t td[5] = {(cuuint64_t)d, (cuuint64_t)Hkv, (cuuint64_t)Nmax, (cuuint64_t)B, layers};
    cuuint64_t ts[4] = {(cuuint64_t)d * e, (cuuint64_t)Hkv * d * e, (cuuint64_t)Nmax * Hkv * d * e, t_ls};
    cuuint32_t tb[5] = {64, 1, kTileN, 1, 1};
    const bool ok = encode_map(&maps[0], q, 5, qd, qs, qb) && encode_map(&maps[1], k_cache, 4, cd, cs, cb) &&
                    encode_map(&maps[2], v_cache, 4, cd, cs, cb) &&
                    (in_cache ? (maps[3] = maps[1], maps[4] = maps[2], true)      // placeholders the kernel never uses
                              : (encode_map(&maps[3], k_tree, 5, td, ts, tb) && encode_map(&maps[4], v_tree, 5, td, ts, tb)));
    if (!ok) return tv::fail(TV_ERR_CUDA, "tree_verify_attn: cuTensorMapEncodeTiled failed");
  }
  AttnParams prm{};
  prm.prefix_len = prefix_len;
  prm.n_nodes = n_nodes;
  prm.anc_bits = anc_bits;
  prm.out = out;
  prm.lse = lse;
  prm.status = status;
  // The launch touches the workspace only after its grid-dependency wait, that is after every earlier kernel of
  // the stream has completed: consecutive launches may share it although they overlap on the device.
  char* ws = static_cast<char*>(workspace);
  prm.flags = reinterpret_cast<unsigned long long*>(ws + g.flags_off);
  prm.part_ml = reinterpret_cast<float*>(ws + g.ml_off);
  prm.part_o = reinterpret_cast<tv_bf16*>(ws + g.o_off);
  prm.epoch = next_epoch();
  prm.B = B; prm.Nmax = Nmax; prm.Hq = Hq; prm.Hkv = Hkv; prm.Scap = Scap;
  prm.G = g.G; prm.NPT = g.NPT; prm.NP = g.NP; prm.W = (Nmax + 31) / 32; prm.groups = g.groups;
  prm.TT = (Nmax + kTileN - 1) / kTileN;
  prm.scale = scale;
  prm.tree_in_cache = in_cache ? 1 : 0;
  prm.block_table = block_table;
  prm.max_blocks = max_blocks;
  prm.n_pages = n_pages;
  prm.out_al32 = ((reinterpret_cast<uintptr_t>(out) & 31u) == 0 && (L == 1 || (ls.out * 2) % 32 == 0)) ? 1 : 0;
  prm.q_box_bytes = 64u * (uint32_t)g.G * (uint32_t)g.NPT * 2u;
  prm.trace = g_trace.load(std::memory_order_relaxed);
  prm.scale_log2e = scale * kLog2e;
  prm.early = opt.early ? 1 : 0;
  prm.wait_limit_ns = opt.wait_limit_ns;
  prm.debug = opt.debug;
  prm.L = L;
  prm.out_layer_stride = ls.out;
  cudaError_t e;
  if (d == 128) e = g.MT == 2 ? launch<128, 2>(g, maps, prm, s) : launch<128, 1>(g, maps, prm, s);
  else e = g.MT == 2 ? launch<64, 2>(g, maps, prm, s) : launch<64, 1>(g, maps, prm, s);
  if (e != cudaSuccess) return tv::fail(TV_ERR_CUDA, "tree_verify_attn: launch failed: %s", cudaGetErrorString(e));
  return TV_OK;
}

int attn_entry(const tv_bf16* q,
               const tv_bf16* k_cache, const tv_bf16* v_cache,
               const int32_t* block_table, int n_pages, int max_blocks,
               const tv_bf16* k_tree, const tv_bf16* v_tree,
               const int32_t* prefix_len, const int32_t* n_nodes,
               const uint32_t* anc_bits,
               int L, const LayerStrides& ls, int B, int Nmax, int Hq, int Hkv, int d, int Scap, float scale,
               tv_bf16* out, float* lse,
               void* workspace, size_t workspace_bytes,
               int32_t* status, const AttnOptions& opt, tv_stream stream) {
  TV_REQUIRE(q && k_cache && v_cache && prefix_len && n_nodes && anc_bits && out && status && workspace,
             "tree_verify_attn: NULL pointer");
  TV_REQUIRE((k_tree == nullptr) == (v_tree == nullptr), "tree_verify_attn: k_tree and v_tree must both be given or both be NULL");
  const bool in_cache = (k_tree == nullptr);       // the tree's K/V rows sit in the cache behind the prefix
  TV_REQUIRE(B >= 0 && B <= kMaxB, "tree_verify_attn: need 0 <= B <= 512");
  TV_REQUIRE(Nmax >= 1 && Nmax <= 256, "tree_verify_attn: Nmax must be in 1..256");
  TV_REQUIRE(d == 64 || d == 128, "tree_verify_attn: d must be 64 or 128");
  TV_REQUIRE(Hq >= 1 && Hkv >= 1 && Hq % Hkv == 0 && Hq / Hkv <= kTileM, "tree_verify_attn: need Hq %% Hkv == 0 and Hq/Hkv <= 128");
  TV_REQUIRE(Scap >= 1 && scale > 0.f, "tree_verify_attn: need Scap >= 1 and scale > 0");
  TV_REQUIRE(tv::aligned16(q) && tv::aligned16(k_cache) && tv::aligned16(v_cache) && tv::aligned16(k_tree) &&
                 tv::aligned16(v_tree) && tv::aligned16(out),
             "tree_verify_attn: tensors must be 16-byte aligned");
  TV_REQUIRE((reinterpret_cast<uintptr_t>(workspace) & 255u) == 0, "tree_verify_attn: workspace must be 256-byte aligned");
  if (B == 0 || L == 0) return TV_OK;
  const Geometry g = geometry(B, Nmax, Hq, Hkv, d, true);
  const long long tiles_per_layer = (long long)B * Hkv * ((Scap + kTileN - 1) / kTileN + 2 + kSetupCost);
  TV_REQUIRE(tiles_per_layer < (1ll << 31), "tree_verify_attn: B * Hkv * Scap is too large for the tile scheduler");
  if (g.sms > 160) return tv::fail(TV_ERR_INVALID_ARG, "tree_verify_attn: device with more than 160 SMs is not supported");
  if (workspace_bytes < g.layers_off + g.per_layer)
    return tv::fail(TV_ERR_WORKSPACE, "tree_verify_attn: workspace of %zu bytes, need %zu", workspace_bytes,
                    g.layers_off + g.per_layer);
  // Layers that share a launch: as many as the workspace has stretches for and as the 31-bit tile space holds.
  long long per_launch = (long long)((workspace_bytes - g.layers_off) / g.per_layer);
  const long long by_tiles = ((1ll << 31) - 1) / tiles_per_layer;
  if (per_launch > by_tiles) per_launch = by_tiles;
  if (per_launch > 65535) per_launch = 65535;
  AttnOptions o = opt;
  for (int l0 = 0; l0 < L; l0 += (int)per_launch) {
    const int nl = L - l0 < per_launch ? L - l0 : (int)per_launch;
    const tv_bf16* kc = k_cache + (size_t)l0 * ls.cache;
    const tv_bf16* vc = v_cache + (size_t)l0 * ls.cache;
    const int rc = attn_launch(q + (size_t)l0 * ls.q, kc, vc, block_table, n_pages, max_blocks,
                               in_cache ? kc : k_tree + (size_t)l0 * ls.tree, in_cache ? vc : v_tree + (size_t)l0 * ls.tree,
                               in_cache, prefix_len, n_nodes, anc_bits, nl, ls, B, Nmax, Hq, Hkv, d, Scap, scale,
                               out + (size_t)l0 * ls.out, lse ? lse + (size_t)l0 * B * Hq * Nmax : nullptr, workspace, status,
                               o, (cudaStream_t)stream);
    if (rc != TV_OK) return rc;
    o.early = true;       // behind a tree_verify_attn launch of this very call the inputs are stable
  }
  return TV_OK;
}

}  // namespace

// Tuning aid, live only in a library built with -DTV_TRACE: while a device buffer of 160 * 4 * 256 u64 is
// registered here, every tree_verify_attn launch records a per-CTA, per-role timeline (tag << 48 |
// globaltimer ns) into it.  NULL switches it off.
extern "C" TV_API void tv_debug_set_attn_trace(unsigned long long* device_buffer) {
  g_trace.store(device_buffer, std::memory_order_relaxed);
}

// Test aid for the failure path: tree_verify_attn with the limit of every bounded wait set to wait_limit_ns and,
// with mode bit 0, a producer warp that issues no copy at all, so that the first wait of the MMA issuer expires;
// with mode bit 1, pieces of cut units that never announce their partials, so that the poll of the merging piece expires.
// The launch must then end by itself with TV_ST_TIMEOUT in status[] of every sequence and leave the GPU usable.
extern "C" TV_API int tv_debug_attn_expire(const tv_bf16* q, const tv_bf16* k_cache, const tv_bf16* v_cache,
                                           const tv_bf16* k_tree, const tv_bf16* v_tree, const int32_t* prefix_len,
                                           const int32_t* n_nodes, const uint32_t* anc_bits, int B, int Nmax, int Hq,
                                           int Hkv, int d, int Scap, float scale, tv_bf16* out, float* lse,
                                           void* workspace, size_t workspace_bytes, int32_t* status,
                                           unsigned long long wait_limit_ns, int mode, tv_stream stream) {
  AttnOptions opt;
  opt.wait_limit_ns = wait_limit_ns;
  opt.debug = mode;
  return attn_entry(q, k_cache, v_cache, nullptr, 0, 0, k_tree, v_tree, prefix_len, n_nodes, anc_bits, 1, LayerStrides{}, B,
                    Nmax, Hq, Hkv, d, Scap, scale, out, lse, workspace, workspace_bytes, status, opt, stream);
}

extern "C" TV_API int tv_debug_attn_stream_only(const tv_bf16* q, const tv_bf16* k_cache, const tv_bf16* v_cache,
                                                const tv_bf16* k_tree, const tv_bf16* v_tree, const int32_t* prefix_len,
                                                const int32_t* n_nodes, const uint32_t* anc_bits, int L, int B, int Nmax,
                                                int Hq, int Hkv, int d, int Scap, int64_t q_layer_stride,
                                                int64_t cache_layer_stride, int64_t tree_layer_stride, tv_bf16* out,
                                                int64_t out_layer_stride, void* workspace, size_t workspace_bytes,
                                                int32_t* status, tv_stream stream) {
  TV_REQUIRE(L >= 0 && L <= 65535, "tv_debug_attn_stream_only: need 0 <= L <= 65535");
  TV_REQUIRE(q_layer_stride % 8 == 0 && cache_layer_stride % 8 == 0 && tree_layer_stride % 8 == 0 && out_layer_stride % 8 == 0,
             "tv_debug_attn_stream_only: layer strides must be multiples of 8 elements");
  AttnOptions opt;
  opt.early = true;
  opt.debug = 4;
  LayerStrides ls;
  ls.q = q_layer_stride;
  ls.cache = cache_layer_stride;
  ls.tree = tree_layer_stride;
  ls.out = out_layer_stride;
  return attn_entry(q, k_cache, v_cache, nullptr, 0, 0, k_tree, v_tree, prefix_len, n_nodes, anc_bits, L, ls, B, Nmax, Hq,
                    Hkv, d, Scap, 1.0f, out, nullptr, workspace, workspace_bytes, status, opt, stream);
}

extern "C" size_t tv_attn_workspace_bytes(int B, int Nmax, int Hq, int Hkv, int d, int Scap) {
  (void)Scap;
  if (B <= 0 || Nmax <= 0 || Hq <= 0 || Hkv <= 0 || Hq % Hkv != 0 || Hq / Hkv > kTileM || d <= 0) return 256;
  return geometry(B, Nmax, Hq, Hkv, d, false).total;
}

extern "C" int tree_verify_attn(const tv_bf16* q,
                                const tv_bf16* k_cache, const tv_bf16* v_cache,
                                const tv_bf16* k_tree, const tv_bf16* v_tree,
                                const int32_t* prefix_len, const int32_t* n_nodes,
                                const uint32_t* anc_bits,
                                int B, int Nmax, int Hq, int Hkv, int d, int Scap, float scale,
                                tv_bf16* out, float* lse,
                                void* workspace, size_t workspace_bytes,
                                int32_t* status, tv_stream stream) {
  return attn_entry(q, k_cache, v_cache, nullptr, 0, 0, k_tree, v_tree, prefix_len, n_nodes, anc_bits, 1, LayerStrides{}, B,
                    Nmax, Hq, Hkv, d, Scap, scale, out, lse, workspace, workspace_bytes, status, AttnOptions{}, stream);
}

extern "C" int tree_verify_attn_paged(const tv_bf16* q,
                                      const tv_bf16* k_pages, const tv_bf16* v_pages,
                                      const int32_t* block_table,
                                      const tv_bf16* k_tree, const tv_bf16* v_tree,
                                      const int32_t* prefix_len, const int32_t* n_nodes,
                                      const uint32_t* anc_bits,
                                      int B, int Nmax, int Hq, int Hkv, int d, int n_pages, int max_blocks, float scale,
                                      tv_bf16* out, float* lse,
                                      void* workspace, size_t workspace_bytes,
                                      int32_t* status, tv_stream stream) {
  TV_REQUIRE(block_table && k_tree && v_tree, "tree_verify_attn_paged: NULL pointer");
  TV_REQUIRE(n_pages >= 1 && max_blocks >= 1 && max_blocks <= (1 << 20) && (long long)n_pages * Hkv < (1ll << 31),
             "tree_verify_attn_paged: need n_pages >= 1, 1 <= max_blocks <= 2^20, n_pages * Hkv < 2^31");
  return attn_entry(q, k_pages, v_pages, block_table, n_pages, max_blocks, k_tree, v_tree, prefix_len, n_nodes, anc_bits,
                    1, LayerStrides{}, B, Nmax, Hq, Hkv, d, max_blocks * kTileN, scale, out, lse, workspace, workspace_bytes,
                    status, AttnOptions{}, stream);
}

extern "C" int tree_verify_attn_layers(const tv_bf16* q,
                                       const tv_bf16* k_cache, const tv_bf16* v_cache,
                                       const tv_bf16* k_tree, const tv_bf16* v_tree,
                                       const int32_t* prefix_len, const int32_t* n_nodes,
                                       const uint32_t* anc_bits,
                                       int L, int B, int Nmax, int Hq, int Hkv, int d, int Scap, float scale,
                                       int64_t q_layer_stride, int64_t cache_layer_stride, int64_t tree_layer_stride,
                                       tv_bf16* out, int64_t out_layer_stride, float* lse,
                                       void* workspace, size_t workspace_bytes,
                                       int32_t* status, unsigned flags, tv_stream stream) {
  TV_REQUIRE(L >= 0 && L <= 65535, "tree_verify_attn_layers: need 0 <= L <= 65535");
  TV_REQUIRE(q_layer_stride % 8 == 0 && cache_layer_stride % 8 == 0 && tree_layer_stride % 8 == 0 && out_layer_stride % 8 == 0,
             "tree_verify_attn_layers: layer strides must be multiples of 8 elements");
  TV_REQUIRE((flags & ~(unsigned)(TV_ATTN_STABLE_INPUTS | TV_ATTN_LAUNCH_PER_LAYER)) == 0, "tree_verify_attn_layers: unknown flag");
  AttnOptions opt;
  opt.early = (flags & TV_ATTN_STABLE_INPUTS) != 0;
  LayerStrides ls;
  ls.q = q_layer_stride;
  ls.cache = cache_layer_stride;
  ls.tree = tree_layer_stride;
  ls.out = out_layer_stride;
  if (flags & TV_ATTN_LAUNCH_PER_LAYER) {      // exactly what L calls of tree_verify_attn issue
    for (int l = 0; l < L; ++l) {
      const int rc = attn_entry(q + (size_t)l * ls.q, k_cache + (size_t)l * ls.cache, v_cache + (size_t)l * ls.cache, nullptr,
                                0, 0, k_tree ? k_tree + (size_t)l * ls.tree : nullptr,
                                v_tree ? v_tree + (size_t)l * ls.tree : nullptr, prefix_len, n_nodes, anc_bits, 1,
                                LayerStrides{}, B, Nmax, Hq, Hkv, d, Scap, scale, out + (size_t)l * ls.out,
                                lse ? lse + (size_t)l * B * Hq * Nmax : nullptr, workspace, workspace_bytes, status, opt,
                                stream);
      if (rc != TV_OK) return rc;
      opt.early = true;      // behind a tree_verify_attn launch of this very call the inputs are stable
    }
    return TV_OK;
  }
  return attn_entry(q, k_cache, v_cache, nullptr, 0, 0, k_tree, v_tree, prefix_len, n_nodes, anc_bits, L, ls, B, Nmax, Hq,
                    Hkv, d, Scap, scale, out, lse, workspace, workspace_bytes, status, opt, stream);
}

extern "C" int tree_verify_attn_paged_layers(const tv_bf16* q,
                                             const tv_bf16* k_pages, const tv_bf16* v_pages,
                                             const int32_t* block_table,
                                             const tv_bf16* k_tree, const tv_bf16* v_tree,
                                             const int32_t* prefix_len, const int32_t* n_nodes,
                                             const uint32_t* anc_bits,
                                             int L, int B, int Nmax, int Hq, int Hkv, int d, int n_pages, int max_blocks,
                                             float scale,
                                             int64_t q_layer_stride, int64_t page_layer_stride, int64_t tree_layer_stride,
                                             tv_bf16* out, int64_t out_layer_stride, float* lse,
                                             void* workspace, size_t workspace_bytes,
                                             int32_t* status, unsigned flags, tv_stream stream) {
  TV_REQUIRE(block_table && k_tree && v_tree, "tree_verify_attn_paged_layers: NULL pointer");
  TV_REQUIRE(n_pages >= 1 && max_blocks >= 1 && max_blocks <= (1 << 20) && (long long)n_pages * Hkv < (1ll << 31),
             "tree_verify_attn_paged_layers: need n_pages >= 1, 1 <= max_blocks <= 2^20, n_pages * Hkv < 2^31");
  TV_REQUIRE(L >= 0 && L <= 65535, "tree_verify_attn_paged_layers: need 0 <= L <= 65535");
  TV_REQUIRE(q_layer_stride % 8 == 0 && page_layer_stride % 8 == 0 && tree_layer_stride % 8 == 0 && out_layer_stride % 8 == 0,
             "tree_verify_attn_paged_layers: layer strides must be multiples of 8 elements");
  TV_REQUIRE((flags & ~(unsigned)TV_ATTN_STABLE_INPUTS) == 0, "tree_verify_attn_paged_layers: unknown flag");
  AttnOptions opt;
  opt.early = (flags & TV_ATTN_STABLE_INPUTS) != 0;
  LayerStrides ls;
  ls.q = q_layer_stride;
  ls.cache = page_layer_stride;
  ls.tree = tree_layer_stride;
  ls.out = out_layer_stride;
  return attn_entry(q, k_pages, v_pages, block_table, n_pages, max_blocks, k_tree, v_tree, prefix_len, n_nodes, anc_bits, L,
                    ls, B, Nmax, Hq, Hkv, d, max_blocks * kTileN, scale, out, lse, workspace, workspace_bytes, status, opt,
                    stream);
}
