// Reading one row of a [rows, V] bf16 tensor in 16-byte vectors whatever V is.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "treeverify.h"

namespace tv {

// The row is covered by the aligned 16-byte vectors of memory it lies in: vector i holds entries 8 i - off .. 8 i - off + 7.
// vector() gives the vectors that lie wholly inside the row and -inf for all others; edge() gives the entries that are
// left, at most seven before the first such vector and at most seven behind the last one.  (Putting the outer vectors
// together inside vector() cost registers and kept a thread's loads from being issued together.)
struct LogitsRow {
  const uint16_t* row;
  int off, V;
  __device__ __forceinline__ LogitsRow(const tv_bf16* logits, long long r, int V_) : row(logits + r * V_), V(V_) {
    off = (int)((reinterpret_cast<uintptr_t>(row) & 15u) >> 1);
  }
  __device__ __forceinline__ uint4 vector(int i) const {
    const int v = 8 * i - off;
    return v >= 0 && v <= V - 8 ? __ldcs(reinterpret_cast<const uint4*>(row + v))
                                : make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u);
  }
  // Entry number t (0..15) of those no whole vector holds, or -1.
  __device__ __forceinline__ int edge(int t) const {
    const int head = min((8 - off) & 7, V);               // entries before the first aligned vector
    const int tail = head + ((V - head) & ~7);            // first entry behind the last one
    const int v = t < 8 ? t : tail + t - 8;
    return t < 8 ? (v < head ? v : -1) : (v < V ? v : -1);
  }
};

}  // namespace tv
