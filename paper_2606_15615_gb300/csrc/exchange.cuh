// Grid-wide exchanges that carry their data, shared by the fused preparation
// kernel and decide_kernel: every block of a co-resident grid publishes words
// and reads the other blocks', without a barrier or a fence.
#pragma once

#include "common.cuh"

namespace moeca {

// Tagged words of the grid-wide exchanges: payload in the low 32 bits, the
// launch's epoch in the high 32.
__device__ __forceinline__ unsigned long long tag_word(uint32_t payload, unsigned epoch) {
  return (static_cast<unsigned long long>(epoch) << 32) | payload;
}
__device__ __forceinline__ void st_word(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_word(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Read n tagged words p[idx(0)] .. p[idx(n - 1)] and hand their payloads to
// f(j, payload) in order j = 0..n-1.  Words are fetched kB at a time; while
// any word of a batch still carries another epoch, the batch's stale words
// are fetched again (one round trip per retry).  Returns false once
// `deadline` (%globaltimer) has passed.
template <int kB, typename Idx, typename F>
__device__ __forceinline__ bool read_tagged(const unsigned long long* p, int n, Idx idx, unsigned epoch,
                                            unsigned long long deadline, F&& f) {
  for (int j0 = 0; j0 < n; j0 += kB) {
    unsigned long long v[kB];
#pragma unroll
    for (int u = 0; u < kB; ++u) v[u] = 0ull;  // epoch 0 is never used: every word starts stale
    for (;;) {
#pragma unroll
      for (int u = 0; u < kB; ++u)
        if (j0 + u < n && static_cast<unsigned>(v[u] >> 32) != epoch) v[u] = ld_word(p + idx(j0 + u));
      bool all = true;
#pragma unroll
      for (int u = 0; u < kB; ++u) all &= j0 + u >= n || static_cast<unsigned>(v[u] >> 32) == epoch;
      if (all) break;
      if (globaltimer() > deadline) return false;
    }
#pragma unroll
    for (int u = 0; u < kB; ++u)
      if (j0 + u < n) f(j0 + u, static_cast<uint32_t>(v[u]));
  }
  return true;
}

}  // namespace moeca
