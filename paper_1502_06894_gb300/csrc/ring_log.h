// ring_log.h -- which copies a ring of shared-memory stages has in flight.
// Plain C++, so that its bookkeeping also runs (and is tested) on the host.
#pragma once

#ifdef __CUDACC__
#define RING_LOG_FN __host__ __device__ __forceinline__
#else
#define RING_LOG_FN inline
#endif

namespace corr {

// Per slot, the last stage whose copies were issued into it, plus one (0:
// none).  Several warps issue, and nothing orders the issues of different
// slots, so that one count of stages could end too small (a copy in flight not
// seen) or include a stage that was never issued.  A slot's own issues are
// ordered: stage q goes into slot q % stages, and only after every warp has
// read stage q - stages.  That also means that a slot's earlier copies have
// landed, so that the last one is all there is to wait for.
template <int N>
struct RingLog {
  volatile int last[N];

  RING_LOG_FN void clear() {
    for (int i = 0; i < N; ++i) last[i] = 0;
  }
  RING_LOG_FN void note(int slot, int q) { last[slot] = q + 1; }
  // wait(slot, parity) for the last copies of every slot of a ring of `stages`
  template <typename Wait>
  RING_LOG_FN void for_each(int stages, Wait wait) const {
    for (int slot = 0; slot < stages; ++slot)
      if (const int n = last[slot]) wait(slot, (unsigned)(((n - 1) / stages) & 1));
  }
};

}  // namespace corr
