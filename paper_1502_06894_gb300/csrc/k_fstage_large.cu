// k_fstage_large.cu -- the F step (k_fstage_impl.cuh) for transforms of 4096 to 16384 samples.
#include "k_fstage_impl.cuh"

namespace corr {

cudaError_t fstage_large_init_constants() { return init_w32(); }

template <int L>
static cudaError_t launch_L(const FParams& p, cudaStream_t st) {
  if constexpr (L >= 256) {
    if (p.G == 16) return launch_LG<L, 16, false>(p, st);
    if (p.G == 32) return launch_LG<L, 32, false>(p, st);
  }
  return launch_LG<L, 0, false>(p, st);
}

cudaError_t launch_fstage_large(const FParams& p, cudaStream_t s) {
  switch (p.nchan) {
    case 2048: return launch_L<2048>(p, s);
    case 4096: return launch_L<4096>(p, s);
    case 8192: return launch_L<8192>(p, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace corr
