// k_fstage_1024.cu -- the F step (k_fstage_impl.cuh) for transforms of 2048 samples.
#include "k_fstage_impl.cuh"

namespace corr {

cudaError_t fstage_1024_init_constants() { return init_w32(); }

template <int L>
static cudaError_t launch_L(const FParams& p, cudaStream_t st) {
  if constexpr (L >= 256) {
    if (p.G == 16) return launch_LG<L, 16, false>(p, st);
    if (p.G == 32) return launch_LG<L, 32, false>(p, st);
  }
  return launch_LG<L, 0, false>(p, st);
}

cudaError_t launch_fstage_1024(const FParams& p, cudaStream_t s) {
  switch (p.nchan) {
    case 1024: return launch_L<1024>(p, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace corr
