// k_fstage_pre_large.cu -- the pre-F form of the F step (k_fstage_pre.cu) for transforms of 1024 to 8192 points.
#include "k_fstage_impl.cuh"

namespace corr {

cudaError_t fstage_pre_large_init_constants() { return init_w32(); }

template <int L>
static cudaError_t launch_L(const FParams& p, cudaStream_t st) {
  if constexpr (L >= 256) {
    if (p.G == 16) return launch_LG<L, 16, true>(p, st);
    if (p.G == 32) return launch_LG<L, 32, true>(p, st);
  }
  return launch_LG<L, 0, true>(p, st);
}

cudaError_t launch_fstage_pre_large(const FParams& p, cudaStream_t s) {
  switch (2 * p.nchan) {
    case 1024: return launch_L<1024>(p, s);
    case 2048: return launch_L<2048>(p, s);
    case 4096: return launch_L<4096>(p, s);
    case 8192: return launch_L<8192>(p, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace corr
