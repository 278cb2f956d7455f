// k_fstage_small.cu -- the F step (k_fstage_impl.cuh) for transforms of up to 1024 samples.
#include "k_fstage_impl.cuh"

namespace corr {

cudaError_t fstage_small_init_constants() { return init_w32(); }

template <int L>
static cudaError_t launch_L(const FParams& p, cudaStream_t st) {
  if constexpr (L >= 256) {
    if (p.G == 16) return launch_LG<L, 16, false>(p, st);
    if (p.G == 32) return launch_LG<L, 32, false>(p, st);
  }
  return launch_LG<L, 0, false>(p, st);
}

cudaError_t launch_fstage_small(const FParams& p, cudaStream_t s) {
  switch (p.nchan) {
    case 4: return launch_L<4>(p, s);
    case 8: return launch_L<8>(p, s);
    case 16: return launch_L<16>(p, s);
    case 32: return launch_L<32>(p, s);
    case 64: return launch_L<64>(p, s);
    case 128: return launch_L<128>(p, s);
    case 256: return launch_L<256>(p, s);
    case 512: return launch_L<512>(p, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace corr
