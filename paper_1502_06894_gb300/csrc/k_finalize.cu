// k_finalize.cu -- integration end: baseline weights and normalisation.
//
// W_ab counts the FFT blocks of the integration that are valid at both
// stations a and b; blocks valid at only one end were stored as zero spectra
// and so add nothing to V_ab.  The output is V_ab / (W_ab * N) (zero when
// W_ab = 0), which puts the autocorrelation of 2-bit data at the mean power of
// the quantised levels.  The KZ partial accumulators are summed in a fixed
// order.
#include "corr_internal.cuh"

#include <algorithm>

namespace corr {

// Blocks valid at both stations of baseline bl, counted by `threads` threads
// from index i0; the caller adds their counts up.  Bound by the latency of its
// loads, which take 16 blocks each where the rows of `valid` start at multiples
// of 16 bytes (a handle pads them; in the static scratch they are as long as the
// integration): 62500 blocks took a CTA 120 us with byte loads, 11 us now.
__device__ __forceinline__ int count_valid(const FinParams& p, int bl, int i0, int threads) {
  int a = 0, q = bl;  // baseline index -> (a, b)
  while (q >= p.S - a) { q -= p.S - a; ++a; }
  const int b = a + q;
  const uint8_t* va = p.valid + (size_t)a * p.ld;
  const uint8_t* vb = p.valid + (size_t)b * p.ld;
  int cnt = 0;
  const int vec = p.ld % 16 == 0 ? p.M : 0;  // bytes of 0 or 1
#pragma unroll 4
  for (int i = 16 * i0; i < vec; i += 16 * threads) {
    const uint4 x = *reinterpret_cast<const uint4*>(va + i), y = *reinterpret_cast<const uint4*>(vb + i);
    const uint32_t w[4] = {x.x & y.x, x.y & y.y, x.z & y.z, x.w & y.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int n = p.M - i - 4 * q;  // blocks of the integration in this word
      cnt += __popc(n >= 4 ? w[q] : n > 0 ? w[q] & ((1u << (8 * n)) - 1u) : 0u);
    }
  }
  for (int i = vec + i0; i < p.M; i += threads) cnt += va[i] & vb[i];
  return cnt;
}

// The same for two consecutive baselines (n = 1: one) and a warp, with four loads
// in flight (16 stations, 60000 blocks: 160 us baseline by baseline, 100; four at
// once, 94, take registers that the writes below miss).
__device__ __forceinline__ void count_valid2(const FinParams& p, int bl, int n, int lane, int (&cnt)[2]) {
  const uint8_t *va[2], *vb[2];
  int a = 0, b = bl;
  while (b >= p.S - a) { b -= p.S - a; ++a; }
  b += a;
#pragma unroll
  for (int u = 0; u < 2; ++u) {  // beyond the n-th: the last one again, not used
    va[u] = p.valid + (size_t)a * p.ld;
    vb[u] = p.valid + (size_t)b * p.ld;
    cnt[u] = 0;
    if (u + 1 < n && ++b == p.S) b = ++a;
  }
  if (p.ld % 16 != 0) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (u < n) cnt[u] = count_valid(p, bl + u, lane, 32);
    return;
  }
  for (int i = 16 * lane; i < p.M; i += 16 * 32) {
    uint4 x[2], y[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      x[u] = *reinterpret_cast<const uint4*>(va[u] + i);
      y[u] = *reinterpret_cast<const uint4*>(vb[u] + i);
    }
    uint32_t mask[4];  // blocks of the integration only
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int left = p.M - i - 4 * k;
      mask[k] = left >= 4 ? ~0u : left > 0 ? (1u << (8 * left)) - 1u : 0u;
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
      cnt[u] += __popc(x[u].x & y[u].x & mask[0]) + __popc(x[u].y & y[u].y & mask[1]) +
                __popc(x[u].z & y[u].z & mask[2]) + __popc(x[u].w & y[u].w & mask[3]);
  }
}

// 1 / (W N) of a baseline times `unscale`: in FP64, which this GPU runs at a
// 64th of its FP32 rate, so one thread of a CTA forms it, not every element.
// That thread also writes the weight, in the first CTA of the baseline's row.
__device__ __forceinline__ float fin_scale(const FinParams& p, int bl, int w, float unscale) {
  if (p.weights && blockIdx.x == 0) p.weights[bl] = (double)w;
  return w > 0 ? (float)((double)unscale / ((double)w * (double)p.N)) : 0.f;
}

// The same for a CTA of 256 threads and one baseline (blockIdx.y): every CTA
// of the row counts for itself, which costs less than a launch before it.
__device__ __forceinline__ float cta_scale(const FinParams& p, float unscale) {
  __shared__ float s_scale;
  __shared__ int s_count[8];
  int cnt = count_valid(p, blockIdx.y, threadIdx.x, 256);
  for (int o = 16; o > 0; o >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, o);
  if ((threadIdx.x & 31) == 0) s_count[threadIdx.x >> 5] = cnt;
  __syncthreads();
  if (threadIdx.x == 0) {
    int w = 0;
    for (int q = 0; q < 8; ++q) w += s_count[q];
    s_scale = fin_scale(p, blockIdx.y, w, unscale);
  }
  __syncthreads();
  return s_scale;
}

// Partial sums [KZ][nbl][G][nchan] -> out.  A CTA takes elements of one
// baseline (blockIdx.y), shared by KG groups of 256 / KG threads: group q adds
// partials q, q + KG, ... and the groups' sums are added in order.  Up to 8
// partials (KG = 1): one streaming pass of eight loads in flight per thread,
// bound by HBM (2080 baselines x 131072 values, one partial, 4.4 GB: 5.5 ms
// with an FP64 quotient per element, 0.62 ms now).  Above, the sum of one
// element is a long chain of loads and the output small (a two-station scan
// has 768 values of 456 partials: 66 us as one chain, 9.5 us now), so sixteen
// groups share it.
template <int KG>
__global__ void __launch_bounds__(256) k_finalize(FinParams p) {
  constexpr int EL = 256 / KG, PER = KG == 1 ? 8 : 1;  // a thread takes PER elements, EL apart, at a time
  const int bl = blockIdx.y;
  const size_t per = (size_t)p.G * p.nchan;
  const size_t total = (size_t)nbl_of(p.S) * per;
  __shared__ float2 s_sum[KG > 1 ? 256 : 1];
  const float sc = cta_scale(p, p.unscale);
  const bool failed = p.err && *p.err != 0;
  const float nan = __int_as_float(0x7fc00000);
  const int q = threadIdx.x / EL;
  for (size_t k0 = (size_t)blockIdx.x * EL * PER; k0 < per; k0 += (size_t)gridDim.x * EL * PER) {
    const size_t k = k0 + threadIdx.x % EL;
    float2 v[PER];
#pragma unroll
    for (int u = 0; u < PER; ++u) v[u] = make_float2(0.f, 0.f);
#pragma unroll(KG > 1 ? 8 : 1)
    for (int kz = q; kz < p.KZ; kz += KG) {
      const float2* src = p.part + (size_t)kz * total + (size_t)bl * per + k;
      float2 x[PER];
#pragma unroll
      for (int u = 0; u < PER; ++u) x[u] = k + u * EL < per ? __ldcs(src + u * EL) : make_float2(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < PER; ++u) v[u] = make_float2(v[u].x + x[u].x, v[u].y + x[u].y);
    }
    if constexpr (KG > 1) {
      __syncthreads();  // the sums of the elements before have been read
      s_sum[threadIdx.x] = v[0];
      __syncthreads();
      if (q != 0) continue;
#pragma unroll
      for (int g = 1; g < KG; ++g) {
        const float2 x = s_sum[g * EL + threadIdx.x];
        v[0].x += x.x;
        v[0].y += x.y;
      }
    }
#pragma unroll
    for (int u = 0; u < PER; ++u)
      if (k + u * EL < per)
        p.out[(size_t)bl * per + k + u * EL] = failed ? make_float2(nan, nan) : make_float2(v[u].x * sc, v[u].y * sc);
  }
}

// CTAs along a baseline's elements: one per `each` of them, but no more than
// `most` an SM over all baselines, since every CTA counts the baseline's valid
// blocks.
static unsigned row_ctas(size_t elements, size_t each, int rows, int most = 32) {
  const size_t need = (elements + each - 1) / each, room = std::max(1, 152 * most / rows);
  return (unsigned)std::min(need, room);
}

// Sixteen groups of threads share an element's partials where one chain would
// be long or leave the chip idle: above 8 partials, but for up to 16 of outputs
// that give every SM a CTA of chains (190 baselines x 12 streams x 256 channels,
// 9 partials: 55 us in groups, 18 in chains).
static bool shared_sums(int KZ, size_t values) { return KZ > 16 || (KZ > 8 && values < (size_t)152 * 2048); }

cudaError_t launch_finalize(const FinParams& p, cudaStream_t s) {
  const size_t per = (size_t)p.G * p.nchan;
  const int nbl = nbl_of(p.S);
  if (shared_sums(p.KZ, per * nbl))
    k_finalize<16><<<dim3(row_ctas(per, 16, nbl, 8), nbl), 256, 0, s>>>(p);
  else
    k_finalize<1><<<dim3(std::max(row_ctas(per, 2048, nbl), (unsigned)((per + 8191) / 8192)), nbl), 256, 0, s>>>(p);
  return cudaGetLastError();
}

// Tensor-core partial sums are laid out [G][nchan][nbl] (baseline fastest, as
// the X kernel's epilogue adds them), the output is [nbl][G][nchan]: 32 x 32
// values are turned through shared memory so that both the reads and the
// writes are 256-byte runs.  Bound by HBM: 2080 baselines x 131072 channels
// (2.2 GB each way) took 6.0 ms with 8-byte reads 16 KB apart and an FP64
// quotient per value, 0.64 ms now, 6.8 TB/s.
constexpr int kTurn = 32;
__global__ void __launch_bounds__(256) k_finalize_tc(FinParams p, float unscale) {
  __shared__ float2 tile[kTurn][kTurn + 1];
  __shared__ float s_sc[kTurn];
  const int nbl = nbl_of(p.S);
  const size_t per = (size_t)p.G * p.nchan;
  const int bl0 = blockIdx.y * kTurn;
  for (int r = 2 * threadIdx.y; r < kTurn && bl0 + r < nbl; r += 16) {  // a warp per pair of baselines
    const int n = min(2, nbl - bl0 - r);
    int cnt[2];
    count_valid2(p, bl0 + r, n, threadIdx.x, cnt);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      for (int o = 16; o > 0; o >>= 1) cnt[u] += __shfl_down_sync(0xffffffffu, cnt[u], o);
      if (threadIdx.x == 0 && u < n) s_sc[r + u] = fin_scale(p, bl0 + r + u, cnt[u], unscale);
    }
  }
  for (size_t gk0 = (size_t)blockIdx.x * kTurn; gk0 < per; gk0 += (size_t)gridDim.x * kTurn) {
    __syncthreads();  // the tile before has been written out
#pragma unroll
    for (int r = 0; r < kTurn; r += 8) {
      const size_t gk = gk0 + r + threadIdx.y;
      const int bl = bl0 + threadIdx.x;
      if (gk < per && bl < nbl) tile[r + threadIdx.y][threadIdx.x] = __ldcs(p.part + gk * nbl + bl);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kTurn; r += 8) {
      const int row = r + threadIdx.y;
      const size_t gk = gk0 + threadIdx.x;
      if (gk < per && bl0 + row < nbl) {
        const float2 v = tile[threadIdx.x][row];
        p.out[(size_t)(bl0 + row) * per + gk] = make_float2(v.x * s_sc[row], v.y * s_sc[row]);
      }
    }
  }
}

cudaError_t launch_finalize_tc(const FinParams& p, float unscale, cudaStream_t s) {
  const size_t per = (size_t)p.G * p.nchan;
  const int rows = (nbl_of(p.S) + kTurn - 1) / kTurn;
  k_finalize_tc<<<dim3(row_ctas(per, kTurn, rows), rows), dim3(kTurn, 8), 0, s>>>(p, unscale);
  return cudaGetLastError();
}

// Both hands of two polarisations.  The X step ran over 2S virtual stations
// v = pol * S + station per subband, so V_ab^pq is the virtual product
// P[p S + a][q S + b] when p S + a <= q S + b and its conjugate otherwise
// (for a = b and pq = 10: the conjugate of the 01 product).
__device__ __forceinline__ int cross_source(int S, int a, int b, int pq, bool& flip) {
  int v1 = (pq >> 1) * S + a, v2 = (pq & 1) * S + b;
  flip = v1 > v2;
  if (flip) {
    const int t = v1;
    v1 = v2;
    v2 = t;
  }
  return bl_index(v1, v2, 2 * S);
}

// A CTA takes one baseline (blockIdx.y) and a run of (subband, hand, channel)
// values, shared by KG groups of threads as in k_finalize: the X step of few
// rows leaves over a hundred partials (two stations, 1024 channels: 114), whose
// sum in one chain would round more often than the sums that it adds, and, with
// few values, is all latency (two stations, 256 channels, 228 partials: 195 us, 12
// us now).
template <bool TC, int KG>
__global__ void __launch_bounds__(256) k_finalize_cross(FinParams p, float unscale) {
  constexpr int EL = 256 / KG;
  __shared__ float2 s_sum[KG > 1 ? 256 : 1];
  const int S = p.S, nsub = p.G, nch = p.nchan;
  const int nblv = nbl_of(2 * S);
  const int bl = blockIdx.y;
  const float sc = cta_scale(p, unscale);
  int a = 0, q = bl;
  while (q >= S - a) { q -= S - a; ++a; }
  const int b = a + q;
  const int per = nsub * 4 * nch;
  const int g = threadIdx.x / EL;
  for (int e0 = blockIdx.x * EL; e0 < per; e0 += gridDim.x * EL) {
    const int e = e0 + threadIdx.x % EL;
    const bool mine = e < per;
    const int k = e & (nch - 1);  // a power of two of channels
    const int r = e / nch;
    const int pq = r & 3, sb = r >> 2;
    bool flip;
    const int blv = cross_source(S, a, b, pq, flip);
    float2 v = make_float2(0.f, 0.f);
#pragma unroll(KG > 1 ? 8 : 4)
    for (int kz = g; kz < p.KZ && mine; kz += KG) {
      const float2 x = TC ? p.part[(((size_t)kz * nsub + sb) * nch + k) * nblv + blv]
                          : p.part[(((size_t)kz * nblv + blv) * nsub + sb) * nch + k];
      v.x += x.x;
      v.y += x.y;
    }
    if constexpr (KG > 1) {
      __syncthreads();  // the sums of the values before have been read
      s_sum[threadIdx.x] = v;
      __syncthreads();
      if (g != 0) continue;
      float2 x[KG];  // added up in pairs, with fewer roundings than one by one
#pragma unroll
      for (int h = 0; h < KG; ++h) x[h] = s_sum[h * EL + threadIdx.x];
#pragma unroll
      for (int h = KG / 2; h > 0; h /= 2)
#pragma unroll
        for (int u = 0; u < h; ++u) x[u] = make_float2(x[u].x + x[u + h].x, x[u].y + x[u + h].y);
      v = x[0];
    }
    if (flip) v.y = -v.y;
    if (mine) p.out[(size_t)bl * per + e] = make_float2(v.x * sc, v.y * sc);
  }
}

cudaError_t launch_finalize_cross(const FinParams& p, bool tc, float unscale, cudaStream_t s) {
  const int per = p.G * 4 * p.nchan, nbl = nbl_of(p.S);
  const dim3 few(row_ctas(per, 16, nbl, 8), nbl), grid(row_ctas(per, 1024, nbl), nbl);
  if (tc)
    k_finalize_cross<true, 1><<<grid, 256, 0, s>>>(p, unscale);
  else if (shared_sums(p.KZ, (size_t)per * nbl))
    k_finalize_cross<false, 16><<<few, 256, 0, s>>>(p, unscale);
  else
    k_finalize_cross<false, 1><<<grid, 256, 0, s>>>(p, unscale);
  return cudaGetLastError();
}

}  // namespace corr
