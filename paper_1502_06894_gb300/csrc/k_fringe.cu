// k_fringe.cu -- delay-rate fringe search of one baseline's visibilities
// (the wide-window fringe search the paper lists for RadioAstron, Sec. 2).
//
// For visibilities V[t][k] (t: sub-integration, k: channel) the map is the
// zero-padded two-dimensional inverse DFT, unnormalised,
//     M[r][l] = sum_t sum_k V[t][k] exp(+2 pi i (k l / Nd + t r / Nr)),
// and the peak is the largest |M|, the smaller flat index r * Nd + l on ties.
// Two passes of k_cfft_inv: over channels for every sub-integration, then over
// sub-integrations for every lag, whose last pass also finds the peak.
#include "../../include/corr.h"
#include "k_fstage_impl.cuh"

#include <atomic>
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace corr {

namespace {

// What FP32 leaves of c_w32 and c_w32n: exp(-2 pi i m / 32) to twice the bits.
__constant__ float2 c_w32_low[32];
__constant__ float2 c_w32n_low[32];

// a W_32^m with the constant's low part: rounded like a product by the exact
// root.  The few constants of a 32-point butterfly meet every value of a
// transform, so their own roundings would not average out: with FP32 constants
// alone a search is less exact than one of radix-2 passes.
struct TurnW32Exact {
  __device__ __forceinline__ float2 operator()(float2 a, int m) const {
    const float2 low = f2fma(swp(a), c_w32n_low[m], f2mul(a, bc(c_w32_low[m].x)));
    return f2fma(swp(a), c_w32n[m], f2fma(a, bc(c_w32[m].x), low));
  }
};

}  // namespace

cudaError_t fringe_init_constants() {
  cudaError_t e = init_w32();
  if (e != cudaSuccess) return e;
  float2 h[32], hn[32];
  for (int m = 0; m < 32; ++m) {
    const double a = -2.0 * 3.14159265358979323846 * (double)m / 32.0;
    h[m] = make_float2((float)(cos(a) - (double)(float)cos(a)), (float)(sin(a) - (double)(float)sin(a)));
    hn[m] = make_float2(-h[m].y, h[m].y);
  }
  if ((e = cudaMemcpyToSymbol(c_w32_low, h, sizeof(h))) != cudaSuccess) return e;
  return cudaMemcpyToSymbol(c_w32n_low, hn, sizeof(hn));
}

namespace {

constexpr int kMaxFft = 16384;

// The peak of one search: `best` orders by amplitude, then by smaller index.
struct PeakSlot {
  unsigned long long best;
  unsigned int done;  // finished CTAs of the second pass
  float2 value;       // the map at the peak, written by the last of them
};

// A search holds one slot from its first launch until it has read the peak
// back (the call waits for that), so concurrent searches on other threads and
// streams have slots of their own.
constexpr int kPeakSlots = 64;
__device__ PeakSlot g_peak_slots[kPeakSlots];
std::atomic<unsigned long long> g_peak_taken{0};

// Radices of a transform of n = R0 R1 R2 points.  A thread holds 32 points
// (n if fewer) in every pass.
template <int n> struct Radices {
  static constexpr int R0 = n <= 32 ? n : n == 64 ? 8 : (n == 512 || n == 1024 || n == 16384) ? 32 : 16;
  static constexpr int R1 = n <= 32 ? 1 : (n == 64 || n == 128) ? 8 : (n == 1024 || n == 16384) ? 32 : 16;
  static constexpr int R2 = n / R0 / R1;  // 1, 8, 16 or 32
  static constexpr int T = n <= 32 ? 1 : n / 32;
  static_assert(R0 * R1 * R2 == n, "radices");
};

// Transforms per CTA: rows (consecutive in memory) fill about 256 threads;
// of columns up to 16 (one 128-byte line a row of the map) as long as their
// points fit 64 KB of shared memory and 256 threads, more for short ones.
template <int n, bool COLS> struct Batch {
  static constexpr int T = Radices<n>::T;
  static constexpr int C = T >= 256 ? 1 : COLS ? (n <= 64 ? 128 / T : n <= 256 ? 32 : 8192 / n) : 256 / T > 64 ? 64 : 256 / T;
  // complex values in shared memory: the points (rows padded, see at()), and the second pass's twiddles
  static constexpr int POINTS = Radices<n>::R1 == 1 ? 0 : COLS ? n * C : C * (n + n / Radices<n>::R0 + 1);
  static constexpr int TWIDDLES = Radices<n>::R0 * (Radices<n>::R1 - 1);
};

// Position of point i of transform c in shared memory: columns side by side
// (the threads of a warp run over columns), rows one after another with a
// padding element after every R0 points.
template <int n, bool COLS>
__device__ __forceinline__ int at(int i, int c) {
  if constexpr (COLS) return i * Batch<n, COLS>::C + c;
  else return c * (n + n / Radices<n>::R0 + 1) + padp<Radices<n>::R0>(i);
}

// W_N^m, rounded once: sincospif of an argument that is exact.  The transforms
// work on swapped (imaginary, real) values, which turns the forward butterflies
// of dft_reg into inverse ones, so the twiddles here are the forward ones.
template <int N>
__device__ __forceinline__ float2 root(int m) {
  float sn, cs;
  sincospif(-2.0f * (float)m / (float)N, &sn, &cs);
  return make_float2(cs, sn);
}

// v[r] *= W_{NS R}^{k r}.  The second pass has few k, so the CTA forms all its
// factors once, [r - 1][k] in `table`.  The third pass has one k a butterfly: r
// splits into its low bits a and its high bits b, and a factor is one product of
// W^{k a} and W^{k b} at most (ten sines and cosines for 32 points; with the
// powers k 2^i alone, five, a factor is up to four roundings away and the search
// less exact than one of radix-2 passes).
template <int R, int NS, bool TABLE>
__device__ __forceinline__ void cfft_twiddle(float2 (&v)[R], int k, const float2* table) {
  if constexpr (TABLE) {
#pragma unroll
    for (int r = 1; r < R; ++r) v[r] = cmul(v[r], table[(r - 1) * NS + k]);
    return;
  }
  constexpr int LO = ilog2c(R) / 2, NA = 1 << LO, NB = R / NA;
  float2 A[NA];
#pragma unroll
  for (int a = 1; a < NA; ++a) A[a] = root<NS * R>(k * a);
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const float2 B = b ? root<NS * R>(k * b * NA) : make_float2(1.f, 0.f);
#pragma unroll
    for (int a = 0; a < NA; ++a)
      if (a || b) v[b * NA + a] = cmul(v[b * NA + a], a && b ? cmul(A[a], B) : a ? A[a] : B);
  }
}

// A middle or last pass: R points a butterfly from shared memory; the middle
// one back to it, the last one to `store`.
template <int n, int R, int NS, bool COLS, typename Store>
__device__ __forceinline__ void cfft_pass(float2* buf, const float2* table, int t, int c, Store store) {
  constexpr int T = Radices<n>::T, PER = n / R / T;
  constexpr bool last = NS * R == n;
  float2 v[PER][R];
#pragma unroll
  for (int u = 0; u < PER; ++u)
#pragma unroll
    for (int r = 0; r < R; ++r) v[u][r] = buf[at<n, COLS>(t + u * T + r * (n / R), c)];
  if constexpr (!last) __syncthreads();
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int j = t + u * T, k = j & (NS - 1);
    cfft_twiddle<R, NS, NS == Radices<n>::R0>(v[u], k, table);
    dft_reg<R>(v[u], TurnW32Exact());
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if constexpr (last) store(k + r * NS, v[u][r]);
      else buf[at<n, COLS>((j / NS) * NS * R + k + r * NS, c)] = v[u][r];
    }
  }
  if constexpr (!last) __syncthreads();
}

// Amplitude bits (non-negative floats order like their bit patterns) above
// the complement of the flat index: the largest key is the largest amplitude
// with the smallest index.
__device__ __forceinline__ unsigned long long peak_key(float2 v, uint32_t e) {
  const float a = sqrtf(v.x * v.x + v.y * v.y);
  return ((unsigned long long)__float_as_uint(a) << 32) | (unsigned long long)(0xFFFFFFFFu - e);
}

// Inverse transforms of n points, C per CTA: transform q (a row, or with COLS
// a column) has point i at in[q * in_q + i * in_i] for i < in_len, zero above,
// and writes point i to out[q * out_q + i * out_i].
//
// Bound by the map's one write and by latency (a few waves of CTAs at most).
// The points stay in registers (radix 8..32 passes) and cross shared memory
// once or twice; the first pass reads global memory, the last one writes it.
// The rows' results lie in the map's own first in_len rows: a CTA of the
// second pass reads its columns before it writes them, whole 128-byte lines
// for transforms of up to 512 points, so the search needs no work space.
// 256 x 1024 values into 512 x 8192 bins: 14.3 + 21.7 us (radix-2 passes in
// shared memory, a transposed write of the lags and a pass of its own for the
// peak took 66.6 + 70.7 + 11.0 us).
template <int n, bool COLS, bool PEAK>
__global__ void __launch_bounds__(Radices<n>::T * Batch<n, COLS>::C)
k_cfft_inv(const float2* in, int in_len, int64_t in_q, int64_t in_i, float2* out, int64_t out_q, int64_t out_i,
           int count, PeakSlot* slot) {
  using P = Radices<n>;
  constexpr int T = P::T, C = Batch<n, COLS>::C, PER = n / P::R0 / T;
  extern __shared__ __align__(16) float2 cfft_buf[];
  const int c = COLS ? threadIdx.x % C : threadIdx.x / T;
  const int t = COLS ? threadIdx.x / C : threadIdx.x % T;
  const int q = blockIdx.x * C + c;
  const bool mine = q < count;
  if (!PEAK && blockIdx.x == 0 && threadIdx.x == 0) {  // the next pass finds the slot cleared
    slot->best = 0ull;
    slot->done = 0u;
  }
  unsigned long long key = 0ull;
  auto store = [&](int i, float2 v) {
    if (!mine) return;
    v = swp(v);
    out[q * out_q + i * out_i] = v;
    if constexpr (PEAK) {
      const unsigned long long k = peak_key(v, (uint32_t)(q * out_q + i * out_i));
      key = k > key ? k : key;
    }
  };
  float2 v[PER][P::R0];
#pragma unroll
  for (int u = 0; u < PER; ++u)
#pragma unroll
    for (int r = 0; r < P::R0; ++r) {
      const int i = t + u * T + r * (n / P::R0);
      v[u][r] = mine && i < in_len ? swp(in[q * in_q + i * in_i]) : make_float2(0.f, 0.f);
    }
  float2* table = cfft_buf + Batch<n, COLS>::POINTS;
  if constexpr (P::R1 > 1)  // while the points arrive
    for (int e = threadIdx.x; e < Batch<n, COLS>::TWIDDLES; e += T * C)
      table[e] = root<P::R0 * P::R1>((e / P::R0 + 1) * (e % P::R0));
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    dft_reg<P::R0>(v[u], TurnW32Exact());
#pragma unroll
    for (int r = 0; r < P::R0; ++r) {
      if constexpr (P::R1 == 1) store(r, v[u][r]);
      else cfft_buf[at<n, COLS>((t + u * T) * P::R0 + r, c)] = v[u][r];
    }
  }
  if constexpr (P::R1 > 1) {
    __syncthreads();
    cfft_pass<n, P::R1, P::R0, COLS>(cfft_buf, table, t, c, store);
    if constexpr (P::R2 > 1) cfft_pass<n, P::R2, P::R0 * P::R1, COLS>(cfft_buf, table, t, c, store);
  }
  if constexpr (PEAK) {
    __threadfence();  // the map's values, for the CTA that reads the peak's
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long other = __shfl_down_sync(0xffffffffu, key, o);
      key = other > key ? other : key;
    }
    __shared__ unsigned long long ws[32];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = key;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < (int)(blockDim.x >> 5); ++w) key = ws[w] > key ? ws[w] : key;
      atomicMax(&slot->best, key);
      __threadfence();
      if (atomicAdd(&slot->done, 1u) == gridDim.x - 1) {
        __threadfence();
        const unsigned long long best = atomicMax(&slot->best, 0ull);
        slot->value = __ldcg(out + (0xFFFFFFFFu - (uint32_t)best));
      }
    }
  }
}

template <int n, bool COLS, bool PEAK>
cudaError_t launch_cfft_n(const float2* in, int in_len, int64_t in_q, int64_t in_i, float2* out, int64_t out_q,
                          int64_t out_i, int count, PeakSlot* slot, cudaStream_t st) {
  constexpr int C = Batch<n, COLS>::C;
  constexpr size_t smem = sizeof(float2) * (Batch<n, COLS>::POINTS + Batch<n, COLS>::TWIDDLES);
  cudaError_t e = cudaFuncSetAttribute(k_cfft_inv<n, COLS, PEAK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_cfft_inv<n, COLS, PEAK><<<(count + C - 1) / C, Radices<n>::T * C, smem, st>>>(in, in_len, in_q, in_i, out, out_q,
                                                                                 out_i, count, slot);
  return cudaGetLastError();
}

template <bool COLS, bool PEAK, typename... A>
cudaError_t launch_cfft(int n, A... a) {
  switch (n) {
    case 2: return launch_cfft_n<2, COLS, PEAK>(a...);
    case 4: return launch_cfft_n<4, COLS, PEAK>(a...);
    case 8: return launch_cfft_n<8, COLS, PEAK>(a...);
    case 16: return launch_cfft_n<16, COLS, PEAK>(a...);
    case 32: return launch_cfft_n<32, COLS, PEAK>(a...);
    case 64: return launch_cfft_n<64, COLS, PEAK>(a...);
    case 128: return launch_cfft_n<128, COLS, PEAK>(a...);
    case 256: return launch_cfft_n<256, COLS, PEAK>(a...);
    case 512: return launch_cfft_n<512, COLS, PEAK>(a...);
    case 1024: return launch_cfft_n<1024, COLS, PEAK>(a...);
    case 2048: return launch_cfft_n<2048, COLS, PEAK>(a...);
    case 4096: return launch_cfft_n<4096, COLS, PEAK>(a...);
    case 8192: return launch_cfft_n<8192, COLS, PEAK>(a...);
    case 16384: return launch_cfft_n<16384, COLS, PEAK>(a...);
    default: return cudaErrorInvalidValue;
  }
}

bool is_fft_length(int n) { return n >= 2 && n <= kMaxFft && (n & (n - 1)) == 0; }

// A slot for one search, given back when it goes out of scope; slots beyond
// the static ones come from the stream's memory pool.
struct PeakLease {
  PeakSlot* dev = nullptr;
  int index = -1;
  cudaStream_t st;
  explicit PeakLease(cudaStream_t s) : st(s) {
    unsigned long long taken = g_peak_taken.load();
    while (~taken) {
      const int i = __builtin_ctzll(~taken);
      if (!g_peak_taken.compare_exchange_weak(taken, taken | (1ull << i))) continue;
      index = i;
      void* base = nullptr;
      if (cudaGetSymbolAddress(&base, g_peak_slots) == cudaSuccess) dev = reinterpret_cast<PeakSlot*>(base) + i;
      return;
    }
    void* p = nullptr;
    if (cudaMallocAsync(&p, sizeof(PeakSlot), st) == cudaSuccess) dev = reinterpret_cast<PeakSlot*>(p);
  }
  ~PeakLease() {
    if (index >= 0) g_peak_taken.fetch_and(~(1ull << index));
    else if (dev) cudaFreeAsync(dev, st);
  }
  PeakLease(const PeakLease&) = delete;
};

}  // namespace

}  // namespace corr

using namespace corr;

extern "C" int corr_fringe_search(const float* dev_vis, int nsub, int nchan, int pad_rate, int pad_delay,
                                  float* dev_map, int* peak_rate, int* peak_lag, float* peak_amp,
                                  float* peak_value, void* cuda_stream) {
  if (!dev_vis || !dev_map || nsub < 1 || nchan < 1) return CORR_EINVAL;
  if (!is_fft_length(pad_rate) || !is_fft_length(pad_delay) || pad_rate < nsub || pad_delay < nchan ||
      (int64_t)pad_rate * pad_delay > ((int64_t)1 << 26))
    return CORR_EINVAL;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const float2* V = reinterpret_cast<const float2*>(dev_vis);
  float2* M = reinterpret_cast<float2*>(dev_map);
  const int64_t count = (int64_t)pad_rate * pad_delay;
  cudaError_t e = fstage_ensure_constants();
  PeakLease lease(st);
  // the lag transforms [nsub][pad_delay]: the map's first rows, unless the
  // visibilities themselves lie in the map
  float2* X1 = M;
  void* buf = nullptr;
  const uintptr_t v0 = (uintptr_t)V, v1 = v0 + sizeof(float2) * (size_t)nsub * nchan, m0 = (uintptr_t)M,
                  m1 = m0 + sizeof(float2) * (size_t)count;
  if (!lease.dev || (v0 < m1 && m0 < v1 &&
                     cudaMallocAsync(&buf, sizeof(float2) * (size_t)pad_delay * nsub, st) != cudaSuccess)) {
    cudaGetLastError();
    return CORR_ENOMEM;
  }
  if (buf) X1 = reinterpret_cast<float2*>(buf);
  // over channels: row t of V -> X1[t][l]; over sub-integrations: column l of X1 -> M[r][l]
  if (e == cudaSuccess)
    e = launch_cfft<false, false>(pad_delay, V, nchan, (int64_t)nchan, (int64_t)1, X1, (int64_t)pad_delay, (int64_t)1, nsub,
                                  lease.dev, st);
  if (e == cudaSuccess)
    e = launch_cfft<true, true>(pad_rate, (const float2*)X1, nsub, (int64_t)1, (int64_t)pad_delay, M, (int64_t)1,
                                (int64_t)pad_delay, pad_delay, lease.dev, st);
  PeakSlot peak = {};
  if (e == cudaSuccess) e = cudaMemcpyAsync(&peak, lease.dev, sizeof(peak), cudaMemcpyDeviceToHost, st);
  // on an error too: the slot is given back only when nothing in flight writes it
  const cudaError_t waited = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = waited;
  if (buf) cudaFreeAsync(buf, st);
  const int64_t idx = (int64_t)(0xFFFFFFFFu - (uint32_t)(peak.best & 0xFFFFFFFFull));
  if (e == cudaSuccess && (idx < 0 || idx >= count)) e = cudaErrorUnknown;
  if (e != cudaSuccess) {
    cudaGetLastError();
    return CORR_ECUDA;
  }
  if (peak_rate) *peak_rate = (int)(idx / pad_delay);
  if (peak_lag) *peak_lag = (int)(idx % pad_delay);
  if (peak_amp) {
    const uint32_t bits = (uint32_t)(peak.best >> 32);
    memcpy(peak_amp, &bits, sizeof(float));
  }
  if (peak_value) {
    peak_value[0] = peak.value.x;
    peak_value[1] = peak.value.y;
  }
  return CORR_OK;
}
