// k_xstage.cu -- the X step of the FX correlator on CUDA cores in FP32 (the
// paper, Abstract: after the Fourier transform every station pair is
// cross-multiplied).  For each stream g and channel k, over the FFT blocks of
// a chunk:  V_ab[k] += X_a[k] conj(X_b[k]) for every baseline a <= b
// (autocorrelations included, parallel hands only).
//
// A lane owns one channel of one stream and all baselines of a tile of TS
// stations (a <= b), or of two different tiles (TS x TS), in registers, so
// each value read from shared memory meets TS others.  Up to 12 stations are
// one tile (k_xmac); more are split into tiles of 5 to 8, and the warps of a
// CTA hold up to 12 tile pairs of the same 32 channels, so that a station's
// values are fetched once for all of them (k_xpairs).  The blocks of a chunk
// are split into KZ ranges; each range sums at most 256 blocks in registers
// and then adds that partial into its own FP32 accumulator slice part[kz], one
// add per element and launch, so results are deterministic and the FP32 sums
// stay short (hierarchical accumulation).
#include "corr_internal.cuh"

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <cudaTypedefs.h>

#include <string.h>

#include <algorithm>
#include <type_traits>

namespace corr {

namespace {

// acc + x conj(y) on packed FP32 pairs: acc + x (y.x, y.x) + xr (y.y, y.y)
// with xr = (x.y, -x.x), formed once per loaded value: two f32x2 fused
// multiply-adds per baseline instead of four scalar ones.
__device__ __forceinline__ float2 cmac_conj(float2 acc, float2 x, float2 xr, float2 y) {
  return __ffma2_rn(xr, make_float2(y.y, y.y), __ffma2_rn(x, make_float2(y.x, y.x), acc));
}
__device__ __forceinline__ float2 rot_conj(float2 x) { return __fmul2_rn(make_float2(x.y, x.x), make_float2(1.f, -1.f)); }
// An autocorrelation needs only |x|^2: the accumulator keeps (sum re^2,
// sum im^2), one f32x2 FMA per block; auto_value() forms the visibility.
__device__ __forceinline__ float2 cmac_auto(float2 acc, float2 x) { return __ffma2_rn(x, x, acc); }
__device__ __forceinline__ float2 auto_value(float2 acc) { return make_float2(acc.x + acc.y, 0.f); }

constexpr long long kXDrainLimit = 1LL << 26;  // spins per wait while draining after an abort
constexpr int kMaxStages = 8;                  // ring depth
constexpr int kGroupWarps = 12;                // tile pairs per CTA (168 registers a thread at TS = 8)
constexpr int kGroupTiles = 8;                 // station tiles a CTA stages
constexpr int kOneTile = 12;                   // stations held as one tile
constexpr int kMaxXStations = 2 * kMaxStations;

// What one CTA of the many-station form works on: the station tiles that it
// stages, and per warp the places in that list of its tile pair (equal: the
// baselines inside a tile).
struct XGroup {
  uint8_t nwarp, ntile;
  uint8_t tile[kGroupTiles];
  uint8_t wa[kGroupWarps], wb[kGroupWarps];
};
constexpr int kMaxTiles = kMaxXStations / 8;  // 8 is the tile above 64 stations
constexpr int kMaxGroups = 2 * (kMaxTiles * (kMaxTiles + 1) / 2) / kGroupWarps;
struct XGroups {
  int n;
  XGroup g[kMaxGroups];
};

__device__ __forceinline__ uint32_t xs_u32(const void* ptr) { return (uint32_t)__cvta_generic_to_shared(ptr); }

// One spectrum value of lane `i` from the ring as FP32 (the FP16 / E4M3
// values carry X * 2^-sigma; the normalisation takes the 2^(2 sigma) back out).
template <int IN>
__device__ __forceinline__ float2 ring_value(const unsigned char* st, int i) {
  if constexpr (IN == 0) {
    return reinterpret_cast<const float2*>(st)[i];
  } else if constexpr (IN == 1) {
    return __half22float2(reinterpret_cast<const __half2*>(st)[i]);
  } else {
    const __half2_raw h = __nv_cvt_fp8x2_to_halfraw2(reinterpret_cast<const __nv_fp8x2_storage_t*>(st)[i], __NV_E4M3);
    return __half22float2(__half2(h));
  }
}

constexpr int spec_bytes(int in) { return in == 0 ? 8 : (in == 1 ? 4 : 2); }  // per complex value

// Bounded wait for a phase of an mbarrier: gives up when the CTA's abort flag
// is set or after `limit` polls.
__device__ __forceinline__ bool ring_poll(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
               : "=r"(ok)
               : "r"(xs_u32(bar)), "r"(parity)
               : "memory");
  return ok;
}
__device__ __forceinline__ bool ring_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, long long limit) {
  for (long long it = 0; it < limit; ++it) {
    if (ring_poll(bar, parity)) return true;
    if ((it & 1023) == 1023 && *abort_flag) return false;
  }
  return false;
}

// A ring of shared-memory stages filled by tensor copies.  Each stage has an
// mbarrier `full` (the copies' byte count) and `empty` (one arrival per
// reading warp).  At its iteration q one of the warps, each in its turn, refills
// the slot of stage q - 2: issuing copies holds a warp up for most of a
// thousand cycles, and waiting for the slowest reader of stage q - 1 would
// hold up the whole CTA (64 stations x 8 streams x 4096 channels x 128 blocks:
// 1.58 ms; warp 0 refilling each time 1.69, slot q - 1 instead 2.33).
struct Ring {
  uint64_t *full, *empty;
  volatile int* abort_flag;
  RingLog<kMaxStages>* log;  // the copies issued
  int stages;
  long long limit;

  __device__ __forceinline__ void init(int readers) {
    if (threadIdx.x == 0) {
      for (int i = 0; i < stages; ++i) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(xs_u32(&full[i])));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(xs_u32(&empty[i])), "r"(readers));
      }
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      *abort_flag = 0;
      log->clear();
    }
    __syncthreads();
  }
  // at stage q, held in `slot` with parity `phase`: the place of stage q - 2, once every warp has read it (-1: gave
  // up, here or in another warp before)
  __device__ __forceinline__ int reclaim(int slot, uint32_t phase) const {
    const int old = slot >= 2 ? slot - 2 : slot - 2 + stages;
    const int stop = *abort_flag;  // read first: its latency passes behind the wait's
    if (ring_wait(&empty[old], old > slot ? phase ^ 1 : phase, abort_flag, limit) && !stop) return old;
    *abort_flag = 1;
    return -1;
  }
  // a warp has read stage slot `slot`
  __device__ __forceinline__ void release(int slot) const {
    __syncwarp();
    if ((threadIdx.x & 31) == 0)
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(xs_u32(&empty[slot])) : "memory");
  }
  // After an abort, with every warp of the CTA past its last issue: let the
  // copies in flight land before the CTA's shared memory goes away.
  __device__ __forceinline__ void drain(int* err) const {
    log->for_each(stages, [&](int slot, unsigned parity) {
      for (long long it = 0; it < kXDrainLimit; ++it)
        if (ring_poll(&full[slot], parity)) break;
    });
    if (err) atomicExch(err, 1);
  }
};

// The accumulators of one tile pair and their update by one block: `ra` and
// `rb` point at the tiles' staged rows of this lane's channel.
template <int TS, int IN, bool DIAG>
__device__ __forceinline__ void tile_block(float2 (&acc)[TS][TS], const unsigned char* ra, const unsigned char* rb,
                                           int row_bytes) {
  float2 b[TS];
#pragma unroll
  for (int j = 0; j < TS; ++j) b[j] = ring_value<IN>(rb + j * row_bytes, 0);
#pragma unroll
  for (int i = 0; i < TS; ++i) {
    const float2 a = DIAG ? b[i] : ring_value<IN>(ra + i * row_bytes, 0);
    const float2 ar = rot_conj(a);
#pragma unroll
    for (int j = DIAG ? i : 0; j < TS; ++j)
      acc[i][j] = (DIAG && j == i) ? cmac_auto(acc[i][j], a) : cmac_conj(acc[i][j], a, ar, b[j]);
  }
}

// Add a tile pair's sums to the partial sums: part[baseline * row] of this
// lane's stream and channel, one add per element and launch (the first
// launch of an integration writes them, so that nothing clears them before).
template <int TS, bool DIAG>
__device__ __forceinline__ void add_tile(const float2 (&acc)[TS][TS], float2* part, size_t row, int a0, int b0, int S,
                                         int first) {
#pragma unroll
  for (int i = 0; i < TS; ++i)
#pragma unroll
    for (int j = DIAG ? i : 0; j < TS; ++j)
      if (a0 + i < S && b0 + j < S) {
        float2* dst = part + (size_t)bl_index(a0 + i, b0 + j, S) * row;
        if (first)
          *dst = DIAG && j == i ? auto_value(acc[i][j]) : acc[i][j];
        else if (DIAG && j == i)
          atomicAdd(&dst->x, auto_value(acc[i][j]).x);
        else
          asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(dst), "f"(acc[i][j].x), "f"(acc[i][j].y) : "memory");
      }
}

// CTAs per SM of the one-tile form: TS (TS + 1) accumulators a lane.
constexpr int one_tile_ctas(int TS) { return TS <= 5 ? 6 : TS <= 8 ? 4 : TS <= 11 ? 3 : 2; }

struct XShape {
  int nb;          // blocks per ring stage
  int nst;         // ring stages
  int cg;          // channel groups of 32, one warp each (k_xmac)
  int pitch;       // channels per staged row: 32 cg, or nchan if fewer
  int tile_bytes;  // nb blocks of one tile, rounded up to the copies' 128-byte alignment
  int stage_bytes;
};

// Up to 12 stations: one CTA of cg warps takes 32 cg channels of stream
// blockIdx.y and block range blockIdx.z.  Its ring's stages hold nb blocks of
// all stations, [block][station][channel], each filled by one tensor copy.
// Every wait is bounded (timeout -> *err; the CTA stops and lets its copies
// land).
//
// FP32 spectra: bound by HBM.  FP16 / E4M3 spectra: by the FMA pipe and the
// register moves of its paired operands (one lane for all 55 baselines of ten
// stations reads 10 values a block, where two lanes with half the baselines
// each read 17).  A stage takes as many blocks as four of them fit: a copy
// costs the copy engine about 13 cycles per row of up to 1 KB on top of about
// 60, and a stage its warps' waits.  Ten stations x 16 streams x 1024
// channels, 819 blocks: FP32 167 us (6.4 TB/s), FP16 129, E4M3 123 us; with two
// lanes a channel and two barriers a stage 178, 151 and 150 us.
template <int TS, int IN>
__global__ void __launch_bounds__(128, one_tile_ctas(TS))
k_xmac(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ XParams p, const XShape sh) {
  extern __shared__ __align__(128) unsigned char ring_raw[];
  unsigned char* data = ring_raw + ((128u - (xs_u32(ring_raw) & 127u)) & 127u);
  __shared__ __align__(8) uint64_t s_full[kMaxStages], s_empty[kMaxStages];
  __shared__ volatile int s_abort;
  __shared__ RingLog<kMaxStages> s_log;
  constexpr int EB = spec_bytes(IN);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k0 = blockIdx.x * 32 * sh.cg;
  const int k = k0 + threadIdx.x;
  const int g = blockIdx.y, kz = blockIdx.z;
  const int b_lo = (int)((int64_t)p.CB * kz / p.KZ);
  const int b_hi = (int)((int64_t)p.CB * (kz + 1) / p.KZ);
  if (b_hi <= b_lo && !p.first) return;  // an empty range of the first chunk writes zeros
  const int nst = (b_hi - b_lo + sh.nb - 1) / sh.nb;
  const int row_bytes = sh.pitch * EB;
  Ring ring{s_full, s_empty, &s_abort, &s_log, sh.nst, p.wait_limit};
  ring.init(sh.cg);
  auto issue = [&](int q, int slot) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(xs_u32(&s_full[slot])),
                 "r"(sh.nb * TS * row_bytes)
                 : "memory");
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(xs_u32(data) + (uint32_t)(slot * sh.stage_bytes)),
        "l"(reinterpret_cast<uint64_t>(&tmap)), "r"(2 * k0), "r"(0), "r"(g * p.CB + b_lo + q * sh.nb),
        "r"(xs_u32(&s_full[slot]))
        : "memory");
    s_log.note(slot, q);
  };
  if (threadIdx.x == 0)
    for (int q = 0; q < sh.nst && q < nst; ++q) issue(q, q);

  float2 acc[TS][TS];
#pragma unroll
  for (int i = 0; i < TS; ++i)
#pragma unroll
    for (int j = i; j < TS; ++j) acc[i][j] = make_float2(0.f, 0.f);
  int slot = 0, turn = 0;
  uint32_t phase = 0;
  // lanes beyond the staged channels read the row's first value (their sums are not used)
  const int lane_off = ((int)threadIdx.x < sh.pitch ? (int)threadIdx.x : 0) * EB;
  for (int q = 0; q < nst; ++q) {
    if (q >= 2 && q - 2 + sh.nst < nst && warp == turn && lane == 0) {
      const int old = ring.reclaim(slot, phase);
      if (old >= 0) issue(q - 2 + sh.nst, old);
    }
    if (++turn == sh.cg) turn = 0;
    __syncwarp();
    if (!ring_wait(&s_full[slot], phase, &s_abort, p.wait_limit)) {
      s_abort = 1;
      break;
    }
    const unsigned char* st = data + slot * sh.stage_bytes + lane_off;
    const int nb = min(sh.nb, b_hi - b_lo - q * sh.nb);
    for (int bi = 0; bi < nb; ++bi, st += TS * row_bytes) tile_block<TS, IN, true>(acc, st, st, row_bytes);
    ring.release(slot);
    if (++slot == sh.nst) {
      slot = 0;
      phase ^= 1;
    }
  }
  if (k < p.nchan) {
    const size_t row = (size_t)p.G * p.nchan;
    add_tile<TS, true>(acc, p.part + (size_t)kz * nbl_of(TS) * row + (size_t)g * p.nchan + k, row, 0, 0, TS,
                       p.first);
  }
  __syncthreads();
  if (s_abort && threadIdx.x == 0) ring.drain(p.err);
}

// More than 12 stations: one CTA takes the tile pairs of group blockIdx.x %
// groups (the groups of the same 32 channels are neighbours, so that they
// share L2 lines), stream blockIdx.y and block range blockIdx.z.  A ring stage
// holds nb blocks of the group's tiles, [tile][block][station][channel], one
// tensor copy per tile.
//
// Bound by the FMA pipe and the register moves of its paired operands: at TS =
// 8 a warp issues 136 packed FMAs (two cycles each) for 16 shared-memory loads
// a block.  Twelve pairs a CTA need a station's values from L2 less than half
// as often as single 8 x 8 pairs, whose L2 traffic bound the step before.
// Copies of 256-byte rows run at about 13 cycles a row plus 60 a copy, hence
// several blocks per copy (single blocks reach 3.9 TB/s where the FMAs consume
// 5.5); 16-byte cp.async copies by the multiplying warps took as much of their
// time again as the multiplications (2.08 ms for 64 stations x 8 streams x
// 4096 channels x 128 blocks, 1.60 ms now, 43 TFLOP/s; single 8 x 8 pairs took
// 3.25 ms).
template <int TS>
__global__ void __launch_bounds__(32 * kGroupWarps, 1)
k_xpairs(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ XParams p, const XShape sh,
         const __grid_constant__ XGroups groups) {
  extern __shared__ __align__(128) unsigned char ring_raw[];
  unsigned char* data = ring_raw + ((128u - (xs_u32(ring_raw) & 127u)) & 127u);
  __shared__ __align__(8) uint64_t s_full[kMaxStages], s_empty[kMaxStages];
  __shared__ volatile int s_abort;
  __shared__ RingLog<kMaxStages> s_log;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const XGroup& gr = groups.g[blockIdx.x % groups.n];
  const int k0 = blockIdx.x / groups.n * 32;
  const int g = blockIdx.y, kz = blockIdx.z, S = p.S;
  const int b_lo = (int)((int64_t)p.CB * kz / p.KZ);
  const int b_hi = (int)((int64_t)p.CB * (kz + 1) / p.KZ);
  if (b_hi <= b_lo && !p.first) return;  // an empty range of the first chunk writes zeros
  const int nst = (b_hi - b_lo + sh.nb - 1) / sh.nb;
  const int row_bytes = sh.pitch * 8, nwarp = gr.nwarp;
  Ring ring{s_full, s_empty, &s_abort, &s_log, sh.nst, p.wait_limit};
  ring.init(nwarp);
  auto issue = [&](int q, int slot) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(xs_u32(&s_full[slot])),
                 "r"(gr.ntile * sh.nb * TS * row_bytes)
                 : "memory");
    for (int i = 0; i < gr.ntile; ++i)
      asm volatile(
          "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
          "[%5];" ::"r"(xs_u32(data) + (uint32_t)(slot * sh.stage_bytes + i * sh.tile_bytes)),
          "l"(reinterpret_cast<uint64_t>(&tmap)), "r"(2 * k0), "r"((int)gr.tile[i] * TS),
          "r"(g * p.CB + b_lo + q * sh.nb), "r"(xs_u32(&s_full[slot]))
          : "memory");
    s_log.note(slot, q);
  };
  if (threadIdx.x == 0)
    for (int q = 0; q < sh.nst && q < nst; ++q) issue(q, q);

  // lanes beyond the staged channels read the row's first value (their sums are not used)
  const int lane_off = (lane < sh.pitch ? lane : 0) * 8;
  auto run = [&](auto diag, int wa, int wb) {
    constexpr bool DIAG = decltype(diag)::value;
    float2 acc[TS][TS];
#pragma unroll
    for (int i = 0; i < TS; ++i)
#pragma unroll
      for (int j = DIAG ? i : 0; j < TS; ++j) acc[i][j] = make_float2(0.f, 0.f);
    int slot = 0, turn = 0;
    uint32_t phase = 0;
    for (int q = 0; q < nst; ++q) {
      if (q >= 2 && q - 2 + sh.nst < nst && warp == turn && lane == 0) {
        const int old = ring.reclaim(slot, phase);
        if (old >= 0) issue(q - 2 + sh.nst, old);
      }
      if (++turn == nwarp) turn = 0;
      __syncwarp();
      if (!ring_wait(&s_full[slot], phase, &s_abort, p.wait_limit)) {
        s_abort = 1;
        break;
      }
      const unsigned char* st = data + slot * sh.stage_bytes + lane_off;
      const int nb = min(sh.nb, b_hi - b_lo - q * sh.nb);
      for (int bi = 0; bi < nb; ++bi, st += TS * row_bytes)
        tile_block<TS, 0, DIAG>(acc, st + wa * sh.tile_bytes, st + wb * sh.tile_bytes, row_bytes);
      ring.release(slot);
      if (++slot == sh.nst) {
        slot = 0;
        phase ^= 1;
      }
    }
    if (k0 + lane < p.nchan) {
      const size_t row = (size_t)p.G * p.nchan;
      add_tile<TS, DIAG>(acc, p.part + (size_t)kz * nbl_of(S) * row + (size_t)g * p.nchan + k0 + lane, row,
                         gr.tile[wa] * TS, gr.tile[wb] * TS, S, p.first);
    }
  };
  if (warp < nwarp) {  // a CTA with fewer pairs than the largest one has warps without work
    const int wa = gr.wa[warp], wb = gr.wb[warp];
    if (wa == wb) run(std::true_type{}, wa, wb);
    else run(std::false_type{}, wa, wb);
  }
  __syncthreads();
  if (s_abort && threadIdx.x == 0) ring.drain(p.err);
}

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
    cudaGetLastError();
    return (PFN_cuTensorMapEncodeTiled_v12000) nullptr;
  }();
  return fn;
}

// Stations per tile above kOneTile: the size whose tile pairs cost least per
// block, counting packed FMAs (an autocorrelation takes one, a baseline two,
// a station one) and each shared-memory load as two of them.  Small tiles
// waste less on stations beyond S, large ones load less: 20 stations go as
// 7 + 7 + 6, not 8 + 8 + 4 or 4 x 5.
int tile_size(int S) {
  if (S > 64) return 8;
  int best = 8;
  long cost = 0;
  for (int ts = 8; ts >= 5; --ts) {
    const long nt = (S + ts - 1) / ts;
    const long c = nt * (ts * ts + 3 * ts) + nt * (nt - 1) / 2 * (2 * ts * ts + 5 * ts);
    if (ts == 8 || c < cost) {
      best = ts;
      cost = c;
    }
  }
  return best;
}

// Tile pairs in CTAs: in blocks of 4 x 4 tiles, so that consecutive pairs
// share tiles (64 stations: 36 pairs in three CTAs that stage 6, 8 and 5 of
// the 8 tiles).  A CTA of 12 warps fills an SM; with fewer pairs, CTAs of a
// size that several of them nearly fill one.
XGroups make_groups(int nt) {
  struct Pair { int a, b; };
  Pair pairs[kMaxTiles * (kMaxTiles + 1) / 2];
  int n = 0;
  for (int I = 0; I < nt; I += 4)
    for (int J = I; J < nt; J += 4)
      for (int a = I; a < std::min(I + 4, nt); ++a)
        for (int b = std::max(a, J); b < std::min(J + 4, nt); ++b) pairs[n++] = {a, b};
  const int least = (n + kGroupWarps - 1) / kGroupWarps;
  int size = kGroupWarps;
  double best = 0.0;
  for (int ng = least; ng < least + 3; ++ng) {
    const int sz = (n + ng - 1) / ng;
    const double warps = (double)(kGroupWarps / sz) * n / ng;
    if (warps > best) {
      best = warps;
      size = sz;
    }
  }
  XGroups out;
  memset(&out, 0, sizeof(out));
  for (int q = 0; q < n;) {
    XGroup& x = out.g[out.n++];
    for (; q < n && x.nwarp < size; ++q) {
      int at[2];
      const int t[2] = {pairs[q].a, pairs[q].b};
      int have = x.ntile;
      for (int e = 0; e < 2; ++e) {
        int i = 0;
        while (i < have && x.tile[i] != t[e]) ++i;
        if (i == have) {
          if (have == kGroupTiles) { i = -1; }
          else x.tile[have++] = (uint8_t)t[e];
        }
        at[e] = i;
        if (i < 0) break;
      }
      if (at[0] < 0 || at[1] < 0) break;  // no room for its tiles: the next CTA's first pair
      x.ntile = (uint8_t)have;
      x.wa[x.nwarp] = (uint8_t)at[0];
      x.wb[x.nwarp++] = (uint8_t)at[1];
    }
    // pairs inside a tile have half the work: first, so that they go to
    // different schedulers (warp % 4)
    for (int w = 0, d = 0; w < x.nwarp; ++w)
      if (x.wa[w] == x.wb[w]) {
        std::swap(x.wa[w], x.wa[d]);
        std::swap(x.wb[w], x.wb[d++]);
      }
  }
  return out;
}

struct XPlan {
  int ts, cg, pitch, ngroup, warps, ctas_per_sm;
  int tiles;  // staged per CTA, at most
};

XPlan plan_for(int S, int nchan, XGroups* groups) {
  XPlan x;
  if (S <= kOneTile) {
    x.ts = S;
    x.cg = nchan >= 128 ? 4 : (nchan + 31) / 32;
    x.pitch = std::min(nchan, 32 * x.cg);
    x.ngroup = x.tiles = 1;
    x.warps = x.cg;
    x.ctas_per_sm = one_tile_ctas(S);
    return x;
  }
  x.ts = tile_size(S);
  x.cg = 1;
  x.pitch = std::min(nchan, 32);
  const XGroups g = make_groups((S + x.ts - 1) / x.ts);
  x.ngroup = g.n;
  x.warps = x.tiles = 0;
  for (int i = 0; i < g.n; ++i) {
    x.warps = std::max(x.warps, (int)g.g[i].nwarp);
    x.tiles = std::max(x.tiles, (int)g.g[i].ntile);
  }
  x.ctas_per_sm = kGroupWarps / x.warps;
  if (groups) *groups = g;
  return x;
}

// The ring of a launch: at least four stages (more if a block is small) of up
// to `most` blocks in a CTA's share of 216 KB of shared memory, and the tensor
// map: the spectra as [stream x block][station][2 nchan scalars], FP32, FP16
// or single bytes (E4M3 pairs); a copy takes 2 pitch scalars (a multiple of 16
// bytes, from a multiple of 64 scalars) x TS stations (zeros beyond S) x nb
// blocks.
template <int TS, int IN>
cudaError_t ring_shape(const XParams& p, const XPlan& x, int most, XShape* sh, CUtensorMap* tm, size_t* smem) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  if (!enc) return cudaErrorNotSupported;
  constexpr int EB = spec_bytes(IN);
  const int block_bytes = TS * x.pitch * EB, budget = 216 * 1024 / x.ctas_per_sm;
  sh->cg = x.cg;
  sh->pitch = x.pitch;
  sh->nb = std::max(1, std::min({most, p.CB / std::max(1, p.KZ), budget / 4 / (x.tiles * block_bytes)}));
  sh->tile_bytes = (sh->nb * block_bytes + 127) & ~127;
  sh->stage_bytes = x.tiles * sh->tile_bytes;
  sh->nst = std::min(kMaxStages, budget / sh->stage_bytes);
  *smem = 128 + (size_t)sh->nst * sh->stage_bytes;
  cuuint64_t dims[3] = {(cuuint64_t)2 * p.nchan, (cuuint64_t)p.S, (cuuint64_t)p.G * p.CB};
  cuuint64_t strides[2] = {(cuuint64_t)p.nchan * EB, (cuuint64_t)p.S * p.nchan * EB};
  cuuint32_t box[3] = {(cuuint32_t)(2 * x.pitch), (cuuint32_t)TS, (cuuint32_t)sh->nb};
  cuuint32_t estr[3] = {1, 1, 1};
  const CUtensorMapDataType dt =
      IN == 0 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : (IN == 1 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8);
  return enc(tm, dt, 3, const_cast<float2*>(p.spec), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? cudaSuccess
             : cudaErrorInvalidValue;
}

template <int TS, int IN>
cudaError_t launch_one_in(const XParams& p_in, const XPlan& x, cudaStream_t s) {
  XParams p = p_in;
  p.wait_limit = wait_limit();
  XShape sh;
  CUtensorMap tm;
  size_t smem = 0;
  cudaError_t e = ring_shape<TS, IN>(p, x, 16, &sh, &tm, &smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_xmac<TS, IN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_xmac<TS, IN><<<dim3((p.nchan + 32 * x.cg - 1) / (32 * x.cg), p.G, p.KZ), 32 * x.cg, smem, s>>>(tm, p, sh);
  return cudaGetLastError();
}

template <int TS>
cudaError_t launch_one(const XParams& p, const XPlan& x, cudaStream_t s) {
  if (p.in_kind == 1) return launch_one_in<TS, 1>(p, x, s);
  if (p.in_kind == 2) return launch_one_in<TS, 2>(p, x, s);
  return launch_one_in<TS, 0>(p, x, s);
}

template <int TS>
cudaError_t launch_pairs(const XParams& p_in, const XPlan& x, const XGroups& groups, cudaStream_t s) {
  XParams p = p_in;
  p.wait_limit = wait_limit();
  XShape sh;
  CUtensorMap tm;
  size_t smem = 0;
  cudaError_t e = ring_shape<TS, 0>(p, x, 4, &sh, &tm, &smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_xpairs<TS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_xpairs<TS><<<dim3(x.ngroup * ((p.nchan + 31) / 32), p.G, p.KZ), 32 * x.warps, smem, s>>>(tm, p, sh, groups);
  return cudaGetLastError();
}

}  // namespace

// Block ranges per chunk.  At least one per 256 blocks, and where that leaves
// sums of more than 24 blocks, (but for an eighth) as many as make 912 ranges of
// 128 channels and 8 x 8 stations: the error of an integration grows with the
// length of its FP32 register sums (43 stations x 5 streams x 512 channels, 104
// blocks: 2.65e-7 from 64 bits in three ranges, 2.90e-7 in one).  Above that the
// number whose CTAs fill whole waves of the SMs, weighed against each CTA's
// start and end (worth about 12 blocks) and the partial sums it adds to memory
// (read and written, against the spectra read).
int xstage_kz(int CB, int S, int G, int nchan) {
  const XPlan x = plan_for(S, nchan, nullptr);
  const int64_t base = (int64_t)x.ngroup * ((nchan + 32 * x.cg - 1) / (32 * x.cg)) * G;
  const int64_t slots = (int64_t)152 * x.ctas_per_sm;
  const int64_t nt = S <= kOneTile ? 1 : (S + 7) / 8;
  const int64_t tiles = (int64_t)((nchan + 127) / 128) * G * (nt * (nt + 1) / 2);
  const int64_t ranges = (912 + tiles - 1) / tiles;
  const int least = (int)std::max<int64_t>({1, (CB + 255) / 256, std::min<int64_t>((CB + 23) / 24, ranges - ranges / 8)});
  const int most = (int)std::min<int64_t>(CB, std::max<int64_t>(least, 3 * slots / base + 1));
  int best = least;
  double score = 0.0;
  for (int kz = least; kz <= most; ++kz) {
    const int64_t ctas = base * kz, waves = (ctas + slots - 1) / slots;
    const double nb = (double)CB / kz;
    const double v = (double)ctas / (double)(waves * slots) * nb / (nb + 12.0) / (1.0 + (S + 1.0) / nb);
    if (v > score) {
      score = v;
      best = kz;
    }
  }
  return std::min(best, std::max(1, CB));
}

bool xstage_reduced_supported(int S, int nchan) {
  return S >= 1 && S <= kOneTile && nchan >= 128 && nchan % 128 == 0 && tensor_map_encoder() != nullptr;
}

cudaError_t launch_xstage(const XParams& p, cudaStream_t s) {
  if (p.CB <= 0) return cudaSuccess;
  if (p.in_kind != 0 && !xstage_reduced_supported(p.S, p.nchan)) return cudaErrorNotSupported;
  if (p.S > kMaxXStations) return cudaErrorInvalidValue;
  XGroups groups;
  const XPlan x = plan_for(p.S, p.nchan, &groups);
  if (p.S <= kOneTile) {
    switch (x.ts) {
      case 1: return launch_one<1>(p, x, s);
      case 2: return launch_one<2>(p, x, s);
      case 3: return launch_one<3>(p, x, s);
      case 4: return launch_one<4>(p, x, s);
      case 5: return launch_one<5>(p, x, s);
      case 6: return launch_one<6>(p, x, s);
      case 7: return launch_one<7>(p, x, s);
      case 8: return launch_one<8>(p, x, s);
      case 9: return launch_one<9>(p, x, s);
      case 10: return launch_one<10>(p, x, s);
      case 11: return launch_one<11>(p, x, s);
      case 12: return launch_one<12>(p, x, s);
      default: return cudaErrorInvalidValue;
    }
  }
  switch (x.ts) {
    case 5: return launch_pairs<5>(p, x, groups, s);
    case 6: return launch_pairs<6>(p, x, groups, s);
    case 7: return launch_pairs<7>(p, x, groups, s);
    default: return launch_pairs<8>(p, x, groups, s);
  }
}

}  // namespace corr
