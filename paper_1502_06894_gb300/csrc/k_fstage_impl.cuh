// k_fstage_impl.cuh -- the F-step kernel template shared by the real-transform
// (post-F rotation) and the pre-F rotation translation units.  Internal: each
// including translation unit gets its own copy of the radix-32 constant table
// (c_w32) and loads it through its own init function.
#pragma once
#include "corr_internal.cuh"

#include <cuda_fp8.h>

#include <algorithm>
#include <type_traits>
#include <math.h>

namespace corr {

// Complex value -> two E4M3 bytes (Re in the low byte), round to nearest,
// saturating at +-448.
__device__ __forceinline__ uint32_t fp8x2(float re, float im) {
  return (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(re, im), __NV_SATFINITE, __NV_E4M3);
}


static __constant__ float2 c_w32[32];   // exp(-2 pi i m / 32)
static __constant__ float2 c_w32n[32];  // (-Im, Im) of the same, the second operand of a packed product

static cudaError_t init_w32() {
  float2 h[32], hn[32];
  for (int m = 0; m < 32; ++m) {
    double a = -2.0 * 3.14159265358979323846 * (double)m / 32.0;
    h[m] = make_float2((float)cos(a), (float)sin(a));
    hn[m] = make_float2(-h[m].y, h[m].y);
  }
  cudaError_t e = cudaMemcpyToSymbol(c_w32, h, sizeof(h));
  if (e != cudaSuccess) return e;
  return cudaMemcpyToSymbol(c_w32n, hn, sizeof(hn));
}

__host__ __device__ constexpr int ilog2c(int x) { return x <= 1 ? 0 : 1 + ilog2c(x >> 1); }
__host__ __device__ constexpr int bitrevc(int x, int bits) {
  int r = 0;
  for (int i = 0; i < bits; ++i) r |= ((x >> i) & 1) << (bits - 1 - i);
  return r;
}

// Complex arithmetic on packed FP32 pairs: one f32x2 instruction (add, mul
// or fma) computes both parts of a complex value with the rounding of two
// scalar instructions, which halves the instructions of the FFT butterflies
// and products (the F kernels are bound by instruction issue); the swapped
// and broadcast operands below are operand selections, not extra moves.
__device__ __forceinline__ float2 f2add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 f2sub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 f2mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 f2fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 swp(float2 a) { return make_float2(a.y, a.x); }
__device__ __forceinline__ float2 bc(float x) { return make_float2(x, x); }

// a b = (a.x b.x - a.y b.y, a.y b.x + a.x b.y) = a (b.x, b.x) + swap(a) (-b.y, b.y)
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return f2fma(swp(a), make_float2(-b.y, b.y), f2mul(a, bc(b.x)));
}
// a W_32^m, the second operand pair read ready-made from c_w32n
struct TurnW32 {
  __device__ __forceinline__ float2 operator()(float2 a, int m) const {
    return f2fma(swp(a), c_w32n[m], f2mul(a, bc(c_w32[m].x)));
  }
};

// Shared FFT buffers insert one padding element after every P elements (P =
// the first pass's radix): pass 0 stores each thread's P outputs contiguously,
// so without padding the threads of a half-warp would hit the same banks.
template <int P>
__device__ __forceinline__ int padp(int i) { return i + (i >> ilog2c(P)); }

// In-register DFT of R points (R <= 32): radix-2 decimation in frequency,
// natural-order input, output permuted back to natural order.  A difference
// whose twiddle is -i stays unrotated: the next stage adds it through the
// multiply-add that its butterfly needs anyway (the product by +-1 is exact, so
// the rounding is that of the rotation and the addition), which takes 228
// packed instructions for 32 points instead of 243, the bound of this routine
// (two cycles each: 491 -> 460 cycles).  `turn(d, m)` is d W_32^m.
template <int R, typename Turn = TurnW32>
__device__ __forceinline__ void dft_reg(float2 (&v)[R], Turn turn = Turn()) {
  constexpr int LOG = ilog2c(R);
#pragma unroll
  for (int st = 0; st < LOG; ++st) {
    const int half = R >> (st + 1);
#pragma unroll
    for (int i = 0; i < R; i += 2 * half) {
#pragma unroll
      for (int k = 0; k < half; ++k) {
        const float2 a = v[i + k], b = v[i + k + half];
        // the first element of a group of differences: b stands for -i b
        const bool turned = st > 0 && k == 0 && ((i / (2 * half)) & 1);
        const float2 pm = make_float2(1.f, -1.f), mp = make_float2(-1.f, 1.f);
        v[i + k] = turned ? f2fma(swp(b), pm, a) : f2add(a, b);
        const float2 d = turned ? f2fma(swp(b), mp, a) : f2sub(a, b);
        const int m = k * (32 / (2 * half));  // W_{2 half}^k = W_32^m
        v[i + k + half] = (m == 0 || m == 8) ? d : turn(d, m);
      }
    }
  }
  float2 t[R];
#pragma unroll
  for (int r = 0; r < R; ++r) t[r] = v[bitrevc(r, LOG)];
#pragma unroll
  for (int r = 0; r < R; ++r) v[r] = t[r];
}

// Barrier of one FFT group of T threads (groups are T consecutive threads).
// Groups skip their transform independently (a block that is not valid), so
// a group never waits for lanes outside it: groups smaller than a warp sync
// on their own lane mask, larger ones on a named barrier of their own.
template <int T>
__device__ __forceinline__ void gsync(int grp) {
  if constexpr (T == 1) {
    // one thread: program order suffices
  } else if constexpr (T < 32) {
    const unsigned lane = threadIdx.x & 31u;
    __syncwarp(((1u << T) - 1u) << (lane & ~(unsigned)(T - 1)));
  } else if constexpr (T == 32) {
    __syncwarp();
  } else {
    asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(T) : "memory");
  }
}

// v[r] *= W^{kr} for r = 1..R-1 from wp[i] = W^{k 2^i}.  r splits into its
// low LO bits a and its high bits b: W^{kr} = A[a] B[b] with A[a] = W^{ka}
// and B[b] = W^{k 2^LO b}, each the product of the wp of its bits.  Only the
// two short tables stay live (not one power per r), and every index is fixed
// at compile time, so all values stay in registers.
template <int N, int r = 1>
__device__ __forceinline__ void power_table(float2 (&A)[N], const float2* wp) {
  if constexpr (r < N) {
    constexpr int hb = ilog2c(r);
    if constexpr (r == (1 << hb))
      A[r] = wp[hb];
    else
      A[r] = cmul(A[r - (1 << hb)], wp[hb]);
    power_table<N, r + 1>(A, wp);
  }
}

template <int R, int NA, int NB, int r = 1>
__device__ __forceinline__ void apply_powers(float2 (&v)[R], const float2 (&A)[NA], const float2 (&B)[NB]) {
  if constexpr (r < R) {
    constexpr int a = r % NA, b = r / NA;
    if constexpr (a != 0 && b != 0)
      v[r] = cmul(cmul(v[r], A[a]), B[b]);
    else if constexpr (a != 0)
      v[r] = cmul(v[r], A[a]);
    else
      v[r] = cmul(v[r], B[b]);
    apply_powers<R, NA, NB, r + 1>(v, A, B);
  }
}

template <int R, int LOGR>
__device__ __forceinline__ void twiddle_products(float2 (&v)[R], const float2 (&wp)[LOGR]) {
  constexpr int LO = LOGR / 2;
  constexpr int NA = 1 << LO, NB = 1 << (LOGR - LO);
  float2 A[NA], B[NB];
  power_table<NA>(A, wp);
  power_table<NB>(B, wp + LO);
  apply_powers<R, NA, NB>(v, A, B);
}

// A later Stockham pass: read R points per butterfly group, twiddle, DFT,
// write back in place (all reads of the group finish before any write).
// W_{NS R}^{k r} = W_L^{k r L/(NS R)} = W_N^{TWS k r L/(NS R)} (TWS = N / L:
// 2 for the real transform packed into L = N/2 points, 1 for the complex
// N-point transform of the pre-F rotation).  For the last pass (NS R = L)
// from the shared table s_twl[r NS + k] when given; otherwise the powers
// W^k, W^2k, W^4k, ... come from the global table and W^{kr} is their
// product over the bits of r (at most log2 R - 1 multiplications deep),
// which keeps the memory pipeline, the bottleneck of the large transforms,
// to log2 R loads per butterfly group.  Those loads depend on the thread
// only, so they are issued first and their latency passes while the group
// reads its points and waits at the barrier.  With s_twp (transforms of
// 2048+ points) the powers come from a shared table [i][k] of the pass
// instead: consecutive k in consecutive words, read after the barrier.
//
// stockham_values leaves the results of butterfly group j = t + uT, point
// (j / NS) NS R + (j mod NS) + r NS, in v[u][r].  `load(u, r)` reads its point
// j + r L/R, `loaded()` follows the reads.
template <int L, int R, int NS, int T, int TWS, typename Load, typename Loaded>
__device__ __forceinline__ void stockham_values(Load load, Loaded loaded, int t, const float2* __restrict__ twN,
                                                const float2* __restrict__ s_twl, const float2* __restrict__ s_twp,
                                                float2 (&v)[L / R / T][R]) {
  constexpr int GROUPS = L / R;
  constexpr int PER = GROUPS / T;
  constexpr int LOGR = ilog2c(R);
  static_assert(PER >= 1 && GROUPS % T == 0, "bad FFT plan");
  const bool tab = NS * R == L && s_twl != nullptr;
  const bool ptab = !tab && s_twp != nullptr;  // the powers from the shared table of this pass
  float2 wp[PER][LOGR];
  if (!tab && !ptab) {
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int k = (t + u * T) & (NS - 1);
#pragma unroll
      for (int i = 0; i < LOGR; ++i) wp[u][i] = __ldg(&twN[TWS * k * (1 << i) * (L / (NS * R))]);
    }
  }
#pragma unroll
  for (int u = 0; u < PER; ++u)
#pragma unroll
    for (int r = 0; r < R; ++r) v[u][r] = load(u, r);
  loaded();
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int k = (t + u * T) & (NS - 1);
    if (tab) {
#pragma unroll
      for (int r = 1; r < R; ++r) v[u][r] = cmul(v[u][r], s_twl[r * NS + k]);
    } else {
      if (ptab) {
#pragma unroll
        for (int i = 0; i < LOGR; ++i) wp[u][i] = s_twp[i * NS + k];
      }
      twiddle_products<R, LOGR>(v[u], wp[u]);
    }
    dft_reg<R>(v[u]);
  }
}

template <int L, int R, int NS, int T, int P, int TWS = 2>
__device__ __forceinline__ void stockham_pass(float2* __restrict__ buf, int t, int grp,
                                              const float2* __restrict__ twN,
                                              const float2* __restrict__ s_twl = nullptr,
                                              const float2* __restrict__ s_twp = nullptr) {
  constexpr int PER = L / R / T;
  float2 v[PER][R];
  stockham_values<L, R, NS, T, TWS>([&](int u, int r) { return buf[padp<P>(t + u * T + r * (L / R))]; },
                                    [&] { gsync<T>(grp); }, t, twN, s_twl, s_twp, v);
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int j = t + u * T;
    const int idxD = (j / NS) * NS * R + (j & (NS - 1));
#pragma unroll
    for (int r = 0; r < R; ++r) buf[padp<P>(idxD + r * NS)] = v[u][r];
  }
  gsync<T>(grp);
}

// Where a three-pass transform keeps the points between its second and third
// pass.  The second pass writes each result back to the place that it read the
// operand of the same number from, which no other thread touches: no barrier
// between its reads and its writes.  Butterfly group j2 = t + uT of the third
// pass finds its operand r at
template <int L, int R0, int R1, int T>
__device__ __forceinline__ int third_place(int t, int u, int r) {
  static_assert(T % R0 == 0, "places");
  return padp<R0>(r * R0 + (t & (R0 - 1)) + (t / R0 + (T / R0) * u) * (L / R1));
}

// FFT plans: L = N/2 complex points; radices R0*R1*R2 = L; T threads per FFT.
template <int L> struct Plan;
template <> struct Plan<4>    { static constexpr int R0 = 4,  R1 = 1,  R2 = 1, T = 1; };
template <> struct Plan<8>    { static constexpr int R0 = 8,  R1 = 1,  R2 = 1, T = 1; };
template <> struct Plan<16>   { static constexpr int R0 = 16, R1 = 1,  R2 = 1, T = 1; };
template <> struct Plan<32>   { static constexpr int R0 = 32, R1 = 1,  R2 = 1, T = 1; };
template <> struct Plan<64>   { static constexpr int R0 = 8,  R1 = 8,  R2 = 1, T = 8; };
template <> struct Plan<128>  { static constexpr int R0 = 16, R1 = 8,  R2 = 1, T = 8; };
template <> struct Plan<256>  { static constexpr int R0 = 16, R1 = 16, R2 = 1, T = 16; };
template <> struct Plan<512>  { static constexpr int R0 = 32, R1 = 16, R2 = 1, T = 16; };
template <> struct Plan<1024> { static constexpr int R0 = 32, R1 = 32, R2 = 1, T = 32; };
template <> struct Plan<2048> { static constexpr int R0 = 16, R1 = 16, R2 = 8, T = 128; };
template <> struct Plan<4096> { static constexpr int R0 = 16, R1 = 16, R2 = 16, T = 256; };
template <> struct Plan<8192> { static constexpr int R0 = 32, R1 = 16, R2 = 16, T = 256; };

template <int L> struct Groups {
  static constexpr int T = Plan<L>::T;
  // 256 threads per CTA (64 one-thread transforms for the smallest sizes);
  // 4096-point complex transforms (8192-sample blocks) run three independent
  // 256-thread transforms per CTA of 768 threads, so that barriers stay
  // within a transform, three of them are in flight per SM and 24 warps hide
  // the latency of the twiddle loads
  static constexpr int NGRP = T == 1 ? 64 : (L == 4096 ? 3 : 256 / T);
};

// The tensor-core F step runs teams of 8 groups (one per block of its 8),
// one stream per team and round.
template <int L> struct GroupsTC {
  static constexpr int NGRP = Groups<L>::NGRP >= 8 ? Groups<L>::NGRP : 8;
};

template <int L> constexpr int kBufPad() { return L + L / Plan<L>::R0 + 1; }

// Shared tables for N <= 2048: the last Stockham pass's twiddles W_L^{k r}
// (L entries, [r][k]) and the real-split twiddles W_N^k for k <= L/2.
template <int L> struct Tw {
  static constexpr bool on = L >= 64 && L <= 1024;
  static constexpr int size = on ? L + L / 2 + 1 : 1;
};

// Fill the shared tables: s_lut16[c0 | c1 << 2] = (l[c0], l[c1]) / 2 (the
// halving takes the 1/2 of the real-FFT split into the input, exactly), and,
// when Tw<L>::on, the twiddle tables (last pass: NS = L / R_last).
template <int L, int RLAST, int TWS = 2>
__device__ __forceinline__ void fill_tables(float2* s_lut16, float2* s_tw, const FParams& p) {
  const int tid = threadIdx.x;
  if (tid < 16) {
    const float l[4] = {p.lut0, p.lut1, p.lut2, p.lut3};
    s_lut16[tid] = make_float2(0.5f * l[tid & 3], 0.5f * l[tid >> 2]);
  }
  if constexpr (Tw<L>::on) {
    constexpr int NS = L / RLAST;
    for (int e = tid; e < L; e += blockDim.x) {
      const int r = e / NS, k = e - r * NS;
      s_tw[e] = __ldg(&p.twN[TWS * k * r]);
    }
    for (int k = tid; k <= L / 2; k += blockDim.x) s_tw[L + k] = __ldg(&p.twN[k]);
  }
}

// Shared tables of the powers W^{k 2^i} (k < NS, i < log2 R) of the passes
// after the first, for transforms of 2048+ points: [i][k] per pass, the
// second pass's table after the first's.
template <int L> struct PassTw {
  static constexpr bool on = L >= 2048;
  static constexpr int n1 = Plan<L>::R1 > 1 ? ilog2c(Plan<L>::R1) * Plan<L>::R0 : 0;
  static constexpr int n2 = Plan<L>::R2 > 1 ? ilog2c(Plan<L>::R2) * Plan<L>::R0 * Plan<L>::R1 : 0;
  static constexpr int size = on ? n1 + n2 : 1;
};

template <int L, int R, int NS, int TWS>
__device__ __forceinline__ void fill_pass_table(float2* dst, const float2* __restrict__ twN) {
  constexpr int LOGR = ilog2c(R);
  for (int e = threadIdx.x; e < LOGR * NS; e += blockDim.x) {
    const int i = e / NS, k = e - i * NS;
    dst[e] = __ldg(&twN[TWS * k * (1 << i) * (L / (NS * R))]);
  }
}

template <int L, int TWS>
__device__ __forceinline__ void fill_pass_tables(float2* s_twp, const float2* __restrict__ twN) {
  if constexpr (PassTw<L>::on) {
    using P = Plan<L>;
    if constexpr (P::R1 > 1) fill_pass_table<L, P::R1, P::R0, TWS>(s_twp, twN);
    if constexpr (P::R2 > 1) fill_pass_table<L, P::R2, P::R0 * P::R1, TWS>(s_twp + PassTw<L>::n1, twN);
  }
}

template <int L> struct LastRadix {
  static constexpr int v = Plan<L>::R2 > 1 ? Plan<L>::R2 : (Plan<L>::R1 > 1 ? Plan<L>::R1 : Plan<L>::R0);
};

// ---- real split and rotation ----
// Channels k and L-k come from the same pair Z[k], Z[L-k] of the N/2-point
// transform:  X[k] = E + W O,  X[L-k] = conj(E - W O),  W = W_N^k.  Z is the
// transform of the halved samples, so E = Z[k] + conj Z[L-k] and
// O = -i (Z[k] - conj Z[L-k]) carry the split's factor 1/2.
__device__ __forceinline__ void split_values(float2 Zk, float2 Zm, float2 w, float2& Xa, float2& Xb) {
  const float2 pm = make_float2(1.f, -1.f), mp = make_float2(-1.f, 1.f);
  const float2 E = f2fma(Zm, pm, Zk);             // (Zk.x + Zm.x, Zk.y - Zm.y)
  const float2 Ec = f2fma(Zk, pm, Zm);            // conj E
  const float2 O = f2fma(swp(Zk), pm, swp(Zm));   // (Zk.y + Zm.y, Zm.x - Zk.x)
  const float2 WO = cmul(O, w);
  Xa = f2add(E, WO);
  Xb = f2fma(WO, mp, Ec);                         // (E.x - WO.x, WO.y - E.y)
}

template <int L, int R0>
__device__ __forceinline__ void split_pair(const float2* __restrict__ fbuf, float2 w, int k, int km, float2& Xa,
                                           float2& Xb) {
  split_values(fbuf[padp<R0>(k)], fbuf[padp<R0>(km)], w, Xa, Xb);
}

// The split's twiddles W_N^k along a thread's channels k = t + qT: from the
// shared table for N <= 2048; above, W_N^t from the global table times
// W_N^{qT} by a walk (one product per channel instead of a global load
// whose latency the large transforms cannot hide; QF <= 16 steps add a few
// ulp).
template <int L, int T>
struct SplitTw {
  float2 w, step;
  __device__ __forceinline__ SplitTw(const float2* __restrict__ s_tw, const float2* __restrict__ twN, int t) {
    if constexpr (!Tw<L>::on) {
      w = __ldg(&twN[t]);
      step = __ldg(&twN[T]);
    }
  }
  __device__ __forceinline__ float2 get(const float2* __restrict__ s_tw, int k) const {
    if constexpr (Tw<L>::on) return s_tw[L + k];
    else return w;
  }
  __device__ __forceinline__ void next() {
    if constexpr (!Tw<L>::on) w = cmul(w, step);
  }
};

// The rotation exp(+2 pi i (phi + k delta)) along a thread's channels
// k = t + qT (and L - k): the first factor of each sequence comes from the
// fast sine/cosine of the argument reduced to [-pi, pi] (abs. error ~4e-7),
// later ones by a walk z <- z + z (e^{i theta} - 1), theta = +-2 pi T delta.
// |delta| <= 1/(2N) turns per channel (the fractional delay is at most half
// a sample), so |theta| <= pi T / N <= 0.2 and e^{i theta} - 1 comes from its
// Taylor series to theta^8 (remainder < 1e-12); written as an increment the
// walk has no systematic drift of |z| from rounding cos(theta).
__device__ __forceinline__ float2 cis_turns(float ph) {
  ph -= rintf(ph);
  float sn, cs;
  __sincosf(6.28318530717958648f * ph, &sn, &cs);
  return make_float2(cs, sn);
}

__device__ __forceinline__ void walk_step(float T_delta, float& cm1, float& sn) {
  const float th = 6.28318530717958648f * T_delta;
  const float t2 = th * th;
  // sin th = th (1 - th^2/3! + th^4/5! - th^6/7!)
  sn = th * fmaf(t2, fmaf(t2, fmaf(t2, -1.0f / 5040.0f, 1.0f / 120.0f), -1.0f / 6.0f), 1.0f);
  // cos th - 1 = th^2 (-1/2! + th^2/4! - th^4/6! + th^6/8!)
  cm1 = t2 * fmaf(t2, fmaf(t2, fmaf(t2, 1.0f / 40320.0f, -1.0f / 720.0f), 1.0f / 24.0f), -0.5f);
}

// z + z (cm1 + i sn) = (z + z cm1) + swap(z) (-sn, sn)
__device__ __forceinline__ float2 walk(float2 z, float cm1, float sn) {
  return f2fma(swp(z), make_float2(-sn, sn), f2fma(z, bc(cm1), z));
}

template <int OUT>
__device__ __forceinline__ void store_spec(void* out, size_t idx, float2 X, float scale) {
  if constexpr (OUT == 0) {
    reinterpret_cast<float2*>(out)[idx] = X;
  } else if constexpr (OUT == 1) {
    reinterpret_cast<__half2*>(out)[idx] = __floats2half2_rn(X.x * scale, X.y * scale);
  } else {
    reinterpret_cast<uint16_t*>(out)[idx] = (uint16_t)fp8x2(X.x * scale, X.y * scale);
  }
}

// Split, rotate and store the L/2 + 1 channel pairs of one transform; a
// block that is not valid stores zeros.
template <int L, int T, int R0, int OUT>
__device__ __forceinline__ void split_rotate_store(const float2* __restrict__ fbuf, const float2* __restrict__ s_tw,
                                                   const float2* __restrict__ twN, int t, bool ok, float phi,
                                                   float delta, void* out, size_t obase, float scale) {
  constexpr int HALF = L / 2;
  constexpr int QF = HALF / T;  // k = t + qT < HALF for q < QF; k = HALF is thread 0's extra
  const float2 zero = make_float2(0.f, 0.f);
  if (!ok) {
#pragma unroll 4
    for (int q = 0; q < QF; ++q) {
      const int k = t + q * T;
      store_spec<OUT>(out, obase + k, zero, scale);
      if (k != 0) store_spec<OUT>(out, obase + (L - k), zero, scale);
    }
    if (t == 0) store_spec<OUT>(out, obase + HALF, zero, scale);
    return;
  }
  float2 z = cis_turns(fmaf((float)t, delta, phi));
  float2 y = cis_turns(fmaf((float)(L - t), delta, phi));
  float cm1, sn;
  walk_step((float)T * delta, cm1, sn);
  SplitTw<L, T> tw(s_tw, twN, t);
#pragma unroll 4
  for (int q = 0; q < QF; ++q) {
    const int k = t + q * T;
    const int km = (L - k) & (L - 1);
    float2 Xa, Xb;
    split_pair<L, R0>(fbuf, tw.get(s_tw, k), k, km, Xa, Xb);
    store_spec<OUT>(out, obase + k, cmul(Xa, z), scale);
    if (k != 0) store_spec<OUT>(out, obase + km, cmul(Xb, y), scale);
    z = walk(z, cm1, sn);
    y = walk(y, cm1, -sn);
    tw.next();
  }
  if (t == 0) {  // k = HALF: X[HALF] = E + W_N^{N/4} O; z has walked to it
    float2 Xa, Xb;
    split_pair<L, R0>(fbuf, make_float2(0.f, -1.f), HALF, HALF, Xa, Xb);
    store_spec<OUT>(out, obase + HALF, cmul(Xa, z), scale);
  }
}

// Split, rotate and store from the registers of one warp's transform.  Z[L - k]
// of k = t + qT is element Q - 1 - q of thread T - t (element Q - q of thread 0
// itself), so half the values cross lanes by shuffles, where the shared-memory
// form writes and reads all of them: 32 shared-memory cycles a 1024-point
// transform instead of 128.
template <int L, int T, int OUT, int PER, int R>
__device__ __forceinline__ void split_rotate_shuffle(const float2 (&z_)[PER][R], const float2* __restrict__ s_tw, int t,
                                                     float phi, float delta, void* out, size_t obase, float scale) {
  constexpr int Q = L / T;
  static_assert(PER * R == Q, "last pass");
  auto v = [&](int q) { return z_[q % PER][q / PER]; };  // Z[t + q T]
  const unsigned mask = T == 32 ? 0xffffffffu : ((1u << T) - 1u) << (threadIdx.x & 31u & ~(unsigned)(T - 1));
  const int partner = (T - t) & (T - 1);
  float2 z = cis_turns(fmaf((float)t, delta, phi));
  float2 y = cis_turns(fmaf((float)(L - t), delta, phi));
  float cm1, sn;
  walk_step((float)T * delta, cm1, sn);
#pragma unroll
  for (int q = 0; q < Q / 2; ++q) {
    const int k = t + q * T;
    const float2 give = t == 0 ? v((Q - q) % Q) : v(Q - 1 - q);
    const float2 Zm = make_float2(__shfl_sync(mask, give.x, partner, T), __shfl_sync(mask, give.y, partner, T));
    float2 Xa, Xb;
    split_values(v(q), Zm, s_tw[L + k], Xa, Xb);
    store_spec<OUT>(out, obase + k, cmul(Xa, z), scale);
    if (q > 0 || t != 0) store_spec<OUT>(out, obase + (L - k), cmul(Xb, y), scale);
    z = walk(z, cm1, sn);
    y = walk(y, cm1, -sn);
  }
  if (t == 0) {  // k = L/2: X = E + W_N^{N/4} O; z has walked to it
    float2 Xa, Xb;
    split_values(v(Q / 2), v(Q / 2), make_float2(0.f, -1.f), Xa, Xb);
    store_spec<OUT>(out, obase + L / 2, cmul(Xa, z), scale);
  }
}

// The same for a transform of several warps and three passes: the thread's own
// results v[u][r] = Z[t + (r PER + u) T] stay in registers, the upper half of
// them also goes to the places that its operands came from, where the thread
// of the partner channels reads them.  (Writing and reading all results, with
// barriers around every pass's writes, took six barriers a transform where
// this takes four: 2.7e8 samples of 4096-point transforms 510 us, 475 now, of
// 2048-point ones 434 and 418, pre-F 680 and 647.)
template <int L, int R0, int R1, int T, int OUT, int PER, int R>
__device__ __forceinline__ void split_rotate_places(const float2 (&z_)[PER][R], float2* __restrict__ fbuf, int t, int grp,
                                                    const float2* __restrict__ twN, float phi, float delta, void* out,
                                                    size_t obase, float scale) {
  constexpr int Q = L / T;
  static_assert(PER * R == Q, "last pass");
  auto v = [&](int q) { return z_[q % PER][q / PER]; };  // Z[t + q T]
#pragma unroll
  for (int q = Q / 2; q < Q; ++q) fbuf[third_place<L, R0, R1, T>(t, q % PER, q / PER)] = v(q);
  gsync<T>(grp);
  const int tp = (T - t) & (T - 1);  // thread of Z[L - k], element Q - 1 - q (Q - q for thread 0)
  float2 z = cis_turns(fmaf((float)t, delta, phi));
  float2 y = cis_turns(fmaf((float)(L - t), delta, phi));
  float cm1, sn;
  walk_step((float)T * delta, cm1, sn);
  SplitTw<L, T> tw(nullptr, twN, t);
#pragma unroll
  for (int q = 0; q < Q / 2; ++q) {
    const int k = t + q * T;
    const int qp = Q - 1 - q + (t == 0 ? 1 : 0);
    const float2 Zm = q == 0 && t == 0 ? v(0) : fbuf[third_place<L, R0, R1, T>(tp, qp % PER, qp / PER)];
    float2 Xa, Xb;
    split_values(v(q), Zm, tw.get(nullptr, k), Xa, Xb);
    store_spec<OUT>(out, obase + k, cmul(Xa, z), scale);
    if (q > 0 || t != 0) store_spec<OUT>(out, obase + (L - k), cmul(Xb, y), scale);
    z = walk(z, cm1, sn);
    y = walk(y, cm1, -sn);
    tw.next();
  }
  if (t == 0) {  // k = L/2: X = E + W_N^{N/4} O; z has walked to it
    float2 Xa, Xb;
    split_values(v(Q / 2), v(Q / 2), make_float2(0.f, -1.f), Xa, Xb);
    store_spec<OUT>(out, obase + L / 2, cmul(Xa, z), scale);
  }
}

// Byte offset of the packed-word staging area after the NGRP FFT buffers,
// rounded up to 16 bytes for the 16-byte shared-memory stores.
template <int L>
constexpr size_t kWordsOffset(int NGRP) {
  return ((size_t)NGRP * kBufPad<L>() * sizeof(float2) + 15) & ~(size_t)15;
}

__host__ __device__ inline int wslot_words(int N, int G) {
  // window bits 2*N*G plus up to 31 bits of misalignment, up to 3 lead words
  // before the window, one word of shift (G = 16) and one spare word
  return (((2 * N * G + 31 + 31) >> 5) + 3 + 1 + 1 + 3) & ~3;
}

// Asynchronous global -> shared copies (LDGSTS) for the window staging.
__device__ __forceinline__ void cp_async16(void* sdst, const void* gsrc) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(sdst)),
               "l"(gsrc)
               : "memory");
}
__device__ __forceinline__ void cp_async8(void* sdst, const void* gsrc) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(sdst)),
               "l"(gsrc)
               : "memory");
}
__device__ __forceinline__ void cp_async4(void* sdst, const void* gsrc) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(sdst)),
               "l"(gsrc)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Stage the packed windows of `nslots` blocks (chunk blocks bb0...) into
// wbuf (slot stride wslot words) with asynchronous copies (plain loads from
// pinned host memory unless ASYNC): 16-byte copies where the words lie inside
// the station's data, single words at its end.
// The copy of slot sl starts at the 16-byte aligned word a0 = w0 & ~3; with
// GC = 16 (one word per sample time) word w0 goes to an even index so that
// every sample pair is one aligned 64-bit load (odd leads are copied word by
// word, one word further on); with GC = 32 (two words per sample time, so
// the lead is 0 or 2) word w0 goes to a 16-byte boundary so that a sample
// pair is one aligned 16-byte load (a lead of 2 is copied in 8-byte pieces,
// two words further on).  s_ok / s_boff receive each slot's validity and the
// bit offset of its window from the slot's first word.
template <int N, int GC, bool ASYNC>
__device__ __forceinline__ void stage_windows(const FParams& p, const StationView& sv, int s, int G, int bb0,
                                              int nslots, uint32_t* wbuf, int wslot, int* s_ok, int* s_boff) {
  // several windows: a share of the warps each, so that their descriptor
  // loads (and the copies behind them) run side by side, not one after another
  const int ways = min(nslots, (int)(blockDim.x >> 5));
  const int nt = (int)(blockDim.x / ways) & ~31;  // threads per window
  const int tid = threadIdx.x % nt, way = threadIdx.x / nt;
  for (int sl = way < ways ? way : nslots; sl < nslots; sl += ways) {
    const int d = p.blk0 + bb0 + sl;
    const bool ok = p.valid[(size_t)s * p.ld + d] != 0;
    int64_t w0 = 0;
    int boff = 0, nw = 0;
    if (ok) {
      const int64_t rel = p.start[(size_t)s * p.ld + d] - sv.sample0;
      const int64_t bit0 = 2 * rel * G;
      w0 = bit0 >> 5;
      boff = (int)(bit0 & 31);
      nw = (boff + 2 * N * G + 31) >> 5;
      if (w0 + nw > sv.nwords) nw = (int)(sv.nwords - w0);
    }
    const int lead = (int)(w0 & 3);
    // GC = 16: the window's first word at an even index; GC = 32 (lead 0
    // or 2): at a 16-byte boundary
    const int shift = (GC == 16) ? (lead & 1) : (GC == 32 ? ((4 - lead) & 3) : 0);
    uint32_t* dst = wbuf + sl * wslot + shift;
    const int64_t a0 = w0 - lead;
    const int ntot = nw + lead;
    const int nvec = ntot >> 2;
    if (sv.host && (!ASYNC || nvec >= 32)) {
      // pinned host memory over the host link: plain 16-byte loads keep more
      // of the link's requests in flight than the async copies (with ASYNC:
      // 4 stations x 20 streams x 1024 channels, 6e8 station-samples, 3.59 ms
      // by copies behind the step before, 2.98 by loads).  Windows of less than
      // a load for each lane are all latency, which the copies leave behind
      // that step (one stream x 64 channels: 9.7 ms by loads, 8.5 by copies).
      const uint4* src4 = reinterpret_cast<const uint4*>(sv.words + a0);
      for (int q = tid; q < nvec; q += nt) {
        if (a0 + 4 * q + 4 <= sv.nwords) {
          const uint4 x = __ldg(src4 + q);
          if (shift) {
            dst[4 * q] = x.x;
            dst[4 * q + 1] = x.y;
            dst[4 * q + 2] = x.z;
            dst[4 * q + 3] = x.w;
          } else {
            reinterpret_cast<uint4*>(dst)[q] = x;
          }
        } else {
          for (int u = 0; u < 4; ++u)
            if (a0 + 4 * q + u < sv.nwords) dst[4 * q + u] = __ldg(&sv.words[a0 + 4 * q + u]);
        }
      }
      for (int q = 4 * nvec + tid; q < ntot; q += nt)
        if (a0 + q < sv.nwords) dst[q] = __ldg(&sv.words[a0 + q]);
    } else {
      for (int q = tid; q < nvec; q += nt) {
        if (a0 + 4 * q + 4 <= sv.nwords) {
          if (shift == 2) {
            cp_async8(dst + 4 * q, sv.words + a0 + 4 * q);
            cp_async8(dst + 4 * q + 2, sv.words + a0 + 4 * q + 2);
          } else if (shift) {
#pragma unroll
            for (int u = 0; u < 4; ++u) cp_async4(dst + 4 * q + u, sv.words + a0 + 4 * q + u);
          } else {
            cp_async16(dst + 4 * q, sv.words + a0 + 4 * q);
          }
        } else {
          for (int u = 0; u < 4; ++u)
            if (a0 + 4 * q + u < sv.nwords) cp_async4(dst + 4 * q + u, sv.words + a0 + 4 * q + u);
        }
      }
      for (int q = 4 * nvec + tid; q < ntot; q += nt)
        if (a0 + q < sv.nwords) cp_async4(dst + q, sv.words + a0 + q);
    }
    if (tid == 0) {
      s_ok[sl] = ok ? 1 : 0;
      s_boff[sl] = boff + 32 * (lead + shift);
    }
  }
}

// Compile-time stream count GC (0: runtime p.G).  With GC = 16 a sample-time
// group is exactly one 32-bit word (a sample pair is one aligned 64-bit
// load: the staging puts the window's first word at an even index); with
// GC = 32 it is two words.
template <int GC>
__device__ __forceinline__ void load_pair(const uint32_t* __restrict__ wsl, int boff, int G, int m, int j,
                                          uint32_t& c0, uint32_t& c1) {
  if constexpr (GC == 16) {
    // the staging put the window's first word at an even index
    const uint2 w = *reinterpret_cast<const uint2*>(wsl + 2 * m);
    c0 = (w.x >> (2 * j)) & 3u;
    c1 = (w.y >> (2 * j)) & 3u;
  } else if constexpr (GC == 32) {
    // the staging put the window's first word at a 16-byte boundary: the
    // four words of a sample pair are one aligned 16-byte load
    const uint4 w = *reinterpret_cast<const uint4*>(wsl + 4 * m);
    const bool hi = (j >> 4) != 0;
    c0 = ((hi ? w.y : w.x) >> (2 * (j & 15))) & 3u;
    c1 = ((hi ? w.w : w.z) >> (2 * (j & 15))) & 3u;
  } else {
    const int bit = boff + 2 * (2 * m * G + j);
    c0 = (wsl[bit >> 5] >> (bit & 31)) & 3u;
    const int bit1 = bit + 2 * G;
    c1 = (wsl[bit1 >> 5] >> (bit1 & 31)) & 3u;
  }
}

// Transpose a 16 x 16 matrix of 2-bit fields: field i of word j becomes field
// j of word i.
__device__ __forceinline__ void transpose_fields(uint32_t (&a)[16]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t x = a[i], y = a[i + 8];
    a[i] = __byte_perm(x, y, 0x5410);
    a[i + 8] = __byte_perm(x, y, 0x7632);
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int i = (q & 3) + 2 * (q & 4);
    const uint32_t x = a[i], y = a[i + 4];
    a[i] = __byte_perm(x, y, 0x6240);
    a[i + 4] = __byte_perm(x, y, 0x7351);
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int i = (q & 1) + 2 * (q & 6);
    const uint32_t x = a[i], y = a[i + 2], m = 0x0F0F0F0Fu;
    a[i] = (x & m) | ((y << 4) & ~m);
    a[i + 2] = ((x >> 4) & m) | (y & ~m);
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int i = 2 * q;
    const uint32_t x = a[i], y = a[i + 1], m = 0x33333333u;
    a[i] = (x & m) | ((y << 2) & ~m);
    a[i + 1] = ((x >> 2) & m) | (y & ~m);
  }
}

// The first pass's codes, stream by stream.  The staged window interleaves the
// streams, so that each transform had to read all of it: 32 64-bit loads and
// as many shifts and masks a thread for a 1024-point transform, an eighth of
// the kernel's shared-memory traffic.  Here the CTA turns the window once for
// all streams: thread t of a transform takes points t + r T, r < R0, whose
// codes (two samples a point; one in the pre-F form) become the 2-bit fields
// of W words, [slot][stream][word][thread], read as W consecutive loads.
template <int L, bool PRE> struct Codes {
  static constexpr int T = Plan<L>::T, R0 = Plan<L>::R0;
  static constexpr int F = R0 * (PRE ? 1 : 2);   // fields per thread
  static constexpr int W = (F + 15) / 16;
  static constexpr bool on = L >= 64 && L <= 4096 && L / R0 == T;  // one point group a thread
};

// One stream (post-F form): the window is a row of 4-bit point codes, and the
// words of eight threads come from an 8 x 8 transpose of them.
template <int L>
__device__ __forceinline__ void turn_codes_one(const uint32_t* __restrict__ wbuf, int wslot, const int* s_ok,
                                               const int* s_boff, int nslots, uint32_t* codes) {
  using C = Codes<L, false>;
  constexpr int T = C::T, W = C::W;
  for (int e = threadIdx.x; e < nslots * W * (T / 8); e += blockDim.x) {
    const int t8 = e % (T / 8);
    const int w = e / (T / 8) % W;
    const int sl = e / (T / 8) / W;
    if (!s_ok[sl]) continue;
    const int boff = s_boff[sl];
    const uint32_t* wsl = wbuf + sl * wslot;
    uint32_t a[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {  // points 8 t8 .. 8 t8 + 7 of row r = 8 w + i
      const int bit = boff + 4 * (8 * t8 + (8 * w + i) * T);
      a[i] = __funnelshift_r(wsl[bit >> 5], wsl[(bit >> 5) + 1], bit & 31);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t x = a[i], y = a[i + 4];
      a[i] = __byte_perm(x, y, 0x5410);
      a[i + 4] = __byte_perm(x, y, 0x7632);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = (q & 1) + 2 * (q & 2);
      const uint32_t x = a[i], y = a[i + 2];
      a[i] = __byte_perm(x, y, 0x6240);
      a[i + 2] = __byte_perm(x, y, 0x7351);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = 2 * q;
      const uint32_t x = a[i], y = a[i + 1], m = 0x0F0F0F0Fu;
      a[i] = (x & m) | ((y << 4) & ~m);
      a[i + 1] = ((x >> 4) & m) | (y & ~m);
    }
    uint4* dst = reinterpret_cast<uint4*>(codes + (sl * W + w) * T + 8 * t8);
    dst[0] = make_uint4(a[0], a[1], a[2], a[3]);
    dst[1] = make_uint4(a[4], a[5], a[6], a[7]);
  }
}

// Streams [j0, j0 + jb) of `nslots` staged windows into `codes`.
template <int L, int GC, bool PRE>
__device__ __forceinline__ void turn_codes(const uint32_t* __restrict__ wbuf, int wslot, const int* s_ok,
                                           const int* s_boff, int nslots, int G, int j0, int jb, uint32_t* codes) {
  using C = Codes<L, PRE>;
  constexpr int T = C::T, W = C::W, F = C::F;
  if constexpr (GC == 0 && !PRE && T >= 8) {
    if (G == 1) return turn_codes_one<L>(wbuf, wslot, s_ok, s_boff, nslots, codes);
  }
  const int halves = (jb + 15) >> 4;  // 16 streams at a time
  for (int e = threadIdx.x; e < nslots * halves * W * T; e += blockDim.x) {
    const int t = e % T;
    int q = e / T;
    const int w = q % W;
    q /= W;
    const int sl = q / halves, h = q - sl * halves;
    if (!s_ok[sl]) continue;
    const int boff = s_boff[sl];
    const uint32_t* wsl = wbuf + sl * wslot + (GC ? (boff >> 5) : 0);
    uint32_t a[16];
#pragma unroll
    for (int f = 0; f < 16; f += PRE ? 1 : 2) {
      const int fi = 16 * w + f;
      const int m = t + (PRE ? fi : fi >> 1) * T;  // point
      if (F < 16 && f >= F) {
        a[f] = 0u;
        if (!PRE) a[f + 1] = 0u;
      } else if constexpr (GC == 16 && PRE) {
        a[f] = wsl[m];
      } else if constexpr (GC == 16) {  // the staging put the window's first word at an even index
        const uint2 x = *reinterpret_cast<const uint2*>(wsl + 2 * m);
        a[f] = x.x;
        a[f + 1] = x.y;
      } else if constexpr (GC == 32 && PRE) {
        a[f] = wsl[2 * m + (j0 >> 4) + h];
      } else if constexpr (GC == 32) {
        a[f] = wsl[4 * m + (j0 >> 4) + h];
        a[f + 1] = wsl[4 * m + 2 + (j0 >> 4) + h];
      } else {
        const int bit = boff + 2 * ((PRE ? m : 2 * m) * G + j0 + 16 * h);
        a[f] = __funnelshift_r(wsl[bit >> 5], wsl[(bit >> 5) + 1], bit & 31);
        if constexpr (!PRE) {
          const int bit1 = bit + 2 * G;
          a[f + 1] = G <= 8 ? a[f] >> (2 * G) : __funnelshift_r(wsl[bit1 >> 5], wsl[(bit1 >> 5) + 1], bit1 & 31);
        }
      }
    }
    transpose_fields(a);
    uint32_t* dst = codes + ((size_t)(sl * jb + 16 * h) * W + w) * T + t;
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (16 * h + j < jb) dst[j * W * T] = a[j];
  }
}

// CTAs per SM the register allocation must allow: larger FFTs run one group
// of 128-256 threads per FFT, so without a bound the compiler takes up to
// 255 registers and a single CTA fills the SM's register file.  (4096- and
// 8192-point transforms keep one CTA of 768 / 256 threads per SM: their
// buffers and staged windows fill shared memory anyway.)
template <int L> struct MinBlocks {
  static constexpr int v = (L >= 64 && L <= 1024) ? 2 : (L == 2048 ? 3 : 1);
};
// the tensor-core F step keeps its 8 groups' spectra in shared memory
template <int L> struct MinBlocksTC {
  static constexpr int v = Groups<L>::T * GroupsTC<L>::NGRP > 256 ? 1 : MinBlocks<L>::v;
};

// Row of the spectra output for stream j, chunk block bb, station s:
// [stream][block][station], or with both hands of two polarisations
// [subband][block][pol][station], which puts the 2S (station, pol) pairs of a
// subband side by side for the X step.
__device__ __forceinline__ size_t spec_row(const FParams& p, int j, int bb, int s) {
  if (p.cross) {
    const int sb = j / p.npol, pol = j - sb * p.npol;
    return ((size_t)(sb * p.CB + bb) * p.npol + pol) * p.S + s;
  }
  return ((size_t)j * p.CB + bb) * p.S + s;
}

// One sample of stream j: sample-time group m of the staged window.
template <int GC>
__device__ __forceinline__ uint32_t load_one(const uint32_t* __restrict__ wsl, int boff, int G, int m, int j) {
  if constexpr (GC == 16) {
    return (wsl[m] >> (2 * j)) & 3u;
  } else if constexpr (GC == 32) {
    return (wsl[2 * m + (j >> 4)] >> (2 * (j & 15))) & 3u;
  } else {
    const int bit = boff + 2 * (m * G + j);
    return (wsl[bit >> 5] >> (bit & 31)) & 3u;
  }
}

// Pre-F fringe rotation of sample m of a block: exp(+2 pi i phi_m) with
// phi_m = phi0 + m * delta_s (turns), phi0 = the phase at the block's first
// sample (FP64 on the host side of the delay kernel, reduced to [0, 1)) and
// delta_s = dhi + dlo the phase step per sample, split so that dhi has at
// most 10 significant bits: m * dhi is then exact in FP32 for m < 2^14, its
// whole turns drop out exactly, and phi_m carries an error of ~1e-7 turns.
__device__ __forceinline__ float2 prerot(int m, float phi0, float dhi, float dlo) {
  const float fm = (float)m;
  float a = fm * dhi;
  a -= rintf(a);
  return cis_turns(fmaf(fm, dlo, phi0) + a);
}

// The rotation over the r T samples (r < R0) between the points that a thread
// of the first pass takes: the same for all threads and both polarisations of
// a (slot, subband), so the CTA forms it once per step (with the accurate sine
// and cosine) and a point costs one complex product instead of a sine, a
// cosine and two reductions of its own phase, whose special-function and
// issue slots bound the pre-F form with the transform's (2048 points: 705 us
// per 2.7e8 samples, 680 with the table; 647 now, with the middle pass in place).
template <int L>
__device__ __forceinline__ void fill_rotations(const FParams& p, int s, int bb0, int nslots, const int* s_ok, float2* rot) {
  constexpr int R0 = Plan<L>::R0, T = Plan<L>::T;
  for (int e = threadIdx.x; e < nslots * p.nsub * R0; e += blockDim.x) {
    const int r = e % R0;
    const int sb = e / R0 % p.nsub, sl = e / R0 / p.nsub;
    if (!s_ok[sl]) continue;
    const float2 dph = p.dphi[((size_t)s * p.nsub + sb) * p.ld + p.blk0 + bb0 + sl];
    const float fm = (float)(r * T);
    float a = fm * dph.x;  // exact, see prerot
    a -= rintf(a);
    float sn, cs;
    sincospif(2.0f * fmaf(fm, dph.y, a), &sn, &cs);
    rot[e] = make_float2(cs, sn);
  }
}

// Store of the pre-F path: channels k = 0..L/2-1 of the complex L-point
// transform, times the fractional-delay slope exp(+2 pi i k delta) (the
// fringe phase was applied before the transform), by the same walk as the
// post-F store.  v(q) is Z[t + qT]: the thread's own results of the last pass,
// which need not pass through shared memory.
template <int L, int T, int OUT>
__device__ __forceinline__ void store_zeros_pre(int t, void* out, size_t obase) {
#pragma unroll 4
  for (int q = 0; q < L / 2 / T; ++q) store_spec<OUT>(out, obase + t + q * T, make_float2(0.f, 0.f), 1.f);
}

template <int L, int T, int OUT, typename V>
__device__ __forceinline__ void rotate_store_pre(V v, int t, float delta, void* out, size_t obase, float scale) {
  constexpr int Q = (L / 2) / T;
  static_assert(Q >= 1 && (L / 2) % T == 0, "plan");
  float2 z = cis_turns((float)t * delta);
  float cm1, sn;
  walk_step((float)T * delta, cm1, sn);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    store_spec<OUT>(out, obase + t + q * T, cmul(v(q), z), scale);
    z = walk(z, cm1, sn);
  }
}

// The F kernel.  PRE = false: the N = 2L real samples of a block as an
// L-point complex transform (even/odd samples packed), real split, post-F
// rotation.  PRE = true: the N = L real samples rotated one by one by the
// fringe phase into an L-point complex transform, then the fractional-delay
// slope.  TURN: the codes come stream by stream from turn_codes, jb streams at
// a time; else each transform decodes the staged window itself.
//
// Bound by the mix of the FMA pipe (51%), the shared-memory pipe (59%) and
// instruction issue (54%) at the 16 warps that 32 points a thread leave an SM:
// no one of its parts, taken out, gives more than 9%.  Ten stations x 16
// streams x 1024 channels, 819 blocks (2.7e8 samples): 328 us; 376 us when each
// transform decoded the interleaved window (shared-memory pipe 71%) and passed
// its last pass through shared memory again.
template <int L, int GC, bool PRE, bool TURN>
__global__ void __launch_bounds__(Groups<L>::T * Groups<L>::NGRP, MinBlocks<L>::v)
k_fstage(FParams p, int slots, int wslot, int nseq, int jb) {
  using P = Plan<L>;
  constexpr int T = P::T;
  constexpr int NGRP = Groups<L>::NGRP;
  constexpr int N = PRE ? L : 2 * L;   // real samples per block
  constexpr int TWS = PRE ? 1 : 2;     // twN holds W_N^m; the transform needs W_L
  constexpr int BUF = kBufPad<L>();
  constexpr int R0 = P::R0;
  constexpr int PER0 = L / R0 / T;
  // the last pass's results stay in registers: the pre-F form's store needs only a thread's own,
  // the real split half of another thread's, by a shuffle within a warp or through shared memory
  // (8192 points, 32 a thread at 8 warps per SM: 590 us so, 575 with all results in shared memory)
  constexpr bool REGS = PRE || (T <= 32 && Tw<L>::on && P::R1 > 1) || (P::R2 > 1 && L <= 4096);
  static_assert(PER0 >= 1, "plan");

  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* fbuf_all = reinterpret_cast<float2*>(smem_raw);
  static_assert(kWordsOffset<L>(NGRP) % 16 == 0, "staging area must be 16-byte aligned");
  uint32_t* wbuf = reinterpret_cast<uint32_t*>(smem_raw + kWordsOffset<L>(NGRP));
  uint32_t* codes = wbuf + slots * wslot;  // TURN
  float2* rot = reinterpret_cast<float2*>(codes + (size_t)slots * jb * Codes<L, PRE>::W * T);  // TURN and PRE: [slot][subband][R0]

  const int tid = threadIdx.x;
  const int grp = tid / T;
  const int t = tid - grp * T;
  float2* fbuf = fbuf_all + grp * BUF;
  const int s = blockIdx.y;
  const int G = GC ? GC : p.G;
  const StationView sv = p.st[s];

  // this CTA: nseq steps of `slots` blocks each, from chunk block `first`;
  // the windows of step it+1 are copied asynchronously while step it is
  // transformed: into the staging area itself once its codes are turned, else
  // into the other half of a double buffer
  const int first = blockIdx.x * nseq * slots;
  if (first >= p.CB) return;

  __shared__ int s_boff[2][64];
  __shared__ int s_ok[2][64];
  __shared__ float2 s_lut16[16];
  __shared__ float2 s_tw[Tw<L>::size];
  __shared__ float2 s_twp[PassTw<L>::size];
  fill_tables<L, LastRadix<L>::v, TWS>(s_lut16, s_tw, p);
  fill_pass_tables<L, TWS>(s_twp, p.twN);

  stage_windows<N, GC, false>(p, sv, s, G, first, min(slots, p.CB - first), wbuf, wslot, s_ok[0], s_boff[0]);
  cp_async_commit();
  for (int it = 0; it < nseq; ++it) {
    const int bb0 = first + it * slots;
    if (bb0 >= p.CB) break;  // uniform over the CTA
    const int nslots = min(slots, p.CB - bb0);
    const int nb = it & 1;
    const bool more = it + 1 < nseq && bb0 + slots < p.CB;
    uint32_t* wcur = wbuf;
    if constexpr (TURN) {
      cp_async_wait<0>();
    } else {
      wcur = wbuf + nb * slots * wslot;
      if (more)
        stage_windows<N, GC, TURN>(p, sv, s, G, bb0 + slots, min(slots, p.CB - bb0 - slots), wbuf + (nb ^ 1) * slots * wslot,
                             wslot, s_ok[nb ^ 1], s_boff[nb ^ 1]);
      cp_async_commit();
      cp_async_wait<1>();  // this step's windows have landed (the next step's may still fly)
    }
    __syncthreads();

    for (int j0 = 0; j0 < G; j0 += jb) {
    const int nj = min(jb, G - j0);
    if constexpr (TURN) {
      if constexpr (PRE) {
        if (j0 == 0) fill_rotations<L>(p, s, bb0, nslots, s_ok[nb], rot);
      }
      turn_codes<L, GC, PRE>(wcur, wslot, s_ok[nb], s_boff[nb], nslots, G, j0, nj, codes);
      __syncthreads();
      if (more && j0 + jb >= G) {  // the window has been read
        stage_windows<N, GC, TURN>(p, sv, s, G, bb0 + slots, min(slots, p.CB - bb0 - slots), wbuf, wslot, s_ok[nb ^ 1],
                             s_boff[nb ^ 1]);
        cp_async_commit();
      }
    }
    const int ntasks = nslots * nj;
    for (int base = 0; base < ntasks; base += NGRP) {
      const int task = base + grp;
      const bool active = task < ntasks;
      const int sl = active ? task / nj : 0;
      const int j = active ? j0 + task - sl * nj : 0;
      const bool ok = active && s_ok[nb][sl];
      const int boff = s_boff[nb][sl];
      // for GC = 16 / 32 the window starts on a word boundary: skip the lead
      // (and shift) words
      const uint32_t* wsl = wcur + sl * wslot + (GC ? (boff >> 5) : 0);
      const int d = p.blk0 + bb0 + sl;
      // the block's phase terms, loaded now so that their latency passes
      // during the transform
      const float delta = ok ? p.delta[(size_t)s * p.ld + d] : 0.f;
      const float phi = (ok && !PRE) ? p.phi[((size_t)s * p.nsub + j / p.npol) * p.ld + d] : 0.f;
      constexpr int NCH = PRE ? L / 2 : L;
      const size_t obase = spec_row(p, j, bb0 + sl, s) * (size_t)NCH;

      // ---- pass 0: unpack straight into registers (NS = 1, no twiddles);
      //      the transform of a block that is not valid is skipped ----
      if (ok) {
        uint32_t cw[Codes<L, PRE>::W];
        if constexpr (TURN) {
#pragma unroll
          for (int w = 0; w < Codes<L, PRE>::W; ++w) cw[w] = codes[(task * Codes<L, PRE>::W + w) * T + t];
        }
        float2 v[PER0][R0];
        if constexpr (PRE) {
          const size_t ps = ((size_t)s * p.nsub + j / p.npol) * p.ld + d;
          const float phi0 = p.phi[ps];
          const float2 dph = p.dphi[ps];
          // s_lut16[c] = (l[c] / 2, l[0] / 2): twice its real part is level c
          if constexpr (TURN) {
            const float2 z0 = prerot(t, phi0, dph.x, dph.y);
            const float2* w = rot + (size_t)(sl * p.nsub + j / p.npol) * R0;
#pragma unroll
            for (int r = 0; r < R0; ++r) {
              const float lev = 2.0f * s_lut16[(cw[r >> 4] >> (2 * (r & 15))) & 3u].x;
              v[0][r] = f2mul(r == 0 ? z0 : cmul(z0, w[r]), bc(lev));
            }
          } else {
#pragma unroll
            for (int u = 0; u < PER0; ++u) {
              const int jj = t + u * T;
#pragma unroll
              for (int r = 0; r < R0; ++r) {
                const int m = jj + r * (L / R0);
                const float lev = 2.0f * s_lut16[load_one<GC>(wsl, boff, G, m, j)].x;
                v[u][r] = f2mul(prerot(m, phi0, dph.x, dph.y), bc(lev));
              }
            }
          }
        } else {
#pragma unroll
          for (int u = 0; u < PER0; ++u) {
            const int jj = t + u * T;
#pragma unroll
            for (int r = 0; r < R0; ++r) {
              if constexpr (TURN) {
                v[u][r] = s_lut16[(cw[r >> 3] >> (4 * (r & 7))) & 15u];
              } else {
                uint32_t c0, c1;
                load_pair<GC>(wsl, boff, G, jj + r * (L / R0), j, c0, c1);
                v[u][r] = s_lut16[c0 | (c1 << 2)];
              }
            }
          }
        }
#pragma unroll
        for (int u = 0; u < PER0; ++u) {
          const int jj = t + u * T;
          dft_reg<R0>(v[u]);
          if constexpr (P::R1 > 1 || !REGS) {
#pragma unroll
            for (int r = 0; r < R0; ++r) fbuf[padp<R0>(jj * R0 + r)] = v[u][r];
          }
        }
        // the passes after the first; the last one's results stay in registers
        // where their thread (pre-F) or warp (post-F) can finish them
        constexpr int RL = LastRadix<L>::v, PERL = L / RL / T;
        const float2* twl = Tw<L>::on ? s_tw : nullptr;
        const float2* twp1 = PassTw<L>::on ? s_twp : nullptr;
        const float2* twp2 = PassTw<L>::on ? s_twp + PassTw<L>::n1 : nullptr;
        if constexpr (P::R1 > 1) gsync<T>(grp);
        if constexpr (P::R2 > 1 && REGS) {  // the second of three passes, in place
          constexpr int R = P::R1, PER = L / R / T;
          float2 w[PER][R];
          stockham_values<L, R, P::R0, T, TWS>([&](int u, int r) { return fbuf[padp<R0>(t + u * T + r * (L / R))]; }, [] {}, t,
                                               p.twN, nullptr, twp1, w);
#pragma unroll
          for (int u = 0; u < PER; ++u)
#pragma unroll
            for (int r = 0; r < R; ++r) fbuf[padp<R0>(t + u * T + r * (L / R))] = w[u][r];
          gsync<T>(grp);
        }
        if constexpr (REGS) {
          float2 z[PERL][RL];  // Z[t + q T] = z[q % PERL][q / PERL]
          if constexpr (P::R2 > 1) {
            stockham_values<L, RL, L / RL, T, TWS>(
                [&](int u, int r) { return fbuf[third_place<L, R0, P::R1, T>(t, u, r)]; }, [] {}, t, p.twN, twl, twp2, z);
          } else if constexpr (P::R1 > 1) {
            stockham_values<L, RL, L / RL, T, TWS>(
                [&](int u, int r) { return fbuf[padp<R0>(t + u * T + r * (L / RL))]; }, [&] { gsync<T>(grp); }, t, p.twN, twl,
                twp1, z);
          } else {
#pragma unroll
            for (int r = 0; r < RL; ++r) z[0][r] = v[0][r];
          }
          auto finish = [&](auto kind) {
            constexpr int OUT = decltype(kind)::value;
            if constexpr (PRE)
              rotate_store_pre<L, T, OUT>([&](int q) { return z[q % PERL][q / PERL]; }, t, delta, p.out, obase, p.scale);
            else if constexpr (P::R2 > 1)
              split_rotate_places<L, R0, P::R1, T, OUT>(z, fbuf, t, grp, p.twN, phi, delta, p.out, obase, p.scale);
            else
              split_rotate_shuffle<L, T, OUT>(z, s_tw, t, phi, delta, p.out, obase, p.scale);
          };
          if (p.out_kind == 1) finish(std::integral_constant<int, 1>{});
          else if (p.out_kind == 2) finish(std::integral_constant<int, 2>{});
          else finish(std::integral_constant<int, 0>{});
        } else if constexpr (P::R1 > 1) {
          if constexpr (P::R2 > 1) stockham_pass<L, P::R1, P::R0, T, P::R0, TWS>(fbuf, t, grp, p.twN, nullptr, twp1);
          stockham_pass<L, RL, L / RL, T, P::R0, TWS>(fbuf, t, grp, p.twN, twl, P::R2 > 1 ? twp2 : twp1);
        } else {
          gsync<T>(grp);
        }
      }

      // ---- store (real split and post-F rotation, or the pre-F path's
      //      slope); a block that is not valid stores zeros ----
      if (active && !(REGS && ok)) {
        if constexpr (PRE) {
          if (p.out_kind == 1)
            store_zeros_pre<L, T, 1>(t, p.out, obase);
          else if (p.out_kind == 2)
            store_zeros_pre<L, T, 2>(t, p.out, obase);
          else
            store_zeros_pre<L, T, 0>(t, p.out, obase);
        } else {
          if (p.out_kind == 1)
            split_rotate_store<L, T, R0, 1>(fbuf, s_tw, p.twN, t, ok && !REGS, phi, delta, p.out, obase, p.scale);
          else if (p.out_kind == 2)
            split_rotate_store<L, T, R0, 2>(fbuf, s_tw, p.twN, t, ok && !REGS, phi, delta, p.out, obase, p.scale);
          else
            split_rotate_store<L, T, R0, 0>(fbuf, s_tw, p.twN, t, ok && !REGS, phi, delta, p.out, obase, p.scale);
        }
      }
      gsync<T>(grp);
    }
    __syncthreads();  // every read of this step's windows and codes is done before they are overwritten
    }
  }
}

template <int L, int GC, bool PRE, bool TURN>
static cudaError_t launch_turn(const FParams& p, int slots, int wslot, int jb, int nseq, size_t smem, cudaStream_t st) {
  cudaError_t e =
      cudaFuncSetAttribute(k_fstage<L, GC, PRE, TURN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int per_cta = slots * nseq;
  dim3 grid((p.CB + per_cta - 1) / per_cta, p.S);
  k_fstage<L, GC, PRE, TURN><<<grid, Plan<L>::T * Groups<L>::NGRP, smem, st>>>(p, slots, wslot, nseq, jb);
  return cudaGetLastError();
}

template <int L, int GC, bool PRE>
static cudaError_t launch_LG(const FParams& p, cudaStream_t st) {
  constexpr int NGRP = Groups<L>::NGRP;
  const int N = PRE ? L : 2 * L;
  const int wslot = wslot_words(N, p.G);
  const size_t fixed = sizeof(float2) * (Tw<L>::size + PassTw<L>::size) + 2048;
  auto resident = [&](size_t smem) { return (int)std::min<size_t>(MinBlocks<L>::v, 227 * 1024 / (smem + fixed)); };
  auto window = [&](int slots) { return (size_t)slots * wslot * sizeof(uint32_t); };
  auto turned = [&](int slots, int jb) {
    return kWordsOffset<L>(NGRP) + window(slots) +
           sizeof(uint32_t) * (size_t)slots * jb * Codes<L, PRE>::W * Codes<L, PRE>::T +
           (PRE ? sizeof(float2) * (size_t)slots * p.nsub * Codes<L, PRE>::R0 : 0);
  };
  static int sm_count = 0;
  if (!sm_count) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      sm_count = 152;
  }
  // Steps per CTA.  A start (tables, first windows) costs about a fifth of one
  // round of transforms, so a CTA whose step is one round takes eight steps
  // (1024 samples, 8 streams: 412 us against 489 with one step each); from four
  // rounds a step on, more and shorter CTAs even out the last wave better
  // (2048 samples, 16 streams: 328 us against 338 with two steps).  At least
  // four waves stay.
  auto steps_per_cta = [&](int slots, int ctas) {
    const int rounds = std::max(1, slots * p.G / NGRP);
    const int64_t steps = (int64_t)((p.CB + slots - 1) / slots) * p.S;
    const int64_t most = std::max<int64_t>(1, steps / ((int64_t)4 * ctas * sm_count));
    // the 8192-point form has one round per stream and stages the next windows into a buffer of their own
    if (L > 4096 && rounds >= 4) return (int)std::max<int64_t>(1, std::min<int64_t>(4, most / 2));
    return (int)std::min<int64_t>(rounds >= 4 ? 1 : (8 + rounds - 1) / rounds, most);
  };
  // blocks a CTA takes at a time: as many as give every group a transform
  const int base = std::max(1, std::min(64, NGRP / p.G));
  // Codes turned stream by stream: the turned codes of all streams (of 16 at a
  // time if more do not fit) beside the windows, as long as they cost no CTA
  // per SM.  A step ends at barriers, so it takes four rounds of transforms if
  // the windows fit and two waves of CTAs stay (1024 samples, 8, 16, 32
  // streams, which two blocks make 1, 2 and 4 rounds: 422, 353, 318 us).
  if constexpr (Codes<L, PRE>::on) {
    const int most = std::max(1, resident(kWordsOffset<L>(NGRP) + window(base)));
    const int64_t keep = (int64_t)p.CB * p.S / ((int64_t)2 * most * sm_count);  // blocks a CTA, for two waves
    int slots = (int)std::min<int64_t>(std::min(64, (4 * NGRP + p.G - 1) / p.G), std::max<int64_t>(base, keep));
    while (slots > base && resident(turned(slots, p.G)) < most) --slots;
    if (slots > base)
      return launch_turn<L, GC, PRE, true>(p, slots, wslot, p.G, steps_per_cta(slots, most), turned(slots, p.G), st);
    for (const int jb : {p.G, 16})
      if (jb <= p.G && resident(turned(base, jb)) >= most)
        return launch_turn<L, GC, PRE, true>(p, base, wslot, jb, steps_per_cta(base, most), turned(base, jb), st);
  }
  if constexpr (!Codes<L, PRE>::on || (L == 2048 && !PRE && GC != 16)) {  // (2048 points, more than 17 streams)
    const size_t one = kWordsOffset<L>(NGRP) + window(base), two = one + window(base);
    const int nseq = resident(two) == MinBlocks<L>::v ? steps_per_cta(base, resident(two)) : 1;
    const size_t smem = nseq > 1 ? two : one;
    if (resident(smem) < 1) return cudaErrorInvalidConfiguration;
    return launch_turn<L, GC, PRE, false>(p, base, wslot, p.G, nseq, smem, st);
  }
  return cudaErrorInvalidConfiguration;
}

}  // namespace corr
