// Line FFTs with 64 values per thread: a length-R line (R = RA RB) in two
// register-resident stages and one exchange through shared memory.
//
// The radix-16 stages of fft_block.cuh move every element of a 2048- or
// 4096-point line through shared memory twice, read a twiddle per element and
// stage, and wait at two barriers of 16 warps per stage; the passes built on
// them keep the shared-memory pipe 50-78 % busy and the issue slots 40-47 %
// (one-launch ncu captures), with DRAM at a third of its rate.  Here a thread
// transforms RA (then RB) points in registers, so a line goes through shared
// memory once, a tile of 8192 values needs 128 threads (barriers of four
// warps), and 64 independent loads per thread keep the memory system busy at
// three CTAs of four warps per SM (at most 168 registers).
//
// Stage 1: butterfly t < RB reads x[t + RB j], j < RA, and leaves output k at
// RA t + k; stage 2: butterfly t < RA reads x[t + RA j], j < RB, scales input j
// by w^{j t}, w = exp(-+2 pi i / R), and output k is X[t + RA k].  In shared
// memory the line is RB rows of RA values with one value of padding per row,
// so stage 1 writes rows and stage 2 reads columns without bank conflicts.
// Stage 2's twiddles are factored: j = NB a + b gives w^{NB a t} w^{b t}, the
// first applied before the inner DFTs over a, the second after them.  There the RB-point DFT
// has a factor of its own, exp(-+2 pi i b ka / RB) for output ka; WideTw reads the
// product of the two, rounded once, from a table (a value passes three products instead
// of four: an FP32 line of 2048 points is off by 1.05e-7 relative to 64 bits, by
// 1.13e-7 with two products, by 1.05e-7 with three radix-16 stages).  The column pass
// after F2f multiplies twice (WideTwPair): it keeps NA + NB - 2 (10 for RB = 32) values in
// registers for its butterflies and has none to spare.
#pragma once
#include "fft_block.cuh"

namespace pond {

constexpr int WIDE_V = 64;                  // values per thread
constexpr int WIDE_NT = TILE / WIDE_V;      // threads per tile

// cos(2 pi k / 64), k = 0 .. 16
__host__ __device__ constexpr float cos64(int k) {
  constexpr float c[17] = {1.00000000000000000f, 0.99518472667219693f, 0.98078528040323043f, 0.95694033573220882f,
                           0.92387953251128674f, 0.88192126434835505f, 0.83146961230254524f, 0.77301045336273699f,
                           0.70710678118654757f, 0.63439328416364549f, 0.55557023301960229f, 0.47139673682599781f,
                           0.38268343236508984f, 0.29028467725446233f, 0.19509032201612833f, 0.09801714032956077f,
                           0.00000000000000000f};
  k &= 63;
  return k <= 16 ? c[k] : k <= 32 ? -c[32 - k] : k <= 48 ? -c[k - 32] : c[64 - k];
}
__host__ __device__ constexpr float sin64(int k) { return cos64(k + 48); }   // cos(x - pi/2)

// a exp(-+2 pi i e / 64), e a compile-time constant after unrolling.
template <bool INV>
__device__ __forceinline__ float2 tw64(float2 a, int e) {
  e &= 63;
  if (e == 0) return a;
  if (e == 16) return rot90<INV>(a);
  if (e == 32) return make_float2(-a.x, -a.y);
  if (e == 48) return rot90<!INV>(a);
  if (e == 8) return rot45<INV>(a);
  if (e == 24) return rot135<INV>(a);
  return cmul(a, make_float2(cos64(e), INV ? sin64(e) : -sin64(e)));
}

// How an N-point register DFT splits: N = NA NB, input j = NB a + b, output k = ka + NA kb.
template <int N> struct WideSplit;
template <> struct WideSplit<64> { static constexpr int NA = 8, NB = 8; };
template <> struct WideSplit<32> { static constexpr int NA = 4, NB = 8; };
template <> struct WideSplit<16> { static constexpr int NA = 4, NB = 4; };
template <> struct WideSplit<8> { static constexpr int NA = 2, NB = 4; };

// N-point DFT of v, natural order in and out.  before(v, a) may scale input
// NB a + b ahead of the inner DFT over a; between(v, b, ka) scales its output ka
// after it, by the DFT's own factor exp(-+2 pi i b ka / N) among others.
template <int N, bool INV, class Before, class Between>
__device__ __forceinline__ void wide_dft(float2* v, Before before, Between between) {
  constexpr int NA = WideSplit<N>::NA, NB = WideSplit<N>::NB;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    float2 x[NA];
#pragma unroll
    for (int a = 0; a < NA; ++a) x[a] = before(v[NB * a + b], a);
    Dft<NA, INV>::run(x);
#pragma unroll
    for (int ka = 0; ka < NA; ++ka) v[NB * ka + b] = between(x[ka], b, ka);
  }
#pragma unroll
  for (int ka = 0; ka < NA; ++ka) Dft<NB, INV>::run(v + NB * ka);
  // v[NB ka + kb] = X[ka + NA kb]: to natural order (register renaming only)
  float2 y[N];
#pragma unroll
  for (int ka = 0; ka < NA; ++ka)
#pragma unroll
    for (int kb = 0; kb < NB; ++kb) y[ka + NA * kb] = v[NB * ka + kb];
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = y[i];
}

template <int N, bool INV>
__device__ __forceinline__ void wide_dft(float2* v) {
  wide_dft<N, INV>(v, [](float2 x, int) { return x; },
                   [](float2 x, int b, int ka) { return tw64<INV>(x, b * ka * (64 / N)); });
}

// Stage 2's twiddles of butterfly t, w = exp(-2 pi i / (RA RB)): w^{NB a t} (a = 1 .. NA-1)
// and w^{b (t + RA ka)} (b = 1 .. NB-1), which is w^{b t} times the RB-point DFT's own factor.
// In memory (FP64-built): a row of RA entries per (b, ka), then one per a.
template <int RA, int RB> struct WideTw {
  static constexpr int NA = WideSplit<RB>::NA, NB = WideSplit<RB>::NB;
  static constexpr int ROWS = NB * NA - 1;
  static constexpr int SIZE = ROWS * RA;
  float2 wa[NA - 1];
  const float2* wb;
  __device__ __forceinline__ void load(const float2* __restrict__ tw, int t) {
    wb = tw + t;
#pragma unroll
    for (int a = 1; a < NA; ++a) wa[a - 1] = __ldg(tw + ((NB - 1) * NA + a - 1) * RA + t);
  }
  // the twiddled RB-point DFT
  template <bool INV> __device__ __forceinline__ void dft(float2* v) const {
    wide_dft<RB, INV>(
        v, [&](float2 x, int a) { return a == 0 ? x : cmul(x, INV ? cconj(wa[a - 1]) : wa[a - 1]); },
        [&](float2 x, int b, int ka) {
          if (b == 0) return x;
          const float2 w = __ldg(wb + ((b - 1) * NA + ka) * RA);
          return cmul(x, INV ? cconj(w) : w);
        });
  }
};

// The same with w^{b t} alone, in registers, and the DFT's own factor multiplied after it; from
// the ka = 0 rows of the same table.
template <int RA, int RB> struct WideTwPair {
  static constexpr int NA = WideSplit<RB>::NA, NB = WideSplit<RB>::NB;
  float2 wa[NA - 1], wb[NB - 1];
  __device__ __forceinline__ void load(const float2* __restrict__ tw, int t) {
#pragma unroll
    for (int b = 1; b < NB; ++b) wb[b - 1] = __ldg(tw + (b - 1) * NA * RA + t);
#pragma unroll
    for (int a = 1; a < NA; ++a) wa[a - 1] = __ldg(tw + ((NB - 1) * NA + a - 1) * RA + t);
  }
  template <bool INV> __device__ __forceinline__ void dft(float2* v) const {
    wide_dft<RB, INV>(
        v, [&](float2 x, int a) { return a == 0 ? x : cmul(x, INV ? cconj(wa[a - 1]) : wa[a - 1]); },
        [&](float2 x, int b, int ka) {
          return tw64<INV>(b == 0 ? x : cmul(x, INV ? cconj(wb[b - 1]) : wb[b - 1]), b * ka * (64 / RB));
        });
  }
};

// Line stride of nl lines of RB rows of RA values: lanes that run over the lines
// first (16 / nl rows of each per half-warp) fall in distinct banks.
template <int RA, int RB>
__host__ __device__ constexpr int wide_stride() {
  constexpr int base = (RA + 1) * RB, nl = TILE / (RA * RB) > 16 ? 16 : TILE / (RA * RB);
  return base + ((16 / nl - base) & 15);
}

}  // namespace pond
