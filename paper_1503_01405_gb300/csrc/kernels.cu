// Segment kernels of the coherent-dedispersion path (PONDER Sec. 3.7).
//
// Overlap-save segments of N real int8 samples go through three or four FFT passes
// over a spectrum of L = N/2 complex bins (passes.cuh, passes_wide.cuh; FP32
// instantiations here), several consecutive segments to a launch, then fold and decimation:
//
//  k_fold_dec      : fold (FP64 phase) and decimation of a launch's segments.
//  k_fold_partial / k_fold_merge : deterministic fold of a series (FP64 phase).
//  k_decimate      : deterministic decimation of P into the time series.
#include <cuda_runtime.h>
#include <stdint.h>

#include "passes.cuh"
#include "passes_wide.cuh"

namespace pond {

// ---------------------------------------------------------------------------
// Tables (built once per plan, FP64 on the device)
// ---------------------------------------------------------------------------

// Concatenated stage twiddle tables of a length-R line FFT (see fft_block.cuh):
// entry (j-1) LS + k of the stage after sub-transforms of length LS holds
// exp(-2 pi i j k / (LS RAD)).
__global__ void k_make_stage_tw(float2* out, int R) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  int off = 0;
  for (int ls = 1; ls < R; ls *= stage_radix(R, ls)) {
    const int rad = stage_radix(R, ls);
    if (ls == 1) continue;
    const int n = (rad - 1) * ls;
    if (m >= off && m < off + n) {
      const int j = (m - off) / ls + 1, k = (m - off) % ls;
      double sn, cs;
      sincospi(-2.0 * (double)(j * k) / (double)(ls * rad), &sn, &cs);
      out[m] = make_float2((float)cs, (float)sn);
    }
    off += n;
  }
}

// Stage 2's twiddles of the (ra, rb) line FFT (fft_wide.cuh), rb = na nb: row
// (b - 1) na + ka (b = 1 .. nb-1, ka < na) holds w^{b (t + ra ka)}, row (nb - 1) na + a - 1
// (a = 1 .. na-1) w^{nb a t}, t < ra, w = exp(-2 pi i / (ra rb)).
__global__ void k_make_wide_tw(float2* out, int ra, int rb, int na, int nb) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (nb * na - 1) * ra) return;
  const int row = i / ra, t = i % ra;
  const int e = row < (nb - 1) * na ? (row / na + 1) * (t + ra * (row % na)) : nb * (row - (nb - 1) * na + 1) * t;
  double s, c;
  sincospi(-2.0 * (double)e / (double)(ra * rb), &s, &c);
  out[i] = make_float2((float)c, (float)s);
}

// Anchor a covers the 2^clog bins k = 2^clog a + d (d < 2^clog); it holds the
// Taylor coefficients of the dedispersion phase phi(k) = sgn * c(f_k) (cycles)
// about k_a = 2^clog a + 2^(clog-1): phi(k_a) mod 1 in Q0.32, phi'(k_a) and
// phi''(k_a)/2 mod 1 in Q0.64 (so the polynomial up to d^2 is exact mod 1 in
// integer arithmetic), phi'''(k_a)/6 in FP32.  c(f) = alpha f^2 / (f0 + f)
// with alpha = K 1e6 DM / f0^2 (Eq. 4), f = k du - |bw|/2 (upper sideband) or
// |bw|/2 - k du (inverted).  The planner picks clog so that the dropped
// quartic term stays below 1e-9 cycles.
__device__ __forceinline__ unsigned long long frac_q064(double x) {
  const double fr = x - floor(x);                 // in [0, 1), exact in FP64
  const double t = fr * 4294967296.0;             // exact scaling
  const double h = floor(t);
  const long long l = llrint((t - h) * 4294967296.0);
  return ((unsigned long long)h << 32) + (unsigned long long)l;   // a carry from l = 2^32 wraps mod 2^64
}

__global__ void k_make_chirp_anchors(ChirpAnchor* anc, long long nanc, int clog, double du, double half,
                                     double f0, double alpha, int sgn) {
  const long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= nanc) return;
  const long long span = 1ll << clog;
  const double ka = (double)(a * span + span / 2);
  const double f = sgn > 0 ? __dsub_rn(__dmul_rn(ka, du), half) : __dsub_rn(half, __dmul_rn(ka, du));
  const double g = f0 + f;
  const double q = f0 * f0 / (g * g);
  const double c = alpha * f * f / g;
  const double d1 = alpha * (1.0 - q);
  const double d2 = 2.0 * alpha * q / g;
  const double d3 = -6.0 * alpha * q / (g * g);
  const double phi0 = sgn * c;
  const double phi1 = du * d1;
  const double phi2 = sgn * du * du * d2 * 0.5;
  const double phi3 = du * du * du * d3 / 6.0;
  const double fr0 = phi0 - floor(phi0);
  ChirpAnchor r;
  r.p0 = (unsigned)((unsigned long long)llrint(fr0 * 4294967296.0) & 0xffffffffull);
  r.p1 = frac_q064(phi1);
  r.p2 = frac_q064(phi2);
  r.p3 = (float)phi3;
  r.pad[0] = r.pad[1] = 0u;
  anc[a] = r;
}

// Three-level table for exponents e < 2^24: entry 256 l + j holds
// w^(j 2^(8 l)), w = exp(sign 2 pi i / 2^logn) (FP64 sincospi).
__global__ void k_make_tw3(float2* out, int logn, int sign) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 768) return;
  const long long e = (long long)(i & 255) << (8 * (i >> 8));
  double s, c;
  sincospi(2.0 * sign * (double)e / (double)(1ll << logn), &s, &c);
  out[i] = make_float2((float)c, (float)s);
}

// ---------------------------------------------------------------------------
// Two-level twiddle tables: w^e = hi[e >> 12] * lo[e & 4095], w = exp(+-2 pi i / n)
// ---------------------------------------------------------------------------

__global__ void k_make_tw2(float2* lo, float2* hi, int logn, int sign) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const double inv = 2.0 * sign / (double)(1ll << logn);
  double s, c;
  if (i < TW2_LO) {
    sincospi(inv * (double)i, &s, &c);
    lo[i] = make_float2((float)c, (float)s);
  }
  const long long nhi = logn > TW2_LOG ? (1ll << (logn - TW2_LOG)) : 1;
  if (i < nhi) {
    sincospi(inv * (double)((long long)i << TW2_LOG), &s, &c);
    hi[i] = make_float2((float)c, (float)s);
  }
}

// ---------------------------------------------------------------------------
// Fold (Sec. 3.4 fold thread): deterministic per-warp histograms
// ---------------------------------------------------------------------------

constexpr int FOLD_WARPS = 4;
constexpr int FOLD_U = 4;        // 32-sample groups in flight per warp

// The fold's phase rules: phase(g) in cycles and whether it is known to run
// forwards over samples [ga, gb] in its FP64 evaluation.  Each FP64 operation
// is rounded on its own, so bins are those of a plain evaluation.
struct ConstPeriod {
  double inc;
  __device__ __forceinline__ double operator()(long long g) const { return __dmul_rn((double)g, inc); }
  __device__ __forceinline__ bool forwards(long long, long long) const { return true; }   // one rounded product: monotone
};

// Polynomial phase model, Horner's rule.
struct PhaseRule {
  FoldPhase r;
  __device__ __forceinline__ double operator()(long long g) const {
    const double tau = __dsub_rn(__dmul_rn((double)g, r.dt), r.t_ref);
    double x = r.c[r.nc - 1];
    for (int k = r.nc - 2; k >= 0; --k) x = __dadd_rn(__dmul_rn(x, tau), r.c[k]);
    return x;
  }
  __device__ bool forwards(long long ga, long long gb) const {
    return phase_forwards(r.c, r.nc, r.dt, r.t_ref, ga, gb);
  }
};

// bin = min(floor((phi - floor(phi)) nbins), nbins - 1); key = floor(phi) nbins + bin.
__device__ __forceinline__ int phase_bin(double x, int nbins, double* key = nullptr) {
  const double q = floor(x);
  const int t = (int)__dmul_rn(__dsub_rn(x, q), (double)nbins), b = t < nbins - 1 ? t : nbins - 1;
  if (key) *key = q * (double)nbins + (double)b;   // an integer below 2^53: exact
  return b;
}

// Fold a window of 32 FOLD_RUN channel samples [c, ..) of P (global index g + i) whose
// phase runs forwards: lane l takes FOLD_RUN consecutive samples, evaluates the phase at
// the first and last of them and, where the bin changes in between, finds the
// change by bisection, so a window costs two to seven phase evaluations per lane
// instead of FOLD_RUN (an SM retires two FP64 operations per clock, which bounded the
// per-sample form: a 2^20-sample segment 34.7 -> 7 us, nine segments of 113k samples with a
// phase model 579 -> 83 us).  Each lane's one or two FP32 sums are joined with its neighbours' of the
// same bin in FP64, in lane order.  False (nothing added) when a lane's samples span more
// than two bins or the window comes back to a bin.
constexpr int FOLD_RUN = 32, FOLD_WIN = 32 * FOLD_RUN;
template <class Rule>
__device__ __forceinline__ bool fold_window(const float* __restrict__ P, long long c, long long g, const Rule& rule,
                                            int nbins, int b0, double* myh, int* myc) {
  const int lane = threadIdx.x & 31;
  float v[FOLD_RUN];
  const float4* src = reinterpret_cast<const float4*>(P + c) + lane * (FOLD_RUN / 4);
#pragma unroll
  for (int i = 0; i < FOLD_RUN / 4; ++i) {
    const float4 q = __ldg(src + i);
    v[4 * i] = q.x;
    v[4 * i + 1] = q.y;
    v[4 * i + 2] = q.z;
    v[4 * i + 3] = q.w;
  }
  const long long ga = g + lane * FOLD_RUN;
  double kf, kt;
  const int bf = phase_bin(rule(ga), nbins, &kf), bt = phase_bin(rule(ga + FOLD_RUN - 1), nbins, &kt);
  int split = FOLD_RUN;   // samples before the change of bin
  bool ok = true;
  if (__any_sync(0xffffffffu, kf != kt)) {
    int lo = 0, hi = FOLD_RUN - 1;   // key(lo) = kf, key(hi) > kf
    double kh = kt;
#pragma unroll 1
    for (int s = 0; s < 5; ++s) {
      const int mid = (lo + hi) >> 1;
      double km;
      phase_bin(rule(ga + mid), nbins, &km);
      if (km > kf) {
        hi = mid;
        kh = km;
      } else {
        lo = mid;
      }
    }
    if (kf != kt) {
      split = hi;
      ok = kh == kt;
    }
  }
  const double k0 = __shfl_sync(0xffffffffu, kf, 0), k1 = __shfl_sync(0xffffffffu, kt, 31);
  if (!__all_sync(0xffffffffu, ok) || !(k1 - k0 < (double)nbins)) return false;
  float sl = 0.f, sr = 0.f;
  {
    float l[4] = {0.f, 0.f, 0.f, 0.f}, r[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < FOLD_RUN; ++i) {
      l[i & 3] += i < split ? v[i] : 0.f;
      r[i & 3] += i < split ? 0.f : v[i];
    }
    sl = (l[0] + l[1]) + (l[2] + l[3]);
    sr = (r[0] + r[1]) + (r[2] + r[3]);
  }
  // chain of the lanes' last bins: lane l continues lane l-1's sum when all its
  // samples lie in that bin
  const bool two = split < FOLD_RUN;
  const double kp = __shfl_up_sync(0xffffffffu, kt, 1), kn = __shfl_down_sync(0xffffffffu, kf, 1);
  const bool joins = lane > 0 && kp == kf;   // the first part belongs to the previous lane's bin
  double s = two ? (double)sr : (double)sl;
  int n = two ? FOLD_RUN - split : FOLD_RUN;
  bool open = joins && !two;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const double ps = __shfl_up_sync(0xffffffffu, s, d);
    const int pn = __shfl_up_sync(0xffffffffu, n, d);
    const bool po = __shfl_up_sync(0xffffffffu, open, d);
    if (lane >= d && open) {
      s += ps;
      n += pn;
      open = po;
    }
  }
  const double ps = __shfl_up_sync(0xffffffffu, s, 1);
  const int pn = __shfl_up_sync(0xffffffffu, n, 1);
  if (two) {
    const int e = bf >= b0 ? bf - b0 : bf - b0 + nbins;
    myh[e] += joins ? ps + (double)sl : (double)sl;
    myc[e] += joins ? pn + split : split;
  }
  __syncwarp();
  if (lane == 31 || kn != kt) {
    const int e = bt >= b0 ? bt - b0 : bt - b0 + nbins;
    myh[e] += s;
    myc[e] += n;
  }
  __syncwarp();
  return true;
}

// Fold 32 channel samples, one per lane, into the warp's histogram (b < 0: none).
__device__ __forceinline__ void fold_group(int b, float p, int nbins, int b0, double* myh, int* myc, float* mybuf) {
  const int lane = threadIdx.x & 31;
  const bool ok = b >= 0;
  const unsigned peers = __match_any_sync(0xffffffffu, b);
  const int first = __ffs(peers) - 1;
  const int last = 31 - __clz(peers);
  const unsigned span = (last == 31 ? 0xffffffffu : ((1u << (last + 1)) - 1u)) & ~((1u << first) - 1u);
  if (__all_sync(0xffffffffu, peers == span)) {
    // every bin's lanes are contiguous: segmented scan in a fixed tree order
    float x = p;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const float y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane - d >= first) x += y;
    }
    if (ok && lane == last) {
      const int e = b >= b0 ? b - b0 : b - b0 + nbins;
      myh[e] += (double)x;
      myc[e] += last - first + 1;
    }
  } else {
    // a period shorter than a warp: the group leader sums its lanes in order
    mybuf[lane] = p;
    __syncwarp();
    if (ok && lane == first) {
      float sum = 0.f;
      unsigned m = peers;
      while (m) {
        sum += mybuf[__ffs(m) - 1];
        m &= m - 1;
      }
      const int e = b >= b0 ? b - b0 : b - b0 + nbins;
      myh[e] += (double)sum;
      myc[e] += __popc(peers);
    }
  }
  __syncwarp();
}

// Fold channel samples [c0, c1) of P (global index g0 + c) into this warp's
// histogram; FOLD_WARPS warps share the chunk.  From two windows on, whole windows whose
// phase runs forwards go through fold_window (a single one would leave to one warp
// what four share sample by sample: 15,600 samples 5 against 20 us); the
// rest goes sample by sample, FOLD_U groups of 32 per warp and
// step (their loads and phases in flight before the groups are added in order).
// Bin b is kept at entry (b - b0) mod nbins, so a chunk that spans a short cyclic
// run of bins starting at b0 needs only that run's entries.
template <class Rule>
__device__ __forceinline__ void fold_chunk(const float* __restrict__ P, long long c0, long long c1, long long g0,
                                           const Rule& rule, int nbins, int b0, double* myh, int* myc, float* mybuf) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto by_sample = [&](long long a, long long e, int step) {
    for (long long base = a; base < e; base += step) {
      float pv[FOLD_U];
      int bv[FOLD_U];
#pragma unroll
      for (int u = 0; u < FOLD_U; ++u) {
        const long long i = base + u * 32 + lane;
        pv[u] = 0.f;
        bv[u] = -1;
        if (i < e) {
          pv[u] = __ldg(P + i);
          bv[u] = phase_bin(rule(g0 + i), nbins);
        }
      }
#pragma unroll
      for (int u = 0; u < FOLD_U; ++u) fold_group(bv[u], pv[u], nbins, b0, myh, myc, mybuf);
    }
  };
  long long tail = c0;
  if ((reinterpret_cast<uintptr_t>(P + c0) & 15) == 0 && c1 - c0 >= 2 * FOLD_WIN &&
      rule.forwards(g0 + c0, g0 + c1)) {
    const int nwin = (int)((c1 - c0) / FOLD_WIN);
    for (int i = w; i < nwin; i += FOLD_WARPS) {
      const long long c = c0 + (long long)i * FOLD_WIN;
      if (!fold_window(P, c, g0 + c, rule, nbins, b0, myh, myc)) by_sample(c, c + FOLD_WIN, 32 * FOLD_U);
    }
    tail = c0 + (long long)nwin * FOLD_WIN;
  }
  by_sample(tail + (long long)w * 32 * FOLD_U, c1, FOLD_WARPS * 32 * FOLD_U);
}

// Shared-memory layout of the fold kernels: [FOLD_WARPS][nbins] FP64 sums,
// [FOLD_WARPS][nbins] int32 hits, [FOLD_WARPS][32] FP32 staging.
struct FoldSmem {
  double* hsum;
  int* hcnt;
  float* pbuf;
};

__device__ __forceinline__ FoldSmem fold_smem_init(unsigned char* fsm, int nbins, int used) {
  FoldSmem f;
  f.hsum = reinterpret_cast<double*>(fsm);
  f.hcnt = reinterpret_cast<int*>(f.hsum + FOLD_WARPS * nbins);
  f.pbuf = reinterpret_cast<float*>(f.hcnt + FOLD_WARPS * nbins);
  for (int i = threadIdx.x; i < FOLD_WARPS * used; i += blockDim.x) {
    const int k = (i / used) * nbins + i % used;
    f.hsum[k] = 0.0;
    f.hcnt[k] = 0;
  }
  __syncthreads();
  return f;
}

// One CTA per chunk of channel samples: the CTA's histogram (warps added in
// order) is written to row blockIdx.x of the partials.
__global__ void __launch_bounds__(FOLD_WARPS * 32) k_fold_partial(const float* __restrict__ P, long long n,
                                                                  long long g0, double inc, int nbins,
                                                                  long long chunk, double* __restrict__ psum,
                                                                  int* __restrict__ phits) {
  extern __shared__ unsigned char fsm[];
  const FoldSmem f = fold_smem_init(fsm, nbins, nbins);
  const int w = threadIdx.x >> 5;
  const long long c0 = (long long)blockIdx.x * chunk;
  fold_chunk(P, c0, min(n, c0 + chunk), g0, ConstPeriod{inc}, nbins, 0, f.hsum + w * nbins, f.hcnt + w * nbins,
             f.pbuf + w * 32);
  __syncthreads();
  for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
    double s = 0.0;
    int h = 0;
#pragma unroll
    for (int k = 0; k < FOLD_WARPS; ++k) {
      s += f.hsum[k * nbins + b];
      h += f.hcnt[k * nbins + b];
    }
    psum[(size_t)blockIdx.x * nbins + b] = s;
    phits[(size_t)blockIdx.x * nbins + b] = h;
  }
}

__device__ __forceinline__ long long ceil_div_ll(long long a, long long b) { return (a + b - 1) / b; }

// Series samples spanning at most DEC_SPAN channel samples load them together.
constexpr int DEC_SPAN = 16;

// The sum of P[g0 .. g0 + n) over g in [a, e) by one thread (spans under 64 samples).
__device__ __forceinline__ float dec_span(const float* __restrict__ P, long long a, long long e) {
  float s = 0.f;
  if (e - a <= DEC_SPAN) {
    // loads issued together, added in sample order
    float v[DEC_SPAN];
#pragma unroll
    for (int i = 0; i < DEC_SPAN; ++i) v[i] = a + i < e ? __ldg(P + a + i) : 0.f;
#pragma unroll
    for (int i = 0; i < DEC_SPAN; ++i)
      if (a + i < e) s += v[i];
  } else {
    for (long long g = a; g < e; ++g) s += __ldg(P + g);
  }
  return s;
}

// The same by one warp: four partial sums per lane, then a fixed tree.
__device__ __forceinline__ float dec_span_warp(const float* __restrict__ P, long long a, long long e, int lane) {
  float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
  long long g = a + lane;
  for (; g + 96 < e; g += 128) {
    s0 += __ldg(P + g);
    s1 += __ldg(P + g + 32);
    s2 += __ldg(P + g + 64);
    s3 += __ldg(P + g + 96);
  }
  if (g < e) s0 += __ldg(P + g);
  if (g + 32 < e) s1 += __ldg(P + g + 32);
  if (g + 64 < e) s2 += __ldg(P + g + 64);
  float s = (s0 + s1) + (s2 + s3);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  return s;
}

// Fold + decimation of the valid spans of nseg consecutive segments in one launch.
// The first parts nseg CTAs fold: CTA (y, x) adds chunk x of segment y to partial
// row (s mod slots) parts + x, which accumulates over the stream and is merged
// when the profile is read; a launch holds at most `slots` segments, so no two of
// its CTAs share a row and every row takes its segments in order however they
// are grouped.  The other CTAs own the series samples j: one thread per j for spans under
// 64 channel samples, else one warp.  A sample that straddles segments adds one
// sum per segment, in order, as separate launches would.  No atomics.
template <bool MODEL>
__global__ void __launch_bounds__(FOLD_WARPS * 32) k_fold_dec(const float* __restrict__ P, FoldSegs f, FoldPhase rule,
                                                              int nbins, int slots, int parts, long long chunk,
                                                              long long num, long long den, long long j_lo,
                                                              long long nj, float* __restrict__ T,
                                                              int* __restrict__ C, long long ring,
                                                              double* __restrict__ psum,
                                                              long long* __restrict__ phits) {
  extern __shared__ unsigned char fsm[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nfold = parts * f.nseg;
  if ((int)blockIdx.x < nfold) {
    const int y = blockIdx.x / parts, x = blockIdx.x - y * parts;
    const long long n = min(f.S_c, f.n_left - y * f.S_c), c0 = x * chunk, c1 = min(n, c0 + chunk);
    if (c1 <= c0) return;
    const long long gy = f.g0 + y * f.S_c;
    // at the constant period the phase grows with g, so a chunk shorter than one
    // period (with a margin of two bins) covers the cyclic run of bins
    // of its first and last sample; a phase model keeps every bin
    int b0 = 0, used = nbins;
    if (!MODEL && (double)(c1 - 1 - c0) * rule.inc < 1.0 - 2.0 / nbins) {
      const ConstPeriod cp{rule.inc};
      b0 = phase_bin(cp(gy + c0), nbins);
      const int b1 = phase_bin(cp(gy + c1 - 1), nbins);
      used = (b1 >= b0 ? b1 - b0 : b1 - b0 + nbins) + 1;
    }
    const FoldSmem fs = fold_smem_init(fsm, nbins, used);
    const float* Py = P + y * f.M;
    if constexpr (MODEL)
      fold_chunk(Py, c0, c1, gy, PhaseRule{rule}, nbins, b0, fs.hsum + w * nbins, fs.hcnt + w * nbins, fs.pbuf + w * 32);
    else
      fold_chunk(Py, c0, c1, gy, ConstPeriod{rule.inc}, nbins, b0, fs.hsum + w * nbins, fs.hcnt + w * nbins, fs.pbuf + w * 32);
    __syncthreads();
    const size_t row = (size_t)((f.s0 + y) % slots) * parts + x;
    for (int e = threadIdx.x; e < used; e += blockDim.x) {
      double s = 0.0;
      int h = 0;
#pragma unroll
      for (int q = 0; q < FOLD_WARPS; ++q) {
        s += fs.hsum[q * nbins + e];
        h += fs.hcnt[q * nbins + e];
      }
      const int b = b0 + e < nbins ? b0 + e : b0 + e - nbins;
      psum[row * nbins + b] += s;
      phits[row * nbins + b] += h;
    }
    return;
  }
  const long long g_end = f.g0 + f.n_left;
  const bool by_warp = num >= 64 * den;
  const long long jj = by_warp ? (long long)(blockIdx.x - nfold) * FOLD_WARPS + w
                               : (long long)(blockIdx.x - nfold) * (FOLD_WARPS * 32) + threadIdx.x;
  if (jj >= nj) return;
  const long long j = j_lo + jj, slot = j % ring;
  long long a = max(ceil_div_ll(j * num, den), f.g0);
  const long long e = min(ceil_div_ll((j + 1) * num, den), g_end);
  const int c = (int)max(e - a, 0ll);
  const bool owner = !by_warp || lane == 0;
  float t = owner ? T[slot] : 0.f;
  while (a < e) {   // uniform over a warp in the by_warp form
    const long long y = (a - f.g0) / f.S_c, base = f.g0 + y * f.S_c, ey = min(e, base + f.S_c);
    t += by_warp ? dec_span_warp(P + y * f.M, a - base, ey - base, lane) : dec_span(P + y * f.M, a - base, ey - base);
    a = ey;
  }
  if (owner) {
    T[slot] = t;
    C[slot] += c;
  }
}

// A CTA merges 32 consecutive bins: warp y of W sums parts y, y + W, y + 2 W, ... in
// order (lanes read 32 consecutive bins of a part: coalesced), then lane x of
// warp 0 adds the warp sums of bin x in a fixed order.  ACC adds the
// result to the profile, otherwise it replaces it.
constexpr int MERGE_WARPS = 8, SNAP_WARPS = 32;

template <typename H, bool ACC, int W>
__global__ void __launch_bounds__(W * 32) k_fold_merge(const double* __restrict__ psum,
                                                                 const H* __restrict__ phits, int nparts,
                                                                 int nbins, double* __restrict__ prof_sum,
                                                                 long long* __restrict__ prof_hits) {
  __shared__ double ss[W][32];
  __shared__ long long sh[W][32];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  const int b = blockIdx.x * 32 + x;
  double s = 0.0;
  long long h = 0;
  if (b < nbins) {
#pragma unroll 4
    for (int k = y; k < nparts; k += W) {
      s += __ldg(psum + (size_t)k * nbins + b);
      h += (long long)__ldg(phits + (size_t)k * nbins + b);
    }
  }
  ss[y][x] = s;
  sh[y][x] = h;
  __syncthreads();
  if (y == 0 && b < nbins) {
    double t = 0.0;
    long long c = 0;
#pragma unroll
    for (int k = 0; k < W; ++k) {
      t += ss[k][x];
      c += sh[k][x];
    }
    if (ACC) {
      prof_sum[b] += t;
      prof_hits[b] += c;
    } else {
      prof_sum[b] = t;
      prof_hits[b] = c;
    }
  }
}

// ---------------------------------------------------------------------------
// Decimation: T[j] += sum of P[g], floor(g den / num) = j; one warp per j
// ---------------------------------------------------------------------------

// One warp per series sample j (spans of 64 or more channel samples): four
// independent partial sums keep four loads in flight per lane, combined in a
// fixed order, then a fixed xor-tree over the lanes.
__global__ void k_decimate(const float* __restrict__ P, long long n, long long g0, long long num,
                           long long den, long long j_lo, long long nj, float* __restrict__ T,
                           int* __restrict__ C, long long ring) {
  const long long jj = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (jj >= nj) return;
  const long long j = j_lo + jj;
  long long ga = ceil_div_ll(j * num, den), gb = ceil_div_ll((j + 1) * num, den);
  ga = max(ga, g0);
  gb = min(gb, g0 + n);
  float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
  long long g = ga + lane;
  for (; g + 96 < gb; g += 128) {
    s0 += __ldg(P + (g - g0));
    s1 += __ldg(P + (g + 32 - g0));
    s2 += __ldg(P + (g + 64 - g0));
    s3 += __ldg(P + (g + 96 - g0));
  }
  if (g < gb) s0 += __ldg(P + (g - g0));
  if (g + 32 < gb) s1 += __ldg(P + (g + 32 - g0));
  if (g + 64 < gb) s2 += __ldg(P + (g + 64 - g0));
  float s = (s0 + s1) + (s2 + s3);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane == 0) {
    const long long slot = j % ring;
    T[slot] += s;
    C[slot] += (int)max(gb - ga, 0ll);
  }
}

// One thread per series sample j (spans shorter than 64 channel samples): the
// span is summed in index order; neighbouring threads read neighbouring spans.
__global__ void k_decimate_short(const float* __restrict__ P, long long n, long long g0, long long num,
                                 long long den, long long j_lo, long long nj, float* __restrict__ T,
                                 int* __restrict__ C, long long ring) {
  const long long jj = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (jj >= nj) return;
  const long long j = j_lo + jj;
  long long ga = ceil_div_ll(j * num, den), gb = ceil_div_ll((j + 1) * num, den);
  ga = max(ga, g0);
  gb = min(gb, g0 + n);
  float s = 0.f;
  for (long long g = ga; g < gb; ++g) s += __ldg(P + (g - g0));
  const long long slot = j % ring;
  T[slot] += s;
  C[slot] += (int)max(gb - ga, 0ll);
}

// k_decimate_short for the trials of one batched launch: blockIdx.y = trial t,
// reading P + t pstride and adding to series row rows[t].
__global__ void k_decimate_short_multi(const float* __restrict__ P, long long pstride, long long n, long long g0,
                                       long long num, long long den, long long j_lo, long long nj,
                                       float* __restrict__ T, int* __restrict__ C, long long ring,
                                       const int* __restrict__ rows) {
  const long long jj = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (jj >= nj) return;
  const int row = __ldg(rows + blockIdx.y);
  P += blockIdx.y * pstride;
  const long long j = j_lo + jj;
  long long ga = ceil_div_ll(j * num, den), gb = ceil_div_ll((j + 1) * num, den);
  ga = max(ga, g0);
  gb = min(gb, g0 + n);
  float s = 0.f;
  for (long long g = ga; g < gb; ++g) s += __ldg(P + (g - g0));
  const long long slot = (size_t)row * ring + j % ring;
  T[slot] += s;
  C[slot] += (int)max(gb - ga, 0ll);
}

// Chirp table of a batched lane whose DMs are whole multiples of dDM: entry
// k2 R1 + k1 (the spectrum's row layout, bin k = k2 + R2 k1) holds the phase of
// Eq. 4's inverse at bin k for one DM step, sgn dDM c(f_k) mod 1, as a Q0.32
// word (FP64, the same formula as the anchors' phase term).
__global__ void k_make_chirp_table(unsigned* tab, int logR1, int logR2, double du, double half, double f0,
                                   double alpha, int sgn) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (1ll << (logR1 + logR2))) return;
  const long long k2 = i >> logR1, k1 = i & ((1ll << logR1) - 1);
  const double k = (double)(k2 + (k1 << logR2));
  const double f = sgn > 0 ? __dsub_rn(__dmul_rn(k, du), half) : __dsub_rn(half, __dmul_rn(k, du));
  const double g = f0 + f;
  const double phi = sgn * (alpha * f * f / g);
  const double fr = phi - floor(phi);
  tab[i] = (unsigned)((unsigned long long)llrint(fr * 4294967296.0) & 0xffffffffull);
}

// The inverse filter of Eq. 4 per bin as FP32 (cos, -sin) of 2 pi phi(k), in
// F2f's order (runs): row k2, then the position j in a run of 64 columns, then the run c (bin
// k2 + R2 (64 c + j) at k2 R1 + j NCH + c, NCH = R1 / 64), or the spectrum's (bin k2 + R2 k1 at
// k2 R1 + k1).  phi in FP64 with the
// anchors' formula, reduced mod 1, then FP64 sincospi, rounded once to FP32.
__global__ void k_make_chirp_c64(float2* tab, int logR1, int logR2, bool runs, double du, double half, double f0, double alpha,
                                 int sgn) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (1ll << (logR1 + logR2))) return;
  const long long k2 = i >> logR1, e = i & ((1ll << logR1) - 1);
  const long long k1 = runs ? ((e & ((1ll << (logR1 - 6)) - 1)) << 6) + (e >> (logR1 - 6)) : e;
  const double k = (double)(k2 + (k1 << logR2));
  const double f = sgn > 0 ? __dsub_rn(__dmul_rn(k, du), half) : __dsub_rn(half, __dmul_rn(k, du));
  const double g = f0 + f;
  const double phi = sgn * (alpha * f * f / g);
  double r = phi - floor(phi);
  if (r > 0.5) r -= 1.0;
  double sn, cs;
  sincospi(2.0 * r, &sn, &cs);
  tab[i] = make_float2((float)cs, (float)-sn);
}

// A trial's phase words (anchor_word), in the same order as the table above.
__global__ void k_make_chirp_words(unsigned* words, int logR1, int logR2, const ChirpAnchor* __restrict__ anc, int clog) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (1ll << (logR1 + logR2))) return;
  const long long k2 = i >> logR1, e = i & ((1ll << logR1) - 1), nch = 1ll << (logR1 - 6);
  const unsigned k = (unsigned)(k2 + ((((e & (nch - 1)) << 6) + (e >> (logR1 - 6))) << logR2));
  words[i] = anchor_word(anc[k >> clog], clog, k);
}

// Byte copy between device buffers (any alignment): 16-byte words of dst, each from the
// one to five aligned 4-byte words of src that hold its bytes; single bytes at the ends.
// (A byte at a time where the sides disagree, the carry of an N / S stream pushed in odd
// pieces took 141 us per push.)
__global__ void k_copy_bytes(int8_t* __restrict__ dst, const int8_t* __restrict__ src, long long n) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long head = min(n, (long long)(-(uintptr_t)dst & 15)), n16 = (n - head) >> 4;
  const int8_t* s = src + head;
  uint4* d = reinterpret_cast<uint4*>(dst + head);
  const unsigned mis = (unsigned)((uintptr_t)s & 15), sh = (mis & 3) * 8;
  if (mis == 0) {
    for (long long i = i0; i < n16; i += stride) d[i] = __ldg(reinterpret_cast<const uint4*>(s) + i);
  } else {
    const unsigned* w = reinterpret_cast<const unsigned*>(s - (mis & 3));
    for (long long i = i0; i < n16; i += stride) {
      const unsigned* p = w + 4 * i;
      const unsigned a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2), e = __ldg(p + 3), f = sh ? __ldg(p + 4) : 0u;
      d[i] = make_uint4(__funnelshift_r(a, b, sh), __funnelshift_r(b, c, sh), __funnelshift_r(c, e, sh),
                        __funnelshift_r(e, f, sh));
    }
  }
  for (long long i = i0; i < head; i += stride) dst[i] = src[i];
  for (long long i = head + (n16 << 4) + i0; i < n; i += stride) dst[i] = src[i];
}

// ---------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------

// Host (mapped, pinned) -> device copy by a few CTAs: each thread keeps four
// 16-byte loads in flight, so 8 CTAs stream host memory (191 GB/s alone, the
// link's 211 GB/s from 16 CTAs on) faster than the passes consume it while
// leaving the other SMs to them.  Both pointers 16-byte aligned.
__global__ void __launch_bounds__(512) k_copy_host(uint4* __restrict__ dst, const uint4* __restrict__ src,
                                                    long long n16) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (; i + 3 * stride < n16; i += 4 * stride) {
    const uint4 a = __ldcs(src + i), b = __ldcs(src + i + stride), c = __ldcs(src + i + 2 * stride),
                d = __ldcs(src + i + 3 * stride);
    dst[i] = a;
    dst[i + stride] = b;
    dst[i + 2 * stride] = c;
    dst[i + 3 * stride] = d;
  }
  for (; i < n16; i += stride) dst[i] = __ldcs(src + i);
}

cudaError_t launch_copy_host(int8_t* dst, const int8_t* src, long long n, int blocks, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  if ((((uintptr_t)dst | (uintptr_t)src) & 15) != 0) return launch_copy_bytes(dst, src, n, st);
  const long long body = n & ~15ll;
  if (body > 0)
    k_copy_host<<<blocks, 512, 0, st>>>(reinterpret_cast<uint4*>(dst), reinterpret_cast<const uint4*>(src), body >> 4);
  if (n > body) return launch_copy_bytes(dst + body, src + body, n - body, st);
  return cudaGetLastError();
}

cudaError_t launch_copy_bytes(int8_t* dst, const int8_t* src, long long n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  // at most two CTAs per SM: the copy runs beside segment passes, whose CTAs
  // cannot share an SM with a third resident CTA
  const long long words = std::max(1ll, n >> 4);
  const unsigned blocks = (unsigned)std::min<long long>((words + 255) / 256, 304);
  k_copy_bytes<<<blocks, 256, 0, st>>>(dst, src, n);
  return cudaGetLastError();
}

cudaError_t launch_chirp_c64(float2* tab, const Geom& g, bool runs, double du, double half, double f0, double alpha, int sgn,
                             cudaStream_t st) {
  const long long n = g.L;
  k_make_chirp_c64<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(tab, g.logR1, g.logR2, runs, du, half, f0, alpha, sgn);
  return cudaGetLastError();
}

cudaError_t launch_chirp_words(unsigned* words, const Geom& g, const ChirpAnchor* anc, int clog, cudaStream_t st) {
  k_make_chirp_words<<<(unsigned)((g.L + 255) / 256), 256, 0, st>>>(words, g.logR1, g.logR2, anc, clog);
  return cudaGetLastError();
}

cudaError_t launch_chirp_table(unsigned* tab, const Geom& g, double du, double half, double f0, double alpha, int sgn,
                               cudaStream_t st) {
  const long long n = g.L;
  k_make_chirp_table<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(tab, g.logR1, g.logR2, du, half, f0, alpha, sgn);
  return cudaGetLastError();
}

cudaError_t launch_decimate_multi(const float* P, long long pstride, long long n, long long g0, long long num,
                                  long long den, long long j_lo, long long nj, float* T, int* C, long long ring,
                                  const int* rows, int ntr, cudaStream_t st) {
  if (n <= 0 || nj <= 0) return cudaSuccess;
  if (num >= 64 * den) return cudaErrorInvalidValue;   // short spans only (batched plans decimate by a few)
  const dim3 grid((unsigned)((nj + 255) / 256), (unsigned)ntr);
  k_decimate_short_multi<<<grid, 256, 0, st>>>(P, pstride, n, g0, num, den, j_lo, nj, T, C, ring, rows);
  return cudaGetLastError();
}

cudaError_t launch_stage_tw(float2* out, int R, cudaStream_t st) {
  const int n = stage_table_size(R);
  if (n > 0) k_make_stage_tw<<<(n + 255) / 256, 256, 0, st>>>(out, R);
  return cudaGetLastError();
}

int stage_tw_entries(int R) { return stage_table_size(R); }

#define POND_WIDE_RB(X) X(8) X(16) X(32) X(64)

int wide_tw_entries(int R, bool last64) {
  switch (R / 64) {
#define CASE(RB) case RB: return last64 ? WideTw<RB, 64>::SIZE : WideTw<64, RB>::SIZE;
    POND_WIDE_RB(CASE)
#undef CASE
    default: return 0;
  }
}

cudaError_t launch_wide_tw(float2* out, int R, bool last64, cudaStream_t st) {
  const int n = wide_tw_entries(R, last64);
  if (n == 0) return cudaSuccess;
  int na = 8, nb = 8;   // split of the last radix
  switch (last64 ? 64 : R / 64) {
#define CASE(RB) case RB: na = WideSplit<RB>::NA; nb = WideSplit<RB>::NB; break;
    POND_WIDE_RB(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
  k_make_wide_tw<<<(n + 255) / 256, 256, 0, st>>>(out, last64 ? R / 64 : 64, last64 ? 64 : R / 64, na, nb);
  return cudaGetLastError();
}

cudaError_t launch_tw2(float2* lo, float2* hi, int logn, int sign, cudaStream_t st) {
  const long long nhi = logn > TW2_LOG ? (1ll << (logn - TW2_LOG)) : 1;
  const long long n = std::max<long long>(TW2_LO, nhi);
  k_make_tw2<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(lo, hi, logn, sign);
  return cudaGetLastError();
}

cudaError_t launch_tw3(float2* out, int logn, int sign, cudaStream_t st) {
  k_make_tw3<<<3, 256, 0, st>>>(out, logn, sign);
  return cudaGetLastError();
}

cudaError_t launch_tables(ChirpAnchor* anc, long long nanc, int clog, double du, double half,
                          double f0, double alpha, int sgn, cudaStream_t st) {
  k_make_chirp_anchors<<<(unsigned)((nanc + 127) / 128), 128, 0, st>>>(anc, nanc, clog, du, half, f0, alpha, sgn);
  return cudaGetLastError();
}

// Fused schedule: F2f for R1 = 512..4096 with J = 64, Ic for R2 = 16..2048
// (the radix-16 form to 512, the 64-values-per-thread form from 512).
#define POND_FUSED_R1(X) X(512) X(1024) X(2048) X(4096)
#define POND_FUSED_R2(X) X(16) X(32) X(64) X(128) X(256) X(512)

bool fused_geometry(const Geom& g) {
  return g.logM - g.logR2 == 6 && g.logR1 >= 9 && g.logR1 <= 12 && g.logR2 >= 4 && g.logR2 <= 11;
}

namespace {
template <int R2>
size_t smem_inv_cols_det(int nl) {
  return ((size_t)stage_table_size(R2) + (size_t)nl * col_stride<R2>()) * sizeof(float2);
}
}  // namespace

cudaError_t launch_fwd_rows_inv(const Geom& g, const float2* in, float2* out, Tw2 tw2L,
                                const float2* wtw, const ChirpAnchor* anc, int clog, const float2* ctab,
                                cudaStream_t st, int nseg) {
  const RowTile rt = row_tile(g.logR1, g.logR2);
  const dim3 tiles((unsigned)nseg, (unsigned)(g.L / TILE));   // segments fastest
  switch (1 << g.logR1) {
#define CASE(R)                                                                                             \
  case R:                                                                                                   \
    if (ctab)                                                                                               \
      k_fwd_rows_w<R, ROW_TABLE><<<tiles, WIDE_NT, fwd_rows_smem_bytes<R>(rt), st>>>(in, out, rt, tw2L, wtw, anc, clog, ctab); \
    else                                                                                                    \
      k_fwd_rows_w<R, ROW_ANCHORS><<<tiles, WIDE_NT, fwd_rows_smem_bytes<R>(rt), st>>>(in, out, rt, tw2L, wtw, anc, clog, ctab); \
    break;
    POND_FUSED_R1(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// Ir with the anchor chirp over ntr trials (mc), or over the one trial anc1 (mc.anc null).
static cudaError_t launch_inv_rows_anchor(const Geom& g, const float2* in, float2* out, int ntr, Tw2 tw2L,
                                          MultiChirp mc, const ChirpAnchor* anc1, int clog1, cudaStream_t st) {
  const RowTile rt = row_tile(g.logR1, g.logR2);
  const unsigned tiles = (unsigned)(g.L / TILE);
  const dim3 grid((unsigned)ntr, tiles);
  switch (1 << g.logR1) {
#define CASE(R)                                                                                             \
  case R:                                                                                                   \
    k_inv_rows_anchor<R><<<grid, WIDE_NT, anchor_smem_bytes<R>(rt), st>>>(in, out, g.L, rt, tw2L, mc, anc1, \
                                                                          clog1);                           \
    break;
    POND_FUSED_R1(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_inv_rows_chirp(const Geom& g, const float2* in, float2* out, Tw2 tw2L, const unsigned* words,
                                  const ChirpAnchor* anc, int clog, cudaStream_t st) {
  if (words) {
    MultiChirp mc{};
    mc.words = words;
    return launch_inv_rows_chirp_multi(g, in, out, 1, tw2L, mc, false, st);
  }
  return launch_inv_rows_anchor(g, in, out, 1, tw2L, MultiChirp{}, anc, clog, st);
}

cudaError_t launch_inv_rows_chirp_multi(const Geom& g, const float2* in, float2* out, int ntr, Tw2 tw2L,
                                        MultiChirp mc, bool table, cudaStream_t st) {
  if (ntr < 1) return cudaErrorInvalidValue;
  if (!table && !mc.words) return launch_inv_rows_anchor(g, in, out, ntr, tw2L, mc, nullptr, 0, st);
  const RowTile rt = row_tile(g.logR1, g.logR2);
  const unsigned tiles = (unsigned)(g.L / TILE);
  if (!table) {
    // trials per CTA: four waves of three CTAs per SM, then as many trials as leave them
    const int tpc = std::max(1, std::min(ntr, (int)((long long)tiles * ntr / (12ll * std::max(1, g.sms)))));
    const dim3 grid((unsigned)((ntr + tpc - 1) / tpc), tiles);
    switch (1 << g.logR1) {
#define CASE(R)                                                                                             \
  case R:                                                                                                   \
    k_inv_rows_words<R><<<grid, WIDE_NT, anchor_smem_bytes<R>(rt), st>>>(in, out, g.L, rt, tw2L, mc.words,  \
                                                                         ntr, tpc);                         \
    break;
      POND_FUSED_R1(CASE)
#undef CASE
      default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
  }
  // table form: one CTA per row tile runs every trial
  switch (1 << g.logR1) {
#define CASE(R)                                                                                             \
  case R:                                                                                                   \
    k_inv_rows_table<R><<<tiles, TAB_GROUPS * WIDE_NT, table_smem_bytes<R>(rt), st>>>(in, out, g.L, rt,    \
                                                                                      tw2L, mc, ntr);       \
    break;
    POND_FUSED_R1(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

int fused_groups(const Geom& g) {
  const int nl = std::min(TILE >> g.logR2, g.nchan);
  return g.nchan / nl;
}

cudaError_t launch_inv_cols_det(const Geom& g, const float2* in, float* P, float* part, int* cnt, float2* vout,
                                long long vstride, long long vofs, const MSpan& span, const float2* tw,
                                const float2* wtw, cudaStream_t st, int nu) {
  const int R2 = 1 << g.logR2, R1 = 1 << g.logR1;
  const int nl = std::min(TILE / R2, g.nchan);
  const dim3 grid((unsigned)(R1 / nl), (unsigned)nu);
  const float scale = 1.0f / (float)(1u << g.logM);
  const int lognch = g.logR1 - (g.logM - g.logR2);
  // several trials or segments: each has its own L-element input, M-element P, partials and tickets
  const TrialStride ts = nu > 1 ? TrialStride{g.L, g.M, (long long)fused_groups(g) * g.M, FUSED_J}
                                 : TrialStride{0, 0, 0, 0};
  // 512-, 1024- and 2048-point columns that fill a tile (at least TILE / R2
  // sub-channels; always so from 1024 on) take the form with 64 values per
  // thread: per launch of 32 trials of the 2048-point column pass 755 -> 548 us,
  // of up to 21 trials of the 512-point one 30.7 -> 21.3 us.  Shorter columns
  // have no 64-point first stage to fill, and half tiles leave half the threads idle.
  if (R2 >= 512 && nl * R2 == TILE) {
    const int logG = lognch - (13 - g.logR2);
    switch (R2) {
#define CASE(R)                                                                                                  \
  case R:                                                                                                        \
    if (vout)                                                                                                    \
      k_inv_cols_det_w<R, true><<<grid, WIDE_NT, wide_smem_bytes<64, R / 64>(), st>>>(                          \
          in, P, part, cnt, vout, vstride, vofs, logG, g.logM - g.logR2, span, scale, wtw, ts);            \
    else                                                                                                         \
      k_inv_cols_det_w<R, false><<<grid, WIDE_NT, wide_smem_bytes<64, R / 64>(), st>>>(                         \
          in, P, part, cnt, vout, vstride, vofs, logG, g.logM - g.logR2, span, scale, wtw, ts);            \
    return cudaGetLastError();
      CASE(512) CASE(1024) CASE(2048)
#undef CASE
      default: break;
    }
  }
  switch (R2) {
#define CASE(R) case R: k_inv_cols_det<R><<<grid, NT, smem_inv_cols_det<R>(nl), st>>>(in, P, part, cnt, vout, vstride, vofs, g.logR1, lognch, g.logM - g.logR2, span, scale, tw, ts); break;
    POND_FUSED_R2(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t set_kernel_attributes() {
  cudaError_t e = set_attributes_t<false>();
  // The small kernels that run between and beside the passes take the passes' division of
  // L1 and shared memory: an SM changes it only when idle, and the CTAs of the next
  // kernel crowd on the SMs that could (after a carry copy at the default division
  // a segment's fold took 31.8 us instead of 8.1, four 64-bit-bound CTAs to an SM).  Not
  // the copy from host memory: its loads in flight need the L1 (end to end 1057 -> 1230 us), nor
  // the per-trial forms' decimation (24 trials at nfft 2^20: 2,132 us without, 2,230 with).
  auto shared_first = [&](auto* f) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  };
  shared_first(k_copy_bytes);
  shared_first(k_decimate_short_multi);
#define SET_F(R)                                                                                               \
  {                                                                                                            \
    const RowTile rt{0, 0, 0, row_stride_max(R), row_stride_max(R)};                                           \
    auto attr = [&](auto* f, size_t bytes) {                                                                   \
      if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes); \
    };                                                                                                         \
    attr(k_fwd_rows_w<R, ROW_SPECTRUM>, fwd_rows_smem_bytes<R>(rt));                                           \
    attr(k_fwd_rows_w<R, ROW_ANCHORS>, fwd_rows_smem_bytes<R>(rt));                                            \
    attr(k_fwd_rows_w<R, ROW_TABLE>, fwd_rows_smem_bytes<R>(rt));                                              \
    attr(k_inv_rows_words<R>, anchor_smem_bytes<R>(rt));                                                       \
    attr(k_inv_rows_anchor<R>, anchor_smem_bytes<R>(rt));                                                      \
    attr(k_inv_rows_table<R>, table_smem_bytes<R>(rt));                                                        \
  }
  POND_FUSED_R1(SET_F)
#undef SET_F
#define SET_C(R) \
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_inv_cols_det<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_inv_cols_det<R>(TILE / R));
  POND_FUSED_R2(SET_C)
#undef SET_C
#define SET_W(R)                                                                                                     \
  if (e == cudaSuccess)                                                                                              \
    e = cudaFuncSetAttribute(k_inv_cols_det_w<R, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,                \
                             wide_smem_bytes<64, R / 64>());                                                         \
  if (e == cudaSuccess)                                                                                              \
    e = cudaFuncSetAttribute(k_inv_cols_det_w<R, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,                 \
                             wide_smem_bytes<64, R / 64>());
  SET_W(512) SET_W(1024) SET_W(2048)
#undef SET_W
#define SET_I(R)                                                                                                     \
  if (e == cudaSuccess)                                                                                              \
    e = cudaFuncSetAttribute(k_inv_cols_w<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, wide_smem_bytes<64, R / 64>()); \
  if (e == cudaSuccess)                                                                                              \
    e = cudaFuncSetAttribute(k_inv_rows_w<R, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, inv_rows_w_smem<R>(0)); \
  if (e == cudaSuccess)                                                                                              \
    e = cudaFuncSetAttribute(k_inv_rows_w<R, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, inv_rows_w_smem<R>(0));
  SET_I(512) SET_I(1024) SET_I(2048) SET_I(4096)
#undef SET_I
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_fold_partial, cudaFuncAttributeMaxDynamicSharedMemorySize, fold_smem_bytes(MAX_NBINS));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_fold_dec<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, fold_smem_bytes(MAX_NBINS));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_fold_dec<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, fold_smem_bytes(MAX_NBINS));
  return e;
}

// The pass launchers pick the FP32 or the tensor-core instantiation.
cudaError_t launch_fwd_cols(const Geom& g, const SegSrc& in, float2* out, const float2* tw, cudaStream_t st, int nseg) {
  return g.tc_terms ? launch_fwd_cols_tc(g, in, out, tw, st, nseg) : launch_fwd_cols_t<false>(g, in, out, tw, st, nseg);
}

cudaError_t launch_fwd_rows(const Geom& g, const float2* in, float2* out, const float2* tw3L, Tw2 tw2L, const float2* tw,
                            const float2* wtw, cudaStream_t st, int nseg) {
  if (g.tc_terms) return launch_fwd_rows_tc(g, in, out, tw3L, tw2L, tw, st, nseg);
  const RowTile rt = row_tile(g.logR1, g.logR2);
  const dim3 tiles((unsigned)nseg, (unsigned)(g.L / TILE));   // segments fastest
  if (g.L >= TILE) {
    switch (1 << g.logR1) {
#define CASE(R)                                                                                             \
  case R:                                                                                                   \
    k_fwd_rows_w<R, ROW_SPECTRUM><<<tiles, WIDE_NT, fwd_rows_smem_bytes<R>(rt), st>>>(in, out, rt, tw2L, wtw, nullptr, 0, nullptr); \
    return cudaGetLastError();
      POND_FUSED_R1(CASE)
#undef CASE
      default: break;
    }
  }
  return launch_fwd_rows_t<false>(g, in, out, tw3L, tw2L, tw, st, nseg);
}

// Lines of 512 and more points take 64 values per thread (I1 with the chirp from a table;
// the anchors of batched trials stay with the radix-16 form, which stages them).
cudaError_t launch_inv_cols(const Geom& g, const float2* in, float2* out, const ChirpAnchor* anc,
                            int clog, const float2* ctab, const float2* tw, const float2* wtw, cudaStream_t st, int nseg) {
  if (g.tc_terms) return launch_inv_cols_tc(g, in, out, anc, clog, tw, st, nseg);
  if (ctab) {
    const dim3 grid((unsigned)nseg, (unsigned)(g.L / TILE));   // segments fastest
    switch (1 << g.logQ2) {
#define CASE(R)                                                                                                     \
  case R:                                                                                                           \
    k_inv_cols_w<R><<<grid, WIDE_NT, wide_smem_bytes<64, R / 64>(), st>>>(in, out, g.logQ1, g.logM, g.logR1, g.logR2, \
                                                                          ctab, wtw);                               \
    return cudaGetLastError();
      CASE(512) CASE(1024) CASE(2048) CASE(4096)
#undef CASE
      default: return cudaErrorInvalidValue;
    }
  }
  return launch_inv_cols_t<false>(g, in, out, anc, clog, tw, st, nseg);
}

// The table form reads runs of 2^(logQ2 - 6 - s) consecutive bins, s = logR2 - logQ1: from four
// on (a 32-byte sector) it wins (2^22 bins, runs of four: 44.0 us against 49.1 per segment),
// at two it does not (2^23 bins: 61.8 us against 45.4).
bool inv_cols_table(const Geom& g) {
  return g.L >= TILE && g.logQ2 >= 9 && g.logQ2 <= 12 && g.logQ2 - 6 - (g.logR2 - g.logQ1) >= 2;
}

cudaError_t launch_inv_rows(const Geom& g, const float2* buf, float* P, float2* vout, long long vstride,
                            long long vofs, const MSpan& span, const float2* tw3M, const float2* tw, const float2* wtw,
                            cudaStream_t st, int nseg) {
  if (g.tc_terms) return launch_inv_rows_tc(g, buf, P, vout, vstride, vofs, span, tw3M, tw, st, nseg);
  if (g.L >= TILE) {
    const dim3 grid((unsigned)(g.L / TILE), (unsigned)nseg);
    const int lognch = g.logL - g.logM;
    const float scale = 1.0f / (float)(1u << g.logM);
    switch (1 << g.logQ1) {
#define CASE(R)                                                                                                     \
  case R:                                                                                                           \
    if (vout)                                                                                                       \
      k_inv_rows_w<R, true><<<grid, WIDE_NT, inv_rows_w_smem<R>(lognch), st>>>(                                     \
          buf, P, vout, vstride, vofs, g.logQ2, g.logM, lognch, span, scale, tw3M, wtw);                            \
    else                                                                                                            \
      k_inv_rows_w<R, false><<<grid, WIDE_NT, inv_rows_w_smem<R>(lognch), st>>>(                                    \
          buf, P, vout, vstride, vofs, g.logQ2, g.logM, lognch, span, scale, tw3M, wtw);                            \
    return cudaGetLastError();
      CASE(512) CASE(1024) CASE(2048) CASE(4096)
#undef CASE
      default: break;
    }
  }
  return launch_inv_rows_t<false>(g, buf, P, vout, vstride, vofs, span, tw3M, tw, st, nseg);
}

size_t fold_smem_bytes(int nbins) {
  return (size_t)FOLD_WARPS * nbins * (sizeof(double) + sizeof(int)) + FOLD_WARPS * 32 * sizeof(float);
}

int fold_parts(long long n, long long* chunk) {
  long long c = std::max<long long>(1024, (n + MAX_FOLD_PARTS - 1) / MAX_FOLD_PARTS);
  c = (c + 127) / 128 * 128;
  *chunk = c;
  return (int)((n + c - 1) / c);
}

cudaError_t launch_fold(const float* P, long long n, long long g0, double inc, int nbins, double* psum,
                        int* phits, double* prof_sum, long long* prof_hits, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  long long chunk;
  const int parts = fold_parts(n, &chunk);
  k_fold_partial<<<parts, FOLD_WARPS * 32, fold_smem_bytes(nbins), st>>>(P, n, g0, inc, nbins, chunk, psum, phits);
  k_fold_merge<int, true, MERGE_WARPS><<<(nbins + 31) / 32, MERGE_WARPS * 32, 0, st>>>(psum, phits, parts, nbins, prof_sum,
                                                                          prof_hits);
  return cudaGetLastError();
}

// Segments per launch: 2^25 bins' worth (four segments of a 2^24-point plan, so
// that a pass runs many waves of CTAs), at most 16.
int fold_slots(const Geom& g) { return (int)std::max<long long>(1, std::min<long long>(16, (1ll << 25) / g.L)); }

// Fold CTAs per segment: one window per warp, more where the partial rows of all slots
// would exceed 1024.  Segments of 2^14 samples and less go by sample in CTAs of 1024:
// a launch of one segment would otherwise be one to four CTAs.
static long long fold_chunk_len(const Geom& g) {
  const long long most = std::max(1, std::min(MAX_FOLD_PARTS, 1024 / fold_slots(g)));
  const long long step = g.S_c <= 1 << 14 ? 1024 : (long long)FOLD_WARPS * FOLD_WIN;
  return ((g.S_c + most - 1) / most + step - 1) / step * step;
}
int fold_parts_seg(const Geom& g) { return (int)((g.S_c + fold_chunk_len(g) - 1) / fold_chunk_len(g)); }

cudaError_t launch_fold_dec(const Geom& g, const float* P, const FoldSegs& f, const FoldPhase& ph, int nbins, long long num,
                            long long den, float* T, int* C, long long ring, double* psum, long long* phits,
                            cudaStream_t st) {
  if (f.n_left <= 0) return cudaSuccess;
  const int slots = fold_slots(g), parts = fold_parts_seg(g);
  if (f.nseg > slots) return cudaErrorInvalidValue;
  const long long chunk = fold_chunk_len(g);
  const long long j_lo = (f.g0 * den) / num, nj = ((f.g0 + f.n_left - 1) * den) / num - j_lo + 1;
  const long long per = num >= 64 * den ? FOLD_WARPS : FOLD_WARPS * 32;
  const unsigned blocks = (unsigned)(parts * f.nseg + (nj + per - 1) / per);
  if (ph.nc > 0)
    k_fold_dec<true><<<blocks, FOLD_WARPS * 32, fold_smem_bytes(nbins), st>>>(P, f, ph, nbins, slots, parts, chunk, num, den,
                                                                            j_lo, nj, T, C, ring, psum, phits);
  else
    k_fold_dec<false><<<blocks, FOLD_WARPS * 32, fold_smem_bytes(nbins), st>>>(P, f, ph, nbins, slots, parts, chunk, num,
                                                                             den, j_lo, nj, T, C, ring, psum, phits);
  return cudaGetLastError();
}

cudaError_t launch_fold_snapshot(const double* psum, const long long* phits, int rows, int nbins, double* prof_sum,
                                 long long* prof_hits, cudaStream_t st) {
  k_fold_merge<long long, false, SNAP_WARPS><<<(nbins + 31) / 32, SNAP_WARPS * 32, 0, st>>>(psum, phits, rows, nbins,
                                                                                          prof_sum, prof_hits);
  return cudaGetLastError();
}

cudaError_t launch_decimate(const float* P, long long n, long long g0, long long num, long long den,
                            long long j_lo, long long nj, float* T, int* C, long long ring, cudaStream_t st) {
  if (n <= 0 || nj <= 0) return cudaSuccess;
  if (num < 64 * den) {   // fewer than 64 channel samples per series sample
    k_decimate_short<<<(unsigned)((nj + 255) / 256), 256, 0, st>>>(P, n, g0, num, den, j_lo, nj, T, C, ring);
  } else {
    const long long threads = nj * 32;
    k_decimate<<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(P, n, g0, num, den, j_lo, nj, T, C, ring);
  }
  return cudaGetLastError();
}

}  // namespace pond
