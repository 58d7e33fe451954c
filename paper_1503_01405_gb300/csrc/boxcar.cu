// Boxcar S/N single-pulse detector over the series of a batch of DM trials.
//
// The paper names automatic transient detection as future work (Sec. 5); this
// is the plain matched-filter search over the dedispersed series that the
// batched trials produce:
//   mu_d = median(T_d), sigma_d = 1.4826 median|T_d - mu_d| (exact order
//   statistics; an even count takes the FP64 mean of the two middle values),
//   S_w(d, t) = (sum_{i<w} T_d[t+i] - w mu_d) / (sigma_d sqrt(w)), w = 1..64
//   (powers of two), the sum accumulated in FP64 in index order,
//   s(d, t) = max_w S_w, w*(d, t) its smallest maximising width,
//   candidate: s >= threshold and no point within |dd| <= 2 trials and
//   |dt| <= w* samples has a larger s (an equal s wins when it comes earlier
//   in (trial, sample) order).
// Every floating-point step is one correctly rounded IEEE operation (explicit
// _rn intrinsics, no contraction), so the FP64 oracle reproduces each S value
// bit for bit and the integer decisions agree exactly.
//
// An SM retires two FP64 operations per clock, so S is evaluated in FP64 only
// where it can matter.  k_screen sums the boxcars in FP32 with a bound on the
// rounding, and a point whose every sum stays below the threshold by more than
// that bound can neither be a candidate nor suppress one (a suppressing point has
// the larger s).  The few points left are listed, evaluated exactly and compared
// among themselves (2^25 points: 12.5 ms when every point was evaluated in FP64).
// The median and the MAD are exact order statistics of a bracket around them that
// a sample of the row predicts and the row's counts confirm; a row where they do
// not falls back to a radix select (4.3 ms for 128 rows of 250,000 samples by
// radix select alone, one CTA per row).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <mutex>
#include <vector>

#include "../../include/pond.h"
#include "pond_internal.h"

namespace pond {

constexpr int NW = 7;                       // widths 1, 2, 4, ..., 64
constexpr int WMAX = 64;
constexpr int BOX_THREADS = 256;

__device__ __forceinline__ unsigned f32_key(float v) {
  const unsigned u = __float_as_uint(v);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float f32_unkey(unsigned k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// k-th smallest (0-based) of n keys produced by key(i), MSB-first radix select
// with 8-bit digits; all threads of the CTA call it and get the same result.
template <typename K, int BITS, typename F>
__device__ K radix_select(long long n, long long k, F key, unsigned* hist, K* sh_prefix, long long* sh_k) {
  K prefix = 0, mask = 0;
  for (int shift = BITS - 8; shift >= 0; shift -= 8) {
    for (int b = threadIdx.x; b < 256; b += blockDim.x) hist[b] = 0;
    __syncthreads();
    for (long long i = threadIdx.x; i < n; i += blockDim.x) {
      const K x = key(i);
      if ((x & mask) == prefix) atomicAdd(&hist[(unsigned)((x >> shift) & 0xff)], 1u);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      long long c = 0;
      int b = 0;
      for (; b < 255; ++b) {
        if (c + hist[b] > k) break;
        c += hist[b];
      }
      *sh_k = k - c;
      *sh_prefix = prefix | ((K)b << shift);
    }
    __syncthreads();
    k = *sh_k;
    prefix = *sh_prefix;
    mask |= (K)0xff << shift;
    __syncthreads();
  }
  return prefix;
}

// mu and mad of a row by radix selects over all of it.
__device__ void robust_by_radix(const float* __restrict__ T, long long n, unsigned* hist, unsigned long long* shp,
                                long long* shk, double* mu_out, double* mad_out) {
  auto k32 = [&](long long i) -> unsigned { return f32_key(T[i]); };
  unsigned* pu = reinterpret_cast<unsigned*>(shp);
  double mu;
  {
    const float a = f32_unkey(radix_select<unsigned, 32>(n, (n - 1) / 2, k32, hist, pu, shk));
    if (n % 2) {
      mu = (double)a;
    } else {
      const float b = f32_unkey(radix_select<unsigned, 32>(n, n / 2, k32, hist, pu, shk));
      mu = __dmul_rn(__dadd_rn((double)a, (double)b), 0.5);
    }
  }
  // |T - mu| >= 0: its FP64 bit pattern orders like the value
  auto k64 = [&](long long i) -> unsigned long long {
    return (unsigned long long)__double_as_longlong(fabs(__dsub_rn((double)T[i], mu)));
  };
  double mad;
  {
    const double a = __longlong_as_double((long long)radix_select<unsigned long long, 64>(n, (n - 1) / 2, k64, hist,
                                                                                        shp, shk));
    if (n % 2) {
      mad = a;
    } else {
      const double b = __longlong_as_double((long long)radix_select<unsigned long long, 64>(n, n / 2, k64, hist,
                                                                                          shp, shk));
      mad = __dmul_rn(__dadd_rn(a, b), 0.5);
    }
  }
  *mu_out = mu;
  *mad_out = mad;
}

// What a row's sample predicts and its counts: the median lies among keys [klo, khi],
// `below` of the row's keys are smaller; the samples at one MAD from the median lie in
// [a1, a2] or [b1, b2], `mid` of the row's lie between the two.
struct Bracket {
  unsigned klo, khi;
  float a1, a2, b1, b2;
  float r_lo, r_hi;          // predicted bounds of the MAD
  unsigned below, mid, nc, nd;
  int bad;                   // NaN seen
};

// FP32 screening constants of a row: mu = mh + ml, th[q] the least sum over 2^q
// samples (less mu each) that can reach the threshold, rounded down.
struct Screen {
  float mh, ml, th[NW];
  int on;                    // sigma > 0
};

// One CTA per row: bracket from SAMPLE values, SAMPLE_DEV ranks (five standard
// deviations of a sample rank) to either side.
constexpr int SAMPLE = 8192, SAMPLE_DEV = 226, SORT_THREADS = 1024;
__global__ void __launch_bounds__(SORT_THREADS) k_bracket(const float* __restrict__ series, long long n,
                                                        long long stride, Bracket* __restrict__ out) {
  __shared__ unsigned key[SAMPLE];
  __shared__ int s_lo, s_hi;
  const float* T = series + (size_t)blockIdx.x * stride;
  const int tid = threadIdx.x;
  constexpr int V = SAMPLE / SORT_THREADS;   // element tid + SORT_THREADS u in register u
  unsigned x[V];
#pragma unroll
  for (int u = 0; u < V; ++u) {
    // spread over the row, the place inside each stretch scattered
    const int i = tid + u * SORT_THREADS;
    const long long a = (long long)i * n / SAMPLE, w = ((long long)(i + 1) * n) / SAMPLE - a;
    x[u] = f32_key(__ldg(T + min(n - 1, a + (w > 1 ? (long long)((unsigned)i * 2654435761u % (unsigned)w) : 0))));
  }
  if (tid == 0) {
    s_lo = -1;
    s_hi = SORT_THREADS;
  }
  // bitonic sort: partners SORT_THREADS apart and more meet in registers, under 32 apart
  // by shuffles, the 30 steps between through shared memory
#pragma unroll 1
  for (int k = 2; k <= SAMPLE; k <<= 1) {
#pragma unroll 1
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= SORT_THREADS) {
        const int d = j / SORT_THREADS, kk = k / SORT_THREADS;
#pragma unroll
        for (int u = 0; u < V; ++u)
#pragma unroll
          for (int e = 1; e < V; e <<= 1)
            if (e == d && (u & e) == 0) {
              const unsigned lo = min(x[u], x[u | e]), hi = max(x[u], x[u | e]);
              const bool up = (u & kk) == 0;
              x[u] = up ? lo : hi;
              x[u | e] = up ? hi : lo;
            }
      } else {
        const bool low = (tid & j) == 0;
        unsigned y[V];
        if (j >= 32) {
          __syncthreads();
#pragma unroll
          for (int u = 0; u < V; ++u) key[tid + u * SORT_THREADS] = x[u];
          __syncthreads();
#pragma unroll
          for (int u = 0; u < V; ++u) y[u] = key[(tid ^ j) + u * SORT_THREADS];
        } else {
#pragma unroll
          for (int u = 0; u < V; ++u) y[u] = __shfl_xor_sync(0xffffffffu, x[u], j);
        }
#pragma unroll
        for (int u = 0; u < V; ++u) {
          const bool up = ((tid + u * SORT_THREADS) & k) == 0;
          x[u] = up == low ? min(x[u], y[u]) : max(x[u], y[u]);
        }
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < V; ++u) key[tid + u * SORT_THREADS] = x[u];
  __syncthreads();
  const float m = f32_unkey(key[SAMPLE / 2]);
  const float span = f32_unkey(key[SAMPLE / 4 * 3]) - f32_unkey(key[SAMPLE / 4]);   // about two MADs
  // radius of thread tid and the sample values within it
  const float r = span * ((float)tid / (float)(SORT_THREADS - 1));
  auto rank_of = [&](unsigned v) {   // sample keys < v
    int lo = 0, hi = SAMPLE;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (key[mid] < v) lo = mid + 1;
      else hi = mid;
    }
    return lo;
  };
  const int in = rank_of(f32_key(m + r)) - rank_of(f32_key(m - r));
  if (in <= SAMPLE / 2 - SAMPLE_DEV) atomicMax(&s_lo, tid);
  if (in >= SAMPLE / 2 + SAMPLE_DEV) atomicMin(&s_hi, tid);
  __syncthreads();
  if (tid == 0) {
    Bracket b{};
    b.klo = key[SAMPLE / 2 - SAMPLE_DEV];
    b.khi = key[SAMPLE / 2 + SAMPLE_DEV];
    const float step = span / (float)(SORT_THREADS - 1), lo = f32_unkey(b.klo), hi = f32_unkey(b.khi);
    b.r_lo = s_lo < 0 ? 0.f : step * (float)s_lo;
    b.r_hi = s_hi >= SORT_THREADS ? INFINITY : step * (float)s_hi;
    b.a1 = lo - b.r_hi;
    b.a2 = hi - b.r_lo;
    b.b1 = lo + b.r_lo;
    b.b2 = hi + b.r_hi;
    out[blockIdx.x] = b;
  }
}

// Counts each row against its bracket and collects the values inside: list C (median)
// and list D (one MAD out).  Grid (chunks of COLLECT values, rows).
constexpr int COLLECT_THREADS = 256, COLLECT_V = 32, COLLECT = COLLECT_THREADS * COLLECT_V;
__global__ void __launch_bounds__(COLLECT_THREADS) k_collect(const float* __restrict__ series, long long n,
                                                           long long stride, Bracket* __restrict__ br,
                                                           float* __restrict__ C, float* __restrict__ D,
                                                           unsigned ccap, unsigned dcap) {
  __shared__ unsigned part[4][COLLECT_THREADS / 32];
  __shared__ unsigned s_base[2];
  const int row = blockIdx.y, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const float* T = series + (size_t)row * stride;
  const Bracket b = br[row];
  const long long i0 = (long long)blockIdx.x * COLLECT;
  // value u of the thread: sample 4 (tid + COLLECT_THREADS (u / 4)) + u % 4 of the chunk
  const int left = (int)min(n - i0, (long long)COLLECT);
  float v[COLLECT_V];
  if (left == COLLECT && ((reinterpret_cast<uintptr_t>(T + i0)) & 15) == 0) {
#pragma unroll
    for (int u = 0; u < COLLECT_V; u += 4) {
      const float4 q = __ldg(reinterpret_cast<const float4*>(T + i0) + tid + COLLECT_THREADS * (u / 4));
      v[u] = q.x;
      v[u + 1] = q.y;
      v[u + 2] = q.z;
      v[u + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int u = 0; u < COLLECT_V; ++u) {
      const int i = 4 * (tid + COLLECT_THREADS * (u / 4)) + u % 4;
      v[u] = i < left ? __ldg(T + i0 + i) : 0.f;
    }
  }
  // [0] values of C, [1] of D, [2] keys below, [3] values between
  unsigned cnt[4] = {0, 0, 0, 0};
  bool nan = false;
  unsigned inc = 0, ind = 0;
#pragma unroll
  for (int u = 0; u < COLLECT_V; ++u) {
    const float x = v[u];
    const unsigned k = f32_key(x);
    const bool ok = 4 * (tid + COLLECT_THREADS * (u / 4)) + u % 4 < left;
    nan |= ok && x != x;
    if (ok) {
      if (k >= b.klo && k <= b.khi) inc |= 1u << u;
      if ((x >= b.a1 && x <= b.a2) || (x >= b.b1 && x <= b.b2)) ind |= 1u << u;
      cnt[2] += k < b.klo;
      cnt[3] += x > b.a2 && x < b.b1;
    }
  }
  cnt[0] = __popc(inc);
  cnt[1] = __popc(ind);
  unsigned before[2];   // values of this warp's earlier lanes
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    unsigned x = cnt[q];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    if (q < 2) before[q] = x - cnt[q];
    if (lane == 31) part[q][w] = x;
  }
  if (__any_sync(0xffffffffu, nan) && lane == 0) br[row].bad = 1;
  __syncthreads();
  if (tid < 4) {
    unsigned s = 0;
    for (int q = 0; q < COLLECT_THREADS / 32; ++q) {
      const unsigned x = part[tid][q];
      part[tid][q] = s;
      s += x;
    }
    if (tid == 0) s_base[0] = atomicAdd(&br[row].nc, s);
    if (tid == 1) s_base[1] = atomicAdd(&br[row].nd, s);
    if (tid == 2) atomicAdd(&br[row].below, s);
    if (tid == 3) atomicAdd(&br[row].mid, s);
  }
  __syncthreads();
  unsigned pc = s_base[0] + part[0][w] + before[0], pd = s_base[1] + part[1][w] + before[1];
#pragma unroll
  for (int u = 0; u < COLLECT_V; ++u) {
    if ((inc >> u) & 1u) {
      if (pc < ccap) C[(size_t)row * ccap + pc] = v[u];
      ++pc;
    }
    if ((ind >> u) & 1u) {
      if (pd < dcap) D[(size_t)row * dcap + pd] = v[u];
      ++pd;
    }
  }
}

// The values of list (m of them) with ranks k1 <= k2, exactly: bin(x) is a
// monotone map to [0, NB) up to `slack` bins; the values in the ranks' bins (widened by slack)
// are ranked by their exact keys.  False when they are too many.
constexpr int SEL_NB = 4096, SEL_CAND = 1024;
struct SelSmem {
  unsigned hist[SEL_NB];
  unsigned long long cand[SEL_CAND];
  unsigned warp[32];
  unsigned ncand, below;
  int b1, b2;
  unsigned long long out[2];
};
template <class Bin, class Key>
__device__ bool select_ranks(SelSmem& s, const float* __restrict__ list, unsigned m, long long k1, long long k2,
                             int slack, Bin bin, Key key) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;   // SORT_THREADS threads
  for (int i = tid; i < SEL_NB; i += SORT_THREADS) s.hist[i] = 0;
  if (tid == 0) {
    s.ncand = s.below = 0;
    s.b1 = s.b2 = -1;
  }
  __syncthreads();
  for (unsigned i = tid; i < m; i += SORT_THREADS) atomicAdd(&s.hist[bin(list[i])], 1u);
  __syncthreads();
  // exclusive prefix over the bins, four per thread
  constexpr int PER = SEL_NB / SORT_THREADS;
  unsigned c[PER], sum = 0;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    c[i] = s.hist[PER * tid + i];
    sum += c[i];
  }
  unsigned x = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) s.warp[w] = x;
  __syncthreads();
  if (tid < 32) {
    unsigned t = s.warp[tid];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, t, d);
      if (lane >= d) t += y;
    }
    s.warp[tid] = t;
  }
  __syncthreads();
  unsigned p = (w ? s.warp[w - 1] : 0u) + x - sum;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    if (k1 >= (long long)p && k1 < (long long)(p + c[i])) s.b1 = PER * tid + i;
    if (k2 >= (long long)p && k2 < (long long)(p + c[i])) s.b2 = PER * tid + i;
    s.hist[PER * tid + i] = p;
    p += c[i];
  }
  __syncthreads();
  if (s.b1 < 0 || s.b2 < 0) return false;
  const int lo = max(0, s.b1 - slack), hi = min(SEL_NB - 1, s.b2 + slack);
  const unsigned below = s.hist[lo];
  for (unsigned i = tid; i < m; i += SORT_THREADS) {
    const float v = list[i];
    const int b = bin(v);
    if (b >= lo && b <= hi) {
      const unsigned q = atomicAdd(&s.ncand, 1u);
      if (q < SEL_CAND) s.cand[q] = key(v);
    }
  }
  __syncthreads();
  if (s.ncand > SEL_CAND) return false;
  for (unsigned i = tid; i < s.ncand; i += SORT_THREADS) {
    const unsigned long long me = s.cand[i];
    unsigned rank = below;
    for (unsigned j = 0; j < s.ncand; ++j) {
      const unsigned long long o = s.cand[j];
      rank += o < me || (o == me && j < i);
    }
    if ((long long)rank == k1) s.out[0] = me;
    if ((long long)rank == k2) s.out[1] = me;
  }
  __syncthreads();
  return true;
}

// One CTA per row: mu and sigma from the lists where the counts confirm the bracket, else
// (or without brackets, br null) from the whole row; and the row's screening constants for
// threshold thr.
__global__ void __launch_bounds__(SORT_THREADS) k_robust_stats(const float* __restrict__ series, long long n,
                                                             long long stride, const Bracket* __restrict__ br,
                                                             const float* __restrict__ C, const float* __restrict__ D,
                                                             unsigned ccap, unsigned dcap, double thr,
                                                             double* __restrict__ mu_out, double* __restrict__ sig_out,
                                                             Screen* __restrict__ screen) {
  __shared__ SelSmem s;
  __shared__ unsigned long long shp;
  __shared__ long long shk;
  const int row = blockIdx.x;
  const Bracket b = br ? br[row] : Bracket{};
  const long long k1 = (n - 1) / 2, k2 = n / 2;
  double mu = 0.0, mad = 0.0;
  bool ok = br && !b.bad && b.nc <= ccap && b.nd <= dcap && k1 >= (long long)b.below && k2 - (long long)b.below < (long long)b.nc;
  if (ok) {
    const int shift = max(0, 32 - __clz(b.khi - b.klo) - 12);   // (khi - klo) >> shift < SEL_NB
    ok = select_ranks(s, C + (size_t)row * ccap, b.nc, k1 - b.below, k2 - b.below, 0,
                      [&](float x) { return (int)((f32_key(x) - b.klo) >> shift); },
                      [&](float x) { return (unsigned long long)f32_key(x); });
    if (ok) {
      const float lo = f32_unkey((unsigned)s.out[0]), hi = f32_unkey((unsigned)s.out[1]);
      mu = n % 2 ? (double)lo : __dmul_rn(__dadd_rn((double)lo, (double)hi), 0.5);
      __syncthreads();   // s.out read
      auto dist = [&](float x) { return fabs(__dsub_rn((double)x, mu)); };
      // distances in FP32 for the bins: two rounded differences, so to 2 ulps of themselves
      const float mh = (float)mu, ml = (float)(mu - (double)mh);
      const float w = f32_unkey(b.khi) - f32_unkey(b.klo);
      const float d0 = fmaxf(0.f, b.r_lo - w), width = (b.r_hi + w - d0) / (float)SEL_NB;
      const float err = 4.8e-7f * (b.r_hi + w + fabsf(ml));
      const float inv = 1.f / width;
      ok = b.mid <= k1 && width > 8.f * err && isfinite(inv) &&
           select_ranks(s, D + (size_t)row * dcap, b.nd, k1 - b.mid, k2 - b.mid, 1,
                        [&](float x) {
                          const float d = fabsf((x - mh) - ml);
                          return min(SEL_NB - 1, (int)fmaxf(0.f, (d - d0) * inv));
                        },
                        [&](float x) { return (unsigned long long)__double_as_longlong(dist(x)); });
      if (ok) {
        const double r1 = __longlong_as_double((long long)s.out[0]), r2 = __longlong_as_double((long long)s.out[1]);
        // every value between a2 and b1 is at most r1 away, every value outside [a1, b2] at least r2
        ok = (double)b.a2 <= mu && mu <= (double)b.b1 && dist(b.a2) <= r1 && dist(b.b1) <= r1 && dist(b.a1) >= r2 &&
             dist(b.b2) >= r2;
        mad = n % 2 ? r1 : __dmul_rn(__dadd_rn(r1, r2), 0.5);
      }
    }
  }
  __syncthreads();
  if (!ok) robust_by_radix(series + (size_t)row * stride, n, s.hist, &shp, &shk, &mu, &mad);
  if (threadIdx.x == 0) {
    const double sg = __dmul_rn(1.4826, mad);
    mu_out[row] = mu;
    sig_out[row] = sg;
    Screen z;
    z.mh = (float)mu;
    z.ml = (float)(mu - (double)z.mh);
    z.on = sg > 0;
    for (int q = 0; q < NW; ++q) {
      const double t = thr * sg * sqrt((double)(1 << q));
      z.th[q] = isinf(t) ? (float)t : (float)(t - fabs(t) * 2.4e-7);   // below t after rounding to FP32
    }
    screen[row] = z;
  }
}

// s and w* of one point, exactly (point t of a row of n samples).
__device__ __forceinline__ double boxcar_point(const float* T, long long left, double m, double sg, int* width) {
  double best = -INFINITY, acc = 0.0;
  int bw = 0, done = 0;
#pragma unroll
  for (int q = 0; q < NW; ++q) {
    const int w = 1 << q;
    if (w > left) break;
    for (int i = done; i < w; ++i) acc = __dadd_rn(acc, (double)T[i]);
    done = w;
    const double num = __dsub_rn(acc, __dmul_rn((double)w, m));
    const double s = __ddiv_rn(num, __dmul_rn(sg, __dsqrt_rn((double)w)));
    if (s > best) {
      best = s;
      bw = w;
    }
  }
  *width = bw;
  return best;
}

// FP32 screen of all points: bit i of word (row, t / 32) set when point t may reach
// the threshold; the set points of a word are listed from base[word] on.  A warp takes
// SCREEN_T points (and the 64 samples after them), 16 consecutive samples per lane, and doubles
// the boxcars by adding the neighbouring lanes' sums.  A sum of w samples is off
// by at most w maxabs 2^-20 (each sample less mu to 2 ulps, six additions).
constexpr int SCREEN_WARPS = 8, SCREEN_T = 448, SCREEN_W = SCREEN_T / 32;
template <bool VEC>
__global__ void __launch_bounds__(SCREEN_WARPS * 32) k_screen(const float* __restrict__ series, int ndm, long long n,
                                                            long long stride, const Screen* __restrict__ sc,
                                                            unsigned* __restrict__ bits, unsigned* __restrict__ base,
                                                            uint2* __restrict__ hot, unsigned hotcap,
                                                            unsigned long long* __restrict__ nhot) {
  const int lane = threadIdx.x & 31;
  const long long chunks = (n + SCREEN_T - 1) / SCREEN_T;
  const long long job = (long long)blockIdx.x * SCREEN_WARPS + (threadIdx.x >> 5);
  if (job >= chunks * ndm) return;
  const int row = (int)(job / chunks);
  const long long c = job - (long long)row * chunks, t0 = c * SCREEN_T;
  const float* T = series + (size_t)row * stride + t0;
  const Screen z = sc[row];
  const int left = (int)min(n - t0, 512ll);   // samples of the row from t0 on (512: all the warp sees)
  float a[16];
  if (VEC && left == 512) {
    const float4* p = reinterpret_cast<const float4*>(T) + lane * 4;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 v = __ldg(p + i);
      a[4 * i] = v.x;
      a[4 * i + 1] = v.y;
      a[4 * i + 2] = v.z;
      a[4 * i + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) a[i] = lane * 16 + i < left ? __ldg(T + lane * 16 + i) : z.mh;
  }
  float mx = 0.f;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    a[i] = (a[i] - z.mh) - z.ml;
    mx = fmaxf(mx, fabsf(a[i]));
  }
  bool odd = false;   // a value that is not finite: the bound says nothing
#pragma unroll
  for (int i = 0; i < 16; ++i) odd |= !(fabsf(a[i]) <= 3.4e38f);
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
  const bool any_odd = __any_sync(0xffffffffu, odd);
  // near the row's end a boxcar that does not fit is summed over what there is: that may
  // set a bit for nothing, never clear one.  The points are marked one by one only in
  // warps where some width's largest sum reaches its threshold.
  float a1[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) a1[i] = a[i];
  auto grow = [](float (&s)[16], int h) {   // s[i] += the sum that starts h samples on
    if (h < 16) {
      float nx[16];
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (i < h) nx[i] = __shfl_down_sync(0xffffffffu, s[i], 1);
#pragma unroll
      for (int i = 0; i < 16; ++i) s[i] += i + h < 16 ? s[i + h < 16 ? i + h : 0] : nx[(i + h) & 15];
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i) s[i] += __shfl_down_sync(0xffffffffu, s[i], h / 16);
    }
  };
  float th[NW];
  bool reach = any_odd || !(mx <= 1e36f);   // (sums that could overflow: mark by one)
#pragma unroll
  for (int q = 0; q < NW; ++q) {
    if (q > 0) grow(a, 1 << (q - 1));
    th[q] = z.th[q] - (float)(1 << q) * 9.5367432e-7f * mx;   // w maxabs 2^-20
    float m = a[0];
#pragma unroll
    for (int i = 1; i < 16; ++i) m = fmaxf(m, a[i]);
    reach |= !(m < th[q]);
  }
  unsigned mask = 0;
  if (__any_sync(0xffffffffu, reach)) {
#pragma unroll
    for (int q = 0; q < NW; ++q) {
      if (q > 0) grow(a1, 1 << (q - 1));
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (!(a1[i] < th[q])) mask |= 1u << i;
    }
  }
  if (any_odd) mask = 0xffffu;
  const int t_lane = lane * 16;
  if (!z.on || lane >= SCREEN_T / 16 || t_lane >= left) mask = 0;
  else if (left - t_lane < 16) mask &= (1u << (left - t_lane)) - 1u;
  const unsigned other = __shfl_down_sync(0xffffffffu, mask, 1);
  const unsigned word = (lane & 1) ? 0u : mask | (other << 16);
  const unsigned long long wi = (unsigned long long)job * SCREEN_W + (lane >> 1);
  const bool owner = !(lane & 1) && lane < SCREEN_T / 16;
  if (owner) bits[wi] = word;
  if (!__any_sync(0xffffffffu, word != 0)) return;
  const unsigned cnt = __popc(word);
  unsigned x = cnt;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  unsigned long long start = 0;
  if (lane == 31) start = atomicAdd(nhot, (unsigned long long)x);
  start = __shfl_sync(0xffffffffu, start, 31);
  unsigned long long pos = start + x - cnt;
  if (owner) base[wi] = (unsigned)min(pos, (unsigned long long)hotcap);
  for (unsigned m = word; m; m &= m - 1, ++pos)
    if (pos < hotcap) hot[pos] = make_uint2((unsigned)row, (unsigned)(t0 + t_lane + __ffs(m) - 1));
}

// The listed points' exact s and w*.
__global__ void __launch_bounds__(128) k_exact(const float* __restrict__ series, long long n, long long stride,
                                             const double* __restrict__ mu, const double* __restrict__ sig,
                                             const uint2* __restrict__ hot, unsigned hotcap,
                                             const unsigned long long* __restrict__ nhot, double* __restrict__ S,
                                             unsigned char* __restrict__ W) {
  if (*nhot > hotcap) return;   // the host takes the dense form
  const unsigned m = (unsigned)*nhot;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    const uint2 p = hot[i];
    int w;
    S[i] = boxcar_point(series + (size_t)p.x * stride + p.y, n - p.y, mu[p.x], sig[p.x], &w);
    W[i] = (unsigned char)w;
  }
}

__device__ __forceinline__ pond_cand make_cand(int d, long long t, int w, double s) {
  pond_cand c;
  c.trial = d;
  c.width = w;
  c.index = t;
  c.snr = s;
  c.dm = 0.0;
  c.score = -1.f;
  c.reserved = 0;
  return c;
}

// Candidates among the listed points: no larger s within |dd| <= radius and |dt| <= w*
// (points that are not listed lie below the threshold).
__global__ void __launch_bounds__(128) k_suppress_hot(const uint2* __restrict__ hot, unsigned hotcap,
                                                    const unsigned long long* __restrict__ nhot,
                                                    const double* __restrict__ S, const unsigned char* __restrict__ W,
                                                    const unsigned* __restrict__ bits,
                                                    const unsigned* __restrict__ base, int ndm, long long n, double thr,
                                                    int radius, pond_cand* __restrict__ out, long long cap,
                                                    unsigned long long* __restrict__ count) {
  if (*nhot > hotcap) return;
  const unsigned m = (unsigned)*nhot;
  const long long words = (n + SCREEN_T - 1) / SCREEN_T * SCREEN_W;   // per row
  // a warp per point: lanes over the (row, word) pairs of its neighbourhood
  const int lane = threadIdx.x & 31;
  for (unsigned i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < m; i += gridDim.x * blockDim.x >> 5) {
    const double s = S[i];
    if (!(s >= thr)) continue;
    const uint2 p = hot[i];
    const int d = (int)p.x, w = W[i];
    const long long t = p.y;
    const int d0 = max(0, d - radius), d1 = min(ndm - 1, d + radius);
    const long long a = max(0ll, t - w), b = min(n - 1, t + w), q0 = a / 32;
    const int per = (int)(b / 32 - q0) + 1, pairs = per * (d1 - d0 + 1);
    bool lost = false;
    for (int e = lane; e < pairs && !lost; e += 32) {
      const int dd = d0 + e / per;
      const long long q = q0 + e % per;
      const unsigned word = bits[(size_t)dd * words + q];
      unsigned in = word;
      if (q == q0) in &= 0xffffffffu << (a & 31);
      if (q == b / 32 && (b & 31) != 31) in &= (2u << (b & 31)) - 1u;
      if (!in) continue;
      const unsigned bs = base[(size_t)dd * words + q];
      for (; in && !lost; in &= in - 1) {
        const int bit = __ffs(in) - 1;
        const long long tt = q * 32 + bit;
        if (dd == d && tt == t) continue;
        const double o = S[bs + __popc(word & ((1u << bit) - 1u))];
        lost = o > s || (o == s && (dd < d || (dd == d && tt < t)));
      }
    }
    if (__any_sync(0xffffffffu, lost) || lane) continue;
    const unsigned long long k = atomicAdd(count, 1ull);
    if ((long long)k < cap) out[k] = make_cand(d, t, w, s);
  }
}

// s(d, t) and w*(d, t); grid (ceil(n / BOX_THREADS), ndm).
__global__ void __launch_bounds__(BOX_THREADS) k_boxcar(const float* __restrict__ series, long long n,
                                                       long long stride, const double* __restrict__ mu,
                                                       const double* __restrict__ sig, double* __restrict__ S,
                                                       unsigned char* __restrict__ W) {
  __shared__ float tile[BOX_THREADS + WMAX];
  const int d = blockIdx.y;
  const long long t0 = (long long)blockIdx.x * BOX_THREADS;
  const float* T = series + (size_t)d * stride;
  for (int i = threadIdx.x; i < BOX_THREADS + WMAX; i += BOX_THREADS)
    tile[i] = (t0 + i < n) ? T[t0 + i] : 0.f;
  __syncthreads();
  const long long t = t0 + threadIdx.x;
  if (t >= n) return;
  double best = -INFINITY;
  int bw = 0;
  if (sig[d] > 0) best = boxcar_point(tile + threadIdx.x, n - t, mu[d], sig[d], &bw);
  S[(size_t)d * n + t] = best;
  W[(size_t)d * n + t] = (unsigned char)bw;
}

// Candidates: local maxima of s over |dd| <= 2 trials and |dt| <= w* samples.
__global__ void k_suppress(const double* __restrict__ S, const unsigned char* __restrict__ W, int ndm, long long n,
                           double thr, int radius, pond_cand* __restrict__ out, long long cap,
                           unsigned long long* __restrict__ count) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)ndm * n) return;
  const double s = S[idx];
  if (!(s >= thr)) return;
  const int d = (int)(idx / n);
  const long long t = idx - (long long)d * n;
  const int w = W[idx];
  const int d0 = max(0, d - radius), d1 = min(ndm - 1, d + radius);
  const long long a = max(0ll, t - w), b = min(n - 1, t + w);
  for (int dd = d0; dd <= d1; ++dd)
    for (long long tt = a; tt <= b; ++tt) {
      if (dd == d && tt == t) continue;
      const double o = S[(size_t)dd * n + tt];
      const bool earlier = dd < d || (dd == d && tt < t);
      if (o > s || (o == s && earlier)) return;
    }
  const unsigned long long k = atomicAdd(count, 1ull);
  if ((long long)k < cap) out[k] = make_cand(d, t, w, s);
}

// Scratch of a call: stream-ordered allocations from a pool of the library's own per
// device, which keeps up to SCRATCH_KEPT bytes between calls and gives the rest back.  What
// it keeps the driver takes when another allocation of the process would fail (seen with
// cudaMalloc beyond the free memory).
constexpr unsigned long long SCRATCH_KEPT = 256ull << 20;
cudaError_t scratch_pool(cudaMemPool_t* out) {
  static std::mutex mu;
  static cudaMemPool_t pools[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (!pools[dev]) {
    cudaMemPoolProps pr{};
    pr.allocType = cudaMemAllocationTypePinned;
    pr.handleTypes = cudaMemHandleTypeNone;
    pr.location.type = cudaMemLocationTypeDevice;
    pr.location.id = dev;
    cudaMemPool_t p = nullptr;
    e = cudaMemPoolCreate(&p, &pr);
    if (e != cudaSuccess) return e;
    unsigned long long keep = SCRATCH_KEPT;
    e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e != cudaSuccess) {
      cudaMemPoolDestroy(p);
      return e;
    }
    pools[dev] = p;
  }
  *out = pools[dev];
  return cudaSuccess;
}

// One block of scratch cut into aligned pieces: sizes first, then pointers.
struct Scratch {
  unsigned char* p = nullptr;
  size_t bytes = 0;
  size_t cut(size_t n) {
    const size_t o = bytes;
    bytes += (n + 255) / 256 * 256;
    return o;
  }
  template <class T> T* at(size_t o) const { return reinterpret_cast<T*>(p + o); }
};

int boxcar_fail(cudaError_t e) {
  return set_error(e == cudaErrorMemoryAllocation ? POND_E_OOM : POND_E_CUDA, cudaGetErrorString(e));
}

// Copy the candidates to the caller, sorted by (trial, index).  v may hold the first of them.
int deliver(std::vector<pond_cand>& v, unsigned long long found, long long dcap, const pond_cand* dc, pond_cand* out,
            size_t cap, size_t* n_found, cudaStream_t st) {
  const size_t have = (size_t)std::min<unsigned long long>(v.size(), found);
  v.resize((size_t)std::min<unsigned long long>(found, (unsigned long long)dcap));
  if (v.size() > have) {
    cudaError_t e = cudaMemcpyAsync(v.data() + have, dc + have, (v.size() - have) * sizeof(pond_cand),
                                    cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return set_error(POND_E_CUDA, cudaGetErrorString(e));
  }
  *n_found = (size_t)found;
  if (found > (unsigned long long)dcap) return set_error(POND_E_OVERRUN, "boxcar: more candidates than capacity");
  std::sort(v.begin(), v.end(), [](const pond_cand& x, const pond_cand& y) {
    return x.trial != y.trial ? x.trial < y.trial : x.index < y.index;
  });
  if (v.size() > cap) return set_error(POND_E_OVERRUN, "boxcar: more candidates than capacity");
  std::copy(v.begin(), v.end(), out);
  return POND_OK;
}

// Every point in FP64: for thresholds that most points pass, and lists that overflow.  The
// caller's scratch is given back first (its rows' mu and sigma are kept), so a
// call never holds more than the larger of the two forms.
int run_dense(const float* d_series, int ndm, long long n, long long stride, double thr, Scratch* sc, const double* mu,
              const double* sig, pond_cand* host_out, size_t cap, size_t* n_found, cudaStream_t st) {
  const long long dcap = std::max<long long>(1024, (long long)cap);
  double *stats = nullptr, *S = nullptr;
  unsigned char* W = nullptr;
  pond_cand* dc = nullptr;
  unsigned long long* cnt = nullptr;
  cudaError_t e = cudaSuccess;
  auto take = [&](auto** p, size_t count) {
    if (e == cudaSuccess) e = cudaMalloc(p, count * sizeof(**p));
  };
  take(&stats, 2 * (size_t)ndm);
  if (e == cudaSuccess) e = cudaMemcpyAsync(stats, mu, ndm * sizeof(double), cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(stats + ndm, sig, ndm * sizeof(double), cudaMemcpyDeviceToDevice, st);
  cudaFreeAsync(sc->p, st);
  sc->p = nullptr;
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  take(&S, (size_t)ndm * n);
  take(&W, (size_t)ndm * n);
  take(&dc, (size_t)dcap);
  take(&cnt, 1);
  if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), st);
  unsigned long long found = 0;
  if (e == cudaSuccess) {
    const dim3 grid((unsigned)((n + BOX_THREADS - 1) / BOX_THREADS), (unsigned)ndm);
    k_boxcar<<<grid, BOX_THREADS, 0, st>>>(d_series, n, stride, stats, stats + ndm, S, W);
    const long long tot = (long long)ndm * n;
    k_suppress<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(S, W, ndm, n, thr, 2, dc, dcap, cnt);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&found, cnt, sizeof found, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  std::vector<pond_cand> v;
  const int rc = e == cudaSuccess ? deliver(v, found, dcap, dc, host_out, cap, n_found, st) : boxcar_fail(e);
  cudaFree(stats);
  cudaFree(S);
  cudaFree(W);
  cudaFree(dc);
  cudaFree(cnt);
  return rc;
}

int run_boxcar(const float* d_series, int ndm, long long n, long long stride, double thr, pond_cand* host_out,
               size_t cap, size_t* n_found, cudaStream_t st) {
  *n_found = 0;
  if (ndm <= 0 || n <= 0) return POND_OK;
  // At a threshold of 1 and more under half of a noise row's points reach the exact
  // evaluation; the list holds a sixteenth of all points, and a block where more reach it
  // takes the dense form.  (Points are listed with 32-bit sample indices.)
  bool sparse = thr >= 1.0 && n < (1ll << 31);
  const long long dcap = std::max<long long>(1024, (long long)cap), tot = (long long)ndm * n;
  const long long chunks = (n + SCREEN_T - 1) / SCREEN_T, jobs = chunks * ndm;
  unsigned ccap = (unsigned)std::min<long long>(n, n / 8 + 8192), dlist = (unsigned)std::min<long long>(n, n / 4 + 16384);
  const unsigned hotcap = (unsigned)std::min<long long>(1ll << 30, std::max<long long>(1 << 16, tot / 16));
  constexpr size_t FIRST = 512;   // candidates copied with the counters
  struct Head {
    unsigned long long nhot, found;
    pond_cand first[FIRST];
  };
  Scratch sc;
  size_t o_mu = 0, o_sig = 0, o_br = 0, o_scr = 0, o_C = 0, o_D = 0, o_head = 0, o_bits = 0, o_base = 0, o_hot = 0, o_S = 0,
         o_W = 0;
  auto lay_out = [&]() {
    sc.bytes = 0;
    o_mu = sc.cut(ndm * sizeof(double));
    o_sig = sc.cut(ndm * sizeof(double));
    o_br = sc.cut(ndm * sizeof(Bracket));
    o_scr = sc.cut(ndm * sizeof(Screen));
    o_C = sc.cut((size_t)ndm * ccap * sizeof(float));
    o_D = sc.cut((size_t)ndm * dlist * sizeof(float));
    if (!sparse) return;
    // counters, then the candidates
    o_head = sc.cut(offsetof(Head, first) + (size_t)std::max<long long>(dcap, FIRST) * sizeof(pond_cand));
    o_bits = sc.cut((size_t)jobs * SCREEN_W * sizeof(unsigned));
    o_base = sc.cut((size_t)jobs * SCREEN_W * sizeof(unsigned));
    o_hot = sc.cut((size_t)hotcap * sizeof(uint2));
    o_S = sc.cut((size_t)hotcap * sizeof(double));
    o_W = sc.cut(hotcap);
  };
  cudaMemPool_t pool = nullptr;
  cudaError_t e = scratch_pool(&pool);
  if (e != cudaSuccess) return boxcar_fail(e);
  lay_out();
  e = cudaMallocFromPoolAsync(reinterpret_cast<void**>(&sc.p), sc.bytes, pool, st);
  if (e == cudaErrorMemoryAllocation) {
    // no room for the lists: every row by radix selects, every point in FP64
    cudaGetLastError();
    sparse = false;
    ccap = dlist = 0;
    lay_out();
    e = cudaMallocFromPoolAsync(reinterpret_cast<void**>(&sc.p), sc.bytes, pool, st);
  }
  if (e != cudaSuccess) return boxcar_fail(e);
  double *mu = sc.at<double>(o_mu), *sig = sc.at<double>(o_sig);
  Bracket* br = sc.at<Bracket>(o_br);
  // A bracket sorts 8192 values whatever the row's length (50 us for the two rows of an SM), so many short
  // rows go by radix selects in small CTAs: 20,000 rows of 100 samples 2,060 us (6,520 with
  // brackets), 2,000 of 2,000 590 (750), 1,333 of 3,000 552 (511); 64 rows
  // of 1,000 142 (111).
  const bool radix = n <= 2048 && ndm > 304;
  if (radix) br = nullptr;
  else k_bracket<<<ndm, SORT_THREADS, 0, st>>>(d_series, n, stride, br);
  const dim3 cg((unsigned)((n + COLLECT - 1) / COLLECT), (unsigned)ndm);
  if (!radix)
    k_collect<<<cg, COLLECT_THREADS, 0, st>>>(d_series, n, stride, br, sc.at<float>(o_C), sc.at<float>(o_D), ccap, dlist);
  k_robust_stats<<<ndm, radix ? 256 : SORT_THREADS, 0, st>>>(d_series, n, stride, br, sc.at<float>(o_C), sc.at<float>(o_D), ccap,
                                               dlist, thr, mu, sig, sc.at<Screen>(o_scr));
  e = cudaGetLastError();
  int rc = POND_OK;
  bool dense = !sparse;
  if (e == cudaSuccess && sparse) {
    unsigned char* head = sc.at<unsigned char>(o_head);
    auto* nhot = reinterpret_cast<unsigned long long*>(head + offsetof(Head, nhot));
    auto* count = reinterpret_cast<unsigned long long*>(head + offsetof(Head, found));
    auto* dc = reinterpret_cast<pond_cand*>(head + offsetof(Head, first));
    unsigned *bits = sc.at<unsigned>(o_bits), *base = sc.at<unsigned>(o_base);
    uint2* hot = sc.at<uint2>(o_hot);
    e = cudaMemsetAsync(head, 0, offsetof(Head, first), st);
    const unsigned blocks = (unsigned)((jobs + SCREEN_WARPS - 1) / SCREEN_WARPS);
    const bool vec = (reinterpret_cast<uintptr_t>(d_series) & 15) == 0 && stride % 4 == 0;
    if (vec)
      k_screen<true><<<blocks, SCREEN_WARPS * 32, 0, st>>>(d_series, ndm, n, stride, sc.at<Screen>(o_scr), bits, base,
                                                           hot, hotcap, nhot);
    else
      k_screen<false><<<blocks, SCREEN_WARPS * 32, 0, st>>>(d_series, ndm, n, stride, sc.at<Screen>(o_scr), bits, base,
                                                            hot, hotcap, nhot);
    k_exact<<<304, 128, 0, st>>>(d_series, n, stride, mu, sig, hot, hotcap, nhot, sc.at<double>(o_S),
                                 sc.at<unsigned char>(o_W));
    k_suppress_hot<<<1216, 128, 0, st>>>(hot, hotcap, nhot, sc.at<double>(o_S), sc.at<unsigned char>(o_W), bits, base,
                                        ndm, n, thr, 2, dc, dcap, count);
    if (e == cudaSuccess) e = cudaGetLastError();
    Head h;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, head, sizeof h, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess) {
      dense = h.nhot > hotcap;
      if (!dense) {
        std::vector<pond_cand> v(h.first, h.first + std::min<unsigned long long>(h.found, FIRST));
        rc = deliver(v, h.found, dcap, dc, host_out, cap, n_found, st);
      }
    }
  }
  if (e == cudaSuccess && dense)
    rc = run_dense(d_series, ndm, n, stride, thr, &sc, mu, sig, host_out, cap, n_found, st);
  if (e != cudaSuccess) rc = boxcar_fail(e);
  if (sc.p) cudaFreeAsync(sc.p, st);
  return rc;
}

}  // namespace pond

extern "C" int pond_boxcar(const float* d_series, int32_t ndm, int64_t n, int64_t stride, double threshold,
                           pond_cand* out, size_t cap, size_t* n_found, void* cuda_stream) {
  if (!n_found || (cap > 0 && !out) || ndm < 0 || n < 0 || stride < n || (ndm > 0 && n > 0 && !d_series))
    return pond::set_error(POND_E_ARG, "pond_boxcar: bad argument");
  return pond::run_boxcar(d_series, ndm, n, stride, threshold, out, cap, n_found,
                          static_cast<cudaStream_t>(cuda_stream));
}
