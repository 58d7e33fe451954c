// Fold with a polynomial phase model into a pulse stack (PONDER Sec. 3.4: the
// fold uses the period predicted by TEMPO2; Sec. 4: a stack of single pulses,
// one row per rotation).
//
// phi(g) = sum_i c_i tau^i, tau = g dt - t_ref, by Horner's rule with every
// multiply and add rounded on its own (explicit _rn intrinsics, no contraction;
// the host evaluates the same expression with products kept unfused), so that
// rotation q = floor(phi) and bin b = min(floor((phi - q) nbins), nbins - 1)
// are decided exactly as a plain FP64 evaluation decides them.
//
// The key K(g) = q nbins + b never decreases along the series for a phase
// model that runs forwards, so the samples of
// one (rotation, bin) pair form one contiguous run.  k_stack_starts evaluates K
// where it changes, checks that it grows and writes the first sample of every key's run; one
// thread per stack cell (row, bin) then adds the samples of its rotations' runs in
// sample order in FP64, unless the check failed: no atomics, no partials to merge, and
// the sums are those of a sequential loop over the series.  The phase evaluations bound
// the kernels (an SM retires two FP64 operations per clock): with the check evaluating two keys per
// sample and every cell finding its runs by binary search on K, a 60 s series (976,562
// samples, 1024 bins) took 58 + 137 us, now 19 + 9; the call with its two read-backs
// of 0.7 MB 340 us, now about 175.  Where there are more than eight keys per
// sample (bins much finer than the sampling) the table of starts is not
// worth its size and the cells search, as they do without scratch.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <condition_variable>
#include <cstdio>
#include <mutex>
#include <string>

#include "../../include/pond.h"
#include "pond_internal.h"

namespace {

constexpr int MAX_COEF = 8;
constexpr int CELL_THREADS = 256;

struct PhaseModel {
  double c[MAX_COEF];
  int nc;
  double dt, t_ref;
  long long g0;
  int nbins;
};

struct Key {
  long long q;   // rotation
  int b;         // bin
};

__device__ __forceinline__ Key key_at(const PhaseModel& m, long long i) {
  const double tau = __dsub_rn(__dmul_rn((double)(m.g0 + i), m.dt), m.t_ref);
  double x = m.c[m.nc - 1];
  for (int k = m.nc - 2; k >= 0; --k) x = __dadd_rn(__dmul_rn(x, tau), m.c[k]);
  const double q = floor(x);
  const int b = (int)__dmul_rn(__dsub_rn(x, q), (double)m.nbins);
  return Key{(long long)q, b < m.nbins - 1 ? b : m.nbins - 1};
}

__device__ __forceinline__ long long key_value(const PhaseModel& m, long long i) {
  const Key k = key_at(m, i);
  return k.q * m.nbins + k.b;
}

// Lowest i in [lo, hi] with K(g0 + i) >= K (hi when there is none).
__device__ long long first_at_or_after(const PhaseModel& m, long long lo, long long hi, long long K) {
  while (lo < hi) {
    const long long mid = lo + ((hi - lo) >> 1);
    if (key_value(m, mid) >= K) hi = mid;
    else lo = mid + 1;
  }
  return lo;
}

// Flags of the calls in flight, one each: set when K decreases somewhere along that call's
// series.  Device memory of the module, so a call needs no allocation for its flag.
constexpr int FLAGS = 64;
__device__ int g_backwards[FLAGS];

__device__ __forceinline__ double phase_at(const PhaseModel& m, long long i) {
  const double tau = __dsub_rn(__dmul_rn((double)(m.g0 + i), m.dt), m.t_ref);
  double x = m.c[m.nc - 1];
  for (int k = m.nc - 2; k >= 0; --k) x = __dadd_rn(__dmul_rn(x, tau), m.c[k]);
  return x;
}

// start[K - K0] = first sample i with key >= K, for K0 <= K <= K0 + nk.  A warp takes
// windows of 32 run samples.  Where the phase is known to run forwards over a window a
// lane takes run consecutive samples: the keys at its first sample and at the next
// lane's tell which keys begin in between, and each one's first sample is predicted from
// the phases at the ends and corrected with exact keys (two evaluations per key).
// Elsewhere every sample's key is evaluated and compared with the one before.  A run of 32 needs
// the fewest evaluations; a short series takes shorter ones, whose keys follow one another on
// fewer steps, until RUN_LANES lanes share it (a call over 20,000 samples, 1.5 keys a
// sample: 47 us, 108 at 32; 80,000 samples: 56 and 108; 65,536 lanes 62, 4,096 71).
constexpr int MAX_RUN = 32;
constexpr long long RUN_LANES = 16384;
int run_length(long long n) {
  int run = MAX_RUN;
  while (run > 1 && n / run < RUN_LANES) run /= 2;
  return run;
}
__global__ void __launch_bounds__(128) k_stack_starts(PhaseModel m, long long n, long long K0, long long nk,
                                                    unsigned* __restrict__ start, int* __restrict__ backwards, int run) {
  const int window = 32 * run;
  const int lane = threadIdx.x & 31;
  const long long warps = gridDim.x * 4ll;
  auto put = [&](long long lo, long long hi, long long i) {   // keys lo .. hi start at sample i
    for (long long q = max(lo, K0); q <= min(hi, K0 + nk); ++q) start[q - K0] = (unsigned)i;
  };
  for (long long base = (blockIdx.x * 4ll + (threadIdx.x >> 5)) * window; base < n; base += warps * window) {
    const long long end = min(n, base + window);   // the window and the step to the next one
    if (base == 0 && lane == 0) put(K0, key_value(m, 0), 0);
    if (end == n && lane == 0) put(key_value(m, n - 1) + 1, K0 + nk, n);
    const long long last = min(end, n - 1);
    if (pond::phase_forwards(m.c, m.nc, m.dt, m.t_ref, m.g0 + base, m.g0 + last)) {
      const long long a = base + lane * run, e = min(last, a + run);
      if (a >= e) continue;
      const double xa = phase_at(m, a), xe = phase_at(m, e);
      const long long ka = key_value(m, a), ke = key_value(m, e);
      const float per = (float)(e - a) / (float)(xe - xa);
      for (long long k = ka + 1; k <= ke;) {
        // the first sample at or after the start of bin k
        const double lead = (double)k / (double)m.nbins - xa;
        long long i = a + max(1ll, min((long long)ceilf((float)lead * per), e - a));
        long long ki = key_value(m, i);
        while (ki < k) ki = key_value(m, ++i);            // ends: key(e) = ke >= k
        for (long long kp; i - 1 > a && (kp = key_value(m, i - 1)) >= k;) {
          ki = kp;
          --i;
        }
        put(k, ki, i);
        k = ki + 1;
      }
    } else {
      // steps i -> i + 1 of samples base .. last, each key against the next
      for (long long i0 = base; i0 < last; i0 += 31) {
        const long long i = min(i0 + lane, last);
        const long long k = key_value(m, i);
        const long long prev = __shfl_up_sync(0xffffffffu, k, 1);
        if (lane > 0 && i0 + lane <= last) {
          if (k < prev) *backwards = 1;
          put(prev + 1, k, i);
        }
      }
    }
  }
}

// Cell (row, b) from the table of starts (rows as in k_stack_cells); nothing when the model
// runs backwards (the table then has entries that no sample wrote).
__global__ void __launch_bounds__(CELL_THREADS) k_stack_sums(const float* __restrict__ y, long long n, PhaseModel m,
                                                             int mode, long long n_sub, long long q_first,
                                                             long long rows, const unsigned* __restrict__ start,
                                                             const int* __restrict__ backwards,
                                                             double* __restrict__ S, long long* __restrict__ H) {
  if (*backwards) return;
  const long long cell = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (cell >= rows * m.nbins) return;
  const long long row = cell / m.nbins;
  const int b = (int)(cell - row * m.nbins);
  long long lo = 0, hi = n, qa = row, qb = row;   // rotations from q_first
  if (mode != POND_STACK_ROTATION) {
    lo = row * n_sub;
    hi = min(n, lo + n_sub);
    qa = key_at(m, lo).q - q_first;
    qb = key_at(m, hi - 1).q - q_first;
  }
  double s = 0.0;
  long long h = 0;
  for (long long q = qa; q <= qb; ++q) {
    const unsigned* p = start + q * m.nbins + b;
    const long long a = max(lo, (long long)p[0]), e = min(hi, (long long)p[1]);
    long long i = a;
    for (; i + 4 <= e; i += 4) {   // four loads in flight, added in order
      const float v0 = __ldg(y + i), v1 = __ldg(y + i + 1), v2 = __ldg(y + i + 2), v3 = __ldg(y + i + 3);
      s = __dadd_rn(__dadd_rn(__dadd_rn(__dadd_rn(s, (double)v0), (double)v1), (double)v2), (double)v3);
    }
    for (; i < e; ++i) s = __dadd_rn(s, (double)__ldg(y + i));
    if (e > a) h += e - a;
  }
  S[cell] = s;
  H[cell] = h;
}

__global__ void k_stack_check(PhaseModel m, long long n, int* __restrict__ backwards) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i + 1 < n;
       i += (long long)gridDim.x * blockDim.x)
    if (key_value(m, i + 1) < key_value(m, i)) *backwards = 1;
}

// Cell (row, b): ROTATION rows are rotations q_first + row; SUBINT rows are the
// samples [row n_sub, min(n, (row + 1) n_sub)) with every rotation they touch.
__global__ void __launch_bounds__(CELL_THREADS) k_stack_cells(const float* __restrict__ y, long long n, PhaseModel m,
                                                              int mode, long long n_sub, long long q_first,
                                                              long long rows, double* __restrict__ S,
                                                              long long* __restrict__ H) {
  const long long cell = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (cell >= rows * m.nbins) return;
  const long long row = cell / m.nbins;
  const int b = (int)(cell - row * m.nbins);
  long long lo = 0, hi = n, qa, qb;
  if (mode == POND_STACK_ROTATION) {
    qa = qb = q_first + row;
  } else {
    lo = row * n_sub;
    hi = min(n, lo + n_sub);
    qa = key_at(m, lo).q;
    qb = key_at(m, hi - 1).q;
  }
  double s = 0.0;
  long long h = 0;
  for (long long q = qa; q <= qb; ++q) {
    const long long K = q * m.nbins + b;
    const long long a = first_at_or_after(m, lo, hi, K);
    const long long e = first_at_or_after(m, a, hi, K + 1);
    for (long long i = a; i < e; ++i) s = __dadd_rn(s, (double)__ldg(y + i));
    if (e > a) h += e - a;
  }
  S[cell] = s;
  H[cell] = h;
}

double rounded(double x) {
  volatile double v = x;
  return v;
}

// The host's evaluation of the same rotation, for the row count.
long long host_rotation(const PhaseModel& m, long long i) {
  const double tau = rounded((double)(m.g0 + i) * m.dt) - m.t_ref;
  double x = m.c[m.nc - 1];
  for (int k = m.nc - 2; k >= 0; --k) x = rounded(x * tau) + m.c[k];
  return (long long)std::floor(x);
}

int stack_args(int64_t n, int64_t g0, double dt_s, const double* coef, int32_t ncoef, double t_ref_s, int32_t nbins,
               int32_t mode, int64_t n_sub, PhaseModel* m, int64_t* rows, int64_t* first_rotation) {
  if (!rows || !first_rotation || (!coef && ncoef > 0))
    return pond::set_error(POND_E_ARG, "pond_fold_stack: null pointer");
  if (n < 0 || g0 < 0 || !(dt_s > 0) || !std::isfinite(dt_s) || !std::isfinite(t_ref_s) || ncoef < 1 ||
      ncoef > MAX_COEF || nbins < 1 || nbins > pond::MAX_NBINS ||
      !(mode == POND_STACK_ROTATION || (mode == POND_STACK_SUBINT && n_sub >= 1)))
    return pond::set_error(POND_E_ARG,
                           "pond_fold_stack: need n, g0 >= 0, dt > 0, 1..8 coefficients, nbins 1..4096, "
                           "mode ROTATION or SUBINT with n_sub >= 1");
  for (int k = 0; k < ncoef; ++k)
    if (!std::isfinite(coef[k])) return pond::set_error(POND_E_ARG, "pond_fold_stack: coefficient not finite");
  *m = PhaseModel{};
  for (int k = 0; k < ncoef; ++k) m->c[k] = coef[k];
  m->nc = ncoef;
  m->dt = dt_s;
  m->t_ref = t_ref_s;
  m->g0 = g0;
  m->nbins = nbins;
  if (n == 0) {
    *rows = 0;
    *first_rotation = 0;
    return POND_OK;
  }
  const long long q0 = host_rotation(*m, 0);
  *first_rotation = q0;
  *rows = mode == POND_STACK_ROTATION ? std::max(0ll, host_rotation(*m, n - 1) - q0 + 1) : (n + n_sub - 1) / n_sub;
  return POND_OK;
}

// A call's own flag, from before its first launch to after it has waited for its stream;
// waits for another call to end when all are taken.
class Flag {
 public:
  Flag() {
    std::unique_lock<std::mutex> lock(mu());
    freed().wait(lock, [] { return taken() != ~0ull; });
    while ((taken() >> i_) & 1) ++i_;
    taken() |= 1ull << i_;
  }
  ~Flag() {
    {
      std::lock_guard<std::mutex> lock(mu());
      taken() &= ~(1ull << i_);
    }
    freed().notify_one();
  }
  Flag(const Flag&) = delete;
  Flag& operator=(const Flag&) = delete;
  cudaError_t address(int** out) const {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_backwards);
    *out = static_cast<int*>(p) + i_;
    return e;
  }

 private:
  static std::mutex& mu() {
    static std::mutex m;
    return m;
  }
  static std::condition_variable& freed() {
    static std::condition_variable c;
    return c;
  }
  static unsigned long long& taken() {
    static unsigned long long t = 0;
    return t;
  }
  static_assert(FLAGS == 64, "one bit per flag");
  int i_ = 0;
};

}  // namespace

extern "C" int pond_stack_rows(int64_t n, int64_t g0, double dt_s, const double* coef, int32_t ncoef, double t_ref_s,
                               int32_t nbins, int32_t mode, int64_t n_sub, int64_t* rows, int64_t* first_rotation) {
  PhaseModel m;
  return stack_args(n, g0, dt_s, coef, ncoef, t_ref_s, nbins, mode, n_sub, &m, rows, first_rotation);
}

extern "C" int pond_fold_stack(const float* d_series, int64_t n, int64_t g0, double dt_s, const double* coef,
                               int32_t ncoef, double t_ref_s, int32_t nbins, int32_t mode, int64_t n_sub,
                               double* d_sum, int64_t* d_hits, int64_t rows_cap, int64_t* rows,
                               int64_t* first_rotation, void* cuda_stream) {
  PhaseModel m;
  int rc = stack_args(n, g0, dt_s, coef, ncoef, t_ref_s, nbins, mode, n_sub, &m, rows, first_rotation);
  if (rc) return rc;
  if (*rows > rows_cap) {
    char msg[160];
    snprintf(msg, sizeof msg, "pond_fold_stack: %lld rows needed, room for %lld", (long long)*rows,
             (long long)rows_cap);
    return pond::set_error(POND_E_OVERRUN, msg);
  }
  if (n == 0) return POND_OK;
  if (!d_series || !d_sum || !d_hits) return pond::set_error(POND_E_ARG, "pond_fold_stack: null device pointer");
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  auto failed = [](cudaError_t e) {
    return pond::set_error(e == cudaErrorMemoryAllocation ? POND_E_OOM : POND_E_CUDA,
                           (std::string("pond_fold_stack: ") + cudaGetErrorString(e)).c_str());
  };
  const char* backwards = "pond_fold_stack: the phase model runs backwards over the series";
  const long long cells = *rows * (long long)nbins, q_last = host_rotation(m, n - 1);
  const unsigned cell_blocks = (unsigned)((cells + CELL_THREADS - 1) / CELL_THREADS);
  const Flag own;
  int *flag = nullptr, back = 0;
  cudaError_t e = own.address(&flag);
  if (e == cudaSuccess) e = cudaMemsetAsync(flag, 0, sizeof(int), st);
  if (e != cudaSuccess) return failed(e);
  // the table holds a start per key (4 bytes of scratch): used while there are at most eight keys
  // per sample and the scratch can be had; the cells search without one
  const double keys = ((double)q_last - (double)*first_rotation + 1.0) * nbins;
  const unsigned blocks = (unsigned)std::min<long long>((n + 255) / 256, 4096);
  unsigned* start = nullptr;
  long long nk = 0;
  if (q_last >= *first_rotation && keys <= 8.0 * (double)n + 65536.0 && n < (1ll << 32)) {
    nk = (q_last - *first_rotation + 1) * nbins;
    cudaMemPool_t pool = nullptr;
    e = pond::scratch_pool(&pool);
    if (e == cudaSuccess)
      e = cudaMallocFromPoolAsync(reinterpret_cast<void**>(&start), (size_t)(nk + 1) * sizeof(unsigned), pool, st);
    if (e == cudaErrorMemoryAllocation) {
      cudaGetLastError();
      start = nullptr;
    } else if (e != cudaSuccess) {
      return failed(e);
    }
  }
  if (start) {
    const long long K0 = *first_rotation * (long long)nbins;
    const int run = run_length(n);
    const long long cta = 4 * 32 * run;
    k_stack_starts<<<(unsigned)std::min<long long>((n + cta - 1) / cta, 4096), 128, 0, st>>>(m, n, K0, nk, start, flag, run);
    if (cells > 0)
      k_stack_sums<<<cell_blocks, CELL_THREADS, 0, st>>>(d_series, n, m, mode, n_sub, *first_rotation, *rows, start,
                                                         flag, d_sum, reinterpret_cast<long long*>(d_hits));
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&back, flag, sizeof(int), cudaMemcpyDeviceToHost, st);
    cudaFreeAsync(start, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return failed(e);
    return back ? pond::set_error(POND_E_ARG, backwards) : POND_OK;
  }
  k_stack_check<<<blocks, 256, 0, st>>>(m, n, flag);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(&back, flag, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return failed(e);
  if (back) return pond::set_error(POND_E_ARG, backwards);
  if (cells > 0) {
    k_stack_cells<<<cell_blocks, CELL_THREADS, 0, st>>>(d_series, n, m, mode, n_sub, *first_rotation, *rows, d_sum,
                                                        reinterpret_cast<long long*>(d_hits));
    e = cudaGetLastError();
    if (e != cudaSuccess) return failed(e);
  }
  return POND_OK;
}
