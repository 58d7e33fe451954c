// Internal types shared by the kernels and the C-ABI layer.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "../../include/pond.h"

namespace pond {

constexpr int CHIRP_LOG_MAX = 15;            // at most 2^15 bins per chirp anchor
constexpr int MAX_NBINS = 4096;              // fold bins (per-warp FP64 histograms in smem)
constexpr int MAX_FOLD_PARTS = 304;          // CTAs of launch_fold (2 per SM)

// Taylor coefficients of the dedispersion phase phi (cycles) about an anchor
// bin: phi(k_a + d) = phi0 + phi1 d + phi2 d^2 + phi3 d^3.  The first three
// terms are evaluated exactly mod 1 in 64-bit fixed point (d is an integer),
// so only the small cubic term is rounded in FP32.
struct __align__(16) ChirpAnchor {
  unsigned long long p1;   // phi1 mod 1, Q0.64
  unsigned long long p2;   // phi2 mod 1, Q0.64
  unsigned p0;             // phi0 mod 1, Q0.32
  float p3;                // phi3
  unsigned pad[2];
};

// Chirps of the trials of one batched launch.  Table form (the lane's DMs are
// whole multiples n_d of one step dDM): atab[k] = frac(sgn dDM c(f_k)) in Q0.32,
// built once per lane in FP64, and trial d's phase at bin k is n_d atab[k]
// mod 2^32, an exact integer product (its error is n_d times the table's
// rounding, below 2^-33 cycles per step).  Anchor form: each trial's own
// anchor table (chirp_from).
struct MultiChirp {
  const unsigned* atab;            // table form: [L], bin k2 + R2 k1 at k2 R1 + k1
  const unsigned* nmul;            // table form: per trial of the launch, n_d
  const unsigned* words;           // anchor form: [trial][L] phase words (launch_chirp_words), or null
  const ChirpAnchor* const* anc;   // anchor form: per trial of the launch
  const int* clog;                 // anchor form: per trial of the launch
};

// Two-level twiddle table for exponents e < n: w^e = hi[e >> 12] * lo[e & 4095].
constexpr int TW2_LOG = 12;
constexpr int TW2_LO = 1 << TW2_LOG;
struct Tw2 {
  const float2* lo;
  const float2* hi;
};

// A segment's int8 input as up to two runs: samples [0, a_len) from a,
// [a_len, a_len + b_len) from b, zeros beyond.
// One segment's input: bytes [0, a_len) of run a, then [0, b_len) of run b, then
// zeros.  Real sample m is byte m (ch = 1) or the sum of bytes 2m, 2m + 1 (ch = 2:
// the two halves' interleaved int8 samples, added in phase); a_len is a whole
// number of samples.
struct SegIn {
  const int8_t* a;
  long long a_len;
  const int8_t* b;
  long long b_len;
  int vec8;   // ch 1, both runs 8-byte aligned with a_len % 8 == 0: F1 may load 8 bytes at a time
  int ch = 1;
  int pair4 = 0;  // ch 2, both runs 4-byte aligned with a_len, b_len % 4 == 0: F1 may load
                  // one complex sample's two N / S pairs (4 bytes) at a time
  int pair2 = 0;  // ch 1, both runs 2-byte aligned with even lengths: one complex sample (2 bytes) at a time
};

// The input of consecutive segments, one per blockIdx.x or .y of a launch.  Byte r of
// the stream, counted from the first new byte: carry_end[r] for r < 0, d[r] for
// 0 <= r < avail, zero beyond.  Segment y starts at byte r0 + y step and spans
// `bytes` bytes; F1 forms its two runs and alignment flags from these.
struct SegSrc {
  const int8_t* carry_end;
  const int8_t* d;
  long long avail, r0, step, bytes;
  int ch;
};

// Emitted span of segment y of a launch: m_lo <= m < min(m_hi, m_end - y m_step).
// Batched launches (blockIdx.y = trial) have m_step = 0.
struct MSpan {
  int m_lo, m_hi;
  long long m_end, m_step;
#ifdef __CUDACC__
  __device__ __forceinline__ int hi(unsigned y) const {
    const long long e = m_end - (long long)y * m_step;
    return e < m_hi ? (int)e : m_hi;
  }
#endif
};

constexpr int TC_W_BYTES = 3 * 32 * 32 * 2;   // W16 hi, mid, lo parts of one direction

// Tensor-core stage arguments: the W16 parts of one transform direction
// (hi, mid, lo BF16 in the operand layout, 6 KiB), the product terms (3 or 5)
// and the plan's error flag (set when a bounded MMA wait expires).
struct TcArgs {
  const uint4* w;
  int terms;
  int* err;
};

// Geometry of a plan: segment and pass decomposition.
struct Geom {
  long long N, L, M;     // real samples per segment, spectrum bins kept, samples per sub-channel
  int nchan;
  int logL, logM;
  int logR1, logR2;      // forward: L = R1 * R2 (F2 rows of R1, F1 columns of R2)
  int logQ1, logQ2;      // inverse: M = Q1 * Q2 (I2 rows of Q1, I1 columns of Q2)
  long long n_past, n_fut, S_c, S;
  int sms;               // streaming multiprocessors of the device
  int tc_terms = 0;      // 0: FP32 stages; 3 or 5: split-BF16 tensor-core radix-16 stages
  TcArgs tc_fwd{}, tc_inv{};
};

cudaError_t set_kernel_attributes();
// Largest batch a classifier accepts (its scratch size).
int cnn_max_batch(pond_cnn_t net);
cudaError_t set_kernel_attributes_tc();
// One CTA waiting on a barrier nothing arrives on (bounded by limit_ns); status 1 = gave up.
cudaError_t launch_wait_probe(unsigned long long limit_ns, int* status, unsigned long long* waited);
// W16 parts for the tensor-core stages, host-built: [fwd, inv][hi, mid, lo] in
// the K-major operand layout (2 x 6 KiB).
void build_w16_parts(uint16_t* out);
// The library's own stream-ordered memory pool of the current device (scratch of the
// entry points without a handle): it keeps a bounded amount between calls.
cudaError_t scratch_pool(cudaMemPool_t* out);
int run_boxcar(const float* d_series, int ndm, long long n, long long stride, double thr, pond_cand* host_out,
               size_t cap, size_t* n_found, cudaStream_t st);
// Record msg as the calling thread's last error (pond_last_error) and return code.
int set_error(int code, const char* msg);
cudaError_t launch_tables(ChirpAnchor* anc, long long nanc, int clog, double du, double half,
                          double f0, double alpha, int sgn, cudaStream_t st);
cudaError_t launch_tw2(float2* lo, float2* hi, int logn, int sign, cudaStream_t st);
// Three-level table (768 entries) of w^e, w = exp(sign 2 pi i / 2^logn), e < 2^24.
cudaError_t launch_tw3(float2* out, int logn, int sign, cudaStream_t st);
cudaError_t launch_stage_tw(float2* out, int R, cudaStream_t st);
int stage_tw_entries(int R);
// Stage-2 twiddles of the 64-values-per-thread FFT of length R (512 .. 4096; none
// otherwise), radices (64, R / 64) or, last64, (R / 64, 64).
cudaError_t launch_wide_tw(float2* out, int R, bool last64, cudaStream_t st);
int wide_tw_entries(int R, bool last64);
// Passes over nseg consecutive segments per launch: segment y reads
// and writes its own L elements of the buffers (M of P).  ctab (I1) non-null: the chirp from that
// table in the spectrum's layout; wtw: launch_wide_tw of the line length.
cudaError_t launch_fwd_cols(const Geom& g, const SegSrc& in, float2* out, const float2* tw, cudaStream_t st,
                            int nseg = 1);
// wtw: launch_wide_tw of R1 (rows of 512 and more; tw: the radix-16 tables of the others)
cudaError_t launch_fwd_rows(const Geom& g, const float2* in, float2* out, const float2* tw3L, Tw2 tw2L, const float2* tw,
                            const float2* wtw, cudaStream_t st, int nseg = 1);
cudaError_t launch_inv_cols(const Geom& g, const float2* in, float2* out, const ChirpAnchor* anc,
                            int clog, const float2* ctab, const float2* tw, const float2* wtw, cudaStream_t st,
                            int nseg = 1);
cudaError_t launch_inv_rows(const Geom& g, const float2* buf, float* P, float2* vout, long long vstride,
                            long long vofs, const MSpan& span, const float2* tw3M, const float2* tw, const float2* wtw,
                            cudaStream_t st, int nseg = 1);
// whether I1 of this geometry can take the chirp from a table (launch_chirp_c64, runs = false)
bool inv_cols_table(const Geom& g);
// Fused schedule (F1, F2f, Ic) for single-trial FP32 plans whose geometry has
// J = M / R2 = FUSED_J; fused_groups = sub-channel groups per m1 in Ic.
constexpr int FUSED_J = 64;
bool fused_geometry(const Geom& g);
int fused_groups(const Geom& g);
// ctab non-null: the chirp from that per-bin table (launch_chirp_c64), else from the anchors
cudaError_t launch_fwd_rows_inv(const Geom& g, const float2* in, float2* out, Tw2 tw2L,
                                const float2* wtw, const ChirpAnchor* anc, int clog, const float2* ctab,
                                cudaStream_t st, int nseg = 1);
cudaError_t launch_chirp_c64(float2* tab, const Geom& g, bool runs, double du, double half, double f0, double alpha, int sgn,
                             cudaStream_t st);
// words: the trial's launch_chirp_words, or null (from its anchors)
cudaError_t launch_inv_rows_chirp(const Geom& g, const float2* in, float2* out, Tw2 tw2L, const unsigned* words,
                                  const ChirpAnchor* anc, int clog, cudaStream_t st);
// nu > 1: one launch over nu trials or segments, the u-th reading in + u L and writing
// P + u M, part + u G M, cnt + u FUSED_J (G = fused_groups); wtw: launch_wide_tw of R2
// (null: the radix-16 stages with their tables tw)
cudaError_t launch_inv_cols_det(const Geom& g, const float2* in, float* P, float* part, int* cnt, float2* vout,
                                long long vstride, long long vofs, const MSpan& span, const float2* tw,
                                const float2* wtw, cudaStream_t st, int nu = 1);
// Batched lanes: Ir over ntr trials in one launch (trial t writes out + t L),
// the chirp from the lane's Q0.32 table (table = true) or each trial's anchors
cudaError_t launch_inv_rows_chirp_multi(const Geom& g, const float2* in, float2* out, int ntr, Tw2 tw2L,
                                        MultiChirp mc, bool table, cudaStream_t st);
// Tensor-core column pass (split-BF16, three terms) for R2 = 2048 and at least
// four sub-channels: same outputs and arguments as launch_inv_cols_det, plus
// its operand block (build_ic_tc_ops, ic_tc_ops_bytes() bytes on the device)
// and the plan's MMA-wait error flag.
bool ic_tc_geometry(const Geom& g);
cudaError_t launch_inv_cols_det_tc(const Geom& g, const float2* in, float* P, float* part, int* cnt, float2* vout,
                                   long long vstride, long long vofs, int m_lo, int m_hi, const uint4* ops, int* err,
                                   cudaStream_t st, int ntr = 1);
void build_ic_tc_ops(unsigned char* out);
int ic_tc_ops_bytes();
// Device-to-device byte copy as a kernel (the carry rewrite between pushes).
cudaError_t launch_copy_bytes(int8_t* dst, const int8_t* src, long long n, cudaStream_t st);
// Host-to-device copy from mapped pinned memory by `blocks` CTAs (the copy engines are not used).
cudaError_t launch_copy_host(int8_t* dst, const int8_t* src, long long n, int blocks, cudaStream_t st);
// Phase words of one trial from its anchors, in F2f's order (row, position in a run, run).
cudaError_t launch_chirp_words(unsigned* words, const Geom& g, const ChirpAnchor* anc, int clog, cudaStream_t st);
cudaError_t launch_chirp_table(unsigned* tab, const Geom& g, double du, double half, double f0, double alpha, int sgn,
                               cudaStream_t st);
cudaError_t launch_decimate_multi(const float* P, long long pstride, long long n, long long g0, long long num,
                                  long long den, long long j_lo, long long nj, float* T, int* C, long long ring,
                                  const int* rows, int ntr, cudaStream_t st);
size_t fold_smem_bytes(int nbins);
int fold_parts(long long n, long long* chunk);
cudaError_t launch_fold(const float* P, long long n, long long g0, double inc, int nbins, double* psum,
                        int* phits, double* prof_sum, long long* prof_hits, cudaStream_t st);
// The fold's phase rule: nc = 0 folds at the constant period (phase g inc);
// 1 <= nc <= 8 evaluates the polynomial phi = sum_i c[i] tau^i, tau = g dt - t_ref
// (Horner's rule, every FP64 operation rounded on its own).
struct FoldPhase {
  double inc = 0;
  int nc = 0;
  double dt = 0, t_ref = 0;
  double c[8] = {};
};
#ifdef __CUDACC__
// True when the FP64 evaluation (Horner's rule) of the phase polynomial c[0 .. nc) in
// tau = g dt - t_ref is known to grow from each sample of [ga, gb] to the next: phi' at the
// middle less its largest change over the span, times dt, exceeds twice the
// evaluation's rounding with room to spare.  False for NaN.
__device__ inline bool phase_forwards(const double* c, int nc, double dt, double t_ref, long long ga, long long gb) {
  const double t0 = (double)ga * dt - t_ref, t1 = (double)gb * dt - t_ref;
  const double tm = 0.5 * (t0 + t1), half = 0.5 * (t1 - t0), ta = fmax(fabs(t0), fabs(t1));
  double d = 0.0, dd = 0.0, mag = 0.0, pm = 1.0, pa1 = 1.0, pa2 = 0.0;
  for (int i = 0; i < nc; ++i) {
    const double a = fabs(c[i]);
    if (i >= 1) {
      d += i * c[i] * pm;
      pm *= tm;
    }
    if (i >= 2) {
      pa2 = i == 2 ? 1.0 : pa2 * ta;
      dd += i * (i - 1) * a * pa2;
    }
    mag += a * pa1;
    pa1 *= ta;
  }
  // tau itself is rounded: to |g dt| + |t_ref| ulps, times the slope
  const double err = 1e-14 * (mag + (fabs(d) + dd * half) * (fabs((double)gb * dt) + fabs(t_ref)));
  return (d - dd * half) * dt > err;
}
#endif
// Fold + decimation of nseg consecutive segments s0 .. (single-DM plans).  Segment y's
// power is P + y M, n_y = min(S_c, n_left - y S_c) samples from g0 + y S_c on.  The
// fold of segment s adds to the fold_parts rows of its slot s mod fold_slots of the
// partials [fold_rows][nbins], which accumulate over the stream, so the sums do not depend
// on how the segments are grouped into launches (nseg <= fold_slots);
// launch_fold_snapshot merges the rows into the profile (replacing it).
struct FoldSegs {
  long long s0, g0, S_c, M, n_left;
  int nseg;
};
int fold_slots(const Geom& g);   // also the most segments per launch
int fold_parts_seg(const Geom& g);
cudaError_t launch_fold_dec(const Geom& g, const float* P, const FoldSegs& f, const FoldPhase& ph, int nbins, long long num,
                            long long den, float* T, int* C, long long ring, double* psum, long long* phits,
                            cudaStream_t st);
cudaError_t launch_fold_snapshot(const double* psum, const long long* phits, int rows, int nbins, double* prof_sum,
                                 long long* prof_hits, cudaStream_t st);
cudaError_t launch_decimate(const float* P, long long n, long long g0, long long num, long long den,
                            long long j_lo, long long nj, float* T, int* C, long long ring, cudaStream_t st);

}  // namespace pond
