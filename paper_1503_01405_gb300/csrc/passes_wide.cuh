// Passes whose line FFTs keep 64 values per thread (fft_wide.cuh).
#pragma once
#include "fft_wide.cuh"
#include "passes.cuh"

namespace pond {

// L2 prefetch distance (CTAs) of these passes, three CTAs per SM.  Batched
// chunk of 128 trials / full-rate stream, ms: 38: 104.3 / 15.98, 114: 103.3 /
// 15.97, 228: 103.5 / 16.09, 456: 105.4 / 16.34, none: 116.6 / 16.40.
constexpr int WIDE_PF = 114;

// Shared memory of a tile of lines of RA x RB.
template <int RA, int RB>
constexpr int wide_smem_bytes() {
  return TILE / (RA * RB) * wide_stride<RA, RB>() * (int)sizeof(float2);
}

// ---------------------------------------------------------------------------
// Ic: column pass after F2f: inverse length-R2 FFTs, discard, detect, sum
// ---------------------------------------------------------------------------

// A CTA takes nl = TILE/R2 adjacent sub-channels of one m1 (one contiguous
// block of F2f's output, rows k2 of nl elements), transforms them along k2
// (v_c[m1 + J m2], m2 < R2), keeps the valid span m_lo <= m < m_hi, and detects.
// Thread (t, h) of stage 2 holds outputs t + 64 k of the 64 / RB lines of half h,
// so |v|^2 is summed over them in registers and once across the halves by
// shuffles: the outputs never return to shared memory.  With G = NCH / nl > 1
// the CTAs of one m1 each write their group's partial sums to part[g][m1][m2];
// the last of the G to finish (an atomic ticket per m1, no waiting) adds the G
// partials in group order into P and clears the ticket.
// P = scale^2 sum_c |v_c|^2.  Bound by DRAM and latency: the block is read once
// (64 MiB per 2^24 segment) and the instruction count falls from 60 to about 35
// per value against the radix-16 form.  Batched full-rate plan, 32 trials per
// launch: 23.6 -> 17.1 us per trial; the 8 s chunk of 128 trials 149 -> 126 ms.
template <int R2, bool VOUT>
__global__ void __launch_bounds__(WIDE_NT, 3) k_inv_cols_det_w(const float2* __restrict__ in, float* __restrict__ P,
                                                               float* __restrict__ part, int* __restrict__ cnt,
                                                               float2* __restrict__ vout, long long vstride,
                                                               long long vofs, int logG, int logJ, MSpan span,
                                                               float scale, const float2* __restrict__ tw,
                                                               TrialStride ts) {
  constexpr int RA = 64, RB = R2 / RA, NL = TILE / R2, BPT = 64 / RB;
  constexpr int WSTR = wide_stride<RA, RB>();
  extern __shared__ float2 smem[];
  __shared__ int s_last;
  const int m_lo = span.m_lo, m_hi = span.hi(blockIdx.y);
  // blockIdx.y is the trial or segment, with its own input, P, partials and tickets
  in += blockIdx.y * ts.in;
  P += blockIdx.y * ts.P;
  part += blockIdx.y * ts.part;
  cnt += blockIdx.y * ts.cnt;
  const int tid = (int)threadIdx.x;
  const int m1 = blockIdx.x >> logG, gi = blockIdx.x & ((1 << logG) - 1);
  const float2* blk = in + (size_t)blockIdx.x * TILE;   // block m1 G + g
  if (tid < 4) {
    // the block of CTA blockIdx.x + WIDE_PF (in launch order, the next unit's
    // blocks after this trial's last), in four quarters
    const unsigned nx = gridDim.x, lin = blockIdx.y * nx + blockIdx.x + WIDE_PF;
    if (lin < nx * gridDim.y) {
      const float2* nb = in - blockIdx.y * ts.in + (size_t)(lin / nx) * ts.in + (size_t)(lin % nx) * TILE;
      constexpr unsigned qb = TILE * (unsigned)sizeof(float2) / 4;
      if (ts.in != 0 || lin / nx == blockIdx.y) prefetch_l2(reinterpret_cast<const char*>(nb) + tid * qb, qb);
    }
  }
  // stage 2's thread: column t, half h (lane bit 4) of the lines
  const int t2 = (tid & 15) | ((tid >> 5) << 4), h = (tid >> 4) & 1;
  WideTwPair<RA, RB> w2;
  {
    // stage 1 straight from global memory: butterfly t of line ci (sub-channels
    // fastest, so consecutive lanes read consecutive elements) reads rows t + RB j
    const int ci = tid & (NL - 1), t = tid / NL;
    float2 v[RA];
#pragma unroll
    for (int j = 0; j < RA; ++j) v[j] = __ldg(blk + tid + j * (RB * NL));
    w2.load(tw, t2);
    wide_dft<RA, true>(v);
    float2* dst = smem + ci * WSTR + (RA + 1) * t;
#pragma unroll
    for (int j = 0; j < RA; ++j) dst[j] = v[j];
  }
  __syncthreads();
  float p[RB];
#pragma unroll
  for (int k = 0; k < RB; ++k) p[k] = 0.f;
#pragma unroll 1   // one copy of the DFT in the instruction cache
  for (int u = 0; u < BPT; ++u) {
    const int line = h * BPT + u;
    const float2* src = smem + line * WSTR + t2;
    float2 v[RB];
#pragma unroll
    for (int j = 0; j < RB; ++j) v[j] = src[j * (RA + 1)];
    w2.template dft<true>(v);
#pragma unroll
    for (int k = 0; k < RB; ++k) {
      p[k] = fmaf(v[k].y, v[k].y, fmaf(v[k].x, v[k].x, p[k]));
      if constexpr (VOUT) {
        const int m = m1 + ((t2 + RA * k) << logJ);
        if (m >= m_lo && m < m_hi)
          vout[(size_t)(gi * NL + line) * vstride + vofs + (m - m_lo)] = cscale(v[k], scale);
      }
    }
  }
  // the two halves of the lines meet in the same warp: half h keeps outputs
  // k = h RB/2 .. of both
  const float s2 = scale * scale;
#pragma unroll
  for (int k = 0; k < RB / 2; ++k) {
    const float mine = h ? p[k + RB / 2] : p[k], other = h ? p[k] : p[k + RB / 2];
    const float q = mine + __shfl_xor_sync(0xffffffffu, other, 16);
    const int m2 = t2 + RA * (k + h * (RB / 2));
    if (logG == 0) {
      const int m = m1 + (m2 << logJ);
      if (m >= m_lo && m < m_hi) P[m - m_lo] = q * s2;
    } else {
      part[((((size_t)gi << logJ) + m1) << ilog2c(R2)) + m2] = q;
    }
  }
  if (logG == 0) return;
  // release: the barrier orders every thread's partials before thread 0's fence
  // and ticket; acquire: the last group's thread 0 fences after its ticket and
  // the barrier orders the CTA's L2 loads of the other groups' partials after it
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    const int t = atomicAdd(cnt + m1, 1);
    s_last = t == (1 << logG) - 1;
    if (s_last) {
      cnt[m1] = 0;   // every group has taken its ticket
      __threadfence();
    }
  }
  __syncthreads();
  if (!s_last) return;
  // four outputs per thread and step: the G partials of each (G <= GMAX) are
  // loaded together, then added in group order
  constexpr int GMAX = 16;
  const size_t gstride = (size_t)1 << (logJ + ilog2c(R2));   // part[g + 1] - part[g]
#pragma unroll 1
  for (int m2 = 4 * tid; m2 < R2; m2 += 4 * WIDE_NT) {
    const float* src = part + (((size_t)m1) << ilog2c(R2)) + m2;
    float4 v[GMAX];
#pragma unroll
    for (int g = 0; g < GMAX; ++g)
      v[g] = g < (1 << logG) ? __ldcg(reinterpret_cast<const float4*>(src + g * gstride)) : make_float4(0, 0, 0, 0);
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int g = 0; g < GMAX; ++g)
      if (g < (1 << logG)) {
        a.x += v[g].x;
        a.y += v[g].y;
        a.z += v[g].z;
        a.w += v[g].w;
      }
    const float o[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = m1 + ((m2 + i) << logJ);
      if (m >= m_lo && m < m_hi) P[m - m_lo] = o[i] * s2;
    }
  }
}

// ---------------------------------------------------------------------------
// Ir: per-trial row pass of batched plans with M = 64 R2
// ---------------------------------------------------------------------------

// A batched plan shares F2's spectrum X[k2 + R2 k1] (row k2, column k1) among
// its trials.  For each trial a row tile (nl = TILE/R1 consecutive rows) takes the
// trial's chirp (Eq. 4) and the length-64 inverse DFT of every (row, sub-channel)
// run of J = 64 consecutive columns, scales output m1 by e^{2 pi i k2 m1 / M} and
// stores it at ((m1 G + g) R2 + k2) nlc + ci, c = g nlc + ci, nlc = min(TILE/R2,
// NCH), the blocks that the column pass reads.
//
// A thread transforms a whole run in registers.  Rows sit in shared memory with
// one value of padding per run and a row stride of RowTile::rstr values, so that a warp's
// lanes, which take the nlc sub-channels of a block first, then the tile's rows,
// read distinct banks and store runs of nl nlc consecutive values.
struct RowTile {
  int logR2, lognl, lognlc;   // rows of the segment, rows per tile, sub-channels per block
  int rstr;                   // row stride in shared memory, values
  int tstr;                   // row stride of the table words (32 lanes on 4-byte banks)
};

template <int R1>
__host__ __device__ constexpr int run_slots() { return TILE / R1; }

// Row stride: NCH runs of 65 values, padded to (16 / nl or nlc, the larger) mod 16
// while a half-warp covers several rows.
inline RowTile row_tile(int logR1, int logR2) {
  RowTile r;
  const int lognch = logR1 - 6;
  r.logR2 = logR2;
  r.lognl = 13 - logR1;
  r.lognlc = 13 - logR2 < lognch ? 13 - logR2 : lognch;
  const int base = 65 << lognch, nlc = 1 << r.lognlc, s = 16 >> r.lognl;
  const int want = nlc >= 16 ? 0 : (nlc > s ? nlc : s);
  r.rstr = base + ((want - base) & 15);
  // lanes of a warp: nlc sub-channels, then min(nl, 32 / nlc) rows, then blocks of nlc
  const int rows = nlc >= 32 ? 1 : (32 / nlc < (1 << r.lognl) ? 32 / nlc : 1 << r.lognl);
  r.tstr = base + (((rows > 1 ? 32 / rows : 0) - base) & 31);
  return r;
}
// largest row stride of a line length (any R2): for shared-memory limits
constexpr int row_stride_max(int R1) { return 65 * (R1 / 64) + 31; }

constexpr int TWK_STR = 65;   // stride of a row's 64 factors e^{2 pi i k2 m1 / M}

// Thread -> run: sub-channels of a block fastest, then rows, then blocks.
struct Run {
  int slot, c;
};
__device__ __forceinline__ Run run_of(const RowTile& rt, int id) {
  Run r;
  r.slot = (id >> rt.lognlc) & ((1 << rt.lognl) - 1);
  r.c = (id & ((1 << rt.lognlc) - 1)) | ((id >> (rt.lognlc + rt.lognl)) << rt.lognlc);
  return r;
}

// A run's bins k0 + R2 j times the chirp from a trial's anchors (chirp_from).
template <class Bin>
__device__ __forceinline__ void run_chirp_anchors(float2* v, const ChirpAnchor* __restrict__ anc, int clog, unsigned k0,
                                                  int logR2, Bin bin) {
  // bins that share an anchor: the run starts at a multiple of min(2^clog, M) plus k2 < R2
  const int amask = clog > logR2 ? (1 << (clog - logR2)) - 1 : 0;
  ChirpAnchor a;
#pragma unroll
  for (int j = 0; j < 64; ++j) {
    const unsigned k = k0 + ((unsigned)j << logR2);
    if ((j & amask) == 0) a = anc[k >> clog];
    v[j] = cmul(bin(j), chirp_from(a, clog, k));
  }
}

// The run's 64-point inverse DFT, the factors twk[m1] and the blocked store.
template <int R1>
__device__ __forceinline__ void run_finish(float2* v, const RowTile& rt, const Run& r, unsigned k2, const float2* twk,
                                           float2* __restrict__ out) {
  constexpr int LOGNCH = ilog2c(R1 / 64);
  wide_dft<64, true>(v);
  const unsigned g = (unsigned)r.c >> rt.lognlc, ci = (unsigned)r.c & ((1u << rt.lognlc) - 1);
  float2* dst = out + ((((g << rt.logR2) + k2) << rt.lognlc) + ci);
  const float2* w = twk + r.slot * TWK_STR;
#pragma unroll
  for (int m1 = 0; m1 < 64; ++m1) dst[(unsigned)m1 << (LOGNCH + rt.logR2)] = cmul(v[m1], w[m1]);
}

// e^{2 pi i k2 m1 / M} = conj(w^{k2 m1 NCH}), w = exp(-2 pi i / L), k2 m1 NCH < L, of
// rows row_of(0 .. nl-1): one product of two table entries (tw2L steps by half a bin).
template <int R1, class RowOf>
__device__ __forceinline__ void make_twk(float2* twk, const Tw2& tw2L, int nl, RowOf row_of) {
  for (int i = threadIdx.x; i < nl * 64; i += blockDim.x) {
    const unsigned k2 = (unsigned)row_of(i >> 6), m1 = (unsigned)(i & 63);
    twk[(i >> 6) * TWK_STR + m1] = cconj(tw2(tw2L, (k2 * m1) << (ilog2c(R1 / 64) + 1)));
  }
}

// Table form: the rows and their Q0.32 table words resident for every trial of the launch.
// Four warps run a trial of the tile, GROUPS trials at a time; a run is read from the
// resident copies and stored from registers, so there is no exchange and no
// barrier after the tile's load.  Bound by the issue slots (chirp and DFT, 34
// instructions per value) next to the 64 MiB that each trial writes (4.8 TB/s).
// Full-rate batched plan: 19.9 us per trial with the runs split over four lanes
// and exchanged through shared memory (78 % of that pipe), 13.5 here (16 in a launch of 16 trials
// that starts with a cold L2); the 8 s chunk of 128 trials 126 -> 103 ms on the device.
constexpr int TAB_GROUPS = 3;   // 384 threads of 168 registers: one CTA per SM

template <int R1>
__global__ void __launch_bounds__(TAB_GROUPS * WIDE_NT, 1)
    k_inv_rows_table(const float2* __restrict__ in, float2* __restrict__ out, long long out_tstride, RowTile rt,
                     Tw2 tw2L, MultiChirp mc, int ntr) {
  constexpr int NLR = run_slots<R1>(), LOGR1 = ilog2c(R1);
  extern __shared__ float2 smem[];
  float2* twk = smem;                              // [NLR][TWK_STR]
  float2* rows = twk + NLR * TWK_STR; // [NLR * rstr]
  unsigned* tabw = reinterpret_cast<unsigned*>(rows + NLR * rt.rstr);
  const int r0 = blockIdx.x * NLR;
  const float2* src = in + ((size_t)r0 << LOGR1);
  const unsigned* tsrc = mc.atab + ((size_t)r0 << LOGR1);
#pragma unroll 8
  for (int i = threadIdx.x; i < TILE; i += TAB_GROUPS * WIDE_NT) {
    const int slot = i >> LOGR1, k1 = i & (R1 - 1), o = k1 + (k1 >> 6);
    rows[slot * rt.rstr + o] = __ldg(src + i);
    tabw[slot * rt.tstr + o] = __ldg(tsrc + i);
  }
  make_twk<R1>(twk, tw2L, NLR, [&](int slot) { return r0 + slot; });
  __syncthreads();   // twk, the rows and their table words
  const Run r = run_of(rt, (int)threadIdx.x & (WIDE_NT - 1));
  const int o = r.slot * rt.rstr + 65 * r.c, ot = r.slot * rt.tstr + 65 * r.c;
  int t = (int)threadIdx.x / WIDE_NT;
  unsigned next = t < ntr ? __ldg(mc.nmul + t) : 0u;
  for (; t < ntr; t += TAB_GROUPS) {
    const unsigned nm = next;
    if (t + TAB_GROUPS < ntr) next = __ldg(mc.nmul + t + TAB_GROUPS);   // ahead of its use
    float2 v[64];
#pragma unroll
    for (int j = 0; j < 64; ++j) v[j] = cmul(rows[o + j], chirp_q32(nm * tabw[ot + j]));
    run_finish<R1>(v, rt, r, (unsigned)(r0 + r.slot), twk, out + (size_t)t * out_tstride);
  }
}

template <int R1>
size_t table_smem_bytes(const RowTile& rt) {
  constexpr int NLR = run_slots<R1>();
  return (size_t)(NLR * TWK_STR + NLR * rt.rstr) * sizeof(float2) +
         (size_t)NLR * rt.tstr * sizeof(unsigned);
}

// Word form: the anchor chirp with its phases read from per-trial tables of Q0.32 words
// ([row][j][c]: consecutive lanes, consecutive words) made from the anchors once
// per plan.  A CTA keeps its rows resident and runs tpc trials of the launch on
// them (blockIdx.x: trials x tpc ..), so a trial reads 4 bytes per bin and
// writes 8.  21 trials of 2^19 bins: 53 us per launch with
// the anchors evaluated per bin and trial, 36 here.  Also one trial per launch, where the
// anchors' evaluation adds to each tile's serial path (2^17 bins, a trial with its column
// pass and decimation: 18 us against 26).
template <int R1>
__global__ void __launch_bounds__(WIDE_NT, 3)
    k_inv_rows_words(const float2* __restrict__ in, float2* __restrict__ out, long long out_tstride, RowTile rt,
                     Tw2 tw2L, const unsigned* __restrict__ words, int ntr, int tpc) {
  constexpr int NLR = run_slots<R1>(), LOGR1 = ilog2c(R1), NCH = R1 / 64;
  extern __shared__ float2 smem[];
  float2* twk = smem;              // [NLR][TWK_STR]
  float2* rows = twk + NLR * TWK_STR;       // [NLR * rstr]
  const int r0 = blockIdx.y * NLR;
  {
    const float2* src = in + ((size_t)r0 << LOGR1);
    float2 v[64];   // the tile: 64 loads in flight per thread
#pragma unroll
    for (int u = 0; u < 64; ++u) v[u] = __ldg(src + threadIdx.x + u * WIDE_NT);
#pragma unroll
    for (int u = 0; u < 64; ++u) {
      const int i = (int)threadIdx.x + u * WIDE_NT, k1 = i & (R1 - 1);
      rows[(i >> LOGR1) * rt.rstr + k1 + (k1 >> 6)] = v[u];
    }
  }
  make_twk<R1>(twk, tw2L, NLR, [&](int slot) { return r0 + slot; });
  __syncthreads();
  const Run r = run_of(rt, (int)threadIdx.x);
  const float2* row = rows + r.slot * rt.rstr + 65 * r.c;
  const unsigned* wr = words + ((size_t)(r0 + r.slot) << LOGR1) + r.c;
  const int t1 = min(ntr, ((int)blockIdx.x + 1) * tpc);
  for (int t = (int)blockIdx.x * tpc; t < t1; ++t) {
    // nothing of the run (its values, its outputs' offsets) is held across trials: 64
    // of each would not fit the registers
    RowTile ro = rt;
    asm volatile("" : "+r"(ro.logR2)::"memory");
    const unsigned* wt = wr + (size_t)t * out_tstride;
    float2 v[64];
#pragma unroll
    for (int j = 0; j < 64; ++j) v[j].x = __uint_as_float(__ldg(wt + j * NCH));
#pragma unroll
    for (int j = 0; j < 64; ++j) v[j] = cmul(row[j], chirp_q32(__float_as_uint(v[j].x)));
    run_finish<R1>(v, ro, r, (unsigned)(r0 + r.slot), twk, out + (size_t)t * out_tstride);
  }
}

// Anchor form: one CTA per (trial, row tile), the chirp evaluated from the trial's anchors
// as the tile is loaded (lanes over consecutive columns: their anchors lie side by side).
// For lanes whose word tables would be too large, and for the length tuner's trial (2^23 bins, one
// trial with its column pass and decimation: 94 us, with the words 82; the whole tile loaded
// first and an anchor per value: 116).
// blockIdx.x is the trial and runs fastest, so the CTAs that share rows are
// adjacent in launch order and all but the first find them in L2.  With mc.anc null
// the launch's one trial takes its anchors from anc1, clog1.
template <int R1>
__global__ void __launch_bounds__(WIDE_NT, 3)
    k_inv_rows_anchor(const float2* __restrict__ in, float2* __restrict__ out, long long out_tstride, RowTile rt,
                      Tw2 tw2L, MultiChirp mc, const ChirpAnchor* __restrict__ anc1, int clog1) {
  constexpr int NLR = run_slots<R1>(), LOGR1 = ilog2c(R1);
  extern __shared__ float2 smem[];
  float2* twk = smem;              // [NLR][TWK_STR]
  float2* rows = twk + NLR * TWK_STR;       // [NLR * rstr]
  const int r0 = blockIdx.y * NLR, t = blockIdx.x;
  const float2* src = in + ((size_t)r0 << LOGR1);
  {
    if (t == 0 && threadIdx.x == 0) {
      // the first trial's CTA of a row tile warms L2 with the rows of a later tile
      const unsigned rn = blockIdx.y + max(1u, (unsigned)WIDE_PF / gridDim.x);
      if (rn < gridDim.y) prefetch_l2(in + (((size_t)rn * NLR) << LOGR1), TILE * (unsigned)sizeof(float2));
    }
    const ChirpAnchor* anc = mc.anc ? mc.anc[t] : anc1;
    const int clog = mc.anc ? __ldg(mc.clog + t) : clog1;
    // 16 values at a time, all rows of CB columns: their anchors fit the registers beside them
    constexpr int CB = 16 / NLR, COLS = R1 / WIDE_NT;
    const bool shared = (1 << clog) >= NLR;   // the tile's rows of a column have one anchor
#pragma unroll 1
    for (int c0 = 0; c0 < COLS; c0 += CB) {
      float2 v[CB][NLR];
#pragma unroll
      for (int q = 0; q < CB; ++q)
#pragma unroll
        for (int slot = 0; slot < NLR; ++slot) v[q][slot] = __ldg(src + slot * R1 + threadIdx.x + (c0 + q) * WIDE_NT);
      ChirpAnchor a[CB];
#pragma unroll
      for (int q = 0; q < CB; ++q)
        a[q] = anc[((unsigned)r0 + ((threadIdx.x + (unsigned)(c0 + q) * WIDE_NT) << rt.logR2)) >> clog];
#pragma unroll
      for (int q = 0; q < CB; ++q) {
        const int k1 = (int)threadIdx.x + (c0 + q) * WIDE_NT;
#pragma unroll
        for (int slot = 0; slot < NLR; ++slot) {
          const unsigned k = (unsigned)(r0 + slot) + ((unsigned)k1 << rt.logR2);
          if (!shared && slot > 0) a[q] = anc[k >> clog];
          rows[slot * rt.rstr + k1 + (k1 >> 6)] = cmul(v[q][slot], chirp_from(a[q], clog, k));
        }
      }
    }
  }
  make_twk<R1>(twk, tw2L, NLR, [&](int slot) { return r0 + slot; });
  __syncthreads();
  const Run r = run_of(rt, (int)threadIdx.x);
  const float2* row = rows + r.slot * rt.rstr + 65 * r.c;
  float2 v[64];
#pragma unroll
  for (int j = 0; j < 64; ++j) v[j] = row[j];
  run_finish<R1>(v, rt, r, (unsigned)(r0 + r.slot), twk, out + (size_t)t * out_tstride);
}

template <int R1>
size_t anchor_smem_bytes(const RowTile& rt) {
  constexpr int NLR = run_slots<R1>();
  return (size_t)(NLR * TWK_STR + NLR * rt.rstr) * sizeof(float2);
}

// ---------------------------------------------------------------------------
// F2, F2f: row FFTs of the forward transform, real-input split, and (F2f) the
// chirp with the first factor of every sub-channel's inverse
// ---------------------------------------------------------------------------

// L2 prefetch distance of F2 and F2f, at most three CTAs per SM (full-rate stream, ms:
// 20: 14.46, 38: 14.59, 114: 15.0, none: 15.4).
constexpr int ROW_PF = 20;

// The two entries of a tw2 lookup, loaded now and multiplied later.
struct Tw2Pair {
  float2 hi, lo;
  Tw2Pair() = default;
  __device__ __forceinline__ Tw2Pair(const Tw2& t, unsigned e)
      : hi(__ldg(t.hi + (e >> TW2_LOG))), lo(__ldg(t.lo + (e & (TW2_LO - 1)))) {}
  __device__ __forceinline__ float2 value() const { return cmul(hi, lo); }
};

enum RowMode { ROW_SPECTRUM = 0, ROW_ANCHORS = 1, ROW_TABLE = 2 };

// Rows k2 and R2 - k2 share a CTA (f2_line), each a (64, RB) line, RB = R1 / 64 =
// NCH.  Stage 1 takes the rows straight from global memory with the inter-pass
// twiddle w^{n1 k2}, n1 = t + RB (8 a + b), factored as w^{8 RB k2 a} (inside the
// first DFT) and w^{k2 (t + RB b)}; stage 2 works in place (a thread reads and writes the
// same column), after which run c of a row is row c of its line.  Then, with
// A = Z[k], B = conj(Z[L-k]), W = exp(-i pi k / L):
//   X[k] = (A + B) / 2 - i W (A - B) / 2,
// evaluated for every bin on its own (both bins of a pair load the same two
// values, so this costs one more shared-memory read per bin and saves the write, the read and
// the barrier of a split spectrum).  W = Wb s[j], Wb per run, s[j] = exp(-i pi j / R1).
//   ROW_SPECTRUM: X[k2 + R2 k1] to row k2, column k1 (the batched trials read it);
//   ROW_TABLE / ROW_ANCHORS (F2f): times the chirp, from the per-bin table (laid out
//   [row][j][c]: consecutive lanes, consecutive words) or the anchors, then the run's
//   length-64 inverse DFT and blocked store (run_finish).
// F2f runs two CTAs per SM: at the 168 registers of three, the run's 64 chirp loads are
// split into batches whose latency shows (101 us per launch at three, 71 at two).  F2 runs
// three for rows of 2048 and 4096 points (33.3 us against 36.9 per 2^23 bins); shorter rows
// belong to segments of at most 128 tiles, which do not fill the SMs once, and take
// the registers instead (2^20 bins beside another trial's passes: 8.0 us against 12.2).
// Bound by instruction issue (40 % in launches of four segments, 31 % in one's) and memory
// latency in turn.  Full rate, launches of four 2^24-point segments: 56 -> 47 us per
// segment; 22.6 M warp instructions per segment against 31.0 M with radix-16 stages.  A launch of one
// segment has 3.4 waves and takes 71 us where 512 threads per tile took 69.  blockIdx.x is
// the segment and runs fastest, so the segments of a launch share the chirp table's
// rows in L2 (launches of four: 215 -> 188 us).
template <int R1, int MODE>
__global__ void __launch_bounds__(WIDE_NT, MODE == ROW_SPECTRUM && R1 > 1024 ? 3 : 2)
    k_fwd_rows_w(const float2* __restrict__ in, float2* __restrict__ out, RowTile rt,
                 Tw2 tw2L, const float2* __restrict__ tw,
                 const ChirpAnchor* __restrict__ anc, int clog, const float2* __restrict__ ctab) {
  constexpr int RB = R1 / 64, NLR = run_slots<R1>(), BPT = 64 / RB, LOGR1 = ilog2c(R1), LOGRB = ilog2c(RB);
  extern __shared__ float2 smem[];
  float2* uni = smem;                          // [NLR][16]: w^{RB k2 b} (b < 8), w^{8 RB k2 a} at 8 + a
  float2* sj = uni + NLR * 16;                 // [64]: exp(-i pi j / R1)
  float2* wbt = sj + 64;                       // [NLR][RB]: exp(-i pi (k2 + 64 R2 c) / L) / 2
  float2* twk = wbt + NLR * RB;                // [NLR][TWK_STR]
  float2* sm = twk + NLR * TWK_STR;   // [NLR * rstr]
  const int tid = (int)threadIdx.x, R2 = 1 << rt.logR2, np = NLR / 2, q0 = blockIdx.y * np;
  in += (size_t)blockIdx.x << (LOGR1 + rt.logR2);
  out += (size_t)blockIdx.x << (LOGR1 + rt.logR2);
  auto row_of = [&](int slot) { return f2_line(slot, q0, np, R2); };
  const unsigned ahead = max(1u, (unsigned)ROW_PF / gridDim.x);
  if (tid < 4 && np == 1 && blockIdx.y + ahead < gridDim.y) {
    // the two rows of a CTA ROW_PF later (q and its mirror R2 - q), and, once per
    // launch of several segments, the same rows of the chirp table
    const int q = q0 + (int)ahead, row = (tid & 1) == 0 ? q : R2 - q;
    if (tid < 2) prefetch_l2(in + ((size_t)row << LOGR1), R1 * (unsigned)sizeof(float2));
    else if (MODE == ROW_TABLE && blockIdx.x == 0)
      prefetch_l2(ctab + ((size_t)row << LOGR1), R1 * (unsigned)sizeof(float2));
  }
  {
    // stage 1: butterfly t of the line, inputs n1 = t + RB j.  The table entries of
    // the twiddles are asked for ahead of the rows, their products formed behind them.
    constexpr int NU = (NLR * 16 + WIDE_NT - 1) / WIDE_NT, NK = MODE != ROW_SPECTRUM ? NLR / 2 : 0;
    const int slot = tid >> LOGRB, t = tid & (RB - 1);
    const unsigned k2 = (unsigned)row_of(slot);
    Tw2Pair pt(tw2L, 2 * k2 * (unsigned)t), pb(tw2L, k2 + ((unsigned)(64 * t) << rt.logR2)), ps, pu[NU], pk[NK + 1];
    if (tid < 64) ps = Tw2Pair(tw2L, (unsigned)tid << rt.logR2);
#pragma unroll
    for (int i = 0; i < NU; ++i) {
      const int q = tid + i * WIDE_NT;
      if (q < NLR * 16)
        pu[i] = Tw2Pair(tw2L, 2 * (unsigned)row_of(q >> 4) * ((unsigned)(q & 7) * (unsigned)((q & 8) ? 8 * RB : RB)));
    }
#pragma unroll
    for (int i = 0; i < NK; ++i) {
      const int q = tid + i * WIDE_NT;
      pk[i] = Tw2Pair(tw2L, ((unsigned)row_of(q >> 6) * (unsigned)(q & 63)) << (LOGRB + 1));
    }
    const float2* src = in + ((size_t)k2 << LOGR1) + t;
    float2 v[64];
#pragma unroll
    for (int j = 0; j < 64; ++j) v[j] = __ldg(src + j * RB);
    const float2 wt = pt.value();
    wbt[tid] = cscale(pb.value(), 0.5f);   // NLR RB = 128 entries
    if (tid < 64) sj[tid] = ps.value();
#pragma unroll
    for (int i = 0; i < NU; ++i)
      if (tid + i * WIDE_NT < NLR * 16) uni[tid + i * WIDE_NT] = pu[i].value();
#pragma unroll
    for (int i = 0; i < NK; ++i) {   // e^{2 pi i k2 m1 / M}, as make_twk
      const int q = tid + i * WIDE_NT;
      twk[(q >> 6) * TWK_STR + (q & 63)] = cconj(pk[i].value());
    }
    __syncthreads();   // uni
    const float2* un = uni + slot * 16;
    wide_dft<64, false>(
        v, [&](float2 x, int a) { return a == 0 ? x : cmul(x, un[8 + a]); },
        [&](float2 x, int b, int ka) { return tw64<false>(cmul(x, b == 0 ? wt : cmul(wt, un[b])), b * ka); });
    float2* dst = sm + slot * rt.rstr + 65 * t;
#pragma unroll
    for (int j = 0; j < 64; ++j) dst[j] = v[j];
  }
  {
    const int t2 = tid & 63;
    WideTw<64, RB> w2;
    w2.load(tw, t2);
    __syncthreads();
#pragma unroll 1
    for (int u = 0; u < BPT; ++u) {
      float2* p = sm + ((tid >> 6) + 2 * u) * rt.rstr + t2;
      float2 v[RB];
#pragma unroll
      for (int j = 0; j < RB; ++j) v[j] = p[65 * j];
      w2.template dft<false>(v);
#pragma unroll
      for (int j = 0; j < RB; ++j) p[65 * j] = v[j];
    }
  }
  __syncthreads();
  // X of (slot, c, j): partner Z[L - k] at column R1 - 1 - k1 of the mirrored row;
  // rows 0 and R2/2 (tile 0) pair with themselves, row 0 at column R1 - k1 (mod R1)
  struct Pair {
    int oa, ob, ob0;   // own value j at oa + j; the partner's at ob - j, for j = 0 at ob0
  };
  auto pair_of = [&](int slot, int c) {
    Pair q;
    const bool self = q0 == 0 && (slot == 0 || slot == np);
    const int ps = self ? slot : (slot < np ? slot + np : slot - np);
    q.oa = slot * rt.rstr + 65 * c;
    q.ob = ps * rt.rstr + 65 * (RB - 1 - c) + 63;
    q.ob0 = q.ob;
    if (self && slot == 0) {
      q.ob += 1;
      q.ob0 = c == 0 ? 0 : 65 * (RB - c);
    }
    return q;
  };
  auto split = [&](float2 A, float2 Z, float2 W) {   // W holds the factor 1/2
    const float2 B = cconj(Z), E = cadd(A, B), WO = cmul(W, csub(A, B));
    return make_float2(fmaf(0.5f, E.x, WO.y), fmaf(0.5f, E.y, -WO.x));
  };
  if constexpr (MODE == ROW_SPECTRUM) {
    // lane: bin j of a run; two runs of a row at a time
    const int j = tid & 63, c0 = tid >> 6;
    const float2 s = sj[j];
#pragma unroll 1
    for (int slot = 0; slot < NLR; ++slot) {
      const Pair q = pair_of(slot, c0);
      const float2 *pa = sm + q.oa + j, *pb = sm + q.ob - j + (j == 0 && q.ob0 != q.ob), *wb = wbt + slot * RB + c0;
      float2* o = out + ((size_t)row_of(slot) << LOGR1) + tid;
#pragma unroll
      for (int i = 0; i < RB / 2; ++i) {
        const float2 Z = i == 0 && j == 0 ? sm[q.ob0] : pb[-130 * i];
        o[128 * i] = split(pa[130 * i], Z, cmul(wb[2 * i], s));
      }
    }
  } else {
    const Run r = run_of(rt, tid);
    const unsigned k2 = (unsigned)row_of(r.slot);
    const Pair q = pair_of(r.slot, r.c);
    const float2 wb = wbt[r.slot * RB + r.c];
    auto bin = [&](int j) { return split(sm[q.oa + j], sm[j == 0 ? q.ob0 : q.ob - j], cmul(wb, sj[j])); };
    float2 v[64];
    if constexpr (MODE == ROW_TABLE) {
      const float2* ct = ctab + ((size_t)k2 << LOGR1) + r.c;
#pragma unroll
      for (int j = 0; j < 64; ++j) v[j] = __ldg(ct + j * RB);
#pragma unroll
      for (int j = 0; j < 64; ++j) v[j] = cmul(bin(j), v[j]);
    } else {
      run_chirp_anchors(v, anc, clog, k2 + ((unsigned)(64 * r.c) << rt.logR2), rt.logR2, bin);
    }
    run_finish<R1>(v, rt, r, k2, twk, out);
  }
}

template <int R1>
size_t fwd_rows_smem_bytes(const RowTile& rt) {
  constexpr int NLR = run_slots<R1>();
  return (size_t)(NLR * 16 + 64 + WIDE_NT + NLR * TWK_STR + NLR * rt.rstr) *
         sizeof(float2);
}

// ---------------------------------------------------------------------------
// I1: per-sub-channel inverse column FFTs (table chirp)
// ---------------------------------------------------------------------------

// Line (c, j1) holds Y[c M + j1 + Q1 j2], j2 < Q2, read from F2's rows (j2 = j2lo + 2^s
// j2hi, s = logR2 - logQ1, at row j1 + Q1 j2lo, column c M/R2 + j2hi) and multiplied
// by the chirp from the plan's per-bin table, which has the spectrum's layout.  The inverse
// transform goes to natural order c M + j1 + Q1 m2.  Lines are (64, RB); lanes run over the
// inputs of a line in stage 1 and over the lines in stage 2 (runs of nl values).
// blockIdx.x is the segment and runs fastest: the segments of a launch share the table in
// L2.  Bound by memory (three streams of 8 bytes a bin, one of them shared).  Launches of
// four segments of 2^20 bins: 28.3 us with the chirp from anchors in the radix-16 form, 17.3 here.
template <int Q2>
__global__ void __launch_bounds__(WIDE_NT, 2)
    k_inv_cols_w(const float2* __restrict__ in, float2* __restrict__ out, int logQ1, int logM, int logR1, int logR2,
                 const float2* __restrict__ ctab, const float2* __restrict__ tw) {
  constexpr int RA = 64, RB = Q2 / 64, NL = TILE / Q2, BPT = 64 / RB, LOGNL = ilog2c(NL);
  constexpr int WSTR = wide_stride<RA, RB>();
  extern __shared__ float2 smem[];
  in += (size_t)blockIdx.x << (logR1 + logR2);
  out += (size_t)blockIdx.x << (logR1 + logR2);
  const int tid = (int)threadIdx.x, l0 = blockIdx.y * NL;
  {
    const int l = l0 + tid / RB, t = tid % RB, s = logR2 - logQ1;
    const unsigned c = (unsigned)l >> logQ1, j1 = (unsigned)l & ((1u << logQ1) - 1), sm = (1u << s) - 1;
    // offset of input j2: additive over the bits of t and of RB j
    auto ofs = [&](unsigned j2) { return (j2 >> s) + ((j2 & sm) << (logQ1 + logR1)); };
    const unsigned o = (c << (logM - logR2)) + (j1 << logR1) + ofs((unsigned)t);
    const float2 *src = in + o, *ct = ctab + o;
    float2 v[RA], h[RA];
#pragma unroll
    for (int j = 0; j < RA; ++j) v[j] = __ldg(src + ofs((unsigned)(RB * j)));
#pragma unroll
    for (int j = 0; j < RA; ++j) h[j] = __ldg(ct + ofs((unsigned)(RB * j)));
#pragma unroll
    for (int j = 0; j < RA; ++j) v[j] = cmul(v[j], h[j]);
    wide_dft<RA, true>(v);
    float2* dst = smem + (tid / RB) * WSTR + (RA + 1) * t;
#pragma unroll
    for (int j = 0; j < RA; ++j) dst[j] = v[j];
  }
  __syncthreads();
  const int b = tid & (NL - 1);
  const unsigned l = (unsigned)(l0 + b);
  float2* o = out + ((l >> logQ1) << logM) + (l & ((1u << logQ1) - 1));
#pragma unroll 1
  for (int u = 0; u < BPT; ++u) {
    const int t = (tid >> LOGNL) + u * (WIDE_NT / NL);
    WideTw<RA, RB> w2;
    w2.load(tw, t);
    const float2* src = smem + b * WSTR + t;
    float2 v[RB];
#pragma unroll
    for (int j = 0; j < RB; ++j) v[j] = src[j * (RA + 1)];
    w2.template dft<true>(v);
#pragma unroll
    for (int k = 0; k < RB; ++k) o[(unsigned)(t + RA * k) << logQ1] = v[k];
  }
}

// ---------------------------------------------------------------------------
// I2: inverse row FFTs, discard, detect, sum over sub-channels
// ---------------------------------------------------------------------------

// Row m2 of sub-channel c: elements j1 < Q1 at c M + m2 Q1 + j1, scaled by
// exp(+2 pi i j1 m2 / M) as they are loaded (factored as in F2f), inverse length-Q1
// transform, sample m2 + Q2 m1.  A CTA takes b2 rows m2 of every sub-channel (lines c b2 +
// bb).  In stage 2 a thread holds outputs m1 = t + 64 k of half of the lines: for
// each bb it sums |v|^2 over its half of the sub-channels in registers, the halves meet
// by shuffles, and the b2 Q1 powers go through shared memory so that neighbouring m
// are stored together.  One sub-channel: the halves take different rows.
// blockIdx.y is the segment.
template <int Q1, bool VOUT>
__global__ void __launch_bounds__(WIDE_NT, 2)
    k_inv_rows_w(const float2* __restrict__ buf, float* __restrict__ P, float2* __restrict__ vout, long long vstride,
                 long long vofs, int logQ2, int logM, int lognch, MSpan span, float scale,
                 const float2* __restrict__ tw3M, const float2* __restrict__ tw) {
  constexpr int RA = 64, RB = Q1 / 64, NL = TILE / Q1, LOGQ1 = ilog2c(Q1);
  constexpr int WSTR = wide_stride<RA, RB>();
  extern __shared__ float2 smem[];
  float2* st3 = smem;                         // [TW3_SN], w = exp(+2 pi i / M)
  float2* sm = st3 + TW3_SN;                  // [NL * WSTR]
  float* pw = reinterpret_cast<float*>(sm + NL * WSTR);   // [b2 Q1]
  buf += (size_t)blockIdx.y << (logM + lognch);
  P += (size_t)blockIdx.y << logM;
  const int m_lo = span.m_lo, m_hi = span.hi(blockIdx.y);
  const int tid = (int)threadIdx.x, logb2 = ilog2c(NL) - lognch, b2 = 1 << logb2, m2_0 = blockIdx.x << logb2;
  {
    const int line = tid / RB, t = tid % RB;
    const unsigned m2 = (unsigned)(m2_0 + (line & (b2 - 1)));
    const float2* src = buf + ((size_t)(line >> logb2) << logM) + ((size_t)m2 << LOGQ1) + t;
    float2 v[RA];
#pragma unroll
    for (int j = 0; j < RA; ++j) v[j] = __ldg(src + RB * j);
    load_tw3(st3, tw3M);
    __syncthreads();   // st3
    // j1 = t + RB (8 a + b): w^{8 RB m2 a} inside the first DFT, w^{m2 (t + RB b)} after it
    float2 wa[7], wb[8];
#pragma unroll
    for (int a = 1; a < 8; ++a) wa[a - 1] = tw3(st3, m2 * (unsigned)(8 * RB * a));
#pragma unroll
    for (int b = 0; b < 8; ++b) wb[b] = tw3(st3, m2 * (unsigned)(t + RB * b));
    wide_dft<RA, true>(
        v, [&](float2 x, int a) { return a == 0 ? x : cmul(x, wa[a - 1]); },
        [&](float2 x, int b, int ka) { return tw64<true>(cmul(x, wb[b]), b * ka); });
    float2* dst = sm + line * WSTR + (RA + 1) * t;
#pragma unroll
    for (int j = 0; j < RA; ++j) dst[j] = v[j];
  }
  const int t2 = (tid & 15) | ((tid >> 5) << 4), h = (tid >> 4) & 1;
  WideTw<RA, RB> w2;
  w2.load(tw, t2);
  __syncthreads();
  const float s2 = scale * scale;
  // lines of this half: sub-channels c0 .. c0 + nc - 1 of rows bb0 .. bb0 + nb - 1
  const int nc = lognch ? 1 << (lognch - 1) : 1, c0 = lognch ? h * nc : 0;
  const int nb = lognch ? b2 : b2 / 2, bb0 = lognch ? 0 : h * nb;
#pragma unroll 1
  for (int bb = bb0; bb < bb0 + nb; ++bb) {
    float p[RB];
#pragma unroll
    for (int k = 0; k < RB; ++k) p[k] = 0.f;
#pragma unroll 1
    for (int c = c0; c < c0 + nc; ++c) {
      const float2* src = sm + ((c << logb2) + bb) * WSTR + t2;
      float2 v[RB];
#pragma unroll
      for (int j = 0; j < RB; ++j) v[j] = src[j * (RA + 1)];
      w2.template dft<true>(v);
#pragma unroll
      for (int k = 0; k < RB; ++k) {
        p[k] = fmaf(v[k].y, v[k].y, fmaf(v[k].x, v[k].x, p[k]));
        if constexpr (VOUT) {
          const int m = m2_0 + bb + ((t2 + RA * k) << logQ2);
          if (m >= m_lo && m < m_hi) vout[(size_t)c * vstride + vofs + (m - m_lo)] = cscale(v[k], scale);
        }
      }
    }
    if (lognch) {
#pragma unroll
      for (int k = 0; k < RB / 2; ++k) {
        const float mine = h ? p[k + RB / 2] : p[k], other = h ? p[k] : p[k + RB / 2];
        const float q = mine + __shfl_xor_sync(0xffffffffu, other, 16);
        pw[((t2 + RA * (k + h * (RB / 2))) << logb2) + bb] = q * s2;
      }
    } else {
#pragma unroll
      for (int k = 0; k < RB; ++k) pw[((t2 + RA * k) << logb2) + bb] = p[k] * s2;
    }
  }
  __syncthreads();
  for (int i = tid; i < Q1 << logb2; i += WIDE_NT) {
    const int m = m2_0 + (i & (b2 - 1)) + ((i >> logb2) << logQ2);
    if (m >= m_lo && m < m_hi) P[m - m_lo] = pw[i];
  }
}

template <int Q1>
constexpr int inv_rows_w_smem(int lognch) {   // the table, the tile and its powers
  return TW3_BYTES + wide_smem_bytes<64, Q1 / 64>() + (TILE >> lognch) * (int)sizeof(float);
}


}  // namespace pond
