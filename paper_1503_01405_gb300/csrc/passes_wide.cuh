// Passes whose line FFTs keep 64 values per thread (fft_wide.cuh).
#pragma once
#include "fft_wide.cuh"
#include "passes.cuh"

namespace pond {

// L2 prefetch distance (CTAs) of these passes, three CTAs per SM.  Batched
// chunk of 128 trials / full-rate stream, ms: 38: 104.3 / 15.98, 114: 103.3 /
// 15.97, 228: 103.5 / 16.09, 456: 105.4 / 16.34, none: 116.6 / 16.40.
constexpr int WIDE_PF = 114;

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
  WideTw<RA, RB> w2;
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

// e^{2 pi i k2 m1 / M} = conj(w^{k2 m1 NCH}), k2 m1 NCH < L, of rows row_of(0 .. nl-1).
template <int R1, class RowOf>
__device__ __forceinline__ void make_twk(float2* twk, const float2* st3, int nl, RowOf row_of) {
  for (int i = threadIdx.x; i < nl * 64; i += blockDim.x) {
    const unsigned k2 = (unsigned)row_of(i >> 6), m1 = (unsigned)(i & 63);
    twk[(i >> 6) * TWK_STR + m1] = cconj(tw3(st3, (k2 * m1) << ilog2c(R1 / 64)));
  }
}

// Table form: the rows and their Q0.32 table words resident for every trial of the launch.
// Four warps run a trial of the tile, GROUPS trials at a time; a run is read from the
// resident copies and stored from registers, so there is no exchange and no
// barrier after the tile's load.  Bound by the issue slots (chirp and DFT, 34
// instructions per value) next to the 64 MiB that each trial writes (4.8 TB/s).
// Full-rate batched plan: 19.9 us per trial with the runs split over four lanes
// and exchanged through shared memory (78 % of that pipe), 13.5 here; the 8 s
// chunk of 128 trials 126 -> 103 ms.
constexpr int TAB_GROUPS = 3;   // 384 threads of 168 registers: one CTA per SM

template <int R1>
__global__ void __launch_bounds__(TAB_GROUPS * WIDE_NT, 1)
    k_inv_rows_table(const float2* __restrict__ in, float2* __restrict__ out, long long out_tstride, RowTile rt,
                     const float2* __restrict__ tw3L, MultiChirp mc, int ntr) {
  constexpr int NLR = run_slots<R1>(), LOGR1 = ilog2c(R1);
  extern __shared__ float2 smem[];
  float2* st3 = smem;                                       // [TW3_SN], w = exp(-2 pi i / L)
  float2* twk = st3 + TW3_SN;                               // [NLR][TWK_STR]
  float2* rows = twk + NLR * TWK_STR + (NLR * TWK_STR & 1); // [NLR * rstr]
  unsigned* tabw = reinterpret_cast<unsigned*>(rows + NLR * rt.rstr);
  const int r0 = blockIdx.x * NLR;
  load_tw3(st3, tw3L);
  const float2* src = in + ((size_t)r0 << LOGR1);
  const unsigned* tsrc = mc.atab + ((size_t)r0 << LOGR1);
#pragma unroll 8
  for (int i = threadIdx.x; i < TILE; i += TAB_GROUPS * WIDE_NT) {
    const int slot = i >> LOGR1, k1 = i & (R1 - 1), o = k1 + (k1 >> 6);
    rows[slot * rt.rstr + o] = __ldg(src + i);
    tabw[slot * rt.tstr + o] = __ldg(tsrc + i);
  }
  __syncthreads();   // st3
  make_twk<R1>(twk, st3, NLR, [&](int slot) { return r0 + slot; });
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
  return (size_t)(TW3_SN + NLR * TWK_STR + (NLR * TWK_STR & 1) + NLR * rt.rstr) * sizeof(float2) +
         (size_t)NLR * rt.tstr * sizeof(unsigned);
}

// Shared memory of a tile of nl lines of RA x RB.
template <int RA, int RB>
constexpr int wide_smem_bytes() {
  return TILE / (RA * RB) * wide_stride<RA, RB>() * (int)sizeof(float2);
}

}  // namespace pond
