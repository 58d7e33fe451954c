// Passes whose line FFTs keep 64 values per thread (fft_wide.cuh).
#pragma once
#include "fft_wide.cuh"
#include "passes.cuh"

namespace pond {

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
                                                               long long vofs, int logG, int logJ, int m_lo, int m_hi,
                                                               float scale, const float2* __restrict__ tw,
                                                               TrialStride ts) {
  constexpr int RA = 64, RB = R2 / RA, NL = TILE / R2, BPT = 64 / RB;
  constexpr int WSTR = wide_stride<RA, RB>();
  extern __shared__ float2 smem[];
  __shared__ int s_last;
  // batched launches: blockIdx.y is the trial, with its own input, P, partials and tickets
  in += blockIdx.y * ts.in;
  P += blockIdx.y * ts.P;
  part += blockIdx.y * ts.part;
  cnt += blockIdx.y * ts.cnt;
  const int tid = (int)threadIdx.x;
  const int m1 = blockIdx.x >> logG, gi = blockIdx.x & ((1 << logG) - 1);
  const float2* blk = in + (size_t)blockIdx.x * TILE;   // block m1 G + g
  if (tid < 4) {
    // the block of CTA blockIdx.x + PF_DIST (in launch order, the next trial's
    // blocks after this trial's last), in four quarters
    const unsigned nx = gridDim.x, lin = blockIdx.y * nx + blockIdx.x + PF_DIST;
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
  for (int u = 0; u < BPT; ++u) {
    const int line = h * BPT + u;
    const float2* src = smem + line * WSTR + t2;
    float2 v[RB];
#pragma unroll
    for (int j = 0; j < RB; ++j) v[j] = src[j * (RA + 1)];
    w2.template dft<true>(v);
#pragma unroll
    for (int k = 0; k < RB; ++k) {
      const float q = u == 0 ? v[k].x * v[k].x : fmaf(v[k].x, v[k].x, p[k]);
      p[k] = fmaf(v[k].y, v[k].y, q);
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

// Shared memory of a tile of nl lines of RA x RB.
template <int RA, int RB>
constexpr int wide_smem_bytes() {
  return TILE / (RA * RB) * wide_stride<RA, RB>() * (int)sizeof(float2);
}

}  // namespace pond
