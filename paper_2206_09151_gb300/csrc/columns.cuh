// What the column kernels of stage A share (columns.cu for P <= 512, stage_a.cu for P >= 1024).
#pragma once

#include <cfloat>
#include <cmath>

#include "recon_internal.h"

namespace recon {

// sin(pi t) for t = hi * 2^-31 in [-1, 1) (hi: the top 32 bits of chi / (2 pi) in
// fixed point, so chi = pi t is already reduced to [-pi, pi) exactly by the integer
// phase).  The hardware sine (__sinf, maximum absolute error 2^-21.4 on [-pi, pi])
// measured faster than an odd polynomial after a quadrant fold, at 5.7e-7 instead of
// 5.2e-7 rel-L2 against the FP64 oracle on the 256^3 / 360-view scan.
__device__ __forceinline__ float sin_half_turns(int32_t hi) {
  return __sinf((float)hi * 1.4629180792671596e-09f);  // hi * 2 pi / 2^32
}

__device__ __forceinline__ float cos_half_turns(int32_t hi) { return __cosf((float)hi * 1.4629180792671596e-09f); }

// sin and cos of chi = pi t for t = hi * 2^-31 in [-1, 1) (hardware sine and cosine).
__device__ __forceinline__ void sincos_half_turns(int32_t hi, float* sn, float* cs) {
  __sincosf((float)hi * 1.4629180792671596e-09f, sn, cs);  // hi * 2 pi / 2^32
}

// The phase of a frequency m runs linearly over the layers (their depths are equidistant), so the
// layer loops add a 32-bit step per layer instead of forming uA_k m (a 32 x 64-bit product) each time:
// hi(k) = hi(k0) + (k - k0) step, k0 the multiple of kPhaseRun below k, whose hi is exact to 2^-32 turns.  The step is
// rounded to the nearest 2^-32 turns: at most kPhaseRun 2^-33 = 2^-27 turns of drift, 4.7e-8 rad, below the hardware
// sine's error of 2^-21.4 (runs of 8, 16 and 64 layers leave the same error against 64 bits, 1.5e-6 for a batch of
// uneven tomograms; 8 cost 3 to 5 % more time).  hi is a function of k alone, however the layers are split.
constexpr int kPhaseRun = 64;
__device__ __forceinline__ uint32_t phase_of(uint64_t uA, uint32_t m) {
  return (uint32_t)(uA >> 32) * m + __umulhi((uint32_t)uA, m);
}
__device__ __forceinline__ uint32_t phase_step(uint64_t dA, uint32_t m) {
  return (uint32_t)((dA * m + 0x80000000ull) >> 32);
}

// The learned eps, at least FLT_MIN; a NaN (of the network's weights) stays one, which fmaxf would hide.
__device__ __forceinline__ float positive_eps(float eps) {
  float e;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(e) : "f"(eps), "f"(FLT_MIN));
  return e;
}

// sn / (sn^2 + eps), eps >= FLT_MIN: one reciprocal (the general divide also scales for subnormal divisors).
__device__ __forceinline__ float inverse_ctf(float sn, float eps) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fmaf(sn, sn, eps)));
  return sn * r;
}

// Column stacks whose volume rows fall between two detector rows: row w is detector rows r_lo + w and
// the next blended, zero outside the detector (the blend commutes with the row transform, so it
// is done on the column's values, once per stack entry instead of once per voxel).
template <class Idx>
__device__ __forceinline__ void store_blended(const float2* buf, float2* out, const StageAConst& c, int j, int step,
                                              Idx idx) {
  for (int w = j; w < c.nw; w += step) {
    const int r = w + c.r_lo;
    const float2 a = r >= 0 && r < c.nv ? buf[idx(r)] : make_float2(0.f, 0.f);
    const float2 b = r + 1 >= 0 && r + 1 < c.nv ? buf[idx(r + 1)] : make_float2(0.f, 0.f);
    out[w] = make_float2(fmaf(c.b_frac, b.x - a.x, a.x), fmaf(c.b_frac, b.y - a.y, a.y));
  }
}

// Layer groups of the column stage: the split of the Nz layers over CTAs that keeps the
// last wave of `slots` resident CTAs fullest, counting the set-up each group repeats (the
// column's forward FFT and weights, `setup` layers' worth of work) as extra work.
inline int pick_layer_groups(int ctas_per_group, int nz_layers, int slots, double setup) {
  int best = 1;
  double best_eff = 0.0;
  const int max_lg = nz_layers / 2 > 0 ? (nz_layers / 2 < 16 ? nz_layers / 2 : 16) : 1;
  for (int lg = 1; lg <= max_lg; ++lg) {
    const double waves = (double)ctas_per_group * lg / slots;
    const double fill = waves / std::ceil(waves);
    const double eff = fill * (double)nz_layers / (nz_layers + setup * lg);
    if (eff > best_eff + 1e-9) {
      best_eff = eff;
      best = lg;
    }
  }
  return best;
}

}  // namespace recon
