// Stage A of the layered UTR path: contrast -> 2D DFT -> per-layer CTF inverse and
// ramp -> inverse 2D DFT -> cropped layer stack (Sec. 2, Eq. 4, 7, 11; ramp of Sec. 2).
//
// Three kernels per block of directions:
//   k_rows_fwd  two image rows packed as one complex row (real + i real), forward FFT,
//               split into the two half spectra                    -> S[n][v][0..P/2]
//   k_cols      (columns.cu for P <= 512, P/16 threads per spectrum column; k_cols16 here for the larger ones) the
//               forward FFT along v (rows >= nv are the zero padding), kept in registers; then for every
//               layer k: multiply by H_k(q) W(q_u), inverse FFT along v, store the stack's rows
//                                                                   -> T[n][k][col][v]
//   k_rows_inv  (rows_inv.cu) two rows of one layer: Hermitian-extend both half spectra, pack
//               as real + i real, inverse FFT, crop u < nu         -> the stack
// For P >= 16 the FFTs are register-resident mixed-radix Stockham transforms
// (fft_reg.cuh); tiny images (P <= 8) use a shared-memory radix-2 transform.
// The image sits at offset 0 of the P x P frame; by the shift invariance of the
// circular filters this equals any other placement with the same crop.
#include <cuda_bf16.h>

#include <cmath>

#include "columns.cuh"
#include "density.cuh"
#include "fft16.cuh"
#include "fft_reg.cuh"
#include "recon_internal.h"

namespace recon {
namespace {

using fft::cmul;
using fft::padded;

constexpr int kThreads = 256;

template <int P>
__host__ __device__ constexpr int groups_per_cta() {
  return kThreads / (P / 8) > 0 ? kThreads / (P / 8) : 1;
}

__device__ __forceinline__ float contrast_of(float x, int input_mode) {
  // RECON_INPUT_INTENSITY: g = ln(I/I_in), floored at 1e-6 (left side of Eq. 4)
  return input_mode == 0 ? logf(fmaxf(x, 1e-6f)) : x;
}

// sin(chi_k) from x = chi/(2 pi) modulo 1 in 64-bit fixed point.  The constants are
// fractions of a turn, so the products with the integer squared frequency m are exact
// modulo 2 pi: the range reduction of chi (hundreds of radians at the band edge) loses
// nothing, and the top 32 bits give chi in [-pi, pi) to 2^-31 turns.
__device__ __forceinline__ float sin_from_turns(uint64_t x) {
  const int32_t hi = (int32_t)(x >> 32);
  return sinpif((float)hi * 4.656612873077393e-10f);  // hi * 2^-31 = chi / pi in [-1, 1)
}

// The stack stores horizontal tap pairs: entry (row v + 1, column c) of a layer holds
// (Y[v][c - 1], Y[v][c]) for c in [0, nu], zero outside the image, so a bilinear row is
// one 8-byte (float32) or 4-byte (bfloat16) load.
template <typename PairT>
__device__ __forceinline__ PairT make_pair(float a, float b);
template <>
__device__ __forceinline__ float2 make_pair<float2>(float a, float b) { return make_float2(a, b); }
template <>
__device__ __forceinline__ __nv_bfloat162 make_pair<__nv_bfloat162>(float a, float b) {
  return __floats2bfloat162_rn(a, b);
}

// ------------------------------------------------------------------ register FFT kernels
template <int P>
__global__ void __launch_bounds__(kThreads) k_rows_fwd(const float* __restrict__ images, float2* __restrict__ S,
                                                        const float2* __restrict__ twg, StageAConst c,
                                                        int dir_begin) {
  constexpr int TT = P / 8, G = groups_per_cta<P>(), L = fft::buffer_len(P, G), NT = fft::pass_table_len(P);
  __shared__ float2 tw[NT];
  __shared__ float2 buf_all[G * L];
  const int g = threadIdx.x / TT, j = threadIdx.x % TT;
  float2* buf = buf_all + g * L;
  for (int i = threadIdx.x; i < NT; i += kThreads) tw[i] = twg[i];
  const int n = blockIdx.y;
  const int v0 = 2 * (blockIdx.x * G + g);
  const bool row1 = v0 < c.nv, row2 = v0 + 1 < c.nv;
  const float* im = images + (size_t)(dir_begin + n) * c.nu * c.nv;
  float2 x[8];
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const int u = j + s * TT;
    const bool in = u < c.nu;
    const float x1 = (row1 && in) ? contrast_of(im[(size_t)v0 * c.nu + u], c.input_mode) : 0.f;
    const float x2 = (row2 && in) ? contrast_of(im[(size_t)(v0 + 1) * c.nu + u], c.input_mode) : 0.f;
    x[s] = make_float2(x1, x2);
  }
  __syncthreads();
  fft::block_fft<P, false>(x, buf, tw, j);
  __syncthreads();
#pragma unroll
  for (int s = 0; s < 8; ++s) buf[padded(j + s * TT)] = x[s];
  __syncthreads();
  if (!row1) return;
  float2* s1 = S + ((size_t)n * c.nv + v0) * c.half;
  for (int m = j; m < c.half; m += TT) {
    const float2 zm = buf[padded(m & (P - 1))];
    const float2 zc = buf[padded((P - m) & (P - 1))];
    // X1 = (Z[m] + conj Z[P-m]) / 2,  X2 = (Z[m] - conj Z[P-m]) / (2i)
    s1[m] = make_float2(0.5f * (zm.x + zc.x), 0.5f * (zm.y - zc.y));
    if (row2) s1[c.half + m] = make_float2(0.5f * (zm.y + zc.y), -0.5f * (zm.x - zc.x));
  }
}

// ------------------------------------------------------------------ 16-value kernels (P >= 1024)
// The same column and row stages with the 16-value FFT of fft16.cuh: three passes and two
// exchanges per length-2048 transform instead of four and three, exchange addresses that
// are a per-thread base plus constants, and (in the column kernel) double-buffered
// exchanges, so two group barriers per transform instead of six.
constexpr int kThreads16 = 256;

template <int P>
__host__ __device__ constexpr int cols16_per_cta() {
  return kThreads16 / (P / 16);
}

// Column stage: a group of P/16 threads per spectrum column, cols16_per_cta columns per CTA.
// The forward FFT along v stays in registers, multiplied once by the column's weight (ramp
// or density weight, with the filter prefactor and 1/P^2); per layer: the CTF filter,
// inverse FFT, store v < nv.  ONE: one filtered layer, its phases formed where they are used: the sums' registers
// cost 8 % there (200 directions of 512 x 16: 481 us, 447 without, 436 before there were sums).
template <int P, int FILT, bool DENS, bool BLEND, bool ONE>
__global__ void __launch_bounds__(kThreads16, FILT == 3 ? 1 : 2) k_cols16(const float2* __restrict__ S, float2* __restrict__ T,
                                                          const float2* __restrict__ twg,
                                                          const uint64_t* __restrict__ uA,
                                                          const float* __restrict__ ramp,
                                                          const DirParams* __restrict__ dirs,
                                                          const float* __restrict__ dens,
                                                          const double* __restrict__ band_sum,
                                                          const float* __restrict__ eps_tab, int n_bins,
                                                          int bin_width, StageAConst c, int dir_begin) {
  constexpr int TT = P / 16, CB = cols16_per_cta<P>(), L = fft16::buffer_len(P), NT = fft16::table_len(P);
  extern __shared__ __align__(16) float2 smem16[];
  float2* tw = smem16;
  const int g = threadIdx.x / TT, j = threadIdx.x % TT;
  float2* buf0 = smem16 + NT + (2 * g) * L;
  float2* buf1 = buf0 + L;
  for (int i = threadIdx.x; i < NT; i += kThreads16) tw[i] = twg[i];
  const int n = blockIdx.y;
  const int col = blockIdx.x * CB + g;
  const bool ok = col < c.half;
  const int colc = ok ? col : c.half - 1;
  const float2* Sn = S + (size_t)n * c.nv * c.half;
  float2 xg[16];
#pragma unroll
  for (int s = 0; s < 16; ++s) {
    const int v = j + s * TT;
    xg[s] = v < c.nv ? Sn[(size_t)v * c.half + colc] : make_float2(0.f, 0.f);
  }
  __syncthreads();  // twiddle table
  const fft::GroupSync gsync{1 + g, TT};
  fft16::group_fft_db<P, false>(xg, buf0, buf1, tw, j, gsync);  // G(col, m_v) at m_v = j + s*TT
  // ramp (single-axis scans) or sampling-density weight (any geometry), 1/P^2 included, and
  // with a filter its prefactor lambda / (4 pi sqrt(1+sigma^2)): layer-independent, so
  // folded into the spectrum once
  {
    const float pref = FILT != 0 ? c.pref : 1.f;
    if constexpr (DENS) {
      const DirParams& dp = dirs[dir_begin + n];
#pragma unroll
      for (int s = 0; s < 16; ++s) {
        const int m = j + s * TT;
        const int mv = m < P / 2 ? m : m - P;
        float wv = density_weight(c.dens, dens, band_sum, dp.af, dp.bf, (float)colc, (float)mv);
        const bool nyq_u = colc == P / 2, nyq_v = m == P / 2;  // the Nyquist bin is its own alias
        if (nyq_u || nyq_v) {
          const float w2 = density_weight(c.dens, dens, band_sum, dp.af, dp.bf, nyq_u ? -(float)colc : (float)colc,
                                          (nyq_v && !nyq_u) ? -(float)mv : (float)mv);
          wv = 0.5f * (wv + w2);
        }
        wv *= pref;
        xg[s] = make_float2(xg[s].x * wv, xg[s].y * wv);
      }
    } else {
      const float wv = ramp[colc] * pref;
#pragma unroll
      for (int s = 0; s < 16; ++s) xg[s] = make_float2(xg[s].x * wv, xg[s].y * wv);
    }
  }
  // chi/(2 pi) in 2^-32 turns, as in k_cols
  const auto msq = [&](int s, int jj) {
    const int m = jj + s * TT;
    const int mv = m < P / 2 ? m : m - P;
    return (uint32_t)(colc * colc + mv * mv);
  };
  const auto base_hi = [&](uint64_t m) { return (uint32_t)((c.uC * (m * m) - c.uW) >> 32); };
  uint32_t bins[FILT == 2 ? 4 : 1];  // radial bins (exact isqrt, at most 256 of them), four to a word
  if constexpr (FILT == 2) {
#pragma unroll
    for (int s = 0; s < 16; ++s) {
      const uint32_t q2 = msq(s, j);
      int r = (int)sqrtf((float)q2);
      while ((uint32_t)r * (uint32_t)r > q2) --r;
      while ((uint32_t)(r + 1) * (uint32_t)(r + 1) <= q2) ++r;
      const uint32_t b = (uint32_t)min(r / bin_width, n_bins - 1);
      bins[s / 4] = s % 4 ? bins[s / 4] | b << 8 * (s % 4) : b;
    }
  }
  const uint64_t* uAn = uA + (size_t)(dir_begin + n) * (c.nz_layers + (FILT == 3 ? 1 : 0));
  float sp[FILT == 3 ? 16 : 1], cp[FILT == 3 ? 16 : 1];
  if constexpr (FILT == 3) {  // image-plane sin chi / (sin^2 chi + eps), cos chi / (cos^2 chi + eps)
    const uint64_t uR = uAn[c.nz_layers];
#pragma unroll
    for (int s = 0; s < 16; ++s) {
      float sn, cs;
      sincos_half_turns((int32_t)(phase_of(uR, msq(s, j)) + base_hi(msq(s, j))), &sn, &cs);
      sp[s] = c.pair_mode == 0 ? __fdividef(sn, fmaf(sn, sn, c.eps)) : (c.pair_mode == 1 ? 1.f : 0.f);
      cp[s] = c.pair_mode == 0 ? __fdividef(cs, fmaf(cs, cs, c.eps)) : (c.pair_mode == 1 ? 0.f : -1.f);
    }
  }
  // this thread's rows w = j + s TT - r_lo of T (s < 8: nv <= P/2, P being at least twice the image
  // size), stored where 0 <= w < nw
  float2* Tj = T + ((size_t)n * c.nz_layers * c.half + col) * c.tp + (BLEND ? 0 : j - c.r_lo);
  bool keep[8];
#pragma unroll
  for (int s = 0; s < 8; ++s) keep[s] = ok && (unsigned)(j + s * TT - c.r_lo) < (unsigned)c.nw;
  const int lg = (c.nz_layers + gridDim.z - 1) / gridDim.z;
  const int k_begin = blockIdx.z * lg;
  const int k_end = min(c.nz_layers, k_begin + lg);
  constexpr int NF = FILT != 0 && !ONE ? 16 : 1;
  uint32_t hi[NF], step[NF];  // phase of the layer, per layer
  const float eps0 = fmaxf(c.eps, FLT_MIN);                   // Tikhonov eps
  for (int kr = k_begin, kr_end; kr < k_end; kr = kr_end) {  // runs of kPhaseRun layers
    kr_end = min(k_end, kr - kr % kPhaseRun + kPhaseRun);
    if constexpr (FILT != 0 && !ONE) {
      const int k0 = kr - kr % kPhaseRun;
      int jj = j;  // formed again for each run, not kept in registers over the layers
      asm volatile("" : "+r"(jj));
      const uint64_t uA0 = uAn[k0], dA = k0 + 1 < c.nz_layers ? uAn[k0 + 1] - uA0 : 0;
#pragma unroll
      for (int s = 0; s < 16; ++s) {
        const uint32_t m = msq(s, jj);
        step[s] = phase_step(dA, m);
        hi[s] = phase_of(uA0, m) + (FILT == 3 ? 0 : base_hi(m)) + (uint32_t)(kr - k0) * step[s];
      }
    }
    for (int k = kr; k < kr_end; ++k) {
      const float* eps_k = eps_tab + ((size_t)n * c.nz_layers + k) * n_bins;
      float2 x[16];
#pragma unroll
      for (int s = 0; s < 16; ++s) {
        if constexpr (FILT == 0) {
          x[s] = xg[s];
        } else {
          float f;
          uint32_t h;
          if constexpr (ONE) {
            h = phase_of(uAn[0], msq(s, j)) + (FILT == 3 ? 0 : base_hi(msq(s, j)));
          } else {
            h = hi[s];
            hi[s] += step[s];
          }
          if constexpr (FILT == 3) {  // Re{bracket * exp(-i phi_k)}, phi_k = pi lambda z_k q^2
            float sn, cs;
            sincos_half_turns((int32_t)h, &sn, &cs);
            f = fmaf(sp[s], cs, -cp[s] * sn);
          } else {  // real part of the Eq. 11 bracket
            const float e = FILT == 2 ? positive_eps(__ldg(eps_k + (bins[s / 4] >> 8 * (s % 4) & 255u))) : eps0;
            f = inverse_ctf(sin_half_turns((int32_t)h), e);
          }
          x[s] = make_float2(xg[s].x * f, xg[s].y * f);
        }
      }
      fft16::group_fft_db<P, true>(x, buf0, buf1, tw, j, gsync);
      float2* out = Tj + (size_t)k * c.half * c.tp;
      if constexpr (!BLEND) {
        // elements s >= 8 (v >= P/2) are never kept, so the last pass's butterflies that only feed them are
        // dropped
#pragma unroll
        for (int s = 0; s < 8; ++s)
          if (keep[s]) out[s * TT] = x[s];
      } else {
        // the transform's second pass, before its last barrier, was the last to read buf0
#pragma unroll
        for (int s = 0; s < 8; ++s) buf0[fft16::pad(j + s * TT)] = x[s];
        gsync();
        if (ok) store_blended(buf0, out, c, j, TT, [](int v) { return fft16::pad(v); });
        gsync();  // the next transform's first pass writes buf0
      }
    }
  }
}

template <int P>
constexpr size_t cols16_smem() {
  return sizeof(float2) * ((size_t)fft16::table_len(P) + 2 * (size_t)cols16_per_cta<P>() * fft16::buffer_len(P));
}

// ------------------------------------------------------------------ radix-2 fallback (P <= 8)
__device__ __forceinline__ int bitrev(int i, int logP) { return (int)(__brev((unsigned)i) >> (32 - logP)); }

template <bool INV>
__device__ void fft_radix2(float2* data, int P, int logP, const float2* tw) {
  const int halfP = P >> 1;
  for (int s = 0; s < logP; ++s) {
    const int half = 1 << s;
    const int tw_shift = logP - 1 - s;
    __syncthreads();
    for (int jj = threadIdx.x; jj < halfP; jj += blockDim.x) {
      const int pos = jj & (half - 1);
      const int i1 = ((jj - pos) << 1) + pos;
      float2 w = tw[pos << tw_shift];
      if (INV) w.y = -w.y;
      const float2 a = data[i1];
      const float2 wb = cmul(w, data[i1 + half]);
      data[i1] = make_float2(a.x + wb.x, a.y + wb.y);
      data[i1 + half] = make_float2(a.x - wb.x, a.y - wb.y);
    }
  }
  __syncthreads();
}

__global__ void k_small_rows_fwd(const float* __restrict__ images, float2* __restrict__ S,
                                 const float2* __restrict__ twg, StageAConst c, int dir_begin) {
  __shared__ float2 tw[8];
  __shared__ float2 z[8];
  const int n = blockIdx.y;
  const int v0 = blockIdx.x * 2;
  const bool two = v0 + 1 < c.nv;
  const float* im = images + (size_t)(dir_begin + n) * c.nu * c.nv;
  for (int i = threadIdx.x; i < c.P; i += blockDim.x) tw[i] = twg[i];
  for (int i = threadIdx.x; i < c.P; i += blockDim.x) {
    float x1 = 0.f, x2 = 0.f;
    if (i < c.nu) {
      x1 = contrast_of(im[(size_t)v0 * c.nu + i], c.input_mode);
      if (two) x2 = contrast_of(im[(size_t)(v0 + 1) * c.nu + i], c.input_mode);
    }
    z[bitrev(i, c.logP)] = make_float2(x1, x2);
  }
  fft_radix2<false>(z, c.P, c.logP, tw);
  float2* s1 = S + ((size_t)n * c.nv + v0) * c.half;
  for (int m = threadIdx.x; m < c.half; m += blockDim.x) {
    const float2 zm = z[m & (c.P - 1)];
    const float2 zc = z[(c.P - m) & (c.P - 1)];
    s1[m] = make_float2(0.5f * (zm.x + zc.x), 0.5f * (zm.y - zc.y));
    if (two) s1[c.half + m] = make_float2(0.5f * (zm.y + zc.y), -0.5f * (zm.x - zc.x));
  }
}

__global__ void k_small_cols(const float2* __restrict__ S, float2* __restrict__ T, const float2* __restrict__ twg,
                             const uint64_t* __restrict__ uA, const float* __restrict__ ramp,
                             const DirParams* __restrict__ dirs, const float* __restrict__ dens,
                             const double* __restrict__ band_sum, const float* __restrict__ eps_tab, int n_bins,
                             int bin_width, StageAConst c, int dir_begin) {
  __shared__ float2 tw[8];
  __shared__ float2 G[8];
  __shared__ float2 Wk[8];
  const int n = blockIdx.y;
  const int col = blockIdx.x;  // one column per CTA
  for (int i = threadIdx.x; i < c.P; i += blockDim.x) tw[i] = twg[i];
  const float2* Sn = S + (size_t)n * c.nv * c.half;
  for (int v = threadIdx.x; v < c.P; v += blockDim.x)
    G[bitrev(v, c.logP)] = v < c.nv ? Sn[(size_t)v * c.half + col] : make_float2(0.f, 0.f);
  fft_radix2<false>(G, c.P, c.logP, tw);
  const uint64_t* uAn = uA + (size_t)(dir_begin + n) * (c.nz_layers + (c.filter == 3 ? 1 : 0));
  const int hP = c.P >> 1;
  for (int k = 0; k < c.nz_layers; ++k) {
    for (int m = threadIdx.x; m < c.P; m += blockDim.x) {
      const int mv = m < (c.P >> 1) ? m : m - c.P;
      const uint64_t msq = (uint64_t)(col * col + mv * mv);
      float f = ramp[col];
      if (c.dens.enabled) {
        const DirParams& dp = dirs[dir_begin + n];
        f = density_weight(c.dens, dens, band_sum, dp.af, dp.bf, (float)col, (float)mv);
        const bool nyq_u = col == hP, nyq_v = m == hP;  // the Nyquist bin is its own alias
        if (nyq_u || nyq_v)
          f = 0.5f * (f + density_weight(c.dens, dens, band_sum, dp.af, dp.bf, nyq_u ? -(float)col : (float)col,
                                         (nyq_v && !nyq_u) ? -(float)mv : (float)mv));
      }
      if (c.filter == 3) {  // opposite-pair filter: image-plane chi, depth phase of layer k
        float sn, cs, sz, cz;
        sincos_half_turns((int32_t)((uAn[c.nz_layers] * msq + c.uC * (msq * msq) - c.uW) >> 32), &sn, &cs);
        sincos_half_turns((int32_t)((uAn[k] * msq) >> 32), &sz, &cz);
        const float sp = c.pair_mode == 0 ? __fdividef(sn, fmaf(sn, sn, c.eps)) : (c.pair_mode == 1 ? 1.f : 0.f);
        const float cp = c.pair_mode == 0 ? __fdividef(cs, fmaf(cs, cs, c.eps)) : (c.pair_mode == 1 ? 0.f : -1.f);
        f *= c.pref * (sp * cz - cp * sz);
      } else if (c.filter) {
        const float sn = sin_from_turns(uAn[k] * msq + c.uC * (msq * msq) - c.uW);
        float e = c.eps;
        if (c.filter == 2) {
          int r = 0;
          while ((uint64_t)(r + 1) * (uint64_t)(r + 1) <= msq) ++r;
          const int b = r / bin_width;
          e = eps_tab[((size_t)n * c.nz_layers + k) * n_bins + (b < n_bins - 1 ? b : n_bins - 1)];
        }
        f *= c.pref * __fdividef(sn, fmaf(sn, sn, e));
      }
      Wk[bitrev(m, c.logP)] = make_float2(G[m].x * f, G[m].y * f);
    }
    fft_radix2<true>(Wk, c.P, c.logP, tw);
    float2* out = T + (((size_t)n * c.nz_layers + k) * c.half + col) * c.nv;
    for (int v = threadIdx.x; v < c.nv; v += blockDim.x) out[v] = Wk[v];
    __syncthreads();
  }
}

template <typename PairT>
__global__ void k_small_rows_inv(const float2* __restrict__ T, PairT* __restrict__ stack,
                                 const float2* __restrict__ twg, StageAConst c) {
  __shared__ float2 tw[8];
  __shared__ float2 z[8];
  const int n = blockIdx.z, k = blockIdx.y;
  const int v0 = blockIdx.x * 2;
  const bool two = v0 + 1 < c.nv;
  for (int i = threadIdx.x; i < c.P; i += blockDim.x) tw[i] = twg[i];
  const float2* Tk = T + ((size_t)n * c.nz_layers + k) * c.half * c.nv;
  const int hP = c.P >> 1;
  for (int m = threadIdx.x; m < c.P; m += blockDim.x) {
    const int mm = m <= hP ? m : c.P - m;
    float2 a = Tk[(size_t)mm * c.nv + v0];
    float2 b = two ? Tk[(size_t)mm * c.nv + v0 + 1] : make_float2(0.f, 0.f);
    if (m == 0 || m == hP) {
      a.y = 0.f;
      b.y = 0.f;
    } else if (m > hP) {
      a.y = -a.y;
      b.y = -b.y;
    }
    z[bitrev(m, c.logP)] = make_float2(a.x - b.y, a.y + b.x);
  }
  fft_radix2<true>(z, c.P, c.logP, tw);
  PairT* L = stack + ((size_t)n * c.nz_layers + k) * c.layer_elems;
  const int sp = c.su;
  for (int cc = threadIdx.x; cc <= c.nu; cc += blockDim.x) {
    const float2 left = cc >= 1 ? z[cc - 1] : make_float2(0.f, 0.f);
    const float2 right = cc < c.nu ? z[cc] : make_float2(0.f, 0.f);
    L[(size_t)(v0 + 1) * sp + cc] = make_pair<PairT>(left.x, right.x);
    if (two) L[(size_t)(v0 + 2) * sp + cc] = make_pair<PairT>(left.y, right.y);
    if (v0 == 0) L[cc] = make_pair<PairT>(0.f, 0.f);
    if (v0 + 2 >= c.nv) L[(size_t)(c.nv + 1) * sp + cc] = make_pair<PairT>(0.f, 0.f);
  }
}

// ------------------------------------------------------------------ finiteness scan
__global__ void k_count_nonfinite(const float* __restrict__ x, size_t n, unsigned int* __restrict__ count) {
  unsigned int bad = 0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    bad += isfinite(x[i]) ? 0u : 1u;
  for (int o = 16; o > 0; o >>= 1) bad += __shfl_down_sync(0xffffffffu, bad, o);
  if ((threadIdx.x & 31) == 0 && bad) atomicAdd(count, bad);
}

// ------------------------------------------------------------------ launch
template <int P, int FILT, bool DENS, bool BLEND, bool ONE>
cudaError_t launch_cols16_t(const StageAConst& c, const Workspace& ws, const float2* twq, int d0, int cnt, int sms,
                          cudaStream_t stream) {
  constexpr size_t smem = cols16_smem<P>();
  static unsigned long long attr_set = 0;  // devices on which the shared-memory limit is raised
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 64 || !(attr_set >> dev & 1ull)) {
    const cudaError_t e =
        cudaFuncSetAttribute(k_cols16<P, FILT, DENS, BLEND, ONE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (dev < 64) attr_set |= 1ull << dev;
  }
  constexpr int CB = cols16_per_cta<P>();
  const int col_groups = (c.half + CB - 1) / CB;
  // set-up per group: the forward FFT (about one layer's work), and with the density
  // weighting about one more for the weights' trilinear lookups
  const int lg = pick_layer_groups(col_groups * cnt, c.nz_layers, (FILT == 3 ? 1 : 2) * sms, DENS ? 2.2 : 1.2);
  k_cols16<P, FILT, DENS, BLEND, ONE><<<dim3(col_groups, cnt, lg), kThreads16, smem, stream>>>(
      ws.S, ws.T, twq, ws.uA, ws.ramp, ws.dirs, ws.dens, ws.band_sum, ws.eps, ws.n_bins, ws.bin_width, c, d0);
  return cudaGetLastError();
}

template <int P, int FILT, bool DENS, bool BLEND>
cudaError_t launch_cols16(const StageAConst& c, const Workspace& ws, const float2* twq, int d0, int cnt, int sms,
                          cudaStream_t stream) {
  if constexpr (FILT != 0 && !DENS)
    if (c.nz_layers == 1) return launch_cols16_t<P, FILT, DENS, BLEND, true>(c, ws, twq, d0, cnt, sms, stream);
  return launch_cols16_t<P, FILT, DENS, BLEND, false>(c, ws, twq, d0, cnt, sms, stream);
}

// The row stage of one sub-block into the stacks from direction s0 of the block on.
cudaError_t launch_rows(const StageAConst& c, const Workspace& ws, int s0, int cnt, cudaStream_t stream) {
  const size_t entry = c.cols ? (c.stack_bf16 ? 2 : 4) : (c.stack_bf16 ? 4 : 8);
  const size_t layer = c.cols ? (size_t)c.nu * c.wp : (size_t)c.layer_elems;
  return launch_rows_inv(c, ws.T, (char*)ws.stack + (size_t)s0 * c.nz_layers * layer * entry, ws.twp, cnt, stream);
}

template <int P>
cudaError_t launch_reg(const StageAConst& c, const Workspace& ws, const float* images, int dir_begin, int dir_count,
                       cudaStream_t stream, EventRecorder* rec, const StageAHook* hook) {
  constexpr int G = groups_per_cta<P>();
  // Sub-blocks of c.sub_block directions: S and T of one sub-block stay in L2 between the
  // column and the row kernels; each sub-block writes its part of the block's stack.
  const int sub = c.sub_block > 0 ? c.sub_block : dir_count;
  const int sms = device_sm_count();
  for (int s0 = 0; s0 < dir_count; s0 += sub) {
    const int cnt = min(sub, dir_count - s0);
    const int d0 = dir_begin + s0;
    k_rows_fwd<P><<<dim3((c.nv + 2 * G - 1) / (2 * G), cnt), kThreads, 0, stream>>>(images, ws.S, ws.twp, c, d0);
    if (hook) {
      const cudaError_t e = hook->fn(hook->ctx, d0, cnt, stream);
      if (e != cudaSuccess) return e;
    }
    if (rec) rec->mark(0, stream);
    const bool dens = c.dens.enabled != 0;
    if constexpr (P >= 1024) {
      // 16-value FFTs (fft16.cuh); their twiddle table follows the 8-value one
      const float2* twq = ws.twp + (P - 8);
      cudaError_t e;
#define RECON_K_COLS16(F)                                                                                       \
  (dens ? (c.b_frac != 0.f ? launch_cols16<P, F, true, true>(c, ws, twq, d0, cnt, sms, stream)                   \
                           : launch_cols16<P, F, true, false>(c, ws, twq, d0, cnt, sms, stream))                 \
        : (c.b_frac != 0.f ? launch_cols16<P, F, false, true>(c, ws, twq, d0, cnt, sms, stream)                  \
                           : launch_cols16<P, F, false, false>(c, ws, twq, d0, cnt, sms, stream)))
      e = c.filter == 0 ? RECON_K_COLS16(0)
                        : (c.filter == 3 ? RECON_K_COLS16(3) : (c.filter == 2 ? RECON_K_COLS16(2) : RECON_K_COLS16(1)));
#undef RECON_K_COLS16
      if (e != cudaSuccess) return e;
    } else {
      const cudaError_t e = launch_columns(c, ws, d0, cnt, stream);
      if (e != cudaSuccess) return e;
    }
    if (rec) rec->mark(1, stream);
    const cudaError_t e = launch_rows(c, ws, s0, cnt, stream);
    if (e != cudaSuccess) return e;
    if (rec) rec->mark(2, stream);
  }
  return cudaGetLastError();
}

template <int P>
cudaError_t rows_fwd_only(const StageAConst& c, float2* S, const float2* twp, const float* images, int first,
                          int count, cudaStream_t stream) {
  constexpr int G = groups_per_cta<P>();
  k_rows_fwd<P><<<dim3((c.nv + 2 * G - 1) / (2 * G), count), kThreads, 0, stream>>>(images, S, twp, c, first);
  return cudaGetLastError();
}

cudaError_t launch_small(const StageAConst& c, const Workspace& ws, const float* images, int dir_begin,
                         int dir_count, cudaStream_t stream, EventRecorder* rec) {
  k_small_rows_fwd<<<dim3((c.nv + 1) / 2, dir_count), 32, 0, stream>>>(images, ws.S, ws.tw, c, dir_begin);
  if (rec) rec->mark(0, stream);
  k_small_cols<<<dim3(c.half, dir_count), 32, 0, stream>>>(ws.S, ws.T, ws.tw, ws.uA, ws.ramp, ws.dirs, ws.dens,
                                                          ws.band_sum, ws.eps, ws.n_bins, ws.bin_width, c,
                                                          dir_begin);
  if (rec) rec->mark(1, stream);
  const dim3 gi((c.nv + 1) / 2, c.nz_layers, dir_count);
  if (c.stack_bf16)
    k_small_rows_inv<__nv_bfloat162><<<gi, 32, 0, stream>>>(ws.T, (__nv_bfloat162*)ws.stack, ws.tw, c);
  else
    k_small_rows_inv<float2><<<gi, 32, 0, stream>>>(ws.T, (float2*)ws.stack, ws.tw, c);
  if (rec) rec->mark(2, stream);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_stage_a(const StageAConst& c, const Workspace& ws, const float* images, int dir_begin,
                           int dir_count, cudaStream_t stream, EventRecorder* ev, const StageAHook* hook) {
  if (dir_count <= 0) return cudaSuccess;
  switch (c.P) {
    case 16: return launch_reg<16>(c, ws, images, dir_begin, dir_count, stream, ev, hook);
    case 32: return launch_reg<32>(c, ws, images, dir_begin, dir_count, stream, ev, hook);
    case 64: return launch_reg<64>(c, ws, images, dir_begin, dir_count, stream, ev, hook);
    case 128: return launch_reg<128>(c, ws, images, dir_begin, dir_count, stream, ev, hook);
    case 256: return launch_reg<256>(c, ws, images, dir_begin, dir_count, stream, ev, hook);
    case 512: return launch_reg<512>(c, ws, images, dir_begin, dir_count, stream, ev, hook);
    case 1024: return launch_reg<1024>(c, ws, images, dir_begin, dir_count, stream, ev, hook);
    case 2048: return launch_reg<2048>(c, ws, images, dir_begin, dir_count, stream, ev, hook);
    default: return hook ? cudaErrorInvalidValue : launch_small(c, ws, images, dir_begin, dir_count, stream, ev);
  }
}

cudaError_t launch_count_nonfinite(const float* x, size_t n, unsigned int* count, cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  const size_t want = (n + 255) / 256;
  const size_t cap = (size_t)device_sm_count() * 8;
  k_count_nonfinite<<<(unsigned)(want < cap ? want : cap), 256, 0, stream>>>(x, n, count);
  return cudaGetLastError();
}

cudaError_t launch_rows_fwd(const StageAConst& c, float2* S, const float2* twp, const float* images, int first,
                            int count, cudaStream_t stream) {
  if (count <= 0) return cudaSuccess;
  switch (c.P) {
    case 16: return rows_fwd_only<16>(c, S, twp, images, first, count, stream);
    case 32: return rows_fwd_only<32>(c, S, twp, images, first, count, stream);
    case 64: return rows_fwd_only<64>(c, S, twp, images, first, count, stream);
    case 128: return rows_fwd_only<128>(c, S, twp, images, first, count, stream);
    case 256: return rows_fwd_only<256>(c, S, twp, images, first, count, stream);
    case 512: return rows_fwd_only<512>(c, S, twp, images, first, count, stream);
    case 1024: return rows_fwd_only<1024>(c, S, twp, images, first, count, stream);
    case 2048: return rows_fwd_only<2048>(c, S, twp, images, first, count, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace recon
