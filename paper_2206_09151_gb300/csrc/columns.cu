// Stage A's column stage for P <= 512: per spectrum column the forward FFT along v, the layer-independent
// weight, and for every layer the CTF filter and the inverse FFT.
//
// What bounds it is instruction issue (the filter's sine and reciprocal, the transform), so
// everything that a layer repeats is kept down:
//   - A thread holds 16 values as two 8-value parts, in the frequency domain m = j + s T and (T - j) + s T (T =
//     P/8): mirror images of each other, and the filter depends on m^2 only, so 9 filter values serve 16
//     spectrum values (the ninth is the Nyquist bin, which only j = 0 uses).
//   - A column's P/16 threads lie in one warp: the exchanges need no barrier beyond the warp's.
//   - In the other passes the parts are j and j + P/16, which share the middle pass's twiddles and have
//     addresses a constant apart.
//   - The phase is a 32-bit sum per layer (columns.cuh).
// 120 directions x 32 layers of 256 x 256 (P = 512): 970 us with 8 values per thread, a filter value for each
// and groups of two warps; 885 with the phase sums and 2 CTAs of up to 128 registers per SM instead of 3 of 80 (937
// with 3); 805 with the mirrored parts.  The pair filter's layers (swapped order, 60 directions x 32): 561, 470; two
// layers (200 directions of 200 x 200): 225, 218, but 257 with an amplitude and an angle per frequency, one cosine
// per layer, in place of the sine and the cosine (32 layers 461).
// Forming the exchange addresses again per layer, or reading one part after the other, trades the 27 registers that
// spill per layer for as many instructions: 1 to 9 % slower.
// The CTA's columns are consecutive in (direction, column), so that the last column (Nyquist) of a direction
// does not leave most of a CTA idle.
#include "columns.cuh"
#include "density.cuh"
#include "fft_reg.cuh"
#include "recon_internal.h"

namespace recon {
namespace {

template <int P>
struct ColsT {
  static constexpr int T = P / 8, TT = P / 16;  // parts and threads per column
  static constexpr int NTH = P >= 256 ? 256 : (P >= 64 ? P : 32);
  static constexpr int CB = NTH / TT;           // columns per CTA
  // entries between the columns' buffers: half-warps that span columns (TT < 16) and the fill, which runs over
  // the columns, find them on distinct banks
  static constexpr int L = P + (TT < 16 ? TT : (CB >= 16 ? 1 : 16 / CB));
  static constexpr int NT = fft::pass_table_len(P);
};

// The radix-R pass at sub-length Ns of part b: read (not for the first pass), twiddles, DFT ...
template <int P, int R, int Ns, bool INV>
__device__ __forceinline__ void part_load(float2 (&v)[8], const float2* buf, const float2* tw, int b) {
  constexpr int T = P / 8, NB = 8 / R, STRIDE = P / R;
#pragma unroll
  for (int q = 0; q < NB; ++q)
#pragma unroll
    for (int r = 0; r < R; ++r) v[q * R + r] = buf[fft::padded(b + q * T + r * STRIDE)];
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const float2* twk = tw + (Ns - 8) + ((b + q * T) & (Ns - 1)) * (R - 1) - 1;
#pragma unroll
    for (int r = 1; r < R; ++r) {
      float2 w = twk[r];
      if (INV) w.y = -w.y;
      v[q * R + r] = fft::cmul(v[q * R + r], w);
    }
    fft::dftR<R, INV>(v + q * R);
  }
}
// ... and write (not for the last pass).
template <int P, int R, int Ns>
__device__ __forceinline__ void part_store(const float2 (&v)[8], float2* buf, int b0) {
  constexpr int T = P / 8, NB = 8 / R;
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int b = b0 + q * T;
    const int base = (b / Ns) * Ns * R + (b & (Ns - 1));
#pragma unroll
    for (int r = 0; r < R; ++r) buf[fft::padded(base + r * Ns)] = v[q * R + r];
  }
}
// The passes from sub-length Ns on; the last one takes parts j and `last`, the others j and j + P/16.
template <int P, int Ns, bool INV>
__device__ __forceinline__ void passes(float2 (&a)[8], float2 (&b)[8], float2* buf, const float2* tw, int j, int last) {
  constexpr int rem = P / Ns, R = rem % 8 == 0 ? 8 : rem, NB = 8 / R;
  float2 va[8], vb[8];
  const int jb = Ns * R == P ? last : j + P / 16;
  __syncwarp();
  part_load<P, R, Ns, INV>(va, buf, tw, j);
  part_load<P, R, Ns, INV>(vb, buf, tw, jb);
  if constexpr (Ns * R == P) {
#pragma unroll
    for (int q = 0; q < NB; ++q)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        a[q + r * NB] = va[q * R + r];
        b[q + r * NB] = vb[q * R + r];
      }
  } else {
    __syncwarp();
    part_store<P, R, Ns>(va, buf, j);
    part_store<P, R, Ns>(vb, buf, jb);
    passes<P, Ns * R, INV>(a, b, buf, tw, j, last);
  }
}
// Length-P transform of the parts j and `first` (in a, b) into the parts j and `last`.
template <int P, bool INV>
__device__ __forceinline__ void transform(float2 (&a)[8], float2 (&b)[8], float2* buf, const float2* tw, int j,
                                          int first, int last) {
  fft::dft8<INV>(a);
  fft::dft8<INV>(b);
  __syncwarp();  // the last reads of the buffer
  part_store<P, 8, 1>(a, buf, j);
  part_store<P, 8, 1>(b, buf, first);
  passes<P, 8, INV>(a, b, buf, tw, j, last);
}

// FILT: 0 ramp only (filter off), 1 Tikhonov eps, 2 learned eps table, 3 the opposite-pair form of Eq. 10 /
// 11 (real part of the complex bracket at the image plane carried to the layer depth); DENS: density
// weighting (any geometry) instead of the ramp; BLEND: rows between two detector rows (c.b_frac != 0).
template <int P, int FILT, bool DENS, bool BLEND>
__global__ void __launch_bounds__(ColsT<P>::NTH, P >= 256 ? 2 : 4)
    k_cols(const float2* __restrict__ S, float2* __restrict__ T_out, const float2* __restrict__ twg,
           const uint64_t* __restrict__ uA, const float* __restrict__ ramp, const DirParams* __restrict__ dirs,
           const float* __restrict__ dens, const double* __restrict__ band_sum, const float* __restrict__ eps_tab,
           int n_bins, int bin_width, StageAConst c, int dir_begin, int cnt) {
  using C = ColsT<P>;
  constexpr int T = C::T, TT = C::TT, CB = C::CB, L = C::L;
  __shared__ float2 tw[C::NT];
  __shared__ float2 buf_all[CB * L];
  const int g = threadIdx.x / TT, j = threadIdx.x % TT;
  const int jb = j ? T - j : T / 2;  // the mirrored part; 0 and T / 2 are their own mirror images
  float2* buf = buf_all + g * L;
  for (int i = threadIdx.x; i < C::NT; i += C::NTH) tw[i] = twg[i];
  const int columns = cnt * c.half, first = blockIdx.x * CB;
  {  // coalesced fill of rows v < nv of the CTA's columns
    const int t = threadIdx.x % CB, f = min(first + t, columns - 1), n = f / c.half;
    const float2* Sc = S + (size_t)n * c.nv * c.half + (f - n * c.half);
    for (int v = threadIdx.x / CB; v < c.nv; v += C::NTH / CB) buf_all[t * L + fft::padded(v)] = Sc[(size_t)v * c.half];
  }
  const bool ok = first + g < columns;
  const int flat = ok ? first + g : columns - 1, n = flat / c.half, col = flat - n * c.half;
  __syncthreads();
  float2 ga[8], gb[8];  // the column's spectrum at m = j + s T and jb + s T, kept for all layers
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const int v = j + s * T;
    ga[s] = v < c.nv ? buf[fft::padded(v)] : make_float2(0.f, 0.f);
    gb[s] = v + TT < c.nv ? buf[fft::padded(v + TT)] : make_float2(0.f, 0.f);
  }
  transform<P, false>(ga, gb, buf, tw, j, j + TT, jb);

  {  // ramp (single-axis scans) or sampling-density weight (any geometry), 1/P^2 included, and with a
     // filter its prefactor lambda / (4 pi sqrt(1+sigma^2))
    const float pref = FILT != 0 ? c.pref : 1.f;
    const DirParams& dp = dirs[dir_begin + n];
    const float wr = DENS ? 0.f : ramp[col] * pref;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        float wv = wr;
        if constexpr (DENS) {
          const int m = (h ? jb : j) + s * T;
          const int mv = m < P / 2 ? m : m - P;
          wv = density_weight(c.dens, dens, band_sum, dp.af, dp.bf, (float)col, (float)mv);
          // the Nyquist bin is its own alias (+-P/2): mean over both, so that W stays even
          const bool nyq_u = col == P / 2, nyq_v = m == P / 2;
          if (nyq_u || nyq_v) {
            const float w2 = density_weight(c.dens, dens, band_sum, dp.af, dp.bf, nyq_u ? -(float)col : (float)col,
                                            (nyq_v && !nyq_u) ? -(float)mv : (float)mv);
            wv = 0.5f * (wv + w2);
          }
          wv *= pref;
        }
        float2& x = h ? gb[s] : ga[s];
        x = make_float2(x.x * wv, x.y * wv);
      }
  }
  // The filter values: slot i < 4 at m = j + i T, i < 8 at jb + (i - 4) T, 8 at P / 2.  chi/(2 pi) in 2^-32
  // turns needs only the top 32 bits of the 64-bit fixed-point sum: uA_k m is formed as hi(uA) m +
  // umulhi(lo(uA), m), and the layer-independent part uC m^2 - uW apart (dropped low-word carries cost at most
  // 2^-32 turns).
  constexpr int NF = FILT != 0 ? 9 : 1;
  const auto msq = [&](int i, int jj) {
    const int m = i < 4 ? jj + i * T : (i < 8 ? (jj ? T - jj : T / 2) + (i - 4) * T : P / 2);
    return (uint32_t)(col * col + m * m);
  };
  const auto base_hi = [&](uint64_t m) { return (uint32_t)((c.uC * (m * m) - c.uW) >> 32); };
  int bin[FILT == 2 ? 9 : 1];  // learned regulariser: the radial bin of each frequency (isqrt, exact integers)
  if constexpr (FILT == 2) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const uint32_t q2 = msq(i, j);
      int r = (int)sqrtf((float)q2);
      while ((uint32_t)r * (uint32_t)r > q2) --r;
      while ((uint32_t)(r + 1) * (uint32_t)(r + 1) <= q2) ++r;
      const int b = r / bin_width;
      bin[i] = b < n_bins - 1 ? b : n_bins - 1;
    }
  }
  // the opposite-pair filter keeps one constant more per direction: the image-plane phase constant after the
  // Nz per-layer depth constants
  const uint64_t* uAn = uA + (size_t)(dir_begin + n) * (c.nz_layers + (FILT == 3 ? 1 : 0));
  // The pair filter at a layer is Re{bracket exp(-i phi_k)} = sp cos phi_k - cp sin phi_k, phi_k = pi lambda z_k
  // q^2, of the image-plane sp = sin chi / (sin^2 chi + eps) and cp = cos chi / (cos^2 chi + eps).
  float sp[FILT == 3 ? 9 : 1], cp[FILT == 3 ? 9 : 1];
  if constexpr (FILT == 3) {
    const uint64_t uR = uAn[c.nz_layers];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      float sn, cs;
      sincos_half_turns((int32_t)(phase_of(uR, msq(i, j)) + base_hi(msq(i, j))), &sn, &cs);
      sp[i] = c.pair_mode == 0 ? __fdividef(sn, fmaf(sn, sn, c.eps)) : (c.pair_mode == 1 ? 1.f : 0.f);
      cp[i] = c.pair_mode == 0 ? __fdividef(cs, fmaf(cs, cs, c.eps)) : (c.pair_mode == 1 ? 0.f : -1.f);
    }
  }
  // this thread's rows w = v - r_lo of T, v = j + s TT (nv <= P/2: s < 8), stored where 0 <= w < nw
  float2* Tj = T_out + ((size_t)n * c.nz_layers * c.half + col) * c.tp + (BLEND ? 0 : j - c.r_lo);
  uint32_t keep = 0;
#pragma unroll
  for (int s = 0; s < 8; ++s) keep |= ok && (unsigned)(j + s * TT - c.r_lo) < (unsigned)c.nw ? 1u << s : 0u;
  asm volatile("" : "+r"(keep));  // one register, not eight predicates' inputs
  const int lg = (c.nz_layers + gridDim.y - 1) / gridDim.y;  // this CTA's layers: group blockIdx.y of equal groups
  const int k_begin = blockIdx.y * lg;
  const int k_end = min(c.nz_layers, k_begin + lg);
  const float eps0 = fmaxf(c.eps, FLT_MIN);  // Tikhonov eps
  uint32_t hi[NF], step[NF] = {};            // phase of the layer, per layer
  if (FILT != 0 && c.nz_layers > 1) {
    const uint64_t dA = uAn[1] - uAn[0];
#pragma unroll
    for (int i = 0; i < NF; ++i) step[i] = phase_step(dA, msq(i, j));
  }
  for (int kr = k_begin, kr_end; kr < k_end; kr = kr_end) {  // runs of kPhaseRun layers
    kr_end = min(k_end, kr - kr % kPhaseRun + kPhaseRun);
    if constexpr (FILT != 0) {
      const int k0 = kr - kr % kPhaseRun;
      int jj = j;  // formed again for each run, not kept in registers over the layers
      asm volatile("" : "+r"(jj));
      const uint64_t uA0 = uAn[k0];
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const uint32_t m = msq(i, jj);
        hi[i] = phase_of(uA0, m) + (FILT == 3 ? 0u : base_hi(m)) + (uint32_t)(kr - k0) * step[i];
      }
    }
    for (int k = kr; k < kr_end; ++k) {
      const float* eps_k = eps_tab + ((size_t)n * c.nz_layers + k) * n_bins;
      float2 a[8], b[8];
      if constexpr (FILT == 0) {
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          a[s] = ga[s];
          b[s] = gb[s];
        }
      } else {
        float f[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          if constexpr (FILT == 3) {
            float sn, cs;
            sincos_half_turns((int32_t)hi[i], &sn, &cs);
            f[i] = fmaf(sp[i], cs, -cp[i] * sn);
          } else {  // real part of the Eq. 11 bracket
            const float e = FILT == 2 ? positive_eps(__ldg(eps_k + bin[i])) : eps0;
            f[i] = inverse_ctf(sin_half_turns((int32_t)hi[i]), e);
          }
          hi[i] += step[i];
        }
        // the upper halves mirror the other part's lower half, those of parts 0 and T / 2 their own
        float ua[4], ub[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          ua[s] = j ? f[7 - s] : (s == 0 ? f[8] : f[4 - s]);
          ub[s] = j ? f[3 - s] : f[7 - s];
        }
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          const float fa = s < 4 ? f[s] : ua[s - 4], fb = s < 4 ? f[4 + s] : ub[s - 4];
          a[s] = make_float2(ga[s].x * fa, ga[s].y * fa);
          b[s] = make_float2(gb[s].x * fb, gb[s].y * fb);
        }
      }
      transform<P, true>(a, b, buf, tw, j, jb, j + TT);
      float2* out = Tj + (size_t)k * c.half * c.tp;
      if constexpr (!BLEND) {
        // rows v >= P/2 are never kept (their last butterflies drop)
#pragma unroll
        for (int s = 0; s < 8; ++s)
          if (keep >> s & 1u) out[s * TT] = s & 1 ? b[s / 2] : a[s / 2];
      } else {
        __syncwarp();  // the transform's last reads of the buffer
#pragma unroll
        for (int s = 0; s < 8; ++s) buf[fft::padded(j + s * TT)] = s & 1 ? b[s / 2] : a[s / 2];
        __syncwarp();
        if (ok) store_blended(buf, out, c, j, TT, [](int v) { return fft::padded(v); });
      }
    }
  }
}

template <int P, int FILT, bool DENS, bool BLEND>
cudaError_t launch(const StageAConst& c, const Workspace& ws, int d0, int cnt, cudaStream_t stream) {
  using C = ColsT<P>;
  const int groups = (int)(((long long)cnt * c.half + C::CB - 1) / C::CB);
  // set-up per layer group: the forward FFT (about a layer's work), and with the density weighting about one
  // more for the weights' trilinear lookups
  const int resident = (P >= 256 ? 2 : 4) * (256 / C::NTH > 4 ? 4 : 256 / C::NTH);
  const int lg = pick_layer_groups(groups, c.nz_layers, resident * device_sm_count(), DENS ? 2.2 : 1.2);
  k_cols<P, FILT, DENS, BLEND><<<dim3(groups, lg), C::NTH, 0, stream>>>(
      ws.S, ws.T, ws.twp, ws.uA, ws.ramp, ws.dirs, ws.dens, ws.band_sum, ws.eps, ws.n_bins, ws.bin_width, c, d0, cnt);
  return cudaGetLastError();
}
template <int P, int FILT>
cudaError_t launch(const StageAConst& c, const Workspace& ws, int d0, int cnt, cudaStream_t s) {
  if (c.b_frac != 0.f)
    return c.dens.enabled ? launch<P, FILT, true, true>(c, ws, d0, cnt, s) : launch<P, FILT, false, true>(c, ws, d0, cnt, s);
  return c.dens.enabled ? launch<P, FILT, true, false>(c, ws, d0, cnt, s) : launch<P, FILT, false, false>(c, ws, d0, cnt, s);
}
template <int P>
cudaError_t launch(const StageAConst& c, const Workspace& ws, int d0, int cnt, cudaStream_t s) {
  switch (c.filter) {
    case 0: return launch<P, 0>(c, ws, d0, cnt, s);
    case 2: return launch<P, 2>(c, ws, d0, cnt, s);
    case 3: return launch<P, 3>(c, ws, d0, cnt, s);
    default: return launch<P, 1>(c, ws, d0, cnt, s);
  }
}

}  // namespace

cudaError_t launch_columns(const StageAConst& c, const Workspace& ws, int dir_begin, int cnt, cudaStream_t s) {
  switch (c.P) {
    case 16: return launch<16>(c, ws, dir_begin, cnt, s);
    case 32: return launch<32>(c, ws, dir_begin, cnt, s);
    case 64: return launch<64>(c, ws, dir_begin, cnt, s);
    case 128: return launch<128>(c, ws, dir_begin, cnt, s);
    case 256: return launch<256>(c, ws, dir_begin, cnt, s);
    case 512: return launch<512>(c, ws, dir_begin, cnt, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace recon
