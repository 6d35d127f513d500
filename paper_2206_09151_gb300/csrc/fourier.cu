// The method's two 3D-Fourier-space forms, beside the layered real-space path:
//
// Eq. 12 (one defocus R for every view): the CT step -- the layered reconstruction of the
// contrasts with the Ewald placement and no CTF bracket, as two real volumes V_c, V_s
// (per-layer cos and sin of pi lambda z_k q^2, run by the stage-A kernels) -- is packed as
// V_c + i V_s into a zero-padded grid and transformed once; the CTF inversion is then one
// pass over that spectrum:
//   F3 delta(q) = lambda / (4 pi sqrt(1+sigma^2)) [s'(q) V_c^(q) - c'(q) V_s^(q)],
//   V_c^(q) = (Z(q) + conj Z(-q)) / 2,  V_s^(q) = (Z(q) - conj Z(-q)) / (2 i),
//   s' = sin chi / (sin^2 chi + eps), c' = cos chi / (cos^2 chi + eps), chi at the
//   in-plane frequency q_perp of the Ewald-paraboloid point q (q_perp^2 = 2 q^2 /
//   (sqrt(1 + lambda^2 q^2) + 1)); chi reaches hundreds of radians, so its exact part is
//   taken modulo one turn in 64-bit fixed point and only a small correction in FP32.
// The spectrum of the CT step stays in the workspace, so other (sigma, eps) rerun only the
// phase pass and the inverse transform.
//
// The Fourier-gridding UTR (Sec. 2 after Eq. 11): every 2D DFT coefficient of every view,
// taken about the detector centre and multiplied by the bracket of Eq. 11 at its own R_n
// (fixed-point phase, as in stage A), is spread with trilinear weights over the 8 cells
// around its point Rot_n^T (q_u, q_v, -lambda q^2 / 2) of the padded volume's DFT grid
// (float atomics); S sums the weights.  Then F = acc / (S + eps_S), eps_S = 1e-3 x the
// mean of S over its non-zero cells; with the noise filter of Sec. 3, F = 0 where the
// gridded contrast (the same splat without the bracket) over S + eps_S is below
// NSR M / sqrt(S).  The phase back to the grid origin and 1/Delta are applied before the
// inverse transform.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "fft3.cuh"
#include "recon_internal.h"

namespace recon {
namespace {

__device__ __forceinline__ int signed_bin(int m, int P) { return m < P / 2 ? m : m - P; }

// Load functor of the first forward pass of Eq. 12's transform: line l = (z, y) of V_c + i V_s,
// zero outside the volume's n0 columns.
struct VolumePair {
  static constexpr bool kAlong = true;
  const float* vc;
  const float* vs;
  int n0, off0;
  __device__ __forceinline__ void begin() {}
  __device__ __forceinline__ float2 load(long long l, int v) const {
    const int i = v - off0;
    return i >= 0 && i < n0 ? make_float2(vc[l * n0 + i], vs[l * n0 + i]) : make_float2(0.f, 0.f);
  }
};

// Store functor of that pass: line (z, y) goes to its place in the padded grid.
struct GridLines {
  static constexpr bool kAlong = true;
  float2* grid;
  int n1, off1, off2;
  long long P0, P1;
  __device__ __forceinline__ void store(long long l, int v, float2 x) const {
    const unsigned z = (unsigned)l / (unsigned)n1;  // fewer than 2^20 lines
    grid[((z + off2) * P1 + ((unsigned)l - z * n1) + off1) * P0 + v] = x;
  }
};

// Constants of the phase pass (host-built in FP64 per call).  With power-of-two grid sides,
// K = sum_a (Pmax / P3_a)^2 m_a^2 is an integer and q^2 = K / (Pmax Delta)^2, so the phase in
// turns, chi / (2 pi) = (lambda R / 2) q_perp^2 + (Cs lambda^3 / 4) q_perp^4 - omega / (2 pi),
// splits into an exact part, uR K + uC K^2 - uW in 64-bit fixed point (2^-64 turns, modulo
// 1; uR, uC, uW the fractional parts of the per-unit constants) with q_perp^2 replaced by
// q^2, and the Ewald correction q_perp^2 = q^2 c(x), c = 2 / (1 + sqrt(1 + x)), x =
// lambda^2 q^2: (lambda R / 2) q^2 (c - 1) + (Cs lambda^3 / 4) q^4 (c^2 - 1), a fraction of a
// turn, in FP32.
struct SwapPhaseConst {
  uint64_t uR, uC, uW;
  float kx;          // x per unit K
  float uRf, uCf;    // lambda R / (2 (Pmax Delta)^2) and Cs lambda^3 / (4 (Pmax Delta)^4), turns
  float pref, eps;   // lambda / (4 pi sqrt(1 + sigma^2)), the Tikhonov eps
  int lx, ly;        // log2 of P3[0], P3[1]
  int sx, sy, sz;    // (Pmax / P3_a)^2
};

// Load functor of the first inverse pass (along z) of Eq. 12's CTF inversion: F3 delta at
// (ix, iy, iz), line l = iy P0 + ix with iy <= P1 / 2, from the kept spectrum at q and -q.  The
// result is Hermitian (V_c, V_s are real volumes and s', c' are even), so this half is all of it.
struct SwapPhase {
  static constexpr bool kAlong = false;
  const float2* Z;
  int P0, P1, P2;
  SwapPhaseConst k;
  __device__ __forceinline__ void begin() {}
  struct Raw {
    float2 a, b;  // Z(q), Z(-q)
  };
  static constexpr int kBatch = 8;  // 256^3: 452 us, 471 by 2, 555 with the loads between the arithmetic
  __device__ __forceinline__ Raw fetch(long long l, int iz) const {
    const int mx = P0 - 1, my = P1 - 1, mz = P2 - 1;
    const int ix = (int)(l & mx), iy = (int)(l >> k.lx);
    const int jx = (P0 - ix) & mx, jy = (P1 - iy) & my, jz = (P2 - iz) & mz;
    return Raw{Z[((((long long)iz << k.ly) + iy) << k.lx) + ix], Z[((((long long)jz << k.ly) + jy) << k.lx) + jx]};
  }
  __device__ __forceinline__ float2 finish(long long l, int iz, const Raw& raw) const {
    const int ix = (int)(l & (P0 - 1)), iy = (int)(l >> k.lx);
    const float2 a = raw.a, b = raw.b;  // conj Z(-q) is (b.x, -b.y)
    // V_c = (a + conj b) / 2, V_s = (a - conj b) / (2 i)
    const float vcr = 0.5f * (a.x + b.x), vci = 0.5f * (a.y - b.y);
    const float vsr = 0.5f * (a.y + b.y), vsi = -0.5f * (a.x - b.x);
    const int ux = signed_bin(ix, P0), uy = signed_bin(iy, P1), uz = signed_bin(iz, P2);
    const uint64_t K = (uint64_t)k.sx * (uint64_t)(ux * ux) + (uint64_t)k.sy * (uint64_t)(uy * uy) +
                       (uint64_t)k.sz * (uint64_t)(uz * uz);
    const uint64_t ph = k.uR * K + k.uC * (K * K) - k.uW;  // modulo 2^64 = modulo one turn
    const float Kf = (float)K;
    const float x = k.kx * Kf;
    const float r = 1.f + sqrtf(1.f + x);
    const float cm1 = -x / (r * r);  // c - 1
    const float corr = k.uRf * Kf * cm1 + k.uCf * Kf * Kf * (cm1 * (cm1 + 2.f));  // turns
    const int32_t h = (int32_t)(uint32_t)(ph >> 32) + __float2int_rn((corr - rintf(corr)) * 4294967296.0f);
    float sn, cn;
    __sincosf((float)h * 1.4629180792671596e-09f, &sn, &cn);  // h * 2 pi / 2^32
    const float sp = k.pref * __fdividef(sn, fmaf(sn, sn, k.eps));
    const float cp = k.pref * __fdividef(cn, fmaf(cn, cn, k.eps));
    return make_float2(sp * vcr - cp * vsr, sp * vci - cp * vsi);
  }
};

// ------------------------------------------------------------------ gridding
// The accumulators are [P3z][P3x][P3y], y fastest: consecutive lanes of the splat hold consecutive
// m_v of one column, and in a scan about y those fall on consecutive cells, so a warp's
// atomics to one of the 8 corners are one contiguous run.  A cell's sums are one vector
// (contrast x bracket, and with the noise filter the contrast too) and its weight a scalar beside it:
// two reductions per corner (red.global.add.v4.f32 / .v2.f32) instead of five scalar ones.
// A corner of weight zero adds nothing and is left out: in a scan about y half of the corners,
// whose samples lie on the grid's y planes.  L2 atomics bound it: 192^3 volume, 180 views,
// noise filter: 13.5 ms with scalar atomics and x fastest, 1.13 ms now.
template <bool RAW>
struct Cell;
template <>
struct Cell<true> {
  using type = float4;
};
template <>
struct Cell<false> {
  using type = float2;
};

__device__ __forceinline__ void cell_add(float4* p, float w, float2 z, float2 g) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(w * z.x), "f"(w * z.y), "f"(w * g.x),
               "f"(w * g.y)
               : "memory");
}
__device__ __forceinline__ void cell_add(float2* p, float w, float2 z, float2) {
  asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(w * z.x), "f"(w * z.y) : "memory");
}

// A sample's arithmetic in a written-out order of its fused products, since k_grid_resum forms the same terms again:
// its point (q_u, q_v, q_z) in DFT bins of each grid axis, ...
__device__ __forceinline__ void sample_point(const GridDir& d, const Fourier3Const& f, int mu, int mv, float qz,
                                             float (&g)[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a)
    g[a] = fmaf(qz, d.r[6 + a], fmaf((float)mu, d.r[a], (float)mv * d.r[3 + a])) * f.scale[a];
}
// ... and its contrast about the detector centre: G0 (for the mirrored half conj G0) times
// exp(i pi (mu (nu - 1) + mv (nv - 1)) / P), exact phase.
__device__ __forceinline__ float2 centred(float2 G0, bool mirror, const StageAConst& c, int mu, int mv) {
  const int k = (mu * (c.nu - 1) + mv * (c.nv - 1)) % (2 * c.P);
  float ps, pc;
  sincospif((float)k / (float)c.P, &ps, &pc);
  return mirror ? make_float2(fmaf(G0.y, ps, G0.x * pc), fmaf(G0.x, ps, -(G0.y * pc)))
                : make_float2(fmaf(G0.x, pc, -(G0.y * ps)), fmaf(G0.x, ps, G0.y * pc));
}

template <typename CellT>
__device__ __forceinline__ void splat(CellT* acc, float* S, const Fourier3Const& f, const float g[3], float2 z,
                                      float2 gc) {
  int b[3];
  float fr[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float fl = floorf(g[a]);
    b[a] = (int)fl;
    fr[a] = g[a] - fl;
  }
#pragma unroll
  for (int dz = 0; dz < 2; ++dz)
#pragma unroll
    for (int dy = 0; dy < 2; ++dy)
#pragma unroll
      for (int dx = 0; dx < 2; ++dx) {
        const float w = (dx ? fr[0] : 1.f - fr[0]) * (dy ? fr[1] : 1.f - fr[1]) * (dz ? fr[2] : 1.f - fr[2]);
        const int ix = (b[0] + dx) & (f.P3[0] - 1), iy = (b[1] + dy) & (f.P3[1] - 1), iz = (b[2] + dz) & (f.P3[2] - 1);
        const long long c = ((long long)iz * f.P3[0] + ix) * f.P3[1] + iy;
        if (w != 0.f) {
          atomicAdd(&S[c], w);
          cell_add(acc + c, w, z, gc);
        }
      }
}

// One thread per coefficient (n, col, m_v) of the half spectra G [n][col][P]; columns 1 ..
// P/2 - 1 also stand for their mirrors (-col, -m_v) (conjugate contrast, same bracket).
template <typename CellT>
__global__ void k_grid_splat(const float2* __restrict__ G, const GridDir* __restrict__ dirs, int dir_begin,
                             int n_dirs, StageAConst c, Fourier3Const f, CellT* __restrict__ acc,
                             float* __restrict__ S) {
  const int P = c.P, half = c.half;
  const long long total = (long long)n_dirs * half * P;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const long long line = i >> c.logP;
    const int mvi = (int)(i & (P - 1)), n = (int)(line / half), col = (int)(line - (long long)n * half);
    const GridDir& d = dirs[dir_begin + n];
    const int mu = col == P / 2 ? -P / 2 : col;  // the Nyquist column is bin -P/2 of the full grid
    const int mv = signed_bin(mvi, P);
    const float2 G0 = G[((long long)n * half + col) * P + mvi];
    const float2 gc = centred(G0, false, c, mu, mv);
    // Eq. 11's bracket at this view's R_n: chi / (2 pi) in 2^-64 turns, exact modulo 1
    const uint32_t m2 = (uint32_t)(mu * mu + mv * mv);
    const uint64_t m64 = m2;
    const uint32_t hi = (uint32_t)((d.uR * m64 + c.uC * (m64 * m64) - c.uW) >> 32);
    float sn, cn;
    sincospif((float)(int32_t)hi * 4.656612873077393e-10f, &sn, &cn);  // hi * 2^-31 = chi / pi
    const float sp = sn / fmaf(sn, sn, c.eps), cp = cn / fmaf(cn, cn, c.eps);
    // Z = pref G_c (s' - i c')
    const float2 z = make_float2(c.pref * (gc.x * sp + gc.y * cp), c.pref * (gc.y * sp - gc.x * cp));
    // the point (q_u, q_v, -lambda q^2 / 2) in DFT bins of each grid axis
    const float qz = -d.qz_coef * (float)m2;  // in units of 1 / (P delta)
    float g[3];
    sample_point(d, f, mu, mv, qz, g);
    splat(acc, S, f, g, z, gc);
    if (col >= 1 && col < P / 2) {  // the mirror (-mu, -mv): conjugate contrast, same bracket
      // its own bin (-P/2 stays -P/2 on the Nyquist row) and its own centring phase
      const int mvm = mv == -P / 2 ? mv : -mv;
      const float2 gm = centred(G0, true, c, -mu, mvm);
      const float2 zm = make_float2(c.pref * (gm.x * sp + gm.y * cp), c.pref * (gm.y * sp - gm.x * cp));
      float h[3];
      sample_point(d, f, -mu, mvm, qz, h);
      splat(acc, S, f, h, zm, gm);
    }
  }
}

// Sum and count of the non-zero cells of S: per thread in FP32 over its strided cells, then
// in FP64 across the warp and the grid.
__global__ void k_grid_stats(const float* __restrict__ S, long long n, double* __restrict__ stats) {
  float sum = 0.f;
  unsigned int cnt = 0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float s = S[i];
    if (s > 0.f) {
      sum += s;
      ++cnt;
    }
  }
  double ds = sum, dc = (double)cnt;
  for (int o = 16; o > 0; o >>= 1) {
    ds += __shfl_down_sync(0xffffffffu, ds, o);
    dc += __shfl_down_sync(0xffffffffu, dc, o);
  }
  if ((threadIdx.x & 31) == 0 && dc > 0.0) {
    atomicAdd(&stats[0], ds);
    atomicAdd(&stats[1], dc);
  }
}

// The noise filter keeps or drops whole cells by comparing float sums of atomics with a threshold, so for a cell
// next to it the order in which the atomics land would decide, and the volume change by a plane wave (1e-4 of its
// norm) from call to call.  Cells within kNearBand of the threshold (far more than the sums' rounding; some thousand
// of 79 million for 192^3, 180 views) are noted by the pass that takes the decision, summed again in one fixed order
// (k_grid_resum), and where those sums decide otherwise, the cell is added to or taken out of the pass's result
// (k_grid_settle).  A note list that is full leaves its other cells as they were taken.  The order is that in which
// the additions land in practice, so that volumes stay what they were: of the sums that six calls of the splat with
// scalar atomics repeat, it gives 98 to 99 % to the bit, sums in 64 bits 91 %, which decided otherwise in 6 volumes of 17.
// 192^3, 180 views: the call 2.67 ms, 2.66 without.
constexpr float kNearBand = 0x1p-15f;

// The two sides of the filter's comparison, |contrast| against its noise at a cell of weight s, inv = 1 / (s + eps_S).
__device__ __forceinline__ void noise_sides(float s, float inv, float x, float y, float nsr_m, float* signal,
                                            float* noise) {
  // squares fused in this order: the decision must not hang on how a compiler contracts them
  *signal = sqrtf(fmaf(y, y, x * x)) * inv;
  *noise = nsr_m * rsqrtf(fmaxf(s, 1e-30f));
}

__device__ __forceinline__ float grid_eps(const double* stats) {
  return stats[1] > 0.0 ? (float)(1e-3 * stats[0] / stats[1]) : 1.f;
}

// Load functor of the first inverse pass (along z) of the gridding: the Hermitian part, (F(q) +
// conj F(-q)) / 2, of the quotient F = acc / (S + eps_S) with the noise filter and the phase from
// the volume centre to the frame origin.  Line l = ix P3y + iy with ix <= P3x / 2.
template <bool RAW>
struct GridQuotient {
  static constexpr bool kAlong = false;
  const typename Cell<RAW>::type* acc;
  const float* S;
  const double* stats;
  int P3x, P3y, P3z, lx, ly;  // sides, log2 of x and y
  int kx, ky, kz;             // 2 c_a Pmax / P3_a, c_a = off_a + (n_a - 1) / 2 the volume's centre
  int turn;                   // 2 Pmax
  float inv_pmax, inv_delta, nsr_m, eps_s;
  NearCells near;
  __device__ __forceinline__ void begin() { eps_s = grid_eps(stats); }
  using Acc = typename Cell<RAW>::type;
  struct Raw {
    float s, sm;  // the cells at q and -q: weight,
    Acc a, am;    // sums
  };
  static constexpr int kBatch = 2;  // 192^3: 739 us, 1193 by 4 and 1043 by 8 (fewer warps), 1213 with early returns between
  __device__ __forceinline__ long long cell(int ix, int iy, int iz) const {
    return ((((long long)iz << lx) + ix) << ly) + iy;
  }
  __device__ __forceinline__ Acc sums(float s, long long i) const {
    Acc a = {};
    if (s != 0.f) a = acc[i];  // else nothing was added to the cell
    return a;
  }
  __device__ __forceinline__ Raw fetch(long long l, int iz) const {
    const int iy = (int)(l & (P3y - 1)), ix = (int)(l >> ly);
    const long long i = cell(ix, iy, iz);
    const long long m = cell((P3x - ix) & (P3x - 1), (P3y - iy) & (P3y - 1), (P3z - iz) & (P3z - 1));
    Raw r;
    r.s = S[i];
    r.sm = S[m];
    r.a = sums(r.s, i);
    r.am = sums(r.sm, m);
    return r;
  }
  __device__ __forceinline__ float2 quotient(int ix, int iy, int iz, float s, const Acc& a, bool note) const {
    if (s == 0.f) return make_float2(0.f, 0.f);
    const float inv = 1.f / (s + eps_s);
    if constexpr (RAW) {
      float signal, noise;
      noise_sides(s, inv, a.z, a.w, nsr_m, &signal, &noise);
      const bool keep = s > 0.f && signal >= noise;
      if (note && fabsf(signal - noise) < kNearBand * noise) {
        const unsigned int at = atomicAdd(near.count, 1u);
        if (at < near.cap) {
          near.cells[at] = 2 * (unsigned long long)cell(ix, iy, iz) + (keep ? 1 : 0);
          for (int q = 0; q < 3; ++q) near.sums[3 * (size_t)at + q] = 0.f;
        }
      }
      if (!keep) return make_float2(0.f, 0.f);
    }
    return placed(ix, iy, iz, make_float2(a.x * inv, a.y * inv));
  }
  // F with the phase from the volume centre to the frame origin, over Delta.
  __device__ __forceinline__ float2 placed(int ix, int iy, int iz, float2 F) const {
    // exp(-2 pi i sum_a m_a c_a / P3_a): the turns are T / (2 Pmax), T = sum_a m_a (2 c_a)
    // (Pmax / P3_a) an exact integer, reduced modulo 2 Pmax (a power of two)
    const int T = (signed_bin(ix, P3x) * kx + signed_bin(iy, P3y) * ky + signed_bin(iz, P3z) * kz) & (turn - 1);
    float ps, pc;
    sincospif(-(float)T * inv_pmax, &ps, &pc);
    return make_float2((F.x * pc - F.y * ps) * inv_delta, (F.x * ps + F.y * pc) * inv_delta);
  }
  __device__ __forceinline__ float2 finish(long long l, int iz, const Raw& r) const {
    const int iy = (int)(l & (P3y - 1)), ix = (int)(l >> ly);
    // every cell is noted once: where it is q itself, the cells beyond the half where they are -q
    const float2 a = quotient(ix, iy, iz, r.s, r.a, true);
    const float2 b = quotient((P3x - ix) & (P3x - 1), (P3y - iy) & (P3y - 1), (P3z - iz) & (P3z - 1), r.sm, r.am,
                              ix > 0 && ix < P3x / 2);
    return make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y));
  }
};

// The order of a noted cell's additions: CTAs kResident at a time (5 per SM, as the splat with scalar atomics ran),
// each in grid strides; those views that pass at the same time one after the other, and of a view the corners in
// the order of the splat's code (bit 3: the mirrored half after the direct one), then the samples.
constexpr int kResident = 5 * 152;
__device__ __forceinline__ unsigned long long landing_key(unsigned sample, unsigned stride, int view, int corner,
                                                          int in_view) {
  const unsigned long long turn = sample / stride, wave = sample % stride / 256 / kResident;
  // 4, 12, 20, 4 and 22 bits: a launch has at most 2^27 samples (1 GiB of spectra), 246 000 views of 32 x 17 of them
  return ((((wave << 12 | turn) << 20 | (unsigned)view) << 4 | (unsigned)corner) << 22) | (unsigned)in_view;
}

// The noted cells' sums over `n_dirs` views, a warp per cell: its lanes over the views (and the periodic images of the
// cell), a few of which have samples near the cell's projection onto their axes; over those samples, listing the ones
// that reach the cell; over the list for the contrasts; then the terms one by one by their keys.  Cells of more than
// kTerms terms (the lowest frequencies, or volumes much smaller than the images; the median is 2) take them in 64 bits.
constexpr int kTerms = 1024, kResumWarps = 2;
struct Terms {
  unsigned long long key[kTerms];
  float v[3][kTerms];
  unsigned short order[kTerms];
};
__global__ void k_grid_resum(const float2* __restrict__ G, const GridDir* __restrict__ dirs, int dir_begin, int n_dirs,
                             StageAConst c, Fourier3Const f, int lx, int ly, float reach, unsigned stride,
                             NearCells near) {
  __shared__ Terms terms_all[kResumWarps];
  __shared__ int n_terms_all[kResumWarps];
  Terms& terms = terms_all[threadIdx.x >> 5];
  int& n_terms = n_terms_all[threadIdx.x >> 5];
  const int P = c.P, lane = threadIdx.x & 31;
  const unsigned int n = min(*near.count, near.cap);
  for (unsigned int e = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < n; e += (gridDim.x * blockDim.x) >> 5) {
    const long long cell = (long long)(near.cells[e] >> 1);
    const int at[3] = {signed_bin((int)(cell >> ly) & (f.P3[0] - 1), f.P3[0]), signed_bin((int)cell & (f.P3[1] - 1), f.P3[1]),
                       signed_bin((int)(cell >> (lx + ly)), f.P3[2])};
    // samples per cell (powers of two); the grid is periodic: samples, up to reach P off, land on a cell's images too
    const float per[3] = {1.f / f.scale[0], 1.f / f.scale[1], 1.f / f.scale[2]};
    const int side = 2 * (int)(reach + 1.f) + 1;
    double sum[3] = {0.0, 0.0, 0.0};
    __syncwarp();
    if (lane == 0) n_terms = 0;
    __syncwarp();
    // whether view v has samples around the point s3 (in samples along the grid's axes), and their window
    const auto window = [&](int v, const float (&s3)[3], int (&lo)[2], int (&n)[2]) {
      const GridDir& d = dirs[dir_begin + v];
      float p[3], h[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        p[q] = s3[0] * d.r[3 * q] + s3[1] * d.r[3 * q + 1] + s3[2] * d.r[3 * q + 2];
        // half widths, in samples, of the cell's reach along the view's axes, and what rounding may add
        h[q] = 0.05f + fabsf(d.r[3 * q]) * per[0] + fabsf(d.r[3 * q + 1]) * per[1] + fabsf(d.r[3 * q + 2]) * per[2];
      }
      // q_z at the projection, and how far it varies over the window
      const float qz0 = -d.qz_coef * (p[0] * p[0] + p[1] * p[1]);
      const float vary = d.qz_coef * (2.f * (fabsf(p[0]) * h[0] + fabsf(p[1]) * h[1]) + h[0] * h[0] + h[1] * h[1]);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        lo[q] = max(-P / 2, (int)ceilf(p[q] - h[q]));
        n[q] = min(P / 2 - 1, (int)floorf(p[q] + h[q])) - lo[q] + 1;
      }
      return fabsf(p[2] - qz0) <= h[2] + vary && n[0] > 0 && n[1] > 0;
    };
    for (int image = 0; image < side * side * side; ++image) {
      const int b[3] = {at[0] + (image % side - side / 2) * f.P3[0], at[1] + (image / side % side - side / 2) * f.P3[1],
                        at[2] + (image / (side * side) - side / 2) * f.P3[2]};
      float s3[3];
      bool out = false;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        s3[a] = (float)b[a] * per[a];
        out |= fabsf(s3[a]) > reach * (float)P + 2.f * per[a];
      }
      if (out) continue;
      for (int first = 0; first < n_dirs; first += 32) {
        int lo[2], n_w[2];
        unsigned todo = __ballot_sync(0xffffffffu, first + lane < n_dirs && window(first + lane, s3, lo, n_w));
        for (; todo; todo &= todo - 1) {  // the lanes over the window's samples
          const int v = first + __ffs(todo) - 1;
          window(v, s3, lo, n_w);
          const GridDir& d = dirs[dir_begin + v];
          for (int q0 = lane; q0 < n_w[0] * n_w[1]; q0 += 32) {
            const int mu = lo[0] + q0 / n_w[1], mv = lo[1] + q0 % n_w[1];
            float g[3], w[3];
            sample_point(d, f, mu, mv, -d.qz_coef * (float)(uint32_t)(mu * mu + mv * mv), g);
            bool hit = true;
            int corner = 0;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
              const float fl = floorf(g[a]);
              const int to = b[a] - (int)fl;  // 0 or 1: the cell is a corner of the sample's
              hit &= to == 0 || to == 1;
              corner |= (to & 1) << a;
              w[a] = to ? g[a] - fl : 1.f - (g[a] - fl);
            }
            const float wt = w[0] * w[1] * w[2];
            if (!hit || wt == 0.f) continue;
            const bool mirror = mu < 0 && mu > -P / 2;  // from column -mu, whose row -P/2 stays
            const int col = abs(mu), row = mirror && mv > -P / 2 ? -mv : mv;
            const int in_view = col * P + (row & (P - 1));
            const int at_term = atomicAdd(&n_terms, 1);
            if (at_term < kTerms) {
              terms.key[at_term] =
                  landing_key((unsigned)v * c.half * P + in_view, stride, v, corner + (mirror ? 8 : 0), in_view);
              terms.v[0][at_term] = wt;
            } else {
              const float2 gc = centred(G[(long long)v * c.half * P + in_view], mirror, c, mu, mv);
              sum[0] += (double)wt;
              sum[1] += (double)__fmul_rn(wt, gc.x);
              sum[2] += (double)__fmul_rn(wt, gc.y);
            }
          }
          __syncwarp();
        }
      }
    }
    __syncwarp();
    const int m = n_terms;
    float* const total = near.sums + 3 * (size_t)e;
    for (int q = lane; q < min(m, kTerms); q += 32) {
      const unsigned long long key = terms.key[q];
      const int in_view = (int)(key & 0x3FFFFF), v = (int)(key >> 26 & 0xFFFFF), col = in_view >> c.logP;
      const bool mirror = key >> 25 & 1;
      const int row = signed_bin(in_view & (P - 1), P);
      const int mu = mirror ? -col : (col == P / 2 ? -P / 2 : col), mv = mirror && row > -P / 2 ? -row : row;
      const float2 gc = centred(G[(long long)v * c.half * P + in_view], mirror, c, mu, mv);
      const float wt = terms.v[0][q];
      const float t[3] = {wt, __fmul_rn(wt, gc.x), __fmul_rn(wt, gc.y)};
      terms.v[1][q] = t[1];
      terms.v[2][q] = t[2];
#pragma unroll
      for (int i = 0; i < 3; ++i) sum[i] += (double)t[i];
    }
    __syncwarp();
    if (m > kTerms) {
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        for (int o = 16; o > 0; o >>= 1) sum[q] += __shfl_down_sync(0xffffffffu, sum[q], o);
        if (lane == 0) total[q] = (float)(total[q] + sum[q]);
      }
      continue;
    }
    for (int q = lane; q < m; q += 32) {
      int rank = 0;
      for (int k = 0; k < m; ++k) rank += terms.key[k] < terms.key[q];  // the keys are distinct
      terms.order[rank] = (unsigned short)q;
    }
    __syncwarp();
    float acc = lane < 3 ? total[lane] : 0.f;
    if (lane < 3)
      for (int k = 0; k < m; ++k) acc += terms.v[lane][terms.order[k]];
    if (lane < 3) total[lane] = acc;
  }
}

// A warp per noted cell: where the ordered sums decide otherwise, the cell's share of its z lines (transformed
// already, planes off .. off + n of H) is added or taken out.
__global__ void k_grid_settle(const GridQuotient<true> in, float2* __restrict__ H, int off, int n) {
  const int lane = threadIdx.x & 31;
  const unsigned int noted = min(*in.near.count, in.near.cap);
  const float eps_s = grid_eps(in.stats);
  const long long plane = (long long)(in.P3x / 2 + 1) * in.P3y;
  for (unsigned int e = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < noted; e += (gridDim.x * blockDim.x) >> 5) {
    const long long cell = (long long)(in.near.cells[e] >> 1);
    const bool kept = in.near.cells[e] & 1;
    const float* t = in.near.sums + 3 * (size_t)e;
    const float sum = t[0];
    float signal, noise;
    noise_sides(sum, 1.f / (sum + eps_s), t[1], t[2], in.nsr_m, &signal, &noise);
    const bool keep = signal >= noise;
    if (!(sum > 0.f) || keep == kept) continue;
    const int iy = (int)cell & (in.P3y - 1), ix = (int)(cell >> in.ly) & (in.P3x - 1), iz = (int)(cell >> (in.lx + in.ly));
    const float inv = (keep ? 0.5f : -0.5f) / (in.S[cell] + eps_s);  // half: of the Hermitian part
    const float4 a = in.acc[cell];
    const float2 F = in.placed(ix, iy, iz, make_float2(a.x * inv, a.y * inv));
#pragma unroll
    for (int m = 0; m < 2; ++m) {  // as q, and conjugate as -q
      const int jx = m ? (in.P3x - ix) & (in.P3x - 1) : ix, jy = m ? (in.P3y - iy) & (in.P3y - 1) : iy;
      const int jz = m ? (in.P3z - iz) & (in.P3z - 1) : iz;
      if (jx > in.P3x / 2) continue;
      const float Fy = m ? -F.y : F.y;
      for (int z = lane; z < n; z += 32) {
        float ps, pc;
        sincospif(2.f * (float)((jz * (z + off)) & (in.P3z - 1)) / (float)in.P3z, &ps, &pc);
        float2* h = H + z * plane + (long long)jx * in.P3y + jy;
        atomicAdd(&h->x, F.x * pc - Fy * ps);
        atomicAdd(&h->y, F.x * ps + Fy * pc);
      }
    }
  }
}

// frac(t) in 2^-64 turns (t >= 0)
uint64_t turns_fixed(double t) {
  double fr = t - std::floor(t);
  if (!(fr < 1.0)) fr = 0.0;
  const double scaled = std::ldexp(fr, 64);
  return scaled >= 18446744073709551616.0 ? 0 : (uint64_t)scaled;
}

int log2_int(int p) {
  int l = 0;
  while ((1 << l) < p) ++l;
  return l;
}

unsigned grid_blocks(long long n) {
  const long long cap = (long long)device_sm_count() * 16;
  const long long want = (n + 255) / 256;
  return (unsigned)(want < cap ? (want > 0 ? want : 1) : cap);
}

}  // namespace

cudaError_t launch_swap_forward(const float* vc, const float* vs, float2* Z, const Fourier3Const& f,
                                const float2* const tw[3], cudaStream_t s) {
  const long long P0 = f.P3[0], P1 = f.P3[1];
  const VolumePair in{vc, vs, f.n[0], f.off[0]};
  const GridLines out{Z, f.n[1], f.off[1], f.off[2], P0, P1};
  cudaError_t e = fft3::launch_lines<false>(f.P3[0], in, out, (long long)f.n[1] * f.n[2], tw[0], s);
  // y lines of the planes that hold the volume, then every z line
  float2* Zv = Z + f.off[2] * P0 * P1;
  const int lx = log2_int(f.P3[0]);
  const fft3::Columns y_in{Zv, lx, P0 * P1, P0, f.off[1], f.off[1] + f.n[1]}, y_out{Zv, lx, P0 * P1, P0, 0, f.P3[1]};
  if (e == cudaSuccess) e = fft3::launch_lines<false>(f.P3[1], y_in, y_out, P0 * f.n[2], tw[1], s);
  const fft3::Columns z_in{Z, 62, 0, P0 * P1, f.off[2], f.off[2] + f.n[2]}, z_out{Z, 62, 0, P0 * P1, 0, f.P3[2]};
  if (e == cudaSuccess) e = fft3::launch_lines<false>(f.P3[2], z_in, z_out, P0 * P1, tw[2], s);
  return e;
}

size_t swap_half_cells(const Fourier3Const& f) { return fft3::half_cells(f.P3, f.n[2]); }

// axes of the gridding's half spectrum: y fastest, halved along x
static void grid_axes(const Fourier3Const& f, int P[3], int n[3], int off[3]) {
  const int perm[3] = {1, 0, 2};
  for (int a = 0; a < 3; ++a) {
    P[a] = f.P3[perm[a]];
    n[a] = f.n[perm[a]];
    off[a] = f.off[perm[a]];
  }
}

size_t grid_half_cells(const Fourier3Const& f) {
  int P[3], n[3], off[3];
  grid_axes(f, P, n, off);
  return fft3::half_cells(P, n[2]);
}

cudaError_t launch_swap_phase(const float2* Z, float2* H, float* vol, const Fourier3Const& f, double R, double sigma,
                              double eps, double cs, const float2* const tw[3], cudaStream_t s) {
  SwapPhaseConst k;
  const int Pmax = std::max(f.P3[0], std::max(f.P3[1], f.P3[2]));
  const double pd2 = (double)Pmax * f.delta * (double)Pmax * f.delta;  // (Pmax Delta)^2
  const double cR = f.lam * R / (2.0 * pd2);                            // turns per unit K
  const double cC = cs * f.lam * f.lam * f.lam / (4.0 * pd2 * pd2);     // turns per unit K^2
  const double cW = std::atan(sigma) / (2.0 * 3.14159265358979323846);
  k.uR = turns_fixed(cR);
  k.uC = turns_fixed(cC);
  k.uW = turns_fixed(cW);
  k.kx = (float)(f.lam * f.lam / pd2);
  k.uRf = (float)cR;
  k.uCf = (float)cC;
  k.pref = (float)(f.lam / (4.0 * 3.14159265358979323846 * std::sqrt(1.0 + sigma * sigma)));
  k.eps = (float)eps;
  k.lx = log2_int(f.P3[0]);
  k.ly = log2_int(f.P3[1]);
  k.sx = (Pmax / f.P3[0]) * (Pmax / f.P3[0]);
  k.sy = (Pmax / f.P3[1]) * (Pmax / f.P3[1]);
  k.sz = (Pmax / f.P3[2]) * (Pmax / f.P3[2]);
  const SwapPhase in{Z, f.P3[0], f.P3[1], f.P3[2], k};
  const cudaError_t e = fft3::inverse_first(in, H, f.P3, f.n, f.off, tw, s);
  return e == cudaSuccess ? fft3::inverse_rest<true>(H, vol, f.P3, f.n, f.off, tw, s) : e;
}

cudaError_t launch_grid_splat(const float2* G, const GridDir* dirs, int dir_begin, int n_dirs, const StageAConst& c,
                              const Fourier3Const& f, void* acc, float* S, bool with_raw, cudaStream_t s) {
  if (n_dirs <= 0) return cudaSuccess;
  const unsigned blocks = grid_blocks((long long)n_dirs * c.half * c.P);
  if (with_raw)
    k_grid_splat<float4><<<blocks, 256, 0, s>>>(G, dirs, dir_begin, n_dirs, c, f, (float4*)acc, S);
  else
    k_grid_splat<float2><<<blocks, 256, 0, s>>>(G, dirs, dir_begin, n_dirs, c, f, (float2*)acc, S);
  return cudaGetLastError();
}

unsigned int grid_near_cap(const Fourier3Const& f) {
  const long long cells = (long long)f.P3[0] * f.P3[1] * f.P3[2];
  return (unsigned int)std::min<long long>(1 << 18, std::max<long long>(1024, cells / 64));
}

template <bool RAW>
static GridQuotient<RAW> grid_quotient(const GridSums& g, const Fourier3Const& f) {
  const int Pmax = std::max(f.P3[0], std::max(f.P3[1], f.P3[2]));
  GridQuotient<RAW> in;
  in.acc = (const typename Cell<RAW>::type*)g.acc;
  in.S = g.S;
  in.stats = g.stats;
  in.P3x = f.P3[0];
  in.P3y = f.P3[1];
  in.P3z = f.P3[2];
  in.lx = log2_int(f.P3[0]);
  in.ly = log2_int(f.P3[1]);
  in.kx = (2 * f.off[0] + f.n[0] - 1) * (Pmax / f.P3[0]);
  in.ky = (2 * f.off[1] + f.n[1] - 1) * (Pmax / f.P3[1]);
  in.kz = (2 * f.off[2] + f.n[2] - 1) * (Pmax / f.P3[2]);
  in.turn = 2 * Pmax;
  in.inv_pmax = 1.f / (float)Pmax;  // a power of two: exact
  in.inv_delta = (float)(1.0 / f.delta);
  in.nsr_m = g.nsr_m;
  in.eps_s = 0.f;  // set on the device from stats
  in.near = g.near;
  return in;
}

cudaError_t launch_grid_quotient(const GridSums& g, const Fourier3Const& f, const float2* const tw[3], cudaStream_t s) {
  const long long nb = (long long)f.P3[0] * f.P3[1] * f.P3[2];
  cudaError_t e = cudaMemsetAsync(g.stats, 0, 2 * sizeof(double), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(g.near.count, 0, sizeof(unsigned int), s);
  if (e != cudaSuccess) return e;
  k_grid_stats<<<grid_blocks(nb), 256, 0, s>>>(g.S, nb, g.stats);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  int P[3], n[3], off[3];
  grid_axes(f, P, n, off);
  const float2* const twp[3] = {tw[1], tw[0], tw[2]};
  return g.nsr_m > 0.f ? fft3::inverse_first(grid_quotient<true>(g, f), g.H, P, n, off, twp, s)
                       : fft3::inverse_first(grid_quotient<false>(g, f), g.H, P, n, off, twp, s);
}

cudaError_t launch_grid_resum(const GridSums& g, const float2* G, const GridDir* dirs, int dir_begin, int n_dirs,
                              const StageAConst& c, const Fourier3Const& f, cudaStream_t s) {
  // samples reach sqrt(2) P / 2 in the image plane and lambda / (4 Delta) P along the beam.  Beyond 8 pixels of
  // wavelength (no image resolves that) the images of a cell are too many to try: its sums stay 0 and settle nothing
  const double reach = 0.7072 + f.lam / (4.0 * f.delta);
  if (reach > 2.8) return cudaSuccess;
  k_grid_resum<<<device_sm_count() * 10, 32 * kResumWarps, 0, s>>>(G, dirs, dir_begin, n_dirs, c, f, log2_int(f.P3[0]),
                                                     log2_int(f.P3[1]), (float)reach,
                                                     256 * grid_blocks((long long)n_dirs * c.half * c.P), g.near);
  return cudaGetLastError();
}

cudaError_t launch_grid_finish(const GridSums& g, float* vol, const Fourier3Const& f, const float2* const tw[3],
                               cudaStream_t s) {
  if (g.nsr_m > 0.f) {
    k_grid_settle<<<device_sm_count(), 128, 0, s>>>(grid_quotient<true>(g, f), g.H, f.off[2], f.n[2]);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  int P[3], n[3], off[3];
  grid_axes(f, P, n, off);
  const float2* const twp[3] = {tw[1], tw[0], tw[2]};
  return fft3::inverse_rest<false>(g.H, vol, P, n, off, twp, s);
}

}  // namespace recon
