// Line FFTs of the padded 3D grids of the two 3D-Fourier forms (Eq. 12's CTF inversion after
// the CT step; the Fourier-gridding reconstruction, Sec. 2 after Eq. 11).  A transform is
// three passes of line FFTs, one per axis, and only the part of the grid that each pass
// needs is touched: a forward pass reads the rows that hold the volume (the rest of the padded
// grid is zero and is never stored), an inverse pass writes the rows that later passes keep.
// The producer of a pass (reading the volumes, the CTF phase, the gridded quotient) is its
// load functor and the volume is written by its last pass, so no grid-sized array is read or
// written only to be scaled, packed or cropped.  The inverse result is the real part of the
// transform, i.e. the transform of the spectrum's Hermitian part, so the inverse passes run
// on half of the spectrum along axis 1 and end with a complex-to-real pass.
//
// HBM traffic bounds these passes (512^3 grid of a 256^3 volume: forward 2.2 GB, inverse 1.9 GB
// against 7.5 GB and 10.8 GB when each pass ran over the whole grid): a CTA of 512 threads
// takes CB = 512 / T neighbouring lines, T threads per line, so a pass across rows moves at
// least 32 and for lengths up to 512 at least 64 contiguous bytes, all of a thread's loads in
// flight before its first shared-memory store.
#pragma once

#include <type_traits>

#include <cuda_runtime.h>

#include "fft16.cuh"
#include "fft_reg.cuh"
#include "recon_internal.h"

namespace recon {
namespace fft3 {

constexpr int kThreads = 512;

// Lengths 2-8: a thread per line, the whole line in registers; 16-512: fft_reg.cuh; 1024-2048:
// fft16.cuh.
template <int P>
struct Engine {
  static constexpr bool kDirect = P <= 8, kWide = P >= 1024;
  static constexpr int T = kDirect ? 1 : (kWide ? P / 16 : P / 8);  // threads per line
  static constexpr int V = P / T;                                    // values per thread
  static constexpr int CB = kThreads / T;                            // lines per CTA
  static constexpr int L = kDirect ? P + 1 : (kWide ? fft16::buffer_len(P) : fft::buffer_len(P, CB));
  static constexpr int NT = kDirect ? 0 : (kWide ? fft16::table_len(P) : fft::pass_table_len(P));
  __device__ static int idx(int v) { return kDirect ? v : (kWide ? fft16::pad(v) : fft::padded(v)); }

  template <bool INV>
  __device__ static void run(float2 (&x)[V], float2* buf, const float2* tw, int j, int g) {
    if constexpr (kDirect) {
      fft::dftR<P, INV>(x);
    } else if constexpr (kWide) {
      fft16::group_fft_sb<P, INV>(x, buf, tw, j, fft::GroupSync{1 + g, T});
    } else {
      fft::block_fft<P, INV>(x, buf, tw, j, fft::GroupSync{1 + g, T});
    }
  }
};

// Element v of line l of a complex array, for v in [lo, hi); zero (on load) or dropped (on store)
// outside.  Rows: a line's elements are consecutive, lines `pitch` apart.  Columns: neighbouring
// lines are consecutive, (l >> inner_log2) outer + (l mod 2^inner_log2) + v step.
struct Rows {
  static constexpr bool kAlong = true;
  float2* data;
  long long pitch;
  int lo, hi;
  __device__ __forceinline__ void begin() {}
  __device__ __forceinline__ float2 load(long long l, int v) const {
    return v >= lo && v < hi ? data[l * pitch + v] : make_float2(0.f, 0.f);
  }
  __device__ __forceinline__ void store(long long l, int v, float2 x) const {
    if (v >= lo && v < hi) data[l * pitch + v] = x;
  }
};
struct Columns {
  static constexpr bool kAlong = false;
  float2* data;
  int inner_log2;
  long long outer, step;
  int lo, hi;
  __device__ __forceinline__ void begin() {}
  __device__ __forceinline__ float2* at(long long l, int v) const {
    return data + (l >> inner_log2) * outer + (l & ((1LL << inner_log2) - 1)) + v * step;
  }
  __device__ __forceinline__ float2 load(long long l, int v) const {
    return v >= lo && v < hi ? *at(l, v) : make_float2(0.f, 0.f);
  }
  __device__ __forceinline__ void store(long long l, int v, float2 x) const {
    if (v >= lo && v < hi) *at(l, v) = x;
  }
};

// Line and element of a thread's k-th value: element by element along the lines, or CB
// neighbouring lines per element.
template <int P, bool ALONG>
__device__ __forceinline__ void place(int k, int& t, int& v) {
  constexpr int CB = Engine<P>::CB;
  if constexpr (!ALONG) {
    t = threadIdx.x % CB;
    v = threadIdx.x / CB + k * (kThreads / CB);
  } else if constexpr (P >= kThreads) {
    t = k / (P / kThreads);
    v = threadIdx.x + (k % (P / kThreads)) * kThreads;
  } else {
    t = threadIdx.x / P + k * (kThreads / P);
    v = threadIdx.x % P;
  }
}

// Load functors with arithmetic behind their loads give them apart: fetch() returns what it read (Raw), finish() makes
// the value of it, kBatch values at a time, so that the loads of a batch are in flight together (the
// divisions and roots of finish() branch, and no load moves over a branch).
template <class In, class = void>
struct Batch {
  static constexpr int N = 0;
};
template <class In>
struct Batch<In, std::void_t<typename In::Raw>> {
  static constexpr int N = In::kBatch;
};

template <int P, bool INV, class In, class Out>
__global__ void __launch_bounds__(kThreads) k_lines(const In in_arg, const Out out, long long n_lines,
                                                    const float2* __restrict__ twg) {
  using E = Engine<P>;
  extern __shared__ float2 smem3[];
  float2* tw = smem3;
  float2* buf_all = smem3 + E::NT;
  const int g = threadIdx.x / E::T, j = threadIdx.x % E::T;
  float2* buf = buf_all + g * E::L;
  for (int i = threadIdx.x; i < E::NT; i += kThreads) tw[i] = twg[i];
  const long long l0 = (long long)blockIdx.x * E::CB;
  In in = in_arg;
  in.begin();
  float2 val[E::V];  // a CTA's CB lines of P elements are V per thread
  if constexpr (Batch<In>::N > 0) {
    constexpr int N = Batch<In>::N < E::V ? Batch<In>::N : E::V;
    static_assert(E::V % N == 0, "whole batches");
#pragma unroll
    for (int k0 = 0; k0 < E::V; k0 += N) {
      typename In::Raw raw[N];
#pragma unroll
      for (int k = 0; k < N; ++k) {
        int t, v;
        place<P, In::kAlong>(k0 + k, t, v);
        raw[k] = in.fetch(l0 + t < n_lines ? l0 + t : n_lines - 1, v);
      }
#pragma unroll
      for (int k = 0; k < N; ++k) {
        int t, v;
        place<P, In::kAlong>(k0 + k, t, v);
        val[k0 + k] = l0 + t < n_lines ? in.finish(l0 + t, v, raw[k]) : make_float2(0.f, 0.f);
      }
    }
  } else {
#pragma unroll
    for (int k = 0; k < E::V; ++k) {
      int t, v;
      place<P, In::kAlong>(k, t, v);
      val[k] = l0 + t < n_lines ? in.load(l0 + t, v) : make_float2(0.f, 0.f);
    }
  }
#pragma unroll
  for (int k = 0; k < E::V; ++k) {
    int t, v;
    place<P, In::kAlong>(k, t, v);
    buf_all[t * E::L + E::idx(v)] = val[k];
  }
  __syncthreads();
#pragma unroll
  for (int s = 0; s < E::V; ++s) val[s] = buf[E::idx(j + s * E::T)];
  E::template run<INV>(val, buf, tw, j, g);
  fft::GroupSync{1 + g, E::T}();  // the transform's last reads of the line's buffer
#pragma unroll
  for (int s = 0; s < E::V; ++s) buf[E::idx(j + s * E::T)] = val[s];
  __syncthreads();
#pragma unroll
  for (int k = 0; k < E::V; ++k) {
    int t, v;
    place<P, Out::kAlong>(k, t, v);
    if (l0 + t < n_lines) out.store(l0 + t, v, buf_all[t * E::L + E::idx(v)]);
  }
}

// The last inverse pass: half spectra along axis 1 to real rows of the volume.  Two lines
// (neighbours along axis 0) share one complex transform as real + i imaginary.  H [n2][half][P0]
// holds the lines; axis 0 is cropped to n0 entries from off0, axis 1 to n1 from off1.
// ROWS0: the volume is [n2][n1][n0] (axis 0 fastest), else [n2][n0][n1].
struct RealOut {
  const float2* H;
  float* vol;
  int n0, n1, n2, off0, off1, P0;
  float scale;
};

template <int P>
__host__ __device__ constexpr int c2r_stride() {  // odd: the fill's columns spread over the banks
  return (P / 2 + 1) | 1;
}

template <int P>
constexpr size_t c2r_smem() {
  using E = Engine<P>;
  size_t n = (size_t)E::CB * E::L;
  const size_t tile = (size_t)2 * E::CB * c2r_stride<P>();
  if (tile > n) n = tile;
  const size_t rows = ((size_t)P * (2 * E::CB + 1) + 1) / 2;
  if (rows > n) n = rows;
  return sizeof(float2) * (E::NT + n);
}

template <int P, bool ROWS0>
__global__ void __launch_bounds__(kThreads) k_lines_c2r(const RealOut o, const float2* __restrict__ twg) {
  using E = Engine<P>;
  constexpr int H1 = P / 2 + 1, HS = c2r_stride<P>();
  constexpr int FILL = (2 * E::CB * H1 + kThreads - 1) / kThreads;
  extern __shared__ float2 smem3[];
  float2* tw = smem3;
  float2* tile = smem3 + E::NT;
  const int g = threadIdx.x / E::T, j = threadIdx.x % E::T;
  float2* buf = tile + g * E::L;
  for (int i = threadIdx.x; i < E::NT; i += kThreads) tw[i] = twg[i];
  const int pairs = (o.n0 + 1) / 2;
  const int units = o.n2 * pairs, u0 = blockIdx.x * E::CB;  // at most 1024 * 512
  {
    float2 tmp[FILL];
#pragma unroll
    for (int it = 0; it < FILL; ++it) {
      const int q = threadIdx.x + it * kThreads;
      const int t = q % (2 * E::CB), m = q / (2 * E::CB);
      const int u = u0 + (t >> 1);
      tmp[it] = make_float2(0.f, 0.f);
      if (m < H1 && u < units) {
        const int z = u / pairs;
        const int i0 = 2 * (u - z * pairs) + (t & 1);
        if (i0 < o.n0) tmp[it] = o.H[((long long)z * H1 + m) * o.P0 + o.off0 + i0];
      }
    }
#pragma unroll
    for (int it = 0; it < FILL; ++it) {
      const int q = threadIdx.x + it * kThreads;
      const int t = q % (2 * E::CB), m = q / (2 * E::CB);
      if (m < H1) tile[t * HS + m] = tmp[it];
    }
  }
  __syncthreads();
  const float2* X1 = tile + 2 * g * HS;
  const float2* X2 = X1 + HS;
  float2 x[E::V];
#pragma unroll
  for (int s = 0; s < E::V; ++s) {
    const int m = j + s * E::T, mm = m <= P / 2 ? m : P - m;
    float2 a = X1[mm], b = X2[mm];
    if (m == 0 || m == P / 2) a.y = b.y = 0.f;  // real bins
    if (m > P / 2) {                            // X[m] = conj X[P - m]
      a.y = -a.y;
      b.y = -b.y;
    }
    x[s] = make_float2(a.x - b.y, a.y + b.x);  // a + i b
  }
  __syncthreads();
  E::template run<true>(x, buf, tw, j, g);
  if constexpr (ROWS0) {
    float* rows = reinterpret_cast<float*>(tile);  // [P][2 CB + 1]: rows along axis 0 for the stores
    __syncthreads();
#pragma unroll
    for (int s = 0; s < E::V; ++s) {
      rows[(j + s * E::T) * (2 * E::CB + 1) + 2 * g] = x[s].x * o.scale;
      rows[(j + s * E::T) * (2 * E::CB + 1) + 2 * g + 1] = x[s].y * o.scale;
    }
    __syncthreads();
#pragma unroll 4
    for (int q = threadIdx.x; q < 2 * E::CB * o.n1; q += kThreads) {
      const int t = q % (2 * E::CB), i1 = q / (2 * E::CB);
      const int u = u0 + (t >> 1);
      if (u >= units) continue;
      const int z = u / pairs;
      const int i0 = 2 * (u - z * pairs) + (t & 1);
      if (i0 < o.n0) o.vol[((long long)z * o.n1 + i1) * o.n0 + i0] = rows[(i1 + o.off1) * (2 * E::CB + 1) + t];
    }
  } else {
    const int u = u0 + g;
    if (u >= units) return;
    const int z = u / pairs;
    const int i0 = 2 * (u - z * pairs);
    float* r1 = o.vol + ((long long)z * o.n0 + i0) * o.n1 - o.off1;
#pragma unroll
    for (int s = 0; s < E::V; ++s) {
      const int v = j + s * E::T;
      if (v < o.off1 || v >= o.off1 + o.n1) continue;
      r1[v] = x[s].x * o.scale;
      if (i0 + 1 < o.n0) r1[o.n1 + v] = x[s].y * o.scale;
    }
  }
}

// Host side: the launch of one pass for a run-time length.
template <int P, bool INV, class In, class Out>
cudaError_t launch_lines_p(const In& in, const Out& out, long long n_lines, const float2* tw, cudaStream_t s) {
  using E = Engine<P>;
  constexpr size_t smem = sizeof(float2) * ((size_t)E::NT + (size_t)E::CB * E::L);
  if (smem > 48 * 1024) {
    const cudaError_t e =
        cudaFuncSetAttribute(k_lines<P, INV, In, Out>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  k_lines<P, INV, In, Out><<<(unsigned)((n_lines + E::CB - 1) / E::CB), kThreads, smem, s>>>(in, out, n_lines, tw);
  return cudaGetLastError();
}

// calls f.template operator()<P>() for the grid side P (a power of two, 2 .. 2048)
template <class F>
cudaError_t with_length(int P, F&& f) {
  switch (P) {
    case 2: return f.template operator()<2>();
    case 4: return f.template operator()<4>();
    case 8: return f.template operator()<8>();
    case 16: return f.template operator()<16>();
    case 32: return f.template operator()<32>();
    case 64: return f.template operator()<64>();
    case 128: return f.template operator()<128>();
    case 256: return f.template operator()<256>();
    case 512: return f.template operator()<512>();
    case 1024: return f.template operator()<1024>();
    case 2048: return f.template operator()<2048>();
    default: return cudaErrorInvalidValue;
  }
}

template <bool INV, class In, class Out>
struct LinesCall {
  const In& in;
  const Out& out;
  long long n_lines;
  const float2* tw;
  cudaStream_t s;
  template <int P>
  cudaError_t operator()() const {
    return launch_lines_p<P, INV>(in, out, n_lines, tw, s);
  }
};

template <bool INV, class In, class Out>
cudaError_t launch_lines(int P, const In& in, const Out& out, long long n_lines, const float2* tw, cudaStream_t s) {
  return with_length(P, LinesCall<INV, In, Out>{in, out, n_lines, tw, s});
}

template <bool ROWS0>
struct RealCall {
  const RealOut& o;
  const float2* tw;
  cudaStream_t s;
  template <int P>
  cudaError_t operator()() const {
    constexpr size_t smem = c2r_smem<P>();
    if (smem > 48 * 1024) {
      const cudaError_t e =
          cudaFuncSetAttribute(k_lines_c2r<P, ROWS0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    const long long units = (long long)o.n2 * ((o.n0 + 1) / 2);
    k_lines_c2r<P, ROWS0>
        <<<(unsigned)((units + Engine<P>::CB - 1) / Engine<P>::CB), kThreads, smem, s>>>(o, tw);
    return cudaGetLastError();
  }
};

// The inverse passes: the first one, along axis 2, from the producing load `in` into the half spectrum H [n2][P1 / 2
// + 1][P0] (P, n, off per axis, 0 fastest), and the others, the cropped real volume to vol.
template <class In>
cudaError_t inverse_first(const In& in, float2* H, const int P[3], const int n[3], const int off[3],
                          const float2* const tw[3], cudaStream_t s) {
  const long long plane = (long long)(P[1] / 2 + 1) * P[0];
  const Columns z{H - (long long)off[2] * plane, 62, 0, plane, off[2], off[2] + n[2]};
  return launch_lines<true>(P[2], in, z, plane, tw[2], s);
}
template <bool ROWS0>
cudaError_t inverse_rest(float2* H, float* vol, const int P[3], const int n[3], const int off[3],
                         const float2* const tw[3], cudaStream_t s) {
  const Rows x{H, P[0], 0, P[0]}, xc{H, P[0], off[0], off[0] + n[0]};
  cudaError_t e = launch_lines<true>(P[0], x, xc, (long long)n[2] * (P[1] / 2 + 1), tw[0], s);
  const RealOut o{H, vol, n[0], n[1], n[2], off[0], off[1], P[0], (float)(1.0 / ((double)P[0] * P[1] * P[2]))};
  if (e == cudaSuccess) e = with_length(P[1], RealCall<ROWS0>{o, tw[1], s});
  return e;
}

// Complex cells of the half spectrum that the inverse passes work in.
inline size_t half_cells(const int P[3], int n2) { return (size_t)n2 * (P[1] / 2 + 1) * P[0]; }

}  // namespace fft3
}  // namespace recon
