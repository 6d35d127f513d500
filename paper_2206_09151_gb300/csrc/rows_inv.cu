// Stage A's row stage for P <= 2048: the spectra of every row of a layer (T, from the column kernels)
// to the rows of the interpolation stack.
//
// A CTA takes G row pairs of one layer; each pair is one complex inverse FFT of length P (row 2p in the
// real part, row 2p + 1 in the imaginary part).  What bounds it is the shared-memory / L1 pipe
// and behind that the bytes of T and of the stack, so everything here is about fewer trips through it:
//   - the lanes of a warp run over the row pairs first, so the loads from T ([column][row],
//     a row pair is 16 bytes) and the stores to column stacks ([column][row]) are contiguous across
//     lanes without passing through shared memory;
//   - a thread holds the first pass's butterflies j and P/R - j, whose inputs are each other's
//     Hermitian mirror images: every value of the half spectrum is loaded once, and
//     straight into the registers of the pass that uses it;
//   - the later passes take butterflies j + q P/2R, whose twiddles in the middle pass are the same.
// The lanes along the row, a group of threads per pair, staged the half spectra and the output in shared
// memory and read every spectrum value twice: 836 us for 120 directions x 32 layers of 256 x 256
// (P = 512, column stack), 523 us now, 5.8 TB/s; 3 directions x 64 layers of 1024 x 1024 (P = 2048, bfloat16
// tap pairs) 791 us, 680 now; 15 x 64 of 512 x 512 (P = 1024, the same) 1038 us, 654 now.
// Measured and not kept: an L2 prefetch of the tile that the SM takes next (the same to 5 % slower, the loads are
// not what waits), 3 CTAs of 80 registers at P = 512 (6 % slower than 4 of 64), at P = 2048 two pairs per
// CTA (35 % slower, 32-byte pieces of T) or four radix-8 passes of 16 values per thread (4 to 19 % slower).
#include <cuda_bf16.h>

#include <atomic>

#include "fft16.cuh"
#include "recon_internal.h"

namespace recon {
namespace {

template <int P>
struct RowsT {
  static constexpr int R = P >= 1024 ? 16 : 8;  // radix of the passes (the last one takes what is left)
  static constexpr int V = 2 * R;               // values a thread holds of its pair
  static constexpr int TT = P / V;              // threads per pair
  static constexpr int G = P >= 2048 ? 4 : (P >= 512 ? 8 : (P >= 256 ? 16 : 32));  // pairs per CTA
  static constexpr int NTH = G * TT;
  static constexpr int NT = P - R;              // twiddle table entries (fft_reg.cuh, fft16.cuh)
  static constexpr int MINB = P >= 1024 ? 2 : 4;
  static constexpr size_t smem = sizeof(float2) * ((size_t)NT + (size_t)G * P);
};

// Exchange entry of element i of pair p: i' G + p.  A half-warp's 64-bit accesses touch 16 / G
// neighbouring butterflies of G pairs; the low bits of i' carry the bits above the first radix, so that these
// are on distinct bank pairs in every pass (G >= 16: always).
template <int P>
__device__ __forceinline__ int swz(int i) {
  using C = RowsT<P>;
  constexpr int M = C::G >= 16 ? 0 : 16 / C::G - 1;
  return i ^ ((i / C::R) & M);
}

template <int R>
__device__ __forceinline__ void dft(float2* v) {
  fft16::dftR<R, true>(v);
}

// The passes from sub-length Ns on, the values of the passes before in `buf`.  On return v[q R + r] is
// element (j + q TT) + r P/R for the last pass's radix R (returned through last_radix).
template <int P, int Ns>
__device__ __forceinline__ void passes(float2 (&v)[RowsT<P>::V], float2* buf, const float2* tw, int j, int p) {
  using C = RowsT<P>;
  constexpr int rem = P / Ns, R = rem % C::R == 0 ? C::R : rem, NB = C::V / R, STRIDE = P / R;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NB; ++q)
#pragma unroll
    for (int r = 0; r < R; ++r) v[q * R + r] = buf[swz<P>(j + q * C::TT + r * STRIDE) * C::G + p];
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const float2* twk = tw + (Ns - C::R) + ((j + q * C::TT) & (Ns - 1)) * (R - 1) - 1;
#pragma unroll
    for (int r = 1; r < R; ++r) {
      const float2 w = twk[r];
      v[q * R + r] = fft::cmul(v[q * R + r], make_float2(w.x, -w.y));
    }
    dft<R>(v + q * R);
  }
  if constexpr (Ns * R < P) {
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int b = j + q * C::TT;
#pragma unroll
      for (int r = 0; r < R; ++r) buf[swz<P>((b / Ns) * Ns * R + (b & (Ns - 1)) + r * Ns) * C::G + p] = v[q * R + r];
    }
    passes<P, Ns * R>(v, buf, tw, j, p);
  }
}
template <int P>
__host__ __device__ constexpr int last_radix() {
  int ns = RowsT<P>::R;
  while ((P / ns) % RowsT<P>::R == 0 && P / ns > RowsT<P>::R) ns *= RowsT<P>::R;
  return P / ns;
}

template <bool WIDE>
__device__ __forceinline__ float4 row_pair(const float2* p, bool row2) {
  if constexpr (WIDE) return *reinterpret_cast<const float4*>(p);
  const float2 a = p[0], b = row2 ? p[1] : make_float2(0.f, 0.f);
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void store_pair(float* out, float2 v) { *reinterpret_cast<float2*>(out) = v; }
__device__ __forceinline__ void store_pair(__nv_bfloat16* out, float2 v) {
  *reinterpret_cast<__nv_bfloat162*>(out) = __floats2bfloat162_rn(v.x, v.y);
}
__device__ __forceinline__ void store_taps(float2* out, float a, float b) { *out = make_float2(a, b); }
__device__ __forceinline__ void store_taps(__nv_bfloat162* out, float a, float b) { *out = __floats2bfloat162_rn(a, b); }

// Entry: the stack's, a tap pair (float2, bfloat162) or with COLS a single value.  WIDE: c.tp is even, so that a row
// pair of T is one 16-byte load (a scratch too small for the even pitch takes two 8-byte ones).
template <int P, typename Entry, bool COLS, bool WIDE>
__global__ void __launch_bounds__(RowsT<P>::NTH, RowsT<P>::MINB) k_rows_inv(const float2* __restrict__ T,
                                                                          Entry* __restrict__ stack,
                                                                          const float2* __restrict__ twg,
                                                                          StageAConst c) {
  using C = RowsT<P>;
  constexpr int R = C::R, G = C::G, H = P / 2 + 1, B = P / R;  // B: butterflies of the first pass
  extern __shared__ __align__(16) float2 smem_rows[];
  float2 *tw = smem_rows, *buf = smem_rows + C::NT;
  const int p = threadIdx.x % G, j = threadIdx.x / G;
  const int n = blockIdx.z, k = blockIdx.y, vbase = blockIdx.x * 2 * G, v0 = vbase + 2 * p;
  float2 z[C::V];
  {
    // columns j + s B and (B - j) + s B, s < R / 2, of rows v0 and v0 + 1; j = 0 takes B / 2 for the second
    const int jb = j ? B - j : B / 2;
    const float2* Tk = T + (((size_t)n * c.nz_layers + k) * H) * c.tp + v0;
    const bool row1 = v0 < c.nw, row2 = v0 + 1 < c.nw;
    float4 a[R / 2], b[R / 2], ny = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int s = 0; s < R / 2; ++s) {
      a[s] = b[s] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (row1) {
        a[s] = row_pair<WIDE>(Tk + (size_t)(j + s * B) * c.tp, row2);
        b[s] = row_pair<WIDE>(Tk + (size_t)(jb + s * B) * c.tp, row2);
      }
    }
    if (row1 && j == 0) ny = row_pair<WIDE>(Tk + (size_t)(P / 2) * c.tp, row2);
    for (int i = threadIdx.x; i < C::NT; i += C::NTH) tw[i] = twg[i];
    if (!row2) {
#pragma unroll
      for (int s = 0; s < R / 2; ++s) a[s].z = a[s].w = b[s].z = b[s].w = 0.f;
      ny.z = ny.w = 0.f;
    }
    if (j == 0) a[0].y = a[0].w = 0.f;  // C2R: DC and Nyquist bins are real
    float2 ca[R / 2], cb[R / 2];        // the mirror images conj X1 + i conj X2
#pragma unroll
    for (int s = 0; s < R / 2; ++s) {
      z[s] = make_float2(a[s].x - a[s].w, a[s].y + a[s].z);
      z[R + s] = make_float2(b[s].x - b[s].w, b[s].y + b[s].z);
      ca[s] = make_float2(a[s].x + a[s].w, a[s].z - a[s].y);
      cb[s] = make_float2(b[s].x + b[s].w, b[s].z - b[s].y);
    }
#pragma unroll
    for (int s = 0; s < R / 2; ++s) {  // butterfly j's upper half mirrors butterfly B - j's lower half, and
      z[R - 1 - s] = cb[s];            // the other way round; 0 and B / 2 mirror themselves
      z[2 * R - 1 - s] = ca[s];
    }
    if (j == 0) {
#pragma unroll
      for (int s = 0; s < R / 2; ++s) z[2 * R - 1 - s] = cb[s];
#pragma unroll
      for (int s = 1; s < R / 2; ++s) z[R - s] = ca[s];
      z[R / 2] = make_float2(ny.x, ny.z);
    }
    dft<R>(z);
    dft<R>(z + R);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      buf[swz<P>(j * R + r) * G + p] = z[r];
      buf[swz<P>(jb * R + r) * G + p] = z[R + r];
    }
  }
  passes<P, R>(z, buf, tw, j, p);
  // elements u < nu <= P/2 (P is at least twice the image size) are kept: the last pass's butterflies that only
  // feed the others drop
  constexpr int RL = last_radix<P>(), NB = C::V / RL, STRIDE = P / RL;
  if constexpr (COLS) {
    if (v0 >= c.wp) return;
    Entry* out = stack + ((size_t)n * c.nz_layers + k) * c.nu * c.wp + v0;
#pragma unroll
    for (int q = 0; q < NB; ++q)
#pragma unroll
      for (int r = 0; r < RL / 2; ++r) {
        const int u = j + q * C::TT + r * STRIDE;
        if (u < c.nu) store_pair(out + (size_t)u * c.wp, z[q * RL + r]);
      }
  } else {
    // through shared memory, so that the stores run along the rows: pair p's values at p PS + u
    constexpr int PS = P / 2 + (G >= 16 ? 1 : 16 / G);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NB; ++q)
#pragma unroll
      for (int r = 0; r < RL / 2; ++r) buf[p * PS + j + q * C::TT + r * STRIDE] = z[q * RL + r];
    __syncthreads();
    const int po = threadIdx.x / C::TT, jo = threadIdx.x % C::TT, v = vbase + 2 * po, sp = c.su;
    Entry* Lk = stack + ((size_t)n * c.nz_layers + k) * c.layer_elems;
    if (v < c.nv) {
      const bool two = v + 1 < c.nv;
      const float2* y = buf + po * PS;
      Entry *r1 = Lk + (size_t)(v + 1) * sp, *r2 = r1 + sp;
      for (int cc = jo; cc <= c.nu; cc += C::TT) {  // pair column: (Y[cc - 1], Y[cc])
        const float2 left = cc >= 1 ? y[cc - 1] : make_float2(0.f, 0.f);
        const float2 right = cc < c.nu ? y[cc] : make_float2(0.f, 0.f);
        store_taps(r1 + cc, left.x, right.x);
        if (two) store_taps(r2 + cc, left.y, right.y);
      }
    }
    if (blockIdx.x == 0)  // top border row
      for (int i = threadIdx.x; i < sp; i += C::NTH) store_taps(Lk + i, 0.f, 0.f);
    if (vbase + 2 * G >= c.nv)  // bottom border row
      for (int i = threadIdx.x; i < sp; i += C::NTH) store_taps(Lk + (size_t)(c.nv + 1) * sp + i, 0.f, 0.f);
  }
}

template <int P, typename Entry, bool COLS, bool WIDE>
cudaError_t launch(const StageAConst& c, const float2* T, void* stack, const float2* twp, int cnt, cudaStream_t stream) {
  using C = RowsT<P>;
  static std::atomic<unsigned long long> attr_set{0};  // devices on which the shared-memory limit is raised
  if constexpr (C::smem > 48 * 1024) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 64 || !(attr_set.load() >> dev & 1ull)) {
      const cudaError_t e =
          cudaFuncSetAttribute(k_rows_inv<P, Entry, COLS, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::smem);
      if (e != cudaSuccess) return e;
      if (dev < 64) attr_set.fetch_or(1ull << dev);
    }
  }
  const float2* tw = twp + (P >= 1024 ? P - 8 : 0);  // the 16-value table follows the 8-value one
  const dim3 grid((c.nw + 2 * C::G - 1) / (2 * C::G), c.nz_layers, cnt);
  k_rows_inv<P, Entry, COLS, WIDE><<<grid, C::NTH, C::smem, stream>>>(T, (Entry*)stack, tw, c);
  return cudaGetLastError();
}
template <int P, bool WIDE>
cudaError_t launch(const StageAConst& c, const float2* T, void* stack, const float2* twp, int cnt, cudaStream_t s) {
  if (c.cols)
    return c.stack_bf16 ? launch<P, __nv_bfloat16, true, WIDE>(c, T, stack, twp, cnt, s)
                        : launch<P, float, true, WIDE>(c, T, stack, twp, cnt, s);
  return c.stack_bf16 ? launch<P, __nv_bfloat162, false, WIDE>(c, T, stack, twp, cnt, s)
                      : launch<P, float2, false, WIDE>(c, T, stack, twp, cnt, s);
}
template <int P>
cudaError_t launch(const StageAConst& c, const float2* T, void* stack, const float2* twp, int cnt, cudaStream_t s) {
  return c.tp & 1 ? launch<P, false>(c, T, stack, twp, cnt, s) : launch<P, true>(c, T, stack, twp, cnt, s);
}

}  // namespace

cudaError_t launch_rows_inv(const StageAConst& c, const float2* T, void* stack, const float2* twp, int cnt,
                            cudaStream_t s) {
  switch (c.P) {
    case 16: return launch<16>(c, T, stack, twp, cnt, s);
    case 32: return launch<32>(c, T, stack, twp, cnt, s);
    case 64: return launch<64>(c, T, stack, twp, cnt, s);
    case 128: return launch<128>(c, T, stack, twp, cnt, s);
    case 256: return launch<256>(c, T, stack, twp, cnt, s);
    case 512: return launch<512>(c, T, stack, twp, cnt, s);
    case 1024: return launch<1024>(c, T, stack, twp, cnt, s);
    case 2048: return launch<2048>(c, T, stack, twp, cnt, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace recon
