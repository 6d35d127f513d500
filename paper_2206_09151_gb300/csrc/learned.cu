// Learned regulariser of the CTF inverse: eps_theta = softplus(MLP(x)) per (direction n,
// layer k, radial bin b) replaces the Tikhonov eps of Eq. 11 (chosen "ad hoc" in Sec. 3).
// Features x: log10 of the bin's signal-to-noise ratio (radial power spectrum of the
// contrast over the Poisson floor (NSR M)^2 per DFT coefficient, the Parseval scaling of
// Sec. 3's noise filter) / 3, clamped to [-1, 2]; the bin-centre radius / (P/2); the layer's
// effective defocus lambda (R_n - z_k) / delta^2 / 100.  Network 3 -> 64 -> 64 -> 1 (ReLU),
// FP32 weights W1[64][3], b1, W2[64][64], b2, w3, b3.
//
// Kernels:
//   k_cols_forward<P>  column FFTs of the row spectra (as in k_cols), then the radial power
//                      sum_{q in b} mult |G(q)|^2 (mult = 2 for the columns standing for two
//                      of the full grid) and, for training, the column spectra themselves
//   k_eps_table        one thread per (n, k, b): SNR, features, MLP, eps (and the features, for training)
//   k_train_loss       per frequency of every (image, layer): H G - T, the loss sums and
//                      d loss / d eps_b
//   k_mlp_backward     backpropagation of d loss / d eps to the 4481 parameters
//   k_adam             Adam (Kingma and Ba 2015) on the parameters
#include <cuda_runtime.h>

#include "columns.cuh"
#include "fft_reg.cuh"
#include "learned.cuh"
#include "recon_internal.h"

namespace recon {
namespace {

constexpr int kThreads = 256;
constexpr int H = kMlpHidden;

template <int P>
__host__ __device__ constexpr int groups() {
  return kThreads / (P / 8) > 0 ? kThreads / (P / 8) : 1;
}

__device__ __forceinline__ int isqrt_u32(uint32_t x) {
  int r = (int)sqrtf((float)x);
  while ((uint32_t)r * (uint32_t)r > x) --r;
  while ((uint32_t)(r + 1) * (uint32_t)(r + 1) <= x) ++r;
  return r;
}

__device__ __forceinline__ int radial_bin(const LearnConst& lc, uint32_t msq) {
  const int b = isqrt_u32(msq) / lc.bin_width;
  return b < lc.n_bins - 1 ? b : lc.n_bins - 1;
}

__device__ __forceinline__ float softplus(float o) { return o > 20.f ? o : log1pf(expf(o)); }

// ----------------------------------------------------------------- column forward FFT
template <int P>
__global__ void __launch_bounds__(kThreads) k_cols_forward(const float2* __restrict__ S, float2* __restrict__ G_out,
                                                            float* __restrict__ pow, const float2* __restrict__ twg,
                                                            StageAConst c, LearnConst lc) {
  constexpr int TT = P / 8, CB = groups<P>(), L = fft::buffer_len(P, CB), NT = fft::pass_table_len(P);
  __shared__ float2 tw[NT];
  __shared__ float2 buf_all[CB * L];
  __shared__ float hist[kMaxBins];
  const int g = threadIdx.x / TT, j = threadIdx.x % TT;
  float2* buf = buf_all + g * L;
  for (int i = threadIdx.x; i < NT; i += kThreads) tw[i] = twg[i];
  for (int i = threadIdx.x; i < lc.n_bins; i += kThreads) hist[i] = 0.f;
  const int n = blockIdx.y;
  const int c0 = blockIdx.x * CB;
  const int col = c0 + g;
  const float2* Sn = S + (size_t)n * c.nv * c.half;
  for (int idx = threadIdx.x; idx < c.nv * CB; idx += kThreads) {
    const int t = idx % CB, v = idx / CB;
    buf_all[t * L + fft::padded(v)] = (c0 + t < c.half) ? Sn[(size_t)v * c.half + c0 + t] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  float2 x[8];
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const int v = j + s * TT;
    x[s] = v < c.nv ? buf[fft::padded(v)] : make_float2(0.f, 0.f);
  }
  fft::block_fft<P, false>(x, buf, tw, j);
  const bool ok = col < c.half;
  if (ok && G_out) {
    float2* out = G_out + ((size_t)n * c.half + col) * P;
#pragma unroll
    for (int s = 0; s < 8; ++s) out[j + s * TT] = x[s];
  }
  if (pow) {
    if (ok) {
      const float mult = (col == 0 || col == P / 2) ? 1.f : 2.f;
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        const int m = j + s * TT;
        const int mv = m < P / 2 ? m : m - P;
        const int b = radial_bin(lc, (uint32_t)(col * col + mv * mv));
        atomicAdd(&hist[b], mult * (x[s].x * x[s].x + x[s].y * x[s].y));
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < lc.n_bins; i += kThreads)
      if (hist[i] != 0.f) atomicAdd(&pow[(size_t)n * lc.n_bins + i], hist[i]);
  }
}

// ----------------------------------------------------------------- MLP forward
__device__ __forceinline__ void features(const LearnConst& lc, const float* __restrict__ pow,
                                         const float* __restrict__ cnt, const float* __restrict__ x2tab, int n,
                                         int k, int b, int n_layers, float x[3]) {
  const float N0 = lc.noise_floor;
  const float pw = pow[(size_t)n * lc.n_bins + b] / fmaxf(cnt[b], 1.f);
  const float snr = fmaxf(pw - N0, 1e-3f * N0) / N0;
  x[0] = fminf(fmaxf(log10f(snr), -3.f), 6.f) * (1.f / 3.f);
  x[1] = ((float)b + 0.5f) * (float)lc.bin_width * lc.inv_half_p;
  x[2] = x2tab[(size_t)n * n_layers + k];
}

// The network's parameters in shared memory with W2 transposed, W2T[q][i], so that a
// hidden unit q's weights into four consecutive units i are one 16-byte load.
struct MlpWeights {
  float W1[3 * H], b1[H], W2T[H][H], b2[H], w3[H], b3;
};
__device__ __forceinline__ void load_weights(MlpWeights& w, const float* __restrict__ theta) {
  for (int i = threadIdx.x; i < kMlpParams; i += blockDim.x) {
    const float v = theta[i];
    int o = i;
    if (o < 3 * H) { w.W1[o] = v; continue; }
    if ((o -= 3 * H) < H) { w.b1[o] = v; continue; }
    if ((o -= H) < H * H) { w.W2T[o % H][o / H] = v; continue; }
    if ((o -= H * H) < H) { w.b2[o] = v; continue; }
    if ((o -= H) < H) { w.w3[o] = v; continue; }
    w.b3 = v;
  }
}

// One row (direction, layer, bin) per thread: its 64 second-layer sums stay in registers as 32
// packed FP32x2 pairs while the first layer's units q pass by, so the sums are 64 independent
// chains (a row-by-row product was one dependent chain of 64 per unit) and a unit q costs 16
// shared 16-byte loads and 32 packed FMAs.  Every sum runs over q in ascending order.  For
// training the row's inputs are kept (16 bytes a row) and the backward pass recomputes the
// activations: storing them cost 132 scattered 4-byte stores per row (46 592 rows, 128^2
// images: 83 us with the stores, 29 us now).
__global__ void __launch_bounds__(kThreads) k_eps_table(const float* __restrict__ pow, const float* __restrict__ cnt,
                                                         const float* __restrict__ x2tab,
                                                         const float* __restrict__ theta, float* __restrict__ eps,
                                                         float4* __restrict__ inputs, LearnConst lc, int n_dirs,
                                                         int n_layers, int dir_begin) {
  __shared__ __align__(16) MlpWeights w;
  load_weights(w, theta);
  __syncthreads();
  const size_t rows = (size_t)n_dirs * n_layers * lc.n_bins;
  const size_t row = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= rows) return;
  const int b = (int)(row % lc.n_bins);
  const int k = (int)((row / lc.n_bins) % n_layers);
  const int n = (int)(row / ((size_t)lc.n_bins * n_layers));
  float x[3];
  features(lc, pow, cnt, x2tab, n, k, b, n_layers, x);
  x[2] = x2tab[(size_t)(dir_begin + n) * n_layers + k];
  float2 a[H / 2];
#pragma unroll
  for (int i = 0; i < H / 2; ++i) a[i] = make_float2(w.b2[2 * i], w.b2[2 * i + 1]);
#pragma unroll 2
  for (int q = 0; q < H; ++q) {
    const float h =
        fmaxf(fmaf(w.W1[3 * q], x[0], fmaf(w.W1[3 * q + 1], x[1], fmaf(w.W1[3 * q + 2], x[2], w.b1[q]))), 0.f);
    const float2 hh = make_float2(h, h);
#pragma unroll
    for (int i = 0; i < H / 4; ++i) {
      const float4 v = *reinterpret_cast<const float4*>(&w.W2T[q][4 * i]);
      a[2 * i] = __ffma2_rn(make_float2(v.x, v.y), hh, a[2 * i]);
      a[2 * i + 1] = __ffma2_rn(make_float2(v.z, v.w), hh, a[2 * i + 1]);
    }
  }
  float o = w.b3;
#pragma unroll
  for (int i = 0; i < H / 2; ++i) {
    o = fmaf(w.w3[2 * i], fmaxf(a[i].x, 0.f), o);
    o = fmaf(w.w3[2 * i + 1], fmaxf(a[i].y, 0.f), o);
  }
  if (inputs) inputs[row] = make_float4(x[0], x[1], x[2], 0.f);
  eps[row] = softplus(o) * lc.eps_scale;
}

// ----------------------------------------------------------------- training loss
// Loss and d loss / d eps of one image over kLossCols spectrum columns: a thread keeps its
// kLossCols * P / 256 frequencies' spectrum values, phase integers and bins over all layers.
// The bins of a warp's 32 consecutive frequencies are equal in runs, so each run is summed by
// shuffles and one lane adds it to the shared histogram: a shared float atomic per frequency
// was a compare-and-swap loop contended by the whole warp.  The loss sums are float pairs
// (sum and rounding error, two-sum) per thread and FP64 only across threads: FP64 arithmetic per
// frequency bound the kernel before (32 images, 128^2, 16 layers: 473 us, now 131 us).
constexpr int kLossCols = 4;
constexpr int kLossLayers = 8;  // layers per pass over the shared histograms (one barrier pair for all)

struct TwoSum {
  float s = 0.f, e = 0.f;
  __device__ __forceinline__ void add(float v) {
    const float t = s + v, b = t - s;
    e += (s - (t - b)) + (v - b);
    s = t;
  }
  // an overflowed sum is infinite, its rounding error not a number
  __device__ __forceinline__ double value() const { return isinf(s) ? (double)s : (double)s + e; }
};

template <int P>
__global__ void __launch_bounds__(kThreads) k_train_loss(const float2* __restrict__ G, const float2* __restrict__ T,
                                                          const float* __restrict__ eps,
                                                          const uint64_t* __restrict__ uA, StageAConst c,
                                                          LearnConst lc, double* __restrict__ sums,
                                                          double* __restrict__ deps) {
  // a histogram per warp where a warp's runs have distinct bins (32 consecutive frequencies of one
  // column and one sign of m_v, P >= 64): plain adds; else one for the CTA, with atomics
  constexpr int W = P >= 64 ? kThreads / 32 : 1;
  __shared__ float hist[W][kLossLayers][kMaxBins];
  __shared__ double part[2][kThreads / 32];
  constexpr int E = (kLossCols * P + kThreads - 1) / kThreads;
  const int n = blockIdx.y, nl = c.nz_layers;
  const int lane = threadIdx.x & 31;
  const size_t plane = (size_t)c.half * P;
  const size_t first = (size_t)blockIdx.x * kLossCols * P;
  float2 g[E];
  uint32_t msq[E], info[E];  // info: bin | head << 8 | "lane + 2^i is in my run" << (9 + i)
  uint32_t base[E];
  float mult[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const size_t idx = first + (size_t)e * kThreads + threadIdx.x;
    const bool in = e * kThreads + threadIdx.x < kLossCols * P && idx < plane;
    const int col = in ? (int)(idx / P) : 0, m = in ? (int)(idx % P) : 0;
    const int mv = m < P / 2 ? m : m - P;
    msq[e] = (uint32_t)(col * col + mv * mv);
    const uint64_t m64 = msq[e];
    base[e] = (uint32_t)((c.uC * (m64 * m64) - c.uW) >> 32);
    g[e] = in ? G[(size_t)n * plane + idx] : make_float2(0.f, 0.f);
    mult[e] = !in ? 0.f : ((col == 0 || col == P / 2) ? 1.f : 2.f);
    const int b = radial_bin(lc, msq[e]);
    const int left = __shfl_up_sync(0xffffffffu, b, 1);
    const bool head = lane == 0 || left != b;
    const uint32_t heads = __ballot_sync(0xffffffffu, head);
    info[e] = (uint32_t)b | (head ? 256u : 0u);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      // no run starts in (lane, lane + 2^i]
      const uint32_t span = (((2u << ((1 << i) - 1)) - 1u) << lane) << 1;
      if (lane + (1 << i) < 32 && (heads & span) == 0) info[e] |= 512u << i;
    }
  }
  TwoSum num, den;
  for (int k0 = 0; k0 < nl; k0 += kLossLayers) {
    for (int i = threadIdx.x; i < W * kLossLayers * kMaxBins; i += kThreads) (&hist[0][0][0])[i] = 0.f;
    __syncthreads();
    const int kn = min(kLossLayers, nl - k0);
#pragma unroll 2
    for (int kk = 0; kk < kn; ++kk) {
      const int k = k0 + kk;
      const uint64_t uAk = uA[(size_t)n * nl + k];
      const uint32_t a_hi = (uint32_t)(uAk >> 32), a_lo = (uint32_t)uAk;
      const float* eps_k = eps + ((size_t)n * nl + k) * lc.n_bins;
      const float2* Tk = T + ((size_t)n * nl + k) * plane + first + threadIdx.x;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const float2 tq = mult[e] != 0.f ? Tk[e * kThreads] : make_float2(0.f, 0.f);
        const uint32_t hi = a_hi * msq[e] + __umulhi(a_lo, msq[e]) + base[e];
        const float sn = sin_half_turns((int32_t)hi);
        const float inv = __frcp_rn(fmaf(sn, sn, eps_k[info[e] & 255u]));
        const float Hq = c.pref * sn * inv;
        const float rx = Hq * g[e].x - tq.x, ry = Hq * g[e].y - tq.y;
        num.add(mult[e] * (rx * rx + ry * ry));
        den.add(mult[e] * (tq.x * tq.x + tq.y * tq.y));
        float d = -2.f * mult[e] * (rx * g[e].x + ry * g[e].y) * (Hq * inv);  // dH / d eps = -Hq inv
#pragma unroll
        for (int i = 0; i < 5; ++i) {
          const float o = __shfl_down_sync(0xffffffffu, d, 1 << i);
          if (info[e] & (512u << i)) d += o;
        }
        if (info[e] & 256u) {
          float* h = &hist[W > 1 ? threadIdx.x >> 5 : 0][kk][info[e] & 255u];
          if constexpr (W > 1) *h += d;
          else atomicAdd(h, d);
        }
        if constexpr (W > 1) __syncwarp();
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kn * lc.n_bins; i += kThreads) {
      float v = 0.f;
#pragma unroll
      for (int w = 0; w < W; ++w) v += hist[w][i / lc.n_bins][i % lc.n_bins];
      if (v != 0.f) atomicAdd(&deps[((size_t)n * nl + k0) * lc.n_bins + i], (double)v);
    }
    __syncthreads();
  }
  double a = num.value(), d = den.value();
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    d += __shfl_down_sync(0xffffffffu, d, o);
  }
  if (lane == 0) {
    part[0][threadIdx.x >> 5] = a;
    part[1][threadIdx.x >> 5] = d;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a = d = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) {
      a += part[0][w];
      d += part[1][w];
    }
    atomicAdd(&sums[0], a);
    atomicAdd(&sums[1], d);
  }
}

// ----------------------------------------------------------------- backward and Adam
// Backpropagation as small matrix products: a CTA takes chunks of 128 rows, recomputes their
// activations from the inputs (A2 = H1 W2^T), forms D1 = D2 W2 and adds D2^T H1 to its share of
// the gradient, which stays in registers over all its chunks and is added to the global
// gradient once at the end.  A thread's blocks are 8 rows x 4 units of A2 and D1 and 4 x 4 of dW2,
// so a shared-memory float feeds two to three FMAs (its return bandwidth is what bounds the
// products).  Before, 4481 contended shared atomics per row bound the kernel (46 592 rows:
// 4.30 ms, now 52 us).  Rows beyond the last count as zero through d_o = 0.
constexpr int kBwRows = 128, kBwPitch = kBwRows + 4;  // [unit][row] arrays, rows padded against bank conflicts

struct BwShared {
  MlpWeights w;
  alignas(16) float W2[H][H];         // [i][q]
  alignas(16) float h1[H][kBwPitch];  // relu(a1), [unit][row]
  alignas(16) float d2[H][kBwPitch];  // d loss / d a2; before that the 16 partial sums of each row's output
  float4 x[kBwRows];
  float d_o[kBwRows];
};

__global__ void __launch_bounds__(kThreads, 2) k_mlp_backward(const float4* __restrict__ inputs,
                                                            const double* __restrict__ deps,
                                                            const double* __restrict__ sums,
                                                            const float* __restrict__ theta, float* __restrict__ grad,
                                                            size_t rows) {
  static_assert(H == 64 && kThreads == 256 && kBwRows == 128, "16 x 16 threads of 8 rows x 4 units");
  extern __shared__ __align__(16) unsigned char smem_bw[];
  BwShared& m = *reinterpret_cast<BwShared*>(smem_bw);
  load_weights(m.w, theta);
  for (int i = threadIdx.x; i < H * H; i += kThreads) m.W2[i / H][i % H] = theta[4 * H + i];
  // rows ra .. ra + 3 and ra + 64 .. ra + 67, units u0 .. u0 + 3; dW2 rows i = ti + 16 a, columns q = tq + 16 b
  const int ra = (threadIdx.x & 15) * 4, u0 = (threadIdx.x >> 4) * 4;
  const int tq = threadIdx.x & 15, ti = threadIdx.x >> 4;
  float gW2[4][4] = {}, gw3[4] = {}, gb2[4] = {}, gb1[4] = {}, gW1[4][3] = {}, gb3 = 0.f;
  const double inv_den = 1.0 / sums[1];
  // D[row][unit] += sum_q A[q][row] B[q][unit]
  auto product = [&](const float(*A)[kBwPitch], const float(*B)[H], float(&acc)[8][4]) {
#pragma unroll 4
    for (int q = 0; q < H; ++q) {
      const float4 a0 = *reinterpret_cast<const float4*>(&A[q][ra]);
      const float4 a1 = *reinterpret_cast<const float4*>(&A[q][ra + 64]);
      const float4 b = *reinterpret_cast<const float4*>(&B[q][u0]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[r][i] = fmaf(bv[i], av[r], acc[r][i]);
    }
  };
  for (size_t r0 = (size_t)blockIdx.x * kBwRows; r0 < rows; r0 += (size_t)gridDim.x * kBwRows) {
    __syncthreads();  // weights in place; the previous chunk's arrays are free
    if (threadIdx.x < kBwRows)
      m.x[threadIdx.x] =
          r0 + threadIdx.x < rows ? inputs[r0 + threadIdx.x] : make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float* W1 = m.w.W1 + 3 * (u0 + i);
      const float b1 = m.w.b1[u0 + i];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const float4 x = m.x[ra + 64 * h + r];
          v[r] = fmaxf(fmaf(W1[0], x.x, fmaf(W1[1], x.y, fmaf(W1[2], x.z, b1))), 0.f);
        }
        *reinterpret_cast<float4*>(&m.h1[u0 + i][ra + 64 * h]) = make_float4(v[0], v[1], v[2], v[3]);
      }
    }
    __syncthreads();
    float acc[8][4];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[r][i] = m.w.b2[u0 + i];
    product(m.h1, m.w.W2T, acc);  // a2
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      float o = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) o = fmaf(m.w.w3[u0 + i], fmaxf(acc[r][i], 0.f), o);
      m.d2[threadIdx.x >> 4][ra + (r & 3) + (r >> 2) * 64] = o;
    }
    __syncthreads();
    if (threadIdx.x < kBwRows) {
      float o = m.w.b3;
#pragma unroll
      for (int t = 0; t < 16; ++t) o += m.d2[t][threadIdx.x];
      const float d_eps = r0 + threadIdx.x < rows ? (float)(deps[r0 + threadIdx.x] * inv_den) : 0.f;
      const float d_o = d_eps / (1.f + expf(-o));  // softplus' = sigmoid
      m.d_o[threadIdx.x] = d_o;
      gb3 += d_o;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float w3 = m.w.w3[u0 + i];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const float a2 = acc[4 * h + r][i], d_o = m.d_o[ra + 64 * h + r];
          v[r] = a2 > 0.f ? d_o * w3 : 0.f;
          gw3[i] = fmaf(d_o, fmaxf(a2, 0.f), gw3[i]);
          gb2[i] += v[r];
        }
        *reinterpret_cast<float4*>(&m.d2[u0 + i][ra + 64 * h]) = make_float4(v[0], v[1], v[2], v[3]);
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[r][i] = 0.f;
    product(m.d2, m.W2, acc);  // d loss / d h1
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int row = ra + (r & 3) + (r >> 2) * 64;
      const float4 x = m.x[row];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float d = m.h1[u0 + i][row] > 0.f ? acc[r][i] : 0.f;
        gb1[i] += d;
        gW1[i][0] = fmaf(d, x.x, gW1[i][0]);
        gW1[i][1] = fmaf(d, x.y, gW1[i][1]);
        gW1[i][2] = fmaf(d, x.z, gW1[i][2]);
      }
    }
#pragma unroll 2
    for (int r = 0; r < kBwRows; r += 4) {
      float4 h[4], d[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        h[a] = *reinterpret_cast<const float4*>(&m.h1[tq + 16 * a][r]);
        d[a] = *reinterpret_cast<const float4*>(&m.d2[ti + 16 * a][r]);
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
          gW2[a][b] = fmaf(d[a].w, h[b].w,
                           fmaf(d[a].z, h[b].z, fmaf(d[a].y, h[b].y, fmaf(d[a].x, h[b].x, gW2[a][b]))));
    }
  }
  // the 16 row groups of a unit are one half-warp: sum, then one global add per unit
  auto reduce = [](float v) {
#pragma unroll
    for (int s = 8; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
    return v;
  };
  float* const d_b1 = grad + 3 * H;
  float* const d_W2 = d_b1 + H;
  float* const d_b2 = d_W2 + H * H;
  float* const d_w3 = d_b2 + H;
  const bool lead = (threadIdx.x & 15) == 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float v3 = reduce(gw3[i]), v2 = reduce(gb2[i]), v1 = reduce(gb1[i]);
    const float w0 = reduce(gW1[i][0]), w1 = reduce(gW1[i][1]), w2 = reduce(gW1[i][2]);
    if (lead) {
      atomicAdd(&d_w3[u0 + i], v3);
      atomicAdd(&d_b2[u0 + i], v2);
      atomicAdd(&d_b1[u0 + i], v1);
      atomicAdd(&grad[3 * (u0 + i)], w0);
      atomicAdd(&grad[3 * (u0 + i) + 1], w1);
      atomicAdd(&grad[3 * (u0 + i) + 2], w2);
    }
  }
  gb3 = reduce(gb3);
  if (lead && threadIdx.x < kBwRows) atomicAdd(&d_w3[H], gb3);
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) atomicAdd(&d_W2[(ti + 16 * a) * H + tq + 16 * b], gW2[a][b]);
}

__global__ void k_adam(float* __restrict__ theta, float* __restrict__ grad, float* __restrict__ m1,
                       float* __restrict__ m2, int step, float lr, const double* __restrict__ sums,
                       float* __restrict__ loss_out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0 && loss_out) *loss_out = (float)(sums[0] / sums[1]);
  if (i >= kMlpParams) return;
  const float b1 = 0.9f, b2 = 0.999f;
  const float g = grad[i];
  const float m = b1 * m1[i] + (1.f - b1) * g;
  const float v = b2 * m2[i] + (1.f - b2) * g * g;
  m1[i] = m;
  m2[i] = v;
  const float mh = m / (1.f - powf(b1, (float)step));
  const float vh = v / (1.f - powf(b2, (float)step));
  theta[i] -= lr * mh / (sqrtf(vh) + 1e-8f);
  grad[i] = 0.f;
}

__global__ void k_loss_only(const double* __restrict__ sums, float* __restrict__ loss_out) {
  if (threadIdx.x == 0 && blockIdx.x == 0) *loss_out = (float)(sums[0] / sums[1]);
}

template <int P>
cudaError_t cols_forward_p(const StageAConst& c, const LearnConst& lc, const float2* S, float2* G_out, float* pow,
                           const float2* twp, int n_dirs, cudaStream_t s) {
  constexpr int G = groups<P>();
  k_cols_forward<P><<<dim3((c.half + G - 1) / G, n_dirs), kThreads, 0, s>>>(S, G_out, pow, twp, c, lc);
  return cudaGetLastError();
}

template <int P>
cudaError_t train_loss_p(const StageAConst& c, const LearnConst& lc, const float2* G, const float2* T,
                         const float* eps, const uint64_t* uA, int n_img, double* sums, double* deps,
                         cudaStream_t s) {
  k_train_loss<P><<<dim3((c.half + kLossCols - 1) / kLossCols, n_img), kThreads, 0, s>>>(G, T, eps, uA, c, lc, sums,
                                                                                        deps);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_cols_forward(const StageAConst& c, const LearnConst& lc, const float2* S, float2* G_out,
                                float* pow, const float2* twp, int n_dirs, cudaStream_t s) {
  if (n_dirs <= 0) return cudaSuccess;
  switch (c.P) {
    case 16: return cols_forward_p<16>(c, lc, S, G_out, pow, twp, n_dirs, s);
    case 32: return cols_forward_p<32>(c, lc, S, G_out, pow, twp, n_dirs, s);
    case 64: return cols_forward_p<64>(c, lc, S, G_out, pow, twp, n_dirs, s);
    case 128: return cols_forward_p<128>(c, lc, S, G_out, pow, twp, n_dirs, s);
    case 256: return cols_forward_p<256>(c, lc, S, G_out, pow, twp, n_dirs, s);
    case 512: return cols_forward_p<512>(c, lc, S, G_out, pow, twp, n_dirs, s);
    case 1024: return cols_forward_p<1024>(c, lc, S, G_out, pow, twp, n_dirs, s);
    case 2048: return cols_forward_p<2048>(c, lc, S, G_out, pow, twp, n_dirs, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_eps_table(const LearnConst& lc, const float* pow, const float* cnt, const float* x2tab,
                             const float* theta, float* eps, float4* inputs, int n_dirs, int n_layers, int dir_begin,
                             cudaStream_t s) {
  const size_t rows = (size_t)n_dirs * n_layers * lc.n_bins;
  if (rows == 0) return cudaSuccess;
  k_eps_table<<<(unsigned)((rows + kThreads - 1) / kThreads), kThreads, 0, s>>>(pow, cnt, x2tab, theta, eps, inputs,
                                                                                lc, n_dirs, n_layers, dir_begin);
  return cudaGetLastError();
}

cudaError_t launch_train_step(const StageAConst& c, const LearnConst& lc, const float2* G, const float2* T,
                              const float* eps, const uint64_t* uA, const float4* inputs, const float* theta_dev,
                              float* theta_upd, float* grad, float* m1, float* m2, int n_img, double* sums,
                              double* deps, int step, float lr, float* loss_out, cudaStream_t s) {
  const size_t rows = (size_t)n_img * c.nz_layers * lc.n_bins;
  cudaError_t e;
  switch (c.P) {
    case 16: e = train_loss_p<16>(c, lc, G, T, eps, uA, n_img, sums, deps, s); break;
    case 32: e = train_loss_p<32>(c, lc, G, T, eps, uA, n_img, sums, deps, s); break;
    case 64: e = train_loss_p<64>(c, lc, G, T, eps, uA, n_img, sums, deps, s); break;
    case 128: e = train_loss_p<128>(c, lc, G, T, eps, uA, n_img, sums, deps, s); break;
    case 256: e = train_loss_p<256>(c, lc, G, T, eps, uA, n_img, sums, deps, s); break;
    case 512: e = train_loss_p<512>(c, lc, G, T, eps, uA, n_img, sums, deps, s); break;
    case 1024: e = train_loss_p<1024>(c, lc, G, T, eps, uA, n_img, sums, deps, s); break;
    case 2048: e = train_loss_p<2048>(c, lc, G, T, eps, uA, n_img, sums, deps, s); break;
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  // two CTAs per SM: the per-CTA share of the gradient (4481 global atomics) is paid once for all
  // of a CTA's rows
  constexpr size_t smem = sizeof(BwShared);
  e = cudaFuncSetAttribute(k_mlp_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const size_t chunks = (rows + kBwRows - 1) / kBwRows, cap = 2 * (size_t)device_sm_count();
  k_mlp_backward<<<(unsigned)(chunks < cap ? chunks : cap), kThreads, smem, s>>>(inputs, deps, sums, theta_dev, grad,
                                                                                rows);
  if (step > 0)
    k_adam<<<(kMlpParams + 255) / 256, 256, 0, s>>>(theta_upd, grad, m1, m2, step, lr, sums, loss_out);
  else
    k_loss_only<<<1, 32, 0, s>>>(sums, loss_out);
  return cudaGetLastError();
}

}  // namespace recon
