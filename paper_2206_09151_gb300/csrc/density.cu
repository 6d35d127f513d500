// Sampling-matrix construction for the density weighting of arbitrary scans (see
// density.cuh): the trilinear splat of every direction's sub-sampled DFT grid, and the
// band sum that sets the regulariser eps_S.
#include "density.cuh"

namespace recon {
namespace {

// Adds w0 and w1 to cells `i` and i + 1: one 16-byte vector reduction where they lie in one aligned group of four
// (the other two get zeros), else one each.
__device__ __forceinline__ void add_two(float* S, int i, float w0, float w1) {
  const int a = i & 3;
  if (a == 3) {
    atomicAdd(S + i, w0);
    atomicAdd(S + i + 1, w1);
    return;
  }
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(S + (i - a)), "f"(a == 0 ? w0 : 0.f),
               "f"(a == 0 ? w1 : (a == 1 ? w0 : 0.f)), "f"(a == 1 ? w1 : (a == 2 ? w0 : 0.f)), "f"(a == 2 ? w1 : 0.f)
               : "memory");
}

// The samples at q; their mirror images at -q are added by k_density_mirror.  L2 atomics bound it: 240
// directions of 128 x 128 samples (P = 2048) 97 us, 266 with 16 scalar atomics per sample, both signs here; the
// mirror pass 24 us, the band sum alone took 36 with 64-bit divisions.
__global__ void k_density_splat(const DirParams* __restrict__ dirs, DensityConst dc, int P, float* __restrict__ S) {
  const int n = blockIdx.y;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int n1 = dc.n_samples1;
  if (i >= n1 * n1) return;
  const DirParams& d = dirs[n];
  const float mu = (float)(-P / 2 + (i % n1) * dc.s);
  const float mv = (float)(-P / 2 + (i / n1) * dc.s);
  const float qx = (mu * d.af[0] + mv * d.bf[0]) * dc.inv_s;
  const float qy = (mu * d.af[1] + mv * d.bf[1]) * dc.inv_s;
  const float qz = (mu * d.af[2] + mv * d.bf[2]) * dc.inv_s;
  const float w = 0.5f * (float)(dc.s * dc.s);  // the sample at q and its mirror -q, half weight each
  const float bx = floorf(qx), by = floorf(qy), bz = floorf(qz);
  const float fx = qx - bx, fy = qy - by, fz = qz - bz;
  const int ix = (int)bx + dc.Gh, iy = (int)by + dc.Gh, iz = (int)bz + dc.Gh;
#pragma unroll
  for (int dz = 0; dz < 2; ++dz)
#pragma unroll
    for (int dy = 0; dy < 2; ++dy) {
      const float wt = (dy ? fy : 1.f - fy) * (dz ? fz : 1.f - fz) * w;
      add_two(S, ((iz + dz) * dc.G + (iy + dy)) * dc.G + ix, (1.f - fx) * wt, fx * wt);  // G <= 187: 32-bit indices
    }
}

// S(q) + S(-q) into both cells, and the sum over the band.
__global__ void k_density_mirror(float* __restrict__ S, DensityConst dc, double* __restrict__ out) {
  __shared__ double part[32];
  const int total = dc.G * dc.G * dc.G;
  const int r2max = (dc.Gh - 2) * (dc.Gh - 2);
  double acc = 0.0;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c <= total / 2; c += gridDim.x * blockDim.x) {
    const int row = c / dc.G, x = c - row * dc.G - dc.Gh;
    const int z = row / dc.G - dc.Gh, y = row - (z + dc.Gh) * dc.G - dc.Gh;
    const int m = total - 1 - c;  // the cell at -q (total / 2: the centre, its own mirror image)
    const float both = S[c] + S[m];
    S[c] = S[m] = both;
    if (x * x + y * y + z * z <= r2max) acc += c == m ? (double)both : 2.0 * both;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    acc = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (threadIdx.x == 0) atomicAdd(out, acc);
  }
}

}  // namespace

cudaError_t launch_density_setup(const DensityConst& dc, const DirParams* dirs, int n_dir, int P, float* S,
                                 double* band_sum, cudaStream_t stream) {
  const size_t cells = (size_t)dc.G * dc.G * dc.G;
  cudaError_t e = cudaMemsetAsync(S, 0, cells * sizeof(float), stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(band_sum, 0, sizeof(double), stream);
  if (e != cudaSuccess) return e;
  if (n_dir > 0) {
    const int n = dc.n_samples1 * dc.n_samples1;
    k_density_splat<<<dim3((n + 255) / 256, n_dir), 256, 0, stream>>>(dirs, dc, P, S);
  }
  k_density_mirror<<<device_sm_count() * 4, 256, 0, stream>>>(S, dc, band_sum);
  return cudaGetLastError();
}

}  // namespace recon
