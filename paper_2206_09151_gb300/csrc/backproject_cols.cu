// The per-scan kernel of the column-stack backprojection (see backproject_cols.cuh) and its host side.
#include <cooperative_groups.h>

#include <algorithm>

#include "backproject_cols.cuh"

namespace recon {
namespace {

namespace cg = cooperative_groups;

// The CTAs of a cluster (cluster size = gridDim.x / tiles along i) share the tile's directions.
template <typename ST, int J, bool LAYERS>
__global__ void __launch_bounds__(cols::kThreads, 2) k_backproject_cols(const __grid_constant__ CUtensorMap map,
                                                                        const DirParams* __restrict__ dirs,
                                                                        BackprojConst c, int dir_begin, int dir_count,
                                                                        float* __restrict__ vol, int accumulate) {
  using T = cols::Tile<J>;
  extern __shared__ __align__(128) unsigned char smem_cols[];  // TMA destinations: 128-byte aligned
  __shared__ unsigned long long s_bars[2 * cols::kStages];
  const cols::Ring ring = cols::init_ring(s_bars, smem_cols, cols::fixed_bytes<J>(), c.cols_stage);
  cg::cluster_group cluster = cg::this_cluster();
  const int S = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int bx = blockIdx.x / S, by = blockIdx.y, bz = blockIdx.z;
  const int d0 = (int)((long long)dir_count * rank / S), d1 = (int)((long long)dir_count * (rank + 1) / S);
  cols::Pair acc[cols::kB * cols::kB][2];
  cols::tile_sums<ST, J, LAYERS>(bx, by, bz, dirs, &map, c, dir_begin, d0, d1, smem_cols, ring, 0, acc);
  if (S == 1) {
    cols::write_tile<J>(bx, by, bz, c, vol, accumulate != 0, acc);
    if (bz == 0 && c.nw < c.ny && !accumulate) cols::clear_beside<J>(bx, by, c, vol);
    return;
  }
  // each CTA leaves its sums in shared memory as [k][j][i], adds the cluster's of its share of the tile's rows
  // and writes them
  float* dump = reinterpret_cast<float*>(smem_cols);
  __syncthreads();  // the ring is done with
  const int g = threadIdx.x / T::LANES, jl = threadIdx.x % T::LANES;
  const int x0 = (g % (T::TI / cols::kB)) * cols::kB, z0 = (g / (T::TI / cols::kB)) * cols::kB;
#pragma unroll
  for (int v = 0; v < cols::kB * cols::kB; ++v)
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      float* p = dump + ((z0 + v % cols::kB) * J + jl * 4 + 2 * r) * T::DUMP_PITCH + x0 + v / cols::kB;
      const float2 x = cols::unpack(acc[v][r]);
      p[0] = x.x;
      p[T::DUMP_PITCH] = x.y;
    }
  cluster.sync();
  const int i0 = bx * T::TI, k0 = by * cols::kTK, jb = c.j_lo + bz * J;
  const int rows = cols::kTK * J, r0 = rows * rank / S, r1 = rows * (rank + 1) / S;
  for (int q = threadIdx.x; q < (r1 - r0) * T::TI; q += cols::kThreads) {
    const int i = i0 + q % T::TI, r = r0 + q / T::TI, k = k0 + r / J, w = r % J;
    if (i >= c.nx || k >= c.nz || bz * J + w >= c.nw) continue;
    const int at = r * T::DUMP_PITCH + q % T::TI;
    float v = 0.f;
    for (int p = 0; p < S; ++p) v += cluster.map_shared_rank(dump, p)[at];
    float* o = vol + ((size_t)k * c.ny + jb + w) * c.nx + i;
    *o = accumulate ? *o + v : v;
  }
  if (bz == 0 && rank == 0 && c.nw < c.ny && !accumulate) cols::clear_beside<J>(bx, by, c, vol);
  cluster.sync();  // no CTA leaves while another reads its sums
}

// Persistent form for a batch: CTA b takes the (tomogram, tile) items b, b + gridDim.x, ...; a warp goes on to
// the next item when it has written its part of one.
struct Item {
  const BatchBp* d;
  int bx, by, bz;
};
__device__ __forceinline__ Item batch_item(const BatchBp* __restrict__ desc, int n_desc, unsigned it) {
  int lo = 0, hi = n_desc - 1;
  while (lo < hi) {  // the last tomogram whose first item is at or before it
    const int mid = (lo + hi + 1) >> 1;
    if (desc[mid].first_item <= it) lo = mid;
    else hi = mid - 1;
  }
  const BatchBp* d = desc + lo;
  const unsigned t = it - (unsigned)d->first_item;
  return Item{d, (int)(t % d->gx), (int)((t / d->gx) % d->gy), (int)(t / (unsigned)(d->gx * d->gy))};
}
template <typename ST, int J>
__device__ __noinline__ uint32_t cols_item(const Item& it, unsigned char* smem, const cols::Ring& ring, uint32_t uses) {
  const BackprojConst& c = it.d->c;
  cols::Pair acc[cols::kB * cols::kB][2];
  if (uses != cols::kFailed)
    uses = cols::tile_sums<ST, J, true>(it.bx, it.by, it.bz, it.d->dirs, &it.d->map, c, it.d->dir_begin, 0,
                                        it.d->dir_count, smem, ring, uses, acc);
  else  // a wait of an earlier item ran out: the warp is out of step with the ring and leaves no voxel unwritten
    cols::nan_sums(acc);
  cols::write_tile<J>(it.bx, it.by, it.bz, c, it.d->vol, it.d->accumulate != 0, acc);
  if (it.bz == 0 && c.nw < c.ny && !it.d->accumulate) cols::clear_beside<J>(it.bx, it.by, c, it.d->vol);
  return uses;
}
// J: rows per tile of the launch's tomograms; stage_bytes: their largest stage (one ring serves them all, so that
// a box of the next item never overlaps one that another warp still reads)
template <int J>
__global__ void __launch_bounds__(cols::kThreads, 2) k_backproject_cols_persistent(const BatchBp* __restrict__ desc,
                                                                                 int n_desc, unsigned total,
                                                                                 int stage_bytes) {
  extern __shared__ __align__(128) unsigned char smem_cols[];
  __shared__ unsigned long long s_bars[2 * cols::kStages];
  const cols::Ring ring = cols::init_ring(s_bars, smem_cols, cols::fixed_bytes<J>(), stage_bytes);
  uint32_t uses = 0;
  const BatchBp* fenced = nullptr;
  for (unsigned n = blockIdx.x; n < total; n += gridDim.x) {
    const Item it = batch_item(desc, n_desc, n);
    if (it.d != fenced) acquire_map(&it.d->map);  // by every warp: each issues loads
    fenced = it.d;
    uses = it.d->c.stack_bf16 ? cols_item<__nv_bfloat16, J>(it, smem_cols, ring, uses)
                              : cols_item<float, J>(it, smem_cols, ring, uses);
  }
}

constexpr int kMaxSmem = 220 * 1024;  // what a plan's boxes may take

// CTAs that run at once in clusters of S, by CTAs per SM (1 or 2): clusters do not fill every SM of a GPC.  As
// cudaOccupancyMaxActiveClusters gives it on a GB300.
constexpr int kSlots[2][9] = {{0, 152, 152, 138, 144, 140, 138, 105, 120}, {0, 304, 304, 291, 296, 290, 276, 266, 288}};
constexpr int kMaxSplit = 8;

// Time of `ctas` CTAs, `slots` at once, in times of one that has its SM to itself: two on one SM take 1.43 of it.
double wave_units(long long ctas, long long slots, int per_sm) {
  const double full = per_sm == 2 ? 1.43 : 1.0;
  const long long rest = ctas % slots;
  return (double)(ctas / slots) * full + (rest == 0 ? 0.0 : (rest * per_sm > slots ? full : 1.0));
}
// A CTA's time in directions (0.63 us each, dir_cost times that): its share of them and what it spends around them,
// 2.8, or 11 where a cluster shares them (sums left in shared memory and added across it).
double split_units(long long tiles, int S, int per_sm, int dirs, double dir_cost) {
  return wave_units(tiles * S, kSlots[per_sm - 1][S], per_sm) * ((dirs + S - 1) / S * dir_cost + (S == 1 ? 2.8 : 11.0));
}
// CTAs that share a tile's directions.  A split pays where the tiles leave SMs idle: 45 tiles, 60 directions 45
// us whole, 27 in four; 128 tiles, 60 directions 45 whole, 51 in two.  Over 250 scans (32^3 to 288^3, flat and tall
// volumes, 12 to 120 directions, 1 to 32 layers), each run with every split, the choice loses 2 % of the time on
// average; counting 5 directions around either lost 14 % (208^3, 30 directions in two: 127 us instead of 101).
int pick_split(long long tiles, int per_sm, int dirs) {
  int best = 1;
  for (int S = 2; S <= kMaxSplit && dirs >= 2 * S; ++S)
    if (split_units(tiles, S, per_sm, dirs, 1.0) < split_units(tiles, best, per_sm, dirs, 1.0)) best = S;
  return best;
}

// The column stacks of `dirs` directions at `stack` as a 4D tensor (rows, columns, layers, directions) with
// the plan's box.
cudaError_t encode_cols(const BackprojConst& c, const void* stack, int dirs, CUtensorMap* map) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_tiled();
  if (!enc) return cudaErrorNotSupported;
  const size_t es = c.stack_bf16 ? 2 : 4;
  const cuuint64_t dims[4] = {(cuuint64_t)c.wp, (cuuint64_t)c.nu, (cuuint64_t)c.nz_layers, (cuuint64_t)dirs};
  const cuuint64_t strides[3] = {(cuuint64_t)c.wp * es, (cuuint64_t)c.nu * c.wp * es,
                                 (cuuint64_t)c.nz_layers * c.nu * c.wp * es};
  const cuuint32_t bdim[4] = {(cuuint32_t)c.cols_j, (cuuint32_t)c.cols_w, (cuuint32_t)c.cols_l, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUresult r = enc(map, es == 2 ? CU_TENSOR_MAP_DATA_TYPE_UINT16 : CU_TENSOR_MAP_DATA_TYPE_UINT32, 4,
                         const_cast<void*>(stack), dims, strides, bdim, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <typename ST, int J, bool LAYERS>
cudaError_t launch_cols_t(const BackprojConst& c, const DirParams* dirs, const void* stack, int dir_begin,
                          int dir_count, float* volume, int accumulate, cudaStream_t stream) {
  using T = cols::Tile<J>;
  auto* kernel = k_backproject_cols<ST, J, LAYERS>;
  const size_t smem = cols_smem_bytes(c);
  static std::atomic<unsigned long long> raised{0};
  cudaError_t e = raise_smem_limit(raised, (const void*)kernel, kMaxSmem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, cols::kThreads, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const unsigned gi = (c.nx + T::TI - 1) / T::TI, gk = (c.nz + cols::kTK - 1) / cols::kTK, gj = (c.nw + J - 1) / J;
  const int S = pick_split((long long)gi * gk * gj, per_sm > 1 ? 2 : 1, dir_count);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(gi * S, gk, gj);
  cfg.blockDim = dim3(cols::kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = S;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  CUtensorMap map;
  e = encode_cols(c, stack, dir_count, &map);
  if (e != cudaSuccess) return e;
  e = cudaLaunchKernelEx(&cfg, kernel, map, dirs, c, dir_begin, dir_count, volume, accumulate);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t take_wait_failures(unsigned int* n, cudaStream_t stream) {
  void* count = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&count, cols::wait_failures);
  if (e == cudaSuccess) e = cudaMemcpyAsync(n, count, sizeof *n, cudaMemcpyDeviceToHost, stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  if (e == cudaSuccess && *n) e = cudaMemsetAsync(count, 0, sizeof *n, stream);
  if (e == cudaSuccess && *n) e = cudaStreamSynchronize(stream);
  return e;
}

size_t cols_smem_bytes(const BackprojConst& c) {
  const size_t fixed = c.cols_j == 64 ? cols::fixed_bytes<64>() : cols::fixed_bytes<32>();
  const size_t dump = c.cols_j == 64 ? cols::Tile<64>::kDumpBytes : cols::Tile<32>::kDumpBytes;
  return std::max(fixed + cols::kStages * (size_t)c.cols_stage, dump);
}

void cols_setup(BackprojConst& c, const DirParams* dirs, int n_dirs) {
  c.cols_j = 0;
  // the volume rows that detector rows fall on: j + b_int (and the row after it) inside the detector
  c.j_lo = std::max(0, -c.b_int - (c.b_frac != 0.f ? 1 : 0));
  c.nw = std::min(c.ny, c.nv - c.b_int) - c.j_lo;
  if (!c.axis_y || c.staged || c.layer_linear || n_dirs <= 0 || c.nw < 1) return;
  // a bfloat16 stack keeps rounded detector rows: rows between two of them are blended after
  // the rounding, which the column stack cannot
  if (c.stack_bf16 && c.b_frac != 0.f) return;
  const int per16 = c.stack_bf16 ? 8 : 4;
  c.wp = (c.nw + per16 - 1) / per16 * per16;
  // rows per tile: the one that wastes less of its last tile; 64 rows share the per-voxel work of a
  // direction among twice as many voxels (about 8 % of the time)
  const int pad64 = (c.nw + 63) / 64 * 64, pad32 = (c.nw + 31) / 32 * 32;
  const int prefer = pad64 <= 1.08 * pad32 ? 64 : 32;
  for (const int J : {prefer, 96 - prefer}) {
    const int TI = J == 64 ? cols::Tile<64>::TI : cols::Tile<32>::TI;
    long long W = cols::kLineCols, L = 1;
    for (int n = 0; n < n_dirs; ++n) {
      const DirParams& p = dirs[n];
      const long long a0 = std::abs(p.a[0]), a2 = std::abs(p.a[2]);
      // u over the tile (a 2^-9 pixel margin for the FP32 coordinates).  Where u rises along the lines, their
      // first taps lie over the tile less 3 steps, and 4 more columns follow; where it falls, the tap
      // above the first u is the last column
      const long long ea = a0 * (TI - 1) + a2 * (cols::kTK - 1) + (1LL << (kPixFracBits - 9));
      const long long et =
          std::abs((long long)p.t[1]) * (TI - 1) + std::abs((long long)p.t[3]) * (cols::kTK - 1);
      W = std::max(W, ((ea - 3 * std::max(a0, a2)) >> kPixFracBits) + 1 + cols::kLineCols);
      W = std::max(W, (ea >> kPixFracBits) + 4);
      L = std::max(L, std::min<long long>((et >> 24) + 2, c.nz_layers));
    }
    if (W > 256 || L > 256) continue;  // TMA box sides
    c.cols_j = J;
    c.cols_w = (int)W;
    c.cols_l = (int)L;
    c.cols_stage = (int)((W * L * J * (c.stack_bf16 ? 2 : 4) + 127) / 128 * 128);
    if (cols_smem_bytes(c) <= (size_t)kMaxSmem) return;
    c.cols_j = 0;
  }
}

// Not for flat volumes whose rows fill half of a tile's 32 or less, where the single-axis kernel, 16 rows per CTA, finds
// them all on the detector and the tiles fill the SMs by themselves: 300 x 16 x 300 voxels, 60 directions 64 us,
// the pairs 42; 256 x 16 x 256 (128 tiles) 45, 38.  With fewer tiles the split makes up for it (100 x 20 x 100: 20, 55).
bool cols_pay(const BackprojConst& c) {
  const long long tiles = (long long)((c.nx + cols::Tile<32>::TI - 1) / cols::Tile<32>::TI) * ((c.nz + cols::kTK - 1) / cols::kTK);
  const bool flat = c.ny <= 16 && c.b_frac == 0.f && c.b_int >= -1 && c.b_int + 15 <= c.nv;
  return !flat || tiles < 120;
}

cudaError_t describe_backproject_cols(const BackprojConst& c, BatchBp* out) {
  const int TI = c.cols_j == 64 ? cols::Tile<64>::TI : cols::Tile<32>::TI;
  out->gx = (c.nx + TI - 1) / TI;
  out->gy = (c.nz + cols::kTK - 1) / cols::kTK;
  out->gz = (c.nw + c.cols_j - 1) / c.cols_j;
  return encode_cols(c, out->stack, out->dir_count, &out->map);
}

template <int J>
static cudaError_t launch_persistent_t(const BatchBp* desc, int n_desc, unsigned total, size_t smem, cudaStream_t stream) {
  auto* kernel = k_backproject_cols_persistent<J>;
  static std::atomic<unsigned long long> raised{0};
  cudaError_t e = raise_smem_limit(raised, (const void*)kernel, kMaxSmem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, cols::kThreads, smem);
  if (e != cudaSuccess) return e;
  const unsigned ctas = (unsigned)(device_sm_count() * (per_sm < 1 ? 1 : per_sm));
  const int stage_bytes = (int)((smem - cols::fixed_bytes<J>()) / cols::kStages / 128 * 128);
  kernel<<<ctas < total ? ctas : total, cols::kThreads, smem, stream>>>(desc, n_desc, total, stage_bytes);
  return cudaGetLastError();
}
cudaError_t launch_backproject_cols_persistent(const BatchBp* desc_dev, int n_desc, unsigned long long total, int rows,
                                               size_t smem, cudaStream_t stream) {
  if (total == 0) return cudaSuccess;
  if (total > 0x7FFFFFFFull) return cudaErrorInvalidValue;
  return rows == 64 ? launch_persistent_t<64>(desc_dev, n_desc, (unsigned)total, smem, stream)
                    : launch_persistent_t<32>(desc_dev, n_desc, (unsigned)total, smem, stream);
}

cudaError_t launch_backproject_cols(const BackprojConst& c, const DirParams* dirs, const void* stack, int dir_begin,
                                    int dir_count, float* volume, int accumulate, cudaStream_t stream) {
  if (dir_count <= 0 || c.nx <= 0 || c.ny <= 0 || c.nz <= 0) return cudaSuccess;
#define RECON_COLS(ST, J)                                                                                            \
  (c.nz_layers > 1 ? launch_cols_t<ST, J, true>(c, dirs, stack, dir_begin, dir_count, volume, accumulate, stream)    \
                   : launch_cols_t<ST, J, false>(c, dirs, stack, dir_begin, dir_count, volume, accumulate, stream))
  if (c.stack_bf16) return c.cols_j == 64 ? RECON_COLS(__nv_bfloat16, 64) : RECON_COLS(__nv_bfloat16, 32);
  return c.cols_j == 64 ? RECON_COLS(float, 64) : RECON_COLS(float, 32);
#undef RECON_COLS
}

}  // namespace recon
