// Stage B of single-axis scans about the volume y axis from a column stack: a device body
// shared by the per-scan kernel and the persistent batch kernel (backproject_cols.cu).
//
// In such a scan a voxel column (i, k) takes, from each direction, one layer and one detector
// coordinate u for all its voxels along y.  The column stack [direction][layer][u][w] keeps the
// detector rows w that the volume's y rows fall on consecutive, one value each (not the tap
// pairs of the general kernels, half their bytes), so a 16-byte load takes 4 voxels' samples of one
// detector column and the coordinate work is shared by J = 32 or 64 rows.
//
// What bounds it is the return bandwidth of the loads (128 bytes per SM and clock): gathers of
// tap pairs bring 8 bytes per voxel and direction.  Here neighbouring voxel columns share detector
// columns through registers.  A thread owns a 4 x 4 block of voxel columns x 4 rows and takes it,
// per direction, as 4 lines of 4 along the axis on which u moves more, by |du| in [0.707, 1] per
// voxel: counted from the line's first left tap, the left taps are then 0, {0, 1}, {1, 2}, {2, 3},
// so 5 consecutive detector columns serve the line (5 bytes per voxel and direction) and voxel m
// takes columns m - 1 .. m + 1 with weights max(0, 1 - |u - column|), 3 FMAs instead of 2, with no
// branch and no index into registers.  (Reloading only the columns that change between
// neighbours needs 3 bytes, but loads under a predicate cost more in moves than they save: 5.7 ms
// against 4.3 ms for 512 x 256 x 512 voxels and 360 views.)  The depth moves least along the same axis:
// a line whose voxels fall in two layers runs once per layer with the other voxels' weights zero.
//
// A CTA owns TI x 16 voxel columns x J rows (TI = 16 for J = 64, 32 for J = 32), 64 sums per thread
// over all its directions.  Per direction one TMA load brings the box of layers x detector columns that
// the tile can touch (one box size for all directions; columns off the detector are
// zero-filled) into a ring of three shared-memory stages, and each line has a record (the
// fraction of the first u, and its row of the box).  The 8 warps take turns at preparing a
// direction two ahead and otherwise advance on their own (a barrier per direction for the whole
// CTA cost a seventh of the time, as warps differ in the lines that span layers; a ninth warp for
// the preparation costs the others 24 registers).  Every wait is bounded; one that runs out leaves NaN
// in the warp's voxels, in the batch's persistent form in those of its later items too, and is counted for recon_sync.  A cluster of CTAs may share a tile's directions; their sums are
// added in rank order through distributed shared memory, so the result does not depend on timing.
#pragma once

#include <cuda_bf16.h>

#include "recon.h"
#include "recon_internal.h"
#include "tma.cuh"

namespace recon {
namespace cols {

constexpr uint32_t kFailed = 0xFFFFFFFFu;
constexpr int kThreads = 256, kWarps = kThreads / 32, kB = 4, kTK = 16, kStages = 3;
constexpr int kLineCols = 5;  // detector columns of a line of 4 voxels

template <int J>
struct Tile {
  static constexpr int LANES = J / 4;              // lanes per block of voxel columns (4 rows each)
  static constexpr int GROUPS = kThreads / LANES;  // blocks of 4 x 4 voxel columns
  static constexpr int TI = GROUPS * kB * kB / kTK;  // 16 (J = 64) or 32 (J = 32)
  static constexpr int LINES = GROUPS * kB;
  static constexpr int DUMP_PITCH = TI + 1;
  static constexpr size_t kDumpBytes = sizeof(float) * kTK * J * DUMP_PITCH;
};

struct Info {  // per (tile, direction)
  float fa, af0, af2;  // tile-origin u (its fraction) and its steps
  int shift;           // integer origin minus the box's first column
  uint32_t t, ti, tk;  // tile-origin depth minus the box's first layer and its steps, 2^-24 layer units
  int top;             // last layer of the box
  int c0, L0;          // the staged box's first column and layer
  int along_k, down;   // the lines run along k (else i); u falls along them
  float du;            // |step of u| along the lines
  uint32_t dt;         // step of the depth along the lines
  int pad[2];
};
static_assert(sizeof(Info) == 64, "Info layout");

struct Record {    // per line
  float d;         // distance of the first voxel's u from its first tap, in the lines' direction of u
  uint32_t place;  // row of the box (layer x columns) of that tap; bit 31: more than one layer
};
template <int J>
struct Stage {  // beside the box, written by the warp that prepares the direction
  Record rec[Tile<J>::LINES];
  uint32_t depth[Tile<J>::LINES];  // the first voxel's depth
  Info info;
};

constexpr int kOwn = 16;  // of the directions that a warp prepares (every 8th), it forms the infos of 16 at a time

// Dynamic shared memory: the stages' records, the warps' infos, then the boxes (128-byte aligned).
template <int J>
__host__ __device__ constexpr size_t fixed_bytes() {
  return (kStages * sizeof(Stage<J>) + kWarps * kOwn * sizeof(Info) + 127) / 128 * 128;
}

__device__ unsigned int wait_failures;  // warps whose wait ran out, since recon_sync last took it

constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23: x + kMagic, rounded down, holds floor(x) in its low mantissa bits
constexpr int kMagicBits = 0x4B400000;

__device__ __forceinline__ Info make_info(const DirParams& p, const BackprojConst& c, int i0, int k0, int ti_n) {
  Info f;
  const long long a = p.a[3] + p.a[0] * i0 + p.a[2] * k0;  // p.a[1] = 0; 2^-40 pixel
  const int ia = (int)(a >> kPixFracBits);
  f.fa = (float)((a & ((1LL << kPixFracBits) - 1)) >> (kPixFracBits - 24)) * 0x1p-24f;
  f.af0 = p.af[0];
  f.af2 = p.af[2];
  f.t = (uint32_t)p.t[0] + (uint32_t)p.t[1] * (uint32_t)i0 + (uint32_t)p.t[3] * (uint32_t)k0;
  f.ti = (uint32_t)p.t[1];
  f.tk = (uint32_t)p.t[3];
  f.along_k = fabsf(f.af2) > fabsf(f.af0);
  const float du = f.along_k ? f.af2 : f.af0;
  const uint32_t dt = f.along_k ? f.tk : f.ti;
  f.down = du < 0.f;
  f.du = fabsf(du);
  f.dt = dt;
  // u is a chain of FMAs, monotone in the voxel indices, and the depth an exact integer sum: the
  // extremes are at the tile's corners.  Corners beyond the volume lie up to 58 layers (the deepest box) off the
  // stack's at most 96: counted from its middle, so that 32 bits hold the depth (clamping the corners to the
  // volume instead cost the kernel 8 %: 442 us against 410 for 320^3, 60 directions)
  constexpr int kMiddle = RECON_MAX_LAYERS / 2;
  const uint32_t tm = f.t - ((uint32_t)kMiddle << 24);
  float umin = 1e30f;
  int lmin = INT32_MAX;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int x = q & 1 ? ti_n - 1 : 0, z = q & 2 ? kTK - 1 : 0;
    umin = fminf(umin, fmaf(f.af0, (float)x, fmaf(f.af2, (float)z, f.fa)));
    lmin = min(lmin, (int32_t)(tm + f.ti * (uint32_t)x + f.tk * (uint32_t)z) >> 24);
  }
  // where u falls along the lines, their 5 columns end at the tap above the first u, up to one column
  // below the tile's least u
  const int cmin = (int)floorf(umin) - f.down;
  f.c0 = ia + cmin;
  f.shift = -cmin;
  // the box's layers: clamped to the stack's, as the voxels' are
  f.L0 = max(min(lmin + kMiddle, c.nz_layers - c.cols_l), 0);
  f.t -= (uint32_t)f.L0 << 24;
  f.top = c.cols_l - 1;
  return f;
}

// Packed pairs of float32 in 64-bit registers (FP32x2 arithmetic).
typedef unsigned long long Pair;
__device__ __forceinline__ Pair pack(float lo, float hi) {
  Pair p;
  asm("mov.b64 %0, {%1, %2};" : "=l"(p) : "f"(lo), "f"(hi));
  return p;
}
__device__ __forceinline__ float2 unpack(Pair p) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(p));
  return f;
}
__device__ __forceinline__ Pair fma2(Pair a, Pair b, Pair c) {
  Pair d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// 4 rows of one detector column as two pairs.
template <typename ST>
struct Col {
  Pair v[2];
};
template <typename ST>
__device__ __forceinline__ void load_col(Col<ST>& c, uint32_t a);
template <>
__device__ __forceinline__ void load_col<float>(Col<float>& c, uint32_t a) {
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(c.v[0]), "=l"(c.v[1]) : "r"(a));
}
template <>
__device__ __forceinline__ void load_col<__nv_bfloat16>(Col<__nv_bfloat16>& c, uint32_t a) {
  uint32_t x, y;
  asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(x), "=r"(y) : "r"(a));
  c.v[0] = pack(__uint_as_float(x << 16), __uint_as_float(x & 0xFFFF0000u));
  c.v[1] = pack(__uint_as_float(y << 16), __uint_as_float(y & 0xFFFF0000u));
}

// One line: the 5 columns at shared address `a`, `step` bytes apart (backwards where u falls along the
// line); the voxels' sums at acc[P0], acc[P0 + S], ...  d: distance of the first u from the first
// column; one[m]: 1, or 0 to leave voxel m out (MASK).
template <typename ST, bool MASK, int P0, int S>
__device__ __forceinline__ void line(uint32_t a, uint32_t step, float d, float du, const float (&one)[kB],
                                     Pair (&acc)[kB * kB][2]) {
  Col<ST> y[kLineCols];
#pragma unroll
  for (int q = 0; q < kLineCols; ++q) load_col<ST>(y[q], a + q * step);
  {
    const float w1 = MASK ? d * one[0] : d, w0 = MASK ? __saturatef(one[0] - d) : 1.f - d;
    const Pair w0p = pack(w0, w0), w1p = pack(w1, w1);
#pragma unroll
    for (int r = 0; r < 2; ++r) acc[P0][r] = fma2(w1p, y[1].v[r], fma2(w0p, y[0].v[r], acc[P0][r]));
  }
#pragma unroll
  for (int m = 1; m < kB; ++m) {
    // t = u - (first column + m) in [-1, 1]: weights of the columns m - 1, m, m + 1
    const float t = fmaf((float)m, du, d) - (float)m;
    const float w0 = MASK ? __saturatef(one[m] - 1.f - t) : __saturatef(-t);
    const float w1 = MASK ? __saturatef(one[m] - fabsf(t)) : 1.f - fabsf(t);
    const float w2 = MASK ? __saturatef(one[m] - 1.f + t) : __saturatef(t);
    const Pair w0p = pack(w0, w0), w1p = pack(w1, w1), w2p = pack(w2, w2);
#pragma unroll
    for (int r = 0; r < 2; ++r)
      acc[P0 + m * S][r] = fma2(w2p, y[m + 1].v[r],
                                fma2(w1p, y[m].v[r], fma2(w0p, y[m - 1].v[r], acc[P0 + m * S][r])));
  }
}

// A line whose voxels (or those of another block of the warp) fall in several layers: one pass per layer of
// the warp's line that spans most; a block without that layer reads its first one with zero weights.
template <typename ST, int ROWB, int P0, int S>
__device__ __forceinline__ void layered_line(const Record& r, uint32_t t0, const Info& f, float du, uint32_t step,
                                             int W, uint32_t box, Pair (&acc)[kB * kB][2]) {
  const uint32_t dt = f.dt;
  const int top = f.top;
  int layer[kB];
#pragma unroll
  for (int m = 0; m < kB; ++m) layer[m] = min(max((int32_t)(t0 + m * dt) >> 24, 0), top);
  const int dir = layer[3] < layer[0] ? -1 : 1, span = (layer[3] - layer[0]) * dir;
  const int passes = __reduce_max_sync(0xffffffffu, span);
  const uint32_t first = r.place & 0x7FFFFFFFu;
#pragma unroll 1
  for (int p = 0; p <= passes; ++p) {
    const int now = layer[0] + p * dir;
    const bool mine = p <= span;
    float one[kB];
#pragma unroll
    for (int m = 0; m < kB; ++m) one[m] = mine && layer[m] == now ? 1.f : 0.f;
    line<ST, true, P0, S>(box + (mine ? first + (uint32_t)(p * dir * W) : first) * ROWB, step, r.d, du, one, acc);
  }
}

// The four lines of a thread's block for one direction, along k (K) or i.  Sums are [i of the block x 4 + k].
// One layer in the stack: no line can span two, and the four run as one piece of code (their loads overlap:
// 4.34 ms instead of 4.70 for the 360-view, 512 x 256 x 512 scan).  With LAYERS each line asks for itself.
template <typename ST, int ROWB, bool LAYERS, bool K, int l = 0>
__device__ __forceinline__ void block(const Record* rec, const uint32_t* depth, const Info& f, float du, uint32_t step,
                                      int W, uint32_t box, Pair (&acc)[kB * kB][2]) {
  if constexpr (l < kB) {
    constexpr int P0 = K ? l * kB : l, S = K ? 1 : kB;
    const Record r = rec[l];
    if (LAYERS && __any_sync(0xffffffffu, (int)r.place < 0)) {
      layered_line<ST, ROWB, P0, S>(r, depth[l], f, du, step, W, box, acc);
    } else {
      const float one[kB] = {1.f, 1.f, 1.f, 1.f};
      line<ST, false, P0, S>(box + r.place * ROWB, step, r.d, du, one, acc);
    }
    block<ST, ROWB, LAYERS, K, l + 1>(rec, depth, f, du, step, W, box, acc);
  }
}

// The ring: stage s's "full" mbarrier (the preparing warp's arrival and the box's bytes) and "empty" one (an
// arrival per warp).  `uses` counts the boxes that have passed; every warp steps it alike.
struct Ring {
  uint32_t full, empty;  // shared addresses of the first of each
  uint32_t boxes;        // shared address of the first box
  uint32_t stage_bytes;
};

__device__ __forceinline__ unsigned long long wait_limit(const BackprojConst& c) {
  return c.cols_probe_ns ? (unsigned long long)c.cols_probe_ns : kWaitNs;
}

// One warp: the records of a tile for one direction (d of the block that `map` describes) and the load of its
// box, into stage `use` mod kStages; false if the wait for the stage ran out.
template <typename ST, int J>
__device__ __forceinline__ bool prepare(int bz, const Info& f, const CUtensorMap* map, const BackprojConst& c, int d,
                                        unsigned char* smem, const Ring& ring, uint32_t use) {
  using T = Tile<J>;
  constexpr int ROWB = J * (int)sizeof(ST);
  const int lane = threadIdx.x & 31, W = c.cols_w;
  const uint32_t s = use % kStages;
  if (!__all_sync(0xffffffffu, mbar_wait(ring.empty + 8 * s, ((use / kStages) & 1u) ^ 1u, wait_limit(c)))) return false;
  Stage<J>& st = reinterpret_cast<Stage<J>*>(smem)[s];
#pragma unroll
  for (int q = 0; q < T::LINES / 32; ++q) {
    // line rl of block g
    const int n = lane + q * 32, rl = n % kB, g = n / kB;
    const int x = (g % (T::TI / kB)) * kB + (f.along_k ? rl : 0), z = (g / (T::TI / kB)) * kB + (f.along_k ? 0 : rl);
    const float u = fmaf(f.af0, (float)x, fmaf(f.af2, (float)z, f.fa));
    // the tap below u, or above it where u falls along the line (the magic-number add rounds down or up)
    const float tap = f.down ? __fadd_ru(u, kMagic) : __fadd_rd(u, kMagic);
    // inside the box by its construction; clamped all the same, so that no address leaves it
    const int lo = f.down ? kLineCols - 1 : 0;
    const int col = min(max(__float_as_int(tap) - kMagicBits + f.shift, lo), W - kLineCols + lo);
    const uint32_t t = f.t + f.ti * (uint32_t)x + f.tk * (uint32_t)z;
    const int la = min(max((int32_t)t >> 24, 0), f.top);
    const int lb = min(max((int32_t)(t + 3 * f.dt) >> 24, 0), f.top);
    st.rec[n] = Record{fabsf(u - (tap - kMagic)), (uint32_t)(la * W + col) | (la != lb ? 0x80000000u : 0u)};
    st.depth[n] = t;
  }
  if (lane == 0) st.info = f;
  __syncwarp();
  if (lane == 0) {
    mbar_expect_tx(ring.full + 8 * s, (uint32_t)(W * c.cols_l * ROWB));  // releases the records above
    if (!c.cols_probe_ns) tma_load_4d(ring.boxes + s * ring.stage_bytes, map, bz * J, f.c0, f.L0, d, ring.full + 8 * s);
  }
  return true;
}

__device__ __forceinline__ void nan_sums(Pair (&acc)[kB * kB][2]) {
  const float nan = __int_as_float(0x7FC00000);
#pragma unroll
  for (int v = 0; v < kB * kB; ++v) acc[v][0] = acc[v][1] = pack(nan, nan);
}

// The sums of tile (bx, by, bz) over the directions [d0, d1) of a block.  Returns the new count; a warp whose
// wait ran out has NaN sums and returns kFailed, after the loads still in flight.
template <typename ST, int J, bool LAYERS>
__device__ __forceinline__ uint32_t tile_sums(int bx, int by, int bz, const DirParams* __restrict__ dirs,
                                              const CUtensorMap* map, const BackprojConst& c, int dir_begin, int d0,
                                              int d1, unsigned char* smem, const Ring& ring, uint32_t uses,
                                              Pair (&acc)[kB * kB][2]) {
  using T = Tile<J>;
  constexpr int ROWB = J * (int)sizeof(ST);
  const Stage<J>* stages = reinterpret_cast<const Stage<J>*>(smem);
  const int tid = threadIdx.x, g = tid / T::LANES, jl = tid % T::LANES, warp = tid >> 5;
  const int count = d1 - d0;
#pragma unroll
  for (int v = 0; v < kB * kB; ++v) acc[v][0] = acc[v][1] = 0;
  bool ok = true;
  Info* own = reinterpret_cast<Info*>(smem + kStages * sizeof(Stage<J>)) + warp * kOwn;
  auto ready = [&](int n) {  // direction d0 + n, one of this warp's
    const int q = n / kWarps, lane = tid & 31;
    if (q % kOwn == 0) {
      const int m = n + lane * kWarps;
      __syncwarp();
      if (lane < kOwn && m < count) own[lane] = make_info(dirs[dir_begin + d0 + m], c, bx * T::TI, by * kTK, T::TI);
      __syncwarp();
    }
    return prepare<ST, J>(bz, own[q % kOwn], map, c, d0 + n, smem, ring, uses + n);
  };
  if (warp < kStages - 1 && warp < count) ok = ready(warp);
  uint32_t s = uses % kStages, parity = (uses / kStages) & 1u;
  for (int n = 0; ok && n < count; ++n) {
    ok = __all_sync(0xffffffffu, mbar_wait(ring.full + 8 * s, parity, wait_limit(c)));
    if (!ok) break;
    const Stage<J>& st = stages[s];
    const uint32_t box = ring.boxes + s * ring.stage_bytes + (uint32_t)(jl * 4 * (int)sizeof(ST));
    const Record* rec = st.rec + g * kB;
    const uint32_t* depth = st.depth + g * kB;
    const float du = st.info.du;
    const uint32_t step = st.info.down ? 0u - (uint32_t)ROWB : (uint32_t)ROWB;
    if (st.info.along_k) block<ST, ROWB, LAYERS, true>(rec, depth, st.info, du, step, c.cols_w, box, acc);
    else block<ST, ROWB, LAYERS, false>(rec, depth, st.info, du, step, c.cols_w, box, acc);
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(ring.empty + 8 * s);
    if (++s == kStages) {
      s = 0;
      parity ^= 1u;
    }
    const int ahead = n + kStages - 1;  // into the stage of direction n - 1
    if (ahead < count && ahead % kWarps == warp) ok = ready(ahead);
  }
  if (ok) return uses + (uint32_t)count;
  // every load of this tile lands (or runs out as well) before the warp gives up the shared memory
  if ((tid & 31) == 0) {
    const uint32_t end = uses + (uint32_t)count;
    for (uint32_t m = end - uses > kStages ? end - kStages : uses; m < end; ++m)
      mbar_wait(ring.full + 8 * (m % kStages), (m / kStages) & 1u, wait_limit(c));
  }
  __syncwarp();
  if ((tid & 31) == 0) atomicAdd(&wait_failures, 1u);
  nan_sums(acc);
  return kFailed;
}

// A thread's sums straight into the volume: 4 consecutive i per load and store, the two blocks of a
// half-warp pair side by side along i.
template <int J>
__device__ __forceinline__ void write_tile(int bx, int by, int bz, const BackprojConst& c, float* __restrict__ vol,
                                           bool accumulate, const Pair (&acc)[kB * kB][2]) {
  using T = Tile<J>;
  const int g = threadIdx.x / T::LANES, jl = threadIdx.x % T::LANES;
  const int i = bx * T::TI + (g % (T::TI / kB)) * kB, kb = by * kTK + (g / (T::TI / kB)) * kB, w = bz * J + jl * 4;
  const bool whole = i + kB <= c.nx && (c.nx & 3) == 0 && ((uintptr_t)vol & 15) == 0;
#pragma unroll
  for (int k = 0; k < kB; ++k) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (kb + k >= c.nz || w + j >= c.nw) continue;
      float v[kB];
#pragma unroll
      for (int x = 0; x < kB; ++x) {
        const float2 p = unpack(acc[x * kB + k][j >> 1]);
        v[x] = j & 1 ? p.y : p.x;
      }
      float* o = vol + ((size_t)(kb + k) * c.ny + c.j_lo + w + j) * c.nx + i;
      if (whole) {
        float4* o4 = reinterpret_cast<float4*>(o);
        float4 r = make_float4(v[0], v[1], v[2], v[3]);
        if (accumulate) {
          const float4 was = *o4;
          r = make_float4(was.x + r.x, was.y + r.y, was.z + r.z, was.w + r.w);
        }
        *o4 = r;
      } else {
#pragma unroll
        for (int x = 0; x < kB; ++x)
          if (i + x < c.nx) o[x] = accumulate ? o[x] + v[x] : v[x];
      }
    }
  }
}

// Sets up the ring in a kernel's shared memory (every thread calls it).
__device__ __forceinline__ Ring init_ring(unsigned long long* bars, unsigned char* smem, size_t fixed, int stage_bytes) {
  Ring r;
  r.full = (uint32_t)__cvta_generic_to_shared(bars);
  r.empty = r.full + 8 * kStages;
  r.boxes = (uint32_t)__cvta_generic_to_shared(smem + fixed);
  r.stage_bytes = (uint32_t)stage_bytes;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(r.full + 8 * s, 1);
      mbar_init(r.empty + 8 * s, kWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  return r;
}

// Volume rows beside the detector take nothing: cleared by the tiles of the first row block.
template <int J>
__device__ __forceinline__ void clear_beside(int bx, int by, const BackprojConst& c, float* __restrict__ vol) {
  using T = Tile<J>;
  const int beside = c.ny - c.nw;
  for (int q = threadIdx.x; q < T::TI * kTK * beside; q += kThreads) {
    const int i = bx * T::TI + q % T::TI, r = q / T::TI, k = by * kTK + r / beside;
    int j = r % beside;
    if (j >= c.j_lo) j += c.nw;
    if (i < c.nx && k < c.nz) vol[((size_t)k * c.ny + j) * c.nx + i] = 0.f;
  }
}

}  // namespace cols
}  // namespace recon
