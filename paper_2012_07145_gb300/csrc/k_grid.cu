// Bilateral grid (the bilateral grid app of Sec. 6, after Chen, Paris and
// Durand): the splat of a gray image into a grid of s x s pixel cells and
// range levels of size r, and the trilinear slice of the blurred grid back to
// the image.  The grid is a (ceil(W/s)+1) x (ceil(H/s)+1) image of 2 GZ
// channels: channel 2z holds the sum of the values of range level z, channel
// 2z+1 their count.  The blur between them (a point-wise op along the range
// levels and two 5-tap stencils) is one streaming kernel, k_grid_blur, below;
// any other grouping of those stages runs on the generic kernel.
//
// k_grid_splat: one thread per cell (any s) or four (s = 8, k_grid_splat8: two
//   pixel rows each, their copies added in a fixed order); each walks its
//   pixels in row order and adds them to its range level's pair of
//   accumulators, which sit in lane-private shared memory (every access of a
//   warp hits 32 banks), so the sums are formed in the same order every time.
// k_grid_slice: per pixel, trilinear interpolation (x, then y, then the range
//   level) of the value and the weight, then their ratio; four pixels of a row
//   per thread.
#include <cuda_runtime.h>

#include "hp_internal.h"
#include "stage_math.cuh"

namespace hp {

namespace {

constexpr int kSplatThreads = 128;
constexpr int kMaxGZ = 31;

__device__ __forceinline__ float gray_at(const ImgView& v, int x, int y) {
  return fminf(fmaxf(load_px(v, 0, x, y), 0.0f), 1.0f);
}

__device__ __forceinline__ int range_level(float v, float inv_r, int gz) {
  return iclamp((int)floorf(__fmaf_rn(v, inv_r, 0.5f)), 0, gz - 1);
}

// Any cell size s: one thread per cell walks its s x s pixels in row order.
__global__ void __launch_bounds__(kSplatThreads) k_grid_splat(const GridArgs a) {
  grid_dep_sync();
  __shared__ float acc[2 * kMaxGZ * kSplatThreads];
  const int t = threadIdx.x;
  const int gx = blockIdx.x * kSplatThreads + t, gy = blockIdx.y;
  if (gx >= a.grid.w) return;  // no barrier below: each thread owns its column of acc
  for (int j = 0; j < 2 * a.gz; ++j) acc[j * kSplatThreads + t] = 0.0f;
  const int W = a.in.w, H = a.in.h;
  const int s = a.s;
  for (int j = 0; j < s; ++j) {
    const int y = iclamp(gy * s + j - s / 2, 0, H - 1);
    for (int i = 0; i < s; ++i) {
      const float v = gray_at(a.in, iclamp(gx * s + i - s / 2, 0, W - 1), y);
      const int z = range_level(v, a.inv_r, a.gz);
      float* p = acc + 2 * z * kSplatThreads + t;
      p[0] = __fadd_rn(p[0], v);
      p[kSplatThreads] = __fadd_rn(p[kSplatThreads], 1.0f);
    }
  }
  for (int j = 0; j < 2 * a.gz; ++j)
    reinterpret_cast<float*>((char*)a.grid.data + (long long)j * a.grid.ps + (long long)gy * a.grid.rs)[gx] =
        acc[j * kSplatThreads + t];
}

// The splat of 8 x 8-pixel cells: a block of 4 warps takes 32 consecutive
// cells of a grid row, lane = cell, warp w = the cell's pixel rows 2w and 2w+1
// (two 128-bit loads per row for interior cells); each warp accumulates into
// its own lane-private copy, then the four copies are added in warp order.  The
// copies take the shared memory of the grid's own range levels (11 KB at 11, not
// the 32 KB of the most): every block of a 2560x1536 image is resident at once.
__global__ void __launch_bounds__(128) k_grid_splat8(const GridArgs a) {
  grid_dep_sync();
  extern __shared__ float accs[];   // [4][2 gz][32]
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float* const acc = accs + w * 2 * a.gz * 32 + lane;
  const int gx = blockIdx.x * 32 + lane, gy = blockIdx.y;
  const bool valid = gx < a.grid.w;
  for (int j = 0; j < 2 * a.gz; ++j) acc[j * 32] = 0.0f;
  if (valid) {
    const int W = a.in.w, H = a.in.h;
    const int x0 = gx * 8 - 4;
    const bool inner = x0 >= 0 && x0 + 7 <= W - 1 && a.in.dtype == HP_F32;
#pragma unroll
    for (int jj = 0; jj < 2; ++jj) {
      const int y = iclamp(gy * 8 + 2 * w + jj - 4, 0, H - 1);
      float v[8];
      if (inner) {
        const float4* row = reinterpret_cast<const float4*>((const char*)a.in.data + (long long)y * a.in.rs) + (x0 >> 2);
        const float4 f0 = __ldg(row), f1 = __ldg(row + 1);
        v[0] = f0.x; v[1] = f0.y; v[2] = f0.z; v[3] = f0.w; v[4] = f1.x; v[5] = f1.y; v[6] = f1.z; v[7] = f1.w;
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = fminf(fmaxf(v[i], 0.0f), 1.0f);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = gray_at(a.in, iclamp(x0 + i, 0, W - 1), y);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int z = range_level(v[i], a.inv_r, a.gz);
        acc[2 * z * 32] = __fadd_rn(acc[2 * z * 32], v[i]);
        acc[(2 * z + 1) * 32] = __fadd_rn(acc[(2 * z + 1) * 32], 1.0f);
      }
    }
  }
  __syncthreads();
  if (!valid) return;
  for (int j = w; j < 2 * a.gz; j += 4) {
    const float* p = accs + j * 32 + lane;
    const int copy = 2 * a.gz * 32;
    const float t = __fadd_rn(__fadd_rn(__fadd_rn(p[0], p[copy]), p[2 * copy]), p[3 * copy]);
    reinterpret_cast<float*>((char*)a.grid.data + (long long)j * a.grid.ps + (long long)gy * a.grid.rs)[gx] = t;
  }
}

__device__ __forceinline__ float lerp(float a, float b, float f) { return __fmaf_rn(f, __fsub_rn(b, a), a); }

// Four consecutive pixels of one row per thread (a warp: 128 pixels; a block:
// 8 rows): one 128-bit load of the image and one 128-bit store of the output
// where the row allows, and the grid-row addresses shared by the four pixels.
// Each pixel's arithmetic is the per-pixel expression above, unchanged.
__global__ void __launch_bounds__(256) k_grid_slice(const GridArgs a) {
  grid_dep_sync();
  const int xb = (blockIdx.x * 32 + (threadIdx.x & 31)) * 4;
  const int y = blockIdx.y * 8 + (threadIdx.x >> 5);
  if (xb >= a.in.w || y >= a.in.h) return;
  const ImgView& g = a.grid;
  const float gyf = __fmul_rn((float)y, a.inv_s);
  const float fly = floorf(gyf), fy = __fsub_rn(gyf, fly);
  const int y0 = iclamp((int)fly, 0, g.h - 1), y1 = iclamp((int)fly + 1, 0, g.h - 1);
  const char* g0 = (const char*)g.data + (long long)y0 * g.rs;
  const char* g1 = (const char*)g.data + (long long)y1 * g.rs;
  const int n = imin(4, a.in.w - xb);
  const bool vec = n == 4 && a.in.dtype == HP_F32 && (((size_t)a.in.data | (size_t)a.in.rs | (size_t)a.out.data | (size_t)a.out.rs) & 15) == 0;
  float v[4];
  if (vec) {
    const float4 q = __ldg(reinterpret_cast<const float4*>((const char*)a.in.data + (long long)y * a.in.rs) + (xb >> 2));
    v[0] = fminf(fmaxf(q.x, 0.0f), 1.0f); v[1] = fminf(fmaxf(q.y, 0.0f), 1.0f);
    v[2] = fminf(fmaxf(q.z, 0.0f), 1.0f); v[3] = fminf(fmaxf(q.w, 0.0f), 1.0f);
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = gray_at(a.in, imin(xb + k, a.in.w - 1), y);
  }
  float o[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float gxf = __fmul_rn((float)(xb + k), a.inv_s), gzf = __fmul_rn(v[k], a.inv_r);
    const float flx = floorf(gxf), flz = floorf(gzf);
    const float fx = __fsub_rn(gxf, flx), fz = __fsub_rn(gzf, flz);
    const int x0 = iclamp((int)flx, 0, g.w - 1), x1 = iclamp((int)flx + 1, 0, g.w - 1);
    const int z0 = iclamp((int)flz, 0, a.gz - 1), z1 = iclamp((int)flz + 1, 0, a.gz - 1);
    float r[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {  // value, weight
      float zs[2];
#pragma unroll
      for (int d = 0; d < 2; ++d) {
        const long long off = (long long)(2 * (d ? z1 : z0) + q) * g.ps;
        const float* p0 = reinterpret_cast<const float*>(g0 + off);
        const float* p1 = reinterpret_cast<const float*>(g1 + off);
        const float a0 = lerp(__ldg(p0 + x0), __ldg(p0 + x1), fx);
        const float a1 = lerp(__ldg(p1 + x0), __ldg(p1 + x1), fx);
        zs[d] = lerp(a0, a1, fy);
      }
      r[q] = lerp(zs[0], zs[1], fz);
    }
    o[k] = r[1] > 0.0f ? __fdiv_rn(r[0], r[1]) : v[k];
  }
  float* orow = reinterpret_cast<float*>((char*)a.out.data + (long long)y * a.out.rs);
  if (vec) {
    reinterpret_cast<float4*>(orow)[xb >> 2] = make_float4(o[0], o[1], o[2], o[3]);
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (k < n) orow[xb + k] = o[k];
  }
}

typedef unsigned long long u64;

__device__ __forceinline__ u64 pack2(float a, float b) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// lerp of (value, weight) at once: b - a and the fused step, each rounded once as in lerp().
__device__ __forceinline__ u64 lerp2(u64 a, u64 b, float f) {
  const u64 minus = pack2(-1.0f, -1.0f);
  return fma2(pack2(f, f), fma2(a, minus, b), a);
}

// The slice of a grid in pair layout (see grid_pair_levels): a cell's (value,
// weight) pairs lie together, level by level, the last level twice, so a corner of
// a pixel's two range levels is two adjacent 64-bit loads at one address instead
// of four 32-bit ones from four planes, and the pair is interpolated by the paired
// FP32 instructions.  Bound by issue: 2560x1536, s = 8, 11 levels: 28.2 us from
// planes, 18.8 as pairs with clamped levels and a type switch per pixel, about 14
// so.  SAME: the cell size is a power of two >= 4,
// so a thread's four pixels (rows 4 q .. 4 q + 3 of a column) lie in one cell, whose
// corner addresses they share.  F32: the image is f32.
// The next kernel is not let in early (grid_dep_wait, not grid_dep_sync): where
// realizes follow one another without a graph it is the next splat, whose
// shared memory asks for another split of the SM's memory than this kernel's
// cache, and its waiting blocks held this grid's up (640x480: 13.7 us a realize
// let in early, 10.0 so; 1000x700 16.5 and 12.4; replays 12.4 and 14.4 either way).
template <bool SAME, bool F32>
__global__ void __launch_bounds__(256) k_grid_slice_pairs(const GridArgs a) {
  grid_dep_wait();
  const int x = blockIdx.x * 32 + (threadIdx.x & 31);
  const int yb = blockIdx.y * 32 + (threadIdx.x >> 5) * 4;
  const int W = a.in.w, H = a.in.h;
  if (x >= W || yb >= H) return;
  const int gw = a.grid.w, gh = a.grid.h, gzp = grid_pair_levels(a.gz);
  const float gxf = __fmul_rn((float)x, a.inv_s);
  const float flx = floorf(gxf), fx = __fsub_rn(gxf, flx);
  const int x0 = iclamp((int)flx, 0, gw - 1) * gzp, x1 = iclamp((int)flx + 1, 0, gw - 1) * gzp;
  const u64* const g = (const u64*)a.grid.data;
  const long long pitch = (long long)gw * gzp;   // pairs per grid row
  const u64 *b00 = g, *b10 = g, *b01 = g, *b11 = g;   // the cell's corners at level 0
  float v[4];
  {
    const char* p = (const char*)a.in.data + (long long)yb * a.in.rs;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float t = F32 ? __ldg(reinterpret_cast<const float*>(p) + x) : load_px(a.in, 0, x, imin(yb + k, H - 1));
      v[k] = fminf(fmaxf(t, 0.0f), 1.0f);
      if (yb + k + 1 < H) p += a.in.rs;
    }
  }
  float fly = 0.0f;
  char* q = (char*)a.out.data + (long long)yb * a.out.rs + 4LL * x;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float gyf = __fmul_rn((float)(yb + k), a.inv_s), gzf = __fmul_rn(v[k], a.inv_r);
    if (!SAME || k == 0) {
      fly = floorf(gyf);
      const u64* r0 = g + iclamp((int)fly, 0, gh - 1) * pitch;
      const u64* r1 = g + iclamp((int)fly + 1, 0, gh - 1) * pitch;
      b00 = r0 + x0; b10 = r0 + x1; b01 = r1 + x0; b11 = r1 + x1;
    }
    // 0 <= v <= 1, so the level is in [0, gz - 1] without a clamp and the next
    // one is in the layout
    const int z = (int)gzf;
    const float fy = __fsub_rn(gyf, fly), fz = __fsub_rn(gzf, (float)z);
    const u64 lo = lerp2(lerp2(__ldg(b00 + z), __ldg(b10 + z), fx), lerp2(__ldg(b01 + z), __ldg(b11 + z), fx), fy);
    const u64 hi = lerp2(lerp2(__ldg(b00 + z + 1), __ldg(b10 + z + 1), fx),
                         lerp2(__ldg(b01 + z + 1), __ldg(b11 + z + 1), fx), fy);
    float val, wt;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(val), "=f"(wt) : "l"(lerp2(lo, hi, fz)));
    const float o = wt > 0.0f ? __fdiv_rn(val, wt) : v[k];
    if (yb + k < H) *reinterpret_cast<float*>(q) = o;
    q += a.out.rs;
  }
}

}  // namespace

int grid_max_levels() { return kMaxGZ; }

int launch_grid_splat(const GridArgs& a, void* stream) {
  if (a.gz < 1 || a.gz > kMaxGZ || a.s < 1 || a.grid.dtype != HP_F32 || a.grid.c < 2 * a.gz) return (int)cudaErrorInvalidValue;
  if (a.s == 8) {
    dim3 grid8((a.grid.w + 31) / 32, a.grid.h, 1);
    { const int le_ = launch_kernel(k_grid_splat8, grid8, dim3(128), 4 * 2 * a.gz * 32 * sizeof(float), stream, a); if (le_) return le_; }
  } else {
    dim3 grid((a.grid.w + kSplatThreads - 1) / kSplatThreads, a.grid.h, 1);
    { const int le_ = launch_kernel(k_grid_splat, grid, dim3(kSplatThreads), 0, stream, a); if (le_) return le_; }
  }
  __atomic_add_fetch(&g_launches, 1ULL, __ATOMIC_RELAXED);
  return (int)cudaGetLastError();
}

int launch_grid_slice(const GridArgs& a, void* stream) {
  if (a.gz < 1 || a.grid.dtype != HP_F32 || a.out.dtype != HP_F32 || a.grid.c < 2 * a.gz) return (int)cudaErrorInvalidValue;
  dim3 grid((a.in.w + 127) / 128, (a.in.h + 7) / 8, 1);
  if (a.pairs) grid = dim3((a.in.w + 31) / 32, (a.in.h + 31) / 32, 1);
  auto kern = !a.pairs ? k_grid_slice : a.in.dtype != HP_F32 ? k_grid_slice_pairs<false, false>
              : a.s >= 4 && (a.s & (a.s - 1)) == 0 ? k_grid_slice_pairs<true, true> : k_grid_slice_pairs<false, true>;
  { const int le_ = launch_kernel(kern, grid, dim3(256), 0, stream, a); if (le_) return le_; }
  __atomic_add_fetch(&g_launches, 1ULL, __ATOMIC_RELAXED);
  return (int)cudaGetLastError();
}


// ---- the blur of the grid (the group: range-level blur, x blur, y blur) ----
//
// k_grid_blur: one warp per strip of 28 grid columns (lanes 0, 1, 30, 31 only
// feed their neighbours) and a chunk of 4 range levels, values and weights,
// walking down a run of grid rows.  Per row it loads the chunk's levels and two
// more on each side (clamped), blurs along the levels, then along x (neighbours
// by warp shuffles); the y blur is five accumulators per level, each fed its taps
// in order as the rows arrive, so the float operations are those of the three
// stages one after the other (128 registers, 16 bytes spilled).  Read by slices alone, the result is stored in
// pair layout (one lane's 4 levels are two 128-bit stores), else in planes.
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kZC = 4;          // range levels per unit
constexpr int kBlurStrip = 28;  // grid columns per warp

struct GridBlurParams {
  GridBlurArgs a;
  int strips, zchunks, runs, units;
};

struct BlurRun {
  const GridBlurParams& P;
  int x, z0, y0, nout, T;
  bool prod;
  float acc[2][kZC][5];
  float ld[2][kZC + 4];  // the row's levels z0-2 .. z0+kZC+1 (clamped), in flight

  __device__ __forceinline__ explicit BlurRun(const GridBlurParams& p) : P(p) {}

  __device__ __forceinline__ void fetch(int t) {
    const ImgView& g = P.a.in;
    const int y = iclamp(y0 - 2 + t, 0, g.h - 1);
    const int xc = iclamp(x, 0, g.w - 1);
    const char* row = (const char*)g.data + (long long)y * g.rs;
#pragma unroll
    for (int i = 0; i < kZC + 4; ++i) {
      const float* p = reinterpret_cast<const float*>(row + 2 * iclamp(z0 - 2 + i, 0, P.a.gz - 1) * g.ps) + xc;
      ld[0][i] = __ldg(p);
      ld[1][i] = __ldg(reinterpret_cast<const float*>(reinterpret_cast<const char*>(p) + g.ps));
    }
  }

  // Input row t (grid row y0 - 2 + t) into the accumulators; PH = t mod 5.
  // Row t is tap j of output row t - j (run-relative, outputs 0 .. nout-1):
  // tap 0 starts output t, tap 4 completes output t - 4.
  template <int PH>
  __device__ __forceinline__ void row(int t) {
    float v[2][kZC + 4];
#pragma unroll
    for (int i = 0; i < kZC + 4; ++i) { v[0][i] = ld[0][i]; v[1][i] = ld[1][i]; }
    if (t + 1 < T) fetch(t + 1);
    const float w[5] = {0.0625f, 0.25f, 0.375f, 0.25f, 0.0625f};
    const int ofin = t - 4;
    const bool st = prod && ofin >= 0 && ofin < nout;
    float done[2][kZC];
#pragma unroll
    for (int q = 0; q < kZC; ++q)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float zb = tap5_binomial16(v[k][q], v[k][q + 1], v[k][q + 2], v[k][q + 3], v[k][q + 4]);
        const float l2 = __shfl_up_sync(kFull, zb, 2), l1 = __shfl_up_sync(kFull, zb, 1);
        const float r1 = __shfl_down_sync(kFull, zb, 1), r2 = __shfl_down_sync(kFull, zb, 2);
        const float h = tap5(w, l2, l1, zb, r1, r2);
        // slot of output t - j is (t - j) mod 5 = (PH - j) mod 5
        float (&s)[5] = acc[k][q];
        done[k][q] = __fmaf_rn(w[4], h, s[(PH + 1) % 5]);        // output t - 4: tap 4, complete
        s[(PH + 2) % 5] = __fmaf_rn(w[3], h, s[(PH + 2) % 5]);   // output t - 3
        s[(PH + 3) % 5] = __fmaf_rn(w[2], h, s[(PH + 3) % 5]);   // output t - 2
        s[(PH + 4) % 5] = __fmaf_rn(w[1], h, s[(PH + 4) % 5]);   // output t - 1
        s[PH] = __fmul_rn(w[0], h);                              // output t: tap 0
      }
    if (!st) return;
    const ImgView& o = P.a.out;
    if (P.a.pairs) {
      const int gzp = grid_pair_levels(P.a.gz);
      float* p = (float*)o.data + (((long long)(y0 + ofin) * o.w + x) * gzp + z0) * 2;
      // level gz holds level gz - 1 again
#pragma unroll
      for (int q = kZC - 1; q > 0; --q)
        if (z0 + q == P.a.gz) { done[0][q] = done[0][q - 1]; done[1][q] = done[1][q - 1]; }
#pragma unroll
      for (int q = 0; q < kZC; q += 2)
        if (z0 + q < gzp)
          *reinterpret_cast<float4*>(p + 2 * q) = make_float4(done[0][q], done[1][q], done[0][q + 1], done[1][q + 1]);
      if (z0 + kZC == P.a.gz) *reinterpret_cast<float2*>(p + 2 * kZC) = make_float2(done[0][kZC - 1], done[1][kZC - 1]);
    } else {
#pragma unroll
      for (int q = 0; q < kZC; ++q)
        if (z0 + q < P.a.gz) {
          char* p = (char*)o.data + (long long)2 * (z0 + q) * o.ps + (long long)(y0 + ofin) * o.rs;
          reinterpret_cast<float*>(p)[x] = done[0][q];
          reinterpret_cast<float*>(p + o.ps)[x] = done[1][q];
        }
    }
  }

  __device__ __forceinline__ void run(int u) {
    const int lane = threadIdx.x & 31;
    const int strip = u % P.strips;
    int rest = u / P.strips;
    const int zc = rest % P.zchunks;
    const int run_idx = rest / P.zchunks;
    x = strip * kBlurStrip + lane - 2;
    prod = lane >= 2 && lane < 2 + kBlurStrip && x < P.a.in.w;
    z0 = zc * kZC;
    y0 = run_idx * P.a.rows;
    nout = imin(P.a.rows, P.a.in.h - y0);
    T = nout + 4;  // grid rows y0 - 2 .. y0 + nout + 1
#pragma unroll
    for (int q = 0; q < kZC; ++q)
#pragma unroll
      for (int s = 0; s < 5; ++s) acc[0][q][s] = acc[1][q][s] = 0.0f;
    fetch(0);
    for (int t = 0; t < T; t += 5) {
      row<0>(t);
      if (t + 1 >= T) break;
      row<1>(t + 1);
      if (t + 2 >= T) break;
      row<2>(t + 2);
      if (t + 3 >= T) break;
      row<3>(t + 3);
      if (t + 4 >= T) break;
      row<4>(t + 4);
    }
  }
};

__global__ void __launch_bounds__(256, 2) k_grid_blur(const GridBlurParams P) {
  grid_dep_wait();
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int u = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < P.units; u += nw) {
    BlurRun r(P);
    r.run(u);
  }
}

}  // namespace

int grid_blur_units(const GridBlurArgs& a) {
  const int strips = (a.in.w + kBlurStrip - 1) / kBlurStrip;
  const int zchunks = (a.gz + kZC - 1) / kZC;
  return strips * zchunks * ((a.in.h + a.rows - 1) / a.rows);
}

int launch_grid_blur(const GridBlurArgs& a, int grid, void* stream) {
  if (a.gz < 1 || a.rows < 1 || grid < 1 || a.in.dtype != HP_F32 || a.out.dtype != HP_F32 || a.in.c < 2 * a.gz ||
      a.out.c < 2 * a.gz)
    return (int)cudaErrorInvalidValue;
  GridBlurParams kp;
  kp.a = a;
  kp.strips = (a.in.w + kBlurStrip - 1) / kBlurStrip;
  kp.zchunks = (a.gz + kZC - 1) / kZC;
  kp.runs = (a.in.h + a.rows - 1) / a.rows;
  kp.units = kp.strips * kp.zchunks * kp.runs;
  { const int le_ = launch_kernel(k_grid_blur, dim3(grid), dim3(256), 0, stream, kp); if (le_) return le_; }
  __atomic_add_fetch(&g_launches, 1ULL, __ATOMIC_RELAXED);
  return (int)cudaGetLastError();
}

}  // namespace hp
