// Register-resident stencil chain: d consecutive 5x5 separable stencil stages
// with the tile's pixels held in registers from the first stage to the last.
//
// One CTA computes a tile 256 columns wide and R rows per warp tall.  A lane
// owns 8 columns x R rows of it, loads them once, applies every stage in place
// and stores the pixels that are still exact.  Per stage
//   - the x pass runs row by row in place; a lane's four neighbour columns come
//     from the adjacent lanes by shuffles (half a shuffle per pixel);
//   - each warp hands the x-pass results of its outer two rows on either side
//     to the warps above and below through shared memory (two alternating
//     buffers, one CTA barrier per stage);
//   - the y pass runs in place over column pairs with the paired FP32
//     instructions (adjacent columns sit in adjacent registers, so the pairs
//     need no moves).
// What is computed is 10 FP32 operations per pixel and stage, nothing twice
// inside a tile; a tile's outer 2d rows and columns are a halo whose values go
// wrong from the edge inwards by 2 per stage and are not stored (none at the
// image's edges, where the tile starts at the edge and clamps).  The tiled kernel
// (k_chain.cu) spends 15.5 FP32 operations per pixel-stage on halo and x passes
// recomputed per row segment, and as much again on shared-memory round trips,
// addresses and barriers.
// Measured, 32 stages: 2560x1536 f32 154.2 -> 109.2 us (8 stages a launch, 20
// rows a thread), 1919x1079 bf16 152.5 -> 91.3; 640x480 f32, 16 stages 59.5 ->
// 20.5.  Pixels computed per pixel stored (halo): 1.50 at 2560x1536 and 1.76 at
// 1919x1079, 8 stages a launch.  Bound by issue: a row of 256 columns takes a warp about 125 cycles a
// stage, 80 of them on the FP32 pipe, the rest exposed latency of the shuffles at
// 2 to 4 warps per partition; a launch adds about 7 us (loads, stores, the wait
// for the previous grid), which is why few deep launches win.  One cooperative
// launch with halos exchanged between tiles measured no better: an exchange
// (border stores, release, flags, loads) takes 5 us.
//
// Boundary condition (clamp to edge on each stage's own producer): the two rows
// and columns past the image's last are made copies of it before every stage,
// and those before the first are taken from the edge itself.
//
// Every value uses the separable x-then-y fma order of stage_math.cuh and is
// rounded to the chain's storage type after each stage, so the result is
// bit-identical to every other schedule.
#include <cuda_runtime.h>

#include "hp_internal.h"
#include "stage_math.cuh"

namespace hp {

namespace {

constexpr int kCols = 8;                 // columns per lane
constexpr int kTileW = 32 * kCols;       // columns per tile, halo included
constexpr unsigned kFull = 0xffffffffu;
constexpr int kExchFloats = 2 * 4 * kTileW;  // per warp: two buffers of two top and two bottom rows

struct ResParams {
  ImgView in, out;
  int depth;
  int hx;              // halo columns per side (2 depth, rounded up to whole lanes)
  int step_x, step_y;  // tile pitch: the columns and rows an inner tile stores
  float w[kResidentMaxDepth][10];
};

typedef unsigned long long u64;

__device__ __forceinline__ u64 pack2(float a, float b) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(u64 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
  u64 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Two values rounded to the storage type (0: f32, 1: f16, 2: bf16).
template <int RND>
__device__ __forceinline__ void round2(float& a, float& b) {
  if (RND == 1) {
    const float2 f = __half22float2(__floats2half2_rn(a, b));
    a = f.x; b = f.y;
  } else if (RND == 2) {
    const float2 f = __bfloat1622float2(__floats2bfloat162_rn(a, b));
    a = f.x; b = f.y;
  }
}

// Pixels between memory and registers.  The code of a row is kept to a few instructions: it is
// unrolled over the rows, and what a tile runs once is paid for in instruction
// fetches.
template <int RND>
__device__ __forceinline__ void load8(const char* p, float (&v)[kCols]) {
  if (RND == 0) {
    const float4* q = reinterpret_cast<const float4*>(p);
    const float4 a = *q;
    const float4 b = q[1];
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  } else {
    const uint4 t = *reinterpret_cast<const uint4*>(p);
    const unsigned u[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 f = RND == 1 ? __half22float2(*reinterpret_cast<const __half2*>(&u[i]))
                                : __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u[i]));
      v[2 * i] = f.x; v[2 * i + 1] = f.y;
    }
  }
}

template <int RND>
__device__ __forceinline__ void store8(char* p, const float (&v)[kCols]) {
  if (RND == 0) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4*>(p + 16) = make_float4(v[4], v[5], v[6], v[7]);
  } else {
    unsigned u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (RND == 1) {
        const __half2 h = __floats2half2_rn(v[2 * i], v[2 * i + 1]);
        u[i] = *reinterpret_cast<const unsigned*>(&h);
      } else {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        u[i] = *reinterpret_cast<const unsigned*>(&h);
      }
    }
    *reinterpret_cast<uint4*>(p) = make_uint4(u[0], u[1], u[2], u[3]);
  }
}

// The first n columns of a lane that the image's right edge cuts.
template <int RND>
__device__ __forceinline__ void load_cut(const char* p, int n, float (&v)[kCols]) {
#pragma unroll
  for (int k = 0; k < kCols - 1; ++k) {
    if (k >= n) break;
    if (RND == 0) v[k] = reinterpret_cast<const float*>(p)[k];
    if (RND == 1) v[k] = __half2float(reinterpret_cast<const __half*>(p)[k]);
    if (RND == 2) v[k] = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p)[k]);
  }
}

template <int RND>
__device__ __forceinline__ void store_cut(char* p, int n, const float (&v)[kCols]) {
#pragma unroll
  for (int k = 0; k < kCols - 1; ++k) {
    if (k >= n) break;
    if (RND == 0) reinterpret_cast<float*>(p)[k] = v[k];
    if (RND == 1) reinterpret_cast<__half*>(p)[k] = __float2half_rn(v[k]);
    if (RND == 2) reinterpret_cast<__nv_bfloat16*>(p)[k] = __float2bfloat16_rn(v[k]);
  }
}

// x pass of one row in place: columns x0 - 2 .. x0 + 9 of the row, the outer
// four from the adjacent lanes.  `first`: the lane holds the image's column 0;
// `last`: it holds the last column (or lies past it).  TAPS: a tap stays in the
// operand cache for eight instructions (78 -> 71 cycles a row at 20 rows per
// thread; the instances with fewer registers spill with it).
template <bool TAPS>
__device__ __forceinline__ void xpass(float (&v)[kCols], const float* w, bool first, bool last) {
  float l2 = __shfl_up_sync(kFull, v[6], 1), l1 = __shfl_up_sync(kFull, v[7], 1);
  float r1 = __shfl_down_sync(kFull, v[0], 1), r2 = __shfl_down_sync(kFull, v[1], 1);
  l2 = first ? v[0] : l2;
  l1 = first ? v[0] : l1;
  r1 = last ? v[7] : r1;
  r2 = last ? v[7] : r2;
  const float e[kCols + 4] = {l2, l1, v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], r1, r2};
  float h[kCols];
  if (TAPS) {  // tap by tap over the eight columns (tap5's order in each)
#pragma unroll
    for (int k = 0; k < kCols; ++k) h[k] = __fmul_rn(w[0], e[k]);
#pragma unroll
    for (int j = 1; j < 5; ++j)
#pragma unroll
      for (int k = 0; k < kCols; ++k) h[k] = __fmaf_rn(w[j], e[k + j], h[k]);
  } else {
#pragma unroll
    for (int k = 0; k < kCols; ++k) h[k] = tap5(w, e[k], e[k + 1], e[k + 2], e[k + 3], e[k + 4]);
  }
#pragma unroll
  for (int k = 0; k < kCols; ++k) v[k] = h[k];
}

// Columns C and C + 1 of the lane that holds the image's last column, C - 1.
template <int C, int R>
__device__ __forceinline__ void copy_edge_cols(float (&v)[R][kCols], bool here) {
#pragma unroll
  for (int r = 0; r < R; ++r) {
    v[r][C] = here ? v[r][C - 1] : v[r][C];
    if (C + 1 < kCols) v[r][C + 1 < kCols ? C + 1 : C] = here ? v[r][C - 1] : v[r][C + 1 < kCols ? C + 1 : C];
  }
}

// An exchanged row: the lanes' first four columns, then their last four, so
// that a quarter warp's 128-bit accesses are contiguous.
__device__ __forceinline__ void put_row(float* row, int lane, const float (&v)[kCols]) {
  *reinterpret_cast<float4*>(row + 4 * lane) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(row + 128 + 4 * lane) = make_float4(v[4], v[5], v[6], v[7]);
}

template <int R, int RND, int MAXW>
__global__ void __launch_bounds__(32 * MAXW, 1) k_chain_resident(const __grid_constant__ ResParams kp) {
  grid_dep_sync();
  extern __shared__ __align__(16) float exch[];
  constexpr int kBytes = RND == 0 ? 4 : 2;
  constexpr bool kTaps = MAXW == 8 && !(R == 20 && RND == 0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int W = kp.in.w, H = kp.in.h;
  const int sx = blockIdx.x * kp.step_x, sy = blockIdx.y * kp.step_y;
  const int x0 = sx + kCols * lane, y0 = sy + R * warp;
  const bool active = y0 < H;                       // warps past the last row only keep the barrier
  const bool first = x0 == 0, last = x0 + kCols >= W;
  const bool ragged_cols = (W % kCols) != 0 && sx + kTileW > W;   // a lane of the tile holds columns past the last
  const bool ragged_rows = y0 + R > H;
  const bool own_below = warp == nw - 1 || y0 + R >= H;  // no rows below, or copies of the last
  const int cut = x0 < W && last ? W - x0 : kCols;   // columns of the lane inside the image (lanes past it: unused)
  const bool whole = x0 + kCols <= W;
  float v[R][kCols];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int k = 0; k < kCols; ++k) v[r][k] = 0.0f;
  if (active) {
    const char* p = (const char*)kp.in.data + (long long)blockIdx.z * kp.in.ps + (long long)y0 * kp.in.rs + (long long)x0 * kBytes;
    if (whole) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        load8<RND>(p, v[r]);
        if (y0 + r + 1 < H) p += kp.in.rs;   // rows past the last: copies of it
      }
    } else if (cut < kCols) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        load_cut<RND>(p, cut, v[r]);
        if (y0 + r + 1 < H) p += kp.in.rs;
      }
    }
  }
#pragma unroll 1
  for (int s = 0; s < kp.depth; ++s) {
    const float* const w = kp.w[s];
    float* const mine = exch + (s & 1) * nw * 4 * kTileW + warp * 4 * kTileW;
    if (active) {
      // the two columns and rows past the image's last are copies of it (the
      // passes reach no further)
      if (ragged_cols) {
        switch (W % kCols) {
          case 1: copy_edge_cols<1>(v, cut < kCols); break;
          case 2: copy_edge_cols<2>(v, cut < kCols); break;
          case 3: copy_edge_cols<3>(v, cut < kCols); break;
          case 4: copy_edge_cols<4>(v, cut < kCols); break;
          case 5: copy_edge_cols<5>(v, cut < kCols); break;
          case 6: copy_edge_cols<6>(v, cut < kCols); break;
          default: copy_edge_cols<7>(v, cut < kCols);
        }
      }
      if (ragged_rows) {
#pragma unroll
        for (int r = 1; r < R; ++r)
          if (y0 + r == H) {
#pragma unroll
            for (int k = 0; k < kCols; ++k) {
              v[r][k] = v[r - 1][k];
              if (r + 1 < R) v[r + 1 < R ? r + 1 : r][k] = v[r - 1][k];
            }
          }
      }
      float wx[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) wx[k] = w[k];
      // the rows the neighbours wait for first
      xpass<kTaps>(v[0], wx, first, last);
      xpass<kTaps>(v[1], wx, first, last);
      put_row(mine, lane, v[0]);
      put_row(mine + kTileW, lane, v[1]);
      xpass<kTaps>(v[R - 2], wx, first, last);
      xpass<kTaps>(v[R - 1], wx, first, last);
      put_row(mine + 2 * kTileW, lane, v[R - 2]);
      put_row(mine + 3 * kTileW, lane, v[R - 1]);
#pragma unroll
      for (int r = 2; r < R - 2; ++r) xpass<kTaps>(v[r], wx, first, last);
    }
    __syncthreads();
    if (active) {
      u64 wy[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) wy[k] = pack2(w[5 + k], w[5 + k]);
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        float4 a0, a1, b0, b1;   // the rows -2, -1, R and R + 1 of this half
        const float* q = mine + 128 * half + 4 * lane;
        if (warp == 0) {
          a0 = a1 = make_float4(v[0][4 * half], v[0][4 * half + 1], v[0][4 * half + 2], v[0][4 * half + 3]);
        } else {
          a0 = *reinterpret_cast<const float4*>(q - 2 * kTileW);
          a1 = *reinterpret_cast<const float4*>(q - 1 * kTileW);
        }
        if (own_below) {
          b0 = b1 = make_float4(v[R - 1][4 * half], v[R - 1][4 * half + 1], v[R - 1][4 * half + 2], v[R - 1][4 * half + 3]);
        } else {
          b0 = *reinterpret_cast<const float4*>(q + 4 * kTileW);
          b1 = *reinterpret_cast<const float4*>(q + 5 * kTileW);
        }
#pragma unroll
        for (int pr = 0; pr < 2; ++pr) {
          const int c = 4 * half + 2 * pr;
          u64 m2 = pr ? pack2(a0.z, a0.w) : pack2(a0.x, a0.y);
          u64 m1 = pr ? pack2(a1.z, a1.w) : pack2(a1.x, a1.y);
          const u64 e0 = pr ? pack2(b0.z, b0.w) : pack2(b0.x, b0.y);
          const u64 e1 = pr ? pack2(b1.z, b1.w) : pack2(b1.x, b1.y);
          u64 cur = pack2(v[0][c], v[0][c + 1]), n1 = pack2(v[1][c], v[1][c + 1]);
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const u64 n2 = r + 2 < R ? pack2(v[r + 2 < R ? r + 2 : 0][c], v[r + 2 < R ? r + 2 : 0][c + 1]) : r + 2 == R ? e0 : e1;
            u64 o = mul2(wy[0], m2);
            o = fma2(wy[1], m1, o);
            o = fma2(wy[2], cur, o);
            o = fma2(wy[3], n1, o);
            o = fma2(wy[4], n2, o);
            m2 = m1; m1 = cur; cur = n1; n1 = n2;
            unpack2(o, v[r][c], v[r][c + 1]);
            round2<RND>(v[r][c], v[r][c + 1]);
          }
        }
      }
    }
  }
  // the columns and rows the tile stores: all but the halo, which only lies on
  // sides inside the image
  const int cx0 = blockIdx.x > 0 ? sx + kp.hx : 0, cx1 = blockIdx.x + 1 < gridDim.x ? sx + kp.hx + kp.step_x : W;
  const int ry0 = blockIdx.y > 0 ? sy + 2 * kp.depth : 0;
  const int ry1 = blockIdx.y + 1 < gridDim.y ? sy + 2 * kp.depth + kp.step_y : H;
  if (!active || x0 < cx0 || x0 >= cx1) return;
  char* q = (char*)kp.out.data + (long long)blockIdx.z * kp.out.ps + (long long)y0 * kp.out.rs + (long long)x0 * kBytes;
  const int lo = ry0 - y0, hi = ry1 - y0;
  if (whole) {
#pragma unroll
    for (int r = 0; r < R; ++r, q += kp.out.rs)
      if (r >= lo && r < hi) store8<RND>(q, v[r]);
  } else {
#pragma unroll
    for (int r = 0; r < R; ++r, q += kp.out.rs)
      if (r >= lo && r < hi) store_cut<RND>(q, cut, v[r]);
  }
}

typedef void (*ResKernel)(ResParams);

// Rows per thread and the warps an SM's registers hold at that many (128, 168
// or 255 registers a thread).
struct ResShape {
  int rows, max_warps;
};
constexpr ResShape kShapes[] = {{5, 16}, {6, 16}, {8, 16}, {9, 12}, {11, 12}, {14, 8}, {17, 8}, {20, 8}};
constexpr int kNumShapes = sizeof kShapes / sizeof kShapes[0];

template <int RND>
ResKernel by_rows(int i) {
  switch (i) {
    case 0: return k_chain_resident<5, RND, 16>;
    case 1: return k_chain_resident<6, RND, 16>;
    case 2: return k_chain_resident<8, RND, 16>;
    case 3: return k_chain_resident<9, RND, 12>;
    case 4: return k_chain_resident<11, RND, 12>;
    case 5: return k_chain_resident<14, RND, 8>;
    case 6: return k_chain_resident<17, RND, 8>;
    default: return k_chain_resident<20, RND, 8>;
  }
}

int halo_cols(int depth) { return (2 * depth + kCols - 1) / kCols * kCols; }

// Tiles along an axis of n pixels: the first reaches `full`, every later one adds `step`.
int tiles_along(int n, int full, int step) { return n <= full ? 1 : 1 + (n - full + step - 1) / step; }

}  // namespace

int resident_smem_bytes(int threads) { return threads / 32 * kExchFloats * 4; }

// The tile shape of a w x h image with `planes` planes: fills a.seg (rows per
// thread), a.threads, a.tile_w/h (the columns and rows an inner tile stores) and
// a.tiles_x/y by the least estimated time; a caller's nonzero a.seg or a.threads
// is kept.  The estimate's figures are measured (2560x1536 f32): a warp's stage
// takes 125 cycles per row of 256 columns on its partition of the SM (80 on the
// FP32 pipe), and a wave of tiles 6000 cycles besides its loads and stores.
// Returns 0, or 1 where no shape fits.
int resident_shape(ChainArgs& a, int w, int h, int planes) {
  const int hx = halo_cols(a.depth), step_x = kTileW - 2 * hx;
  if (a.depth < 1 || a.depth > kResidentMaxDepth || step_x < kCols) return 1;
  constexpr long long sms = 152;
  double best = 0;
  ChainArgs b = a;
  bool found = false;
  for (int i = 0; i < kNumShapes; ++i) {
    const int R = kShapes[i].rows;
    if (a.seg && a.seg != R) continue;
    for (int nw = 1; nw <= kShapes[i].max_warps; ++nw) {
      if (a.threads && a.threads != 32 * nw) continue;
      const int rows = R * nw, step_y = rows - 4 * a.depth;
      if (rows < h && step_y < 1) continue;
      const int nx = tiles_along(w, kTileW, step_x), ny = step_y < 1 ? 1 : tiles_along(h, rows, step_y);
      const long long tiles = (long long)nx * ny * planes;
      const long long slots = sms * (kShapes[i].max_warps / nw);   // CTAs resident at once
      const long long waves = (tiles + slots - 1) / slots;
      auto wave = [&](long long ctas) {
        const int k = (int)((ctas + sms - 1) / sms);               // CTAs on the fullest SM
        return a.depth * (((k * nw + 3) / 4) * R * 125.0 + 150.0) + 6000.0 + k * nw * R * kTileW * 8.0 / 50.0;
      };
      const double cost = (waves - 1) * wave(slots) + wave(tiles - (waves - 1) * slots);
      if (found && cost >= best) continue;
      found = true;
      best = cost;
      b.seg = R;
      b.threads = 32 * nw;
      b.tile_w = step_x;
      b.tile_h = step_y < 1 ? rows : step_y;
      b.tiles_x = nx;
      b.tiles_y = ny;
    }
  }
  if (!found) return 1;
  b.resident = 1;
  a = b;
  return 0;
}

int launch_chain_resident(const ChainArgs& a, void* stream) {
  const int rnd = a.in.dtype == HP_F32 ? 0 : a.in.dtype == HP_F16 ? 1 : 2;
  int i = 0;
  while (i < kNumShapes && kShapes[i].rows != a.seg) ++i;
  if (i == kNumShapes) return (int)cudaErrorInvalidValue;
  ResKernel kern = rnd == 0 ? by_rows<0>(i) : rnd == 1 ? by_rows<1>(i) : by_rows<2>(i);
  static bool configured[3 * kNumShapes] = {};
  if (!configured[rnd * kNumShapes + i]) {
    int e = allow_max_dynamic_smem((const void*)kern);
    if (e) return e;
    configured[rnd * kNumShapes + i] = true;
  }
  ResParams kp;
  memset(&kp, 0, sizeof kp);
  kp.in = a.in;
  kp.out = a.out;
  kp.depth = a.depth;
  kp.hx = halo_cols(a.depth);
  kp.step_x = a.tile_w;
  kp.step_y = a.tile_h;
  memcpy(kp.w, a.w, sizeof(float) * 10 * a.depth);
  const int le = launch_kernel(kern, dim3(a.tiles_x, a.tiles_y, a.in.c), dim3(a.threads), resident_smem_bytes(a.threads),
                               stream, kp);
  if (le) return le;
  __atomic_add_fetch(&g_launches, 1ULL, __ATOMIC_RELAXED);
  return (int)cudaGetLastError();
}

}  // namespace hp
