// Max filter, streaming (the max filter app of Sec. 6): per channel, the
// maximum over the (2RX+1) x (2RY+1) window at clamped coordinates, for a
// group of one window-maximum stage (square, horizontal or vertical) or of a
// horizontal and a vertical one of the same radius (the same values as the
// square window: the clamp acts on each coordinate separately).
//
// f32 and bf16 inputs: one warp per strip of 120 columns of one plane walks down
// a run of rows, four rows at a time.  They arrive as TMA boxes of 4 rows x 128
// columns through a ring of 3 shared-memory slots private to the warp.  Pixels outside the image
// arrive as NaN, which a maximum ignores: a window clamped at an edge holds the
// same in-image pixels as one cut there, so edges need no code.  A lane owns 4
// columns (lanes 0 and 31 none).
//   - Horizontal: blocks of 4 columns; output k of a block is the maximum of a
//     suffix of the block on its left, of its own columns and of a prefix of the
//     block on its right, all three read from shared memory.
//   - Vertical: blocks of 4 rows, one box each; the output at row j of a block
//     is the maximum of the block's first j + 1 rows and of suffixes of the two
//     blocks before it, which are kept as running suffix maxima (8 registers per
//     column for any radius), not as 2r + 1 rows.
// A warp runs one unit and every lane tests the box's barrier itself, so the
// ring needs no bookkeeping across units.  Bound by the loads' latency, then by
// memory: 2560x1536 RGB f32 9x9 takes 17.5 us in a stream of realizes (94 MB: 0.80
// of the measured copy rate).  As graph replays it is 20.6, against 39.3 with
// 2r + 1 rows of maxima in registers, a row loop unrolled as often, and a ring
// across units that one lane waited on; with the blocks but that ring it was 31.8.
//
// Other input types: one warp per strip of 120 columns, rows loaded from global
// memory, the next row's loads in flight while a row is processed; the
// horizontal maxima from the neighbour lanes' values (shuffles), a ring of
// 2RY + 1 rows of them in registers.
//
// Maxima are exact, so the order of the comparisons does not matter; the
// group's storage roundings are applied to the final maximum (rounding is
// monotone, so rounding the maximum equals the maximum of rounded values).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstring>

#include "hp_internal.h"
#include "stage_math.cuh"
#include "tma.cuh"

namespace hp {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kStripW = 120;    // output columns per warp
constexpr int kBoxRows = 4;     // rows per TMA box, and of a block of the vertical maxima
constexpr int kRing = 3;        // boxes per warp ring
constexpr int kBarBytes = 512;  // mbarriers of up to 16 warps x kRing

struct MaxParams {
  CUtensorMap tmap;
  MaxArgs a;
  int strips, runs, units;
};

// TMA boxes start at the strip's first column less 4 (lane 0's), less `pad`
// columns where that start is not 16-byte aligned (2-byte inputs); a box row
// is a multiple of 16 bytes, and every slot starts on a 128-byte boundary (the
// shared-memory destination of a tensor copy).
struct BoxGeom {
  int pad, box_w, box_bytes, slot_bytes;
};

__host__ __device__ constexpr BoxGeom box_geom(int esize) {
  BoxGeom g{};
  g.pad = esize == 2 ? 4 : 0;
  g.box_w = esize == 2 ? 136 : 128;
  g.box_bytes = g.box_w * kBoxRows * esize;
  g.slot_bytes = (g.box_bytes + 127) / 128 * 128;
  return g;
}

// A run of rows of one strip of one plane: input rows y0 - RY .. y0 + nout + RY - 1.
struct Unit {
  int plane, xs, y0, nout, n_in, nbox;
};

__device__ __forceinline__ Unit unit_geom(const MaxParams& P, int u, int ry) {
  Unit U;
  const int per_plane = P.strips * P.runs;
  U.plane = u / per_plane;
  const int v = u - U.plane * per_plane;
  const int run = v / P.strips, strip = v - run * P.strips;
  U.xs = strip * kStripW;
  U.y0 = run * P.a.rows;
  U.nout = imin(P.a.rows, P.a.in.h - U.y0);
  U.n_in = U.nout + 2 * ry;
  U.nbox = (U.n_in + kBoxRows - 1) / kBoxRows;
  return U;
}

template <int IDT>
__device__ __forceinline__ void load4_smem(const unsigned char* p, float (&v)[4]) {
  if (IDT == HP_F32) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
    const uint2 q = *reinterpret_cast<const uint2*>(p);
    const unsigned u[2] = {q.x, q.y};
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const unsigned short lo = (unsigned short)(u[i] & 0xffffu), hi = (unsigned short)(u[i] >> 16);
      if (IDT == HP_BF16) {
        v[2 * i] = __bfloat162float(__ushort_as_bfloat16(lo));
        v[2 * i + 1] = __bfloat162float(__ushort_as_bfloat16(hi));
      } else {
        v[2 * i] = __half2float(__ushort_as_half(lo));
        v[2 * i + 1] = __half2float(__ushort_as_half(hi));
      }
    }
  }
}

template <int IDT>
__device__ __forceinline__ void load_row(const MaxArgs& a, int plane, int y, int x0, bool vec, float (&v)[4]) {
  const char* row = (const char*)a.in.data + (long long)plane * a.in.ps + (long long)y * a.in.rs;
  if (IDT == HP_F32 && vec) {
    const float4 q = __ldg(reinterpret_cast<const float4*>(row) + (x0 >> 2));
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else if (IDT == HP_BF16 && vec) {
    const uint2 q = __ldg(reinterpret_cast<const uint2*>(row) + (x0 >> 2));
    v[0] = __bfloat162float(__ushort_as_bfloat16((unsigned short)(q.x & 0xffffu)));
    v[1] = __bfloat162float(__ushort_as_bfloat16((unsigned short)(q.x >> 16)));
    v[2] = __bfloat162float(__ushort_as_bfloat16((unsigned short)(q.y & 0xffffu)));
    v[3] = __bfloat162float(__ushort_as_bfloat16((unsigned short)(q.y >> 16)));
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = load_px(a.in, plane, iclamp(x0 + k, 0, a.in.w - 1), y);
  }
}

template <int IDT, int RX, int RY, bool RND>
struct MaxRun {
  static constexpr int N = 2 * RY + 1;  // rows of the ring of horizontal maxima = rows per unrolled step
  const MaxParams& P;
  int plane, x0, y0, nout, lane, n_in;
  bool vec, prod;
  float ring[N][4];
  float nxt[4];    // the next input row, in flight

  __device__ __forceinline__ explicit MaxRun(const MaxParams& p) : P(p) {}

  __device__ __forceinline__ void fetch(int t, float (&dst)[4]) {
    load_row<IDT>(P.a, plane, iclamp(y0 - RY + t, 0, P.a.in.h - 1), x0, vec, dst);
  }

  // Input row t of the run into ring slot S (the load of row t + 1 is issued
  // first); from t = 2RY on, output row t - 2RY.
  template <int S>
  __device__ __forceinline__ void row(int t) {
    float v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = nxt[k];
    if (t + 1 < n_in) fetch(t + 1, nxt);
    // a[0..11]: the left lane's 4 columns, this lane's, the right lane's
    float a[12];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      a[k] = __shfl_up_sync(kFull, v[k], 1);
      a[4 + k] = v[k];
      a[8 + k] = __shfl_down_sync(kFull, v[k], 1);
    }
    // column k's window is a[4 + k - RX .. 4 + k + RX]
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float m = a[4 + k - RX];
#pragma unroll
      for (int i = 5 + k - RX; i <= 4 + k + RX; ++i) m = fmaxf(m, a[i]);
      ring[S][k] = m;
    }
    if (t >= 2 * RY) {
      float o[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float m = ring[0][k];
#pragma unroll
        for (int s = 1; s < N; ++s) m = fmaxf(m, ring[s][k]);
        o[k] = RND ? round_storage(P.a.st_out, round_storage(P.a.st_mid, m)) : m;
      }
      if (prod) {
        const int y = y0 + t - 2 * RY;
        const ImgView& ov = P.a.out;
        if (!RND && x0 + 3 < ov.w) {
          reinterpret_cast<float4*>((char*)ov.data + (long long)plane * ov.ps + (long long)y * ov.rs)[x0 >> 2] =
              make_float4(o[0], o[1], o[2], o[3]);
        } else {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (x0 + k < ov.w) store_px(ov, plane, x0 + k, y, o[k]);
        }
      }
    }
  }

  template <int SS>
  __device__ __forceinline__ bool step(int t) {
    if (t + SS >= n_in) return false;
    row<SS>(t + SS);
    return true;
  }

  __device__ __forceinline__ void run(int u) {
    lane = threadIdx.x & 31;
    const int per_plane = P.strips * P.runs;
    plane = u / per_plane;
    const int v = u - plane * per_plane;
    const int run_idx = v / P.strips, strip = v - run_idx * P.strips;
    x0 = strip * kStripW + 4 * (lane - 1);
    const int W = P.a.in.w;
    vec = x0 >= 0 && x0 + 3 <= W - 1;
    prod = lane >= 1 && lane <= 30 && x0 < W;
    y0 = run_idx * P.a.rows;
    nout = imin(P.a.rows, P.a.in.h - y0);
    n_in = nout + 2 * RY;
    fetch(0, nxt);
    for (int t = 0; t < n_in; t += N) {
      if (!step<0>(t)) return;
      if (N > 1 && !step<(N > 1 ? 1 : 0)>(t)) return;
      if (N > 2 && !step<(N > 2 ? 2 : 0)>(t)) return;
      if (N > 3 && !step<(N > 3 ? 3 : 0)>(t)) return;
      if (N > 4 && !step<(N > 4 ? 4 : 0)>(t)) return;
      if (N > 5 && !step<(N > 5 ? 5 : 0)>(t)) return;
      if (N > 6 && !step<(N > 6 ? 6 : 0)>(t)) return;
      if (N > 7 && !step<(N > 7 ? 7 : 0)>(t)) return;
      if (N > 8 && !step<(N > 8 ? 8 : 0)>(t)) return;
    }
  }
};

__device__ __forceinline__ float max3(float a, float b, float c) { return fmaxf(fmaxf(a, b), c); }

// Horizontal maxima of the lane's 4 columns of a box row at p (the columns on
// either side are the neighbour lanes'; lanes 0 and 31 read past the row and
// produce nothing).
template <int IDT, int RX>
__device__ __forceinline__ void hmax4(const unsigned char* p, float (&h)[4]) {
  constexpr int kStep = 4 * (IDT == HP_F32 ? 4 : 2);
  float m[4];
  load4_smem<IDT>(p, m);
  if (RX == 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) h[k] = m[k];
    return;
  }
  float l[4], r[4];
  load4_smem<IDT>(p - kStep, l);
  load4_smem<IDT>(p + kStep, r);
#pragma unroll
  for (int k = 2; k >= 4 - RX && k >= 0; --k) l[k] = fmaxf(l[k], l[k + 1]);  // suffixes
#pragma unroll
  for (int k = 1; k < RX && k < 4; ++k) r[k] = fmaxf(r[k], r[k - 1]);        // prefixes
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    constexpr int kNone = -1;
    const int first = k - RX > 0 ? k - RX : 0, last = k + RX < 3 ? k + RX : 3;
    float o = m[first];
#pragma unroll
    for (int i = first + 1; i <= last; ++i) o = fmaxf(o, m[i]);
    const int li = k - RX < 0 ? 4 + k - RX : kNone, ri = k + RX > 3 ? k + RX - 4 : kNone;
    if (li != kNone) o = fmaxf(o, l[li < 0 ? 0 : li]);
    if (ri != kNone) o = fmaxf(o, r[ri < 0 ? 0 : ri]);
    h[k] = o;
  }
}

// A run of rows of one strip of one plane, its input rows taken from the warp's
// TMA ring, one block (box) of four at a time: box i lives in slot i % kRing and
// completes phase (i / kRing) & 1 of that slot's mbarrier.
template <int IDT, int RX, int RY, bool RND>
struct MaxRunTma {
  static constexpr int kEsize = IDT == HP_F32 ? 4 : 2;
  const MaxParams& P;
  const Unit& U;
  unsigned char* const slots;
  uint64_t* const bars;
  const int lane;
  bool vec, part, cut;  // the lane stores its four columns at once / one by one, up to the image's edge; any lane does
  char* row;            // the output row of the next input row (before the run's first: not stored)
  int s, phase;         // slot and phase of the next box

  __device__ __forceinline__ MaxRunTma(const MaxParams& P_, const Unit& U_, unsigned char* slots_, uint64_t* bars_,
                                       int lane_)
      : P(P_), U(U_), slots(slots_), bars(bars_), lane(lane_), s(0), phase(0) {
    const ImgView& ov = P.a.out;
    const int c0 = U.xs - 4 + 4 * lane;
    const bool prod = lane >= 1 && lane <= 30 && c0 < ov.w;
    vec = prod && c0 + 3 < ov.w && (!RND || ov.dtype == HP_BF16);
    part = prod && !vec;
    cut = __any_sync(kFull, part);
    row = (char*)ov.data + (long long)U.plane * ov.ps + (long long)(U.y0 - 2 * RY) * ov.rs +
          (long long)c0 * (RND ? dtype_size(ov.dtype) : 4);
  }

  __device__ __forceinline__ void issue(int i, int slot) {
    constexpr BoxGeom g = box_geom(kEsize);
    // the warp's reads of this slot (its previous box) come before the copy
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_arrive_expect_tx(bars + slot, (unsigned)g.box_bytes);
    tma_load_3d(slots + slot * g.slot_bytes, &P.tmap, U.xs - 4 - g.pad, U.y0 - RY + i * kBoxRows, U.plane, bars + slot);
  }

  // Block i of the run: X holds the suffix maxima of block i - 2, Y those of
  // block i - 1; X becomes this block's.
  __device__ __forceinline__ bool block(int i, float (&X)[4][4], float (&Y)[4][4]) {
    constexpr BoxGeom g = box_geom(kEsize);
    // every lane waits for the box itself (usually there: one test)
    if (!__all_sync(kFull, mbar_try_wait(bars + s, phase) || mbar_wait_poll(bars + s, phase, 2000000000ull))) return false;
    const unsigned char* p = slots + s * g.slot_bytes + (4 * lane + g.pad) * kEsize;
    const int t = 4 * i - 2 * RY;  // output row (of the run) of the block's row 0
    float pre[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float h[4], o[4];
      hmax4<IDT, RX>(p + j * g.box_w * kEsize, h);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        pre[k] = j ? fmaxf(pre[k], h[k]) : h[k];
        // rows before the block that the window holds: the last n of block
        // i - 1, and beyond its four the last n - 4 of block i - 2; n < 0 (radius
        // 1 and 0): only the last 2 RY + 1 of the block's own rows
        constexpr int two = 2 * RY;
        const int n = two - j;
        float m = pre[k];
        if (n >= 4) m = fmaxf(m, Y[0][k]);
        if (n > 0 && n < 4) m = fmaxf(m, Y[(4 - n) & 3][k]);
        if (n > 4) m = fmaxf(m, X[(8 - n) & 3][k]);
        if (n < 0) {
          m = h[k];
#pragma unroll
          for (int d = 1; d <= two; ++d) m = fmaxf(m, X[(j - d) & 3][k]);
        }
        o[k] = RND ? round_storage(P.a.st_out, round_storage(P.a.st_mid, m)) : m;
        X[j][k] = h[k];
      }
      const bool in_run = (unsigned)(t + j) < (unsigned)U.nout;
      if (vec && in_run) {
        if (!RND) {
          *reinterpret_cast<float4*>(row) = make_float4(o[0], o[1], o[2], o[3]);
        } else {
          const __nv_bfloat162 a = __floats2bfloat162_rn(o[0], o[1]), c = __floats2bfloat162_rn(o[2], o[3]);
          *reinterpret_cast<uint2*>(row) =
              make_uint2(*reinterpret_cast<const unsigned*>(&a), *reinterpret_cast<const unsigned*>(&c));
        }
      }
      if (cut) {
        if (part && in_run) {
          const int c0 = U.xs - 4 + 4 * lane;
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (c0 + k < P.a.out.w) store_px(P.a.out, U.plane, c0 + k, U.y0 + t + j, o[k]);
        }
      }
      row += P.a.out.rs;
    }
    __syncwarp();   // every lane has read the box
    if (lane == 0 && i + kRing < U.nbox) issue(i + kRing, s);
    phase ^= s == kRing - 1;
    s = s == kRing - 1 ? 0 : s + 1;
#pragma unroll
    for (int j = 2; j >= 0; --j)
#pragma unroll
      for (int k = 0; k < 4; ++k) X[j][k] = fmaxf(X[j][k], X[j + 1][k]);
    return true;
  }

  // False: a box never arrived.
  __device__ __forceinline__ bool run() {
    if (lane == 0)
      for (int i = 0; i < kRing && i < U.nbox; ++i) issue(i, i);
    float A[4][4], B[4][4];
    const float none = __int_as_float(0x7fffffff);   // NaN: no rows yet
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int k = 0; k < 4; ++k) A[j][k] = B[j][k] = none;
#pragma unroll 1
    for (int i = 0; i < U.nbox; i += 2) {
      if (!block(i, A, B)) return false;
      if (i + 1 < U.nbox && !block(i + 1, B, A)) return false;
    }
    return true;
  }
};

// RND: a storage rounding or a non-f32 output (else plain maxima, float4 stores).
// Three CTAs per SM, except the vertical-only windows of radius 3 and 4, whose
// ring of 2r+1 row maxima needs more registers than that leaves (they run at
// two CTAs per SM rather than spill).
template <int RX, int RY>
constexpr int max_rows_min_blocks() { return RX == 0 && RY >= 3 ? 2 : 3; }

template <int IDT, int RX, int RY, bool RND>
__global__ void __launch_bounds__(256, max_rows_min_blocks<RX, RY>()) k_max_rows(const MaxParams P) {
  grid_dep_wait();
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int u = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < P.units; u += nw) {
    MaxRun<IDT, RX, RY, RND> r(P);
    r.run(u);
  }
}

// Two CTAs of 8 warps per SM: 96 KB of boxes in flight are enough, and more CTAs
// would spill (2560x1536 RGB f32 9x9, replayed: 20.6 us at two, 22.4 at three, 24.7 at four).
template <int IDT, int RX, int RY, bool RND>
__global__ void __launch_bounds__(256, 2) k_max_rows_tma(const __grid_constant__ MaxParams P) {
  grid_dep_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* base = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int u = blockIdx.x * nw + warp;
  if (u >= P.units) return;
  uint64_t* const bars = reinterpret_cast<uint64_t*>(base) + warp * kRing;
  unsigned char* const slots = base + kBarBytes + warp * kRing * box_geom(IDT == HP_F32 ? 4 : 2).slot_bytes;
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < kRing; ++i) mbar_init(bars + i, 1);
    fence_mbar_init();
  }
  __syncwarp();
  const Unit U = unit_geom(P, u, RY);
  MaxRunTma<IDT, RX, RY, RND> r(P, U, slots, bars, lane);
  if (!r.run()) {
    // a box never arrived: report, and wait (bounded) for copies still in
    // flight into this warp's slots (a slot's phase is at most one behind)
    if (lane == 0) {
      atomicExch(P.a.err, 1);
      for (int i = 0; i < kRing; ++i) mbar_wait_poll(bars + i, i < r.s ? r.phase ^ 1 : r.phase, 100000000ull);
    }
    __syncwarp();
  }
}

typedef void (*MaxKernel)(MaxParams);

// shape 0: square window, 1: horizontal only, 2: vertical only; f32 and bf16
// inputs take the TMA ring
template <int IDT, int R, bool RND>
MaxKernel by_shape(int shape) {
  if (IDT == HP_F32 || IDT == HP_BF16) {
    constexpr int T = IDT == HP_F32 || IDT == HP_BF16 ? IDT : HP_F32;
    return shape == 1 ? k_max_rows_tma<T, R, 0, RND> : shape == 2 ? k_max_rows_tma<T, 0, R, RND>
                                                                  : k_max_rows_tma<T, R, R, RND>;
  }
  return shape == 1 ? k_max_rows<IDT, R, 0, RND> : shape == 2 ? k_max_rows<IDT, 0, R, RND> : k_max_rows<IDT, R, R, RND>;
}

template <int IDT, bool RND>
MaxKernel by_radius(int r, int shape) {
  return r == 1 ? by_shape<IDT, 1, RND>(shape) : r == 2 ? by_shape<IDT, 2, RND>(shape)
                : r == 3 ? by_shape<IDT, 3, RND>(shape) : by_shape<IDT, 4, RND>(shape);
}

// The input type's index (0: f32 to f32, 1: f32 with a rounding, 2: bf16, 3: others).
int input_kind(const MaxArgs& a) {
  const bool plain = a.st_mid == HP_F32 && a.st_out == HP_F32 && a.out.dtype == HP_F32;
  return a.in.dtype == HP_F32 ? (plain ? 0 : 1) : a.in.dtype == HP_BF16 ? 2 : 3;
}

MaxKernel pick_kernel(const MaxArgs& a) {
  switch (input_kind(a)) {
    case 0: return by_radius<HP_F32, false>(a.radius, a.shape);
    case 1: return by_radius<HP_F32, true>(a.radius, a.shape);
    case 2: return by_radius<HP_BF16, true>(a.radius, a.shape);
    default: return by_radius<-1, true>(a.radius, a.shape);
  }
}

bool uses_tma(const MaxArgs& a) { return a.in.dtype == HP_F32 || a.in.dtype == HP_BF16; }

}  // namespace

int max_rows_strip_w() { return kStripW; }

// Whether the input arrives in boxes of rows, one run per warp.
bool max_rows_boxed(const MaxArgs& a) { return uses_tma(a); }

int max_rows_smem_bytes(const MaxArgs& a, int threads) {
  if (!uses_tma(a)) return 0;
  return 2 * 128 + kBarBytes + (threads / 32) * kRing * box_geom(a.in.dtype == HP_F32 ? 4 : 2).slot_bytes;
}

// CTAs for `units` runs: one run per warp (TMA), or at most the resident CTAs,
// whose warps stride over the runs.  For 1 << 30 units: the resident CTAs.
int max_rows_grid(const MaxArgs& a, int units, int threads) {
  const int nw = threads / 32;
  const int need = (units + nw - 1) / nw;
  if (uses_tma(a) && units < 1 << 30) return need;
  int dev = 0, sms = 0, per_sm = 0;
  const MaxKernel kern = pick_kernel(a);
  const int smem = max_rows_smem_bytes(a, threads);
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      (smem && allow_max_dynamic_smem((const void*)kern) != 0) ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    return need < 2 * 152 ? need : 2 * 152;  // no device to ask: two CTAs on each of 152 SMs
  }
  return need < sms * per_sm ? need : sms * per_sm;
}

int launch_max_rows(const MaxArgs& a, int grid, void* stream) {
  if (a.radius < 1 || a.radius > 4 || a.shape < 0 || a.shape > 2 || a.rows < 1 || a.threads < 32 || a.threads > 256 || a.threads % 32 || grid < 1)
    return (int)cudaErrorInvalidValue;
  MaxParams kp;
  memset(&kp, 0, sizeof kp);
  kp.a = a;
  kp.strips = (a.in.w + kStripW - 1) / kStripW;
  kp.runs = (a.in.h + a.rows - 1) / a.rows;
  kp.units = kp.strips * kp.runs * a.in.c;
  const MaxKernel kern = pick_kernel(a);
  const int smem = max_rows_smem_bytes(a, a.threads);
  if (smem) {
    // once per kernel: it is four runtime calls, and a direct launch pays them on every realize
    static bool configured[3][4][3] = {};
    bool& done = configured[input_kind(a)][a.radius - 1][a.shape];
    if (!done) {
      int e = allow_max_dynamic_smem((const void*)kern);
      if (e) return e;
      done = true;
    }
    const int esize = a.in.dtype == HP_F32 ? 4 : 2;
    const CUtensorMapDataType tdt = a.in.dtype == HP_F32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    if (encode_tmap_3d(&kp.tmap, tdt, esize, a.in.data, a.in.w, a.in.h, a.in.c, a.in.rs, a.in.ps,
                       box_geom(esize).box_w, kBoxRows, 1, true))
      return (int)cudaErrorInvalidValue;
  }
  { const int le_ = launch_kernel(kern, dim3(grid), dim3(a.threads), smem, stream, kp); if (le_) return le_; }
  __atomic_add_fetch(&g_launches, 1ULL, __ATOMIC_RELAXED);
  return (int)cudaGetLastError();
}

}  // namespace hp
