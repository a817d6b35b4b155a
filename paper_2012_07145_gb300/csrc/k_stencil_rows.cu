// Streaming single 5x5 stencil, optionally followed by the unsharp-mask
// combine (out = in + amount (in - blur)), per channel plane.
//
// Each warp owns a strip of output columns, four per lane, of one plane and
// walks down a run of rows, four at a time.  Input rows arrive as TMA boxes
// (kBoxRows rows, 128 columns) through a ring of shared-memory slots private to
// the warp, so the loads of later rows overlap the arithmetic on the current
// ones and no barrier wider than the warp is taken.  A warp runs one unit (run of
// rows) and every lane tests a box's barrier itself: a ring that ran on into the
// warp's next unit, waited on by one lane, cost more in bookkeeping than the
// arithmetic.  The x pass reads the two columns on either side from shared
// memory, the y pass runs over the x-pass results of the last eight rows (two
// blocks, alternating, so nothing is moved), and the unsharp combine keeps the
// two input rows it is behind.  The stencil and combine expressions are those of
// stage_math.cuh, so the result is bit-identical to every other schedule.
// Bound by memory: unsharp 4096x3072 RGB f32 takes 47.2 us in a stream of realizes
// (302 MB: 0.94 of the measured copy rate), 50.4 replayed; with the ring across
// units, one row at a time and a queue of row registers, 68.7 replayed.
//
// Boundary condition (clamp to edge on the stencil's input): in strips that
// touch the left or right image edge the two columns outside it are written into
// the arrived box; rows outside take the nearest edge row's x-pass result.
#include <cuda.h>
#include <cuda_runtime.h>

#include "hp_internal.h"
#include "stage_math.cuh"
#include "tma.cuh"

namespace hp {

namespace {

// Box heights stay a power of two: boxes of 3 or 5 rows measured several
// times slower to arrive than boxes of 2 or 4.
constexpr int kBoxRows = 4;      // rows per TMA box
constexpr int kRing = 3;         // boxes per warp ring
constexpr int kBarBytes = 512;   // mbarriers of up to 16 warps x kRing
constexpr unsigned kFull = 0xffffffffu;

struct StripGeom {
  int halo_lanes;  // lanes on each side that only feed neighbours
  int strip_w;     // output columns per strip: 4 (32 - 2 halo_lanes)
  int slot_bytes;  // one ring slot: 128 columns x kBoxRows rows
};

// A TMA box must start on a 16-byte boundary: 4 columns of a 4-byte input, 8
// of a 2-byte one; that sets the halo lanes (two columns of halo are needed).
__host__ __device__ inline StripGeom strip_geom(int esize) {
  StripGeom g;
  g.halo_lanes = esize == 4 ? 1 : 2;
  g.strip_w = 4 * (32 - 2 * g.halo_lanes);
  g.slot_bytes = 128 * kBoxRows * esize;
  return g;
}

struct SRowsParams {
  CUtensorMap tmap;
  ChainArgs a;  // depth 1: storage[0], w[0] (wx then wy), epilogue, amount
  int strips, runs, units, rows;  // per plane: strips x runs units of `rows` output rows
};

struct Unit {
  int x0, oy, plane, nout, nbox;  // x0: image column of lane 0's first column
};

__device__ __forceinline__ Unit unit_geom(const SRowsParams& kp, const StripGeom& g, int u) {
  Unit U;
  const int per_plane = kp.strips * kp.runs;
  U.plane = u / per_plane;
  const int v = u - U.plane * per_plane;
  const int run = v / kp.strips, s = v - run * kp.strips;
  U.x0 = s * g.strip_w - 4 * g.halo_lanes;
  U.oy = run * kp.rows;
  U.nout = min(kp.rows, kp.a.out.h - U.oy);
  U.nbox = (U.nout + 4 + kBoxRows - 1) / kBoxRows;
  return U;
}

// Four columns at p, and the two on either side.
template <bool F32>
__device__ __forceinline__ void load8(const unsigned char* p, int dtype, float (&v)[8]) {
  if (F32 || dtype == HP_F32) {
    const float2 l = *reinterpret_cast<const float2*>(p - 8);
    const float4 q = *reinterpret_cast<const float4*>(p);
    const float2 r = *reinterpret_cast<const float2*>(p + 16);
    v[0] = l.x; v[1] = l.y; v[2] = q.x; v[3] = q.y; v[4] = q.z; v[5] = q.w; v[6] = r.x; v[7] = r.y;
  } else {
    const uint2 q = *reinterpret_cast<const uint2*>(p);
    const unsigned u[4] = {*reinterpret_cast<const unsigned*>(p - 4), q.x, q.y, *reinterpret_cast<const unsigned*>(p + 8)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const unsigned short lo = (unsigned short)(u[i] & 0xffffu), hi = (unsigned short)(u[i] >> 16);
      if (dtype == HP_BF16) {
        v[2 * i] = __bfloat162float(__ushort_as_bfloat16(lo));
        v[2 * i + 1] = __bfloat162float(__ushort_as_bfloat16(hi));
      } else {
        v[2 * i] = __half2float(__ushort_as_half(lo));
        v[2 * i + 1] = __half2float(__ushort_as_half(hi));
      }
    }
  }
}

// The binomial [1,4,6,4,1]/16 taps (the unsharp blur, the same float values
// the pipeline stores) as compile-time constants.
__device__ __forceinline__ float tap5_binomial_const(float a, float b, float c, float d, float e) {
  float s = __fmul_rn(0.0625f, a);
  s = __fmaf_rn(0.25f, b, s);
  s = __fmaf_rn(0.375f, c, s);
  s = __fmaf_rn(0.25f, d, s);
  return __fmaf_rn(0.0625f, e, s);
}

// One run of rows of one strip of one plane.  Box i lives in slot i % kRing and
// completes phase (i / kRing) & 1 of that slot's mbarrier; its rows are input
// rows 4 i .. 4 i + 3 of the run (image rows oy - 2 + ...), and row t of the run
// emits output row t - 4.  F32 = every storage type is f32 (no rounding, one
// 128-bit store per lane and row).  BIN: both passes take the binomial taps
// (checked bit for bit on the host), compiled as constants.
template <bool F32, bool EPI, bool BIN>
struct StripRun {
  const SRowsParams& kp;
  const StripGeom& g;
  const Unit& U;
  unsigned char* const slots;
  uint64_t* const bars;
  const int lane, c0, esize;
  const bool vedge;          // the run reads rows outside the image
  float wx[5], wy[5];
  bool vec, part, cut;       // the lane stores its four columns at once / one by one, up to the edge; any lane does
  char* out_row;             // output row of the next input row
  int s, phase;              // slot and phase of the next box
  float behind[2][4];        // the last two input rows (unsharp)

  __device__ __forceinline__ StripRun(const SRowsParams& kp_, const StripGeom& g_, const Unit& U_, unsigned char* slots_,
                                      uint64_t* bars_, int lane_)
      : kp(kp_), g(g_), U(U_), slots(slots_), bars(bars_), lane(lane_), c0(U_.x0 + 4 * lane_),
        esize(F32 || kp_.a.in.dtype == HP_F32 ? 4 : 2), vedge(U_.oy < 2 || U_.oy + U_.nout + 2 > kp_.a.in.h), s(0), phase(0) {
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      wx[k] = kp.a.w[0][k];
      wy[k] = kp.a.w[0][5 + k];
    }
    const ImgView& ov = kp.a.out;
    const bool mine = lane >= g.halo_lanes && lane < 32 - g.halo_lanes && c0 < ov.w;
    const int osize = F32 ? 4 : dtype_size(ov.dtype);
    vec = mine && c0 + 3 < ov.w && (osize == 4 ? ov.dtype == HP_F32 : osize == 2 && ov.dtype != HP_U16);
    part = mine && !vec;
    cut = __any_sync(kFull, part);
    out_row = (char*)ov.data + (long long)U.plane * ov.ps + (long long)(U.oy - 4) * ov.rs + (long long)c0 * osize;
#pragma unroll
    for (int k = 0; k < 4; ++k) behind[0][k] = behind[1][k] = 0.0f;
  }

  __device__ __forceinline__ void issue(int i, int slot) {
    // the warp's accesses to this slot (its previous box) come before the copy
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_arrive_expect_tx(bars + slot, (unsigned)g.slot_bytes);
    tma_load_3d(slots + slot * g.slot_bytes, &kp.tmap, U.x0, U.oy - 2 + i * kBoxRows, U.plane, bars + slot);
  }

  // In a strip at the left or right edge: the two columns outside the image,
  // where the box holds them, become the edge column (16 lanes, one value each).
  __device__ __forceinline__ void fill_edges(unsigned char* box) {
    const int W = kp.a.in.w;
    const int row = lane & 3, k = (lane >> 2) & 1;
    const int edge = (lane < 8 ? 0 : W - 1) - U.x0, to = lane < 8 ? edge - 1 - k : edge + 1 + k;
    if (lane < 16 && edge >= 0 && edge < 128 && to >= 0 && to < 128) {
      unsigned char* r = box + row * 128 * esize;
      if (esize == 4) {
        reinterpret_cast<float*>(r)[to] = reinterpret_cast<const float*>(r)[edge];
      } else {
        reinterpret_cast<unsigned short*>(r)[to] = reinterpret_cast<const unsigned short*>(r)[edge];
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // before the slot's next copy
    __syncwarp();
  }

  __device__ __forceinline__ float tap_x(float a, float b, float c, float d, float e) const {
    return BIN ? tap5_binomial_const(a, b, c, d, e) : tap5(wx, a, b, c, d, e);
  }
  __device__ __forceinline__ float tap_y(float a, float b, float c, float d, float e) const {
    return BIN ? tap5_binomial_const(a, b, c, d, e) : tap5(wy, a, b, c, d, e);
  }

  // Box i: A holds the x-pass results of the four rows before it, B receives its own.
  __device__ __forceinline__ bool block(int i, float (&A)[4][4], float (&B)[4][4]) {
    const ChainArgs& a = kp.a;
    // every lane waits for the box itself (usually there: one test)
    if (!__all_sync(kFull, mbar_try_wait(bars + s, phase) || mbar_wait_poll(bars + s, phase, 2000000000ull))) return false;
    unsigned char* const box = slots + s * g.slot_bytes;
    if (U.x0 < 0 || U.x0 + 128 > a.in.w) fill_edges(box);
    const unsigned char* p = box + lane * 4 * esize;
    float raw[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float v[8];
      load8<F32>(p + j * 128 * esize, a.in.dtype, v);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        raw[j][k] = v[k + 2];
        B[j][k] = tap_x(v[k], v[k + 1], v[k + 2], v[k + 3], v[k + 4]);
      }
      if (vedge) {
        const int r = U.oy - 2 + 4 * i + j;
        if (r == 0) {  // rows -2 and -1 are row 0 (rows 2 and up of the run: j >= 2)
#pragma unroll
          for (int k = 0; k < 4; ++k) { B[(j + 3) & 3][k] = B[j][k]; B[(j + 2) & 3][k] = B[j][k]; }
        }
        if (r >= a.in.h) {  // rows H and H + 1 are row H - 1
#pragma unroll
          for (int k = 0; k < 4; ++k) B[j][k] = j ? B[(j + 3) & 3][k] : A[3][k];
        }
      }
      const int t = 4 * i + j - 4;   // output row of the run
      const bool in_run = (unsigned)t < (unsigned)U.nout;
      float o[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float r0 = j < 1 ? A[0][k] : j < 2 ? A[1][k] : j < 3 ? A[2][k] : A[3][k];
        const float r1 = j < 1 ? A[1][k] : j < 2 ? A[2][k] : j < 3 ? A[3][k] : B[0][k];
        const float r2 = j < 1 ? A[2][k] : j < 2 ? A[3][k] : j < 3 ? B[0][k] : B[1][k];
        const float r3 = j < 1 ? A[3][k] : j < 2 ? B[0][k] : j < 3 ? B[1][k] : B[2][k];
        float b = tap_y(r0, r1, r2, r3, B[j][k]);
        if (!F32) b = round_storage(a.storage[0], b);
        if (EPI) {
          b = op_unsharp(j < 2 ? behind[j & 1][k] : raw[j < 2 ? 0 : j - 2][k], b, a.amount);
          if (!F32) b = round_storage(a.out.dtype, b);
        }
        o[k] = b;
      }
      if (vec && in_run) {
        if (F32 || a.out.dtype == HP_F32) {
          *reinterpret_cast<float4*>(out_row) = make_float4(o[0], o[1], o[2], o[3]);
        } else if (a.out.dtype == HP_BF16) {
          const __nv_bfloat162 q0 = __floats2bfloat162_rn(o[0], o[1]), q1 = __floats2bfloat162_rn(o[2], o[3]);
          *reinterpret_cast<uint2*>(out_row) =
              make_uint2(*reinterpret_cast<const unsigned*>(&q0), *reinterpret_cast<const unsigned*>(&q1));
        } else {
          const __half2 q0 = __floats2half2_rn(o[0], o[1]), q1 = __floats2half2_rn(o[2], o[3]);
          *reinterpret_cast<uint2*>(out_row) =
              make_uint2(*reinterpret_cast<const unsigned*>(&q0), *reinterpret_cast<const unsigned*>(&q1));
        }
      }
      if (cut) {
        if (part && in_run) {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (c0 + k < a.out.w) store_px(a.out, U.plane, c0 + k, U.oy + t, o[k]);
        }
      }
      out_row += a.out.rs;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) { behind[0][k] = raw[2][k]; behind[1][k] = raw[3][k]; }
    __syncwarp();   // every lane has read the box
    if (lane == 0 && i + kRing < U.nbox) issue(i + kRing, s);
    phase ^= s == kRing - 1;
    s = s == kRing - 1 ? 0 : s + 1;
    return true;
  }

  // False: a box never arrived.
  __device__ __forceinline__ bool run() {
    if (lane == 0)
      for (int i = 0; i < kRing && i < U.nbox; ++i) issue(i, i);
    float A[4][4], B[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int k = 0; k < 4; ++k) A[j][k] = 0.0f;
#pragma unroll 1
    for (int i = 0; i < U.nbox; i += 2) {
      if (!block(i, A, B)) return false;
      if (i + 1 < U.nbox && !block(i + 1, B, A)) return false;
    }
    return true;
  }
};

template <bool F32, bool EPI, bool BIN>
__global__ void __maxnreg__(BIN ? 96 : 128) k_stencil_rows(const __grid_constant__ SRowsParams kp) {
  grid_dep_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* base = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const StripGeom g = strip_geom(F32 || kp.a.in.dtype == HP_F32 ? 4 : 2);
  const int u = blockIdx.x * nw + warp;
  if (u >= kp.units) return;
  uint64_t* const bars = reinterpret_cast<uint64_t*>(base) + warp * kRing;
  unsigned char* const slots = base + kBarBytes + warp * kRing * g.slot_bytes;
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < kRing; ++i) mbar_init(bars + i, 1);
    fence_mbar_init();
  }
  __syncwarp();
  const Unit U = unit_geom(kp, g, u);
  StripRun<F32, EPI, BIN> run(kp, g, U, slots, bars, lane);
  if (!run.run()) {
    // a box never arrived: report, and wait (bounded) for copies still in
    // flight into this warp's slots (a slot's phase is at most one behind)
    if (lane == 0) {
      atomicExch(kp.a.err, 1);
      for (int i = 0; i < kRing; ++i) mbar_wait_poll(bars + i, i < run.s ? run.phase ^ 1 : run.phase, 100000000ull);
    }
    __syncwarp();
  }
}

typedef void (*SRowsKernel)(SRowsParams);

// Whether both passes' taps are the binomial ones, bit for bit.
bool binomial_taps(const ChainArgs& a) {
  static const float b[5] = {0.0625f, 0.25f, 0.375f, 0.25f, 0.0625f};
  return memcmp(a.w[0], b, sizeof b) == 0 && memcmp(a.w[0] + 5, b, sizeof b) == 0;
}

template <bool BIN>
SRowsKernel pick_fe(bool f32, bool epi) {
  if (epi) return f32 ? k_stencil_rows<true, true, BIN> : k_stencil_rows<false, true, BIN>;
  return f32 ? k_stencil_rows<true, false, BIN> : k_stencil_rows<false, false, BIN>;
}

SRowsKernel pick_kernel(const ChainArgs& a, int* variant) {
  const bool f32 = a.in.dtype == HP_F32 && a.storage[0] == HP_F32 && a.out.dtype == HP_F32;
  const bool epi = a.epilogue == 1;
  const bool bin = binomial_taps(a);
  *variant = (f32 ? 0 : 1) + (epi ? 2 : 0) + (bin ? 4 : 0);
  return bin ? pick_fe<true>(f32, epi) : pick_fe<false>(f32, epi);
}

}  // namespace

int stencil_rows_strip_w(int in_dtype) { return strip_geom(in_dtype == HP_F32 ? 4 : 2).strip_w; }

int stencil_rows_smem_bytes(int threads, int in_dtype) {
  const StripGeom g = strip_geom(in_dtype == HP_F32 ? 4 : 2);
  return 2 * 128 + kBarBytes + (threads / 32) * kRing * g.slot_bytes;  // alignment, and room for lane 31's right columns
}

// CTAs for `units` runs, one per warp; for 1 << 30 units: the CTAs that fill every
// SM at the kernel's occupancy.
int stencil_rows_grid(const ChainArgs& a, int units, int threads, int smem_bytes) {
  const int nw = threads / 32;
  const int need = (units + nw - 1) / nw;
  if (units < 1 << 30) return need;
  int dev = 0, sms = 0, per_sm = 0, variant = 0;
  SRowsKernel kern = pick_kernel(a, &variant);
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      allow_max_dynamic_smem((const void*)kern) != 0 ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem_bytes) != cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    return need < 2 * 152 ? need : 2 * 152;  // no device to ask: two CTAs on each of 152 SMs
  }
  return need < sms * per_sm ? need : sms * per_sm;
}

int launch_stencil_rows(const ChainArgs& a, int rows, int grid, int smem_bytes, void* stream) {
  int variant;
  SRowsKernel kern = pick_kernel(a, &variant);
  static bool configured[8] = {};
  if (!configured[variant]) {
    int e = allow_max_dynamic_smem((const void*)kern);
    if (e) return e;
    configured[variant] = true;
  }
  SRowsParams kp;
  memset(&kp, 0, sizeof kp);
  kp.a = a;
  const int dt = a.in.dtype;
  const int esize = dt == HP_F32 ? 4 : 2;
  const StripGeom g = strip_geom(esize);
  kp.strips = (a.out.w + g.strip_w - 1) / g.strip_w;
  kp.runs = (a.out.h + rows - 1) / rows;
  kp.rows = rows;
  kp.units = kp.strips * kp.runs * a.out.c;
  CUtensorMapDataType tdt = dt == HP_F32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                            : dt == HP_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  if (encode_tmap_3d(&kp.tmap, tdt, esize, a.in.data, a.in.w, a.in.h, a.in.c, a.in.rs, a.in.ps, 128, kBoxRows, 1))
    return (int)cudaErrorInvalidValue;
  { const int le_ = launch_kernel(kern, dim3(grid), dim3(a.threads), smem_bytes, stream, kp); if (le_) return le_; }
  __atomic_add_fetch(&g_launches, 1ULL, __ATOMIC_RELAXED);
  return (int)cudaGetLastError();
}

}  // namespace hp
