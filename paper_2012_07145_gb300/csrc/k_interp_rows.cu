// One level of the interpolate app's composite (Sec. 6 app list), streaming:
// I_l = D_l over U(I_{l+1}) for the 4 premultiplied channels, and at the
// finest level the division by coverage, out = I_0.rgb / I_0.a.
//
// One warp per strip of 30 coarse columns walks down a run of coarse rows.
// Lane l owns coarse column m = 30 s + l - 1 and the fine columns 2m and 2m+1.
// Per coarse row it loads the 4 channels of I_{l+1} at its column and takes
// the x pass of the upsample for its two fine columns (coarse neighbours m-1,
// m+1 by warp shuffles): even fine columns 1/8, 6/8, 1/8 over m-1, m, m+1; odd
// ones 1/2, 1/2 over m, m+1.  A window of three x-passed coarse rows (in
// registers) gives the y pass of fine rows 2n (1/8, 6/8, 1/8 over n-1, n, n+1)
// and 2n+1 (1/2, 1/2 over n, n+1); the composite with D_l follows per pixel.
// Lanes 0 and 31 only feed their neighbours.  The two fine rows of D_l a
// coarse step composites arrive as one TMA box (68 fine columns from a 16-byte
// aligned start, 2 rows, the 4 planes) through a ring of 3 shared-memory slots
// private to the warp (a warp runs one run): three are issued with the run, each
// next one once its slot is read, so the fine loads are in flight well ahead of
// their use without holding registers.  The operations are those of the
// per-pixel expressions (x pass over each coarse row, then the y pass, in tap
// order; op_over, op_unpremul), so results are bit-identical to the generic
// kernel.  All stages are stored as f32 (the host checks).  Bound by issue and the
// coarse rows' latency: the finest level of 2560x1536 takes 26.7 us alone (0.69 of
// the measured copy rate).
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstring>

#include "hp_internal.h"
#include "stage_math.cuh"
#include "tma.cuh"

namespace hp {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kStripW = 30;   // coarse columns per warp
constexpr int kBoxW = 68;     // fine columns per box: lanes 0..31's 64, from 4 left of lane 1's first (16-byte aligned)
constexpr int kBoxBytes = kBoxW * 2 * 4 * 4;          // 2 fine rows x 4 planes x f32
constexpr int kSlotBytes = (kBoxBytes + 127) / 128 * 128;  // slots start on 128-byte boundaries
constexpr int kRing = 3;      // boxes per warp ring
constexpr int kBarBytes = 512;  // mbarriers of up to 16 warps x kRing

struct InterpParams {
  CUtensorMap tmap;  // the fine level D_l: (W, H, planes), box (kBoxW, 2, 4)
  InterpArgs a;
  int strips, units;
};

// One run of coarse rows of one strip.  Box j (fine rows 2 (n0 + j) and
// 2 (n0 + j) + 1) lives in slot j % kRing of the warp's ring and completes phase
// (j / kRing) & 1 of that slot's mbarrier.  PREMUL: the fine image is not yet
// premultiplied (the premultiply stage is folded in).
template <bool FINAL, bool PREMUL>
struct InterpRun {
  const InterpParams& P;
  unsigned char* const slots;
  uint64_t* const bars;
  int m, cm, X0, X1, n0, nrun, c0, c1;  // c0, c1: X0, X1 as columns of the box
  bool pair, prod, ok1;
  int s, phase;               // slot and phase of the next box
  const float* box;           // the box being read
  float hx[3][4][2];  // x-passed coarse rows (window slot, channel, fine column)
  float raw[4];       // the next coarse row, in flight

  __device__ __forceinline__ InterpRun(const InterpParams& p, unsigned char* slots_, uint64_t* bars_)
      : P(p), slots(slots_), bars(bars_), s(0), phase(0), box(nullptr) {}

  __device__ __forceinline__ void issue(int strip, int j, int slot) const {
    // the warp's reads of this slot (its previous box) come before the copy
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_arrive_expect_tx(bars + slot, (unsigned)kBoxBytes);
    tma_load_3d(slots + slot * kSlotBytes, &P.tmap, 2 * (strip * kStripW) - 4, 2 * (n0 + j), 0, bars + slot);
  }

  __device__ __forceinline__ void load_raw(int q) {
    const ImgView& c = P.a.coarse;
    const char* row = (const char*)c.data + (long long)iclamp(n0 - 1 + q, 0, c.h - 1) * c.rs;
#pragma unroll
    for (int ch = 0; ch < 4; ++ch) raw[ch] = __ldg(reinterpret_cast<const float*>(row + ch * c.ps) + cm);
  }

  template <int S>
  __device__ __forceinline__ void xpass() {
#pragma unroll
    for (int ch = 0; ch < 4; ++ch) {
      const float l = __shfl_up_sync(kFull, raw[ch], 1);
      const float r = __shfl_down_sync(kFull, raw[ch], 1);
      hx[S][ch][0] = __fmaf_rn(0.125f, r, __fmaf_rn(0.75f, raw[ch], __fmul_rn(0.125f, l)));
      hx[S][ch][1] = __fmaf_rn(0.5f, r, __fmul_rn(0.5f, raw[ch]));
    }
  }

  // Fine row Y (row ODD of the current box) from window slots of coarse rows
  // n-1 (A), n (B), n+1 (C).
  template <bool ODD, int A, int B, int C>
  __device__ __forceinline__ void emit(int Y) const {
    float d[4][2];
#pragma unroll
    for (int ch = 0; ch < 4; ++ch) {
      const float* q = box + (2 * ch + (ODD ? 1 : 0)) * kBoxW;
      if (pair) {
        const float2 v = *reinterpret_cast<const float2*>(q + c0);
        d[ch][0] = v.x;
        d[ch][1] = v.y;
      } else {
        d[ch][0] = q[c0];
        d[ch][1] = q[c1];
      }
    }
    if (PREMUL) {
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) {
        d[ch][0] = op_premul(d[ch][0], d[3][0], ch);
        d[ch][1] = op_premul(d[ch][1], d[3][1], ch);
      }
    }
    float o[4][2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
#pragma unroll
      for (int ch = 0; ch < 4; ++ch) {
        const float u = ODD ? __fmaf_rn(0.5f, hx[C][ch][j], __fmul_rn(0.5f, hx[B][ch][j]))
                            : __fmaf_rn(0.125f, hx[C][ch][j], __fmaf_rn(0.75f, hx[B][ch][j], __fmul_rn(0.125f, hx[A][ch][j])));
        o[ch][j] = op_over(d[ch][j], d[3][j], u);
      }
      if (FINAL) {
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) o[ch][j] = op_unpremul(o[ch][j], o[3][j]);
      }
    }
    if (!prod) return;
    const ImgView& ov = P.a.out;
    char* orow = (char*)ov.data + (long long)Y * ov.rs;
#pragma unroll
    for (int ch = 0; ch < (FINAL ? 3 : 4); ++ch) {
      float* q = reinterpret_cast<float*>(orow + ch * ov.ps);
      if (ok1 && P.a.vec) {
        reinterpret_cast<float2*>(q)[X0 >> 1] = make_float2(o[ch][0], o[ch][1]);
      } else {
        q[X0] = o[ch][0];
        if (ok1) q[X1] = o[ch][1];
      }
    }
  }

  // False: a box never arrived.
  template <int PH>
  __device__ __forceinline__ bool step(int strip, int i, int lane) {
    constexpr int A = PH, B = (PH + 1) % 3, C = (PH + 2) % 3;
    xpass<C>();
    if (i + 3 <= nrun + 1) load_raw(i + 3);
    // every lane waits for the box itself (usually there: one test)
    if (!__all_sync(kFull, mbar_try_wait(bars + s, phase) || mbar_wait_poll(bars + s, phase, 2000000000ull))) return false;
    box = reinterpret_cast<const float*>(slots + s * kSlotBytes);
    const int Y = 2 * (n0 + i);
    emit<false, A, B, C>(Y);
    if (Y + 1 < P.a.fine.h) emit<true, A, B, C>(Y + 1);
    __syncwarp();   // every lane has read the box
    if (lane == 0 && i + kRing < nrun) issue(strip, i + kRing, s);
    phase ^= s == kRing - 1;
    s = s == kRing - 1 ? 0 : s + 1;
    return true;
  }

  __device__ __forceinline__ bool run(int strip, int run_idx) {
    const int lane = threadIdx.x & 31;
    const int W = P.a.fine.w;
    m = strip * kStripW + lane - 1;
    cm = iclamp(m, 0, P.a.coarse.w - 1);
    X0 = iclamp(2 * m, 0, W - 1);
    X1 = iclamp(2 * m + 1, 0, W - 1);
    c0 = X0 - (2 * (strip * kStripW) - 4);
    c1 = X1 - (2 * (strip * kStripW) - 4);
    pair = 2 * m >= 0 && 2 * m + 1 <= W - 1;
    prod = lane >= 1 && lane <= kStripW && 2 * m <= W - 1;
    ok1 = prod && 2 * m + 1 <= W - 1;
    n0 = run_idx * P.a.rows;
    nrun = imin(P.a.rows, P.a.coarse.h - n0);
    if (lane == 0)
      for (int j = 0; j < kRing && j < nrun; ++j) issue(strip, j, j);
    load_raw(0);
    xpass<0>();
    load_raw(1);
    xpass<1>();
    load_raw(2);
    for (int i = 0; i < nrun; i += 3) {
      if (!step<0>(strip, i, lane)) return false;
      if (i + 1 >= nrun) break;
      if (!step<1>(strip, i + 1, lane)) return false;
      if (i + 2 >= nrun) break;
      if (!step<2>(strip, i + 2, lane)) return false;
    }
    return true;
  }
};

template <bool FINAL, bool PREMUL>
__global__ void __launch_bounds__(256, 3) k_interp_rows(const __grid_constant__ InterpParams P) {
  grid_dep_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* base = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int u = blockIdx.x * nw + warp;
  if (u >= P.units) return;
  uint64_t* const bars = reinterpret_cast<uint64_t*>(base) + warp * kRing;
  unsigned char* const slots = base + kBarBytes + warp * kRing * kSlotBytes;
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < kRing; ++i) mbar_init(bars + i, 1);
    fence_mbar_init();
  }
  __syncwarp();
  InterpRun<FINAL, PREMUL> r(P, slots, bars);
  if (!r.run(u % P.strips, u / P.strips)) {
    // a box never arrived: report, and wait (bounded) for copies still in
    // flight into this warp's slots (a slot's phase is at most one behind)
    if (lane == 0) {
      atomicExch(P.a.err, 1);
      for (int i = 0; i < kRing; ++i) mbar_wait_poll(bars + i, i < r.s ? r.phase ^ 1 : r.phase, 100000000ull);
    }
    __syncwarp();
  }
}

typedef void (*InterpKernel)(InterpParams);

InterpKernel pick_kernel(const InterpArgs& a) {
  if (a.premul) return a.final_div ? k_interp_rows<true, true> : k_interp_rows<false, true>;
  return a.final_div ? k_interp_rows<true, false> : k_interp_rows<false, false>;
}

}  // namespace

int interp_rows_strip_w() { return kStripW; }

int interp_rows_smem_bytes(int threads) { return 128 + kBarBytes + (threads / 32) * kRing * kSlotBytes; }

// CTAs for `units` runs, one per warp; for 1 << 30 units: the CTAs that fill every
// SM at the kernel's occupancy.
int interp_rows_grid(const InterpArgs& a, int units, int threads) {
  const int nw = threads / 32;
  const int need = (units + nw - 1) / nw;
  if (units < 1 << 30) return need;
  int dev = 0, sms = 0, per_sm = 0;
  const InterpKernel kern = pick_kernel(a);
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      allow_max_dynamic_smem((const void*)kern) != 0 ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, interp_rows_smem_bytes(threads)) != cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    return need < 2 * 152 ? need : 2 * 152;  // no device to ask: two CTAs on each of 152 SMs
  }
  return need < sms * per_sm ? need : sms * per_sm;
}

int launch_interp_rows(const InterpArgs& a_in, int grid, void* stream) {
  InterpArgs a = a_in;
  if (a.rows < 1 || a.threads < 32 || a.threads > 256 || a.threads % 32 || grid < 1) return (int)cudaErrorInvalidValue;
  if (a.fine.dtype != HP_F32 || a.coarse.dtype != HP_F32 || a.out.dtype != HP_F32 || a.fine.c < 4 || a.coarse.c < 4 ||
      a.out.c < (a.final_div ? 3 : 4))
    return (int)cudaErrorInvalidValue;
  auto al = [](const ImgView& v) { return (long long)(size_t)v.data % 8 == 0 && v.rs % 8 == 0 && v.ps % 8 == 0; };
  a.vec = al(a.fine) && al(a.out);
  InterpParams kp;
  memset(&kp, 0, sizeof kp);
  kp.a = a;
  kp.strips = (a.coarse.w + kStripW - 1) / kStripW;
  kp.units = kp.strips * ((a.coarse.h + a.rows - 1) / a.rows);
  const InterpKernel kern = pick_kernel(a);
  // once per kernel: it is four runtime calls, and a direct launch pays them on every realize
  static bool configured[4] = {};
  bool& done = configured[(a.premul ? 2 : 0) + (a.final_div ? 1 : 0)];
  if (!done) {
    int e = allow_max_dynamic_smem((const void*)kern);
    if (e) return e;
    done = true;
  }
  if (encode_tmap_3d(&kp.tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, a.fine.data, a.fine.w, a.fine.h, a.fine.c, a.fine.rs,
                     a.fine.ps, kBoxW, 2, 4))
    return (int)cudaErrorInvalidValue;
  { const int le_ = launch_kernel(kern, dim3(grid), dim3(a.threads), interp_rows_smem_bytes(a.threads), stream, kp); if (le_) return le_; }
  __atomic_add_fetch(&g_launches, 1ULL, __ATOMIC_RELAXED);
  return (int)cudaGetLastError();
}

}  // namespace hp
