// The coarse end of a pyramid in one launch: every downsample below a level of at
// most kTailPixels pixels and every level step back up to it, by one CTA in shared
// memory.  A launch of its own per level and direction costs about 3 us each
// whatever its size; these levels together are a few thousand pixels.
//   - interpolate: D_i = downsample(D_{i-1}), then I_i = D_i over upsample(I_{i+1})
//     in place of D_i (a thread holds the four channels of its pixel);
//   - local Laplacian: G_i = downsample(G_{i-1}) for the K remaps and gray, then
//     R_i = blend of L_i at gray + upsample(R_{i+1}), beside the stacks.
// Values are those of the per-level kernels: x pass of each row, then the y pass,
// taps in order, clamped indices, the same point-wise expressions.
// Threads are dealt out over a level's values, not its rows, so that a level is the
// same few steps of the CTA whatever its shape (a warp per row took 177 us a realize
// for a 16x20000 image, 10 levels, and 275 for its local Laplacian, against 76 and 99
// with a launch per level; 52 and 77 dealt out).
// Bound by the barriers and shared-memory latency of one CTA: 2559x1535 RGBA, levels
// 6 to 9 (40x24 to 5x3) and back in place of six launches, 103.0 -> 98.6 us in all.
#include <cuda_runtime.h>

#include <cstring>

#include "hist_common.cuh"
#include "hp_internal.h"
#include "stage_math.cuh"

namespace hp {

namespace {

constexpr int kThreads = 1024;

struct TailParams {
  PyrTailArgs a;
  int off[kTailLevels];   // float offset of level i's stack in shared memory
  int roff[kTailLevels];  // local Laplacian: of R_i
  FastDiv w[kTailLevels], h[kTailLevels];  // a value's row and column, channel and row
};

// Downsampled value at (x, y) of a w x h plane.
__device__ __forceinline__ float down_at(const float* p, int w, int h, int x, int y) {
  int cx[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) cx[k] = iclamp(2 * x - 2 + k, 0, w - 1);
  float r[5];
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    const float* q = p + iclamp(2 * y - 2 + j, 0, h - 1) * w;
    r[j] = tap5_binomial16(q[cx[0]], q[cx[1]], q[cx[2]], q[cx[3]], q[cx[4]]);
  }
  return tap5_binomial16(r[0], r[1], r[2], r[3], r[4]);
}

// The coarse rows and columns under a fine pixel, and its parities.
struct UpAt {
  int x0, x1, x2, y0, y1, y2;  // clamped m - 1, m, m + 1; rows as offsets
  bool ox, oy;
  __device__ __forceinline__ UpAt(int X, int Y, int w, int h) {
    const int m = X >> 1, n = Y >> 1;
    x0 = iclamp(m - 1, 0, w - 1); x1 = iclamp(m, 0, w - 1); x2 = iclamp(m + 1, 0, w - 1);
    y0 = iclamp(n - 1, 0, h - 1) * w; y1 = iclamp(n, 0, h - 1) * w; y2 = iclamp(n + 1, 0, h - 1) * w;
    ox = X & 1; oy = Y & 1;
  }
  __device__ __forceinline__ float row(const float* q) const {
    const float c = q[x1], r = q[x2];
    if (ox) return __fmaf_rn(0.5f, r, __fmul_rn(0.5f, c));
    return __fmaf_rn(0.125f, r, __fmaf_rn(0.75f, c, __fmul_rn(0.125f, q[x0])));
  }
  __device__ __forceinline__ float at(const float* p) const {
    const float b = row(p + y1), c = row(p + y2);
    if (oy) return __fmaf_rn(0.5f, c, __fmul_rn(0.5f, b));
    return __fmaf_rn(0.125f, c, __fmaf_rn(0.75f, b, __fmul_rn(0.125f, row(p + y0))));
  }
};

template <bool LL>
__global__ void __launch_bounds__(kThreads) k_pyr_tail(const __grid_constant__ TailParams P) {
  grid_dep_wait();
  extern __shared__ float sm[];
  const PyrTailArgs& a = P.a;
  const int C = a.channels;
  {  // the finest level of the tail
    const int w = a.w[0], h = a.h[0];
    for (int i = threadIdx.x; i < C * h * w; i += kThreads) {
      const int r = fastdiv(i, P.w[0]), x = i - r * w, c = fastdiv(r, P.h[0]), y = r - c * h;
      sm[i] = __ldg(reinterpret_cast<const float*>((const char*)a.src.data + c * a.src.ps + (long long)y * a.src.rs) + x);
    }
  }
  for (int l = 1; l < a.levels; ++l) {
    __syncthreads();
    const int w = a.w[l], h = a.h[l], fw = a.w[l - 1], fh = a.h[l - 1];
    const float* f = sm + P.off[l - 1];
    float* o = sm + P.off[l];
    for (int i = threadIdx.x; i < C * h * w; i += kThreads) {
      const int r = fastdiv(i, P.w[l]), x = i - r * w, c = fastdiv(r, P.h[l]), y = r - c * h;
      o[i] = down_at(f + c * fw * fh, fw, fh, x, y);
    }
  }
  for (int l = a.levels - 2; l >= 0; --l) {
    __syncthreads();
    const int w = a.w[l], n = w * a.h[l], cw = a.w[l + 1], ch = a.h[l + 1], cn = cw * ch;
    float* d = sm + P.off[l];
    const float* cs = sm + P.off[l + 1];
    for (int i = threadIdx.x; i < n; i += kThreads) {
      const int y = fastdiv(i, P.w[l]), x = i - y * w;
      const UpAt u(x, y, cw, ch);
      char* out = (char*)a.out.data + (long long)y * a.out.rs + 4LL * x;
      if (LL) {
        const float* cr = l + 2 == a.levels ? cs + a.rn_ch * cn : sm + P.roff[l + 1];
        int k0;
        float f;
        ll_interp_index(d[a.K * n + i], a.K, &k0, &f);
        const float L0 = __fsub_rn(d[k0 * n + i], u.at(cs + k0 * cn));
        const float L1 = __fsub_rn(d[(k0 + 1) * n + i], u.at(cs + (k0 + 1) * cn));
        const float r = __fadd_rn(op_ll_blend(L0, L1, f), u.at(cr));
        if (l) sm[P.roff[l] + i] = r;
        else *reinterpret_cast<float*>(out) = r;
      } else {
        const float al = d[3 * n + i];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float v = op_over(d[c * n + i], al, u.at(cs + c * cn));
          if (l) d[c * n + i] = v;
          else *reinterpret_cast<float*>(out + c * a.out.ps) = v;
        }
      }
    }
  }
}

// Float offsets of a tail's levels; returns the floats in all.
long long layout(const PyrTailArgs& a, int* off, int* roff) {
  long long at = 0;
  for (int l = 0; l < a.levels; ++l) {
    off[l] = (int)at;
    at += (long long)a.w[l] * a.h[l] * a.channels;
  }
  for (int l = 0; l < a.levels; ++l) {
    roff[l] = (int)at;
    if (a.ll && l > 0 && l + 1 < a.levels) at += (long long)a.w[l] * a.h[l];
  }
  return at;
}

}  // namespace

int pyr_tail_threads() { return kThreads; }

// Shared memory of a tail, or 0 where it does not fit one CTA.
int pyr_tail_smem_bytes(const PyrTailArgs& a) {
  int off[kTailLevels], roff[kTailLevels];
  if (a.levels < 2 || a.levels > kTailLevels || (long long)a.w[0] * a.h[0] > kTailPixels) return 0;
  const long long b = layout(a, off, roff) * 4;
  return b <= kSmemLimit ? (int)b : 0;
}

int launch_pyr_tail(const PyrTailArgs& a, void* stream) {
  const int smem = pyr_tail_smem_bytes(a);
  if (!smem || a.src.dtype != HP_F32 || a.out.dtype != HP_F32 || a.src.c < a.channels) return (int)cudaErrorInvalidValue;
  TailParams kp;
  memset(&kp, 0, sizeof kp);
  kp.a = a;
  layout(a, kp.off, kp.roff);
  for (int l = 0; l < a.levels; ++l) {
    kp.w[l] = make_fastdiv(a.w[l]);
    kp.h[l] = make_fastdiv(a.h[l]);
  }
  auto kern = a.ll ? k_pyr_tail<true> : k_pyr_tail<false>;
  static bool configured[2] = {};
  if (!configured[a.ll ? 1 : 0]) {
    const int e = allow_max_dynamic_smem((const void*)kern);
    if (e) return e;
    configured[a.ll ? 1 : 0] = true;
  }
  const int le = launch_kernel(kern, dim3(1), dim3(kThreads), smem, stream, kp);
  if (le) return le;
  __atomic_add_fetch(&g_launches, 1ULL, __ATOMIC_RELAXED);
  return (int)cudaGetLastError();
}

}  // namespace hp
