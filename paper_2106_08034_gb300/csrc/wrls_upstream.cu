// The denoiser's per-frame inputs from the renderer's raw data:
//   k_reconstruct : pixel reconstruction filter (Sec. 4, Table 2: the samples f_j of a pixel
//                   are filtered into I~_j; Sec. 6: separable Gaussian kernel), plus the
//                   variance of each pixel's sample mean;
//   k_velocity    : per-pixel backward motion from the first-collision world position
//                   (Sec. 5.3; Sec. 6 "Optical flow estimation"), projected with the previous
//                   frame's view-projection matrix.
#include <math.h>
#include <string.h>

#include <type_traits>

#include "wrls_internal.h"

namespace wrls {

// Reconstruction tiles: 32 x 8 pixels.
constexpr int kRecTW = 32, kRecTH = 8;
constexpr int kRecSW = kRecTW + 2, kRecSH = kRecTH + 2, kRecSP = kRecSW * kRecSH;

struct ReconArgs {
  float k2;      // log2(e) / (2 sigma^2): g(dx) g(dy) = 2^(-(dx^2 + dy^2) k2)
  float radius;  // support: |dx|, |dy| <= radius (binary32)
};

// I~_j = sum_k g(x_k - x_j) g(y_k - y_j) f_k / sum_k g g over the samples of the 3x3 pixels
// around j. Samples: ((s * 5 + k) * H + y) * W + x, k = r, g, b, ox, oy. One CTA per 32 x 8
// tile; the 34 x 10 windows of CH sample indices at a time are staged in shared
// memory (one barrier pair per chunk). A sample with a non-finite colour or offset, or
// outside the image, is staged with an infinite offset, which no support contains.
// The kernel is bound by its instructions and by the latency of each staging phase. With R = 2 each
// thread filters two vertically adjacent pixels: a staged sample is read once for both (30 shared loads a
// pixel and sample index instead of 45) and the two rows that reach both pixels run as packed
// pairs. Where all offsets of the chunk lie within radius - 1 of the pixel centre (always, with
// the default radius) the support needs no test. The terms of a pixel are added sample by sample, row by
// row, by the same operations in both forms. 1080p, us, R = 2 with 2 sample indices at a time: 2 samples a
// pixel with variance 54.1 -> 50.2, without 51.4 -> 41.5, 3 samples 72.0 -> 68.6, 16 samples 333 -> 317. (Four rows a
// thread: 55-63, fewer warps; 4 sample indices at a time: 58.8; 1: 75.)
// On small images, whose CTAs are all resident at once, twice the warps and half the phases are
// worth more: R = 1 with 4 sample indices at a time. With variance, R = 2 / R = 1, us: 128x128 4 samples 8.3 / 4.5, 16
// samples 29.4 / 13.6; 300x200 4 samples 9.0 / 5.3; 500x400 (800 tiles) 4 samples 12.0 / 11.1; 643x361 (966) without
// variance 10.9 / 11.1; 1280x720 33.1 / 36.0.
constexpr int kRecOneChunk = 4;    // sample indices at a time with one pixel a thread
constexpr int kRecOneBelow = 6;    // tiles an SM below which a thread takes one pixel

template <bool VAR, int R, int CH>
__global__ void __launch_bounds__(32 * kRecTH / R, 6 * R)
    k_reconstruct(const ReconArgs a, const int W, const int H, const int spp, const float* smp,
                  float* __restrict__ out, float* __restrict__ var) {
  constexpr int kWarps = kRecTH / R;
  __shared__ float sm[CH][5][kRecSP];
  const int bx0 = blockIdx.x * kRecTW, by0 = blockIdx.y * kRecTH;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int x = bx0 + lane, y0 = by0 + warp * R;
  const size_t np = (size_t)W * H;
  static_assert(R == 1 || R == 2, "a thread's pixels are the halves of its sums");
  float2 n0 = make_float2(0.0f, 0.0f), n1 = n0, n2 = n0, den = n0;
  // own samples, shifted by the first valid one (k): sums and sum of squares
  float k0[R] = {}, k1[R] = {}, k2[R] = {}, m0[R] = {}, m1[R] = {}, m2[R] = {}, q[R] = {};
  int cnt[R] = {};
  // near: every valid offset of the staged samples is within radius - 1, so that the support holds
  // all of the 3x3 neighbours and needs no test (rounding is monotone and radius representable)
  const float margin = a.radius - 1.0f;
  bool wide = false;
  auto stage = [&](int c, int s, int ly, int lx) {
    const int gx = bx0 - 1 + lx, gy = by0 - 1 + ly, ew = ly * kRecSW + lx;
    float r = 0.0f, g = 0.0f, b = 0.0f, ox = INFINITY, oy = INFINITY;
    if ((unsigned)gx < (unsigned)W && (unsigned)gy < (unsigned)H) {
      const float* base = smp + (size_t)s * 5 * np + (size_t)gy * W + gx;
      r = ld_global(base);
      g = ld_global(base + np);
      b = ld_global(base + 2 * np);
      ox = ld_global(base + 3 * np);
      oy = ld_global(base + 4 * np);
      // 0 * v is NaN for a non-finite v
      const float t = fmaf(oy, 0.0f, fmaf(ox, 0.0f, fmaf(b, 0.0f, fmaf(g, 0.0f, r * 0.0f))));
      if (t != t) {
        r = g = b = 0.0f;
        ox = oy = INFINITY;
      } else {
        wide = wide || !(fmaxf(fabsf(ox), fabsf(oy)) <= margin);
      }
    }
    sm[c][0][ew] = r;
    sm[c][1][ew] = g;
    sm[c][2][ew] = b;
    sm[c][3][ew] = ox;
    sm[c][4][ew] = oy;
  };
  pdl_wait();
  for (int s0 = 0; s0 < spp; s0 += CH) {
    const int ns = min(CH, spp - s0);
    if (R == 1) {
      for (int e = threadIdx.x; e < kRecSP * ns; e += 32 * kWarps) {
        const int c = e / kRecSP, ew = e - c * kRecSP;
        stage(c, s0 + c, ew / kRecSW, ew % kRecSW);
      }
    } else {
      for (int c = 0; c < ns; ++c) {  // a warp takes whole rows, the two left-over columns last
        // (unrolled: the loads of all of a thread's rows are in flight together)
#pragma unroll
        for (int k = 0; k < (kRecSH + kWarps - 1) / kWarps; ++k)
          if (warp + k * kWarps < kRecSH) stage(c, s0 + c, warp + k * kWarps, lane);
        const int e = threadIdx.x;
        if (e < 2 * kRecSH) stage(c, s0 + c, e >> 1, kRecTW + (e & 1));
      }
    }
    const bool near = !__syncthreads_or(wide);
    for (int c = 0; c < ns; ++c) {
      const float* w0 = &sm[c][0][warp * R * kRecSW + lane];  // window row and column of dy = dx = -1 of pixel 0
      auto filter = [&](auto all) {
        constexpr bool ALL = decltype(all)::value;
#pragma unroll
        for (int wr = 0; wr < R + 2; ++wr)
#pragma unroll
          for (int dx = -1; dx <= 1; ++dx) {
            const float* e = w0 + wr * kRecSW + dx + 1;
            const float r = e[0], g = e[kRecSP], b = e[2 * kRecSP], ox = e[3 * kRecSP], oy = e[4 * kRecSP];
            const float ux = (float)dx + ox;
            const float ux2 = ALL || fabsf(ux) <= a.radius ? ux * ux : INFINITY;  // weight 2^-inf = 0
            if (R == 2 && (wr == 1 || wr == 2)) {  // both pixels, packed
              const float2 uy = f2add(make_float2(oy, oy), make_float2((float)(wr - 1), (float)(wr - 2)));
              const float2 t = f2mul(f2fma(uy, uy, make_float2(ux2, ux2)), make_float2(-a.k2, -a.k2));
              float2 w = make_float2(ex2_approx(t.x), ex2_approx(t.y));
              if (!ALL) w = make_float2(fabsf(uy.x) <= a.radius ? w.x : 0.0f, fabsf(uy.y) <= a.radius ? w.y : 0.0f);
              n0 = f2fma(w, make_float2(r, r), n0);
              n1 = f2fma(w, make_float2(g, g), n1);
              n2 = f2fma(w, make_float2(b, b), n2);
              den = f2add(den, w);
            } else {
              const bool lower = R == 2 && wr == 3;  // the last window row reaches the lower pixel alone
              const float uy = (float)(lower ? 1 : wr - 1) + oy;
              float w = ex2_approx(fmaf(uy, uy, ux2) * -a.k2);
              if (!ALL) w = fabsf(uy) <= a.radius ? w : 0.0f;
              if (!lower) {
                n0.x = fmaf(w, r, n0.x);
                n1.x = fmaf(w, g, n1.x);
                n2.x = fmaf(w, b, n2.x);
                den.x += w;
              } else {
                n0.y = fmaf(w, r, n0.y);
                n1.y = fmaf(w, g, n1.y);
                n2.y = fmaf(w, b, n2.y);
                den.y += w;
              }
            }
          }
      };
      if (near) filter(std::integral_constant<bool, true>{});
      else filter(std::integral_constant<bool, false>{});
      if (VAR) {
        const float* e = w0 + kRecSW + 1;
#pragma unroll
        for (int i = 0; i < R; ++i, e += kRecSW) {
          const float r = e[0], g = e[kRecSP], b = e[2 * kRecSP];
          const bool own = e[3 * kRecSP] < INFINITY;  // own sample is valid (an invalid one adds 0)
          if (cnt[i] == 0) {
            k0[i] = r;
            k1[i] = g;
            k2[i] = b;
          }
          const float dr = own ? r - k0[i] : 0.0f, dg = own ? g - k1[i] : 0.0f, db = own ? b - k2[i] : 0.0f;
          m0[i] += dr;
          m1[i] += dg;
          m2[i] += db;
          q[i] = fmaf(dr, dr, fmaf(dg, dg, fmaf(db, db, q[i])));
          cnt[i] += own ? 1 : 0;
        }
      }
    }
    __syncthreads();
  }
  if (x >= W) return;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    if (y0 + i >= H) break;
    const size_t j = (size_t)(y0 + i) * W + x;
    const float d = i ? den.y : den.x;
    const float inv = d > 0.0f ? 1.0f / d : __int_as_float(0x7fc00000);
    out[j] = (i ? n0.y : n0.x) * inv;
    out[np + j] = (i ? n1.y : n1.x) * inv;
    out[2 * np + j] = (i ? n2.y : n2.x) * inv;
    if (VAR) {
      if (cnt[i] < 2) {
        var[j] = __int_as_float(0x7fc00000);
      } else {
        // sum over channels of sum_s (f - mean)^2 = sum u^2 - (sum u)^2 / n, u = f - k
        const float fn = (float)cnt[i];
        const float ss = q[i] - fmaf(m2[i], m2[i], fmaf(m1[i], m1[i], m0[i] * m0[i])) / fn;
        var[j] = fmaxf(ss, 0.0f) / (3.0f * (fn - 1.0f)) / fn;
      }
    }
  }
}

struct Mat4 {
  float m[16];
};

// V pixels a thread: 4 with 128-bit accesses where every plane's rows allow it (W a multiple of 4,
// 16-byte aligned buffers), else 1. A streaming kernel: 1080p 12.4 -> 10.3 us, 8.0 with the launch set up
// beside the kernel before (20 B a pixel, 6.1 us at the copy rate). Neither form lets the next launch in
// before its CTAs end: on small images the next kernel's would crowd on the SMs that are free first
// (reconstruction and velocity in turn, 500x400, 4 samples: 21.4 -> 13.0 us), and beside the many CTAs of one
// pixel a thread they contend (1080p 12.4 -> 18.8 us).
template <int V>
__global__ void k_velocity(const Mat4 M, const int W, const int H, const int miss_policy,
                           const float* world, float* __restrict__ mot) {
  const int x0 = (blockIdx.x * blockDim.x + threadIdx.x) * V, y = blockIdx.y;
  pdl_wait();
  if (x0 >= W || y >= H) return;
  const size_t np = (size_t)W * H, j = (size_t)y * W + x0;
  float p[3][V], v[2][V];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (V == 4) {
      const float4 t = ld_global(reinterpret_cast<const float4*>(world + c * np + j));
      p[c][0] = t.x;
      p[c][V > 1 ? 1 : 0] = t.y;
      p[c][V > 2 ? 2 : 0] = t.z;
      p[c][V > 3 ? 3 : 0] = t.w;
    } else {
      p[c][0] = ld_global(world + c * np + j);
    }
  }
  const float nan = __int_as_float(0x7fc00000);
#pragma unroll
  for (int k = 0; k < V; ++k) {
    const float X = p[0][k], Y = p[1][k], Z = p[2][k];
    if (!(isfinite(X) && isfinite(Y) && isfinite(Z))) {
      v[0][k] = v[1][k] = miss_policy == 0 ? 0.0f : nan;
      continue;
    }
    const float cw = fmaf(M.m[12], X, fmaf(M.m[13], Y, fmaf(M.m[14], Z, M.m[15])));
    if (!(cw > 0.0f)) {
      v[0][k] = v[1][k] = nan;
      continue;
    }
    const float cx = fmaf(M.m[0], X, fmaf(M.m[1], Y, fmaf(M.m[2], Z, M.m[3])));
    const float cy = fmaf(M.m[4], X, fmaf(M.m[5], Y, fmaf(M.m[6], Z, M.m[7])));
    const float iw = 1.0f / cw;
    v[0][k] = fmaf(cx * iw + 1.0f, 0.5f * (float)W, -0.5f) - (float)(x0 + k);
    v[1][k] = fmaf(1.0f - cy * iw, 0.5f * (float)H, -0.5f) - (float)y;
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    if (V == 4)
      *reinterpret_cast<float4*>(mot + c * np + j) =
          make_float4(v[c][0], v[c][V > 1 ? 1 : 0], v[c][V > 2 ? 2 : 0], v[c][V > 3 ? 3 : 0]);
    else
      mot[c * np + j] = v[c][0];
  }
}

}  // namespace wrls

using namespace wrls;

static bool in_range(int w, int h) { return w >= 1 && h >= 1 && w <= 16384 && h <= 16384; }

static bool overlap_bytes(const void* a, size_t an, const void* b, size_t bn) {
  if (!a || !b) return false;
  const char* x = (const char*)a;
  const char* y = (const char*)b;
  return x < y + bn && y < x + an;
}

extern "C" {

void wrls_recon_params_default(wrls_recon_params* p) {
  if (!p) return;
  memset(p, 0, sizeof(*p));
  p->struct_size = sizeof(wrls_recon_params);
  p->sigma = 0.5f;
  p->radius = 1.5f;
}

wrls_status wrls_reconstruct(int width, int height, int spp, const float* samples, const wrls_recon_params* p,
                             float* radiance, float* variance, void* cuda_stream) {
  NvtxRange nvtx("wrls_reconstruct");
  if (!p || p->struct_size != sizeof(wrls_recon_params)) {
    set_error("wrls_reconstruct: params NULL or struct_size != sizeof(wrls_recon_params)");
    return WRLS_ERR_INVALID_ARG;
  }
  if (!in_range(width, height) || spp < 1 || spp > 1024 || !samples || !radiance) {
    set_error("wrls_reconstruct: bad size (%d x %d, spp %d) or NULL samples/radiance", width, height, spp);
    return WRLS_ERR_INVALID_ARG;
  }
  if (!(p->sigma > 0.0f) || !(p->radius > 0.0f && p->radius <= 1.5f)) {
    set_error("wrls_reconstruct: sigma must be > 0 and radius in (0, 1.5]");
    return WRLS_ERR_INVALID_ARG;
  }
  if (((uintptr_t)samples | (uintptr_t)radiance | (uintptr_t)variance) & 3u) {
    set_error("wrls_reconstruct: buffers must be 4-byte aligned");
    return WRLS_ERR_INVALID_ARG;
  }
  const size_t np = (size_t)width * height;
  if (overlap_bytes(radiance, 12 * np, samples, 20 * np * spp) || overlap_bytes(variance, 4 * np, samples, 20 * np * spp) ||
      overlap_bytes(radiance, 12 * np, variance, 4 * np)) {
    set_error("wrls_reconstruct: outputs overlap each other or the samples");
    return WRLS_ERR_INVALID_ARG;
  }
  ReconArgs a;
  // k2 stays above 0 (sigma up to infinity: a box filter, weight 2^-0 = 1 within the support), so that
  // the infinite offset of a missing sample or of one outside the image gives 2^-inf = 0, not inf * 0 = NaN
  a.k2 = fmaxf((float)(1.4426950408889634 / (2.0 * (double)p->sigma * (double)p->sigma)), 1.17549435e-38f);
  a.radius = p->radius;
  const dim3 grid((width + kRecTW - 1) / kRecTW, (height + kRecTH - 1) / kRecTH);
  cudaStream_t cs = (cudaStream_t)cuda_stream;
  const bool one = (int)(grid.x * grid.y) < kRecOneBelow * sm_count();  // one pixel a thread (see the kernel)
  cudaError_t e = launch_kernel(one ? (variance ? k_reconstruct<true, 1, kRecOneChunk> : k_reconstruct<false, 1, kRecOneChunk>)
                                    : (variance ? k_reconstruct<true, 2, 2> : k_reconstruct<false, 2, 2>),
                                grid, one ? 32 * kRecTH : 32 * kRecTH / 2, 0, cs, pdl_allowed(cs), a, width, height, spp, samples,
                                radiance, variance);
  if (e != cudaSuccess) {
    set_error("wrls_reconstruct: launch: %s", cudaGetErrorString(e));
    return WRLS_ERR_CUDA;
  }
  return WRLS_OK;
}

wrls_status wrls_velocity_from_world(int width, int height, const float* world, const float* prev_view_proj,
                                     int miss_policy, float* motion, void* cuda_stream) {
  NvtxRange nvtx("wrls_velocity_from_world");
  if (!in_range(width, height) || !world || !prev_view_proj || !motion || miss_policy < 0 || miss_policy > 1) {
    set_error("wrls_velocity_from_world: bad size (%d x %d), NULL pointer or miss_policy %d", width, height,
              miss_policy);
    return WRLS_ERR_INVALID_ARG;
  }
  if (((uintptr_t)world | (uintptr_t)motion) & 3u) {
    set_error("wrls_velocity_from_world: buffers must be 4-byte aligned");
    return WRLS_ERR_INVALID_ARG;
  }
  const size_t np = (size_t)width * height;
  if (overlap_bytes(motion, 8 * np, world, 12 * np)) {
    set_error("wrls_velocity_from_world: motion overlaps world");
    return WRLS_ERR_INVALID_ARG;
  }
  Mat4 M;
  for (int i = 0; i < 16; ++i) {
    if (!isfinite(prev_view_proj[i])) {
      set_error("wrls_velocity_from_world: prev_view_proj[%d] is not finite", i);
      return WRLS_ERR_INVALID_ARG;
    }
    M.m[i] = prev_view_proj[i];
  }
  const bool vec = width % 4 == 0 && (((uintptr_t)world | (uintptr_t)motion) & 15u) == 0;
  cudaStream_t cs = (cudaStream_t)cuda_stream;
  cudaError_t e = launch_kernel(vec ? k_velocity<4> : k_velocity<1>, dim3(((vec ? width / 4 : width) + 127) / 128, height), 128, 0,
                                cs, vec && pdl_allowed(cs), M, width, height, miss_policy, world, motion);
  if (e != cudaSuccess) {
    set_error("wrls_velocity_from_world: launch: %s", cudaGetErrorString(e));
    return WRLS_ERR_CUDA;
  }
  return WRLS_OK;
}

}  // extern "C"
