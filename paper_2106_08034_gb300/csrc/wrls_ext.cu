// Extended predictor and weights (streams whose parameters select them):
//   - G-buffer entries in the predictor, p = [1, z, g_1..g_n] (or [1, g_1..g_n] without the
//     temporal feature), d up to 8: the regression on auxiliary G-buffer features of RLS
//     denoisers that Sec. 2.1 and Sec. 5.2-5.3 discuss (and argue against for noisy
//     path-traced G-buffers);
//   - the sample-variance weight that Sec. 5.3 sets aside: Eq. 13 with the squared colour
//     distance replaced by its expectation 3 sigma^2 under the per-pixel variance;
//   - nearest-pixel reprojection (floor(q + 0.5) per axis, binary32).
// Everything else is the paper's step for step: reprojection, Eq. 12 feature with the 3x3
// clamp, Eq. 13 / Eq. 14 / Eq. 8 / Eq. 9 / Eq. 11, restarts, missing samples, the wind-up
// guard and the 5x5 bilateral cross-prediction blend (Sec. 5.3).
//
// State: binary32 planes, d = predictor dimension: beta[c][a] (plane c*d + a), the upper
// triangle of P row by row (d(d+1)/2 planes), z (3 planes). With d = 4 and the temporal
// feature this is the paper layout of the fast kernels.
//
// The update stages a 40 x 10 window of the previous state per 32 x 8 tile by TMA (three boxes: z, P,
// beta) and takes one pixel a thread; the blend takes two adjacent columns x two rows a thread
// from a TMA-filled 72 x 12 window (blend_mode 1, images smaller than the window and small images without
// G-buffer entries: one column a thread, plain loads).
#include <type_traits>

#include "wrls_internal.h"
#include "wrls_tiles.cuh"

namespace wrls {

template <int D, bool F>
struct ExtDim {
  static constexpr int kG = D - (F ? 4 : 1);  // G-buffer entries of p
  static constexpr int kNP = D * (D + 1) / 2;
  static constexpr int kBeta = 0;
  static constexpr int kP = 3 * D;
  static constexpr int kZ = 3 * D + kNP;
  static constexpr int kNS = kZ + 3;
  static constexpr int kG0 = F ? 4 : 1;  // index of the first G-buffer entry in p
};

// Index of P(a, b), a <= b, in the packed upper triangle (row by row).
__host__ __device__ constexpr int sym_index(int d, int a, int b) { return a * d - a * (a - 1) / 2 + (b - a); }

__device__ __forceinline__ bool finite3(const float v[3]) {
  return isfinite(v[0]) && isfinite(v[1]) && isfinite(v[2]);
}

constexpr int kExtTW = 32, kExtTH = 8;

// Shared memory of an update CTA: the staged window (kStageW x kStageH, as the paper-mode update's) of
// the previous state in three sections, each a TMA box of its own: z, P, beta.
template <int D, bool F>
struct ExtStage {
  using L = ExtDim<D, F>;
  static constexpr int pad(int planes) { return (planes * kStagePix + 31) / 32 * 32; }  // 128-byte multiple
  static constexpr int kOffZ = 0, kOffP = pad(3), kOffB = kOffP + pad(L::kNP);
  static constexpr int kFloats = kOffB + pad(3 * D);
  static constexpr int kSmemBytes = kFloats * 4 + 128;
  // CTAs per SM (256 threads): as many as the window leaves room for, within 64 registers a thread
  static constexpr int kMinCtas = kSmemBytes > 72 * 1024 ? 2 : kSmemBytes > 54 * 1024 ? 3 : 4;
};

// Taps from the staged window, or from the state copy where a tile's footprint exceeds it.
// at(section offset, first plane of the section, plane, tap offset).
struct ExtStaged {
  const float* w;
  __device__ __forceinline__ float at(int off, int first, int p, int o) const { return w[off + (p - first) * kStagePix + o]; }
};
struct ExtGlobal {
  const float* base;
  size_t ps;
  __device__ __forceinline__ float at(int, int, int p, int o) const { return ld_global(base + (size_t)p * ps + (uint32_t)o); }
};

struct ExtTaps {
  int o[4];    // offsets of the taps (x0, y0), (x1, y0), (x0, y1), (x1, y1)
  float w[4];  // bilinear weights
};

// N planes from plane p0 (a section of the state) at the reprojected position. TAPS = 4, 2 (fy = 0:
// the lower taps have weight exactly 0) or 1 (nearest pixel: the value itself).
template <int TAPS, int N, class Src>
__device__ __forceinline__ void ext_gather(const Src& s, const ExtTaps& t, int off, int p0, float* v) {
#pragma unroll
  for (int p = 0; p < N; ++p) {
    const float a = s.at(off, p0, p0 + p, t.o[0]);
    if (TAPS == 1) {
      v[p] = a;
    } else {
      const float b = s.at(off, p0, p0 + p, t.o[1]);
      if (TAPS == 2) v[p] = t.w[0] * a + t.w[1] * b;
      else v[p] = t.w[0] * a + t.w[1] * b + (t.w[2] * s.at(off, p0, p0 + p, t.o[2]) + t.w[3] * s.at(off, p0, p0 + p, t.o[3]));
    }
  }
}

// One pixel's update: Eq. 12 feature, weight, Eq. 14 / 11 / 8 / 9. The state is taken and stored part
// by part (z, P, one channel's model at a time), so that a thread holds P and little else, and
// ready(k) waits for section k of the staged window only when it is needed. TAPS = 0: restart.
template <int D, bool F, int TAPS, class Src, class Ready>
__device__ __forceinline__ void ext_update_pixel(const ExtParams& ep, const Src& src, const ExtTaps& t, const bool valid,
                                                 const float I[3], const bool missing, const float lo[3],
                                                 const float hi[3], const float* var,
                                                 const float* gbuf, const size_t npix, const size_t j,
                                                 float* __restrict__ dst, const size_t ps, const bool inside,
                                                 Ready&& ready) {
  using L = ExtDim<D, F>;
  using S = ExtStage<D, F>;
  const KParams& kp = ep.kp;
  float z[3];
  if (!ready(0)) return;
  if (TAPS > 0) ext_gather<TAPS ? TAPS : 1, 3>(src, t, S::kOffZ, L::kZ, z);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (TAPS > 0 && valid) {
      if (lo[0] <= hi[0]) z[c] = fminf(fmaxf(z[c], lo[c]), hi[c]);
      z[c] = missing ? z[c] : fmaf(kp.alpha, z[c], kp.one_m_alpha * I[c]);
    } else {
      z[c] = missing ? 0.0f : I[c];
    }
  }
  // predictor p = [1, z, g] of frame t; a non-finite G-buffer value enters as 0, weight 0
  float p[D];
  p[0] = 1.0f;
  if (F) {
    p[F ? 1 : 0] = z[0];
    p[F ? 2 : 0] = z[1];
    p[F ? 3 : 0] = z[2];
  }
  bool g_ok = true;
#pragma unroll
  for (int i = 0; i < L::kG; ++i) {
    const float g = inside ? ld_global(gbuf + (size_t)i * npix + j) : 0.0f;
    const bool f = isfinite(g);
    p[L::kG0 + i] = f ? g : 0.0f;
    g_ok = g_ok && f;
  }
  // weight: Eq. 13, RLS (w = 1) or the sample-variance weight
  float w;
  if (missing || !g_ok) {
    w = 0.0f;
  } else if (kp.weight_mode == 1) {
    w = 1.0f;
  } else {
    const float nI = sqrtf(I[0] * I[0] + I[1] * I[1] + I[2] * I[2]);
    const float nz = sqrtf(z[0] * z[0] + z[1] * z[1] + z[2] * z[2]);
    const float m = fminf(nI, nz) + kp.eps;
    if (kp.weight_mode == 2) {
      const float v = inside ? ld_global(var + j) : 0.0f;
      w = (isfinite(v) && v >= 0.0f) ? ex2_approx(-(v / (m * m)) * ep.wv_k) : 0.0f;
    } else {
      const float d0 = I[0] - z[0], d1 = I[1] - z[1], d2 = I[2] - z[2];
      w = ex2_approx(-((d0 * d0 + d1 * d1 + d2 * d2) / (m * m)) * kp.w_k);
    }
  }
  // k = P p, s = p^T P p; Eq. 14 gain q^w = (w / (lambda + w s)) k
  float P[L::kNP], k[D];
  if (!ready(1)) return;
  if (TAPS > 0) ext_gather<TAPS ? TAPS : 1, L::kNP>(src, t, S::kOffP, L::kP, P);
  if (TAPS == 0 || !valid) {
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
      for (int b = a; b < D; ++b) P[sym_index(D, a, b)] = a == b ? kp.p0_delta : 0.0f;
  }
#pragma unroll
  for (int a = 0; a < D; ++a) {
    float acc = 0.0f;
#pragma unroll
    for (int b = 0; b < D; ++b) acc = fmaf(P[a <= b ? sym_index(D, a, b) : sym_index(D, b, a)], p[b], acc);
    k[a] = acc;
  }
  float s = 0.0f;
#pragma unroll
  for (int a = 0; a < D; ++a) s = fmaf(p[a], k[a], s);
  const float gain = w / (kp.lambda + w * s);
  // Eq. 11: P <- (P - q^w p^T P) / lambda, p^T P = k^T
#pragma unroll
  for (int a = 0; a < D; ++a)
#pragma unroll
    for (int b = a; b < D; ++b) {
      const int e = sym_index(D, a, b);
      P[e] = (P[e] - gain * k[a] * k[b]) * kp.inv_lambda;
    }
  if (kp.p_trace_max > 0.0f) {
    float tr = 0.0f;
    bool bad = false;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const float v = P[sym_index(D, a, a)];
      tr += v;
      bad = bad || !(v > 0.0f);
    }
    if (bad || tr > kp.p_trace_max) {
#pragma unroll
      for (int a = 0; a < D; ++a)
#pragma unroll
        for (int b = a; b < D; ++b) P[sym_index(D, a, b)] = a == b ? kp.p0_delta : 0.0f;
    }
  }
  if (inside) {
#pragma unroll
    for (int q = 0; q < L::kNP; ++q) dst[(size_t)(L::kP + q) * ps] = P[q];
#pragma unroll
    for (int c = 0; c < 3; ++c) dst[(size_t)(L::kZ + c) * ps] = z[c];
  }
  if (!ready(2)) return;
  const bool use = !(missing || !g_ok);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float beta[D];
    if (TAPS > 0) {
      // plane indices run through the whole beta section
#pragma unroll
      for (int a = 0; a < D; ++a) {
        float v[1];
        ext_gather<TAPS ? TAPS : 1, 1>(src, t, S::kOffB + (c * D + a) * kStagePix, L::kBeta + c * D + a, v);
        beta[a] = v[0];
      }
    }
    if (TAPS == 0 || !valid) {
#pragma unroll
      for (int a = 0; a < D; ++a) beta[a] = 0.0f;
      if (kp.init_mode == 1) {
        if (F) beta[F ? c + 1 : 0] = 1.0f;
        else beta[0] = z[c];
      }
    }
    float pred = 0.0f;
#pragma unroll
    for (int a = 0; a < D; ++a) pred = fmaf(p[a], beta[a], pred);
    const float ge = gain * (use ? I[c] - pred : 0.0f);  // Eq. 8, Eq. 9
    if (inside) {
#pragma unroll
      for (int a = 0; a < D; ++a) dst[(size_t)(L::kBeta + c * D + a) * ps] = fmaf(ge, k[a], beta[a]);
    }
  }
}

// Update of a 32 x 8 tile, one pixel a thread. As in the paper-mode update, the footprint of the
// tile's taps is reduced over the CTA and, where it fits the window, every state plane of it is
// copied to shared memory by TMA (three boxes in the order the update needs them: z, P, beta).
// Cached loads of the taps (the form before) were bound by their latency at 2 CTAs of 128
// registers and thrashed L1 under general motion. Measured on a 1080p frame, orbit / pan, us: d = 8
// 469 / 284 -> 216 / 210 (540 algorithmic bytes a pixel: 165 us at the copy rate), d = 5 180 -> 112,
// variance weight d = 4 136 -> 96, nearest pixel d = 4 91 -> 87. More CTAs at fewer registers without
// the window: d = 8 304 (2 CTAs) to 351 (4).
template <int D, bool F>
__global__ void __launch_bounds__(kExtTW * kExtTH, ExtStage<D, F>::kMinCtas)
    k_update_ext(const ExtParams ep, const int W, const int H, const int reset, const int stage_ok,
                 const float* prev, float* __restrict__ next, const int pitch, const size_t ps,
                 const __grid_constant__ ExtStageMaps maps, const float* rad,
                 const float* mot, const float* var, const float* gbuf, int* err) {
  using L = ExtDim<D, F>;
  using S = ExtStage<D, F>;
  const KParams& kp = ep.kp;
  extern __shared__ unsigned char dsmem[];
  float* stage = reinterpret_cast<float*>(align128(dsmem));
  __shared__ int4 red[kExtTH];
  __shared__ alignas(8) uint64_t bar[3];
  if (threadIdx.x < 3) mbar_init(&bar[threadIdx.x], 1);
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int x = blockIdx.x * kExtTW + lane, y = blockIdx.y * kExtTH + warp;
  const bool inside = x < W && y < H;
  const size_t npix = (size_t)W * H, j = (size_t)y * W + x;

  // reprojection q = j + v_j (Table 2), binary32; NaN motion fails every comparison
  float qx = 0.0f, qy = 0.0f;
  bool valid = false;
  if (inside) {
    qx = (float)x + ld_global(mot + j);
    qy = (float)y + ld_global(mot + npix + j);
    valid = !reset && qx >= 0.0f && qx <= (float)(W - 1) && qy >= 0.0f && qy <= (float)(H - 1);
  }
  const bool nearest = ep.reproj_filter == 1;
  // (nearest pixel: the tap is floor(q + 0.5), in binary32)
  const float rx = nearest ? floorf(qx + 0.5f) : floorf(qx), ry = nearest ? floorf(qy + 0.5f) : floorf(qy);
  const int x0 = (int)rx, y0 = (int)ry;
  const bool any = __any_sync(0xffffffffu, valid);
  // a warp whose valid pixels all have an integral vertical motion component reads the upper taps only
  const bool fy0 = __all_sync(0xffffffffu, !valid || qy == ry);
  int lo_x = __reduce_min_sync(0xffffffffu, valid ? x0 : 0x7fffffff), hi_x = __reduce_max_sync(0xffffffffu, valid ? x0 : -1);
  int lo_y = __reduce_min_sync(0xffffffffu, valid ? y0 : 0x7fffffff), hi_y = __reduce_max_sync(0xffffffffu, valid ? y0 : -1);
  if (lane == 0) red[warp] = make_int4(lo_x, hi_x, lo_y, hi_y);
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kExtTH; ++k) {
    const int4 r = red[k];
    lo_x = min(lo_x, r.x); hi_x = max(hi_x, r.y);
    lo_y = min(lo_y, r.z); hi_y = max(hi_y, r.w);
  }
  pdl_next(kp);
  const int more = nearest ? 0 : 1;
  const int X0 = lo_x & ~3, Y0 = lo_y;  // TMA box origin: 16-byte aligned column
  const bool fits = stage_ok && hi_x >= 0 && min(hi_x + more, W - 1) - X0 < kStageW && min(hi_y + more, H - 1) - Y0 < kStageH;
  if (fits && threadIdx.x == 0) {
    mbar_expect_tx(&bar[0], 3u * kStagePix * 4u);
    tma_load_3d(stage + S::kOffZ, &maps.z, X0, Y0, L::kZ, &bar[0]);
    mbar_expect_tx(&bar[1], (uint32_t)L::kNP * kStagePix * 4u);
    tma_load_3d(stage + S::kOffP, &maps.p, X0, Y0, L::kP, &bar[1]);
    mbar_expect_tx(&bar[2], 3u * D * kStagePix * 4u);
    if (!kp.debug_withhold_copy) tma_load_3d(stage + S::kOffB, &maps.beta, X0, Y0, L::kBeta, &bar[2]);
  }
  float I[3] = {0.0f, 0.0f, 0.0f}, lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  bool missing = true;
  if (inside) {
#pragma unroll
    for (int c = 0; c < 3; ++c) I[c] = ld_global(rad + c * npix + j);
    missing = !finite3(I);
    if (kp.clamp_mode == 0) {
      // Psi = clamp to the 3x3 min/max of the finite samples: a neighbour outside the image is
      // replaced by the nearest one inside, which is in the window as well; a missing sample
      // enters as NaN, which fminf / fmaxf skip
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx) {
          const size_t jj = (size_t)min(max(y + dy, 0), H - 1) * W + min(max(x + dx, 0), W - 1);
          const float In[3] = {ld_global(rad + jj), ld_global(rad + npix + jj), ld_global(rad + 2 * npix + jj)};
          const bool fin = finite3(In);
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const float v = fin ? In[c] : __int_as_float(0x7fc00000);
            lo[c] = fminf(lo[c], v);
            hi[c] = fmaxf(hi[c], v);
          }
        }
    }
  }
  ExtTaps t;
  {
    const float fx = qx - rx, fy = qy - ry;
    t.w[0] = (1.0f - fx) * (1.0f - fy);
    t.w[1] = fx * (1.0f - fy);
    t.w[2] = (1.0f - fx) * fy;
    t.w[3] = fx * fy;
    // offsets in the window or in a plane of the copy; a restarted pixel reads offset 0
    const int row = fits ? kStageW : pitch;
    const int b = valid ? (y0 - (fits ? Y0 : 0)) * row + x0 - (fits ? X0 : 0) : 0;
    const int dx = valid && x0 < W - 1 ? 1 : 0, dy = valid && y0 < H - 1 ? row : 0;
    t.o[0] = b;
    t.o[1] = b + dx;
    t.o[2] = b + dy;
    t.o[3] = b + dy + dx;
  }
  float* dst = next + (size_t)y * pitch + x;
  auto pixel = [&](auto taps, const auto& src, auto&& ready) {
    ext_update_pixel<D, F, decltype(taps)::value>(ep, src, t, valid, I, missing, lo, hi, var, gbuf, npix, j, dst, ps, inside,
                                                  ready);
  };
  using T0 = std::integral_constant<int, 0>;
  using T1 = std::integral_constant<int, 1>;
  using T2 = std::integral_constant<int, 2>;
  using T4 = std::integral_constant<int, 4>;
  auto landed = [&](int k) {
    if (mbar_wait_bounded(&bar[k], 0)) return true;
    atomicExch(err, (int)WRLS_ERR_TIMEOUT);
    const long long t0 = clock64();
    for (int m = 0; m < 3; ++m) mbar_wait_until(&bar[m], 0, t0);  // the copies may still be in flight
    return false;
  };
  auto at_once = [](int) { return true; };
  if (!any) {
    pixel(T0{}, ExtGlobal{prev, ps}, at_once);
    if (fits)
      for (int m = 0; m < 3; ++m)
        if (!landed(m)) return;  // leave no copy in flight behind
  } else if (fits) {
    const ExtStaged src{stage};
    if (nearest) pixel(T1{}, src, landed);
    else if (fy0) pixel(T2{}, src, landed);
    else pixel(T4{}, src, landed);
  } else {
    const ExtGlobal src{prev, ps};
    if (nearest) pixel(T1{}, src, at_once);
    else pixel(T4{}, src, at_once);
  }
}

constexpr int kExtSW = kExtTW + 4, kExtSH = kExtTH + 4, kExtSP = kExtSW * kExtSH;
constexpr float kExtFarZ = 1e18f;  // feature of an out-of-image neighbour: its blend weight is 0

// 5x5 blend: out_i = sum_k b_ik (p_i beta_k) / sum_k b_ik (blend_mode 1: p_k beta_k), with
// b_ik = 2^(spatial_ik - |z_i - z_k|^2 max(r_i, r_k)), r = log2(e) / (h_s^2 (|z| + eps)^2):
// the Eq. 13 distance of the two features, min(|z_i|, |z_k|) taken through max(r_i, r_k).
// A CTA of 32 x 4 threads blends a 32 x 8 tile; each thread produces two vertically adjacent
// outputs, so that every neighbour read from shared memory serves both (6 x 5 reads for two
// outputs instead of 2 x 25).
constexpr int kExtBlendRows = 2;

template <int D, bool F>
__device__ __forceinline__ void ext_predictor_g(const float* gbuf, size_t npix, size_t j, float p[D]) {
  using L = ExtDim<D, F>;
#pragma unroll
  for (int i = 0; i < L::kG; ++i) {
    const float g = ld_global(gbuf + (size_t)i * npix + j);
    p[L::kG0 + i] = isfinite(g) ? g : 0.0f;
  }
}

template <int D, bool F>
__global__ void __launch_bounds__(kExtTW * kExtTH / kExtBlendRows)
    k_blend_ext(const ExtParams ep, const int W, const int H, const float* cur, const int pitch,
                const size_t ps, const float* gbuf, float* __restrict__ out) {
  using L = ExtDim<D, F>;
  constexpr int NPL = 3 * D + 4;  // beta planes, z (3), range factor
  constexpr int NT = kExtTW * kExtTH / kExtBlendRows;
  static_assert(NPL * kExtSP * 4 <= 48 * 1024, "blend window exceeds static shared memory");
  __shared__ float sm[NPL * kExtSP];
  const KParams& kp = ep.kp;
  const int bx0 = blockIdx.x * kExtTW, by0 = blockIdx.y * kExtTH;
  const int tid = threadIdx.y * kExtTW + threadIdx.x;
  pdl_wait();
  for (int e = tid; e < kExtSP; e += NT) {
    const int gx = bx0 - 2 + e % kExtSW, gy = by0 - 2 + e / kExtSW;
    if (gx >= 0 && gx < W && gy >= 0 && gy < H) {
      const float* src = cur + (size_t)gy * pitch + gx;
#pragma unroll
      for (int a = 0; a < 3 * D; ++a) sm[a * kExtSP + e] = ld_global(src + (L::kBeta + a) * ps);
      const float z0 = ld_global(src + (L::kZ + 0) * ps), z1 = ld_global(src + (L::kZ + 1) * ps),
                  z2 = ld_global(src + (L::kZ + 2) * ps);
      sm[(3 * D + 0) * kExtSP + e] = z0;
      sm[(3 * D + 1) * kExtSP + e] = z1;
      sm[(3 * D + 2) * kExtSP + e] = z2;
      const float nz = sqrtf(z0 * z0 + z1 * z1 + z2 * z2) + kp.eps;
      sm[(3 * D + 3) * kExtSP + e] = kp.range_k / (nz * nz);
    } else {
#pragma unroll
      for (int a = 0; a < 3 * D; ++a) sm[a * kExtSP + e] = 0.0f;
      sm[(3 * D + 0) * kExtSP + e] = kExtFarZ;
      sm[(3 * D + 1) * kExtSP + e] = kExtFarZ;
      sm[(3 * D + 2) * kExtSP + e] = kExtFarZ;
      sm[(3 * D + 3) * kExtSP + e] = 0.0f;
    }
  }
  __syncthreads();
  pdl_next(kp);
  const int x = bx0 + threadIdx.x;
  const int ty0 = threadIdx.y * kExtBlendRows;  // first of the thread's two rows in the tile
  const size_t npix = (size_t)W * H;
  // the two outputs' features, range factors and predictors
  float zi[kExtBlendRows][3], ri[kExtBlendRows], pi[kExtBlendRows][D];
#pragma unroll
  for (int r = 0; r < kExtBlendRows; ++r) {
    const int ei = (ty0 + r + 2) * kExtSW + threadIdx.x + 2;
    zi[r][0] = sm[(3 * D + 0) * kExtSP + ei];
    zi[r][1] = sm[(3 * D + 1) * kExtSP + ei];
    zi[r][2] = sm[(3 * D + 2) * kExtSP + ei];
    ri[r] = sm[(3 * D + 3) * kExtSP + ei];
    pi[r][0] = 1.0f;
    if (F) {
      pi[r][1] = zi[r][0];
      pi[r][2] = zi[r][1];
      pi[r][3] = zi[r][2];
    }
    const int y = by0 + ty0 + r;
#pragma unroll
    for (int i = 0; i < L::kG; ++i) pi[r][L::kG0 + i] = 0.0f;
    if (x < W && y < H) ext_predictor_g<D, F>(gbuf, npix, (size_t)y * W + x, pi[r]);
  }
  float num[kExtBlendRows][3] = {}, den[kExtBlendRows] = {};
#pragma unroll
  for (int wy = 0; wy < 4 + kExtBlendRows; ++wy)  // window rows ty0 .. ty0 + 5 (relative)
#pragma unroll
    for (int dx = 0; dx < 5; ++dx) {
      const int e = (ty0 + wy) * kExtSW + threadIdx.x + dx;
      const float zk0 = sm[(3 * D + 0) * kExtSP + e], zk1 = sm[(3 * D + 1) * kExtSP + e],
                  zk2 = sm[(3 * D + 2) * kExtSP + e];
      const float rk = sm[(3 * D + 3) * kExtSP + e];
      float bk[3 * D];
#pragma unroll
      for (int a = 0; a < 3 * D; ++a) bk[a] = sm[a * kExtSP + e];
      float own[3] = {0.0f, 0.0f, 0.0f};  // blend_mode 1: neighbour k's own prediction
      if (kp.blend_mode != 0) {
        const int xx = x + dx - 2, yy = by0 + ty0 + wy - 2;
        const bool in = xx >= 0 && xx < W && yy >= 0 && yy < H;
        float pk[D];
        pk[0] = 1.0f;
        if (F) {
          pk[1] = in ? zk0 : 0.0f;
          pk[2] = in ? zk1 : 0.0f;
          pk[3] = in ? zk2 : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < L::kG; ++i) pk[L::kG0 + i] = 0.0f;
        if (in) ext_predictor_g<D, F>(gbuf, npix, (size_t)yy * W + xx, pk);
#pragma unroll
        for (int a = 0; a < D; ++a) {
          own[0] = fmaf(pk[a], bk[0 * D + a], own[0]);
          own[1] = fmaf(pk[a], bk[1 * D + a], own[1]);
          own[2] = fmaf(pk[a], bk[2 * D + a], own[2]);
        }
      }
#pragma unroll
      for (int r = 0; r < kExtBlendRows; ++r) {
        const int dy = wy - r;  // this neighbour's row offset (0..4) for output r
        if (dy < 0 || dy > 4) continue;  // resolved at compile time
        const float a0 = zi[r][0] - zk0, a1 = zi[r][1] - zk1, a2 = zi[r][2] - zk2;
        const float b = ex2_approx(blend_exponent(kp.spatial[dy * 5 + dx], a0, a1, a2, fmaxf(ri[r], rk)));
        float p0 = own[0], p1 = own[1], p2 = own[2];
        if (kp.blend_mode == 0) {
          p0 = p1 = p2 = 0.0f;
#pragma unroll
          for (int a = 0; a < D; ++a) {
            p0 = fmaf(pi[r][a], bk[0 * D + a], p0);
            p1 = fmaf(pi[r][a], bk[1 * D + a], p1);
            p2 = fmaf(pi[r][a], bk[2 * D + a], p2);
          }
        }
        num[r][0] = fmaf(b, p0, num[r][0]);
        num[r][1] = fmaf(b, p1, num[r][1]);
        num[r][2] = fmaf(b, p2, num[r][2]);
        den[r] += b;
      }
    }
#pragma unroll
  for (int r = 0; r < kExtBlendRows; ++r) {
    const int y = by0 + ty0 + r;
    if (x >= W || y >= H) continue;
    const size_t j = (size_t)y * W + x;
    const float inv = 1.0f / den[r];
    out[j] = num[r][0] * inv;
    out[npix + j] = num[r][1] * inv;
    out[2 * npix + j] = num[r][2] * inv;
  }
}

// blend_mode 0 with packed pairs: a CTA of 32 x 4 threads blends a 64 x 8 tile, each thread two
// adjacent columns x two rows, from a 72 x 12 window (origin 4 columns left, 2 rows above the
// tile) of the beta and z planes filled by TMA. As in the paper-mode blend, the neighbours of
// the two columns at an even dx are the halves of one aligned 64-bit load, so those 15 of 25
// offsets take one packed instruction for both columns, and a window value is loaded once for
// up to four outputs. The z planes land on their own mbarrier, so that the range factors are
// computed while the beta planes are in flight. Outputs equal k_blend_ext's bit for bit.
// What bounds the one-column kernel is its shared loads, 28 x 30 for two outputs at d = 8 (420 an
// output against 126 here). Measured on a 1080p frame, us: d = 8 195.6 -> 115.0, d = 5 161.6 -> 75.9,
// d = 4 110.2 -> 63.7, d = 3 without the feature 86.8 -> 53.8. blend_mode 1 needs the neighbours'
// G-buffer values beside their models and keeps the one-column kernel.
constexpr int kExt2W = 64, kExt2H = 8, kExt2SH = kExt2H + 4, kExt2Plane = kBlendBoxW2 * kExt2SH;
template <int D>
constexpr int ext2_smem_bytes() { return (3 * D + 4) * kExt2Plane * 4 + 128; }

template <int D, bool F>
__global__ void __launch_bounds__(128)
    k_blend_ext2(const ExtParams ep, const int W, const int H, const __grid_constant__ ExtMaps maps,
                 const float* gbuf, float* __restrict__ out, int* err) {
  using L = ExtDim<D, F>;
  constexpr int P = kExt2Plane, SW = kBlendBoxW2, Z = 3 * D;  // window planes: beta, z (3), range factor
  extern __shared__ unsigned char dsmem[];
  float* w = reinterpret_cast<float*>(align128(dsmem));
  __shared__ alignas(8) uint64_t zbar, bbar;
  const KParams& kp = ep.kp;
  const int bx0 = blockIdx.x * kExt2W, by0 = blockIdx.y * kExt2H;
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  pdl_wait();
  if (threadIdx.x == 0) {
    mbar_init(&zbar, 1);
    mbar_init(&bbar, 1);
    mbar_expect_tx(&zbar, 3u * P * 4u);
    tma_load_3d(w + Z * P, &maps.z, bx0 - 4, by0 - 2, L::kZ, &zbar);
    mbar_expect_tx(&bbar, 3u * D * P * 4u);
    if (!kp.debug_withhold_copy) tma_load_3d(w, &maps.beta, bx0 - 4, by0 - 2, 0, &bbar);
  }
  // G-buffer entries of the thread's predictors (.x: column 2 tx, .y: column 2 tx + 1)
  const size_t npix = (size_t)W * H;
  const int x = bx0 + 2 * tx, y0 = by0 + 2 * ty;
  float2 pi[2][D];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int a = 0; a < L::kG; ++a) {
      float2 g = make_float2(0.0f, 0.0f);
      const float* s = gbuf + (size_t)a * npix + (size_t)(y0 + i) * W + x;
      if (y0 + i < H && x < W) g.x = ld_global(s);
      if (y0 + i < H && x + 1 < W) g.y = ld_global(s + 1);
      pi[i][L::kG0 + a] = make_float2(isfinite(g.x) ? g.x : 0.0f, isfinite(g.y) ? g.y : 0.0f);
    }
  __syncthreads();  // the barriers are initialised
  bool ok = mbar_wait_bounded(&zbar, 0);
  const bool inner = bx0 >= 4 && bx0 + 68 <= W && by0 >= 2 && by0 + 10 <= H;
  if (!inner) ok = ok && mbar_wait_bounded(&bbar, 0);  // far records overwrite the beta planes too
  if (ok)
    for (int i = threadIdx.x; i < P; i += 128) {
      const int gx = bx0 - 4 + i % SW, gy = by0 - 2 + i / SW;
      if (inner || (gx >= 0 && gx < W && gy >= 0 && gy < H)) {
        const float z0 = w[Z * P + i], z1 = w[(Z + 1) * P + i], z2 = w[(Z + 2) * P + i];
        const float nz = sqrtf(z0 * z0 + z1 * z1 + z2 * z2) + kp.eps;
        w[(Z + 3) * P + i] = kp.range_k / (nz * nz);
      } else {
#pragma unroll
        for (int p = 0; p < 3 * D; ++p) w[p * P + i] = 0.0f;
        w[Z * P + i] = w[(Z + 1) * P + i] = w[(Z + 2) * P + i] = kExtFarZ;
        w[(Z + 3) * P + i] = 0.0f;
      }
    }
  ok = ok && mbar_wait_bounded(&bbar, 0);
  if (__syncthreads_or(!ok)) {
    if (threadIdx.x == 0) atomicExch(err, (int)WRLS_ERR_TIMEOUT);
    const long long t0 = clock64();
    mbar_wait_until(&zbar, 0, t0);  // the copies may still be in flight
    mbar_wait_until(&bbar, 0, t0);
    return;
  }
  pdl_next(kp);
  float2 zi[2][3], ri[2], den[2], acc[2][3];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int e = (2 * ty + i + 2) * SW + 2 * tx + 4;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      zi[i][c] = *reinterpret_cast<const float2*>(w + (Z + c) * P + e);
      acc[i][c] = make_float2(0.0f, 0.0f);
      if (F) pi[i][F ? c + 1 : 0] = zi[i][c];
    }
    ri[i] = *reinterpret_cast<const float2*>(w + (Z + 3) * P + e);
    den[i] = make_float2(0.0f, 0.0f);
  }
  // a neighbour's weight of one output: half h of output row i against half k of the pair
  auto half = [](float2 v, int h) { return h ? v.y : v.x; };
#pragma unroll 1
  for (int kr = 0; kr < 6; ++kr) {
    const float* row = w + (2 * ty + kr) * SW + 2 * tx + 2;
#pragma unroll
    for (int pair = 0; pair < 3; ++pair) {
      float2 b[3 * D], zk[3];
#pragma unroll
      for (int p = 0; p < 3 * D; ++p) b[p] = *reinterpret_cast<const float2*>(row + p * P + 2 * pair);
#pragma unroll
      for (int c = 0; c < 3; ++c) zk[c] = *reinterpret_cast<const float2*>(row + (Z + c) * P + 2 * pair);
      const float2 rk = *reinterpret_cast<const float2*>(row + (Z + 3) * P + 2 * pair);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int dy = kr - 2 - i;
        if (dy < -2 || dy > 2) continue;
        const float* sp = kp.spatial + (dy + 2) * 5 + 2;
        auto single = [&](int h, int k, int dx) {
          const float e0 = half(zi[i][0], h) - half(zk[0], k), e1 = half(zi[i][1], h) - half(zk[1], k),
                      e2 = half(zi[i][2], h) - half(zk[2], k);
          const float wt = ex2_approx(blend_exponent(sp[dx], e0, e1, e2, fmaxf(half(ri[i], h), half(rk, k))));
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            float v = half(b[c * D], k);
#pragma unroll
            for (int a = 1; a < D; ++a) v = fmaf(half(pi[i][a], h), half(b[c * D + a], k), v);
            if (h) acc[i][c].y = fmaf(wt, v, acc[i][c].y);
            else acc[i][c].x = fmaf(wt, v, acc[i][c].x);
          }
          if (h) den[i].y += wt;
          else den[i].x += wt;
        };
        if (pair >= 1) single(1, 0, 2 * pair - 3);
        {
          const float2 e0 = f2sub(zi[i][0], zk[0]), e1 = f2sub(zi[i][1], zk[1]), e2 = f2sub(zi[i][2], zk[2]);
          const float s = sp[2 * pair - 2];
          const float2 t = blend_exponent2(make_float2(s, s), e0, e1, e2,
                                           make_float2(-fmaxf(ri[i].x, rk.x), -fmaxf(ri[i].y, rk.y)));
          const float2 wt = make_float2(ex2_approx(t.x), ex2_approx(t.y));
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            float2 v = b[c * D];
#pragma unroll
            for (int a = 1; a < D; ++a) v = f2fma(pi[i][a], b[c * D + a], v);
            acc[i][c] = f2fma(wt, v, acc[i][c]);
          }
          den[i] = f2add(den[i], wt);
        }
        if (pair <= 1) single(0, 1, 2 * pair - 1);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    if (y0 + i >= H) break;
    const float2 inv = make_float2(1.0f / den[i].x, 1.0f / den[i].y);
    float* d = out + (size_t)(y0 + i) * W + x;
#pragma unroll
    for (int c = 0; c < 3; ++c, d += npix) {
      if (x < W) d[0] = acc[i][c].x * inv.x;
      if (x + 1 < W) d[1] = acc[i][c].y * inv.y;
    }
  }
}

__global__ void k_read_state_ext(const int W, const int H, const float* __restrict__ cur, const int pitch,
                                 const size_t ps, const int nplanes, float* __restrict__ dst) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (x >= W || y >= H) return;
  const size_t npix = (size_t)W * H, j = (size_t)y * W + x;
  const float* src = cur + (size_t)y * pitch + x;
  for (int p = 0; p < nplanes; ++p) dst[p * npix + j] = src[p * ps];
}

__global__ void k_write_state_ext(const int W, const int H, float* __restrict__ cur, const int pitch,
                                  const size_t ps, const int nplanes, const float* __restrict__ src) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (x >= W || y >= H) return;
  const size_t npix = (size_t)W * H, j = (size_t)y * W + x;
  float* dst = cur + (size_t)y * pitch + x;
  for (int p = 0; p < nplanes; ++p) dst[p * ps] = src[p * npix + j];
}

template <int D, bool F>
static cudaError_t launch_ext_t(const ExtParams& ep, const StateDesc& prev, const StateDesc& next, bool reset,
                                const float* rad, const float* mot, const float* var, const float* gbuf, int* err,
                                cudaStream_t cs) {
  constexpr int bytes = ExtStage<D, F>::kSmemBytes;
  static KernelSetup setup;  // per instantiation
  const cudaError_t e = setup(k_update_ext<D, F>, kExtTW * kExtTH, bytes);
  if (e != cudaSuccess) return e;
  const dim3 grid((prev.W + kExtTW - 1) / kExtTW, (prev.H + kExtTH - 1) / kExtTH);
  return launch_kernel(k_update_ext<D, F>, grid, kExtTW * kExtTH, bytes, cs, hint_pdl(ep.kp), ep, prev.W, prev.H, reset ? 1 : 0,
                       prev.stage_ok ? 1 : 0, (const float*)prev.base, (float*)next.base, prev.pitch, prev.plane_stride,
                       prev.esmaps, rad, mot, var, gbuf, err);
}

template <int D, bool F>
static cudaError_t launch_ext_blend_t(const ExtParams& ep, const StateDesc& cur, const float* gbuf, float* out,
                                      int* err, cudaStream_t cs) {
  // Without G-buffer entries (d = 4 or 1) the one-column blend is the faster one on images whose CTAs
  // leave SMs idle: half the outputs a thread, twice the CTAs. Nearest pixel, us a frame through per-frame
  // calls / sequence, two columns -> one: 128x128 9.7 / 9.3 -> 7.3 / 7.8, 200x150 9.7 / 11.6 -> 8.9 / 10.9, 320x240 (300
  // tiles) 10.9 / 12.2 -> 10.1 / 12.8; 361x363 (552) 13.7 / 14.1 -> 14.7 / 15.3. With G-buffer entries, whose
  // window and predictors two columns share, it is slower at every size (128x128, d = 5 11.1 -> 12.8).
  const bool few = ExtDim<D, F>::kG == 0 && ((cur.W + kExtTW - 1) / kExtTW) * ((cur.H + kExtTH - 1) / kExtTH) <= 2 * sm_count();
  if (ep.kp.blend_mode == 0 && cur.ext_tma_ok && !few) {
    constexpr int bytes = ext2_smem_bytes<D>();
    static KernelSetup setup;  // per instantiation
    const cudaError_t e = setup(k_blend_ext2<D, F>, 128, bytes);
    if (e != cudaSuccess) return e;
    const dim3 grid((cur.W + kExt2W - 1) / kExt2W, (cur.H + kExt2H - 1) / kExt2H);
    return launch_kernel(k_blend_ext2<D, F>, grid, 128, bytes, cs, hint_pdl(ep.kp), ep, cur.W, cur.H, cur.emaps, gbuf, out, err);
  }
  const dim3 grid((cur.W + kExtTW - 1) / kExtTW, (cur.H + kExtTH - 1) / kExtTH);
  return launch_kernel(k_blend_ext<D, F>, grid, dim3(kExtTW, kExtTH / kExtBlendRows), 0, cs, hint_pdl(ep.kp), ep, cur.W, cur.H,
                       (const float*)cur.base, cur.pitch, cur.plane_stride, gbuf, out);
}

int ext_dim(const wrls_params& p) { return (p.feature_mode == 0 ? 4 : 1) + p.n_gbuf; }

int ext_planes(int d) { return 3 * d + d * (d + 1) / 2 + 3; }

#define WRLS_EXT_DISPATCH(FN, ...)                                 \
  switch ((ep.kp.feature_mode == 0 ? 0 : 16) + d) {                \
    case 4: return FN<4, true>(__VA_ARGS__);                       \
    case 5: return FN<5, true>(__VA_ARGS__);                       \
    case 6: return FN<6, true>(__VA_ARGS__);                       \
    case 7: return FN<7, true>(__VA_ARGS__);                       \
    case 8: return FN<8, true>(__VA_ARGS__);                       \
    case 17: return FN<1, false>(__VA_ARGS__);                     \
    case 18: return FN<2, false>(__VA_ARGS__);                     \
    case 19: return FN<3, false>(__VA_ARGS__);                     \
    case 20: return FN<4, false>(__VA_ARGS__);                     \
    case 21: return FN<5, false>(__VA_ARGS__);                     \
    default: return cudaErrorInvalidValue;                         \
  }

cudaError_t launch_ext_update(const ExtParams& ep, int d, const StateDesc& prev, const StateDesc& next, bool reset,
                              const float* rad, const float* mot, const float* var, const float* gbuf, int* err,
                              cudaStream_t cs) {
  WRLS_EXT_DISPATCH(launch_ext_t, ep, prev, next, reset, rad, mot, var, gbuf, err, cs)
}

cudaError_t launch_ext_blend(const ExtParams& ep, int d, const StateDesc& cur, const float* gbuf, float* out, int* err,
                             cudaStream_t cs) {
  WRLS_EXT_DISPATCH(launch_ext_blend_t, ep, cur, gbuf, out, err, cs)
}

cudaError_t launch_write_state_ext(const StateDesc& cur, int nplanes, const float* src, cudaStream_t cs) {
  const dim3 grid((cur.W + 127) / 128, cur.H);
  k_write_state_ext<<<grid, 128, 0, cs>>>(cur.W, cur.H, (float*)cur.base, cur.pitch, cur.plane_stride, nplanes, src);
  return cudaGetLastError();
}

cudaError_t launch_read_state_ext(const StateDesc& cur, int nplanes, float* dst, cudaStream_t cs) {
  const dim3 grid((cur.W + 127) / 128, cur.H);
  k_read_state_ext<<<grid, 128, 0, cs>>>(cur.W, cur.H, (const float*)cur.base, cur.pitch, cur.plane_stride, nplanes,
                                         dst);
  return cudaGetLastError();
}

}  // namespace wrls
