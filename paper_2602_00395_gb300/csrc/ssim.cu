// gs_dssim_cotangents: the image-space vectors of the pixel loss
// (1 - lambda) L1 + lambda D-SSIM of Eq. pixel_loss (Sec. 3.2, D-SSIM = 1 - SSIM,
// m = 6 H W per view) for the reverse pass (GS_LOSS_COTANGENT):
//   stream 0   dL/dC = ((1 - lambda) sign(r) - lambda sum_p dS_p/dC) / (2m)
//   stream k   (1 - lambda)/(4 max(|r|, floor))/m . d_k + A[lambda/(4 max(1 - S, floor))/m . dS[d_k]]
// with d_k = J z_k the image tangents, dS[d] the directional derivative of the
// SSIM map and A its adjoint.  SSIM of one channel uses the 11 x 11 Gaussian
// window of standard deviation 1.5 (zeros outside the image), C1 = 0.01^2,
// C2 = 0.03^2.  As a function of the window means mx = G*x, Ex2 = G*(x^2),
// Exy = G*(x y) of the rendered channel x (the target's are constants):
//   A[a] = G*(a dS/dmx) + 2 x G*(a dS/dEx2) + y G*(a dS/dExy)   (G is symmetric)
//   dS[d] = dS/dmx G*d + dS/dEx2 G*(2 x d) + dS/dExy G*(y d)
//
// Two kernels: the first filters the image, the target and the probes' tangents
// and writes the SSIM map's partials and each probe's weighted derivative; the
// second filters those and writes the cotangents of all streams.  Both work on
// 32 x 32 output tiles of one (view, channel) plane: the inputs of the tile and
// its 5-pixel halo go to shared memory by asynchronous copies (zero outside the
// image), up to three pairs of products at a time are filtered horizontally into
// shared memory, then vertically into registers, and an epilogue combines the
// filtered values at each pixel.  Packing the products that are filtered alike
// (image and target, the two probes) and running two kernels instead of four
// (S is no longer stored, the partials are read once) took 8 views of 1080p with
// two probes from 3.31 to 2.17 ms: issue slots 61-66 %, shared memory 70 % of
// its bandwidth.  Three blocks of 256 threads run per SM; with 2 x 4 pixels of
// row pairs per thread and all products of a tile filtered at once, two blocks of
// 192 fitted and the loads' latency showed (3.47 ms).
#include <cmath>

#include "common.cuh"

namespace gs {
namespace {

constexpr int kR = 5, kTile = 32, kIn = kTile + 2 * kR;  // 42
constexpr int kSsimThreads = 256;
constexpr float kC1 = 1e-4f, kC2 = 9e-4f;

struct Plane {
  int W, H, planes;  // planes = views x 3
};
struct Window {  // the symmetric window: w[|d|] for offsets d = -5..5
  float w[kR + 1];
};

// Shared memory.  Two quantities that are filtered alike are held as pairs, so
// that a packed instruction filters both.  Rows are an odd number of pairs long:
// the horizontal pass gives consecutive lanes consecutive rows.
constexpr int kInRow = 43, kInPlane = kIn * kInRow;    // staged inputs, [kIn][kInRow]
constexpr int kHRow = 33, kHPlane = kIn * kHRow;       // horizontal sums, [kIn][kHRow]
constexpr int kGroup = 3;                              // pairs filtered at a time

// Starts the copies of a plane's tile (with halo) into dst[(ty * kInRow + tx) * stride].
__device__ __forceinline__ void load_tile(const float* __restrict__ src, int W, int H, int x0, int y0, float* dst,
                                          int stride) {
#pragma unroll
  for (int n = 0; n < (kIn * kIn + kSsimThreads - 1) / kSsimThreads; ++n) {
    const int q = n * kSsimThreads + (int)threadIdx.x;
    if (q >= kIn * kIn) break;
    const int ty = q / kIn, tx = q - ty * kIn;
    const int gx = x0 - kR + tx, gy = y0 - kR + ty;
    const bool in = gx >= 0 && gx < W && gy >= 0 && gy < H;
    cp_async4_or_zero(dst + (ty * kInRow + tx) * stride, in ? src + (size_t)gy * W + gx : src, in);
  }
}

// Horizontal window sums of NPAIR pairs of products (prod(at, p) of the inputs at
// index `at`) for all kIn rows and kTile columns.  A thread covers kCols columns
// of one row and forms each product once; every sum adds its 11 terms in window
// order.
constexpr int kCols = 4, kRows = 4;
template <int NPAIR, class Prod>
__device__ __forceinline__ void filter_rows(f32x2* s_h, const Window& win, Prod prod) {
  for (int q = threadIdx.x; q < kIn * (kTile / kCols); q += kSsimThreads) {
    const int cg = q / kIn, row = q - cg * kIn;
    f32x2 acc[NPAIR][kCols];
#pragma unroll
    for (int o = 0; o < NPAIR; ++o)
#pragma unroll
      for (int j = 0; j < kCols; ++j) acc[o][j] = 0ull;
#pragma unroll
    for (int c = 0; c < kCols + 2 * kR; ++c) {
      f32x2 p[NPAIR];
      prod(row * kInRow + cg * kCols + c, p);
#pragma unroll
      for (int j = 0; j < kCols; ++j) {
        const int dd = c - j;
        if (dd >= 0 && dd <= 2 * kR) {
          const f32x2 w = dup2(win.w[dd < kR ? kR - dd : dd - kR]);
#pragma unroll
          for (int o = 0; o < NPAIR; ++o) acc[o][j] = fma2(w, p[o], acc[o][j]);
        }
      }
    }
#pragma unroll
    for (int o = 0; o < NPAIR; ++o)
#pragma unroll
      for (int j = 0; j < kCols; ++j) s_h[o * kHPlane + row * kHRow + cg * kCols + j] = acc[o][j];
  }
}

// Vertical window sums at the thread's pixels: rows oy0 .. oy0 + kRows - 1 of
// column ox, each horizontal sum read once.
template <int NPAIR>
__device__ __forceinline__ void filter_columns(const f32x2* s_h, const Window& win, int oy0, int ox,
                                               f32x2 (&out)[NPAIR][kRows]) {
#pragma unroll
  for (int o = 0; o < NPAIR; ++o) {
#pragma unroll
    for (int j = 0; j < kRows; ++j) out[o][j] = 0ull;
#pragma unroll
    for (int c = 0; c < kRows + 2 * kR; ++c) {
      const f32x2 h = s_h[o * kHPlane + (oy0 + c) * kHRow + ox];
#pragma unroll
      for (int j = 0; j < kRows; ++j) {
        const int dd = c - j;
        if (dd >= 0 && dd <= 2 * kR) out[o][j] = fma2(dup2(win.w[dd < kR ? kR - dd : dd - kR]), h, out[o][j]);
      }
    }
  }
}
// The output pixels of a thread.
__device__ __forceinline__ void out_block(int& oy0, int& ox) {
  ox = threadIdx.x % kTile;
  oy0 = (threadIdx.x / kTile) * kRows;
}
static_assert(kSsimThreads * kRows == kTile * kTile, "one block of kRows pixels per thread");

__device__ __forceinline__ float lo2(f32x2 v) {
  float a, b;
  unpack2(v, a, b);
  return a;
}
__device__ __forceinline__ float hi2(f32x2 v) {
  float a, b;
  unpack2(v, a, b);
  return b;
}

// SSIM and its partials by the raw window moments at one pixel
__device__ __forceinline__ void ssim_at(float mx, float my, float ex2, float ey2, float exy, float& S, float& dmx,
                                        float& dex2, float& dexy) {
  const float sx2 = ex2 - mx * mx, sy2 = ey2 - my * my, sxy = exy - mx * my;
  const float A1 = 2.f * mx * my + kC1, A2 = 2.f * sxy + kC2;
  const float B1 = mx * mx + my * my + kC1, B2 = sx2 + sy2 + kC2;
  const float iB = 1.f / (B1 * B2);
  S = A1 * A2 * iB;
  const float d_mx = 2.f * A2 * iB * (my - mx * A1 / B1);
  const float d_sx2 = -S / B2;
  const float d_sxy = 2.f * A1 * iB;
  dmx = d_mx - 2.f * mx * d_sx2 - my * d_sxy;
  dex2 = d_sx2;
  dexy = d_sxy;
}

// The SSIM map's partials P1..P3 by the window moments, the objective's sum, and
// for each of NP probes a_k = lambda/(4 max(1 - S, floor))/m . dS[d_k].  The
// planes of d and a are `stride` floats apart.
template <int NP>
__global__ void __launch_bounds__(kSsimThreads, 3) ssim_map_kernel(
    const float* __restrict__ img, const float* __restrict__ tgt, const float* __restrict__ d, Plane pl, size_t stride,
    Window win, float lambda, float inv_2m, float wscale, float floor_, float* __restrict__ P1, float* __restrict__ P2,
    float* __restrict__ P3, float* __restrict__ a, float* __restrict__ loss) {
  extern __shared__ __align__(16) f32x2 smem2[];
  f32x2* s_xy = smem2;             // (image, target)
  f32x2* s_d = s_xy + kInPlane;    // the probes' tangents
  f32x2* s_h = smem2 + (NP > 0 ? 2 : 1) * kInPlane;
  __shared__ float s_red[kSsimThreads / 32];
  const int x0 = blockIdx.x * kTile, y0 = blockIdx.y * kTile;
  const size_t off = (size_t)blockIdx.z * pl.W * pl.H;
  load_tile(img + off, pl.W, pl.H, x0, y0, reinterpret_cast<float*>(s_xy), 2);
  load_tile(tgt + off, pl.W, pl.H, x0, y0, reinterpret_cast<float*>(s_xy) + 1, 2);
#pragma unroll
  for (int k = 0; k < NP; ++k)
    load_tile(d + (size_t)k * stride + off, pl.W, pl.H, x0, y0, reinterpret_cast<float*>(s_d) + k, 2);
  cp_async_wait_all();
  __syncthreads();
  int oy0, ox;
  out_block(oy0, ox);
  float lsum = 0.f, g1[kRows], g2[kRows], g3[kRows], wv[kRows];
  {
    filter_rows<3>(s_h, win, [&](int at, f32x2 (&p)[3]) {
      p[0] = s_xy[at];
      p[1] = mul2(p[0], p[0]);
      p[2] = pack2(lo2(p[0]) * hi2(p[0]), 0.f);
    });
    __syncthreads();
    f32x2 f[3][kRows];
    filter_columns<3>(s_h, win, oy0, ox, f);
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      float s;
      ssim_at(lo2(f[0][j]), hi2(f[0][j]), lo2(f[1][j]), hi2(f[1][j]), lo2(f[2][j]), s, g1[j], g2[j], g3[j]);
      const int gx = x0 + ox, gy = y0 + oy0 + j;
      wv[j] = wscale / (4.f * fmaxf(1.f - s, floor_));
      if (gx >= pl.W || gy >= pl.H) continue;
      const size_t at = off + (size_t)gy * pl.W + gx;
      P1[at] = g1[j];
      P2[at] = g2[j];
      P3[at] = g3[j];
      const f32x2 xy = s_xy[(oy0 + j + kR) * kInRow + ox + kR];
      lsum += ((1.f - lambda) * fabsf(lo2(xy) - hi2(xy)) + lambda * (1.f - s)) * inv_2m;
    }
  }
  if constexpr (NP > 0) {
    constexpr int NPAIR = NP == 2 ? 3 : 2;
    __syncthreads();  // the sums have been read
    filter_rows<NPAIR>(s_h, win, [&](int at, f32x2 (&p)[NPAIR]) {
      const f32x2 xy = s_xy[at], dk = s_d[at];
      const float x2 = 2.f * lo2(xy), y = hi2(xy);
      if constexpr (NP == 2) {
        p[0] = dk;
        p[1] = mul2(dup2(x2), dk);
        p[2] = mul2(dup2(y), dk);
      } else {
        p[0] = pack2(lo2(dk), x2 * lo2(dk));
        p[1] = pack2(y * lo2(dk), 0.f);
      }
    });
    __syncthreads();
    f32x2 f[NPAIR][kRows];
    filter_columns<NPAIR>(s_h, win, oy0, ox, f);
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      const int gx = x0 + ox, gy = y0 + oy0 + j;
      if (gx >= pl.W || gy >= pl.H) continue;
      const size_t at = off + (size_t)gy * pl.W + gx;
      if constexpr (NP == 2) {
        a[at] = wv[j] * (g1[j] * lo2(f[0][j]) + g2[j] * lo2(f[1][j]) + g3[j] * lo2(f[2][j]));
        a[stride + at] = wv[j] * (g1[j] * hi2(f[0][j]) + g2[j] * hi2(f[1][j]) + g3[j] * hi2(f[2][j]));
      } else {
        a[at] = wv[j] * (g1[j] * lo2(f[0][j]) + g2[j] * hi2(f[0][j]) + g3[j] * lo2(f[1][j]));
      }
    }
  }
  if (loss) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = lsum;
    __syncthreads();
    if (threadIdx.x == 0) {
      float t = 0.f;
      for (int w = 0; w < kSsimThreads / 32; ++w) t += s_red[w];
      atomicAdd(loss, t);
    }
  }
}

// The cotangent images: the gradient stream (GRAD; the map's adjoint with
// weights all 1) and NA probe streams (the adjoint of the weight planes a_k),
// each with its L1 part.  The planes of a, d and cot are `stride` floats apart.
template <int NA, bool GRAD>
__global__ void __launch_bounds__(kSsimThreads, 3) ssim_cot_kernel(
    const float* __restrict__ a, const float* __restrict__ img, const float* __restrict__ tgt, Plane pl, size_t stride,
    Window win, const float* __restrict__ P1, const float* __restrict__ P2, const float* __restrict__ P3,
    const float* __restrict__ d, float lambda, float inv_m, float floor_, float* __restrict__ cot) {
  extern __shared__ __align__(16) f32x2 smem2[];
  f32x2* s_p = smem2;                // (P1, P2)
  f32x2* s_a = s_p + kInPlane;       // the probes' weights
  f32x2* s_h = s_p + (NA > 0 ? 2 : 1) * kInPlane;
  float* s_p3 = reinterpret_cast<float*>(s_h + kGroup * kHPlane);
  const int x0 = blockIdx.x * kTile, y0 = blockIdx.y * kTile;
  const size_t off = (size_t)blockIdx.z * pl.W * pl.H;
  load_tile(P1 + off, pl.W, pl.H, x0, y0, reinterpret_cast<float*>(s_p), 2);
  load_tile(P2 + off, pl.W, pl.H, x0, y0, reinterpret_cast<float*>(s_p) + 1, 2);
  load_tile(P3 + off, pl.W, pl.H, x0, y0, s_p3, 1);
#pragma unroll
  for (int k = 0; k < NA; ++k)
    load_tile(a + (size_t)k * stride + off, pl.W, pl.H, x0, y0, reinterpret_cast<float*>(s_a) + k, 2);
  int oy0, ox;
  out_block(oy0, ox);
  float x[kRows], y[kRows];
  const int gx = x0 + ox, gy0 = y0 + oy0;
  const size_t at0 = off + (size_t)gy0 * pl.W + gx;
#pragma unroll
  for (int j = 0; j < kRows; ++j) {
    const bool in = gx < pl.W && gy0 + j < pl.H;
    x[j] = in ? __ldg(img + at0 + (size_t)j * pl.W) : 0.f;
    y[j] = in ? __ldg(tgt + at0 + (size_t)j * pl.W) : 0.f;
  }
  cp_async_wait_all();
  __syncthreads();
  if constexpr (GRAD) {
    filter_rows<2>(s_h, win, [&](int at, f32x2 (&p)[2]) {
      p[0] = s_p[at];
      p[1] = pack2(s_p3[at], 0.f);
    });
    __syncthreads();
    f32x2 f[2][kRows];
    filter_columns<2>(s_h, win, oy0, ox, f);
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      if (gx >= pl.W || gy0 + j >= pl.H) continue;
      const float r = x[j] - y[j], A = lo2(f[0][j]) + 2.f * x[j] * hi2(f[0][j]) + y[j] * lo2(f[1][j]);
      cot[at0 + (size_t)j * pl.W] = 0.5f * inv_m * ((1.f - lambda) * (float)((r > 0.f) - (r < 0.f)) - lambda * A);
    }
  }
  if constexpr (NA > 0) {
    constexpr int NPAIR = NA == 2 ? 3 : 2;
    float* out = cot + (GRAD ? stride : 0);
    float dv[NA][kRows];
#pragma unroll
    for (int k = 0; k < NA; ++k)
#pragma unroll
      for (int j = 0; j < kRows; ++j)
        dv[k][j] = gx < pl.W && gy0 + j < pl.H ? __ldg(d + (size_t)k * stride + at0 + (size_t)j * pl.W) : 0.f;
    if (GRAD) __syncthreads();  // the sums have been read
    filter_rows<NPAIR>(s_h, win, [&](int at, f32x2 (&p)[NPAIR]) {
      const f32x2 p12 = s_p[at], ak = s_a[at];
      const float p3 = s_p3[at];
      if constexpr (NA == 2) {
        p[0] = mul2(ak, dup2(lo2(p12)));
        p[1] = mul2(ak, dup2(hi2(p12)));
        p[2] = mul2(ak, dup2(p3));
      } else {
        p[0] = mul2(dup2(lo2(ak)), p12);
        p[1] = pack2(lo2(ak) * p3, 0.f);
      }
    });
    __syncthreads();
    f32x2 f[NPAIR][kRows];
    filter_columns<NPAIR>(s_h, win, oy0, ox, f);
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      if (gx >= pl.W || gy0 + j >= pl.H) continue;
      const float l1 = (1.f - lambda) * inv_m / (4.f * fmaxf(fabsf(x[j] - y[j]), floor_));
#pragma unroll
      for (int k = 0; k < NA; ++k) {
        float f0, f1, f2;
        if constexpr (NA == 2) {
          f0 = k ? hi2(f[0][j]) : lo2(f[0][j]);
          f1 = k ? hi2(f[1][j]) : lo2(f[1][j]);
          f2 = k ? hi2(f[2][j]) : lo2(f[2][j]);
        } else {
          f0 = lo2(f[0][j]);
          f1 = hi2(f[0][j]);
          f2 = lo2(f[1][j]);
        }
        out[(size_t)k * stride + at0 + (size_t)j * pl.W] = l1 * dv[k][j] + (f0 + 2.f * x[j] * f1 + y[j] * f2);
      }
    }
  }
}

// Shared memory of the kernels: their pair planes, the sums of a group, and P3.
size_t map_smem(int np) { return sizeof(f32x2) * ((np > 0 ? 2 : 1) * kInPlane + kGroup * kHPlane); }
size_t cot_smem(int na) { return map_smem(na) + sizeof(float) * kInPlane; }

Window window() {
  double g[kR + 1], s = 0.0;
  for (int i = 0; i <= kR; ++i) g[i] = std::exp(-(double)(i * i) / (2.0 * 1.5 * 1.5));
  for (int i = -kR; i <= kR; ++i) s += g[i < 0 ? -i : i];
  Window w;
  for (int i = 0; i <= kR; ++i) w.w[i] = (float)(g[i] / s);
  return w;
}

template <class F>
cudaError_t allow_smem(F* f, size_t bytes, bool& done) {
  if (done) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute((const void*)f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  done = e == cudaSuccess;
  return e;
}

// Planes of the call and where they are.
struct SsimArgs {
  Plane pl;
  size_t stride;
  Window win;
  const float *img, *tgt, *d;
  float lambda, inv_m, floor_;
  float *P1, *P2, *P3, *a, *cot, *loss;
};

template <int NP>
cudaError_t launch_ssim(const SsimArgs& s, bool grad, cudaStream_t st) {
  const dim3 grid((s.pl.W + kTile - 1) / kTile, (s.pl.H + kTile - 1) / kTile, s.pl.planes);
  const size_t sm_map = map_smem(NP), sm_cot = cot_smem(NP);
  static bool map_done = false, cot_done[2] = {false, false};
  cudaError_t e = allow_smem(ssim_map_kernel<NP>, sm_map, map_done);
  if (e != cudaSuccess) return e;
  ssim_map_kernel<NP><<<grid, kSsimThreads, sm_map, st>>>(s.img, s.tgt, s.d, s.pl, s.stride, s.win, s.lambda,
                                                          0.5f * s.inv_m, s.lambda * s.inv_m, s.floor_, s.P1, s.P2,
                                                          s.P3, s.a, s.loss);
  if (grad) {
    if ((e = allow_smem(ssim_cot_kernel<NP, true>, sm_cot, cot_done[1])) != cudaSuccess) return e;
    ssim_cot_kernel<NP, true><<<grid, kSsimThreads, sm_cot, st>>>(s.a, s.img, s.tgt, s.pl, s.stride, s.win, s.P1, s.P2,
                                                                  s.P3, s.d, s.lambda, s.inv_m, s.floor_, s.cot);
  } else if constexpr (NP > 0) {
    if ((e = allow_smem(ssim_cot_kernel<NP, false>, sm_cot, cot_done[0])) != cudaSuccess) return e;
    ssim_cot_kernel<NP, false><<<grid, kSsimThreads, sm_cot, st>>>(s.a, s.img, s.tgt, s.pl, s.stride, s.win, s.P1,
                                                                   s.P2, s.P3, s.d, s.lambda, s.inv_m, s.floor_, s.cot);
  }
  return cudaSuccess;
}

}  // namespace
}  // namespace gs

extern "C" size_t gs_dssim_workspace_size(gs_frame frame, int32_t nu) {
  if (frame.n_views < 1 || frame.width < 1 || frame.height < 1 || nu < 0 || nu > 2) return 0;
  const size_t plane = (size_t)frame.n_views * 3 * frame.width * frame.height;
  return plane * sizeof(float) * (4 + (size_t)nu);  // three partials, one weight map per probe (and one plane spare)
}

extern "C" gs_status gs_dssim_cotangents(gs_frame frame, const float* image, const float* target,
                                         const float* image_tangent, int32_t nu, float lambda, float gn_floor,
                                         int32_t want_grad, float* cot, float* loss_out, void* workspace,
                                         size_t workspace_bytes, int32_t* status, void* stream) {
  using namespace gs;
  (void)status;
  GS_REQUIRE(image && target && cot, "gs_dssim_cotangents: null argument");
  GS_REQUIRE(frame.n_views >= 1 && frame.width >= 1 && frame.height >= 1, "gs_dssim_cotangents: bad frame");
  GS_REQUIRE(nu >= 0 && nu <= 2 && (nu == 0 || image_tangent), "gs_dssim_cotangents: bad nu=%d or no tangents", nu);
  GS_REQUIRE(want_grad || nu > 0, "gs_dssim_cotangents: nothing to compute");
  GS_REQUIRE(lambda >= 0.f && lambda <= 1.f && gn_floor > 0.f, "gs_dssim_cotangents: bad lambda or floor");
  const size_t need = gs_dssim_workspace_size(frame, nu);
  GS_REQUIRE(workspace && workspace_bytes >= need, "gs_dssim_cotangents: workspace needs %zu bytes, got %zu", need,
             workspace_bytes);
  cudaStream_t st = (cudaStream_t)stream;
  SsimArgs a;
  a.pl = Plane{frame.width, frame.height, frame.n_views * 3};
  const size_t plane = a.stride = (size_t)a.pl.planes * a.pl.W * a.pl.H;
  float* ws = (float*)workspace;
  a.win = window();
  a.img = image;
  a.tgt = target;
  a.d = image_tangent;
  a.lambda = lambda;
  a.inv_m = (float)(1.0 / (6.0 * frame.width * frame.height * frame.n_views));
  a.floor_ = gn_floor;
  a.P1 = ws;
  a.P2 = ws + plane;
  a.P3 = ws + 2 * plane;
  a.a = ws + 3 * plane;
  a.cot = cot;
  a.loss = loss_out;
  const cudaError_t e = nu == 0 ? launch_ssim<0>(a, want_grad != 0, st)
                        : nu == 1 ? launch_ssim<1>(a, want_grad != 0, st) : launch_ssim<2>(a, want_grad != 0, st);
  if (e != cudaSuccess) return check_launch("gs_dssim_cotangents: smem attribute");
  return check_launch("gs_dssim_cotangents");
}
