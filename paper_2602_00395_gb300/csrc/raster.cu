// Rasteriser forward and reverse passes of arXiv 2602.00395:
//
//   gs_raster_fwd  front-to-back alpha blending per pixel (Sec. 3.1), with the
//                  forward-mode tangents J z_k of the Hutchinson probes fused in
//                  (Sec. 4.1; the paper's forward-mode AD of the rasteriser, Sec. 5)
//   gs_raster_bwd  reverse pass for the gradient g = (1/m) J^T F (Sec. 4.1) and,
//                  in the same sweep, the Gauss-Newton products J^T diag(w) J z_k
//   gs_hvp_diag    the Gauss-Newton products alone
//
// Both blends run one warp per CTA on one 8 x 8 pixel block of a tile, two pixels
// per thread held as a packed FP32 pair.  A warp walks its tile's list in
// chunks of 32 positions, keeps the splats whose alpha >= 1/255 footprint can
// reach its block, and stages those records in shared memory by asynchronous
// copies, one buffer ahead of the one it blends.  Nothing is shared with the
// tile's other blocks, so no block waits for another (but see below).  The reverse
// pass walks the list back to front, recovers T_i = T_{i+1} / (1 - a_i) from the final
// transmittance (nothing per pair is stored), sums each splat's 9 x streams partial
// derivatives over the block's 64 pixels in a fixed order, and adds them with
// float4 reductions; with two probes beside the gradient a tile's warps walk its list
// in step, sharing a ring of TMA-staged batches.  The projection's reverse pass (2-D
// cotangents -> 11 + 3K parameter rows) runs one thread per Gaussian and sums
// over the views.
#include "common.cuh"

namespace gs {
namespace {

struct alignas(16) Rec {
  float4 a;  // mx, my, A, B
  float4 b;  // C, opacity, r, g
  float4 c;  // b, depth, radius bits, unused
};
static_assert(sizeof(Rec) == 48, "record size");

__device__ __forceinline__ float ex2_approx(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// The splat at a thread's two pixels, which share their column: dx and the
// negated centres -py of the pair give dy, then power and exp(power) per pixel.
// One function with a fixed rounding sequence, so that the forward and reverse
// kernels take identical decisions.
__device__ __forceinline__ void splat_gauss2(const Rec& r, float pxc, f32x2 npy, float& dx, f32x2& dy,
                                             float (&power)[2], f32x2& G) {
  dx = __fsub_rn(r.a.x, pxc);
  dy = add2(dup2(r.a.y), npy);
  const f32x2 q = fma2(dup2(r.b.x), mul2(dy, dy), dup2(__fmul_rn(r.a.z, __fmul_rn(dx, dx))));
  const f32x2 pw = fma2(dup2(-0.5f), q, mul2(dup2(-r.a.w), mul2(dup2(dx), dy)));
  unpack2(pw, power[0], power[1]);
  // e^p = 2^(p log2 e)
  float l[2];
  unpack2(mul2(pw, dup2(1.4426950408889634f)), l[0], l[1]);
  G = pack2(ex2_approx(l[0]), ex2_approx(l[1]));
}

// 1: the blends also test a splat's footprint ellipse itself, not only its
// bounding box, against each 8 x 8 pixel block (0: the box alone).
#ifndef GS_EXACT_BLOCK_TEST
#define GS_EXACT_BLOCK_TEST 1
#endif

// False only if no pixel centre of the 8 x 8 block with first centre (x0, y0)
// can reach alpha >= 1/255: the minimum over the rectangle [x0, x0 + 7] x
// [y0, y0 + 7] of q(u) = A ux^2 + 2 B ux uy + C uy^2, u = p - mean (-2 x the
// power), is above 2 ln(255 o) by more than a slack that covers the FP32
// rounding of both this test and the blends' own evaluation (1e-4 of the
// terms' largest magnitude on the rectangle, 1e-3 relative and absolute, each
// hundreds of times their error bounds).  With the origin outside the rectangle
// the convex q takes its minimum on an edge, where it is a parabola in one
// coordinate.  A conic that is not positive definite is never rejected.
__device__ __forceinline__ bool footprint_meets_block(const Rec& r, float x0, float y0) {
  const float A = r.a.z, B = r.a.w, C = r.b.x;
  if (!(A > 0.f && C > 0.f && A * C > B * B)) return true;
  const float thr = 2.f * __logf(255.f * r.b.y);
  const float xl = x0 - r.a.x, xh = xl + 7.f, yl = y0 - r.a.y, yh = yl + 7.f;
  const float X = fmaxf(fabsf(xl), fabsf(xh)), Y = fmaxf(fabsf(yl), fabsf(yh));
  const float slack = 1e-4f * (A * X * X + 2.f * fabsf(B) * X * Y + C * Y * Y) + 1e-3f * fabsf(thr) + 1e-3f;
  if (xl <= 0.f && xh >= 0.f && yl <= 0.f && yh >= 0.f) return thr + slack >= 0.f;
  const float bc = B / C, ba = B / A;
  auto on_x_edge = [&](float ux) {  // q on ux = const, minimised over uy in [yl, yh]
    const float uy = fminf(fmaxf(-bc * ux, yl), yh);
    return A * ux * ux + 2.f * B * ux * uy + C * uy * uy;
  };
  auto on_y_edge = [&](float uy) {
    const float ux = fminf(fmaxf(-ba * uy, xl), xh);
    return A * ux * ux + 2.f * B * ux * uy + C * uy * uy;
  };
  const float qmin = fminf(fminf(on_x_edge(xl), on_x_edge(xh)), fminf(on_y_edge(yl), on_y_edge(yh)));
  return qmin <= thr + slack;
}

// ------------------------------------------------------------ pixel blocks
// A tile is cut into 8 x 8 pixel blocks, block w at (w % (tile_w/8), w / (tile_w/8)),
// and a lane renders pixels (lx, ly) and (lx, ly + 4) of its warp's block.
// Compact blocks meet few splats; two pixels per thread halve the per-splat
// overheads and share a column.
constexpr int kPixPerThread = 2;

// The 8 x 8 block of a one-warp CTA: its view and tile (the heaviest tiles first
// when an order is given), its number w in the tile and its first pixel.
struct PixelBlock {
  int view, tile, w, x0, y0;
};
__device__ __forceinline__ PixelBlock pixel_block(const uint32_t* __restrict__ order, const gs_frame& fr, int Tx, int T,
                                                  int log_blocks) {
  PixelBlock p;
  p.w = (int)(blockIdx.x & ((1u << log_blocks) - 1u));
  const int ordinal = (int)(blockIdx.x >> log_blocks);
  const int blk = order ? (int)min(__ldg(order + ordinal), (gridDim.x >> log_blocks) - 1) : ordinal;
  p.view = blk / T;
  p.tile = blk - p.view * T;
  const int ty = p.tile / Tx, tx = p.tile - ty * Tx, bw = fr.tile_w >> 3;
  p.x0 = tx * fr.tile_w + (p.w % bw) * 8;
  p.y0 = ty * fr.tile_h + (p.w / bw) * 8;
  return p;
}

// True if the splat can reach alpha >= 1/255 at some pixel centre of the 8 x 8
// block whose first pixel centre is (x0, y0).  The record's last word holds the
// half-extents of the bounding box of that footprint, widened and rounded up by
// the projection (footprint_extents); a block inside the box is then tested
// against the ellipse (footprint_meets_block).  Both tests are conservative, so a
// block that fails them skips only splats that every pixel of it skips anyway:
// results are unchanged.
__device__ __forceinline__ bool block_sees(const Rec& r, float x0, float y0) {
  const uint32_t e = __float_as_uint(r.c.w);
  const float hx = __half2float(__ushort_as_half((unsigned short)(e & 0xffffu)));
  const float hy = __half2float(__ushort_as_half((unsigned short)(e >> 16)));
  return r.a.x + hx >= x0 && r.a.x - hx <= x0 + 7.f && r.a.y + hy >= y0 && r.a.y - hy <= y0 + 7.f &&
         (!GS_EXACT_BLOCK_TEST || footprint_meets_block(r, x0, y0));
}

// ------------------------------------------------------------------ forward
// Blend state of a thread's two pixels: colour, transmittance, the probe tangents
// of both, and each pixel's list position after its last blended splat.
template <int NU>
struct FwdPair {
  f32x2 C[3], T;
  f32x2 Cd[NU > 0 ? NU : 1][3], Td[NU > 0 ? NU : 1];
  f32x2 npy;  // negated pixel centres
  float pxc;
  uint32_t last[2];
  bool done[2];
};

// One splat's front-to-back update of the two pixels, with the decisions as
// selects: a pixel that does not blend the splat (it is done or skips it, or the
// splat would take T below kTMin, which ends the pixel instead) adds exact
// zeros and keeps T, its tangents and its last position.  tk: the splat's
// rewritten tangent records (see raster_fwd_kernel).  With the power's tangent
// pd, a blended pixel gets C += c a T, C' += c' a T + c (a' T + a T'),
// T' <- T' (1 - a) - T a', T <- T (1 - a), a' = a (o'/o + pd) (0 for a capped alpha).
template <int NU>
__device__ __forceinline__ void fwd_visit(FwdPair<NU>& p, const Rec& r, const Rec* tk, uint32_t pos) {
  float dx, power[2], oG[2], al[2], Tn[2];
  f32x2 dy, G;
  splat_gauss2(r, p.pxc, p.npy, dx, dy, power, G);
  unpack2(mul2(dup2(r.b.y), G), oG[0], oG[1]);
  bool on[2], bl[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    al[q] = fminf(kAlphaMax, oG[q]);
    on[q] = !p.done[q] && power[q] <= 0.f && al[q] >= kAlphaMin;
  }
  if (!__any_sync(0xffffffffu, on[0] || on[1])) return;
  const f32x2 alp = pack2(al[0], al[1]);
  unpack2(mul2(p.T, fma2(alp, dup2(-1.f), dup2(1.f))), Tn[0], Tn[1]);
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    bl[q] = on[q] && !(Tn[q] < kTMin);
    p.done[q] = p.done[q] || (on[q] && !bl[q]);
    p.last[q] = bl[q] ? pos + 1 : p.last[q];
  }
  const f32x2 a = pack2(bl[0] ? al[0] : 0.f, bl[1] ? al[1] : 0.f);
  const f32x2 om = fma2(a, dup2(-1.f), dup2(1.f)), w = mul2(a, p.T);
  if constexpr (NU > 0) {
    const bool live0 = bl[0] && !(oG[0] > kAlphaMax), live1 = bl[1] && !(oG[1] > kAlphaMax);
#pragma unroll
    for (int k = 0; k < NU; ++k) {
      const Rec t = tk[k];
      const float p0 = fmaf(dx, fmaf(t.a.x, dx, t.a.w), t.b.y), p1 = fmaf(t.a.y, dx, t.b.x);
      float ad0, ad1;
      unpack2(mul2(alp, fma2(dy, fma2(dy, dup2(t.a.z), dup2(p1)), dup2(p0))), ad0, ad1);
      const f32x2 adT = mul2(pack2(live0 ? ad0 : 0.f, live1 ? ad1 : 0.f), p.T);
      const f32x2 sk = fma2(a, p.Td[k], adT);
      p.Cd[k][0] = fma2(dup2(r.b.z), sk, fma2(dup2(t.b.z), w, p.Cd[k][0]));
      p.Cd[k][1] = fma2(dup2(r.b.w), sk, fma2(dup2(t.b.w), w, p.Cd[k][1]));
      p.Cd[k][2] = fma2(dup2(r.c.x), sk, fma2(dup2(t.c.x), w, p.Cd[k][2]));
      p.Td[k] = fma2(adT, dup2(-1.f), mul2(p.Td[k], om));
    }
  }
  p.C[0] = fma2(dup2(r.b.z), w, p.C[0]);
  p.C[1] = fma2(dup2(r.b.w), w, p.C[1]);
  p.C[2] = fma2(dup2(r.c.x), w, p.C[2]);
  p.T = mul2(p.T, om);  // a pixel that blends nothing has om = 1
}

// Minimum resident CTAs (warps) per SM requested from the compiler for the
// forward kernel, by the number of probes, and the splats per staging buffer
// (larger buffers pause less often, smaller ones leave room for more warps).
// Measured on 1M Gaussians, 8 views of 1080p: without a probe 32 CTAs and
// buffers of 32 (0.762 ms; 28 CTAs 0.821, buffers of 16 0.790), with one 30 and
// 16 (1.053; 24 CTAs 1.165), with two 21 and 24 (80 registers, so 24 CTAs run;
// 1.370; 20 CTAs and 16 1.487, 25 CTAs 1.486, buffers of 16 1.399, of 32 1.432).
#ifndef GS_FWD_MB0
#define GS_FWD_MB0 32
#endif
#ifndef GS_FWD_MB1
#define GS_FWD_MB1 30
#endif
#ifndef GS_FWD_MB2
#define GS_FWD_MB2 21
#endif
#ifndef GS_FWD_BUF0
#define GS_FWD_BUF0 32
#endif
#ifndef GS_FWD_BUF1
#define GS_FWD_BUF1 16
#endif
#ifndef GS_FWD_BUF2
#define GS_FWD_BUF2 24
#endif
// Splats per staging buffer, at most 32.
__host__ __device__ constexpr int fwd_buffer(int nu) { return nu == 0 ? GS_FWD_BUF0 : nu == 1 ? GS_FWD_BUF1 : GS_FWD_BUF2; }
__host__ __device__ constexpr int fwd_min_blocks(int nu) { return nu == 0 ? GS_FWD_MB0 : nu == 1 ? GS_FWD_MB1 : GS_FWD_MB2; }

// The pairs' mask bytes as aligned 32-bit words: byte q is byte head + q of
// `words` (head < 4), and `count` words from `first` on lie within the array.  The
// bytes of the array outside them, at most three at each end, have every bit set
// instead (the reverse pass then tests the splat at the pixels, which is as right).
struct MaskWords {
  uint32_t* words;  // NULL: no masks, or none but set bits
  uint32_t head, first, count;
};

// The kernel is bound by issue slots (65 %) and the FMA pipe (50 %).  As CTAs of a
// tile's four warps that met at two barriers per staged batch, with scalar
// pixels, it took 1.702 ms with two probes (now 1.370), 1.414 with one (1.053)
// and 1.085 without (0.762); 100k Gaussians, 1297 x 840, one probe 0.293 ms
// (0.243).  Instructions per launch of two views: 411M, now 293M.
// masks: cleared before the launch (the blocks of a tile set their own bits of the
// same bytes).
template <int NU>
__global__ void __launch_bounds__(32, fwd_min_blocks(NU)) raster_fwd_kernel(
    const float4* __restrict__ rec, const float4* __restrict__ tan, const uint32_t* __restrict__ vals,
    const uint32_t* __restrict__ ranges, const uint32_t* __restrict__ order, int n_pad, gs_frame fr, int Tx, int T,
    int log_blocks, float* __restrict__ image, float* __restrict__ final_T, uint32_t* __restrict__ n_contrib,
    float* __restrict__ image_tan, MaskWords masks) {
  constexpr int kFwdBuf = fwd_buffer(NU);
  constexpr int kPieces = 3 * (1 + NU);  // 16-byte pieces of a splat's record and tangents
  // two buffers of staged splats (the record, whose radius word is replaced by
  // the list position, then its tangents), and the splats' indices and positions
  __shared__ Rec buf[2][kFwdBuf * (1 + NU)];
  __shared__ uint2 s_who[2][kFwdBuf];
  const int lane = threadIdx.x;
  const PixelBlock pb = pixel_block(order, fr, Tx, T, log_blocks);
  const int view = pb.view;
  if (pb.x0 >= fr.width || pb.y0 >= fr.height) return;
  const size_t tslot = 2 * ((size_t)view * T + pb.tile);
  const uint32_t start = __ldg(ranges + tslot);
  const int n = (int)(__ldg(ranges + tslot + 1) - start), nc = (n + 31) >> 5;
  const float wx0 = (float)pb.x0 + 0.5f, wy0 = (float)pb.y0 + 0.5f;  // the block's first pixel centre
  const int px = pb.x0 + (lane & 7), py = pb.y0 + (lane >> 3);       // and (px, py + 4)

  FwdPair<NU> p;
  p.C[0] = p.C[1] = p.C[2] = 0ull;
  p.T = dup2(1.f);
#pragma unroll
  for (int k = 0; k < NU; ++k) p.Cd[k][0] = p.Cd[k][1] = p.Cd[k][2] = p.Td[k] = 0ull;
  p.pxc = (float)px + 0.5f;
  p.npy = pack2(-((float)py + 0.5f), -((float)(py + 4) + 0.5f));
  p.last[0] = p.last[1] = 0;
  p.done[0] = !(px < fr.width && py < fr.height);
  p.done[1] = !(px < fr.width && py + 4 < fr.height);

  // Chunks of 32 list positions, front to back: a lane holds one position's
  // index two chunks ahead and its record one chunk ahead of the test whether
  // the splat can reach this block.
  const float4* vrec = rec + 3 * (size_t)view * n_pad;
  int c = 0;
  auto index_of = [&](int cc) -> uint32_t {
    const int q = cc * 32 + lane;
    return q < n ? __ldg(vals + start + (uint32_t)q) : 0xffffffffu;
  };
  auto record_of = [&](uint32_t g, Rec& r) {
    if (g == 0xffffffffu) return;
    const float4* src = vrec + 3 * (size_t)g;  // what block_sees reads
    r.a = __ldg(src);
    const float2 Co = __ldg(reinterpret_cast<const float2*>(src + 1));
    r.b.x = Co.x;
    r.b.y = Co.y;
    r.c.w = __ldg(reinterpret_cast<const float*>(src + 2) + 3);
  };
  uint32_t gi = index_of(0), gi1 = index_of(1), gi2 = 0, bits = 0;
  Rec rn{};
  record_of(gi, rn);
  // tests chunk c (index gi, record rn), marks its visible pairs, and starts the
  // loads of the chunks after it
  auto test = [&]() {
    bits = 0;
    if (c >= nc) return;
    bits = __ballot_sync(0xffffffffu, gi != 0xffffffffu && block_sees(rn, wx0, wy0));
    if (masks.words && lane <= 8) {
      // byte q of the masks is pair q's: the chunk's bits, shifted to the words'
      // boundaries, four at a time spread over a word's bytes at bit w
      const uint32_t at = start + (uint32_t)(c * 32) + masks.head, word = (at >> 2) + lane;
      const uint32_t nib = (uint32_t)(((uint64_t)bits << (at & 3u)) >> (4 * lane)) & 15u;
      if (nib && word - masks.first < masks.count)
        atomicOr(masks.words + word, ((nib * 0x204081u) & 0x01010101u) << pb.w);
    }
    record_of(gi1, rn);
    gi2 = index_of(c + 2);
  };
  test();
  auto fill = [&](int b) {
    int cnt = 0;
    while (c < nc) {
      const int at = cnt + __popc(bits & ((1u << lane) - 1u));
      const bool mine = ((bits >> lane) & 1u) && at < kFwdBuf;
      if (mine) s_who[b][at] = make_uint2(gi, (uint32_t)(c * 32 + lane));
      cnt += __popc(bits);
      if (cnt > kFwdBuf) {  // the rest of the chunk goes to the next buffer
        bits &= ~__ballot_sync(0xffffffffu, mine);
        cnt = kFwdBuf;
        break;
      }
      ++c;
      gi = gi1;
      gi1 = gi2;
      test();
    }
    __syncwarp();
    const float4* src = NU > 0 ? tan + (size_t)kPieces * ((size_t)view * n_pad) : vrec;
    for (int q = lane; q < cnt * kPieces; q += 32) {
      const int e = q / kPieces;
      cp_async16(reinterpret_cast<float4*>(buf[b]) + q, src + (size_t)kPieces * s_who[b][e].x + (q - e * kPieces));
    }
    cp_async_commit();
    return cnt;
  };

  int cur = 0, cnt = fill(0);
  while (cnt > 0) {
    const int cnt_next = fill(cur ^ 1);
    cp_async_wait_prior();  // all but the newest group: this buffer has landed
    __syncwarp();
    if (lane < cnt) {
      // the list position, and the probe tangents of the splat's power and
      // opacity rewritten as pd + o'/o = (a dx + d) dx + f + (b dx + e) dy + c dy^2
      Rec* rp = &buf[cur][lane * (1 + NU)];
      const float4 ra = rp->a;
      const float rC = rp->b.x, o = rp->b.y;
      rp->c.z = __uint_as_float(s_who[cur][lane].y);
#pragma unroll
      for (int k = 0; k < NU; ++k) {
        Rec* tp = rp + 1 + k;
        const float4 ta = tp->a;  // dmx, dmy, dA, dB
        const float dC = tp->b.x;
        tp->a = make_float4(-0.5f * ta.z, -ta.w, -0.5f * dC, -(ra.z * ta.x + ra.w * ta.y));
        tp->b.x = -(rC * ta.y + ra.w * ta.x);
        tp->b.y = __fdividef(tp->b.y, o);
      }
    }
    __syncwarp();
    for (int j = 0; j < cnt; ++j) {
      const Rec r = buf[cur][j * (1 + NU)];
      fwd_visit<NU>(p, r, &buf[cur][j * (1 + NU) + 1], __float_as_uint(r.c.z));
    }
    if (__all_sync(0xffffffffu, p.done[0] && p.done[1])) break;
    __syncwarp();  // the buffer may be refilled
    cur ^= 1;
    cnt = cnt_next;
  }
  cp_async_wait_all();  // a buffer staged ahead of an early end lands before the CTA does

  const size_t HW = (size_t)fr.width * fr.height, at = (size_t)py * fr.width + px;
  auto store = [&](float* plane, f32x2 v) {
    float lo, hi;
    unpack2(v, lo, hi);
    if (px < fr.width && py < fr.height) plane[at] = lo;
    if (px < fr.width && py + 4 < fr.height) plane[at + 4 * (size_t)fr.width] = hi;
  };
#pragma unroll
  for (int ch = 0; ch < 3; ++ch) store(image + ((size_t)view * 3 + ch) * HW, p.C[ch]);
  store(final_T + (size_t)view * HW, p.T);
  store(reinterpret_cast<float*>(n_contrib) + (size_t)view * HW,
        pack2(__uint_as_float(p.last[0]), __uint_as_float(p.last[1])));
#pragma unroll
  for (int k = 0; k < NU; ++k)
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) store(image_tan + (((size_t)k * fr.n_views + view) * 3 + ch) * HW, p.Cd[k][ch]);
}

// ------------------------------------------------------------------ reverse
// Two kernels.  With one or two streams a warp per CTA walks its own 8 x 8 block
// (raster_bwd_kernel); with three, the gradient's and two probes', a tile's warps
// walk its list in step (raster_bwd_tile_kernel).  Both sum a splat's products over
// a block in the same fixed order (see merge_slots).
// Minimum resident CTAs (warps) per SM requested from the compiler for
// raster_bwd_kernel, by the number of cotangent streams; what counts is the warps of
// one of the SM's four schedulers, whose registers they share.  Without a probe 28
// (72 registers; 24: 1.577 against 1.563 ms per call of 1M Gaussians, 8 views of
// 1080p, 32, with spills: 1.612), with one 20 (95 registers; 16: 2.524, 24, with
// spills: 2.512 against 2.378).  Against CTAs of a tile's four warps sharing a ring of
// TMA-staged batches, with a reduce-scatter of every splat's row: none 2.29 -> 1.56
// ms, one 3.10 -> 2.38; 100k Gaussians, 1297 x 840, one probe 0.66 -> 0.45 ms.
#ifndef GS_BWD_MB1
#define GS_BWD_MB1 28
#endif
#ifndef GS_BWD_MB2
#define GS_BWD_MB2 20
#endif
__host__ __device__ constexpr int bwd_min_blocks(int S) { return S == 1 ? GS_BWD_MB1 : GS_BWD_MB2; }

// Row stride (floats) of the per-view 2-D cotangents: 9 per stream, padded to
// whole float4s so that rows can be added and read as vectors.
__host__ __device__ constexpr int cot_stride(int streams) { return (9 * streams + 3) & ~3; }
// Place of entry k of stream st in a row of S streams.  The last two streams are
// interleaved, so that the projection's reverse pass reads two probes as packed
// pairs; the first of three follows them.
__host__ __device__ constexpr int cot_index(int S, int st, int k) {
  return S == 1 ? k : st < S - 2 ? 18 + k : 2 * k + (st - (S - 2));
}

// The reverse pass's workspace: a header, then the cotangent rows the reverse
// blend adds into.  They must be zero when the blend starts.  The projection
// reverse, which reads every row, leaves each row it read zero, and its last
// block records in the header that the first clear_floats floats are zero;
// the next call then clears nothing.  Any other header (zeros, foreign bytes, a
// call that stopped between the blend and the projection reverse) makes the next
// call clear the rows first; the blend marks the rows dirty when it starts.  The
// record is the caller's to drop (zeros over the header) where a former workspace
// was written to by something else: only reading every row would show that.
constexpr int kLossSlots = GS_BATCH_MAX;
struct CotHeader {
  uint64_t magic;         // kCotClear while clear_floats is valid
  uint64_t clear_floats;  // leading floats of the rows known to be zero
  uint32_t done_blocks;   // projection-reverse blocks finished in this call
  uint32_t reserved;
  double loss[kLossSlots];  // the objective's partial sums: of each view (a batch), or spread over the slots
};
constexpr uint64_t kCotClear = 0x9d2c5680a3b1f4e7ull;
constexpr size_t kCotHeaderBytes = GS_RASTER_BWD_HEADER;
static_assert(sizeof(CotHeader) <= kCotHeaderBytes, "workspace header");

// Zero the first 4 n4 floats of the rows unless the header says they are zero;
// reset the projection reverse's block count.
__global__ void cot_prepare_kernel(CotHeader* __restrict__ h, float4* __restrict__ cot, size_t n4) {
  const bool clear = h->magic == kCotClear && h->clear_floats >= 4 * n4;
  if (blockIdx.x == 0 && threadIdx.x == 0) h->done_blocks = 0;
  if (blockIdx.x == 0 && threadIdx.x < kLossSlots) h->loss[threadIdx.x] = 0.0;
  if (clear) return;
  for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < n4; k += (size_t)gridDim.x * blockDim.x)
    cot[k] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// The objective's sums onto the caller's: one per view of a batch (loss_views),
// or all slots onto one value (loss_views 0).
__device__ __forceinline__ void add_loss(const CotHeader* h, float* loss_out, int loss_views) {
  double all = 0.0;
  for (int k = 0; k < kLossSlots; ++k) {
    if (k < loss_views) atomicAdd(loss_out + k, (float)h->loss[k]);
    all += h->loss[k];
  }
  if (loss_views == 0) atomicAdd(loss_out, (float)all);
}
// The same where no projection-reverse block runs (no Gaussians).
__global__ void add_loss_kernel(const CotHeader* h, float* loss_out, int loss_views) { add_loss(h, loss_out, loss_views); }

// End of a projection-reverse block: after every thread's zeroing stores, the
// last block to finish records that the first `floats` floats are zero.
__device__ __forceinline__ void cot_mark_clear(CotHeader* h, uint64_t floats, float* loss_out, int loss_views) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0 && atomicAdd(&h->done_blocks, 1u) == gridDim.x - 1) {
    __threadfence();
    if (loss_out) add_loss(h, loss_out, loss_views);
    h->clear_floats = floats;
    h->magic = kCotClear;
  }
}

__device__ __forceinline__ float rcp_approx(float x) {  // at most 1 ulp off
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Reverse-pass state of a thread's two pixels: the negated cotangent -dL/dC of
// each stream, the transmittance being recovered back to front, the negated
// colour suffix -sum_{j>i} a_j T_j c_j, and the list position after each pixel's
// last blended splat.
template <int S>
struct BwdPair {
  f32x2 nw[S][3];
  f32x2 T, ns[3];
  f32x2 npy;  // negated pixel centres
  float pxc;
  uint32_t nc[2];
};

// p[0..3] += v, p 16-byte aligned: a reduction, which returns nothing (the
// atomicAdd on a float4 fetches the old value back).
__device__ __forceinline__ void red_add4(float* p, float4 v) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z),
               "f"(v.w)
               : "memory");
}

// The cotangents dL/dC of each stream at the thread's two pixels, of the block whose
// first pixel is (bx0, by0), and their transmittance and list end (none of an empty
// list, len = 0); returns the objective's terms there.
template <int NU, bool GRAD>
__device__ __forceinline__ float bwd_pixels(BwdPair<(GRAD ? 1 : 0) + NU>& pp, int bx0, int by0, int view, uint32_t len,
                                            const gs_frame& fr, const float* __restrict__ image,
                                            const float* __restrict__ target, const float* __restrict__ final_T,
                                            const uint32_t* __restrict__ n_contrib,
                                            const float* __restrict__ image_tan, int loss_kind, float gn_floor,
                                            float inv_m) {
  constexpr int S = (GRAD ? 1 : 0) + NU;
  const int lane = threadIdx.x & 31;
  const size_t HW = (size_t)fr.width * fr.height;
  float lossp = 0.f;
  float wv[kPixPerThread][S][3], Tv[kPixPerThread], pyc[kPixPerThread];
#pragma unroll
  for (int q = 0; q < kPixPerThread; ++q) {
    const int px = bx0 + (lane & 7), py = by0 + (lane >> 3) + 4 * q;
    pp.pxc = (float)px + 0.5f;
    pyc[q] = (float)py + 0.5f;
    Tv[q] = 0.f;
    pp.nc[q] = 0;
#pragma unroll
    for (int st = 0; st < S; ++st) wv[q][st][0] = wv[q][st][1] = wv[q][st][2] = 0.f;
    if (!(px < fr.width && py < fr.height)) continue;
    const size_t at0 = (size_t)py * fr.width + px;
    if (len) {
      Tv[q] = final_T[(size_t)view * HW + at0];
      pp.nc[q] = n_contrib[(size_t)view * HW + at0];
    }
    if (loss_kind == GS_LOSS_COTANGENT) {  // the caller's cotangent images, one per stream
#pragma unroll
      for (int st = 0; st < S; ++st)
#pragma unroll
        for (int ch = 0; ch < 3; ++ch)
          wv[q][st][ch] = target[(((size_t)st * fr.n_views + view) * 3 + ch) * HW + at0];
      continue;
    }
    if (loss_kind == GS_LOSS_WEIGHTED) {  // dL/dC (gradient stream), then the weights of w . J z_k
      const float* wimg = target + (GRAD ? (size_t)fr.n_views * 3 * HW : 0);
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) {
        if constexpr (GRAD) wv[q][0][ch] = target[((size_t)view * 3 + ch) * HW + at0];
        const float wt = wimg[((size_t)view * 3 + ch) * HW + at0];
#pragma unroll
        for (int k = 0; k < NU; ++k)
          wv[q][(GRAD ? 1 : 0) + k][ch] = wt * image_tan[(((size_t)k * fr.n_views + view) * 3 + ch) * HW + at0];
      }
      continue;
    }
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      const size_t at = ((size_t)view * 3 + ch) * HW + at0;
      const float r = image[at] - target[at];
      const float ar = fabsf(r);
      float lam;
      if (loss_kind == GS_LOSS_L1) {
        lossp += 0.5f * inv_m * ar;
        lam = 0.25f / fmaxf(ar, gn_floor);
      } else {
        lossp += 0.5f * inv_m * r * r;
        lam = 1.f;
      }
      if constexpr (GRAD)
        wv[q][0][ch] = (loss_kind == GS_LOSS_L1) ? (0.5f * inv_m) * ((r > 0.f) - (r < 0.f)) : inv_m * r;
#pragma unroll
      for (int k = 0; len && k < NU; ++k)
        wv[q][(GRAD ? 1 : 0) + k][ch] =
            inv_m * lam * image_tan[(((size_t)k * fr.n_views + view) * 3 + ch) * HW + at0];
    }
  }
  pp.T = pack2(Tv[0], Tv[1]);
  pp.npy = pack2(-pyc[0], -pyc[1]);
  pp.ns[0] = pp.ns[1] = pp.ns[2] = 0ull;
#pragma unroll
  for (int st = 0; st < S; ++st) {
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      pp.nw[st][ch] = pack2(-wv[0][st][ch], -wv[1][st][ch]);
    }
  }
  return lossp;
}

// Adds the warp's terms to the objective's sums (see CotHeader).
__device__ __forceinline__ void add_block_loss(float lossp, int slot, CotHeader* cot_hdr) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) lossp += __shfl_xor_sync(0xffffffffu, lossp, o);
  if ((threadIdx.x & 31) == 0 && lossp != 0.f) atomicAdd(&cot_hdr->loss[slot], (double)lossp);
}

// One splat, at list position pos, at the thread's two pixels: which blend it, the
// g = dL/d(power) of each stream and -a T, and the pixels' state in front of it.
// Returns the lanes that blend it (0: nothing else is set).
template <int S>
__device__ __forceinline__ uint32_t bwd_visit(BwdPair<S>& pp, const Rec& r, uint32_t pos, bool (&on)[2], float& dx,
                                              f32x2& dy, f32x2 (&gp)[S], f32x2& naT) {
  float power[2], oG[2], na[2], ac[2], om[2];
  f32x2 G;
  splat_gauss2(r, pp.pxc, pp.npy, dx, dy, power, G);
  unpack2(mul2(dup2(r.b.y), G), oG[0], oG[1]);
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const float al = fminf(kAlphaMax, oG[q]);
    on[q] = pos < pp.nc[q] && power[q] <= 0.f && al >= kAlphaMin;
    na[q] = on[q] ? -al : 0.f;
    ac[q] = on[q] && !(oG[q] > kAlphaMax) ? -al : 0.f;  // a capped alpha has zero derivative
  }
  const uint32_t act = __ballot_sync(0xffffffffu, on[0] || on[1]);
  if (!act) return 0u;
  // recover T_i = T_{i+1} / (1 - a); dC/da = c T_i - suffix / (1 - a), and
  // dL/d(power) = a (w . dC/da) per stream.  A pixel that does not blend the
  // splat has a = 0: its state stays as it is and it contributes exact zeros.
  const f32x2 nap = pack2(na[0], na[1]);
  unpack2(add2(dup2(1.f), nap), om[0], om[1]);
  const f32x2 inv = pack2(rcp_approx(om[0]), rcp_approx(om[1]));
  const f32x2 Ti = mul2(pp.T, inv), nac = pack2(ac[0], ac[1]);
  naT = mul2(nap, Ti);
  const float rgb[3] = {r.b.z, r.b.w, r.c.x};
  f32x2 da[3];
#pragma unroll
  for (int ch = 0; ch < 3; ++ch) {
    da[ch] = fma2(dup2(rgb[ch]), Ti, mul2(pp.ns[ch], inv));
    pp.ns[ch] = fma2(dup2(rgb[ch]), naT, pp.ns[ch]);
  }
#pragma unroll
  for (int s = 0; s < S; ++s)
    gp[s] = mul2(fma2(pp.nw[s][2], da[2], fma2(pp.nw[s][0], da[0], mul2(pp.nw[s][1], da[1]))), nac);
  pp.T = Ti;
  return act;
}

// A splat that at most this many lanes blend is added by those lanes, each the row
// of its two pixels, instead of through the sums over the block: part of the fixed
// order too (a quarter of the splats that a block blends; without it raster_bwd_kernel
// takes 1.557 instead of 1.584 ms with no probe, 2.425 instead of 2.378 with one).
constexpr int kSparseLanes = 8;
// The row of a lane's two pixels: their products summed in one fused operation.
template <int S>
__device__ __forceinline__ void lane_row(const f32x2 (&gp)[S], f32x2 naT, const f32x2 (&nw)[S][3], float dx, f32x2 dy,
                                         float* v) {
  float y0, y1, t0, t1;
  unpack2(dy, y0, y1);
  unpack2(naT, t0, t1);
#pragma unroll
  for (int s = 0; s < S; ++s) {
    float g0, g1;
    unpack2(gp[s], g0, g1);
    v[cot_index(S, s, 0)] = fmaf(dx, g1, __fmul_rn(dx, g0));
    v[cot_index(S, s, 1)] = fmaf(y1, g1, __fmul_rn(y0, g0));
    v[cot_index(S, s, 2)] = fmaf(__fmul_rn(dx, dx), g1, __fmul_rn(__fmul_rn(dx, dx), g0));
    v[cot_index(S, s, 3)] = fmaf(__fmul_rn(dx, y1), g1, __fmul_rn(__fmul_rn(dx, y0), g0));
    v[cot_index(S, s, 4)] = fmaf(__fmul_rn(y1, y1), g1, __fmul_rn(__fmul_rn(y0, y0), g0));
    v[cot_index(S, s, 5)] = g0 + g1;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      float w0, w1;
      unpack2(nw[s][ch], w0, w1);
      v[cot_index(S, s, 6 + ch)] = fmaf(w1, t1, __fmul_rn(w0, t0));
    }
  }
#pragma unroll
  for (int k = 9 * S; k < cot_stride(S); ++k) v[k] = 0.f;
}
template <int S>
__device__ __forceinline__ void add_lane(const f32x2 (&gp)[S], f32x2 naT, const f32x2 (&nw)[S][3], float dx, f32x2 dy,
                                         float* __restrict__ row) {
  float v[cot_stride(S)];
  lane_row<S>(gp, naT, nw, dx, dy, v);
#pragma unroll
  for (int k = 0; k < cot_stride(S); k += 4) red_add4(row + k, make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]));
}

// Shared memory of one warp's merge of the partial derivatives of one or two
// streams (see raster_bwd_kernel): kMergeSlots splats' per-pixel values, S + 1 pairs
// per lane, and the negated cotangents -w of the warp's pixels, 3 S pairs per lane.
// A slot holds g of one stream beside -a T, or of two side by side, then -a T.
constexpr int kMergeSlots = 4;
__host__ __device__ constexpr int merge_slot_pairs(int S) { return 32 * (S + 1); }
__host__ __device__ constexpr int merge_w_stride(int S) { return 3 * S; }
__host__ __device__ constexpr int merge_pairs(int S) { return kMergeSlots * merge_slot_pairs(S) + 32 * merge_w_stride(S); }

// The merge of up to kMergeSlots splats of one warp into their cotangent rows.
// A row's entries per stream are the sums over pixels of (dx, dy, dx^2, dx dy,
// dy^2, 1) g, g = dL/d(power), and of (w_r, w_g, w_b) a T.  So a pixel needs to
// hand over only S + 1 values (g of each stream, -a T), not 9 S, and -w stays in
// shared memory.  power = -(A dx^2 + C dy^2)/2 - B dx dy is linear in the conic,
// which the projection's reverse pass applies: dL/dA = -M(dx^2)/2, dL/dB =
// -M(dx dy), dL/dC = -M(dy^2)/2, dL/dmx = -(A M(dx) + B M(dy)), dL/dmy =
// -(B M(dx) + C M(dy)), dL/d(logit) = M(1) (1 - o).
// For a needle those products cancel by the square of its axis ratio, so the
// order of the moments' sums shows in its scale and rotation: it is fixed.  A
// pixel's product is added to that of the pixel four rows below it (one fused
// operation), then rows y and y + 2, rows y and y + 1, columns x and x + 4, x and
// x + 1, x and x + 2; the pixels' g come from the suffix of each colour.  Summing
// whole columns first and keeping one suffix per stream took 1.40 and 2.02 ms
// instead of 1.56 and 2.38 (no probe and one), and moved single entries of the
// gradient by 1e-3 of its root mean square.
// Lanes 8 s .. 8 s + 7 sum splat s, lane & 7 the column of the 8 x 8 block.  A lane
// holds rows (0, 1), (2, 3), (4, 5), (6, 7) as pairs, with two streams first their
// moments, which it writes over the slots' values, then the colours, so that half
// the row is live at a time; lane (s, quad) then adds the eight columns of its four
// entries and issues one float4 reduction.
// smx, smy, sgi: mean and index of the lane's splat; count: slots in use.
template <int S>
__device__ __forceinline__ void merge_slots(f32x2* slots, const f32x2* sw, int count, float wx0, float wy0, float smx,
                                            float smy, uint32_t sgi, float* __restrict__ cot_view) {
  constexpr int NVP = cot_stride(S), NQ = NVP / 4;
  static_assert(S <= 2, "streams");
  constexpr int kA = S == 2 ? 12 : 0, kB = NVP - kA;  // floats of a column's first and second part
  constexpr int kQA = kA / 4, kQB = kB / 4;
  // two float4s 8 floats apart: swapped in columns 4..7, so that eight lanes' are on distinct banks
  auto swizzle = [](int col) { return S == 2 ? col >> 2 : 0; };
  const int lane = threadIdx.x & 31, sl = lane >> 3, x = lane & 7;
  f32x2* my = slots + sl * merge_slot_pairs(S);
  float* rows = reinterpret_cast<float*>(my);
  const float dx = smx - (wx0 + (float)x);
  const f32x2 dx2 = dup2(dx), dxx2 = dup2(dx * dx);
  f32x2 dy[4];  // of rows (0, 1), (2, 3), (4, 5), (6, 7)
#pragma unroll
  for (int r = 0; r < 4; ++r)
    dy[r] = add2(dup2(smy), pack2(-(wy0 + (float)(2 * r)), -(wy0 + (float)(2 * r + 1))));
  // sums over a column of g times (dx, dy, dx^2, dx dy, dy^2, 1); lo, hi: g of rows
  // 0..3 and 4..7
  auto moments = [&](const float (&lo)[4], const float (&hi)[4], float (&m)[6]) {
    const f32x2 g0 = pack2(lo[0], lo[1]), g1 = pack2(lo[2], lo[3]), g2 = pack2(hi[0], hi[1]), g3 = pack2(hi[2], hi[3]);
    auto column = [&](f32x2 k0, f32x2 k1, f32x2 k2, f32x2 k3) {
      return sum2(add2(fma2(k2, g2, mul2(k0, g0)), fma2(k3, g3, mul2(k1, g1))));
    };
    m[0] = column(dx2, dx2, dx2, dx2);
    m[1] = column(dy[0], dy[1], dy[2], dy[3]);
    m[2] = column(dxx2, dxx2, dxx2, dxx2);
    m[3] = column(mul2(dx2, dy[0]), mul2(dx2, dy[1]), mul2(dx2, dy[2]), mul2(dx2, dy[3]));
    m[4] = column(mul2(dy[0], dy[0]), mul2(dy[1], dy[1]), mul2(dy[2], dy[2]), mul2(dy[3], dy[3]));
    m[5] = sum2(add2(add2(g0, g1), add2(g2, g3)));
  };
  __syncwarp();
  if constexpr (S == 2) {  // the moments of two streams
    float lo[2][4], hi[2][4], m[2][6];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(my + 2 * (r * 8 + x));
      unpack2(t.x, lo[0][r], hi[0][r]);
      unpack2(t.y, lo[1][r], hi[1][r]);
    }
    moments(lo[0], hi[0], m[0]);
    moments(lo[1], hi[1], m[1]);
    __syncwarp();  // every lane has read these values
#pragma unroll
    for (int q = 0; q < 3; ++q)
      *reinterpret_cast<float4*>(rows + x * kA + 4 * q) =
          make_float4(m[0][2 * q], m[1][2 * q], m[0][2 * q + 1], m[1][2 * q + 1]);
  }
  {
    float b[kB];
    f32x2 c[3 * S];
#pragma unroll
    for (int k = 0; k < 3 * S; ++k) c[k] = 0ull;
    float lo[4], hi[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int at = r * 8 + x;
      f32x2 naT;
      if constexpr (S == 1) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(my + 2 * at);
        unpack2(t.x, lo[r], hi[r]);
        naT = t.y;
      } else {
        naT = my[64 + at];
      }
      const f32x2* wp = sw + at * merge_w_stride(S);
#pragma unroll
      for (int k = 0; k < 3 * S; k += S) {
        if constexpr (S == 1) {
          c[k] = fma2(naT, wp[k], c[k]);
        } else {
          const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(wp + k);
          c[k] = fma2(naT, t.x, c[k]);
          c[k + 1] = fma2(naT, t.y, c[k + 1]);
        }
      }
    }
#pragma unroll
    for (int s = 0; s < S; ++s)
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) b[cot_index(S, s, 6 + ch) - kA] = sum2(c[3 * s + ch]);
    if constexpr (S == 1) {
      float m[6];
      moments(lo, hi, m);
#pragma unroll
      for (int k = 0; k < 6; ++k) b[cot_index(S, 0, k) - kA] = m[k];
    }
#pragma unroll
    for (int k = 9 * S - kA; k < kB; ++k) b[k] = 0.f;
    __syncwarp();  // every lane has read these values
#pragma unroll
    for (int q = 0; q < kQB; ++q)
      *reinterpret_cast<float4*>(rows + 128 * (S - 1) + x * kB + 4 * (q ^ swizzle(x))) =
          make_float4(b[4 * q], b[4 * q + 1], b[4 * q + 2], b[4 * q + 3]);
  }
  __syncwarp();
  if (x < NQ && sl < count) {  // quad x of the lane's own splat
    const bool first = x < kQA;
    const float* part = rows + (first ? 4 * x : 128 * (S - 1));
    const int stride = first ? kA : kB;
    auto quad = [&](int k) {
      return *reinterpret_cast<const ulonglong2*>(part + k * stride + (first ? 0 : 4 * ((x - kQA) ^ swizzle(k))));
    };
    f32x2 a[2], b[2];
#pragma unroll
    for (int k = 0; k < 4; k += 2) {  // columns 0, 4, 1, 5 and 2, 6, 3, 7
      const ulonglong2 t = quad(k), u = quad(k + 4), v = quad(k + 1), w = quad(k + 5);
      a[k / 2] = add2(add2(t.x, u.x), add2(v.x, w.x));
      b[k / 2] = add2(add2(t.y, u.y), add2(v.y, w.y));
    }
    float4 q;
    unpack2(add2(a[0], a[1]), q.x, q.y);
    unpack2(add2(b[0], b[1]), q.z, q.w);
    if (q.x != 0.f || q.y != 0.f || q.z != 0.f || q.w != 0.f)
      red_add4(cot_view + (size_t)sgi * NVP + 4 * x, q);
  }
  __syncwarp();  // the slots may be written again
}

// A lane's cotangents from shared memory; volatile, so that they are read here and
// not held in registers across a merge, where they would be spilled.
template <int S>
__device__ __forceinline__ void load_w(f32x2 (&nw)[S][3], const f32x2* sw) {
#pragma unroll
  for (int k = 0; k < 3 * S; ++k) {
    if constexpr (S == 1) {
      asm volatile("ld.shared.b64 %0, [%1];" : "=l"(nw[k / 3][k % 3]) : "r"(smem_u32(sw + k)));
    } else if (k % 2 == 0) {
      asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];"
                   : "=l"(nw[k / 3][k % 3]), "=l"(nw[(k + 1) / 3][(k + 1) % 3])
                   : "r"(smem_u32(sw + k)));
    }
  }
}
template <int NU, bool GRAD>
__global__ void __launch_bounds__(32, bwd_min_blocks((GRAD ? 1 : 0) + NU)) raster_bwd_kernel(
    const float4* __restrict__ rec, const uint32_t* __restrict__ vals, const uint32_t* __restrict__ ranges,
    const uint32_t* __restrict__ order, int n_pad, gs_frame fr, int Tx, int T, int log_blocks,
    const float* __restrict__ image, const float* __restrict__ target, const float* __restrict__ final_T,
    const uint32_t* __restrict__ n_contrib, const float* __restrict__ image_tan, int loss_kind, float gn_floor,
    float inv_m, float* __restrict__ cot, bool want_loss, bool loss_per_view, CotHeader* cot_hdr,
    const uint8_t* __restrict__ masks, const int32_t* status) {
  constexpr int S = (GRAD ? 1 : 0) + NU;  // cotangent streams
  constexpr int NVP = cot_stride(S);      // padded row stride of their 9 S values
  static_assert(S <= 2, "three streams take raster_bwd_tile_kernel");
  // the merge slots, then the negated cotangents (see merge_slots), and two
  // buffers of staged records, whose last two words hold the Gaussian index
  // and the list position instead of the record's radius and extents
  __shared__ __align__(16) f32x2 slots[merge_pairs(S)];
  __shared__ Rec buf[2][32];
  f32x2* s_w = slots + kMergeSlots * merge_slot_pairs(S);
  const int lane = threadIdx.x;
  if (blockIdx.x == 0 && lane == 0) cot_hdr->clear_floats = 0;  // the rows are being added into
  const PixelBlock pb = pixel_block(order, fr, Tx, T, log_blocks);
  const int view = pb.view, wb = pb.w, bx0 = pb.x0, by0 = pb.y0;
  if (bx0 >= fr.width || by0 >= fr.height) return;
  const size_t tslot = 2 * ((size_t)view * T + pb.tile);
  const uint32_t start = __ldg(ranges + tslot), len = __ldg(ranges + tslot + 1) - start;
  if (len == 0 && !want_loss) return;
  const float wx0 = (float)bx0 + 0.5f, wy0 = (float)by0 + 0.5f;  // the block's first pixel centre

  BwdPair<S> pp;
  const float lossp = bwd_pixels<NU, GRAD>(pp, bx0, by0, view, len, fr, image, target, final_T, n_contrib, image_tan,
                                           loss_kind, gn_floor, inv_m);
#pragma unroll
  for (int k = 0; k < 3 * S; ++k) s_w[lane * merge_w_stride(S) + k] = pp.nw[k / 3][k % 3];
  if (want_loss) add_block_loss(lossp, loss_per_view ? view : (int)(blockIdx.x % kLossSlots), cot_hdr);
  // list positions this block still needs (n_contrib never exceeds the tile's
  // list); none after a wait that ran out in an earlier call
  const uint32_t nw = min(__reduce_max_sync(0xffffffffu, max(pp.nc[0], pp.nc[1])), len);
  if (__any_sync(0xffffffffu, nw == 0 || (status && (*(volatile const int32_t*)status & GS_FLAG_TIMEOUT)))) return;
  const int n = (int)nw;

  // Chunks of 32 list positions, back to front: each lane reads the index and
  // visibility of one position (the forward pass's mask bit when given, else
  // the footprint test), a chunk ahead of its use.
  int c = (n - 1) >> 5;
  uint32_t gi = 0, gi_next = 0;
  bool see = false, see_next = false;
  auto fetch = [&](int cc, uint32_t& g, bool& v) {
    const int p = cc * 32 + lane;
    v = false;
    if (cc < 0 || p >= n) return;
    g = __ldg(vals + start + (uint32_t)p);
    if (masks) {
      v = ((__ldg(masks + start + (uint32_t)p) >> wb) & 1u) != 0;
    } else {
      const float4* src = rec + 3 * ((size_t)view * n_pad + g);
      Rec r;
      r.a = __ldg(src);
      r.b = __ldg(src + 1);
      r.c = __ldg(src + 2);
      v = block_sees(r, wx0, wy0);
    }
  };
  fetch(c, gi, see);
  fetch(c - 1, gi_next, see_next);
  // Stages the visible splats of the next chunks, as many whole chunks as fit,
  // into b (asynchronous copies, one group per call); returns their count.
  auto fill = [&](Rec* b) {
    int cnt = 0;
    while (c >= 0) {
      const uint32_t bits = __ballot_sync(0xffffffffu, see);
      const int k = __popc(bits);
      if (cnt + k > 32) break;
      if (see) {
        Rec* d = b + cnt + __popc(bits & (0xfffffffeu << lane));  // the last position first
        const float4* src = rec + 3 * ((size_t)view * n_pad + gi);
        cp_async16(&d->a, src);
        cp_async16(&d->b, src + 1);
        cp_async4(&d->c.x, src + 2);
        *reinterpret_cast<uint2*>(&d->c.z) = make_uint2(gi, (uint32_t)(c * 32 + lane));
      }
      cnt += k;
      --c;
      gi = gi_next;
      see = see_next;
      fetch(c - 1, gi_next, see_next);
    }
    cp_async_commit();
    return cnt;
  };

  int used = 0;  // merge slots filled (warp-uniform)
  float smx = 0.f, smy = 0.f;
  uint32_t sgi = 0;
  float* cot_view = cot + (size_t)view * n_pad * NVP;
  int cur = 0, cnt = fill(buf[0]);
  while (cnt > 0) {
    const int cnt_next = fill(buf[cur ^ 1]);
    cp_async_wait_prior();  // all but the newest group: this buffer has landed
    __syncwarp();
    for (int j = 0; j < cnt; ++j) {
      const Rec r = buf[cur][j];
      const uint32_t pos = __float_as_uint(r.c.w);
      bool on[2];
      float dx;
      f32x2 dy, gp[S], naT;
      const uint32_t act = bwd_visit<S>(pp, r, pos, on, dx, dy, gp, naT);
      if (!act) continue;
      if (__popc(act) <= kSparseLanes) {
        if (on[0] || on[1])
          add_lane<S>(gp, naT, pp.nw, dx, dy, cot_view + (size_t)__float_as_uint(r.c.z) * NVP);
        continue;
      }
      // the lane's values of this splat into its merge slot
      f32x2* my = slots + used * merge_slot_pairs(S);
      if constexpr (S == 1) {
        *reinterpret_cast<ulonglong2*>(my + 2 * lane) = make_ulonglong2(gp[0], naT);
      } else {
        *reinterpret_cast<ulonglong2*>(my + 2 * lane) = make_ulonglong2(gp[0], gp[1]);
        my[64 + lane] = naT;
      }
      if ((lane >> 3) == used) {
        smx = r.a.x;
        smy = r.a.y;
        sgi = __float_as_uint(r.c.z);
      }
      if (++used == kMergeSlots) {
        merge_slots<S>(slots, s_w, kMergeSlots, wx0, wy0, smx, smy, sgi, cot_view);
        used = 0;
        // the cotangents again, so that they take no registers during a merge
        load_w<S>(pp.nw, s_w + lane * merge_w_stride(S));
      }
    }
    __syncwarp();  // the buffer may be refilled
    cur ^= 1;
    cnt = cnt_next;
  }
  if (used) merge_slots<S>(slots, s_w, used, wx0, wy0, smx, smy, sgi, cot_view);
}

// ------------------------------------------------ reverse, three streams
// A CTA per tile, a warp per 8 x 8 block.  The warps share a ring of kBwdStages
// batches (one record per thread) that they release one by one: a warp moves on as
// soon as a batch has landed and reads only the splats its block sees; the last warp
// to release a buffer refills it with the batch kBwdStages further on.  So a
// tile's warps walk its list in step, and the order in which their blocks add to a
// splat's row is nearly the same in every run.  With a warp per CTA (raster_bwd_kernel's
// way, 2.83 ms for 1M Gaussians, 8 views of 1080p) near ties between blocks went
// either way: the rotation of a nearly round splat, whose terms cancel to 1e-5 of
// their size, moved by 3e-4 of itself between a request alone and the same one in a
// batch; here by less than a tenth of that in 250 runs.  With one stream or two the
// same comparison moves by a twentieth of that, and the walk in step takes 2.00
// instead of 1.56 ms (no probe) and 2.67 instead of 2.38 (one).
// Sums over the block are a reduce-scatter over the warp (the order of
// merge_slots).  Scalar pixels and 7 CTAs took 3.40 ms; pairs 2.94 at 8 CTAs per SM
// (64 registers, 24 bytes of spills; 7: 3.09, 6: 3.19).  In 16 x 32 tiles 3.17.
constexpr int kBwdStages = 3;
#ifndef GS_BWD_TILE_MB
#define GS_BWD_TILE_MB 8
#endif
// ring header: one mbarrier and one release counter per stage, 16-byte aligned
constexpr size_t kBwdRingHdr = (kBwdStages * (sizeof(uint64_t) + sizeof(uint32_t)) + 15) / 16 * 16;
__host__ __device__ constexpr size_t bwd_ring_bytes(int batch) {
  return kBwdRingHdr + (size_t)kBwdStages * batch * (sizeof(Rec) + sizeof(uint32_t)) +
         ((size_t)kBwdStages * batch + 15) / 16 * 16;  // and the staged block masks, one byte per record
}

// The calling warp fills ring stage s with batch b of the list (use u of the
// ring): its lanes store the Gaussian indices (and, given the forward pass's
// block masks, each record's mask byte) and issue one bulk copy per record,
// then lane 0 records u as the stage's last fill and arms the stage's barrier
// with the byte count.  The copies may complete before that arrival (the
// phase cannot complete while the arrival is pending), and the arrival releases
// the index stores to the warps that wait on the phase.
__device__ __forceinline__ void stage_batch_warp(int s, int u, int b, int batch, uint32_t start, int n, int view,
                                                 int n_pad, const uint32_t* __restrict__ vals,
                                                 const float4* __restrict__ rec, const uint8_t* __restrict__ masks,
                                                 Rec* buf, uint32_t* s_idx, uint8_t* s_bits, uint64_t* full,
                                                 int* fill_use) {
  const int lane = threadIdx.x & 31;
  const int cnt = min(batch, n - b * batch);
  __syncwarp();
  fence_proxy_async();  // the ring slot's earlier reads come before the copies' writes
  for (int q = lane; q < cnt; q += 32) {
    const uint32_t gi = __ldg(vals + start + (uint32_t)(b * batch + q));
    s_idx[s * batch + q] = gi;
    if (masks) s_bits[s * batch + q] = __ldg(masks + start + (uint32_t)(b * batch + q));
    bulk_g2s(&buf[s * batch + q], rec + 3 * ((size_t)view * n_pad + gi), sizeof(Rec), &full[s]);
  }
  __syncwarp();
  if (lane == 0) {
    fill_use[s] = u;
    mbar_arrive_expect_tx(&full[s], (uint32_t)(cnt * (int)sizeof(Rec)));
  }
}

// Warp sums of v[0..31] delivered as quads: afterwards every lane L with
// (L & 3) == 0 holds in q[0..3] the warp-wide sums of v[L .. L+3].  Three
// reduce-scatter stages (lane bits 4, 3, 2) then a butterfly over bits 1, 0.
__device__ __forceinline__ void warp_reduce_quads(float (&v)[32], float (&q)[4]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o >= 4; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float send = up ? v[i] : v[i + o];
      const float keep = up ? v[i + o] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float x = v[i];
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    q[i] = x;
  }
}

template <int NU, bool GRAD, int NT>
__global__ void __launch_bounds__(NT, GS_BWD_TILE_MB * 128 / NT) raster_bwd_tile_kernel(
    const float4* __restrict__ rec, const uint32_t* __restrict__ vals, const uint32_t* __restrict__ ranges,
    const uint32_t* __restrict__ order, int n_pad, gs_frame fr, int Tx, int T, const float* __restrict__ image,
    const float* __restrict__ target, const float* __restrict__ final_T, const uint32_t* __restrict__ n_contrib,
    const float* __restrict__ image_tan, int loss_kind, float gn_floor, float inv_m, float* __restrict__ cot,
    bool want_loss, bool loss_per_view, CotHeader* cot_hdr, const uint8_t* __restrict__ masks, int32_t* status) {
  constexpr int S = (GRAD ? 1 : 0) + NU, NVP = cot_stride(S), K = kBwdStages;
  static_assert(NVP <= 32, "streams");
  extern __shared__ __align__(16) unsigned char smem[];
  const int nthr = blockDim.x, nwarps = nthr >> 5, batch = nthr;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem);                             // K phase barriers
  uint32_t* released = reinterpret_cast<uint32_t*>(smem + K * sizeof(uint64_t));  // K release counters
  Rec* buf = reinterpret_cast<Rec*>(smem + kBwdRingHdr);
  uint32_t* s_idx = reinterpret_cast<uint32_t*>(buf + K * batch);
  uint8_t* s_bits = reinterpret_cast<uint8_t*>(s_idx + K * batch);  // block masks of the staged records
  __shared__ uint32_t s_max;
  __shared__ int s_abort;
  __shared__ int s_fill_use[K];  // ring use of each stage's last fill (-1: none)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // the tile of this block: the heaviest tiles first when an order is given
  const int blk = order ? (int)min(__ldg(order + blockIdx.x), gridDim.x - 1) : (int)blockIdx.x;
  const int view = blk / T, tile = blk - view * T, ty = tile / Tx, tx = tile - ty * Tx, bw = fr.tile_w >> 3;
  const int bx0 = tx * fr.tile_w + (warp % bw) * 8, by0 = ty * fr.tile_h + (warp / bw) * 8;
  const size_t tslot = 2 * ((size_t)view * T + tile);
  const uint32_t start = __ldg(ranges + tslot), len = __ldg(ranges + tslot + 1) - start;
  if (blockIdx.x == 0 && tid == 0) cot_hdr->clear_floats = 0;  // the rows are being added into
  if (len == 0 && !want_loss) return;
  const float wx0 = (float)bx0 + 0.5f, wy0 = (float)by0 + 0.5f;  // the block's first pixel centre
  BwdPair<S> pp;
  const float lossp = bwd_pixels<NU, GRAD>(pp, bx0, by0, view, len, fr, image, target, final_T, n_contrib, image_tan,
                                           loss_kind, gn_floor, inv_m);
  if (want_loss) add_block_loss(lossp, loss_per_view ? view : (int)((blockIdx.x * nwarps + warp) % kLossSlots), cot_hdr);
  if (tid == 0) {
    s_max = 0;
    // a stage wait that ran out in an earlier block: skip the list walk
    s_abort = status ? (*(volatile int32_t*)status & GS_FLAG_TIMEOUT) : 0;
    for (int k = 0; k < K; ++k) {
      mbar_init(&full[k], 1);
      released[k] = 0;
      s_fill_use[k] = -1;
    }
    fence_mbar_init();
  }
  __syncthreads();
  const uint32_t warp_nc = __reduce_max_sync(0xffffffffu, max(pp.nc[0], pp.nc[1]));  // positions this warp needs
  if (lane == 0 && warp_nc) atomicMax(&s_max, warp_nc);
  __syncthreads();
  const int n = s_abort ? 0 : (int)min(s_max, len);  // n_contrib never exceeds the tile's list
  const int nb = (n + batch - 1) / batch;
  // batch b is use u = nb - 1 - b of the ring: stage u % K, its (u / K)-th fill
  for (int u = warp; u < min(K, nb); u += nwarps)
    stage_batch_warp(u, u, nb - 1 - u, batch, start, n, view, n_pad, vals, rec, masks, buf, s_idx, s_bits, full,
                     s_fill_use);
  float* cot_view = cot + (size_t)view * n_pad * NVP;
  bool ok = true;
  for (int u = 0; u < nb; ++u) {
    const int st = u % K, b = nb - 1 - u;
    // every lane waits (bounded) for the stage's phase: each acquires the copies
    // and indices.  A warp whose wait ran out stops at once: it releases no
    // further stage, so no later round completes and nothing is refilled
    // behind it; the other warps run into their own bounded waits.
    const bool landed = mbar_wait_bounded(&full[st], (uint32_t)((u / K) & 1), status);
    ok = __all_sync(0xffffffffu, landed) != 0;
    if (!ok) break;
    const int cnt = min(batch, n - b * batch);
    const Rec* bb = buf + st * batch;
    // the warp walks, back to front, only the splats its block can see (the
    // forward pass's mask bit when given, else the same footprint test) and
    // that lie before its last contributor: one ballot per 32 splats
    const uint8_t* sb = s_bits + st * batch;
    for (int j0 = ((cnt - 1) & ~31); (uint32_t)(b * batch) < warp_nc && j0 >= 0; j0 -= 32) {
      const int jl = j0 + lane;
      uint32_t bits = __ballot_sync(
          0xffffffffu, jl < cnt && (uint32_t)(b * batch + jl) < warp_nc &&
                           (masks ? ((sb[jl] >> warp) & 1u) != 0 : block_sees(bb[jl], wx0, wy0)));
      while (bits) {
        const int hb = 31 - __clz(bits);
        bits &= ~(1u << hb);
        const int j = j0 + hb;
        const Rec r = bb[j];
        bool on[2];
        float dx;
        f32x2 dy, gp[S], naT;
        const uint32_t act = bwd_visit<S>(pp, r, (uint32_t)(b * batch + j), on, dx, dy, gp, naT);
        if (!act) continue;
        float* row = cot_view + (size_t)s_idx[st * batch + j] * NVP;
        if (__popc(act) <= kSparseLanes) {
          if (on[0] || on[1]) add_lane<S>(gp, naT, pp.nw, dx, dy, row);
          continue;
        }
        float v[32], q[4];
        lane_row<S>(gp, naT, pp.nw, dx, dy, v);
#pragma unroll
        for (int k = NVP; k < 32; ++k) v[k] = 0.f;
        warp_reduce_quads(v, q);
        if ((lane & 3) == 0 && lane < NVP && (q[0] != 0.f || q[1] != 0.f || q[2] != 0.f || q[3] != 0.f))
          red_add4(row + lane, make_float4(q[0], q[1], q[2], q[3]));
      }
    }
    // release the stage: the warp's reads of it are ordered before its count,
    // and the last warp to count it, ordered after all counts, refills it
    __syncwarp();
    uint32_t last = 0;
    if (lane == 0) {
      __threadfence_block();
      last = atomicAdd(&released[st], 1u) == (uint32_t)(nwarps - 1);
      if (last) {
        released[st] = 0;
        __threadfence_block();
      }
    }
    last = __shfl_sync(0xffffffffu, last, 0);
    if (last && u + K < nb)
      stage_batch_warp(st, u + K, nb - 1 - (u + K), batch, start, n, view, n_pad, vals, rec, masks, buf, s_idx,
                       s_bits, full, s_fill_use);
  }
  // Drain after a failed wait: a stage is refilled only by a warp that saw its
  // previous fill land, so each stage has at most one fill in flight, its last.
  // One thread per stage waits (bounded) for that fill, so that no bulk copy is
  // still writing into this block's shared memory, or completing on its
  // barrier, when the block exits.  Without a failure every fill has landed.
  if (__syncthreads_or(!ok) && tid < K && s_fill_use[tid] >= 0)
    mbar_wait_bounded(&full[tid], (uint32_t)((s_fill_use[tid] / K) & 1), status);
}

// ------------------------------------------------ projection reverse pass
// Reverse pass of the EWA projection and SH colour for one Gaussian, summed over
// views.  The chain rule, written out:
//   conic = Sigma'^-1:   dA/da = -c^2/det^2, dA/db = 2bc/det^2, dA/dc = 1/det - ac/det^2,
//                        dB/da = bc/det^2, dB/db = -1/det - 2b^2/det^2, dB/dc = ab/det^2,
//                        dC/da = 1/det - ac/det^2, dC/db = 2ab/det^2, dC/dc = -a^2/det^2
//   Sigma' = J Sc J^T:   dSc = J^T Gs J, dJ = 2 Gs J Sc, Gs = [[ga, gb/2], [gb/2, gc]]
//   J(t):                the slope clamp cuts the t_x (t_y) path, J02 = -fx uc / tz
//   Sc = W Sigma W^T:    dSigma = W^T dSc W = (W^T J^T) Gs (J W), summed as the 6
//                        entries of a symmetric matrix from a0 = W^T j0, a1 = W^T j1
//                        (j0, j1 the rows of J);   mean2D(t) and t = W mu + t_w
//   Sigma = M M^T:       dM = 2 dSigma M, M = R diag(s), s = exp(log s)
//   R(q / |q|):          dq = (dqn - qn (qn . dqn)) / |q|
//   colour:              dSH_k = Y_k dc (0 where clamped), dmu += P_perp grad_Y . (sum sh dc) / |d|
// One thread per Gaussian.  A first pass over the views computes each view's
// geometry once and applies it to every cotangent stream (geometric rows); a
// second pass per stream accumulates the SH rows, reusing the clamp decisions
// recorded in the first.  The first pass also keeps the clamped colour
// cotangents of the first kStashViews views in shared memory, so the second
// pass reads them there instead of from L2.  The probe streams are combined into
// hz = (1/nu) sum_k z_k . (G z_k).
constexpr int kPbwdThreads = 128;
// Resident CTAs per SM requested for the projection reverse, by the number of
// cotangent streams.  A fourth CTA with three streams spills and has no room for
// the stash (2.633 against 2.610 ms per call of 1M Gaussians, 8 views, two
// probes); without a probe a fifth CTA: 1.415 against 1.510 ms, with one a fourth:
// 2.050 against 2.093.
__host__ __device__ constexpr int pbwd_min_blocks(int streams) { return streams == 3 ? 3 : streams == 2 ? 4 : 5; }
constexpr int kClampViews = 21;  // clamp bits kept for the first 21 views (3 per view)
constexpr int kStashViews = 8;   // views whose colour cotangents pass 2 reads from shared memory

// dynamic shared memory of the projection reverse: min(V, kStashViews) x 3S x kPbwdThreads floats
__host__ __device__ constexpr size_t pbwd_stash_bytes(int n_views, int streams) {
  return (size_t)(n_views < kStashViews ? n_views : kStashViews) * 3 * streams * kPbwdThreads * sizeof(float);
}

struct ViewGeom {
  float Rc[3][3], tc[3], fx, fy;
};

__device__ __forceinline__ void load_view(const gs_camera* cam, ViewGeom& v) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
#pragma unroll
    for (int b = 0; b < 3; ++b) v.Rc[a][b] = cam->viewmat[4 * a + b];
    v.tc[a] = cam->viewmat[4 * a + 3];
  }
  v.fx = cam->fx;
  v.fy = cam->fy;
}

// Unit view direction and distance from the camera centre to mu.
__device__ __forceinline__ void view_direction(const ViewGeom& v, const float mu[3], float d[3], float& dn) {
  float cp[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) cp[q] = -(v.Rc[0][q] * v.tc[0] + v.Rc[1][q] * v.tc[1] + v.Rc[2][q] * v.tc[2]);
  const float d0 = mu[0] - cp[0], d1 = mu[1] - cp[1], d2 = mu[2] - cp[2];
  dn = sqrtf(d0 * d0 + d1 * d1 + d2 * d2);
  d[0] = d0 / dn;
  d[1] = d1 / dn;
  d[2] = d2 / dn;
}

// One stream's arithmetic, or two probes' at once as packed pairs (1M Gaussians, 8
// views, two probes: the call 2.760 -> 2.610 ms; the loads' latency at 12 warps
// per SM, and 3 TB/s of rows read and cleared, are what is left).
__device__ __forceinline__ float vmul(float a, float b) { return a * b; }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ f32x2 vmul(f32x2 a, float b) { return mul2(a, dup2(b)); }
__device__ __forceinline__ f32x2 vfma(f32x2 a, float b, f32x2 c) { return fma2(a, dup2(b), c); }

// What a view's geometry gives every stream: coefficients of the moments in
// dL/d(conic, mean), of those in dL/d(Sigma', J, t), and W.
struct ViewTerms {
  float cs[2][2];             // dL/d(mx, my) by the moments of dx, dy
  float k2[3][3];             // dL/d(a, b, c) of Sigma' by the moments of dx^2, dx dy, dy^2
  float j00[2], j02[2], j11[2], j12[2];  // dL/dJ by dL/d(a, b) or dL/d(b, c)
  float tx[2], ty[2], tz[6];  // dL/dt by dL/d(mx, my) and dL/dJ
  float a0[3], a1[3];
};
template <class T>
struct GeoSums {
  T mu[3], S[6], ol;  // dL/dmu, the entries (0,0) (0,1) (0,2) (1,1) (1,2) (2,2) of dL/dSigma, dL/d(logit)
};
// mo: the view's moments of (dx, dy, dx^2, dx dy, dy^2, 1) dL/d(power).
// Which product of a sum is rounded before it is added matters: the conic of a
// needle cancels, and two orders differ by as much as the blend's atomics do (a
// scale's entry by 4e-3 of the gradient's root mean square, 9e-4 in this order and
// that of the scalar kernel).
template <class T>
__device__ __forceinline__ void add_view(GeoSums<T>& g, const T (&mo)[6], const ViewTerms& v, const float (&Rc)[3][3],
                                         float one_minus_o) {
  const T cs0 = vfma(mo[0], v.cs[0][0], vmul(mo[1], v.cs[0][1])), cs1 = vfma(mo[0], v.cs[1][0], vmul(mo[1], v.cs[1][1]));
  T q[3];
#pragma unroll
  for (int e = 0; e < 3; ++e) q[e] = vfma(mo[4], v.k2[e][2], vfma(mo[2], v.k2[e][0], vmul(mo[3], v.k2[e][1])));
  const T ga = q[0], gb = q[1], gc = q[2];
  const T gJ00 = vfma(gb, v.j00[1], vmul(ga, v.j00[0])), gJ02 = vfma(gb, v.j02[1], vmul(ga, v.j02[0]));
  const T gJ11 = vfma(gc, v.j11[1], vmul(gb, v.j11[0])), gJ12 = vfma(gc, v.j12[1], vmul(gb, v.j12[0]));
  const T gt0 = vfma(gJ02, v.tx[1], vmul(cs0, v.tx[0])), gt1 = vfma(gJ12, v.ty[1], vmul(cs1, v.ty[0]));
  const T gt2 = vfma(gJ12, v.tz[5], vfma(gJ02, v.tz[4], vfma(gJ11, v.tz[3], vfma(gJ00, v.tz[2],
                     vfma(cs1, v.tz[1], vmul(cs0, v.tz[0]))))));
#pragma unroll
  for (int e = 0; e < 3; ++e) g.mu[e] = vfma(gt2, Rc[2][e], vfma(gt1, Rc[1][e], vfma(gt0, Rc[0][e], g.mu[e])));
  // dSigma += ga a0 a0^T + gb/2 (a0 a1^T + a1 a0^T) + gc a1 a1^T = u a0^T + w a1^T
  constexpr int kSymP[6] = {0, 0, 0, 1, 1, 2}, kSymQ[6] = {0, 1, 2, 1, 2, 2};
  const T hb = vmul(gb, 0.5f);
  T u[3], w[3];
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    u[e] = vfma(ga, v.a0[e], vmul(hb, v.a1[e]));
    w[e] = vfma(hb, v.a0[e], vmul(gc, v.a1[e]));
  }
#pragma unroll
  for (int e = 0; e < 6; ++e) g.S[e] = vfma(w[kSymP[e]], v.a1[kSymQ[e]], vfma(u[kSymP[e]], v.a0[kSymQ[e]], g.S[e]));
  g.ol = vfma(mo[5], one_minus_o, g.ol);
}
// The colour's dependence on mu through the view direction d (distance 1 / idn):
// gdc[ch] the direction gradient of channel ch's colour, gcol its cotangent.
template <class T>
__device__ __forceinline__ void add_view_colour(GeoSums<T>& g, const T (&gcol)[3], const float (&gdc)[3][3],
                                                const float (&d)[3], float idn) {
  T gd[3];
#pragma unroll
  for (int e = 0; e < 3; ++e)
    gd[e] = vfma(gcol[2], gdc[2][e], vfma(gcol[1], gdc[1][e], vmul(gcol[0], gdc[0][e])));
  const T dot = vfma(gd[2], d[2], vfma(gd[1], d[1], vmul(gd[0], d[0])));
#pragma unroll
  for (int e = 0; e < 3; ++e) g.mu[e] = vfma(vfma(dot, -d[e], gd[e]), idn, g.mu[e]);
}

// Column i (of n Gaussians, parameter pitch n_pad) summed over views cams[0..V),
// its cotangent row of view v at (v * cot_pitch + i) * NVP of cot.  Called by
// every thread of a kPbwdThreads block, warp by warp.
template <int DEG, int NU, bool GRAD>
__device__ __forceinline__ void project_bwd_column(const float* __restrict__ P, int n, int n_pad, int i,
                                                   const gs_camera* __restrict__ cams, int V, gs_frame fr,
                                                   float* __restrict__ cot, int cot_pitch, ProbeArg pa,
                                                   float* __restrict__ grad, float* __restrict__ hz) {
  constexpr int S = (GRAD ? 1 : 0) + NU;
  constexpr int NVP = cot_stride(S);
  constexpr int K = (DEG + 1) * (DEG + 1);
  // the block's SH coefficients, staged once and read per view from shared
  // memory (volatile: re-read, not held in registers across the view loops)
  __shared__ __align__(16) float s_sh[3 * K][kPbwdThreads];
  {
    const int lane = threadIdx.x & 31;
    stage_rows<3 * K>(&s_sh[0][threadIdx.x - lane], kPbwdThreads, P + (size_t)kRowSH * n_pad, n_pad, i - lane);
    cp_async_wait_all();
    __syncwarp();
  }
  const volatile float* vsh = &s_sh[0][0];
  auto sh_of = [&](int k, int ch) { return vsh[(3 * k + ch) * kPbwdThreads + threadIdx.x]; };
  // colour cotangents (0 where clamped) of views v < kStashViews, one column per thread
  extern __shared__ float s_pbwd_stash[];
  auto stash = [&](int v, int j) -> float& { return s_pbwd_stash[(v * 3 * S + j) * kPbwdThreads + threadIdx.x]; };
  if (i >= n) return;
  const uint64_t seed = pa.seed;
  const int64_t step = NU > 0 ? probe_step(pa) : 0;
  auto ld = [&](int r) { return __ldg(P + (size_t)r * n_pad + i); };
  const float mu[3] = {ld(0), ld(1), ld(2)};
  float qx = ld(6), qy = ld(7), qz = ld(8), qw = ld(9);
  const float qlen = sqrtf(qx * qx + qy * qy + qz * qz + qw * qw);
  qx /= qlen; qy /= qlen; qz /= qlen; qw /= qlen;
  float R[3][3];
  R[0][0] = 1.f - 2.f * (qy * qy + qz * qz);
  R[0][1] = 2.f * (qx * qy - qw * qz);
  R[0][2] = 2.f * (qx * qz + qw * qy);
  R[1][0] = 2.f * (qx * qy + qw * qz);
  R[1][1] = 1.f - 2.f * (qz * qz + qx * qx);
  R[1][2] = 2.f * (qy * qz - qw * qx);
  R[2][0] = 2.f * (qx * qz - qw * qy);
  R[2][1] = 2.f * (qy * qz + qw * qx);
  R[2][2] = 1.f - 2.f * (qx * qx + qy * qy);
  float sc[3], M[3][3], Sg[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a) sc[a] = expf(ld(3 + a));
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) M[a][b] = R[a][b] * sc[b];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) Sg[a][b] = M[a][0] * M[b][0] + M[a][1] * M[b][1] + M[a][2] * M[b][2];
  const float opac = 1.f / (1.f + expf(-ld(10)));

  // ---- pass 1: geometric rows of every stream
  // (two probes as a pair, the other streams one by one)
  constexpr int kOne = NU == 2 ? S - 2 : S;
  GeoSums<float> g1[kOne > 0 ? kOne : 1] = {};
  GeoSums<f32x2> g2 = {};
  uint64_t clamp_bits = 0;  // bit 3 v + c: colour channel c clamped at 0 in view v (v < kClampViews)
  uint64_t read_rows = 0;   // bit v: the row of view v held a nonzero value (cleared at the end; v >= 64 always)
#pragma unroll 1
  for (int v = 0; v < V; ++v) {
    float c[NVP];
    bool any = false;
    const float4* row4 = reinterpret_cast<const float4*>(cot + ((size_t)v * cot_pitch + i) * NVP);
#pragma unroll
    for (int q = 0; q < NVP / 4; ++q) {
      const float4 x4 = row4[q];
      c[4 * q + 0] = x4.x; c[4 * q + 1] = x4.y; c[4 * q + 2] = x4.z; c[4 * q + 3] = x4.w;
      any = any || x4.x != 0.f || x4.y != 0.f || x4.z != 0.f || x4.w != 0.f;
    }
    if (v < 64) read_rows |= (uint64_t)any << v;
    if (!any) {
      if (v < kStashViews) {
#pragma unroll
        for (int j = 0; j < 3 * S; ++j) stash(v, j) = 0.f;
      }
      continue;
    }
    ViewGeom vg;
    load_view(cams + v, vg);
    const float fx = vg.fx, fy = vg.fy;
    float t[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) t[a] = vg.Rc[a][0] * mu[0] + vg.Rc[a][1] * mu[1] + vg.Rc[a][2] * mu[2] + vg.tc[a];
    float Sc[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      float tmp[3];
#pragma unroll
      for (int b = 0; b < 3; ++b) tmp[b] = vg.Rc[a][0] * Sg[0][b] + vg.Rc[a][1] * Sg[1][b] + vg.Rc[a][2] * Sg[2][b];
#pragma unroll
      for (int b = 0; b < 3; ++b) Sc[a][b] = tmp[0] * vg.Rc[b][0] + tmp[1] * vg.Rc[b][1] + tmp[2] * vg.Rc[b][2];
    }
    const float limx = kSlopeClamp * 0.5f * (float)fr.width / fx;
    const float limy = kSlopeClamp * 0.5f * (float)fr.height / fy;
    const float itz = 1.f / t[2];
    const float u = t[0] * itz, vv = t[1] * itz;
    const bool clx = u < -limx || u > limx, cly = vv < -limy || vv > limy;
    const float uc = fminf(fmaxf(u, -limx), limx), vc = fminf(fmaxf(vv, -limy), limy);
    const float J00 = fx * itz, J02 = -fx * uc * itz, J11 = fy * itz, J12 = -fy * vc * itz;
    const float a = J00 * J00 * Sc[0][0] + 2.f * J00 * J02 * Sc[0][2] + J02 * J02 * Sc[2][2] + kDilation;
    const float bb = J00 * J11 * Sc[0][1] + J00 * J12 * Sc[0][2] + J02 * J11 * Sc[1][2] + J02 * J12 * Sc[2][2];
    const float cc = J11 * J11 * Sc[1][1] + 2.f * J11 * J12 * Sc[1][2] + J12 * J12 * Sc[2][2] + kDilation;
    const float det = a * cc - bb * bb;
    const float idet = 1.f / det, id2 = idet * idet;
    // rows of J taken back to world axes: a0 = W^T j0, a1 = W^T j1
    float a0[3], a1[3];
#pragma unroll
    for (int p2 = 0; p2 < 3; ++p2) {
      a0[p2] = vg.Rc[0][p2] * J00 + vg.Rc[2][p2] * J02;
      a1[p2] = vg.Rc[1][p2] * J11 + vg.Rc[2][p2] * J12;
    }
    float JS0[3], JS1[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      JS0[q] = J00 * Sc[0][q] + J02 * Sc[2][q];
      JS1[q] = J11 * Sc[1][q] + J12 * Sc[2][q];
    }
    const float itz2 = itz * itz, itz3 = itz2 * itz;
    // conic of this view, to turn the blend's moments into dL/d(mx, my, A, B, C)
    const float cA = cc * idet, cB = -bb * idet, cCc = a * idet, dac = idet - a * cc * id2;
    const ViewTerms vt = {
        {{-cA, -cB}, {-cB, -cCc}},
        {{0.5f * cc * cc * id2, -bb * cc * id2, -0.5f * dac},
         {-bb * cc * id2, idet + 2.f * bb * bb * id2, -a * bb * id2},
         {-0.5f * dac, -a * bb * id2, 0.5f * a * a * id2}},
        {2.f * JS0[0], JS1[0]}, {2.f * JS0[2], JS1[2]}, {JS0[1], 2.f * JS1[1]}, {JS0[2], 2.f * JS1[2]},
        {J00, clx ? 0.f : -fx * itz2}, {J11, cly ? 0.f : -fy * itz2},
        {-fx * t[0] * itz2, -fy * t[1] * itz2, -fx * itz2, -fy * itz2, clx ? fx * uc * itz2 : 2.f * fx * t[0] * itz3,
         cly ? fy * vc * itz2 : 2.f * fy * t[1] * itz3},
        {a0[0], a0[1], a0[2]}, {a1[0], a1[1], a1[2]}};
#pragma unroll
    for (int st = 0; st < kOne; ++st) {
      float mo[6];
#pragma unroll
      for (int k = 0; k < 6; ++k) mo[k] = c[cot_index(S, st, k)];
      add_view(g1[st], mo, vt, vg.Rc, 1.f - opac);
    }
    if constexpr (NU == 2) {
      f32x2 mo[6];
#pragma unroll
      for (int k = 0; k < 6; ++k) mo[k] = pack2(c[2 * k], c[2 * k + 1]);
      add_view(g2, mo, vt, vg.Rc, 1.f - opac);
    }
    // colour: clamp decisions, and the dependence of colour on mu through the view direction
    float d[3], dn;
    view_direction(vg, mu, d, dn);
    float Y[K];
    sh_basis<DEG>(d[0], d[1], d[2], Y);
    // per channel: the raw colour (its clamp decision) and, for the colour's
    // dependence on mu, the direction gradient of sum_k sh_k Y_k; the SH
    // coefficients come from the staged copy instead of registers
    bool clamped[3];
    float gdc[3][3];
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      float shc[K];
#pragma unroll
      for (int k = 0; k < K; ++k) shc[k] = sh_of(k, ch);
      float raw = 0.5f;
#pragma unroll
      for (int k = 0; k < K; ++k) raw += Y[k] * shc[k];
      clamped[ch] = raw < 0.f;
      if (clamped[ch] && v < kClampViews) clamp_bits |= 1ull << (3 * v + ch);
      if constexpr (DEG > 0) sh_basis_grad<DEG>(d[0], d[1], d[2], shc, gdc[ch]);
    }
    if (v < kStashViews) {
#pragma unroll
      for (int st = 0; st < S; ++st)
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) stash(v, 3 * st + ch) = clamped[ch] ? 0.f : c[cot_index(S, st, 6 + ch)];
    }
    if constexpr (DEG > 0) {
      const float idn = 1.f / dn;
#pragma unroll
      for (int st = 0; st < kOne; ++st) {
        float gcol[3];
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) gcol[ch] = clamped[ch] ? 0.f : c[cot_index(S, st, 6 + ch)];
        add_view_colour(g1[st], gcol, gdc, d, idn);
      }
      if constexpr (NU == 2) {
        f32x2 gcol[3];
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) gcol[ch] = clamped[ch] ? 0ull : pack2(c[12 + 2 * ch], c[13 + 2 * ch]);
        add_view_colour(g2, gcol, gdc, d, idn);
      }
    }
  }

  // ---- geometric rows: Sigma = M M^T, M = R diag(s); R(q / |q|)
  const float qn[4] = {qx, qy, qz, qw};
  float hz_geo[kRowSH];
#pragma unroll
  for (int r = 0; r < kRowSH; ++r) hz_geo[r] = 0.f;
  const float inv_nu = NU > 0 ? 1.f / (float)NU : 0.f;
#pragma unroll
  for (int st = 0; st < S; ++st) {
    GeoSums<float> g;
    if (st < kOne) {
      g = g1[st < kOne ? st : 0];
    } else {
      auto half = [&](f32x2 v) {
        float lo, hi;
        unpack2(v, lo, hi);
        return st - kOne ? hi : lo;
      };
#pragma unroll
      for (int e = 0; e < 3; ++e) g.mu[e] = half(g2.mu[e]);
#pragma unroll
      for (int e = 0; e < 6; ++e) g.S[e] = half(g2.S[e]);
      g.ol = half(g2.ol);
    }
    const float gS[3][3] = {{g.S[0], g.S[1], g.S[2]}, {g.S[1], g.S[3], g.S[4]}, {g.S[2], g.S[4], g.S[5]}};
    float gM[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) gM[a][b] = 2.f * (gS[a][0] * M[0][b] + gS[a][1] * M[1][b] + gS[a][2] * M[2][b]);
    float rowv[kRowSH];
    float gR[3][3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      rowv[3 + b] = (gM[0][b] * R[0][b] + gM[1][b] * R[1][b] + gM[2][b] * R[2][b]) * sc[b];
#pragma unroll
      for (int a = 0; a < 3; ++a) gR[a][b] = gM[a][b] * sc[b];
    }
    const float x = qx, y = qy, z = qz, ww = qw;
    float gq[4];
    gq[0] = 2.f * y * gR[0][1] + 2.f * z * gR[0][2] + 2.f * y * gR[1][0] - 4.f * x * gR[1][1] - 2.f * ww * gR[1][2] +
            2.f * z * gR[2][0] + 2.f * ww * gR[2][1] - 4.f * x * gR[2][2];
    gq[1] = -4.f * y * gR[0][0] + 2.f * x * gR[0][1] + 2.f * ww * gR[0][2] + 2.f * x * gR[1][0] + 2.f * z * gR[1][2] -
            2.f * ww * gR[2][0] + 2.f * z * gR[2][1] - 4.f * y * gR[2][2];
    gq[2] = -4.f * z * gR[0][0] - 2.f * ww * gR[0][1] + 2.f * x * gR[0][2] + 2.f * ww * gR[1][0] - 4.f * z * gR[1][1] +
            2.f * y * gR[1][2] + 2.f * x * gR[2][0] + 2.f * y * gR[2][1];
    gq[3] = -2.f * z * gR[0][1] + 2.f * y * gR[0][2] + 2.f * z * gR[1][0] - 2.f * x * gR[1][2] - 2.f * y * gR[2][0] +
            2.f * x * gR[2][1];
    const float qd = gq[0] * x + gq[1] * y + gq[2] * z + gq[3] * ww;
#pragma unroll
    for (int a = 0; a < 3; ++a) rowv[a] = g.mu[a];
#pragma unroll
    for (int cq = 0; cq < 4; ++cq) rowv[6 + cq] = (gq[cq] - qn[cq] * qd) / qlen;
    rowv[10] = g.ol;
    if (GRAD && st == 0) {
#pragma unroll
      for (int r = 0; r < kRowSH; ++r) grad[(size_t)r * n_pad + i] = rowv[r];
    } else {
      const int k = st - (GRAD ? 1 : 0);
      const uint64_t zneg = probe_signs(seed, step, k, (uint64_t)i, kRowSH + 3 * K);
#pragma unroll
      for (int r = 0; r < kRowSH; ++r) {
        const bool neg = (zneg >> r) & 1ull;
        hz_geo[r] += (neg ? -rowv[r] : rowv[r]) * inv_nu;
      }
    }
  }
  if constexpr (NU > 0) {
#pragma unroll
    for (int r = 0; r < kRowSH; ++r) hz[(size_t)r * n_pad + i] = hz_geo[r];
  }

  // ---- pass 2: SH rows, dSH_k = sum_v Y_k(d_v) dc_v.  The gradient stream
  // alone; two probe streams in one walk over the views: z1 . G1 + z2 . G2 =
  // z1 . (G1 + (z1 z2) G2), so the sums of Y (dc1 + dc2) and Y (dc1 - dc2) are
  // kept and each row's sign product picks one.
  // colour cotangent of view v, stream st (clamps applied for v < kStashViews)
  auto colour_cot = [&](int v, int st, float (&g)[3]) {
    if (v < kStashViews) {
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) g[ch] = stash(v, 3 * st + ch);
    } else {
      const float* cv = cot + ((size_t)v * cot_pitch + i) * NVP;
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) g[ch] = cv[cot_index(S, st, 6 + ch)];
    }
  };
  // basis of view v and its clamp decisions (true: channel clamped at 0)
  auto view_basis = [&](int v, float (&Y)[K], bool (&cl)[3]) {
    ViewGeom vg;
    load_view(cams + v, vg);
    float d[3], dn;
    view_direction(vg, mu, d, dn);
    sh_basis<DEG>(d[0], d[1], d[2], Y);
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      if (v < kStashViews) {
        cl[ch] = false;  // already applied
      } else if (v < kClampViews) {
        cl[ch] = (clamp_bits >> (3 * v + ch)) & 1ull;
      } else {
        float raw = 0.5f;
#pragma unroll
        for (int k = 0; k < K; ++k) raw += Y[k] * sh_of(k, ch);
        cl[ch] = raw < 0.f;
      }
    }
  };
  auto sh_rows_single = [&](int st) {
    float g_sh[K][3];
#pragma unroll
    for (int k = 0; k < K; ++k) g_sh[k][0] = g_sh[k][1] = g_sh[k][2] = 0.f;
#pragma unroll 1
    for (int v = 0; v < V; ++v) {
      float gcol[3];
      colour_cot(v, st, gcol);
      if (gcol[0] == 0.f && gcol[1] == 0.f && gcol[2] == 0.f) continue;
      float Y[K];
      bool cl[3];
      view_basis(v, Y, cl);
#pragma unroll
      for (int ch = 0; ch < 3; ++ch)
        if (cl[ch]) gcol[ch] = 0.f;
#pragma unroll
      for (int k = 0; k < K; ++k)
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) g_sh[k][ch] += Y[k] * gcol[ch];
    }
    if (GRAD && st == 0) {
#pragma unroll
      for (int k = 0; k < K; ++k)
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) grad[(size_t)(kRowSH + 3 * k + ch) * n_pad + i] = g_sh[k][ch];
    } else {
      const uint64_t zneg = probe_signs(seed, step, st - (GRAD ? 1 : 0), (uint64_t)i, kRowSH + 3 * K);
#pragma unroll
      for (int k = 0; k < K; ++k)
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
          const int r = kRowSH + 3 * k + ch;
          const bool neg = (zneg >> r) & 1ull;
          hz[(size_t)r * n_pad + i] = (neg ? -g_sh[k][ch] : g_sh[k][ch]) * inv_nu;
        }
    }
  };
  if constexpr (GRAD) sh_rows_single(0);
  if constexpr (NU == 1) sh_rows_single(GRAD ? 1 : 0);
  if constexpr (NU == 2) {
    constexpr int s1 = GRAD ? 1 : 0, s2 = s1 + 1;
    f32x2 spm[K][3];  // sums of Y (dc1 + dc2) and of Y (dc1 - dc2)
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) spm[k][ch] = 0ull;
#pragma unroll 1
    for (int v = 0; v < V; ++v) {
      float g1[3], g2[3];
      colour_cot(v, s1, g1);
      colour_cot(v, s2, g2);
      if (g1[0] == 0.f && g1[1] == 0.f && g1[2] == 0.f && g2[0] == 0.f && g2[1] == 0.f && g2[2] == 0.f) continue;
      float Y[K];
      bool cl[3];
      view_basis(v, Y, cl);
      f32x2 gpm[3];
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) gpm[ch] = cl[ch] ? 0ull : pack2(g1[ch] + g2[ch], g1[ch] - g2[ch]);
#pragma unroll
      for (int k = 0; k < K; ++k)
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) spm[k][ch] = vfma(gpm[ch], Y[k], spm[k][ch]);
    }
    const uint64_t zn1 = probe_signs(seed, step, 0, (uint64_t)i, kRowSH + 3 * K);
    const uint64_t zn2 = probe_signs(seed, step, 1, (uint64_t)i, kRowSH + 3 * K);
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) {
        const int r = kRowSH + 3 * k + ch;
        const bool n1 = (zn1 >> r) & 1ull, same = ((zn1 ^ zn2) >> r & 1ull) == 0;
        float sum, diff;
        unpack2(spm[k][ch], sum, diff);
        const float val = same ? sum : diff;
        hz[(size_t)r * n_pad + i] = (n1 ? -val : val) * inv_nu;
      }
  }
  // leave the rows read above zero for the next call (CotHeader)
  for (int v = 0; v < V; ++v) {
    if (v < 64 && !((read_rows >> v) & 1ull)) continue;
    float4* row4 = reinterpret_cast<float4*>(cot + ((size_t)v * cot_pitch + i) * NVP);
#pragma unroll
    for (int q = 0; q < NVP / 4; ++q) row4[q] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

template <int DEG, int NU, bool GRAD>
__global__ void __launch_bounds__(kPbwdThreads, pbwd_min_blocks((GRAD ? 1 : 0) + NU)) project_bwd_kernel(const float* __restrict__ P, int n, int n_pad,
                                                  const gs_camera* __restrict__ cams, gs_frame fr,
                                                  float* __restrict__ cot, ProbeArg pa, float* __restrict__ grad,
                                                  float* __restrict__ hz, CotHeader* cot_hdr, uint64_t cot_floats,
                                                  float* loss_out) {
  const int i = blockIdx.x * kPbwdThreads + threadIdx.x;
  project_bwd_column<DEG, NU, GRAD>(P, n, n_pad, i, cams, fr.n_views, fr, cot, n_pad, pa, grad, hz);
  cot_mark_clear(cot_hdr, cot_floats, loss_out, 0);
}

// A batch: item b's share of the grid takes its columns through the reverse of
// its own projection, from its slot of the cotangents (pitch cot_pitch), with
// its own probe step, into its own gradient and Hutchinson rows.
template <int DEG, int NU, bool GRAD>
__global__ void __launch_bounds__(kPbwdThreads, pbwd_min_blocks((GRAD ? 1 : 0) + NU)) project_bwd_batch_kernel(BatchArg ba, gs_frame fr, float* __restrict__ cot,
                                                        int cot_pitch, ProbeArg pa, CotHeader* cot_hdr,
                                                        uint64_t cot_floats, float* loss_out) {
  constexpr int NVP = cot_stride((GRAD ? 1 : 0) + NU);
  const int b = batch_item(ba, (int)blockIdx.x);
  const int i = ((int)blockIdx.x - ba.first_block[b]) * kPbwdThreads + threadIdx.x;
  pa.t = ba.t[b];
  pa.t_dev = nullptr;
  project_bwd_column<DEG, NU, GRAD>(ba.P[b], ba.n[b], ba.n_pad[b], i, ba.cam[b], 1, fr,
                                    cot + (size_t)b * cot_pitch * NVP, cot_pitch, pa, ba.grad[b], ba.hz[b]);
  cot_mark_clear(cot_hdr, cot_floats, loss_out, ba.n_items);
}

// ------------------------------------------------------------------ host side
struct TileGrid {
  int Tx, Ty, T;
};
TileGrid tile_grid(gs_frame fr) {
  TileGrid g;
  g.Tx = (fr.width + fr.tile_w - 1) / fr.tile_w;
  g.Ty = (fr.height + fr.tile_h - 1) / fr.tile_h;
  g.T = g.Tx * g.Ty;
  return g;
}

int log_tile_blocks(gs_frame fr) {  // 8 x 8 blocks per tile, a power of two
  int b = 0;
  while ((64 << b) < fr.tile_w * fr.tile_h) ++b;
  return b;
}

template <class F>
cudaError_t allow_smem(F* f, size_t bytes) {
  return cudaFuncSetAttribute((const void*)f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Clears the masks and cuts them into whole words (see MaskWords).
bool clear_masks(uint8_t* p, size_t bytes, MaskWords& m, cudaStream_t st) {
  if (!p) return true;
  m.head = (uint32_t)((uintptr_t)p & 3);
  const size_t lead = (4 - m.head) & 3, tail = (m.head + bytes) & 3;
  if (bytes < 8 || bytes > 0xfffffff0u)  // no whole word, or byte numbers that 32 bits do not hold
    return cudaMemsetAsync(p, 0xff, bytes, st) == cudaSuccess;
  m.words = reinterpret_cast<uint32_t*>(p - m.head);
  m.first = m.head ? 1 : 0;
  m.count = (uint32_t)((m.head + bytes) >> 2) - m.first;
  return cudaMemsetAsync(p, 0, bytes, st) == cudaSuccess &&
         (!lead || cudaMemsetAsync(p, 0xff, lead, st) == cudaSuccess) &&
         (!tail || cudaMemsetAsync(p + bytes - tail, 0xff, tail, st) == cudaSuccess);
}

template <int NU>
gs_status launch_fwd(const gs_projected* proj, const gs_sorted* sorted, int n_pad, gs_frame fr, float* image,
                     float* final_T, uint32_t* n_contrib, float* image_tan, cudaStream_t st) {
  const TileGrid g = tile_grid(fr);
  MaskWords masks{};
  if (!clear_masks(sorted->masks, sorted->capacity, masks, st)) return check_launch("gs_raster_fwd: memset");
  const int log_blocks = log_tile_blocks(fr);
  const unsigned blocks = (unsigned)((size_t)fr.n_views * g.T << log_blocks);
  raster_fwd_kernel<NU><<<blocks, 32, 0, st>>>(
      reinterpret_cast<const float4*>(proj->rec), reinterpret_cast<const float4*>(proj->tangent), sorted->vals,
      sorted->ranges, sorted->order, n_pad, fr, g.Tx, g.T, log_blocks, image, final_T, n_contrib, image_tan,
      masks);
  return check_launch("gs_raster_fwd");
}

size_t bwd_cot_floats(int32_t n_pad, gs_frame fr, int streams) {
  return (size_t)fr.n_views * n_pad * cot_stride(streams);
}

// The reverse call's workspace: its header, the rows, and how many floats of
// them this call uses.
struct CotWs {
  CotHeader* hdr;
  float* cot;
  uint64_t floats;
};

// Point ws at the workspace and have the rows zero before the blend: the
// prepare kernel clears them unless the header says they already are.
cudaError_t cot_prepare(void* workspace, uint64_t floats, CotWs& ws, cudaStream_t st) {
  ws.hdr = reinterpret_cast<CotHeader*>(workspace);
  ws.cot = reinterpret_cast<float*>(reinterpret_cast<char*>(workspace) + kCotHeaderBytes);
  ws.floats = floats;
  const size_t n4 = floats / 4;  // rows are whole float4s
  const unsigned blocks = (unsigned)std::max<size_t>(1, std::min<size_t>((n4 + 255) / 256, 152 * 8));
  cot_prepare_kernel<<<blocks, 256, 0, st>>>(ws.hdr, reinterpret_cast<float4*>(ws.cot), n4);
  return cudaGetLastError();
}

template <int DEG, int NU, bool GRAD>
void launch_pbwd(const gs_params* x, const gs_camera* cams, gs_frame fr, CotWs ws, const gs_probe* probe,
                 float* grad, float* hz, float* loss_out, cudaStream_t st) {
  constexpr int S = (GRAD ? 1 : 0) + NU;
  const size_t smem = pbwd_stash_bytes(fr.n_views, S);
  static size_t attr = 0;
  if (smem > attr) {
    if (allow_smem(project_bwd_kernel<DEG, NU, GRAD>, smem) != cudaSuccess) return;  // the caller reports the error
    attr = smem;
  }
  const dim3 pg((x->n + kPbwdThreads - 1) / kPbwdThreads), pb(kPbwdThreads);
  project_bwd_kernel<DEG, NU, GRAD><<<pg, pb, smem, st>>>(x->data, x->n, x->n_pad, cams, fr, ws.cot,
                                                          probe_arg(probe), grad, hz, ws.hdr, ws.floats, loss_out);
}

// The reverse blend over the frame, then the projection's reverse pass: of the
// one scene x (ba NULL), or of each batch item from its slot (ba given: records
// and cotangents at pitch n_pad, each view its own objective, m = 3 H W).
template <int NU, bool GRAD>
void launch_bwd_kernels(const gs_params* x, const BatchArg* ba, int n_pad, int deg, const gs_camera* cams,
                        const gs_projected* proj, const gs_sorted* sorted, gs_frame fr, const float* image,
                        const float* target, const float* final_T, const uint32_t* n_contrib, const float* image_tan,
                        const gs_probe* probe, gs_loss loss, float* grad, float* hz, float* loss_out, CotWs ws,
                        int32_t* status, cudaStream_t st) {
  const TileGrid g = tile_grid(fr);
  const double views_per_objective = ba ? 1.0 : (double)fr.n_views;
  const float inv_m = (float)(1.0 / (3.0 * (double)fr.width * fr.height * views_per_objective));
  const float4* rec = reinterpret_cast<const float4*>(proj->rec);
  if constexpr (GRAD && NU == 2) {
    const int nthr = fr.tile_w * fr.tile_h / kPixPerThread;
    auto* kern = nthr <= 128 ? raster_bwd_tile_kernel<NU, GRAD, 128> : raster_bwd_tile_kernel<NU, GRAD, 256>;
    kern<<<(unsigned)((size_t)fr.n_views * g.T), nthr, bwd_ring_bytes(nthr), st>>>(
        rec, sorted->vals, sorted->ranges, sorted->order, n_pad, fr, g.Tx, g.T, image, target, final_T, n_contrib,
        image_tan, loss.kind, loss.gn_floor, inv_m, ws.cot, loss_out != nullptr, ba != nullptr, ws.hdr, sorted->masks,
        status);
  } else {
    const int log_blocks = log_tile_blocks(fr);
    const unsigned blocks = (unsigned)((size_t)fr.n_views * g.T << log_blocks);
    raster_bwd_kernel<NU, GRAD><<<blocks, 32, 0, st>>>(
        rec, sorted->vals, sorted->ranges, sorted->order, n_pad, fr, g.Tx, g.T, log_blocks, image, target, final_T,
        n_contrib, image_tan, loss.kind, loss.gn_floor, inv_m, ws.cot, loss_out != nullptr, ba != nullptr, ws.hdr,
        sorted->masks, status);
  }
  if (loss_out && (ba ? ba->first_block[ba->n_items] : x->n) == 0)
    add_loss_kernel<<<1, 1, 0, st>>>(ws.hdr, loss_out, ba ? ba->n_items : 0);
  if (ba) {
    if (ba->first_block[ba->n_items] == 0) return;
    constexpr int S = (GRAD ? 1 : 0) + NU;
    const size_t sm = pbwd_stash_bytes(1, S);
    const ProbeArg pa = probe_arg(probe);
    const dim3 grid(ba->first_block[ba->n_items]), blk(kPbwdThreads);
#define GS_PBWD_BATCH(D)                                                                           \
  do {                                                                                             \
    static size_t battr = 0;                                                                       \
    if (sm > battr) {                                                                              \
      if (allow_smem(project_bwd_batch_kernel<D, NU, GRAD>, sm) != cudaSuccess) return;            \
      battr = sm;                                                                                  \
    }                                                                                              \
    project_bwd_batch_kernel<D, NU, GRAD><<<grid, blk, sm, st>>>(*ba, fr, ws.cot, n_pad, pa, ws.hdr, \
                                                                 ws.floats, loss_out);             \
  } while (0)
    switch (deg) {
      case 0: GS_PBWD_BATCH(0); break;
      case 1: GS_PBWD_BATCH(1); break;
      case 2: GS_PBWD_BATCH(2); break;
      default: GS_PBWD_BATCH(3); break;
    }
#undef GS_PBWD_BATCH
    return;
  }
  if (x->n == 0) return;
  switch (x->sh_degree) {
    case 0: launch_pbwd<0, NU, GRAD>(x, cams, fr, ws, probe, grad, hz, loss_out, st); break;
    case 1: launch_pbwd<1, NU, GRAD>(x, cams, fr, ws, probe, grad, hz, loss_out, st); break;
    case 2: launch_pbwd<2, NU, GRAD>(x, cams, fr, ws, probe, grad, hz, loss_out, st); break;
    default: launch_pbwd<3, NU, GRAD>(x, cams, fr, ws, probe, grad, hz, loss_out, st); break;
  }
}

// The kernels of one reverse call for the stream counts: the gradient stream
// (want_grad) and nu probe streams.
void launch_bwd_streams(bool want_grad, int nu, const gs_params* x, const BatchArg* ba, int n_pad, int deg,
                        const gs_camera* cams, const gs_projected* proj, const gs_sorted* sorted, gs_frame frame,
                        const float* image, const float* target, const float* final_T, const uint32_t* n_contrib,
                        const float* image_tangent, const gs_probe* probe, gs_loss loss, float* gptr, float* hptr,
                        float* loss_out, CotWs ws, int32_t* status, cudaStream_t st) {
#define GS_BWD_ARGS x, ba, n_pad, deg, cams, proj, sorted, frame, image, target, final_T, n_contrib, image_tangent, \
                    probe, loss, gptr, hptr, loss_out, ws, status, st
  if (want_grad) {
    if (nu == 0) launch_bwd_kernels<0, true>(GS_BWD_ARGS);
    else if (nu == 1) launch_bwd_kernels<1, true>(GS_BWD_ARGS);
    else launch_bwd_kernels<2, true>(GS_BWD_ARGS);
  } else {
    if (nu == 1) launch_bwd_kernels<1, false>(GS_BWD_ARGS);
    else launch_bwd_kernels<2, false>(GS_BWD_ARGS);
  }
#undef GS_BWD_ARGS
}

gs_status run_bwd(bool want_grad, const gs_params* x, const gs_camera* cams, gs_frame frame, const gs_projected* proj,
                  const gs_sorted* sorted, const float* image, const float* target, const float* final_T,
                  const uint32_t* n_contrib, const float* image_tangent, const gs_probe* probe, gs_loss loss,
                  gs_params* grad, gs_params* hz, float* loss_out, void* workspace, size_t workspace_bytes,
                  int32_t* status, void* stream, const char* name) {
  GS_REQUIRE(x && cams && proj && sorted && image && target && final_T && n_contrib, "%s: null argument", name);
  GS_REQUIRE(proj->rec && sorted->vals && sorted->ranges && x->data, "%s: null device buffer", name);
  GS_REQUIRE(on_16_bytes(proj->rec), "%s: rec must be 16-byte aligned", name);
  GS_REQUIRE(frame_ok(frame), "%s: bad frame", name);
  GS_REQUIRE(x->n >= 0 && x->n_pad >= x->n && x->n_pad % 4 == 0, "%s: bad n/n_pad", name);
  GS_REQUIRE(loss.kind == GS_LOSS_L1 || loss.kind == GS_LOSS_L2 || loss.kind == GS_LOSS_COTANGENT ||
                 loss.kind == GS_LOSS_WEIGHTED,
             "%s: bad loss kind %d", name, loss.kind);
  const bool given = loss.kind == GS_LOSS_COTANGENT;
  const int nu = ((image_tangent || given) && probe) ? probe->nu : 0;
  GS_REQUIRE(loss.kind != GS_LOSS_WEIGHTED || nu == 0 || image_tangent, "%s: weighted loss needs image_tangent",
             name);
  if (nu < 0 || nu > 2 || x->sh_degree < 0 || x->sh_degree > 3) {
    set_error("%s: unsupported nu=%d sh_degree=%d", name, nu, x->sh_degree);
    return GS_ERR_UNSUPPORTED;
  }
  GS_REQUIRE(want_grad || nu > 0, "%s: needs image_tangent and a probe with nu >= 1", name);
  GS_REQUIRE(!want_grad || (grad && grad->data), "%s: null grad", name);
  GS_REQUIRE(nu == 0 || (hz && hz->data), "%s: probes given but hz is NULL", name);
  auto same = [&](const gs_params* p) { return !p || (p->n == x->n && p->n_pad == x->n_pad && p->sh_degree == x->sh_degree); };
  GS_REQUIRE(same(grad) && same(hz), "%s: grad/hz layout differs from x", name);
  const int streams = (want_grad ? 1 : 0) + nu;
  const size_t floats = bwd_cot_floats(x->n_pad, frame, streams);
  const size_t need = kCotHeaderBytes + floats * sizeof(float);
  GS_REQUIRE(workspace && workspace_bytes >= need, "%s: workspace needs %zu bytes, got %zu", name, need,
             workspace_bytes);
  GS_REQUIRE(((uintptr_t)workspace & 15) == 0, "%s: workspace must be 16-byte aligned", name);
  cudaStream_t st = (cudaStream_t)stream;
  CotWs ws;
  if (cot_prepare(workspace, floats, ws, st) != cudaSuccess) return check_launch(name);
  float* gptr = want_grad ? grad->data : nullptr;
  float* hptr = nu ? hz->data : nullptr;
  launch_bwd_streams(want_grad, nu, x, nullptr, x->n_pad, x->sh_degree, cams, proj, sorted, frame, image, target,
                     final_T, n_contrib, image_tangent, probe, loss, gptr, hptr, loss_out, ws, status, st);
  return check_launch(name);
}

}  // namespace
}  // namespace gs

extern "C" gs_status gs_raster_fwd(const gs_projected* proj, const gs_sorted* sorted, int32_t n_pad, gs_frame frame,
                                   const gs_probe* probe, float* image, float* final_T, uint32_t* n_contrib,
                                   float* image_tangent, int32_t* status, void* stream) {
  using namespace gs;
  (void)status;
  GS_REQUIRE(proj && sorted && proj->rec && sorted->vals && sorted->ranges, "gs_raster_fwd: null argument");
  GS_REQUIRE(image && final_T && n_contrib, "gs_raster_fwd: null output");
  GS_REQUIRE(frame_ok(frame), "gs_raster_fwd: bad frame (tile %dx%d)", frame.tile_w, frame.tile_h);
  GS_REQUIRE(n_pad >= 0 && n_pad % 4 == 0, "gs_raster_fwd: bad n_pad");
  const int nu = (probe && image_tangent) ? probe->nu : 0;
  if (nu < 0 || nu > 2) {
    set_error("gs_raster_fwd: unsupported nu=%d", nu);
    return GS_ERR_UNSUPPORTED;
  }
  GS_REQUIRE(nu == 0 || proj->tangent, "gs_raster_fwd: probes given but proj->tangent is NULL");
  GS_REQUIRE(on_16_bytes(proj->rec) && (nu == 0 || on_16_bytes(proj->tangent)),
             "gs_raster_fwd: rec and tangent must be 16-byte aligned");
  cudaStream_t st = (cudaStream_t)stream;
  if (nu == 0) return launch_fwd<0>(proj, sorted, n_pad, frame, image, final_T, n_contrib, nullptr, st);
  if (nu == 1) return launch_fwd<1>(proj, sorted, n_pad, frame, image, final_T, n_contrib, image_tangent, st);
  return launch_fwd<2>(proj, sorted, n_pad, frame, image, final_T, n_contrib, image_tangent, st);
}

extern "C" size_t gs_raster_bwd_workspace_size(int32_t n_pad, gs_frame frame, int32_t nu) {
  if (n_pad < 0 || nu < 0 || nu > 2 || !gs::frame_ok(frame)) return 0;
  return gs::kCotHeaderBytes + gs::bwd_cot_floats(n_pad, frame, 1 + nu) * sizeof(float);
}

extern "C" gs_status gs_raster_bwd(const gs_params* x, const gs_camera* cams, gs_frame frame, const gs_projected* proj,
                                   const gs_sorted* sorted, const float* image, const float* target,
                                   const float* final_T, const uint32_t* n_contrib, const float* image_tangent,
                                   const gs_probe* probe, gs_loss loss, gs_params* grad, gs_params* hz,
                                   float* loss_out, void* workspace, size_t workspace_bytes, int32_t* status,
                                   void* stream) {
  return gs::run_bwd(true, x, cams, frame, proj, sorted, image, target, final_T, n_contrib, image_tangent, probe, loss,
                     grad, hz, loss_out, workspace, workspace_bytes, status, stream, "gs_raster_bwd");
}

extern "C" gs_status gs_hvp_diag(const gs_params* x, const gs_camera* cams, gs_frame frame, const gs_projected* proj,
                                 const gs_sorted* sorted, const float* image, const float* target, const float* final_T,
                                 const uint32_t* n_contrib, const float* image_tangent, const gs_probe* probe,
                                 gs_loss loss, gs_params* hz, void* workspace, size_t workspace_bytes, int32_t* status,
                                 void* stream) {
  return gs::run_bwd(false, x, cams, frame, proj, sorted, image, target, final_T, n_contrib, image_tangent, probe, loss,
                     nullptr, hz, nullptr, workspace, workspace_bytes, status, stream, "gs_hvp_diag");
}

extern "C" gs_status gs_raster_bwd_batch(const gs_batch_item* items, int32_t n_items, int32_t n_pad_max,
                                         gs_frame frame, const gs_projected* proj, const gs_sorted* sorted,
                                         const float* image, const float* target, const float* final_T,
                                         const uint32_t* n_contrib, const float* image_tangent, const gs_probe* probe,
                                         gs_loss loss, float* loss_out, void* workspace, size_t workspace_bytes,
                                         int32_t* status, void* stream) {
  using namespace gs;
  const char* name = "gs_raster_bwd_batch";
  GS_REQUIRE(items && proj && sorted && image && target && final_T && n_contrib, "%s: null argument", name);
  GS_REQUIRE(proj->rec && sorted->vals && sorted->ranges, "%s: null device buffer", name);
  GS_REQUIRE(on_16_bytes(proj->rec), "%s: rec must be 16-byte aligned", name);
  GS_REQUIRE(n_items >= 1 && n_items <= GS_BATCH_MAX, "%s: n_items=%d outside [1, %d]", name, n_items, GS_BATCH_MAX);
  GS_REQUIRE(frame_ok(frame) && frame.n_views == n_items, "%s: bad frame (n_views must equal n_items)", name);
  GS_REQUIRE(n_pad_max >= 4 && n_pad_max % 4 == 0, "%s: bad n_pad_max=%d", name, n_pad_max);
  GS_REQUIRE(loss.kind == GS_LOSS_L1 || loss.kind == GS_LOSS_L2 || loss.kind == GS_LOSS_COTANGENT ||
                 loss.kind == GS_LOSS_WEIGHTED,
             "%s: bad loss kind %d", name, loss.kind);
  const bool given = loss.kind == GS_LOSS_COTANGENT;
  const int nu = ((image_tangent || given) && probe) ? probe->nu : 0;
  const int deg = items[0].x.sh_degree;
  if (nu < 0 || nu > 2 || deg < 0 || deg > 3) {
    set_error("%s: unsupported nu=%d sh_degree=%d", name, nu, deg);
    return GS_ERR_UNSUPPORTED;
  }
  GS_REQUIRE(loss.kind != GS_LOSS_WEIGHTED || nu == 0 || image_tangent, "%s: weighted loss needs image_tangent",
             name);
  for (int b = 0; b < n_items; ++b) {
    const gs_batch_item& it = items[b];
    auto same = [&](const gs_params& p) { return p.n == it.x.n && p.n_pad == it.x.n_pad && p.sh_degree == deg; };
    GS_REQUIRE(it.x.data && it.cam && it.grad.data && same(it.x) && same(it.grad),
               "%s: item %d needs x, cam and a gradient of x's layout", name, b);
    GS_REQUIRE(nu == 0 || (it.hz.data && same(it.hz) && it.t >= 1), "%s: item %d needs hz and t >= 1 with probes",
               name, b);
    GS_REQUIRE(it.x.n >= 0 && it.x.n <= n_pad_max && it.x.n_pad % 4 == 0, "%s: item %d: bad n=%d n_pad=%d", name,
               b, it.x.n, it.x.n_pad);
  }
  const size_t floats = bwd_cot_floats(n_pad_max, frame, 1 + nu);
  const size_t need = kCotHeaderBytes + floats * sizeof(float);
  GS_REQUIRE(workspace && workspace_bytes >= need, "%s: workspace needs %zu bytes, got %zu", name, need,
             workspace_bytes);
  GS_REQUIRE(((uintptr_t)workspace & 15) == 0, "%s: workspace must be 16-byte aligned", name);
  cudaStream_t st = (cudaStream_t)stream;
  CotWs ws;
  if (cot_prepare(workspace, floats, ws, st) != cudaSuccess) return check_launch(name);
  const BatchArg ba = batch_arg(items, n_items, [](const gs_batch_item& it) {
    return (it.x.n + kPbwdThreads - 1) / kPbwdThreads;
  });
  launch_bwd_streams(true, nu, nullptr, &ba, n_pad_max, deg, nullptr, proj, sorted, frame, image, target, final_T,
                     n_contrib, image_tangent, probe, loss, nullptr, nullptr, loss_out, ws, status, st);
  return check_launch(name);
}
