// dRadon/ds precompute: the Grangeat intermediate function S_lambda (Eq. 1) of
// every projection on an (alpha, s) grid.
//
//   line table           (FP64, geometry_kernel) the parameters of the detector lines
//                        (x - cx) cos a + (y - cy) sin a = sigma as 32.32 fixed-point
//                        coordinates along the interpolation axis (exact integer
//                        stepping, no FP64 in the hot loop).
//   weight_kernel        cosine pre-weight g D / sqrt(D^2 + u^2 + v^2) of each
//                        projection, stored as interpolation pairs (v[i],
//                        v[i+1] - v[i]) twice: along image rows and along image
//                        columns, each with a zero margin on both sides wide enough
//                        for the 32 lines of a warp.
//   joseph_kernel        one warp per (view, alpha, 31 consecutive s_n), a block's
//                        warps on consecutive alpha rows (shared image band): Joseph
//                        line sums (step over rows for |cos a| >= |sin a|, else over
//                        columns, linear interpolation along the other axis), one
//                        8-byte pair load and one FMA per tap.  The half-step
//                        difference in s is formed between neighbouring lanes (warp
//                        shuffle) on 8-row partial sums, so that it never cancels
//                        two large FP32 sums (Kahan-compensated across blocks); the
//                        (D^2 + s^2)/D^2 weight is applied at the end.  Lanes read
//                        consecutive pairs of one image row: coalesced, L1/L2
//                        resident.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "ecc_internal.cuh"
#include "kernels.cuh"

namespace ecc {

namespace {

// Weighted projection as interpolation pairs (v[i], v[i+1] - v[i]) along the
// interpolation axis: row-major [H][pitch_r] (pairs along x) and transposed
// [W][pitch_c] (pairs along y), the image from element pad on, zeros elsewhere
// (the pair before the image carries (0, v[0])).  A block (32, 8) covers 32x32
// pairs starting one pixel before the image; the weighted values of a 33x33 tile
// are computed once into shared memory and both planes are written coalesced.  The
// blocks beside the margins write their zeros.
__global__ void weight_kernel(const float* __restrict__ images, const RadonView* rv, int W, int H,
                              int pad, int pitch_r, int pitch_c, float2* __restrict__ wimg, size_t plane) {
  wait_for_previous();
  __shared__ float tile[33][34];
  const int v = blockIdx.z;
  const float* g = images + (size_t)v * W * H;
  float2* R = wimg + (size_t)v * plane;
  float2* T = R + (size_t)H * pitch_r;
  const RadonView r = rv[v];
  const int bx = (int)blockIdx.x * 32 - 1, by = (int)blockIdx.y * 32 - 1;
  for (int i = threadIdx.y * 32 + threadIdx.x; i < 33 * 33; i += 256) {
    const int ty = i / 33, tx = i % 33;
    const int x = bx + tx, y = by + ty;
    float w = 0.0f;
    if (x >= 0 && x < W && y >= 0 && y < H) {
      const float du = (float)x - r.u0, dv = (float)y - r.v0;
      w = g[(size_t)y * W + x] * (r.D / sqrtf(r.D * r.D + du * du + dv * dv));
    }
    tile[ty][tx] = w;
  }
  __syncthreads();
  for (int j = 0; j < 4; ++j) {
    const int tx = threadIdx.x, ty = threadIdx.y + 8 * j;
    const int x = bx + tx, y = by + ty;
    // pairs along x for image rows
    if (y >= 0 && y < H && x >= -1 && x < W)
      R[(size_t)y * pitch_r + x + pad] = make_float2(tile[ty][tx], tile[ty][tx + 1] - tile[ty][tx]);
    // pairs along y for image columns (threads run along y: coalesced)
    const int xo = bx + ty, yo = by + tx;
    if (xo >= 0 && xo < W && yo >= -1 && yo < H)
      T[(size_t)xo * pitch_c + yo + pad] = make_float2(tile[tx][ty], tile[tx + 1][ty] - tile[tx][ty]);
  }
  // margins: [0, pad - 1) before the image's pairs, [W + pad, W + 2 pad) behind them (H for columns)
  const float2 zero = make_float2(0.0f, 0.0f);
  for (int side = 0; side < 2; ++side) {
    const int n = side ? pad : pad - 1;
    if (blockIdx.x == (side ? gridDim.x - 1 : 0))
      for (int j = threadIdx.y; j < 32; j += 8) {
        const int y = by + j;
        for (int i = threadIdx.x; y >= 0 && y < H && i < n; i += 32)
          R[(size_t)y * pitch_r + (side ? W + pad : 0) + i] = zero;
      }
    if (blockIdx.y == (side ? gridDim.y - 1 : 0))
      for (int j = threadIdx.y; j < 32; j += 8) {
        const int x = bx + j;
        for (int i = threadIdx.x; x >= 0 && x < W && i < n; i += 32)
          T[(size_t)x * pitch_c + (side ? H + pad : 0) + i] = zero;
      }
  }
}

// ---------------------------------------------------------------- Joseph line sums
//
// One warp per (view, alpha row, 31 consecutive s_n): lane i follows the line at
// the half-step offset s_{k0+i} - ds/2 (lane 31 provides the line after the last
// output).  The weighted image is stored as pairs (v[i], v[i+1] - v[i]) along the
// interpolation axis, so one tap is one 8-byte load and one FMA; lanes read
// consecutive pairs of one image row (coalesced, L1-resident).  A warp walks only
// the image rows where some of its lines meet the image (exact row range), in
// blocks of 16 rows: exact 32.32 fixed-point position at the block's first row,
// then FP32 offsets u * dy (|u| < 16, error < 2e-6 px); floor and element offset
// come from one round-down add against 1.5 * 2^23 + u * pitch.  Taps are summed
// over 8 rows, and the 8-row sum's difference to the next lane's line is added to
// a Kahan-compensated accumulator, so the half-step difference in s never cancels
// two large FP32 sums.
constexpr int kRowsPerAnchor = 16;
constexpr int kRowsPerBlock = 8;
constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23: float ulp 1 for [2^23, 2^24)
constexpr unsigned kMagicBits = 0x4B400000u;
constexpr int kMaxPad = 160;  // wider margins: clamped variant

__device__ __forceinline__ void kahan_add(float q, float& acc, float& comp) {
  const float y = q - comp;
  const float t = acc + y;
  comp = (t - acc) - y;
  acc = t;
}

constexpr int kAlphaPerBlock = 8;  // warps per block

struct JosephArgs {
  int W, H, n_alpha, n_s;
  int pad, pitch_r, pitch_c;  // float2 elements
  size_t plane;               // float2 elements per view
  float ds;
};

// Taps of rows u in [ua, ub) of one anchor block (all 16 rows when FULL).
template <bool CLAMP, bool FULL>
__device__ __forceinline__ void joseph_block(const float2* rp, float f0, float dyf, float lo_c, float hi_c,
                                             const float (&Mu)[kRowsPerAnchor], int ua, int ub, float& acc,
                                             float& comp) {
#pragma unroll
  for (int i = 0; i < kRowsPerAnchor / kRowsPerBlock; ++i) {
    float s = 0.0f;
#pragma unroll
    for (int uu = 0; uu < kRowsPerBlock; ++uu) {
      const int u = i * kRowsPerBlock + uu;
      if (FULL || (u >= ua && u < ub)) {
        float xf = fmaf((float)u, dyf, f0);
        if (CLAMP) xf = fminf(fmaxf(xf, lo_c), hi_c);
        const float t = __fadd_rd(xf, Mu[u]);
        const float f = xf - (t - Mu[u]);
        const float2 vd = rp[__float_as_uint(t)];
        s += fmaf(f, vd.y, vd.x);
      }
    }
    const float nb = __shfl_down_sync(0xffffffffu, s, 1);
    kahan_add(nb - s, acc, comp);
  }
}

// Three blocks per SM (80 registers): the kernel waits on its loads, and with registers to
// spare the compiler issues 16 rows' loads together.  Left to itself it takes 64 (a view of
// 256 x 256 on the 256 x 363 grid 28.5 us, now 20.4; 12 views of 620 x 480 1.296 ms, now
// 1.268; a 976 x 976 view 450 us, now 435); two blocks are 1 % faster on many views and 3 %
// slower on two.  (Several warps along one line, and the next rows' loads issued before these
// rows' sums, did not pay: 31 us stayed 31 us for two views, more views got slower.)
template <bool CLAMP>
__global__ void __launch_bounds__(32 * kAlphaPerBlock, 3) joseph_kernel(const RadonRow* table,
                                                                         const RadonView* rv,
                                                                         const float2* wimg,
                                                                         JosephArgs g, float* __restrict__ out_f32,
                                                                         __nv_bfloat16* __restrict__ out_bf16) {
  wait_for_previous();
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  // the warps of a block take the same 31 outputs of consecutive alpha rows: their
  // image bands largely overlap and are shared through L1
  const int v = blockIdx.z, m = (int)blockIdx.y * kAlphaPerBlock + warp;
  if (m >= g.n_alpha) return;  // warp-uniform
  const int k0 = 31 * (int)blockIdx.x;
  const int k = k0 + lane;
  const RadonRow row = table[(size_t)v * g.n_alpha + m];
  const bool rows = row.rows_mode != 0;
  const float2* img = wimg + (size_t)v * g.plane + (rows ? 0 : (size_t)g.H * g.pitch_r);
  const int pitch = rows ? g.pitch_r : g.pitch_c;
  const int n_steps = rows ? g.H : g.W;
  const int limit = rows ? g.W : g.H;
  // image rows where some lane of the warp is inside the interpolation support
  int s_lo = 0, s_hi = n_steps;
  {
    const float scale = 1.0f / 65536.0f;
    const float xa = (float)((row.B0 + (long long)k0 * row.STEP) >> 16) * scale;
    const float xb = (float)((row.B0 + (long long)(k0 + 31) * row.STEP) >> 16) * scale;
    const float dy = (float)(row.DY >> 16) * scale;
    const float mn = fminf(xa, xb) - 2.0f, mx = fmaxf(xa, xb) + 2.0f;
    const float lo_t = -1.0f, hi_t = (float)limit;
    if (fabsf(dy) > 1e-6f) {
      const float s1 = (lo_t - mx) / dy, s2 = (hi_t - mn) / dy;
      // clamp in float first: nearly axis-parallel lines give huge bounds
      const float cap = (float)n_steps + 4.0f;
      const float sl = fminf(fmaxf(fminf(s1, s2), -4.0f), cap);
      const float sh = fminf(fmaxf(fmaxf(s1, s2), -4.0f), cap);
      s_lo = max(0, (int)floorf(sl) - 1);
      s_hi = min(n_steps, (int)ceilf(sh) + 2);
    } else if (mx < lo_t || mn > hi_t) {
      s_hi = 0;
    }
    if (s_hi < s_lo) s_hi = s_lo;
  }
  const float dyf = (float)((double)row.DY * (1.0 / 4294967296.0));
  const long long DY16 = (long long)kRowsPerAnchor * row.DY;
  float Mu[kRowsPerAnchor];
#pragma unroll
  for (int u = 0; u < kRowsPerAnchor; ++u) Mu[u] = kMagic + (float)(u * pitch);
  long long X = row.B0 + (long long)k * row.STEP + (long long)s_lo * row.DY;
  float acc = 0.0f, comp = 0.0f;
  // row pointers are biased by -kMagicBits elements, so that a tap's element is the
  // pointer plus the bit pattern of its round-down sum (one 32x32+64 multiply-add)
  const uint64_t img_b = reinterpret_cast<uint64_t>(img) - 8ull * kMagicBits;
  for (int j0 = s_lo; j0 < s_hi; j0 += kRowsPerAnchor) {
    const int xi0 = (int)(X >> 32);
    const float f0 = __uint_as_float(0x3f800000u | ((unsigned)X >> 9)) - 1.0f;
    const float2* rp = reinterpret_cast<const float2*>(img_b + 8ull * (uint64_t)((long long)j0 * pitch + g.pad + xi0));
    const float lo_c = (float)(-2 - xi0), hi_c = (float)(limit - xi0);
    const int n = s_hi - j0;
    if (n >= kRowsPerAnchor)
      joseph_block<CLAMP, true>(rp, f0, dyf, lo_c, hi_c, Mu, 0, n, acc, comp);
    else
      joseph_block<CLAMP, false>(rp, f0, dyf, lo_c, hi_c, Mu, 0, n, acc, comp);
    X += DY16;
  }
  if (lane < 31 && k < g.n_s) {
    const RadonView r = rv[v];
    const float sn = ((float)k - 0.5f * (float)(g.n_s - 1)) * g.ds;
    const float spp = sn - (r.u0 - 0.5f * (float)(g.W - 1)) * row.ca - (r.v0 - 0.5f * (float)(g.H - 1)) * row.sa;
    const float wgt = (r.D * r.D + spp * spp) / (r.D * r.D);
    const float val = (acc - comp) * (row.inv_len / g.ds) * wgt;
    const size_t o = ((size_t)v * g.n_alpha + m) * g.n_s + k;
    if (out_bf16)
      out_bf16[o] = __float2bfloat16_rn(val);
    else
      out_f32[o] = val;
  }
}

// FP16 storage: per-view scale = max|S| / 2^14 (1 if the view is all zero), so
// every stored value is in FP16's normal range; stored = S / scale.  A block takes
// kQuantBlock values of a view, 16 a thread, as four 16-byte loads in flight where the
// views' rows allow it (a multiple of four values a view, outputs on 8 bytes) and as 16
// single ones elsewhere: one value a thread at a time left both passes waiting on their
// loads (64 MB of 173 views: 35 and 47 us, now 18 and 33).  The max of a view is folded
// from its blocks by an atomic max on the bit pattern (non-negative floats order as
// their bits) in the view's slot, zero before.
constexpr int kQuantBlock = 256 * 16;

// Applies f to the values of this thread, f(index in the view, values).
template <class F>
__device__ __forceinline__ void quant_values(const float* p, size_t per_view, bool vec, F f) {
  const size_t i0 = (size_t)blockIdx.x * kQuantBlock;
  if (vec) {
    float4 x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const size_t i = i0 + 4 * (256 * j + threadIdx.x);
      x[j] = i < per_view ? *reinterpret_cast<const float4*>(p + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) f(i0 + 4 * (256 * j + threadIdx.x), x[j]);
  } else {
    float x[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const size_t i = i0 + 256 * j + threadIdx.x;
      x[j] = i < per_view ? p[i] : 0.0f;
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) f(i0 + 256 * j + threadIdx.x, x[j]);
  }
}

__global__ void __launch_bounds__(256) absmax_kernel(const float* s32, size_t per_view, bool vec, RadonView* rv) {
  wait_for_previous();
  struct {
    float m = 0.0f;
    __device__ void operator()(size_t, float x) { m = fmaxf(m, fabsf(x)); }
    __device__ void operator()(size_t, const float4& x) {
      m = fmaxf(fmaxf(m, fmaxf(fabsf(x.x), fabsf(x.y))), fmaxf(fabsf(x.z), fabsf(x.w)));
    }
  } most;
  quant_values(s32 + (size_t)blockIdx.y * per_view, per_view, vec, [&](size_t i, const auto& x) { most(i, x); });
  float m = most.m;
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0 && m > 0.0f) atomicMax(&rv[blockIdx.y].max_bits, __float_as_uint(m));
}

__global__ void __launch_bounds__(256) quantize_f16_kernel(const float* s32, size_t per_view, bool vec, const RadonView* rv,
                                                           float* __restrict__ scales, __half* __restrict__ out) {
  wait_for_previous();
  const float m = __uint_as_float(rv[blockIdx.y].max_bits);
  const float scale = m > 0.0f ? m / 16384.0f : 1.0f;
  if (blockIdx.x == 0 && threadIdx.x == 0) scales[blockIdx.y] = scale;
  struct {
    __half* o;
    size_t n;
    float scale;
    __device__ void operator()(size_t i, float x) const {
      if (i < n) o[i] = __float2half_rn(x / scale);
    }
    __device__ void operator()(size_t i, const float4& x) const {
      if (i >= n) return;
      const auto two = [&](float a, float b) {
        return (unsigned)__half_as_ushort(__float2half_rn(a / scale)) |
               (unsigned)__half_as_ushort(__float2half_rn(b / scale)) << 16;
      };
      *reinterpret_cast<uint2*>(o + i) = make_uint2(two(x.x, x.y), two(x.z, x.w));
    }
  } put{out + (size_t)blockIdx.y * per_view, per_view, scale};
  quant_values(s32 + (size_t)blockIdx.y * per_view, per_view, vec, [&](size_t i, const auto& x) { put(i, x); });
}

}  // namespace

int radon_pad(int W, int H, int n_s) {
  // span of 32 neighbouring lines along the interpolation axis (|cos| or |sin| >=
  // 1/sqrt 2 in their mode) plus the margins of the per-warp row range
  const double ds = sqrt((double)W * W + (double)H * H) / (n_s - 1);
  const int need = (int)ceil(31.0 * ds * 1.41421356237309515 + 8.0);
  return need <= kMaxPad ? need : 2;  // 2: clamped variant
}

size_t radon_plane_bytes(int W, int H, int n_s) {
  const int pad = radon_pad(W, H, n_s);
  return sizeof(float2) * ((size_t)H * (W + 2 * pad) + (size_t)W * (H + 2 * pad));
}

size_t radon_f16_stage_bytes(int n_alpha, int n_s, int batch_views) {
  return sizeof(float) * (size_t)n_alpha * n_s * batch_views;
}

static size_t stage_bytes(int n_alpha, int n_s, int dtype, int batch) {
  return dtype == 1 ? radon_f16_stage_bytes(n_alpha, n_s, batch) : 0;
}

RadonPlan radon_plan_by_view(int n_views, int W, int H, int n_alpha, int n_s, int dtype) {
  RadonPlan p{};
  const size_t plane = radon_plane_bytes(W, H, n_s);
  const size_t max_batch_bytes = (size_t)256 << 20;  // weighted images of a batch, unless one view takes more
  p.batch = (int)std::max<size_t>(1, std::min<size_t>((size_t)n_views, max_batch_bytes / plane));
  p.lead = p.batch;
  p.wimg_bytes = plane * (size_t)p.batch;
  p.stage_bytes = stage_bytes(n_alpha, n_s, dtype, p.batch);
  return p;
}

RadonPlan radon_plan(int n_scan, int n_views, int W, int H, int n_alpha, int n_s, int dtype,
                     const RadonRoom& room) {
  const int least = ViewsPlan::min_views(W, H, n_alpha, n_s);
  if (least > 0 && n_scan >= least) {
    for (int axes = 2; axes >= 1; --axes) {
      const size_t gb = ViewsPlan::group_bytes(axes, W, H, n_alpha, n_s);
      int groups = (int)std::min<size_t>((size_t)(n_views + 31) / 32, room.wimg / gb);
      auto batch = [&] { return std::min(n_views, groups * 32); };
      auto stage = [&] { return stage_bytes(n_alpha, n_s, dtype, batch()); };
      while (groups > 0 && (stage() > room.stage || gb * groups + stage() > room.total)) --groups;
      if (groups == 0) continue;
      RadonPlan p{};
      p.views = true;
      p.batch = p.lead = batch();
      p.wimg_bytes = gb * groups;
      p.stage_bytes = stage();
      return p;
    }
  }
  return radon_plan_by_view(n_views, W, H, n_alpha, n_s, dtype);
}

// FP16 storage of nb views staged in FP32: per-view maximum, scale, quantisation.
static cudaError_t quantize_batch(const float* stage, size_t per_view, int nb, RadonView* rv, float* scales,
                                  __half* out, const LaunchHooks& hooks, cudaStream_t stream) {
  const unsigned bpv = (unsigned)((per_view + kQuantBlock - 1) / kQuantBlock);
  const bool vec = per_view % 4 == 0 && reinterpret_cast<uintptr_t>(out) % 8 == 0;
  for (int v = 0; v < nb; v += 65535) {
    const dim3 grid(bpv, std::min(65535, nb - v));
    const float* s = stage + per_view * v;
    hooks.on_begin("absmax_kernel", stream);
    launch_behind(absmax_kernel, grid, 256, 0, stream, s, per_view, vec, rv + v);
    hooks.on_end("absmax_kernel", stream);
    hooks.on_begin("quantize_f16_kernel", stream);
    launch_behind(quantize_f16_kernel, grid, 256, 0, stream, s, per_view, vec, rv + v, scales + v, out + per_view * v);
    hooks.on_end("quantize_f16_kernel", stream);
  }
  return cudaGetLastError();
}

cudaError_t launch_radon(int n_views, const float* images, int W, int H, int n_alpha, int n_s, int dtype,
                         void* sino_out, float* scales_out, const RadonRow* table, void* wimg, float* stage,
                         const RadonPlan& plan, int* status, const LaunchHooks& hooks, cudaStream_t stream,
                         const cudaEvent_t* batch_ready) {
  RadonView* rv = plan.weights(const_cast<RadonRow*>(table), n_views, n_alpha);
  JosephArgs jg;
  jg.W = W;
  jg.H = H;
  jg.n_alpha = n_alpha;
  jg.n_s = n_s;
  jg.pad = radon_pad(W, H, n_s);
  const bool clamp = jg.pad == 2;
  jg.pitch_r = W + 2 * jg.pad;
  jg.pitch_c = H + 2 * jg.pad;
  jg.plane = radon_plane_bytes(W, H, n_s) / sizeof(float2);
  jg.ds = (float)(sqrt((double)W * W + (double)H * H) / (n_s - 1));
  const int n_chunks = (n_s + 30) / 31;
  const size_t per_view = (size_t)n_alpha * n_s;
  float2* wv = reinterpret_cast<float2*>(wimg);
  const bool behind = batch_ready == nullptr;  // behind an event a batch's first kernel is launched plainly
  const int passes = plan.passes(n_views);
  for (int pass = 0; pass < passes; ++pass) {
    const int v0 = plan.begin(pass), nb = plan.count(pass, n_views);
    cudaError_t e;
    if (batch_ready && (e = cudaStreamWaitEvent(stream, batch_ready[pass], 0)) != cudaSuccess) return e;
    const float* im = images + (size_t)v0 * W * H;
    const size_t oo = (size_t)v0 * per_view;
    float* of = dtype == 0 ? (float*)sino_out + oo : (dtype == 1 ? stage : nullptr);
    __nv_bfloat16* ob = dtype == 2 ? (__nv_bfloat16*)sino_out + oo : nullptr;
    if (plan.views) {
      e = launch_radon_views(table, rv + v0, nb, im, W, H, n_alpha, n_s, wimg, plan.wimg_bytes, of, ob, status, plan.wait_ns,
                             behind, hooks, stream);
      if (e != cudaSuccess) return e;
    } else {
      hooks.on_begin("weight_kernel", stream);
      launch_at(behind, weight_kernel, dim3((W + 32) / 32, (H + 32) / 32, nb), dim3(32, 8), 0, stream, im, rv + v0, W,
                H, jg.pad, jg.pitch_r, jg.pitch_c, wv, jg.plane);
      hooks.on_end("weight_kernel", stream);
      e = cudaGetLastError();
      if (e != cudaSuccess) return e;
      const RadonRow* tb = table + (size_t)v0 * n_alpha;
      const dim3 grid(n_chunks, (n_alpha + kAlphaPerBlock - 1) / kAlphaPerBlock, nb), block(32 * kAlphaPerBlock);
      hooks.on_begin("joseph_kernel", stream);
      if (clamp)
        launch_behind(joseph_kernel<true>, grid, block, 0, stream, tb, rv + v0, wv, jg, of, ob);
      else
        launch_behind(joseph_kernel<false>, grid, block, 0, stream, tb, rv + v0, wv, jg, of, ob);
      hooks.on_end("joseph_kernel", stream);
      e = cudaGetLastError();
      if (e != cudaSuccess) return e;
    }
    if (dtype == 1) {
      e = quantize_batch(stage, per_view, nb, rv + v0, scales_out + v0, (__half*)sino_out + oo, hooks, stream);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

}  // namespace ecc
