// dRadon/ds precompute of many views at once: the detector lines are the same for
// every view of a scan (they depend on the detector and the grid only), so one walk
// along a line serves a group of 32 views.
//
//   weight_views_kernel  cosine pre-weight of each projection and its differences
//                        d_i = v[i+1] - v[i] along image rows or image columns (zero
//                        outside the detector, from one cell before it), views
//                        innermost: [step][cell][32 views], 128 bytes per cell.
//   radon_views_kernel   S on the grid.  By the fundamental theorem on the piecewise
//                        linear image row, the difference of two neighbouring lines'
//                        taps at one step is the sum of d over the cells between their
//                        positions x_k < x_(k+1):
//                          (1 - f_k) d[i_k] + (cells in between) + f_(k+1) d[i_(k+1)],
//                        i = floor(x), f = x - i.  With lines less than two cells apart
//                        there is at most one cell in between, so a line costs one load
//                        (1.15 with the cells in between, averaged over the angles) and
//                        two FMAs, and the half-step difference of Eq. 1 is accumulated
//                        directly: no difference of two large sums is ever taken.  Every
//                        line's position is exact (32.32 fixed point), and the sums of
//                        32 steps are folded into a second level in tensor memory.
//
// Work split: a lane follows 16 lines of one alpha row for four views; a warp holds four
// neighbouring alpha rows x 32 views.  Where the four rows' lines are in one cell, the
// warp's 16-byte loads fall into the same 128 bytes of shared memory, which are read once
// (3.2 wavefronts a load instead of 4 on the 620 x 480 grid).  A CTA takes 16 warps = A
// neighbouring alpha rows x 64 / A neighbouring chunks of 16 lines.  Their lines cross one
// image step within a window of some dozen cells; each step's window (contiguous in memory)
// is brought into a ring of shared-memory slots by one bulk asynchronous copy, which the
// warps issue in turn some steps ahead.  The 64 accumulators of a lane stay in registers.
//
// Measured on 496 views of 620 x 480, 768 x 768 grid, the whole precompute: 23.5 ms (view by
// view: 56.0; lines stepped in FP32 and sums of one level, which are less accurate than
// view by view on noise: 22.3).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "ecc_internal.cuh"
#include "kernels.cuh"

namespace ecc {

namespace {

constexpr int kWarps = 16;        // per CTA: 128 registers a thread
constexpr int kRows = 4;          // alpha rows per warp
constexpr int kUnits = kWarps * kRows;  // (alpha row, chunk of lines) per CTA
constexpr int kLines = 16;        // lines (and outputs) per lane
constexpr int kGroup = 32;        // views per group
constexpr unsigned kCell = 4 * kGroup;  // bytes of one cell
constexpr int kLag = 2;           // steps between a slot's last use and its refill
constexpr int kRing = 190 * 1024; // shared memory of the slots
constexpr int kMinSlots = 4;
constexpr int kMaxSlots = 16;
constexpr int kMaxSteps = 2048;   // of the window table
constexpr unsigned kAll = 0xffffffffu;  // lanes of a warp

struct ViewsArgs {
  int W, H, n_alpha, n_s;
  int n_views;             // of this launch (all groups)
  int A;                   // alpha rows per CTA (64 / A chunks of lines each)
  int r1, r2;              // steps are image rows for m < r1 and m >= r2, else columns
  int axis;                // planes present: 0 rows, 1 columns, 2 both
  int pad;                 // zero cells on either side of a step
  int win;                 // most cells of a window
  size_t cols0;            // floats from the row planes to the column planes
  float ds;
  unsigned long long wait_ns;  // a wait gives up after this long
  unsigned hint;           // longest suspension of one of its tries, in ns
};

typedef unsigned long long u64;

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ u64 now_ns() {
  u64 t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
// One try, in which the hardware may suspend the warp for up to `hint` ns (polling without
// the hint took 35 instructions a step).
__device__ __forceinline__ bool mbar_try(unsigned bar, unsigned parity, unsigned hint) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2, %3;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(hint)
      : "memory");
  return ok != 0;
}
// Waits for the phase of `parity` to complete, by one thread; false if that took longer than
// the limit, or if a wait of the CTA has given up meanwhile (failed, or NULL).
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, u64 limit_ns, unsigned hint,
                                          volatile int* failed) {
  if (mbar_try(bar, parity, hint)) return true;
  const u64 t0 = now_ns();
  for (;;) {
    const bool out = now_ns() - t0 >= limit_ns || (failed && *failed);
    if (mbar_try(bar, parity, hint)) return true;
    if (out) break;
  }
  if (failed) *failed = 1;
  return false;
}
// The same by a whole warp, with one verdict for all lanes: lanes that disagreed would part,
// some to the next step's warp barriers and some to the CTA's, and wait there for each other.
__device__ __forceinline__ bool mbar_wait_warp(unsigned bar, unsigned parity, u64 limit_ns, unsigned hint,
                                               volatile int* failed) {
  if (__all_sync(kAll, mbar_try(bar, parity, hint))) return true;
  const u64 t0 = now_ns();
  for (;;) {
    const bool out = now_ns() - t0 >= limit_ns || *failed;
    if (__all_sync(kAll, mbar_try(bar, parity, hint))) return true;
    if (__any_sync(kAll, out)) break;
  }
  *failed = 1;
  return false;
}
__device__ __forceinline__ void bulk_copy(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// ---------------------------------------------------------------- weighting
//
// Weighted projections as differences along one axis or both, views innermost.  A block
// takes 32 x 8 cells of the 32 views of a group: the weighted values of 33 x 9 pixels are
// computed once into shared memory (reads coalesced along image rows) and the planes are
// written in runs of 128 bytes.  The blocks beside the margins write their zeros.
constexpr int kTileX = 32, kTileY = 8;
constexpr int kTilePitch = 33;

__global__ void __launch_bounds__(256) weight_views_kernel(const float* __restrict__ images, const RadonView* rv,
                                                           ViewsArgs g, float* __restrict__ planes) {
  wait_for_previous();
  __shared__ float tile[(kTileX + 1) * (kTileY + 1) * kTilePitch];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int bx = (int)blockIdx.x * kTileX - 1, by = (int)blockIdx.y * kTileY - 1;
  const int v0 = (int)blockIdx.z * kGroup;
  auto put = [&](int v, int ty, int tx, const RadonView& r) {
    const int x = bx + tx, y = by + ty;
    float w = 0.0f;
    if (v0 + v < g.n_views && y >= 0 && y < g.H && x >= 0 && x < g.W) {
      const float du = (float)x - r.u0, dv = (float)y - r.v0;
      w = images[((size_t)(v0 + v) * g.H + y) * g.W + x] * (r.D / sqrtf(r.D * r.D + du * du + dv * dv));
    }
    tile[(ty * (kTileX + 1) + tx) * kTilePitch + v] = w;
  };
  for (int v = warp; v < 32; v += 8) {
    const RadonView r = rv[min(v0 + v, g.n_views - 1)];
#pragma unroll
    for (int ty = 0; ty <= kTileY; ++ty) put(v, ty, lane, r);
  }
  for (int i = threadIdx.x; i < 32 * (kTileY + 1); i += 256) {  // the last column
    const int v = i / (kTileY + 1);
    put(v, i % (kTileY + 1), kTileX, rv[min(v0 + v, g.n_views - 1)]);
  }
  __syncthreads();
  const int pitch_r = g.W + 1 + 2 * g.pad, pitch_c = g.H + 1 + 2 * g.pad;
  if (g.axis != 1) {
    float* __restrict__ rows = planes + (size_t)blockIdx.z * g.H * pitch_r * kGroup;
    for (int i = warp; i < kTileX * kTileY; i += 8) {
      const int tx = i % kTileX, ty = 1 + i / kTileX;
      const int x = bx + tx, y = by + ty;
      if (y < g.H && x < g.W) {
        const float* p = tile + (ty * (kTileX + 1) + tx) * kTilePitch + lane;
        rows[((size_t)y * pitch_r + x + 1 + g.pad) * kGroup + lane] = p[kTilePitch] - p[0];
      }
    }
    const int y = by + 1 + warp;  // margins: a row per warp
    if (y < g.H && blockIdx.x == 0)
      for (int i = 0; i < g.pad; ++i) rows[((size_t)y * pitch_r + i) * kGroup + lane] = 0.0f;
    if (y < g.H && blockIdx.x == gridDim.x - 1)
      for (int i = 0; i < g.pad; ++i) rows[((size_t)y * pitch_r + g.W + 1 + g.pad + i) * kGroup + lane] = 0.0f;
  }
  if (g.axis != 0) {
    float* __restrict__ cols = planes + g.cols0 + (size_t)blockIdx.z * g.W * pitch_c * kGroup;
    for (int i = warp; i < kTileX * kTileY; i += 8) {
      const int ty = i % kTileY, tx = 1 + i / kTileY;
      const int x = bx + tx, y = by + ty;
      if (y < g.H && x < g.W) {
        const float* p = tile + (ty * (kTileX + 1) + tx) * kTilePitch + lane;
        cols[((size_t)x * pitch_c + y + 1 + g.pad) * kGroup + lane] = p[(kTileX + 1) * kTilePitch] - p[0];
      }
    }
    for (int t = warp; t < kTileX; t += 8) {
      const int x = bx + 1 + t;
      if (x < g.W && blockIdx.y == 0)
        for (int i = 0; i < g.pad; ++i) cols[((size_t)x * pitch_c + i) * kGroup + lane] = 0.0f;
      if (x < g.W && blockIdx.y == gridDim.y - 1)
        for (int i = 0; i < g.pad; ++i) cols[((size_t)x * pitch_c + g.H + 1 + g.pad + i) * kGroup + lane] = 0.0f;
    }
  }
}

// ---------------------------------------------------------------- line sums

// Steps where some line of a chunk may meet the image: lines at x_a .. x_b (at step 0)
// moving by dy per step, support (-1, cells).  Margins of a step and two cells.
__device__ __forceinline__ void step_range(float xa, float xb, float dy, int steps, int cells, int& lo, int& hi) {
  const float mn = fminf(xa, xb) - 2.0f, mx = fmaxf(xa, xb) + 2.0f;
  lo = 0;
  hi = steps;
  if (fabsf(dy) > 1e-6f) {
    const float s1 = (-1.0f - mx) / dy, s2 = ((float)cells - mn) / dy;
    const float cap = (float)steps + 4.0f;
    lo = max(0, (int)floorf(fminf(fmaxf(fminf(s1, s2), -4.0f), cap)) - 1);
    hi = min(steps, (int)ceilf(fminf(fmaxf(fmaxf(s1, s2), -4.0f), cap)) + 2);
  } else if (mx < -1.0f || mn > (float)cells) {
    hi = 0;
  }
  if (hi < lo) hi = lo;
}

__device__ __forceinline__ float4 load4(unsigned addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
// o += w d for four views, two FMAs per instruction.  (Through the intrinsic: the same
// instruction as inline assembly on 64-bit registers cost a move for every operand.)
__device__ __forceinline__ void fma4(float4& o, float w, const float4& d) {
  const float2 ww = make_float2(w, w);
  const float2 a = __ffma2_rn(ww, make_float2(d.x, d.y), make_float2(o.x, o.y));
  const float2 b = __ffma2_rn(ww, make_float2(d.z, d.w), make_float2(o.z, o.w));
  o = make_float4(a.x, a.y, b.x, b.y);
}

// Weights of a position with fraction n / 2^32: f of the cell it is in, g = 1 - f.
__device__ __forceinline__ float frac_f(unsigned n) { return __uint2float_rn(n) * 0x1p-32f; }
__device__ __forceinline__ float frac_g(unsigned n) { return fmaf(__uint2float_rn(n), -0x1p-32f, 1.0f); }

// Lines I and I + 1 of a lane at one step.  b + I cells: the cell after line I - 1's, n the
// fraction of its position.  A line is s = 1 + step / 2^32 cells after the one before, so
// that a carry out of the fractions' sum means a move by two cells (predicates p, q): the
// cell in between goes to the output as it is; m holds it (registers that only some lanes
// write would stay live around the loop if they were not kept across steps).  Loads and
// predicated sums of both lines first, then their FMAs, so that no two neighbouring
// instructions depend on one another.  NEAR: lanes with `below` set have s = step / 2^32,
// and no carry means that the position stays in its cell (predicates r, t): the output is
// then (f1 - f) d, of which the line before has put in (1 - f) d.
template <bool NEAR, int I>
__device__ __forceinline__ void two_lines(unsigned& b, unsigned& n, unsigned step, bool below, float4 (&m)[2],
                                          float4 (&acc)[kLines]) {
  unsigned n1, n2;
  float4 d1, d2;
  float4 &o = acc[I - 1], &o2 = acc[I];
  float w1, w2;
  if (NEAR) {
    unsigned stay1, stay2;
    asm volatile(
        "{\n .reg .pred p, q, r, t, u;\n"
        " setp.ne.u32 u, %31, 0;\n"
        " add.u32 %0, %29, %30;\n"
        " setp.ge.and.u32 r, %0, %29, u;\n @r sub.u32 %2, %2, 128;\n"
        " setp.lt.and.u32 p, %0, %29, !u;\n @p ld.shared.v4.f32 {%11, %12, %13, %14}, [%2 + %32];\n"
        " @p add.u32 %2, %2, 128;\n"
        " ld.shared.v4.f32 {%19, %20, %21, %22}, [%2 + %32];\n"
        " add.u32 %1, %0, %30;\n"
        " setp.ge.and.u32 t, %1, %0, u;\n @t sub.u32 %2, %2, 128;\n"
        " setp.lt.and.u32 q, %1, %0, !u;\n @q ld.shared.v4.f32 {%15, %16, %17, %18}, [%2 + %33];\n"
        " @q add.u32 %2, %2, 128;\n"
        " ld.shared.v4.f32 {%23, %24, %25, %26}, [%2 + %33];\n"
        " selp.u32 %27, 1, 0, r;\n selp.u32 %28, 1, 0, t;\n"
        " @p add.f32 %3, %3, %11;\n @p add.f32 %4, %4, %12;\n @p add.f32 %5, %5, %13;\n @p add.f32 %6, %6, %14;\n"
        " @q add.f32 %7, %7, %15;\n @q add.f32 %8, %8, %16;\n @q add.f32 %9, %9, %17;\n @q add.f32 %10, %10, %18;\n}"
        : "=&r"(n1), "=&r"(n2), "+r"(b), "+f"(o.x), "+f"(o.y), "+f"(o.z), "+f"(o.w), "+f"(o2.x), "+f"(o2.y),
          "+f"(o2.z), "+f"(o2.w), "+f"(m[0].x), "+f"(m[0].y), "+f"(m[0].z), "+f"(m[0].w), "+f"(m[1].x), "+f"(m[1].y),
          "+f"(m[1].z), "+f"(m[1].w), "=&f"(d1.x), "=&f"(d1.y), "=&f"(d1.z), "=&f"(d1.w), "=&f"(d2.x), "=&f"(d2.y),
          "=&f"(d2.z), "=&f"(d2.w), "=&r"(stay1), "=&r"(stay2)
        : "r"(n), "r"(step), "r"((unsigned)below), "n"(I * 128), "n"(I * 128 + 128));
    w1 = stay1 ? -frac_g(n1) : frac_f(n1);
    w2 = stay2 ? -frac_g(n2) : frac_f(n2);
  } else {
    asm volatile(
        "{\n .reg .pred p, q;\n"
        " add.u32 %0, %27, %28;\n"
        " setp.lt.u32 p, %0, %27;\n @p ld.shared.v4.f32 {%11, %12, %13, %14}, [%2 + %29];\n"
        " @p add.u32 %2, %2, 128;\n"
        " ld.shared.v4.f32 {%19, %20, %21, %22}, [%2 + %29];\n"
        " add.u32 %1, %0, %28;\n"
        " setp.lt.u32 q, %1, %0;\n @q ld.shared.v4.f32 {%15, %16, %17, %18}, [%2 + %30];\n"
        " @q add.u32 %2, %2, 128;\n"
        " ld.shared.v4.f32 {%23, %24, %25, %26}, [%2 + %30];\n"
        " @p add.f32 %3, %3, %11;\n @p add.f32 %4, %4, %12;\n @p add.f32 %5, %5, %13;\n @p add.f32 %6, %6, %14;\n"
        " @q add.f32 %7, %7, %15;\n @q add.f32 %8, %8, %16;\n @q add.f32 %9, %9, %17;\n @q add.f32 %10, %10, %18;\n}"
        : "=&r"(n1), "=&r"(n2), "+r"(b), "+f"(o.x), "+f"(o.y), "+f"(o.z), "+f"(o.w), "+f"(o2.x), "+f"(o2.y),
          "+f"(o2.z), "+f"(o2.w), "+f"(m[0].x), "+f"(m[0].y), "+f"(m[0].z), "+f"(m[0].w), "+f"(m[1].x), "+f"(m[1].y),
          "+f"(m[1].z), "+f"(m[1].w), "=&f"(d1.x), "=&f"(d1.y), "=&f"(d1.z), "=&f"(d1.w), "=&f"(d2.x), "=&f"(d2.y),
          "=&f"(d2.z), "=&f"(d2.w)
        : "r"(n), "r"(step), "n"(I * 128), "n"(I * 128 + 128));
    w1 = frac_f(n1);
    w2 = frac_f(n2);
  }
  fma4(o, w1, d1);
  fma4(o2, w2, d2);
  fma4(o2, frac_g(n1), d1);
  if constexpr (I + 1 < kLines) fma4(acc[I + 1], frac_g(n2), d2);
  n = n2;
  if constexpr (I + 2 < kLines) two_lines<NEAR, I + 2>(b, n, step, below, m, acc);
}

// One step of a lane's lines: the first at cell address b and fraction n, each next one
// `step` further (its fraction; 1 + step / 2^32 cells, or without the 1 where `below`).
// NEAR: some line spacing of the warp is below one cell, so that two lines may share a cell.
template <bool NEAR>
__device__ __forceinline__ void walk_step(unsigned b, unsigned n, unsigned step, bool below, float4 (&m)[2],
                                          float4 (&acc)[kLines]) {
  fma4(acc[0], frac_g(n), load4(b));
  two_lines<NEAR, 1>(b, n, step, below, m, acc);
}

// Second level of the sums, in tensor memory (a lane's 64 accumulators take all its
// registers, the ring all shared memory): every kFold steps the accumulators are added to
// it and keep what the addition rounds off, which the next fold takes along.  Rounding then
// grows with the kFold steps of a block instead of all of up to 2048.  Error over max|S|
// against 64 bits, in a restatement on the CPU over 40 grids of 160 to 976 pixels: of white
// noise at most 0.57 times that of the view-by-view form (one level, lines stepped in FP32:
// 3.7), of smooth images 0.26 times (1.5).  Blocks of 16 steps: 0.51 and 0.14.
constexpr int kFold = 32;
constexpr unsigned kTmemCols = 64 * kWarps / 4;  // a warp owns 32 lanes and 64 columns

// Where a warp's part starts: its 32 lanes in the upper half of the address, its columns below.
__device__ __forceinline__ unsigned tmem_of(unsigned base, int warp) {
  return base + ((unsigned)(warp & 3) << 21) + 64u * (unsigned)(warp >> 2);
}
// Eight columns of the lane's second level (more at a time would spill).  The wait belongs
// to the load: the registers are not valid before it.
__device__ __forceinline__ void tmem_load(unsigned at, float4 (&v)[2]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
      " tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[0].z), "=f"(v[0].w), "=f"(v[1].x), "=f"(v[1].y), "=f"(v[1].z), "=f"(v[1].w)
      : "r"(at)
      : "memory");
}
__device__ __forceinline__ void tmem_store(unsigned at, const float4 (&v)[2]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};" ::"f"(v[0].x),
               "f"(v[0].y), "f"(v[0].z), "f"(v[0].w), "f"(v[1].x), "f"(v[1].y), "f"(v[1].z), "f"(v[1].w), "r"(at)
               : "memory");
}
__device__ __forceinline__ void tmem_stored() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// s += y, y = what that rounds off.
__device__ __forceinline__ void fold1(float& s, float& y) {
  const float t = s + y;
  y = y - (t - s);
  s = t;
}
__device__ __forceinline__ void fold(unsigned at, float4 (&acc)[kLines]) {
#pragma unroll
  for (int c = 0; c < kLines / 2; ++c) {
    float4 s[2];
    tmem_load(at + 8 * c, s);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      float4& y = acc[2 * c + i];
      fold1(s[i].x, y.x);
      fold1(s[i].y, y.y);
      fold1(s[i].z, y.z);
      fold1(s[i].w, y.w);
    }
    tmem_store(at + 8 * c, s);
  }
  tmem_stored();
}

__global__ void __launch_bounds__(32 * kWarps, 1) radon_views_kernel(const RadonRow* table, const RadonView* rv,
                                                                     const float* planes, ViewsArgs g,
                                                                     float* __restrict__ out_f32,
                                                                     __nv_bfloat16* __restrict__ out_bf16,
                                                                     int* __restrict__ status) {
  wait_for_previous();
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) u64 bars[2 * kMaxSlots];
  __shared__ unsigned windows[kMaxSteps];   // of each step: start in the plane, cells << 16
  __shared__ int range[kWarps][2];          // steps of each warp
  __shared__ longlong2 line[kUnits];        // first line of each unit at step 0, advance per step
  __shared__ long long span[kUnits];        // from its first line to its last
  __shared__ int armed[kMaxSlots];          // parity of the last phase a slot's copies were issued in, -1: none
  __shared__ int failed, widest;
  __shared__ unsigned tmem_base;
  const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
  const int sub = lane >> 3, vl = lane & 7;
  // alpha rows of the tile: tiles of the two segments stepping over rows, then of the columns
  const int t1 = (g.r1 + g.A - 1) / g.A, t2 = t1 + (g.n_alpha - g.r2 + g.A - 1) / g.A;
  const int ty = (int)blockIdx.y + (g.axis == 1 ? t2 : 0);
  const bool cols = ty >= t2;
  const int m0 = cols ? g.r1 + (ty - t2) * g.A : ty >= t1 ? g.r2 + (ty - t1) * g.A : ty * g.A;
  const int m_end = cols ? g.r2 : ty >= t1 ? g.n_alpha : g.r1;
  const int steps = cols ? g.W : g.H, cells = cols ? g.H : g.W;
  const int pitch = cells + 1 + 2 * g.pad;
  const float* plane =
      planes + (cols ? g.cols0 : 0) + (size_t)blockIdx.z * steps * pitch * kGroup;
  const int blocks = g.A / kRows;  // of the alpha rows of one warp
  const int m_warp = m0 + (warp % blocks) * kRows;
  const int my_m = min(m_warp + sub, m_end - 1);
  const int k0 = ((int)blockIdx.x * (kWarps / blocks) + warp / blocks) * kLines;
  const bool live = m_warp + sub < m_end && k0 < g.n_s;
  const RadonRow row = table[my_m];
  // lines in the order of increasing position: k0 .. k0 + 16, or back where the step is negative
  const bool rev = row.STEP < 0;
  const long long step_q = rev ? -row.STEP : row.STEP;
  const unsigned step = (unsigned)step_q;      // fraction of the line spacing
  const bool below = step_q < (1ll << 32);     // the spacing is below one cell (and below two always)
  const long long first = row.B0 + (long long)(rev ? k0 + kLines : k0) * row.STEP;  // at step 0
  int lo_w = 0, hi_w = 0;
  if (live) {
    const float q = 1.0f / 65536.0f;
    step_range((float)(first >> 16) * q, (float)((first + kLines * step_q) >> 16) * q, (float)(row.DY >> 16) * q, steps,
               cells, lo_w, hi_w);
  }
  {  // a warp walks the steps of all its lines
    const bool some = hi_w > lo_w;
    lo_w = __reduce_min_sync(0xffffffffu, some ? lo_w : steps);
    hi_w = __reduce_max_sync(0xffffffffu, some ? hi_w : 0);
    if (hi_w < lo_w) hi_w = lo_w;
  }
  const bool near = __any_sync(0xffffffffu, below);
  const unsigned bar0 = smem_u32(bars);
  if (lane == 0) {
    range[warp][0] = lo_w;
    range[warp][1] = hi_w;
  }
  if (vl == 0) {
    const int u = warp * kRows + sub;
    line[u] = make_longlong2(first, row.DY);
    span[u] = kLines * step_q;
  }
  if (threadIdx.x == 0) {
    failed = widest = 0;
    for (int i = 0; i < kMaxSlots; ++i) {
      armed[i] = -1;
      mbar_init(bar0 + 8 * i, 1);
      mbar_init(bar0 + 8 * (kMaxSlots + i), kWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {  // the only CTA of its SM (shared memory), so that the columns are free
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "n"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  int j_lo = steps, j_hi = 0;
  for (int w = 0; w < kWarps; ++w)
    if (range[w][1] > range[w][0]) {
      j_lo = min(j_lo, range[w][0]);
      j_hi = max(j_hi, range[w][1]);
    }
  const int n_steps = max(j_hi - j_lo, 0);
  // the window of every step: the cells between the first and the last line of the warps
  // that walk it, with one of margin on either side for the FP32 rounding of positions
  int most = 0;
  for (int n = threadIdx.x; n < n_steps; n += 32 * kWarps) {
    int mn = 0x3fffffff, mx = -0x3fffffff;
    for (int w = 0; w < kWarps; ++w)
      if (j_lo + n >= range[w][0] && j_lo + n < range[w][1])
#pragma unroll
        for (int u = w * kRows; u < (w + 1) * kRows; ++u) {
          const longlong2 l = line[u];
          const long long X = l.x + (long long)(j_lo + n) * l.y;
          mn = min(mn, (int)(X >> 32) - 1);
          mx = max(mx, (int)((X + span[u]) >> 32) + 1);
        }
    const int at = min(max(mn + 1 + g.pad, 0), pitch - 1);
    const int cnt = mx >= mn ? min(min(mx - mn + 1, g.win), pitch - at) : 0;
    windows[n] = (unsigned)at | (unsigned)cnt << 16;
    most = max(most, cnt);
  }
  most = __reduce_max_sync(0xffffffffu, most);
  if (lane == 0) atomicMax(&widest, most);
  __syncthreads();
  const unsigned slot_bytes = (unsigned)max(widest, 1) * kCell;
  const int slots = min(kMaxSlots, (int)((unsigned)kRing / slot_bytes));
  const unsigned slot0 = smem_u32(smem);
  bool ok = true;
  // one lane: copies the window of step n into its slot, whose phase has this parity
  auto refill = [&](int n, int slot, int parity) {
    const unsigned w = windows[n], bytes = (w >> 16) * kCell, bar = bar0 + 8 * slot;
    armed[slot] = parity;
    mbar_expect(bar, bytes);
    if (bytes)
      bulk_copy(slot0 + slot * slot_bytes, plane + ((size_t)(j_lo + n) * pitch + (w & 0xffffu)) * kGroup, bytes, bar);
  };
  if (lane == 0)
    for (int n = warp; n < min(slots, n_steps); n += kWarps) refill(n, n, 0);
  __syncwarp();

  float4 acc[kLines];
#pragma unroll
  for (int i = 0; i < kLines; ++i) acc[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  float4 m[2] = {acc[0], acc[0]};
  for (int c = 0; c < kLines / 2; ++c) tmem_store(tmem_of(tmem_base, warp) + 8 * c, m);  // zeros
  tmem_stored();
  auto walk = [&](auto near_lines) {
    long long X = first + (long long)lo_w * row.DY;
    const int n_lo = lo_w - j_lo, n_hi = hi_w - j_lo;
    unsigned slot_at = slot0 + vl * 16 + (1 + g.pad) * kCell;
    const unsigned slot_end = slot_at + slots * slot_bytes;
    unsigned full = bar0, turn = 0;   // of step n
    int slot_r = 0, turn_r = 0;       // of step n - kLag: the slot to refill
    unsigned window_at = smem_u32(windows);
    for (int n = 0; n < n_steps; ++n, window_at += 4) {
      if (n >= kLag) {
        if ((n & (kWarps - 1)) == warp && n - kLag + slots < n_steps) {
          if (lane == 0 && mbar_wait(bar0 + 8 * (kMaxSlots + slot_r), turn_r, g.wait_ns, g.hint, &failed))
            refill(n - kLag + slots, slot_r, turn_r ^ 1);
          __syncwarp();
        }
        if (++slot_r == slots) {
          slot_r = 0;
          turn_r ^= 1;
        }
      }
      ok = mbar_wait_warp(full, turn, g.wait_ns, g.hint, &failed);
      if (!ok) break;  // warp-uniform
      if (n >= n_lo && n < n_hi) {
        // exact positions of all lines: whole cells and a 32-bit fraction
        unsigned window;
        asm volatile("ld.shared.u16 %0, [%1];" : "=r"(window) : "r"(window_at));
        const unsigned b = slot_at + (unsigned)((int)(X >> 32) - (int)window) * kCell;
        walk_step<decltype(near_lines)::value>(b, (unsigned)X, step, below, m, acc);
        X += row.DY;
        if (((n - n_lo) & (kFold - 1)) == kFold - 1) fold(tmem_of(tmem_base, warp), acc);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(full + 8 * kMaxSlots);
      full += 8;
      slot_at += slot_bytes;
      if (slot_at == slot_end) {
        slot_at -= slots * slot_bytes;
        full = bar0;
        turn ^= 1;
      }
    }
  };
  if (near)
    walk(std::true_type{});
  else
    walk(std::false_type{});
  // each accumulator and its second level together
#pragma unroll
  for (int c = 0; c < kLines / 2; ++c) {
    float4 s[2];
    tmem_load(tmem_of(tmem_base, warp) + 8 * c, s);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      float4& a = acc[2 * c + i];
      a = make_float4(s[i].x + a.x, s[i].y + a.y, s[i].z + a.z, s[i].w + a.w);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  // A wait that gave up is reported.  No warp issues copies any more; those in flight land
  // before the shared memory is given back.
  const bool gave_up = __syncthreads_or(!ok || failed);
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(kTmemCols) : "memory");
  }
  if (gave_up) {
    if (threadIdx.x < kMaxSlots && armed[threadIdx.x] >= 0)
      mbar_wait(bar0 + 8 * threadIdx.x, (unsigned)armed[threadIdx.x], kWaitNs, g.hint, nullptr);
    if (threadIdx.x == 0) atomicOr(status, kStatusTimeout);
    __syncthreads();
    return;
  }
  // transpose through shared memory: [alpha row][view][line], then runs of 16 outputs
  constexpr int kPitch = kLines + 1;
  float* __restrict__ mine = reinterpret_cast<float*>(smem) + warp * (kRows * kGroup * kPitch);
  const float norm = row.inv_len / g.ds * (rev ? -1.0f : 1.0f);
#pragma unroll
  for (int i = 0; i < kLines; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e)
      mine[(sub * kGroup + vl * 4 + e) * kPitch + (rev ? kLines - 1 - i : i)] =
          (e == 0 ? acc[i].x : e == 1 ? acc[i].y : e == 2 ? acc[i].z : acc[i].w) * norm;
  __syncwarp();
  const int vbase = (int)blockIdx.z * kGroup;
  for (int a = 0; a < kRows; ++a) {
    const int ma = m_warp + a;
    if (ma >= m_end) break;
    const float ca = table[ma].ca, sa = table[ma].sa;
    for (int i = lane; i < kGroup * kLines; i += 32) {
      const int v = vbase + i / kLines, k = k0 + i % kLines;
      if (v < g.n_views && k < g.n_s) {
        const RadonView r = rv[v];
        const float sn = ((float)k - 0.5f * (float)(g.n_s - 1)) * g.ds;
        const float spp = sn - (r.u0 - 0.5f * (float)(g.W - 1)) * ca - (r.v0 - 0.5f * (float)(g.H - 1)) * sa;
        const float val =
            mine[(a * kGroup + i / kLines) * kPitch + i % kLines] * ((r.D * r.D + spp * spp) / (r.D * r.D));
        const size_t o = ((size_t)v * g.n_alpha + ma) * g.n_s + k;
        if (out_bf16)
          out_bf16[o] = __float2bfloat16_rn(val);
        else
          out_f32[o] = val;
      }
    }
  }
}

// ---------------------------------------------------------------- plan

double spacing(int W, int H, int n_s) {  // of the lines in cells, at 45 degrees (the widest)
  return std::sqrt((double)W * W + (double)H * H) / (n_s - 1) * 1.41421356237309515;
}

// Zero cells on either side of a step: where one line of a warp is inside the image,
// others may be up to the width of its chunk and the turn of its alpha rows outside.
int pad_of(int W, int H, int n_alpha, double s_max) {
  const double turn = 3.14159265358979323846 / n_alpha * (kRows - 1);
  const double lines = kLines * s_max + 4.0;
  const double reach = 0.5 * std::sqrt((double)W * W + (double)H * H) + lines + 16.0;
  return (int)std::ceil(lines + 1.41421356237309515 * turn * reach * (1.0 + turn)) + 8;
}

// Cells that the lines of one CTA can span at one step: its chunks side by side and the
// turn of its alpha rows about the detector centre, over the half diagonal and the
// lines that reach past it.
int window_of(int A, int W, int H, int n_alpha, double s_max) {
  const double lines = (double)(kUnits / A) * kLines * s_max;
  const double reach = 0.5 * std::sqrt((double)W * W + (double)H * H) + 0.5 * lines + 8.0;
  const double da = 3.14159265358979323846 / n_alpha * (A - 1);
  return (int)std::ceil(lines + 1.41421356237309515 * da * reach * (1.0 + da)) + 5;
}

}  // namespace

size_t ViewsPlan::group_bytes(int axes, int W, int H, int n_alpha, int n_s) {
  const size_t pad = (size_t)pad_of(W, H, n_alpha, spacing(W, H, n_s));
  const size_t rows = (size_t)H * (W + 1 + 2 * pad), cols = (size_t)W * (H + 1 + 2 * pad);
  return (axes == 2 ? rows + cols : std::max(rows, cols)) * kCell;
}

// Alpha rows per CTA: those with the narrowest window; 0: none fits, or neighbouring lines
// are two cells or more apart.
static int alphas_of(int W, int H, int n_alpha, int n_s) {
  const double s_max = spacing(W, H, n_s);
  if (s_max > 1.999 || std::max(W, H) > kMaxSteps) return 0;
  int best = 0, best_win = kRing / (int)(kMinSlots * kCell) + 1;
  for (int A = kUnits; A >= kRows; A /= 2) {
    const int w = window_of(A, W, H, n_alpha, s_max);
    if (w < best_win) {
      best = A;
      best_win = w;
    }
  }
  return best;
}

struct Tiles {  // CTAs of one group: alpha rows per CTA, tiles of the row and column modes, chunks of lines
  int A, r1, r2, rows, cols, chunks;
};
static Tiles tiles_of(int W, int H, int n_alpha, int n_s) {
  Tiles t{};
  t.A = alphas_of(W, H, n_alpha, n_s);
  t.r1 = n_alpha / 4 + 1;  // rows: 4 m <= n_alpha or 4 m >= 3 n_alpha
  t.r2 = (3 * n_alpha + 3) / 4;
  if (t.A == 0) return t;
  const int per = kUnits / t.A * kLines;
  t.rows = (t.r1 + t.A - 1) / t.A + (n_alpha - t.r2 + t.A - 1) / t.A;
  t.cols = (t.r2 - t.r1 + t.A - 1) / t.A;
  t.chunks = (n_s + per - 1) / per;
  return t;
}

// A group takes as long as about 16 views of the view-by-view form where its CTAs fill the
// GPU for some waves (one group of 16 views against 15 view by view, in us: 1,778 and 1,646 on
// 620 x 480, 6,411 and 6,363 on 976 x 976), and longer in proportion where they do not
// (300 x 260, 221 CTAs a group: 23 views 506, view by view 22 take 484; 256 x 256, 102 CTAs:
// 48 and 47 views 434 and 484).  Where lines are closer together than a cell (windows with
// more lines) it takes up to half as long again; there from the second group on, whose last
// views may be few (168 views of 18 x 126, ds = 0.46: 188 and 188).  A rule on the sizes
// alone, at which the two forms took about the same time on ten grids: two waves of a GPU of
// 152 SMs.
int ViewsPlan::min_views(int W, int H, int n_alpha, int n_s) {
  const Tiles t = tiles_of(W, H, n_alpha, n_s);
  if (t.A == 0) return 0;
  const double ctas = (double)(t.rows + t.cols) * t.chunks;
  const bool close = std::sqrt((double)W * W + (double)H * H) / (n_s - 1) < 0.99;
  const double least = std::max(close ? 48.0 : 16.0, 16.0 * 304.0 / ctas * (close ? 1.5 : 1.0));
  return (int)std::ceil(least);
}

cudaError_t launch_radon_views(const RadonRow* table, const RadonView* rv, int n_views, const float* images, int W,
                               int H, int n_alpha, int n_s, void* scratch, size_t scratch_bytes, float* of,
                               __nv_bfloat16* ob, int* status, u64 wait_ns, bool behind, const LaunchHooks& hooks,
                               cudaStream_t stream) {
  const double s_max = spacing(W, H, n_s);
  ViewsArgs g{};
  g.W = W;
  g.H = H;
  g.n_alpha = n_alpha;
  g.n_s = n_s;
  g.ds = (float)(std::sqrt((double)W * W + (double)H * H) / (n_s - 1));
  g.wait_ns = wait_ns;
  g.hint = (unsigned)std::min<u64>(wait_ns, 20000);
  const Tiles t = tiles_of(W, H, n_alpha, n_s);
  g.A = t.A;
  g.r1 = t.r1;
  g.r2 = t.r2;
  g.pad = pad_of(W, H, n_alpha, s_max);
  g.win = window_of(g.A, W, H, n_alpha, s_max);
  const size_t out_bytes = sizeof(float) * kWarps * kRows * kGroup * (kLines + 1);
  const size_t shared = std::max((size_t)kRing, out_bytes);
  cudaError_t e = cudaFuncSetAttribute(radon_views_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shared);
  if (e != cudaSuccess) return e;
  const size_t grid = (size_t)n_alpha * n_s, px = (size_t)W * H;
  const size_t pitch_r = (size_t)W + 1 + 2 * g.pad;
  // the planes of both axes at once, or of one at a time where both do not fit
  const int axes = ViewsPlan::group_bytes(2, W, H, n_alpha, n_s) > scratch_bytes ? 1 : 2;
  const int fit = (int)std::min<size_t>(4096, scratch_bytes / ViewsPlan::group_bytes(axes, W, H, n_alpha, n_s));
  float* planes = static_cast<float*>(scratch);
  for (int v = 0; v < n_views; v += fit * kGroup) {
    g.n_views = std::min(n_views - v, fit * kGroup);
    const int groups = (g.n_views + kGroup - 1) / kGroup;
    for (int pass = 0; pass < (axes == 2 ? 1 : 2); ++pass) {
      g.axis = axes == 2 ? 2 : pass;
      g.cols0 = g.axis == 2 ? (size_t)groups * H * pitch_r * kGroup : 0;
      hooks.on_begin("weight_views_kernel", stream);
      launch_at(behind, weight_views_kernel, dim3((W + kTileX) / kTileX, (H + kTileY) / kTileY, groups), 256, 0, stream,
                images + (size_t)v * px, rv + v, g, planes);
      hooks.on_end("weight_views_kernel", stream);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      const int tiles = (g.axis != 1 ? t.rows : 0) + (g.axis != 0 ? t.cols : 0);
      if (tiles == 0) continue;
      hooks.on_begin("radon_views_kernel", stream);
      launch_behind(radon_views_kernel, dim3(t.chunks, tiles, groups), 32 * kWarps, shared, stream, table, rv + v,
                    planes, g, of ? of + (size_t)v * grid : nullptr, ob ? ob + (size_t)v * grid : nullptr, status);
      hooks.on_end("radon_views_kernel", stream);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

}  // namespace ecc
