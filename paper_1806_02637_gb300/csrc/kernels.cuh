// Kernel declarations shared by the translation units of the library.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include "ecc_internal.cuh"

namespace ecc {

// pairs [p_begin, p_end) of the row-major a < b enumeration (pairs == NULL) or of the list
__global__ void view_grad_theta_kernel(int n_views, long long n_pairs, const int32_t* pairs, const float2* gq,
                                       const ViewTan* vtan, double* grad);
constexpr int kGradQThreads = 64;
__global__ void pair_grad_q_kernel(long long n_pairs, const PairRec* prs, const ViewRec* views, const double* Gpp,
                                   float2* gq, const double* partial, int n_partial, double* total);
__global__ void view_grad_P_kernel(int n_views, long long n_pairs, const int32_t* pairs, const float2* gq,
                                   const ViewTanP* vtan, double* grad_P);

// Line parameters of the Joseph line sums at one alpha row (32.32 fixed point).
struct RadonRow {
  long long B0;    // coordinate along the interpolation axis at rho index 0, step 0
  long long STEP;  // per rho index
  long long DY;    // per step along the integration axis
  float inv_len;   // path length per step: 1/|cos a| (rows) or 1/|sin a| (columns)
  float ca, sa;    // cos, sin of alpha
  int rows_mode;   // 1: step over image rows, interpolate in x; 0: columns
};

struct RadonView {  // per-view weights (FP32 copies of the FP64 set-up)
  float u0, v0, D;
  unsigned max_bits;  // max |S| of a view staged for FP16, as bits
};

// The FP64 work of a call that depends on its geometry alone, in one launch: what is not
// wanted is NULL.
struct Geometry {
  int n_views, W, H;
  const double* P;       // [n_views][12]
  const double* motion;  // [n_views][6] or NULL
  ViewRec* views;        // per-view set-up
  int* status;
  RadonView* weights;    // of the dRadon/ds precompute
  ViewTan* tan;          // tangents with respect to the motion
  ViewTanP* tanP;        // and with respect to P
  int n_alpha, n_s;
  float4* alpha_dir;     // alpha-row directions
  RadonRow* table;       // line table of the precompute, `copies` times
  int copies;
};

// Callbacks around every kernel launch (launch counting and optional CUDA-event
// timing by the context).
struct LaunchHooks {
  void (*begin)(void* ctx, const char* name, cudaStream_t s) = nullptr;
  void (*end)(void* ctx, const char* name, cudaStream_t s) = nullptr;
  void* ctx = nullptr;
  void on_begin(const char* n, cudaStream_t s) const {
    if (begin) begin(ctx, n, s);
  }
  void on_end(const char* n, cudaStream_t s) const {
    if (end) end(ctx, n, s);
  }
};

// Kernels of a call that are launched behind the one before (programmatic dependent launch)
// wait for its end and its stores as their first step: their launch and their blocks' start
// overlap its end.  What earlier kernels write is then not read-only for their duration: they
// take it through pointers without const __restrict__ and never through __ldg, whose loads may
// be non-coherent and may move ahead of the wait.  Starting early takes 2 us to 5 us off a
// call of several short kernels (motion gradient of 248 views 285 -> 282 us, evaluation of one
// pair 37.2 -> 35.0 us, two-view precompute 43.8 -> 40.8 us).  Launched plainly: the first
// kernel of a call, which waits for whatever the stream did before; pair_setup_kernel and ecc_pair_kernel, because an SM that
// never falls idle between them keeps the first one's split of L1 and shared memory, at which
// fewer blocks of the second fit (evaluation of the 496-view scan 567 -> 747 us).
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() {
  let_next_start();
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <class... K, class... A>
void launch_at(bool behind, void (*kernel)(K...), dim3 grid, dim3 block, size_t shared, cudaStream_t stream,
               A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = shared;
  c.stream = stream;
  c.attrs = &at;
  c.numAttrs = behind ? 1 : 0;
  cudaLaunchKernelEx(&c, kernel, K(args)...);  // the caller reads cudaGetLastError
}
template <class... K, class... A>
void launch_behind(void (*kernel)(K...), dim3 grid, dim3 block, size_t shared, cudaStream_t stream, A... args) {
  launch_at(true, kernel, grid, block, shared, stream, args...);
}

// Fixed-order sum of n block partials by one block of THREADS threads: as many chunks as
// slots, one after the other, then a tree, whatever THREADS.
constexpr int kSumSlots = 1024;
template <int THREADS>
__device__ __forceinline__ void reduce_fixed(const double* partial, int n, double* __restrict__ total,
                                             double* s) {
  const int per = (n + kSumSlots - 1) / kSumSlots;
#pragma unroll 4
  for (int t = threadIdx.x; t < kSumSlots; t += THREADS) {
    double acc = 0.0;
    const int end = min(n, (t + 1) * per);
    for (int i = t * per; i < end; ++i) acc += partial[i];
    s[t] = acc;
  }
  __syncthreads();
  for (int w = kSumSlots / 2; w > 0; w >>= 1) {
    for (int t = threadIdx.x; t < w; t += THREADS) s[t] += s[t + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = s[0];
}

// Parameters of the pair kernel for one scan (device pointers).
struct PairArgs {
  long long n_pairs;
  const PairRec* prs;
  const float4* ctile;      // tile-centre directions (hi.x, hi.y, lo.x, lo.y)
  int n_tiles;
  const float4* alpha_dir;  // alpha-row directions (cos, sin as double-float pairs)
  const void* sino;
  const float* scales;  // FP16 storage only, else NULL
  int n_alpha, n_s, K;
  // grid constants (set by pair_args_grid): alpha rows per radian, s bins per pixel
  // (FP32 and as a double-float pair), and (n_s - 1) / 2 as a double-float pair
  float inv_dalpha, inv_ds_f, inv_ds_hi, inv_ds_lo, half_hi, half_lo;
  float cauchy_c;
  double* per_pair;
  int32_t* nk_out;
  double* block_partial;
  double* Gpp;  // adjoint output, NULL for the plain evaluation
  int* status;  // device status word (kStatus* bits OR-ed in), or NULL
};

inline void pair_args_grid(PairArgs& g, int n_alpha, int n_s, int W, int H) {
  const double inv_ds = (double)(n_s - 1) / std::sqrt((double)W * W + (double)H * H);
  const double inv_dalpha = (double)n_alpha / 3.14159265358979323846;
  const double half = 0.5 * (n_s - 1);
  g.n_alpha = n_alpha;
  g.n_s = n_s;
  g.inv_dalpha = (float)inv_dalpha;
  g.inv_ds_f = (float)inv_ds;
  g.inv_ds_hi = (float)inv_ds;
  g.inv_ds_lo = (float)(inv_ds - (double)g.inv_ds_hi);
  g.half_hi = (float)half;
  g.half_lo = (float)(half - (double)g.half_hi);
}

// How a dRadon/ds precompute runs.  Scans with enough views whose grid qualifies follow the
// detector lines once for many views (radon_views.cu), others view by view (radon.cu); the
// two round differently.  The choice depends on the grid, on the number of views of the scan
// (n_scan: of this call, or of the scan that the call's views are part of) and on the scratch
// that the call may take.  The many-view sums do not depend on how the views are grouped.
constexpr unsigned long long kWaitNs = 1000000000ull;  // a bounded device wait gives up after this long
struct RadonPlan {
  unsigned long long wait_ns = kWaitNs;
  bool views;          // many views at once
  int batch;           // views per pass over the scratch
  int lead;            // views of the first pass; each next one takes four times as many, up to batch
  int passes(int n_views) const {
    long long v = 0, size = lead;
    int p = 0;
    for (; v < n_views && size < batch; ++p, size = std::min<long long>(4 * size, batch)) v += size;
    return p + (int)(v < n_views ? (n_views - v + batch - 1) / batch : 0);
  }
  int begin(int pass) const {
    long long v = 0, size = lead;
    int p = 0;
    for (; p < pass && size < batch; ++p, size = std::min<long long>(4 * size, batch)) v += size;
    return (int)std::min<long long>(v + (pass - p) * size, 0x7fffffff);
  }
  int count(int pass, int n_views) const { return std::min(begin(pass + 1), n_views) - begin(pass); }
  size_t wimg_bytes;   // weighted images
  size_t stage_bytes;  // FP32 staging of FP16 storage
  // the line table (copies of n_alpha rows) and the per-view weights after it
  int copies(int n_views) const { return views ? 1 : n_views; }
  size_t table_bytes(int n_views, int n_alpha) const {
    return sizeof(RadonRow) * (size_t)copies(n_views) * n_alpha + sizeof(RadonView) * (size_t)n_views;
  }
  RadonView* weights(RadonRow* table, int n_views, int n_alpha) const {
    return reinterpret_cast<RadonView*>(table + (size_t)copies(n_views) * n_alpha);
  }
};
// Scratch that a many-view plan may take: weighted images, FP16 staging, and both together.
struct RadonRoom {
  size_t wimg = SIZE_MAX, stage = SIZE_MAX, total = SIZE_MAX;
};
// The many-view form in as many groups of 32 views at once as fit the room.  Where none fits,
// or the scan does not qualify, the plan is the view-by-view form's, which follows no limit.
RadonPlan radon_plan(int n_scan, int n_views, int W, int H, int n_alpha, int n_s, int dtype, const RadonRoom& room);
RadonPlan radon_plan_by_view(int n_views, int W, int H, int n_alpha, int n_s, int dtype);

// Many-view form, in groups of 32 views.
struct ViewsPlan {
  // least number of views for which the many-view form is taken; 0: the grid does not qualify
  static int min_views(int W, int H, int n_alpha, int n_s);
  // scratch of one group with the planes of both axes (2) or of one at a time (1)
  static size_t group_bytes(int axes, int W, int H, int n_alpha, int n_s);
};

// Launchers (return cudaError_t of the launch).
cudaError_t launch_geometry(const Geometry& g, const LaunchHooks& hooks, cudaStream_t stream);
cudaError_t launch_pair_setup(int n_views, long long n_pairs, const int32_t* pairs, const ViewRec* views, int W, int H,
                              int K, PairRec* out, float4* ctile, int n_tiles, bool reuse_sampling, int* status,
                              const LaunchHooks& hooks, cudaStream_t stream);
cudaError_t launch_radon(int n_views, const float* images, int W, int H, int n_alpha, int n_s, int dtype,
                         void* sino_out, float* scales_out, const RadonRow* table, void* wimg, float* stage,
                         const RadonPlan& plan, int* status, const LaunchHooks& hooks, cudaStream_t stream,
                         const cudaEvent_t* batch_ready = nullptr);  // per pass: wait before reading its images
cudaError_t launch_radon_views(const RadonRow* table, const RadonView* rv, int n_views, const float* images, int W,
                               int H, int n_alpha, int n_s, void* planes, size_t plane_bytes, float* of,
                               __nv_bfloat16* ob, int* status, unsigned long long wait_ns, bool behind,
                               const LaunchHooks& hooks, cudaStream_t stream);

cudaError_t launch_ecc_pairs(long long n_pairs, const PairRec* prs, const float4* ctile, int n_tiles,
                             const float4* alpha_dir, const void* sino, const float* scales, int dtype,
                             int n_alpha, int n_s, int K, int W, int H, double cauchy_c, double* per_pair, int32_t* nk_out,
                             double* block_partial, double* Gpp, int* status, int* n_blocks_out,
                             const LaunchHooks& hooks, cudaStream_t stream);

cudaError_t launch_reduce(const double* partial, int n, double* total, const LaunchHooks& hooks,
                          cudaStream_t stream);

// ---------------------------------------------------------------- serving rounds
// One active job of a serving round (device copy of the scheduler's table).  Every
// round evaluates each job's total and, with do_grad, its gradient and one step
// theta <- theta - step * grad.  The kernels below cover all jobs of a round; a
// flattened index (view, pair or pair block) is mapped to its job by binary search
// over the per-job prefix offsets (n_jobs + 1 entries each).
struct ServeJob {
  PairArgs pair;  // pair kernel parameters (block_partial and Gpp set, per_pair/nk_out NULL)
  int dtype;
  int n_views, W, H, n_tiles;
  int do_grad;
  double step;
  const double* P;   // [n_views][12]
  double* theta;     // [n_views][6]
  double* grad;      // [n_views][6]
  ViewRec* views;
  ViewTan* vtan;
  float2* gpp;        // [n_pairs][30] d e / d (C, up, cofc) of views a and b, double-float pairs
  double* total_out;  // this round's total
  int* status;
  // motion model: per-view (theta stepped directly) or Akima spline of node values
  int model, n_nodes, mask;  // mask: estimated parameters (bits 0..5)
  double h;                  // node spacing in views
  const double* theta0;      // [n_views][6] fixed part (motion0)
  double* nodes;             // [n_nodes][6]
  double* jac;               // [n_views][6][6] d theta / d nodes (local window)
  int* jbase;                // [n_views][6] first node of the window
};

__host__ __device__ inline int serve_job_of(const long long* off, int n_jobs, long long i) {
  int lo = 0, hi = n_jobs - 1;  // last job with off[j] <= i
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= i) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Per-view set-up and tangents; per-pair set-up.
cudaError_t launch_serve_setup(const ServeJob* jobs, const long long* voff, const long long* poff, int n_jobs,
                               long long n_views, long long n_pairs, cudaStream_t stream);
// Pair kernel over all jobs' pair blocks: a persistent grid that takes blocks from a
// counter (reset here), then each job's fixed-order total.
cudaError_t launch_serve_pairs(const ServeJob* jobs, const long long* boff, int n_jobs,
                               unsigned long long* counter, int grid, cudaStream_t stream);
int serve_pairs_blocks_per_sm();
// Motion of the round: theta = theta0 + spline(nodes) for spline jobs (and the
// window Jacobians); per-view jobs keep their theta.
cudaError_t launch_serve_motion(const ServeJob* jobs, const long long* voff, int n_jobs, long long n_views,
                                cudaStream_t stream);
// Pair gradients, per-view gradient sums and the gradient steps.
cudaError_t launch_serve_grad(const ServeJob* jobs, const long long* voff, const long long* poff, int n_jobs,
                              long long n_views, long long n_pairs, cudaStream_t stream);

}  // namespace ecc
