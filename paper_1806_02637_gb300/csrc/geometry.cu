// Per-view and per-pair set-up of the ECC path (no matrix inverse anywhere): FP64 per
// view, double-float (about 48 bits, on the FP32 pipes) per pair.
//
//  geometry_kernel    one thread per view: rigid motion P' = P T(theta), scaling,
//                     source as the meet of the rows of P (Eq. 4/5), cofactor
//                     matrix, intrinsics; in the same launch the views' tangents for
//                     the gradients, the alpha-row directions and the line table.
//  pair_setup_kernel  one thread per pair: pencil frame around the baseline, the
//                     3x2 maps kappa -> epipolar line (the inverse-free form of
//                     Eq. 13/14), valid arcs from the detector corners, the sampled
//                     arc, the integer ranges of valid samples and the direction of
//                     each 32-sample tile centre.
#include "df.cuh"
#include "dual.cuh"
#include "motion.cuh"
#include "ecc_internal.cuh"
#include "kernels.cuh"

namespace ecc {

namespace {

__host__ __device__ inline void sc_pair(double x, double* s, double* c) { sincos(x, s, c); }
template <int N>
__device__ inline void sc_pair(const Dual<N>& x, Dual<N>* s, Dual<N>* c) { sincos(x, s, c); }

// a b + c, one rounding on doubles: written out, so that the records do not depend on what the
// compiler contracts.
__host__ __device__ inline double mad(double a, double b, double c) { return fma(a, b, c); }
template <int N>
__host__ __device__ inline Dual<N> mad(const Dual<N>& a, const Dual<N>& b, const Dual<N>& c) {
  return a * b + c;
}
template <int N>
__host__ __device__ inline Dual<N> mad(double a, const Dual<N>& b, const Dual<N>& c) {
  return a * b + c;
}

// a b - c d with one rounding less (fused), or all three.
__host__ __device__ inline double cross2(double a, double b, double c, double d, bool fused) {
#ifdef __CUDA_ARCH__
  return fused ? fma(a, b, -__dmul_rn(c, d)) : __dsub_rn(__dmul_rn(a, b), __dmul_rn(c, d));
#else
  return fused ? fma(a, b, -(c * d)) : a * b - c * d;
#endif
}
template <int N>
__host__ __device__ inline Dual<N> cross2(const Dual<N>& a, const Dual<N>& b, const Dual<N>& c, const Dual<N>& d,
                                          bool) {
  return a * b - c * d;
}

// A view's geometry while its lanes work on it.
template <class T>
struct ViewWork {
  T sc[6];   // sin, cos of the motion's angles
  T R[9];
  T Pm[12];  // P T(theta)
  T V[30];   // scaled P; 15 minors of its rows; (W - 1) / 2, (H - 1) / 2, 1
  T S[11];   // X0 .. X3, u0, v0, m1.m1, |m3 x m1|^2, centred third cofactor row
  T q[15];   // C, up, cofc
  T D;
  __host__ __device__ const T& u0() const { return S[4]; }
  __host__ __device__ const T& v0() const { return S[5]; }
};

// Minor k of the rows of P, x[i] y[j] - x[j] y[i]: p, q, r, s, -t, u of rows 1 and 2 (Eq. 5's
// Pluecker coordinates), then the cofactor rows m2 x m3, m3 x m1, m1 x m2.
__host__ __device__ inline int minor_code(int k) {  // x, y, i, j in two bits each
#define ECC_M(x, y, i, j) ((unsigned long long)((x) | (y) << 2 | (i) << 4 | (j) << 6))
  constexpr unsigned long long lo = ECC_M(0, 1, 2, 3) | ECC_M(0, 1, 1, 3) << 8 | ECC_M(0, 1, 1, 2) << 16 |
                                    ECC_M(0, 1, 0, 3) << 24 | ECC_M(0, 1, 2, 0) << 32 | ECC_M(0, 1, 0, 1) << 40 |
                                    ECC_M(1, 2, 1, 2) << 48 | ECC_M(1, 2, 2, 0) << 56;
  constexpr unsigned long long hi = ECC_M(1, 2, 0, 1) | ECC_M(2, 0, 1, 2) << 8 | ECC_M(2, 0, 2, 0) << 16 |
                                    ECC_M(2, 0, 0, 1) << 24 | ECC_M(0, 1, 1, 2) << 32 | ECC_M(0, 1, 2, 0) << 40 |
                                    ECC_M(0, 1, 0, 1) << 48;
#undef ECC_M
  return (int)((k < 8 ? lo >> (8 * k) : hi >> (8 * (k - 8))) & 255);
}

// Sum k of three products of V: the source's homogeneous coordinates, the dot products, the
// centred third cofactor row.  One product: sign, two places in V.
__host__ __device__ inline unsigned long long sum_code(int k) {
#define ECC_P(neg, i, j) ((unsigned long long)((neg) << 10 | (i) << 5 | (j)))
#define ECC_S(p0, p1, p2) ((p0) | (p1) << 11 | (p2) << 22)
  switch (k) {
    case 0: return ECC_S(ECC_P(1, 13, 10), ECC_P(0, 12, 9), ECC_P(0, 14, 11));
    case 1: return ECC_S(ECC_P(1, 12, 8), ECC_P(0, 15, 10), ECC_P(0, 16, 11));
    case 2: return ECC_S(ECC_P(1, 15, 9), ECC_P(0, 13, 8), ECC_P(0, 17, 11));
    case 3: return ECC_S(ECC_P(1, 14, 8), ECC_P(1, 16, 9), ECC_P(1, 17, 10));
    case 4: return ECC_S(ECC_P(0, 1, 9), ECC_P(0, 0, 8), ECC_P(0, 2, 10));
    case 5: return ECC_S(ECC_P(0, 5, 9), ECC_P(0, 4, 8), ECC_P(0, 6, 10));
    case 6: return ECC_S(ECC_P(0, 1, 1), ECC_P(0, 0, 0), ECC_P(0, 2, 2));
    case 7: return ECC_S(ECC_P(0, 22, 22), ECC_P(0, 21, 21), ECC_P(0, 23, 23));
    default: {
      const int c = k - 8;
      return ECC_S(ECC_P(0, 28, 21 + c), ECC_P(0, 27, 18 + c), ECC_P(0, 29, 24 + c));
    }
  }
#undef ECC_S
#undef ECC_P
}

// Per-view geometry, by L lanes: the moved matrix P T(theta), T = [R t; 0 1],
// R = Rz(rz) Ry(ry) Rx(rx); scaled P (third row of M unit, det M > 0), source as the meet of
// the rows (Eq. 4, then Eq. 5 with p entering with the opposite sign), up axis m3 x m1,
// cofactor rows (m2 x m3, m3 x m1, m1 x m2; l = cof(M) n) with the third row for centred
// detector coordinates, principal point and source-detector distance.  Returns false (in
// every lane) for a degenerate P.
//
// P(k) and th(k) give the matrix and the motion; sync() makes the lanes' stores to w visible
// to each other.  T is double, or Dual for tangents.  One lane alone (L = 1, the host)
// computes the same.  By lanes because an FP64 instruction holds its pipe 16 cycles and a
// dependent one waits far longer: one thread's 1570 instructions per view took 10 us however
// few the views (two views: launch of 15.3 us by threads, 11.6 us by lanes; 248 views and
// their motion tangents: 20.7 + 22.5 us in two launches, 18.0 us in this one).
template <int L, class T, class FP, class FT, class Sync>
__host__ __device__ bool view_geometry(FP P, FT th, bool moved, int W, int H, int lane, ViewWork<T>& w, Sync sync) {
  if (moved) {
    for (int k = lane; k < 3; k += L) sc_pair(th(k), &w.sc[2 * k], &w.sc[2 * k + 1]);
    sync();
    for (int k = lane; k < 9; k += L) {
      const int r = k / 3, c = k % 3;
      const T sx = w.sc[0], cx = w.sc[1], sy = w.sc[2], cy = w.sc[3], sz = w.sc[4], cz = w.sc[5];
      const T x = r == 0 ? cz : sz;
      const T a = r == 2 ? cy : x * sy;  // column 1: a sx + e cx, column 2: a cx + e sx
      const T e = r == 2 ? T(0.0) : (r == 0 ? (c == 1 ? -sz : sz) : (c == 1 ? cz : -cz));
      const T f = c == 1 ? sx : cx, g = c == 1 ? cx : sx;
      w.R[k] = c == 0 ? (r == 2 ? -sy : x * cy) : (k == 2 ? mad(e, g, a * f) : mad(a, f, e * g));
    }
    sync();
  }
  for (int k = lane; k < 12; k += L) {
    if (moved) {
      const int i = k & ~3, j = k & 3;
      const T x = j < 3 ? w.R[j] : th(3), y = j < 3 ? w.R[3 + j] : th(4), z = j < 3 ? w.R[6 + j] : th(5);
      const T s = mad(P(i + 2), z, mad(P(i), x, P(i + 1) * y));
      w.Pm[k] = j < 3 ? s : s + T(P(k));
    } else {
      w.Pm[k] = T(P(k));
    }
  }
  if (lane == 0) {
    w.V[27] = T(0.5 * (W - 1));
    w.V[28] = T(0.5 * (H - 1));
    w.V[29] = T(1.0);
  }
  sync();
  const T* m1 = w.Pm;
  const T* m2 = w.Pm + 4;
  const T* m3 = w.Pm + 8;
  const T det = m1[0] * (m2[1] * m3[2] - m2[2] * m3[1]) + m1[1] * (m2[2] * m3[0] - m2[0] * m3[2]) +
                m1[2] * (m2[0] * m3[1] - m2[1] * m3[0]);
  const T n3 = sqrt(mad(m3[2], m3[2], mad(m3[0], m3[0], m3[1] * m3[1])));
  bool ok = isfinite(value(det)) && isfinite(value(n3)) && value(det) != 0.0 && value(n3) > 0.0;
  for (int k = 0; k < 12; ++k) ok = ok && isfinite(value(w.Pm[k]));  // NaN / Inf anywhere, the motion's included
  const T sc = ok ? T(copysign(1.0, value(det))) / n3 : T(0.0);
  for (int k = lane; k < 12; k += L) w.V[k] = w.Pm[k] * sc;
  sync();
  for (int k = lane; k < 15; k += L) {
    const int m = minor_code(k);
    const T* x = w.V + 4 * (m & 3);
    const T* y = w.V + 4 * (m >> 2 & 3);
    const int i = m >> 4 & 3, j = m >> 6;
    // t and its copy in m1 x m2 with three roundings, as one shared difference of products
    w.V[12 + k] = cross2(x[i], y[j], x[j], y[i], k != 4 && k != 13);
  }
  sync();
  for (int k = lane; k < 11; k += L) {
    const unsigned long long m = sum_code(k);
    T x[3];
    for (int i = 0; i < 3; ++i) {
      x[i] = w.V[m >> (11 * i + 5) & 31];
      if (m >> (11 * i + 10) & 1) x[i] = -x[i];
    }
    w.S[k] = mad(x[2], w.V[m >> 22 & 31], mad(x[1], w.V[m >> 11 & 31], x[0] * w.V[m & 31]));
  }
  sync();
  ok = ok && value(w.S[3]) != 0.0;
  const T iw = ok ? T(1.0) / w.S[3] : T(0.0);
  const T nu = sqrt(w.S[7]);
  ok = ok && value(nu) > 0.0;
  for (int k = lane; k < 15; k += L)
    w.q[k] = k < 3 ? w.S[k] * iw : (k < 6 ? (ok ? w.V[18 + k] / nu : T(0.0)) : (k < 12 ? w.V[12 + k] : w.S[k - 4]));
  const T dd = mad(-w.S[4], w.S[4], w.S[6]);
  ok = ok && value(dd) > 0.0;
  const T D = ok ? sqrt(dd) : T(0.0);
  if (lane == 0) w.D = D;
  sync();
  for (int k = 0; k < 3; ++k) ok = ok && isfinite(value(w.q[k]));
  return ok;
}

// The view's record from its finished geometry, written by its lanes.
template <int L>
__host__ __device__ void write_view(const ViewWork<double>& w, bool ok, int lane, ViewRec* out) {
  for (int k = lane; k < 15; k += L) {
    if (k < 12) out->P[k] = w.V[k];
    (k < 3 ? out->C[k] : (k < 6 ? out->up[k - 3] : out->cofc[k - 6])) = w.q[k];
    const df q = df_from_double(w.q[k]);
    out->qdf[2 * k] = q.hi;
    out->qdf[2 * k + 1] = q.lo;
  }
  if (lane == 0) {
    out->u0 = w.u0();
    out->v0 = w.v0();
    out->D = w.D;
    out->status = ok ? 0 : 1;
    out->pad = 0;
  }
}

// Lanes per view, and per tangent direction: the FP64 pipe's time per direction falls with
// fewer lanes, the chain of dependent instructions grows.
constexpr int kViewLanes = 16, kTanLanes = 8;

union GeometryShared {
  ViewWork<double> view[32 / kViewLanes];
  ViewWork<Dual<1>> tan[32 / kTanLanes];
  __device__ GeometryShared() {}
};

// View i (of n) by its kViewLanes of the warp; lanes past the end work on the last view and
// write nothing.  P and motion (or NULL) are the view's own.
__device__ const ViewWork<double>& device_view(const double* __restrict__ P, const double* __restrict__ motion, int W,
                                               int H, GeometryShared& sh, bool write, ViewRec* out, int* status) {
  const int lane = threadIdx.x % kViewLanes;
  ViewWork<double>& w = sh.view[threadIdx.x / kViewLanes];
  const bool ok = view_geometry<kViewLanes, double>([=](int k) { return P[k]; }, [=](int k) { return motion[k]; },
                                                    motion != nullptr, W, H, lane, w, [] { __syncwarp(); });
  if (write) {
    write_view<kViewLanes>(w, ok, lane, out);
    if (!ok && lane == 0) atomicOr(status, kStatusDegenerateView);
  }
  return w;
}

// Tangents of the per-view geometry q = (C, up, cofc), forward mode in FP64, one direction
// per kTanLanes of the warp: with respect to motion parameter j (out[15][6], ViewTan) or,
// WRT_P, to entry j of the unmoved P (out[15][12], ViewTanP; the view uses P T(theta)).  A
// degenerate view's pairs carry no gradient; zero tangents keep its row at 0 (its NaN / Inf
// geometry would otherwise turn 0 x tangent into NaN).
template <bool WRT_P>
__device__ void device_tangent(const double* __restrict__ P, const double* __restrict__ motion, int j, int W, int H,
                               GeometryShared& sh, bool write, double* __restrict__ out) {
  using D1 = Dual<1>;
  const int lane = threadIdx.x % kTanLanes;
  ViewWork<D1>& w = sh.tan[threadIdx.x / kTanLanes];
  auto seeded = [](double x, bool one) {
    D1 d(x);
    d.d[0] = one ? 1.0 : 0.0;
    return d;
  };
  auto th = [=](int k) { return seeded(motion ? motion[k] : 0.0, !WRT_P && k == j); };
  bool ok;
  if (WRT_P)
    ok = view_geometry<kTanLanes, D1>([=](int k) { return seeded(P[k], k == j); }, th, motion != nullptr, W, H, lane, w,
                                      [] { __syncwarp(); });
  else
    ok = view_geometry<kTanLanes, D1>([=](int k) { return P[k]; }, th, true, W, H, lane, w, [] { __syncwarp(); });
  if (write)
    for (int k = lane; k < 15; k += kTanLanes) out[(WRT_P ? 12 : 6) * k + j] = ok ? w.q[k].d[0] : 0.0;
}

// Line parameters of alpha row m of the Joseph line sums, as 32.32 fixed-point coordinates
// along the interpolation axis (the x axis for rows, the y axis for columns).
__device__ RadonRow radon_row(int m, int W, int H, int n_alpha, int n_s) {
  constexpr double kTwo32 = 4294967296.0;
  double sa, ca;
  sincospi((double)m / (double)n_alpha, &sa, &ca);
  const bool rows = (4 * m <= n_alpha) || (4 * m >= 3 * n_alpha);
  const double ds = sqrt((double)W * W + (double)H * H) / (n_s - 1);
  const double cx = 0.5 * (W - 1), cy = 0.5 * (H - 1);
  const double p = rows ? ca : sa, q = rows ? sa : ca, cp = rows ? cx : cy, cq = rows ? cy : cx;
  RadonRow r;
  r.B0 = llrint((cp + (cq * q - 0.5 * n_s * ds) / p) * kTwo32);
  r.STEP = llrint(ds / p * kTwo32);
  r.DY = llrint(-q / p * kTwo32);
  r.inv_len = (float)(1.0 / fabs(p));
  r.ca = (float)ca;
  r.sa = (float)sa;
  r.rows_mode = rows ? 1 : 0;
  return r;
}

}  // namespace

// All FP64 work of a call that depends on its geometry alone, in one launch: blocks of one
// warp take views, tangent directions, alpha rows or table rows, by ranges of the block
// index.  One warp per block because the FP64 pipe of an SM is what they would share.  (Set-up
// and line table of two views: 14.4 + 13.9 us in two launches, 10.4 us in this one.)
struct GeometryRanges {
  int views, tan, tanP, alpha, table;  // blocks of each kind
};

__global__ void __launch_bounds__(32) geometry_kernel(Geometry g, GeometryRanges n) {
  let_next_start();
  __shared__ GeometryShared sh;
  int b = (int)blockIdx.x;
  if (b < n.views) {
    const int i = b * (32 / kViewLanes) + threadIdx.x / kViewLanes;
    const int v = min(i, g.n_views - 1);
    const bool write = i < g.n_views;
    const ViewWork<double>& w = device_view(g.P + 12 * v, g.motion ? g.motion + 6 * v : nullptr, g.W, g.H, sh, write,
                                            g.views + v, g.status);
    if (g.weights && write && threadIdx.x % kViewLanes == 0) {
      RadonView o;
      o.u0 = (float)w.u0();
      o.v0 = (float)w.v0();
      o.D = (float)w.D;
      o.max_bits = 0;
      g.weights[v] = o;
    }
    return;
  }
  b -= n.views;
  if (b < n.tan) {
    const long long i = (long long)b * (32 / kTanLanes) + threadIdx.x / kTanLanes, last = 6ll * g.n_views - 1;
    const int v = (int)(min(i, last) / 6), j = (int)(min(i, last) % 6);
    device_tangent<false>(g.P + 12 * v, g.motion ? g.motion + 6 * v : nullptr, j, g.W, g.H, sh, i <= last,
                          &g.tan[v].dC[0][0]);
    return;
  }
  b -= n.tan;
  if (b < n.tanP) {
    const long long i = (long long)b * (32 / kTanLanes) + threadIdx.x / kTanLanes, last = 12ll * g.n_views - 1;
    const int v = (int)(min(i, last) / 12), j = (int)(min(i, last) % 12);
    device_tangent<true>(g.P + 12 * v, g.motion ? g.motion + 6 * v : nullptr, j, g.W, g.H, sh, i <= last,
                         &g.tanP[v].d[0][0]);
    return;
  }
  b -= n.tanP;
  if (b < n.alpha) {
    const int m = 32 * b + threadIdx.x;
    if (m >= g.n_alpha) return;
    double s, c;
    sincospi((double)m / (double)g.n_alpha, &s, &c);
    g.alpha_dir[m] = split_dir(c, s);
    return;
  }
  b -= n.alpha;
  const long long i = 32ll * b + threadIdx.x;
  if (i < (long long)g.copies * g.n_alpha) g.table[i] = radon_row((int)(i % g.n_alpha), g.W, g.H, g.n_alpha, g.n_s);
}

cudaError_t launch_geometry(const Geometry& g, const LaunchHooks& hooks, cudaStream_t stream) {
  auto blocks = [](bool on, long long n, int per) { return on ? (int)((n + per - 1) / per) : 0; };
  GeometryRanges n;
  n.views = blocks(g.views != nullptr, g.n_views, 32 / kViewLanes);
  n.tan = blocks(g.tan != nullptr, 6ll * g.n_views, 32 / kTanLanes);
  n.tanP = blocks(g.tanP != nullptr, 12ll * g.n_views, 32 / kTanLanes);
  n.alpha = blocks(g.alpha_dir != nullptr, g.n_alpha, 32);
  n.table = blocks(g.table != nullptr, (long long)g.copies * g.n_alpha, 32);
  hooks.on_begin("geometry_kernel", stream);
  geometry_kernel<<<n.views + n.tan + n.tanP + n.alpha + n.table, 32, 0, stream>>>(g, n);
  hooks.on_end("geometry_kernel", stream);
  return cudaGetLastError();
}

namespace {

// Double-float vector helpers of the per-pair set-up.
__host__ __device__ inline df qget(const ViewRec& v, int k) { return df{v.qdf[2 * k], v.qdf[2 * k + 1]}; }
__host__ __device__ inline df df_dot3(const df* a, const df* b) {
  return df_add(df_add(df_mul(a[0], b[0]), df_mul(a[1], b[1])), df_mul(a[2], b[2]));
}
__host__ __device__ inline df df_cross2(df ax, df ay, df bx, df by) { return df_sub(df_mul(ax, by), df_mul(ay, bx)); }
__host__ __device__ inline df df_sel(bool c, df a, df b) { return c ? a : b; }

// Frame of the pencil of epipolar planes around the baseline C_a -> C_b, in
// double-float: u = baseline direction, w = (up_a + up_b) made orthogonal to u (below
// |w| = 1e-6 the world axis least aligned with u, the first within 1e-9 of the
// smallest |u_k| so that ties are not left to rounding), v = w x u; the plane at kappa
// has normal cos(kappa) w + sin(kappa) v.  Normalisations are products by reciprocal
// square roots.  Returns false for coincident sources.
__host__ __device__ bool pencil_frame_df(const ViewRec& va, const ViewRec& vb, df* w, df* v) {
  df d[3], rr[3], u[3];
  for (int k = 0; k < 3; ++k) {
    d[k] = df_sub(qget(vb, k), qget(va, k));
    rr[k] = df_add(qget(va, 3 + k), qget(vb, 3 + k));
  }
  const df nd2 = df_dot3(d, d);
  if (!(nd2.hi > 0.0f)) return false;
  const df ind = df_rsqrt(nd2);
  for (int k = 0; k < 3; ++k) u[k] = df_mul(d[k], ind);
  const df ru = df_dot3(rr, u);
  for (int k = 0; k < 3; ++k) w[k] = df_sub(rr[k], df_mul(ru, u[k]));
  df nw2 = df_dot3(w, w);
  if (nw2.hi < 1e-12f) {
    // the first axis within 1e-9 of the smallest |u_k|: ties are not left to rounding
    const double ua[3] = {fabs(df_to_double(u[0])), fabs(df_to_double(u[1])), fabs(df_to_double(u[2]))};
    const double best = fmin(ua[0], fmin(ua[1], ua[2]));
    const int ax = ua[0] <= best + 1e-9 ? 0 : (ua[1] <= best + 1e-9 ? 1 : 2);
    const df ui = ax == 0 ? u[0] : (ax == 1 ? u[1] : u[2]);
    for (int k = 0; k < 3; ++k) w[k] = df_sub(df{k == ax ? 1.0f : 0.0f, 0.0f}, df_mul(ui, u[k]));
    nw2 = df_dot3(w, w);
  }
  const df inw = df_rsqrt(nw2);
  for (int k = 0; k < 3; ++k) w[k] = df_mul(w[k], inw);
  v[0] = df_cross2(w[1], w[2], u[1], u[2]);
  v[1] = df_cross2(w[2], w[0], u[2], u[0]);
  v[2] = df_cross2(w[0], w[1], u[0], u[1]);
  return true;
}

// Reverse mode of pencil_frame_df (the same steps in double-float): given gw = d e / d w
// and gv = d e / d v, returns d e / d (Ca, Cb, up) in gCa, gCb and gup (the same for both
// up axes, which enter as their sum).  Each step's adjoint follows from its forward
// rule: v = w x u gives w' += u x v', u' += v' x w; y = x / |x| gives
// x' = (y' - (y'.y) y) / |x|; w_t = r - (r.u) u gives r' = w_t' - (w_t'.u) u and
// u' -= (w_t'.u) r + (r.u) w_t' (for the fallback axis e: u' -= (w_t'.u) e_ax + u_ax w_t').
__host__ __device__ bool pencil_frame_adjoint_df(const ViewRec& va, const ViewRec& vb, const df* gw, const df* gv,
                                                 df* w, df* v, df* gCa, df* gCb, df* gup) {
  df d[3], rr[3], u[3], wt[3];
  for (int k = 0; k < 3; ++k) {
    d[k] = df_sub(qget(vb, k), qget(va, k));
    rr[k] = df_add(qget(va, 3 + k), qget(vb, 3 + k));
  }
  const df nd2 = df_dot3(d, d);
  if (!(nd2.hi > 0.0f)) return false;
  const df ind = df_rsqrt(nd2);
  for (int k = 0; k < 3; ++k) u[k] = df_mul(d[k], ind);
  const df ru = df_dot3(rr, u);
  for (int k = 0; k < 3; ++k) wt[k] = df_sub(rr[k], df_mul(ru, u[k]));
  df nw2 = df_dot3(wt, wt);
  int ax = -1;
  if (nw2.hi < 1e-12f) {
    const double ua[3] = {fabs(df_to_double(u[0])), fabs(df_to_double(u[1])), fabs(df_to_double(u[2]))};
    const double best = fmin(ua[0], fmin(ua[1], ua[2]));
    ax = ua[0] <= best + 1e-9 ? 0 : (ua[1] <= best + 1e-9 ? 1 : 2);
    const df ui = ax == 0 ? u[0] : (ax == 1 ? u[1] : u[2]);
    for (int k = 0; k < 3; ++k) wt[k] = df_sub(df{k == ax ? 1.0f : 0.0f, 0.0f}, df_mul(ui, u[k]));
    nw2 = df_dot3(wt, wt);
  }
  const df inw = df_rsqrt(nw2);
  for (int k = 0; k < 3; ++k) w[k] = df_mul(wt[k], inw);
  v[0] = df_cross2(w[1], w[2], u[1], u[2]);
  v[1] = df_cross2(w[2], w[0], u[2], u[0]);
  v[2] = df_cross2(w[0], w[1], u[0], u[1]);
  // reverse
  df gwt_in[3], gu[3], gwt[3];
  gwt_in[0] = df_add(gw[0], df_cross2(u[1], u[2], gv[1], gv[2]));  // d e / d w from v = w x u
  gwt_in[1] = df_add(gw[1], df_cross2(u[2], u[0], gv[2], gv[0]));
  gwt_in[2] = df_add(gw[2], df_cross2(u[0], u[1], gv[0], gv[1]));
  gu[0] = df_cross2(gv[1], gv[2], w[1], w[2]);  // d e / d u from v = w x u
  gu[1] = df_cross2(gv[2], gv[0], w[2], w[0]);
  gu[2] = df_cross2(gv[0], gv[1], w[0], w[1]);
  const df gww = df_dot3(gwt_in, w);
  for (int k = 0; k < 3; ++k) gwt[k] = df_mul(df_sub(gwt_in[k], df_mul(gww, w[k])), inw);
  const df gwu = df_dot3(gwt, u);
  if (ax < 0) {
    for (int k = 0; k < 3; ++k) {
      gup[k] = df_sub(gwt[k], df_mul(gwu, u[k]));
      gu[k] = df_sub(gu[k], df_add(df_mul(gwu, rr[k]), df_mul(ru, gwt[k])));
    }
  } else {
    const df ui = ax == 0 ? u[0] : (ax == 1 ? u[1] : u[2]);
    for (int k = 0; k < 3; ++k) {
      gup[k] = df{0.0f, 0.0f};
      gu[k] = df_sub(gu[k], df_mul(ui, gwt[k]));
    }
    gu[ax] = df_sub(gu[ax], gwu);
  }
  const df guu = df_dot3(gu, u);
  for (int k = 0; k < 3; ++k) {
    const df gd = df_mul(df_sub(gu[k], df_mul(guu, u[k])), ind);
    gCb[k] = gd;
    gCa[k] = df_neg(gd);
  }
  return true;
}

// Valid arc of the pencil for one view: the plane at kappa (c = (cos, sin)) meets
// the detector rectangle iff the values g_c . c at the four corners do not all have
// the same strict sign, g_c = A^T x_c.  If the g_c lie in a half plane (epipole
// outside), the valid directions (mod pi) run counter-clockwise from rot90(g_min)
// over the angle between the extreme g's; otherwise every plane is valid.  The
// corner values, the sign tests (each cross product once, with its antisymmetry for
// the reversed order) and the angle run in double-float.
__host__ __device__ __noinline__ df view_arc(const df* A, int W, int H, df* clo) {
  const float hw = 0.5f * (float)W, hh = 0.5f * (float)H;  // exact
  const float xs[4] = {-hw, hw, hw, -hw};
  const float ys[4] = {-hh, -hh, hh, hh};
  df sc = df_mul(A[0], A[0]);
  for (int k = 1; k < 6; ++k) sc = df_add(sc, df_mul(A[k], A[k]));
  df gx[4], gy[4], n2[4];
  bool degenerate = false;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    gx[c] = df_add(df_add(df_mul_f(A[0], xs[c]), df_mul_f(A[2], ys[c])), A[4]);
    gy[c] = df_add(df_add(df_mul_f(A[1], xs[c]), df_mul_f(A[3], ys[c])), A[5]);
    n2[c] = df_add(df_mul(gx[c], gx[c]), df_mul(gy[c], gy[c]));
    if (!(n2[c].hi > 1e-28f * sc.hi)) degenerate = true;
  }
  // cross products g_i x g_j (i < j); g_j x g_i = -(g_i x g_j)
  const float c01 = df_cross2(gx[0], gy[0], gx[1], gy[1]).hi, c02 = df_cross2(gx[0], gy[0], gx[2], gy[2]).hi;
  const float c03 = df_cross2(gx[0], gy[0], gx[3], gy[3]).hi, c12 = df_cross2(gx[1], gy[1], gx[2], gy[2]).hi;
  const float c13 = df_cross2(gx[1], gy[1], gx[3], gy[3]).hi, c23 = df_cross2(gx[2], gy[2], gx[3], gy[3]).hi;
  // corner i is the minimum if g_i x g_j >= 0 for every j, the maximum if <= 0
  const bool mn0 = c01 >= 0.0f && c02 >= 0.0f && c03 >= 0.0f, mx0 = c01 <= 0.0f && c02 <= 0.0f && c03 <= 0.0f;
  const bool mn1 = -c01 >= 0.0f && c12 >= 0.0f && c13 >= 0.0f, mx1 = -c01 <= 0.0f && c12 <= 0.0f && c13 <= 0.0f;
  const bool mn2 = -c02 >= 0.0f && -c12 >= 0.0f && c23 >= 0.0f, mx2 = -c02 <= 0.0f && -c12 <= 0.0f && c23 <= 0.0f;
  const bool mn3 = -c03 >= 0.0f && -c13 >= 0.0f && -c23 >= 0.0f, mx3 = -c03 <= 0.0f && -c13 <= 0.0f && -c23 <= 0.0f;
  const int imin = mn0 ? 0 : (mn1 ? 1 : (mn2 ? 2 : (mn3 ? 3 : -1)));
  const int imax = mx0 ? 0 : (mx1 ? 1 : (mx2 ? 2 : (mx3 ? 3 : -1)));
  if (degenerate || imin < 0 || imax < 0) {
    clo[0] = df{0.0f, 0.0f};
    clo[1] = df{-1.0f, 0.0f};
    return df_pi();
  }
  // (scalars and selects only: no dynamically indexed local arrays)
  const df ax_ = df_sel(imin == 0, gx[0], df_sel(imin == 1, gx[1], df_sel(imin == 2, gx[2], gx[3])));
  const df ay_ = df_sel(imin == 0, gy[0], df_sel(imin == 1, gy[1], df_sel(imin == 2, gy[2], gy[3])));
  const df an2 = df_sel(imin == 0, n2[0], df_sel(imin == 1, n2[1], df_sel(imin == 2, n2[2], n2[3])));
  const df bx_ = df_sel(imax == 0, gx[0], df_sel(imax == 1, gx[1], df_sel(imax == 2, gx[2], gx[3])));
  const df by_ = df_sel(imax == 0, gy[0], df_sel(imax == 1, gy[1], df_sel(imax == 2, gy[2], gy[3])));
  const df cr = df_cross2(ax_, ay_, bx_, by_);
  const df dt = df_add(df_mul(ax_, bx_), df_mul(ay_, by_));
  df phi = df_atan2(cr, dt);
  if (df_lt0(phi)) phi = df{0.0f, 0.0f};
  const df ing = df_rsqrt(an2);
  clo[0] = df_neg(df_mul(ay_, ing));
  clo[1] = df_mul(ax_, ing);
  return phi;
}

}  // namespace

// Per-pair set-up: frame, kappa -> line maps, valid arcs, the sampled arc, the
// integer ranges of valid samples and the tile-centre directions (ctile, n_tiles
// entries).  With previous != NULL the sampling of *previous is kept and only the maps
// follow the geometry.  GB300 issues FP64 at 1/64 of the FP32 rate, so everything
// here runs in double-float (about 48 bits) on the FP32 pipes from the views'
// double-float copies: the frame, the maps, the corner values and signs, the angles
// (df_atan2, df_sincos), the step and the positions whose floors give the integer
// ranges.
//
// LANES = 2: lanes 2 i and 2 i + 1 of a warp (side 0, 1; the whole warp calls) take one
// view's map and arc each, which go to r.Af[0], and the same steps otherwise; each writes
// every other tile direction.  The values are the same.
template <int LANES>
__host__ __device__ PairRec setup_pair(int a, int b, int n_views, const ViewRec* views, int W, int H, int K,
                                       float4* ctile, int n_tiles, const PairRec* previous, int side = 0) {
  const bool reuse_sampling = previous != nullptr;
  PairRec r;
  const bool in_range = a >= 0 && b >= 0 && a < n_views && b < n_views;
  if (!in_range) {  // caller's pair list names a view that does not exist
    a = 0;
    b = 0;
  }
  r.a = a;
  r.b = b;
  r.status = 0;
  r.r0lo = r.r0hi = r.r1lo = r.r1hi = 0;
  r.nk = 0;
  r.dk = 0.0;
  r.dk_hi = r.dk_lo = 0.0f;
  for (int i = 0; i < 24; ++i) (&r.Af[0][0])[i] = 0.0f;
  r.c0[0] = 1.0;
  r.c0[1] = 0.0;
  const ViewRec& va = views[a];
  const ViewRec& vb = views[b];
  constexpr int kSides = LANES == 1 ? 2 : 1;  // of this lane
  df w[3], v[3];
  df Ad[kSides][6];
  df len[2] = {}, cl[2][2] = {};
  bool ok = in_range && va.status == 0 && vb.status == 0 && a != b && pencil_frame_df(va, vb, w, v);
  if (ok) {
    const ViewRec* vv[2] = {LANES == 1 || side == 0 ? &va : &vb, &vb};
    for (int s = 0; s < kSides; ++s)
      for (int i = 0; i < 3; ++i) {
        const df row[3] = {qget(*vv[s], 6 + 3 * i), qget(*vv[s], 7 + 3 * i), qget(*vv[s], 8 + 3 * i)};
        Ad[s][2 * i + 0] = df_dot3(row, w);
        Ad[s][2 * i + 1] = df_dot3(row, v);
      }
    for (int s = 0; s < kSides; ++s)
      for (int i = 0; i < 6; ++i) {
        r.Af[s][2 * i] = Ad[s][i].hi;
        r.Af[s][2 * i + 1] = Ad[s][i].lo;
      }
    if (!reuse_sampling)
      for (int s = 0; s < kSides; ++s) len[s] = view_arc(Ad[s], W, H, cl[s]);
  }
#ifdef __CUDA_ARCH__
  if (LANES == 2) {
    auto other = [](df x) { return df{__shfl_xor_sync(0xffffffffu, x.hi, 1), __shfl_xor_sync(0xffffffffu, x.lo, 1)}; };
    const df lo = other(len[0]), xo = other(cl[0][0]), yo = other(cl[0][1]);
    len[1] = df_sel(side == 0, lo, len[0]);
    cl[1][0] = df_sel(side == 0, xo, cl[0][0]);
    cl[1][1] = df_sel(side == 0, yo, cl[0][1]);
    len[0] = df_sel(side == 0, len[0], lo);
    cl[0][0] = df_sel(side == 0, cl[0][0], xo);
    cl[0][1] = df_sel(side == 0, cl[0][1], yo);
  }
#endif
  if (ok && reuse_sampling) {
    // keep the planes sampled by the previous call (kappa arcs and validity
    // frozen); only the kappa -> line maps follow the new geometry
    const PairRec old = *previous;
    r.dk = old.dk;
    r.c0[0] = old.c0[0];
    r.c0[1] = old.c0[1];
    r.dk_hi = old.dk_hi;
    r.dk_lo = old.dk_lo;
    r.r0lo = old.r0lo;
    r.r0hi = old.r0hi;
    r.r1lo = old.r1lo;
    r.r1hi = old.r1hi;
    r.nk = old.nk;
    ok = old.status == 0;
  } else if (ok) {
    const df lena = len[0], lenb = len[1];
    // sample the shorter arc; ties (equal in exact arithmetic for mirror-symmetric
    // pairs) go to view a within a relative tolerance, not by rounding
    const bool samp_a = df_sub(lena, lenb).hi <= 1e-9f * fmaxf(lena.hi, lenb.hi);
    const df len_s = samp_a ? lena : lenb, len_o = samp_a ? lenb : lena;
    const df csx = samp_a ? cl[0][0] : cl[1][0], csy = samp_a ? cl[0][1] : cl[1][1];
    const df cox = samp_a ? cl[1][0] : cl[0][0], coy = samp_a ? cl[1][1] : cl[0][1];
    const df dk = df_div_f(len_s, (float)K);
    r.dk = df_to_double(dk);
    r.dk_hi = dk.hi;
    r.dk_lo = dk.lo;
    // one sincos: the rotations by dk, 16 dk and 32 dk follow by angle doubling (the
    // angle error doubles with each step: about 1e-13 rad after six)
    df sh, ch;
    df_sincos(df_mul_f(dk, 0.5f), &sh, &ch);
    auto twice = [](df& s_, df& c_) {
      const df s2 = df_mul_f(df_mul(s_, c_), 2.0f);
      c_ = df_sub(df_mul(c_, c_), df_mul(s_, s_));
      s_ = s2;
    };
    auto rotate = [](df c, df s, df x, df y, df* ox, df* oy) {
      *ox = df_sub(df_mul(c, x), df_mul(s, y));
      *oy = df_add(df_mul(s, x), df_mul(c, y));
    };
    {
      df c0x, c0y;
      rotate(ch, sh, csx, csy, &c0x, &c0y);
      r.c0[0] = df_to_double(c0x);
      r.c0[1] = df_to_double(c0y);
    }
    // valid samples of the other view: y_k = delta0 + (k + 1/2) dk, valid iff
    // y_k <= len_o or pi <= y_k <= pi + len_o (angles mod pi from its arc start)
    const df pi = df_pi();
    if (!df_lt0(df_sub(len_o, pi))) {
      r.r0lo = 0;
      r.r0hi = K;
      r.r1lo = r.r1hi = K;
    } else if (dk.hi > 0.0f) {
      df d0 = df_atan2(df_cross2(cox, coy, csx, csy), df_add(df_mul(cox, csx), df_mul(coy, csy)));
      if (df_lt0(d0)) d0 = df_add(d0, pi);
      if (!df_lt0(df_sub(d0, pi))) d0 = df_sub(d0, pi);
      const df idk = df_recip(dk);
      const df half = {0.5f, 0.0f};
      // floor / ceil of the sample positions (integer-valued FP32; K is exact in FP32)
      float fr;
      const float e0 = df_floor_frac(df_sub(df_mul(df_sub(len_o, d0), idk), half), &fr);
      float s1 = df_floor_frac(df_sub(df_mul(df_sub(pi, d0), idk), half), &fr);
      if (fr > 0.0f) s1 += 1.0f;
      const float e1 = df_floor_frac(df_sub(df_mul(df_sub(df_add(pi, len_o), d0), idk), half), &fr);
      const float Kf = (float)K;
      const int hi0 = (int)fminf(fmaxf(e0 + 1.0f, 0.0f), Kf);
      const int lo1 = (int)fminf(fmaxf(s1, (float)hi0), Kf);
      const int hi1 = (int)fminf(fmaxf(e1 + 1.0f, (float)lo1), Kf);
      r.r0lo = 0;
      r.r0hi = hi0;
      r.r1lo = lo1;
      r.r1hi = hi1;
    }
    r.nk = (r.r0hi - r.r0lo) + (r.r1hi - r.r1lo);
    // directions of the tile centres: tile t holds samples [32t, min(32t + 32, K)),
    // centred at ((k_begin + k_end) / 2) dk from the arc start; full tiles step by 32 dk
    df s16 = sh, c16 = ch;
    for (int i = 0; i < 5; ++i) twice(s16, c16);  // 16 dk
    df s32 = s16, c32 = c16;
    twice(s32, c32);  // 32 dk
    df cx0, cy0;
    rotate(c16, s16, csx, csy, &cx0, &cy0);
    float4* ct = ctile;
    for (int t = 0; t < n_tiles; ++t) {
      if (LANES == 2 && (t & 1) != side) {
      } else if (32 * t + 32 <= K) {
        ct[t] = make_float4(cx0.hi, cy0.hi, cx0.lo, cy0.lo);
      } else {  // last, partial tile
        df sp, cp, px, py;
        df_sincos(df_mul_f(dk, 0.5f * (float)(32 * t + K)), &sp, &cp);
        rotate(cp, sp, csx, csy, &px, &py);
        ct[t] = make_float4(px.hi, py.hi, px.lo, py.lo);
      }
      df nx, ny;
      rotate(c32, s32, cx0, cy0, &nx, &ny);
      cx0 = nx;
      cy0 = ny;
    }
  }
  if (!ok) r.status = 1;
  return r;
}

// One thread per pair, or two.
template <int LANES>
__global__ void pair_setup_kernel(int n_views, long long n_pairs, const int32_t* __restrict__ pairs,
                                  const ViewRec* __restrict__ views, int W, int H, int K,
                                  PairRec* __restrict__ out, float4* __restrict__ ctile, int n_tiles,
                                  int reuse_sampling, int* __restrict__ status) {
  const long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / LANES;
  if (LANES == 1 && i >= n_pairs) return;
  const long long p = i < n_pairs ? i : n_pairs - 1;  // LANES = 2: the warp stays whole
  const int side = LANES == 1 ? 0 : threadIdx.x & 1;
  int a, b;
  if (pairs) {
    a = pairs[2 * p];
    b = pairs[2 * p + 1];
  } else {
    pair_from_index(p, n_views, &a, &b);
  }
  PairRec prev;
  if (reuse_sampling) prev = out[p];
  if (LANES == 2) __syncwarp();  // both have read it
  PairRec r = setup_pair<LANES>(a, b, n_views, views, W, H, K, ctile + p * n_tiles, n_tiles,
                                reuse_sampling ? &prev : nullptr, side);
  if (LANES == 1) {
    if (r.status) atomicOr(status, kStatusDegeneratePair);
    out[p] = r;
    return;
  }
  if (i >= n_pairs) return;
  PairRec& o = out[p];
  for (int k = 0; k < 12; ++k) o.Af[side][k] = r.Af[0][k];
  if (side == 0) {
    if (r.status) atomicOr(status, kStatusDegeneratePair);
    o.dk_hi = r.dk_hi;
    o.dk_lo = r.dk_lo;
    o.c0[0] = r.c0[0];
    o.c0[1] = r.c0[1];
    o.dk = r.dk;
    o.a = r.a;
    o.b = r.b;
    o.r0lo = r.r0lo;
    o.r0hi = r.r0hi;
    o.r1lo = r.r1lo;
    o.r1hi = r.r1hi;
    o.nk = r.nk;
    o.status = r.status;
  }
}

// Two threads per pair while that leaves a scheduler with one warp: a pair's steps wait on
// each other, and the second thread takes one view's map and arc off the first (evaluation of
// one pair 35.2 -> 33.8 us, of a list without allocation 55.7 -> 53.3 us, gradient of 7140
// pairs 107.0 -> 104.7 us).  With more pairs the instructions bound the kernel, and two
// threads execute more of them than one.
cudaError_t launch_pair_setup(int n_views, long long n_pairs, const int32_t* pairs, const ViewRec* views, int W, int H,
                              int K, PairRec* out, float4* ctile, int n_tiles, bool reuse_sampling, int* status,
                              const LaunchHooks& hooks, cudaStream_t stream) {
  int dev = 0, n_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  hooks.on_begin("pair_setup_kernel", stream);
  if (2 * n_pairs <= 4 * 32 * (long long)n_sm)
    pair_setup_kernel<2><<<(unsigned)((2 * n_pairs + 63) / 64), 64, 0, stream>>>(
        n_views, n_pairs, pairs, views, W, H, K, out, ctile, n_tiles, reuse_sampling, status);
  else
    pair_setup_kernel<1><<<(unsigned)((n_pairs + 127) / 128), 128, 0, stream>>>(
        n_views, n_pairs, pairs, views, W, H, K, out, ctile, n_tiles, reuse_sampling, status);
  hooks.on_end("pair_setup_kernel", stream);
  return cudaGetLastError();
}

// Gradient of one pair's e with respect to the per-view quantities the pair reads,
// q = (C[3], up[3], cofc[9]) of view a, then of view b (30 values), from
// G = d e / d A (the pair kernel's adjoint, FP32 values): A = cofc [w v] is linear in
// cofc, and the frame (w, v) is differentiated in reverse mode
// (pencil_frame_adjoint_df).  Double-float throughout; out holds (hi, lo) pairs.
__device__ void pair_grad_q(const PairRec& pr, const ViewRec* views, const double* G,
                            float2* __restrict__ out) {
  if (pr.status != 0 || pr.nk <= 0) {
    for (int j = 0; j < 30; ++j) out[j] = make_float2(0.0f, 0.0f);
    return;
  }
  const ViewRec& va = views[pr.a];
  const ViewRec& vb = views[pr.b];
  const ViewRec* vv[2] = {&va, &vb};
  df g[12];
  for (int i = 0; i < 12; ++i) g[i] = df{(float)G[i], 0.0f};  // an FP32 value: exact
  // d e / d w and d e / d v through A = cofc [w v]
  df gw[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, gv[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
  for (int s = 0; s < 2; ++s)
    for (int i = 0; i < 3; ++i) {
      const df g0 = g[6 * s + 2 * i], g1 = g[6 * s + 2 * i + 1];
      for (int k = 0; k < 3; ++k) {
        const df cof = qget(*vv[s], 6 + 3 * i + k);
        gw[k] = df_add(gw[k], df_mul(g0, cof));
        gv[k] = df_add(gv[k], df_mul(g1, cof));
      }
    }
  df w[3], v[3], gCa[3], gCb[3], gup[3];
  if (!pencil_frame_adjoint_df(va, vb, gw, gv, w, v, gCa, gCb, gup)) {
    for (int j = 0; j < 30; ++j) out[j] = make_float2(0.0f, 0.0f);
    return;
  }
  auto put = [&](int j, df x) { out[j] = make_float2(x.hi, x.lo); };
  for (int s = 0; s < 2; ++s)
    for (int i = 0; i < 3; ++i) {
      const df g0 = g[6 * s + 2 * i], g1 = g[6 * s + 2 * i + 1];
      for (int k = 0; k < 3; ++k) put(15 * s + 6 + 3 * i + k, df_add(df_mul(g0, w[k]), df_mul(g1, v[k])));
    }
  for (int k = 0; k < 3; ++k) {
    put(k, gCa[k]);
    put(3 + k, gup[k]);
    put(15 + k, gCb[k]);
    put(18 + k, gup[k]);
  }
}

// The first block sums the total meanwhile (a launch of its own before this one held up the
// gradient by 8 us).
__global__ void __launch_bounds__(kGradQThreads)
    pair_grad_q_kernel(long long n_pairs, const PairRec* prs, const ViewRec* views, const double* Gpp,
                       float2* __restrict__ gq, const double* partial,
                       int n_partial, double* __restrict__ total) {
  __shared__ double s[kSumSlots];
  wait_for_previous();
  if (blockIdx.x == 0) {
    reduce_fixed<kGradQThreads>(partial, n_partial, total, s);
    return;
  }
  const long long p = (long long)(blockIdx.x - 1) * kGradQThreads + threadIdx.x;
  if (p >= n_pairs) return;
  pair_grad_q(prs[p], views, Gpp + 12 * p, gq + 30 * p);
}

// Per-view sum of the pairs' q gradients in a fixed order (one block of 256 threads
// per view), in double-float: on return sh[k][0] (k < 15) holds d total / d q_k of view
// lam as a (hi, lo) pair.  With pairs == NULL the pairs of a view are found by the
// row-major a < b enumeration, otherwise by scanning the pair list.
__device__ void reduce_q_block(int lam, int n_views, long long n_pairs, const int32_t* __restrict__ pairs,
                               const float2* gq, float2 (*sh)[256]) {
  df acc[15];
  for (int k = 0; k < 15; ++k) acc[k] = df{0.0f, 0.0f};
  auto add = [&](const float2* q) {
    for (int k = 0; k < 15; ++k) {
      const float2 x = q[k];
      acc[k] = df_add(acc[k], df{x.x, x.y});
    }
  };
  if (pairs) {
    for (long long p = threadIdx.x; p < n_pairs; p += blockDim.x) {
      const int a = pairs[2 * p], b = pairs[2 * p + 1];
      if (a == lam) add(gq + 30 * p);
      if (b == lam) add(gq + 30 * p + 15);
    }
  } else {
    const long long n = n_views;
    for (int o = threadIdx.x; o < n_views; o += blockDim.x) {
      if (o == lam) continue;
      const long long a = o < lam ? o : lam, b = o < lam ? lam : o;
      const long long p = a * (2 * n - a - 1) / 2 + (b - a - 1);
      const int off = o < lam ? 15 : 0;  // this view is b of the pair when o < lam
      add(gq + 30 * p + off);
    }
  }
  for (int k = 0; k < 15; ++k) sh[k][threadIdx.x] = make_float2(acc[k].hi, acc[k].lo);
  __syncthreads();
  // a level's 15 wdt sums spread over all threads (by the first wdt threads alone the levels
  // took 15 sums in a row each)
  for (int wdt = 128; wdt > 0; wdt >>= 1) {
    for (int i = threadIdx.x; i < 15 * wdt; i += 256) {
      const int k = i / wdt, t = i % wdt;
      const float2 x = sh[k][t], y = sh[k][t + wdt];
      const df z = df_add(df{x.x, x.y}, df{y.x, y.y});
      sh[k][t] = make_float2(z.hi, z.lo);
    }
    __syncthreads();
  }
}

__device__ __forceinline__ double sh_value(const float2 (*sh)[256], int k) {
  return (double)sh[k][0].x + (double)sh[k][0].y;
}

// d total / d theta of one view from its q gradient (sh[k][0]) and the tangents
// d q / d theta (C, up, cofc rows).
__device__ __forceinline__ double contract_theta(const float2 (*sh)[256], const ViewTan& t, int j) {
  double g = 0.0;
  for (int k = 0; k < 3; ++k) g += sh_value(sh, k) * t.dC[k][j];
  for (int k = 0; k < 3; ++k) g += sh_value(sh, 3 + k) * t.dup[k][j];
  for (int k = 0; k < 9; ++k) g += sh_value(sh, 6 + k) * t.dcofc[k][j];
  return g;
}

// grad[view][6] = d total / d theta (one block of 256 threads per view).
__global__ void __launch_bounds__(256) view_grad_theta_kernel(int n_views, long long n_pairs,
                                                              const int32_t* __restrict__ pairs,
                                                              const float2* gq, const ViewTan* vtan,
                                                              double* __restrict__ grad) {
  wait_for_previous();
  __shared__ float2 sh[15][256];
  const int lam = blockIdx.x;
  reduce_q_block(lam, n_views, n_pairs, pairs, gq, sh);
  if (threadIdx.x < 6) grad[6 * lam + threadIdx.x] = contract_theta(sh, vtan[lam], threadIdx.x);
}

// grad_P[view][12] = d total / d P (one block of 256 threads per view).
__global__ void __launch_bounds__(256) view_grad_P_kernel(int n_views, long long n_pairs,
                                                          const int32_t* __restrict__ pairs,
                                                          const float2* gq, const ViewTanP* vtan,
                                                          double* __restrict__ grad_P) {
  wait_for_previous();
  __shared__ float2 sh[15][256];
  const int lam = blockIdx.x;
  reduce_q_block(lam, n_views, n_pairs, pairs, gq, sh);
  if (threadIdx.x < 12) {
    const ViewTanP& t = vtan[lam];
    double g = 0.0;
    for (int k = 0; k < 15; ++k) g += sh_value(sh, k) * t.d[k][threadIdx.x];
    grad_P[12 * lam + threadIdx.x] = g;
  }
}

// ---------------------------------------------------------------- serving rounds
// Blocks of one warp as in geometry_kernel: first the views, then (of jobs that take a
// gradient step) the tangent directions.
__global__ void __launch_bounds__(32) serve_view_kernel(const ServeJob* __restrict__ jobs,
                                                        const long long* __restrict__ voff, int n_jobs, long long total,
                                                        int view_blocks) {
  __shared__ GeometryShared sh;
  if ((int)blockIdx.x < view_blocks) {
    const long long t = (long long)blockIdx.x * (32 / kViewLanes) + threadIdx.x / kViewLanes, i = min(t, total - 1);
    const int j = serve_job_of(voff, n_jobs, i);
    const ServeJob& J = jobs[j];
    const long long v = i - voff[j];
    device_view(J.P + 12 * v, J.theta + 6 * v, J.W, J.H, sh, t < total, J.views + v, J.status);
    return;
  }
  const long long t = (long long)((int)blockIdx.x - view_blocks) * (32 / kTanLanes) + threadIdx.x / kTanLanes;
  const long long i = min(t, 6 * total - 1) / 6;
  const int j = serve_job_of(voff, n_jobs, i), dir = (int)(min(t, 6 * total - 1) % 6);
  const ServeJob& J = jobs[j];
  if (!__any_sync(0xffffffffu, J.do_grad)) return;
  const long long v = i - voff[j];
  device_tangent<false>(J.P + 12 * v, J.theta + 6 * v, dir, J.W, J.H, sh, J.do_grad && t < 6 * total,
                        &J.vtan[v].dC[0][0]);
}

__global__ void serve_pair_setup_kernel(const ServeJob* __restrict__ jobs, const long long* __restrict__ poff,
                                        int n_jobs, long long total) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const int j = serve_job_of(poff, n_jobs, i);
  const ServeJob& J = jobs[j];
  const long long p = i - poff[j];
  int a, b;
  pair_from_index(p, J.n_views, &a, &b);
  const PairRec r = setup_pair<1>(a, b, J.n_views, J.views, J.W, J.H, J.pair.K,
                               const_cast<float4*>(J.pair.ctile) + p * J.n_tiles, J.n_tiles, nullptr);
  if (r.status) atomicOr(J.status, kStatusDegeneratePair);
  const_cast<PairRec*>(J.pair.prs)[p] = r;
}

__global__ void serve_pair_grad_kernel(const ServeJob* __restrict__ jobs, const long long* __restrict__ poff,
                                       int n_jobs, long long total) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const int j = serve_job_of(poff, n_jobs, i);
  const ServeJob& J = jobs[j];
  if (!J.do_grad) return;
  const long long p = i - poff[j];
  pair_grad_q(J.pair.prs[p], J.views, J.pair.Gpp + 12 * p, J.gpp + 30 * p);
}

__global__ void __launch_bounds__(256) serve_view_grad_kernel(const ServeJob* __restrict__ jobs,
                                                              const long long* __restrict__ voff, int n_jobs) {
  __shared__ float2 sh[15][256];
  const long long i = blockIdx.x;
  const int j = serve_job_of(voff, n_jobs, i);
  const ServeJob& J = jobs[j];
  if (!J.do_grad) return;  // block-uniform
  const int lam = (int)(i - voff[j]);
  reduce_q_block(lam, J.n_views, J.pair.n_pairs, nullptr, J.gpp, sh);
  if (threadIdx.x < 6) J.grad[6 * lam + threadIdx.x] = contract_theta(sh, J.vtan[lam], threadIdx.x);
}

// Per-view jobs: theta <- theta - step * grad for the estimated parameters.
__global__ void serve_step_kernel(const ServeJob* __restrict__ jobs, const long long* __restrict__ voff, int n_jobs,
                                  long long total) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 6 * total) return;
  const int j = serve_job_of(voff, n_jobs, i / 6);
  const ServeJob& J = jobs[j];
  const long long k = i - 6 * voff[j];
  if (!J.do_grad || J.model != kMotionPerView || !(J.mask >> (int)(k % 6) & 1)) return;
  J.theta[k] = J.theta[k] - J.step * J.grad[k];
}

// Spline jobs: theta = theta0 + Akima(nodes) for the estimated parameters, and the
// window Jacobian of each (view, parameter).
__global__ void serve_spline_kernel(const ServeJob* __restrict__ jobs, const long long* __restrict__ voff,
                                    int n_jobs, long long total) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 6 * total) return;
  const int j = serve_job_of(voff, n_jobs, i / 6);
  const ServeJob& J = jobs[j];
  if (J.model != kMotionAkima) return;
  const long long k = i - 6 * voff[j];
  const int p = (int)(k % 6);
  const long long v = k / 6;
  if (!(J.mask >> p & 1)) {
    J.theta[k] = J.theta0[k];
    return;
  }
  const AkimaPoint a = akima_point(J.nodes + p, 6, J.n_nodes, J.h, (double)v);
  J.theta[k] = J.theta0[k] + a.value;
  for (int q = 0; q < 6; ++q) J.jac[6 * k + q] = a.d[q];
  J.jbase[k] = a.base;
}

// Spline jobs: node gradient d total / d y_(n, p) = sum over the views whose window
// holds node n of jac * grad, summed in view order; then the step on the nodes.
// One thread per (node, parameter) of a job, one block per job.
__global__ void serve_node_step_kernel(const ServeJob* __restrict__ jobs) {
  const ServeJob& J = jobs[blockIdx.x];
  if (!J.do_grad || J.model != kMotionAkima) return;
  for (int t = threadIdx.x; t < 6 * J.n_nodes; t += blockDim.x) {
    const int node = t / 6, p = t % 6;
    if (!(J.mask >> p & 1)) continue;
    // windows [i - 2, i + 3] hold node n for intervals i in [n - 3, n + 2]: views in
    // [(n - 3) h, (n + 3) h]
    const long long v0 = (long long)fmax(0.0, floor((node - 3) * J.h));
    const long long v1 = (long long)fmin((double)(J.n_views - 1), ceil((node + 3) * J.h));
    double g = 0.0;
    for (long long v = v0; v <= v1; ++v) {
      const long long k = 6 * v + p;
      const int q = node - J.jbase[k];
      if (q >= 0 && q < 6) g += J.jac[6 * k + q] * J.grad[k];
    }
    J.nodes[t] = J.nodes[t] - J.step * g;
  }
}

cudaError_t launch_serve_motion(const ServeJob* jobs, const long long* voff, int n_jobs, long long n_views,
                                cudaStream_t stream) {
  if (n_views > 0)
    serve_spline_kernel<<<(unsigned)((6 * n_views + 127) / 128), 128, 0, stream>>>(jobs, voff, n_jobs, n_views);
  return cudaGetLastError();
}

cudaError_t launch_serve_setup(const ServeJob* jobs, const long long* voff, const long long* poff, int n_jobs,
                               long long n_views, long long n_pairs, cudaStream_t stream) {
  if (n_views > 0) {
    const long long view_blocks = (n_views + 32 / kViewLanes - 1) / (32 / kViewLanes);
    const long long tan_blocks = (6 * n_views + 32 / kTanLanes - 1) / (32 / kTanLanes);
    serve_view_kernel<<<(unsigned)(view_blocks + tan_blocks), 32, 0, stream>>>(jobs, voff, n_jobs, n_views,
                                                                               (int)view_blocks);
  }
  if (n_pairs > 0)
    serve_pair_setup_kernel<<<(unsigned)((n_pairs + 127) / 128), 128, 0, stream>>>(jobs, poff, n_jobs, n_pairs);
  return cudaGetLastError();
}

cudaError_t launch_serve_grad(const ServeJob* jobs, const long long* voff, const long long* poff, int n_jobs,
                              long long n_views, long long n_pairs, cudaStream_t stream) {
  if (n_pairs > 0)
    serve_pair_grad_kernel<<<(unsigned)((n_pairs + 63) / 64), 64, 0, stream>>>(jobs, poff, n_jobs, n_pairs);
  if (n_views > 0) {
    serve_view_grad_kernel<<<(unsigned)n_views, 256, 0, stream>>>(jobs, voff, n_jobs);
    serve_step_kernel<<<(unsigned)((6 * n_views + 255) / 256), 256, 0, stream>>>(jobs, voff, n_jobs, n_views);
    serve_node_step_kernel<<<n_jobs, 128, 0, stream>>>(jobs);
  }
  return cudaGetLastError();
}

}  // namespace ecc

// Internal host entry point (tests only, not part of the public ABI): runs the
// per-view and per-pair set-up above on the CPU for views (a, b) of a scan so
// that the set-up logic can be checked without a GPU.
//   P host FP64 [n_views][12], motion host FP64 [n_views][6] or NULL
//   info_out [8]: sampled-arc start direction of sample 0 (c0x, c0y), dk, nk,
//                 status, r0hi, r1lo, r1hi
//   A_out [12]: the kappa -> line maps of views a and b
extern "C" int ecc_internal_setup_pair_host(int n_views, const double* P, const double* motion, int W, int H, int K,
                                            int a, int b, double* info_out, double* A_out) {
  if (n_views < 1 || a < 0 || b < 0 || a >= n_views || b >= n_views || K < 1) return -1;
  ecc::ViewRec views[2];
  for (int s = 0; s < 2; ++s) {
    const double* p = P + 12 * (s ? b : a);
    const double* m = motion ? motion + 6 * (s ? b : a) : nullptr;
    ecc::ViewWork<double> w;
    const bool ok = ecc::view_geometry<1, double>([=](int k) { return p[k]; }, [=](int k) { return m[k]; },
                                                  m != nullptr, W, H, 0, w, [] {});
    ecc::write_view<1>(w, ok, 0, &views[s]);
  }
  const int n_tiles = (K + 31) / 32;
  float4* ct = new float4[n_tiles];
  const ecc::PairRec r = ecc::setup_pair<1>(0, 1, 2, views, W, H, K, ct, n_tiles, nullptr);
  delete[] ct;
  info_out[0] = r.c0[0];
  info_out[1] = r.c0[1];
  info_out[2] = r.dk;
  info_out[3] = r.nk;
  info_out[4] = r.status;
  info_out[5] = r.r0hi;
  info_out[6] = r.r1lo;
  info_out[7] = r.r1hi;
  for (int i = 0; i < 12; ++i) A_out[i] = (double)(&r.Af[0][0])[2 * i] + (double)(&r.Af[0][0])[2 * i + 1];
  return 0;
}

// Internal host entry point (tests only): the Akima spline point of the motion
// model, computed by the same code as the serving kernels.
//   y host FP64 [n] node values, h node spacing, x position; out[0] value, out[1..6]
//   derivatives with respect to y[base .. base + 5]; *base receives base.
extern "C" int ecc_internal_akima_host(const double* y, int n, double h, double x, double* out, int* base) {
  if (!y || !out || !base || n < 3 || !(h > 0.0)) return -1;
  const ecc::AkimaPoint a = ecc::akima_point(y, 1, n, h, x);
  out[0] = a.value;
  for (int k = 0; k < 6; ++k) out[1 + k] = a.d[k];
  *base = a.base;
  return 0;
}

// Internal host entry point (tests only): the double-float angle functions of the
// per-pair set-up on the CPU.  op 0: out[2i], out[2i + 1] = sin, cos of x[i] (|x| <= 4);
// op 1: out[i] = atan2(x[i], y[i]).  Inputs are split into double-float pairs first.
extern "C" int ecc_internal_df_math_host(int op, const double* x, const double* y, int n, double* out) {
  if (!x || !out || n < 0 || (op == 1 && !y) || op < 0 || op > 1) return -1;
  for (int i = 0; i < n; ++i) {
    if (op == 0) {
      ecc::df s, c;
      ecc::df_sincos(ecc::df_from_double(x[i]), &s, &c);
      out[2 * i] = ecc::df_to_double(s);
      out[2 * i + 1] = ecc::df_to_double(c);
    } else {
      out[i] = ecc::df_to_double(ecc::df_atan2(ecc::df_from_double(x[i]), ecc::df_from_double(y[i])));
    }
  }
  return 0;
}

// Internal host entry point (tests only): the pencil frame of two sources and its
// reverse mode (pencil_frame_df, pencil_frame_adjoint_df) on the CPU.
//   Ca, Cb, upa, upb [3] host FP64; gw, gv [3] the incoming d e / d w, d e / d v
//   w_v_out [6] = w, v; grad_out [9] = d e / d Ca, d e / d Cb, d e / d up (each up axis)
// Returns -1 for coincident sources.
extern "C" int ecc_internal_frame_adjoint_host(const double* Ca, const double* Cb, const double* upa,
                                               const double* upb, const double* gw, const double* gv,
                                               double* w_v_out, double* grad_out) {
  ecc::ViewRec va{}, vb{};
  for (int k = 0; k < 3; ++k) {
    const ecc::df ca = ecc::df_from_double(Ca[k]), cb = ecc::df_from_double(Cb[k]);
    const ecc::df ua = ecc::df_from_double(upa[k]), ub = ecc::df_from_double(upb[k]);
    va.qdf[2 * k] = ca.hi; va.qdf[2 * k + 1] = ca.lo;
    vb.qdf[2 * k] = cb.hi; vb.qdf[2 * k + 1] = cb.lo;
    va.qdf[6 + 2 * k] = ua.hi; va.qdf[6 + 2 * k + 1] = ua.lo;
    vb.qdf[6 + 2 * k] = ub.hi; vb.qdf[6 + 2 * k + 1] = ub.lo;
  }
  ecc::df g_w[3], g_v[3], w[3], v[3], gCa[3], gCb[3], gup[3];
  for (int k = 0; k < 3; ++k) {
    g_w[k] = ecc::df_from_double(gw[k]);
    g_v[k] = ecc::df_from_double(gv[k]);
  }
  if (!ecc::pencil_frame_adjoint_df(va, vb, g_w, g_v, w, v, gCa, gCb, gup)) return -1;
  for (int k = 0; k < 3; ++k) {
    w_v_out[k] = ecc::df_to_double(w[k]);
    w_v_out[3 + k] = ecc::df_to_double(v[k]);
    grad_out[k] = ecc::df_to_double(gCa[k]);
    grad_out[3 + k] = ecc::df_to_double(gCb[k]);
    grad_out[6 + k] = ecc::df_to_double(gup[k]);
  }
  return 0;
}
