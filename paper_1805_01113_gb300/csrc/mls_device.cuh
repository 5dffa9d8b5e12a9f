// Device-side building blocks of the MLS transfer library: grid description,
// home-cell location, per-axis support geometry and the two shape-function
// evaluations (exact-MLS, Eqs. 3-6; fast-MLS, Eqs. 9-10).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace mls {

// One grid axis.  Cell i spans [faces[i], faces[i+1]); `uniform` axes also
// carry lo and h so the home cell comes from one multiply plus a face check.
// IEEE operations rounded to nearest with no contraction, so that a fixed
// order of operations is reproducible bit for bit by any IEEE implementation.
template <typename R> struct Ops;
template <> struct Ops<float> {
  static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
  static __device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
  static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
  static __device__ __forceinline__ float div(float a, float b) { return __fdiv_rn(a, b); }
  static __device__ __forceinline__ float sqrt_(float a) { return __fsqrt_rn(a); }
  static __device__ __forceinline__ float nan_() { return __int_as_float(0x7fc00000); }
};
template <> struct Ops<double> {
  static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
  static __device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
  static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
  static __device__ __forceinline__ double div(double a, double b) { return __ddiv_rn(a, b); }
  static __device__ __forceinline__ double sqrt_(double a) { return __dsqrt_rn(a); }
  static __device__ __forceinline__ double nan_() { return __longlong_as_double(0x7ff8000000000000ULL); }
};

// Marker of a triangle (Section 3): centroid C = ((V1+V2)+V3)/3 and area
// |(V2-V1)x(V3-V1)|/2, in this order of operations.
template <typename R>
__device__ __forceinline__ void triangle_marker(const R a[3], const R b[3], const R c[3], R x[3], R& area) {
  using O = Ops<R>;
  R e1[3], e2[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    x[d] = O::div(O::add(O::add(a[d], b[d]), c[d]), R(3));
    e1[d] = O::sub(b[d], a[d]);
    e2[d] = O::sub(c[d], a[d]);
  }
  const R nx = O::sub(O::mul(e1[1], e2[2]), O::mul(e1[2], e2[1]));
  const R ny = O::sub(O::mul(e1[2], e2[0]), O::mul(e1[0], e2[2]));
  const R nz = O::sub(O::mul(e1[0], e2[1]), O::mul(e1[1], e2[0]));
  area = O::mul(R(0.5), O::sqrt_(O::add(O::add(O::mul(nx, nx), O::mul(ny, ny)), O::mul(nz, nz))));
}

template <typename R>
struct Axis {
  const R* faces;   // n+1 values (device)
  const R* widths;  // n values (device)
  R lo, hi, h;      // faces[0], faces[n], width when uniform
  R inv_h;          // 1/h when uniform (rounded)
  int n;
  int periodic;
  int uniform;
  // Non-uniform axes: [lo, hi) cut into nbk equal buckets; bucket[b] is the
  // cell containing the bucket's lower edge (device, nbk values).
  const int* bucket;
  R inv_bw;         // nbk / (hi - lo) (rounded)
  int nbk;
};

template <typename R>
struct Grid {
  Axis<R> ax[3];
};

// Spreading tiles: 2^l home cells per axis; bins = tiles + 1 (the last bin
// collects dropped markers).
struct Tiles {
  int l[3];
  int nb[3];
  int nbins;
};

// Home cell of coordinate x on one axis: face_i <= x < face_{i+1}.  Returns -1
// outside [faces[0], faces[n]) or for NaN.  Uniform axes guess i from
// (x - lo) * (1/h), other axes take the cell of x's bucket; the guess is then
// corrected against the face array, so the result agrees with the exact
// comparison whatever the rounding of the guess (a bucket holds only a few
// faces, so the corrections take few steps).
template <typename R>
__device__ __forceinline__ int locate_axis(const Axis<R>& a, R x) {
  if (!(x >= a.lo && x < a.hi)) return -1;
  int i;
  if (a.uniform) {
    R s = (x - a.lo) * a.inv_h;
    i = (int)s;
    i = i < 0 ? 0 : (i > a.n - 1 ? a.n - 1 : i);
    if (x < a.faces[i]) --i;
    else if (x >= a.faces[i + 1]) ++i;
  } else {
    int b = (int)((x - a.lo) * a.inv_bw);
    b = b < 0 ? 0 : (b > a.nbk - 1 ? a.nbk - 1 : b);
    i = __ldg(a.bucket + b);
    while (i > 0 && x < a.faces[i]) --i;
    while (i < a.n - 1 && x >= a.faces[i + 1]) ++i;
  }
  return i;
}

// A home index is usable when the 3-wide support stays on the grid (always on
// periodic axes, which wrap).
template <typename R>
__device__ __forceinline__ bool support_ok(const Axis<R>& a, int i) {
  return i >= 0 && (a.periodic || (i >= 1 && i <= a.n - 2));
}

__device__ __forceinline__ int wrap(int j, int n, int periodic) {
  if (periodic) return j < 0 ? j + n : (j >= n ? j - n : j);
  return j < 0 ? 0 : (j >= n ? n - 1 : j);
}

template <typename R>
__device__ __forceinline__ R width_of(const Axis<R>& a, int j) {
  return a.uniform ? a.h : a.widths[j];
}

// Geometry of the 3 support nodes of one axis, in units of the home cell's
// width: xi[a] = (x_node - x_l)/Delta_home, node widths w[a] (physical), the
// marker's position frac in [0, 1) across the home cell, t = frac - 1/2, its
// offset from the home-cell centre, and the distances dm, dp of the two
// neighbour nodes from that centre (xi = -dm - t, -t, dp - t).
template <typename R>
struct AxisNodes {
  R xi[3];
  R w[3];
  R frac;
  R t;
  R dm, dp;
};

// On a uniform axis both width ratios are exactly 1 and the offset is
// (x - face_i) * (1/h), which equals (x - face_i)/h when h is a power of two.
template <typename R>
__device__ __forceinline__ AxisNodes<R> axis_nodes(const Axis<R>& a, int i, R x) {
  AxisNodes<R> s;
  if (a.uniform) {
    s.frac = (x - a.faces[i]) * a.inv_h;
    s.t = s.frac - R(0.5);
    s.xi[0] = R(-1) - s.t;
    s.xi[1] = -s.t;
    s.xi[2] = R(1) - s.t;
    s.w[0] = s.w[1] = s.w[2] = a.h;
    s.dm = s.dp = R(1);
    return s;
  }
  const R wh = width_of(a, i);
  const R wm = width_of(a, wrap(i - 1, a.n, a.periodic));
  const R wp = width_of(a, wrap(i + 1, a.n, a.periodic));
  s.frac = (x - a.faces[i]) / wh;
  s.t = s.frac - R(0.5);
  s.dm = R(0.5) + R(0.5) * (wm / wh);
  s.dp = R(0.5) + R(0.5) * (wp / wh);
  s.xi[0] = -s.dm - s.t;
  s.xi[1] = -s.t;
  s.xi[2] = s.dp - s.t;
  s.w[0] = wm;
  s.w[1] = wh;
  s.w[2] = wp;
  return s;
}

// Node geometry at a prescribed offset t with neighbour/home width ratios
// rm, rp (used to tabulate fast-MLS shape functions on the sub-Eulerian mesh).
template <typename R>
__device__ __forceinline__ AxisNodes<R> axis_nodes_at(R t, R wm, R wh, R wp) {
  AxisNodes<R> s;
  s.t = t;
  s.frac = t + R(0.5);
  s.dm = R(0.5) + R(0.5) * (wm / wh);
  s.dp = R(0.5) + R(0.5) * (wp / wh);
  s.xi[0] = -s.dm - t;
  s.xi[1] = -t;
  s.xi[2] = s.dp - t;
  s.w[0] = wm;
  s.w[1] = wh;
  s.w[2] = wp;
  return s;
}

template <typename R> __device__ __forceinline__ R dev_exp(R v);
// Single precision takes the hardware exponential: for the arguments here
// (|v| <= 4 with eps = 1) its relative error is a few ulp, far inside the
// single-precision tolerance of the shape functions.
template <> __device__ __forceinline__ float dev_exp<float>(float v) { return __expf(v); }
template <> __device__ __forceinline__ double dev_exp<double>(double v) { return exp(v); }

// 1/d: the hardware reciprocal in single precision (1 ulp), IEEE in double.
__device__ __forceinline__ float recip(float d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  return r;
}
__device__ __forceinline__ double recip(double d) { return 1.0 / d; }

// 1/sqrt(d): the hardware reciprocal square root in single precision (about
// 1 ulp), IEEE operations in double.
__device__ __forceinline__ float inv_sqrt(float d) { return rsqrtf(d); }
__device__ __forceinline__ double inv_sqrt(double d) { return 1.0 / sqrt(d); }

// 4x4 symmetric positive definite solve by Cholesky, A packed lower-triangular
// row by row: a00 a10 a11 a20 a21 a22 a30 a31 a32 a33.
template <typename R>
struct Chol4 {
  R l10, l20, l21, l30, l31, l32;
  R i0, i1, i2, i3;   // reciprocals of the diagonal of L
  bool ok;

  __device__ __forceinline__ void factor(const R a[10]) {
    R d0 = a[0];
    ok = d0 > R(0);
    i0 = inv_sqrt(d0);
    l10 = a[1] * i0;
    l20 = a[3] * i0;
    l30 = a[6] * i0;
    R d1 = a[2] - l10 * l10;
    ok = ok && d1 > R(0);
    i1 = inv_sqrt(d1);
    l21 = (a[4] - l20 * l10) * i1;
    l31 = (a[7] - l30 * l10) * i1;
    R d2 = a[5] - l20 * l20 - l21 * l21;
    ok = ok && d2 > R(0);
    i2 = inv_sqrt(d2);
    l32 = (a[8] - l30 * l20 - l31 * l21) * i2;
    R d3 = a[9] - l30 * l30 - l31 * l31 - l32 * l32;
    ok = ok && d3 > R(0);
    i3 = inv_sqrt(d3);
  }

  __device__ __forceinline__ void solve(const R b[4], R y[4]) const {
    R z0 = b[0] * i0;
    R z1 = (b[1] - l10 * z0) * i1;
    R z2 = (b[2] - l20 * z0 - l21 * z1) * i2;
    R z3 = (b[3] - l30 * z0 - l31 * z1 - l32 * z2) * i3;
    y[3] = z3 * i3;
    y[2] = (z2 - l32 * y[3]) * i2;
    y[1] = (z1 - l21 * y[2] - l31 * y[3]) * i1;
    y[0] = (z0 - l10 * y[1] - l20 * y[2] - l30 * y[3]) * i0;
  }
};

// ---- exact-MLS shape functions in closed form (Eqs. 3-6) ---------------------
// The Gaussian weight and the 27-node stencil are tensor products, so the
// moment matrix A = sum_k W_k p_k p_k^T is diagonal in the products of per-axis
// polynomials that are orthogonal under that axis's three normalised weights
// n_a = w_a / sum w: P0 = 1, P1 = xi - m, P2 = P1^2 - s P1 - v, with the mean m
// and the variance v of xi.  The linear basis spans P0 and the three P1, the
// quadratic basis [1, xi_x, .., xi_z xi_x] all products of total degree <= 2,
// so Phi^T = e_0^T A^-1 B (Eq. 6, p(x_l) = e_0 in the marker-centred basis) is
//   phi_abc = sum_{i+j+k <= 1 or 2} E_i,a[x] E_j,b[y] E_k,c[z],
//   E_i,a = n_a P_i(0) P_i(xi_a) / sum_a n_a P_i(xi_a)^2.
// Nothing is assembled, factored or refined.  Offsets are taken from the
// home-cell centre, where the middle node sits, so the mean offset mu keeps its
// relative accuracy when the outer weights are tiny (narrow cells between wide
// ones); E_2, a difference of values of order one, keeps its absolute accuracy.  It replaced a 4 x 4 (or
// 10 x 10) Cholesky solve with a refinement step per marker, which issued 124 M
// (276 M) warp instructions on 4 M markers at 64 (166) registers; the quadratic
// build with its interpolation went from 944 to 544 us there, with half the
// error (2.7e-7 to 1.2e-7 against double precision).
constexpr int kQuad = 10;  // size of the quadratic basis (the linear one has 4)

// One axis: E_0, E_1 (and E_2 for the quadratic basis) at the three nodes, and
// the moments the condition number needs.
template <typename R, int MB>
struct AxisForm {
  R e0[3], e1[3], e2[MB == 4 ? 1 : 3];
  R m, v, iv, g;  // mean and variance of xi under n, 1 / v, g = m / v
  R c3, q2;    // quadratic: third central moment and sum_a n_a P2(xi_a)^2
};

// Weights relative to the middle node's: w_a / w_1 = exp(-(xi_a^2 - xi_1^2)/eps^2),
// with xi_0^2 - xi_1^2 = dm (dm + 2 t) and xi_2^2 - xi_1^2 = dp (dp - 2 t).  A
// middle node that is not the nearest (next to a narrower cell) scales by the
// largest instead, so that no weight overflows.  Returns false when the
// variance is not a normal positive number (the weights of the outer nodes
// vanish or an input is NaN); phi is then not defined in this precision.
template <int MB, typename R>
__device__ __forceinline__ bool axis_form(const AxisNodes<R>& s, R inv_eps2, AxisForm<R, MB>& f) {
  R a0 = -(s.dm * (s.dm + R(2) * s.t)) * inv_eps2, a2 = -(s.dp * (s.dp - R(2) * s.t)) * inv_eps2, w1 = R(1);
  const R top = a0 > a2 ? a0 : a2;
  if (top > R(0)) {
    a0 -= top;
    a2 -= top;
    w1 = dev_exp<R>(-top);
  }
  const R w0 = dev_exp<R>(a0), w2 = dev_exp<R>(a2);
  const R inv = recip(w0 + w1 + w2);
  f.e0[0] = w0 * inv;
  f.e0[1] = w1 * inv;
  f.e0[2] = w2 * inv;
  const R mu = f.e0[2] * s.dp - f.e0[0] * s.dm;
  const R c[3] = {-s.dm - mu, -mu, s.dp - mu};
  R nc[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) nc[a] = f.e0[a] * c[a];
  f.v = nc[0] * c[0] + nc[1] * c[1] + nc[2] * c[2];
  f.m = mu - s.t;
  f.iv = recip(f.v);
  f.g = f.m * f.iv;
#pragma unroll
  for (int a = 0; a < 3; ++a) f.e1[a] = -(nc[a] * f.g);
  if constexpr (MB != 4) {
    // On three nodes E_0 + E_1 + E_2 interpolates: the Lagrange weights at the marker.
    const R id = recip(s.dm + s.dp), im = recip(s.dm), ip = recip(s.dp);
    const R l0 = s.xi[1] * s.xi[2] * (im * id), l1 = -(s.xi[0] * s.xi[2]) * (im * ip), l2 = s.xi[0] * s.xi[1] * (ip * id);
    f.e2[0] = l0 - f.e0[0] - f.e1[0];
    f.e2[1] = l1 - f.e0[1] - f.e1[1];
    f.e2[2] = l2 - f.e0[2] - f.e1[2];
    f.c3 = nc[0] * c[0] * c[0] + nc[1] * c[1] * c[1] + nc[2] * c[2] * c[2];
    // The Gram determinant of 1, P1, P2 on three nodes is v sum n P2^2 and also
    // n_0 n_1 n_2 times the squared Vandermonde determinant.  As c4 - c3^2/v - v^2
    // the sum would be rounding noise of either sign once an outer weight is tiny.
    const R vd = s.dm * s.dp * (s.dm + s.dp);
    f.q2 = (f.e0[0] * vd) * (f.e0[2] * vd) * f.e0[1] * recip(f.v);
  }
  return f.v > (sizeof(R) == 4 ? R(1e-30) : R(1e-290));
}

// Derivatives of E_0 and E_1 of one axis along it, per physical length (inv_h =
// 1 / home width).  With beta = 2/eps^2 and c_a the offsets from the mean node,
// d n_a = beta n_a c_a, d m = beta v - 1 and d v = beta c3 (c3 = sum n c^3), so
//   d E_1,a = -(d(n_a c_a) g + n_a c_a d g),  d(n_a c_a) = beta n_a (c_a^2 - v),
//   d g = beta - (1 + beta g c3) / v.
template <typename R>
__device__ __forceinline__ void axis_slopes(const AxisNodes<R>& s, const AxisForm<R, 4>& f, R inv_eps2, R inv_h,
                                            R d0[3], R d1[3]) {
  const R beta = R(2) * inv_eps2;
  const R mu = f.e0[2] * s.dp - f.e0[0] * s.dm;
  const R c[3] = {-s.dm - mu, -mu, s.dp - mu};
  R nc[3], c3 = R(0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    nc[a] = f.e0[a] * c[a];
    c3 += nc[a] * c[a] * c[a];
  }
  const R bh = beta * inv_h, bg = bh * f.g, dg = (beta - (R(1) + beta * f.g * c3) * f.iv) * inv_h;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    d0[a] = bh * nc[a];
    d1[a] = -(bg * (nc[a] * c[a] - f.e0[a] * f.v) + nc[a] * dg);
  }
}

// cond_1(A) = ||A||_1 ||A^-1||_1 for the linear basis: with weights of unit sum
// A = [1 m^T; m diag(v) + m m^T] and A^-1 = [1 + m.g, -g^T; -g, diag(1/v)].
template <typename R>
__device__ __forceinline__ R cond1(const AxisForm<R, 4> f[3]) {
  const R am[3] = {fabs(f[0].m), fabs(f[1].m), fabs(f[2].m)};
  const R ag[3] = {fabs(f[0].g), fabs(f[1].g), fabs(f[2].g)};
  const R sum = am[0] + am[1] + am[2];
  R an = R(1) + sum, in = R(1) + (am[0] * ag[0] + am[1] * ag[1] + am[2] * ag[2]) + (ag[0] + ag[1] + ag[2]);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    an = fmax(an, am[d] * (R(1) + sum) + f[d].v);
    in = fmax(in, ag[d] + recip(f[d].v));
  }
  return an * in;
}

// The same for the quadratic basis, column by column, from the raw moments r_k
// (k <= 4) of each axis and the monomial coefficients of the orthogonal
// products: P2 = xi^2 - al xi + be, al = 2 m + s, be = m^2 + s m - v, with
// s = c3 / v; the fourth central moment is q2 + s c3 + v^2.
template <typename R>
__device__ __forceinline__ R cond1(const AxisForm<R, kQuad> f[3]) {
  R r[3][5], iv[3], i2[3], al[3], be[3], m[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const R v = f[d].v, c3 = f[d].c3;
    m[d] = f[d].m;
    iv[d] = recip(v);
    const R mm = m[d] * m[d], s = c3 * iv[d], c4 = f[d].q2 + s * c3 + v * v;
    r[d][0] = R(1);
    r[d][1] = m[d];
    r[d][2] = v + mm;
    r[d][3] = c3 + m[d] * (R(3) * v + mm);
    r[d][4] = c4 + m[d] * (R(4) * c3 + m[d] * (R(6) * v + mm));
    i2[d] = recip(f[d].q2);
    al[d] = R(2) * m[d] + s;
    be[d] = mm + s * m[d] - v;
#pragma unroll
    for (int k = 0; k < 5; ++k) r[d][k] = fabs(r[d][k]);
  }
  // Columns of A: the monomial x^p y^q z^t against the ten of the basis.
  auto col = [&](int p, int q, int t) {
    const R x0 = r[0][p], x1 = r[0][p + 1], y0 = r[1][q], y1 = r[1][q + 1], z0 = r[2][t], z1 = r[2][t + 1];
    return x0 * y0 * (z0 + z1 + r[2][t + 2]) + (x1 + r[0][p + 2]) * y0 * z0 + x0 * (y1 + r[1][q + 2]) * z0 +
           x1 * y1 * z0 + x0 * y1 * z1 + x1 * y0 * z1;
  };
  R an = fmax(fmax(fmax(col(0, 0, 0), col(1, 0, 0)), fmax(col(0, 1, 0), col(0, 0, 1))),
              fmax(fmax(col(2, 0, 0), col(0, 2, 0)), fmax(col(0, 0, 2), col(1, 1, 0))));
  an = fmax(an, fmax(col(0, 1, 1), col(1, 0, 1)));
  // Columns of A^-1, by the same monomials.
  R c0 = R(1), off0 = R(0), in = R(0);
  R lin[3], row1[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    lin[d] = iv[d] + al[d] * al[d] * i2[d];
    row1[d] = -m[d] * iv[d] - al[d] * be[d] * i2[d];
    c0 += m[d] * m[d] * iv[d] + be[d] * be[d] * i2[d];
    off0 += fabs(be[d]) * i2[d];
  }
  R cross[3];  // |(xi_d, xi_e)| for the pairs d, e = (0,1), (1,2), (2,0)
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int d = q, e = (q + 1) % 3;
    const R pv = iv[d] * iv[e];
    lin[d] += m[e] * m[e] * pv;
    lin[e] += m[d] * m[d] * pv;
    row1[d] -= m[e] * m[e] * m[d] * pv;
    row1[e] -= m[d] * m[d] * m[e] * pv;
    c0 += m[d] * m[d] * m[e] * m[e] * pv;
    off0 += fabs(m[d] * m[e]) * pv;
    cross[q] = fabs(m[d] * m[e]) * pv;
    in = fmax(in, pv * (R(1) + fabs(m[d]) + fabs(m[e]) + fabs(m[d] * m[e])));
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int e = (d + 1) % 3, g = (d + 2) % 3;
    off0 += fabs(row1[d]);
    in = fmax(in, i2[d] * (R(1) + fabs(al[d]) + fabs(be[d])));
    in = fmax(in, fabs(row1[d]) + lin[d] + cross[d] + cross[g] + fabs(al[d]) * i2[d] +
                      iv[d] * (fabs(m[e]) * iv[e] + fabs(m[g]) * iv[g]));
  }
  return an * fmax(in, c0 + off0);
}

// An upper bound of cond_1(A) that costs a few operations: for a symmetric
// positive definite matrix of size n, cond_1 <= n tr(A) tr(A^-1), and both
// traces are sums of products of per-axis terms.  A marker below the limit by
// this bound is below it; only the others evaluate cond1.
template <typename R>
__device__ __forceinline__ R cond_bound(const AxisForm<R, kQuad> f[3]) {
  R q2[3], q4[3], t1[3], t2[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const R v = f[d].v, c3 = f[d].c3, m = f[d].m, mm = m * m, iv = recip(v), s = c3 * iv;
    q2[d] = v + mm;
    q4[d] = f[d].q2 + s * c3 + v * v + m * (R(4) * c3 + m * (R(6) * v + mm));
    t1[d] = (R(1) + mm) * iv;
    const R al = R(2) * m + s, be = mm + s * m - v;
    t2[d] = (R(1) + al * al + be * be) * recip(f[d].q2);
  }
  const R ta = R(1) + q2[0] + q2[1] + q2[2] + q4[0] + q4[1] + q4[2] + q2[0] * q2[1] + q2[1] * q2[2] + q2[2] * q2[0];
  const R ti = R(1) + t1[0] + t1[1] + t1[2] + t2[0] + t2[1] + t2[2] + t1[0] * t1[1] + t1[1] * t1[2] + t1[2] * t1[0];
  return R(kQuad) * ta * ti;
}

// Whether cond_1(A) exceeds `limit`.  NaN counts as exceeding, and so does a
// norm of P2 that is no normal number (its reciprocal would be infinite, and
// fmax passes NaN over).
template <typename R>
__device__ __forceinline__ bool cond_above(const AxisForm<R, 4> f[3], R limit) {
  return !(cond1(f) <= limit);
}
template <typename R>
__device__ __forceinline__ bool cond_above(const AxisForm<R, kQuad> f[3], R limit) {
  const R tiny = sizeof(R) == 4 ? R(1e-37) : R(1e-300);
  if (!(f[0].q2 > tiny && f[1].q2 > tiny && f[2].q2 > tiny)) return true;
  if (cond_bound(f) <= R(0.99) * limit) return false;
  return !(cond1(f) <= limit);
}

// The three axes of a marker; false when phi is not defined in this precision.
template <int MB, typename R>
__device__ __forceinline__ bool exact_form(const AxisNodes<R> s[3], R inv_eps2, AxisForm<R, MB> f[3]) {
  bool ok = true;
#pragma unroll
  for (int d = 0; d < 3; ++d) ok = axis_form<MB>(s[d], inv_eps2, f[d]) && ok;
  return ok;
}

// Streams phi_k, k = 9c + 3b + a, as polynomials of E_i[x] whose coefficients
// are formed once per (b, c).
template <int MB, typename R, typename Sink>
__device__ __forceinline__ void exact_emit(const AxisForm<R, MB> f[3], Sink&& sink) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const R z0 = f[2].e0[c], z01 = z0 + f[2].e1[c];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const R y0 = f[1].e0[b], y1 = f[1].e1[b];
      const R k0 = y0 * z0, k1 = y0 * z01 + y1 * z0;
      if constexpr (MB == 4) {
#pragma unroll
        for (int a = 0; a < 3; ++a) sink(a, b, c, f[0].e0[a] * k1 + f[0].e1[a] * k0);
      } else {
        const R k2 = y0 * (z01 + f[2].e2[c]) + (y1 * z01 + f[1].e2[b] * z0);
#pragma unroll
        for (int a = 0; a < 3; ++a) sink(a, b, c, f[0].e0[a] * k2 + (f[0].e1[a] * k1 + f[0].e2[a] * k0));
      }
    }
  }
}

// c_l of Eq. 8, A_l h_l / sum_k phi_k dV_k with h_l = sum_k phi_k (Dx_k + Dy_k
// + Dz_k)/3, without the 27 terms: E_i sums to 1 over an axis for i = 0 and to
// 0 otherwise, so sum_k phi_k Dx_k = sum_a (E_0 + E_1 (+ E_2))_a Dx_a, and
// sum_k phi_k dV_k combines the per-axis sums V_i = sum_a E_i,a D_a as phi
// combines E_i.  Returns 0 when sum_k phi_k dV_k is 0.
template <int MB, typename R>
__device__ __forceinline__ R exact_scale(const AxisNodes<R> s[3], const AxisForm<R, MB> f[3], R area) {
  R V[3][3], h = R(0);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    V[d][0] = f[d].e0[0] * s[d].w[0] + f[d].e0[1] * s[d].w[1] + f[d].e0[2] * s[d].w[2];
    V[d][1] = f[d].e1[0] * s[d].w[0] + f[d].e1[1] * s[d].w[1] + f[d].e1[2] * s[d].w[2];
    V[d][2] = R(0);
    if constexpr (MB != 4) V[d][2] = f[d].e2[0] * s[d].w[0] + f[d].e2[1] * s[d].w[1] + f[d].e2[2] * s[d].w[2];
    h += V[d][0] + V[d][1] + V[d][2];
  }
  const R k0 = V[1][0] * V[2][0], k1 = V[1][0] * (V[2][0] + V[2][1]) + V[1][1] * V[2][0];
  R vol = V[0][0] * k1 + V[0][1] * k0;
  if constexpr (MB != 4)
    vol = V[0][0] * (V[1][0] * (V[2][0] + V[2][1] + V[2][2]) + V[1][1] * (V[2][0] + V[2][1]) + V[1][2] * V[2][0]) +
          V[0][1] * k1 + V[0][2] * k0;
  return vol != R(0) ? (area * (h / R(3))) / vol : R(0);
}

// All 27 exact shape functions (table path).
template <typename R, int MB = 4>
__device__ __forceinline__ bool shape_exact(const AxisNodes<R> s[3], R inv_eps2, R phi[27]) {
  AxisForm<R, MB> f[3];
  if (!exact_form<MB>(s, inv_eps2, f)) return false;
  exact_emit<MB>(f, [&](int a, int b, int c, R v) { phi[9 * c + 3 * b + a] = v; });
  return true;
}

// Running sums for c_l of Eq. 8 while phi is streamed out.
template <typename R>
struct ScaleSums {
  R mx[3], my[3], mz[3], vol;
  __device__ __forceinline__ ScaleSums() {
#pragma unroll
    for (int q = 0; q < 3; ++q) mx[q] = my[q] = mz[q] = R(0);
    vol = R(0);
  }
  __device__ __forceinline__ void add(const AxisNodes<R> s[3], int a, int b, int c, R p) {
    mx[a] += p;
    my[b] += p;
    mz[c] += p;
    vol += p * (s[0].w[a] * s[1].w[b] * s[2].w[c]);
  }
  // The three nodes (0..2, b, c) of one row.
  __device__ __forceinline__ void add_row(const AxisNodes<R> s[3], int b, int c, const R p[3]) {
    const R r = p[0] + p[1] + p[2];
#pragma unroll
    for (int a = 0; a < 3; ++a) mx[a] += p[a];
    my[b] += r;
    mz[c] += r;
    vol += (p[0] * s[0].w[0] + p[1] * s[0].w[1] + p[2] * s[0].w[2]) * (s[1].w[b] * s[2].w[c]);
  }
  // c_l = A_l h_l / sum_k phi_k dV_k, h_l = sum_k phi_k (Dx_k + Dy_k + Dz_k)/3.
  __device__ __forceinline__ R scale(const AxisNodes<R> s[3], R area) const {
    R hsum = R(0);
#pragma unroll
    for (int q = 0; q < 3; ++q) hsum += mx[q] * s[0].w[q] + my[q] * s[1].w[q] + mz[q] * s[2].w[q];
    return (area * (hsum / R(3))) / vol;
  }
};

}  // namespace mls
