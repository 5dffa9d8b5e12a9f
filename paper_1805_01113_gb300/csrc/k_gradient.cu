// Gradients of interpolated fields at the markers from the derivatives of the
// exact-MLS shape functions (Section 2: MLS gives values and spatial
// derivatives; the solver needs velocity and pressure gradients at markers).
#include "build_common.cuh"
#include "transfer_common.cuh"

namespace mls {

template <typename R> constexpr int kGradThreads = sizeof(R) == 4 ? kBlock : kBlockF64;

// One axis of a marker's derivative: the linear basis functions E_0, E_1 and
// their slopes at the three nodes.
template <typename R>
struct AxisSlopes {
  R e0[3], e1[3], d0[3], d1[3];
};

// Functions that sum to zero (E_0: to one) over the nodes, against the outer
// values' differences from the middle one, which then enters through them alone.
template <typename R>
__device__ __forceinline__ R ends(const R w[3], R lo, R hi) {
  return w[0] * lo + w[2] * hi;
}

// The value at node a of a function with that sum, from the outer two (so that
// the middle one need not be kept for the rare use of this).
template <typename R>
__device__ __forceinline__ R of_node(const R w[3], R sum, int a) {
  return a == 0 ? w[0] : a == 2 ? w[2] : sum - w[0] - w[2];
}

// The derivatives of phi at node (n_x, n_y, n_z).
template <typename R>
__device__ __forceinline__ void node_slopes(const AxisSlopes<R> f[3], const int n[3], R out[3]) {
  R e0[3], e1[3], d0[3], d1[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    e0[d] = of_node(f[d].e0, R(1), n[d]);
    e1[d] = of_node(f[d].e1, R(0), n[d]);
    d0[d] = of_node(f[d].d0, R(0), n[d]);
    d1[d] = of_node(f[d].d1, R(0), n[d]);
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int a = (d + 1) % 3, b = (d + 2) % 3;
    out[d] = d0[d] * (e0[a] * (e0[b] + e1[b]) + e1[a] * e0[b]) + d1[d] * (e0[a] * e0[b]);
  }
}

// One component's derivatives as the plain sum over the nodes, where a value of
// the stencil is not finite (or a difference overflows): an infinity then
// reaches the derivatives with its own weight's sign only.
template <typename R, typename FT>
__device__ __forceinline__ void plain_sum(const AxisSlopes<R> f[3], const FT* __restrict__ u, const int xs[3],
                                          const int rows[3][3], R out[3]) {
  out[0] = out[1] = out[2] = R(0);
#pragma unroll 1
  for (int k = 0; k < 27; ++k) {
    const int n[3] = {k % 3, k / 3 % 3, k / 9};
    R w[3];
    node_slopes(f, n, w);
    int o = n[0] == 0 ? xs[0] : n[0] == 1 ? xs[1] : xs[2];
#pragma unroll
    for (int q = 0; q < 9; ++q)
      if (q == k / 3) o += rows[q / 3][q % 3];
    const R v = load_field<R, FT>(u + o);
#pragma unroll
    for (int d = 0; d < 3; ++d) out[d] += w[d] * v;
  }
}

// The sums in double precision, node by node for all components at once: the
// contraction below has a quarter more operations, and FP64 units are what this
// form waits for (433 us on 261 120 markers in 128^3; contracted, a sixth more).
// The field is taken relative to a mean of the home cell and its six neighbours,
// which leaves less to round than the home cell's own value where the field varies
// from cell to cell (48^3, up to 16 waves per box: 3.4 against 4.0e-16).
template <typename FT>
__device__ __forceinline__ void node_sum(const AxisSlopes<double> f[3], const FT* __restrict__ u, int64_t N,
                                         const int xs[3], const int rows[3][3], double out[3][3]) {
  double mid[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    auto at = [&](int x, int y, int z) { return load_field<double, FT>(u + c * N + rows[z][y] + xs[x]); };
    const double own = at(1, 1, 1);
    mid[c] = 0.125 * (((at(0, 1, 1) + at(2, 1, 1)) + (at(1, 0, 1) + at(1, 2, 1))) +
                      ((at(1, 1, 0) + at(1, 1, 2)) + (own + own)));
#pragma unroll
    for (int d = 0; d < 3; ++d) out[c][d] = 0.0;
  }
#pragma unroll
  for (int cz = 0; cz < 3; ++cz) {
    const double z0 = f[2].e0[cz], z01 = z0 + f[2].e1[cz], dz0 = f[2].d0[cz], dz01 = dz0 + f[2].d1[cz];
#pragma unroll
    for (int cy = 0; cy < 3; ++cy) {
      const double y0 = f[1].e0[cy], y1 = f[1].e1[cy], dy0 = f[1].d0[cy], dy1 = f[1].d1[cy];
      const double k0 = y0 * z0, k1 = y0 * z01 + y1 * z0;
      const double ky0 = dy0 * z0, ky1 = dy0 * z01 + dy1 * z0;
      const double kz0 = y0 * dz0, kz1 = y0 * dz01 + y1 * dz0;
#pragma unroll
      for (int cx = 0; cx < 3; ++cx) {
        const double e0 = f[0].e0[cx], e1 = f[0].e1[cx];
        const double w[3] = {f[0].d0[cx] * k1 + f[0].d1[cx] * k0, e0 * ky1 + e1 * ky0, e0 * kz1 + e1 * kz0};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const double v = load_field<double, FT>(u + c * N + rows[cz][cy] + xs[cx]) - mid[c];
#pragma unroll
          for (int d = 0; d < 3; ++d) out[c][d] += w[d] * v;
        }
      }
    }
  }
}

// G[c][d][l] = sum_k d_d phi_k^l u_c,k.  One thread per marker in tile order.
// phi_abc = E_0,a (E_0,b (E_0 + E_1)_c + E_1,b E_0,c) + E_1,a E_0,b E_0,c, and a
// derivative along an axis replaces that axis's E by its slopes.  The sums are
// contracted axis by axis over differences between neighbouring nodes, in which
// a constant part of the field cancels before any rounding: with the field's own
// values the error of a smooth field grows as its gradient falls, and with the
// field relative to the home cell's value, rounded per node, a rough one loses.
// Wave numbers up to 16 per box, error over the gradient's norm, by own values,
// by home-relative ones and so: 1.4, 1.8 and 1.2e-7 in 48^3, 3.4, 1.24 and 0.85e-7
// in 384^3.  The 81 gathers of a marker go through the cache hierarchy (the
// markers of a home cell are adjacent, so a warp's gathers share lines) and are
// what the kernel waits for: 271 us on 4 M markers in 512^3 at 64 registers, 300
// at 80, against 38 us for the bytes; the home-relative sum took 282.
template <typename R, typename FT>
__global__ void __launch_bounds__(kGradThreads<R>, sizeof(R) == 4 ? 4 : 1)
    k_interp_gradient(Dims D, Grid<R> g, const R* __restrict__ x, const int32_t* __restrict__ home,
                      const int32_t* __restrict__ perm, int64_t M, R inv_eps2, const FT* __restrict__ u,
                      R* __restrict__ G) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= M) return;
  const int64_t m = perm[j];
  const int32_t hc = home[j];
  bool ok = hc >= 0;
  AxisSlopes<R> f[3];
  int xs[3], rows[3][3];
  if (ok) {
    int i[3];
    decode_home(hc, D, i);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const AxisNodes<R> s = axis_nodes(g.ax[d], i[d], x[d * M + m]);
      AxisForm<R, 4> a;
      ok = axis_form<4>(s, inv_eps2, a) && ok;
      axis_slopes(s, a, inv_eps2, R(1) / s.w[1], f[d].d0, f[d].d1);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        f[d].e0[q] = a.e0[q];
        f[d].e1[q] = a.e1[q];
      }
    }
    support_offsets(g, i, xs, rows);
  }
  if (!ok) {
#pragma unroll
    for (int q = 0; q < 9; ++q) G[q * M + m] = R(0);
    return;
  }
  const int64_t N = (int64_t)D.n[0] * D.n[1] * D.n[2];
  if constexpr (sizeof(R) == 8) {
    R out[3][3];
    node_sum<FT>(f, u, N, xs, rows, out);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (!isfinite(out[c][0] + out[c][1] + out[c][2])) plain_sum<R, FT>(f, u + c * N, xs, rows, out[c]);
#pragma unroll
      for (int d = 0; d < 3; ++d) G[(3 * c + d) * M + m] = out[c][d];
    }
    return;
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const FT* uc = u + c * N;
    R out[3] = {R(0), R(0), R(0)}, v_mid = R(0), w_mid = R(0);
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const int cz = t == 0 ? 1 : t == 1 ? 0 : 2;   // the middle plane first: the others are taken against it
      R v[3], e0[3], e1[3], d0[3], d1[3];           // per row: the middle node and the sums over x without it
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const FT* ur = uc + rows[cz][b];
        v[b] = load_field<R, FT>(ur + xs[1]);
        const R lo = load_field<R, FT>(ur + xs[0]) - v[b], hi = load_field<R, FT>(ur + xs[2]) - v[b];
        e0[b] = ends(f[0].e0, lo, hi);
        e1[b] = ends(f[0].e1, lo, hi);
        d0[b] = ends(f[0].d0, lo, hi);
        d1[b] = ends(f[0].d1, lo, hi);
      }
      const R e0l = (e0[0] - e0[1]) + (v[0] - v[1]), e0h = (e0[2] - e0[1]) + (v[2] - v[1]);
      const R e1l = e1[0] - e1[1], e1h = e1[2] - e1[1];
      const R d0l = d0[0] - d0[1], d0h = d0[2] - d0[1], d1l = d1[0] - d1[1], d1h = d1[2] - d1[1];
      const AxisSlopes<R>& y = f[1];
      // Sums over the plane: the coefficient of E_0 + E_1 along z, and that of E_0.
      const R x1 = d0[1] + ends(y.e0, d0l, d0h), x0 = d1[1] + ends(y.e0, d1l, d1h) + ends(y.e1, d0l, d0h);
      const R y1 = ends(y.d0, e0l, e0h), y0 = ends(y.d0, e1l, e1h) + ends(y.d1, e0l, e0h);
      const R w1 = e0[1] + ends(y.e0, e0l, e0h), w0 = e1[1] + ends(y.e0, e1l, e1h) + ends(y.e1, e0l, e0h);
      const R z0 = f[2].e0[cz], z01 = z0 + f[2].e1[cz], dz0 = f[2].d0[cz], dz01 = dz0 + f[2].d1[cz];
      out[0] += z01 * x1 + z0 * x0;
      out[1] += z01 * y1 + z0 * y0;
      out[2] += dz0 * w0;
      if (cz == 1) {
        v_mid = v[1];
        w_mid = w1;
      } else {
        out[2] += dz01 * ((w1 - w_mid) + (v[1] - v_mid));
      }
    }
    if (!isfinite(out[0] + out[1] + out[2])) plain_sum<R, FT>(f, uc, xs, rows, out);
#pragma unroll
    for (int d = 0; d < 3; ++d) G[(3 * c + d) * M + m] = out[d];
  }
}

template <typename R, typename FT>
static void launch_gradient(const mls_ctx* ctx, const mls_transfer* T, const void* x, const void* u, void* G,
                            cudaStream_t s) {
  const unsigned nt = block_threads(T->M, kGradThreads<R>);
  k_interp_gradient<R, FT><<<blocks_for(T->M, nt), nt, 0, s>>>(
      dims_of(ctx), device_grid<R>(ctx), (const R*)x, T->home, T->perm, T->M,
      (R)(1.0 / (ctx->opt.eps * ctx->opt.eps)), (const FT*)u, (R*)G);
}

cudaError_t launch_interp_gradient(const mls_ctx* ctx, const mls_transfer* T, const void* x, const void* u, void* G,
                                   cudaStream_t s) {
  if (T->M == 0) return cudaSuccess;
  if (ctx->opt.real == MLS_F64)
    launch_gradient<double, double>(ctx, T, x, u, G, s);
  else if (ctx->opt.field == MLS_F32)
    launch_gradient<float, float>(ctx, T, x, u, G, s);
  else
    launch_gradient<float, __nv_bfloat16>(ctx, T, x, u, G, s);
  return cudaGetLastError();
}

}  // namespace mls
