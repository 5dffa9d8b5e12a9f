// Euler-to-Lagrange interpolation (gather) and Lagrange-to-Euler spreading
// (scatter through shared-memory tile accumulators in single precision,
// direct global reductions in double precision).
#include "spread_runs.cuh"

namespace mls {

// U_l = sum_k phi_k^l u_k for the 3 components (text after Eq. 6), double
// precision.  One thread per stored marker; the 27 phi values are read with
// unit stride across the warp, the field through the read-only path.
template <typename R, typename FT>
__global__ void __launch_bounds__(kBlock) k_interp(Dims D, const R* __restrict__ phi, const int32_t* __restrict__ home,
                                                   const int32_t* __restrict__ perm, int64_t M, int64_t cap,
                                                   const FT* __restrict__ u, R* __restrict__ U) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= M) return;
  const int64_t m = perm[j];
  const int32_t h = home[j];
  if (h < 0) {
    U[m] = R(0);
    U[M + m] = R(0);
    U[2 * M + m] = R(0);
    return;
  }
  int i[3];
  decode_home(h, D, i);
  int xs[3], ys[3], zs[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    xs[a] = wrap(i[0] + a - 1, D.n[0], D.periodic[0]);
    ys[a] = wrap(i[1] + a - 1, D.n[1], D.periodic[1]);
    zs[a] = wrap(i[2] + a - 1, D.n[2], D.periodic[2]);
  }
  const int64_t N = (int64_t)D.n[0] * D.n[1] * D.n[2];
  R s0 = R(0), s1 = R(0), s2 = R(0);
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int64_t row = ((int64_t)zs[c] * D.n[1] + ys[b]) * D.n[0];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const R p = phi[(9 * c + 3 * b + a) * cap + j];
        const int64_t o = row + xs[a];
        s0 += p * load_field<R, FT>(u + o);
        s1 += p * load_field<R, FT>(u + N + o);
        s2 += p * load_field<R, FT>(u + 2 * N + o);
      }
    }
  U[m] = s0;
  U[M + m] = s1;
  U[2 * M + m] = s2;
}

// U_l = sum_k phi_k^l u_k (text after Eq. 6), single precision, with F also the
// direct forcing F = (V_b - U) / dt: a block lists the runs of
// kChunkPer * kInterpThreads stored markers and a thread per run gathers the
// run's velocities through the cache hierarchy.  Dropped markers get U = F = 0.
// For spreading tiles of more than 2^9 or fewer than 2^8 cells, whose staged rows
// leave too few blocks per SM or hold too few markers (k_tile_pass): it does not
// depend on the tile's shape.  4 M markers in 512^3 take 164 to 174 us at 64
// registers (79 us for the bytes), staged 246 to 288 in tiles of 2^10 and 2^11
// cells and 194 in tiles of 2^6.
template <typename FT, bool FORCE>
__global__ void __launch_bounds__(kInterpThreads, 8) k_interp_runs(Dims D, const float* __restrict__ phi,
                                                                   const int32_t* __restrict__ home,
                                                                   const int32_t* __restrict__ perm, int64_t M,
                                                                   int64_t cap, InterpOut<float, FT> io) {
  constexpr int NT = kInterpThreads, CHUNK = kChunkPer * NT;
  __shared__ int runs[CHUNK];
  __shared__ int s_cnt[kChunkPer * (NT / 32)];
  const unsigned j0 = blockIdx.x * (unsigned)CHUNK, end = (unsigned)min((int64_t)j0 + CHUNK, M);
  const int n = list_runs<NT>(home, j0, end, j0, runs, s_cnt, [](unsigned, int) {}, [] {}, [] {});
  for (int t = threadIdx.x; t < n; t += NT) {
    const Run r(runs[t]);
    const int64_t g = j0 + (r.first & ~3);
    const int in = r.first & 3;
    const int32_t h = home[j0 + r.first];
    if (h < 0) {
      for (int k = in; k < in + r.len; ++k) io.store_zero(perm[g + k], M);
      continue;
    }
    int i[3];
    decode_home(h, D, i);
    float4 U[3];
    if ((cap & 3) == 0)
      gather_run<FT, true>(D, i, io.u, phi + g, cap, M - g, U);
    else
      gather_run<FT, false>(D, i, io.u, phi + g, cap, M - g, U);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (k >= in && k < in + r.len) {
        const int64_t m = perm[g + k];
        if constexpr (FORCE) {
          io.store(m, M, at(U[0], k), at(U[1], k), at(U[2], k));
        } else {
#pragma unroll
          for (int q = 0; q < 3; ++q) io.U[q * M + m] = at(U[q], k);
        }
      }
  }
}

// f_k += sum_l c_l phi_k^l F_l (text after Eq. 7), single precision.
// Persistent blocks walk the list of non-empty spreading tiles, taking up to
// 512 markers of a tile at a time: a thread per marker forms c_l F_l and the
// chunk's runs are listed, then a thread per run adds its 27 x 3 sums into the
// shared-memory accumulator with native 32-bit integer atomics in fixed point
// (chunk_scale), and the rows the runs touched are added to f and reset.  A
// chunk with non-finite forces is added to f directly.
// On 32 M markers in 1024^3 it takes 1.72 ms and on 4 M in 512^3 257 us, against
// 0.70 ms and 87 us for the bytes: issue (39 % active), the shared-memory pipe
// and the waits between a tile's phases share the rest, at 28 warps per SM.  A
// thread per marker issuing its own 81 atomics, chunks of 128 markers, took
// 2.06 ms and 318 us.
template <typename FT, bool VEC, int LX, int LY = 0, int LZ = 0>
__global__ void __launch_bounds__(kSpreadThreads, 8) k_spread(Dims D, Tiles tl, const float* __restrict__ phi,
                                                           const float* __restrict__ cl,
                                                           const int32_t* __restrict__ home,
                                                           const int32_t* __restrict__ perm,
                                                           const int32_t* __restrict__ items,
                                                           const int32_t* __restrict__ n_items_p,
                                                           const int32_t* __restrict__ offsets,
                                                           const int32_t* __restrict__ counts, int64_t M, int64_t cap,
                                                           int max_bits, const float* __restrict__ F,
                                                           FT* __restrict__ f) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int NT = kSpreadThreads, CHUNK = kChunkPer * NT;
  const int ly = LY ? LY : tl.l[1], lz = LZ ? LZ : tl.l[2];   // compile-time when specialised
  const AccShape A(LX, ly, lz);
  const SpreadSmem L(LX, ly, lz, run_smem_bytes(NT));
  int* acc = reinterpret_cast<int*>(smem_raw);
  float* sv = reinterpret_cast<float*>(smem_raw + L.chunk);
  int* runs = reinterpret_cast<int*>(sv + 3 * CHUNK);
  unsigned char* tags = smem_raw + L.tags;
  __shared__ float s_red[3 * (NT / 32)];
  __shared__ int s_cnt[kChunkPer * (NT / 32)];
  __shared__ Scale s_scale;
  const int tid = threadIdx.x;
  const int n_items = *n_items_p;
  const bool quad = (cap & 3) == 0;
  unsigned char tag = 0;
  for (int e = tid; e < 3 * A.ACC; e += NT) acc[e] = 0;
  for (int r = tid; r < A.AY * A.AZ; r += NT) tags[r] = 0;

  // Every block takes tiles of about equal total weight, neighbours in the list;
  // with fewer tiles than blocks, a share of one.
  if (n_items == 0) return;
  __shared__ int s_range[2];
  const int parts = min((int)gridDim.x / n_items, 8);
  if (parts > 0) {
    if (tid < 2) s_range[tid] = min(n_items, (int)blockIdx.x / parts + tid);
  } else if (tid < 64) {
    const int64_t all = offsets[tl.nbins - 1] + (int64_t)kTileWeight * n_items;
    const int64_t g = blockIdx.x + (tid >> 5);
    const int at = g == gridDim.x ? n_items : tile_at(items, offsets, n_items, all * g / gridDim.x);
    if ((tid & 31) == 0) s_range[tid >> 5] = at;
  }
  __syncthreads();
  int it = s_range[0];
  const int last = s_range[1];
  int b = it < last ? items[it] : 0;
  unsigned start = offsets[b], end = start + counts[b];
  if (parts > 1) tile_part(blockIdx.x % parts, parts, start, end);
  for (; it < last; ++it) {
    if (it + 1 < last) b = items[it + 1];       // the next tile's header, while this one is worked on
    unsigned next_start = start, next_end = end;
    for (unsigned j0 = start & ~3u; j0 < end; j0 += CHUNK) {
      tag = tag == 255 ? 1 : tag + 1;
      float sum[3] = {0.f, 0.f, 0.f};
      const int n = list_runs<NT>(
          home, start, end, j0, runs, s_cnt,
          [&](unsigned j, int at) {
            const int64_t m = perm[j];
            const float c = cl[j];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              const float v = c * F[q * M + m];
              sv[q * CHUNK + at] = v;
              sum[q] += fabsf(v);
            }
          },
          [&] { publish_sums<NT>(sum, s_red); },
          [&] {
            if (tid < 3) chunk_scale<NT>(s_red, tid, min(scale_bits(min(end, j0 + CHUNK) - max(start, j0)), max_bits), &s_scale);
          });
      if (it + 1 < last) {
        next_start = offsets[b];
        next_end = next_start + counts[b];
      }
      const ChunkScale kind = chunk_kind(s_scale);
      if (kind == kZero) continue;
      int o[3];
      decode_home(home[start], D, o);
      o[0] &= ~((1 << LX) - 1);
      o[1] &= ~((1 << ly) - 1);
      o[2] &= ~((1 << lz) - 1);
      if (kind == kFixed) {
        if (quad)
          add_runs<FT, true, NT, CHUNK>(D, o, n, runs, home, sv, j0, phi, cap, M, s_scale, acc, A.AX, A.PS, A.ACC,
                                        A.AY, tags, tag, f);
        else
          add_runs<FT, false, NT, CHUNK>(D, o, n, runs, home, sv, j0, phi, cap, M, s_scale, acc, A.AX, A.PS,
                                         A.ACC, A.AY, tags, tag, f);
        if (quad && it + 1 < last && j0 + CHUNK >= end)
          prefetch_tile(phi, home, perm, cl, cap, next_start, next_end);
        __syncthreads();
        flush_rows<FT, VEC, LX, NT>(D, o, A, acc, tags, tag, s_scale.unit, f);
      } else {
        for (int t = tid; t < n; t += NT) {
          const Run r(runs[t]);
          int i[3];
          decode_home(home[j0 + r.first], D, i);
          for (int k = 0; k < 81; ++k)
            add_direct<FT>(D, i, r, k / 3, k % 3, phi, cap, (int64_t)j0 + r.first, sv, CHUNK, f);
        }
        __syncthreads();
      }
    }
    start = next_start;
    end = next_end;
  }
}

// Double-precision spreading (the small double-precision workloads): one
// thread per stored marker adds its 27 x 3 terms c_l phi_k F_l straight into
// f with native global double reductions.  Shared-memory accumulation, as in
// single precision, needs double shared atomics, which are compare-and-swap
// loops on this GPU and serialise badly where markers crowd few cells.
__global__ void __launch_bounds__(kBlock) k_spread_f64(Dims D, const double* __restrict__ phi,
                                                       const double* __restrict__ cl, const int32_t* __restrict__ home,
                                                       const int32_t* __restrict__ perm, int64_t M, int64_t cap,
                                                       const double* __restrict__ F, double* __restrict__ f) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= M) return;
  const int32_t h = home[j];
  if (h < 0) return;
  int i[3];
  decode_home(h, D, i);
  const int64_t m = perm[j];
  const double c = cl[j];
  const double v0 = c * F[m], v1 = c * F[M + m], v2 = c * F[2 * M + m];
  const int64_t N = (int64_t)D.n[0] * D.n[1] * D.n[2];
#pragma unroll
  for (int cz = 0; cz < 3; ++cz) {
    const int gz = wrap(i[2] + cz - 1, D.n[2], D.periodic[2]);
#pragma unroll
    for (int cy = 0; cy < 3; ++cy) {
      const int64_t row = ((int64_t)gz * D.n[1] + wrap(i[1] + cy - 1, D.n[1], D.periodic[1])) * D.n[0];
#pragma unroll
      for (int cx = 0; cx < 3; ++cx) {
        const double p = phi[(9 * cz + 3 * cy + cx) * cap + j];
        const int64_t o = row + wrap(i[0] + cx - 1, D.n[0], D.periodic[0]);
        atomicAdd(f + o, p * v0);
        atomicAdd(f + N + o, p * v1);
        atomicAdd(f + 2 * N + o, p * v2);
      }
    }
  }
}

static size_t spread_smem_bytes(const mls_ctx* ctx) {
  if (ctx->opt.real == MLS_F64) return 0;   // the double-precision spread uses no shared memory
  return (size_t)SpreadSmem(ctx->tiles.l[0], ctx->tiles.l[1], ctx->tiles.l[2], run_smem_bytes(kSpreadThreads)).total;
}

// The limit on the tile shape: three components of 4 bytes for the tile and its
// halo, with 4 columns on either side when the x extent is a multiple of 4 (1
// otherwise) and 9 bytes per row.  What the kernels need beside any tile that
// passes (at most a tenth of 200 KB for wider rows, 8 KB for a chunk) fits a
// block.
bool spread_tile_fits(const mls_ctx* ctx) {
  if (ctx->opt.real == MLS_F64) return true;
  const int* l = ctx->tiles.l;
  const int ay = (1 << l[1]) + 2, az = (1 << l[2]) + 2, ax = (1 << l[0]) + (spread_vec(ctx) ? 8 : 2);
  return (((12 * az * (ay * ax + 4) + 15) & ~15) + 9 * ay * az + 15) / 16 * 16 <= 200 * 1024 + 256;
}

template <typename K>
static cudaError_t configure_kernel(mls_ctx* ctx, K kernel, int smem) {
  cudaError_t e = raise_smem_limit((const void*)kernel, smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0, sms = 0, dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kSpreadThreads, smem);
  if (e != cudaSuccess) return e;
  ctx->spread_grid = (per_sm > 0 ? per_sm : 1) * sms;
  ctx->spread_threads = kSpreadThreads;
  return cudaSuccess;
}

template <typename FT, bool VEC>
static const void* spread_kernel(int lx, int ly, int lz) {
  // Tile shapes the tile-shape tuner tries get compile-time accumulator strides.
  if (VEC) {
    if (lx == 3 && ly == 3 && lz == 3) return (const void*)k_spread<FT, VEC, 3, 3, 3>;
    if (lx == 3 && ly == 3 && lz == 2) return (const void*)k_spread<FT, VEC, 3, 3, 2>;
    if (lx == 4 && ly == 3 && lz == 3) return (const void*)k_spread<FT, VEC, 4, 3, 3>;
    if (lx == 4 && ly == 4 && lz == 3) return (const void*)k_spread<FT, VEC, 4, 4, 3>;
    if (lx == 4 && ly == 4 && lz == 2) return (const void*)k_spread<FT, VEC, 4, 4, 2>;
    if (lx == 5 && ly == 3 && lz == 3) return (const void*)k_spread<FT, VEC, 5, 3, 3>;
  }
  switch (lx) {
    case 1: return VEC ? nullptr : (const void*)k_spread<FT, false, 1>;
    case 2: return (const void*)k_spread<FT, VEC, 2>;
    case 3: return (const void*)k_spread<FT, VEC, 3>;
    case 4: return (const void*)k_spread<FT, VEC, 4>;
    default: return (const void*)k_spread<FT, VEC, 5>;
  }
}

cudaError_t spread_configure(mls_ctx* ctx) {
  const int smem = (int)spread_smem_bytes(ctx);
  const int lx = ctx->tiles.l[0], ly = ctx->tiles.l[1], lz = ctx->tiles.l[2];
  if (ctx->opt.real == MLS_F64) return cudaSuccess;
  const bool bf = ctx->opt.field == MLS_BF16;
  if (spread_vec(ctx)) {
    // The scalar variant also runs when f is not aligned for the vector reductions (same layout size or smaller).
    cudaError_t e = configure_kernel(ctx, bf ? spread_kernel<__nv_bfloat16, false>(lx, ly, lz) : spread_kernel<float, false>(lx, ly, lz),
                                     smem);
    if (e != cudaSuccess) return e;
    return configure_kernel(ctx, bf ? spread_kernel<__nv_bfloat16, true>(lx, ly, lz) : spread_kernel<float, true>(lx, ly, lz), smem);
  }
  return configure_kernel(ctx, bf ? spread_kernel<__nv_bfloat16, false>(lx, ly, lz) : spread_kernel<float, false>(lx, ly, lz), smem);
}

template <typename FT>
static void launch_interp_runs(const mls_ctx* ctx, const mls_transfer* T, const void* u, void* U, const void* Vb,
                               double dt, void* F, cudaStream_t s) {
  constexpr int64_t chunk = kChunkPer * kInterpThreads;
  const int64_t N = (int64_t)ctx->n[0] * ctx->n[1] * ctx->n[2];
  const InterpOut<float, FT> io{(const FT*)u, (float*)U, N, (const float*)Vb, F ? (float)(1.0 / dt) : 0.f, (float*)F};
  auto kern = F ? k_interp_runs<FT, true> : k_interp_runs<FT, false>;
  kern<<<(unsigned)((T->M + chunk - 1) / chunk), kInterpThreads, 0, s>>>(dims_of(ctx), (const float*)T->phi, T->home,
                                                                        T->perm, T->M, T->cap, io);
}

cudaError_t launch_interp(const mls_ctx* ctx, const mls_transfer* T, const void* u, void* U, cudaStream_t s,
                          const void* Vb, double dt, void* F) {
  if (T->M == 0) return cudaSuccess;
  const unsigned nt = block_threads(T->M, kBlock);
  if (ctx->opt.real == MLS_F64)
    k_interp<double, double><<<blocks_for(T->M, nt), nt, 0, s>>>(
        dims_of(ctx), (const double*)T->phi, T->home, T->perm, T->M, T->cap, (const double*)u, (double*)U);
  else if (ctx->tile_grid[0] > 0)
    return launch_tiles(ctx, T, u, Vb, dt, U, F, nullptr, s);
  else if (ctx->opt.field == MLS_BF16)
    launch_interp_runs<__nv_bfloat16>(ctx, T, u, U, Vb, dt, F, s);
  else
    launch_interp_runs<float>(ctx, T, u, U, Vb, dt, F, s);
  return cudaGetLastError();
}

template <typename FT, bool VEC>
static cudaError_t launch_spread_one(const mls_ctx* ctx, const mls_transfer* T, const void* F, void* f,
                                     cudaStream_t s) {
  Dims D = dims_of(ctx);
  Tiles tl = ctx->tiles;
  const float* phi = (const float*)T->phi;
  const float* c = (const float*)T->c;
  int64_t M = T->M, cap = T->cap;
  // Accumulating |phi| < 1/2 only (two scale bits) sends the node next to the
  // marker past the accumulator where phi exceeds that: with the quadratic basis
  // (0.61 at a cell centre, eps = 1), and with the linear one at
  // (1 + 2 exp(-1/eps^2))^-3 > 1/2, eps < 0.7.  There one bit is the most.
  int max_bits = ctx->opt.basis == 4 && ctx->opt.eps >= 0.75 ? 2 : 1;
  void* args[] = {&D, &tl, (void*)&phi, (void*)&c, (void*)&T->home, (void*)&T->perm, (void*)&T->items,
                  (void*)&T->n_items, (void*)&T->offsets, (void*)&T->counts, &M, &cap, &max_bits, (void*)&F, &f};
  return cudaLaunchKernel(spread_kernel<FT, VEC>(tl.l[0], tl.l[1], tl.l[2]), dim3(ctx->spread_grid), dim3(ctx->spread_threads), args,
                          spread_smem_bytes(ctx), s);
}

cudaError_t launch_spread(const mls_ctx* ctx, const mls_transfer* T, const void* F, void* f, cudaStream_t s) {
  if (T->M == 0) return cudaSuccess;
  const unsigned nt = block_threads(T->M, kBlock);
  if (ctx->opt.real == MLS_F64)
    k_spread_f64<<<blocks_for(T->M, nt), nt, 0, s>>>(
        dims_of(ctx), (const double*)T->phi, (const double*)T->c, T->home, T->perm, T->M, T->cap,
        (const double*)F, (double*)f);
  else if (ctx->opt.field == MLS_BF16)
    return spread_vec_aligned(ctx, f) ? launch_spread_one<__nv_bfloat16, true>(ctx, T, F, f, s)
                                      : launch_spread_one<__nv_bfloat16, false>(ctx, T, F, f, s);
  else if (spread_vec_aligned(ctx, f))
    return launch_spread_one<float, true>(ctx, T, F, f, s);
  else return launch_spread_one<float, false>(ctx, T, F, f, s);
  return cudaGetLastError();
}

}  // namespace mls
