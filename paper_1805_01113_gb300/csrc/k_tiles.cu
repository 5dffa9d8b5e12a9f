// Interpolation and direct forcing by spreading tiles, single precision: a tile's
// field rows are staged in shared memory and a thread per marker gathers from
// there; direct forcing then adds the marker's terms to a second brick and
// flushes it to f in the same pass.
#include "spread_runs.cuh"

namespace mls {

// Copies of W = 4, 2 or 1 cells into a float brick; bfloat16 through registers.
template <int W>
__device__ __forceinline__ void stage(float* dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (W == 4)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
  else if constexpr (W == 2)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ float2 widen(unsigned two) {
  return make_float2(__uint_as_float(two << 16), __uint_as_float(two & 0xffff0000u));
}
template <int W>
__device__ __forceinline__ void stage(float* dst, const __nv_bfloat16* src) {
  if constexpr (W == 4) {
    const uint2 w = __ldg(reinterpret_cast<const uint2*>(src));
    const float2 lo = widen(w.x), hi = widen(w.y);
    *reinterpret_cast<float4*>(dst) = make_float4(lo.x, lo.y, hi.x, hi.y);
  } else if constexpr (W == 2) {
    *reinterpret_cast<float2*>(dst) = widen(__ldg(reinterpret_cast<const unsigned*>(src)));
  } else {
    *dst = to_f<__nv_bfloat16>(__ldg(src));
  }
}

// The rows with the tag, of all three components, from the field into the brick
// (AccShape; the work is split as in flush_rows, in groups of W cells; pairs take
// the halo cells with them).  Cells and rows outside a walled axis, or beyond one
// period, belong to no support and are left out: a row can carry an equal tag of
// 255 tiles ago.
template <typename FT, int W, int LX, int NT>
__device__ __forceinline__ void stage_rows(const Dims& D, const int o[3], const AccShape& A, float* brick,
                                           const unsigned char* tags, unsigned char tag, const FT* __restrict__ u) {
  constexpr int TX = 1 << LX;
  constexpr int GROUPS = W == 4 ? TX / 4 : W == 2 ? TX / 2 + 2 : 0, CELLS = W == 4 ? 2 : W == 2 ? 0 : TX + 2;
  const int rows = A.AY * A.AZ;
  const int64_t N = (int64_t)D.n[0] * D.n[1] * D.n[2];
  for (int e = threadIdx.x; e < (GROUPS + CELLS) * rows; e += NT) {
    const bool group = CELLS == 0 || (W > 1 && e < GROUPS * rows);
    const int s = group ? e : e - GROUPS * rows;
    const int row = group ? s / (GROUPS ? GROUPS : 1) : s / (CELLS ? CELLS : 1), q = s - row * (group ? GROUPS : CELLS);
    if (tags[row] != tag) continue;
    const int ey = row % A.AY, ez = row / A.AY;
    const int x = W == 2 ? 2 * q - 2 : group ? 4 * q : W == 4 ? (q == 0 ? -1 : TX) : q - 1;
    int gx = o[0] + x;
    if (gx < 0 || gx >= D.n[0]) {
      if (!D.periodic[0]) continue;
      gx = gx < 0 ? gx + D.n[0] : gx - D.n[0];
      if (gx < 0 || gx >= D.n[0]) continue;
    }
    const int gy = wrap(o[1] - 1 + ey, D.n[1], D.periodic[1]), gz = wrap(o[2] - 1 + ez, D.n[2], D.periodic[2]);
    if (gy >= D.n[1] || gz >= D.n[2]) continue;
    float* a = brick + AccShape::kFront + ez * A.PS + ey * A.AX + x;
    const FT* ur = u + (int64_t)((gz * D.n[1] + gy) * D.n[0] + gx);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (group)
        stage<W>(a + c * A.ACC, ur + c * N);
      else
        stage<1>(a + c * A.ACC, ur + c * N);
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Shared memory: the field brick, the accumulator when the pass spreads, a tag
// per row of either.
static int tile_pass_smem(int lx, int ly, int lz, bool spread) {
  const AccShape A(lx, ly, lz);
  return ((spread ? 6 : 3) * A.ACC * 4 + A.AY * A.AZ + 15) & ~15;
}

// One pass over the non-empty tiles: U_l = sum_k phi_k^l u_k and, when asked for,
// F_l = (V_b,l - U_l) / dt; with SPREAD also f_k += sum_l c_l phi_k^l F_l, by
// chunks of NT markers in fixed point as k_spread does.  Markers without support
// get U = F = 0.
// Tiles go to the blocks in turn.  There are ten times as many blocks as fit the
// device, or one per 1 024 markers, so that a crowded tile delays only what its
// block has left, but no more than one per 48 (64) markers; where tiles are fewer
// than blocks, a crowded tile is shared by up to eight.  (4 M markers in 512^3: 210
// with the blocks that fit, 187 with twice, 161 with ten times as many.)
// Bound by the shared-memory pipe (81 loads a marker and, with SPREAD, as many
// atomics and conversions) and a tile's chain of phases.  In microseconds,
// against the gather through L1 by runs of markers (k_interp_runs), and against
// that gather and the spread: 55 040 markers in 64^3 8.3 (12.3), forcing 15.1
// (26.9); 1.04 M in 200^3 46 (49), 110 (129); 2.72 M in 256^3 97 (126), 262 (306);
// 4 M in a 512^3 channel 161 (174), 407 (509), of which the bytes take 79 and 166;
// 32 M in 1024^3 1 250 (1 235), 3 010 (3 390).  By runs the gathers of a warp fall
// in few L1 sets where rows are a multiple of 128 bytes; they are faster by up to
// 15 % on some boxes between (280 000 markers in 200^3: 17.5, here 20.2).  Runs
// gathered from the staged rows took 278 in the channel: listing them costs more
// than it saves.
// Blocks have 128 threads, and 256 where they spread tiles of 2^9 cells or more,
// which hold enough markers for that.
constexpr int kTileWaves = 10;   // blocks per resident block

template <typename FT, int W, bool SPREAD, int NT, int LX, int LY = 0, int LZ = 0>
__global__ void __launch_bounds__(NT, (SPREAD ? 1024 : 1536) / NT) k_tile_pass(Dims D, Tiles tl, const float* __restrict__ phi,
                                                              const float* __restrict__ cl,
                                                              const int32_t* __restrict__ home,
                                                              const int32_t* __restrict__ perm,
                                                              const int32_t* __restrict__ items,
                                                              const int32_t* __restrict__ n_items_p,
                                                              const int32_t* __restrict__ offsets,
                                                              const int32_t* __restrict__ counts, int64_t M,
                                                              int64_t cap, int resident,
                                                              InterpOut<float, FT> io, FT* __restrict__ f) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int ly = LY ? LY : tl.l[1], lz = LZ ? LZ : tl.l[2];
  const AccShape A(LX, ly, lz);
  float* brick = reinterpret_cast<float*>(smem_raw);
  int* acc = reinterpret_cast<int*>(brick + 3 * A.ACC);
  unsigned char* tags = reinterpret_cast<unsigned char*>(acc + (SPREAD ? 3 * A.ACC : 0));
  __shared__ float s_red[3 * (NT / 32)];
  __shared__ Scale s_scale;
  const int tid = threadIdx.x;
  const int n_items = *n_items_p;
  const int64_t d0 = offsets[tl.nbins - 1];
  for (int64_t j = d0 + (int64_t)blockIdx.x * NT + tid; j < M; j += (int64_t)gridDim.x * NT) io.store_zero(perm[j], M);
  if (n_items == 0) return;
  for (int r = tid; r < A.AY * A.AZ; r += NT) tags[r] = 0;
  if constexpr (SPREAD)
    for (int e = tid; e < 3 * A.ACC; e += NT) acc[e] = 0;
  __syncthreads();
  // The first n_items blocks take the tiles' first shares, so that blocks without
  // a share come last.  A share has 128 markers or more, and 512 where the tiles
  // fill the device.
  const int least = n_items < resident ? 128 : 512;
  const int parts = max(1, min((int)gridDim.x / n_items, 8)), part = parts > 1 ? (int)blockIdx.x / n_items : 0;
  if (part >= parts) return;
  const int step = parts > 1 ? n_items : (int)gridDim.x;
  unsigned char tag = 0;
  for (int it = (int)blockIdx.x - part * n_items; it < n_items; it += step) {
    const int b = items[it];
    unsigned start = offsets[b], end = start + counts[b];
    if (parts > 1) {
      const int sharing = min(parts, max(1, (int)(end - start) / least));
      if (part >= sharing) break;
      tile_part(part, sharing, start, end);
      if (start >= end) break;
    }
    tag = tag == 255 ? 1 : tag + 1;
    int o[3];
    decode_home(home[start], D, o);
    o[0] &= ~((1 << LX) - 1);
    o[1] &= ~((1 << ly) - 1);
    o[2] &= ~((1 << lz) - 1);
    for (unsigned j = start + tid; j < end; j += NT) {
      int i[3];
      decode_home(home[j], D, i);
      unsigned char* t = tags + (i[2] - o[2]) * A.AY + i[1] - o[1];
#pragma unroll
      for (int cz = 0; cz < 3; ++cz)
#pragma unroll
        for (int cy = 0; cy < 3; ++cy) t[cz * A.AY + cy] = tag;
    }
    __syncthreads();
    stage_rows<FT, W, LX, NT>(D, o, A, brick, tags, tag, io.u);
    __syncthreads();
    for (unsigned j0 = start; j0 < end; j0 += NT) {
      const unsigned j = j0 + tid;
      const bool act = j < end;
      float p[27], v[3] = {0.f, 0.f, 0.f};
      int at = 0, i[3] = {0, 0, 0};
      if (act) {
        const int64_t m = perm[j];
#pragma unroll
        for (int k = 0; k < 27; ++k) p[k] = phi[k * cap + j];
        decode_home(home[j], D, i);
        at = AccShape::kFront + (i[2] - o[2]) * A.PS + (i[1] - o[1]) * A.AX + (i[0] - o[0]) - 1;
        float U[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < 27; ++k)
#pragma unroll
          for (int q = 0; q < 3; ++q) U[q] += p[k] * brick[at + k / 9 * A.PS + k / 3 % 3 * A.AX + k % 3 + q * A.ACC];
        if constexpr (SPREAD) {
          const float c = cl[j];
#pragma unroll
          for (int q = 0; q < 3; ++q) v[q] = c * ((io.Vb[q * M + m] - U[q]) * io.inv_dt);
        }
        io.store(m, M, U[0], U[1], U[2]);
      }
      if constexpr (SPREAD) {
        float sum[3] = {fabsf(v[0]), fabsf(v[1]), fabsf(v[2])};
        publish_sums<NT>(sum, s_red);
        __syncthreads();
        const int bits = scale_bits(min(end - j0, (unsigned)NT));
        if (tid < 3) chunk_scale<NT>(s_red, tid, bits, &s_scale);
        __syncthreads();
        const ChunkScale kind = chunk_kind(s_scale);
        if (kind == kZero) continue;
        if (act) {
          // Fixed point where |phi| is below the limit (NaN is not), the rest to f directly.
          float most = 0.f;
#pragma unroll
          for (int k = 0; k < 27; k += 3) most = max_abs(max_abs(most, p[k], p[k + 1]), p[k + 2], 0.f);
          if (kind == kFixed && most < s_scale.limit) {
            // Lanes of one home cell would add to one word in the same instruction:
            // every third lane starts with another component, and every third of
            // those with another column.
            const int c0 = tid % 3, c1 = c0 == 2 ? 0 : c0 + 1, c2 = c0 == 0 ? 2 : c0 - 1;
            const float q0 = (c0 == 0 ? v[0] : c0 == 1 ? v[1] : v[2]) * s_scale.inv[c0];
            const float q1 = (c1 == 0 ? v[0] : c1 == 1 ? v[1] : v[2]) * s_scale.inv[c1];
            const float q2 = (c2 == 0 ? v[0] : c2 == 1 ? v[1] : v[2]) * s_scale.inv[c2];
            int *a0 = acc + at + c0 * A.ACC, *a1 = acc + at + c1 * A.ACC, *a2 = acc + at + c2 * A.ACC;
            const int x0 = tid / 3 % 3, x1 = x0 == 2 ? 0 : x0 + 1, x2 = x0 == 0 ? 2 : x0 - 1;
#pragma unroll
            for (int r = 0; r < 9; ++r) {
              const float e0 = p[3 * r], e1 = p[3 * r + 1], e2 = p[3 * r + 2];
              const float t[3] = {x0 == 0 ? e0 : x0 == 1 ? e1 : e2, x0 == 0 ? e1 : x0 == 1 ? e2 : e0,
                                  x0 == 0 ? e2 : x0 == 1 ? e0 : e1};
              const int o = r / 3 * A.PS + r % 3 * A.AX;
#pragma unroll
              for (int x = 0; x < 3; ++x) {
                const int w = o + (x == 0 ? x0 : x == 1 ? x1 : x2);
                atomicAdd(a0 + w, __float2int_rn(t[x] * q0));
                atomicAdd(a1 + w, __float2int_rn(t[x] * q1));
                atomicAdd(a2 + w, __float2int_rn(t[x] * q2));
              }
            }
          } else {
            const int64_t N = io.N;
#pragma unroll
            for (int k = 0; k < 27; ++k) {
              const int64_t cell = ((int64_t)wrap(i[2] + k / 9 - 1, D.n[2], D.periodic[2]) * D.n[1] +
                                    wrap(i[1] + k / 3 % 3 - 1, D.n[1], D.periodic[1])) * D.n[0] +
                                   wrap(i[0] + k % 3 - 1, D.n[0], D.periodic[0]);
#pragma unroll
              for (int q = 0; q < 3; ++q) add_field<float, FT>(f + q * N + cell, p[k] * v[q]);
            }
          }
        }
        __syncthreads();
        if (kind == kFixed) flush_rows<FT, W == 4, LX, NT>(D, o, A, acc, tags, tag, s_scale.unit, f);
      }
    }
    if constexpr (SPREAD) __syncthreads();   // flushed by the tile's tags before the next tile sets its own
  }
}

template <typename FT, int W, bool SPREAD, int NT>
static const void* tile_kernel_of(const int l[3]) {
  if (l[0] == 3 && l[1] == 3 && l[2] == 3) return (const void*)k_tile_pass<FT, W, SPREAD, NT, 3, 3, 3>;
  if (l[0] == 3 && l[1] == 3 && l[2] == 2) return (const void*)k_tile_pass<FT, W, SPREAD, NT, 3, 3, 2>;
  switch (l[0]) {
    case 1: return (const void*)k_tile_pass<FT, W == 4 ? 2 : W, SPREAD, NT, 1>;
    case 2: return (const void*)k_tile_pass<FT, W, SPREAD, NT, 2>;
    case 3: return (const void*)k_tile_pass<FT, W, SPREAD, NT, 3>;
    case 4: return (const void*)k_tile_pass<FT, W, SPREAD, NT, 4>;
    default: return (const void*)k_tile_pass<FT, W, SPREAD, NT, 5>;
  }
}

static int tile_threads(const int l[3], bool spread) { return spread && l[0] + l[1] + l[2] >= 9 ? 256 : 128; }

template <typename FT, int W, bool SPREAD>
static const void* tile_kernel(const int l[3]) {
  if constexpr (SPREAD)
    if (tile_threads(l, true) == 256) return tile_kernel_of<FT, W, true, 256>(l);
  return tile_kernel_of<FT, W, SPREAD, 128>(l);
}

// One pass for direct forcing exists for float fields only (launch_direct_forcing).
static const void* tile_kernel(const mls_ctx* ctx, int width, bool spread) {
  const int* l = ctx->tiles.l;
  if (ctx->opt.field == MLS_BF16)
    return width == 4   ? tile_kernel<__nv_bfloat16, 4, false>(l)
           : width == 2 ? tile_kernel<__nv_bfloat16, 2, false>(l)
                        : tile_kernel<__nv_bfloat16, 1, false>(l);
  if (spread)
    return width == 4 ? tile_kernel<float, 4, true>(l) : width == 2 ? tile_kernel<float, 2, true>(l)
                                                                    : tile_kernel<float, 1, true>(l);
  return width == 4 ? tile_kernel<float, 4, false>(l) : width == 2 ? tile_kernel<float, 2, false>(l)
                                                                   : tile_kernel<float, 1, false>(l);
}

// Cells per copy: groups that start on their own boundary in every row.
static int copy_width(const mls_ctx* ctx, const void* u) {
  const uintptr_t cell = ctx->opt.field == MLS_F32 ? 4 : 2, a = reinterpret_cast<uintptr_t>(u);
  const int w = ctx->n[0] % 4 == 0 && a % (4 * cell) == 0 ? 4 : ctx->n[0] % 2 == 0 && a % (2 * cell) == 0 ? 2 : 1;
  return w == 4 && ctx->tiles.l[0] < 2 ? 2 : w;
}

// Tiles of 2^8 and 2^9 cells, and for direct forcing smaller ones too.  Larger ones
// leave few blocks per SM: 2.56 M markers in 512^3 take 125 and 128 us in tiles of
// (3,3,3) and (3,3,2), 202 in (4,3,3), 207 in (4,4,3) and 223 in (5,3,3), by runs
// 134 to 156 in all; direct forcing 348 and 305, 398, 490 and 510, in two kernels
// 387 and 416, 398, 437 and 432.  In (3,2,2) 155 (150), direct forcing 369 (483).
cudaError_t tiles_configure(mls_ctx* ctx) {
  ctx->tile_grid[0] = ctx->tile_grid[1] = 0;
  const int cells = ctx->tiles.l[0] + ctx->tiles.l[1] + ctx->tiles.l[2];
  if (ctx->opt.real == MLS_F64 || cells > 9) return cudaSuccess;
  cudaError_t e;
  int sms = 0;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device)) != cudaSuccess) return e;
  for (int spread = 0; spread < 2; ++spread) {
    const int smem = tile_pass_smem(ctx->tiles.l[0], ctx->tiles.l[1], ctx->tiles.l[2], spread != 0);
    if (!spread && cells < 8) continue;
    if (spread && ctx->opt.field == MLS_BF16) continue;
    int least = 64;
    for (int width = 1; width <= 4; width *= 2) {
      const void* k = tile_kernel(ctx, width, spread != 0);
      int per_sm = 0;
      if ((e = raise_smem_limit(k, smem)) != cudaSuccess ||
          (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
               &per_sm, k, tile_threads(ctx->tiles.l, spread != 0), smem)) != cudaSuccess)
        return e;
      least = std::min(least, per_sm);
    }
    ctx->tile_grid[spread] = std::max(least, 1) * sms * kTileWaves;
  }
  return cudaSuccess;
}

template <typename FT>
static cudaError_t launch_tiles_of(const mls_ctx* ctx, const mls_transfer* T, const void* u, const void* Vb, double dt,
                                   void* U, void* F, void* f, cudaStream_t s) {
  Dims D = dims_of(ctx);
  Tiles tl = ctx->tiles;
  const float* phi = (const float*)T->phi;
  const float* c = (const float*)T->c;
  int64_t M = T->M, cap = T->cap;
  const int64_t N = (int64_t)ctx->n[0] * ctx->n[1] * ctx->n[2];
  InterpOut<float, FT> io{(const FT*)u, (float*)U, N, (const float*)Vb, F ? (float)(1.0 / dt) : 0.f, (float*)F};
  int resident = ctx->tile_grid[f ? 1 : 0] / kTileWaves;
  void* args[] = {&D, &tl, (void*)&phi, (void*)&c, (void*)&T->home, (void*)&T->perm, (void*)&T->items,
                  (void*)&T->n_items, (void*)&T->offsets, (void*)&T->counts, &M, &cap, &resident, &io, &f};
  const int wu = copy_width(ctx, u), width = f && wu == 4 && !spread_vec_aligned(ctx, f) ? 2 : wu;
  const int64_t most = std::max<int64_t>(ctx->tile_grid[f ? 1 : 0], M / 1024);
  const unsigned grid = (unsigned)std::min<int64_t>(most, std::max<int64_t>(kSMs, M / (f ? 64 : 48)));
  return cudaLaunchKernel(tile_kernel(ctx, width, f != nullptr), dim3(grid),
                          dim3(tile_threads(tl.l, f != nullptr)), args, tile_pass_smem(tl.l[0], tl.l[1], tl.l[2], f != nullptr), s);
}

cudaError_t launch_tiles(const mls_ctx* ctx, const mls_transfer* T, const void* u, const void* Vb, double dt, void* U,
                         void* F, void* f, cudaStream_t s) {
  return ctx->opt.field == MLS_BF16 ? launch_tiles_of<__nv_bfloat16>(ctx, T, u, Vb, dt, U, F, f, s)
                                    : launch_tiles_of<float>(ctx, T, u, Vb, dt, U, F, f, s);
}

}  // namespace mls
