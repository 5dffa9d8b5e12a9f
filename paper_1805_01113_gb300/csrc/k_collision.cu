// Coarse-grained collision detection on the Eulerian mesh (Section 4): a cell
// whose markers belong to more than one body is a collision cell, and every
// marker in it is flagged.  The markers are already grouped by spreading tile,
// so each tile's cell states live in shared memory for the duration of one
// block iteration instead of in a zeroed global array.
#include "transfer_common.cuh"

namespace mls {

// Groups of threads (warps or whole blocks) walk the non-empty tiles.  For a
// tile: zero the state of its 2^(lx+ly+lz) home cells; every marker with a body index b > 0 claims its cell
// with compare-and-swap (0 -> b) and, finding another index there, sets the
// cell to -1; then every marker reads its cell: -1 flags it.  The occupied
// cells are written to `coll` when requested.  The final state of a cell does
// not depend on the order of the updates (an empty cell takes the first index,
// any second index makes it -1, and -1 is never overwritten).
// Returns the colliding markers that the thread found.
// Bound by the chain of dependent loads of a tile (its header, the order, the
// body indices); the markers of a tile of up to four per thread are loaded once,
// and the next tile's header is loaded ahead.
template <bool WARP>
__device__ __forceinline__ unsigned long long collide_tiles(const Dims& D, const Tiles& tl,
                                                            const int32_t* __restrict__ home,
                                                            const int32_t* __restrict__ perm,
                                                            const int32_t* __restrict__ items, int n_items,
                                                            const int32_t* __restrict__ offsets,
                                                            const int32_t* __restrict__ counts,
                                                            const int32_t* __restrict__ body,
                                                            int32_t* __restrict__ flag, int32_t* __restrict__ coll) {
  extern __shared__ __align__(16) int state_all[];
  constexpr int G = WARP ? 32 : kSpreadThreads, PER = 4, GROUPS = kSpreadThreads / G;
  const int lx = tl.l[0], ly = tl.l[1], lz = tl.l[2];
  const int TC = 1 << (lx + ly + lz);
  const int tid = threadIdx.x % G, group = threadIdx.x / G;
  int* state = state_all + group * TC;
  auto sync = [] {
    if (WARP) __syncwarp();
    else __syncthreads();
  };
  const int stride = gridDim.x * GROUPS;
  unsigned long long found = 0;
  int it = blockIdx.x * GROUPS + group;
  int b = it < n_items ? items[it] : 0, start = 0, n = 0;
  if (it < n_items) {
    start = offsets[b];
    n = counts[b];
  }
  for (; it < n_items; it += stride) {
    const bool more = it + stride < n_items;
    const int bn = more ? items[it + stride] : 0;
    int m[PER], bid[PER], cell[PER];
    int ox = 0, oy = 0, oz = 0;
    auto load = [&](int w0) {
      int h[PER];
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        const int i = w0 + q * G + tid;
        h[q] = i < n ? home[start + i] : 0;
        m[q] = i < n ? perm[start + i] : -1;
      }
#pragma unroll
      for (int q = 0; q < PER; ++q) bid[q] = m[q] >= 0 ? body[m[q]] : 0;
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        int i[3];
        decode_home(h[q], D, i);
        cell[q] = ((((i[2] & ((1 << lz) - 1)) << ly) | (i[1] & ((1 << ly) - 1))) << lx) | (i[0] & ((1 << lx) - 1));
        if (m[q] >= 0) {
          ox = i[0] & ~((1 << lx) - 1);
          oy = i[1] & ~((1 << ly) - 1);
          oz = i[2] & ~((1 << lz) - 1);
        }
      }
    };
    for (int c = tid; c < TC; c += G) state[c] = 0;
    sync();
    for (int w0 = 0; w0 < n; w0 += PER * G) {
      load(w0);
#pragma unroll
      for (int q = 0; q < PER; ++q)
        if (bid[q] > 0) {
          const int old = atomicCAS(&state[cell[q]], 0, bid[q]);
          if (old != 0 && old != bid[q]) state[cell[q]] = -1;
        }
    }
    const int next_start = more ? offsets[bn] : 0, next_n = more ? counts[bn] : 0;
    sync();
    for (int w0 = 0; w0 < n; w0 += PER * G) {
      if (n > PER * G) load(w0);
#pragma unroll
      for (int q = 0; q < PER; ++q)
        if (m[q] >= 0) {
          const int hit = bid[q] > 0 && state[cell[q]] == -1;
          flag[m[q]] = hit;
          found += hit;
        }
    }
    if (coll) {
      // Thread 0 always has a marker of the tile, so it knows the tile's first cell.
      if constexpr (WARP) {
        ox = __shfl_sync(0xffffffffu, ox, 0);
        oy = __shfl_sync(0xffffffffu, oy, 0);
        oz = __shfl_sync(0xffffffffu, oz, 0);
      } else {
        ox = (b % tl.nb[0]) << lx;
        oy = ((b / tl.nb[0]) % tl.nb[1]) << ly;
        oz = (b / (tl.nb[0] * tl.nb[1])) << lz;
      }
      for (int c = tid; c < TC; c += G) {
        const int s = state[c];
        if (s == 0) continue;
        const int gx = ox + (c & ((1 << lx) - 1)), gy = oy + ((c >> lx) & ((1 << ly) - 1)), gz = oz + (c >> (lx + ly));
        coll[((int64_t)gz * D.n[1] + gy) * D.n[0] + gx] = s;
      }
    }
    sync();
    b = bn;
    start = next_start;
    n = next_n;
  }
  return found;
}

// A warp per tile keeps four times as many tiles in flight as a block per tile
// and needs no block barriers: 5.1 M markers in 384^3, with the clearing of the
// cell array, 126 -> 108 us.  Where the tiles do not fill the device with blocks,
// or twice over while they hold fewer than 512 markers on average, a tile's own
// chain is what takes time and a block walks it sooner: 1.4 M markers of a dense
// packing in 64^3 21 against 51 us, 16 000 markers in 48^3 3.4 against 5.8; 11.2 M
// on 4 096 tiles in 128^3 take 129 by warps and 157 by blocks.
// SMALL: the states of a block's four warps fit (tiles of up to 2^10 cells).
template <bool SMALL>
__global__ void __launch_bounds__(kSpreadThreads) k_collisions(Dims D, Tiles tl, const int32_t* __restrict__ home,
                                                               const int32_t* __restrict__ perm,
                                                               const int32_t* __restrict__ items,
                                                               const int32_t* __restrict__ n_items_p,
                                                               const int32_t* __restrict__ offsets,
                                                               const int32_t* __restrict__ counts, int64_t M,
                                                               const int32_t* __restrict__ body,
                                                               int32_t* __restrict__ flag, int32_t* __restrict__ coll,
                                                               unsigned long long* __restrict__ n_colliding) {
  const int n_items = *n_items_p, lane = threadIdx.x & 31;
  const int64_t d0 = offsets[tl.nbins - 1];
  const int blocks = gridDim.x;
  unsigned long long found;
  if (!SMALL || n_items < blocks || (n_items < 2 * blocks && d0 < 512 * (int64_t)n_items))
    found = collide_tiles<false>(D, tl, home, perm, items, n_items, offsets, counts, body, flag, coll);
  else
    found = collide_tiles<true>(D, tl, home, perm, items, n_items, offsets, counts, body, flag, coll);
  // Markers without support: never flagged.
  for (int64_t j = d0 + (int64_t)blockIdx.x * kSpreadThreads + threadIdx.x; j < M;
       j += (int64_t)gridDim.x * kSpreadThreads)
    flag[perm[j]] = 0;
  if (n_colliding) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) found += __shfl_xor_sync(0xffffffffu, found, o);
    if (lane == 0 && found) atomicAdd(n_colliding, found);
  }
}

// Four tiles' states fit the default 48 KB of a block several times over (2^10
// cells: 16 KB, 14 blocks per SM).
static bool collide_small(const mls_ctx* ctx) {
  return ctx->tiles.l[0] + ctx->tiles.l[1] + ctx->tiles.l[2] <= 10;
}
static size_t collide_smem(const mls_ctx* ctx) {
  const int* l = ctx->tiles.l;
  return ((size_t)4 << (l[0] + l[1] + l[2])) * (collide_small(ctx) ? kSpreadThreads / 32 : 1);
}

cudaError_t launch_collisions(const mls_ctx* ctx, const mls_transfer* T, const int32_t* body, int32_t* flag,
                              int32_t* coll, unsigned long long* n_colliding, cudaStream_t s) {
  if (T->M == 0) return cudaSuccess;
  auto kern = collide_small(ctx) ? k_collisions<true> : k_collisions<false>;
  kern<<<ctx->collision_grid, kSpreadThreads, collide_smem(ctx), s>>>(dims_of(ctx), ctx->tiles, T->home, T->perm,
                                                                      T->items, T->n_items, T->offsets, T->counts,
                                                                      T->M, body, flag, coll, n_colliding);
  return cudaGetLastError();
}

cudaError_t collision_configure(mls_ctx* ctx) {
  auto kern = collide_small(ctx) ? k_collisions<true> : k_collisions<false>;
  const int smem = (int)collide_smem(ctx);
  cudaError_t e;
  if ((e = raise_smem_limit((const void*)kern, smem)) != cudaSuccess) return e;
  int per_sm = 0, sms = 0;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kSpreadThreads, smem)) != cudaSuccess)
    return e;
  ctx->collision_grid = (per_sm > 0 ? per_sm : 1) * sms;
  return cudaSuccess;
}

}  // namespace mls
