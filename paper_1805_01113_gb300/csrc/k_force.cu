// Direct forcing (Section 2, text after Eq. 6 and Eq. 7): U_l = sum_k phi_k^l u_k,
// F_l = (V_b,l - U_l) / dt, f_k += sum_l c_l phi_k^l F_l.  In single precision
// one pass over the tiles; as interpolation (forming F) and spread where the tiles
// are large (tiles_configure), f shares memory with u, or f is bfloat16: the
// pass adds a tile to f every 256 markers and the spread every 512, and each
// addition rounds to 8 bits (2.1 against 2.0e-3 of f on 2.56 M markers in 512^3).
#include "transfer_common.cuh"

namespace mls {

// F_l = (V_b,l - U_l) / dt in place over U, double precision: tile order j,
// caller index perm[j]; markers without support (home < 0) get F = 0.
__global__ void __launch_bounds__(kBlock) k_force_from_u(const int32_t* __restrict__ home,
                                                         const int32_t* __restrict__ perm, int64_t M,
                                                         const double* __restrict__ Vb, double inv_dt,
                                                         double* __restrict__ UF) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= M) return;
  const int64_t m = perm[j];
  const bool ok = home[j] >= 0;
#pragma unroll
  for (int q = 0; q < 3; ++q) UF[q * M + m] = ok ? (Vb[q * M + m] - UF[q * M + m]) * inv_dt : 0.0;
}

static bool one_pass(const mls_ctx* ctx, const void* u, const void* f) {
  const int64_t bytes = 12LL * ctx->n[0] * ctx->n[1] * ctx->n[2];
  const char *a = (const char*)u, *b = (const char*)f;
  return ctx->tile_grid[1] > 0 && ctx->opt.field == MLS_F32 && (a + bytes <= b || b + bytes <= a);
}

cudaError_t launch_direct_forcing(const mls_ctx* ctx, const mls_transfer* T, const void* u, const void* Vb,
                                  double dt, void* U, void* F, void* f, cudaStream_t s) {
  if (T->M == 0) return cudaSuccess;
  cudaError_t e;
  if (ctx->opt.real == MLS_F64) {
    if ((e = launch_interp(ctx, T, u, U ? U : F, s)) != cudaSuccess) return e;
    if (U && (e = cudaMemcpyAsync(F, U, (size_t)3 * T->M * 8, cudaMemcpyDeviceToDevice, s)) != cudaSuccess) return e;
    const unsigned nt = block_threads(T->M, kBlock);
    k_force_from_u<<<blocks_for(T->M, nt), nt, 0, s>>>(T->home, T->perm, T->M, (const double*)Vb, 1.0 / dt, (double*)F);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  } else if (one_pass(ctx, u, f)) {
    return launch_tiles(ctx, T, u, Vb, dt, U, F, f, s);
  } else if ((e = launch_interp(ctx, T, u, U, s, Vb, dt, F)) != cudaSuccess) {
    return e;
  }
  return launch_spread(ctx, T, F, f, s);
}

}  // namespace mls
