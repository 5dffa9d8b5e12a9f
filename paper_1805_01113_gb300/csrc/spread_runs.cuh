// Accumulation of the forces of runs in a tile's shared-memory accumulator.
#pragma once

#include "runs.cuh"

namespace mls {

// Shared memory of a chunk of kChunkPer * nt markers: c_l F_l (three arrays),
// then one word per run.
__host__ __device__ constexpr int run_smem_bytes(int nt) { return 4 * kChunkPer * nt * 4; }

// Asks L2 for what the next tile's markers [start, end) need: home, perm, c
// and their 27 phi (rows of a capacity that is a multiple of 4).
__device__ __forceinline__ void prefetch_tile(const float* __restrict__ phi, const int32_t* __restrict__ home,
                                              const int32_t* __restrict__ perm, const float* __restrict__ cl,
                                              int64_t cap, unsigned start, unsigned end) {
  const unsigned t = threadIdx.x;
  if (t < 30 && end > start) {
    const unsigned j = start & ~3u, bytes = (((end + 3u) & ~3u) - j) * 4u;
    const void* p = t < 27   ? (const void*)(phi + t * cap + j)
                    : t == 27 ? (const void*)(home + j)
                    : t == 28 ? (const void*)(perm + j)
                              : (const void*)(cl + j);
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
  }
}

// A tile's own cost in markers: its two chains of loads, three barriers and the
// flush.  Blocks take ranges of equal weight; on 32 M markers (204 a tile) the
// spread takes 3.4 ms with weight 0, 2.36 with 64, 1.72 with 180 and 2.05 with
// 500, and on 2.56 M (105 a tile) 150 to 250 are equal.  Tiles dealt out round
// robin instead left the blocks up to 1.6 times their mean.
constexpr int kTileWeight = 180;

// First of the n tiles before which markers and tiles weigh at least `target`;
// by a whole warp, 32 probes at a time.
__device__ __forceinline__ int tile_at(const int32_t* __restrict__ items, const int32_t* __restrict__ offsets, int n,
                                       int64_t target) {
  int lo = 0, hi = n;                                   // the answer lies in [lo, hi]
  while (lo < hi) {
    const int step = (hi - lo + 31) / 32, p = lo + (int)(threadIdx.x & 31) * step;
    const bool before = p < hi && offsets[items[p]] + (int64_t)kTileWeight * p < target;
    const int k = __popc(__ballot_sync(0xffffffffu, before));   // probes lo .. lo + (k - 1) step are before it
    if (k == 0) return lo;
    hi = min(hi, lo + k * step);
    lo = lo + (k - 1) * step + 1;
  }
  return lo;
}

// Share `part` of `parts` (whole groups of 32 markers) of a tile's markers, for
// blocks that would otherwise be idle: a small workload takes as long as a tile's
// chain from load to flush.  The spread of 15 360 markers on three bodies in 64^3
// takes 6.0 us by up to eight shares, 11.3 by whole tiles.
__device__ __forceinline__ void tile_part(int part, int parts, unsigned& start, unsigned& end) {
  const unsigned first = start & ~3u, share = ((end - first + parts - 1) / parts + 31u) & ~31u;
  const unsigned from = first + part * share;
  start = max(start, from);
  end = min(end, from + share);
}

// max(|a|, |b|, |c|), NaN if one is.
__device__ __forceinline__ float max_abs(float a, float b, float c) {
  float r;
  asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// One node's term of a run in fixed point (the same bits wherever it is formed).
__device__ __forceinline__ int run_term(float4 p, float4 v) {
  return __float2int_rn(__fmaf_rn(p.x, v.x, __fmaf_rn(p.y, v.y, __fmaf_rn(p.z, v.z, __fmul_rn(p.w, v.w)))));
}

// Sums of |c_l F_l| of the markers a thread saw, per component, to red[].
template <int NT>
__device__ __forceinline__ void publish_sums(float sum[3], float* red) {
#pragma unroll
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum[q] += __shfl_xor_sync(0xffffffffu, sum[q], o);
  if ((threadIdx.x & 31) == 0) {
    red[3 * (threadIdx.x >> 5)] = sum[0];
    red[3 * (threadIdx.x >> 5) + 1] = sum[1];
    red[3 * (threadIdx.x >> 5) + 2] = sum[2];
  }
}

// Fixed-point scale of a chunk.  Terms with |phi| < 2^(1 - e) are accumulated
// (e = scale_bits), so no cell's sum exceeds 2^(1 - e) S, S the chunk's sum of
// |c_l F_l| of that component (rounded up by 1e-4, which covers its own
// rounding); with S < 2^ex the unit 2^(ex - 30 - e) keeps every sum inside 32
// bits.  e grows with the chunk so that the unit is never coarser than 2^-22 of
// the largest |c_l F_l|, which equal forces need: S is at most 2^(7 + e) times
// the largest.  With e = 0 for all chunks a full chunk of equal forces had a unit
// four times as coarse and an error of 2.4e-7 of f, against 0.74e-7 so (1 024 000
// markers of 5 120-face bodies in 128^3); forces that differ have a finer unit,
// the sum being smaller (noise: 1.9e-6, now 4.9e-7 there).  The launch caps e at 1
// where phi itself exceeds 1/2.
__device__ __forceinline__ int scale_bits(unsigned markers) { return markers <= 128 ? 0 : markers <= 256 ? 1 : 2; }
enum ChunkScale { kZero, kFixed, kDirect };
struct Scale {
  float unit[3], inv[3], limit;   // |phi| below the limit is accumulated
  int kind[3];
};
// Component q of the scale, by one thread, from the warps' sums.
template <int NT>
__device__ __forceinline__ void chunk_scale(const float* red, int q, int bits, Scale* out) {
  float s = red[q];
  for (int w = 1; w < NT / 32; ++w) s += red[3 * w + q];
  out->kind[q] = s == 0.f ? kZero : kFixed;
  s *= 1.0001f;
  if (!isfinite(s)) out->kind[q] = kDirect;
  // The exponent field of s < 2^ex is ex + 126 (0 below the normal numbers).
  const int sh = min(30 + bits + 126 - (int)((__float_as_uint(s) >> 23) & 255u), 126);
  out->inv[q] = __uint_as_float((unsigned)(127 + sh) << 23);
  out->unit[q] = __uint_as_float((unsigned)(127 - sh) << 23);
  out->limit = __uint_as_float((unsigned)(128 - bits) << 23);   // 2^(1 - bits)
}
__device__ __forceinline__ ChunkScale chunk_kind(const Scale& s) {
  return (ChunkScale)max(s.kind[0], max(s.kind[1], s.kind[2]));
}

// Adds component q of a run's markers at its node k straight to the field.
template <typename FT>
__device__ __forceinline__ void add_direct(const Dims& D, const int i[3], const Run& r, int k, int q,
                                           const float* __restrict__ phi, int64_t cap, int64_t j,
                                           const float* sv, int chunk, FT* __restrict__ f) {
  const int64_t N = (int64_t)D.n[0] * D.n[1] * D.n[2];
  const int gx = wrap(i[0] + k % 3 - 1, D.n[0], D.periodic[0]);
  const int gy = wrap(i[1] + (k / 3) % 3 - 1, D.n[1], D.periodic[1]);
  const int gz = wrap(i[2] + k / 9 - 1, D.n[2], D.periodic[2]);
  const int64_t o = ((int64_t)gz * D.n[1] + gy) * D.n[0] + gx;
  for (int l = 0; l < r.len; ++l) {
    const float p = phi[k * cap + j + l];
    add_field<float, FT>(f + q * N + o, p * sv[q * chunk + r.first + l]);
  }
}

// Adds a chunk's runs into the accumulator (AccShape) and tags the rows they
// touch: a thread takes one plane of a run's stencil, so that its nine loads of
// phi are in flight together and the 58 to 85 runs of a tile fill the block (a
// thread per run waited for phi row by row).  No branch lies between the loads
// and the atomics: one per node made the compiler wait for every load in turn
// (3.6 against 2.1 ms on 32 M markers).
// Lanes of one warp often own runs of one cell, and lanes that add to one word
// in the same instruction are serialised, so every third lane starts with
// another component: only its pointers differ (wavefronts per atomic on a
// model of the mixed bodies: 4.9 without, 2.9 with ACC = 8 or 20 mod 32).
// Terms with some |phi| >= limit (chunk_scale's 2^(1 - e)) or a NaN in their
// group of four go to f directly.
template <typename FT, bool QUAD, int NT, int CHUNK>
__device__ __forceinline__ void add_runs(const Dims& D, const int o[3], int n, const int* runs,
                                         const int32_t* __restrict__ home,
                                         const float* sv, unsigned j0, const float* __restrict__ phi, int64_t cap,
                                         int64_t M, const Scale& S, int* acc, int AX, int PS, int ACC, int AY,
                                         unsigned char* tags, unsigned char tag, FT* __restrict__ f) {
  const int c0 = threadIdx.x % 3, c1 = c0 == 2 ? 0 : c0 + 1, c2 = c0 == 0 ? 2 : c0 - 1;
  const float s0 = S.inv[c0], s1 = S.inv[c1], s2 = S.inv[c2];
  for (int t = threadIdx.x; t < 3 * n; t += NT) {
    const int cz = (t >= n) + (t >= 2 * n);
    const Run r(runs[t - cz * n]);
    const int g = r.first & ~3;
    const float* plane = phi + j0 + g + 9 * cz * cap;
    const int64_t left = M - (int64_t)(j0 + g);
    float4 p[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) p[k] = phi_group<QUAD>(plane + k * cap, left);
    const unsigned in = ((1u << r.len) - 1u) << (r.first & 3);
    auto load = [&](int c, float s) {
      float4 v = *reinterpret_cast<const float4*>(sv + c * CHUNK + g);
      v.x = in & 1u ? v.x * s : 0.f;
      v.y = in & 2u ? v.y * s : 0.f;
      v.z = in & 4u ? v.z * s : 0.f;
      v.w = in & 8u ? v.w * s : 0.f;
      return v;
    };
    const float4 v0 = load(c0, s0), v1 = load(c1, s1), v2 = load(c2, s2);
    int i[3];
    decode_home(home[j0 + r.first], D, i);
    const int y = i[1] - o[1], z = i[2] - o[2] + cz;
    const int base = AccShape::kFront + z * PS + y * AX + (i[0] - o[0]) - 1;
    int* a0 = acc + c0 * ACC + base;
    int* a1 = acc + c1 * ACC + base;
    int* a2 = acc + c2 * ACC + base;
    float most = 0.f;
#pragma unroll
    for (int cy = 0; cy < 3; ++cy) {
      tags[z * AY + y + cy] = tag;
#pragma unroll
      for (int cx = 0; cx < 3; ++cx) {
        const float4 pk = p[3 * cy + cx];
        most = max_abs(max_abs(most, pk.x, pk.y), pk.z, pk.w);
        atomicAdd(a0 + cy * AX + cx, run_term(pk, v0));
        atomicAdd(a1 + cy * AX + cx, run_term(pk, v1));
        atomicAdd(a2 + cy * AX + cx, run_term(pk, v2));
      }
    }
    // What a node with a term out of the limit added is taken back, and its terms
    // go to f.
    const float limit = S.limit;
    if (!(most < limit)) {
      for (int k = 0; k < 9; ++k) {
        const float4 pk = phi_group<QUAD>(plane + k * cap, left);
        if (max_abs(max_abs(0.f, pk.x, pk.y), pk.z, pk.w) < limit) continue;
        const int at = k / 3 * AX + k % 3;
        atomicAdd(a0 + at, -run_term(pk, v0));
        atomicAdd(a1 + at, -run_term(pk, v1));
        atomicAdd(a2 + at, -run_term(pk, v2));
        for (int q = 0; q < 3; ++q)
          add_direct<FT>(D, i, r, 9 * cz + k, q, phi, cap, (int64_t)j0 + r.first, sv, CHUNK, f);
      }
    }
  }
}

// Adds the accumulator rows with the chunk's tag to f (with VEC by 16- or
// 8-byte vector reductions of four cells, the two halo cells of a row singly;
// else cell by cell) and resets them to zero.  The groups of all rows come
// first and the halo cells after them, so that the lanes of a warp do the same.
// Tags count chunks modulo 255 and need no reset: a row with an old equal tag
// holds zeros.
template <typename FT, bool VEC, int LX, int NT>
__device__ __forceinline__ void flush_rows(const Dims& D, const int o[3], const AccShape& A, int* acc,
                                           const unsigned char* tags, unsigned char tag, const float* unit,
                                           FT* __restrict__ f) {
  constexpr int TX = 1 << LX;
  constexpr int GROUPS = VEC ? TX / 4 : 0, CELLS = VEC ? 2 : TX + 2;   // of a row, and the cells added singly
  const int rows = A.AY * A.AZ;
  const int64_t N = (int64_t)D.n[0] * D.n[1] * D.n[2];
  const float u0 = unit[0], u1 = unit[1], u2 = unit[2];
  for (int e = threadIdx.x; e < (GROUPS + CELLS) * rows; e += NT) {
    const bool group = VEC && e < GROUPS * rows;
    const int s = group ? e : e - GROUPS * rows;
    const int row = group ? s / (VEC ? GROUPS : 1) : s / CELLS, q = s - row * (group ? GROUPS : CELLS);
    if (tags[row] != tag) continue;
    const int ey = row % A.AY, ez = row / A.AY;
    int* a = acc + AccShape::kFront + ez * A.PS + ey * A.AX;
    FT* fr = f + (int64_t)((wrap(o[2] - 1 + ez, D.n[2], D.periodic[2]) * D.n[1] +
                            wrap(o[1] - 1 + ey, D.n[1], D.periodic[1])) * D.n[0]);
    if (group) {
      int gx = o[0] + 4 * q;
      if (gx >= D.n[0]) {                        // past the last cell of a periodic axis: the halo of cell n - 1
        gx -= D.n[0];
        if (!D.periodic[0] || gx >= D.n[0]) continue;
      }
      int4* p = reinterpret_cast<int4*>(a + 4 * q);
      const int4 v0 = p[0], v1 = p[A.ACC / 4], v2 = p[A.ACC / 2];
      const int4 z = make_int4(0, 0, 0, 0);
      fr += gx;
      if (v0.x | v0.y | v0.z | v0.w) red_add_v4(fr, v0.x * u0, v0.y * u0, v0.z * u0, v0.w * u0);
      if (v1.x | v1.y | v1.z | v1.w) red_add_v4(fr + N, v1.x * u1, v1.y * u1, v1.z * u1, v1.w * u1);
      if (v2.x | v2.y | v2.z | v2.w) red_add_v4(fr + 2 * N, v2.x * u2, v2.y * u2, v2.z * u2, v2.w * u2);
      p[0] = z;
      p[A.ACC / 4] = z;
      p[A.ACC / 2] = z;
    } else {
      const int x = VEC ? (q == 0 ? -1 : TX) : q - 1;
      int* p = a + x;
      const int v0 = p[0], v1 = p[A.ACC], v2 = p[2 * A.ACC];
      if ((v0 | v1 | v2) == 0) continue;
      p[0] = p[A.ACC] = p[2 * A.ACC] = 0;
      fr += wrap(o[0] + x, D.n[0], D.periodic[0]);
      if constexpr (VEC) {
        if (v0) red_add_end(fr, v0 * u0, q == 0);
        if (v1) red_add_end(fr + N, v1 * u1, q == 0);
        if (v2) red_add_end(fr + 2 * N, v2 * u2, q == 0);
      } else {
        if (v0) add_field<float, FT>(fr, v0 * u0);
        if (v1) add_field<float, FT>(fr + N, v1 * u1);
        if (v2) add_field<float, FT>(fr + 2 * N, v2 * u2);
      }
    }
  }
}

}  // namespace mls
