// Runs of stored markers of one home cell.  The in-tile sort puts the markers
// of a home cell next to each other, and markers of one cell share their 27
// support nodes.  A run is the markers of one home cell inside one aligned
// group of four stored markers, so a thread that owns a run reads phi_k of its
// group with one 16-byte load and each node's field, or adds its terms, once for
// the whole run.
// On the workloads here a run holds 1.8 (1 280-face bodies) to 2.4 (mixed
// bodies) markers; any order of the markers is correct, unsorted ones only
// make shorter runs.
#pragma once

#include "build_common.cuh"
#include "transfer_common.cuh"

namespace mls {

constexpr int kChunkPer = 4;   // markers per thread of a chunk

// A run in one word: first marker in the chunk (at most 2^16 markers) and the
// number of markers less one.
struct Run {
  int first, len;
  __device__ __forceinline__ explicit Run(int w) : first(w >> 2), len((w & 3) + 1) {}
  static __device__ __forceinline__ int pack(int first, int len) { return first << 2 | (len - 1); }
};

// Lists the runs of the stored markers [max(j0, start), min(j0 + kChunkPer NT,
// end)), j0 a multiple of 4.  `each` is called for every one of them (its index
// and its place in the chunk), `before` ahead of the first of the two barriers
// and `between` them.  Returns the number of runs; runs[] and what the
// callbacks wrote may then be read by every thread.
template <int NT, typename Each, typename Before, typename Between>
__device__ __forceinline__ int list_runs(const int32_t* __restrict__ home, unsigned start, unsigned end, unsigned j0,
                                         int* runs, int* cnt, Each&& each, Before&& before, Between&& between) {
  constexpr int W = NT / 32;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  int word[kChunkPer], place[kChunkPer];
#pragma unroll
  for (int i = 0; i < kChunkPer; ++i) {
    word[i] = -1;
    place[i] = 0;
    int n = 0;
    if (j0 + i * NT < end) {
      const unsigned j = j0 + i * NT + tid;
      const bool act = j >= start && j < end;
      bool head = false;
      if (act) {
        head = (j & 3) == 0 || j == start || home[j] != home[j - 1];
        each(j, i * NT + tid);
      }
      const unsigned hm = __ballot_sync(0xffffffffu, head);
      place[i] = __popc(hm & ((1u << lane) - 1u));
      n = __popc(hm);
      if (head) {
        // The run ends at the next head of its group of four, with the group or with the markers.
        const int p = lane & 3;
        const unsigned next = ((hm >> (lane & ~3)) & 15u) >> (p + 1);
        word[i] = Run::pack(i * NT + tid, (int)min(next ? (unsigned)__ffs(next) : 4u - p, end - j));
      }
    }
    if (lane == 0) cnt[i * W + wid] = n;
  }
  before();
  __syncthreads();
  between();
  int total = 0;
#pragma unroll
  for (int i = 0; i < kChunkPer; ++i) {
    if (j0 + i * NT >= end) break;
    int at = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      if (w == wid) at = total;
      total += cnt[i * W + w];
    }
    if (word[i] >= 0) runs[at + place[i]] = word[i];
  }
  __syncthreads();
  return total;
}

// Four markers' phi_k from an aligned group: one 16-byte load when the planes
// are 16-byte aligned (QUAD: a capacity that is a multiple of 4), else four
// loads of the `left` markers that exist.
template <bool QUAD>
__device__ __forceinline__ float4 phi_group(const float* __restrict__ p, int64_t left) {
  if constexpr (QUAD) return __ldg(reinterpret_cast<const float4*>(p));
  return make_float4(p[0], left > 1 ? p[1] : 0.f, left > 2 ? p[2] : 0.f, left > 3 ? p[3] : 0.f);
}

// U = sum_k phi_k u_k of the four markers of an aligned group whose member(s)
// of home cell i form a run (the other components of the result are not
// theirs): each node's velocity is read once for the whole run.
template <typename FT, bool QUAD>
__device__ __forceinline__ void gather_run(const Dims& D, const int i[3], const FT* __restrict__ u,
                                           const float* __restrict__ plane, int64_t cap, int64_t left, float4 U[3]) {
  const int64_t N = (int64_t)D.n[0] * D.n[1] * D.n[2];
  int xs[3], ys[3], zs[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    xs[a] = wrap(i[0] + a - 1, D.n[0], D.periodic[0]);
    ys[a] = wrap(i[1] + a - 1, D.n[1], D.periodic[1]);
    zs[a] = wrap(i[2] + a - 1, D.n[2], D.periodic[2]);
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) U[q] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int cz = 0; cz < 3; ++cz)
#pragma unroll
    for (int cy = 0; cy < 3; ++cy) {
      const FT* ur = u + (int64_t)((zs[cz] * D.n[1] + ys[cy]) * D.n[0]);   // below n_x n_y n_z < 2^31
#pragma unroll
      for (int cx = 0; cx < 3; ++cx) {
        const float4 p = phi_group<QUAD>(plane + (9 * cz + 3 * cy + cx) * cap, left);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const float v = load_field<float, FT>(ur + q * N + xs[cx]);
          U[q].x += p.x * v;
          U[q].y += p.y * v;
          U[q].z += p.z * v;
          U[q].w += p.w * v;
        }
      }
    }
}

__device__ __forceinline__ float at(const float4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

}  // namespace mls
