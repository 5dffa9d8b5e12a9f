// Runs of stored markers of one home cell.  The in-tile sort puts the markers
// of a home cell next to each other, and markers of one cell share their 27
// support nodes.  A run is the markers of one home cell inside one aligned
// group of four stored markers, so a thread that owns a run reads phi_k of its
// group with one 16-byte load and adds a node's terms once for the whole run.
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

}  // namespace mls
