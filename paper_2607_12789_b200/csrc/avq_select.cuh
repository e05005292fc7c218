// Selection of the P parents with the largest importance, for the kernels that hold the importances as float64.
#pragma once

#include <stdint.h>

namespace avq {

constexpr int kSelThreads = 512;   // threads that take part: warps 0 .. 15 of the CTA

// Top-P of w[0 .. M) (non-negative; ties to the lower index): sel[j] = 1 for the chosen parents (zero before), sel_list[0 .. P)
// their indices in ascending order, also written to topp_out unless that is null.  Scratch: cand [M], s_count [32], s_ncand.
// sync() is a barrier of the participating threads; the importances have been published by one, the results are as well.
// Non-negative doubles order like their bit patterns.
// Only candidates are ranked, those at or above a bound that at least P keys reach: the largest of 32 sample keys
// that has P keys at or above it.  (Ranking all of them took 16 of 230 us at M = 512.)
template <typename Sync>
__device__ __forceinline__ void select_parents(const double* w, int M, int P, int* sel, int* sel_list, int* cand, int* s_count,
                                               int* s_ncand, int32_t* topp_out, Sync sync) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const unsigned long long* key = reinterpret_cast<const unsigned long long*>(w);
  if (P >= M) {
    for (int j = tid; j < M; j += kSelThreads) sel[j] = 1;
  } else if (4 * M <= kSelThreads) {
    // Few parents: four or more threads rank each of them at once, without a bound and its barriers.
    int lt = 2;                                             // 2^lt threads share a parent's scan
    while (lt < 4 && (M << (lt + 1)) <= kSelThreads) ++lt;
    const int j = tid >> lt, part = tid & ((1 << lt) - 1);
    const unsigned long long kj = key[min(j, M - 1)];
    int rank = 0;
#pragma unroll 4
    for (int k = part; k < M; k += 1 << lt) {
      const unsigned long long kk = key[k];
      rank += (kk > kj) | ((kk == kj) & (k < j));
    }
    for (int o = 1; o < (1 << lt); o <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
    if (j < M && part == 0 && rank < P) sel[j] = 1;
  } else {
    unsigned long long bound = 0;
    {
      const unsigned long long smp0 = key[2 * warp * M / 32], smp1 = key[(2 * warp + 1) * M / 32];
      int c = 0;                                            // keys at or above the two samples, 16 bits each
#pragma unroll 4
      for (int j = lane; j < M; j += 32) {
        const unsigned long long kj = key[j];
        c += (kj >= smp0) + ((kj >= smp1) << 16);
      }
      c = __reduce_add_sync(0xffffffffu, c);
      if (lane < 2) s_count[2 * warp + lane] = (c >> (16 * lane)) & 0xFFFF;
      if (tid == 0) *s_ncand = 0;
      sync();
      if (s_count[lane] >= P) bound = key[lane * M / 32];
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, bound, o);
        bound = other > bound ? other : bound;
      }
    }
    for (int j0 = 0; j0 < M; j0 += kSelThreads) {            // in any order, one addition per warp
      const int j = j0 + tid;
      const bool on = j < M && key[j] >= bound;
      const uint32_t bal = __ballot_sync(0xffffffffu, on);
      int base = 0;
      if (lane == 0 && bal) base = atomicAdd(s_ncand, __popc(bal));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (on) cand[base + __popc(bal & ((1u << lane) - 1u))] = j;
    }
    sync();
    const int nc_ = *s_ncand;
    int lt = 0;                                             // 2^lt threads share a candidate's scan
    while (lt < 4 && (nc_ << (lt + 1)) <= kSelThreads) ++lt;
    const int part = tid & ((1 << lt) - 1);
    for (int i0_ = 0; i0_ < nc_; i0_ += kSelThreads >> lt) {   // uniform
      const int i = i0_ + (tid >> lt);
      const int j = i < nc_ ? cand[i] : 0;
      const unsigned long long kj = key[j];
      int rank = 0;
      if (i < nc_) {
#pragma unroll 4
        for (int q = part; q < nc_; q += 1 << lt) {
          const int k = cand[q];
          const unsigned long long kk = key[k];
          rank += (kk > kj) | ((kk == kj) & (k < j));
        }
      }
      for (int o = 1; o < (1 << lt); o <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
      if (i < nc_ && part == 0 && rank < P) sel[j] = 1;
    }
  }
  sync();
  // the ascending list: a warp per 32 parents (M <= 1024: at most 32 words of s_count)
  const int words = (M + 31) >> 5;
  uint32_t mine[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int j = 32 * (warp + 16 * u) + lane;
    mine[u] = __ballot_sync(0xffffffffu, j < M && sel[min(j, M - 1)] != 0);
    if (lane == 0) s_count[warp + 16 * u] = (int)mine[u];
  }
  sync();
  const int ones = __popc((uint32_t)s_count[lane]);         // (words past the last are zero)
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int word = warp + 16 * u;
    if (word < words) {
      const int base = __reduce_add_sync(0xffffffffu, lane < word ? ones : 0);
      if ((mine[u] >> lane) & 1u) sel_list[base + __popc(mine[u] & ((1u << lane) - 1u))] = 32 * word + lane;
    }
  }
  sync();
  if (topp_out)
    for (int r = tid; r < P; r += kSelThreads) topp_out[r] = sel_list[r];
}

}  // namespace avq
