// avq_forward_permuted: the forward pass over query tiles that follow a caller-supplied token order
// (Sec. "Vector Quantization for (A)VQ-Attention": image tokens are reordered along a space-filling curve
// so that a tile holds neighbouring tokens; the curve itself is the caller's business).
//
// Only the grouping of QUERIES into tiles changes the result: per-codeword sums and counts do not depend
// on the order of the keys.  So the call gathers Q into tile order, Qp[i] = Q[perm[i]], runs the forward on it, and
// the output rows go back, Y[perm[i]] = Yp[i]: written to their places by the tensor-core attention kernel itself, by
// a second pass behind the CUDA-core one.  The gather is independent of the key assignment and runs beside it.
#include "avq_internal.h"
#include "avq_tc_common.cuh"

namespace avq {
namespace {

// Rows of `row_vec` 16-byte vectors (at most 64), one (batch, head) per grid row.  gather: dst[i] = src[perm[i]];
// scatter: dst[perm[i]] = src[i].  An index outside [0, N) is flagged; its row is gathered as zeros and not scattered
// at all.  HBM bound; neighbouring threads take neighbouring vectors and a thread has kPermBatch of them in flight
// (one warp per row left most lanes idle: B2 H16 N4096 d64 21 us a pass).
constexpr int kPermThreads = 256, kPermBatch = 4;
__global__ void __launch_bounds__(kPermThreads)
permute_rows_kernel(uint4* __restrict__ dst, const uint4* __restrict__ src, const int32_t* __restrict__ perm,
                    int N, int row_vec, int scatter, int32_t* status_word) {
  tc::pdl_launch_dependents();
  const int per = kPermThreads / row_vec;                // rows a pass of the CTA covers
  const int rr = threadIdx.x / row_vec, v = threadIdx.x - rr * row_vec;
  if (rr >= per) return;
  const long long base = (long long)blockIdx.y * N;
  const long long i0 = (long long)blockIdx.x * per * kPermBatch + rr;
  int j[kPermBatch];
#pragma unroll
  for (int t = 0; t < kPermBatch; ++t) j[t] = i0 + (long long)t * per < N ? __ldg(perm + i0 + (long long)t * per) : -1;
  uint4 x[kPermBatch];
#pragma unroll
  for (int t = 0; t < kPermBatch; ++t) {
    const long long i = i0 + (long long)t * per;
    x[t] = make_uint4(0u, 0u, 0u, 0u);
    if (i < N && j[t] >= 0 && j[t] < N) x[t] = src[(base + (scatter ? i : j[t])) * row_vec + v];
  }
#pragma unroll
  for (int t = 0; t < kPermBatch; ++t) {
    const long long i = i0 + (long long)t * per;
    if (i >= N) continue;
    const bool ok = j[t] >= 0 && j[t] < N;
    if (!ok && v == 0 && status_word) atomicCAS(status_word, 0, DEV_BAD_INDEX);
    if (!scatter) dst[(base + i) * row_vec + v] = x[t];  // the tile needs a defined query row even for a bad index
    else if (ok) dst[(base + j[t]) * row_vec + v] = x[t];
  }
}

avq_status permute_rows(void* dst, const void* src, const int32_t* perm, const avq_problem& p, bool scatter,
                        int32_t* status_word, cudaStream_t st) {
  const size_t es = p.dtype == AVQ_F32 ? 4 : 2;
  const int row_vec = (int)(p.d * es / 16);
  const int rows = kPermThreads / row_vec * kPermBatch;
  const dim3 grid((unsigned)((p.Nq + rows - 1) / rows), (unsigned)(p.B * p.H));
  permute_rows_kernel<<<grid, kPermThreads, 0, st>>>(static_cast<uint4*>(dst), static_cast<const uint4*>(src), perm,
                                                     p.Nq, row_vec, scatter ? 1 : 0, status_word);
  return cuda_ok(cudaGetLastError());
}

inline size_t align256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace
}  // namespace avq

using namespace avq;

extern "C" {

size_t avq_workspace_bytes_permuted(const avq_problem* prob, int32_t P, int32_t block_q) {
  const size_t base = avq_workspace_bytes(prob, P, block_q);
  if (base == 0) return 0;
  const size_t es = prob->dtype == AVQ_F32 ? 4 : 2;
  if ((prob->d * es) % 16 != 0) return 0;
  const size_t qb = align256(es * (size_t)prob->B * prob->H * prob->Nq * prob->d);
  return align256(base) + 2 * qb;
}

avq_status avq_forward_permuted(const avq_problem* prob, const void* Q, const void* K, const void* V,
                                const void* Cp, const void* Cc, int32_t P, int32_t block_q,
                                const int32_t* perm, void* Y, int32_t* topp_out, float* importance_out,
                                void* workspace, size_t workspace_bytes, void* stream) {
  avq_status s = validate_forward(prob, P, block_q);
  if (s != AVQ_OK) return s;
  if (!perm || !Q || !Y) return AVQ_ERR_NULL;
  if (reinterpret_cast<uintptr_t>(perm) & 3u) return AVQ_ERR_ALIGN;
  const size_t es = prob->dtype == AVQ_F32 ? 4 : 2;
  if ((prob->d * es) % 16 != 0) return AVQ_ERR_UNSUPPORTED;
  if (!workspace) return AVQ_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(workspace) & 255u) return AVQ_ERR_ALIGN;
  const size_t need = avq_workspace_bytes_permuted(prob, P, block_q);
  if (need == 0 || workspace_bytes < need) return AVQ_ERR_WORKSPACE;
  const size_t base = align256(avq_workspace_bytes(prob, P, block_q));
  const size_t qb = align256(es * (size_t)prob->B * prob->H * prob->Nq * prob->d);
  char* ws = static_cast<char*>(workspace);
  void* Qp = ws + base;
  void* Yp = ws + base + qb;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (!K || !V || !Cp || !Cc) return AVQ_ERR_NULL;
  for (const void* a : {Q, K, V, Cp, Cc, (const void*)Y, (const void*)topp_out, (const void*)importance_out})
    if (reinterpret_cast<uintptr_t>(a) & 15u) return AVQ_ERR_ALIGN;
  // the forward clears the status header at offset 0, so an index flagged by the gather would be lost: the gather
  // runs without a status word, the write-back (same indices) reports
  s = permute_rows(Qp, Q, perm, *prob, false, nullptr, st);
  if (s != AVQ_OK) return s;
  const Layout L = make_layout(*prob, P, block_q);
  if (use_tensor_path(*prob))
    return forward_core(*prob, Qp, K, V, Cp, Cc, P, block_q, Y, topp_out, importance_out, workspace, L, perm, st);
  s = forward_core(*prob, Qp, K, V, Cp, Cc, P, block_q, Yp, topp_out, importance_out, workspace, L, nullptr, st);
  if (s != AVQ_OK) return s;
  return permute_rows(Y, Yp, perm, *prob, true, static_cast<int32_t*>(workspace), st);
}

}  // extern "C"
