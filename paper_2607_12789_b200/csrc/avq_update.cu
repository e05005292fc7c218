// avq_codebook_update: one training-time update of the hierarchical codebook from a batch of keys
// (appendix "Codeword Clustering During Training").
//
// The data-parallel part reuses the forward's own kernels: the assignment gives every key its parent and
// child under the current codebooks, and the aggregation kernels, fed the KEYS as values, give the
// per-(batch, head) key sums and counts of every child (and of every parent: on the tensor-core path only the part
// that stays with it, the rest is the sum of its children).  ema_project_kernel then folds the
// batch into the per-head EMA statistics, moves each parent to its EMA mean, and places the children at
// the mass-weighted projection of their EMA means onto  mean_c C_{p,c} = C_p
// (Eq. "child_constraint_solve").
#include <cuda_bf16.h>

#include "avq_internal.h"
#include "avq_tc_common.cuh"

namespace avq {
namespace {

constexpr float kMassFloor = 1e-6f;   // a code without EMA mass keeps its position and absorbs the residual

template <typename T> __device__ __forceinline__ float ld_code(const T* p);
template <> __device__ __forceinline__ float ld_code<float>(const float* p) { return *p; }
template <> __device__ __forceinline__ float ld_code<__nv_bfloat16>(const __nv_bfloat16* p) { return __bfloat162float(*p); }
template <typename T> __device__ __forceinline__ void st_code(T* p, float v);
template <> __device__ __forceinline__ void st_code<float>(float* p, float v) { *p = v; }
template <> __device__ __forceinline__ void st_code<__nv_bfloat16>(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

// four consecutive floats of the caller's statistics, which need not be 16-byte aligned
__device__ __forceinline__ float4 ld_stat4(const float* p, bool aligned) {
  if (aligned) return *reinterpret_cast<const float4*>(p);
  return make_float4(p[0], p[1], p[2], p[3]);
}
__device__ __forceinline__ void st_stat4(float* p, const float4& v, bool aligned) {
  if (aligned) *reinterpret_cast<float4*>(p) = v;
  else { p[0] = v.x; p[1] = v.y; p[2] = v.z; p[3] = v.w; }
}

// A thread owns four head dimensions of one (head, parent) with all its children; d / 4 threads per parent, as many
// parents per CTA as fit.  Kp [B,H,M,d], np [B,H,M], Kc [B,H,M,C,d], nc [B,H,M,C]: this batch's key sums and counts
// (leaves: Kp and np hold only the keys that stay with their parent).  CM: children held in registers, C <= CM.
// The kernel is a load round trip and a little arithmetic: the caller's statistics are loaded ahead of the dependency
// wait, the batch's sums in one go behind it (B2 H16 M128 C8 d64: 30.5 us with a thread per dimension and one load at a
// time; 10.8 now, both with cold caches).
constexpr int kEmaThreads = 128;
template <typename T, int CM>
__global__ void __launch_bounds__(kEmaThreads)
ema_project_kernel(const float* Kp, const float* np_, const float* Kc, const float* nc, const T* __restrict__ Cp,
                   const T* __restrict__ Cc, float* Sp, float* Np, float* Sc, float* Nc, T* __restrict__ Cp_out,
                   T* __restrict__ Cc_out, int B, int H, int M, int C, int d, float decay, int leaves, int aligned) {
  const int lanes = d >> 2, per = kEmaThreads / lanes;
  const int mm = threadIdx.x / lanes, k = 4 * (threadIdx.x - mm * lanes);
  const int m = blockIdx.x * per + mm, h = blockIdx.y;
  const bool active = mm < per && m < M;
  const size_t hm = (size_t)h * M + (active ? m : 0);
  float4 sc[CM], sp;
  float Nn[CM], Npn;
  sp = ld_stat4(Sp + hm * d + k, aligned);
  Npn = Np[hm];
#pragma unroll
  for (int c = 0; c < CM; ++c) {
    sc[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    Nn[c] = 0.f;
    if (c < C) {
      sc[c] = ld_stat4(Sc + (hm * C + c) * d + k, aligned);
      Nn[c] = Nc[hm * C + c];
    }
  }
  tc::pdl_wait();                                        // the batch's sums come from the kernel before
  const float g = 1.f - decay;
  float4 ks[CM], kp = make_float4(0.f, 0.f, 0.f, 0.f);
  float n[CM], npar = 0.f;
#pragma unroll
  for (int c = 0; c < CM; ++c) { ks[c] = make_float4(0.f, 0.f, 0.f, 0.f); n[c] = 0.f; }
  for (int b = 0; b < B; ++b) {
    const size_t bhm = ((size_t)b * H + h) * M + (active ? m : 0);
    float4 x[CM];
    float y[CM];
    const float4 xp = tc::ld_after_wait(reinterpret_cast<const float4*>(Kp + bhm * d + k));
    const float yp = tc::ld_after_wait(np_ + bhm);
#pragma unroll
    for (int c = 0; c < CM; ++c)
      if (c < C) {
        x[c] = tc::ld_after_wait(reinterpret_cast<const float4*>(Kc + (bhm * C + c) * d + k));
        y[c] = tc::ld_after_wait(nc + bhm * C + c);
      }
    float4 sum = xp;
    float cnt = yp;
#pragma unroll
    for (int c = 0; c < CM; ++c)
      if (c < C) {
        ks[c].x += x[c].x; ks[c].y += x[c].y; ks[c].z += x[c].z; ks[c].w += x[c].w;
        n[c] += y[c];
        if (leaves) {
          sum.x += x[c].x; sum.y += x[c].y; sum.z += x[c].z; sum.w += x[c].w;
          cnt += y[c];
        }
      }
    kp.x += sum.x; kp.y += sum.y; kp.z += sum.z; kp.w += sum.w;
    npar += cnt;
  }
  __syncthreads();                                       // every thread has read its parent's counts
  if (!active) return;
  float sigma = 0.f;
  Npn = decay * Npn + g * npar;
#pragma unroll
  for (int c = 0; c < CM; ++c)
    if (c < C) {
      Nn[c] = decay * Nn[c] + g * n[c];
      sigma += 1.f / fmaxf(Nn[c], kMassFloor);
    }
  if (k == 0) {
    Np[hm] = Npn;
#pragma unroll
    for (int c = 0; c < CM; ++c)
      if (c < C) Nc[hm * C + c] = Nn[c];
  }
  sp = make_float4(decay * sp.x + g * kp.x, decay * sp.y + g * kp.y, decay * sp.z + g * kp.z, decay * sp.w + g * kp.w);
  st_stat4(Sp + hm * d + k, sp, aligned);
  const float* spv = reinterpret_cast<const float*>(&sp);
  float cp[4], delta[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    cp[e] = Npn > kMassFloor ? spv[e] / Npn : ld_code(Cp + hm * d + k + e);
    st_code(Cp_out + hm * d + k + e, cp[e]);
    delta[e] = -(float)C * cp[e];
  }
#pragma unroll
  for (int c = 0; c < CM; ++c)
    if (c < C) {
      const size_t i = (hm * C + c) * d + k;
      float4 v = make_float4(decay * sc[c].x + g * ks[c].x, decay * sc[c].y + g * ks[c].y, decay * sc[c].z + g * ks[c].z,
                             decay * sc[c].w + g * ks[c].w);
      st_stat4(Sc + i, v, aligned);
      float* mv = reinterpret_cast<float*>(&v);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        mv[e] = Nn[c] > kMassFloor ? mv[e] / Nn[c] : ld_code(Cc + i + e);
        delta[e] += mv[e];
      }
      sc[c] = v;                                         // the EMA mean
    }
#pragma unroll
  for (int c = 0; c < CM; ++c)
    if (c < C) {
      const float wgt = fmaxf(Nn[c], kMassFloor) * sigma;
      const float mv[4] = {sc[c].x, sc[c].y, sc[c].z, sc[c].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) st_code(Cc_out + (hm * C + c) * d + k + e, mv[e] - delta[e] / wgt);
    }
}

template <typename T>
avq_status ema_project(const avq_problem& p, const float* Kp, const float* np_, const float* Kc, const float* nc,
                       const void* Cp, const void* Cc, float decay, float* Sp, float* Np, float* Sc, float* Nc,
                       void* Cp_out, void* Cc_out, bool leaves, cudaStream_t st) {
  const int per = kEmaThreads / (p.d / 4);
  const dim3 grid((unsigned)((p.M + per - 1) / per), (unsigned)p.H);
  const int aligned = ((reinterpret_cast<uintptr_t>(Sp) | reinterpret_cast<uintptr_t>(Sc)) & 15u) == 0;
  auto kern = p.C <= 4 ? ema_project_kernel<T, 4> : (p.C <= 8 ? ema_project_kernel<T, 8> : ema_project_kernel<T, 16>);
  return cuda_ok(tc::launch_pdl(kern, grid, dim3(kEmaThreads), 0, st, true, Kp, np_, Kc, nc, static_cast<const T*>(Cp),
                                static_cast<const T*>(Cc), Sp, Np, Sc, Nc, static_cast<T*>(Cp_out),
                                static_cast<T*>(Cc_out), p.B, p.H, p.M, p.C, p.d, decay, leaves ? 1 : 0, aligned));
}

struct UpdateLayout {
  size_t pidx, cidx, Kc, nc, Kp, np, total;             // Kc .. np adjacent: the assign grid clears them in one pass
};
UpdateLayout update_layout(const avq_problem& p) {
  UpdateLayout L;
  const size_t BH = (size_t)p.B * p.H;
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off = (off + bytes + 255) / 256 * 256; return o; };
  L.pidx = take(4 * BH * p.Nk);
  L.cidx = take(4 * BH * p.Nk);
  L.Kc = take(4 * BH * p.M * p.C * p.d);
  L.nc = take(4 * BH * p.M * p.C);
  L.Kp = take(4 * BH * p.M * p.d);
  L.np = take(4 * BH * p.M);
  L.total = off;
  return L;
}

}  // namespace
}  // namespace avq

using namespace avq;

extern "C" {

size_t avq_codebook_update_workspace_bytes(const avq_problem* prob) {
  if (validate_problem(prob) != AVQ_OK) return 0;
  return update_layout(*prob).total;
}

avq_status avq_codebook_update(const avq_problem* prob, const void* K, const void* Cp, const void* Cc, float decay,
                               float* Sp, float* Np, float* Sc, float* Nc, void* Cp_out, void* Cc_out,
                               void* workspace, size_t workspace_bytes, void* stream) {
  avq_status s = validate_problem(prob);
  if (s != AVQ_OK) return s;
  if (!(decay >= 0.f && decay <= 1.f)) return AVQ_ERR_SHAPE;
  if (prob->C > 16) return AVQ_ERR_UNSUPPORTED;
  if (!K || !Cp || !Cc || !Sp || !Np || !Sc || !Nc || !Cp_out || !Cc_out) return AVQ_ERR_NULL;
  if (!workspace) return AVQ_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(workspace) & 255u) return AVQ_ERR_ALIGN;
  const UpdateLayout L = update_layout(*prob);
  if (workspace_bytes < L.total) return AVQ_ERR_WORKSPACE;
  char* ws = static_cast<char*>(workspace);
  int32_t* pidx = reinterpret_cast<int32_t*>(ws + L.pidx);
  int32_t* cidx = reinterpret_cast<int32_t*>(ws + L.cidx);
  float* Kp = reinterpret_cast<float*>(ws + L.Kp);
  float* np_ = reinterpret_cast<float*>(ws + L.np);
  float* Kc = reinterpret_cast<float*>(ws + L.Kc);
  float* nc = reinterpret_cast<float*>(ws + L.nc);
  // the keys' assignment under the current codebooks, then their sums and counts per codeword
  for (const void* a : {K, Cp, Cc})
    if (reinterpret_cast<uintptr_t>(a) & 15u) return AVQ_ERR_ALIGN;
  const avq_problem& p = *prob;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const bool tensor = use_tensor_path(p);
  if (tensor) {
    s = tc_assign(p, K, Cp, Cc, pidx, cidx, nullptr, ws + L.Kc, L.total - L.Kc, nullptr, false, st);
    if (s == AVQ_OK)
      s = tc_aggregate(p, K, pidx, cidx, Kp, np_, Kc, nc, nullptr, nullptr, nullptr, nullptr, true, true, nullptr, st);
  } else {
    s = simt_assign(p, K, Cp, Cc, pidx, cidx, ws + L.Kc, L.total - L.Kc, st);
    if (s == AVQ_OK) s = simt_aggregate(p, K, pidx, cidx, Kp, np_, Kc, nc, true, nullptr, st);
  }
  if (s != AVQ_OK) return s;
  return p.dtype == AVQ_F32
             ? ema_project<float>(p, Kp, np_, Kc, nc, Cp, Cc, decay, Sp, Np, Sc, Nc, Cp_out, Cc_out, tensor, st)
             : ema_project<__nv_bfloat16>(p, Kp, np_, Kc, nc, Cp, Cc, decay, Sp, Np, Sc, Nc, Cp_out, Cc_out, tensor, st);
}

}  // extern "C"
