// CUDA-core (FFMA) kernels for the three stages of the AVQ-attention forward.
// They carry the float32 path (tensor-core inputs are 16-bit, too coarse for a 1e-4
// output tolerance) and any shape outside the tensor-core envelope, for either dtype.
//
//   assign_simt_kernel     Algorithm 1, parent and child argmin, a tile of 64 keys per CTA
//   aggregate_simt_kernel  Eq. "aggregates": value sums and counts, one warp per 4 keys
//   attend_simt_kernel     Algorithm 2 in its masked form: parent pass, Eq. "importance",
//                          top-P, then one softmax over {unrefined parents} U {children of the
//                          refined parents} with the maximum taken over non-empty codewords
//
// The products (distances, logits, weighted value sums) are register-tiled: both operands of a product are
// staged in shared memory as [contraction index][row or column], a thread keeps an RT x 4 block of results and
// reads RT + 4 operands per step with 16-byte loads.  The logits of bfloat16 inputs are warp-level tensor-core products
// (exact products, float32 sums, as on the FFMA path); everything behind them stays float32.
#include <cuda_bf16.h>
#include <math.h>

#include <type_traits>

#include "avq_internal.h"
#include "avq_select.cuh"
#include "avq_tc_common.cuh"

namespace avq {
namespace {

using tc::ld_after_wait;

template <typename T> __device__ __forceinline__ float ldf(const T* p);
template <> __device__ __forceinline__ float ldf<float>(const float* p) { return __ldg(p); }
template <> __device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16* p) {
  return __bfloat162float(*p);
}
// four consecutive elements (d % 4 == 0 and 16-byte aligned bases: 16 bytes of float, 8 of bfloat16)
__device__ __forceinline__ float4 ld4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p) {
  const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                     __uint_as_float(u.y & 0xFFFF0000u));
}
__device__ __forceinline__ void st4(float* p, const float4& v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void st4(__nv_bfloat16* p, const float4& v) {
  __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
  uint2 u;
  u.x = *reinterpret_cast<uint32_t*>(&lo);
  u.y = *reinterpret_cast<uint32_t*>(&hi);
  *reinterpret_cast<uint2*>(p) = u;
}

constexpr int kThreads = 256;      // of the assign and aggregate kernels: 16 x 16, thread (ty, tx) owns rows ty*4, columns tx*4
constexpr int kCols = 64;          // columns (codewords) of a tile
constexpr int kLdC = kCols + 4;    // row pitch of a [k][column] operand, floats

// The columns of a tile of n <= 64 codewords: thread tx owns tx, tx + 16, tx + 32, tx + 48, which stand side by side in
// the shared-memory operand, so that a narrow tile costs only the columns it has.
__device__ __forceinline__ int code_pos(int c) { return ((c & 15) << 2) | (c >> 4); }

// Copies `rows` rows of d elements (row r at src(r), nullptr = zeros) into dst[k][place(r)], k < d: the transposed
// operand of the register-tiled products.  A warp takes 8 rows x 4 chunks of 4 elements: 64-byte pieces of a
// row in global memory, at most two-way bank conflicts in shared memory.
template <int THREADS, int BATCH, typename Place, typename Src>
__device__ __forceinline__ void load_transposed(float* dst, int ld, int rows, int d, Place place, Src src) {
  constexpr int kWarps = THREADS / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int kc = lane & 3, rr = lane >> 2;
  const int chunks = d >> 2, cblocks = (chunks + 3) >> 2, units = (rows >> 3) * cblocks;
  for (int u = warp; u < units; u += BATCH * kWarps) {    // BATCH loads in flight per trip
    float4 v[BATCH];
    int at[BATCH];
#pragma unroll
    for (int e = 0; e < BATCH; ++e) {
      const int ue = u + e * kWarps, rb = ue / cblocks, cb = ue - rb * cblocks;
      const int r = rb * 8 + rr, c = cb * 4 + kc;
      at[e] = -1;
      v[e] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (ue < units && c < chunks) {
        at[e] = 4 * c * ld + place(r);
        const auto* p = src(r);
        if (p) v[e] = ld4(p + 4 * c);
      }
    }
#pragma unroll
    for (int e = 0; e < BATCH; ++e)
      if (at[e] >= 0) {
        float* o = dst + at[e];
        o[0] = v[e].x; o[ld] = v[e].y; o[2 * ld] = v[e].z; o[3 * ld] = v[e].w;
      }
  }
}

// acc[i][j] += sum_k A[k][ty*RT + i] * B[k][tx*4 + j], j < NJ, k ascending (one accumulator per result: the sums do
// not depend on the tiling)
// With four columns two of them share an instruction (the same rounding; M512 P64 d64, 4096 queries: whole call 203 ->
// 197 us): the loop is short of issue slots next to its shared-memory loads.
template <int RT, int NJ>
__device__ __forceinline__ void mul_tile(float (&acc)[RT][4], const float* A, int lda, const float* B, int ldb, int K,
                                         int ty, int tx) {
  const float* a_ = A + ty * RT;
  const float* b_ = B + tx * 4;
  tc::f32x2 p[RT][2];                                      // NJ == 4: packed pairs of columns
  if constexpr (NJ == 4) {
#pragma unroll
    for (int i = 0; i < RT; ++i) { p[i][0] = tc::pack2(acc[i][0], acc[i][1]); p[i][1] = tc::pack2(acc[i][2], acc[i][3]); }
  }
#pragma unroll 4
  for (int k = 0; k < K; ++k) {
    float a[RT], b[4];
    if constexpr (RT == 4) *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(a_ + k * lda);
    else *reinterpret_cast<float2*>(a) = *reinterpret_cast<const float2*>(a_ + k * lda);
    if constexpr (NJ == 4) *reinterpret_cast<float4*>(b) = *reinterpret_cast<const float4*>(b_ + k * ldb);
    else if constexpr (NJ == 2) *reinterpret_cast<float2*>(b) = *reinterpret_cast<const float2*>(b_ + k * ldb);
    else b[0] = b_[k * ldb];
    if constexpr (NJ == 4) {
      const tc::f32x2 b01 = tc::pack2(b[0], b[1]), b23 = tc::pack2(b[2], b[3]);
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const tc::f32x2 aa = tc::pack2(a[i], a[i]);
        p[i][0] = tc::fma2(aa, b01, p[i][0]);
        p[i][1] = tc::fma2(aa, b23, p[i][1]);
      }
    } else {
#pragma unroll
      for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
  }
  if constexpr (NJ == 4) {
#pragma unroll
    for (int i = 0; i < RT; ++i) { tc::unpack2(p[i][0], acc[i][0], acc[i][1]); tc::unpack2(p[i][1], acc[i][2], acc[i][3]); }
  }
}
template <int RT>
__device__ __forceinline__ void mul_codes(float (&acc)[RT][4], const float* A, int lda, const float* B, int ldb, int K,
                                          int ty, int tx, int n) {
  if (n <= 16) mul_tile<RT, 1>(acc, A, lda, B, ldb, K, ty, tx);
  else if (n <= 32) mul_tile<RT, 2>(acc, A, lda, B, ldb, K, ty, tx);
  else mul_tile<RT, 4>(acc, A, lda, B, ldb, K, ty, tx);
}
__device__ __forceinline__ int code_rows(int n) { return n <= 16 ? 16 : (n <= 32 ? 32 : 64); }

// Two distances closer than this (relative) are re-evaluated in float64.  The float32 direct
// form carries about d * 2^-24 relative error, far below it.
constexpr float kNearTie = 1e-4f;

template <typename T>
__device__ double exact_dist(const T* krow, const T* c, int d) {
  double s = 0.0;
  for (int k = 0; k < d; ++k) {
    double t = (double)ldf(krow + k) - (double)ldf(c + k);
    s += t * t;
  }
  return s;
}

// `rows` rows of d bfloat16 (row r at src(r), nullptr = zeros) into dst[r][k], k < dpad, zeros from d on.
template <int THREADS, typename Src>
__device__ __forceinline__ void load_rows(__nv_bfloat16* dst, int pitch, int rows, int d, int dpad, Src src) {
  const int per = dpad >> 2, units = rows * per;
  for (int u = threadIdx.x; u < units; u += 2 * THREADS) {
    uint2 v[2];
    int at[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int ue = u + e * THREADS, r = ue / per, c = ue - r * per;
      at[e] = ue < units ? r * pitch + 4 * c : -1;
      v[e] = make_uint2(0u, 0u);
      if (ue < units && 4 * c < d) {
        const __nv_bfloat16* p = src(r);
        if (p) v[e] = __ldg(reinterpret_cast<const uint2*>(p + 4 * c));
      }
    }
#pragma unroll
    for (int e = 0; e < 2; ++e)
      if (at[e] >= 0) *reinterpret_cast<uint2*>(dst + at[e]) = v[e];
  }
}
// The same asynchronously (cp.async; the caller waits), each row in pieces of 16 bytes (8 where d is no multiple of 8).
template <int THREADS, int PIECE, typename Src>
__device__ __forceinline__ void load_rows_async(__nv_bfloat16* dst, int pitch, int rows, int d, int dpad, Src src) {
  const int per = dpad / PIECE, step_r = THREADS / per, step_c = THREADS - step_r * per;
  int r = threadIdx.x / per, c = threadIdx.x - r * per;
  for (; r < rows; r += step_r, c += step_c) {
    if (c >= per) { c -= per; if (++r >= rows) break; }
    const __nv_bfloat16* p = src(r);
    const bool there = p != nullptr && PIECE * c < d;
    const uint32_t to = tc::smem_u32(dst + r * pitch + PIECE * c);
    const __nv_bfloat16* from = there ? p + PIECE * c : src(0);
    if constexpr (PIECE == 8)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(from), "r"(there ? 16 : 0) : "memory");
    else
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(to), "l"(from), "r"(there ? 8 : 0) : "memory");
  }
}
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], const __nv_bfloat16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(tc::smem_u32(p)) : "memory");
}
// One warp: s[column][row] = scale * q . c^T for rows r0 .. +15 and columns n0 .. +8 NT - 1
template <int NT>
__device__ __forceinline__ void mma_block(float* s, int ldr, const __nv_bfloat16* q, const __nv_bfloat16* c, int pitch,
                                          int dpad, float scale, int r0, int n0) {
  const int lane = threadIdx.x & 31;
  const __nv_bfloat16* ap = q + (r0 + (lane & 15)) * pitch + (lane >> 4) * 8;
  const __nv_bfloat16* bp = c + (n0 + (lane & 7) + ((lane >> 4) << 3)) * pitch + ((lane >> 3) & 1) * 8;
  float acc[NT][4] = {};
#pragma unroll 4
  for (int k = 0; k < dpad; k += 16) {
    uint32_t a[4];
    ldmatrix4(a, ap + k);
#pragma unroll
    for (int j = 0; j < NT; j += 2) {
      uint32_t b[4];
      ldmatrix4(b, bp + j * 8 * pitch + k);
#pragma unroll
      for (int e = 0; e < 2; ++e)
        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                     : "+f"(acc[j + e][0]), "+f"(acc[j + e][1]), "+f"(acc[j + e][2]), "+f"(acc[j + e][3])
                     : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[2 * e]), "r"(b[2 * e + 1]));
    }
  }
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int j = 0; j < NT; ++j)
#pragma unroll
    for (int e = 0; e < 4; ++e)
      s[(size_t)(n0 + 8 * j + 2 * t + (e & 1)) * ldr + r0 + g + 8 * (e >> 1)] = acc[j][e] * scale;
}

// ------------------------------------------------------------------------------- assign
constexpr int kAssignKeys = 64;    // keys per CTA

// bfloat16: the next tile of codewords is copied while one is used, as long as that leaves two CTAs on an SM (H4 N4096 M512, this
// kernel, us, waiting for each tile and copying ahead: d128 43.9 and 39.3, d256 68.6 and 82.9).
__host__ __device__ inline bool assign_two_tiles(int d) { return d <= 192; }
// Shared memory: float32, keys and codewords as [k][row]; bfloat16, both as rows, two tiles of codewords, and the products
// [column][key]; norms.
__host__ __device__ inline size_t assign_smem_floats(int d, bool mma) {
  if (!mma) return 2 * (size_t)d * kLdC + kAssignKeys + kCols;
  return (assign_two_tiles(d) ? 3 : 2) * (size_t)kAssignKeys * ((size_t)(d + 15) / 16 * 8 + 4) + (size_t)kCols * kLdC + kAssignKeys + kCols;
}

// Parents: 64 keys x 64 codewords at a time, ||k||^2 + ||c||^2 - 2 k.c with float64 rechecks; bfloat16 products on the
// tensor cores (M512 d64, 16384 keys: 74 us with float32 multiply-adds).  Children: four lanes per key,
// direct form.  zero_base / zero_units: 16-byte words this grid clears on the side (the accumulators of the
// aggregation behind it), each CTA a slice of zero_per.
template <typename T>
__global__ void __launch_bounds__(kThreads, 2)
assign_simt_kernel(const T* __restrict__ K, const T* __restrict__ Cp, const T* __restrict__ Cc,
                   int32_t* __restrict__ pidx, int32_t* __restrict__ cidx, int H, int Nk, int d, int M,
                   int C, int parent_stays, uint4* __restrict__ zero_base, size_t zero_units, size_t zero_per) {
  extern __shared__ __align__(16) float smem[];
  constexpr bool kMma = std::is_same<T, __nv_bfloat16>::value;
  const int dpad = (d + 15) & ~15, pitch = dpad + 8;
  float* ks = smem;                                               // [d][kLdC] keys, or rows of pitch bfloat16
  float* cs = ks + (kMma ? (size_t)kAssignKeys * pitch / 2 : (size_t)d * kLdC);   // codewords of the current tile, alike
  const bool two = kMma && assign_two_tiles(d);
  float* cs_next = two ? cs + (size_t)kCols * pitch / 2 : cs;     // bfloat16: of the tile behind it, on their way
  float* prod = cs_next + (size_t)kCols * pitch / 2;              // bfloat16: [kCols][kLdC] products
  float* kn = kMma ? prod + (size_t)kCols * kLdC : cs + (size_t)d * kLdC;   // [kAssignKeys] key norms
  float* cn = kn + kAssignKeys;                                   // [kCols] codeword norms (float32: by code_pos)
  __shared__ int s_par[kAssignKeys];
  __shared__ int s_redo[kAssignKeys];          // 1: parent decided in float64 (its exact distance in s_dp)
  __shared__ double s_dp[kAssignKeys];
  tc::pdl_launch_dependents();
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int bh = blockIdx.y, h = bh % H;
  const int j0 = blockIdx.x * kAssignKeys;
  if (zero_units) {
    const size_t u0 = ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * zero_per, u1 = min(zero_units, u0 + zero_per);
    for (size_t u = u0 + tid; u < u1; u += kThreads) zero_base[u] = make_uint4(0u, 0u, 0u, 0u);
  }
  const T* Kb = K + ((size_t)bh * Nk + j0) * d;
  const int rows = min(kAssignKeys, Nk - j0);
  const T* Cph = Cp + (size_t)h * M * d;
  auto key_row = [&](int r) { return r < rows ? Kb + (size_t)r * d : (const T*)nullptr; };
  auto load_codes = [&](float* to, int m0) {              // bfloat16: a tile of codewords, not waited for
    const int w = min(kCols, M - m0);
    auto row = [&](int r) {
      return r < w ? reinterpret_cast<const __nv_bfloat16*>(Cph) + (size_t)(m0 + r) * d : (const __nv_bfloat16*)nullptr;
    };
    if (d % 8 == 0) load_rows_async<kThreads, 8>(reinterpret_cast<__nv_bfloat16*>(to), pitch, kCols, d, dpad, row);
    else load_rows_async<kThreads, 4>(reinterpret_cast<__nv_bfloat16*>(to), pitch, kCols, d, dpad, row);
  };
  if constexpr (kMma) {
    load_codes(cs, 0);
    load_rows<kThreads>(reinterpret_cast<T*>(ks), pitch, kAssignKeys, d, dpad, key_row);
  } else {                                                // the keys and the first codewords in one go (cs is behind ks)
    const int w = min(kCols, M);
    load_transposed<kThreads, 8>(ks, kLdC, kAssignKeys + code_rows(w), d,
                                 [&](int r) { return r < kAssignKeys ? r : d * kLdC + code_pos(r - kAssignKeys); },
                                 [&](int r) {
                                   if (r < kAssignKeys) return key_row(r);
                                   return r - kAssignKeys < w ? Cph + (size_t)(r - kAssignKeys) * d : (const T*)nullptr;
                                 });
  }
  // squared norm of a staged row (float32: column), four lanes per row (row tid / 4)
  auto row_norm = [&](const float* base) {
    float s = 0.f;
    if constexpr (kMma) {
      const T* rowp = reinterpret_cast<const T*>(base) + (tid >> 2) * pitch;
      for (int k = 4 * (tid & 3); k < dpad; k += 16) {
        const uint2 u = *reinterpret_cast<const uint2*>(rowp + k);
        const float a = __uint_as_float(u.x << 16), b = __uint_as_float(u.x & 0xFFFF0000u);
        const float c = __uint_as_float(u.y << 16), e = __uint_as_float(u.y & 0xFFFF0000u);
        s = fmaf(a, a, s); s = fmaf(b, b, s); s = fmaf(c, c, s); s = fmaf(e, e, s);
      }
    } else {
#pragma unroll 4
      for (int k = tid & 3; k < d; k += 4) {
        const float x = base[(size_t)k * kLdC + (tid >> 2)];
        s = fmaf(x, x, s);
      }
    }
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    return s + __shfl_xor_sync(0xffffffffu, s, 2);
  };

  float d1[4], d2[4];
  int i1[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) { d1[i] = INFINITY; d2[i] = INFINITY; i1[i] = 0; }
  for (int m0 = 0; m0 < M; m0 += kCols) {
    const int w = min(kCols, M - m0);
    if (!kMma && m0 > 0) __syncthreads();
    if constexpr (kMma) {
      if (m0 > 0) {
        if (two) { float* t = cs; cs = cs_next; cs_next = t; }
        else { __syncthreads(); load_codes(cs, m0); }
      }
      tc::cp_async_wait_all();
      __syncthreads();
      if (two && m0 + kCols < M) load_codes(cs_next, m0 + kCols);   // (the tile before has been read)
    } else {
      if (m0 > 0)
        load_transposed<kThreads, 4>(cs, kLdC, code_rows(w), d, [](int r) { return code_pos(r); },
                                     [&](int r) { return r < w ? Cph + (size_t)(m0 + r) * d : (const T*)nullptr; });
      __syncthreads();
    }
    float acc[4][4] = {};
    if (m0 == 0) {
      const float s = row_norm(ks);
      if ((tid & 3) == 0) kn[tid >> 2] = s;
    }
    {
      const float s = row_norm(cs);
      if ((tid & 3) == 0) cn[tid >> 2] = s;
    }
    if constexpr (kMma) {
      const int warp = tid >> 5;
      mma_block<4>(prod, kLdC, reinterpret_cast<const T*>(ks), reinterpret_cast<const T*>(cs), pitch, dpad, 1.f,
                   (warp & 3) * 16, (warp >> 2) * 32);
      __syncthreads();
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 x = *reinterpret_cast<const float4*>(prod + (tx + 16 * j) * kLdC + ty * 4);
        acc[0][j] = x.x; acc[1][j] = x.y; acc[2][j] = x.z; acc[3][j] = x.w;
      }
    } else {
      mul_codes<4>(acc, ks, kLdC, cs, kLdC, d, ty, tx, w);
      __syncthreads();
    }
    {
      const float4 k4 = *reinterpret_cast<const float4*>(kn + ty * 4);
      const float kv[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float c = cn[kMma ? tx + 16 * j : tx * 4 + j];
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i][j] = fmaf(-2.f, acc[i][j], kv[i] + c);
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (tx + 16 * j < w) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float s = acc[i][j];
          if (s < d1[i]) { d2[i] = d1[i]; d1[i] = s; i1[i] = m0 + tx + 16 * j; }
          else if (s < d2[i]) { d2[i] = s; }
        }
      }
  }
  // ---- merge the 16 threads of a key (the lower index wins a tie); near-ties are redone in float64 by them
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
      const float b1 = __shfl_xor_sync(0xffffffffu, d1[i], o), b2 = __shfl_xor_sync(0xffffffffu, d2[i], o);
      const int bi = __shfl_xor_sync(0xffffffffu, i1[i], o);
      d2[i] = fminf(fmaxf(d1[i], b1), fminf(d2[i], b2));
      if (b1 < d1[i] || (b1 == d1[i] && bi < i1[i])) { d1[i] = b1; i1[i] = bi; }
    }
    const int key = ty * 4 + i;
    // norms and products: each carries a rounding error of a small multiple of 2^-24 of the norms, which this bounds
    // with a wide margin
    const float close = 1e-4f * (kn[key] + d2[i]);
    const bool redo = M > 1 && key < rows && !(d2[i] - d1[i] > close);
    double best = INFINITY;
    if (__any_sync(0xffffffffu, redo)) {
      int bi = 0x7fffffff;
      if (redo)
        for (int m = tx; m < M; m += 16) {
          const double s = exact_dist(Kb + (size_t)key * d, Cph + (size_t)m * d, d);
          if (s < best) { best = s; bi = m; }
        }
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob < best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if (redo) { i1[i] = bi < M ? bi : 0; d1[i] = (float)best; }
    }
    if (tx == 0) {
      s_par[key] = i1[i];
      s_redo[key] = redo ? 1 : 0;
      s_dp[key] = best;
    }
  }
  __syncthreads();

  // ---- children of the key's parent: four lanes per key, each over every fourth 4-element chunk
  const int key = tid >> 2, s4 = tid & 3;
  const int par = s_par[key];
  const T* Cch = Cc + ((size_t)h * M + par) * C * d;
  // distances to nr (at most 4) codeword rows c, c + d, ..., this lane's chunks; all loads of 64 elements in flight
  auto dist_part = [&](const T* c, auto nr, int rows_there, float (&sum)[decltype(nr)::value]) {
    constexpr int N = decltype(nr)::value;
#pragma unroll
    for (int x = 0; x < N; ++x) sum[x] = 0.f;
    for (int c0 = s4; c0 < (d >> 2); c0 += 16) {
      float4 v[N][4];
#pragma unroll
      for (int x = 0; x < N; ++x)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (x < rows_there && c0 + 4 * e < (d >> 2)) v[x][e] = ld4(c + (size_t)x * d + 4 * (c0 + 4 * e));
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (c0 + 4 * e < (d >> 2)) {
          const int k = 4 * (c0 + 4 * e);
          float4 kv;
          if constexpr (kMma) {
            const uint2 u = *reinterpret_cast<const uint2*>(reinterpret_cast<const T*>(ks) + key * pitch + k);
            kv = make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                             __uint_as_float(u.y & 0xFFFF0000u));
          } else {
            const float* kp = ks + (size_t)k * kLdC + key;
            kv = make_float4(kp[0], kp[kLdC], kp[2 * kLdC], kp[3 * kLdC]);
          }
#pragma unroll
          for (int x = 0; x < N; ++x)
            if (x < rows_there) {
              const float4 y = make_float4(kv.x - v[x][e].x, kv.y - v[x][e].y, kv.z - v[x][e].z, kv.w - v[x][e].w);
              sum[x] = fmaf(y.x, y.x, sum[x]); sum[x] = fmaf(y.y, y.y, sum[x]);
              sum[x] = fmaf(y.z, y.z, sum[x]); sum[x] = fmaf(y.w, y.w, sum[x]);
            }
        }
    }
#pragma unroll
    for (int x = 0; x < N; ++x) {                         // the four lanes
      sum[x] += __shfl_xor_sync(0xffffffffu, sum[x], 1);
      sum[x] += __shfl_xor_sync(0xffffffffu, sum[x], 2);
    }
  };
  float e1 = INFINITY, e2 = INFINITY;
  int c1 = 0;
  for (int c = 0; c < C; c += 4) {                        // four children at a time
    float sum[4];
    dist_part(Cch + (size_t)c * d, std::integral_constant<int, 4>{}, C - c, sum);
#pragma unroll
    for (int x = 0; x < 4; ++x)
      if (c + x < C) {
        if (sum[x] < e1) { e2 = e1; e1 = sum[x]; c1 = c + x; }
        else if (sum[x] < e2) { e2 = sum[x]; }
      }
  }
  float dpar = 0.f;                                       // the parent's distance in the same form
  if (parent_stays) {
    float sum[1];
    dist_part(Cph + (size_t)par * d, std::integral_constant<int, 1>{}, 1, sum);
    dpar = sum[0];
  }
  double dc64 = -1.0;
  const bool redo = C > 1 && key < rows && !(e2 - e1 > kNearTie * e2);
  if (__any_sync(0xffffffffu, redo)) {
    double best = INFINITY;
    int bi = 0x7fffffff;
    if (redo)
      for (int c = s4; c < C; c += 4) {
        const double s = exact_dist(Kb + (size_t)key * d, Cch + (size_t)c * d, d);
        if (s < best) { best = s; bi = c; }
      }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ob < best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    if (redo) { c1 = bi < C ? bi : 0; dc64 = best; e1 = (float)best; }
  }
  if (s4 == 0 && key < rows) {
    if (parent_stays) {
      const float d1k = dpar;
      bool moved = e1 < d1k;
      if (!(fabsf(e1 - d1k) > kNearTie * fmaxf(e1, d1k))) {
        const double dp64 = s_redo[key] ? s_dp[key] : exact_dist(Kb + (size_t)key * d, Cph + (size_t)par * d, d);
        if (dc64 < 0.0) dc64 = exact_dist(Kb + (size_t)key * d, Cch + (size_t)c1 * d, d);
        moved = dc64 < dp64;
      }
      if (!moved) c1 = -1;
    }
    pidx[(size_t)bh * Nk + j0 + key] = par;
    cidx[(size_t)bh * Nk + j0 + key] = c1;
  }
}

// ------------------------------------------------------------------------------- aggregate
constexpr int kAggKeysPerWarp = 4;

// One warp = 4 keys: lane l adds elements 4l.. of each value row to the parent's and the child's sums with
// 16-byte reductions.  The value rows are the caller's, so they are loaded before the dependency wait.
template <typename T>
__global__ void __launch_bounds__(kThreads)
aggregate_simt_kernel(const T* __restrict__ V, const int32_t* pidx, const int32_t* cidx, float* Vp, float* np_,
                      float* Vc, float* nc, int Nk, int d, int M, int C, int32_t* status_word) {
  tc::pdl_launch_dependents();
  const int bh = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j0 = (blockIdx.x * (kThreads / 32) + warp) * kAggKeysPerWarp;
  const int chunks = d >> 2;                              // <= 64: two per lane
  float4 v[kAggKeysPerWarp][2];
#pragma unroll
  for (int t = 0; t < kAggKeysPerWarp; ++t)
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (j0 + t < Nk && lane + 32 * u < chunks) v[t][u] = ld4(V + ((size_t)bh * Nk + j0 + t) * d + 4 * (lane + 32 * u));
  tc::pdl_wait();
#pragma unroll
  for (int t = 0; t < kAggKeysPerWarp; ++t) {
    const int j = j0 + t;
    if (j >= Nk) break;
    const int a = ld_after_wait(pidx + (size_t)bh * Nk + j);
    const int c = ld_after_wait(cidx + (size_t)bh * Nk + j);
    if (a < 0 || a >= M || c < -1 || c >= C) {            // caller-supplied index out of range: skip the key, flag it
      if (lane == 0 && status_word) atomicCAS(status_word, 0, DEV_BAD_INDEX);
      continue;
    }
    const size_t prow = (size_t)bh * M + a, crow = prow * C + c;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int ch = lane + 32 * u;
      if (ch < chunks) {
        atomicAdd(reinterpret_cast<float4*>(Vp + prow * d) + ch, v[t][u]);
        if (c >= 0) atomicAdd(reinterpret_cast<float4*>(Vc + crow * d) + ch, v[t][u]);
      }
    }
    if (lane == 0) {
      atomicAdd(np_ + prow, 1.0f);
      if (c >= 0) atomicAdd(nc + crow, 1.0f);
    }
  }
}

// ------------------------------------------------------------------------------- attend
struct AttendArgs {
  const void *Q, *Cp, *Cc;
  const float *Vp, *np_, *Vc, *nc;
  void* Y;
  int32_t* topp_out;
  float* importance_out;
  int H, Nq, d, M, C, P, block_q, nblk, stays;
  int correcting; // Algorithm 2's literal child pass: mean-recovered parent logit and Delta A = A_c - A_p
  int tile_m;     // 0: exact importance; else parents visited in tiles of tile_m (Eq. "aproxdenom")
  int Nk;
  uint32_t inv_C; // 2^18 / C rounded up: e / C = e inv_C >> 18 for e < 2^13, C <= 16
  int keep;       // the block's parent logits stay in shared memory between the passes
  float scale;
};

// A running maximum starts at the lowest finite value: while every logit seen is -inf (a product beyond fp32's range) the
// weights are then exp(-inf) = 0, not exp(-inf + inf).
constexpr float kLowest = -3.402823466e38f;
constexpr int kAttThreads = kSelThreads;   // 32 x 16: thread (ty, tx) owns rows ty*RT .. , columns tx*4

// Shared memory of attend_simt_kernel, in floats from the base (doubles first).  All of it is dynamic: the limits the
// launcher compares it with are those of a CTA's dynamic and static memory together.
struct AttendSmem {
  int ldr;                                   // pitch of a [k][row] operand
  size_t w, wpart, q, c, v, s, np, nstay, nseen, sel, list, count, total;   // offsets in floats
};
// RT = 4: 128 query rows at a time (d <= 128), RT = 2: 64 rows.  v == c where the two tiles share one buffer.
// mma: Q and codewords as bfloat16 rows.
__host__ __device__ inline AttendSmem attend_smem_layout(int RT, int DT, int d, int M, int P, int tile_m, int keep,
                                                         bool mma) {
  AttendSmem L;
  L.ldr = 32 * RT + 4;
  const int ntiles = tile_m > 0 ? (M + tile_m - 1) / tile_m : 0;
  size_t o = 0;
  auto take = [&](size_t n) { size_t at = o; o += (n + 3) / 4 * 4; return at; };
  L.w = take(2 * (size_t)M);
  L.wpart = take(2 * (size_t)(kAttThreads / 32) * kCols);
  const size_t pitch = (size_t)(d + 15) / 16 * 8 + 4;       // floats per bfloat16 row: padded to 16 elements, plus 8
  const size_t cbytes = mma ? kCols * pitch : (size_t)d * kLdC, vbytes = (size_t)kCols * DT * 64;
  L.q = take(mma ? 32 * RT * pitch : (size_t)d * L.ldr);
  if (DT <= 2) {
    L.c = take(cbytes);
    L.v = take(vbytes);
  } else {
    L.c = L.v = take(cbytes > vbytes ? cbytes : vbytes);
  }
  L.s = take((size_t)(keep ? (M + kCols - 1) / kCols * kCols : kCols) * L.ldr);
  L.np = take(M);
  L.nstay = take(M);
  L.nseen = take(ntiles);
  L.sel = take(M);
  L.list = take(P > 0 ? P : 1);
  L.count = take(33);
  L.total = o;
  return L;
}

// Logits of columns without keys become -inf: their weight is then exp(-inf) = 0 against any reference, without a branch per
// element around the exponential.
__device__ __forceinline__ void mask_empty(float (&acc)[4], const float (&cnt)[4]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) acc[j] = cnt[j] > 0.f ? acc[j] : -INFINITY;
}
__device__ __forceinline__ float max16(float v) {         // over the 16 threads of a row
#pragma unroll
  for (int o = 8; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float sum16(float v) {
#pragma unroll
  for (int o = 8; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// One CTA = one query block.  Passes over the parents in tiles of 64 codewords:
//   A  logits, row maximum over non-empty parents and denominator (running maximum)
//   B  importance: column sums of A_ij / z_i in float64
//   C  softmax over unrefined parents and the children of the refined ones, weights through shared memory
//      into the value product (running maximum, register accumulators rescaled)
// Where the block's logits fit (a.keep) they are computed once and reused by B and C.  Bound: FFMA issue and
// the shared-memory pipe (RT + 4 operands per 4 RT products).  Against one warp per query row with a lane per
// logit, operands read from global memory for every product: whole forward fp32 B2 H12 N1024 d64 M64 C4 P8
// 2660 -> 82 us, tiled bf16 B1 H4 N4096 d64 M512 C4 P64 12.1 -> 0.36 ms (84 us and 0.40 ms with
// 256 threads); with the bfloat16 logits on the tensor cores 0.27 ms; with the steps since (narrow tiles, candidates only
// ranked, packed multiply-adds, importance tile by tile) 78 us and 0.185 ms; without branches around the exponentials, value
// rows copied asynchronously and small selections ranked at once, 74.6 us (the tiled one has a kernel of its own).
// 512 threads with 4 rows each rather than 256 with 8: the same products per second, twice the warps for everything
// that is a latency (operand loads, exponentials, exchanges), which was most of the time.
// WIDE: one CTA per SM with twice the registers, for grids of a wave at most (they measured 3 % faster there, fp32
// B2 H12 N1024 in 192 CTAs 10 % slower).
template <typename T, int RT, int DT, bool CORR, bool WIDE>
__global__ void __launch_bounds__(kAttThreads, (DT == 1 && !CORR && !WIDE) ? 2 : 1) attend_simt_kernel(const AttendArgs a) {
  extern __shared__ __align__(16) float sm[];
  constexpr int R = 32 * RT, kThreads = kAttThreads;
  const int d = a.d, M = a.M, C = a.C, P = a.P;
  constexpr bool kMma = std::is_same<T, __nv_bfloat16>::value;
  const AttendSmem L = attend_smem_layout(RT, DT, d, M, P, a.tile_m, a.keep, kMma);
  const int ldr = L.ldr;
  double* w = reinterpret_cast<double*>(sm + L.w);
  double* wpart = reinterpret_cast<double*>(sm + L.wpart);   // [16][64]
  float *qs = sm + L.q, *cs = sm + L.c, *vs = sm + L.v, *ss = sm + L.s;
  float *npS = sm + L.np, *nstay = sm + L.nstay, *nseen = sm + L.nseen;
  int *sel = reinterpret_cast<int*>(sm + L.sel), *sel_list = reinterpret_cast<int*>(sm + L.list);
  constexpr int ldv = DT * 64;
  int* cand = reinterpret_cast<int*>(wpart);              // [M] candidates of the selection (the sums are done by then)
  int *s_count = reinterpret_cast<int*>(sm + L.count), *s_ncand = s_count + 32;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, tx = tid & 15, ty = tid >> 4;
  const int blk = blockIdx.x, bh = blockIdx.y, h = bh % a.H;
  const int i0 = blk * a.block_q;
  const int rows = min(a.block_q, a.Nq - i0);
  const int nrt = (rows + R - 1) / R;
  const int ntiles = a.tile_m > 0 ? (M + a.tile_m - 1) / a.tile_m : 0;
  const T* Qb = static_cast<const T*>(a.Q) + ((size_t)bh * a.Nq + i0) * d;
  const T* Cph = static_cast<const T*>(a.Cp) + (size_t)h * M * d;
  const T* Cch = static_cast<const T*>(a.Cc) + (size_t)h * M * C * d;
  const float* Vp = a.Vp + (size_t)bh * M * d;
  const float* Vc = a.Vc + (size_t)bh * M * C * d;
  const float* np_ = a.np_ + (size_t)bh * M;
  const float* nc = a.nc + (size_t)bh * M * C;

  auto row_of = [&](int i) { return ty * RT + i; };
  const int dpad = (d + 15) & ~15, pitch = dpad + 8;
  auto load_q = [&](int rt) {
    auto row = [&](int r) { return rt * R + r < rows ? Qb + (size_t)(rt * R + r) * d : (const T*)nullptr; };
    if constexpr (kMma) load_rows<kThreads>(reinterpret_cast<T*>(qs), pitch, R, d, dpad, row);
    else load_transposed<kThreads, WIDE ? 4 : 2>(qs, ldr, R, d, [](int r) { return r; }, row);
  };
  auto store_s = [&](float* s0, const float (&acc)[RT][4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float* o = s0 + (size_t)(tx + 16 * j) * ldr + ty * RT;
      if constexpr (RT == 4) *reinterpret_cast<float4*>(o) = make_float4(acc[0][j], acc[1][j], acc[2][j], acc[3][j]);
      else *reinterpret_cast<float2*>(o) = make_float2(acc[0][j], acc[1][j]);
    }
  };
  auto load_s = [&](const float* s0, float (&acc)[RT][4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float* o = s0 + (size_t)(tx + 16 * j) * ldr + ty * RT;
      if constexpr (RT == 4) {
        const float4 x = *reinterpret_cast<const float4*>(o);
        acc[0][j] = x.x; acc[1][j] = x.y; acc[2][j] = x.z; acc[3][j] = x.w;
      } else {
        const float2 x = *reinterpret_cast<const float2*>(o);
        acc[0][j] = x.x; acc[1][j] = x.y;
      }
    }
  };

  // Logits of this thread's RT x 4 block of a tile of n columns (row c of the tile at code(c)), by way of s0 where
  // they come from the tensor cores.  Ends with the operands still being read by other threads: the caller
  // synchronises before they are overwritten.
  auto logits = [&](float (&acc)[RT][4], float* s0, int n, auto code) {
    auto row = [&](int c) { return c < n ? code(c) : (const T*)nullptr; };
    if constexpr (kMma) {
      load_rows<kThreads>(reinterpret_cast<T*>(cs), pitch, kCols, d, dpad, row);
      __syncthreads();
      // 32 RT rows x 64 columns over 16 warps: 16 rows x 8 RT columns each
      mma_block<RT>(s0, ldr, reinterpret_cast<const T*>(qs), reinterpret_cast<const T*>(cs), pitch, dpad, a.scale,
                    (warp % (2 * RT)) * 16, (warp / (2 * RT)) * 8 * RT);
      __syncthreads();
      load_s(s0, acc);
    } else {
      load_transposed<kThreads, 2>(cs, kLdC, code_rows(n), d, [](int c) { return code_pos(c); }, row);
      __syncthreads();
#pragma unroll
      for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
      mul_codes<RT>(acc, qs, ldr, cs, kLdC, d, ty, tx, n);
#pragma unroll
      for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] *= a.scale;
    }
  };

  load_q(0);                                              // the caller's Q: before the dependency wait
  tc::pdl_wait();
  for (int j = tid; j < M; j += kThreads) {
    const float n = ld_after_wait(np_ + j);
    npS[j] = n;
    if (a.stays) {                                        // keys that stay with their parent
      float s = 0.f;
      for (int c = 0; c < C; ++c) s += ld_after_wait(nc + (size_t)j * C + c);
      nstay[j] = n - s;
    }
    w[j] = 0.0;
    sel[j] = 0;
  }
  __syncthreads();
  if (tid < ntiles) {                                     // keys of each tile; summed up to a tile where the importance is finished
    float seen = 0.f;
    const int j1 = min(M, (tid + 1) * a.tile_m);
    for (int j = tid * a.tile_m; j < j1; ++j) seen += npS[j];
    nseen[tid] = seen;
  }
  // the choice of parents needs the importances only if there is one to make
  const bool need_w = (P > 0 && P < M) || a.importance_out != nullptr;
  // with a.keep the tiles start at multiples of 64 (validated by the launcher), so S is [M][rows]
  // Passes A and B over one tile of the tiled importance (exact importance: one tile of all parents) before the next,
  // with the maximum and denominator carried on: a tile's weights are taken against the maximum and the denominator seen
  // up to it, so they stay finite however far a later tile's logits lie above them.
  const int span = ntiles ? a.tile_m : M;
  for (int rt = 0; rt < nrt && need_w; ++rt) {
    if (rt > 0) { __syncthreads(); load_q(rt); }
    float m[RT], z[RT];
#pragma unroll
    for (int i = 0; i < RT; ++i) { m[i] = kLowest; z[i] = 0.f; }
    for (int t0 = 0; t0 < M; t0 += span) {
      const int t1 = min(M, t0 + span);
      // ---- pass A
      for (int c0 = t0; c0 < t1;) {
        const int n = min(kCols, t1 - c0);
        float acc[RT][4];
        float* s0 = a.keep ? ss + (size_t)c0 * ldr : ss;
        logits(acc, s0, n, [&](int c) { return Cph + (size_t)(c0 + c) * d; });
        if (!kMma && a.keep) store_s(s0, acc);
        float cnt[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) cnt[j] = tx + 16 * j < n ? npS[c0 + tx + 16 * j] : 0.f;
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          mask_empty(acc[i], cnt);
          float mx = -INFINITY;
#pragma unroll
          for (int j = 0; j < 4; ++j) mx = fmaxf(mx, acc[i][j]);
          mx = max16(mx);
          if (mx > m[i]) {                                // uniform over the 16 threads of the row
            z[i] *= expf(m[i] - mx);
            m[i] = mx;
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) z[i] = fmaf(expf(acc[i][j] - m[i]), cnt[j], z[i]);
        }
        c0 += n;
        __syncthreads();
      }
      // exact: the row's full denominator.  Tiled (appendix "Computing Importance with Tiled Codewords"): the
      // denominator seen up to this codeword's tile (Eq. "aproxdenom").
      double inv[RT];
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const float zi = sum16(z[i]);
        inv[i] = rt * R + row_of(i) < rows && zi != 0.f ? 1.0 / (double)zi : 0.0;
      }
      // ---- pass B
      for (int c0 = t0; c0 < t1;) {
        const int n = min(kCols, t1 - c0);
        float acc[RT][4];
        if (a.keep) load_s(ss + (size_t)c0 * ldr, acc);
        else logits(acc, ss, n, [&](int c) { return Cph + (size_t)(c0 + c) * d; });
        float cnt[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) cnt[j] = tx + 16 * j < n ? npS[c0 + tx + 16 * j] : 0.f;
#pragma unroll
        for (int i = 0; i < RT; ++i) {                    // (rows past the end: their weights do not count)
          mask_empty(acc[i], cnt);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float e = expf(acc[i][j] - m[i]);
            acc[i][j] = rt * R + row_of(i) < rows ? e : 0.f;
          }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          double s = 0.0;
#pragma unroll
          for (int i = 0; i < RT; ++i) s = fma((double)acc[i][j], inv[i], s);
          s += __shfl_xor_sync(0xffffffffu, s, 16);
          if (lane < 16) wpart[warp * kCols + tx + 16 * j] = s;
        }
        __syncthreads();
        if (tid < n) {
          double s = 0.0;
#pragma unroll
          for (int u = 0; u < kThreads / 32; ++u) s += wpart[u * kCols + tid];
          w[c0 + tid] += s;
        }
        c0 += n;
        __syncthreads();
      }
    }
  }
  if (need_w) {
    for (int j = tid; j < M; j += kThreads) {
      double x = w[j] * (double)npS[j];
      if (ntiles) {                                       // extrapolated by the keys seen up to the tile
        float seen = 0.f;
        for (int t = 0; t <= j / a.tile_m; ++t) seen += nseen[t];
        x *= (double)seen / (double)a.Nk;
      }
      w[j] = x;
      if (a.importance_out) a.importance_out[((size_t)bh * a.nblk + blk) * M + j] = (float)x;
    }
  }
  __syncthreads();

  // ---- top-P (ties -> lower index), then an ascending list
  if (P > 0)
    select_parents(w, M, P, sel, sel_list, cand, s_count, s_ncand,
                   a.topp_out ? a.topp_out + ((size_t)bh * a.nblk + blk) * P : nullptr, [] { __syncthreads(); });

  // ---- pass C: merged softmax over unrefined parents, stay residuals and children of refined parents
  T* Yb = static_cast<T*>(a.Y) + ((size_t)bh * a.Nq + i0) * d;
  const int child_w = (kCols / C) * C;                    // whole families per tile
  auto child_row = [&](int e) {                           // e-th child of the selected parents
    const int f = (int)(((uint32_t)e * a.inv_C) >> 18);
    return sel_list[f] * C + (e - f * C);
  };
  const int vch = d >> 2;
  for (int rt = 0; rt < nrt; ++rt) {
    if (rt > 0 || (nrt > 1 && need_w)) { __syncthreads(); load_q(rt); }
    float m[RT], z[RT], o[DT][RT][4];
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      m[i] = kLowest; z[i] = 0.f;
#pragma unroll
      for (int t = 0; t < DT; ++t)
#pragma unroll
        for (int j = 0; j < 4; ++j) o[t][i][j] = 0.f;
    }
    // Value rows of a tile (padding rows and columns zero): vs[c][k], copied without waiting, except a refined parent's (the sum
    // of the keys that stay).  row(c): the row's address, nullptr for zeros; stay(c): it is to be reduced by its children's.
    auto load_v = [&](auto row, auto stay) {
      for (int u = tid; u < kCols * (ldv / 4); u += kThreads) {
        const int c = u / (ldv / 4), ch = u - c * (ldv / 4);
        float* to = vs + c * ldv + 4 * ch;
        const float* from = ch < vch ? row(c) : nullptr;
        if (from == nullptr) {
          *reinterpret_cast<float4*>(to) = make_float4(0.f, 0.f, 0.f, 0.f);
        } else if (const float* child = stay(c)) {
          float4 v = ld_after_wait(reinterpret_cast<const float4*>(from) + ch);
          for (int cc = 0; cc < C; ++cc) {
            const float4 x = ld_after_wait(reinterpret_cast<const float4*>(child + (size_t)cc * d) + ch);
            v.x -= x.x; v.y -= x.y; v.z -= x.z; v.w -= x.w;
          }
          *reinterpret_cast<float4*>(to) = v;
        } else {
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(to)), "l"(from + 4 * ch) : "memory");
        }
      }
    };
    const int ptiles = (M + kCols - 1) / kCols;
    const int ctiles = P > 0 ? (P * C + child_w - 1) / child_w : 0;
    for (int tt = 0; tt < ptiles + ctiles; ++tt) {
      const bool child = tt >= ptiles;
      const int c0 = child ? (tt - ptiles) * child_w : tt * kCols;
      const int n = child ? min(child_w, P * C - c0) : min(kCols, M - c0);
      float acc[RT][4], cnt[4];
      float* sw = ss;                                     // weights of this tile, [column][row]
      auto load_values = [&]() {
        if (child) {
          load_v([&](int c) { return c < n ? Vc + (size_t)child_row(c0 + c) * d : nullptr; },
                 [](int) { return (const float*)nullptr; });
        } else {
          load_v([&](int c) -> const float* {
                   if (c >= n) return nullptr;
                   const bool refined = sel[c0 + c] != 0 && !CORR;
                   return (refined ? (a.stays ? nstay[c0 + c] : 0.f) : npS[c0 + c]) > 0.f ? Vp + (size_t)(c0 + c) * d : nullptr;
                 },
                 [&](int c) { return sel[c0 + c] && !CORR ? Vc + (size_t)(c0 + c) * C * d : nullptr; });
        }
      };
      if (DT <= 2) load_values();                         // its own buffer: the copies fly with the codewords' loads
      if (child) {
        logits(acc, sw, n, [&](int c) { return Cch + (size_t)child_row(c0 + c) * d; });
      } else if (a.keep && need_w) {
        sw = ss + (size_t)c0 * ldr;                       // the tile's logits, overwritten by its weights
        load_s(sw, acc);
      } else {
        logits(acc, sw, n, [&](int c) { return Cph + (size_t)(c0 + c) * d; });
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = tx + 16 * j;
        cnt[j] = 0.f;
        if (c < n) {
          if (child) {
            cnt[j] = ld_after_wait(nc + child_row(c0 + c));
          } else {
            // correcting form: every parent keeps its full term here, the children add differences below
            cnt[j] = (sel[c0 + c] && !CORR) ? (a.stays ? nstay[c0 + c] : 0.f) : npS[c0 + c];
          }
        }
      }
      float mean[CORR ? RT : 1][4];                       // correcting form only
      if (CORR && child) {
        // Eq. "parent_recovery": under parent = mean(children) the parent's logit is the mean of its
        // children's; Eq. "correcting_attention": the child's keys trade the parent's weight for their own
        store_s(sw, acc);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int c = tx + 16 * j, f = c / C * C;
#pragma unroll
          for (int i = 0; i < RT; ++i) {
            float sp = 0.f;
            if (c < n) for (int c2 = 0; c2 < C; ++c2) sp += sw[(size_t)(f + c2) * ldr + row_of(i)];
            mean[CORR ? i : 0][j] = sp / (float)C;
          }
        }
        __syncthreads();
      }
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        mask_empty(acc[i], cnt);
        float mx = -INFINITY;
#pragma unroll
        for (int j = 0; j < 4; ++j) mx = fmaxf(mx, acc[i][j]);
        mx = max16(mx);
        if (mx > m[i]) {
          const float alpha = expf(m[i] - mx);
          z[i] *= alpha;
#pragma unroll
          for (int t = 0; t < DT; ++t)
#pragma unroll
            for (int j = 0; j < 4; ++j) o[t][i][j] *= alpha;
          m[i] = mx;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float av = expf(acc[i][j] - m[i]);
          if (CORR && child) av = cnt[j] > 0.f ? av - expf(mean[CORR ? i : 0][j] - m[i]) : 0.f;
          z[i] = fmaf(av, cnt[j], z[i]);
          acc[i][j] = av;
        }
      }
      store_s(sw, acc);
      if (DT <= 2) tc::cp_async_wait_all();
      __syncthreads();
      if (DT > 2) {                                       // shared buffer: the codewords are done with
        load_values();
        tc::cp_async_wait_all();
        __syncthreads();
      }
#pragma unroll
      for (int t = 0; t < DT; ++t) mul_tile<RT, 4>(o[t], sw, ldr, vs + t * 64, ldv, (n + 3) & ~3, ty, tx);
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      const float inv = 1.f / sum16(z[i]);
      const int r = rt * R + row_of(i);
      if (r < rows) {
#pragma unroll
        for (int t = 0; t < DT; ++t) {
          const int k = t * 64 + tx * 4;
          if (k < d) st4(Yb + (size_t)r * d + k, make_float4(o[t][i][0] * inv, o[t][i][1] * inv, o[t][i][2] * inv, o[t][i][3] * inv));
        }
      }
    }
  }
}

}  // namespace

// The envelope of the entry points (header): what the problem may ask for.  The kernel's own shared memory is
// attend_smem_layout(), at most 227 KiB for every problem inside it.
size_t simt_attend_smem_bytes(int d, int M, int C, int P, int block_q, int tile_m) {
  const size_t ncols = (size_t)M + (size_t)P * C;
  size_t b = sizeof(double) * M;
  b += sizeof(float) * ((size_t)block_q * d + 2 * (size_t)block_q + 2 * (size_t)M + 8 * ncols);
  b += sizeof(int) * ((size_t)M + (size_t)(P > 0 ? P : 1));
  if (tile_m > 0) b += sizeof(float) * ((size_t)block_q + 1) * ((M + tile_m - 1) / tile_m);
  return b;
}

namespace {

constexpr size_t kSmemHalf = 113 * 1024;                  // two CTAs on an SM

template <typename T>
avq_status launch_assign(const avq_problem& p, const void* K, const void* Cp, const void* Cc,
                         int32_t* pidx, int32_t* cidx, void* zero_base, size_t zero_bytes, cudaStream_t st) {
  const size_t smem = sizeof(float) * assign_smem_floats(p.d, std::is_same<T, __nv_bfloat16>::value);
  auto kern = assign_simt_kernel<T>;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return AVQ_ERR_CUDA;
  const avq_status s = open_shared_memory<assign_simt_kernel<T>>(dev);
  if (s != AVQ_OK) return s;
  dim3 grid((p.Nk + kAssignKeys - 1) / kAssignKeys, p.B * p.H);
  kern<<<grid, kThreads, smem, st>>>(static_cast<const T*>(K), static_cast<const T*>(Cp),
                                     static_cast<const T*>(Cc), pidx, cidx, p.H, p.Nk, p.d, p.M, p.C,
                                     (p.flags & AVQ_FLAG_PARENT_STAYS) ? 1 : 0, static_cast<uint4*>(zero_base),
                                     zero_bytes / 16, slice_units(zero_bytes / 16, (size_t)grid.x * grid.y));
  return cuda_ok(cudaGetLastError());
}

template <typename T>
avq_status launch_aggregate(const avq_problem& p, const void* V, const int32_t* pidx, const int32_t* cidx,
                            float* Vp, float* np_, float* Vc, float* nc, bool chained, int32_t* status_word,
                            cudaStream_t st) {
  const int per_cta = kAggKeysPerWarp * (kThreads / 32);
  dim3 grid((p.Nk + per_cta - 1) / per_cta, p.B * p.H);
  return cuda_ok(tc::launch_pdl(aggregate_simt_kernel<T>, grid, dim3(kThreads), 0, st, chained,
                                static_cast<const T*>(V), pidx, cidx, Vp, np_, Vc, nc, p.Nk, p.d, p.M, p.C,
                                status_word));
}

template <typename T, int RT, int DT, bool CORR>
avq_status launch_attend_rdc(AttendArgs a, int B, bool chained, cudaStream_t st) {
  constexpr bool kMma = std::is_same<T, __nv_bfloat16>::value;
  auto bytes = [&](int keep) {
    return sizeof(float) * attend_smem_layout(RT, DT, a.d, a.M, a.P, a.tile_m, keep, kMma).total;
  };
  // The block's logits stay in shared memory when one row tile holds the block and that leaves room for two
  // CTAs per SM (or all of an SM's memory is there for the taking because the grid has a CTA per SM at most).
  int sms = 148, dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return AVQ_ERR_CUDA;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return AVQ_ERR_CUDA;
  const bool one_wave = (int64_t)a.nblk * B * a.H <= sms;
  const size_t most = one_wave ? kSmemMax : kSmemHalf;
  a.keep = (a.block_q <= 32 * RT && (a.tile_m == 0 || a.tile_m % kCols == 0) && bytes(1) <= most) ? 1 : 0;
  const size_t smem = bytes(a.keep);
  if (smem > kSmemMax) return AVQ_ERR_UNSUPPORTED;
  // (the wide variant differs where a CTA may have half an SM's registers otherwise, and in the float32 operand loads)
  constexpr bool kHasWide = !kMma || (DT == 1 && !CORR);
  const bool wide = kHasWide && one_wave;
  auto kern = wide ? attend_simt_kernel<T, RT, DT, CORR, kHasWide> : attend_simt_kernel<T, RT, DT, CORR, false>;
  const avq_status s = wide ? open_shared_memory<attend_simt_kernel<T, RT, DT, CORR, kHasWide>>(dev)
                            : open_shared_memory<attend_simt_kernel<T, RT, DT, CORR, false>>(dev);
  if (s != AVQ_OK) return s;
  return cuda_ok(tc::launch_pdl(kern, dim3(a.nblk, B * a.H), dim3(kAttThreads), smem, st, chained, a));
}

template <typename T, int RT, int DT>
avq_status launch_attend_rd(const AttendArgs& a, int B, bool chained, cudaStream_t st) {
  return a.correcting ? launch_attend_rdc<T, RT, DT, true>(a, B, chained, st)
                      : launch_attend_rdc<T, RT, DT, false>(a, B, chained, st);
}

template <typename T>
avq_status launch_attend(const AttendArgs& a, int B, bool chained, cudaStream_t st) {
  if (simt_attend_smem_bytes(a.d, a.M, a.C, a.P, a.block_q, a.tile_m) > kSimtAttendSmemLimit)
    return AVQ_ERR_UNSUPPORTED;                           // validate_forward rejects these up front
  // 128 rows at a time where the block has them and shared memory holds them (d <= 128), else 64
  if (a.block_q > 64 && a.d <= 64) return launch_attend_rd<T, 4, 1>(a, B, chained, st);
  if (a.block_q > 64 && a.d <= 128) return launch_attend_rd<T, 4, 2>(a, B, chained, st);
  if (a.d <= 64) return launch_attend_rd<T, 2, 1>(a, B, chained, st);
  if (a.d <= 128) return launch_attend_rd<T, 2, 2>(a, B, chained, st);
  return launch_attend_rd<T, 2, 4>(a, B, chained, st);
}

}  // namespace

avq_status simt_assign(const avq_problem& p, const void* K, const void* Cp, const void* Cc,
                       int32_t* parent_idx, int32_t* child_idx, void* zero_base, size_t zero_bytes, cudaStream_t st) {
  if (zero_bytes % 16 != 0) return AVQ_ERR_WORKSPACE;
  return p.dtype == AVQ_F32
             ? launch_assign<float>(p, K, Cp, Cc, parent_idx, child_idx, zero_base, zero_bytes, st)
             : launch_assign<__nv_bfloat16>(p, K, Cp, Cc, parent_idx, child_idx, zero_base, zero_bytes, st);
}

avq_status simt_aggregate(const avq_problem& p, const void* V, const int32_t* parent_idx,
                          const int32_t* child_idx, float* Vp, float* np_, float* Vc, float* nc, bool pre_zeroed,
                          int32_t* status_word, cudaStream_t st) {
  if (!pre_zeroed) {
    const size_t BH = (size_t)p.B * p.H;
    cudaError_t e = cudaMemsetAsync(Vp, 0, sizeof(float) * BH * p.M * p.d, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(np_, 0, sizeof(float) * BH * p.M, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(Vc, 0, sizeof(float) * BH * p.M * p.C * p.d, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(nc, 0, sizeof(float) * BH * p.M * p.C, st);
    if (e != cudaSuccess) return AVQ_ERR_CUDA;
  }
  return p.dtype == AVQ_F32
             ? launch_aggregate<float>(p, V, parent_idx, child_idx, Vp, np_, Vc, nc, pre_zeroed, status_word, st)
             : launch_aggregate<__nv_bfloat16>(p, V, parent_idx, child_idx, Vp, np_, Vc, nc, pre_zeroed, status_word, st);
}

avq_status simt_attend(const avq_problem& p, const void* Q, const void* Cp, const void* Cc,
                       const float* Vp, const float* np_, const float* Vc, const float* nc, int32_t P,
                       int32_t block_q, void* Y, int32_t* topp_out, float* importance_out,
                       int32_t tile_m, bool chained, cudaStream_t st) {
  AttendArgs a;
  a.tile_m = tile_m;
  a.Nk = p.Nk;
  a.Q = Q; a.Cp = Cp; a.Cc = Cc; a.Vp = Vp; a.np_ = np_; a.Vc = Vc; a.nc = nc; a.Y = Y;
  a.topp_out = topp_out; a.importance_out = importance_out;
  a.H = p.H; a.Nq = p.Nq; a.d = p.d; a.M = p.M; a.C = p.C; a.P = P; a.block_q = block_q;
  a.nblk = (p.Nq + block_q - 1) / block_q;
  a.stays = (p.flags & AVQ_FLAG_PARENT_STAYS) ? 1 : 0;
  a.correcting = (p.flags & AVQ_FLAG_CORRECTING) ? 1 : 0;
  a.keep = 0;
  a.inv_C = ((1u << 18) + (uint32_t)p.C - 1) / (uint32_t)p.C;
  a.scale = p.scale;
  return p.dtype == AVQ_F32 ? launch_attend<float>(a, p.B, chained, st)
                            : launch_attend<__nv_bfloat16>(a, p.B, chained, st);
}

}  // namespace avq
