// Tensor-core key assignment (Algorithm 1, parent and child argmin) for bf16 inputs.
//
// One CTA takes a tile of 128 consecutive keys of one (batch, head), or a run of them, 8 warps.  TMA stages each key tile
// and, once per head, the head's parent codebook in shared memory (K-major, 128-byte swizzle); one elected thread issues the
// tcgen05 MMA chain  D[128 x M] = K_tile . Cp^T  into TMEM.
//   parent   (beyond 64 parents; up to that best, runner-up and index by a key per lane) warp w holds keys 32 (w % 4) .. +31 of the column half w / 4 and reads the products in the fragment layout
//            (4 keys x column pairs per lane).  Two passes over ||c||^2 - 2 k.c: the minimum of the row; then the
//            number and the index of the columns within the MMA's rounding of it, added up in one register.  Only
//            when there is more than one such column are all M distances redone in float64 in the direct form
//            (lowest index wins ties).  Three instructions per column and row instead of the six of a running best,
//            runner-up and index, and half of them off the ALU pipe, which bounded the kernel.
//   child    large grids with eight children, and PARENT_STAYS: by warp-level tensor-core products over the keys in the order
//            of their parents (see there).  Else on CUDA cores (a second MMA over all M C children would cost C times the parent GEMM): ||c||^2 - 2 k.c where
//            a norm table is at hand, near-ties in the direct form sum (k - c)^2 in float32 and then in float64; else
//            the direct form throughout, near-ties in float64.
//            Four lanes per key, each over a quarter of the head dimension for all C children of the
//            key's parent (one running sum per child); a transposing butterfly merges the four lanes.
// Bound, with the loop over a key's children, by L1 and shared memory (56 to 69 % busy) and the latency of the child loads, issue
// slots at 39 to 59 %; with products over sorted keys by latency, the barriers around the sort first (2.7 to 3.5 warps wait at one
// per instruction issued), L1 at 39 to 50 %, issue slots at 29 to 52 %.  L2 is at 9 to 19 %.
#include <type_traits>

#include "avq_tc_common.cuh"

namespace avq {
namespace {

using namespace tc;

constexpr int kKeys = 128;
constexpr int kThreadsA = 256;
// CTAs per SM the register budget is set for: the d = 64 kernels are small enough (24-48 KB of shared
// memory, at most 128 TMEM columns up to M = 128) for four to share an SM.
constexpr int assign_min_ctas(int D) { return D == 64 ? 4 : 2; }

__device__ __forceinline__ float bf_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf_hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }

// s + the squares of 8 packed bf16 (mixed-precision multiply-add: exact products, fp32 sum)
__device__ __forceinline__ float norm_bf16x8(float s, const uint4& v) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int e = 0; e < 4; ++e)
    asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %1;\n\tfma.rn.f32.bf16 %0, l, l, %0;\n\tfma.rn.f32.bf16 %0, h, h, %0;\n\t}"
        : "+f"(s) : "r"(w[e]));
  return s;
}
// s += k . c over 8 packed bf16 (same instruction)
__device__ __forceinline__ void dot_bf16x8(float& s, const uint4& k, const uint4& c) {
  const uint32_t x[4] = {k.x, k.y, k.z, k.w}, y[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
  for (int e = 0; e < 4; ++e)
    asm("{\n\t.reg .b16 a, b, c, d;\n\tmov.b32 {a, b}, %1;\n\tmov.b32 {c, d}, %2;\n\tfma.rn.f32.bf16 %0, a, c, %0;\n\tfma.rn.f32.bf16 %0, b, d, %0;\n\t}"
        : "+f"(s) : "r"(x[e]), "r"(y[e]));
}
// One warp: c += a (16 x 16) . b (16 x 8), exact products, fp32 sums
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
struct KeyChunk { f32x2 p[4]; };      // 8 key elements as four fp32 pairs
__device__ __forceinline__ KeyChunk widen8(const uint4& a) {
  KeyChunk k;
  k.p[0] = pack2(bf_lo(a.x), bf_hi(a.x)); k.p[1] = pack2(bf_lo(a.y), bf_hi(a.y));
  k.p[2] = pack2(bf_lo(a.z), bf_hi(a.z)); k.p[3] = pack2(bf_lo(a.w), bf_hi(a.w));
  return k;
}
// sum over 8 elements of (k - c)^2, two lanes of packed fp32 arithmetic (sub.f32x2 / fma.f32x2)
__device__ __forceinline__ float sqdiff8(const KeyChunk& k, const uint4& c) {
  const uint32_t y[4] = {c.x, c.y, c.z, c.w};
  f32x2 acc = 0;   // {0.f, 0.f}
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    f32x2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(k.p[e]), "l"(pack2(bf_lo(y[e]), bf_hi(y[e]))));
    acc = fma2(d, d, acc);
  }
  float lo, hi;
  unpack2(acc, lo, hi);
  return lo + hi;
}

// element `col` (0..D-1) of key row `row` in the swizzled key tile
template <int D>
__device__ __forceinline__ float key_elem(const unsigned char* Ks, int row, int col) {
  const unsigned char* sub = Ks + (col >> 6) * (kKeys * 128);
  return __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(sub + sw128_offset(row, col & 63)));
}

template <int D>
__device__ double exact_dist_smem(const unsigned char* Ks, int row, const __nv_bfloat16* c) {
  double s = 0.0;
  for (int k = 0; k < D; ++k) {
    const double t = (double)key_elem<D>(Ks, row, k) - (double)__bfloat162float(c[k]);
    s += t * t;
  }
  return s;
}

// float64, direct form, by the four lanes (s4) of a key's group: a quarter of the dimensions each
template <int D>
__device__ __forceinline__ double exact4(const unsigned char* Ks, int key, int s4, const __nv_bfloat16* c) {
  double sd = 0.0;
  for (int u = 0; u < D / 32; ++u)
    for (int e = 0; e < 8; ++e) {
      const int col = 8 * (s4 + 4 * u) + e;
      const double x = (double)key_elem<D>(Ks, key, col) - (double)__bfloat162float(c[col]);
      sd += x * x;
    }
  sd += __shfl_xor_sync(0xffffffffu, sd, 1);
  return sd + __shfl_xor_sync(0xffffffffu, sd, 2);
}

// PARENT_STAYS, one warp, four lanes per key: the child of key row `key` (-1: it stays) where norms and products leave open
// which child is nearest or (stay_open) whether that is closer than the parent.  Measured in the direct form in float32, and
// what that leaves open (relative 1e-4) in float64.  Keys that hug their parent are about equally far from its children, and
// products separate little where keys lie far from the origin for their distances: B2 H8 N5000 d128 M96 C8 with 32 added to
// every dimension, us per call: 190 with float64 straight behind the products, 114 so, 118 in the direct form throughout.  (Keys
// that moved are close to one child: without PARENT_STAYS such offsets cost nothing.)  Out of line: keys around the origin
// hardly ever come here, and inlined it took registers from the loop that calls it.
template <int D, int C>
__device__ __noinline__ int settle_child(const unsigned char* Ks, int key, int s4, const __nv_bfloat16* Cch,
                                         const __nv_bfloat16* Cpk, int c1, bool open, bool stay_open, bool moved) {
  auto direct4 = [&](const __nv_bfloat16* c) {
    float sd = 0.f;
#pragma unroll
    for (int u = 0; u < D / 32; ++u) {
      const int cu = s4 + 4 * u;
      sd += sqdiff8(widen8(*reinterpret_cast<const uint4*>(Ks + (cu >> 3) * (kKeys * 128) + sw128_offset(key, (cu & 7) * 8))),
                    __ldg(reinterpret_cast<const uint4*>(c) + cu));
    }
    sd += __shfl_xor_sync(0xffffffffu, sd, 1);
    return sd + __shfl_xor_sync(0xffffffffu, sd, 2);
  };
  if (__any_sync(0xffffffffu, open)) {
    float f1 = INFINITY, f2 = INFINITY;
    int fi = 0;
#pragma unroll 1
    for (int c = 0; c < C; ++c) {
      const float sd = direct4(Cch + (size_t)c * D);
      if (sd < f1) { f2 = f1; f1 = sd; fi = c; }
      else if (sd < f2) { f2 = sd; }
    }
    if (open) c1 = fi;
    open = open && !(f2 - f1 > 1e-4f * f2);
    if (__any_sync(0xffffffffu, open)) {
      double best = INFINITY;
      int bi = 0;
#pragma unroll 1
      for (int c = 0; c < C; ++c) {
        const double sd = exact4<D>(Ks, key, s4, Cch + (size_t)c * D);
        if (sd < best) { best = sd; bi = c; }
      }
      if (open) c1 = bi;
    }
  }
  if (__any_sync(0xffffffffu, stay_open)) {
    const float fc = direct4(Cch + (size_t)c1 * D), fp = direct4(Cpk);
    if (stay_open) moved = fc < fp;
    stay_open = stay_open && !(fabsf(fc - fp) > 1e-4f * fmaxf(fc, fp));
    if (__any_sync(0xffffffffu, stay_open)) {
      const bool closer = exact4<D>(Ks, key, s4, Cch + (size_t)c1 * D) < exact4<D>(Ks, key, s4, Cpk);
      if (stay_open) moved = closer;
    }
  }
  return moved ? c1 : -1;
}

// ||c||^2 of every codeword of every head, once per call: parents [H, M], then children [H, M, C].  Eight lanes per
// codeword row.
template <int D>
__global__ void __launch_bounds__(256) code_norms_kernel(const __nv_bfloat16* __restrict__ Cp,
                                                         const __nv_bfloat16* __restrict__ Cc,
                                                         float* __restrict__ cnorm, int parents, int rows) {
  pdl_launch_dependents();   // the assign grid may start its set-up and loads
  const int row = (blockIdx.x * 256 + threadIdx.x) >> 3, part = threadIdx.x & 7;
  float s = 0.f;
  if (row < rows) {
    const __nv_bfloat16* code = row < parents ? Cp + (size_t)row * D : Cc + (size_t)(row - parents) * D;
    const uint4* src = reinterpret_cast<const uint4*>(code) + part;
#pragma unroll
    for (int t = 0; t < D / 64; ++t) s = norm_bf16x8(s, __ldg(src + 8 * t));
  }
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  s += __shfl_xor_sync(0xffffffffu, s, 4);
  if (row < rows && part == 0) cnorm[row] = s;
  pdl_wait();                // this grid's completion implies that of the one it ran beside
}

enum Form { kOne, kRuns, kSmall };
// NL = 16-byte loads per lane that cover one parent's C x d block of children: C * d / 256.
// STAYS: Algorithm 1's masked scatter - a key moves to its nearest child only if that child is strictly
// closer than the parent (child index -1 otherwise).
// FORM: kOne, one tile per CTA; kRuns, a CTA takes a run of tiles (more loop state in registers); kSmall, one tile per CTA and
// the parents' distances with a key per lane: best, runner-up and index in one pass.
// TABLE: cnorm_g holds the squared norms of all codewords (parents [H, M], then children [H, M, C]); the child distances
// are then ||c||^2 - 2 k.c at one mixed-precision multiply-add per element, half the instructions of the direct form.
// SORTED: children by products over the keys in the order of their parents (always under PARENT_STAYS).
template <int D, int NL, bool STAYS, Form FORM, bool TABLE, bool SORTED>
__global__ void __launch_bounds__(kThreadsA, assign_min_ctas(D))
tc_assign_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmCp,
                 const __nv_bfloat16* __restrict__ Cp, const __nv_bfloat16* __restrict__ Cc,
                 int32_t* __restrict__ pidx, int32_t* __restrict__ cidx, int H, int Nk, int M, int nblk, int total_tiles,
                 uint32_t tmem_cols, int32_t* status_word, uint4* __restrict__ zero_base, size_t zero_units,
                 size_t zero_per, const float* cnorm_g, int beside) {
  // 1024-byte alignment (swizzle atoms) is requested from the launch, not computed from the pointer, so
  // that the compiler keeps every access in the shared address space.
  extern __shared__ __align__(1024) unsigned char smem[];
  constexpr bool RUNS = FORM == kRuns;
  constexpr int kSub = D / 64;                       // 64-column sub-tiles along the head dimension
  constexpr int kKeyBytes = kSub * kKeys * 128;
  const unsigned char* Ks = smem;                    // key tile: kSub x [128 x 128 B]
  unsigned char* Cs = smem + kKeyBytes;              // kSub x [M x 128 B]
  float* cnorm = reinterpret_cast<float*>(Cs + kSub * M * 128);   // [M]
  float* xd = cnorm + M;                             // [2][128] smallest distance of each column half
  float* xs = xd + 2 * kKeys;                        // [2][128] columns close to the minimum: sum of 256 + index (kSmall: runner-up)
  float* xkn = xs + 2 * kKeys;                       // [2][128] halves of ||k||^2
  int* par = reinterpret_cast<int*>(xkn + 2 * kKeys);   // [128] final parent of each key
  int* chi = par + kKeys;                            // [128] final child of each key
  int* hist = chi + kKeys;                           // SORTED: [M] keys per parent
  int* offs = reinterpret_cast<int*>(xs);            // [M] first place of a parent's keys in `order`
  uint8_t* order = reinterpret_cast<uint8_t*>(hist + M);   // SORTED: [128] keys by parent
  uint32_t* cmax_bits = reinterpret_cast<uint32_t*>(SORTED ? order + kKeys : reinterpret_cast<uint8_t*>(hist));   // max ||c||^2 (non-negative float bits)
  uint32_t* tmem_slot = cmax_bits + 1;
  uint64_t* bars = reinterpret_cast<uint64_t*>(tmem_slot + 1);      // [3]
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + 3);
  uint64_t *bar_k = bars, *bar_mma = bars + 1, *bar_c = bars + 2;   // key tile, products, codebook

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform
  const int q = warp & 3, hf = warp >> 2, r = q * 32 + lane;
  const int g = lane >> 2, t4 = lane & 3;            // fragment rows q*32 + g + 8 h, column pairs 2 t4
  // This CTA's run of consecutive tiles (the CTAs with one more are the first ones: every SM gets its share).
  int tile0 = (int)blockIdx.x, tile1 = tile0 + 1;
  if constexpr (RUNS) {
    const int per_cta = total_tiles / gridDim.x, more = total_tiles - per_cta * gridDim.x;
    tile0 = (int)blockIdx.x * per_cta + min((int)blockIdx.x, more);
    tile1 = tile0 + per_cta + ((int)blockIdx.x < more ? 1 : 0);
  }
  int bh = tile0 / nblk, blk = tile0 - bh * nblk;
  const int MH = M >> 1;                             // columns per half (multiple of 16: M % 32 == 0)
  pdl_launch_dependents();   // the next kernel of the call may begin its set-up
  // Inside avq_forward the grid also clears the accumulators of the aggregation that follows (status
  // header, leaf sums, leaf counts: zero_units 16-byte words), each CTA a slice of zero_per; the stores drain
  // while the tile loads.  A bounded wait that expires does so long after CTA 0 has cleared the header.
  if (zero_units) {
    const size_t u0 = blockIdx.x * zero_per, u1 = min(zero_units, u0 + zero_per);
    for (size_t u = u0 + tid; u < u1; u += kThreadsA) zero_base[u] = make_uint4(0u, 0u, 0u, 0u);
  }
  auto load_keys = [&](int b, int t) {               // one thread
    mbar_expect_tx(bar_k, (uint32_t)kKeyBytes);
#pragma unroll
    for (int s = 0; s < kSub; ++s) tma_load_3d(smem + s * kKeys * 128, &tmK, s * 64, t * kKeys, b, bar_k);
  };
  auto load_codes = [&](int b) {
    mbar_expect_tx(bar_c, (uint32_t)(kSub * M * 128));
#pragma unroll
    for (int s = 0; s < kSub; ++s) tma_load_2d(Cs + s * M * 128, &tmCp, s * 64, (b % H) * M, bar_c);
  };
  if (warp == 0 && elect_one()) {
    prefetch_tmap(&tmK);
    prefetch_tmap(&tmCp);
#pragma unroll
    for (int i = 0; i < 3; ++i) mbar_init(&bars[i], 1);
    mbar_fence_init();
    *abort_flag = 0;
    *cmax_bits = 0;
    load_keys(bh, blk);
    load_codes(bh);
  }
  // tcgen05.alloc blocks while the SM's columns are taken (four CTAs of 256 columns share an SM at d = 64,
  // M > 128: two run, two wait here).  The holders need nothing from the waiters and free their columns
  // before they end, so the wait is finite; it is the one device-side wait without a time limit of its own.
  if (warp == 1) {                                   // not the warp that is busy issuing the loads
    tmem_alloc(tmem_slot, tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  auto issue_mma = [&]() {                           // one warp
    if (elect_one()) {
      tc_fence_after();
      const uint32_t idesc = umma_idesc_bf16(kKeys, M);
      const uint64_t kd = umma_desc_sw128(smem_u32(Ks)), cd = umma_desc_sw128(smem_u32(Cs));
#pragma unroll
      for (int k = 0; k < D / 16; ++k)
        umma_bf16(tmem_base, kd + (uint64_t)((k / 4) * (kKeys * 8) + (k % 4) * 2),
                  cd + (uint64_t)((k / 4) * M * 8 + (k % 4) * 2), idesc, k > 0);
      umma_commit(bar_mma);
    }
    __syncwarp();
  };
  uint32_t ph_k = 0, ph_mma = 0, ph_c = 0;
  bool new_head = true;
  for (int tile = tile0;; ++tile) {
  const int h = bh % H, j0 = blk * kKeys;
  const int nbh = blk + 1 == nblk ? bh + 1 : bh, nblk_ = blk + 1 == nblk ? 0 : blk + 1;
  const bool has_next = RUNS && tile + 1 < tile1, next_new_head = has_next && nbh != bh && H > 1;
  // ||c_m||^2 (and its maximum) of a head: from the array the kernel ahead of this one filled, or from the staged
  // codebook
  bool codes = true;
  if (new_head) {
    codes = mbar_wait(bar_c, ph_c, abort_flag, status_word, DEV_TIMEOUT_ASSIGN);
    ph_c ^= 1;
    if (TABLE) pdl_wait();
    for (int m = tid; m < M; m += kThreadsA) {
      float s = 0.f;
      if (TABLE) {
        s = ld_after_wait(cnorm_g + (size_t)h * M + m);
      } else {
#pragma unroll
        for (int sub = 0; sub < kSub; ++sub)
#pragma unroll
          for (int ch = 0; ch < 8; ++ch)
            s = norm_bf16x8(s, *reinterpret_cast<const uint4*>(Cs + sub * M * 128 + sw128_offset(m, ch * 8)));
      }
      cnorm[m] = s;
      atomicMax(cmax_bits, __float_as_uint(s));
    }
  }
  const bool loaded = mbar_wait(bar_k, ph_k, abort_flag, status_word, DEV_TIMEOUT_ASSIGN) && codes;
  ph_k ^= 1;
  if (warp == 0 && loaded) issue_mma();              // (all lanes wait for the same barriers and agree)

  if (SORTED)
    for (int m = tid; m < M; m += kThreadsA) hist[m] = 0;
  {                                                  // half of ||k||^2 per thread
    float s = 0.f;
    constexpr int kChunksHalf = D / 16;              // 16-byte chunks in half a row
#pragma unroll
    for (int cc = 0; cc < kChunksHalf; ++cc) {
      const int ch = hf * kChunksHalf + cc;          // chunk index in the row, 0 .. D/8-1
      s = norm_bf16x8(s, *reinterpret_cast<const uint4*>(Ks + (ch >> 3) * kKeys * 128 + sw128_offset(r, (ch & 7) * 8)));
    }
    xkn[hf * kKeys + r] = s;
  }
  __syncthreads();   // cnorm, cmax visible

  const bool done = mbar_wait(bar_mma, ph_mma, abort_flag, status_word, DEV_TIMEOUT_ASSIGN);
  ph_mma ^= 1;
  tc_fence_after();

  // ---- parents: minimum of ||c||^2 - 2 k.c over this warp's half of the columns
  const uint32_t trow = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(hf * MH);
  const float* cnh = cnorm + hf * MH;
  if constexpr (FORM == kSmall) {
    float d1 = INFINITY, d2 = INFINITY;
    int i1 = 0;
    for (int c0 = 0; c0 < MH; c0 += 16) {
      float dot[16];
      tmem_ld16(trow + c0, dot);                     // warp-collective: executed by every lane
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        const float dist = fmaf(-2.f, dot[e], cnh[c0 + e]);
        d2 = fminf(d2, fmaxf(dist, d1));             // runner-up: second smallest so far
        if (dist < d1) { d1 = dist; i1 = hf * MH + c0 + e; }
      }
    }
    xd[hf * kKeys + r] = d1;
    xs[hf * kKeys + r] = d2;
    par[hf * kKeys + r] = i1;                        // (par and chi, adjacent: [2][128])
  } else {
  const f32x2 minus2 = pack2(-2.f, -2.f);
  float m[4];
#pragma unroll
  for (int h4 = 0; h4 < 4; ++h4) m[h4] = INFINITY;
  auto blocks = [&](auto nb, int c0, auto&& use) {   // distances of nb 8-column blocks from column c0, pair by pair
    constexpr int NBk = decltype(nb)::value;
    uint32_t s[2][4 * NBk];
    tmem_ld_frag<NBk>(trow + c0, s);                 // warp-collective
    f32x2 cn[NBk];
#pragma unroll
    for (int b = 0; b < NBk; ++b) cn[b] = *reinterpret_cast<const f32x2*>(cnh + c0 + 8 * b + 2 * t4);
    tmem_ld_wait_frag<NBk>(s);
#pragma unroll
    for (int b = 0; b < NBk; ++b)
#pragma unroll
      for (int h4 = 0; h4 < 4; ++h4) {
        float lo, hi;
        unpack2(fma2(pack2u(s[h4 >> 1][4 * b + 2 * (h4 & 1)], s[h4 >> 1][4 * b + 2 * (h4 & 1) + 1]), minus2, cn[b]), lo, hi);
        use(h4, c0 + 8 * b, lo, hi);
      }
  };
  auto all_blocks = [&](auto&& use) {
    int c0 = 0;
    if constexpr (D > 64)                            // (the 64-register budget of d = 64 holds 16 columns at a time)
      for (; c0 + 32 <= MH; c0 += 32) blocks(std::integral_constant<int, 4>{}, c0, use);
    for (; c0 < MH; c0 += 16) blocks(std::integral_constant<int, 2>{}, c0, use);
  };
  all_blocks([&](int h4, int, float lo, float hi) { m[h4] = min3(m[h4], lo, hi); });
#pragma unroll
  for (int h4 = 0; h4 < 4; ++h4) m[h4] = quad_min(m[h4]);
  xd[hf * kKeys + q * 32 + g + 8 * t4] = pick4(m, t4);
  asm volatile("bar.sync %0, 64;" ::"r"(q + 1) : "memory");   // the two warps that share these keys
  float lim[4];
  {
    // The MMA accumulates k.c in fp32: its error is a small multiple of 2^-24 * ||k|| * ||c||, which
    // 2e-4 * (||k||^2 + max ||c||^2) bounds with a wide margin.
    const float knorm = xkn[r] + xkn[kKeys + r], cmax = __uint_as_float(*cmax_bits);
    const float l = fminf(xd[r], xd[kKeys + r]) + 2e-4f * (knorm + cmax);
#pragma unroll
    for (int h4 = 0; h4 < 4; ++h4) lim[h4] = __shfl_sync(0xffffffffu, l, g + 8 * h4);
  }
  // ---- the columns within that of the minimum: one, as a rule
  float hits[4] = {0.f, 0.f, 0.f, 0.f};
  {
    const float col0 = (float)(256 + hf * MH + 2 * t4);
    all_blocks([&](int h4, int c, float lo, float hi) {
      const float w0 = col0 + (float)c;
      if (lo <= lim[h4]) hits[h4] += w0;
      if (hi <= lim[h4]) hits[h4] += w0 + 1.f;
    });
  }
#pragma unroll
  for (int h4 = 0; h4 < 4; ++h4) hits[h4] = quad_sum(hits[h4]);
  xs[hf * kKeys + q * 32 + g + 8 * t4] = pick4(hits, t4);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1 && !has_next) tmem_dealloc(tmem_base, tmem_cols);
  const __nv_bfloat16* Cph = Cp + (size_t)h * M * D;
  if (hf == 0) {
    int i1;
    bool open;                                       // more than one parent within the MMA's rounding of the nearest
    if constexpr (FORM == kSmall) {                  // (the lower half holds the lower indices: it wins ties)
      const float a1 = xd[r], a2 = xs[r], b1 = xd[kKeys + r], b2 = xs[kKeys + r];
      i1 = b1 < a1 ? chi[r] : par[r];
      const float close = 2e-4f * (xkn[r] + xkn[kKeys + r] + __uint_as_float(*cmax_bits));
      open = !(fminf(fmaxf(a1, b1), fminf(a2, b2)) - fminf(a1, b1) > close);
    } else {
      const float s = xs[r] + xs[kKeys + r];         // < 512: a single column, 256 + index
      open = !(s >= 256.f && s < 512.f);
      i1 = open ? 0 : (int)s - 256;
    }
    if (done && j0 + r < Nk && open) {
      double best = INFINITY;
      int bi = 0;
      for (int mm = 0; mm < M; ++mm) {
        const double sd = exact_dist_smem<D>(Ks, r, Cph + (size_t)mm * D);
        if (sd < best) { best = sd; bi = mm; }
      }
      i1 = bi;
    }
    par[r] = i1;
    if constexpr (SORTED) {
      if (STAYS) xd[r] = open ? NAN : fminf(xd[r], xd[kKeys + r]);   // distance to the parent, less ||k||^2
      // ---- the keys in the order of their parents (within a parent any): counting sort by the warps of the lower half
      const int rank = atomicAdd(&hist[i1], 1);
      asm volatile("bar.sync 5, 128;" ::: "memory");
      const int per = M >> 5;                          // bins per lane
      int before = 0, n = 0;
      for (int u = 0; u < per; ++u) n += hist[lane * per + u];
      before = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, before, o);
        if (lane >= o) before += up;
      }
      before -= n;
      if (lane >> 3 == q)                              // a quarter of the bins per warp
        for (int u = 0; u < per; ++u) {
          offs[lane * per + u] = before;
          before += hist[lane * per + u];
        }
      asm volatile("bar.sync 5, 128;" ::: "memory");
      order[offs[i1] + rank] = (uint8_t)r;
    }
  }
  __syncthreads();

  if constexpr (SORTED) {
    // ---- children, SORTED: a warp takes 16 keys in the order of their parents.  k . c for all 16 and the children of
    // each parent among them, one (eight children) or two (four) parents per warp-level tensor-core product: 16 keys x 8
    // children; a key takes the columns of its own parent.  Both operands hold the head dimension in the order in which a lane
    // reads 16-byte chunks (lane t of a quad: chunks t, t + 4, ...).  The distance to the parent comes from the parents' products.
    // Bound by the latency of the child rows, one product ahead (the rule and what both forms take: beside the launch).
    constexpr int kC = NL * 256 / D;                   // children per parent (4 or 8)
    constexpr int kPar = 8 / kC;                       // parents per product
    constexpr int kB = D / 32;                         // 16-byte chunks per lane and row
    const int mk = order[warp * 16 + (lane & 15)], mp = par[mk];
    const int prev = __shfl_up_sync(0xffffffffu, mp, 1);
    const uint32_t heads = __ballot_sync(0xffffffffu, lane < 16 && (lane == 0 || mp != prev));   // first key of each parent
    const int nd = __popc(heads);
    int key[2], own[2], cid[2];                        // rows g, g + 8: key, parent, this lane's first child of it
    bool mine[2];                                      // this lane holds children of the row's own parent
    int ord[2];                                        // which of the parents the row's is
    uint4 ka[2][kB];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      key[i] = __shfl_sync(0xffffffffu, mk, g + 8 * i);
      own[i] = __shfl_sync(0xffffffffu, mp, g + 8 * i);
      ord[i] = __popc(heads & ((2u << (g + 8 * i)) - 1u)) - 1;
      mine[i] = kPar == 1 || (ord[i] & 1) == (t4 >> 1);
      cid[i] = kPar == 1 ? 2 * t4 : 2 * (t4 & 1);
#pragma unroll
      for (int b = 0; b < kB; ++b) {
        const int ch = t4 + 4 * b;
        ka[i][b] = *reinterpret_cast<const uint4*>(Ks + (ch >> 3) * (kKeys * 128) + sw128_offset(key[i], (ch & 7) * 8));
      }
    }
    const size_t head_base = (size_t)h * M;
    float nrm[2][2], dot[2][2];                        // of children cid, cid + 1
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      dot[i][0] = dot[i][1] = nrm[i][0] = nrm[i][1] = 0.f;
      if constexpr (TABLE) {
        const float2 n2 = ld_after_wait(reinterpret_cast<const float2*>(cnorm_g + (size_t)H * M + (head_base + own[i]) * kC + cid[i]));
        nrm[i][0] = n2.x;
        nrm[i][1] = n2.y;
      }
    }
    uint32_t rest = heads;
    auto fetch = [&](uint4 (&z)[kB]) {                 // the next product's children: lane 4 g + t, row g
      int src = __ffs(rest) - 1;
      rest &= rest - 1;
      if constexpr (kPar == 2) {
        if (rest && g >= 4) src = __ffs(rest) - 1;
        rest &= rest - 1;
      }
      const int pp = __shfl_sync(0xffffffffu, mp, src);
      const uint4* row = reinterpret_cast<const uint4*>(Cc + ((head_base + pp) * kC + (g & (kC - 1))) * D) + t4;
#pragma unroll
      for (int b = 0; b < kB; ++b) z[b] = __ldg(row + 4 * b);
    };
    auto product = [&](const uint4 (&z)[kB], int u) {
      float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int b = 0; b < kB; ++b) {
        mma_bf16(c, ka[0][b].x, ka[1][b].x, ka[0][b].y, ka[1][b].y, z[b].x, z[b].y);
        mma_bf16(c, ka[0][b].z, ka[1][b].z, ka[0][b].w, ka[1][b].w, z[b].z, z[b].w);
      }
      float n0 = 0.f, n1 = 0.f;
      if constexpr (!TABLE) {                          // ||c||^2 of row g, then of this lane's columns 2 t, 2 t + 1
        float n = 0.f;
#pragma unroll
        for (int b = 0; b < kB; ++b) n = norm_bf16x8(n, z[b]);
        n = quad_sum(n);
        n0 = __shfl_sync(0xffffffffu, n, 8 * t4);
        n1 = __shfl_sync(0xffffffffu, n, 8 * t4 + 4);
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (ord[i] / kPar == u) {
          dot[i][0] = c[2 * i];
          dot[i][1] = c[2 * i + 1];
          if constexpr (!TABLE) { nrm[i][0] = n0; nrm[i][1] = n1; }
        }
    };
    uint4 z[2][kB];
    fetch(z[0]);
    for (int u = 0; u * kPar < nd; u += 2) {
      if ((u + 1) * kPar < nd) fetch(z[1]);
      product(z[0], u);
      if ((u + 1) * kPar < nd) {
        if ((u + 2) * kPar < nd) fetch(z[0]);
        product(z[1], u + 1);
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float a = mine[i] ? fmaf(-2.f, dot[i][0], nrm[i][0]) : INFINITY;
      const float b = mine[i] ? fmaf(-2.f, dot[i][1], nrm[i][1]) : INFINITY;
      float e1 = fminf(a, b), e2 = fmaxf(a, b);
      int c1 = b < a ? cid[i] + 1 : cid[i];
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        const float b1 = __shfl_xor_sync(0xffffffffu, e1, o);
        const float b2 = __shfl_xor_sync(0xffffffffu, e2, o);
        const int cb = __shfl_xor_sync(0xffffffffu, c1, o);
        e2 = fminf(fmaxf(e1, b1), fminf(e2, b2));
        if (b1 < e1 || (b1 == e1 && cb < c1)) { e1 = b1; c1 = cb; }
      }
      // Closer than this two distances are measured again, in the direct form in float32 and then in float64.  A tensor-core
      // product adds 16 exact products to the sum and rounds each of the 17 terms by at most 2^-24 of the largest of them and
      // of the sum: D / 16 steps are off by at most 17 D / 16 2^-24 |k||c|, the norm (chains of at most D / 4 and three
      // additions) by (D/4 + 3) 2^-24 |c|^2, so a distance by less than 1.05e-5 (|k|^2 + |c|^2) at D = 128 and two of them by
      // less than 2.1e-5 (|k|^2 + max |c|^2).  A parent's norm is one chain of D where there is no table, off by 7.7e-6 |c|^2:
      // its distance and a child's together by less than 3.3e-5 |k| |c| + 1.0e-5 |c|^2 with the larger |c|, which is
      // below 2.5e-5 (|k|^2 + |c|^2) for every |k| and |c| (2.5 k^2 - 3.3 k c + 1.5 c^2 has no zero).
      float cmx = mine[i] ? fmaxf(nrm[i][0], nrm[i][1]) : 0.f;
      cmx = quad_max(cmx);
      if (STAYS) cmx = fmaxf(cmx, cnorm[own[i]]);
      const float near = 2.5e-5f * (xkn[key[i]] + xkn[kKeys + key[i]] + cmx);
      const bool live = done && j0 + key[i] < Nk;
      const bool open = live && !(e2 - e1 > near);     // not decided by the products
      const float dp = STAYS ? xd[key[i]] : INFINITY;  // the parent's distance (NaN where that was decided in float64)
      const bool moved = !STAYS || e1 < dp;            // strictly closer
      const bool stay_open = STAYS && live && !(fabsf(e1 - dp) > near);
      if (__any_sync(0xffffffffu, open || stay_open))
        c1 = settle_child<D, kC>(Ks, key[i], t4, Cc + (head_base + own[i]) * kC * D, Cp + (head_base + own[i]) * D, c1, open,
                                 stay_open, moved);
      else if (!moved)
        c1 = -1;
      if (t4 == 0) chi[key[i]] = c1;
    }
  } else {
    // ---- child argmin, four lanes per key: a warp takes 8 keys at a time (two passes over its 16 keys).
    // Lane s of a key's group covers the 16-byte chunks s, s + 4, ... of the key row and of each of the
    // parent's C children (the group reads 64 contiguous bytes of a child row per load), keeps one running
    // sum per child, and a transposing butterfly over the four lanes leaves child s (and s + 4) in lane s.
    // The loads of the next chunk column are in flight while the current one is squared.
    constexpr int kC = NL * 256 / D;                   // children per parent (4 or 8), four at a time
    constexpr int kChunks = D / 8;                     // 16-byte chunks per row
    constexpr int kT = kChunks / 4;                    // chunk columns per lane (2 or 4)
    constexpr int kF = kC / 4;                         // groups of four children
    constexpr int kSteps = 2 * kT * kF;                // (pass, chunk column, group) triples
    const int s4 = lane & 3, grp = lane >> 2;
    const size_t head_base = (size_t)h * M;
    uint4 buf4[2][4];
    auto issue = [&](int step, uint4 (&dst)[4]) {
      const int key = warp * 16 + (step / (kT * kF)) * 8 + grp;
      const uint4* src = reinterpret_cast<const uint4*>(Cc + ((head_base + par[key]) * kC + 4 * (step % kF)) * D) +
                         (s4 + 4 * ((step / kF) % kT));
#pragma unroll
      for (int c = 0; c < 4; ++c) dst[c] = __ldg(src + c * kChunks);
    };
    float sum[kC];
    issue(0, buf4[0]);
    float ncv[2][kC / 4];                                // TABLE: norms of child s4 (and s4 + 4) of this lane's keys
    if constexpr (TABLE) {
#pragma unroll
      for (int pass = 0; pass < 2; ++pass)
#pragma unroll
        for (int i = 0; i < kC / 4; ++i)
          ncv[pass][i] = ld_after_wait(cnorm_g + (size_t)H * M + (head_base + par[warp * 16 + pass * 8 + grp]) * kC + s4 + 4 * i);
    }
    typename std::conditional<TABLE, uint4, KeyChunk>::type kv;
#pragma unroll
    for (int step = 0; step < kSteps; ++step) {
      const int pass = step / (kT * kF), t = (step / kF) % kT, f = step % kF;
      const int key = warp * 16 + pass * 8 + grp;
      if (step + 1 < kSteps) issue(step + 1, buf4[(step + 1) & 1]);
      if (t == 0 && f == 0) {
#pragma unroll
        for (int c = 0; c < kC; ++c) sum[c] = 0.f;
      }
      const int ch = s4 + 4 * t;
      if (f == 0) {
        const uint4 kw = *reinterpret_cast<const uint4*>(Ks + (ch >> 3) * (kKeys * 128) + sw128_offset(key, (ch & 7) * 8));
        if constexpr (TABLE) kv = kw;
        else kv = widen8(kw);
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if constexpr (TABLE) dot_bf16x8(sum[4 * f + c], kv, buf4[step & 1][c]);
        else sum[4 * f + c] += sqdiff8(kv, buf4[step & 1][c]);
      }
      if (t == kT - 1 && f == kF - 1) {
        // transpose-reduce over the group: after the two exchanges lane s holds the total of child s
        // (and of child s + 4 when C = 8)
        const bool hi1 = (s4 & 1) != 0, hi2 = (s4 & 2) != 0;
        float r[kC / 2];
  #pragma unroll
        for (int i = 0; i < kC / 2; ++i) {
          const float send = hi1 ? sum[2 * i] : sum[2 * i + 1];
          const float keep = hi1 ? sum[2 * i + 1] : sum[2 * i];
          r[i] = keep + __shfl_xor_sync(0xffffffffu, send, 1);
        }
        float tot[kC / 4];
  #pragma unroll
        for (int i = 0; i < kC / 4; ++i) {
          const float send = hi2 ? r[2 * i] : r[2 * i + 1];
          const float keep = hi2 ? r[2 * i + 1] : r[2 * i];
          tot[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
        }
        // Closer than this two distances are decided in float64.  Direct form: relative.  With the table: the dot
        // product is a chain of D / 4 exact products in fp32 and two additions, the norms one of D / 8 and three, so a
        // distance is off by at most 2 (D/4 + 2) 2^-24 |k||c| + (D/8 + 3) 2^-24 |c|^2 < 3.3e-6 (|k|^2 + |c|^2) at D = 128,
        // two of them by less than 1e-5 (|k|^2 + max |c|^2).
        float near = 0.f;
        if constexpr (TABLE) {
          float cmx = 0.f;
#pragma unroll
          for (int i = 0; i < kC / 4; ++i) {
            cmx = fmaxf(cmx, ncv[pass][i]);
            tot[i] = fmaf(-2.f, tot[i], ncv[pass][i]);
          }
          cmx = quad_max(cmx);
          near = 1e-5f * (xkn[key] + xkn[kKeys + key] + cmx);
        }
        float e1 = tot[0], e2 = INFINITY;
        int c1 = s4;
        if constexpr (kC == 8) {
          e2 = fmaxf(tot[0], tot[1]);
          if (tot[1] < tot[0]) { e1 = tot[1]; c1 = s4 + 4; }
        }
  #pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
          const float b1 = __shfl_xor_sync(0xffffffffu, e1, o);
          const float b2 = __shfl_xor_sync(0xffffffffu, e2, o);
          const int cb = __shfl_xor_sync(0xffffffffu, c1, o);
          e2 = fminf(fmaxf(e1, b1), fminf(e2, b2));
          if (b1 < e1 || (b1 == e1 && cb < c1)) { e1 = b1; c1 = cb; }
        }
        if constexpr (TABLE) {
          const bool live = done && j0 + key < Nk;
          const bool open = live && !(e2 - e1 > near);   // not decided by the products
          const __nv_bfloat16* Cch = Cc + (head_base + par[key]) * kC * D;
          if (__any_sync(0xffffffffu, open)) {
            double best = INFINITY;
            int bi = 0;
            for (int c = 0; c < kC; ++c) {
              const double sd = exact4<D>(Ks, key, s4, Cch + (size_t)c * D);
              if (sd < best) { best = sd; bi = c; }
            }
            if (open) c1 = bi;
          }
          if (s4 == 0) chi[key] = c1;
        } else if (s4 == 0) {
          double best = INFINITY;
          if (done && j0 + key < Nk && !(e2 - e1 > 1e-4f * e2)) {
            const __nv_bfloat16* Cch = Cc + (head_base + par[key]) * kC * D;
            int bi = 0;
            for (int c = 0; c < kC; ++c) {
              const double sd = exact_dist_smem<D>(Ks, key, Cch + (size_t)c * D);
              if (sd < best) { best = sd; bi = c; }
            }
            c1 = bi;
          }
          chi[key] = c1;
        }
      }
    }
  }
  __syncthreads();
  // When a wait above gave up the indices are meaningless, but they are in range (both argmins start
  // from index 0 and only take loop indices), so the kernels behind this one read nothing out of bounds;
  // they see the recorded status word and skip their work.
  if (tid < kKeys && j0 + tid < Nk) {
    pidx[(size_t)bh * Nk + j0 + tid] = par[tid];
    cidx[(size_t)bh * Nk + j0 + tid] = chi[tid];
  }
  // every thread is past its last read of this key tile (and of the codebook): refill
  if (warp == 0 && has_next && elect_one()) {
    load_keys(nbh, nblk_);
    if (next_new_head) {
      *cmax_bits = 0;
      load_codes(nbh);
    }
  }
  new_head = next_new_head;
  bh = nbh;
  blk = nblk_;
  if (!has_next) break;
  if (next_new_head) __syncthreads();                // cmax_bits is clear
  }   // tiles
  if (beside) pdl_wait();    // this grid's completion then implies that of the one it ran beside
}

int sm_count() {                                      // of the current device; 0: unknown
  static int known[64] = {};
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (dev >= 0 && dev < 64 && known[dev] > 0) return known[dev];
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  if (dev >= 0 && dev < 64) known[dev] = n;
  return n;
}

uint32_t pow2_cols(int n) {
  uint32_t c = 32;
  while ((int)c < n) c <<= 1;
  return c;
}

template <int D, int NL, bool STAYS, Form FORM, bool TABLE, bool SORTED>
avq_status launch_kernel(const CUtensorMap& tmK, const CUtensorMap& tmCp, const avq_problem& p, const void* Cp,
                         const void* Cc, int32_t* pidx, int32_t* cidx, int32_t* status_word, void* zero_base,
                         size_t zero_bytes, const float* cnorm, bool beside, int nblk, int total, size_t smem,
                         unsigned grid, cudaStream_t st) {
  auto kern = tc_assign_kernel<D, NL, STAYS, FORM, TABLE, SORTED>;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return AVQ_ERR_CUDA;
  const avq_status s = open_shared_memory<tc_assign_kernel<D, NL, STAYS, FORM, TABLE, SORTED>>(dev);
  if (s != AVQ_OK) return s;
  // launched as a dependent of the norms kernel when there is one: set-up, loads and the MMA overlap it
  return cuda_ok(launch_pdl(kern, dim3(grid), dim3(kThreadsA), smem, st, cnorm != nullptr || beside, tmK, tmCp,
                            static_cast<const __nv_bfloat16*>(Cp), static_cast<const __nv_bfloat16*>(Cc), pidx, cidx,
                            p.H, p.Nk, p.M, nblk, total, pow2_cols(p.M), status_word,
                            static_cast<uint4*>(zero_base), zero_bytes / 16, slice_units(zero_bytes / 16, grid), cnorm, beside ? 1 : 0));
}

template <int D, int NL, bool STAYS>
avq_status launch(const avq_problem& p, const void* K, const void* Cp, const void* Cc, int32_t* pidx,
                  int32_t* cidx, int32_t* status_word, void* zero_base, size_t zero_bytes, float* cnorm, bool beside,
                  cudaStream_t st) {
  CUtensorMap tmK, tmCp;
  const uint64_t BH = (uint64_t)p.B * p.H;
  {
    const uint64_t dims[3] = {(uint64_t)D, (uint64_t)p.Nk, BH};
    const uint32_t box[3] = {64, (uint32_t)kKeys, 1};
    avq_status s = make_tmap_bf16(&tmK, K, 3, dims, box);
    if (s != AVQ_OK) return s;
  }
  {
    const uint64_t dims[2] = {(uint64_t)D, (uint64_t)p.H * p.M};
    const uint32_t box[2] = {64, (uint32_t)p.M};
    avq_status s = make_tmap_bf16(&tmCp, Cp, 2, dims, box);
    if (s != AVQ_OK) return s;
  }
  // Children by products over sorted keys.  Under PARENT_STAYS, where the loop over each key's children reads the parent's row as
  // well, always (us per call, loop and products: B2 H8 N5000 d128 M96 C8 98.3 and 88.4, H12 N400 d128 M256 C8 67.7 and 47.7,
  // B8 H12 N10167 d64 M32 C8 268 and 230, B2 H16 N4096 d64 M128 C8 81.0 and 77.1, H16 N65536 d64 M256 C4 700 and 700).  Where
  // every key moves, for eight children and grids that hide the sort: d128 H16 N20000 M32 167.7 and 142.6, M64 179.5 and
  // 157.8, M128 247.5 and 234.7, M256 303.4 and 299.4; 288 tiles M64 34.4 and 33.3, M256 56.2 and 53.9, but 48 tiles M64 23.3
  // and 24.0; d64 H16 N20000 M32 92.0 and 85.1, M64 111.3 and 105.4, M128 144.9 and 142.6, M256 224.0 and 224.8; 288 tiles M64
  // 25.7 and 26.5.  Those keys crowd around few parents; where every parent has as many, a warp's 16 keys have more parents and
  // the products gain less: with the norm table H16 N20000 d64 M64 112.4 and 108.6, M128 140.1 and 143.8, d128 M128 246.5 and
  // 245.2; without it, this kernel alone, d64 M64 45.6 and 45.5, M96 48.6 and 52.0, M128 50.3 and 56.4 (crowded keys 49.6 and
  // 49.6), d128 M128 90.6 and 92.7 (91.8 and 82.0).  So at d64 not above 64 parents without the table.  With four children the two about cancel or products lose: d64 H16 N20000 M64 96.5 and 97.9, M256 204.5
  // and 211.5; d128 M128 215.0 and 214.5, M256 256.8 and 259.8.
  constexpr bool kSortedAtAll = STAYS || NL * 256 / D == 8;
  const int nblk = (p.Nk + kKeys - 1) / kKeys;
  if ((uint64_t)nblk * BH > 0x7fffffffull) return AVQ_ERR_UNSUPPORTED;
  const int total = (int)(nblk * BH);
  const int sms = sm_count();
  if (sms <= 0) return AVQ_ERR_CUDA;
  const bool sorted = STAYS || (kSortedAtAll && (D == 128 ? 2 * total >= 3 * sms : total >= 4 * sms && p.M <= (cnorm ? 128 : 64)));
  const size_t smem = (size_t)(D / 64) * (kKeys + p.M) * 128 + sizeof(float) * (p.M + 6 * kKeys) + sizeof(int) * (2 * kKeys + (sorted ? p.M + kKeys / 4 : 0)) + 96;
  const int resident = (int)min((size_t)assign_min_ctas(D), kSmemMax / (smem + 1024));   // CTAs on an SM
  // A wave of CTAs with runs of tiles, the codebook and its norms staying in shared memory, for the largest codebook
  // (64 KB: d128 M256) from four tiles per CTA on (N16384 H16, 6.9 tiles: 72 -> 63 us); with fewer the uneven last round
  // costs more than the set-up it saves (B2 H8 N5000 d128 M96, 2.2 tiles: whole call 111 -> 130 us).  Below M256 the gain
  // is smaller (H16 N16384 d128 C4, whole call with one tile per CTA and with runs: M64 126 and 123, M128 182 and 178, M224
  // 229 and 222) and runs are not taken.  At d64 they cost: M32 by their loop state (B8 H12 N10167: this kernel 122 us and
  // 130), M256 because the resident CTAs take the TMEM columns in turn (N65536: whole call 780 and 960).
  const bool runs = D == 128 && p.M == 256 && (int64_t)total >= 4ll * resident * sms;
  if (cnorm) {
    const int parents = p.H * p.M, rows = parents * (1 + p.C);
    if (launch_pdl(code_norms_kernel<D>, dim3((rows * 8 + 255) / 256), dim3(256), 0, st, beside,
                   static_cast<const __nv_bfloat16*>(Cp), static_cast<const __nv_bfloat16*>(Cc), cnorm, parents,
                   rows) != cudaSuccess)
      return AVQ_ERR_CUDA;
  }
  // Up to 64 parents the fragment layout's exchanges cost more than its cheaper columns save (this kernel alone, us, fragments
  // and a key per lane: H16 d64 C4 N65536 M32 97.8 and 95.2, M64 106.2 and 104.5; d128 N16384 M32 54.0 and 51.9, M64 56.0 and
  // 54.6; beyond, in the form the kernel had with a key per lane throughout: d64 M128 118.5 and 120.8, M256 151 and 166).
  // With the norm table at d64 the loop behind has no registers to spare (whole call N65536 M64 C8: 301.7 and 304.5).
  const bool small = p.M <= 64 && !(D == 64 && cnorm);
  constexpr Form kSmallTable = D == 64 ? kOne : kSmall;
  auto choose = [&](auto sorted_) {
    constexpr bool kSorted = decltype(sorted_)::value;
    auto go = cnorm ? (small ? launch_kernel<D, NL, STAYS, kSmallTable, true, kSorted> : launch_kernel<D, NL, STAYS, kOne, true, kSorted>)
                    : (small ? launch_kernel<D, NL, STAYS, kSmall, false, kSorted> : launch_kernel<D, NL, STAYS, kOne, false, kSorted>);
    if constexpr (D == 128)
      if (runs) go = cnorm ? launch_kernel<D, NL, STAYS, kRuns, true, kSorted> : launch_kernel<D, NL, STAYS, kRuns, false, kSorted>;
    return go;
  };
  auto go = choose(std::integral_constant<bool, STAYS>{});
  if constexpr (kSortedAtAll && !STAYS)
    if (sorted) go = choose(std::true_type{});
  return go(tmK, tmCp, p, Cp, Cc, pidx, cidx, status_word, zero_base, zero_bytes, cnorm, beside, nblk, total, smem,
            (unsigned)(runs ? resident * sms : total), st);
}

}  // namespace

avq_status tc_assign(const avq_problem& p, const void* K, const void* Cp, const void* Cc,
                     int32_t* parent_idx, int32_t* child_idx, int32_t* status_word, void* zero_base,
                     size_t zero_bytes, float* cnorm, bool beside, cudaStream_t st) {
  if (zero_bytes % 16 != 0) return AVQ_ERR_WORKSPACE;
  const bool stays = (p.flags & AVQ_FLAG_PARENT_STAYS) != 0;
#define AVQ_ASSIGN(DD, NN)                                                                                     \
  (stays ? launch<DD, NN, true>(p, K, Cp, Cc, parent_idx, child_idx, status_word, zero_base, zero_bytes, cnorm, beside, st) \
         : launch<DD, NN, false>(p, K, Cp, Cc, parent_idx, child_idx, status_word, zero_base, zero_bytes, cnorm, beside, st))
  if (p.d == 64) return p.C == 4 ? AVQ_ASSIGN(64, 1) : AVQ_ASSIGN(64, 2);
  return p.C == 4 ? AVQ_ASSIGN(128, 2) : AVQ_ASSIGN(128, 4);
#undef AVQ_ASSIGN
}

}  // namespace avq
