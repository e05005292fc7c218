// Tensor-core attention pass of AVQ-attention (Algorithm 2 in its masked form) for bf16 inputs.
//
// One CTA = one query tile of 128 rows of one (batch, head) at a time; 4 NQ warps, warp w holds rows
// 32 (w % 4) .. +31 of the column slice w / 4.  Inside a warp the accumulator is read in the layout of an MMA
// result (tcgen05.ld.16x256b): lane 4 g + t holds rows g, g + 8, g + 16, g + 24 and column pairs 2 t, 2 t + 1 of every
// 8-column block.  Against one row per lane this (a) needs a quarter of the per-column operands (bias, counts) per
// thread, (b) sums a column over its rows mostly in registers (14 shuffles per 64 columns instead of 62), (c) puts
// neighbouring columns into neighbouring registers for the packed fp32 instructions and for the weights' stores.
// Parent codewords (and their value rows) stand in an order of their own in shared memory: inside every group of 8
// rows, codeword 4 v + t at row 2 t + v (the tensor map does it), so that lane t of a quad holds the codewords t,
// t + 4, t + 8, ... of its slice and the denominator's four partial sums stay what they are with one row per lane:
// which parents are selected does not depend on the layout.
// Values enter as per-codeword MEANS with the key counts multiplied into the weights.
// Flow of a tile:
//   parents   S = Q . Cp^T                 tcgen05.mma, fp32 accumulator in TMEM, issued at the end of the tile before
//             read once into registers: row maximum over non-empty parents, exp2, exact denominator z
//                                                                   (Eq. "vqflashattention")
//             importance w_j = n_j sum_i A_ij / z_i from the fp32 weights  (Eq. "importance")
//             top-P, ties to the lower index                        ("Child spawning")
//             bf16 weights A_ij n_j (zero for a refined parent) -> A operand
//             O = (A n) . mean_p           tcgen05.mma
//   children  of the selected parents, in chunks of <= CHW columns: gathered codeword rows,
//             S_c = Q . Cc_sel^T, bf16 weights, O += A_c . Vbar_c   (Algorithm 2, child loop); O is rescaled in
//             TMEM only if the children's weights against the row's reference pass 2^64 (2^8 where a mean exceeds 2^40)
//   Y = O / z, z accumulated from the same bf16-rounded weights as the numerator.
// Empty codewords are excluded from every maximum and contribute nothing (their logit is -inf, their count and
// value sum are zero) - appendix on numerical stability.
// A CTA takes a run of consecutive tiles: codebook, parent values and counts stay in shared memory while the
// (batch, head) does not change.
// Bound by the latency of a tile's phases one after the other (issue slots about half used, tensor pipe 7 to 17 %, no
// memory above a third), not by the tensor cores.  Against one
// row per lane with the weights in shared memory: B1 H16 N16384 d128 M256 C4 P32 183 -> 148 us (floor 31.5, tensor),
// N65536 d64 M256 P64 827 -> 615, B2 H16 N4096 d64 M128 C8 P16 43.5 -> 37.
#include "avq_tc_common.cuh"

namespace avq {
namespace {

using namespace tc;

constexpr int kRows = 128;
// shared-memory row / TMEM column of parent codeword c
__device__ __forceinline__ int parent_pos(int c) { return (c & ~7) | ((c & 3) << 1) | ((c >> 2) & 1); }

struct AttendParams {
  const __nv_bfloat16* Cc;    // [H, M, C, d]
  const __nv_bfloat16* Vcb;   // [B*H, M, C, d]
  const __nv_bfloat16* Vsb;   // [B*H, M, d]  PARENT_STAYS: value sum of the keys that stay / all keys of the parent
  const float* rho;           // [B*H, M]     PARENT_STAYS: keys that stay / all keys of the parent (else nullptr)
  const float* np_;           // [B*H, M]
  const float* nc;            // [B*H, M, C]
  __nv_bfloat16* Y;           // [B*H, Nq, d]
  int32_t* topp_out;          // optional
  float* importance_out;      // optional
  int32_t* status_word;
  const int32_t* perm;        // Y row of query i of the head is perm[i] (else nullptr; an entry out of range is flagged and skipped)
  int H, Nq, M, C, P, nblk;
  int total_tiles;            // nblk * B * H
  int logC;                   // log2(C)
  float scale_log2e;
};

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// The NQ warps that share a quarter of the rows (warp % 4 == q) exchange per-row values through shared
// memory; they synchronise among themselves on named barrier q + 1 instead of stalling the whole CTA.
template <int NQ>
__device__ __forceinline__ void row_sync(int q) {
  asm volatile("bar.sync %0, %1;" ::"r"(q + 1), "r"(32 * NQ) : "memory");
}

// Shared-memory and TMEM plan of one instantiation.
// NQ = warps (column slices) per 32 query rows: 1, 2 or 4.  Small tiles take NQ = 1 so that four CTAs share an SM and
// overlap each other's load / MMA / softmax phases; the largest take NQ = 4.
// CT = parent tile width (32, 64, 128 or 256, >= M), a compile-time constant so that every shared-memory
// offset folds into the instruction stream instead of occupying a register.
template <int D, int NQ, int CT>
struct Plan {
  static constexpr int kThreads = 128 * NQ;
  static constexpr int kSubD = D / 64;
  static constexpr int CHW = CT < 128 ? CT : 128;        // child chunk width
  static constexpr int QT = kSubD * kRows * 128;         // bytes of a query / output tile
  // Weights as the A operand in TMEM: nothing to swizzle or fence, the MMA reads half the shared memory, and the
  // codebook survives the tile.  64 parents with one warp per row have no TMEM columns left (four CTAs of 128 columns share
  // an SM): their weights overwrite the codebook in shared memory, which is then loaded again (8 KB).
  static constexpr bool kTW = !(CT == 64 && D == 64 && NQ == 1);
  // The children's codes and value rows have a buffer each, so that both gathers run ahead of the logits.  The largest
  // tile has room for the values only: the codes go over the parent codebook, whose logits are done by then, and the
  // overwritten half of the codebook is loaded again behind the child logits.  The tile without weights in TMEM gathers
  // the values into the codes' place once the child logits are done (four CTAs fill each other's gaps).
  static constexpr bool kCodesInCA = CT == 256 && D == 128;
  static constexpr bool kSepCV = kTW;
  // The output tile is staged in the child buffers, padded to its size where needed, or, without buffers for both, across
  // the parent values and the child buffer (the parent values are then loaded again).
  static constexpr bool kStageInCC = CT >= 128 || kSepCV;
  static constexpr int child_bytes = CHW * D * 2 * (kSepCV && !kCodesInCA ? 2 : 1);
  static constexpr int stage_pad = kStageInCC && child_bytes < QT ? QT - child_bytes : 0;   // (32 parents only)
  static constexpr int cp_bytes = CT * D * 2;
  static constexpr int ca_bytes = kTW ? cp_bytes : (cp_bytes > kRows * CT * 2 ? cp_bytes : kRows * CT * 2);
  static constexpr int oQ = 0, oCA = QT, oV = oCA + ca_bytes, oCC = oV + CT * D * 2,
                       oCV = oCC + (kSepCV && !kCodesInCA ? CHW * D * 2 : 0);
  static constexpr int oStage = kStageInCC ? oCC : oV;
  static constexpr int oF = oCV + CHW * D * 2 + stage_pad;   // fp32 / word arrays from here
  // Plans of twice the warps per tile (small grids): two neighbouring warps of a row add the denominator as the one warp of
  // the other plan does, the second going on from the first's sums, so that which parents are selected does not depend on
  // how many tiles a call has.
  static constexpr bool kChain = D == 64 && NQ > 1 && CT / NQ == 32;
  static constexpr int chain_floats = kChain ? NQ / 2 * 4 * kRows : 0;
  // TMEM columns: logits, weights (kTW), output.  With 256 logit columns the child logits use half of them and the
  // children's weights go into the other half, so they need not wait for the parents' value MMA.
  static constexpr bool kSepW = CT == 256;
  static constexpr int tW = kTW ? CT : 0, tWc = kSepW ? 128 : tW, tO = CT == 32 ? 64 : (kTW ? CT + CT / 2 : CT);
  static constexpr int tmem_used = tO + D;
  static constexpr uint32_t tmem_cols = tmem_used <= 128 ? 128 : (tmem_used <= 256 ? 256 : 512);
  static_assert(kStageInCC || CT * D * 2 + CHW * D * 2 >= QT, "the output tile fits its staging area");
};

template <int D, int NQ, int CT>
size_t attend_smem(int MC) {
  using L = Plan<D, NQ, CT>;
  return L::oF + 4 * ((size_t)2 * CT + CT + L::CHW + CT + 4 * CT + 2 * NQ * kRows + 2 * CT + MC + CT + 32 + 18 + L::chain_floats) + 8 * 6 + 16;
}

// STAYS = the PARENT_STAYS rule: a refined parent keeps the keys that stayed with it.
// PERM = output rows go to p.perm's places (a branch at run time cost the plain call 1 us of 43).
template <int D, int NQ, int CT, bool STAYS, bool PERM>
__global__ void __launch_bounds__(128 * NQ, 4 / NQ)
tc_attend_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmCp,
                 const __grid_constant__ CUtensorMap tmVpb, const __grid_constant__ CUtensorMap tmY,
                 const AttendParams p) {
  // 1024-byte alignment (swizzle atoms) is requested from the launch, not computed from the pointer, so
  // that the compiler keeps every access in the shared address space.
  extern __shared__ __align__(1024) unsigned char smem[];
  using L = Plan<D, NQ, CT>;
  constexpr int kThreads = L::kThreads, kSubD = L::kSubD, CHW = L::CHW;
  constexpr bool kTW = L::kTW, kSepCV = L::kSepCV;
  constexpr int kVWarp = kThreads / 64;                  // issues S and the value MMAs (warp 0: child logits, TMA)
  constexpr int kLogD = (D == 128) ? 7 : 6;
  constexpr int kLogChunks = kLogD - 3;                  // 16-byte chunks per codeword row
  constexpr int QW = CT / NQ, QWC = CHW / NQ;
  constexpr int NB = QW / 8, NC = QW / 32;               // 8-column blocks and 32-column chunks of a warp's parents
  constexpr int NCC = QWC / 32;                          // and of its children
  const int M = p.M, C = p.C, P = p.P, logC = p.logC;
  unsigned char* Qs = smem + L::oQ;                      // kSubD x [128 x 128 B]
  unsigned char* CA = smem + L::oCA;                     // parent codes: kSubD x [M x 128 B] (kTW false: later the bf16 weights)
  unsigned char* Vs = smem + L::oV;                      // parent value rows: kSubD x [M x 128 B]
  unsigned char* CC = L::kCodesInCA ? CA : smem + L::oCC;   // gathered child codes: kSubD x [rows x 128 B]
  unsigned char* CV = smem + L::oCV;                     // gathered child values
  unsigned char* stage = smem + L::oStage;
  // per-parent operands, by column (parent_pos)
  float* cnt = reinterpret_cast<float*>(smem + L::oF);   // [CT] key counts
  float* bias = cnt + CT;                                // [CT] 0 for non-empty parents, -inf for empty
  // what a parent's term is multiplied by: default rule, the bf16 mask of its weight (0xFFFF, once refined 0);
  // PARENT_STAYS, the share of its own denominator term it keeps (1, once refined its stay share)
  float* keep_f = bias + CT;                             // [CT] STAYS
  uint16_t* keep_m = reinterpret_cast<uint16_t*>(keep_f);   // [CT] default rule
  float* l2n = keep_f + CT;                              // [CHW] log2 of the key counts of the child chunk
  float* w = l2n + CHW;                                  // [CT] importance, by parent
  float* wpart = w + CT;                                 // [4][CT] by column
  float* xm = wpart + 4 * CT;                            // [NQ][128] exchange between the warps of a row
  float* xz = xm + NQ * kRows;                           // [NQ][128]
  uint64_t* cand = reinterpret_cast<uint64_t*>(xz + NQ * kRows);   // [CT] top-P candidates
  float* ncs = reinterpret_cast<float*>(cand + CT);      // [M * C] log2 of the key counts of every child of this (b, h)
  int* sel_list = reinterpret_cast<int*>(ncs + M * C);   // [CT] refined parents
  int* wcount = sel_list + CT;                           // [32] keys at or above a sample key
  uint32_t* nzmask = reinterpret_cast<uint32_t*>(wcount + 32);   // [8] parents with an importance above zero
  uint32_t* selmask = nzmask + 8;                        // [8] refined parents
  int* ncand_s = reinterpret_cast<int*>(selmask + 8);    // candidates listed (+ 1 word of padding)
  uint64_t* bars = reinterpret_cast<uint64_t*>(ncand_s + 2);     // [6]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 6);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* zchain = reinterpret_cast<float*>(tmem_slot + 2);   // [NQ / 2][4][128] kChain
  // it is read in pieces of 16 bytes: the words in front of it, apart from the M C (M is a multiple of 32)
  static_assert(L::oF % 16 == 0 && (11 * CT + CHW + 2 * NQ * kRows + 32 + 8 + 8 + 2 + 2 * 6 + 2) % 4 == 0, "zchain is aligned");

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform
  const int q = warp & 3, cq = warp >> 2, r = q * 32 + lane;   // r: the row this lane stands for in exchanges
  const int g = lane >> 2, t4 = lane & 3;                // fragment rows q*32 + g + 8 h, column pairs 2 t4
  const int colbase = cq * QW;
  uint64_t* bar_q = &bars[0];                            // query tile landed
  uint64_t* bar_v = &bars[1];                            // parent value rows landed
  uint64_t* bar_s = &bars[2];                            // parent or child logits done
  uint64_t* bar_pv = &bars[3];                           // children's value MMA done
  uint64_t* bar_cp = &bars[4];                           // parent codebook landed
  uint64_t* bar_o = &bars[5];                            // parents' value MMA done
  auto issue_q = [&](int bh, int blk) {                  // one thread (as the next two)
    mbar_expect_tx(bar_q, (uint32_t)L::QT);
#pragma unroll
    for (int s = 0; s < kSubD; ++s) tma_load_3d(Qs + s * kRows * 128, &tmQ, s * 64, blk * kRows, bh, bar_q);
  };
  auto issue_cp = [&](int bh, int subs) {                // the first `subs` halves of the codebook
    mbar_expect_tx(bar_cp, (uint32_t)(subs * M * 128));
    for (int s = 0; s < subs; ++s) tma_load_codes(CA + s * M * 128, &tmCp, s * 64, ((bh % p.H) * M) >> 3, bar_cp);
  };
  auto issue_v = [&](int bh) {
    mbar_expect_tx(bar_v, (uint32_t)(kSubD * M * 128));
#pragma unroll
    for (int s = 0; s < kSubD; ++s) tma_load_codes(Vs + s * M * 128, &tmVpb, s * 64, (bh * M) >> 3, bar_v);
  };

  __shared__ int early_exit;
  __shared__ int wide;                                   // the aggregation met a mean beyond kWideMean, infinite or NaN
  // This CTA's run of consecutive tiles.  The CTAs with one tile more are the first ones of the grid: CTAs that
  // share an SM are a multiple of the SM count apart, so every SM gets its share of them.
  const int per = p.total_tiles / gridDim.x, more = p.total_tiles - per * gridDim.x;
  const int tile0 = (int)blockIdx.x * per + min((int)blockIdx.x, more);
  const int tile1 = tile0 + per + ((int)blockIdx.x < more ? 1 : 0);
  int bh = tile0 / p.nblk, blk = tile0 - bh * p.nblk;

  // ---- Part 1 touches only the caller's Q and Cp, so it may run while the kernel that produces the
  // aggregates is still finishing (programmatic dependent launch): barriers, TMEM, the Q / Cp loads and
  // S = Q . Cp^T.
  if (warp == 0 && elect_one()) {
    prefetch_tmap(&tmQ);
    prefetch_tmap(&tmCp);
    prefetch_tmap(&tmVpb);
#pragma unroll
    for (int i = 0; i < 6; ++i) mbar_init(&bars[i], 1);
    mbar_fence_init();
    *abort_flag = 0;
    if (PERM) pdl_wait();                                // Q is then the work of an earlier kernel of the call
    issue_q(bh, blk);
    issue_cp(bh, kSubD);
  }
  // TMEM is allocated before the dependency wait.  tcgen05.alloc blocks until the columns are free and the
  // wait returns only when the kernels before this one have finished; neither can hold the other up: the
  // columns an earlier kernel's CTAs own are released when those CTAs end, which needs nothing from this
  // kernel, and CTAs of this kernel release theirs on every path (including the early exit below).
  if (warp == 1) {                                   // not the warp whose lane is busy issuing the loads
    tmem_alloc(tmem_slot, L::tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16);
  const uint32_t t_s = t_row + (uint32_t)colbase;
  const uint32_t t_sc = t_row + (uint32_t)(cq * QWC);
  const uint32_t t_o = t_row + (uint32_t)(L::tO + cq * (D / NQ));
  const uint32_t idesc_o = umma_idesc_bf16(kRows, D) | (1u << 16);   // B (the value rows) is MN-major
  const float sc = p.scale_log2e;
  uint32_t ph_s = 0, ph_pv = 0, ph_v = 0, ph_o = 0;
  uint32_t ph_q = 0, ph_cp = 0;                          // used by the issuing warp
  const int PC = P * C;
  const int my_cols = min(max(M - colbase, 0), QW);      // multiple of 32

  // Q . rows^T into the logit columns.  (Descriptors count 16-byte units: 2 per 32 bytes, 8 per 128-byte row.)
  auto logits_mma = [&](uint64_t bdesc, int rows) {
    const uint32_t idesc = umma_idesc_bf16(kRows, rows);
    const uint64_t qd = umma_desc_sw128(smem_u32(Qs));
#pragma unroll
    for (int k = 0; k < D / 16; ++k)
      umma_bf16(tmem_base, qd + (uint64_t)((k / 4) * (kRows * 8) + (k % 4) * 2),
                bdesc + (uint64_t)((k / 4) * rows * 8 + (k % 4) * 2), idesc, k > 0);
  };
  // One warp: S = Q . Cp^T of a tile once its operands have landed.
  auto issue_s = [&](bool new_cp) {
    if (elect_one()) {
      bool ok = mbar_wait(bar_q, ph_q, abort_flag, p.status_word, DEV_TIMEOUT_ATTEND);
      if (new_cp) ok = mbar_wait(bar_cp, ph_cp, abort_flag, p.status_word, DEV_TIMEOUT_ATTEND) && ok;
      if (ok) {
        tc_fence_after();
        logits_mma(umma_desc_sw128(smem_u32(CA)), M);
      }
      umma_commit(bar_s);
    }
    __syncwarp();
    ph_q ^= 1;
    if (new_cp) ph_cp ^= 1;
  };
  auto issue_sc = [&](int rows) {                        // one warp: child logits
    if (elect_one()) {
      tc_fence_after();
      logits_mma(umma_desc_sw128(smem_u32(CC)), rows);
      umma_commit(bar_s);
    }
    __syncwarp();
  };
  // One warp: O (+)= weights (TMEM columns from w_col) . value rows
  auto issue_o = [&](const unsigned char* values, int rows, int w_col, bool accumulate, uint64_t* bar) {
    if (elect_one()) {
      tc_fence_after();
      const uint64_t vd = umma_desc_sw128_mn(smem_u32(values), (uint32_t)(rows * 128));
      const uint64_t ad = umma_desc_sw128(smem_u32(CA));
#pragma unroll
      for (int k = 0; k < CT / 16; ++k)
        if (16 * k < rows) {
          if constexpr (kTW)
            umma_bf16_ts(tmem_base + L::tO, tmem_base + w_col + 8 * k, vd + (uint64_t)(128 * k), idesc_o, accumulate || k > 0);
          else
            umma_bf16(tmem_base + L::tO, ad + (uint64_t)((k / 4) * (kRows * 8) + (k % 4) * 2), vd + (uint64_t)(128 * k),
                      idesc_o, accumulate || k > 0);
        }
      umma_commit(bar);
    }
    __syncwarp();
  };
  // Weights of 32 columns (col0 a multiple of 32) of this warp's rows -> A operand: pk[b][h] = block b, row h.
  const uint32_t a_row = smem_u32(CA) + (uint32_t)(r * 128 + ((lane & 7) << 4));
  auto put_weights = [&](int w_col, int col0, const uint32_t (&pk)[4][4]) {
    if constexpr (kTW) {
      const uint32_t v[2][8] = {{pk[0][0], pk[0][1], pk[1][0], pk[1][1], pk[2][0], pk[2][1], pk[3][0], pk[3][1]},
                                {pk[0][2], pk[0][3], pk[1][2], pk[1][3], pk[2][2], pk[2][3], pk[3][2], pk[3][3]}};
      tmem_st_weights(t_row + (uint32_t)(w_col + (col0 >> 1)), v);
    } else {
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int col = col0 + 8 * b;
        stmatrix4((a_row + (uint32_t)((col >> 6) * (kRows * 128))) ^ (uint32_t)(((col >> 3) & 7) << 4), pk[b][0], pk[b][1],
                  pk[b][2], pk[b][3]);
      }
    }
  };
  auto weights_done = [&]() {                            // before the barrier ahead of the MMA that reads them
    if constexpr (kTW) tmem_st_wait();
    cp_async_wait_all();
    fence_proxy_async();
    tc_fence_before();
  };
  // The values a fragment thread needs of rows g + 8 h, from the lane that stands for the row.
  auto to_frag = [&](float v, float (&out)[4]) {
#pragma unroll
    for (int h = 0; h < 4; ++h) out[h] = __shfl_sync(0xffffffffu, v, g + 8 * h);
  };

  if (warp == kVWarp) issue_s(true);
  bool first = true, new_bh = true;                      // new_bh: counts (and V) of another (b, h) than the tile before
  bool store_pending = false;                            // warp 0: a TMA store may still be reading the staging area
  for (int tile = tile0; tile < tile1; ++tile) {
    const int i0 = blk * kRows;
    const int rows_valid = min(kRows, p.Nq - i0);
    const bool has_next = tile + 1 < tile1;
    const int nbh = blk + 1 == p.nblk ? bh + 1 : bh, nblk_ = blk + 1 == p.nblk ? 0 : blk + 1;
    const bool next_new_bh = has_next && nbh != bh;
    const bool next_new_head = next_new_bh && p.H > 1;
    const bool next_new_cp = has_next && (!kTW || next_new_head || (L::kCodesInCA && PC > 0));
    // V of this tile: loaded behind the last use of the one before (below), except for the first tile.  Where its place is the
    // staging area: as soon as the store of the tile before has read that.  (Only ahead of the gather, where the other
    // plans wait for their stores, nothing covered the load: N65536 H16 d64 M64 P0 attend 81.7 -> 75.3 us.)
    if (!L::kStageInCC && warp == 0 && store_pending) {
      if (elect_one()) {
        tma_store_wait_read();
        issue_v(bh);
      }
      store_pending = false;
    }
    const bool new_v = STAYS || !L::kStageInCC || (new_bh | (wide != 0));   // (one load, waited for where it is used)

    if (new_bh) {
      // ---- Part 2 reads what the earlier kernels of this call wrote: status word, counts, value means.  (Loaded
      // with statements the compiler cannot move ahead of the dependency wait.)
      static_assert(2 * CT <= kThreads, "one count load per thread: M * C / 4 <= 2 CT vectors of four");
      if (first) pdl_wait();
      float n_reg = 0.f;
      float4 nc_reg = make_float4(0.f, 0.f, 0.f, 0.f);
      if (tid < M) n_reg = ld_after_wait(p.np_ + (size_t)bh * M + tid);
      if (PC > 0 && tid < ((M * C) >> 2))
        nc_reg = ld_after_wait(reinterpret_cast<const float4*>(p.nc + (size_t)bh * M * C) + tid);
      if (first && warp == 0 && elect_one()) {
        issue_v(bh);
        // a wait that expired in an earlier CTA or kernel of this call: do not start more work (a flagged index is
        // no reason to stop)
        const int32_t word = p.status_word != nullptr ? *reinterpret_cast<volatile int32_t*>(p.status_word) : 0;
        early_exit = word != 0 && word != DEV_BAD_INDEX;
        wide = p.status_word != nullptr ? *reinterpret_cast<volatile int32_t*>(p.status_word + kWideWord) : 0;
      }
      if (tid < CT) {
        cnt[parent_pos(tid)] = n_reg;
        bias[parent_pos(tid)] = n_reg > 0.f ? 0.f : -INFINITY;
      }
      // every child's key count: the gathers below pick theirs from shared memory instead of waiting for a
      // dependent global load once the selection is known (log2 0 = -inf: an empty child's weight is exactly 0)
      if (PC > 0 && tid < ((M * C) >> 2))
        reinterpret_cast<float4*>(ncs)[tid] = make_float4(log2f(nc_reg.x), log2f(nc_reg.y), log2f(nc_reg.z), log2f(nc_reg.w));
      __syncthreads();
      if (first && early_exit) {
        // let the MMA and the load already in flight finish, then leave cleanly
        mbar_wait(bar_s, 0, abort_flag, nullptr, 0);
        mbar_wait(bar_v, 0, abort_flag, nullptr, 0);
        tc_fence_before();
        __syncthreads();
        if (warp == 1) tmem_dealloc(tmem_base, L::tmem_cols);
        return;
      }
      first = false;
    }

    // ---- parents: this thread's logits (4 rows x QW / 8 column pairs) are read from TMEM once and stay in
    // registers through the exponentials, the importance sums and the conversion to bf16.  An empty parent's
    // -inf bias becomes a weight of exactly 0.
    mbar_wait(bar_s, ph_s, abort_flag, p.status_word, DEV_TIMEOUT_ATTEND);
    ph_s ^= 1;
    tc_fence_after();
    if (warp == 0 && PC == 0 && has_next && elect_one()) issue_q(nbh, nblk_);   // no child logits will read this Q tile
    if (warp == 0 && kTW && next_new_cp && !(L::kCodesInCA && PC > 0) && elect_one())
      issue_cp(nbh, kSubD);                              // the codebook of the head that follows
    f32x2 a[4][NB];                                      // [row h][block]
    float m_run[4];                                      // maximum of the rows, log2 units
#pragma unroll
    for (int h = 0; h < 4; ++h) m_run[h] = -INFINITY;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (32 * c < my_cols) {                            // warp-uniform
        uint32_t s[2][16];
        tmem_ld_frag<4>(t_s + 32 * c, s);
        f32x2 bi[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) bi[b] = *reinterpret_cast<const f32x2*>(bias + colbase + 32 * c + 8 * b + 2 * t4);
        tmem_ld_wait_frag<4>(s);
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            const f32x2 v = add2(pack2u(s[h >> 1][4 * b + 2 * (h & 1)], s[h >> 1][4 * b + 2 * (h & 1) + 1]), bi[b]);
            a[h][4 * c + b] = v;
            float lo, hi;
            unpack2(v, lo, hi);
            m_run[h] = max3(m_run[h], lo, hi);
          }
      } else {
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int h = 0; h < 4; ++h) a[h][4 * c + b] = 0;
      }
    }
#pragma unroll
    for (int h = 0; h < 4; ++h) m_run[h] = quad_max(m_run[h]) * sc;   // scale > 0: the maximum commutes with it
    if (NQ > 1) {
      xm[cq * kRows + q * 32 + g + 8 * t4] = pick4(m_run, t4);
      row_sync<NQ>(q);
      float m = xm[r];                                   // of row `lane`
#pragma unroll
      for (int u = 1; u < NQ; ++u) m = fmaxf(m, xm[u * kRows + r]);
      to_frag(m, m_run);
    }
    // m_run is finite: at least one parent holds a key.

    // ---- fp32 weights and the exact denominator.  This lane's columns are the codewords t, t + 4, ... of the slice
    // (kChain: of two warps' slices) in ascending order: one chain per row, the quad adds (0 + 1) + (2 + 3).
    float iz[4];                                         // 1 / z, 0 for rows past the end
    {
      float z[4] = {0.f, 0.f, 0.f, 0.f};
      const f32x2 sc2 = pack2(sc, sc);
      f32x2 nm[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) nm[h] = pack2(-m_run[h], -m_run[h]);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (32 * c < my_cols) {                          // 64 independent exponentials per step
          float2 n2[4];
#pragma unroll
          for (int b = 0; b < 4; ++b) n2[b] = *reinterpret_cast<const float2*>(cnt + colbase + 32 * c + 8 * b + 2 * t4);
#pragma unroll
          for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int h = 0; h < 4; ++h) {
              f32x2& x = a[h][4 * c + b];
              float lo, hi;
              unpack2(fma2(x, sc2, nm[h]), lo, hi);
              lo = ex2(lo);
              hi = ex2(hi);
              if constexpr (!L::kChain) z[h] = fmaf(hi, n2[b].y, fmaf(lo, n2[b].x, z[h]));
              x = pack2(lo, hi);
            }
        }
      }
      constexpr int NZ = L::kChain ? NQ / 2 : NQ;        // chains per row
      const int cz = L::kChain ? cq >> 1 : cq;
      if constexpr (L::kChain) {
        float4* part = reinterpret_cast<float4*>(zchain + cz * 4 * kRows) + q * 32 + lane;
        auto add = [&]() {
          if (my_cols > 0)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              const float2 n2 = *reinterpret_cast<const float2*>(cnt + colbase + 8 * b + 2 * t4);
#pragma unroll
              for (int h = 0; h < 4; ++h) {
                float lo, hi;
                unpack2(a[h][b], lo, hi);
                z[h] = fmaf(hi, n2.y, fmaf(lo, n2.x, z[h]));
              }
            }
        };
        if ((cq & 1) == 0) {                             // warp-uniform
          add();
          *part = make_float4(z[0], z[1], z[2], z[3]);
        }
        row_sync<NQ>(q);
        if (cq & 1) {
          const float4 first_half = *part;
          z[0] = first_half.x; z[1] = first_half.y; z[2] = first_half.z; z[3] = first_half.w;
          add();
        }
      }
#pragma unroll
      for (int h = 0; h < 4; ++h) z[h] = quad_sum(z[h]);
      float zr;                                          // of row `lane`
      if (NQ > 1) {
        if (!L::kChain || (cq & 1)) xz[cz * kRows + q * 32 + g + 8 * t4] = pick4(z, t4);
        row_sync<NQ>(q);
        zr = xz[r];
#pragma unroll
        for (int u = 1; u < NZ; ++u) zr += xz[u * kRows + r];
      } else {
        zr = __shfl_sync(0xffffffffu, pick4(z, t4), 4 * (lane & 7) + (lane >> 3));
      }
      to_frag(r < rows_valid ? 1.f / zr : 0.f, iz);
    }

    // The importances are needed only to choose which parents to refine: with P = 0 (nothing refined) or
    // P >= M (everything refined) the choice is fixed and the pass is skipped unless the caller wants them.
    const bool need_w = (P > 0 && P < M) || p.importance_out != nullptr;
    uint32_t key = 0;                                    // importance of parent `tid` (non-negative float bits)
    int nz = 0;                                          // parents with an importance above zero
    if (tid < CT) {                                      // nothing is refined yet
      if constexpr (STAYS) keep_f[tid] = 1.f;
      else keep_m[tid] = 0xFFFFu;
    }
    if (need_w) {
      // ---- importance: column sums of A_ij / z_i over the 128 rows (4 in registers, 8 lanes, 4 warps)
      f32x2 inv[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) inv[h] = pack2(iz[h], iz[h]);
      f32x2 v[NB];
#pragma unroll
      for (int b = 0; b < NB; ++b)
        v[b] = add2(add2(mul2(a[0][b], inv[0]), mul2(a[2][b], inv[2])), add2(mul2(a[1][b], inv[1]), mul2(a[3][b], inv[3])));
      const f32x2 colsum = reduce_rows<NB>(v, lane);
      const int b = NB == 8 ? g : g >> 1;
      if (NB == 8 || (g & 1) == 0) *reinterpret_cast<f32x2*>(wpart + q * CT + colbase + 8 * b + 2 * t4) = colsum;
      __syncthreads();
      float wj = 0.f;
      if (tid < M) {
        const int c = parent_pos(tid);
        wj = cnt[c] * ((wpart[c] + wpart[CT + c]) + (wpart[2 * CT + c] + wpart[3 * CT + c]));
        w[tid] = fabsf(wj);                              // (a NaN's sign would not order)
        const uint32_t m_ = __ballot_sync(0xffffffffu, wj > 0.f);   // M is a multiple of 32
        if (lane == 0) { nzmask[warp] = m_; selmask[warp] = 0u; }
        if (p.importance_out) p.importance_out[((size_t)bh * p.nblk + blk) * M + tid] = wj;
      }
      if (CT <= 64 && tid >= M && tid < CT) w[tid] = 0.f;
      if (tid == 0) *ncand_s = 0;
      key = __float_as_uint(wj);
      nz = __syncthreads_count(wj > 0.f);
    }

    // ---- top-P, ties to the lower index.  Non-negative floats order like their bit patterns, so the comparisons
    // run on integers.
    auto choose = [&](int j, int pos) {
      sel_list[pos] = j;
      if constexpr (STAYS) keep_f[parent_pos(j)] = __ldg(p.rho + (size_t)bh * M + j);   // the share of its keys that stays with it
      else keep_m[parent_pos(j)] = 0;
    };
    int32_t* topp_out = p.topp_out ? p.topp_out + ((size_t)bh * p.nblk + blk) * P : nullptr;
    if (P >= M) {
      if (!need_w) __syncthreads();                      // keep[] reset above by other threads
      if (tid < M) {
        choose(tid, tid);
        if (topp_out) topp_out[tid] = tid;
      }
    } else if (P > 0) {
      const int K = M >> 5;                              // keys per lane (32 k + lane), <= 8
      const uint32_t below = (1u << lane) - 1u;
      if (nz <= P) {
        // Peaked attention leaves most importances at exactly zero: all others are refined, and as many of the
        // zeros as are missing, lowest index first.  No ranking.
        if (warp < K) {
          int nz_before = 0;
          for (int k = 0; k < warp; ++k) nz_before += __popc(nzmask[k]);
          const uint32_t mk = nzmask[warp];
          const int zr = 32 * warp - nz_before + __popc(~mk & below);   // zeros before this parent
          if (((mk >> lane) & 1u) || zr < P - nz) {
            const int pos = nz_before + __popc(mk & below) + min(zr, P - nz);
            choose(warp * 32 + lane, pos);
            if (topp_out) topp_out[pos] = warp * 32 + lane;
          }
        }
      } else {
        int rank = P, j = 0;                             // parent j of this thread, if it is to be listed
        if constexpr (CT <= 64) {
          // Few parents: 2^kLt threads rank each of them against a share of the others, with no barrier in between.
          // (Candidates as below and all parents so, us per call: H16 N20000 d64 M32 C8 85.2 and 82.6, N65536 M64 259.8 and
          // 256.4, B1 H12 N785 M64 19.0 and 18.6; but N20000 M128 137.2 and 140.7, N9000 M96 71.1 and 73.3.)
          constexpr int kLt = kThreads / CT == 2 ? 1 : 2, kShare = CT >> kLt;
          static_assert((CT << kLt) == kThreads, "every thread has a parent and a share");
          const int part = tid & ((1 << kLt) - 1);
          j = tid >> kLt;
          const uint32_t mine = reinterpret_cast<const uint32_t*>(w)[j];   // (zero from M on: above no other)
          int above = 0;
#pragma unroll
          for (int v = 0; v < kShare / 4; ++v) {
            const uint4 x = reinterpret_cast<const uint4*>(w)[part * (kShare / 4) + v];
            const int k = part * kShare + 4 * v;
            above += (x.x + (k < j) > mine) + (x.y + (k + 1 < j) > mine) + (x.z + (k + 2 < j) > mine) + (x.w + (k + 3 < j) > mine);
          }
#pragma unroll
          for (int o = 1; o < (1 << kLt); o <<= 1) above += __shfl_xor_sync(0xffffffffu, above, o);
          if (part == 0) rank = above;
        } else {
          // Only candidates are ranked, those at or above a bound that at least P keys reach.  The bound is the
          // largest of 32 sample keys (the first 32 parents') that has at least P keys at or above it, else the
          // smallest key above zero; each warp counts for its share of the samples.
          constexpr int kPer = 32 / (kThreads / 32);       // samples per warp
          uint32_t kk[CT / 32];
#pragma unroll
          for (int k = 0; k < CT / 32; ++k) kk[k] = k < K ? reinterpret_cast<const uint32_t*>(w)[32 * k + lane] : 0u;
#pragma unroll
          for (int e = 0; e < kPer; ++e) {
            const uint32_t smp = __shfl_sync(0xffffffffu, kk[0], warp * kPer + e);
            int c = 0;
#pragma unroll
            for (int k = 0; k < CT / 32; ++k) c += kk[k] >= smp;
            c = __reduce_add_sync(0xffffffffu, c);
            if (lane == 0) wcount[warp * kPer + e] = smp > 0u ? c : 0;
          }
          __syncthreads();
          const uint32_t bound = max(__reduce_max_sync(0xffffffffu, wcount[lane] >= P ? kk[0] : 0u), 1u);
          if (warp < K) {                                  // candidates of this warp's 32 parents -> list, in any order
            const uint32_t mk = __ballot_sync(0xffffffffu, key >= bound);
            int base = 0;
            if (lane == 0) base = atomicAdd(ncand_s, __popc(mk));
            base = __shfl_sync(0xffffffffu, base, 0);
            // importance above, complement of the index below: larger means refined earlier, no two are equal
            if ((mk >> lane) & 1u) cand[base + __popc(mk & below)] = ((uint64_t)key << 32) | (uint32_t)(0xFFFF - tid);
          }
          __syncthreads();
          // rank of every candidate among them; 2^lt threads share a candidate.  The list of refined parents is
          // ordered by rank.
          const int ncand = *ncand_s;
          constexpr int kLogT = NQ == 4 ? 9 : (NQ == 2 ? 8 : 7);
          const int lt = max(0, min(4, kLogT - (32 - __clz(ncand - 1))));
          const int i = tid >> lt, part = tid & ((1 << lt) - 1);
          const uint64_t mine = i < ncand ? cand[i] : 0;
          int above = 0;
          for (int k = part; k < ncand; k += 4 << lt) {    // four in flight; past the end only the comparison is masked
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int ku = k + (u << lt);
              above += (cand[min(ku, CT - 1)] > mine) & (ku < ncand);
            }
          }
#pragma unroll
          for (int o = 1; o <= 8; o <<= 1) {
            const int other = __shfl_xor_sync(0xffffffffu, above, o);
            if (o < (1 << lt)) above += other;
          }
          if (i < ncand && part == 0) {
            rank = above;
            j = 0xFFFF - (int)((uint32_t)mine & 0xFFFFu);
          }
        }
        if (rank < P) {
          choose(j, rank);
          if (topp_out) atomicOr(&selmask[j >> 5], 1u << (j & 31));
        }
        if (topp_out) {                                  // the caller's list is ascending
          __syncthreads();
          if (warp < K) {
            const uint32_t mk = selmask[warp];
            int pos = __popc(mk & below);
            for (int k = 0; k < warp; ++k) pos += __popc(selmask[k]);
            if ((mk >> lane) & 1u) topp_out[pos] = tid;
          }
        }
      }
    }
    // the output tile of the tile before must have left its staging area before that is refilled (its store was
    // issued a whole parent pass ago, so this does not wait in practice)
    if (warp == 0 && store_pending) {
      if (elect_one()) tma_store_wait_read();
      store_pending = false;
    }
    __syncthreads();

    // ---- first child chunk: start the asynchronous gather of its codeword rows now; it lands while the
    // weight conversion below runs
    const __nv_bfloat16* Cch = p.Cc + (size_t)(bh % p.H) * M * C * D;
    const __nv_bfloat16* Vch = p.Vcb + (size_t)bh * M * C * D;
    int ncols = min(PC, CHW);
    int np16 = (ncols + 15) & ~15;
    // Rows of a chunk, gathered into a row-per-codeword tile of np16 rows (kSubD sub-tiles of 64 columns): local
    // row e = src[sel_list[(e_first+e)/C] * C + (e_first+e)%C, :]; padding rows are zero.  A thread keeps its
    // 16-byte chunk column and walks down the rows (kThreads is a multiple of the chunks per row).
    auto gather_rows = [&](unsigned char* dst_tile, const __nv_bfloat16* src, int e_first) {
      constexpr int kRowsPerPass = kThreads >> kLogChunks;   // a multiple of 8: a thread's swizzle phase is fixed
      constexpr int kPasses = (CHW + kRowsPerPass - 1) / kRowsPerPass;
      const int ch = tid & ((1 << kLogChunks) - 1), row0 = tid >> kLogChunks;
      const uint32_t dst0 = smem_u32(dst_tile) + (uint32_t)((ch >> 3) * (np16 * 128)) + sw128_offset(row0, (ch & 7) * 8);
      const __nv_bfloat16* src_col = src + ch * 8;
      int sel[kPasses];
#pragma unroll
      for (int it = 0; it < kPasses; ++it) {                 // the list look-ups first, all in flight together
        const int e = e_first + row0 + it * kRowsPerPass;
        sel[it] = (row0 + it * kRowsPerPass < ncols) ? sel_list[e >> logC] : 0;
      }
#pragma unroll
      for (int it = 0; it < kPasses; ++it) {
        const int row = row0 + it * kRowsPerPass;
        const uint32_t dst = dst0 + (uint32_t)(it * kRowsPerPass * 128);
        if (row < ncols) {
          const int e = e_first + row;
          const uint32_t off = (uint32_t)(((sel[it] << logC) + (e & (C - 1))) << kLogD);   // elements: < 2^31
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src_col + off) : "memory");
        } else if (row < np16) {
          asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(dst), "r"(0) : "memory");
        }
      }
    };
    auto gather_codes = [&](int e_first) {
      float l2 = -INFINITY;
      if (tid < ncols) {                                   // CHW <= 128 <= kThreads
        const int e = e_first + tid;
        l2 = ncs[(sel_list[e >> logC] << logC) + (e & (C - 1))];
      }
      gather_rows(CC, Cch, e_first);
      if (tid < CHW) l2n[tid] = l2;
    };
    if (PC > 0) gather_codes(0);

    // ---- bf16 weights -> A operand, and their denominator (this thread's share of its rows; put together at the
    // end of the tile).  Default rule: a refined parent's weight is masked to zero.
    if (new_v) {                                           // parent values have landed (needed by the MMA and the stay rows)
      mbar_wait(bar_v, ph_v, abort_flag, p.status_word, DEV_TIMEOUT_ATTEND);
      ph_v ^= 1;
    }
    if constexpr (STAYS) {
      // a refined parent keeps only the keys that stayed with it (Algorithm 1's masked scatter): its value row
      // becomes the stay residual, Vbar_stay = Vbar_p - sum_c Vbar_c, in the same per-n_p units
      for (int u = tid; u < (min(P, M) << kLogChunks); u += kThreads) {
        const int row = sel_list[u >> kLogChunks], ch = u & ((1 << kLogChunks) - 1);
        *reinterpret_cast<uint4*>(Vs + (ch >> 3) * (M * 128) + sw128_offset(parent_pos(row), (ch & 7) * 8)) =
            __ldg(reinterpret_cast<const uint4*>(p.Vsb + ((size_t)bh * M + row) * D) + ch);
      }
    } else if (wide) {
      // a refined parent's weight of zero does not take an infinite value row out of the product: clear the row
#pragma unroll 1
      for (int u = tid; u < (min(P, M) << kLogChunks); u += kThreads) {
        const int row = sel_list[u >> kLogChunks], ch = u & ((1 << kLogChunks) - 1);
        *reinterpret_cast<uint4*>(Vs + (ch >> 3) * (M * 128) + sw128_offset(parent_pos(row), (ch & 7) * 8)) = make_uint4(0u, 0u, 0u, 0u);
      }
    }
    float z_run[4] = {0.f, 0.f, 0.f, 0.f};
    {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (32 * c < my_cols) {
          uint32_t pk[4][4];
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const f32x2 n2 = *reinterpret_cast<const f32x2*>(cnt + colbase + 32 * c + 8 * b + 2 * t4);
            uint32_t km = 0;
            float2 kf = make_float2(0.f, 0.f);
            if constexpr (STAYS) kf = *reinterpret_cast<const float2*>(keep_f + colbase + 32 * c + 8 * b + 2 * t4);
            else km = *reinterpret_cast<const uint32_t*>(keep_m + colbase + 32 * c + 8 * b + 2 * t4);
#pragma unroll
            for (int h = 0; h < 4; ++h) {
              float lo, hi;
              unpack2(mul2(a[h][4 * c + b], n2), lo, hi);
              pk[b][h] = pack_bf16(lo, hi);
              if constexpr (STAYS) {
                z_run[h] = fmaf(__uint_as_float(pk[b][h] << 16), kf.x, z_run[h]);
                z_run[h] = fmaf(__uint_as_float(pk[b][h] & 0xFFFF0000u), kf.y, z_run[h]);
              } else {
                pk[b][h] &= km;
                add_bf16x2(z_run[h], pk[b][h]);
              }
            }
          }
          put_weights(L::tW, colbase + 32 * c, pk);
        }
      }
    }
    weights_done();
    __syncthreads();

    // ---- the first child chunk's logits, and behind them O = A . Vbar_p: the tensor pipe works in order, the
    // children's logits are waited for, O is not.  An issuing lane is held up at the tensor pipe's pace, so O has
    // another warp, which does its share of the gather first.
    auto pair_barrier = [&](bool wait) {                   // warp 0 arrives, kVWarp waits
      if (wait) asm volatile("bar.sync 5, 64;" ::: "memory");
      else asm volatile("bar.arrive 5, 64;" ::: "memory");
    };
    if (warp == 0 && PC > 0) {
      issue_sc(np16);
      pair_barrier(false);
    }
    if (kSepCV && PC > 0) gather_rows(CV, Vch, 0);         // while the logits are computed
    if (warp == kVWarp) {
      if (PC > 0) pair_barrier(true);
      issue_o(Vs, M, L::tW, false, bar_o);
    }

    // ---- child chunks
    for (int e0 = 0; e0 < PC; e0 += CHW) {
      mbar_wait(bar_s, ph_s, abort_flag, p.status_word, DEV_TIMEOUT_ATTEND);
      ph_s ^= 1;
      tc_fence_after();
      const bool last = e0 + CHW >= PC;
      if (warp == 0 && last && has_next && elect_one()) {  // the last logits are done: Q is dead, and so are the codes
        issue_q(nbh, nblk_);
        if (L::kCodesInCA) issue_cp(nbh, (next_new_head || M < CT) ? kSubD : 1);
      }
      if (e0 > 0) {                                        // the chunk before has left the weights and the value rows
        mbar_wait(bar_pv, ph_pv, abort_flag, p.status_word, DEV_TIMEOUT_ATTEND);
        ph_pv ^= 1;
      }
      if constexpr (!kSepCV) gather_rows(CC, Vch, e0);     // the codes are dead: the values take their place
      else if (e0 > 0) gather_rows(CV, Vch, e0);
      tc_fence_after();
      bool o_done = L::kSepW || e0 > 0;                    // the weights' columns are free
      const int my_c = min(max(np16 - cq * QWC, 0), QWC);  // multiple of 16
      float zc[4];
      // Largest partial sum of the children's weights before the reference moves: 2^64 while no mean exceeds 2^40 (the sums
      // stay below 2^115 then), 2^8 with values beyond that.
      const float largest = wide ? 256.f : 1.8446744e19f;
      for (;;) {
        // bf16 weights exp2(s - m + log2 n) of the children, their sum
        const f32x2 sc2 = pack2(sc, sc);
        f32x2 nm[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) { nm[h] = pack2(-m_run[h], -m_run[h]); zc[h] = 0.f; }
#pragma unroll
        for (int c = 0; c < NCC; ++c)
          if (32 * c < my_c) {                             // warp-uniform
            uint32_t s[2][16];
            tmem_ld_frag<4>(t_sc + 32 * c, s);
            f32x2 ln[4];
#pragma unroll
            for (int b = 0; b < 4; ++b) ln[b] = *reinterpret_cast<const f32x2*>(l2n + cq * QWC + 32 * c + 8 * b + 2 * t4);
            tmem_ld_wait_frag<4>(s);
            uint32_t pk[4][4];
            const bool whole = 32 * c + 16 < my_c;         // else the last 16 columns are not there (no logits, weight zero)
#pragma unroll
            for (int b = 0; b < 4; ++b)
#pragma unroll
              for (int h = 0; h < 4; ++h) {
                if (b >= 2 && !whole) {
                  pk[b][h] = 0u;
                  continue;
                }
                const f32x2 x = pack2u(s[h >> 1][4 * b + 2 * (h & 1)], s[h >> 1][4 * b + 2 * (h & 1) + 1]);
                float lo, hi;
                unpack2(add2(fma2(x, sc2, nm[h]), ln[b]), lo, hi);
                pk[b][h] = pack_bf16(ex2(lo), ex2(hi));
                add_bf16x2(zc[h], pk[b][h]);
              }
            if (!o_done) {
              mbar_wait(bar_o, ph_o, abort_flag, p.status_word, DEV_TIMEOUT_ATTEND);
              tc_fence_after();
              o_done = true;
            }
            put_weights(L::tWc, cq * QWC + 32 * c, pk);
          }
        // Any reference value works as long as numerator and denominator share it: the parents' maximum is kept
        // unless the children's weights grow so large against it that fp32 sums could overflow.  That is found out
        // at the barrier that publishes the weights; the rare case goes round the loop once more.
        weights_done();
        if (!__syncthreads_or(fmaxf(fmaxf(zc[0], zc[1]), fmaxf(zc[2], zc[3])) > largest)) break;
        // ---- row maxima of the chunk (non-empty children); where they exceed the reference it moves up and O and z
        // are rescaled
        float m_c[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int c = 0; c < NCC; ++c)
          if (32 * c < my_c) {
            uint32_t s[2][16];
            tmem_ld_frag<4>(t_sc + 32 * c, s);
            tmem_ld_wait_frag<4>(s);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              const float2 ln = *reinterpret_cast<const float2*>(l2n + cq * QWC + 32 * c + 8 * b + 2 * t4);
#pragma unroll
              for (int h = 0; h < 4; ++h)
                m_c[h] = max3(m_c[h], ln.x + sc * __uint_as_float(s[h >> 1][4 * b + 2 * (h & 1)]),
                              ln.y + sc * __uint_as_float(s[h >> 1][4 * b + 2 * (h & 1) + 1]));
            }
          }
#pragma unroll
        for (int h = 0; h < 4; ++h) m_c[h] = quad_max(m_c[h]);
        if (NQ > 1) {
          xm[cq * kRows + q * 32 + g + 8 * t4] = pick4(m_c, t4);
          row_sync<NQ>(q);
          float m = xm[r];
#pragma unroll
          for (int u = 1; u < NQ; ++u) m = fmaxf(m, xm[u * kRows + r]);
          to_frag(m, m_c);
        }
        float alpha[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          alpha[h] = 1.f;
          if (m_c[h] > m_run[h]) {
            alpha[h] = ex2(m_run[h] - m_c[h]);
            m_run[h] = m_c[h];
          }
          z_run[h] *= alpha[h];
        }
        if (e0 == 0) mbar_wait(bar_o, ph_o, abort_flag, p.status_word, DEV_TIMEOUT_ATTEND);
        tc_fence_after();
        for (int c0 = 0; c0 < D / NQ; c0 += 16) {
          uint32_t o[2][8];
          tmem_ld_frag<2>(t_o + c0, o);
          tmem_ld_wait_frag<2>(o);
#pragma unroll
          for (int h = 0; h < 4; ++h)
#pragma unroll
            for (int e = 0; e < 4; ++e) {                  // blocks 0, 1 x columns 0, 1
              uint32_t& x = o[h >> 1][4 * (e >> 1) + 2 * (h & 1) + (e & 1)];
              x = __float_as_uint(__uint_as_float(x) * alpha[h]);
            }
          tmem_st_frag<2>(t_o + c0, o);
        }
        tmem_st_wait();
        // a second turn sees weights of at most about the chunk's width and ends
      }
#pragma unroll
      for (int h = 0; h < 4; ++h) z_run[h] += zc[h];

      // ---- O += A_c . Vbar_c
      if (warp == kVWarp) issue_o(kSepCV ? CV : CC, np16, L::tWc, true, bar_pv);
      if (!last) {
        ncols = min(PC - e0 - CHW, CHW);
        np16 = (ncols + 15) & ~15;
        if constexpr (!kSepCV) mbar_wait(bar_pv, ph_pv, abort_flag, p.status_word, DEV_TIMEOUT_ATTEND);   // values have left CC
        gather_codes(e0 + CHW);
        cp_async_wait_all();
        fence_proxy_async();
        tc_fence_before();
        __syncthreads();
        if (warp == 0) issue_sc(np16);
      }
    }

    // ---- epilogue: Y = O / z.  The rows' denominators are put together while the last MMA runs.
    float inv[4];
    {
      float zt[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) zt[h] = quad_sum(z_run[h]);
      float z;                                             // of row `lane`
      if (NQ > 1) {
        xz[cq * kRows + q * 32 + g + 8 * t4] = pick4(zt, t4);
        row_sync<NQ>(q);
        z = xz[r];
#pragma unroll
        for (int u = 1; u < NQ; ++u) z += xz[u * kRows + r];
      } else {
        z = __shfl_sync(0xffffffffu, pick4(zt, t4), 4 * (lane & 7) + (lane >> 3));
      }
      to_frag(1.f / z, inv);
    }
    const bool o_ok = mbar_wait(PC > 0 ? bar_pv : bar_o, PC > 0 ? ph_pv : ph_o, abort_flag, p.status_word, DEV_TIMEOUT_ATTEND);
    if (PC > 0) ph_pv ^= 1;
    ph_o ^= 1;                                             // (the children's MMA is behind the parents')
    tc_fence_after();
    // the next tile's logits: every thread has read this tile's, and the last value MMA its weights
    if (kTW && has_next && warp == kVWarp) issue_s(next_new_cp);
    if (warp == 0 && has_next && elect_one()) {
      // the last value MMA has released the weights (here: the codebook's place) and the parent values
      if (!kTW) issue_cp(nbh, kSubD);
      if (L::kStageInCC && (STAYS || next_new_bh || wide)) issue_v(nbh);
    }
    // The output tile is staged in shared memory in the layout of the Q load and written with TMA tile
    // stores; rows past Nq are clipped by the tensor map.
    if (o_ok) {
      constexpr int OW = D / NQ, ONB = OW >= 32 ? 4 : 2;   // output columns of this warp, blocks per step
      const uint32_t st_row = smem_u32(stage) + (uint32_t)(r * 128 + ((lane & 7) << 4));
#pragma unroll
      for (int c = 0; c < OW / (8 * ONB); ++c) {
        uint32_t o[2][4 * ONB];
        tmem_ld_frag<ONB>(t_o + 8 * ONB * c, o);
        tmem_ld_wait_frag<ONB>(o);
#pragma unroll
        for (int b = 0; b < ONB; ++b) {
          uint32_t pk[4];
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            const uint32_t* x = &o[h >> 1][4 * b + 2 * (h & 1)];
            pk[h] = pack_bf16(__uint_as_float(x[0]) * inv[h], __uint_as_float(x[1]) * inv[h]);
          }
          const int col = cq * OW + 8 * ONB * c + 8 * b;
          stmatrix4((st_row + (uint32_t)((col >> 6) * (kRows * 128))) ^ (uint32_t)(((col >> 3) & 7) << 4), pk[0], pk[1], pk[2],
                    pk[3]);
        }
      }
      fence_proxy_async();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0 && o_ok) {
      if (!PERM && elect_one()) {
#pragma unroll
        for (int s2 = 0; s2 < kSubD; ++s2) tma_store_3d(&tmY, stage + s2 * kRows * 128, s2 * 64, i0, bh);
        tma_store_commit();
        if (!has_next) tma_store_wait_read();              // before the CTA may leave
      }
      store_pending = !PERM && has_next;                   // waited for before the staging area is refilled
    }
    if constexpr (PERM) {                                  // every row to its place: d / 8 lanes per row, 16 bytes each
      if (o_ok) {
        for (int u = tid; u < (rows_valid << kLogChunks); u += kThreads) {
          const int row = u >> kLogChunks, ch = u & ((1 << kLogChunks) - 1);
          const int j = __ldg(p.perm + i0 + row);
          const uint4 v = *reinterpret_cast<const uint4*>(stage + (ch >> 3) * (kRows * 128) + sw128_offset(row, (ch & 7) * 8));
          if (j >= 0 && j < p.Nq) reinterpret_cast<uint4*>(p.Y + ((size_t)bh * p.Nq + j) * D)[ch] = v;
          else if (ch == 0 && p.status_word) atomicCAS(p.status_word, 0, DEV_BAD_INDEX);
        }
      }
      fence_proxy_async();
      __syncthreads();                                     // read before the staging area is refilled
      if (!L::kStageInCC && has_next && warp == 0 && elect_one()) issue_v(nbh);
    }
    if (!kTW && has_next && warp == kVWarp) issue_s(true);
    new_bh = next_new_bh;
    bh = nbh;
    blk = nblk_;
  }   // tiles
  if (warp == 1) tmem_dealloc(tmem_base, L::tmem_cols);
}

template <int D, int NQ, int CT, bool STAYS, bool PERM>
avq_status launch_plan(const CUtensorMap& tmQ, const CUtensorMap& tmCp, const CUtensorMap& tmVpb,
                       const CUtensorMap& tmY, const AttendParams& a, bool chained, cudaStream_t st) {
  auto kern = tc_attend_kernel<D, NQ, CT, STAYS, PERM>;
  const size_t smem = attend_smem<D, NQ, CT>(a.M * a.C);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return AVQ_ERR_CUDA;
  const avq_status s = open_shared_memory<tc_attend_kernel<D, NQ, CT, STAYS, PERM>>(dev);
  if (s != AVQ_OK) return s;
  // Grid: one wave of CTAs (4 / NQ per SM), each taking an equal run of tiles.
  static int sm_count[64] = {};
  int sms = (dev >= 0 && dev < 64) ? sm_count[dev] : 0;
  if (sms <= 0) {
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return AVQ_ERR_CUDA;
    if (dev >= 0 && dev < 64) sm_count[dev] = sms;
  }
  int ctas = a.total_tiles;
  if (ctas > (4 / NQ) * sms) ctas = (4 / NQ) * sms;
  // Inside avq_forward (`chained`) the kernel before it in the stream is the aggregate's finalize kernel
  // and Q was complete before the call, so the attention kernel may start as its programmatic dependent.
  // A stand-alone avq_attend is launched plainly: the work before it in the stream may be producing Q.
  return cuda_ok(launch_pdl(kern, dim3((unsigned)ctas), dim3(128 * NQ), smem, st, chained, tmQ, tmCp, tmVpb, tmY, a));
}

template <int D, int NQ, int CT>
avq_status launch_nq(const CUtensorMap& tmQ, const CUtensorMap& tmCp, const CUtensorMap& tmVpb,
                     const CUtensorMap& tmY, const AttendParams& a, bool chained, cudaStream_t st) {
  if (a.perm)
    return a.rho ? launch_plan<D, NQ, CT, true, true>(tmQ, tmCp, tmVpb, tmY, a, chained, st)
                 : launch_plan<D, NQ, CT, false, true>(tmQ, tmCp, tmVpb, tmY, a, chained, st);
  return a.rho ? launch_plan<D, NQ, CT, true, false>(tmQ, tmCp, tmVpb, tmY, a, chained, st)
               : launch_plan<D, NQ, CT, false, false>(tmQ, tmCp, tmVpb, tmY, a, chained, st);
}

template <int D>
avq_status launch(const avq_problem& p, const void* Q, const void* Cp, const void* Cc, const float* np_,
                  const float* nc, const void* Vpb, const void* Vcb, const void* Vsb, const float* rho, int32_t P, void* Y, int32_t* topp_out,
                  float* importance_out, int32_t* status_word, bool chained, const int32_t* perm, cudaStream_t st) {
  const uint64_t BH = (uint64_t)p.B * p.H;
  CUtensorMap tmQ, tmCp, tmVpb, tmY;
  {
    const uint64_t dims[3] = {(uint64_t)D, (uint64_t)p.Nq, BH};
    const uint32_t box[3] = {64, (uint32_t)kRows, 1};
    avq_status s = make_tmap_bf16(&tmQ, Q, 3, dims, box);
    if (s != AVQ_OK) return s;
    s = make_tmap_bf16(&tmY, Y, 3, dims, box);
    if (s != AVQ_OK) return s;
  }
  {
    avq_status s = make_tmap_codes(&tmCp, Cp, D, (uint64_t)p.H * p.M, (uint32_t)p.M);
    if (s != AVQ_OK) return s;
    s = make_tmap_codes(&tmVpb, Vpb, D, BH * p.M, (uint32_t)p.M);
    if (s != AVQ_OK) return s;
  }
  AttendParams a;
  a.Cc = static_cast<const __nv_bfloat16*>(Cc);
  a.Vcb = static_cast<const __nv_bfloat16*>(Vcb);
  a.Vsb = static_cast<const __nv_bfloat16*>(Vsb);
  a.rho = rho;
  a.np_ = np_;
  a.nc = nc;
  a.Y = static_cast<__nv_bfloat16*>(Y);
  a.topp_out = topp_out;
  a.importance_out = importance_out;
  a.status_word = status_word;
  a.perm = perm;
  a.H = p.H; a.Nq = p.Nq; a.M = p.M; a.C = p.C; a.P = P;
  a.nblk = (p.Nq + kRows - 1) / kRows;
  if ((uint64_t)a.nblk * BH > 0x7fffffffull) return AVQ_ERR_UNSUPPORTED;
  a.total_tiles = (int)(a.nblk * BH);
  const int CT = p.M <= 64 ? 64 : (p.M <= 128 ? 128 : 256);
  a.logC = p.C == 8 ? 3 : 2;
  a.scale_log2e = p.scale * 1.4426950408889634f;
  // Warps per query row follow from how many CTAs can share an SM (TMEM columns, shared memory):
  // four small CTAs of 128 threads, two of 256, or one of 512.  A grid too small for that takes twice the warps per
  // tile (attend, B1 H12 d64 M64: N785 10.3 -> 8.7 us, N2000 12.3 -> 10.3).
  int sms = 0, dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return AVQ_ERR_CUDA;
  if constexpr (D == 64) {
    if (CT == 64 && a.total_tiles <= 2 * sms) return launch_nq<D, 2, 64>(tmQ, tmCp, tmVpb, tmY, a, chained, st);
    // (in the 64-parent plan such calls load the codebook again for every tile and wait for their children's values: H16 C4
    // N65536 attend P0 77.4 -> 53.1 us, P4 115 -> 88; N16384 P4 34.0 -> 27.9)
    if (p.M == 32) return launch_nq<D, 1, 32>(tmQ, tmCp, tmVpb, tmY, a, chained, st);
    if (CT == 128 && a.total_tiles <= sms) return launch_nq<D, 4, 128>(tmQ, tmCp, tmVpb, tmY, a, chained, st);
    if (CT == 64) return launch_nq<D, 1, 64>(tmQ, tmCp, tmVpb, tmY, a, chained, st);
    if (CT == 128) return launch_nq<D, 2, 128>(tmQ, tmCp, tmVpb, tmY, a, chained, st);
  } else {
    if (CT == 64) return launch_nq<D, 2, 64>(tmQ, tmCp, tmVpb, tmY, a, chained, st);
    if (CT == 128) return launch_nq<D, 4, 128>(tmQ, tmCp, tmVpb, tmY, a, chained, st);
  }
  return launch_nq<D, 4, 256>(tmQ, tmCp, tmVpb, tmY, a, chained, st);
}

}  // namespace

avq_status tc_attend(const avq_problem& p, const void* Q, const void* Cp, const void* Cc, const float* np_,
                     const float* nc, const void* Vpb, const void* Vcb, const void* Vsb, const float* rho, int32_t P, void* Y, int32_t* topp_out,
                     float* importance_out, int32_t* status_word, bool chained, const int32_t* perm, cudaStream_t st) {
  return p.d == 64 ? launch<64>(p, Q, Cp, Cc, np_, nc, Vpb, Vcb, Vsb, rho, P, Y, topp_out, importance_out, status_word, chained, perm, st)
                   : launch<128>(p, Q, Cp, Cc, np_, nc, Vpb, Vcb, Vsb, rho, P, Y, topp_out, importance_out, status_word, chained, perm, st);
}

}  // namespace avq
