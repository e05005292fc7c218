// Attention pass of avq_forward_tiled on the tensor cores: bfloat16, d = 64, blocks of at most 128 queries, importance tiles of at
// most 256 parents, up to 1024 parents.  The same computation as attend_simt_kernel (tiled importance, selection, merged
// softmax over unrefined parents, stay residuals and children of refined parents) with its precision: weights, value sums and
// their sum stay float32.
//
// One CTA = one query block.  16 warps compute, warp w on rows 32 (w % 4) .. +31 and columns 32 (w / 4) .. +31 of a tile of 128
// codewords, in the fragment layout of the accumulator (lane 4 g + t: rows g + 8 h, column pairs 8 b + 2 t); a 17th warp
// issues the TMA loads and every tcgen05.mma, so that none of the others waits for the tensor pipe.
//   logits   S = Q . C^T, one tcgen05.mma chain per tile; parents' codes by TMA, children's by cp.async gathers, two buffers
//   pass A   per importance tile: maximum, denominator, float64 column sums (importance)
//   pass C   weights and value sums enter the value product as three bfloat16 parts each, rounded to nearest, which hold a
//            float32 exactly (below 2^-110, to 2^-134).  Second and third part are at most 2^-8 and 2^-17 of it.  Of the nine products
//            six are added, the smallest first; the others are at most 2^-24 of the term together, what a float32 multiply-add
//            rounds off.  A tile's product starts from zero and is added to float32 registers while the next tile's weights
//            are computed.
//            Relative error of the float32 output (before its rounding to bfloat16) against 64 bits, CUDA-core kernel and here: M512
//            to M1024 P32 to P64, queries N(0, 1) 4.2e-7 to 4.8e-7 and 3.7e-7 to 4.0e-7, around a few parents 4.2e-7 to 6.7e-7
//            for both; P0 and peaked weights, sums of one or two terms, 1.6e-7 and 1.7e-7.  (Parts cut off instead of
//            rounded left out up to 2^-21 of a term.  Adding the two products of 2^-25 too changed nothing and took 1 us.)
// Bound by the phases of a tile one after the other (exponentials 2000 to 3300 cycles per code tile, splits 1300, column sums
// 2100), with 128 blocks on as many SMs: issue slots 47 % used, tensor pipe 10 %, L1 and shared memory 20 %, L2 6 %.  (96 registers
// with 544 threads: 140 bytes spilled.)  B1 H4 N4096 M512 C4 P64, importance tiles of 128, both cold: 167 us in the CUDA-core
// kernel (whose value product alone takes 55 at the float32 rate), 67 here.  A dedicated issuing warp: the 48 instructions
// of a tile's value product hold their issuer up for 2000 to 3000 cycles.
// A tile with a value sum that is infinite, NaN or beyond bfloat16's largest takes its product on the CUDA cores (an infinity
// times a part that happens to be zero would be NaN).
#include <math.h>

#include "avq_internal.h"
#include "avq_select.cuh"
#include "avq_tc_common.cuh"

namespace avq {
namespace {

using namespace tc;

constexpr int kD = 64;
constexpr int kRows = 128;
constexpr int kTile = 128;                     // codewords per tile
constexpr int kCompute = kSelThreads;          // 16 warps
constexpr int kIssuer = kCompute / 32;         // the warp that issues loads and products
constexpr int kThreadsT = kCompute + 32;
constexpr int kTileBytes = kTile * kD * 2;     // rows of 128 bytes
constexpr int kMaxTiles = 80;                  // M + P C <= 8192
constexpr int kSlots = 8;                      // tiles described at a time (the reason: at describe() below)
constexpr int kStayRow = 1 << 28, kChildRow = 1 << 29;
// TMEM columns: two logit tiles, three weight parts, the value product
constexpr int kColW = 256, kColO = 448;
constexpr float kLargestBf16 = 3.38953139e38f; // 0x7F7F0000
constexpr float kLowest = -3.402823466e38f;    // a running maximum starts at the lowest finite value (weights of -inf logits are then 0)

struct TiledArgs {
  const __nv_bfloat16* Cc;                     // [H, M, C, 64]
  const float *Vp, *np_, *Vc, *nc;
  __nv_bfloat16* Y;
  int32_t* topp_out;
  float* importance_out;
  int32_t* status_word;
  int H, Nq, M, C, P, block_q, nblk, stays, tile_m, Nk;
  uint32_t inv_C;                              // 2^18 / C rounded up
  float scale;
};

struct TiledSmem {
  size_t q, c, v, raw, w, wpart, tcnt, trow, np, nstay, xm, xz, nseen, sel, list, count, bad, bars, total;   // byte offsets
};
__host__ __device__ inline TiledSmem tiled_smem_layout(int M, int P, int tile_m) {
  TiledSmem L;
  size_t o = 0;
  auto take = [&](size_t n) { const size_t at = o; o += (n + 15) / 16 * 16; return at; };
  L.q = take(kTileBytes);
  L.c = take(2 * kTileBytes);
  L.v = take(2 * 3 * kTileBytes);
  L.raw = take(4 * kTile * kD);
  L.w = take(8 * (size_t)M);
  L.wpart = take(8 * 4 * kTile > 4 * (size_t)M ? 8 * 4 * kTile : 4 * (size_t)M);   // also the candidates of the selection
  L.tcnt = take(kSlots * 4 * kTile);
  L.trow = take(kSlots * 4 * kTile);
  L.np = take(4 * (size_t)M);
  L.nstay = take(4 * (size_t)M);
  L.xm = take(2 * 4 * 4 * kRows);
  L.xz = take(4 * 4 * kRows);
  L.nseen = take(4 * (size_t)((M + tile_m - 1) / tile_m));
  L.sel = take(4 * (size_t)M);
  L.list = take(4 * (size_t)(P > 0 ? P : 1));
  L.count = take(4 * 33);
  L.bad = take(4 * kMaxTiles);
  L.bars = take(8 * 6 + 8);
  L.total = o;
  return L;
}

__device__ __forceinline__ void compute_sync() { asm volatile("bar.sync 7, %0;" ::"n"(kCompute) : "memory"); }
// hand-over to the issuing warp
__device__ __forceinline__ void ready_arrive() { asm volatile("bar.arrive 8, %0;" ::"n"(kThreadsT) : "memory"); }
__device__ __forceinline__ void ready_wait() { asm volatile("bar.sync 8, %0;" ::"n"(kThreadsT) : "memory"); }
__device__ __forceinline__ void rows_sync(int q) { asm volatile("bar.sync %0, 128;" ::"r"(q + 1) : "memory"); }

// Two float32 as three pairs of bfloat16 (low half: lo) that add up to them exactly: each rounds to nearest what the ones before
// leave over, which has at most 16 and 7 significant bits.
__device__ __forceinline__ void split3(float lo, float hi, uint32_t (&p)[3]) {
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p[j]) : "f"(hi), "f"(lo));
    if (j < 2) {
      lo -= __uint_as_float(p[j] << 16);
      hi -= __uint_as_float(p[j] & 0xFFFF0000u);
    }
  }
}

__global__ void __launch_bounds__(kThreadsT, 1)
attend_tiled_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmCp, const TiledArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int M = a.M, C = a.C, P = a.P, tile_m = a.tile_m;
  const TiledSmem L = tiled_smem_layout(M, P, tile_m);
  unsigned char *Qs = smem + L.q, *Cs = smem + L.c, *Vs = smem + L.v;
  double *w = reinterpret_cast<double*>(smem + L.w), *wpart = reinterpret_cast<double*>(smem + L.wpart);
  float *tcnt = reinterpret_cast<float*>(smem + L.tcnt), *npS = reinterpret_cast<float*>(smem + L.np);
  float *nstay = reinterpret_cast<float*>(smem + L.nstay), *xm = reinterpret_cast<float*>(smem + L.xm);
  float *xz = reinterpret_cast<float*>(smem + L.xz), *nseen = reinterpret_cast<float*>(smem + L.nseen);
  int *trow = reinterpret_cast<int*>(smem + L.trow), *sel = reinterpret_cast<int*>(smem + L.sel), *sel_list = reinterpret_cast<int*>(smem + L.list);
  int *s_count = reinterpret_cast<int*>(smem + L.count);
  volatile int* bad = reinterpret_cast<volatile int*>(smem + L.bad);   // [tile] it holds a value sum that bfloat16 does not reach
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L.bars);
  uint64_t *bar_q = bars, *bar_c = bars + 1, *bar_s = bars + 3, *bar_o = bars + 5;   // query tile, codes [2], logits [2], product
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 6);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int blk = blockIdx.x, bh = blockIdx.y, h = bh % a.H;
  const int i0 = blk * a.block_q;
  const int rows = min(a.block_q, a.Nq - i0);
  const int ntiles = (M + tile_m - 1) / tile_m;            // importance tiles
  const int per_tile = (tile_m + kTile - 1) / kTile;       // code tiles of each (the last one may have fewer): 1 or 2
  const int last_subs = (M - (ntiles - 1) * tile_m + kTile - 1) / kTile;
  const bool need_w = (P > 0 && P < M) || a.importance_out != nullptr;
  const int na = need_w ? (ntiles - 1) * per_tile + last_subs : 0;   // code tiles of pass A, then those of pass C
  const int ptiles = (M + kTile - 1) / kTile, tiles = ptiles + (P * C + kTile - 1) / kTile;

  if (warp == kIssuer) {
    if (elect_one()) {
      prefetch_tmap(&tmQ);
      prefetch_tmap(&tmCp);
      for (int i = 0; i < 6; ++i) mbar_init(&bars[i], 1);
      mbar_fence_init();
      *abort_flag = 0;
    }
    __syncwarp();
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  if (tid < kMaxTiles) bad[tid] = 0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  if (warp == kIssuer) {
    // ---- loads and products.  Code tile u (pass A, then C) goes through buffer u & 1.
    auto wait = [&](uint64_t* bar, uint32_t parity) {      // all lanes agree
      return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, a.status_word, DEV_TIMEOUT_ATTEND));
    };
    auto load_codes = [&](int u) {
      int c0 = u * kTile;
      if (u < na) c0 = u / per_tile * tile_m + u % per_tile * kTile;
      else if ((c0 = (u - na) * kTile) >= M) return;       // children: the computing warps gather them
      if (elect_one()) {
        mbar_expect_tx(&bar_c[u & 1], kTileBytes);
        tma_load_2d(Cs + (u & 1) * kTileBytes, &tmCp, 0, h * M + c0, &bar_c[u & 1]);
      }
      __syncwarp();
    };
    uint32_t ph_c = 0, ph_s = 0;                           // a bit per barrier
    bool ok = true;
    auto logits = [&](int u, int n, int col, bool loaded) {
      if (loaded) {
        ok = wait(&bar_c[u & 1], (ph_c >> (u & 1)) & 1) && ok;
        ph_c ^= 1u << (u & 1);
      }
      tc_fence_after();
      if (ok && elect_one()) {
        const uint32_t idesc = umma_idesc_bf16(kRows, (n + 15) & ~15);
        const uint64_t qd = umma_desc_sw128(smem_u32(Qs)), cd = umma_desc_sw128(smem_u32(Cs + (u & 1) * kTileBytes));
#pragma unroll
        for (int k = 0; k < kD / 16; ++k) umma_bf16(tmem_base + col, qd + 2 * k, cd + 2 * k, idesc, k > 0);
      }
      __syncwarp();
    };
    auto commit = [&](uint64_t* bar) {
      if (elect_one()) umma_commit(bar);
      __syncwarp();
    };
    auto logits_done = [&](int i) {
      ok = wait(&bar_s[i], (ph_s >> i) & 1) && ok;
      ph_s ^= 1u << i;
    };
    // tile k of pass C (its codes have landed), two ahead of the weights; then the load that takes its buffer
    auto tile_logits = [&](int k) {
      const bool child = k >= ptiles;
      logits(na + k, child ? min(kTile, P * C - (k - ptiles) * kTile) : min(kTile, M - k * kTile), (k & 1) * kTile, !child);
      commit(&bar_s[k & 1]);
    };
    auto next_codes = [&](int k) {
      logits_done(k & 1);
      load_codes(na + k + 2);
    };
    if (elect_one()) {
      mbar_expect_tx(bar_q, kTileBytes);
      tma_load_3d(Qs, &tmQ, 0, i0, bh, bar_q);
    }
    __syncwarp();
    load_codes(0);
    load_codes(1);
    ok = wait(bar_q, 0);
    for (int t = 0, u = 0; t < (need_w ? ntiles : 0); ++t) {
      const int t0 = t * tile_m, subs = t + 1 < ntiles ? per_tile : last_subs;
      if (t > 0) ready_wait();                             // the logits of the tile before have been read
      for (int s = 0; s < subs; ++s) logits(u + s, min(kTile, min(tile_m, M - t0) - s * kTile), s * kTile, true);
      commit(bar_s);
      logits_done(0);
      for (int s = 0; s < subs; ++s) load_codes(u + s + 2);
      u += subs;
    }
    if (need_w) ready_wait();
    tile_logits(0);
    if (ptiles > 1) tile_logits(1);
    next_codes(0);
    if (ptiles > 1) next_codes(1);
    const uint32_t idesc_o = umma_idesc_bf16(kRows, kD) | (1u << 16);   // B (the value rows) is MN-major
    for (int k = 0; k < tiles; ++k) {
      ready_wait();                                        // weights and values of tile k, gathered codes of tile k + 2
      if (k == 0 && ptiles == 1 && tiles > 1) tile_logits(1);
      if (k + 2 < tiles) tile_logits(k + 2);
      const int n = k >= ptiles ? min(kTile, P * C - (k - ptiles) * kTile) : min(kTile, M - k * kTile);
      if (ok && !bad[k] && elect_one()) {
        const uint32_t v0 = smem_u32(Vs + (k & 1) * 3 * kTileBytes);
        const int steps = (n + 15) >> 4;
        bool first = true;
        auto product = [&](int wp, int vp) {
          const uint64_t vd = umma_desc_sw128_mn(v0 + vp * kTileBytes, kTileBytes);
          for (int s = 0; s < steps; ++s) {
            umma_bf16_ts(tmem_base + kColO, tmem_base + kColW + wp * (kTile / 2) + 8 * s, vd + (uint64_t)(128 * s), idesc_o, !first);
            first = false;
          }
        };
        product(0, 2);
        product(2, 0);
        product(1, 1);
        product(0, 1);
        product(1, 0);
        product(0, 0);
      }
      __syncwarp();
      commit(bar_o);
      if (k == 0 && ptiles == 1 && tiles > 1) next_codes(1);
      if (k + 2 < tiles) next_codes(k + 2);
    }
  } else {
    const int q = warp & 3, cq = warp >> 2, r = q * 32 + lane;
    const int g = lane >> 2, t4 = lane & 3;                // fragment rows 32 q + g + 8 h, columns 32 cq + 8 b + 2 t4, + 1
    const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16);
    const float* Vp = a.Vp + (size_t)bh * M * kD;
    const float* Vc = a.Vc + (size_t)bh * M * C * kD;
    const float* np_ = a.np_ + (size_t)bh * M;
    const float* nc = a.nc + (size_t)bh * M * C;
    const __nv_bfloat16* Cch = a.Cc + (size_t)h * M * C * kD;
    auto wait = [&](uint64_t* bar, uint32_t parity) { return mbar_wait(bar, parity, abort_flag, a.status_word, DEV_TIMEOUT_ATTEND); };
    auto to_frag = [&](float v, float (&out)[4]) {         // of rows g + 8 h, from the lane that stands for the row
#pragma unroll
      for (int i = 0; i < 4; ++i) out[i] = __shfl_sync(0xffffffffu, v, g + 8 * i);
    };
    // Over the quad and the four warps of a row, through buffer `buf` of xm.  In pass C a warp may be a turn ahead of one that
    // still reads the maxima of the turn before: the turns take the buffers alternately (through turn k - 2 all are, see describe()).
    auto row_max = [&](float (&m)[4], int buf) {
      float* xb = xm + buf * 4 * kRows;
#pragma unroll
      for (int i = 0; i < 4; ++i) m[i] = quad_max(m[i]);
      xb[cq * kRows + q * 32 + g + 8 * t4] = pick4(m, t4);
      rows_sync(q);
      to_frag(fmaxf(fmaxf(xb[r], xb[kRows + r]), fmaxf(xb[2 * kRows + r], xb[3 * kRows + r])), m);
    };
    auto row_sum = [&](float (&z)[4]) {
#pragma unroll
      for (int i = 0; i < 4; ++i) z[i] = quad_sum(z[i]);
      xz[cq * kRows + q * 32 + g + 8 * t4] = pick4(z, t4);
      rows_sync(q);
      to_frag((xz[r] + xz[kRows + r]) + (xz[2 * kRows + r] + xz[3 * kRows + r]), z);
    };
    // This thread's logits of the tile at TMEM column `col`: e[h][2 b + u], -inf where no key stands behind the column (its
    // weight is then exp(-inf) = 0 against any reference, without a branch); cnt[2 b + u] of its columns.
    auto load_logits = [&](int col, const float* counts, int n, float (&e)[4][8], float (&cnt)[8]) {
      if (32 * cq < n) {                                   // warp-uniform
        uint32_t s[2][16];
        tmem_ld_frag<4>(t_row + col + 32 * cq, s);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int c = 32 * cq + 8 * b + 2 * t4;
          cnt[2 * b] = c < n ? counts[c] : 0.f;
          cnt[2 * b + 1] = c + 1 < n ? counts[c + 1] : 0.f;
        }
        tmem_ld_wait_frag<4>(s);
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int u = 0; u < 2; ++u)
              e[i][2 * b + u] = cnt[2 * b + u] > 0.f ? __uint_as_float(s[i >> 1][4 * b + 2 * (i & 1) + u]) * a.scale : -INFINITY;
      } else {
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          cnt[c] = 0.f;
#pragma unroll
          for (int i = 0; i < 4; ++i) e[i][c] = -INFINITY;
        }
      }
    };

    pdl_wait();                                            // the counts and sums of the kernels before
    for (int j = tid; j < M; j += kCompute) {
      const float n = ld_after_wait(np_ + j);
      npS[j] = n;
      if (a.stays) {                                       // keys that stay with their parent
        float s = 0.f;
        for (int c = 0; c < C; ++c) s += ld_after_wait(nc + (size_t)j * C + c);
        nstay[j] = n - s;
      }
      w[j] = 0.0;
      sel[j] = 0;
    }
    compute_sync();
    if (tid < ntiles) {                                    // keys of each tile
      float seen = 0.f;
      const int j1 = min(M, (tid + 1) * tile_m);
      for (int j = tid * tile_m; j < j1; ++j) seen += npS[j];
      nseen[tid] = seen;
    }

    // ---- pass A: importance, tile by tile: a tile's weights against the maximum and the denominator seen up to it (Eq.
    // "aproxdenom"), so they stay finite however far a later tile's logits lie above them
    uint32_t ph_s = 0;                                     // a bit per barrier
    if (need_w) {
      float m[4] = {kLowest, kLowest, kLowest, kLowest}, z[4] = {0.f, 0.f, 0.f, 0.f};
      bool valid[4];                                       // rows of this block
#pragma unroll
      for (int i = 0; i < 4; ++i) valid[i] = q * 32 + g + 8 * i < rows;
      for (int t0 = 0; t0 < M; t0 += tile_m) {
        const int width = min(tile_m, M - t0), subs = (width + kTile - 1) / kTile;
        wait(bar_s, ph_s & 1);
        ph_s ^= 1;
        tc_fence_after();
        float e[4][8], cnt[8];
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        for (int s = 0; s < subs; ++s) {
          load_logits(s * kTile, npS + t0 + s * kTile, width - s * kTile, e, cnt);
#pragma unroll
          for (int c = 0; c < 8; ++c)
#pragma unroll
            for (int i = 0; i < 4; ++i) mx[i] = fmaxf(mx[i], e[i][c]);
        }
        row_max(mx, 0);                                    // (barriers of all warps at the end of each turn)
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (mx[i] > m[i]) {
            z[i] *= expf(m[i] - mx[i]);
            m[i] = mx[i];
          }
        auto weights = [&](int s) {
          if (subs > 1) load_logits(s * kTile, npS + t0 + s * kTile, width - s * kTile, e, cnt);
#pragma unroll
          for (int c = 0; c < 8; ++c)
#pragma unroll
            for (int i = 0; i < 4; ++i) e[i][c] = expf(e[i][c] - m[i]);
        };
        float zs[4] = {0.f, 0.f, 0.f, 0.f};
        for (int s = 0; s < subs; ++s) {
          weights(s);
#pragma unroll
          for (int c = 0; c < 8; ++c)
#pragma unroll
            for (int i = 0; i < 4; ++i) zs[i] = fmaf(e[i][c], cnt[c], zs[i]);
        }
        row_sum(zs);
        double inv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          z[i] += zs[i];
          inv[i] = valid[i] && z[i] != 0.f ? 1.0 / (double)z[i] : 0.0;   // (a row of the next block may be NaN)
        }
        for (int s = subs - 1; s >= 0; --s) {              // the last code tile's weights are still there
          if (s < subs - 1) weights(s);
          if (s == 0) {                                    // the logits have been read
            tc_fence_before();
            ready_arrive();
          }
          double d[8];
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            d[c] = 0.0;
#pragma unroll
            for (int i = 0; i < 4; ++i) d[c] = fma((double)(valid[i] ? e[i][c] : 0.f), inv[i], d[c]);
          }
          // over the 8 lanes of a column: lane 4 g + t keeps column 8 (g / 2) + 2 t + g % 2
#pragma unroll
          for (int n = 4, bit = 16; n; n >>= 1, bit >>= 1) {
            const bool hi = (lane & bit) != 0;
#pragma unroll
            for (int c = 0; c < 4; ++c)
              if (c < n) d[c] = (hi ? d[c + n] : d[c]) + __shfl_xor_sync(0xffffffffu, hi ? d[c] : d[c + n], bit);
          }
          wpart[q * kTile + 32 * cq + 8 * (g >> 1) + 2 * t4 + (g & 1)] = d[0];
          compute_sync();
          if (tid < min(kTile, width - s * kTile))
            w[t0 + s * kTile + tid] = (wpart[tid] + wpart[kTile + tid]) + (wpart[2 * kTile + tid] + wpart[3 * kTile + tid]);
          compute_sync();
        }
      }
      for (int j = tid; j < M; j += kCompute) {
        float seen = 0.f;                                  // extrapolated by the keys seen up to the tile
        for (int t = 0; t <= j / tile_m; ++t) seen += nseen[t];
        const double x = w[j] * (double)npS[j] * ((double)seen / (double)a.Nk);
        w[j] = x;
        if (a.importance_out) a.importance_out[((size_t)bh * a.nblk + blk) * M + j] = (float)x;
      }
    }
    compute_sync();
    if (P > 0)
      select_parents(w, M, P, sel, sel_list, reinterpret_cast<int*>(wpart), s_count, s_count + 32,
                     a.topp_out ? a.topp_out + ((size_t)bh * a.nblk + blk) * P : nullptr, [] { compute_sync(); });

    // ---- pass C: merged softmax over unrefined parents, stay residuals and children of refined parents
    auto first_of = [&](int k) { return k >= ptiles ? (k - ptiles) * kTile : k * kTile; };
    auto width_of = [&](int k) { return min(kTile, (k >= ptiles ? P * C : M) - first_of(k)); };
    auto child_row = [&](int e) {                          // (e < 2^13, C <= 16: the division by multiplication is exact)
      const int f = (int)(((uint32_t)e * a.inv_C) >> 18);
      return sel_list[f] * C + (e - f * C);
    };
    // What stands behind column tid of tile k: the keys, and the row of their value sums, a child's (kChildRow) or a parent's, less
    // the children's where the parent is refined (kStayRow); -1: none.
    // Tiles 0 to 2 are described before the loop, ahead of a barrier, tile k + 3 in turn k.  No barrier joins all warps in a
    // turn; what orders them is take_product(k - 1) in turn k: it waits for a product that the issuing warp starts behind the
    // arrivals of all warps in turn k - 1.  A warp in turn k therefore knows every other to be through turn k - 2, in which
    // tile k + 1, the furthest it reads (load_values), was described.  And it overwrites the slot of tile k - 5, which was last read
    // in turn k - 4 (a product on the CUDA cores, a turn behind its tile); six slots would do.
    auto describe = [&](int k) {
      if (tid >= kTile || k >= tiles) return;
      float n = 0.f;
      int row = -1;
      if (tid < width_of(k)) {
        const int e = first_of(k) + tid;
        if (k >= ptiles) {
          const int cr = child_row(e);
          n = ld_after_wait(nc + cr);
          row = cr | kChildRow;
        } else {
          n = sel[e] ? (a.stays ? nstay[e] : 0.f) : npS[e];
          if (n > 0.f) row = sel[e] ? e | kStayRow : e;
        }
      }
      tcnt[(k & (kSlots - 1)) * kTile + tid] = n;
      trow[(k & (kSlots - 1)) * kTile + tid] = row;
    };
    // value sums 4 ch .. + 3 of such a row
    auto value_of = [&](int row, int ch) {
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (row >= 0) {
        const int j = row & (kStayRow - 1);
        v = ld_after_wait(reinterpret_cast<const float4*>((row & kChildRow ? Vc : Vp) + (size_t)j * kD) + ch);
        if (row & kStayRow)
          for (int cc = 0; cc < C; ++cc) {
            const float4 x = ld_after_wait(reinterpret_cast<const float4*>(Vc + ((size_t)j * C + cc) * kD) + ch);
            v.x -= x.x; v.y -= x.y; v.z -= x.z; v.w -= x.w;
          }
      }
      return v;
    };
    // Value sums of tile k on their way: rows tid / 16 + 32 i, dimensions 4 (tid % 16) .. + 3, each thread its own.
    const uint32_t own_v = smem_u32(smem + L.raw) + 16 * tid;
    auto load_values = [&](int k) {
      int row[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) row[i] = trow[(k & (kSlots - 1)) * kTile + (tid >> 4) + 32 * i];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t dst = own_v + 16 * kCompute * i;
        if (row[i] >= 0 && (row[i] & kStayRow)) {
          const float4 v = value_of(row[i], tid & 15);
          asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
        } else {                                           // (no row: nothing is read, zeros are written)
          const int j = row[i] < 0 ? 0 : row[i] & (kStayRow - 1);
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst),
                       "l"((row[i] & kChildRow ? Vc : Vp) + (size_t)j * kD + 4 * (tid & 15)), "r"(row[i] < 0 ? 0 : 16) : "memory");
        }
      }
    };
    auto store_values = [&](int k) {
      bool fits = true;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float x[4];
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]) : "r"(own_v + 16 * kCompute * i) : "memory");
#pragma unroll
        for (int e = 0; e < 4; ++e) fits = fits && fabsf(x[e]) <= kLargestBf16;
        uint32_t p[2][3];
        split3(x[0], x[1], p[0]);
        split3(x[2], x[3], p[1]);
        const uint32_t at = smem_u32(Vs + (k & 1) * 3 * kTileBytes) + sw128_offset((tid >> 4) + 32 * i, 4 * (tid & 15));
#pragma unroll
        for (int j = 0; j < 3; ++j)
          asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at + j * kTileBytes), "r"(p[0][j]), "r"(p[1][j]) : "memory");
      }
      if (!fits) bad[k] = 1;
    };
    auto gather_codes = [&](int k) {                       // children's codeword rows of tile k, zeros behind them
      const int n = width_of(k), n16 = (n + 15) & ~15;
      const uint32_t base = smem_u32(Cs + ((na + k) & 1) * kTileBytes);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int c = (tid >> 3) + 64 * i, ch = tid & 7;
        const uint32_t dst = base + sw128_offset(c, 8 * ch);
        if (c < n)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(Cch + (size_t)child_row(first_of(k) + c) * kD + 8 * ch) : "memory");
        else if (c < n16)
          asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(dst), "r"(0) : "memory");
      }
    };
    float o[4][4], z[4], m[4];                             // o[h][2 b + u]: dimensions 16 cq + 8 b + 2 t4 + u
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      z[i] = 0.f;
      m[i] = kLowest;
#pragma unroll
      for (int c = 0; c < 4; ++c) o[i][c] = 0.f;
    }
    uint32_t ph_o = 0;
    // o += the value product of tile k
    auto take_product = [&](int k) {
      wait(bar_o, ph_o);
      ph_o ^= 1;
      tc_fence_after();
      if (!bad[k]) {
        uint32_t x[2][8];
        tmem_ld_frag<2>(t_row + kColO + 16 * cq, x);
        tmem_ld_wait_frag<2>(x);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int c = 0; c < 4; ++c) o[i][c] += __uint_as_float(x[i >> 1][4 * (c >> 1) + 2 * (i & 1) + (c & 1)]);
        return;
      }
      const int n = width_of(k);
#pragma unroll 1
      for (int c = 0; c < n; ++c) {                        // the weights' parts add up to them again
        float wc = 0.f;
#pragma unroll
        for (int j = 2; j >= 0; --j) {
          uint32_t x;
          asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(x) : "r"(t_row + kColW + j * (kTile / 2) + (c >> 1)) : "memory");
          asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(x)::"memory");
          wc += __uint_as_float((c & 1) ? x & 0xFFFF0000u : x << 16);
        }
        float wr[4];
        to_frag(wc, wr);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          const int col = 16 * cq + 8 * b + 2 * t4;
          const float4 v = value_of(trow[(k & (kSlots - 1)) * kTile + c], col >> 2);
          const float v0 = (col & 2) ? v.z : v.x, v1 = (col & 2) ? v.w : v.y;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            o[i][2 * b] = fmaf(wr[i], v0, o[i][2 * b]);
            o[i][2 * b + 1] = fmaf(wr[i], v1, o[i][2 * b + 1]);
          }
        }
      }
      rows_sync(q);                                        // before one of the four warps overwrites its weights
    };
    if (1 >= ptiles && 1 < tiles) {                        // (from tile 2 on behind the logits of tile k - 2)
      // its buffer held a code tile of pass A, whose logits are done, or nothing yet
      gather_codes(1);
    }
    for (int k = 0; k < 3; ++k) describe(k);
    compute_sync();
    load_values(0);
    cp_async_wait_all();
    for (int k = 0; k < tiles; ++k) {
      wait(&bar_s[k & 1], (ph_s >> (k & 1)) & 1);
      ph_s ^= 1u << (k & 1);
      tc_fence_after();
      if (k + 2 < tiles && k + 2 >= ptiles) gather_codes(k + 2);
      store_values(k);
      if (k + 1 < tiles) load_values(k + 1);
      describe(k + 3);
      float e[4][8], cnt[8];
      load_logits((k & 1) * kTile, tcnt + (k & (kSlots - 1)) * kTile, width_of(k), e, cnt);
      float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int c = 0; c < 8; ++c)
#pragma unroll
        for (int i = 0; i < 4; ++i) mx[i] = fmaxf(mx[i], e[i][c]);
      row_max(mx, k & 1);
      float alpha[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float up = fmaxf(m[i], mx[i]);               // (mx may be -inf, m is finite or +inf)
        alpha[i] = up > m[i] ? expf(m[i] - up) : 1.f;
        m[i] = up;
        z[i] *= alpha[i];
      }
#pragma unroll
      for (int c = 0; c < 8; ++c)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          e[i][c] = expf(e[i][c] - m[i]);
          z[i] = fmaf(e[i][c], cnt[c], z[i]);
        }
      if (k > 0) take_product(k - 1);                      // and with it the weights' columns
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) o[i][c] *= alpha[i];
      if (32 * cq < width_of(k)) {
        uint32_t part[3][2][8];
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            uint32_t p[3];
            split3(e[i][2 * b], e[i][2 * b + 1], p);
#pragma unroll
            for (int j = 0; j < 3; ++j) part[j][i >> 1][2 * b + (i & 1)] = p[j];
          }
#pragma unroll
        for (int j = 0; j < 3; ++j) tmem_st_weights(t_row + kColW + j * (kTile / 2) + 16 * cq, part[j]);
        tmem_st_wait();
      }
      cp_async_wait_all();
      fence_proxy_async();
      tc_fence_before();
      ready_arrive();
    }
    take_product(tiles - 1);
    row_sum(z);
    // rows -> shared memory (the query tile's place) -> whole lines of Y
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float inv = 1.f / z[i];
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const __nv_bfloat162 v = __floats2bfloat162_rn(o[i][2 * b] * inv, o[i][2 * b + 1] * inv);
        *reinterpret_cast<__nv_bfloat162*>(Qs + sw128_offset(q * 32 + g + 8 * i, 16 * cq + 8 * b + 2 * t4)) = v;
      }
    }
    compute_sync();
    __nv_bfloat16* Yb = a.Y + ((size_t)bh * a.Nq + i0) * kD;
    for (int u = tid; u < rows * 8; u += kCompute)
      reinterpret_cast<uint4*>(Yb)[u] = *reinterpret_cast<const uint4*>(Qs + sw128_offset(u >> 3, 8 * (u & 7)));
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  if (warp == kIssuer) tmem_dealloc(tmem_base, 512);
}

// A block costs this kernel a tile of 128 rows and tiles of 128 codewords whatever it has of them, on an SM of its own; the CUDA-core
// kernel takes 64 of each at a time, two blocks to an SM.  So small blocks and small codebooks stay there.  Us per call here
// and there, H4 N4096 and H12 N8192, C4, importance tiles of min(M, 128) unless said otherwise:
//   128 rows  M64 P8 39.0 and 39.0, 117.7 and 112.0 (H16 N4096); tiles of 32 0.91 and 0.93 times the other's time
//             M64 P16 0.99 and 1.00 times; M80 P4 0.91 and 0.82 times; M128 P16 0.80 and 0.73 times
//   64 rows   M64 P8 55.9 and 43.1; M128 P16 1.03 and 1.01 times; M160 P16 1.09 and 1.08 times, M200 P10 0.87 and 0.85
//             (tiles of 32: 1.03 and 1.02) times; M128 P28 0.92 and 0.91 times; M256 P64 0.70 and 0.69 times
//   16 rows   M64 P8 144.0 and 99.0; M160 P16 1.09 and 1.10 times, M200 P10 0.83 and 0.83 times, M512 P64 0.61 times
bool tc_tiled_pays(const avq_problem& p, int32_t P, int32_t block_q, int32_t tile_m) {
  const int64_t columns = (int64_t)p.M + (int64_t)P * p.C;
  if (block_q <= 64) return columns >= 240;
  return p.M > (tile_m < 64 ? tile_m : 64) || columns >= 128;
}

}  // namespace

bool tc_tiled_fits(const avq_problem& p, int32_t P, int32_t block_q, int32_t tile_m) {
  return p.dtype == AVQ_BF16 && p.d == kD && block_q <= kRows && tile_m <= 2 * kTile && !(p.flags & AVQ_FLAG_CORRECTING) &&
         tiled_smem_layout(p.M, P, tile_m).total <= kSmemMax && tc_tiled_pays(p, P, block_q, tile_m);
}

avq_status tc_attend_tiled(const avq_problem& p, const void* Q, const void* Cp, const void* Cc, const float* Vp, const float* np_,
                           const float* Vc, const float* nc, int32_t P, int32_t block_q, void* Y, int32_t* topp_out,
                           float* importance_out, int32_t tile_m, int32_t* status_word, cudaStream_t st) {
  const uint64_t BH = (uint64_t)p.B * p.H;
  CUtensorMap tmQ, tmCp;
  {
    const uint64_t dims[3] = {(uint64_t)kD, (uint64_t)p.Nq, BH};
    const uint32_t box[3] = {64, (uint32_t)kRows, 1};
    const avq_status s = make_tmap_bf16(&tmQ, Q, 3, dims, box);
    if (s != AVQ_OK) return s;
  }
  {
    const uint64_t dims[2] = {(uint64_t)kD, (uint64_t)p.H * p.M};
    const uint32_t box[2] = {64, (uint32_t)kTile};
    const avq_status s = make_tmap_bf16(&tmCp, Cp, 2, dims, box);
    if (s != AVQ_OK) return s;
  }
  TiledArgs a;
  a.Cc = static_cast<const __nv_bfloat16*>(Cc);
  a.Vp = Vp; a.np_ = np_; a.Vc = Vc; a.nc = nc;
  a.Y = static_cast<__nv_bfloat16*>(Y);
  a.topp_out = topp_out;
  a.importance_out = importance_out;
  a.status_word = status_word;
  a.H = p.H; a.Nq = p.Nq; a.M = p.M; a.C = p.C; a.P = P; a.block_q = block_q;
  a.nblk = (p.Nq + block_q - 1) / block_q;
  a.stays = (p.flags & AVQ_FLAG_PARENT_STAYS) ? 1 : 0;
  a.tile_m = tile_m;
  a.Nk = p.Nk;
  a.inv_C = ((1u << 18) + (uint32_t)p.C - 1) / (uint32_t)p.C;
  a.scale = p.scale;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return AVQ_ERR_CUDA;
  const avq_status s = open_shared_memory<attend_tiled_kernel>(dev);
  if (s != AVQ_OK) return s;
  return cuda_ok(launch_pdl(attend_tiled_kernel, dim3((unsigned)a.nblk, (unsigned)BH), dim3(kThreadsT),
                            tiled_smem_layout(p.M, P, tile_m).total, st, true, tmQ, tmCp, a));
}

}  // namespace avq
