// Host-side helpers of the tensor-core path: driver entry point for tensor-map encoding.
#include <mutex>

#include "avq_tc_common.cuh"

namespace avq {
namespace tc {

EncodeTiledFn encode_tiled_fn() {
  static EncodeTiledFn fn = []() -> EncodeTiledFn {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

namespace {
// Encoding a tensor map costs a few microseconds of host time and a forward needs six of them, so
// recent encodings are kept: the result depends only on (base, rank, dims, strides, box).
constexpr int kMaxRank = 4;
struct TmapKey {
  const void* base;
  int rank;
  uint64_t dims[kMaxRank];
  uint64_t strides[kMaxRank - 1];   // bytes, of dimensions 1..
  uint32_t box[kMaxRank];
  bool operator==(const TmapKey& o) const {
    if (base != o.base || rank != o.rank) return false;
    for (int i = 0; i < rank; ++i)
      if (dims[i] != o.dims[i] || box[i] != o.box[i]) return false;
    for (int i = 0; i + 1 < rank; ++i)
      if (strides[i] != o.strides[i]) return false;
    return true;
  }
};
// A set-associative table: a call looks at the entries of one set instead of at all of them.
constexpr int kTmapSets = 64, kTmapWays = 4;
std::mutex g_tmap_mu;
TmapKey g_tmap_keys[kTmapSets][kTmapWays];                // rank 0: empty
CUtensorMap g_tmap_vals[kTmapSets][kTmapWays];
uint8_t g_tmap_next[kTmapSets];

unsigned tmap_set(const TmapKey& k) {
  uint64_t h = reinterpret_cast<uintptr_t>(k.base) >> 8;
  h = (h ^ (k.dims[1] * 31) ^ ((uint64_t)k.box[1] << 20) ^ (uint64_t)k.rank << 12) * 0x9E3779B97F4A7C15ull;
  return (unsigned)(h >> 58);
}

avq_status encode(CUtensorMap* map, const TmapKey& key) {
  const unsigned set = tmap_set(key);
  {
    std::lock_guard<std::mutex> lock(g_tmap_mu);
    for (int i = 0; i < kTmapWays; ++i)
      if (g_tmap_keys[set][i] == key) { *map = g_tmap_vals[set][i]; return AVQ_OK; }
  }
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return AVQ_ERR_CUDA;
  cuuint64_t gdim[kMaxRank], gstride[kMaxRank];
  cuuint32_t bdim[kMaxRank], estr[kMaxRank];
  for (int i = 0; i < key.rank; ++i) {
    gdim[i] = key.dims[i];
    bdim[i] = key.box[i];
    estr[i] = 1;
    if (i + 1 < key.rank) gstride[i] = key.strides[i];
  }
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)key.rank, const_cast<void*>(key.base), gdim,
                  gstride, bdim, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return AVQ_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_tmap_mu);
  const int way = g_tmap_next[set]++ % kTmapWays;
  g_tmap_keys[set][way] = key;
  g_tmap_vals[set][way] = *map;
  return AVQ_OK;
}
}  // namespace

avq_status make_tmap_bf16(CUtensorMap* map, const void* base, int rank, const uint64_t* dims,
                          const uint32_t* box) {
  if (rank < 1 || rank > 3) return AVQ_ERR_UNSUPPORTED;
  TmapKey key = {};
  key.base = base;
  key.rank = rank;
  uint64_t pitch = 2;
  for (int i = 0; i < rank; ++i) {
    key.dims[i] = dims[i];
    key.box[i] = box[i];
    pitch *= dims[i];
    if (i + 1 < rank) key.strides[i] = pitch;   // byte stride of dimension i+1
  }
  return encode(map, key);
}

avq_status make_tmap_codes(CUtensorMap* map, const void* base, int d, uint64_t rows, uint32_t box_rows) {
  if (rows % 8 != 0 || box_rows % 8 != 0) return AVQ_ERR_UNSUPPORTED;
  const uint64_t row = 2 * (uint64_t)d;
  TmapKey key = {};
  key.base = base;
  key.rank = 4;
  key.dims[0] = (uint64_t)d; key.dims[1] = 2; key.dims[2] = 4; key.dims[3] = rows / 8;
  key.strides[0] = 4 * row; key.strides[1] = row; key.strides[2] = 8 * row;
  key.box[0] = 64; key.box[1] = 2; key.box[2] = 4; key.box[3] = box_rows / 8;
  return encode(map, key);
}

}  // namespace tc
}  // namespace avq
