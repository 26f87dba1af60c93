// Encoded tensor maps are kept: a caller that launches directly (no CUDA graph) passes the same pointers and shapes
// step after step, and an encode is a driver call.  A map depends on nothing but the arguments of the encode (swizzle,
// interleave, promotion and fill are the same for every map of the library), so the key is those arguments, compared
// byte for byte.  The table holds three maps for each layer of the largest models several times over (a table of 16
// missed on every launch of a 32-layer step): 256 sets of 4, the set chosen by a hash of the key, replaced in turn
// inside a set; one lock per set, held for a copy of 128 bytes.
#include "tensor_map.cuh"

#include <string.h>

#include "common.cuh"

namespace seqtree {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static void* cached = nullptr;  // the driver's entry point, looked up once (the same answer from every thread)
  void* p = __atomic_load_n(&cached, __ATOMIC_ACQUIRE);
  if (p == nullptr) {
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess || p == nullptr)
      return nullptr;
    __atomic_store_n(&cached, p, __ATOMIC_RELEASE);
  }
  return reinterpret_cast<EncodeTiledFn>(p);
}

namespace {
struct MapKey {
  const void* base;
  cuuint64_t dims[5], strides[4];
  cuuint32_t box[5];
  int32_t rank, type;
  int32_t pad;
};
static_assert(sizeof(MapKey) % 8 == 0, "the key is hashed and compared as 64-bit words");
constexpr int kSets = 256, kWays = 4;
struct MapSet {
  MapKey key[kWays];
  CUtensorMap map[kWays];
  int used, next, lock;
};
MapSet g_sets[kSets];

void lock_set(MapSet& s) { while (__atomic_exchange_n(&s.lock, 1, __ATOMIC_ACQUIRE) != 0) { } }
void unlock_set(MapSet& s) { __atomic_store_n(&s.lock, 0, __ATOMIC_RELEASE); }
}  // namespace

bool tensor_map(CUtensorMap* out, CUtensorMapDataType type, unsigned rank, const void* base, const cuuint64_t* dims,
                const cuuint64_t* strides, const cuuint32_t* box) {
  MapKey key;
  memset(&key, 0, sizeof(key));
  key.base = base; key.rank = (int32_t)rank; key.type = (int32_t)type;
  for (unsigned i = 0; i < rank; ++i) { key.dims[i] = dims[i]; key.box[i] = box[i]; }
  for (unsigned i = 0; i + 1 < rank; ++i) key.strides[i] = strides[i];
  uint64_t h = 0;
  for (size_t i = 0; i < sizeof(key) / 8; ++i) {
    uint64_t w;
    memcpy(&w, reinterpret_cast<const char*>(&key) + 8 * i, 8);
    h = (h ^ w) * 0x9E3779B97F4A7C15ull;
    h ^= h >> 29;
  }
  MapSet& set = g_sets[h % kSets];
  lock_set(set);
  for (int w = 0; w < set.used; ++w)
    if (memcmp(&set.key[w], &key, sizeof(key)) == 0) {
      *out = set.map[w];
      unlock_set(set);
      return true;
    }
  unlock_set(set);
  const EncodeTiledFn encode = encode_fn();
  if (encode == nullptr) return false;
  const cuuint32_t ones[5] = {1, 1, 1, 1, 1};
  if (encode(out, type, rank, const_cast<void*>(base), dims, strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return false;
  lock_set(set);
  const int w = set.used < kWays ? set.used++ : (set.next++ % kWays);
  set.key[w] = key;
  set.map[w] = *out;
  unlock_set(set);
  return true;
}

}  // namespace seqtree
