// Host side of the TMA descriptors: encoding, and the table of the maps that are kept.
#include <cudaTypedefs.h>

#include <cstring>
#include <mutex>
#include <unordered_map>

#include "fbq_maps.h"

namespace fbq {
namespace {

struct Key {
    uint64_t v[11];
    bool operator==(const Key &o) const { return memcmp(v, o.v, sizeof v) == 0; }
};
struct KeyHash {
    size_t operator()(const Key &k) const
    {
        uint64_t h = 0x9E3779B97F4A7C15ull;
        for (uint64_t x : k.v) {
            h = (h ^ x) * 0xD6E8FEB86659FD93ull;
            h ^= h >> 32;
        }
        return (size_t)h;
    }
};
Key key_of(const MapSpec &m)
{
    return Key{{(uint64_t)(uintptr_t)m.base, (uint64_t)m.type | (uint64_t)m.ndim << 32, m.dims[0], m.dims[1], m.dims[2], m.strides[0], m.strides[1],
                m.box[0], m.box[1], m.box[2], (uint64_t)m.swizzle}};
}

// A model keeps up to three maps per linear (codes, A, B): a lookup has to cost the same with thousands of them, so
// they sit in a hash table (a list searched from its head cost a decode call of a 32-layer stack tens of microseconds).
// Full, the table starts again from empty: the maps of the weights still in use come back with their next call.
constexpr size_t kKeep = 16384;                     // about 4 MB of host memory
std::mutex g_mu;
std::unordered_map<Key, CUtensorMap, KeyHash> g_maps;

}  // namespace

cudaError_t encode_map(CUtensorMap *out, const MapSpec &m)
{
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult qres;
        const cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
        if (e != cudaSuccess) return e;
        if (qres != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
        encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    const cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = encode(out, m.type, (cuuint32_t)m.ndim, const_cast<void *>(m.base), m.dims, m.strides, m.box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              m.swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t cached_map(CUtensorMap *out, const MapSpec &m)
{
    const Key key = key_of(m);
    std::lock_guard<std::mutex> lk(g_mu);
    const auto it = g_maps.find(key);
    if (it != g_maps.end()) {
        *out = it->second;
        return cudaSuccess;
    }
    if (const cudaError_t e = encode_map(out, m); e != cudaSuccess) return e;
    if (g_maps.size() >= kKeep) g_maps.clear();
    g_maps.emplace(key, *out);
    return cudaSuccess;
}

}  // namespace fbq
