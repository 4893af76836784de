// Tensor maps (TMA descriptors) of the kernels' operands.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

namespace fbq {

struct MapSpec {
    const void *base;
    CUtensorMapDataType type;
    int ndim;                     // 2 or 3
    cuuint64_t dims[3];           // elements, innermost first
    cuuint64_t strides[2];        // bytes between indices of dimension 1, 2
    cuuint32_t box[3];
    CUtensorMapSwizzle swizzle;
};

// Encodes a map.  Reads outside the tensor return zeros.
cudaError_t encode_map(CUtensorMap *out, const MapSpec &spec);
// The same for operands that stay where they are from call to call (weights): maps hold addresses and extents only,
// never data, so they are encoded once per (address, shape) and kept, up to a bounded number.
cudaError_t cached_map(CUtensorMap *out, const MapSpec &spec);

// 2-D map of a row-major matrix with rows of `cols` elements of `elem_bytes` bytes each.
inline MapSpec matrix_map(const void *base, CUtensorMapDataType type, int elem_bytes, size_t cols, size_t rows, int box_cols, int box_rows,
                          CUtensorMapSwizzle swizzle)
{
    MapSpec m{};
    m.base = base;
    m.type = type;
    m.ndim = 2;
    m.dims[0] = cols;
    m.dims[1] = rows;
    m.strides[0] = (cuuint64_t)cols * elem_bytes;
    m.box[0] = (cuuint32_t)box_cols;
    m.box[1] = (cuuint32_t)box_rows;
    m.swizzle = swizzle;
    return m;
}

}  // namespace fbq
