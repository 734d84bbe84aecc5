// Tensor maps of row-major matrices for TMA.
#pragma once
#include <cstdint>
#include <cuda.h>

namespace oprag {

// Row-major rows x d matrix of `dtype` (kBF16 or kF32): boxes of box_rows rows
// of 128 bytes (64 bf16 or 32 floats), 128-byte swizzle; elements past the
// matrix read as zero.
bool encode_rows_map(CUtensorMap* m, const void* base, int64_t rows, int d, int box_rows,
                     int dtype);

}  // namespace oprag
