// Index arithmetic of the tensor-core passes, for host and device code.
#pragma once

#include <cstddef>

#ifdef __CUDACC__
#define SEM3D_HD __host__ __device__ __forceinline__
#else
#define SEM3D_HD inline
#endif

namespace sem3d {

// Offset of row `row` of a y pass (pass 1: row = x index, one batch per z) or
// z pass (pass 2: row = x index + Px * y index, one batch) at column 0, in an
// array of pitch Px.  Planes have fewer than 2^31 entries, a whole array may
// have more than 2^32: nx = 1602 has pitch 1616 in node order and 1632 in
// parity order, so 1602 x 1626 x 1626 crosses 2^32 in the second only.
SEM3D_HD size_t tc_row_offset(int pass, int row, int batch, int Px, int ny) {
  return (size_t)row + (pass == 1 ? (size_t)Px * (size_t)ny * (size_t)batch : 0);
}

}  // namespace sem3d
