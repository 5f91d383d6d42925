// Which elements of the 32 x 32 diagonal block at n0 the state reduction's back substitution reads (k_discrete.cu).
// Compiles for the host too.
#pragma once
#include <cuda_runtime.h>

namespace heat {

// Row n0 + i, column n0 + lane of an nb x nb rate matrix: above the diagonal, inside the matrix (the last block of a
// bin count that is no multiple of 32 passes its end), at or above the column's lowest row with a rate.
__host__ __device__ __forceinline__ bool gth_tile_in(int i, int lane, int n0, int nb, int low) {
    return n0 + lane < nb && i < lane && n0 + i >= low;
}

}  // namespace heat
