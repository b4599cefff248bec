// Row products shared by the kernels that keep whole input rows in registers (simt_row.cu,
// lift_row.cu): rows packed in pairs along the contracted index against operator rows in shared
// memory, every lane reading the same 16 bytes.
#pragma once

#include "tma.cuh"

namespace lc {

__host__ __device__ inline int row_np(int N) { return (N + 3) & ~3; }

// D^T operands of columns c0 .. c0 + 3 against the rows in ur: r[x][m] = out value of element x
template <int NP, int EPT, int LD = NP>  // LD: floats from one operator row to the next
__device__ __forceinline__ void row_columns(const float *Ds, const uint64_t (&ur)[EPT][NP / 2], float (&r)[EPT][4])
{
    uint64_t acc[EPT][4];
#pragma unroll
    for (int x = 0; x < EPT; ++x)
#pragma unroll
        for (int m = 0; m < 4; ++m)
            acc[x][m] = 0;
#pragma unroll
    for (int q = 0; q < NP / 4; ++q) {
        ulonglong2 d[4];
#pragma unroll
        for (int m = 0; m < 4; ++m)
            d[m] = *reinterpret_cast<const ulonglong2 *>(Ds + m * LD + 4 * q);
#pragma unroll
        for (int m = 0; m < 4; ++m)
#pragma unroll
            for (int x = 0; x < EPT; ++x)
                acc[x][m] = fma_f32x2(ur[x][2 * q], d[m].x, acc[x][m]);
#pragma unroll
        for (int m = 0; m < 4; ++m)
#pragma unroll
            for (int x = 0; x < EPT; ++x)
                acc[x][m] = fma_f32x2(ur[x][2 * q + 1], d[m].y, acc[x][m]);
    }
#pragma unroll
    for (int x = 0; x < EPT; ++x)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const float2 v = unpack_f32x2(acc[x][m]);
            r[x][m] = v.x + v.y;
        }
}

}  // namespace lc
