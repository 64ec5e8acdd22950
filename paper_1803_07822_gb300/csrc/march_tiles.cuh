// Tiles of the kernels that march along axis 2 with one plane in shared memory
// (lattice gradient, the adjoint's gather).
#pragma once

#include <cuda_runtime.h>

namespace cslbm {

// Tiles of the marching kernels: TX x TY columns, one thread each, by a chunk
// of planes; the block index counts tiles along axis 0, then 1, then chunks.
constexpr int TX = 32, TY = 8;
struct Tiles {
    int nx, ny, chunk, first, last;  // planes first .. last - 1 in chunks of `chunk`
};
__device__ __forceinline__ void tile_of(const Tiles& T, int lo0, int lo1, int& x0, int& y0, int& za, int& zb)
{
    const int b = blockIdx.x, bx = b % T.nx, r = b / T.nx, by = r % T.ny, bz = r / T.ny;
    x0 = lo0 + bx * TX;
    y0 = lo1 + by * TY;
    za = T.first + bz * T.chunk;
    zb = min(T.last, za + T.chunk);
}

// Chunks of at most 32 planes (a march repeats two planes of its neighbours'),
// shorter ones while there are fewer than eight blocks per SM
inline Tiles tiles_of(int n_sm, int e0, int e1, int first, int last, int ncomp)
{
    Tiles T;
    T.nx = (e0 + TX - 1) / TX;
    T.ny = (e1 + TY - 1) / TY;
    T.first = first;
    T.last = last;
    T.chunk = 32;
    while (T.chunk > 4 && (long long)T.nx * T.ny * ncomp * ((last - first + T.chunk - 1) / T.chunk) < 8LL * n_sm)
        T.chunk /= 2;
    return T;
}
inline dim3 tile_grid(const Tiles& T, int ncomp)
{
    return dim3((unsigned)T.nx * T.ny * ((T.last - T.first + T.chunk - 1) / T.chunk), (unsigned)ncomp);
}

}  // namespace cslbm
