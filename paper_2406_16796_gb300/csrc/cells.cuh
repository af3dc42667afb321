// cells.cuh -- a cell and its neighbours for the one-thread-per-cell kernels: linear
// indexes that already hold the periodic wrap, and whether a neighbour exists (beyond a
// non-periodic side E and B are zero and the axion follows its boundary condition).
// Sizes are 32-bit (grids below 2^30 cells).
#pragma once

#include "axp_internal.h"

namespace axp {

struct Cell {
    int c, x[3];
    int up[3], dn[3];
    bool hu[3], hd[3];
};

// Cell c of an n0 x n1 x n2 grid; MASK: the active axes (an axis left out has one cell).
template <int MASK>
__device__ __forceinline__ void cell_of_index(const int n[3], const int per[3], unsigned c, Cell &q)
{
    const unsigned n0 = n[0], n1 = n[1];
    const unsigned r = c / n0;
    q.c = (int)c;
    q.x[0] = (int)(c - r * n0);
    q.x[1] = (MASK & 4) ? (int)(r % n1) : (int)r;
    q.x[2] = (MASK & 4) ? (int)(r / n1) : 0;
    const int stride[3] = {1, n[0], n[0] * n[1]};
#pragma unroll
    for (int a = 0; a < 3; a++) {
        q.up[a] = q.dn[a] = q.c;
        q.hu[a] = q.hd[a] = true;
        if (!(MASK >> a & 1)) continue;
        const int wrap = (n[a] - 1) * stride[a];
        if (q.x[a] + 1 < n[a]) q.up[a] = q.c + stride[a];
        else { q.up[a] = q.c - wrap; q.hu[a] = per[a]; }
        if (q.x[a] > 0) q.dn[a] = q.c - stride[a];
        else { q.dn[a] = q.c + wrap; q.hd[a] = per[a]; }
    }
}

template <typename T>
__device__ __forceinline__ T ldz(const T *__restrict__ F, int c, bool ok)
{
    return ok ? F[c] : T(0);
}

// index of a cell in the ghost plane of axis a
__device__ __forceinline__ int ghost_index(const int n[3], int a, const Cell &q)
{
    return a == 0 ? q.x[1] + n[1] * q.x[2] : (a == 1 ? q.x[0] + n[0] * q.x[2] : q.x[0] + n[0] * q.x[1]);
}

}  // namespace axp
