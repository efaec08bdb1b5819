// The exchange sum over one unit of work: 32 consecutive pairs (a, d) of a
// transfer Q (one per lane) against all its pairs (b, c),
//   sum_{(b,c)} P_ab P_cd,  P_ab = delta_ab - G[b][a], P_cd = delta_cd - G[d][c].
#pragma once
#include "complex_math.cuh"

namespace ftq {

// Lane sum of the products G[b][a] G[d][c] for the pairs [first, end) of the transfer and
// this lane's pair (al, dl).  G^T is read beside G so that the 32 lanes of a load touch
// neighbouring columns of one row; four partial sums keep eight loads in flight per lane.
template <typename T>
__device__ __forceinline__ T exchange_products(const T* __restrict__ Gw, const T* __restrict__ Gt, int M,
                                               const int* __restrict__ pa, const int* __restrict__ pb, int first,
                                               int end, int al, int dl) {
    const T* gcol = Gw + al;                   // G[b][al] = gcol[b * M]
    const T* tcol = Gt + dl;                   // G[dl][c] = G^T[c][dl] = tcol[c * M]
    T acc[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u].x = acc[u].y = 0;
    int g = first;
#pragma unroll 1
    for (; g + 3 < end; g += 4) {
        T x[4], y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {          // indices are the same for every lane
            x[u] = gcol[pa[g + u] * M];
            y[u] = tcol[pb[g + u] * M];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u] = cfma(x[u], y[u], acc[u]);
    }
    for (; g < end; ++g) acc[0] = cfma(gcol[pa[g] * M], tcol[pb[g] * M], acc[0]);
    return (acc[0] + acc[1]) + (acc[2] + acc[3]);
}

// The same with the deltas.  Since a - d = b - c they meet only at (b, c) = (a, d), and both
// do: 1 - G[a][a] - G[d][d] is added once.
template <typename T>
__device__ __forceinline__ T exchange_unit(const T* __restrict__ Gw, const T* __restrict__ Gt, int M,
                                           const int* __restrict__ pa, const int* __restrict__ pb, int first, int end,
                                           int al, int dl) {
    T r = exchange_products<T>(Gw, Gt, M, pa, pb, first, end, al, dl);
    const T ga = Gw[al * M + al], gd = Gw[dl * M + dl];
    r.x += 1 - ga.x - gd.x;
    r.y -= ga.y + gd.y;
    return r;
}

}  // namespace ftq
