// One Householder reflector of the complex128 factorisations applied to the
// columns of a matrix by a whole block.
#pragma once
#include "complex_math.cuh"

namespace ftq {

// Columns [c0, c1) of B (rows j .. rows - 1, leading dimension ldb) take
// H = I - tau u u^H, u = (u0, A[j + 1 ..][j]) (leading dimension lda).  Two lanes
// share a column, every other row each: the loops over rows are chains of loads and
// FP64 operations whose latency one lane per column left exposed (QRCP at M = 257, 152
// walkers 60.3 -> 41.7 ms, truncated QRCP with 32 walkers 35.8 -> 25.5 ms).  NORMS: cn[c] receives
// the squared norm of the rows below j.
template <bool NORMS>
__device__ __forceinline__ void reflect_columns(const double2* A, int lda, int j, double2* B, int ldb, int rows, int c0,
                                                int c1, double2 u0, double tau, double* cn) {
    const int half = threadIdx.x & 1, per = blockDim.x >> 1;
    for (int cb = c0; cb < c1; cb += per) {                  // the same trips for every lane
        const int c = cb + (int)(threadIdx.x >> 1);
        const bool on = c < c1;
        double2 s = make_double2(0.0, 0.0);
        if (on) {
            if (half == 0) s = cmul(conj(u0), B[(long)j * ldb + c]);
#pragma unroll 4
            for (int r = j + 1 + half; r < rows; r += 2) s = cfma(conj(A[(long)r * lda + j]), B[(long)r * ldb + c], s);
        }
        s.x += __shfl_xor_sync(0xffffffffu, s.x, 1);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, 1);
        s = s * tau;
        double left = 0.0;
        if (on) {
            if (half == 0) B[(long)j * ldb + c] = cfms(u0, s, B[(long)j * ldb + c]);
#pragma unroll 4
            for (int r = j + 1 + half; r < rows; r += 2) {
                const double2 v = cfms(A[(long)r * lda + j], s, B[(long)r * ldb + c]);
                B[(long)r * ldb + c] = v;
                if (NORMS) left += abs2(v);
            }
        }
        if (NORMS) {
            left += __shfl_xor_sync(0xffffffffu, left, 1);
            if (on && half == 0) cn[c] = left;
        }
    }
}

}  // namespace ftq
