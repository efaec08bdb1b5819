// Green's function by a right-looking blocked LU whose updates run on the
// 5th-generation tensor cores, in complex128 and in FP32 (the mixed path).
//
// The algebra is that of k_green: Mt = D_Lb T^-1 D_Rb + D_Ls Y D_Rs, B = Y D_Rs,
// G = I - B Mt^-1 D_Ls, ln det from the pivots.  Here Z = (B Mt^-1)^T comes from
// Mt^T Z = B^T: S = [Mt^T | B^T] (row-major, either part padded to a multiple of
// four columns that nothing reads) is eliminated in panels of NB columns,
// right-hand sides included, and substituted back:
//   k_lu_panel   one block per walker, one row of the panel per thread, held in
//                registers: pivot search by warp reductions, rank-1 updates from
//                a broadcast pivot row, no row is moved until the panel is done.
//   k_lu_tri     one column per thread: the panel's row permutation and the
//                NB x NB triangle (L11 forward, U11 backward) in registers.
//   k_lu_update  C <- C - A B with K = NB on the tensor cores: FP32 operands as
//                three bf16 terms (24 bits, the six products of level i + j <= 2,
//                levels summed apart), complex128 operands as eight base-128 digits
//                under one power of two per row of A and per column of B (see
//                chain_oz.cu; the level sums over 2 NB terms stay below 2^22).
//                FP32 digits with exact sums gave the same errors of G and ln det to
//                two figures and took 1.6 times as long (only behind a stabilisation at M = 515
//                does the truncation of the level sums show: ln det 7e-6 off, 4e-6 with FP64 sums).
// Everything but the panel is spread over (walker, tile) items, so that few
// walkers fill the chip as well as many, and no walker's serial chain of panels
// holds an SM.
#include <algorithm>
#include <cmath>

#include "complex_math.cuh"
#include "df_math.cuh"
#include "digits.cuh"
#include "ftq_internal.h"
#include "green_tail.cuh"
#include "mixed_common.cuh"
#include "tc_common.cuh"

namespace ftq {
namespace {

using namespace tc;

template <typename T> struct Cplx;
template <> struct Cplx<float> { using type = float2; };
template <> struct Cplx<double> { using type = double2; };
template <typename T> using cx = typename Cplx<T>::type;

template <typename T> __device__ __forceinline__ cx<T> mk(T x, T y);
template <> __device__ __forceinline__ float2 mk<float>(float x, float y) { return make_float2(x, y); }
template <> __device__ __forceinline__ double2 mk<double>(double x, double y) { return make_double2(x, y); }

__device__ __forceinline__ float2 cfms(float2 a, float2 b, float2 c) {      // c - a b
    return make_float2(fmaf(-a.x, b.x, fmaf(a.y, b.y, c.x)), fmaf(-a.x, b.y, fmaf(-a.y, b.x, c.y)));
}

// ---------------------------------------------------------------- scales
// Per walker: the factors of both sides split at one, the sum of the logs of
// those split off, and the pivot parity cleared.
template <typename T>
__global__ void __launch_bounds__(256) k_lu_scales(const double2* __restrict__ DR, const double* __restrict__ eps,
                                                  LuScales<T> sc, int M, double lscale, double mu_T) {
    __shared__ double sh[8];
    const int w = blockIdx.x;
    double lsum = 0.0;
    for (int i = threadIdx.x; i < M; i += 256) {
        const double dl = exp(-lscale * (eps[i] - mu_T));
        double b = 1.0, s = dl;
        if (dl > 1.0) { b = 1.0 / dl; s = 1.0; }
        const double2 d = DR[(size_t)w * M + i];
        const double a = sqrt(abs2(d));
        double rb = 1.0;
        double2 rs = d;
        if (a > 1.0) { rb = 1.0 / a; rs = d * (1.0 / a); }
        const size_t o = (size_t)w * M + i;
        sc.dlb[o] = (T)b;
        sc.dls[o] = (T)s;
        sc.drb[o] = (T)rb;
        sc.drs[o] = mk<T>((T)rs.x, (T)rs.y);
        lsum += log(b) + log(rb);
    }
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_down_sync(0xffffffffu, lsum, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = lsum;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < 8; ++i) lsum += sh[i];
        sc.lsum[w] = lsum;
        sc.swaps[w] = 0;
    }
}

// ---------------------------------------------------------------- S = [Mt^T | B^T]
// One block per walker and 32 x 32 tile: S[r][c] = Mt[c][r], S[r][ld / 2 + c] = B[c][r].
__global__ void __launch_bounds__(256) k_lu_form64(const double2* __restrict__ Y, const double2* __restrict__ Tinv,
                                                  double2* __restrict__ S, LuScales<double> sc, int M, int ld) {
    __shared__ double2 tm[32][33], tb[32][33];
    const int w = blockIdx.z, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
    const size_t off = (size_t)w * M * M, so = (size_t)w * M;
    for (int q = wid; q < 32; q += 8) {
        const int c = c0 + q, r = r0 + lane;
        if (c < M && r < M) {
            const size_t e = off + (size_t)c * M + r;
            const double2 b = cmul(Y[e], sc.drs[so + r]);
            tb[q][lane] = b;
            tm[q][lane] = Tinv[e] * (sc.dlb[so + c] * sc.drb[so + r]) + b * sc.dls[so + c];
        }
    }
    __syncthreads();
    for (int q = wid; q < 32; q += 8) {
        const int r = r0 + q, c = c0 + lane;
        if (r < M && c < M) {
            double2* row = S + ((size_t)w * M + r) * ld;
            row[c] = tm[lane][q];
            row[ld / 2 + c] = tb[lane][q];
        }
    }
}

// t s for FP64 t and s = b r in FP32 pairs (48 bits), rounded to FP32 once: the number that
// an FP64 product rounds to, but for rounding ties (none of 4 million products above 1e-33
// differs; below, the pairs' low words run out of exponents).  It is integer and FP32
// work only: with three FP64 multiplications and four conversions per entry the kernel ran at
// the FP64 pipe's rate (1.09 ms at M = 257, 1024 walkers).
__device__ __forceinline__ float scaled(double t, float sh, float sl) {
    const df2 v = df_split_int(t);
    return fmaf(v.h, sh, fmaf(v.h, sl, v.l * sh));
}

// The same from the FP32 planes, whose columns are contiguous along c here.
__global__ void __launch_bounds__(256) k_lu_form32(const float* __restrict__ Ypl, const double2* __restrict__ Tinv,
                                                  float2* __restrict__ S, LuScales<float> sc, Planes P,
                                                  size_t wstride, int M, int ld) {
    __shared__ float2 tm[32][33];
    const int w = blockIdx.z, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
    const size_t off = (size_t)w * M * M, so = (size_t)w * M;
    float2 y[4];
    double2 t[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {                    // every load of the thread in flight at once
        const int c = c0 + wid + 8 * u, r = r0 + lane;
        if (c < M && r < M) t[u] = Tinv[off + (size_t)c * M + r];
        const int r2 = r0 + wid + 8 * u, c2 = c0 + lane;
        if (r2 < M && c2 < M) y[u] = P.load(Ypl + wstride * w, c2, r2);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int q = wid + 8 * u, c = c0 + q, r = r0 + lane;
        if (c < M && r < M) {
            const float bl = sc.dlb[so + c], br = sc.drb[so + r];
            const float sh = bl * br, sl = fmaf(bl, br, -sh);
            tm[q][lane] = make_float2(scaled(t[u].x, sh, sl), scaled(t[u].y, sh, sl));
        }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int q = wid + 8 * u, r = r0 + q, c = c0 + lane;
        if (r < M && c < M) {
            const float2 b = cmul(y[u], sc.drs[so + r]);
            float2* row = S + ((size_t)w * M + r) * ld;
            row[c] = tm[lane][q] + b * sc.dls[so + c];
            row[ld / 2 + c] = b;
        }
    }
}

// ---------------------------------------------------------------- panel
// Factorises rows [jb, M) of columns [jb, jb + nb).  Thread t holds row jb + t.
// The pivot is the row of largest |Re| + |Im| among those left (compared by its
// leading word: 20 bits of mantissa in FP64, all of it in FP32; ties to the
// lower thread).  A row's position is only bookkeeping until the end: the
// permutation is written out for k_lu_tri, which moves the other columns.
__device__ __forceinline__ unsigned pivot_key(float2 v) { return __float_as_uint(fabsf(v.x) + fabsf(v.y)); }
__device__ __forceinline__ unsigned pivot_key(double2 v) { return (unsigned)__double2hiint(fabs(v.x) + fabs(v.y)); }

template <typename T, int NB, int MAXT>
__global__ void __launch_bounds__(MAXT) k_lu_panel(cx<T>* __restrict__ S, LuScales<T> sc, int* __restrict__ status,
                                                   int M, int ld, int jb, int nb) {
    __shared__ unsigned wkey[2][32];
    __shared__ int wthr[2][32], oldpos[2];
    __shared__ cx<T> prow[2][NB];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const int w = blockIdx.x, m = M - jb;
    cx<T>* Sw = S + (size_t)w * M * ld;
    cx<T> a[NB];
    const bool valid = tid < m;
#pragma unroll
    for (int c = 0; c < NB; ++c) a[c] = valid && c < nb ? Sw[(size_t)(jb + tid) * ld + jb + c] : mk<T>(0, 0);
    int pos = tid, flips = 0;
    bool done = !valid;
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        if (j < nb) {
            const int b = j & 1;
            const unsigned key = done ? 0u : pivot_key(a[j]) + 1u;
            const unsigned top = __reduce_max_sync(0xffffffffu, key);
            const unsigned at = __ballot_sync(0xffffffffu, key == top);
            if (lane == 0) {
                wkey[b][warp] = top;
                wthr[b][warp] = warp * 32 + __ffs(at) - 1;
            }
            __syncthreads();
            const unsigned k2 = lane < nw ? wkey[b][lane] : 0u;
            const unsigned top2 = __reduce_max_sync(0xffffffffu, k2);
            const int win = wthr[b][__ffs(__ballot_sync(0xffffffffu, lane < nw && k2 == top2)) - 1];
            if (tid == win) {
#pragma unroll
                for (int c = j; c < NB; ++c) prow[b][c] = a[c];
                oldpos[b] = pos;
            }
            __syncthreads();
            const int op = oldpos[b];
            const cx<T> pv = prow[b][j];
            const T n2 = pv.x * pv.x + pv.y * pv.y;
            const cx<T> ip = mk<T>(pv.x / n2, -pv.y / n2);
            if (tid == win) {
                pos = j;
                done = true;
            } else if (valid && pos == j) {
                pos = op;
            }
            if (tid == 0) {
                flips ^= op != j ? 1 : 0;
                sc.inv[(size_t)w * M + jb + j] = ip;
                if (!(n2 > (T)0)) atomicOr(status, 1);
            }
            if (!done) {
                const cx<T> l = cmul(a[j], ip);
                a[j] = l;
#pragma unroll
                for (int c = j + 1; c < NB; ++c) a[c] = cfms(l, prow[b][c], a[c]);
            }
        }
    }
    if (valid) {
#pragma unroll
        for (int c = 0; c < NB; ++c)
            if (c < nb) Sw[(size_t)(jb + pos) * ld + jb + c] = a[c];
        int* src = sc.perm + (size_t)w * 2 * LU_NB_MAX;
        if (pos < nb) src[pos] = tid;                       // row that ends at position pos of the block
        if (tid < nb) src[LU_NB_MAX + tid] = pos >= nb ? pos : -1;   // where the block's row tid went
    }
    if (tid == 0) sc.swaps[w] ^= flips;
}

// ---------------------------------------------------------------- triangles
// t - sum of d[k] x[k] over k0 <= k < k1 (constants after unrolling).  FP32 products go to
// four sums that meet t last: as one chain, up to 62 roundings at the size of t made these
// triangles the largest error of the FP32 G (rms, on the same chain: M = 57 9.9e-9, now
// 4.9e-9, M = 123 5.2e-9, now 2.0e-9; the CUDA-core LU 6.5e-9 and 4.6e-9) for 0.3% of the time of a
// block of slices.  In FP64 the longer code took 2.5% and changed no error.
template <typename T, int NB>
__device__ __forceinline__ cx<T> less_products(cx<T> t, const cx<T> (&d)[NB], const cx<T> (&x)[NB], int k0, int k1) {
    constexpr int NS = sizeof(T) == 4 ? 4 : 1;
    cx<T> s[NS];
    if constexpr (NS == 1) s[0] = t;
#pragma unroll
    for (int k = 0; k < NB; ++k)
        if (k >= k0 && k < k1) s[k % NS] = cfms(d[k], x[k], NS > 1 && k < k0 + NS ? mk<T>(0, 0) : s[k % NS]);
    if constexpr (NS == 1) return s[0];
    const int n = k1 - k0;
    if (n >= 4) return t + ((s[0] + s[1 % NS]) + (s[2 % NS] + s[3 % NS]));
    cx<T> r = mk<T>(0, 0);
#pragma unroll
    for (int k = 0; k < 3; ++k)
        if (k < n) r = r + s[(k0 + k) % NS];
    return n > 0 ? t + r : t;
}

// One column of S per thread.  Forward: the panel's permutation on its rows,
// then X <- L11^-1 X.  Backward: X <- U11^-1 X.
template <typename T, int NB, bool UPPER, bool PERM = !UPPER>
__global__ void __launch_bounds__(128) k_lu_tri(cx<T>* __restrict__ S, LuScales<T> sc, int M, int ld, int jb, int nb,
                                               int cbeg, int cend) {
    __shared__ cx<T> D[NB][NB];
    __shared__ cx<T> inv[NB];
    __shared__ int src[NB], dst[NB];
    const int w = blockIdx.y, tid = threadIdx.x;
    cx<T>* Sw = S + (size_t)w * M * ld;
    const int nt = blockDim.x;
    for (int e = tid; e < NB * NB; e += nt) {
        const int r = e / NB, c = e % NB;
        D[r][c] = r < nb && c < nb ? Sw[(size_t)(jb + r) * ld + jb + c] : mk<T>(0, 0);
    }
    for (int q = tid; q < NB; q += nt) {
        if (UPPER) inv[q] = q < nb ? sc.inv[(size_t)w * M + jb + q] : mk<T>(0, 0);
        if (!PERM) continue;
        src[q] = q < nb ? sc.perm[(size_t)w * 2 * LU_NB_MAX + q] : 0;
        dst[q] = q < nb ? sc.perm[(size_t)w * 2 * LU_NB_MAX + LU_NB_MAX + q] : -1;
    }
    __syncthreads();
    const int c = cbeg + blockIdx.x * nt + tid;
    if (c >= cend) return;
    cx<T>* col = Sw + (size_t)jb * ld + c;
    cx<T> x[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) x[q] = q < nb ? col[(size_t)(PERM ? src[q] : q) * ld] : mk<T>(0, 0);
    if constexpr (!UPPER) {
        for (int q = 0; PERM && q < nb; ++q)
            if (dst[q] >= 0) col[(size_t)dst[q] * ld] = col[(size_t)q * ld];
#pragma unroll
        for (int q = 1; q < NB; ++q) {
            x[q] = less_products<T, NB>(x[q], D[q], x, 0, q);
        }
    } else {
#pragma unroll
        for (int q = NB - 1; q >= 0; --q) {
            x[q] = cmul(less_products<T, NB>(x[q], D[q], x, q + 1, NB), inv[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < NB; ++q)
        if (q < nb) col[(size_t)q * ld] = x[q];
}

// The forward triangle of the T^-1 update (unit lower, no permutation) with the
// arithmetic of the mixed path's stabilisation: double-FP32 (48 bits) on the FP32
// pipe, whose rate is 64 times that of the FP64 pipe.  One column per thread, kept in
// shared memory ([32][threads] of Re hi, Re lo, Im hi, Im lo), so that the loops stay
// rolled: 48 instructions per complex term would not fit the instruction cache.
__global__ void __launch_bounds__(128) k_tinv_tri_df(double2* __restrict__ S, int M, int ld, int jb, int nb, int cbeg,
                                                    int cend) {
    extern __shared__ unsigned char smem_raw[];
    float4* D = reinterpret_cast<float4*>(smem_raw);         // [32][32]
    float4* X = D + 32 * 32;                                 // [32][threads]
    const int w = blockIdx.y, tid = threadIdx.x, nt = blockDim.x;
    double2* Sw = S + (size_t)w * M * ld;
    for (int e = tid; e < 32 * 32; e += nt) {
        const int r = e >> 5, c = e & 31;
        if (r < nb && c < r) {
            const double2 v = Sw[(size_t)(jb + r) * ld + jb + c];
            const df2 re = df_split_int(v.x), im = df_split_int(v.y);
            D[e] = make_float4(re.h, re.l, im.h, im.l);
        }
    }
    __syncthreads();
    const int c = cbeg + blockIdx.x * nt + tid;
    if (c >= cend) return;
    double2* col = Sw + (size_t)jb * ld + c;
    float4* x = X + tid;
    for (int q = 0; q < nb; ++q) {
        const double2 v = col[(size_t)q * ld];
        df2 re = df_split_int(v.x), im = df_split_int(v.y);
#pragma unroll 4
        for (int k = 0; k < q; ++k) {
            const float4 u = D[q * 32 + k], y = x[k * nt];
            df_msub(re, y.x, y.y, u.x, u.y);                 // s -= x u
            df_madd(re, y.z, y.w, u.z, u.w);
            df_msub(im, y.x, y.y, u.z, u.w);
            df_msub(im, y.z, y.w, u.x, u.y);
        }
        re = df_norm(re);
        im = df_norm(im);
        x[q * nt] = make_float4(re.h, re.l, im.h, im.l);
        col[(size_t)q * ld] = make_double2((double)re.h + (double)re.l, (double)im.h + (double)im.l);
    }
}

// ---------------------------------------------------------------- updates
// C[r0.., c0..) -= S[r, jb .. jb + nb) S[jb .. jb + nb, c] on the tensor cores.
// Work item = (walker, 64 rows, OCT columns); warps 0..7 epilogue (two groups, C
// tiles come and go by TMA: per-thread copies took 60% of an item's time), 8..15
// operand A, 16..19 operand B, 20 control.  Complex as real:
// MMA rows 2 i = Re, 2 i + 1 = Im of row i (so that a warp's lanes hold whole complex
// numbers of 16 rows and meet no bank conflicts in the C tile) and k tiles
// [Re (16) | Im (16)], as in chain_oz.cu.  Stores of operand digits alternate
// between the two rows (A) and the two 8-byte halves (B) over the lanes for the
// same reason.  What bounds the FP32 items is shared-memory wavefronts (63% of the
// pipe; tensor pipe 17%, DRAM 44%, at M = 257, 304 walkers), the complex128 ones the FP64 pipe
// and the integer ALU of the epilogue (49% each).
template <typename T> struct UpCfg;
template <> struct UpCfg<double> { static constexpr int ND = 8, OCT = 32, NST = 2; };
template <> struct UpCfg<float> { static constexpr int ND = 3, OCT = 64, NST = 4; };

constexpr int W_EPI = 8, W_A = 8, W_B = 4;
constexpr int NT_UP = 32 * (W_EPI + W_A + W_B + 1);
constexpr int KT_MAX = 2;                          // k tiles of 16 complex k (NB <= 32)
constexpr int UADIG = 128 * 64;

constexpr int CROW = 512;                          // bytes of a C tile's row (OCT complex numbers)
constexpr int CBOX = 16;                           // rows of one TMA box: tiles end at multiples of NB or at M

template <typename T>
constexpr size_t up_smem() {
    using C = UpCfg<T>;
    return 1024 + (size_t)C::NST * C::ND * (UADIG + C::OCT * 64) + 2 * (size_t)64 * CROW;
}

// The ND digit words of four complex numbers' parts: out[digit] = 4 bf16.
__device__ __forceinline__ void digit_words(const double (&v)[4], int E, uint2 (&out)[8]) {
    float d[4][8];
#pragma unroll
    for (int q = 0; q < 4; ++q) digits8(fixed_point(v[q], E, 4), d[q]);
#pragma unroll
    for (int j = 0; j < 8; ++j) out[j] = make_uint2(pack_hi(d[0][j], d[1][j]), pack_hi(d[2][j], d[3][j]));
}
__device__ __forceinline__ uint32_t bf2(float x, float y) {           // bf16(y) : bf16(x)
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(y), "f"(x));
    return r;
}

// Two FP32 numbers as three bf16 pairs, v = d0 + d1 + d2 to 24 bits.
__device__ __forceinline__ void split3(float x, float y, uint32_t (&d)[3]) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        d[j] = bf2(x, y);
        x -= __uint_as_float(d[j] << 16);
        y -= __uint_as_float(d[j] & 0xffff0000u);
    }
}
__device__ __forceinline__ void digit_words(const float (&v)[4], int, uint2 (&out)[3]) {
    uint32_t a[3], b[3];
    split3(v[0], v[1], a);
    split3(v[2], v[3], b);
#pragma unroll
    for (int j = 0; j < 3; ++j) out[j] = make_uint2(a[j], b[j]);
}

template <typename T>
struct UpArgs {
    cx<T>* S;
    int* status;
    int M, ld, jb, nb, r0, r1, c0, c1, nrb, nct, W;
    long long wait_limit;
};

__device__ __forceinline__ uint32_t hi_abs(double v) { return (uint32_t)__double2hiint(v) & 0x7fffffffu; }
__device__ __forceinline__ uint32_t hi_abs(float) { return 0u; }       // FP32 terms carry their exponents

template <typename T>
__global__ void __launch_bounds__(NT_UP, 1) k_lu_update(const UpArgs<T> p, const __grid_constant__ CUtensorMap map) {
    using C = UpCfg<T>;
    using V = cx<T>;
    constexpr int ND = C::ND, OCT = C::OCT, NST = C::NST;
    constexpr int BDIG = OCT * 64, STAGE = ND * (UADIG + BDIG);
    constexpr bool F64 = sizeof(T) == 8;
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint64_t full[NST], mma_bar[NST], tfull[2], tempty[2], einfo[2], cfull[2];
    __shared__ uint32_t tmem_sh;
    __shared__ volatile int abort_sh;
    __shared__ unsigned short row_e[2][64], col_p[2][W_B][32];    // complex128: exponents of rows, parts of the columns'
    __shared__ __align__(16) unsigned short col_e[2][OCT];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t pad = (1024u - (smem_u32(smem_raw) & 1023u)) & 1023u;
    unsigned char* base = smem_raw + pad;
    unsigned char* ctile = base + (size_t)NST * STAGE;                  // [2][64] rows of CROW bytes
    if (tid == 0) {
        for (int b = 0; b < NST; ++b) {
            mbar_init(&full[b], W_A + W_B);
            mbar_init(&mma_bar[b], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], W_EPI / 2);
            mbar_init(&einfo[b], W_A + W_B);
            mbar_init(&cfull[b], 1);
        }
        abort_sh = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(&tmem_sh, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_sh;
    const int per_walker = p.nrb * p.nct;
    const int nitems = p.W * per_walker;
    const int per = (nitems + (int)gridDim.x - 1) / (int)gridDim.x;
    const int it0 = (int)blockIdx.x * per, it1 = min(nitems, it0 + per);     // this CTA's items
    const int KT = (p.nb + 15) / 16;
    auto wait = [&](uint64_t* bar, uint32_t parity) {
        return mbar_wait_ab(bar, parity, &abort_sh, p.status, p.wait_limit);
    };

    if (warp == W_EPI + W_A + W_B) {
        // ------------------------------------------------ control
        if (lane == 0) {
            int g = 0, last = -1;
            bool ok = true;
            for (int it = it0, li = 0; it < it1 && ok; ++it, ++li) {
                const int bi = li & 1;
                const uint32_t acc = tmem + (uint32_t)(bi * ND * OCT);
                if (li >= 2) ok = wait(&tempty[bi], (uint32_t)(((li - 2) >> 1) & 1));
                for (int kt = 0; kt < KT && ok; ++kt, ++g) {
                    const int s = g % NST;
                    ok = wait(&full[s], (uint32_t)((g / NST) & 1));
                    if (!ok) break;
                    tc_fence_after();
                    unsigned char* st = base + s * STAGE;
                    const uint64_t b0 = sdesc_sw64(st + ND * UADIG);
#pragma unroll
                    for (int k = 0; k < 2; ++k)
#pragma unroll
                        for (int i = 0; i < ND; ++i)
                            mma_f16(acc + (uint32_t)(i * OCT), sdesc_sw64(st + i * UADIG) + (uint64_t)(2 * k),
                                    b0 + (uint64_t)(2 * k), idesc_bf16(OCT * (ND - i)),
                                    (kt > 0 || k > 0 || i > 0) ? 1u : 0u);
                    mma_commit(&mma_bar[s]);
                    if (kt + 1 == KT) mma_commit(&tfull[bi]);
                    last = g;
                }
            }
            // the MMAs end before TMEM is freed, whichever warp gave up (the epilogue's last wait covers them else)
            if (last >= 0) mbar_wait(&mma_bar[last % NST], (uint32_t)((last / NST) & 1));
        }
    } else if (warp >= W_EPI + W_A) {
        // ------------------------------------------------ operand B: rows jb.., columns of the tile
        constexpr int NH = OCT / 32;
        const int wb = warp - (W_EPI + W_A), kq = wb ^ ((lane >> 3) & 1);    // group of 4 complex k
        V raw[NH][KT_MAX][4], nxt[F64 ? 1 : NH][KT_MAX][4];
        auto load = [&](int it, auto& v) {
            const int w = it / per_walker, tile = it % per_walker;
            const V* Sw = p.S + ((size_t)w * p.M + p.jb) * p.ld;
#pragma unroll
            for (int h = 0; h < NH; ++h) {
                const int c = p.c0 + (tile % p.nct) * OCT + 32 * h + lane;
#pragma unroll
                for (int kt = 0; kt < KT_MAX; ++kt)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int k = kt * 16 + kq * 4 + q;
                        v[h][kt][q] = k < p.nb && c < p.c1 ? Sw[(size_t)k * p.ld + c] : mk<T>(0, 0);
                    }
            }
        };
        if (it0 < it1) load(it0, raw);
        int g = 0;
        for (int it = it0, li = 0; it < it1; ++it, ++li) {
            int E = 0;
            if constexpr (!F64)            // operands of the next item on their way during this one
                if (it + 1 < it1) load(it + 1, nxt);
            if constexpr (F64) {
                uint32_t m = 0u;
#pragma unroll
                for (int kt = 0; kt < KT_MAX; ++kt)
#pragma unroll
                    for (int q = 0; q < 4; ++q) m = max(m, max(hi_abs(raw[0][kt][q].x), hi_abs(raw[0][kt][q].y)));
                col_p[li & 1][wb][lane] = (unsigned short)(m >> 20);
                asm volatile("bar.sync 2, %0;" ::"n"(32 * W_B) : "memory");
#pragma unroll
                for (int o = 0; o < W_B; ++o) E = max(E, (int)col_p[li & 1][o][lane]);
                // the previous user of this parity's exponents has read them
                if (li >= 2) wait(&tempty[li & 1], (uint32_t)(((li - 2) >> 1) & 1));
                if (wb == 0) col_e[li & 1][lane] = (unsigned short)E;
                __syncwarp();
                if (lane == 0) mbar_arrive(&einfo[li & 1]);
            }
#pragma unroll
            for (int kt = 0; kt < KT_MAX; ++kt) {
                if (kt >= KT) continue;
                const int s = g % NST;
                const bool ok = g < NST || wait(&mma_bar[s], (uint32_t)((g / NST - 1) & 1));
                ++g;
                if (!ok || abort_sh) continue;
                unsigned char* B = base + s * STAGE + ND * UADIG;
#pragma unroll
                for (int h = 0; h < NH; ++h)
#pragma unroll
                    for (int part = 0; part < 2; ++part) {
                        T v[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) v[q] = part ? raw[h][kt][q].y : raw[h][kt][q].x;
                        uint2 d[ND];
                        digit_words(v, E, d);
                        const uint32_t o = sw64_off(32 * h + lane, 2 * part + (kq >> 1)) + (uint32_t)(kq & 1) * 8u;
#pragma unroll
                        for (int j = 0; j < ND; ++j) *reinterpret_cast<uint2*>(B + j * BDIG + o) = d[j];
                    }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&full[s]);
            }
            if constexpr (F64) {
                if (it + 1 < it1) load(it + 1, raw);
            } else {
#pragma unroll
                for (int h = 0; h < NH; ++h)
#pragma unroll
                    for (int e = 0; e < KT_MAX * 4; ++e) raw[h][e >> 2][e & 3] = nxt[h][e >> 2][e & 3];
            }
        }
    } else if (warp >= W_EPI) {
        // ------------------------------------------------ operand A: rows of the tile, columns jb..
        const int gt = tid - 32 * W_EPI;
        const int r = gt >> 2, kq = gt & 3;
        const uint32_t h8 = (uint32_t)(kq & 1) * 8u;
        // row 2 r (Re C): [Vr | -Vi], row 2 r + 1 (Im C): [Vi | Vr]; odd rows store in the other order
        const bool odd = r & 1;
        const uint32_t oa = sw64_off(2 * r + (odd ? 1 : 0), kq >> 1) + h8;        // first: re (even) or im (odd)
        const uint32_t ob = sw64_off(2 * r + (odd ? 0 : 1), kq >> 1) + h8;        // then the other
        const uint32_t oc = sw64_off(2 * r + (odd ? 1 : 0), 2 + (kq >> 1)) + h8;  // -im (even) or re (odd)
        const uint32_t od = sw64_off(2 * r + (odd ? 0 : 1), 2 + (kq >> 1)) + h8;
        alignas(16) V raw[KT_MAX][4], nxt[KT_MAX][4];
        auto load = [&](int it, auto& raw) {
            const int w = it / per_walker, tile = it % per_walker;
            const int row = p.r0 + (tile / p.nct) * 64 + r;
            const V* Sr = p.S + ((size_t)w * p.M + (row < p.r1 ? row : p.r0)) * p.ld + p.jb;
            constexpr int PER = 16 / (int)sizeof(V);         // 16-byte loads (a row's columns jb .. stay inside it)
#pragma unroll
            for (int kt = 0; kt < KT_MAX; ++kt)
#pragma unroll
                for (int q = 0; q < 4; q += PER) {
                    const int k = kt * 16 + kq * 4 + q;
                    if (k < p.nb && row < p.r1) {
                        const uint4 x = *reinterpret_cast<const uint4*>(Sr + k);
                        *reinterpret_cast<uint4*>(&raw[kt][q]) = x;
#pragma unroll
                        for (int u = 1; u < PER; ++u)
                            if (k + u >= p.nb) raw[kt][q + u] = mk<T>(0, 0);
                    } else {
#pragma unroll
                        for (int u = 0; u < PER; ++u) raw[kt][q + u] = mk<T>(0, 0);
                    }
                }
        };
        if (it0 < it1) load(it0, raw);
        int g = 0;
        for (int it = it0, li = 0; it < it1; ++it, ++li) {
            int E = 0;
            if constexpr (!F64)            // operands of the next item on their way during this one
                if (it + 1 < it1) load(it + 1, nxt);
            if constexpr (F64) {
                if (li >= 2) wait(&tempty[li & 1], (uint32_t)(((li - 2) >> 1) & 1));
                uint32_t m = 0u;
#pragma unroll
                for (int kt = 0; kt < KT_MAX; ++kt)
#pragma unroll
                    for (int q = 0; q < 4; ++q) m = max(m, max(hi_abs(raw[kt][q].x), hi_abs(raw[kt][q].y)));
                m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
                m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
                E = (int)(m >> 20);
                if (kq == 0) row_e[li & 1][r] = (unsigned short)E;
                __syncwarp();
                if (lane == 0) mbar_arrive(&einfo[li & 1]);
            }
#pragma unroll
            for (int kt = 0; kt < KT_MAX; ++kt) {
                if (kt >= KT) continue;
                const int s = g % NST;
                const bool ok = g < NST || wait(&mma_bar[s], (uint32_t)((g / NST - 1) & 1));
                ++g;
                if (!ok || abort_sh) continue;
                unsigned char* A = base + s * STAGE;
                T v[4];
                uint2 dr[ND], di[ND];
#pragma unroll
                for (int q = 0; q < 4; ++q) v[q] = raw[kt][q].x;
                digit_words(v, E, dr);
#pragma unroll
                for (int q = 0; q < 4; ++q) v[q] = raw[kt][q].y;
                digit_words(v, E, di);
#pragma unroll
                for (int i = 0; i < ND; ++i) {
                    unsigned char* Ai = A + i * UADIG;
                    const uint2 dn = make_uint2(di[i].x ^ 0x80008000u, di[i].y ^ 0x80008000u);
                    *reinterpret_cast<uint2*>(Ai + oa) = odd ? di[i] : dr[i];
                    *reinterpret_cast<uint2*>(Ai + ob) = odd ? dr[i] : di[i];
                    *reinterpret_cast<uint2*>(Ai + oc) = odd ? dr[i] : dn;
                    *reinterpret_cast<uint2*>(Ai + od) = odd ? dn : dr[i];
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&full[s]);
            }
            if constexpr (F64) {
                if (it + 1 < it1) load(it + 1, raw);
            } else {
#pragma unroll
                for (int e = 0; e < KT_MAX * 4; ++e) raw[e >> 2][e & 3] = nxt[e >> 2][e & 3];
            }
        }
    } else {
        // ------------------------------------------------ epilogue
        // Two groups of four warps (one per TMEM lane quadrant) take the items in turn, each
        // with its accumulator and its C buffer, so that one group's waits and copies pass
        // under the other's arithmetic (the FP64 pipe bounds the complex128 items).
        const int grp = warp >> 2, quad = warp & 3;
        const int part = lane & 1, rr = quad * 16 + (lane >> 1);
        // column of a chunk of 8 that this lane handles q-th: rows that share banks differ in it
        auto at = [&](int q) { return (q + rr) & 7; };
        constexpr int XF = (int)sizeof(V) / 4;               // floats per element
        int w, row0, col0, boxes;
        auto tile_at = [&](int it) {
            const int tile = it % per_walker;
            w = it / per_walker;
            row0 = p.r0 + (tile / p.nct) * 64;
            col0 = p.c0 + (tile % p.nct) * OCT;
            boxes = (min(64, p.r1 - row0) + CBOX - 1) / CBOX;
        };
        // one thread of the group moves its C tiles (rows beyond M and columns beyond ld are the map's business)
        const bool mover = quad == 0 && lane == 0;
        unsigned char* cbuf = ctile + (size_t)grp * 64 * CROW;
        auto fetch = [&]() {
            mbar_expect_tx(&cfull[grp], (uint32_t)(boxes * CBOX * CROW));
            for (int q = 0; q < boxes; ++q)
                tma_load_3d(cbuf + (size_t)q * CBOX * CROW, &map, col0 * XF, row0 + q * CBOX, w, &cfull[grp]);
        };
        unsigned char* ct = cbuf + (size_t)rr * CROW + part * sizeof(T);
        const int bi = grp;
        int own = 0;                                         // items of this group so far
        int armed = 0;                                       // loads the mover has put on cfull, one phase each
        // Once a wait has given up, this warp touches no C tile any more: the load in flight is the last one
        // armed, so that cfull never has more than one open phase and the buffer more than one writer.
        bool ok = true;
        for (int it = it0 + grp; it < it1; it += 2, ++own) {
            tile_at(it);
            if (mover && ok) {
                if (own > 0) bulk_wait_read();               // the tile stored before has left the buffer
                fetch();
                ++armed;
            }
            __syncwarp();
            const uint32_t ph = (uint32_t)(own & 1);
            ok = ok && wait(&tfull[bi], ph);
            ok = ok && wait(&cfull[bi], ph);
            if constexpr (F64) ok = ok && wait(&einfo[bi], ph);
            ok = __all_sync(0xffffffffu, ok);
            tc_fence_after();
            if (ok) {
                const uint32_t acc = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(bi * ND * OCT);
                const int er = F64 ? row_e[bi][rr] : 0;
#pragma unroll 1
                for (int cc = 0; cc < OCT; cc += 8) {
                    if (col0 + cc >= p.c1) break;
                    uint32_t v[ND][8];
#pragma unroll
                    for (int l = 0; l < ND; ++l) tmem_ld8(acc + (uint32_t)(l * OCT + cc), v[l]);
                    // all eight reads before the first write: the compiler keeps their order otherwise
                    T cv[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        cv[q] = *reinterpret_cast<const T*>(ct + (cc + at(q)) * (int)sizeof(V));
                    tmem_wait_ld();
#pragma unroll
                    for (int l = 0; l < ND; ++l)     // the values are read after the wait
                        asm volatile("" : "+r"(v[l][0]), "+r"(v[l][1]), "+r"(v[l][2]), "+r"(v[l][3]), "+r"(v[l][4]),
                                     "+r"(v[l][5]), "+r"(v[l][6]), "+r"(v[l][7]));
                    T sum[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        if constexpr (F64) {
                            float lv[8];
#pragma unroll
                            for (int l = 0; l < 8; ++l) lv[l] = __uint_as_float(v[l % ND][q]);
                            sum[q] = level_sum(lv);
                        } else {
                            sum[q] = (__uint_as_float(v[2 % ND][q]) + __uint_as_float(v[1][q])) + __uint_as_float(v[0][q]);
                        }
                    }
#pragma unroll
                    for (int b = 1; b < 8; b <<= 1) {        // rotate by rr: entry q takes column at(q)
                        T s0[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) s0[q] = (rr & b) ? sum[(q + b) & 7] : sum[q];
#pragma unroll
                        for (int q = 0; q < 8; ++q) sum[q] = s0[q];
                    }
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        if constexpr (F64) {
                            // -2^n for factors scaled by 2^(1079 - e): products below about 2^-960, 2^60 above
                            // the smallest normal number, vanish; an overflow or NaN shows
                            const int ec = (int)col_e[bi][cc + at(q)];
                            const int n = er + ec - 2 * 1079 + 49 + 1023;
                            const uint32_t hw = er == 0x7ff || ec == 0x7ff
                                                    ? 0x7ff80000u : (0x80000000u | (uint32_t)max(0, min(n, 0x7ff)) << 20);
                            cv[q] = fma(__hiloint2double((int)hw, 0), sum[q], cv[q]);
                        } else {
                            cv[q] -= sum[q];
                        }
                    }
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        *reinterpret_cast<T*>(ct + (cc + at(q)) * (int)sizeof(V)) = cv[q];
                }
            }
            tc_fence_before();
            fence_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[bi]);
            asm volatile("bar.sync %0, %1;" ::"r"(3 + grp), "n"(16 * W_EPI) : "memory");
            if (mover && ok) {
                for (int q = 0; q < boxes; ++q)
                    tma_store_3d(cbuf + (size_t)q * CBOX * CROW, &map, col0 * XF, row0 + q * CBOX, w);
                bulk_commit();
            }
        }
        if (mover && armed > 0) {
            // after an abort the last tile armed may not have been waited for (every earlier one has): it
            // must land before the block ends
            mbar_wait(&cfull[grp], (uint32_t)((armed - 1) & 1));
            bulk_wait();
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// ---------------------------------------------------------------- G and the weight
// G[i][c] = delta_ic - Z[c][i] dls[c], Z in the right half of S.
template <typename T>
__global__ void __launch_bounds__(256) k_lu_green(const cx<T>* __restrict__ S, cx<T>* __restrict__ G, LuScales<T> sc,
                                                 int M, int ld) {
    __shared__ cx<T> t[32][33];
    const int w = blockIdx.z, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int i0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
    for (int q = wid; q < 32; q += 8) {
        const int c = c0 + q, i = i0 + lane;
        if (c < M && i < M) {
            const cx<T> z = S[((size_t)w * M + c) * ld + ld / 2 + i];
            const T s = -sc.dls[(size_t)w * M + c];
            t[q][lane] = mk<T>(fma(z.x, s, c == i ? (T)1 : (T)0), z.y * s);
        }
    }
    __syncthreads();
    for (int q = wid; q < 32; q += 8) {
        const int i = i0 + q, c = c0 + lane;
        if (i < M && c < M) G[((size_t)w * M + i) * M + c] = t[lane][q];
    }
}

template <typename T>
__global__ void __launch_bounds__(128) k_lu_tail(const cx<T>* __restrict__ S, const cx<T>* __restrict__ G,
                                                LuScales<T> sc, double* __restrict__ ws, int* __restrict__ status,
                                                int M, int ld, double kdt, int constraint, int update,
                                                int with_gauss) {
    __shared__ double2 sh[2][4];
    const int w = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double2 ld_m = make_double2(0.0, 0.0), tr = ld_m;
    for (int j = threadIdx.x; j < M; j += 128) {
        const cx<T> u = S[((size_t)w * M + j) * ld + j];
        const cx<T> g = G[((size_t)w * M + j) * M + j];
        ld_m = ld_m + clog(make_double2(u.x, u.y));
        tr = tr + make_double2(g.x, g.y);
    }
    for (int o = 16; o > 0; o >>= 1) {
        ld_m = ld_m + shfl_down(ld_m, o);
        tr = tr + shfl_down(tr, o);
    }
    if (lane == 0) {
        sh[0][wid] = ld_m;
        sh[1][wid] = tr;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < 4; ++i) {
            ld_m = ld_m + sh[0][i];
            tr = tr + sh[1][i];
        }
        green_weight_tail(ws + (size_t)WSTRIDE * w, ld_m, sc.lsum[w], sc.swaps[w], tr, M, kdt, constraint, status,
                          update, with_gauss);
    }
}

// ---------------------------------------------------------------- T^-1 <- T^-1 Pi U^-1
// X U = Z (Z = T^-1 Pi) transposed: U^T X^T = Z^T, a forward substitution in S = [U^T | Z^T]
// with the tensor-core updates above.
//
// k_tinv_diag: D_R = diag(R) (mixed: diag(R_Y) D'), its reciprocals.
// k_tinv_form: S[j][m] = U_mj = R_mj / D_m for m < j, S[j][rhs + i] = T^-1[i][perm j].
// R: FP32 R_Y with D' (mixed path, R_mj = R_Y[m][j] D'_j), or complex128 with Dp null.
template <typename T>
__global__ void __launch_bounds__(256) k_tinv_diag(const cx<T>* __restrict__ R, const double2* __restrict__ Dp,
                                                  double2* __restrict__ dinv, double2* __restrict__ DR,
                                                  int* __restrict__ status, int M) {
    const size_t w = blockIdx.x;
    for (int j = threadIdx.x; j < M; j += 256) {
        const cx<T> r = R[(w * M + j) * M + j];
        double2 d = make_double2(r.x, r.y);
        if (Dp) d = cmul(d, Dp[w * M + j]);
        DR[w * M + j] = d;
        if (!(abs2(d) > 0.0)) atomicOr(status, 1);
        dinv[w * M + j] = cinv(d);
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_tinv_form(const cx<T>* __restrict__ R, const double2* __restrict__ Dp,
                                                  const double2* __restrict__ dinv, const int* __restrict__ perm,
                                                  const double2* __restrict__ Tinv, double2* __restrict__ S, int M,
                                                  int ld) {
    __shared__ double2 tu[32][33];
    __shared__ int pos[32];                                  // position of T^-1's column c0 + q
    const int w = blockIdx.z, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32;    // rows and columns of R, or of T^-1
    const size_t off = (size_t)w * M * M, so = (size_t)w * M;
    double2* Sw = S + so * ld;
    if (c0 + 31 > r0) {
        for (int q = wid; q < 32; q += 8) {
            const int m = r0 + q, j = c0 + lane;
            if (m < j && j < M) {
                const cx<T> r = R[off + (size_t)m * M + j];
                double2 v = make_double2(r.x, r.y);
                if (Dp) v = cmul(v, Dp[so + j]);
                tu[q][lane] = cmul(v, dinv[so + m]);
            }
        }
        __syncthreads();
        for (int q = wid; q < 32; q += 8) {
            const int j = c0 + q, m = r0 + lane;
            if (m < j && j < M) Sw[(size_t)j * ld + m] = tu[lane][q];
        }
        __syncthreads();
    }
    for (int j = threadIdx.x; j < M; j += 256) {
        const int c = perm[so + j] - c0;
        if (c >= 0 && c < 32) pos[c] = j;
    }
    for (int q = wid; q < 32; q += 8) {
        const int i = r0 + q, c = c0 + lane;
        if (i < M && c < M) tu[q][lane] = Tinv[off + (size_t)i * M + c];
    }
    __syncthreads();
    for (int q = wid; q < 32; q += 8) {
        const int c = c0 + q, i = r0 + lane;
        if (c < M && i < M) Sw[(size_t)pos[q] * ld + ld / 2 + i] = tu[lane][q];
    }
}

// T^-1[i][j] = S[j][rhs + i].
__global__ void __launch_bounds__(256) k_tinv_out(const double2* __restrict__ S, double2* __restrict__ Tinv,
                                                 int* __restrict__ status, int M, int ld) {
    __shared__ double2 t[32][33];
    const int w = blockIdx.z, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int i0 = blockIdx.x * 32, j0 = blockIdx.y * 32;
    bool bad = false;
    for (int q = wid; q < 32; q += 8) {
        const int j = j0 + q, i = i0 + lane;
        if (j < M && i < M) {
            const double2 v = S[((size_t)w * M + j) * ld + ld / 2 + i];
            t[q][lane] = v;
            // finite: neither exponent field is all ones
            bad = bad || ((__double2hiint(v.x) & 0x7ff00000) == 0x7ff00000) ||
                  ((__double2hiint(v.y) & 0x7ff00000) == 0x7ff00000);
        }
    }
    if (bad) atomicOr(status, 1);
    __syncthreads();
    for (int q = wid; q < 32; q += 8) {
        const int i = i0 + q, j = j0 + lane;
        if (i < M && j < M) Tinv[((size_t)w * M + i) * M + j] = t[lane][q];
    }
}

template <typename T>
cudaError_t launch_update(ftq_ctx* c, cx<T>* S, int ld, int jb, int nb, int r0, int r1, int c0, int c1,
                          int kind = FTQ_K_GREEN) {
    using C = UpCfg<T>;
    UpArgs<T> a;
    a.S = S;
    a.status = c->status;
    a.M = c->M;
    a.ld = ld;
    a.jb = jb;
    a.nb = nb;
    a.r0 = r0;
    a.r1 = r1;
    a.c0 = c0;
    a.c1 = c1;
    a.nrb = (r1 - r0 + 63) / 64;
    a.nct = (c1 - c0 + C::OCT - 1) / C::OCT;
    a.W = c->W;
    a.wait_limit = c->wait_limit >= 0 ? (long long)c->wait_limit : TC_WAIT_LIMIT;
    if (a.nrb <= 0 || a.nct <= 0) return cudaSuccess;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    constexpr size_t sm = up_smem<T>();
    cudaError_t e = cudaFuncSetAttribute(k_lu_update<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    c->launches[kind] += 1;
    k_lu_update<T><<<std::min(sms, a.W * a.nrb * a.nct), NT_UP, sm, c->stream>>>(
        a, *reinterpret_cast<const CUtensorMap*>(c->lu_map[sizeof(T) == 8]));
    return cudaGetLastError();
}

// The elimination and the substitution on S.
template <typename T, int NB, int MAXT>
cudaError_t lu_solve(ftq_ctx* c, cx<T>* S, const LuScales<T>& sc, int ld) {
    const int M = c->M, W = c->W;
    cudaError_t e = cudaSuccess;
    // blocks of at most 128 columns, as even as whole warps allow
    auto blocks = [](int n) { return (n + 127) / 128; };
    auto threads = [&](int n) { return ((n + blocks(n) - 1) / blocks(n) + 31) / 32 * 32; };
    auto cols = [&](int n, int w) { return dim3((unsigned)((n + threads(n) - 1) / threads(n)), (unsigned)w); };
    const size_t per = (size_t)M * ld;                   // a walker's S
    const int rhs = ld / 2, end = rhs + M;               // columns of the right-hand sides
    for (int jb = 0; jb < M && e == cudaSuccess; jb += NB) {
        const int nb = std::min(NB, M - jb), m = M - jb, c0 = jb + nb;
        c->launches[FTQ_K_GREEN] += 2;
        k_lu_panel<T, NB, MAXT><<<W, (m + 31) / 32 * 32, 0, c->stream>>>(S, sc, c->status, M, ld, jb, nb);
        walker_spans(W, [&](size_t w0, int n) {
            k_lu_tri<T, NB, false><<<cols(end - c0, n), threads(end - c0), 0, c->stream>>>(
                S + per * w0, sc.from(w0, M), M, ld, jb, nb, c0, end);
        });
        e = cudaGetLastError();
        if (e == cudaSuccess) e = launch_update<T>(c, S, ld, jb, nb, c0, M, c0, end);
    }
    for (int jb = (M - 1) / NB * NB; jb >= 0 && e == cudaSuccess; jb -= NB) {
        const int nb = std::min(NB, M - jb);
        c->launches[FTQ_K_GREEN] += 1;
        walker_spans(W, [&](size_t w0, int n) {
            k_lu_tri<T, NB, true><<<cols(M, n), threads(M), 0, c->stream>>>(S + per * w0, sc.from(w0, M), M, ld, jb, nb,
                                                                            rhs, end);
        });
        e = cudaGetLastError();
        if (e == cudaSuccess) e = launch_update<T>(c, S, ld, jb, nb, 0, jb, rhs, end);
    }
    return e;
}

template <typename T>
LuScales<T> scales_of(const ftq_ctx* c) {
    LuScales<T> s;
    const size_t n = (size_t)c->W * c->M;
    double* b = c->lu_scal;
    s.drs = reinterpret_cast<cx<T>*>(b);
    s.inv = reinterpret_cast<cx<T>*>(b + 2 * n);
    s.dlb = reinterpret_cast<T*>(b + 4 * n);
    s.dls = reinterpret_cast<T*>(b + 5 * n);
    s.drb = reinterpret_cast<T*>(b + 6 * n);
    s.lsum = b + 7 * n;
    s.swaps = c->lu_int;
    s.perm = c->lu_int + c->W;
    return s;
}

}  // namespace

int lu_ld(int M) { return 2 * ((M + 3) / 4 * 4); }
size_t lu_scal_doubles(int M, int W) { return (size_t)W * (7 * (size_t)M + 1); }
size_t lu_ints(int W) { return (size_t)W * (1 + 2 * LU_NB_MAX); }

// Smaller bases keep the one-block k_green: at M = 33, 300 walkers a slice takes
// 0.31 ms there and 0.57 ms here (launches and half-empty tiles), at M = 57, 256
// walkers 1.20 against 0.72 ms.  Above, a panel row no longer fits a thread.
bool lu64_supported(int M) { return M >= 48 && M <= 640; }

// Maps of S over the buffers it lives in: [W][M][ld], a row as floats.
cudaError_t lu_make_maps(ftq_ctx* c) {
    const size_t M = c->M, W = c->W, ld = lu_ld(c->M);
    bool ok = tc_map_3d(c->lu_map[1], c->work, 4 * ld, M, W, 16 * ld, 16 * ld * M, CROW / 4, CBOX);
    if (c->w32) ok = ok && tc_map_3d(c->lu_map[0], c->w32, 2 * ld, M, W, 8 * ld, 8 * ld * M, CROW / 4, CBOX);
    return ok ? cudaSuccess : cudaErrorNotSupported;
}

namespace {

template <typename T>
cudaError_t tinv_lu(ftq_ctx* c, const cx<T>* R, const double2* Dp, const int* perm, bool df) {
    const int M = c->M, W = c->W, ld = lu_ld(M), rhs = ld / 2;
    double2* S = c->work;
    double2* dinv = scales_of<double>(c).inv;
    auto tiles = [&](int n) { return dim3((unsigned)((M + 31) / 32), (unsigned)((M + 31) / 32), (unsigned)n); };
    const size_t per = (size_t)M * ld, MM = (size_t)M * M;
    k_tinv_diag<T><<<W, 256, 0, c->stream>>>(R, Dp, dinv, c->DR, c->status, M);
    walker_spans(W, [&](size_t w0, int n) {
        const size_t o = w0 * M;
        k_tinv_form<T><<<tiles(n), 256, 0, c->stream>>>(R + MM * w0, Dp ? Dp + o : nullptr, dinv + o, perm + o,
                                                        c->Tinv + MM * w0, S + per * w0, M, ld);
    });
    c->launches[FTQ_K_TINV] += 2;
    const int nblk = (M + 127) / 128, nt = ((M + nblk - 1) / nblk + 31) / 32 * 32;
    auto cols = [&](int n) { return dim3((unsigned)((M + nt - 1) / nt), (unsigned)n); };
    const size_t sm = sizeof(float4) * (32 * 32 + 32 * (size_t)nt);
    cudaError_t e = cudaGetLastError();
    if (df && e == cudaSuccess)
        e = cudaFuncSetAttribute(k_tinv_tri_df, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(sizeof(float4) * (32 * 32 + 32 * 128)));
    for (int jb = 0; jb < M && e == cudaSuccess; jb += 32) {
        const int nb = std::min(32, M - jb);
        walker_spans(W, [&](size_t w0, int n) {
            double2* Sw = S + per * w0;
            if (df) k_tinv_tri_df<<<cols(n), nt, sm, c->stream>>>(Sw, M, ld, jb, nb, rhs, rhs + M);
            else k_lu_tri<double, 32, false, false><<<cols(n), nt, 0, c->stream>>>(
                Sw, scales_of<double>(c).from(w0, M), M, ld, jb, nb, rhs, rhs + M);
        });
        c->launches[FTQ_K_TINV] += 1;
        e = cudaGetLastError();
        if (e == cudaSuccess) e = launch_update<double>(c, S, ld, jb, nb, jb + nb, M, rhs, rhs + M, FTQ_K_TINV);
    }
    if (e != cudaSuccess) return e;
    walker_spans(W, [&](size_t w0, int n) {
        k_tinv_out<<<tiles(n), 256, 0, c->stream>>>(S + per * w0, c->Tinv + MM * w0, c->status, M, ld);
    });
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_tinv_lu32(ftq_ctx* c) {
    LaunchScope ls(c, FTQ_K_TINV);
    return tinv_lu<float>(c, c->w32, c->hh, c->perm, true);
}

cudaError_t launch_tinv_lu64(ftq_ctx* c, const double2* R, const int* perm) {
    return tinv_lu<double>(c, R, nullptr, perm, false);
}

cudaError_t launch_green_lu64(ftq_ctx* c, const double2* Y, int k, bool update, bool physical) {
    const int M = c->M, W = c->W, ld = lu_ld(M);
    const LuScales<double> sc = scales_of<double>(c);
    const double lscale = physical ? 0.0 : left_scale(c, k);
    auto tiles = [&](int n) { return dim3((unsigned)((M + 31) / 32), (unsigned)((M + 31) / 32), (unsigned)n); };
    const size_t per = (size_t)M * ld, MM = (size_t)M * M;
    LaunchScope ls(c, FTQ_K_GREEN);
    k_lu_scales<double><<<W, 256, 0, c->stream>>>(c->DR, c->tab.eps, sc, M, lscale, c->sys.mu_T);
    walker_spans(W, [&](size_t w0, int n) {
        k_lu_form64<<<tiles(n), 256, 0, c->stream>>>(Y + MM * w0, c->Tinv + MM * w0, c->work + per * w0, sc.from(w0, M), M,
                                                     ld);
    });
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess)
        e = M <= 384 ? lu_solve<double, 32, 384>(c, c->work, sc, ld) : lu_solve<double, 16, 640>(c, c->work, sc, ld);
    if (e != cudaSuccess) return e;
    c->launches[FTQ_K_GREEN] += 3;      // beside the scope's own: form, G and the tail
    walker_spans(W, [&](size_t w0, int n) {
        k_lu_green<double><<<tiles(n), 256, 0, c->stream>>>(c->work + per * w0, c->G + MM * w0, sc.from(w0, M), M, ld);
    });
    k_lu_tail<double><<<W, 128, 0, c->stream>>>(c->work, c->G, sc, c->wstate, c->status, M, ld,
                                               (double)k * c->sys.dtau, c->opts.constraint, update ? 1 : 0,
                                               physical ? 0 : 1);
    return cudaGetLastError();
}

cudaError_t launch_green_lu32(ftq_ctx* c, int k, float2* G, double* ws) {
    const int M = c->M, W = c->W, ld = lu_ld(M);
    const LuScales<float> sc = scales_of<float>(c);
    Planes P;
    P.Kp = c->Kp;
    P.part = (size_t)c->LD * 2 * c->Kp;
    auto tiles = [&](int n) { return dim3((unsigned)((M + 31) / 32), (unsigned)((M + 31) / 32), (unsigned)n); };
    const size_t per = (size_t)M * ld, MM = (size_t)M * M;
    LaunchScope ls(c, FTQ_K_GREEN);
    if (!G) G = c->G32;
    k_lu_scales<float><<<W, 256, 0, c->stream>>>(c->DR, c->tab.eps, sc, M, left_scale(c, k), c->sys.mu_T);
    walker_spans(W, [&](size_t w0, int n) {
        k_lu_form32<<<tiles(n), 256, 0, c->stream>>>(c->Ypl + 2 * P.part * w0, c->Tinv + MM * w0, c->w32 + per * w0,
                                                     sc.from(w0, M), P, 2 * P.part, M, ld);
    });
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess)
        e = M <= 640 ? lu_solve<float, 32, 640>(c, c->w32, sc, ld) : lu_solve<float, 16, 1024>(c, c->w32, sc, ld);
    if (e != cudaSuccess) return e;
    c->launches[FTQ_K_GREEN] += 3;      // beside the scope's own: form, G and the tail
    walker_spans(W, [&](size_t w0, int n) {
        k_lu_green<float><<<tiles(n), 256, 0, c->stream>>>(c->w32 + per * w0, G + MM * w0, sc.from(w0, M), M, ld);
    });
    k_lu_tail<float><<<W, 128, 0, c->stream>>>(c->w32, G, sc, ws ? ws : c->wstate, c->status, M, ld,
                                              (double)k * c->sys.dtau, c->opts.constraint, 1, 1);
    return cudaGetLastError();
}

}  // namespace ftq
