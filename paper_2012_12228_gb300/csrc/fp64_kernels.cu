// Complex128 kernels of the walker slice: force bias and HS fields, Householder
// QRCP stabilisation, and the two-sided stable Green's function with ln det and
// the phaseless weight (the chain is in chain_oz.cu, the estimators in
// estimators.cu).  One walker per thread block for the factorisations.
#include <algorithm>
#include <cmath>

#include "block_reduce.cuh"
#include "complex_math.cuh"
#include "ftq_internal.h"
#include "green_tail.cuh"
#include "reflect.cuh"

namespace ftq {
namespace {

// ---------------------------------------------------------------- init
__global__ void k_init_matrices(double2* Y, double2* Tinv, double2* G, const double* g0, int M, long total) {
    long e = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (e >= total) return;
    int ij = (int)(e % ((long)M * M));
    int i = ij / M, j = ij % M;
    double2 one = make_double2(i == j ? 1.0 : 0.0, 0.0);
    Y[e] = one;
    Tinv[e] = one;
    G[e] = make_double2(i == j ? g0[i] : 0.0, 0.0);
}

__global__ void k_init_walkers(double2* DR, double* ws, int M, int W, double ld0) {
    int w = blockIdx.x;
    for (int i = threadIdx.x; i < M; i += blockDim.x) DR[(long)w * M + i] = make_double2(1.0, 0.0);
    if (threadIdx.x == 0) {
        double* s = ws + (long)WSTRIDE * w;
        for (int q = 0; q < WSTRIDE; ++q) s[q] = 0.0;
        s[2] = 1.0;
        s[3] = ld0;
        s[12] = (double)M;
    }
}

// ---------------------------------------------------------------- force bias
// rho_Q = sum_{(a,b): n_a - n_b = Q} P_ab with P = I - G^T, so for Q != 0
// rho_Q = -sum G[b][a].  <v_A> = 2 i c (rho_Q + rho_-Q), <v_B> = -2 c (rho_Q -
// rho_-Q); xbar = -sqrt(dtau) <v>; y = x - xbar; the V generator
// phi(+Q) = sqrt(dtau) c i (y_A + i y_B), phi(-Q) = sqrt(dtau) c i (y_A - i y_B).
// Sums of G entries: FP64 entries in FP64, FP32 entries as an FP32 pair with the
// rounding errors of its two-sums collected (48 bits and more: a list has at most M
// entries).  A conversion and an addition per part on the FP64 pipe took half of the
// kernel's time on the FP32 G (per slice, before and after, with one pair list for both
// signs of Q: M = 57, 640 walkers 0.059 -> 0.028 ms, M = 257, 1024 walkers 0.92 -> 0.79).
struct SumF64 {
    double2 s = {0.0, 0.0};
    __device__ __forceinline__ void add(double2 g) { s = s + g; }
    __device__ __forceinline__ double2 value() const { return s; }
};
struct SumF32 {
    float2 h = {0.f, 0.f}, l = {0.f, 0.f};
    __device__ __forceinline__ static void two_sum(float& hi, float& lo, float g) {
        const float t = hi + g, b = t - hi;
        lo += (hi - (t - b)) + (g - b);
        hi = t;
    }
    __device__ __forceinline__ void add(float2 g) {
        two_sum(h.x, l.x, g.x);
        two_sum(h.y, l.y, g.y);
    }
    __device__ __forceinline__ double2 value() const {
        return make_double2((double)h.x + (double)l.x, (double)h.y + (double)l.y);
    }
};
template <typename GT> struct SumOf { using type = SumF64; };
template <> struct SumOf<float2> { using type = SumF32; };

template <typename GT>
__global__ void k_force_bias(const GT* __restrict__ G, const double* __restrict__ x,
                             double2* __restrict__ phi, float2* __restrict__ phi32, double* __restrict__ ws,
                             const int* __restrict__ pptr, const int* __restrict__ pa,
                             const int* __restrict__ pb, const double* __restrict__ cq,
                             int M, int nqh, double sdt) {
    __shared__ double2 sh[32];
    const int w = blockIdx.x;
    const GT* Gw = G + (long)w * M * M;
    const double* xw = x + (long)w * 2 * nqh;
    double2* ph = phi + (long)w * (2 * nqh + 1);
    float2* ph32 = phi32 ? phi32 + (long)w * (2 * nqh + 1) : nullptr;
    double2 gauss = make_double2(0.0, 0.0);
    if (threadIdx.x == 0) {
        ph[0] = make_double2(0.0, 0.0);
        if (ph32) ph32[0] = make_float2(0.f, 0.f);
    }
    for (int q = threadIdx.x; q < nqh; q += blockDim.x) {
        // the pairs of -Q are those of +Q reversed: both sums from one list
        typename SumOf<GT>::type sp, sm;
        const int end = pptr[2 + 2 * q];
#pragma unroll 4
        for (int e = pptr[1 + 2 * q]; e < end; ++e) {
            const int a = pa[e], b = pb[e];
            sp.add(Gw[b * M + a]);
            sm.add(Gw[a * M + b]);
        }
        const double2 rp = sp.value() * -1.0, rm = sm.value() * -1.0;
        const double c = cq[q];
        double2 vA = times_i((rp + rm) * (2.0 * c));
        double2 vB = (rp - rm) * (-2.0 * c);
        double2 xbA = vA * (-sdt), xbB = vB * (-sdt);
        double xA = xw[2 * q], xB = xw[2 * q + 1];
        double2 yA = make_double2(xA - xbA.x, -xbA.y);
        double2 yB = make_double2(xB - xbB.x, -xbB.y);
        double2 iyB = times_i(yB);
        const double2 pp = times_i(yA + iyB) * (sdt * c), pm = times_i(yA - iyB) * (sdt * c);
        ph[1 + 2 * q] = pp;
        ph[2 + 2 * q] = pm;
        if (ph32) {
            ph32[1 + 2 * q] = make_float2((float)pp.x, (float)pp.y);
            ph32[2 + 2 * q] = make_float2((float)pm.x, (float)pm.y);
        }
        gauss = gauss + xbA * xA - cmul(xbA, xbA) * 0.5 + xbB * xB - cmul(xbB, xbB) * 0.5;
    }
    gauss = block_sum(gauss, sh);
    if (threadIdx.x == 0) {
        ws[(long)WSTRIDE * w + 5] = gauss.x;
        ws[(long)WSTRIDE * w + 6] = gauss.y;
    }
}

// ---------------------------------------------------------------- QRCP
// Householder QR with column pivoting of C = Y diag(D_R) (Businger-Golub:
// pivot = remaining column of largest norm, ties to the lowest index).
// Reflector H = I - tau u u^H with u = x - beta e_1, beta = -e^{i arg x_0}|x|,
// so H x = beta e_1 and R_jj = beta.  Outputs: Q (next chain start), D_R =
// diag R, T^-1 <- T^-1 Pi^T (D^-1 R)^-1, parity of Pi.
__global__ void __launch_bounds__(1024) k_qrcp(const double2* __restrict__ Yin, double2* __restrict__ Qout,
                       double2* __restrict__ work, double2* __restrict__ work2,
                       double2* __restrict__ DR, double2* __restrict__ Tinv,
                       double2* __restrict__ hh, double* __restrict__ htau,
                       double* __restrict__ ws, int* __restrict__ status, int* __restrict__ perm_out, int M,
                       int in_smem) {
    extern __shared__ unsigned char smem_raw[];
    double* cn = reinterpret_cast<double*>(smem_raw);          // column norms [M]
    int* perm = reinterpret_cast<int*>(cn + M);                 // [M]
    __shared__ double shv[32];
    __shared__ int shi[32];
    __shared__ int nswap;
    const int w = blockIdx.x;
    const long off = (long)w * M * M;
    // small bases: the three matrices in shared memory (fact_smem)
    double2* mats = reinterpret_cast<double2*>(smem_raw + ((12 * (size_t)M + 15) & ~(size_t)15));
    double2* C = in_smem ? mats : work + off;
    double2* Q = in_smem ? mats + M * M : Qout + off;
    double2* XT = in_smem ? mats + 2 * M * M : work2 + off;
    double2* Ti = Tinv + off;
    const double2* Yw = Yin + off;
    double2* u0 = hh + (long)w * M;
    double* tau = htau + (long)w * M;
    const int nt = blockDim.x;

    for (long e = threadIdx.x; e < (long)M * M; e += nt) {
        int c = (int)(e % M);
        C[e] = cmul(Yw[e], DR[(long)w * M + c]);
    }
    for (int c = threadIdx.x; c < M; c += nt) perm[c] = c;
    if (threadIdx.x == 0) nswap = 0;
    __syncthreads();

    // norms of the columns; after that every reflector's update leaves those of the
    // rows below it, so that no pass over the matrix is spent on them
    for (int c = threadIdx.x; c < M; c += nt) {
        double s = 0.0;
        for (int r = 0; r < M; ++r) s += abs2(C[(long)r * M + c]);
        cn[c] = s;
    }
    __syncthreads();
    for (int j = 0; j < M; ++j) {
        double best = -1.0;
        int bidx = M;
        for (int c = j + threadIdx.x; c < M; c += nt) {
            const double s = cn[c];
            if (s > best) { best = s; bidx = c; }
        }
        int pc = block_argmax(best, bidx, shv, shi);
        if (pc >= M) {                       // every candidate norm was NaN
            pc = j;
            if (threadIdx.x == 0) atomicOr(status, 1);
        }
        if (pc != j) {
            for (int r = threadIdx.x; r < M; r += nt) {
                double2 t = C[(long)r * M + j];
                C[(long)r * M + j] = C[(long)r * M + pc];
                C[(long)r * M + pc] = t;
            }
            if (threadIdx.x == 0) {
                int t = perm[j]; perm[j] = perm[pc]; perm[pc] = t;
                double tn = cn[j]; cn[j] = cn[pc]; cn[pc] = tn;
                nswap ^= 1;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double2 al = C[(long)j * M + j];
            double sig = sqrt(cn[j]);
            double aa = sqrt(abs2(al));
            double2 beta = aa > 0.0 ? al * (-sig / aa) : make_double2(-sig, 0.0);
            double uhu = 2.0 * sig * (sig + aa);
            u0[j] = al - beta;
            tau[j] = uhu > 0.0 ? 2.0 / uhu : 0.0;
            C[(long)j * M + j] = beta;
            if (!(sig > 0.0)) atomicOr(status, 1);
        }
        __syncthreads();
        reflect_columns<true>(C, M, j, C, M, M, j + 1, M, u0[j], tau[j], cn);
        __syncthreads();
    }
    // Q = H_0 H_1 ... H_{M-1} by backward accumulation
    for (long e = threadIdx.x; e < (long)M * M; e += nt) {
        int i = (int)(e / M), c = (int)(e % M);
        Q[e] = make_double2(i == c ? 1.0 : 0.0, 0.0);
    }
    __syncthreads();
    for (int j = M - 1; j >= 0; --j) {
        reflect_columns<false>(C, M, j, Q, M, M, j, M, u0[j], tau[j], nullptr);
        __syncthreads();
    }
    if (in_smem)
        for (int e = threadIdx.x; e < M * M; e += nt) Qout[off + e] = Q[e];
    if (perm_out) {                          // T^-1 is updated from R by the kernels of green_lu.cu
        for (int j = threadIdx.x; j < M; j += nt) perm_out[(long)w * M + j] = perm[j];
        if (threadIdx.x == 0) {
            double* s = ws + (long)WSTRIDE * w;
            s[7] = (double)(((int)s[7]) ^ nswap);
        }
        return;
    }
    // D = diag R; U = D^-1 R (strict upper part scaled in place)
    for (int j = threadIdx.x; j < M; j += nt) DR[(long)w * M + j] = C[(long)j * M + j];
    for (long e = threadIdx.x; e < (long)M * M; e += nt) {
        int i = (int)(e / M), c = (int)(e % M);
        if (c > i) C[e] = cdiv(C[e], C[(long)i * M + i]);
    }
    __syncthreads();
    // T^-1 <- T^-1[:, perm] U^-1, one row per thread (XT column-major)
    for (int i = threadIdx.x; i < M; i += nt) {
        for (int j = 0; j < M; ++j) {
            double2 s = Ti[(long)i * M + perm[j]];
            for (int m = 0; m < j; ++m) s = cfms(XT[(long)m * M + i], C[(long)m * M + j], s);
            XT[(long)j * M + i] = s;
        }
        for (int j = 0; j < M; ++j) Ti[(long)i * M + j] = XT[(long)j * M + i];
    }
    if (threadIdx.x == 0) {
        double* s = ws + (long)WSTRIDE * w;
        s[7] = (double)(((int)s[7]) ^ nswap);
    }
}

// ---------------------------------------------------------------- Green's function
// G(tau_k) = (I + R D_L)^-1 with R = Y D_R T, D_L = B_T^(n-k):
//   Mt = D_Lb T^-1 D_Rb + D_Ls Y D_Rs,  G = I - Y D_Rs Mt^-1 D_Ls,
//   ln det(I + A) = -sum ln D_Lb - sum ln D_Rb + ln det Mt + ln det T,
// then ln S_k = 2 (ln det_k - ln det_{k-1}) and the weight (Eqs. import,
// phimport, theta).
//
// L lanes share a column of the LU's updates and a row of the solves: more than one for
// the small bases, where a lane per row left half of a block's lanes idle and the
// sums' latency exposed (green_lanes).
template <int L>
__device__ __forceinline__ double2 lane_sum(double2 s) {
#pragma unroll
    for (int o = 1; o < L; o <<= 1) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
    }
    return s;
}

template <int L>
__global__ void __launch_bounds__(1024) k_green(const double2* __restrict__ Y, const double2* __restrict__ Tinv,
                        const double2* __restrict__ DR, double2* __restrict__ work,
                        double2* __restrict__ work2, double2* __restrict__ G,
                        const double* __restrict__ eps, double* __restrict__ ws,
                        int* __restrict__ status, int M, double lscale, double mu_T,
                        int constraint, int update, int with_gauss, double kdt, int in_smem) {
    extern __shared__ unsigned char smem_raw[];
    double2* drs = reinterpret_cast<double2*>(smem_raw);     // [M]
    double2* invU = drs + M;                                 // [M]
    double* dls = reinterpret_cast<double*>(invU + M);       // [M]
    double* dlb = dls + M;                                   // [M]
    double* drb = dlb + M;                                   // [M]
    int* perm = reinterpret_cast<int*>(drb + M);             // [M]
    __shared__ double shv[32];
    __shared__ int shi[32];
    __shared__ double2 shc[32];
    __shared__ int nswap;
    const int w = blockIdx.x;
    const long off = (long)w * M * M;
    const int nt = blockDim.x;
    const int q = threadIdx.x % L;
    // small bases: both matrices in shared memory (fact_smem)
    double2* mats = reinterpret_cast<double2*>(smem_raw + ((60 * (size_t)M + 15) & ~(size_t)15));
    double2* A = in_smem ? mats : work + off;
    double2* XT = in_smem ? mats + M * M : work2 + off;
    const double2* Yw = Y + off;
    const double2* Tw = Tinv + off;
    double2* Gw = G + off;

    double lsum = 0.0;
    for (int i = threadIdx.x; i < M; i += nt) {
        double dl = exp(-lscale * (eps[i] - mu_T));
        if (dl > 1.0) { dlb[i] = 1.0 / dl; dls[i] = 1.0; } else { dlb[i] = 1.0; dls[i] = dl; }
        double2 d = DR[(long)w * M + i];
        double a = sqrt(abs2(d));
        if (a > 1.0) { drb[i] = 1.0 / a; drs[i] = d * (1.0 / a); } else { drb[i] = 1.0; drs[i] = d; }
        lsum += log(dlb[i]) + log(drb[i]);
        perm[i] = i;
    }
    if (threadIdx.x == 0) nswap = 0;
    __syncthreads();
    for (long e = threadIdx.x; e < (long)M * M; e += nt) {
        int i = (int)(e / M), j = (int)(e % M);
        A[e] = Tw[e] * (dlb[i] * drb[j]) + cmul(Yw[e], drs[j]) * dls[i];
    }
    __syncthreads();
    // LU with partial pivoting, in place
    for (int j = 0; j < M; ++j) {
        double best = -1.0;
        int bidx = M;
        for (int i = j + threadIdx.x; i < M; i += nt) {
            double v = abs1(A[(long)i * M + j]);
            if (v > best) { best = v; bidx = i; }
        }
        int p = block_argmax(best, bidx, shv, shi);
        if (p >= M) {                        // every candidate pivot was NaN
            p = j;
            if (threadIdx.x == 0) atomicOr(status, 1);
        }
        if (p != j) {
            for (int c = threadIdx.x; c < M; c += nt) {
                double2 t = A[(long)j * M + c];
                A[(long)j * M + c] = A[(long)p * M + c];
                A[(long)p * M + c] = t;
            }
            if (threadIdx.x == 0) {
                int t = perm[j]; perm[j] = perm[p]; perm[p] = t;
                nswap ^= 1;
            }
        }
        __syncthreads();
        const double2 piv = A[(long)j * M + j];
        if (!(abs2(piv) > 0.0)) {
            if (threadIdx.x == 0) atomicOr(status, 1);
        }
        const double2 ip = cinv(piv);
        for (int i = j + 1 + threadIdx.x; i < M; i += nt) A[(long)i * M + j] = cmul(A[(long)i * M + j], ip);
        if (threadIdx.x == 0) invU[j] = ip;
        __syncthreads();
        for (int c = j + 1 + (int)threadIdx.x / L; c < M; c += nt / L) {
            const double2 u = A[(long)j * M + c];
            for (int i = j + 1 + q; i < M; i += L) A[(long)i * M + c] = cfms(A[(long)i * M + j], u, A[(long)i * M + c]);
        }
        __syncthreads();
    }
    // ln det Mt = sum ln U_jj + i pi (row-swap parity)
    double2 ldm = make_double2(0.0, 0.0);
    for (int j = threadIdx.x; j < M; j += nt) ldm = ldm + clog(A[(long)j * M + j]);
    ldm = block_sum(ldm, shc);
    lsum = block_sum(lsum, shv);
    // X = (Y D_Rs) U^-1 L^-1 solved row by row (XT column-major), then
    // G[i][perm[m]] = delta - X[i][m] dls[perm[m]].
    // L lanes share a row and its sums (the same trips for every lane of a warp)
    for (int ib = 0; ib < M; ib += nt / L) {
        const int i = ib + (int)threadIdx.x / L;
        const bool on = i < M;
        for (int j = 0; j < M; ++j) {
            double2 s = make_double2(0.0, 0.0);
            if (on) {
                if (q == 0) s = cmul(Yw[(long)i * M + j], drs[j]);
                for (int m = q; m < j; m += L) s = cfms(XT[(long)m * M + i], A[(long)m * M + j], s);
            }
            s = lane_sum<L>(s);
            if (on && q == 0) XT[(long)j * M + i] = cmul(s, invU[j]);
            __syncwarp();
        }
        for (int j = M - 2; j >= 0; --j) {
            double2 s = make_double2(0.0, 0.0);
            if (on) {
                if (q == 0) s = XT[(long)j * M + i];
                for (int m = j + 1 + q; m < M; m += L) s = cfms(XT[(long)m * M + i], A[(long)m * M + j], s);
            }
            s = lane_sum<L>(s);
            if (on && q == 0) XT[(long)j * M + i] = s;
            __syncwarp();
        }
        for (int m = q; m < M && on; m += L) {
            int c = perm[m];
            double2 g = XT[(long)m * M + i] * (-dls[c]);
            if (c == i) g.x += 1.0;
            Gw[(long)i * M + c] = g;
        }
    }
    __syncthreads();
    double2 trg = make_double2(0.0, 0.0);
    for (int i = threadIdx.x; i < M; i += nt) trg = trg + Gw[(long)i * M + i];
    trg = block_sum(trg, shc);
    if (threadIdx.x == 0) {
        green_weight_tail(ws + (long)WSTRIDE * w, ldm, lsum, nswap, trg, M, kdt, constraint, status, update,
                          with_gauss);
    }
}

// The one-block factorisations of bases below lu64_supported's keep their matrices in
// shared memory (two for G, three for the QRCP; at most 106 KB at M = 47) while an SM has
// four walkers at most: their time is latency then.  Per launch at M = 33, 300 walkers: G 378 ->
// 350 us (314 with four lanes per row), QRCP 670 -> 618 us (468 with two lanes per column).
// With more walkers an SM is filled by other blocks: one lane per row or column and the
// matrices in L2, so that more blocks fit (G of ten slices, this and the other: M = 27, 2432
// walkers 7.7 / 13.1 ms, M = 33 18.1 / 22.2, 608 walkers 5.1 / 5.7; a QRCP of M = 33, 2432 walkers
// 4.9 / 5.4 ms).
constexpr int SMEM_M = 47;

bool in_smem(const ftq_ctx* c) { return c->M <= SMEM_M && c->W <= 4 * sm_count(); }

size_t fact_smem(const ftq_ctx* c, size_t vectors, int matrices) {
    return in_smem(c) ? ((vectors + 15) & ~(size_t)15) + sizeof(double2) * matrices * (size_t)c->M * c->M : vectors;
}

// Lanes per row of k_green: four while an SM has one walker and a half, two up to four (M = 33, ten
// slices, 304 walkers 3.15 ms with four lanes, 2.84 with two; 608 walkers 5.73 and 4.66); four
// also where they fit one warp.  Larger bases (M > 640): one.
int green_lanes(const ftq_ctx* c) {
    if (c->M > SMEM_M) return 1;
    const int sms = sm_count();
    return 4 * c->M <= 32 || 2 * c->W <= 3 * sms ? 4 : (c->W <= 4 * sms ? 2 : 1);
}

int fact_threads(int M) {
    int t = ((M + 31) / 32) * 32;
    return t > 1024 ? 1024 : (t < 32 ? 32 : t);
}

}  // namespace

cudaError_t launch_init_walkers(ftq_ctx* c) {
    const int M = c->M, W = c->W;
    double ld0 = 0.0;
    for (int i = 0; i < M; ++i) ld0 += std::log1p(std::exp(-c->sys.beta * (c->sys.eps[i] - c->sys.mu_T)));
    long total = (long)W * M * M;
    LaunchScope ls0(c, FTQ_K_INIT);
    k_init_matrices<<<(unsigned)((total + 255) / 256), 256, 0, c->stream>>>(c->Y ? c->Y : c->zbuf[1], c->Tinv, c->G,
                                                                           c->tab.g0, M, total);
    c->launches[FTQ_K_INIT] += 1;
    k_init_walkers<<<W, 64, 0, c->stream>>>(c->DR, c->wstate, M, W, ld0);
    c->k = 0;
    c->g64_valid = true;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && c->opts.precision != FTQ_FP64) e = mixed_init(c);
    return e;
}

cudaError_t launch_force_bias_any(ftq_ctx* c, const double* x, const void* G, bool g32) {
    LaunchScope ls(c, FTQ_K_FORCE_BIAS);
    if (g32)
        k_force_bias<float2><<<c->W, 256, 0, c->stream>>>(reinterpret_cast<const float2*>(G), x, c->phi, c->phi32,
                                                          c->wstate,
                                                          c->tab.pair_ptr, c->tab.pair_a, c->tab.pair_b, c->tab.cq,
                                                          c->M, c->sys.nq_half, std::sqrt(c->sys.dtau));
    else
        k_force_bias<double2><<<c->W, 256, 0, c->stream>>>(reinterpret_cast<const double2*>(G), x, c->phi,
                                                           c->phi32, c->wstate, c->tab.pair_ptr, c->tab.pair_a, c->tab.pair_b,
                                                           c->tab.cq, c->M, c->sys.nq_half, std::sqrt(c->sys.dtau));
    return cudaGetLastError();
}

cudaError_t launch_force_bias(ftq_ctx* c, const double* x) {
    if (c->opts.precision != FTQ_FP64 && !c->g64_valid) return launch_force_bias_any(c, x, c->G32, true);
    return launch_force_bias_any(c, x, c->G, false);
}

cudaError_t launch_chain(ftq_ctx* c) {
    return c->opts.precision != FTQ_FP64 ? mixed_chain(c) : oz_chain(c);
}

cudaError_t launch_qrcp64(ftq_ctx* c, const double2* Yin, double2* Qout) {
    const int M = c->M;
    const bool small = in_smem(c);
    const size_t sm = fact_smem(c, (sizeof(double) + sizeof(int)) * M, 3);
    const int lanes = M > SMEM_M || small ? 2 : 1;           // per column
    const int nt = std::min(1024, lanes * fact_threads(M));
    if (sm > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_qrcp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
    }
    const bool lu = lu64_supported(M);
    double2* R = lu ? c->zbuf[1] : c->work;      // S of the T^-1 update takes the work buffer
    LaunchScope ls(c, FTQ_K_QRCP);
    k_qrcp<<<c->W, nt, sm, c->stream>>>(Yin, Qout, R, c->work2, c->DR, c->Tinv, c->hh, c->htau,
                                       c->wstate, c->status, lu ? c->perm : nullptr, M, small ? 1 : 0);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && lu) e = launch_tinv_lu64(c, R, c->perm);
    return e;
}

cudaError_t launch_qrcp(ftq_ctx* c) {
    if (c->opts.precision != FTQ_FP64) return mixed_qrcp(c);
    if (c->opts.low_rank_threshold > 0.0) return launch_qrcp_lr(c);
    cudaError_t e = launch_qrcp64(c, c->Y, c->zbuf[0]);
    double2* q = c->zbuf[0];
    c->zbuf[0] = c->Y;
    c->Y = q;
    return e;
}

double left_scale(const ftq_ctx* c, int k) {
    const int power = c->opts.overlap == FTQ_OVERLAP_MODIFIED ? c->sys.n_slices : c->sys.n_slices - k;
    return (double)power * c->sys.dtau;
}

cudaError_t launch_green64(ftq_ctx* c, const double2* Y, int k, bool update, bool physical) {
    const int M = c->M;
    if (c->opts.low_rank_threshold > 0.0) return launch_green_lr(c, Y, k, update, physical);
    if (lu64_supported(M)) return launch_green_lu64(c, Y, k, update, physical);
    const size_t sm = fact_smem(c, (2 * sizeof(double2) + 3 * sizeof(double) + sizeof(int)) * M, 2);
    const double lscale = physical ? 0.0 : left_scale(c, k);
    const int L = green_lanes(c);
    auto kernel = L == 4 ? k_green<4> : (L == 2 ? k_green<2> : k_green<1>);
    const int nt = L > 1 ? (L * M + 31) / 32 * 32 : fact_threads(M);
    if (sm > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    LaunchScope ls(c, FTQ_K_GREEN);
    kernel<<<c->W, nt, sm, c->stream>>>(Y, c->Tinv, c->DR, c->work, c->work2, c->G, c->tab.eps, c->wstate,
                                       c->status, M, lscale, c->sys.mu_T, c->opts.constraint, update ? 1 : 0,
                                       physical ? 0 : 1, (double)k * c->sys.dtau, in_smem(c) ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_green(ftq_ctx* c, int k, bool update) {
    if (c->opts.precision != FTQ_FP64) return mixed_green(c, k);
    cudaError_t e = launch_green64(c, c->Y, k, update);
    // the modified overlap ends with the physical G(beta) and the ratio r
    if (e == cudaSuccess && k == c->sys.n_slices && c->opts.overlap == FTQ_OVERLAP_MODIFIED)
        e = launch_green64(c, c->Y, k, update, true);
    return e;
}

cudaError_t launch_copy_green(ftq_ctx* c, double2* out) {
    if (!c->g64_valid) {
        cudaError_t e0 = mixed_sync_g64(c);
        if (e0 != cudaSuccess) return e0;
    }
    return cudaMemcpyAsync(out, c->G, sizeof(double2) * (size_t)c->W * c->M * c->M, cudaMemcpyDeviceToDevice,
                           c->stream);
}

}  // namespace ftq
