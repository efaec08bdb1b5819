// Density correlation <rho(Q) rho(-Q)> of every walker and its weighted
// average: the numerator of the static structure factor
// S(Q) = <rho(Q) rho(-Q)> / N (Results, structure factor), from
// P = I - G^T by Wick's theorem: Gamma_Q - Lambda_Q + D_Q with
// Gamma_Q = (2 rho_Q)(2 rho_-Q), Lambda_Q = 2 sum_{K1 K2} P_{K1+Q,K2} P_{K2-Q,K1}
// (the exchange sum of the energy estimator) and
// D_Q = 2 sum_{K: K, K+Q in basis} P_{K+Q,K+Q}.
#include <algorithm>
#include <cmath>

#include "complex_math.cuh"
#include "exchange.cuh"
#include "ftq_internal.h"

namespace ftq {
namespace {

// Totals over groups of GS lanes of eight values: the lanes halve the list as they halve the
// distance, seven to nine additions for eight values (a warp's FP64 addition takes 16 cycles
// of the SM).  Lane i GS / 8 of a group holds its total of value i.
template <int GS>
__device__ __forceinline__ double group_totals(double (&v)[8]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int n = 4, o = GS / 2; n >= 1; n >>= 1, o >>= 1)
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const bool up = lane & o;
            const double give = up ? v[i] : v[i + n];
            v[i] = (up ? v[i + n] : v[i]) + __shfl_xor_sync(0xffffffffu, give, o);
        }
#pragma unroll
    for (int o = GS / 16; o >= 1; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}

// The transfers q .. q + 32 / GS - 1 below end_q, one per group of GS lanes; with GS < 32 none
// has more than GS pairs.
template <int GS>
__device__ __forceinline__ void structure_task(const double2* Gw, const double2* Gt, const int* __restrict__ pptr,
                                               const int* __restrict__ pa, const int* __restrict__ pb, double2* out,
                                               int M, int q, int end_q) {
    const int lane = threadIdx.x & 31, gl = lane & (GS - 1), g0 = lane - gl;
    q += lane / GS;
    const bool live = q < end_q;
    const int first = live ? pptr[1 + 2 * q] : 0, end = live ? pptr[2 + 2 * q] : 0;
    double2 rp = make_double2(0.0, 0.0), rm = rp, sa = rp, sb = rp, x = rp;
    for (int e0 = first; e0 < end; e0 += GS) {
        const int e = e0 + gl;
        const bool on = e < end;
        const int a = on ? pa[e] : 0, d = on ? pb[e] : 0;
        const double2 t = exchange_products<double2>(Gw, Gt, M, pa, pb, first, end, a, d);
        if (on) {
            x = x + t;
            rp = rp - Gw[(size_t)d * M + a];                 // P_ad, a != d
            rm = rm - Gw[(size_t)a * M + d];
            sa = sa + Gw[(size_t)a * M + a];
            sb = sb + Gw[(size_t)d * M + d];
        }
    }
    __syncwarp();
    const double2 u = sb - x, v = sa - x;
    double all[8] = {rp.x, rp.y, rm.x, rm.y, u.x, u.y, v.x, v.y};
    const double t = group_totals<GS>(all);
    auto get = [&](int i) { return __shfl_sync(0xffffffffu, t, g0 + i * (GS / 8)); };
    const double2 p = make_double2(2.0 * get(0), 2.0 * get(1)), m = make_double2(2.0 * get(2), 2.0 * get(3));
    const int sl = gl & 1;                                   // lanes 0 and 1 of a group: slots +Q and -Q
    const double2 o = make_double2(get(4 + 2 * sl), get(5 + 2 * sl));
    if (live && gl < 2) out[2 * q + gl] = cmul(p, m) + o * 2.0;
}

// A group of lanes per walker and half-space transfer q (slots 1 + 2 q and 2 + 2 q, whose
// pairs are each other's reversed): both slots at once, since Lambda_-Q = Lambda_Q.
// With the deltas summed over the n pairs (a, d) of Q,
//   Lambda / 2 = X + n - A - B,  D_Q / 2 = n - A,  D_-Q / 2 = n - B,
// X the products of the exchange sum, A = sum G_aa, B = sum G_dd: n drops out, and
// Gamma + 2 (B - X), Gamma + 2 (A - X) are left.
// The FP64 pipe bounds it (four DFMA per exchange term, 16 cycles of an SM each for a whole
// warp), so lanes must not idle: the transfers up to `whole` take a warp each, those up to
// `half` (at most 16 pairs) share one by twos, the rest (at most 8) by fours.  The short
// transfers have the most pairs and come first; the warps of a walker's blocks take the
// tasks in turn.  Whole calls, before both signs shared a sum, then with a warp per transfer,
// and now: M = 33, 1216 walkers 0.72, 1.31 and 0.61 ms; M = 57, 608 walkers 0.82, 1.17 and
// 0.63; M = 257, 128 walkers 14.5, 5.2 and 3.7.  Two blocks per SM at 64 registers, with
// spills, beat one at 96 (M = 171, 152 walkers 1.56 against 2.11 ms).
__global__ void __launch_bounds__(512, 2) k_structure(const double2* __restrict__ G, const double2* __restrict__ Gtr,
                                                  const int* __restrict__ pptr, const int* __restrict__ pa,
                                                  const int* __restrict__ pb, double2* __restrict__ out, int M,
                                                  int nqh, int whole, int half) {
    const int w = blockIdx.y;
    const int warp = blockIdx.x + gridDim.x * (threadIdx.x >> 5), nw = gridDim.x * (blockDim.x >> 5);
    const double2* Gw = G + (size_t)w * M * M;
    const double2* Gt = Gtr + (size_t)w * M * M;
    double2* o = out + (size_t)w * nqh * 2;
    const int twos = (half - whole + 1) / 2, tasks = whole + twos + (nqh - half + 3) / 4;
    for (int t = warp; t < tasks; t += nw) {
        if (t < whole) structure_task<32>(Gw, Gt, pptr, pa, pb, o, M, t, whole);
        else if (t < whole + twos) structure_task<16>(Gw, Gt, pptr, pa, pb, o, M, whole + 2 * (t - whole), half);
        else structure_task<8>(Gw, Gt, pptr, pa, pb, o, M, half + 4 * (t - whole - twos), nqh);
    }
}

// Weights w = exp(ln|w| - s) e^{i arg w} of the alive walkers (s = max ln|w|)
// and their sum; one block.
__global__ void k_struct_weights(const double* __restrict__ ws, double2* __restrict__ wr, double* __restrict__ out,
                                 int W) {
    __shared__ double shm[32];
    __shared__ double2 shc[32];
    const int tid = threadIdx.x, nt = blockDim.x;
    double m = -INFINITY;
    for (int i = tid; i < W; i += nt) {
        const double* s = ws + (long)WSTRIDE * i;
        if (s[2] > 0.5 && isfinite(s[0]) && s[0] > m) m = s[0];
    }
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
    if ((tid & 31) == 0) shm[tid >> 5] = m;
    __syncthreads();
    double ref = shm[0];
    for (int i = 1; i < (nt + 31) / 32; ++i) ref = fmax(ref, shm[i]);
    __syncthreads();
    double2 sum = make_double2(0.0, 0.0);
    double nal = 0.0;
    for (int i = tid; i < W; i += nt) {
        const double* s = ws + (long)WSTRIDE * i;
        double2 v = make_double2(0.0, 0.0);
        if (s[2] > 0.5 && isfinite(s[0])) {
            const double mag = exp(s[0] - ref);
            v = make_double2(mag * cos(s[1]), mag * sin(s[1]));
            nal += 1.0;
        }
        wr[i] = v;
        sum = sum + v;
    }
    for (int o = 16; o > 0; o >>= 1) {
        sum.x += __shfl_down_sync(0xffffffffu, sum.x, o);
        sum.y += __shfl_down_sync(0xffffffffu, sum.y, o);
        nal += __shfl_down_sync(0xffffffffu, nal, o);
    }
    if ((tid & 31) == 0) {
        shc[tid >> 5] = sum;
        shm[tid >> 5] = nal;
    }
    __syncthreads();
    if (tid == 0) {
        double2 t = shc[0];
        double n = shm[0];
        for (int i = 1; i < (nt + 31) / 32; ++i) {
            t = t + shc[i];
            n += shm[i];
        }
        out[0] = t.x;
        out[1] = t.y;
        out[2] = ref;
        out[3] = n;
    }
}

// sum_w w <rho(Q) rho(-Q)>_w for every slot (thread per slot).
__global__ void k_struct_reduce(const double2* __restrict__ wr, const double2* __restrict__ pw,
                                double* __restrict__ out, int W, int nq) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nq) return;
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll 8
    for (int w = 0; w < W; ++w) acc = cfma(wr[w], pw[(long)w * nq + j], acc);
    out[4 + 2 * j] = acc.x;
    out[5 + 2 * j] = acc.y;
}

}  // namespace

cudaError_t launch_structure_factor(ftq_ctx* c, double* per_walker_out) {
    const int W = c->W, nslot = c->nslot, nq = nslot - 1;
    cudaError_t e = cudaSuccess;
    if (!c->sq_walker) {
        e = cudaMalloc(&c->sq_walker, sizeof(double2) * (size_t)W * nq);
        if (e == cudaSuccess) e = cudaMalloc(&c->sq_w, sizeof(double2) * (size_t)W);
        if (e == cudaSuccess) e = cudaMalloc(&c->sq_out, sizeof(double) * (4 + 2 * (size_t)nq));
        if (e != cudaSuccess) return e;
    }
    if (!c->g64_valid) {
        e = mixed_sync_g64(c);
        if (e != cudaSuccess) return e;
    }
    {
        // enough 512-thread blocks for four rounds of two per SM
        int dev = 0, sms = 1;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const int nqh = nq / 2, whole = c->sq_whole, half = c->sq_half;
        const int tasks = whole + (half - whole + 1) / 2 + (nqh - half + 3) / 4;
        const int per = std::max(1, std::min((8 * sms + W - 1) / W, (tasks + 15) / 16));
        LaunchScope ls(c, FTQ_K_ESTIMATORS);
        c->launches[FTQ_K_ESTIMATORS] += 1;
        launch_transpose_g(c, c->G, c->work);
        const size_t MM = (size_t)c->M * c->M;
        walker_spans(W, [&](size_t w0, int n) {
            k_structure<<<dim3((unsigned)per, (unsigned)n), 512, 0, c->stream>>>(
                c->G + MM * w0, c->work + MM * w0, c->tab.pair_ptr, c->tab.pair_a, c->tab.pair_b,
                c->sq_walker + w0 * nq, c->M, nqh, whole, half);
        });
    }
    {
        LaunchScope ls(c, FTQ_K_ESTIMATORS);
        k_struct_weights<<<1, 256, 0, c->stream>>>(c->wstate, c->sq_w, c->sq_out, W);
    }
    {
        LaunchScope ls(c, FTQ_K_ESTIMATORS);
        k_struct_reduce<<<(nq + 127) / 128, 128, 0, c->stream>>>(c->sq_w, c->sq_walker, c->sq_out, W, nq);
    }
    e = cudaGetLastError();
    if (e == cudaSuccess && per_walker_out)
        e = cudaMemcpyAsync(per_walker_out, c->sq_walker, sizeof(double2) * (size_t)W * nq, cudaMemcpyDeviceToDevice,
                            c->stream);
    return e;
}

}  // namespace ftq
