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

// P_ab = <a+_a a_b> = delta_ab - G_ba
__device__ __forceinline__ double2 pel_s(const double2* Gw, int M, int a, int b) {
    const double2 g = Gw[(size_t)b * M + a];
    return make_double2((a == b ? 1.0 : 0.0) - g.x, -g.y);
}

__device__ __forceinline__ double2 warp_total(double2 v) {
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
}

// A warp per walker and half-space transfer q (slots 1 + 2 q and 2 + 2 q, whose
// pairs are each other's reversed): rho and D of both, and Lambda once, since
// Lambda_-Q = Lambda_Q.  The short transfers have the most pairs and come first;
// the warps of a walker's blocks take them in turn.  The FP64 pipe bounds it (four
// DFMA per exchange term).
__global__ void __launch_bounds__(512) k_structure(const double2* __restrict__ G, const double2* __restrict__ Gtr,
                                                  const int* __restrict__ pptr, const int* __restrict__ pa,
                                                  const int* __restrict__ pb, double2* __restrict__ out, int M,
                                                  int nqh) {
    const int w = blockIdx.y, lane = threadIdx.x & 31;
    const int warp = blockIdx.x + gridDim.x * (threadIdx.x >> 5), nw = gridDim.x * (blockDim.x >> 5);
    const double2* Gw = G + (size_t)w * M * M;
    const double2* Gt = Gtr + (size_t)w * M * M;
    for (int q = warp; q < nqh; q += nw) {
        const int first = pptr[1 + 2 * q], end = pptr[2 + 2 * q];
        double2 rp = make_double2(0.0, 0.0), rm = rp, dp = rp, dm = rp, lam = rp;
        for (int e0 = first; e0 < end; e0 += 32) {
            const int e = e0 + lane;
            const bool on = e < end;
            const int a = on ? pa[e] : 0, d = on ? pb[e] : 0;
            const double2 x = exchange_unit<double2>(Gw, Gt, M, pa, pb, first, end, a, d);
            if (on) {
                lam = lam + x;
                rp = rp + pel_s(Gw, M, a, d);
                rm = rm + pel_s(Gw, M, d, a);
                dp = dp + pel_s(Gw, M, a, a);
                dm = dm + pel_s(Gw, M, d, d);
            }
        }
        lam = warp_total(lam);
        rp = warp_total(rp);
        rm = warp_total(rm);
        dp = warp_total(dp);
        dm = warp_total(dm);
        if (lane == 0) {
            const double2 g = cmul(rp * 2.0, rm * 2.0) - lam * 2.0;
            out[((size_t)w * nqh + q) * 2] = g + dp * 2.0;
            out[((size_t)w * nqh + q) * 2 + 1] = g + dm * 2.0;
        }
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
        // enough 512-thread blocks for four rounds of two per SM (M = 257, 128 walkers: one 256-thread
        // block per walker with both signs of Q summed took 14.6 ms)
        int dev = 0, sms = 1;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const int per = std::max(1, std::min((8 * sms + W - 1) / W, (nq / 2 + 15) / 16));
        LaunchScope ls(c, FTQ_K_ESTIMATORS);
        c->launches[FTQ_K_ESTIMATORS] += 1;
        launch_transpose_g(c, c->G, c->work);
        const size_t MM = (size_t)c->M * c->M;
        walker_spans(W, [&](size_t w0, int n) {
            k_structure<<<dim3((unsigned)per, (unsigned)n), 512, 0, c->stream>>>(
                c->G + MM * w0, c->work + MM * w0, c->tab.pair_ptr, c->tab.pair_a, c->tab.pair_b,
                c->sq_walker + w0 * nq, c->M, nq / 2);
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
