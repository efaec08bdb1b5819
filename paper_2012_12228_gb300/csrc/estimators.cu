// UEG estimators (Sec. "Uniform Electron Gas", local energy; Results, the
// time-slice estimates and their average).
//
// Per walker, from P = I - G^T:
//   N = 2 tr P,  E_1 = sum_K |K|^2 P_KK,  rho_Q = sum_{K} P_{K+Q,K},
//   E_2 = sum_q 4 v_q rho_q rho_-q - sum_Q v_Q Lambda_Q,
//   Lambda_Q = sum over the pairs (a, d), (b, c) of transfer Q of P_ab P_cd.
// Lambda_-Q = Lambda_Q (the pairs of -Q are those of +Q reversed, and the sum
// is the trace of a product of two gathered blocks, tr(XY) = tr(YX)), so only
// the half-space transfers are summed and counted twice.
//
// k_est_walkers: persistent blocks over walkers or over equal parts of them (est_parts; a
// walker's G stays in L2 while it is worked on); a warp per slot for rho; for Lambda a warp
// per work unit = 32 consecutive pairs (a, d) of one +Q transfer (one per
// lane), looping over all pairs (b, c) of that transfer (exchange.cuh): G[b][a]
// is read from row b of G and G[d][c] from row c of G^T (written by
// k_transpose_g), so the 32 lanes of a load touch neighbouring columns of
// one row, which needs few sectors; the deltas of P are added once per pair.  With FP32 G
// each lane accumulates v_Q times its partial sum as a compensated float
// pair (two-sum), so no FP64 instruction runs per unit; with complex128 G the
// products and sums are FP64 (the FP64 pipe bounds that variant).
// T = double2 reads a complex128 G; T = float2 the FP32 G of the mixed
// path's slices.
#include <algorithm>
#include <cmath>

#include "block_reduce.cuh"
#include "complex_math.cuh"
#include "exchange.cuh"
#include "ftq_internal.h"

namespace ftq {
namespace {

__device__ __forceinline__ double2 to_d(double2 v) { return v; }
__device__ __forceinline__ double2 to_d(float2 v) { return make_double2(v.x, v.y); }

// P_ab = delta_ab - G_ba in the arithmetic of T
__device__ __forceinline__ double2 pel(const double2* Gw, int M, int a, int b) {
    const double2 g = Gw[(long)b * M + a];
    return make_double2((a == b ? 1.0 : 0.0) - g.x, -g.y);
}
__device__ __forceinline__ float2 pel(const float2* Gw, int M, int a, int b) {
    const float2 g = Gw[(long)b * M + a];
    return make_float2((a == b ? 1.f : 0.f) - g.x, -g.y);
}

// Gt[w] = G[w]^T through 32 x 33 shared tiles; grid (tiles, tiles, W).
template <typename T>
__global__ void k_transpose_g(const T* __restrict__ G, T* __restrict__ Gt, int M) {
    __shared__ T tile[32][33];
    const size_t off = (size_t)blockIdx.z * M * M;
    const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int i = r0 + r, j = c0 + threadIdx.x;
        if (i < M && j < M) tile[r][threadIdx.x] = G[off + (size_t)i * M + j];
    }
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int j = c0 + r, i = r0 + threadIdx.x;
        if (i < M && j < M) Gt[off + (size_t)j * M + i] = tile[threadIdx.x][r];
    }
}

__device__ __forceinline__ double2 warp_sum_d(double2 v) {
    for (int o = 16; o > 0; o >>= 1) v = v + shfl_down(v, o);
    return v;
}

template <typename T>
__global__ void __launch_bounds__(1024) k_est_walkers(const T* __restrict__ G, const T* __restrict__ Gtr,
                                                     const double* __restrict__ ws,
                                                    double* __restrict__ est, const int* __restrict__ pptr,
                                                    const int* __restrict__ pa, const int* __restrict__ pb,
                                                    const uint16_t* __restrict__ vidx, const int4* __restrict__ units,
                                                    int nunits, const double* __restrict__ vq,
                                                    const float2* __restrict__ vqf,
                                                    const double* __restrict__ ksq, int M, int nqh, double E_M,
                                                    int W, int nparts, double* __restrict__ parts) {
    extern __shared__ unsigned char smem_raw[];
    double2* rho = reinterpret_cast<double2*>(smem_raw);     // [2 nqh + 1]
    __shared__ double2 shc[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int item = blockIdx.x; item < W * nparts; item += gridDim.x) {
        const int w = item / nparts, part = item % nparts;
        const T* Gw = G + (size_t)w * M * M;
        const T* Gt = Gtr + (size_t)w * M * M;
        // both slots of every nparts-th transfer (the sums over a alone are the first part's)
        for (int s = warp; part + (s >> 1) * nparts < nqh; s += nw) {
            const int sl = 1 + 2 * (part + (s >> 1) * nparts) + (s & 1);
            double2 r = make_double2(0.0, 0.0);
            for (int e = pptr[sl] + lane; e < pptr[sl + 1]; e += 32) r = r + to_d(pel(Gw, M, pa[e], pb[e]));
            r = warp_sum_d(r);
            if (lane == 0) rho[sl] = r;
        }
        __syncthreads();
        double2 nsum = make_double2(0.0, 0.0), e1 = nsum, e2 = nsum, ex = nsum;
        // FP32 G: v_Q acc accumulated per lane as a compensated float sum
        // (hi + lo, two-sum), so that no FP64 instruction runs per pair
        float exh[2] = {0.f, 0.f}, exl[2] = {0.f, 0.f};
        for (int a = threadIdx.x; a < M && part == 0; a += blockDim.x) {
            const double2 p = to_d(pel(Gw, M, a, a));
            nsum = nsum + p * 2.0;
            e1 = e1 + p * ksq[a];
        }
        for (int q = part + (int)threadIdx.x * nparts; q < nqh; q += blockDim.x * nparts)
            e2 = e2 + cmul(rho[1 + 2 * q], rho[2 + 2 * q]) * (4.0 * vq[q]);
        // The units shorten along the list: with complex128 G every other round of the warps of all
        // parts runs backwards, so that each warp, and with it each part, gets about the same work
        // (M = 171, one block per walker: 2.13 -> 1.38 ms).  FP32 G goes forwards only: the caches
        // bound it, not the longest warp (M = 257, 1024 walkers 8.36 ms, 8.62 with turns).
        const int round = nw * nparts, t = warp * nparts + part;
        for (int u0 = 0, back = 0; u0 < nunits; u0 += round, back ^= 1) {
            const int u = u0 + (sizeof(T) == sizeof(double2) && back ? round - 1 - t : t);
            if (u >= nunits) continue;
            const int4 un = units[u];                  // slot pairs [x, y), chunk from z, v_Q index w
            const int f = un.z + lane;
            const bool on = f < un.y;
            const T acc = exchange_unit<T>(Gw, Gt, M, pa, pb, un.x, un.y, on ? pa[f] : 0, on ? pb[f] : 0);
            if (!on) continue;
            const int qi = un.w;
            if constexpr (sizeof(T) == sizeof(float2)) {
                const float2 v = vqf[qi];
                const float av[2] = {(float)acc.x, (float)acc.y};
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const float pp = av[r] * v.x;
                    float ee = fmaf(av[r], v.x, -pp);
                    ee = fmaf(av[r], v.y, ee);
                    const float sum = exh[r] + pp;
                    const float bb = sum - exh[r];
                    exl[r] += ((exh[r] - (sum - bb)) + (pp - bb)) + ee;
                    exh[r] = sum;
                }
            } else {
                ex = ex + to_d(acc) * vq[qi];
            }
        }
        if constexpr (sizeof(T) == sizeof(float2))
            ex = make_double2((double)exh[0] + (double)exl[0], (double)exh[1] + (double)exl[1]);
        e2 = e2 - ex * 2.0;
        nsum = block_sum(nsum, shc);
        e1 = block_sum(e1, shc);
        e2 = block_sum(e2, shc);
        if (threadIdx.x == 0 && nparts > 1) {
            double* o = parts + 6 * (size_t)item;
            o[0] = e1.x; o[1] = e1.y; o[2] = e2.x; o[3] = e2.y; o[4] = nsum.x; o[5] = nsum.y;
        } else if (threadIdx.x == 0) {
            const double* s = ws + (long)WSTRIDE * w;
            double* o = est + (long)WSTRIDE * w;
            o[0] = s[0]; o[1] = s[1]; o[2] = s[2];
            o[3] = E_M + e1.x + e2.x; o[4] = e1.y + e2.y;
            o[5] = nsum.x; o[6] = nsum.y; o[7] = 0.0;
        }
    }
}

// The parts of every walker summed in order.
__global__ void k_est_combine(const double* __restrict__ parts, const double* __restrict__ ws,
                              double* __restrict__ est, int W, int nparts, double E_M) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= W) return;
    double v[6] = {};
    for (int q = 0; q < nparts; ++q)
        for (int k = 0; k < 6; ++k) v[k] += parts[6 * ((size_t)w * nparts + q) + k];
    const double* s = ws + (long)WSTRIDE * w;
    double* o = est + (long)WSTRIDE * w;
    o[0] = s[0]; o[1] = s[1]; o[2] = s[2];
    o[3] = E_M + v[0] + v[2]; o[4] = v[1] + v[3];
    o[5] = v[4]; o[6] = v[5]; o[7] = 0.0;
}

// sum_w of w, wE, wN with w = exp(ln|w| - s) e^{i arg w}, s = max ln|w| over
// the alive walkers with a finite ln|w| (the others weigh 0); writes
// {Re, Im sum w, Re, Im sum wE, Re, Im sum wN, s, alive} to out, and when
// rec is given also {k, E_k, N_k, alive, Re sum w, s} to rec.
__global__ void k_reduce_walkers(const double* __restrict__ est, double* __restrict__ out, int W,
                                 double* __restrict__ rec, int k) {
    __shared__ double shv[32];
    __shared__ int shi[32];
    __shared__ double2 shc[32];
    double best = -INFINITY;
    int bi = W;
    for (int w = threadIdx.x; w < W; w += blockDim.x)
        if (est[(long)WSTRIDE * w + 2] > 0.5 && isfinite(est[(long)WSTRIDE * w]) && est[(long)WSTRIDE * w] > best) {
            best = est[(long)WSTRIDE * w];
            bi = w;
        }
    int wm = block_argmax(best, bi, shv, shi);
    double s = wm < W ? est[(long)WSTRIDE * wm] : 0.0;
    double2 sw = make_double2(0.0, 0.0), swe = sw, swn = sw;
    double nal = 0.0;
    for (int w = threadIdx.x; w < W; w += blockDim.x) {
        const double* o = est + (long)WSTRIDE * w;
        if (o[2] <= 0.5 || !isfinite(o[0])) continue;     // a non-finite ln|w| weighs 0
        double m = exp(o[0] - s);
        double2 ww = make_double2(m * cos(o[1]), m * sin(o[1]));
        sw = sw + ww;
        swe = swe + cmul(ww, make_double2(o[3], o[4]));
        swn = swn + cmul(ww, make_double2(o[5], o[6]));
        nal += 1.0;
    }
    sw = block_sum(sw, shc);
    swe = block_sum(swe, shc);
    swn = block_sum(swn, shc);
    nal = block_sum(nal, shv);
    if (threadIdx.x == 0) {
        out[0] = sw.x; out[1] = sw.y; out[2] = swe.x; out[3] = swe.y;
        out[4] = swn.x; out[5] = swn.y; out[6] = s; out[7] = nal;
        if (rec) {
            const double2 E = nal > 0.0 ? cdiv(swe, sw) : make_double2(NAN, NAN);
            const double2 N = nal > 0.0 ? cdiv(swn, sw) : make_double2(NAN, NAN);
            rec[0] = (double)k; rec[1] = E.x; rec[2] = E.y; rec[3] = N.x; rec[4] = N.y;
            rec[5] = nal; rec[6] = sw.x; rec[7] = s;
        }
    }
}

// Row 0 of the slice summary: the number of recorded slices and the averages
// of their global estimates (each slice counts once); rows 1.. the records.
__global__ void k_slice_summary(const double* __restrict__ rec, int n, double* __restrict__ out, int rows) {
    __shared__ double2 shc[32];
    double2 e = make_double2(0.0, 0.0), nn = e;
    for (int r = threadIdx.x; r < n; r += blockDim.x) {
        e = e + make_double2(rec[8 * r + 1], rec[8 * r + 2]);
        nn = nn + make_double2(rec[8 * r + 3], rec[8 * r + 4]);
    }
    e = block_sum(e, shc);
    nn = block_sum(nn, shc);
    if (threadIdx.x == 0) {
        const double inv = n > 0 ? 1.0 / n : NAN;
        out[0] = (double)n;
        out[1] = e.x * inv; out[2] = e.y * inv; out[3] = nn.x * inv; out[4] = nn.y * inv;
        out[5] = out[6] = out[7] = 0.0;
    }
    for (int i = threadIdx.x; i < 8 * rows; i += blockDim.x) out[8 + i] = rec[i];
}

template <typename T>
void transpose_g(ftq_ctx* c, const T* G, T* Gt) {
    const unsigned tiles = (unsigned)((c->M + 31) / 32);
    const size_t MM = (size_t)c->M * c->M;
    walker_spans(c->W, [&](size_t w0, int n) {
        k_transpose_g<T><<<dim3(tiles, tiles, (unsigned)n), dim3(32, 8), 0, c->stream>>>(G + MM * w0, Gt + MM * w0, c->M);
    });
}

// Parts of a walker: those that leave the least to the busiest SM.  Blocks take items in
// turn and neighbouring blocks share an SM, so its share is ceil(W n / blocks) items per
// block, each 1 / n of a walker and a fixed cost: 190 / M^2 of a walker's time for complex128
// G, 12 / M + 250 / M^2 for FP32 G.  A part has at least one unit for most warps.  Where the walkers under way read more than 300 MB, twice the L2 and
// more, fewer of them at a time are worth a quarter (complex128, M = 389, 152 walkers: 19.0 ms
// with one part, 11.5 with six).  A split that filled its rounds badly was slower than none:
// FP32, M = 57, 110 walkers in two parts 0.168 ms against 0.100 in one; complex128, M = 147,
// 152 walkers in eight parts 2.07 ms against 1.57 (now 1.00), M = 257, 128 walkers 5.09 (now
// 3.30 in seven parts).
int est_parts(int W, int M, int nunits, int nwarp, int sms, int per_sm, bool f32) {
    const double fixed = f32 ? 12.0 / M + 250.0 / ((double)M * M) : 190.0 / ((double)M * M);
    const double bytes = (f32 ? 16.0 : 32.0) * M * M;                  // G and G^T
    const int blocks = per_sm * sms;
    int best = 1;
    double low = 1e300;
    for (int n = 1; n <= EST_PARTS && (n - 1) * nwarp < nunits; ++n) {
        const long long items = (long long)W * n;
        const double rounds = (double)((items + blocks - 1) / blocks) * (items <= sms ? 1 : per_sm);
        const double walkers = std::min((double)W, (double)blocks / n);
        const double cost = rounds / n * (1.0 + n * fixed) * (walkers * bytes > 300e6 ? 1.25 : 1.0);
        if (cost < low) { low = cost; best = n; }
    }
    return best;
}

template <typename T>
cudaError_t launch_est_walkers(ftq_ctx* c, const T* G) {
    const int nqh = c->sys.nq_half;
    const int M = c->M;
    const size_t sm = sizeof(double2) * (2 * nqh + 1);
    if (sm > 220 * 1024) return cudaErrorInvalidValue;      // the transfer table alone is too large
    static size_t sm_set[2] = {48 * 1024, 48 * 1024};
    const bool f32 = sizeof(T) == sizeof(float2);
    const int which = f32 ? 1 : 0;
    if (sm > sm_set[which]) {
        cudaError_t e = cudaFuncSetAttribute(k_est_walkers<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
        sm_set[which] = sm;
    }
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // FP32 G: one 1024-thread block per SM, so that fewer walkers compete for
    // the L2; complex128 G (FP64-pipe bound): two 512-thread blocks per SM
    const int nthr = f32 ? 1024 : 512;
    const int per_sm = f32 ? 1 : 2;
    const int nparts = est_parts(c->W, M, c->tab.neplus, nthr / 32, sms, per_sm, f32);
    const int grid = c->W * nparts < per_sm * sms ? c->W * nparts : per_sm * sms;
    LaunchScope ls(c, FTQ_K_ESTIMATORS);
    // G^T into the complex128 work buffer (scratch between calls; it holds a
    // complex128 or a complex64 matrix per walker)
    T* Gt = reinterpret_cast<T*>(c->work);
    transpose_g(c, G, Gt);
    c->launches[FTQ_K_ESTIMATORS] += 1;
    k_est_walkers<T><<<grid, nthr, sm, c->stream>>>(G, Gt, c->wstate, c->est, c->tab.pair_ptr, c->tab.pair_a,
                                                    c->tab.pair_b, c->tab.vidx, c->tab.eplus, c->tab.neplus,
                                                    c->tab.vq, c->tab.vqf, c->tab.ksq, M, nqh, c->sys.E_M, c->W,
                                                    nparts, c->est_parts);
    if (nparts > 1) {
        c->launches[FTQ_K_ESTIMATORS] += 1;
        k_est_combine<<<(c->W + 127) / 128, 128, 0, c->stream>>>(c->est_parts, c->wstate, c->est, c->W, nparts,
                                                              c->sys.E_M);
    }
    return cudaGetLastError();
}

}  // namespace

void launch_transpose_g(ftq_ctx* c, const double2* G, double2* Gt) { transpose_g(c, G, Gt); }

cudaError_t launch_estimators(ftq_ctx* c, double* per_walker) {
    if (!c->g64_valid) {
        cudaError_t e0 = mixed_sync_g64(c);
        if (e0 != cudaSuccess) return e0;
    }
    cudaError_t e = launch_est_walkers(c, c->G);
    if (e != cudaSuccess) return e;
    c->launches[FTQ_K_ESTIMATORS] += 1;
    k_reduce_walkers<<<1, 256, 0, c->stream>>>(c->est, c->red, c->W, nullptr, 0);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (per_walker)
        e = cudaMemcpy2DAsync(per_walker, sizeof(double) * 8, c->est, sizeof(double) * WSTRIDE, sizeof(double) * 8,
                              c->W, cudaMemcpyDeviceToDevice, c->stream);
    return e;
}

cudaError_t launch_slice_estimate(ftq_ctx* c, int k) {
    if (c->trk_n >= c->sys.n_slices) return cudaErrorInvalidValue;
    // the mixed path holds G(tau_k) in FP32 for k < n and in complex128 at tau = beta
    cudaError_t e = c->g64_valid ? launch_est_walkers(c, c->G) : launch_est_walkers(c, c->G32);
    if (e != cudaSuccess) return e;
    c->launches[FTQ_K_ESTIMATORS] += 1;
    k_reduce_walkers<<<1, 256, 0, c->stream>>>(c->est, c->red, c->W, c->trk + 8 * (size_t)c->trk_n, k);
    c->trk_n += 1;
    return cudaGetLastError();
}

cudaError_t launch_slice_summary(ftq_ctx* c, double* out_dev, int rows) {
    k_slice_summary<<<1, 256, 0, c->stream>>>(c->trk, c->trk_n, out_dev, rows);
    c->launches[FTQ_K_ESTIMATORS] += 1;
    return cudaGetLastError();
}

}  // namespace ftq
