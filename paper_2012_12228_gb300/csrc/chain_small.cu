// The mixed-precision chain of small bases (M <= 64): all Horner steps of a slice
// in one launch, a walker's V and chain staying in shared memory.
//
// With M <= 64 the real-embedded V (128 rows x 2 Kp, 3xTF32 hi and lo) and the
// chain (NT >= M columns x 2 Kp, hi and lo) fit together, 192 KB at M = 57.  A
// persistent block takes a walker at a time: it generates V's tiles and the scaled
// chain h Y once, then alternates the MMAs of a Horner step (tcgen05 kind::tf32)
// with an epilogue that reads TMEM, adds the U term kept in registers and writes the
// next operand, hi and lo, back to shared memory; planes go to memory after the
// last step only.  The hi * hi products and the cross terms have accumulators of
// their own: a tensor-core addition truncates, and the main sum then takes a third of
// the additions (over the 87 slices of the M = 57 path the drift of the particle
// number falls from 9e-6 to 3e-6 electrons).
//
// What bounded the launch per Horner step was latency: an item of four k tiles, one
// block per SM, 55 us a step at M = 57, 640 walkers for 17 us of traffic.  Here it is the
// epilogue's instructions (2.9 us a step), so a thread has a quarter of a row's
// columns (with half, 4.1 us).  Measured per slice (six steps), before and now: M = 57,
// 640 walkers 335 and 136 us, 64 walkers 113 and 31 us; M = 33, 300 walkers 137 and 45 us;
// M = 7, 64 walkers 62 and 19 us.
#include <algorithm>

#include "complex_math.cuh"
#include "ftq_internal.h"
#include "mixed_common.cuh"
#include "tc_common.cuh"

namespace ftq {
namespace {

using namespace tc;

constexpr int SNT = 512;             // threads: TMEM quadrant = warp & 3, column quarter = warp >> 2
constexpr int SW = SNT / 32;
constexpr int SR = 64 / SW;          // rows of V a warp generates
constexpr int ATILE = 128 * 128;     // bytes of one k tile (32 floats) of V, hi or lo

struct SmallArgs {
    float *Y, *Yf;                   // planes (hi, lo) and the single FP32 plane, in place
    const float2* phi;               // field table [W][nslot]
    const uint16_t* vidx;            // [M][M]
    const float2* h;                 // kinetic half step as float pairs
    int* status;
    int W, M, Kp, LD, NT, nslot, p;
    long long wait_limit;
};

__global__ void __launch_bounds__(SNT, 1) k_chain_slice(const SmallArgs a) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint64_t bar;
    __shared__ uint32_t tmem_sh;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t pad = (1024u - (smem_u32(smem_raw) & 1023u)) & 1023u;
    unsigned char* A = smem_raw + pad;
    const int KT = 2 * a.Kp / 32;                            // k tiles
    const int btile = a.NT * 128;                            // bytes of one k tile of the chain, hi or lo
    unsigned char* B = A + (size_t)KT * 2 * ATILE;
    float2* phs = reinterpret_cast<float2*>(B + (size_t)KT * 2 * btile);
    const uint32_t tcols = 2 * a.NT <= 32 ? 32u : (2 * a.NT <= 64 ? 64u : 128u);
    if (tid == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(&tmem_sh, tcols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_sh;

    const int quad = warp & 3, quarter = warp >> 2;
    const int r = quad * 32 + lane, part = r >> 6, i = r & 63;   // accumulator row
    const int nc = a.NT / 4, c0 = quarter * nc;                  // this thread's columns (4, 8, 12 or 16)
    const size_t rowlen = 2 * (size_t)a.Kp, plane = (size_t)a.LD * rowlen;
    const bool row_ok = i < a.M;
    const ScaleF hi_(row_ok ? a.h[i] : make_float2(0.f, 0.f));
    const uint32_t idesc = idesc_tf32(a.NT), idesc2 = idesc_tf32(2 * a.NT);
    const int kx = part * a.Kp + i;                              // this row's place along the next operand's k
    // slots of V's entries that this thread generates (the same for every walker)
    uint16_t slot[4][SR];
#pragma unroll
    for (int kt = 0; kt < 4; ++kt)
#pragma unroll
        for (int t = 0; t < SR; ++t) {
            const int k = kt * 32 + lane, kc = k >= a.Kp ? k - a.Kp : k, ir = warp + SW * t;
            slot[kt][t] = ir < a.M && kc < a.M ? a.vidx[ir * a.M + kc] : 0;
        }
    uint32_t phase = 0;
    bool ok = true;
    for (int w = blockIdx.x; w < a.W && ok; w += gridDim.x) {
        const float2* ph = a.phi + (size_t)w * a.nslot;
        float* Yw = a.Y + 2 * plane * w;
        float* Fw = a.Yf + plane * w;
        __syncthreads();                                     // the previous walker is done with the table
        for (int s = tid; s < a.nslot; s += SNT) phs[s] = ph[s];
        // the chain, scaled: rows c of [Re | Im]; eight loads of a thread at a time (the
        // compiler keeps a load behind an earlier store to shared memory)
        for (int e0 = warp; e0 < a.NT * KT; e0 += 8 * SW) {
            float y[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int e = e0 + q * SW, c = e / KT, k = (e - c * KT) * 32 + lane;
                const int ii = k >= a.Kp ? k - a.Kp : k;
                y[q] = e < a.NT * KT && c < a.M && ii < a.M ? ScaleF(a.h[ii])(Fw[(size_t)c * rowlen + k]) : 0.f;
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int e = e0 + q * SW, c = e / KT, kt = e - c * KT;
                if (e >= a.NT * KT) break;
                float hh, ll;
                split_tf32(y[q], hh, ll);
                unsigned char* b = B + (size_t)kt * 2 * btile + sw128_off(c, lane);
                *reinterpret_cast<float*>(b) = hh;
                *reinterpret_cast<float*>(b + btile) = ll;
            }
        }
        // the U term h Y of this thread's row and columns
        float u[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const int c = c0 + q;
            u[q] = q < nc && row_ok && c < a.M ? hi_(Fw[(size_t)c * rowlen + kx]) : 0.f;
        }
        __syncthreads();
        // V: rows [Re C (64); Im C (64)], k over [Re Z | Im Z]
#pragma unroll
        for (int kt = 0; kt < 4; ++kt) {
            if (kt >= KT) break;
            const int k = kt * 32 + lane;
            const bool im = k >= a.Kp;
            const int kc = im ? k - a.Kp : k;
            unsigned char* Ah = A + (size_t)kt * 2 * ATILE;
            float2 vv[SR];
#pragma unroll
            for (int t = 0; t < SR; ++t) {
                const int ir = warp + SW * t;
                vv[t] = make_float2(0.f, 0.f);
                if (ir < a.M && kc < a.M) vv[t] = phs[slot[kt][t]];
            }
#pragma unroll
            for (int t = 0; t < SR; ++t) {
                const int ir = warp + SW * t;
                const float2 v = vv[t];
                float hh, ll;
                split_tf32(im ? -v.y : v.x, hh, ll);
                uint32_t o = sw128_off(ir, lane);
                *reinterpret_cast<float*>(Ah + o) = hh;
                *reinterpret_cast<float*>(Ah + ATILE + o) = ll;
                split_tf32(im ? v.x : v.y, hh, ll);
                o += 64 * 128;
                *reinterpret_cast<float*>(Ah + o) = hh;
                *reinterpret_cast<float*>(Ah + ATILE + o) = ll;
            }
        }
        for (int j = a.p; j >= 1 && ok; --j) {
            tc_fence_before();
            fence_async_smem();
            __syncthreads();
            if (tid == 0) {
                tc_fence_after();
                // V_hi times [Z_hi; Z_lo] (rows of one tile) lands on [main | cross], V_lo Z_hi on cross
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    for (int kt = 0; kt < KT; ++kt) {
                        const uint64_t dk = (uint64_t)(2 * k);
                        const uint64_t ah = sdesc_sw128(A + (size_t)kt * 2 * ATILE) + dk;
                        const uint64_t al = sdesc_sw128(A + (size_t)kt * 2 * ATILE + ATILE) + dk;
                        const uint64_t bh = sdesc_sw128(B + (size_t)kt * 2 * btile) + dk;
                        mma_tf32(tmem, ah, bh, idesc2, kt > 0 || k > 0 ? 1u : 0u);
                        mma_tf32(tmem + a.NT, al, bh, idesc, 1u);
                    }
                mma_commit(&bar);
            }
            ok = __syncthreads_and(mbar_wait(&bar, phase, a.wait_limit) ? 1 : 0) != 0;
            if (!ok) break;
            phase ^= 1u;
            tc_fence_after();
            const float alpha = 1.0f / j;
            const uint32_t acc = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)c0;
            uint32_t m[16], x[16];
#pragma unroll
            for (int cc = 0; cc < 16; cc += 4)
                if (cc < nc) {
                    tmem_ld4(acc + cc, m + cc);
                    tmem_ld4(acc + a.NT + cc, x + cc);
                }
            tmem_wait_ld();
            asm volatile("" : "+r"(m[0]), "+r"(m[1]), "+r"(m[2]), "+r"(m[3]), "+r"(m[4]), "+r"(m[5]), "+r"(m[6]), "+r"(m[7]),
                         "+r"(m[8]), "+r"(m[9]), "+r"(m[10]), "+r"(m[11]), "+r"(m[12]), "+r"(m[13]), "+r"(m[14]), "+r"(m[15]));
            asm volatile("" : "+r"(x[0]), "+r"(x[1]), "+r"(x[2]), "+r"(x[3]), "+r"(x[4]), "+r"(x[5]), "+r"(x[6]), "+r"(x[7]),
                         "+r"(x[8]), "+r"(x[9]), "+r"(x[10]), "+r"(x[11]), "+r"(x[12]), "+r"(x[13]), "+r"(x[14]), "+r"(x[15]));
            if (j > 1) {
                // padded rows and columns come out as zeros; rows beyond Kp have no place
                if (i < a.Kp) {
                    unsigned char* bk = B + (size_t)(kx >> 5) * 2 * btile + (kx & 3) * 4;
                    const int ch = (kx >> 2) & 7;
#pragma unroll
                    for (int q = 0; q < 16; ++q)
                        if (q < nc) {
                            const int c = c0 + q;
                            float hh, ll;
                            split_tf32(fmaf(alpha, __uint_as_float(m[q]) + __uint_as_float(x[q]), u[q]), hh, ll);
                            unsigned char* b = bk + c * 128 + (((ch ^ c) & 7) << 4);    // sw128_off(c, kx & 31)
                            *reinterpret_cast<float*>(b) = hh;
                            *reinterpret_cast<float*>(b + btile) = ll;
                        }
                }
            } else if (row_ok) {
#pragma unroll
                for (int q = 0; q < 16; ++q)
                    if (q < nc && c0 + q < a.M) {
                        const float v = hi_(fmaf(alpha, __uint_as_float(m[q]) + __uint_as_float(x[q]), u[q]));
                        float hh, ll;
                        split_tf32(v, hh, ll);
                        const size_t o = (size_t)(c0 + q) * rowlen + kx;
                        Yw[o] = hh;
                        Yw[plane + o] = ll;
                        Fw[o] = v;
                    }
            }
        }
    }
    if (!ok && tid == 0) {
        atomicOr(a.status, 2);
        mbar_wait(&bar, phase);                              // the MMAs in flight end before TMEM is freed
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, tcols);
}

}  // namespace

bool chain_slice_fits(const ftq_ctx* c) {
    return c->M <= 64 && (c->opts.precision == FTQ_MIXED || c->opts.precision == FTQ_MIXED_F64UDT);
}

namespace {

cudaError_t launch_slice(ftq_ctx* c, const ftq_ctx* ruling, float* Y, float* Yf) {
    SmallArgs a;
    a.Y = Y;
    a.Yf = Yf;
    a.phi = c->phi32;
    a.vidx = c->tab.vidx;
    a.h = c->tab.hf;
    a.status = c->status;
    a.W = c->W;
    a.M = c->M;
    a.Kp = c->Kp;
    a.LD = c->LD;
    a.NT = (c->M + 15) / 16 * 16;
    a.nslot = c->nslot;
    a.p = c->opts.exp_order;
    a.wait_limit = ruling->wait_limit >= 0 ? (long long)ruling->wait_limit : TC_WAIT_LIMIT;
    const int KT = 2 * a.Kp / 32;
    const size_t sm = 1024 + (size_t)KT * 2 * (ATILE + a.NT * 128) + sizeof(float2) * a.nslot;
    cudaError_t e = cudaFuncSetAttribute(k_chain_slice, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 1, per_sm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_chain_slice, SNT, sm);
    per_sm = std::max(1, std::min(per_sm, 4));                // 128 TMEM columns at most each
    LaunchScope ls(c, FTQ_K_CHAIN);
    k_chain_slice<<<std::min(a.W, sms * per_sm), SNT, sm, c->stream>>>(a);
    return cudaGetLastError();
}

}  // namespace

// exp(V) and the kinetic factors of one slice applied to the mixed chain, in place.
// `ruling` sets the bounded waits: the context itself, or the batch it is a member of.
cudaError_t chain_slice(ftq_ctx* c, const ftq_ctx* ruling) { return launch_slice(c, ruling, c->Ypl, c->Yf); }

// Time of one Horner step, from slices of a copy of the chain in the Horner buffers (which
// small bases do not use otherwise).
cudaError_t chain_slice_time(ftq_ctx* c, float* ms) {
    const size_t plane = sizeof(float) * (size_t)c->W * c->LD * 2 * c->Kp;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaError_t e = cudaMemcpyAsync(c->zpl[1], c->Yf, plane, cudaMemcpyDeviceToDevice, c->stream);
    if (e == cudaSuccess) e = launch_slice(c, c, c->zpl[0], c->zpl[1]);      // warm-up
    if (e == cudaSuccess) e = cudaEventRecord(e0, c->stream);
    for (int r = 0; r < 3 && e == cudaSuccess; ++r) e = launch_slice(c, c, c->zpl[0], c->zpl[1]);
    if (e == cudaSuccess) e = cudaEventRecord(e1, c->stream);
    if (e == cudaSuccess) e = cudaEventSynchronize(e1);
    float t = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&t, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    *ms = t / (3.f * c->opts.exp_order);
    return e;
}

}  // namespace ftq
