// One Taylor-Horner step of exp(V) on the complex128 chain with the
// 5th-generation tensor cores: the product V Z of each step is formed exactly
// in pieces (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59, 2012) from bf16 digits with tcgen05.mma kind::f16, because
// the FP64 pipe of this part (2 FMA per clock and SM) is 2000 times slower than
// its bf16 tensor pipe.
//
// Digits.  V is scaled by one power of two per walker (its entries all come
// from the walker's field table phi), Z by one per column, to integers of 56
// and 57 bits, written in base 128 as d_0 .. d_7 with |d_j| <= 64 for j >= 1
// and |d_0| <= 128 (V) or 256 (Z): every digit is a bf16 number.  Products
// d_i(V) d_j(Z) of one level l = i + j <= 7 are summed in one FP32 accumulator:
// over at most 512 nonzero real terms (256 complex k) a level's sum stays at or below
// 32768 * 512 = 2^24 for l <= 3 (256 * 128 for l = 0; each further pair adds at
// most 64 * 64), so it is an exact integer.  From l = 4 on the worst case passes
// 2^24 by less than 2x, a rounding of one unit there is below 2^-52 of the
// largest possible sum.  Level sums are combined in 64-bit integers and one
// rounding to FP64.  What is dropped (l >= 8) and the digits' own rounding leave
// a normwise error of V Z of 2.6e-16 to 3e-16 on chains of M = 57 .. 257, below the
// 5e-16 to 8e-16 of an FP64 sum over k (both against a longer format).  The guarantee is
// normwise: an entry 2^-g below the largest of its column (V: of the walker's table) keeps
// 56 - g bits, fewer than FP64's 53 from g = 4 on.  On whole slices G is as close to an 80-bit
// evaluation as with FP64 sums (rms after six slices, M = 257: 1.5e-17 against 2.0e-17 at r_s = 1,
// 5.9e-18 against 8.9e-18 at r_s = 0.5, whose columns are graded most).
//
// Complex product as one real GEMM, as in the mixed chain: for 64 complex rows
// the MMA rows are [Re C ; Im C], a k tile of 16 complex k is [Zr (16) | Zi (16)],
// so its A tile is [[Vr, -Vi], [Vi, Vr]].  The B tiles of the eight digits
// (32 columns each) lie one after the other, so that A_i times the first 8 - i
// of them is ONE MMA with N = 32 (8 - i) that lands on the accumulators of the
// levels i .. 7: 8 MMAs for 36 digit products, at the full tensor rate instead
// of the A-bound one of N = 32.  256 TMEM columns per item, double-buffered.
//
// What bounds it: shared-memory bandwidth (M = 257, 152 walkers: LSU wavefronts 79% of peak beside
// the MMAs' own reads, tensor pipe 29%, DRAM 10%).  Per k tile (16 complex k) the MMAs read
// 136 KB and take 1152 cycles of the tensor pipe; the digits of A are written
// at 64 KB, those of B at 16 KB, and 1024 entries are gathered from the digit table.
// Measured against the tiled FP64 FMA kernel it replaced (74% of the FP64 pipe):
// one slice of six Horner steps at M = 257, 152 walkers 7.7 ms against 132 ms,
// M = 57, 256 walkers 0.46 against 2.8 ms, M = 33, 300 walkers 0.30 against 2.4 ms.
//
// Warps: 0..3 epilogue (TMEM lane quadrants), 4..11 digits of A (gathered from
// the walker's digit table in shared memory when it fits), 12..15 digits of B
// (from FP64 planes), 16 control.  Work item = (walker, 64-row block, 32-column
// tile).  Every wait is bounded; on expiry the kernel latches bit 2 of the
// status word, every role skips its remaining work, and TMEM is freed.
#include <algorithm>
#include <cmath>
#include <vector>

#include "complex_math.cuh"
#include "digits.cuh"
#include "ftq_internal.h"
#include "tc_common.cuh"

namespace ftq {
namespace {

using namespace tc;

constexpr int ND = 8;                       // digits
constexpr int OCT = 32;                     // columns of an item
constexpr int KC = 16;                      // complex k of a k tile
constexpr int ADIG = 128 * 64;              // bytes of one digit's A tile (128 rows x 64 bytes)
constexpr int BDIG = OCT * 64;              // bytes of one digit's B tile
constexpr int STAGE = ND * (ADIG + BDIG);   // 80 KB
constexpr int NSTAGE = 2;
constexpr int W_EPI = 4, W_A = 8, W_B = 4;
constexpr int NT_OZ = 32 * (W_EPI + W_A + W_B + 1);
constexpr int CHUNK_K = 256;                // complex k whose products one accumulator sums
// Planes of a complex128 chain matrix: column c of walker w at
// ((w M + c) 2 + part) Kp, rows contiguous.
struct OzArgs {
    const double* Zin;
    const double* U;
    double* out;                 // planes (nullable with outY)
    double2* outY;               // row-major complex128 (last step), nullable
    const uint4* dig;            // digit table [W][nslot][2]: 8 bf16 digits of Re, of Im
    const int* ev;               // biased exponent of max |phi| per walker
    const uint32_t* cin;         // per column: the largest high word of |Zin|
    uint32_t* cout;              // the same of the output (atomic max), nullable
    const uint16_t* vidx;        // padded slot table [64-row blocks][Kp]
    const double* os;            // row scale of the result, nullable
    const double* rank;          // per-walker rank (stride WSTRIDE), nullable
    int* status;
    double alpha;
    int M, Kp, nslot, nrb, nct, kt0, kt1, W;
    long long wait_limit;
};

__device__ __forceinline__ int item_of(int t, int per, int n, bool spread) {
    // consecutive items per CTA (the walker's table is loaded once), or, with
    // ranks, spread over the CTAs so that skipped tiles leave them balanced
    const int it = spread ? t * (int)gridDim.x + (int)blockIdx.x : (int)blockIdx.x * per + t;
    return it < n && (spread || t < per) ? it : -1;
}

__device__ __forceinline__ void a_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(32 * W_A) : "memory"); }

// TS: the walker's digit table is staged in shared memory
template <bool TS>
__global__ void __launch_bounds__(NT_OZ, 1) k_chain_oz(const OzArgs p) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint64_t full[NSTAGE], mma_bar[NSTAGE], tfull[2], tempty[2];
    __shared__ uint32_t tmem_sh;
    __shared__ volatile int abort_sh;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t pad = (1024u - (smem_u32(smem_raw) & 1023u)) & 1023u;
    unsigned char* base = smem_raw + pad;
    uint4* table = reinterpret_cast<uint4*>(base + (size_t)NSTAGE * STAGE);
    if (tid == 0) {
        for (int b = 0; b < NSTAGE; ++b) {
            mbar_init(&full[b], W_A + W_B);
            mbar_init(&mma_bar[b], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], W_EPI);
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
    const bool spread = p.rank != nullptr;
    const int per = (nitems + (int)gridDim.x - 1) / (int)gridDim.x;
    auto skipped = [&](int w, int c0) { return p.rank && c0 >= (int)p.rank[(long)WSTRIDE * w + 12]; };

    if (warp == W_EPI + W_A + W_B) {
        // ------------------------------------------------ control warp
        if (lane == 0) {
            int g = 0, li = 0, last = -1;
            bool ok = true;
            for (int t = 0, item; ok && (item = item_of(t, per, nitems, spread)) >= 0; ++t) {
                const int w = item / per_walker, tile = item % per_walker;
                if (skipped(w, (tile % p.nct) * OCT)) continue;
                const int bi = li & 1;
                const uint32_t acc = tmem + (uint32_t)(bi * ND * OCT);
                if (li >= 2) ok = mbar_wait_ab(&tempty[bi], (uint32_t)(((li - 2) >> 1) & 1), &abort_sh, p.status, p.wait_limit);
                for (int kt = p.kt0; kt < p.kt1 && ok; ++kt, ++g) {
                    const int s = g % NSTAGE;
                    ok = mbar_wait_ab(&full[s], (uint32_t)((g / NSTAGE) & 1), &abort_sh, p.status, p.wait_limit);
                    if (!ok) break;
                    tc_fence_after();
                    unsigned char* st = base + s * STAGE;
                    const uint64_t b0 = sdesc_sw64(st + ND * ADIG);
#pragma unroll
                    for (int k = 0; k < 2; ++k)          // 16 bf16 = 32 bytes along the row
#pragma unroll
                        for (int i = 0; i < ND; ++i)
                            mma_f16(acc + (uint32_t)(i * OCT), sdesc_sw64(st + i * ADIG) + (uint64_t)(2 * k),
                                    b0 + (uint64_t)(2 * k), idesc_bf16(OCT * (ND - i)),
                                    (kt > p.kt0 || k > 0 || i > 0) ? 1u : 0u);
                    mma_commit(&mma_bar[s]);
                    if (kt + 1 == p.kt1) mma_commit(&tfull[bi]);
                    last = g;
                }
                ++li;
            }
            // the MMAs end before TMEM is freed, whichever warp gave up (the epilogue's last wait covers them else)
            if (last >= 0) mbar_wait(&mma_bar[last % NSTAGE], (uint32_t)((last / NSTAGE) & 1));
        }
    } else if (warp >= W_EPI + W_A) {
        // ------------------------------------------------ digits of Z
        // column, group of 4 complex k (lanes 8..15 and 24..31 take the neighbour's, so that the 8-byte
        // stores of a half warp meet no bank twice)
        const int c = lane, kq = (warp - (W_EPI + W_A)) ^ ((lane >> 3) & 1);
        const uint32_t o_re = sw64_off(c, kq >> 1) + (uint32_t)(kq & 1) * 8u;
        const uint32_t o_im = sw64_off(c, 2 + (kq >> 1)) + (uint32_t)(kq & 1) * 8u;
        int g = 0;
        for (int t = 0, item; (item = item_of(t, per, nitems, spread)) >= 0; ++t) {
            const int w = item / per_walker, tile = item % per_walker;
            const int col0 = (tile % p.nct) * OCT;
            if (skipped(w, col0)) continue;
            const bool live = col0 + c < p.M;
            const double* zr = p.Zin + ((size_t)w * p.M + (live ? col0 + c : 0)) * 2 * p.Kp;
            const int E = live ? (int)(p.cin[(size_t)w * p.M + col0 + c] >> 20) : 0;
            double2 nr[2], ni[2];
            auto load = [&](int kt) {
                const int k = kt * KC + kq * 4;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    nr[h] = *reinterpret_cast<const double2*>(zr + k + 2 * h);
                    ni[h] = *reinterpret_cast<const double2*>(zr + p.Kp + k + 2 * h);
                }
            };
            load(p.kt0);
            for (int kt = p.kt0; kt < p.kt1; ++kt, ++g) {
                const int s = g % NSTAGE, k = kt * KC + kq * 4;
                const double vr[4] = {nr[0].x, nr[0].y, nr[1].x, nr[1].y};
                const double vi[4] = {ni[0].x, ni[0].y, ni[1].x, ni[1].y};
                if (kt + 1 < p.kt1) load(kt + 1);
                if (g >= NSTAGE &&
                    !mbar_wait_ab(&mma_bar[s], (uint32_t)((g / NSTAGE - 1) & 1), &abort_sh, p.status, p.wait_limit))
                    continue;
                if (abort_sh) continue;
                unsigned char* B = base + s * STAGE + ND * ADIG;
#pragma unroll
                for (int part = 0; part < 2; ++part) {
                    float d[4][ND];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const bool on = live && k + q < p.M;
                        digits8(on ? fixed_point(part ? vi[q] : vr[q], E, 4) : 0LL, d[q]);
                    }
#pragma unroll
                    for (int j = 0; j < ND; ++j)
                        *reinterpret_cast<uint2*>(B + j * BDIG + (part ? o_im : o_re)) =
                            make_uint2(pack_hi(d[0][j], d[1][j]), pack_hi(d[2][j], d[3][j]));
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&full[s]);
            }
        }
    } else if (warp >= W_EPI) {
        // ------------------------------------------------ digits of V
        const int gt = tid - 32 * W_EPI;
        const int r = gt >> 2, kq = gt & 3;                 // row of the block, group of 4 complex k
        const uint32_t h8 = (uint32_t)(kq & 1) * 8u;
        const uint32_t t0 = sw64_off(r, kq >> 1) + h8, t1 = sw64_off(r, 2 + (kq >> 1)) + h8;   // rows Re C
        const uint32_t b0 = t0 + 64u * 64u, b1 = t1 + 64u * 64u;                                 // rows Im C
        int g = 0, loaded = -1;
        for (int t = 0, item; (item = item_of(t, per, nitems, spread)) >= 0; ++t) {
            const int w = item / per_walker, tile = item % per_walker;
            if (skipped(w, (tile % p.nct) * OCT)) continue;
            const uint4* dg = p.dig + (size_t)w * p.nslot * 2;
            if constexpr (TS) {
                if (w != loaded) {
                    a_barrier();           // every digit warp is done with the previous walker's table
                    for (int i = gt; i < 2 * p.nslot; i += 32 * W_A) table[i] = dg[i];
                    a_barrier();
                    loaded = w;
                }
            }
            const uint16_t* row = p.vidx + (size_t)((tile / p.nct) * 64 + r) * p.Kp + kq * 4;
            uint2 nx = *reinterpret_cast<const uint2*>(row + p.kt0 * KC);
            for (int kt = p.kt0; kt < p.kt1; ++kt, ++g) {
                const int s = g % NSTAGE;
                const uint32_t sl[4] = {nx.x & 0xffffu, nx.x >> 16, nx.y & 0xffffu, nx.y >> 16};
                if (kt + 1 < p.kt1) nx = *reinterpret_cast<const uint2*>(row + (kt + 1) * KC);
                uint4 re[4], im[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    re[q] = TS ? table[2 * sl[q]] : dg[2 * sl[q]];
                    im[q] = TS ? table[2 * sl[q] + 1] : dg[2 * sl[q] + 1];
                }
                if (g >= NSTAGE &&
                    !mbar_wait_ab(&mma_bar[s], (uint32_t)((g / NSTAGE - 1) & 1), &abort_sh, p.status, p.wait_limit))
                    continue;
                if (abort_sh) continue;
                unsigned char* A = base + s * STAGE;
#pragma unroll
                for (int i = 0; i < ND; ++i) {
                    // digit i sits in half i & 1 of word i >> 1
                    const uint32_t sel = (i & 1) ? 0x7632u : 0x5410u;
                    auto word = [&](const uint4& v) { return i < 2 ? v.x : (i < 4 ? v.y : (i < 6 ? v.z : v.w)); };
                    const uint2 dr = make_uint2(__byte_perm(word(re[0]), word(re[1]), sel),
                                                __byte_perm(word(re[2]), word(re[3]), sel));
                    const uint2 di = make_uint2(__byte_perm(word(im[0]), word(im[1]), sel),
                                                __byte_perm(word(im[2]), word(im[3]), sel));
                    const uint2 dn = make_uint2(di.x ^ 0x80008000u, di.y ^ 0x80008000u);
                    unsigned char* Ai = A + i * ADIG;
                    *reinterpret_cast<uint2*>(Ai + t0) = dr;
                    *reinterpret_cast<uint2*>(Ai + t1) = dn;
                    *reinterpret_cast<uint2*>(Ai + b0) = di;
                    *reinterpret_cast<uint2*>(Ai + b1) = dr;
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&full[s]);
            }
        }
    } else {
        // ------------------------------------------------ epilogue
        const int r = warp * 32 + lane, part = r >> 6;
        int li = 0;
        for (int t = 0, item; (item = item_of(t, per, nitems, spread)) >= 0; ++t) {
            const int w = item / per_walker, tile = item % per_walker;
            const int col0 = (tile % p.nct) * OCT, i = (tile / p.nct) * 64 + (r & 63);
            if (skipped(w, col0)) continue;
            const int bi = li & 1;
            const bool row_ok = i < p.M;
            const double osi = row_ok && p.os ? p.os[i] : 1.0;
            const int ev = p.ev[w];
            const bool ok = mbar_wait_ab(&tfull[bi], (uint32_t)((li >> 1) & 1), &abort_sh, p.status, p.wait_limit);
            tc_fence_after();
            if (ok) {
                const uint32_t acc = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(bi * ND * OCT);
#pragma unroll 1
                for (int cc = 0; cc < OCT; cc += 8) {
                    if (col0 + cc >= p.M) break;
                    uint32_t v[ND][8];
#pragma unroll
                    for (int l = 0; l < ND; ++l) tmem_ld8(acc + (uint32_t)(l * OCT + cc), v[l]);
                    double u[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int c = col0 + cc + q;
                        u[q] = row_ok && c < p.M ? p.U[(((size_t)w * p.M + c) * 2 + part) * p.Kp + i] : 0.0;
                    }
                    tmem_wait_ld();
#pragma unroll
                    for (int l = 0; l < ND; ++l)     // the values are read after the wait
                        asm volatile("" : "+r"(v[l][0]), "+r"(v[l][1]), "+r"(v[l][2]), "+r"(v[l][3]), "+r"(v[l][4]),
                                     "+r"(v[l][5]), "+r"(v[l][6]), "+r"(v[l][7]));
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int c = col0 + cc + q;
                        if (c >= p.M) break;         // uniform over the warp
                        float lv[ND];
#pragma unroll
                        for (int l = 0; l < ND; ++l) lv[l] = __uint_as_float(v[l][q]);
                        const double sum = level_sum(lv);
                        // V is scaled by 2^(1078 - ev), Z by 2^(1079 - ec); the level-7 unit of the
                        // product weighs 2^49 (digit weights 2^(49 - 7 j) of both factors)
                        const int ec = (int)(p.cin[(size_t)w * p.M + c] >> 20);
                        double sc = p.alpha;
                        if (ev == 0x7ff || ec == 0x7ff) sc = __longlong_as_double(0x7ff8000000000000LL);
                        else sc = scale_pow2(sc, ev + ec - 2 * 1078 - 1 + 49);
                        double val = fma(sc, sum, u[q]);
                        if (p.os) val *= osi;
                        if (row_ok) {
                            if (p.outY)
                                reinterpret_cast<double*>(p.outY)[(((size_t)w * p.M + i) * p.M + c) * 2 + part] = val;
                            else
                                p.out[(((size_t)w * p.M + c) * 2 + part) * p.Kp + i] = val;
                        }
                        if (p.cout) {
                            const uint32_t hw = row_ok ? ((uint32_t)__double2hiint(val) & 0x7fffffffu) : 0u;
                            const uint32_t mx = __reduce_max_sync(0xffffffffu, hw);
                            if (lane == q) atomicMax(p.cout + (size_t)w * p.M + c, mx);
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[bi]);
            ++li;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// Z_0 = h Y as planes with its column maxima, and the maxima of the later
// Horner steps cleared.  One block per walker and 32 columns, 32 x 33 tiles.
__global__ void __launch_bounds__(256) k_oz_start(const double2* __restrict__ Y, double* __restrict__ Z,
                                                 const double* __restrict__ h, uint32_t* __restrict__ cmax, int M,
                                                 int Kp, int W, int steps, const double* __restrict__ rank) {
    __shared__ double2 tile[32][33];
    __shared__ uint32_t mx[32];
    const int w = blockIdx.y, c0 = blockIdx.x * 32;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (rank && c0 >= (int)rank[(long)WSTRIDE * w + 12]) return;
    if (threadIdx.x < 32) mx[threadIdx.x] = 0u;
    for (int i0 = 0; i0 < M; i0 += 32) {
        __syncthreads();
        for (int r = wid; r < 32; r += 8) {
            const int i = i0 + r, c = c0 + lane;
            if (i < M && c < M) tile[r][lane] = Y[((size_t)w * M + i) * M + c] * h[i];
        }
        __syncthreads();
        for (int q = wid; q < 32; q += 8) {
            const int i = i0 + lane, c = c0 + q;
            if (c >= M) break;
            uint32_t hw = 0u;
            if (i < M) {
                const double2 v = tile[lane][q];
                double* z = Z + ((size_t)w * M + c) * 2 * Kp + i;
                z[0] = v.x;
                z[Kp] = v.y;
                const uint32_t a = (uint32_t)__double2hiint(v.x) & 0x7fffffffu;
                const uint32_t b = (uint32_t)__double2hiint(v.y) & 0x7fffffffu;
                hw = a > b ? a : b;
            }
            hw = __reduce_max_sync(0xffffffffu, hw);
            if (lane == 0 && hw > mx[q]) mx[q] = hw;      // column q belongs to one warp
        }
    }
    __syncthreads();
    if (threadIdx.x < 32 && c0 + (int)threadIdx.x < M) {
        const size_t o = (size_t)w * M + c0 + threadIdx.x;
        cmax[o] = mx[threadIdx.x];
        for (int s = 1; s <= steps; ++s) cmax[(size_t)s * W * M + o] = 0u;
    }
}

// The walker's field table as digits: exponent of its largest entry, then eight
// bf16 digits of every real and imaginary part.
__global__ void __launch_bounds__(256) k_oz_table(const double2* __restrict__ phi, uint4* __restrict__ dig,
                                                 int* __restrict__ ev, int nslot) {
    __shared__ uint32_t mx;
    const int w = blockIdx.x;
    const double2* ph = phi + (size_t)w * nslot;
    if (threadIdx.x == 0) mx = 0u;
    __syncthreads();
    uint32_t m = 0u;
    for (int s = threadIdx.x; s < nslot; s += 256) {
        const uint32_t a = (uint32_t)__double2hiint(ph[s].x) & 0x7fffffffu;
        const uint32_t b = (uint32_t)__double2hiint(ph[s].y) & 0x7fffffffu;
        m = max(m, max(a, b));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(&mx, m);
    __syncthreads();
    const int E = (int)(mx >> 20);
    if (threadIdx.x == 0) ev[w] = E;
    for (int s = threadIdx.x; s < nslot; s += 256) {
        const double2 v = ph[s];
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            float d[ND];
            digits8(fixed_point(part ? v.y : v.x, E, 3), d);
            dig[((size_t)w * nslot + s) * 2 + part] =
                make_uint4(pack_hi(d[0], d[1]), pack_hi(d[2], d[3]), pack_hi(d[4], d[5]), pack_hi(d[6], d[7]));
        }
    }
}

// Rows [R, M) of a Horner step (a thin band that would cost a whole 64-row
// block): FP64 sums, four lanes per column, the row of V in shared memory.
__global__ void __launch_bounds__(256) k_oz_border(const double* __restrict__ Zin, const double* __restrict__ U,
                                                  double* __restrict__ out, double2* __restrict__ outY,
                                                  const double2* __restrict__ phi, const uint16_t* __restrict__ vidx,
                                                  uint32_t* __restrict__ cmax, const double* __restrict__ os,
                                                  double alpha, int M, int Kp, int nslot, int R,
                                                  const double* __restrict__ rank) {
    extern __shared__ unsigned char smem_raw[];
    double2* v = reinterpret_cast<double2*>(smem_raw);     // [M]
    const int w = blockIdx.y, q = threadIdx.x & 3;
    const int c = blockIdx.x * 64 + (threadIdx.x >> 2);
    if (rank && (int)blockIdx.x * 64 >= (int)rank[(long)WSTRIDE * w + 12]) return;
    const bool on = c < M;
    const size_t col = ((size_t)w * M + (on ? c : 0)) * 2 * Kp;
    for (int i = R; i < M; ++i) {
        __syncthreads();
        for (int k = threadIdx.x; k < M; k += 256) v[k] = phi[(size_t)w * nslot + vidx[(size_t)i * M + k]];
        __syncthreads();
        double2 s = make_double2(0.0, 0.0), s2 = s;
        int k = q;
        for (; k + 4 < M; k += 8) {
            s = cfma(v[k], make_double2(Zin[col + k], Zin[col + Kp + k]), s);
            s2 = cfma(v[k + 4], make_double2(Zin[col + k + 4], Zin[col + Kp + k + 4]), s2);
        }
        if (k < M) s = cfma(v[k], make_double2(Zin[col + k], Zin[col + Kp + k]), s);
        s = s + s2;
        for (int o = 2; o > 0; o >>= 1) {
            s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
            s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
        }
        if (on && q < 2) {
            double val = fma(alpha, q ? s.y : s.x, U[col + (q ? Kp : 0) + i]);
            if (os) val *= os[i];
            if (outY) reinterpret_cast<double*>(outY)[(((size_t)w * M + i) * M + c) * 2 + q] = val;
            else out[col + (q ? Kp : 0) + i] = val;
            if (cmax) atomicMax(cmax + (size_t)w * M + c, (uint32_t)__double2hiint(val) & 0x7fffffffu);
        }
    }
}

// ---------------------------------------------------------------- small bases
// All Horner steps of a slice in one launch, one block per walker: V (built
// once) and the chain in shared memory, an output per thread and pass, FP64 FMA.
__global__ void k_chain_small(double2* __restrict__ Y, const double2* __restrict__ phi,
                              const uint16_t* __restrict__ vidx, const double* __restrict__ h, int p, int M,
                              int nslot, const double* __restrict__ rank) {
    extern __shared__ unsigned char smem_raw[];
    double2* V = reinterpret_cast<double2*>(smem_raw);     // [M][M]
    double2* U = V + M * M;                                // h Y
    double2* Z0 = U + M * M;
    double2* Z1 = Z0 + M * M;
    const int w = blockIdx.x, n = M * M;
    const int cols = rank ? (int)rank[(long)WSTRIDE * w + 12] : M;
    double2* Yw = Y + (size_t)w * n;
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        V[e] = phi[(size_t)w * nslot + vidx[e]];
        U[e] = Yw[e] * h[e / M];
    }
    const double2* in = U;
    double2* out = Z0;
    for (int j = p; j >= 1; --j) {
        __syncthreads();
        const double alpha = 1.0 / j;
        for (int e = threadIdx.x; e < n; e += blockDim.x) {
            const int i = e / M, c = e - i * M;
            if (c >= cols) continue;
            double2 s = make_double2(0.0, 0.0);
            for (int k = 0; k < M; ++k) s = cfma(V[i * M + k], in[k * M + c], s);
            double2 v = U[e] + s * alpha;
            if (j == 1) Yw[e] = v * h[i];
            else out[e] = v;
        }
        in = out;
        out = out == Z0 ? Z1 : Z0;
    }
}

// Bases up to this size run k_chain_small: a 64 x 32 item is mostly padding there,
// and one launch replaces p + 2 (M = 7, 64 walkers: 15 us a slice against 138 us
// for six launches of the tiled kernel).  From M = 27 on the FP64 pipe alone
// would need 2 M^3 = 39,000 cycles per walker and step, the items about 15,000.
constexpr int SMALL_M = 19;

}  // namespace

bool oz_chain_small(int M) { return M <= SMALL_M; }

int oz_kp(int M) { return (M + KC - 1) / KC * KC; }

// Rows the tensor-core items cover: a remainder of at most 8 rows beyond the
// 64-row blocks is left to k_oz_border.
static int oz_rows(int M) {
    const int rem = M % 64;
    return rem == 0 ? M : (M > 64 && rem <= 8 ? M - rem : (M + 63) / 64 * 64);
}

// Slot table with rows of Kp entries, 64-row blocks, zero padded (slot 0 is V's
// zero diagonal).
std::vector<uint16_t> oz_slots(const UegSetup& s) {
    const int Kp = oz_kp(s.M), R = (s.M + 63) / 64 * 64;
    std::vector<uint16_t> v((size_t)R * Kp, 0);
    for (int i = 0; i < s.M; ++i)
        for (int k = 0; k < s.M; ++k) v[(size_t)i * Kp + k] = s.vidx[(size_t)i * s.M + k];
    return v;
}

// One slice's B applied to the complex128 chain c->Y (in place).
cudaError_t oz_chain(ftq_ctx* c) {
    const int M = c->M, W = c->W, p = c->opts.exp_order;
    const double* rank = c->opts.low_rank_threshold > 0.0 ? c->wstate : nullptr;
    if (oz_chain_small(M)) {
        const size_t sm = 4 * sizeof(double2) * (size_t)M * M;
        const int nt = std::min(1024, (M * M + 31) / 32 * 32);
        LaunchScope ls(c, FTQ_K_CHAIN);
        k_chain_small<<<W, nt, sm, c->stream>>>(c->Y, c->phi, c->tab.vidx, c->tab.h, p, M, c->nslot, rank);
        return cudaGetLastError();
    }
    const int Kp = oz_kp(M), R = std::min(oz_rows(M), (M + 63) / 64 * 64);
    double* Z0 = reinterpret_cast<double*>(c->work);       // scratch of the factorisations, free here
    double* Zb[2] = {reinterpret_cast<double*>(c->zbuf[0]), reinterpret_cast<double*>(c->zbuf[1])};
    const size_t col = (size_t)W * M;
    {
        LaunchScope ls(c, FTQ_K_BRIDGE);
        k_oz_table<<<W, 256, 0, c->stream>>>(c->phi, c->oz_dig, c->oz_ev, c->nslot);
    }
    {
        LaunchScope ls(c, FTQ_K_BRIDGE);
        k_oz_start<<<dim3((unsigned)((M + 31) / 32), (unsigned)W), 256, 0, c->stream>>>(c->Y, Z0, c->tab.h, c->oz_cmax,
                                                                                   M, Kp, W, p, rank);
    }
    cudaError_t e = cudaGetLastError();
    OzArgs a{};
    a.U = Z0;
    a.dig = c->oz_dig;
    a.ev = c->oz_ev;
    a.vidx = c->tab.ozidx;
    a.rank = rank;
    a.status = c->status;
    a.M = M;
    a.Kp = Kp;
    a.nslot = c->nslot;
    a.nrb = R < M ? R / 64 : (M + 63) / 64;
    a.nct = (M + OCT - 1) / OCT;
    a.W = W;
    a.wait_limit = c->wait_limit >= 0 ? (long long)c->wait_limit : TC_WAIT_LIMIT;
    constexpr size_t limit = 227 * 1024 - 1024;            // room for the static shared memory
    const size_t tab = 2 * sizeof(uint4) * (size_t)c->nslot;
    size_t sm = 1024 + (size_t)NSTAGE * STAGE;
    const bool ts = sm + tab <= limit;
    if (ts) sm += tab;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    auto kernel = ts ? k_chain_oz<true> : k_chain_oz<false>;
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit);
    const int grid = std::min(sms, W * a.nrb * a.nct);
    const int tiles = Kp / KC;
    // whole k tiles per chunk; one chunk also where only V's zero diagonal keeps a row at CHUNK_K terms (M = 257)
    const int chunks = M - 1 <= CHUNK_K ? 1 : (tiles * KC + CHUNK_K - 1) / CHUNK_K;
    const double* zin = Z0;
    for (int j = p, s = 0; j >= 1 && e == cudaSuccess; --j, ++s) {
        double* zout = Zb[s & 1];
        a.Zin = zin;
        a.cin = c->oz_cmax + s * col;
        a.alpha = 1.0 / j;
        for (int q = 0; q < chunks && e == cudaSuccess; ++q) {
            const bool lastq = q + 1 == chunks;
            a.kt0 = tiles * q / chunks;
            a.kt1 = tiles * (q + 1) / chunks;
            a.U = q == 0 ? Z0 : zout;                      // later chunks add to the partial result
            a.out = zout;
            a.outY = lastq && j == 1 ? c->Y : nullptr;
            a.cout = lastq && j > 1 ? c->oz_cmax + (s + 1) * col : nullptr;
            a.os = lastq && j == 1 ? c->tab.h : nullptr;
            LaunchScope ls(c, FTQ_K_CHAIN);
            kernel<<<grid, NT_OZ, sm, c->stream>>>(a);
            e = cudaGetLastError();
        }
        if (R < M && e == cudaSuccess) {
            LaunchScope ls(c, FTQ_K_BORDER);
            k_oz_border<<<dim3((unsigned)((M + 63) / 64), (unsigned)W), 256, sizeof(double2) * M, c->stream>>>(
                zin, Z0, zout, j == 1 ? c->Y : nullptr, c->phi, c->tab.vidx,
                j > 1 ? c->oz_cmax + (s + 1) * col : nullptr, j == 1 ? c->tab.h : nullptr, 1.0 / j, M, Kp, c->nslot, R,
                rank);
            e = cudaGetLastError();
        }
        zin = zout;
    }
    return e;
}

}  // namespace ftq
