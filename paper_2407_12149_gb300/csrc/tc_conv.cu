// tc_conv.cu -- 3x3 convolutions as implicit GEMMs on the tcgen05 tensor cores.
//
// A tile is 128 consecutive pixels of a channels-last image [B][H][H][C] (whole grid rows, or
// part of one: H is a power of two).  The operand of a tap is the TMA box of those pixels
// shifted by the tap, 16 to 64 channels wide; what falls outside the image is the box's zero
// fill.  So no im2col matrix is written or read: the convolutions' memory traffic is the
// activations themselves, nine shifted reads of which are served by the L2.
//
// k_conv (forward and data gradient), persistent, one CTA per SM, six warps:
//   warp 0     TMA producer: a ring of stages, each one channel chunk of one tap of the pixels
//              (and of the weights, when they do not fit in shared memory as a whole);
//   warp 1     MMA issuer: M = 128, N = the output channels of the tile, K = 16 per instruction,
//              tap by tap and channel by channel -- the order of the im2col matrix's columns;
//   warps 2-5  epilogue, overlapped with the next accumulation (accumulators alternate in TMEM).
// Forward: one accumulation over all taps, bias, ReLU, BF16.  Data gradient: one accumulation
// per tap, the nine FP32 results added in tap order in registers (out-of-range taps add zero).
// Both give the bits of the im2col / col2im forms they replace.
// k_wgrad: dW[tap ci][co] = sum over pixels X(shifted)[p][ci] dZ[p][co]: both operands are
// read pixel-major, i.e. MN-major tiles (64 pixels x 64 or 32 channels), so nothing is
// transposed; the pixel range is cut into splits summed in a fixed order.
//
// Every mbarrier wait is bounded (1 s): when one gives up the other roles stop, the accumulator in
// work is not handed to the epilogue, MMAs and copies in flight are waited for (bounded), the
// event is counted in *status, TMEM is freed and the CTA ends.
// Measured (GB300, 255^2, c0 = 32; im2col + GEMM + col2im before): gradient of 8 samples 17.7 ->
// 2.96 ms, estimates of 16 samples 6.21 -> 1.34 ms (3.34 and 1.72 with 64-bit ring counters; 3.73
// and 2.10 when k_conv ran every layer, without the lines of k_conv_line).
#include <algorithm>
#include <cstring>

#include "tc5.cuh"
#include "tc_conv.cuh"
#include "tc_gemm.cuh"

namespace mgmc {

namespace {

using bf16 = __nv_bfloat16;
using tc5::RingPos;

constexpr int kBM = 128;
constexpr int kConvThreads = 192;
constexpr int kMaxStages = 8;
constexpr size_t kConvSmem = 220 * 1024;   // dynamic shared memory a CTA may use

struct ConvArgs {
    CUtensorMap x, w;     // pixels (box CK x tw x th x tb), weights (box CK x NT)
    long long P;          // pixels
    int H, tw, th, lgH;   // image side, tile width and height
    int taps_c;           // chunks per tap
    int ck;               // channels per chunk
    int wtap_k, wtap_r;   // weight coordinates of tap t: k = t wtap_k + chunk, row = t wtap_r + n0
    int sign;             // shift of tap (ky, kx): sign * (k - 1)
    int nout, ntiles_n;   // output channels, N tiles
    long long tiles;      // pixel tiles x N tiles
    int stages;
    int resident;         // 1: all weights of the N tile stay in shared memory
    const float* bias;
    void* out;
    int* status;
    long long wait_ns;    // bound of the waits (tc_gemm.cuh)
};

// Epilogue warps: one tile's accumulations (`units` of them, from buffer bp on) from TMEM; false
// if a wait gave up.  TMEM lanes 32 (warp % 4) .. + 31 are the warp's, lane = pixel p0 + that.
template <int NT, bool DG, int NBUF, int NTC>
__device__ __forceinline__ bool conv_epilogue(const ConvArgs& g, long long p0, int n_first, int units, RingPos& bp,
                                              unsigned tmem, unsigned long long* tfull, unsigned long long* tempty)
{
    const int quarter = (threadIdx.x >> 5) & 3, lane = threadIdx.x & 31;
    const long long p = p0 + quarter * 32 + lane;
    float acc[DG ? NT : 1];
    for (int a = 0; a < units; ++a, bp.next(NBUF)) {
        const int buf = bp.slot;
        bool ok = mbar_wait(&tfull[buf], bp.par, tc5::role_limit(g.wait_ns));
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) return false;
        tc5::fence_after();
        const unsigned t0 = tmem + ((unsigned)(quarter * 32) << 16) + (unsigned)(buf * NTC);
        if constexpr (DG) {
#pragma unroll
            for (int c0 = 0; c0 < NT; c0 += 32) {
                unsigned r[32];
                tc5::ld32(t0 + c0, r);
                if (a == 0) {
#pragma unroll
                    for (int q = 0; q < 32; ++q) acc[c0 + q] = 0.0f + __uint_as_float(r[q]);
                } else {
#pragma unroll
                    for (int q = 0; q < 32; ++q) acc[c0 + q] += __uint_as_float(r[q]);
                }
            }
        } else {
            for (int c0 = 0; c0 < NT; c0 += 32) {
                unsigned r[32];
                tc5::ld32(t0 + c0, r);
                if (p >= g.P || n_first + c0 >= g.nout) continue;
                __nv_bfloat162 h[16];
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    float2 bb = make_float2(0.f, 0.f);
                    if (n_first + c0 + 2 * q < g.nout)
                        bb = __ldg(reinterpret_cast<const float2*>(g.bias + n_first + c0 + 2 * q));
                    h[q] = __floats2bfloat162_rn(fmaxf(__uint_as_float(r[2 * q]) + bb.x, 0.f),
                                                 fmaxf(__uint_as_float(r[2 * q + 1]) + bb.y, 0.f));
                }
                bf16* o = reinterpret_cast<bf16*>(g.out) + p * g.nout + n_first + c0;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (n_first + c0 + 8 * q < g.nout) *reinterpret_cast<uint4*>(o + 8 * q) = reinterpret_cast<uint4*>(h)[q];
            }
        }
        tc5::fence_before();
        __syncwarp();
        if (lane == 0) tc5::arrive(&tempty[buf]);
    }
    if constexpr (DG) {
        if (p < g.P) {
            float* o = reinterpret_cast<float*>(g.out) + p * g.nout + n_first;
#pragma unroll
            for (int q = 0; q < NT / 4; ++q)
                if (n_first + 4 * q < g.nout)
                    reinterpret_cast<float4*>(o)[q] = make_float4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
        }
    }
    return true;
}

// After a wait gave up, all threads: the MMAs issued (by thread 32) and the copies never consumed
// (stages consumed .. issued - 1 of the ring of n, the weights) may still be in flight and are
// waited for (bounded)
__device__ __forceinline__ void conv_drain(unsigned long long* full, int n, int consumed, int issued,
                                           unsigned long long* wbar, unsigned long long* drained, int* status)
{
    if (threadIdx.x == 32) {
        tc5::commit(drained);
        mbar_wait(drained, 0u);
    }
    if (threadIdx.x == 0) {
        if (wbar) mbar_wait(wbar, 0u);
        for (int k = consumed; k < issued; ++k) mbar_wait(&full[k % n], (unsigned)((k / n) & 1));
        atomicAdd(status, 1);
    }
}

// NT: output channels of a tile; CKB: bytes of a chunk's row; DG: data gradient
template <int NT, int CKB, bool DG>
__global__ void __launch_bounds__(kConvThreads, 1) k_conv(const __grid_constant__ ConvArgs g)
{
    constexpr int A_BYTES = kBM * CKB, B_BYTES = NT * CKB;
    constexpr int NBUF = NT <= 128 ? 4 : 2;
    constexpr int NTC = NT <= 32 ? 32 : NT <= 64 ? 64 : NT <= 128 ? 128 : 256;   // TMEM columns of one accumulator
    constexpr unsigned TCOLS = NBUF * NTC;
    constexpr unsigned SW = tc5::swizzle_of(CKB);
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    unsigned char* sm = smem_align_up<1024>(smem_dyn);
    __shared__ unsigned long long full[kMaxStages], empty[kMaxStages], tfull[4], tempty[4], wbar, drained;
    __shared__ unsigned tmem_slot;
    __shared__ volatile int aborted;
    __shared__ int issued, consumed;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int S = g.stages;
    const int items = 9 * g.taps_c;                       // chunks of one tile
    const int unit = DG ? g.taps_c : items;               // chunks of one accumulation
    const int stage_bytes = A_BYTES + (g.resident ? 0 : B_BYTES);
    unsigned char* const wres = sm;                       // resident weights first
    unsigned char* const ring = sm + (g.resident ? items * B_BYTES : 0);
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s]);
            mbar_init(&empty[s]);
        }
        for (int b = 0; b < 4; ++b) {
            mbar_init(&tfull[b]);
            mbar_init_count(&tempty[b], 4);
        }
        mbar_init(&wbar);
        mbar_init(&drained);
        fence_mbar_init();
        aborted = 0;
        issued = consumed = 0;
    }
    if (warp == 0) tc5::alloc(&tmem_slot, TCOLS);
    tc5::fence_before();
    __syncthreads();
    tc5::fence_after();
    const unsigned tmem = tmem_slot;
    const long long lim = tc5::role_limit(g.wait_ns);
    const int n_first = (int)(blockIdx.x % g.ntiles_n) * NT;   // a CTA keeps its N tile (grid is a multiple)
    const long long step = gridDim.x / g.ntiles_n;
    const long long mtiles = g.tiles / g.ntiles_n;

    if (warp == 0 && lane == 0) {
        if (g.resident) {
            mbar_expect_tx(&wbar, (unsigned)(items * B_BYTES));
            for (int t = 0; t < 9; ++t)
                for (int c = 0; c < g.taps_c; ++c)
                    tma_load_2d(wres + (t * g.taps_c + c) * B_BYTES, &g.w, t * g.wtap_k + c * g.ck,
                                t * g.wtap_r + n_first, &wbar);
        }
        int k = 0;
        RingPos rp;
        for (long long mt = blockIdx.x / g.ntiles_n; mt < mtiles && !aborted; mt += step) {
            const long long p0 = mt * kBM;
            const int j0 = (int)(p0 & (g.H - 1)), i0 = (int)((p0 >> g.lgH) & (g.H - 1));
            const int b0 = (int)(p0 >> (2 * g.lgH));
            for (int t = 0; t < 9 && !aborted; ++t) {
                const int sy = g.sign * (t / 3 - 1), sx = g.sign * (t % 3 - 1);
                for (int c = 0; c < g.taps_c; ++c, ++k, rp.next(S)) {
                    const int s = rp.slot;
                    // a fresh barrier counts as past its phase of parity 1: the first use does not wait
                    if (!mbar_wait(&empty[s], rp.par ^ 1u, lim)) {
                        aborted = 1;
                        break;
                    }
                    unsigned char* st = ring + s * stage_bytes;
                    mbar_expect_tx(&full[s], (unsigned)stage_bytes);
                    tc5::tma_load_4d(st, &g.x, c * g.ck, j0 + sx, i0 + sy, b0, &full[s]);
                    if (!g.resident)
                        tma_load_2d(st + A_BYTES, &g.w, t * g.wtap_k + c * g.ck, t * g.wtap_r + n_first, &full[s]);
                    issued = k + 1;
                }
            }
        }
    } else if (warp == 1 && lane == 0) {
        const unsigned id = tc5::idesc(NT, false);
        int k = 0;
        RingPos rp, bp;
        bool ok = g.wait_ns >= 0 && (!g.resident || mbar_wait(&wbar, 0u));
        for (long long mt = blockIdx.x / g.ntiles_n; mt < mtiles && ok && !aborted; mt += step)
            for (int a = 0; a < items && ok; a += unit, bp.next(NBUF)) {
                const int buf = bp.slot;
                if (!mbar_wait(&tempty[buf], bp.par ^ 1u)) {
                    ok = false;
                    break;
                }
                tc5::fence_after();
                for (int c = 0; c < unit; ++c, ++k, rp.next(S)) {
                    const int s = rp.slot;
                    if (!mbar_wait(&full[s], rp.par)) {
                        ok = false;
                        break;
                    }
                    tc5::fence_after();
                    const unsigned sa = smem_addr(ring + s * stage_bytes);
                    const unsigned sb = g.resident ? smem_addr(wres + (a + c) * B_BYTES) : sa + A_BYTES;
                    const unsigned long long da = tc5::desc(sa, 16, 8 * CKB, SW), db = tc5::desc(sb, 16, 8 * CKB, SW);
#pragma unroll
                    for (int q = 0; q < CKB / 32; ++q)
                        tc5::mma(tmem + (unsigned)(buf * NTC), da + 2ull * q, db + 2ull * q, id, (c > 0 || q > 0) ? 1u : 0u);
                    tc5::commit(&empty[s]);
                    consumed = k + 1;
                }
                if (!ok) break;   // an incomplete accumulator never reaches the epilogue
                tc5::commit(&tfull[buf]);
            }
        if (!ok) aborted = 1;
    } else if (warp >= 2) {
        bool ok = true;
        RingPos bp;
        // the lanes leave the loop together: tcgen05.ld is a warp's
        for (long long mt = blockIdx.x / g.ntiles_n; mt < mtiles && ok && !__any_sync(0xffffffffu, aborted); mt += step)
            ok = conv_epilogue<NT, DG, NBUF, NTC>(g, mt * kBM, n_first, items / unit, bp, tmem, tfull, tempty);
        if (!ok && lane == 0) aborted = 1;
    }
    __syncwarp();
    __syncthreads();
    if (aborted) conv_drain(full, S, consumed, issued, g.resident ? &wbar : nullptr, &drained, g.status);
    tc5::fence_before();
    __syncthreads();
    if (warp == 0) tc5::dealloc(tmem, TCOLS);
}

// The same convolutions on images of side H >= 128 whose weights fit in shared memory: a CTA walks
// down strips of 128 columns, one grid row (tile) at a time, through a ring of lines.  A line is
// the TMA box of 130 pixels (the strip and one more on each side) of one grid row; the tap
// (ky, kx) of a tile is line i + ky - 1 from pixel kx on, an operand that starts kx rows into the
// swizzled box.  Every line is fetched once instead of nine times: the nine-fold reads of k_conv
// ran at the L2's rate (about 15 bytes per clock and SM), this form at a ninth of its traffic.
constexpr int kLinePx = kBM + 2;
template <int NT, int CKB, bool DG>
__global__ void __launch_bounds__(kConvThreads, 1) k_conv_line(const __grid_constant__ ConvArgs g)
{
    constexpr int B_BYTES = NT * CKB;
    constexpr int CHUNK = (kLinePx * CKB + 1023) / 1024 * 1024;   // one channel chunk of a line
    constexpr int NBUF = NT <= 128 ? 4 : 2;
    constexpr int NTC = NT <= 32 ? 32 : NT <= 64 ? 64 : NT <= 128 ? 128 : 256;
    constexpr unsigned TCOLS = NBUF * NTC;
    constexpr unsigned SW = tc5::swizzle_of(CKB);
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    unsigned char* sm = smem_align_up<1024>(smem_dyn);
    __shared__ unsigned long long full[kMaxStages], empty[kMaxStages], tfull[4], tempty[4], wbar, drained;
    __shared__ unsigned tmem_slot;
    __shared__ volatile int aborted;
    __shared__ int issued, consumed;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int NL = g.stages;                       // lines of the ring
    const int items = 9 * g.taps_c;
    const int line_bytes = g.taps_c * CHUNK;
    unsigned char* const ring = sm;
    unsigned char* const wres = sm + NL * line_bytes;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NL; ++s) {
            mbar_init(&full[s]);
            mbar_init(&empty[s]);
        }
        for (int b = 0; b < 4; ++b) {
            mbar_init(&tfull[b]);
            mbar_init_count(&tempty[b], 4);
        }
        mbar_init(&wbar);
        mbar_init(&drained);
        fence_mbar_init();
        aborted = 0;
        issued = consumed = 0;
    }
    if (warp == 0) tc5::alloc(&tmem_slot, TCOLS);
    tc5::fence_before();
    __syncthreads();
    tc5::fence_after();
    const unsigned tmem = tmem_slot;
    const long long lim = tc5::role_limit(g.wait_ns);
    const int n_first = (int)(blockIdx.x % g.ntiles_n) * NT;
    const long long ctas = gridDim.x / g.ntiles_n, cta = blockIdx.x / g.ntiles_n;
    const long long mtiles = g.tiles / g.ntiles_n;
    // tiles in strip order: tile = strip * H + row, strip = image * (H / 128) + column block
    const long long beg = mtiles * cta / ctas, end = mtiles * (cta + 1) / ctas;
    const int spi = g.H >> 7;   // strips per image

    if (warp == 0 && lane == 0) {
        mbar_expect_tx(&wbar, (unsigned)(items * B_BYTES));
        for (int t = 0; t < 9; ++t)
            for (int c = 0; c < g.taps_c; ++c)
                tma_load_2d(wres + (t * g.taps_c + c) * B_BYTES, &g.w, t * g.wtap_k + c * g.ck, t * g.wtap_r + n_first,
                            &wbar);
        int k = 0;
        RingPos rp;
        for (long long t0 = beg; t0 < end && !aborted;) {
            const long long strip = t0 >> g.lgH;
            const long long t1 = min(end, (strip + 1) << g.lgH);
            const int ia = (int)(t0 & (g.H - 1)), ib = ia + (int)(t1 - t0);
            const int b = (int)(strip / spi), j0 = (int)(strip % spi) << 7;
            for (int row = ia - 1; row <= ib; ++row, ++k, rp.next(NL)) {
                const int s = rp.slot;
                if (!mbar_wait(&empty[s], rp.par ^ 1u, lim)) {
                    aborted = 1;
                    break;
                }
                mbar_expect_tx(&full[s], (unsigned)(g.taps_c * kLinePx * CKB));
                for (int c = 0; c < g.taps_c; ++c)
                    tc5::tma_load_4d(ring + s * line_bytes + c * CHUNK, &g.x, c * g.ck, j0 - 1, row, b, &full[s]);
                issued = k + 1;
            }
            t0 = t1;
        }
    } else if (warp == 1 && lane == 0) {
        const unsigned id = tc5::idesc(NT, false);
        RingPos kp, wp, bp;       // the line above the tile, the next line to wait for, the accumulator
        int waited = 0;           // lines known to have arrived
        bool ok = g.wait_ns >= 0 && mbar_wait(&wbar, 0u);
        for (long long t0 = beg; t0 < end && ok && !aborted;) {
            const long long strip = t0 >> g.lgH;
            const long long t1 = min(end, (strip + 1) << g.lgH);
            for (long long t = t0; t < t1 && ok; ++t, kp.next(NL)) {
                for (int q = t == t0 ? 3 : 1; q > 0; --q, ++waited, wp.next(NL)) {
                    ok = mbar_wait(&full[wp.slot], wp.par);
                    if (!ok) break;   // `waited` counts the lines that have arrived
                }
                consumed = waited;
                if (!ok) break;
                for (int tap = 0; tap < 9 && ok; ++tap) {
                    const int buf = bp.slot;
                    if (DG || tap == 0) {
                        ok = mbar_wait(&tempty[buf], bp.par ^ 1u);
                        if (!ok) break;
                        tc5::fence_after();
                    }
                    const int ky = g.sign > 0 ? tap / 3 : 2 - tap / 3, kx = g.sign > 0 ? tap % 3 : 2 - tap % 3;
                    const unsigned la = smem_addr(ring + kp.ahead(ky, NL) * line_bytes) + (unsigned)(kx * CKB);
                    const unsigned lb = smem_addr(wres + tap * g.taps_c * B_BYTES);
                    for (int c = 0; c < g.taps_c; ++c) {
                        const unsigned long long da = tc5::desc(la + c * CHUNK, 16, 8 * CKB, SW);
                        const unsigned long long db = tc5::desc(lb + c * B_BYTES, 16, 8 * CKB, SW);
#pragma unroll
                        for (int q = 0; q < CKB / 32; ++q)
                            tc5::mma(tmem + (unsigned)(buf * NTC), da + 2ull * q, db + 2ull * q, id,
                                     (c > 0 || q > 0 || (!DG && tap > 0)) ? 1u : 0u);
                    }
                    if (DG || tap == 8) {
                        tc5::commit(&tfull[buf]);
                        bp.next(NBUF);
                    }
                }
                if (!ok) break;
                // the line above is done with; after the strip's last row all three are
                tc5::commit(&empty[kp.slot]);
                if (t + 1 == t1) {
                    tc5::commit(&empty[kp.ahead(1, NL)]);
                    tc5::commit(&empty[kp.ahead(2, NL)]);
                }
            }
            kp.next(NL);
            kp.next(NL);
            t0 = t1;
        }
        if (!ok) aborted = 1;
    } else if (warp >= 2) {
        bool ok = true;
        RingPos bp;
        for (long long t = beg; t < end && ok && !__any_sync(0xffffffffu, aborted); ++t) {
            const long long strip = t >> g.lgH;
            const long long row = (strip / spi) * g.H + (t & (g.H - 1));
            ok = conv_epilogue<NT, DG, NBUF, NTC>(g, row * g.H + ((strip % spi) << 7), n_first, DG ? 9 : 1, bp, tmem, tfull,
                                                  tempty);
        }
        if (!ok && lane == 0) aborted = 1;
    }
    __syncwarp();
    __syncthreads();
    if (aborted) conv_drain(full, NL, consumed, issued, &wbar, &drained, g.status);
    tc5::fence_before();
    __syncthreads();
    if (warp == 0) tc5::dealloc(tmem, TCOLS);
}

struct WgradArgs {
    CUtensorMap x, z;        // boxes UC x 64 pixels, UN x 64 pixels
    long long P, k_per_split;
    int H, lgH;
    int cin, nout;
    float* out;              // [splits][9 cin][nout]
    int* status;
    long long wait_ns;
};
constexpr int kWgStages = 4;

// NT: output channels (the whole of them, rounded up to the template), UA / UB: bytes of a
// pixel's row in the staged units of the two operands
template <int NT, int UA, int UB>
__global__ void __launch_bounds__(128, 1) k_wgrad(const __grid_constant__ WgradArgs g)
{
    constexpr int NUA = 256 / UA, NUB = NT * 2 / UB;      // units of 128 rows, of NT columns
    constexpr int A_UNIT = 64 * UA, B_UNIT = 64 * UB;
    constexpr int STAGE = NUA * A_UNIT + NUB * B_UNIT;
    constexpr unsigned TCOLS = NT < 32 ? 32 : NT;
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    unsigned char* sm = smem_align_up<1024>(smem_dyn);
    __shared__ unsigned long long full[kWgStages], empty[kWgStages], done;
    __shared__ unsigned tmem_slot;
    __shared__ int aborted, issued, consumed;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * kBM;
    const long long kbeg = (long long)blockIdx.z * g.k_per_split, kend = min(g.P, kbeg + g.k_per_split);
    const int nkb = kend > kbeg ? (int)((kend - kbeg + 63) / 64) : 0;
    const int rows = 9 * g.cin;
    const int units = min(NUA, (rows - m0 + UA / 2 - 1) / (UA / 2));
    if (threadIdx.x == 0) {
        for (int s = 0; s < kWgStages; ++s) {
            mbar_init(&full[s]);
            mbar_init(&empty[s]);
        }
        mbar_init(&done);
        fence_mbar_init();
        aborted = issued = consumed = 0;
    }
    if (warp == 0) tc5::alloc(&tmem_slot, TCOLS);
    tc5::fence_before();
    __syncthreads();
    tc5::fence_after();
    const unsigned tmem = tmem_slot;
    if (warp == 0 && lane == 0) {
        int kb = 0;
        for (; kb < nkb; ++kb) {
            const int s = kb % kWgStages, use = kb / kWgStages;
            if (use > 0 && !mbar_wait(&empty[s], (unsigned)((use - 1) & 1), tc5::role_limit(g.wait_ns))) {
                aborted = 1;
                break;
            }
            unsigned char* st = sm + s * STAGE;
            const long long p0 = kbeg + 64LL * kb;
            const int j0 = (int)(p0 & (g.H - 1)), i0 = (int)((p0 >> g.lgH) & (g.H - 1)), b0 = (int)(p0 >> (2 * g.lgH));
            mbar_expect_tx(&full[s], (unsigned)(units * A_UNIT + NUB * B_UNIT));
            for (int q = 0; q < units; ++q) {
                const int r = m0 + q * (UA / 2), tap = r / g.cin, c = r % g.cin;
                tc5::tma_load_4d(st + q * A_UNIT, &g.x, c, j0 + tap % 3 - 1, i0 + tap / 3 - 1, b0, &full[s]);
            }
            for (int q = 0; q < NUB; ++q)
                tc5::tma_load_4d(st + NUA * A_UNIT + q * B_UNIT, &g.z, q * (UB / 2), j0, i0, b0, &full[s]);
        }
        issued = kb;
    } else if (warp == 1 && lane == 0) {
        const unsigned id = tc5::idesc(NT, true);
        const int n = g.wait_ns < 0 ? 0 : nkb;
        if (g.wait_ns < 0) aborted = 1;
        int kb = 0;
        for (; kb < n; ++kb) {
            const int s = kb % kWgStages;
            if (!mbar_wait(&full[s], (unsigned)((kb / kWgStages) & 1))) {
                aborted = 1;
                break;
            }
            tc5::fence_after();
            const unsigned sa = smem_addr(sm + s * STAGE), sb = sa + NUA * A_UNIT;
            // MN-major: leading offset = the next 64 / 32 channels (a unit), stride offset = the
            // next 8 pixels; 16 pixels per instruction
            const unsigned long long da = tc5::desc(sa, A_UNIT, 8 * UA, tc5::swizzle_of(UA));
            const unsigned long long db = tc5::desc(sb, B_UNIT, 8 * UB, tc5::swizzle_of(UB));
#pragma unroll
            for (int q = 0; q < 4; ++q)
                tc5::mma(tmem, da + (unsigned long long)(q * 16 * UA >> 4), db + (unsigned long long)(q * 16 * UB >> 4), id,
                         (kb > 0 || q > 0) ? 1u : 0u);
            tc5::commit(&empty[s]);
        }
        consumed = kb;
        tc5::commit(&done);
    }
    __syncwarp();
    const bool ok = mbar_wait(&done, 0u);
    tc5::fence_after();
    __syncthreads();
    const bool good = ok && !aborted && nkb > 0;
    const int row = m0 + warp * 32 + lane;
    for (int c0 = 0; c0 < NT; c0 += 32) {
        unsigned r[32];
        tc5::ld32(tmem + ((unsigned)(warp * 32) << 16) + (unsigned)c0, r);
        if (!good || row >= rows) continue;
        float* o = g.out + ((long long)blockIdx.z * rows + row) * g.nout + c0;
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (c0 + 4 * q < g.nout)
                reinterpret_cast<float4*>(o)[q] = make_float4(__uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1]),
                                                              __uint_as_float(r[4 * q + 2]), __uint_as_float(r[4 * q + 3]));
    }
    if (threadIdx.x == 0 && !good && nkb > 0) {
        atomicAdd(g.status, 1);
        for (int kb = consumed; kb < issued; ++kb) mbar_wait(&full[kb % kWgStages], (unsigned)((kb / kWgStages) & 1));
    }
    tc5::fence_before();
    __syncthreads();
    if (warp == 0) tc5::dealloc(tmem, TCOLS);
}

// ---------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------
CUtensorMapSwizzle swizzle_mode(int bytes)
{
    return bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
}
int chunk_of(int c) { return c % 64 == 0 ? 64 : c % 32 == 0 ? 32 : 16; }
int lg2(int v)
{
    int l = 0;
    while ((1 << l) < v) ++l;
    return l;
}

// image [B][H][H][C], box ck channels x `pixels` consecutive pixels
bool image_map(CUtensorMap* m, const bf16* base, int B, int H, int C, int ck, int pixels)
{
    EncodeTiled fn = tensor_map_encoder();
    if (!fn || !base) return false;
    // kLinePx: a line of k_conv_line, wider than the image at H = 128 (zero fill)
    const int tw = pixels == kLinePx ? kLinePx : std::min(H, pixels);
    const int th = pixels == kLinePx ? 1 : std::min(H, pixels / tw), tb = pixels == kLinePx ? 1 : pixels / (tw * th);
    cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)H, (cuuint64_t)H, (cuuint64_t)B};
    cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)H * C * 2, (cuuint64_t)H * H * C * 2};
    cuuint32_t box[4] = {(cuuint32_t)ck, (cuuint32_t)tw, (cuuint32_t)th, (cuuint32_t)tb};
    cuuint32_t es[4] = {1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16*>(base), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_mode(2 * ck), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
bool matrix_map(CUtensorMap* m, const bf16* base, int cols, int rows, int ck, int box_rows)
{
    EncodeTiled fn = tensor_map_encoder();
    if (!fn || !base) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    cuuint32_t box[2] = {(cuuint32_t)ck, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16*>(base), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_mode(2 * ck), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int NT, int CKB, bool DG>
cudaError_t run_conv(ConvArgs& g, const bf16* img, int B, cudaStream_t st)
{
    const size_t a = (size_t)kBM * CKB, b = (size_t)NT * CKB;
    const size_t w = (size_t)9 * g.taps_c * b;
    const int C = g.ck * g.taps_c;
    g.ntiles_n = (g.nout + NT - 1) / NT;
    const long long mtiles = (g.P + kBM - 1) / kBM;
    g.tiles = mtiles * g.ntiles_n;
    const long long per_n = std::max(1LL, std::min(mtiles, (long long)(sm_count() / g.ntiles_n)));
    const unsigned grid = (unsigned)(per_n * g.ntiles_n);
    // whole lines where a tile is 128 pixels of one grid row and the weights leave room for
    // four lines (three in use, one in flight)
    const size_t line = (size_t)g.taps_c * ((kLinePx * CKB + 1023) / 1024 * 1024);
    if (g.H >= kBM && w + 4 * line <= kConvSmem - 1024) {
        if (!image_map(&g.x, img, B, g.H, C, g.ck, kLinePx)) return cudaErrorInvalidValue;
        g.stages = (int)std::min<size_t>(kMaxStages, (kConvSmem - 1024 - w) / line);
        cudaError_t e =
            cudaFuncSetAttribute(k_conv_line<NT, CKB, DG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kConvSmem);
        if (e != cudaSuccess) return e;
        k_conv_line<NT, CKB, DG><<<grid, kConvThreads, 1024 + w + g.stages * line, st>>>(g);
        return cudaGetLastError();
    }
    if (!image_map(&g.x, img, B, g.H, C, g.ck, kBM)) return cudaErrorInvalidValue;
    // the weights stay resident while they leave the ring at least six stages
    g.resident = w + 6 * a <= kConvSmem - 1024 ? 1 : 0;
    const size_t stage = a + (g.resident ? 0 : b);
    g.stages = (int)std::min<size_t>(kMaxStages, (kConvSmem - 1024 - (g.resident ? w : 0)) / stage);
    const size_t smem = 1024 + (g.resident ? w : 0) + g.stages * stage;
    cudaError_t e = cudaFuncSetAttribute(k_conv<NT, CKB, DG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kConvSmem);
    if (e != cudaSuccess) return e;
    k_conv<NT, CKB, DG><<<grid, kConvThreads, smem, st>>>(g);
    return cudaGetLastError();
}
template <int NT, bool DG>
cudaError_t run_conv_n(ConvArgs& g, const bf16* img, int B, cudaStream_t st)
{
    switch (g.ck) {
        case 64: return run_conv<NT, 128, DG>(g, img, B, st);
        case 32: return run_conv<NT, 64, DG>(g, img, B, st);
        default: return run_conv<NT, 32, DG>(g, img, B, st);
    }
}

template <int NT, int UA, int UB>
cudaError_t run_wgrad(const WgradArgs& g, int splits, cudaStream_t st)
{
    constexpr size_t smem = 1024 + (size_t)kWgStages * (256 / UA * 64 * UA + NT * 2 / UB * 64 * UB);
    cudaError_t e = cudaFuncSetAttribute(k_wgrad<NT, UA, UB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_wgrad<NT, UA, UB><<<dim3((unsigned)((9 * g.cin + kBM - 1) / kBM), 1, (unsigned)splits), 128, smem, st>>>(g);
    return cudaGetLastError();
}
template <int NT, int UB>
cudaError_t run_wgrad_a(const WgradArgs& g, int ua, int splits, cudaStream_t st)
{
    switch (ua) {
        case 64: return run_wgrad<NT, 128, UB>(g, splits, st);
        case 32: return run_wgrad<NT, 64, UB>(g, splits, st);
        default: return run_wgrad<NT, 32, UB>(g, splits, st);
    }
}

}  // namespace

cudaError_t tc_conv_fwd(const bf16* X, int B, int H, int cin, const bf16* W, int cout, const float* bias, bf16* Y,
                        int* status, long long wait_ns, cudaStream_t st)
{
    ConvArgs g;
    std::memset(&g, 0, sizeof(g));
    const int nt = cout <= 32 ? 32 : cout <= 64 ? 64 : cout <= 128 ? 128 : 256;
    g.ck = chunk_of(cin);
    if (!matrix_map(&g.w, W, 9 * cin, cout, g.ck, nt)) return cudaErrorInvalidValue;
    g.P = (long long)B * H * H;
    g.H = H;
    g.lgH = lg2(H);
    g.taps_c = cin / g.ck;
    g.wtap_k = cin;
    g.sign = 1;
    g.nout = cout;
    g.bias = bias;
    g.out = Y;
    g.status = status;
    g.wait_ns = wait_ns;
    switch (nt) {
        case 32: return run_conv_n<32, false>(g, X, B, st);
        case 64: return run_conv_n<64, false>(g, X, B, st);
        case 128: return run_conv_n<128, false>(g, X, B, st);
        default: return run_conv_n<256, false>(g, X, B, st);
    }
}

cudaError_t tc_conv_dgrad(const bf16* dZ, int B, int H, int cin, const bf16* Wt, int cout, float* dX, int* status,
                          long long wait_ns, cudaStream_t st)
{
    ConvArgs g;
    std::memset(&g, 0, sizeof(g));
    const int nt = cin % 128 == 0 ? 128 : cin % 96 == 0 ? 96 : cin % 64 == 0 ? 64 : 32;
    g.ck = chunk_of(cout);
    if (!matrix_map(&g.w, Wt, cout, 9 * cin, g.ck, nt)) return cudaErrorInvalidValue;
    g.P = (long long)B * H * H;
    g.H = H;
    g.lgH = lg2(H);
    g.taps_c = cout / g.ck;
    g.wtap_r = cin;
    g.sign = -1;
    g.nout = cin;
    g.out = dX;
    g.status = status;
    g.wait_ns = wait_ns;
    switch (nt) {
        case 32: return run_conv_n<32, true>(g, dZ, B, st);
        case 64: return run_conv_n<64, true>(g, dZ, B, st);
        case 96: return run_conv_n<96, true>(g, dZ, B, st);
        default: return run_conv_n<128, true>(g, dZ, B, st);
    }
}

cudaError_t tc_conv_wgrad(const bf16* X, const bf16* dZ, int B, int H, int cin, int cout, int splits,
                          long long k_per_split, float* part, int* status, long long wait_ns, cudaStream_t st)
{
    WgradArgs g;
    std::memset(&g, 0, sizeof(g));
    const int ua = chunk_of(cin), ub = chunk_of(cout);
    if (!image_map(&g.x, X, B, H, cin, ua, 64) || !image_map(&g.z, dZ, B, H, cout, ub, 64)) return cudaErrorInvalidValue;
    g.P = (long long)B * H * H;
    g.k_per_split = k_per_split;
    g.H = H;
    g.lgH = lg2(H);
    g.cin = cin;
    g.nout = cout;
    g.out = part;
    g.status = status;
    g.wait_ns = wait_ns;
    switch (cout) {
        case 16: return run_wgrad_a<16, 32>(g, ua, splits, st);
        case 32: return run_wgrad_a<32, 64>(g, ua, splits, st);
        case 64: return run_wgrad_a<64, 128>(g, ua, splits, st);
        case 128: return run_wgrad_a<128, 128>(g, ua, splits, st);
        case 256: return run_wgrad_a<256, 128>(g, ua, splits, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace mgmc
