// tc_gemm.cu -- BF16 GEMM on the 5th-generation (tcgen05) tensor cores:
//   C[M][N] = A[M][K] * B[N][K]^T, FP32 accumulation in tensor memory (TMEM).
//
// k_tc_gemm, for many wide tiles: persistent CTAs of 192 threads, one per SM, each computing 128 x BN
// tiles of C:
//   warp 0, lane 0: TMA producer -- 128 x 64 tiles of A and BN x 64 tiles of B
//                   (128-byte swizzled, the layout the MMA descriptors name) into
//                   a ring of stages, each stage completing on a "full" mbarrier;
//   warp 1, lane 0: MMA issuer -- 4 x tcgen05.mma (M = 128, N = BN, K = 16) per
//                   stage into one of two TMEM accumulators, then tcgen05.commit to the
//                   stage's "empty" mbarrier (frees the stage when the MMAs are done);
//   warps 2 to 5:   epilogue -- a warp reads 32 TMEM lanes (rows of the tile) with
//                   tcgen05.ld and stores them with the epilogue ops, while the issuer
//                   fills the other accumulator and the producer runs ahead into the next tile.
// Tiles are taken in groups of 16 along M, all N tiles of a group before the next group, so that
// the CTAs running together share both operands' tiles in L2.
// k_tc_gemm_tile, for the others: a CTA of 128 threads per tile, the same two roles, then all four
// warps as epilogue.  Two CTAs share an SM where BN <= 64 (80 and 96 KB), and a single tile ends
// sooner: its code is a third as long, and a launch starts with a cold instruction cache.
// What bounds them: the operands' way from L2 to shared memory, (128 + BN) 128 bytes per 128 BN 64
// products.  Both give the same bits.
// Measured (GB300, us, tile / persistent): 65536 x 256 x 2304 102.9 / 89.9, with bias, ReLU and BF16 output
// 112 / 83; 8192^3 809 / 735; 65536 x 128 x 288 29.9 / 27.7; 20000 x 256 x 288 (157 tiles) 24.6 / 23.6;
// 2000 x 512 x 2304 (32 tiles) 21.7 / 25.5; 65536 x 64 x 2304 60.6 / 65.0; 20000 x 32 x 2304 (157
// tiles, two of them in a row in five persistent CTAs) 18.5 / 29.9.
// Every mbarrier wait is bounded (1 s).  When one gives up the other roles stop, the accumulator
// in work is not handed to the epilogue (so what a warp stores, 32 rows of a tile, is always whole), the
// CTA waits (bounded) for its MMAs and copies in flight, counts the event in *status, frees
// its TMEM and ends.
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cstring>

#include "tc5.cuh"
#include "tc_gemm.cuh"

namespace mgmc {

namespace {

// give-ups of the kernels launched without a status word of their own
__device__ int g_gave_up;

using tc5::RingPos;

constexpr int kBM = 128;
constexpr int kBK = 64;        // one 128-byte swizzle row of BF16
constexpr int kThreads = 192;
constexpr int kGroupM = 16;    // tiles along M taken together

template <int BN, bool TILE>
constexpr int gemm_stages()
{
    return TILE || BN == 256 ? 4 : 6;
}
template <int BN, bool TILE>
constexpr size_t gemm_smem()
{
    return (size_t)gemm_stages<BN, TILE>() * (kBM * kBK * 2 + BN * kBK * 2) + 1024;  // + alignment slack
}

// tile t: K split z (slowest), group of kGroupM tiles along M, N tile, M tile of the group
struct Tile {
    int m0, n0, z, kbeg, nkb;
};
template <int BN>
__device__ __forceinline__ Tile tile_at(long long t, int M, int N, int K, int k_per_split)
{
    const int mt = (M + kBM - 1) / kBM, nt = (N + BN - 1) / BN;
    Tile T;
    T.z = (int)(t / ((long long)mt * nt));
    const long long r = t - (long long)T.z * mt * nt;
    const int g = (int)(r / ((long long)kGroupM * nt));
    const int q = (int)(r - (long long)g * kGroupM * nt);
    const int gm = min(kGroupM, mt - g * kGroupM);
    T.m0 = (g * kGroupM + q % gm) * kBM;
    T.n0 = q / gm * BN;
    T.kbeg = T.z * k_per_split;
    const int kend = min(K, T.kbeg + k_per_split);
    T.nkb = (kend - T.kbeg + kBK - 1) / kBK;   // at least one (tc_gemm_plan)
    return T;
}

// one tile from the accumulator at `tmem`: this warp's 32 rows; vec: the rows of C start on 16 bytes.
// ONCE: the CTA takes one tile, so the code is kept short (a launch starts with a cold instruction
// cache: unrolled over the tile's columns, with the element stores unrolled, a tile of BN = 256 took
// 2.5 us longer)
template <int BN, bool ONCE>
__device__ __forceinline__ void gemm_epilogue(unsigned tmem, const Tile& T, void* C, int M, int N, int epi,
                                              bool vec, const float* __restrict__ bias)
{
    const int quarter = (threadIdx.x >> 5) & 3;   // TMEM lanes 32 (warp % 4) .. + 31 are the warp's
    const int row = T.m0 + quarter * 32 + (int)(threadIdx.x & 31);
    auto chunk = [&](int c0) {
        unsigned r[32];
        tc5::ld32(tmem + ((unsigned)(quarter * 32) << 16) + (unsigned)c0, r);
        const int col0 = T.n0 + c0;
        if (row >= M || col0 >= N) return;
        float v[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            float x = __uint_as_float(r[j]);
            if ((epi & kEpiBias) && col0 + j < N) x += bias[col0 + j];
            if (epi & kEpiRelu) x = fmaxf(x, 0.f);
            v[j] = x;
        }
        if (epi & kEpiBF16) {
            __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(C) + (long long)row * N + col0;
            if (vec && col0 + 32 <= N) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    __nv_bfloat162 h[4];
#pragma unroll
                    for (int t = 0; t < 4; ++t) h[t] = __floats2bfloat162_rn(v[8 * q + 2 * t], v[8 * q + 2 * t + 1]);
                    *reinterpret_cast<uint4*>(out + 8 * q) = *reinterpret_cast<uint4*>(h);
                }
            } else if constexpr (ONCE) {
                for (int j = 0; j < 32 && col0 + j < N; ++j) out[j] = __float2bfloat16_rn(v[j]);
            } else {
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    if (col0 + j < N) out[j] = __float2bfloat16_rn(v[j]);
            }
        } else {
            float* out = reinterpret_cast<float*>(C) + (long long)T.z * M * N + (long long)row * N + col0;
            if (vec && col0 + 32 <= N) {
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    *reinterpret_cast<float4*>(out + 4 * q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            } else if constexpr (ONCE) {
                for (int j = 0; j < 32 && col0 + j < N; ++j) out[j] = v[j];
            } else {
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    if (col0 + j < N) out[j] = v[j];
            }
        }
    };
    if constexpr (ONCE) {
#pragma unroll 1
        for (int c0 = 0; c0 < BN; c0 += 32) chunk(c0);
    } else {
        for (int c0 = 0; c0 < BN; c0 += 32) chunk(c0);
    }
}

template <int BN>
__global__ void __launch_bounds__(kThreads, 1)
    k_tc_gemm(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, void* C, int M,
              int N, int K, int k_per_split, long long tiles, int epi, int vec, const float* __restrict__ bias, int* status,
              long long wait_ns)
{
    constexpr int A_BYTES = kBM * kBK * 2;
    constexpr int STAGE_BYTES = A_BYTES + BN * kBK * 2;
    constexpr int S = gemm_stages<BN, false>();
    constexpr unsigned TCOLS = 2 * BN;
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    // 128-byte-swizzled operand tiles start on 1024-byte boundaries
    unsigned char* sm = smem_align_up<1024>(smem_dyn);
    __shared__ unsigned long long full[S], empty[S], tfull[2], tempty[2], drained;
    __shared__ unsigned tmem_slot;
    __shared__ volatile int aborted;
    __shared__ int issued, consumed;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s]);
            mbar_init(&empty[s]);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b]);
            mbar_init_count(&tempty[b], 4);
        }
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
    const long long lim = tc5::role_limit(wait_ns);

    if (warp == 0 && lane == 0) {
        int k = 0;
        RingPos rp;
        for (long long t = blockIdx.x; t < tiles && !aborted; t += gridDim.x) {
            const Tile T = tile_at<BN>(t, M, N, K, k_per_split);
            for (int kb = 0; kb < T.nkb; ++kb, ++k, rp.next(S)) {
                // a fresh barrier counts as past its phase of parity 1: the first use does not wait
                if (!mbar_wait(&empty[rp.slot], rp.par ^ 1u, lim)) {
                    aborted = 1;
                    break;
                }
                unsigned char* st = sm + rp.slot * STAGE_BYTES;
                mbar_expect_tx(&full[rp.slot], STAGE_BYTES);
                tma_load_2d(st, &mapA, T.kbeg + kb * kBK, T.m0, &full[rp.slot]);
                tma_load_2d(st + A_BYTES, &mapB, T.kbeg + kb * kBK, T.n0, &full[rp.slot]);
                issued = k + 1;
            }
        }
    } else if (warp == 1 && lane == 0) {
        const unsigned id = tc5::idesc(BN, false);
        int k = 0;
        RingPos rp, bp;
        bool ok = wait_ns >= 0;
        for (long long t = blockIdx.x; t < tiles && ok && !aborted; t += gridDim.x, bp.next(2)) {
            const Tile T = tile_at<BN>(t, M, N, K, k_per_split);
            if (!mbar_wait(&tempty[bp.slot], bp.par ^ 1u)) {
                ok = false;
                break;
            }
            tc5::fence_after();
            for (int kb = 0; kb < T.nkb; ++kb, ++k, rp.next(S)) {
                if (!mbar_wait(&full[rp.slot], rp.par)) {
                    ok = false;
                    break;
                }
                tc5::fence_after();
                const unsigned sa = smem_addr(sm + rp.slot * STAGE_BYTES);
                const unsigned long long da = tc5::desc(sa, 16, 1024, tc5::swizzle_of(128));
                const unsigned long long db = tc5::desc(sa + A_BYTES, 16, 1024, tc5::swizzle_of(128));
#pragma unroll
                for (int q = 0; q < kBK / 16; ++q)  // K = 16 per MMA: 32 bytes along the swizzled row
                    tc5::mma(tmem + (unsigned)(bp.slot * BN), da + 2ull * q, db + 2ull * q, id, (kb > 0 || q > 0) ? 1u : 0u);
                tc5::commit(&empty[rp.slot]);
                consumed = k + 1;
            }
            if (!ok) break;   // an incomplete accumulator never reaches the epilogue
            tc5::commit(&tfull[bp.slot]);
        }
        if (!ok) aborted = 1;
    } else if (warp >= 2) {
        bool ok = true;
        RingPos bp;
        for (long long t = blockIdx.x; t < tiles; t += gridDim.x, bp.next(2)) {
            // the lanes leave the loop together: tcgen05.ld is a warp's
            if (__any_sync(0xffffffffu, aborted)) break;
            ok = mbar_wait(&tfull[bp.slot], bp.par, lim);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc5::fence_after();
            gemm_epilogue<BN, false>(tmem + (unsigned)(bp.slot * BN), tile_at<BN>(t, M, N, K, k_per_split), C, M, N, epi, vec != 0,
                              bias);
            tc5::fence_before();
            __syncwarp();
            if (lane == 0) tc5::arrive(&tempty[bp.slot]);
        }
        if (!ok && lane == 0) aborted = 1;
    }
    __syncwarp();
    __syncthreads();
    if (aborted) {
        // MMAs issued and copies never consumed may still be in flight: wait for them (bounded)
        if (threadIdx.x == 32) {
            tc5::commit(&drained);
            mbar_wait(&drained, 0u);
        }
        if (threadIdx.x == 0) {
            for (int k = consumed; k < issued; ++k) mbar_wait(&full[k % S], (unsigned)((k / S) & 1));
            atomicAdd(status ? status : &g_gave_up, 1);
        }
    }
    tc5::fence_before();
    __syncthreads();
    if (warp == 0) tc5::dealloc(tmem, TCOLS);
}

// one tile per CTA: blockIdx.x = K split * M tiles + M tile, blockIdx.y = N tile
template <int BN>
__global__ void __launch_bounds__(128)
    k_tc_gemm_tile(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, void* C, int M,
                   int N, int K, int k_per_split, int epi, int vec, const float* __restrict__ bias, int* status,
                   long long wait_ns)
{
    constexpr int A_BYTES = kBM * kBK * 2;
    constexpr int STAGE_BYTES = A_BYTES + BN * kBK * 2;
    constexpr int S = gemm_stages<BN, true>();
    constexpr unsigned TCOLS = BN;
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    unsigned char* sm = smem_align_up<1024>(smem_dyn);
    __shared__ unsigned long long full[S], empty[S], done;
    __shared__ unsigned tmem_slot;
    __shared__ int aborted, issued, consumed;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Tile T;
    const unsigned mt = (unsigned)(M + kBM - 1) / kBM;
    T.z = (int)(blockIdx.x / mt);
    T.m0 = (int)(blockIdx.x - T.z * mt) * kBM;
    T.n0 = blockIdx.y * BN;
    T.kbeg = T.z * k_per_split;
    T.nkb = (min(K, T.kbeg + k_per_split) - T.kbeg + kBK - 1) / kBK;   // at least one (tc_gemm_plan)
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
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
        for (; kb < T.nkb; ++kb) {
            const int s = kb % S, use = kb / S;
            if (use > 0 && !mbar_wait(&empty[s], (unsigned)((use - 1) & 1), tc5::role_limit(wait_ns))) {
                aborted = 1;
                break;
            }
            unsigned char* st = sm + s * STAGE_BYTES;
            mbar_expect_tx(&full[s], STAGE_BYTES);
            tma_load_2d(st, &mapA, T.kbeg + kb * kBK, T.m0, &full[s]);
            tma_load_2d(st + A_BYTES, &mapB, T.kbeg + kb * kBK, T.n0, &full[s]);
        }
        issued = kb;
    } else if (warp == 1 && lane == 0) {
        const unsigned id = tc5::idesc(BN, false);
        const int n = wait_ns < 0 ? 0 : T.nkb;
        if (wait_ns < 0) aborted = 1;
        int kb = 0;
        for (; kb < n; ++kb) {
            const int s = kb % S;
            if (!mbar_wait(&full[s], (unsigned)((kb / S) & 1))) {
                aborted = 1;
                break;
            }
            tc5::fence_after();
            const unsigned sa = smem_addr(sm + s * STAGE_BYTES);
            const unsigned long long da = tc5::desc(sa, 16, 1024, tc5::swizzle_of(128));
            const unsigned long long db = tc5::desc(sa + A_BYTES, 16, 1024, tc5::swizzle_of(128));
#pragma unroll
            for (int q = 0; q < kBK / 16; ++q)
                tc5::mma(tmem, da + 2ull * q, db + 2ull * q, id, (kb > 0 || q > 0) ? 1u : 0u);
            tc5::commit(&empty[s]);
        }
        consumed = kb;
        tc5::commit(&done);   // arrives once every MMA issued above has completed
    }
    __syncwarp();
    const bool ok = mbar_wait(&done, 0u);
    tc5::fence_after();
    const bool good = __syncthreads_and(ok) && !aborted;
    if (good) {
        gemm_epilogue<BN, true>(tmem, T, C, M, N, epi, vec != 0, bias);
    } else if (threadIdx.x == 0) {
        // copies issued but never consumed may still be in flight: wait for them (bounded)
        for (int kb = consumed; kb < issued; ++kb) mbar_wait(&full[kb % S], (unsigned)((kb / S) & 1));
        atomicAdd(status ? status : &g_gave_up, 1);
    }
    tc5::fence_before();
    __syncthreads();
    if (warp == 0) tc5::dealloc(tmem, TCOLS);
}

__global__ void k_reduce_splits(const float* __restrict__ part, int splits, long long count, float* __restrict__ out)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x) {
        float acc = part[i];
        // the loads of 16 partials in flight at a time; the sum stays in order
#pragma unroll 16
        for (int z = 1; z < splits; ++z) acc += part[(long long)z * count + i];
        out[i] = acc;
    }
}

bool encode_bf16(CUtensorMap* m, const void* base, int ld, int rows, int cols, int box_rows)
{
    EncodeTiled fn = tensor_map_encoder();
    if (!fn || !base || (ld & 7) || (reinterpret_cast<uintptr_t>(base) & 15)) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// a kernel's shared-memory opt-in, once per device (each of the first 64 has a bit)
template <typename Kernel>
cudaError_t opt_in(Kernel kernel, size_t smem, std::atomic<unsigned long long>& done)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if (done.load() & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) done.fetch_or(bit);
    return e;
}

// The persistent kernel from one wide tile (BN >= 128) per SM on, one tile per CTA below and for
// narrow tiles (both sides measured in the file's header); gridDim.y takes 65 535 N tiles.
template <int BN>
cudaError_t launch(const TcGemm& g, void* C, int epi, const float* bias, int* status, long long wait_ns,
                   cudaStream_t st)
{
    const long long mt = (g.M + kBM - 1) / kBM, nt = (g.N + BN - 1) / BN, tiles = mt * nt * g.splits;
    // 16-byte stores where every row starts on 16 bytes: C and the row pitch (C may be a view)
    const size_t elem = (epi & kEpiBF16) ? 2 : 4;
    const int vec = (reinterpret_cast<uintptr_t>(C) & 15) == 0 && ((size_t)g.N * elem & 15) == 0;
    if constexpr (BN >= 128) {
        const int sms = sm_count();
        if (tiles >= sms || nt > 65535) {
            static std::atomic<unsigned long long> done{0};
            constexpr size_t smem = gemm_smem<BN, false>();
            const cudaError_t e = opt_in(k_tc_gemm<BN>, smem, done);
            if (e != cudaSuccess) return e;
            k_tc_gemm<BN><<<(unsigned)std::min<long long>(tiles, sms), kThreads, smem, st>>>(
                g.a, g.b, C, g.M, g.N, g.K, g.k_per_split, tiles, epi, vec, bias, status, wait_ns);
            return cudaGetLastError();
        }
    }
    static std::atomic<unsigned long long> done{0};
    constexpr size_t smem = gemm_smem<BN, true>();
    const cudaError_t e = opt_in(k_tc_gemm_tile<BN>, smem, done);
    if (e != cudaSuccess) return e;
    k_tc_gemm_tile<BN><<<dim3((unsigned)(mt * g.splits), (unsigned)nt), 128, smem, st>>>(
        g.a, g.b, C, g.M, g.N, g.K, g.k_per_split, epi, vec, bias, status, wait_ns);
    return cudaGetLastError();
}

}  // namespace

int sm_count()
{
    // a device's count does not change: asked for once (the first 64 devices)
    static std::atomic<int> known[64];
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    if (dev < 64 && (sms = known[dev].load()) > 0) return sms;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 1;
    if (dev < 64) known[dev].store(sms);
    return sms;
}

EncodeTiled tensor_map_encoder()
{
    static EncodeTiled fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<EncodeTiled>(p);
        return (EncodeTiled) nullptr;
    }();
    return fn;
}

bool tc_gemm_plan(TcGemm* g, const void* A, int lda, const void* B, int ldb, int M, int N, int K, int splits)
{
    std::memset(g, 0, sizeof(*g));
    if (M <= 0 || N <= 0 || K <= 0 || lda < K || ldb < K || splits < 1) return false;
    g->M = M;
    g->N = N;
    g->K = K;
    g->bn = N <= 32 ? 32 : N <= 64 ? 64 : N <= 128 ? 128 : 256;
    const int kblocks = (K + kBK - 1) / kBK;
    if (splits > kblocks) splits = kblocks;
    const int per = (kblocks + splits - 1) / splits;
    g->k_per_split = per * kBK;
    g->splits = (kblocks + per - 1) / per;  // every split has at least one K block
    return encode_bf16(&g->a, A, lda, M, K, kBM) && encode_bf16(&g->b, B, ldb, N, K, g->bn);
}

cudaError_t tc_gemm_run(const TcGemm& g, void* C, int epilogue, const float* bias, int* status, long long wait_ns,
                        cudaStream_t st)
{
    if (g.splits > 1 && epilogue != kEpiF32) return cudaErrorInvalidValue;
    switch (g.bn) {
        case 32: return launch<32>(g, C, epilogue, bias, status, wait_ns, st);
        case 64: return launch<64>(g, C, epilogue, bias, status, wait_ns, st);
        case 128: return launch<128>(g, C, epilogue, bias, status, wait_ns, st);
        default: return launch<256>(g, C, epilogue, bias, status, wait_ns, st);
    }
}

cudaError_t tc_gemm_gave_up(int* count, cudaStream_t st)
{
    cudaError_t e = cudaMemcpyFromSymbolAsync(count, g_gave_up, sizeof(int), 0, cudaMemcpyDeviceToHost, st);
    return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
}

cudaError_t tc_reduce_splits(const float* part, int splits, long long count, float* out, cudaStream_t st)
{
    long long blocks = (count + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    k_reduce_splits<<<(unsigned)blocks, 256, 0, st>>>(part, splits, count, out);
    return cudaGetLastError();
}

}  // namespace mgmc
