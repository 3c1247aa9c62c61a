// coarse.cu -- the V-cycle below and including grid `top` in one CTA (Alg. 1
// recursion for the small grids, ending in the exact coarsest Cholesky sample
// of Sec. 3.5).
//
// The state theta_l, the dense right-hand side fdense_l and the operator of every
// grid l <= top live in shared memory for the whole kernel (padded (n+2)^d blocks with
// a zero ghost ring).  The compute warps run a list of phases (a sweep, a low-rank
// step, a residual and restriction, a prolongation, the coarsest sample) the host
// writes at creation; a phase or a colour of a sweep ends in a barrier of those warps.
//
// What bounds it: the latency of a chain of ~65 dependent phases on grids of at most
// a few thousand sites, on one SM (and, in FP64, that SM's FP64 rate), so every phase
// is kept free of anything slow:
//  - everything that set-up fixed -- operator, 1/a_ii and sqrt(a_ii), observation
//    entries, the rows of G where they fit -- is one contiguous image in the layout
//    of the shared memory, written once at creation and fetched by one bulk copy
//    before the wait on the preceding launch;
//  - the noise of a cycle depends on the counter alone: all warps draw the site normals
//    of the first sweep before that wait, kHelp helper threads the others, the low-rank
//    and the coarsest normals beside the first phases;
//  - the m-vector of a low-rank step takes four lanes per observation, is rounded to
//    the path precision once, and G is k-major (coalesced, conflict free);
//  - the residual of a grid is formed once per site, then restricted;
//  - the coarsest sample is one matrix-vector product with the host's gain matrix
//    (n0 <= kCoarseGainMax): A~_0^-1 f + A~_0^-1 B_0 Gamma^-1 d + L_0^-T z, eight lanes a
//    row, instead of two triangular solves of n0 dependent steps each;
//  - n + 1 is a power of two, so a site index is decoded with shifts;
//  - the code is small (loops over items are not unrolled, the draws are functions): every
//    launch starts with a cold instruction cache, and an unrolled version of 170 KB spent
//    30 thousand cycles a launch on instruction fetches.
// The FP32 arithmetic of a site is that of stencil.cuh, with the update's last product and sum rounded apart.
// Measured (GB300, against one CTA per chain with operands staged by loads, per-sweep draws and
// triangular solves): cycle of one 31^2 FP64 chain 137 -> 73 us (52 with the normals of
// normal64.cuh), of a 255^2 FP32 chain 142 -> 97 us (90 with the low-rank launches of tile2d.cu),
// cold launch inside a batch of 32 1023^2 chains 97 -> 38 us.  What is left is the phases' own
// latency (about 600 cycles a colour, 2000 a low-rank step); grids with a compile-time size or
// only four warps on the smallest ones measured no faster.
#include <algorithm>

#include "kernels.cuh"
#include "tma.cuh"

namespace mgmc {

namespace {

constexpr int kHelp = 128;             // helper threads: draw normals beside the phases

// compute threads at most: a colour of a 63^2 grid (2D FP32) has 1024 sites, of a 31^2 one 256
template <typename T, int DIM>
__host__ __device__ constexpr int coarse_max_threads()
{
    return sizeof(T) == 4 && DIM == 2 ? 512 : 256;
}

template <int DIM>
__device__ __forceinline__ int sidx(int S, int i, int j, int k)
{
    return DIM == 3 ? ((k + 1) * S + (j + 1)) * S + (i + 1) : (j + 1) * S + (i + 1);
}

template <int DIM>
__device__ __forceinline__ int soff(int o, int S)
{
    int dx = o % 3 - 1, dy = (o / 3) % 3 - 1, dz = DIM == 3 ? o / 9 - 1 : 0;
    return dx + S * (dy + S * dz);
}

// barrier `id` of the compute warps (id 1) or of all warps
template <int ID>
__device__ __forceinline__ void bar_n(int threads)
{
    asm volatile("bar.sync %0, %1;\n" ::"n"(ID), "r"(threads) : "memory");
}
template <int ID>
__device__ __forceinline__ void bar_arrive(int threads)
{
    asm volatile("bar.arrive %0, %1;\n" ::"n"(ID), "r"(threads) : "memory");
}

// the compute threads
struct Team {
    int nt;
    __device__ __forceinline__ void sync() const { bar_n<1>(nt); }
};

// multiply-add with one rounding, and a plain product, in either precision
__device__ __forceinline__ float mad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return __fma_rn(a, b, c); }

// One grid of the kernel: sizes and its blocks in shared memory.
template <typename T>
struct Blk {
    int n, lg, S, SZ;        // lg = log2(n + 1)
    T *X, *F, *SA, *IV, *CS; // state, dense right-hand side, sqrt(a_ii), 1 / a_ii, coefficient slots (SZ apart)
    bool fine;               // 5/7-point finest grid (one slot: FP64 a_ii, FP32 s kappa^2_i)
    T w;                     // its off-diagonal magnitude
};

// a(l, l + o) from the staged coefficient blocks (slot t at CS + t * SZ)
template <int DIM, typename T>
__device__ __forceinline__ T coef_s(const Blk<T>& b, int ls, int o)
{
    constexpr int C = Offsets<DIM>::C;
    constexpr int NS = Offsets<DIM>::NS;
    if (o > C) return b.CS[(o - C) * b.SZ + ls];
    return b.CS[(NS - 1 - o - C) * b.SZ + ls + soff<DIM>(o, b.S)];
}

// What an update of a site reads besides the state: none of it changes during a sweep.
template <typename T, int DIM>
struct Site {
    T c[Offsets<DIM>::NS];   // couplings, centre = slot 0 (5/7-point grid: only the centre)
    T rhs, iv;
};

// formed: Z already holds rhs = fdense + sqrt(a_ii) z
template <int DIM, typename T>
__device__ __forceinline__ void load_site(Site<T, DIM>& s, const Blk<T>& b, int ls, T z, bool formed)
{
    constexpr int NS = Offsets<DIM>::NS;
    constexpr int C = Offsets<DIM>::C;
    s.c[C] = b.CS[ls];
    if (!b.fine) {
#pragma unroll
        for (int o = 0; o < NS; ++o)
            if (o != C) s.c[o] = coef_s<DIM>(b, ls, o);
    }
    s.iv = b.IV[ls];
    s.rhs = formed ? z : mad(b.SA[ls], z, b.F[ls]);
}

template <int DIM>
__device__ __forceinline__ double upd_s(const Site<double, DIM>& s, const Blk<double>& b, int ls)
{
    const double* X = b.X;
    constexpr int NS = Offsets<DIM>::NS;
    constexpr int C = Offsets<DIM>::C;
    if (b.fine) {
        double lo = X[ls - 1] + X[ls - b.S], hi = X[ls + 1] + X[ls + b.S];
        if (DIM == 3) {
            lo += X[ls - b.S * b.S];
            hi += X[ls + b.S * b.S];
        }
        return mad(b.w, lo + hi, s.rhs) * s.iv;
    }
    // the couplings before and after the centre are summed separately: half the chain
    double lo = s.rhs, hi = 0.0;
#pragma unroll
    for (int o = 0; o < C; ++o) {
        lo = mad(-s.c[o], X[ls + soff<DIM>(o, b.S)], lo);
        hi = mad(-s.c[NS - 1 - o], X[ls + soff<DIM>(NS - 1 - o, b.S)], hi);
    }
    return (lo + hi) * s.iv;
}

// FP32: x + (rhs - A x) / a_ii
template <int DIM>
__device__ __forceinline__ float upd_s(const Site<float, DIM>& s, const Blk<float>& b, int ls)
{
    const float* X = b.X;
    const float xi = X[ls];
    constexpr int NS = Offsets<DIM>::NS;
    constexpr int C = Offsets<DIM>::C;
    float Ax;
    if (b.fine) {
        float lap = (xi - X[ls - b.S]) + (xi - X[ls - 1]) + (xi - X[ls + 1]) + (xi - X[ls + b.S]);
        if (DIM == 3) lap += (xi - X[ls - b.S * b.S]) + (xi - X[ls + b.S * b.S]);
        Ax = fmaf(s.c[C], xi, b.w * lap);
    } else {
        float lap = 0.0f;
#pragma unroll
        for (int o = 0; o < NS; ++o)
            if (o != C) lap = fmaf(s.c[o], X[ls + soff<DIM>(o, b.S)] - xi, lap);
        Ax = fmaf(s.c[C], xi, lap);
    }
    // product and sum rounded apart, so that the bits do not depend on what the compiler contracts
    // (contracted, the error against 64 bits is the same: median ratio 1.0 over 30 seeds and 3 sizes)
    return __fadd_rn(xi, __fmul_rn(s.rhs - Ax, s.iv));
}

// (A x) of the dense part at ls
template <int DIM>
__device__ __forceinline__ double Ax_s(const Blk<double>& b, int ls)
{
    const double* X = b.X;
    if (b.fine) {
        double lo = X[ls - 1] + X[ls - b.S], hi = X[ls + 1] + X[ls + b.S];
        if (DIM == 3) {
            lo += X[ls - b.S * b.S];
            hi += X[ls + b.S * b.S];
        }
        return mad(b.CS[ls], X[ls], -b.w * (lo + hi));
    }
    constexpr int NS = Offsets<DIM>::NS;
    constexpr int C = Offsets<DIM>::C;
    double lo = b.CS[ls] * X[ls], hi = 0.0;
#pragma unroll
    for (int o = 0; o < C; ++o) {
        lo = mad(coef_s<DIM>(b, ls, o), X[ls + soff<DIM>(o, b.S)], lo);
        hi = mad(coef_s<DIM>(b, ls, NS - 1 - o), X[ls + soff<DIM>(NS - 1 - o, b.S)], hi);
    }
    return lo + hi;
}

template <int DIM>
__device__ __forceinline__ float Ax_s(const Blk<float>& b, int ls)
{
    const float* X = b.X;
    const float xi = X[ls];
    if (b.fine) {
        float lap = (xi - X[ls - b.S]) + (xi - X[ls - 1]) + (xi - X[ls + 1]) + (xi - X[ls + b.S]);
        if (DIM == 3) lap += (xi - X[ls - b.S * b.S]) + (xi - X[ls + b.S * b.S]);
        return fmaf(b.CS[ls], xi, b.w * lap);
    }
    constexpr int NS = Offsets<DIM>::NS;
    constexpr int C = Offsets<DIM>::C;
    float lap = 0.0f;
#pragma unroll
    for (int o = 0; o < NS; ++o)
        if (o != C) lap = fmaf(coef_s<DIM>(b, ls, o), X[ls + soff<DIM>(o, b.S)] - xi, lap);
    return fmaf(b.CS[ls], xi, lap);
}

// the it-th item of a cube of side 2^lg
template <int DIM>
__device__ __forceinline__ void cube(int it, int lg, int& i, int& j, int& k)
{
    const int mask = (1 << lg) - 1;
    i = it & mask;
    j = (it >> lg) & mask;
    k = DIM == 3 ? it >> (2 * lg) : 0;
}

// site normals of 4-site group `blk` of one sweep into Z[4 blk ..] in column order (row
// (k, j) of the grid at Z + (k n + j) 4 nq); zeros without noise
template <typename T>
__device__ __noinline__ void draw_group(const CycleState* csp, int level, unsigned slot, T* Z, int blk)
{
    const CycleState& cs = *csp;
    T a0 = T(0), a1 = T(0), b0 = T(0), b1 = T(0);
    if (cs.noise)
        draw_quad_ctr<T>(noise_counter(cs, 0u, 0u, level, slot), (unsigned)blk, (unsigned)cs.seed,
                         (unsigned)(cs.seed >> 32), a0, a1, b0, b1);
    T* z = Z + 4 * blk;
    z[0] = a0;
    z[1] = b0;
    z[2] = a1;
    z[3] = b1;
}

// pair `pair` of the low-rank normals of grid l's sweep `slot` (kind 1) / the coarsest normals (kind 2)
template <typename T>
__device__ __noinline__ void draw_pair_at(const CycleState* csp, unsigned pair, unsigned kind, int l, unsigned slot,
                                          double* out)
{
    T z0 = T(0), z1 = T(0);
    if (csp->noise) draw_pair<T>(*csp, pair, kind, l, slot, z0, z1);
    out[0] = (double)z0;
    out[1] = (double)z1;
}

template <int DIM>
__device__ __forceinline__ int sweep_groups(int n)
{
    return ((n + 3) >> 2) * n * (DIM == 3 ? n : 1);
}

// The colours of one sweep; Z holds the normals (formed: the right-hand sides).
template <int DIM, typename T>
__device__ __forceinline__ void s_sweep(const Blk<T>& b, const T* Z, bool formed, int dir, const Team& tm)
{
    // colour orders (0, 3, 2, 1) and (0, 6, 5, 3, 4, 2, 1, 7) as packed nibbles (no local-memory table)
    constexpr int NCOL = DIM == 2 ? 4 : 8;
    const int n = b.n, ld = ((n + 3) >> 2) << 2;
    const int lh = b.lg - 1, items = 1 << (DIM * lh);
    auto colour = [&](int ci) {
        return (int)(((DIM == 2 ? 0x1230u : 0x71243560u) >> (4 * (dir == 0 ? ci : NCOL - 1 - ci))) & 0xFu);
    };
    // site of item `it` of colour c: shared index ls and normal index zi; false outside the grid
    auto site = [&](int it, int c, int& ls, int& zi) {
        int i, j, k;
        cube<DIM>(it, lh, i, j, k);
        i = 2 * i + (c & 1);
        j = 2 * j + ((c >> 1) & 1);
        k = DIM == 3 ? 2 * k + ((c >> 2) & 1) : 0;
        ls = sidx<DIM>(b.S, i, j, k);
        zi = ((DIM == 3 ? k * n : 0) + j) * ld + i;
        return i < n && j < n && (DIM == 2 || k < n);
    };
#pragma unroll 1
    for (int ci = 0; ci < NCOL; ++ci) {
        const int c = colour(ci);
#pragma unroll 1
        for (int it = threadIdx.x; it < items; it += tm.nt) {
            int ls, zi;
            if (!site(it, c, ls, zi)) continue;
            Site<T, DIM> s;
            load_site<DIM>(s, b, ls, Z[zi], formed);
            b.X[ls] = upd_s<DIM>(s, b, ls);
        }
        tm.sync();
    }
}

// Low-rank area of the dynamic shared memory (see CoarsePlan).
template <typename T>
struct LrArea {
    double *d, *zlr, *zp, *v, *z, *vec, *zc;
    const double* w;
    const int *ss, *ptr;
    T* vt;
};

// theta' = theta*_s - G (B^T theta*_s - d - L_Gamma z') (dir >= 0); with want_dnext
// also d_{l-1} = d_l - B^T theta' = d_l - z + (B^T G) v.  lz: L_Gamma z' (zeros without
// noise).  Sites are shared-memory indices; G is applied in the path precision.
template <typename T>
__device__ __forceinline__ void s_lowrank(const DevLevel<T>& L, const CoarseJob<T>& J, const LrArea<T>& A,
                                          const unsigned char* smem, int m, int l, T* X, int dir, bool want_dnext,
                                          const double* lz, const Team& tm)
{
    const int tid = threadIdx.x;
    const int rows = dir >= 0 ? L.g_rows[dir] : 0;
    const bool sg = J.plan.g_off[l] >= 0;   // G staged: direction 0's columns, then direction 1's
    const T* G = nullptr;                   // k-major: column k at G + k * rows
    const int* gsite = nullptr;
    if (dir >= 0) {
        G = sg ? reinterpret_cast<const T*>(smem + J.plan.g_off[l]) + (dir ? (size_t)L.g_rows[0] * m : 0) : L.gT[dir];
        gsite = sg ? reinterpret_cast<const int*>(smem + J.plan.gs_off[l]) + (dir ? L.g_rows[0] : 0) : L.g_ss[dir];
    }
    // the thread's first row of an unstaged G, issued before z and v are formed
    constexpr int kPre = sizeof(T) == 4 ? 16 : 8;
    T gr[kPre];
    if (!sg && tid < rows) {
#pragma unroll
        for (int k = 0; k < kPre; ++k) gr[k] = k < m ? G[k * rows + tid] : T(0);
    }
    const int gs = tid < rows ? gsite[tid] : 0;
    double* d = A.d + l * m;
#pragma unroll 1
    for (int q = tid; q < ((4 * m + 31) & ~31); q += tm.nt) {
        const int k = q >> 2, p = q & 3;
        double acc = 0.0;
        const double dl = k < m ? d[k] + lz[k] : 0.0;
        if (k < m) {
            if (J.plan.stage_ent) {
                const int* ptr = A.ptr + l * (m + 1);
#pragma unroll 1
                for (int t = ptr[k] + p; t < ptr[k + 1]; t += 4) acc = mad(A.w[t], (double)X[A.ss[t]], acc);
            } else {
#pragma unroll 1
                for (int t = L.bcol_ptr[k] + p; t < L.bcol_ptr[k + 1]; t += 4)
                    acc = mad(L.bcol_w[t], (double)X[L.bcol_ss[t]], acc);
            }
        }
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        if (p == 0 && k < m) {
            const double v = acc - dl;
            A.vt[k] = (T)v;
            A.v[k] = v;
            A.z[k] = acc;
        }
    }
    tm.sync();
    if (tid < rows) {
        T acc = T(0);
        if (sg) {
#pragma unroll 8
            for (int k = 0; k < m; ++k) acc = mad(G[k * rows + tid], A.vt[k], acc);
        } else {
#pragma unroll
            for (int k = 0; k < kPre; ++k)
                if (k < m) acc = mad(gr[k], A.vt[k], acc);
#pragma unroll 1
            for (int k = kPre; k < m; ++k) acc = mad(G[k * rows + tid], A.vt[k], acc);
        }
        X[gs] = X[gs] - acc;
    }
#pragma unroll 1
    for (int r = tid + tm.nt; r < rows; r += tm.nt) {
        T acc = T(0);
#pragma unroll 4
        for (int k = 0; k < m; ++k) acc = mad(G[k * rows + r], A.vt[k], acc);
        const int s = gsite[r];
        X[s] = X[s] - acc;
    }
    if (want_dnext) {
        // four lanes per entry, by the last warps
#pragma unroll 1
        for (int q = tm.nt - 1 - tid; q < ((4 * m + 31) & ~31); q += tm.nt) {
            const int k = q >> 2, p = q & 3;
            double acc = 0.0;
            if (dir >= 0 && k < m)
#pragma unroll 4
                for (int t = p; t < m; t += 4) acc = mad(L.BtG[k * m + t], A.v[t], acc);
            acc += __shfl_xor_sync(0xffffffffu, acc, 1);
            acc += __shfl_xor_sync(0xffffffffu, acc, 2);
            if (p == 0 && k < m) A.d[(l - 1) * m + k] = d[k] - A.z[k] + acc;
        }
    }
    tm.sync();
}

// f_{l-1} = P^T (fdense_l - A theta): the residual once per site into R (laid out like the
// normals of a sweep), then the weighted sums
template <int DIM, typename T>
__device__ __forceinline__ void s_restrict(const Blk<T>& b, T* R, const Blk<T>& c, const Team& tm)
{
    const int n = b.n, ld = ((n + 3) >> 2) << 2;
#pragma unroll 1
    for (int it = threadIdx.x; it < (1 << (DIM * b.lg)); it += tm.nt) {
        int i, j, k;
        cube<DIM>(it, b.lg, i, j, k);
        if (i >= n || j >= n || (DIM == 3 && k >= n)) continue;
        const int ls = sidx<DIM>(b.S, i, j, k);
        R[((DIM == 3 ? k * n : 0) + j) * ld + i] = b.F[ls] - Ax_s<DIM>(b, ls);
    }
    tm.sync();
    const int nc = c.n;
#pragma unroll 1
    for (int it = threadIdx.x; it < (1 << (DIM * c.lg)); it += tm.nt) {
        int I, Jc, K;
        cube<DIM>(it, c.lg, I, Jc, K);
        if (I >= nc || Jc >= nc || (DIM == 3 && K >= nc)) continue;
        T acc = T(0);
#pragma unroll
        for (int pz = 0; pz < (DIM == 3 ? 3 : 1); ++pz)
#pragma unroll
            for (int py = 0; py < 3; ++py)
#pragma unroll
                for (int px = 0; px < 3; ++px) {
                    const T wgt = (T)(pw(px - 1) * pw(py - 1) * (DIM == 3 ? pw(pz - 1) : 1.0));
                    acc = mad(wgt, R[((DIM == 3 ? (2 * K + pz) * n : 0) + 2 * Jc + py) * ld + 2 * I + px], acc);
                }
        c.F[sidx<DIM>(c.S, I, Jc, K)] = acc;
    }
    tm.sync();
}

// theta += P psi: item (I, J[, K]) updates the fine sites 2I, 2I + 1 per axis from the
// coarse sites I - 1, I (fine index 2I: their mean; 2I + 1: coarse I); ghosts are zero
template <int DIM, typename T>
__device__ __forceinline__ void s_prolong(const Blk<T>& c, const Blk<T>& b, const Team& tm)
{
    const int n = b.n;
    constexpr int NZ = DIM == 3 ? 2 : 1;
#pragma unroll 1
    for (int it = threadIdx.x; it < (1 << (DIM * (b.lg - 1))); it += tm.nt) {
        int I, J, K;
        cube<DIM>(it, b.lg - 1, I, J, K);
        T v[NZ][2][2];
#pragma unroll
        for (int a = 0; a < NZ; ++a)
#pragma unroll
            for (int bb = 0; bb < 2; ++bb)
#pragma unroll
                for (int cc = 0; cc < 2; ++cc)
                    v[a][bb][cc] = c.X[sidx<DIM>(c.S, I - 1 + cc, J - 1 + bb, DIM == 3 ? K - 1 + a : 0)];
#pragma unroll
        for (int dz = 0; dz < NZ; ++dz)
#pragma unroll
            for (int dy = 0; dy < 2; ++dy)
#pragma unroll
                for (int dx = 0; dx < 2; ++dx) {
                    const int i = 2 * I + dx, j = 2 * J + dy, k = DIM == 3 ? 2 * K + dz : 0;
                    if (i >= n || j >= n || (DIM == 3 && k >= n)) continue;
                    T acc = T(0);
#pragma unroll
                    for (int a = DIM == 3 ? dz : 0; a < NZ; ++a)
#pragma unroll
                        for (int bb = dy; bb < 2; ++bb)
#pragma unroll
                            for (int cc = dx; cc < 2; ++cc)
                                acc = mad((DIM == 3 && !dz ? T(0.5) : T(1)) * (dy ? T(1) : T(0.5)) *
                                              (dx ? T(1) : T(0.5)),
                                          v[a][bb][cc], acc);
                    const int ls = sidx<DIM>(b.S, i, j, k);
                    b.X[ls] = b.X[ls] + acc;
                }
    }
}

// theta_0 = A~_0^-1 f_0 + L_0^-T z with f_0 = fdense_0 + B_0 Gamma^-1 d_0 (FP64).  zc: the
// standard normals z (zeros without noise).
template <int DIM, typename T>
__device__ __forceinline__ void s_coarsest(const CoarseJob<T>& J, int m, const Blk<T>& b, const double* d, double* vec,
                                           const double* zc, const Team& tm)
{
    const int n = b.n, n0 = J.n0;
    auto at = [&](int s) {
        const int i = s % n, j = (s / n) % n, k = DIM == 3 ? s / (n * n) : 0;
        return sidx<DIM>(b.S, i, j, k);
    };
    if (J.gain) {
        // rows of the gain matrix [A~_0^-1 | A~_0^-1 B_0 Gamma^-1 | L_0^-T] times (fdense_0, d_0, z)
        const int len = 2 * n0 + m;
#pragma unroll 1
        for (int s = threadIdx.x; s < len; s += tm.nt)
            vec[s] = s < n0 ? (double)b.F[at(s)] : (s < n0 + m ? d[s - n0] : zc[s - n0 - m]);
        tm.sync();
#pragma unroll 1
        for (int q = threadIdx.x; q < ((8 * n0 + 31) & ~31); q += tm.nt) {
            const int s = q >> 3, p = q & 7;
            double acc = 0.0;
            if (s < n0) {
                const double* g = J.gain + s * len;
#pragma unroll 4
                for (int t = p; t < len; t += 8) acc = mad(g[t], vec[t], acc);
            }
            acc += __shfl_xor_sync(0xffffffffu, acc, 1);
            acc += __shfl_xor_sync(0xffffffffu, acc, 2);
            acc += __shfl_xor_sync(0xffffffffu, acc, 4);
            if (p == 0 && s < n0) b.X[at(s)] = (T)acc;
        }
        tm.sync();
        return;
    }
    // larger coarsest grids: two triangular solves, the CTA updating the remaining unknowns.  Thread 0's
    // next diagonal entry is loaded a step ahead, a thread's loads of the factor two at a time (a cycle
    // with 961 coarsest unknowns in FP64 / FP32, 225 in FP64: 1657 / 1565 / 324 us; one load after the other
    // 2060 / 1774 / 345.  Four at a time: 83 registers in FP32, and one CTA per SM instead of two)
    double* r = vec;
    const double* chol = J.chol;
#pragma unroll 1
    for (int s = threadIdx.x; s < n0; s += tm.nt) {
        double acc = (double)b.F[at(s)];
#pragma unroll 4
        for (int k = 0; k < m; ++k) acc += J.e0[(long long)k * n0 + s] * d[k];   // (B_0 Gamma^-1 d)_s
        r[s] = acc;
    }
    tm.sync();
    double diag = chol[0];   // thread 0 divides
#pragma unroll 1
    for (int i = 0; i < n0; ++i) {
        if (threadIdx.x == 0) r[i] = r[i] / diag;
        tm.sync();
        if (threadIdx.x == 0 && i + 1 < n0) diag = chol[(i + 1) * (n0 + 1)];
        const double yi = r[i];
#pragma unroll 1
        for (int t = i + 1 + threadIdx.x; t < n0; t += 2 * tm.nt) {
            const int u = t + tm.nt;
            const double ct = chol[t * n0 + i], cu = u < n0 ? chol[u * n0 + i] : 0.0;
            r[t] -= ct * yi;
            if (u < n0) r[u] -= cu * yi;
        }
        tm.sync();
    }
#pragma unroll 1
    for (int s = threadIdx.x; s < n0; s += tm.nt) r[s] += zc[s];
    tm.sync();
    diag = chol[n0 * n0 - 1];
#pragma unroll 1
    for (int i = n0 - 1; i >= 0; --i) {
        if (threadIdx.x == 0) r[i] = r[i] / diag;
        tm.sync();
        if (threadIdx.x == 0 && i > 0) diag = chol[(i - 1) * (n0 + 1)];
        const double xi = r[i];
#pragma unroll 1
        for (int t = threadIdx.x; t < i; t += 2 * tm.nt) {
            const int u = t + tm.nt;
            const double ct = chol[i * n0 + t], cu = u < i ? chol[i * n0 + u] : 0.0;
            r[t] -= ct * xi;
            if (u < i) r[u] -= cu * xi;
        }
        tm.sync();
    }
#pragma unroll 1
    for (int s = threadIdx.x; s < n0; s += tm.nt) b.X[at(s)] = (T)r[s];
    tm.sync();
}

// 8-byte words of a trivially copyable descriptor, all threads of the CTA
template <typename D>
__device__ __forceinline__ void copy_words(D* dst, const D* src)
{
    static_assert(sizeof(D) % 8 == 0, "descriptors are copied as 8-byte words");
    const unsigned long long* s = reinterpret_cast<const unsigned long long*>(src);
    unsigned long long* d = reinterpret_cast<unsigned long long*>(dst);
#pragma unroll 1
    for (int w = threadIdx.x; w < (int)(sizeof(D) / 8); w += blockDim.x) d[w] = s[w];
}

// one element of a global field into shared memory, asynchronously
template <typename T>
__device__ __forceinline__ void cp_elem(T* dst, const T* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(smem_addr(dst)), "l"(src), "n"((int)sizeof(T))
                 : "memory");
}

__host__ __device__ inline int coarse_slots(int dim, bool fine) { return fine ? 1 : (dim == 2 ? 5 : 14); }

template <typename T, int DIM>
__device__ __forceinline__ Blk<T> coarse_blk(const DevLevel<T>& L, const CoarsePlan& p, int l, T* base)
{
    Blk<T> b;
    b.n = L.n;
    b.lg = 31 - __clz(b.n + 1);
    b.S = b.n + 2;
    b.SZ = DIM == 3 ? b.S * b.S * b.S : b.S * b.S;
    b.X = base + p.x_off[l];
    b.F = b.X + b.SZ;
    b.IV = b.F + b.SZ;
    b.CS = b.IV + b.SZ;
    b.SA = p.sa_off[l] >= 0 ? base + p.sa_off[l] : nullptr;   // shared top grid: its right-hand sides are formed
    b.fine = L.fine != 0;
    b.w = L.woff;
    return b;
}

}  // namespace

// The static image of one chain: the first plan.img_bytes of the kernel's dynamic shared
// memory -- zero state and right-hand side, sqrt(a_ii), 1/a_ii, coefficients, the staged rows
// of G and observation entries.  FP32: 1/a_ii and sqrt(a_ii) from one reciprocal square
// root of the FP32 diagonal, as in the other FP32 kernels; FP64: from the host.
template <typename T, int DIM>
__global__ void k_coarse_image(const CoarseJob<T>* __restrict__ job, unsigned char* __restrict__ img)
{
    const CoarseJob<T> J = *job;
    const DevLevel<T>* levels = J.levels;
    const int m = J.P->m;
    T* base = reinterpret_cast<T*>(img);
    const int t0 = blockIdx.x * blockDim.x + threadIdx.x, st = gridDim.x * blockDim.x;
    for (int l = 0; l <= J.top; ++l) {
        const DevLevel<T>& L = levels[l];
        const Blk<T> b = coarse_blk<T, DIM>(L, J.plan, l, base);
        const int nco = coarse_slots(DIM, b.fine);
        for (int s = t0; s < b.SZ; s += st) {
            const int i = s % b.S - 1, j = (s / b.S) % b.S - 1, k = DIM == 3 ? s / (b.S * b.S) - 1 : 0;
            const bool in = i >= 0 && i < b.n && j >= 0 && j < b.n && (DIM == 2 || (k >= 0 && k < b.n));
            const long long e = site_offset(DIM, L.pitch, L.plane, L.base, i, j, k);
            T inv = T(0), sq = T(0);
            if (in) {
                if constexpr (sizeof(T) == 8) {
                    inv = L.isq[e];
                    sq = L.isq[L.alloc + e];
                } else {
                    float a;
                    if (b.fine) {
                        a = fmaf(2.0f * DIM, L.woff, L.diag[e]);
                    } else {
                        float offsum = 0.0f;
#pragma unroll
                        for (int o = 0; o < Offsets<DIM>::NS; ++o)
                            if (o != Offsets<DIM>::C) offsum += coef_at<DIM>(L, e, o);
                        a = L.coef[e] - offsum;
                    }
                    inv_and_sqrt(a, inv, sq);
                }
            }
            b.X[s] = T(0);
            b.F[s] = T(0);
            if (b.SA) b.SA[s] = sq;
            b.IV[s] = inv;
            for (int t = 0; t < nco; ++t) b.CS[t * b.SZ + s] = b.fine ? L.diag[e] : L.coef[(long long)t * L.alloc + e];
        }
        if (m > 0 && J.plan.g_off[l] >= 0) {
            const int r0 = L.g_rows[0], r1 = L.g_rows[1];
            T* G = reinterpret_cast<T*>(img + J.plan.g_off[l]);
            int* gs = reinterpret_cast<int*>(img + J.plan.gs_off[l]);
            for (int q = t0; q < (r0 + r1) * m; q += st) G[q] = q < r0 * m ? L.gT[0][q] : L.gT[1][q - r0 * m];
            for (int q = t0; q < r0 + r1; q += st) gs[q] = q < r0 ? L.g_ss[0][q] : L.g_ss[1][q - r0];
        }
        if (m > 0 && J.plan.stage_ent) {
            double* w = reinterpret_cast<double*>(img + J.plan.ent_off);
            int* ss = reinterpret_cast<int*>(w + J.plan.nent);
            int* ptr = ss + J.plan.nent;
            const int e0 = J.plan.ent0[l], cnt = L.bcol_ptr[m];
            for (int q = t0; q < cnt; q += st) {
                w[e0 + q] = L.bcol_w[q];
                ss[e0 + q] = L.bcol_ss[q];
            }
            for (int k = t0; k <= m; k += st) ptr[l * (m + 1) + k] = e0 + L.bcol_ptr[k];
        }
    }
}

// One CTA per chain (2D batches) or the one chain of a handle; blockDim.x - kHelp compute
// threads.  Their number never changes the arithmetic.  At 80 registers two CTAs of 256 + 128 threads
// share an SM (at 88 one does: 2000 chains of 7^2 in FP32 245 -> 313 us a cycle).
template <typename T, int DIM>
__global__ void __launch_bounds__(coarse_max_threads<T, DIM>() + kHelp) k_coarse_cycle(const CoarseJob<T>* __restrict__ jobs)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(16) CoarseJob<T> J;
    __shared__ __align__(16) DevLevel<T> lv[kCoarseMaxLevels];
    __shared__ __align__(16) DevProblem P;
    __shared__ unsigned long long bar;
    __shared__ CycleState cs_s;
    pdl_launch_dependents();
    copy_words(&J, jobs + blockIdx.x);   // static table
    if (threadIdx.x == 0) {
        mbar_init(&bar);
        fence_mbar_init();
    }
    __syncthreads();
    {
        // the layout the host planned must fit this launch: a mismatch is reported, never run
        unsigned dsz;
        asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dsz));
        if ((unsigned)J.plan.smem_bytes > dsz) {
            pdl_wait();
            if (threadIdx.x == 0) atomicOr(&J.P->cs->status, kStatusLayout);
            return;
        }
    }
    // --- before the wait on the preceding launch: everything that set-up fixed, and noise
    if (threadIdx.x == 0) {
        mbar_expect_tx(&bar, (unsigned)J.plan.img_bytes);
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                smem_addr(smem_raw)),
            "l"(J.image), "r"(J.plan.img_bytes), "r"(smem_addr(&bar))
            : "memory");
    }
    const int top = J.top;
#pragma unroll 1
    for (int l = 0; l <= top; ++l) copy_words(&lv[l], &J.levels[l]);
    copy_words(&P, J.P);
    __syncthreads();
    // the cycle state changes only in the last launch of a cycle, and a cycle is one graph
    // launch, so it is that of the running cycle already
    const CycleState* const csg = P.cs;
    if (threadIdx.x == 0) cs_s = *csg;
    __syncthreads();
    T* const base = reinterpret_cast<T*>(smem_raw);
    const int m = P.m;
    const int NT = (int)blockDim.x - kHelp, NA = (int)blockDim.x;
    LrArea<T> A;
    {
        A.d = reinterpret_cast<double*>(smem_raw + J.plan.lr_off);
        A.zlr = A.d + (top + 1) * m;
        A.zp = A.zlr + (top + 1) * 2 * m;
        A.v = A.zp + (top + 1) * 2 * m;
        A.z = A.v + m;
        A.zc = A.z + m;
        A.vec = A.zc + J.n0;
        A.vt = reinterpret_cast<T*>(A.vec + (J.gain ? 2 * J.n0 + m : J.n0));
        A.w = reinterpret_cast<const double*>(smem_raw + J.plan.ent_off);
        A.ss = reinterpret_cast<const int*>(A.w + J.plan.nent);
        A.ptr = A.ss + J.plan.nent;
    }
    auto blk = [&](int l) { return coarse_blk<T, DIM>(lv[l], J.plan, l, base); };
    // the first sweep's normals, all warps
    if (top > 0) {
        const int ng = sweep_groups<DIM>(lv[top].n);
#pragma unroll 1
        for (int g = threadIdx.x; g < ng; g += NA) draw_group<T>(&cs_s, top, 0u, base + J.plan.zf[top], g);
    }
    const bool ok = mbar_wait(&bar, 0u, cs_s.wait_ns);
    if (__syncthreads_or(!ok)) {
        pdl_wait();
        if (threadIdx.x == 0) {
            atomicOr(&P.cs->status, kStatusTimeout);
            mbar_wait(&bar, 0u);
        }
        __syncthreads();
        return;
    }
    if ((int)threadIdx.x >= NT) {
        // helper warps.  First the low-rank normals L_Gamma z' and the forward normals of the
        // grids below the top (barrier 2: read from the top grid's low-rank step on), then
        // the coarsest and the backward normals (barrier 3: read from the coarsest sample on)
        const int h = (int)threadIdx.x - NT;
        const int pairs = (m + 1) >> 1;
#pragma unroll 1
        for (int q = h; q < 2 * top * pairs; q += kHelp) {
            const int k = 2 * (q % pairs), l = top - (q / pairs) / 2, dir = (q / pairs) & 1;
            double z[2];
            draw_pair_at<T>(&cs_s, (unsigned)(k >> 1), 1u, l, (unsigned)dir, z);
            double* zp = (P.gamma_diag ? A.zlr : A.zp) + (2 * l + dir) * m;
            zp[k] = P.gamma_diag ? P.LG[k * m + k] * z[0] : z[0];
            if (k + 1 < m) zp[k + 1] = P.gamma_diag ? P.LG[(k + 1) * m + k + 1] * z[1] : z[1];
        }
        if (!P.gamma_diag) {
            bar_n<4>(kHelp);
#pragma unroll 1
            for (int q = h; q < 2 * top * m; q += kHelp) {
                const int k = q % m;
                const double* zp = A.zp + 2 * m + (q - k);
                double lz = 0.0;
#pragma unroll 1
                for (int t = 0; t <= k; ++t) lz = mad(P.LG[k * m + t], zp[t], lz);
                A.zlr[2 * m + q] = lz;
            }
        }
        // pass 0: forward normals of the grids below the top; pass 1: the backward ones, coarsest grid first
#pragma unroll 1
        for (int dir = 0; dir < 2; ++dir) {
            if (dir == 1) {
                bar_arrive<2>(NA);
#pragma unroll 1
                for (int q = h; q < (J.n0 + 1) / 2; q += kHelp) {
                    double z[2];
                    draw_pair_at<double>(&cs_s, (unsigned)q, 2u, 0, 0u, z);
                    A.zc[2 * q] = z[0];
                    if (2 * q + 1 < J.n0) A.zc[2 * q + 1] = z[1];
                }
            }
            const int last = (dir == 0 || J.plan.shared_z) ? top - 1 : top;
#pragma unroll 1
            for (int t = 1; t <= last; ++t) {
                const int l = dir == 0 ? last + 1 - t : t;
                const int ng = sweep_groups<DIM>(lv[l].n);
#pragma unroll 1
                for (int g = h; g < ng; g += kHelp)
                    draw_group<T>(&cs_s, l, (unsigned)dir, base + (dir ? J.plan.zb[l] : J.plan.zf[l]), g);
            }
        }
        bar_arrive<3>(NA);
        return;
    }
    pdl_wait();
    {
        // the top grid's right-hand side, d and (finest grid) state come from earlier launches
        const DevLevel<T>& L = lv[top];
        const Blk<T> b = blk(top);
#pragma unroll 1
        for (int it = threadIdx.x; it < (1 << (DIM * b.lg)); it += NT) {
            int i, j, k;
            cube<DIM>(it, b.lg, i, j, k);
            if (i >= b.n || j >= b.n || (DIM == 3 && k >= b.n)) continue;
            const long long e = site_offset(DIM, L.pitch, L.plane, L.base, i, j, k);
            const int ls = sidx<DIM>(b.S, i, j, k);
            if (L.f) cp_elem(b.F + ls, L.f + e);
            if (J.is_finest) cp_elem(b.X + ls, L.x + e);
        }
        for (int k = threadIdx.x; k < m; k += NT) A.d[top * m + k] = L.d[k];
        asm volatile("cp.async.wait_all;\n" ::: "memory");
    }
    bar_n<1>(NT);
    const Team tm{NT};
    bool fwd_ready = false, bwd_ready = false;   // barriers 2 and 3 passed
    int4 nxt = J.ops[0];
#pragma unroll 1
    for (int q = 0; q < J.n_ops; ++q) {
        const int4 op = nxt;
        if (q + 1 < J.n_ops) nxt = J.ops[q + 1];   // its latency passes during this phase
        const int l = op.y;
        const int dir = op.w & 1;
        if (!fwd_ready && op.x != kOpSweep) {
            bar_n<2>(NA);
            fwd_ready = true;
        }
        if (!bwd_ready && op.x == kOpCoarsest) {
            bar_n<3>(NA);
            bwd_ready = true;
        }
        const Blk<T> b = blk(l);
        switch (op.x) {
        case kOpSweep: {
            T* Z = base + (dir ? J.plan.zb[l] : J.plan.zf[l]);
            const bool formed = l == top && J.plan.shared_z;
            if (op.w & 2) {   // not one of the sweeps drawn above
                const int ng = sweep_groups<DIM>(b.n);
#pragma unroll 1
                for (int g = threadIdx.x; g < ng; g += tm.nt) draw_group<T>(&cs_s, l, (unsigned)op.z, Z, g);
#pragma unroll 1
                for (int k = threadIdx.x; k < m; k += tm.nt) {
                    double z[2];
                    draw_pair_at<T>(&cs_s, (unsigned)(k >> 1), 1u, l, (unsigned)op.z, z);
                    A.zp[(2 * l + dir) * m + k] = z[k & 1];
                }
                tm.sync();
#pragma unroll 1
                for (int k = threadIdx.x; k < m; k += tm.nt) {
                    const double* zp = A.zp + (2 * l + dir) * m;
                    double lz = 0.0;
#pragma unroll 1
                    for (int t = 0; t <= k; ++t) lz = mad(P.LG[k * m + t], zp[t], lz);
                    A.zlr[(2 * l + dir) * m + k] = lz;
                }
            }
            if (formed) {
                // the top grid's sweeps share one place for the normals and have no sqrt(a_ii)
                // block: the right-hand sides fdense + sqrt(a_ii) z in one pass
                const int n = b.n, ld = ((n + 3) >> 2) << 2;
#pragma unroll 1
                for (int it = threadIdx.x; it < (1 << (DIM * b.lg)); it += tm.nt) {
                    int i, j, k;
                    cube<DIM>(it, b.lg, i, j, k);
                    if (i >= n || j >= n || (DIM == 3 && k >= n)) continue;
                    const int ls = sidx<DIM>(b.S, i, j, k), zi = ((DIM == 3 ? k * n : 0) + j) * ld + i;
                    T sq;
                    if constexpr (sizeof(T) == 8) {
                        sq = lv[l].isq[lv[l].alloc + site_offset(DIM, lv[l].pitch, lv[l].plane, lv[l].base, i, j, k)];
                    } else {
                        float a, inv;
                        if (b.fine) {
                            a = fmaf(2.0f * DIM, b.w, b.CS[ls]);
                        } else {
                            float offsum = 0.0f;
#pragma unroll
                            for (int o = 0; o < Offsets<DIM>::NS; ++o)
                                if (o != Offsets<DIM>::C) offsum += coef_s<DIM>(b, ls, o);
                            a = b.CS[ls] - offsum;
                        }
                        inv_and_sqrt(a, inv, sq);
                    }
                    Z[zi] = mad(sq, Z[zi], b.F[ls]);
                }
            }
            if (formed || (op.w & 2)) tm.sync();
            s_sweep<DIM>(b, Z, formed, dir, tm);
            break;
        }
        case kOpLowrank:
            if (m > 0)
                s_lowrank(lv[l], J, A, smem_raw, m, l, b.X, (op.w & 2) ? -1 : dir, (op.w & 4) != 0,
                          A.zlr + (2 * l + dir) * m, tm);
            break;
        case kOpRestrict:
            s_restrict<DIM>(b, base + J.plan.zf[l], blk(l - 1), tm);
            break;
        case kOpCoarsest:
            s_coarsest<DIM>(J, m, b, A.d, A.vec, A.zc, tm);
            break;
        case kOpProlong:
            if (op.w & 2) {   // the backward normals share the forward ones' place: drawn beside the prolongation
                const int ng = sweep_groups<DIM>(b.n);
#pragma unroll 1
                for (int g = threadIdx.x; g < ng; g += tm.nt)
                    draw_group<T>(&cs_s, l, 1u, base + J.plan.zb[l], g);
            }
            s_prolong<DIM>(blk(l - 1), b, tm);
            tm.sync();
            break;
        default:
            break;
        }
    }
    // the top grid's final state goes back to global memory
    {
        const DevLevel<T>& L = lv[top];
        const Blk<T> b = blk(top);
#pragma unroll 1
        for (int it = threadIdx.x; it < (1 << (DIM * b.lg)); it += NT) {
            int i, j, k;
            cube<DIM>(it, b.lg, i, j, k);
            if (i >= b.n || j >= b.n || (DIM == 3 && k >= b.n)) continue;
            L.x[site_offset(DIM, L.pitch, L.plane, L.base, i, j, k)] = b.X[sidx<DIM>(b.S, i, j, k)];
        }
    }
}

// Shared-memory plan of grids 0..top (see k_coarse_cycle).  Static image: per grid the state,
// the dense right-hand side, 1/a_ii, the coefficient blocks (1 for the 5/7-point finest grid,
// (3^d + 1)/2 for a Galerkin grid) and sqrt(a_ii); the staged rows of G of as many grids as
// fit, coarsest first; the observation entries.  Then the normals of both sweeps of every
// smoothed grid (its forward part also takes the grid's residual) and the low-rank area.
// When that exceeds `limit` the two sweeps of the top grid share one place for their
// normals and it has no sqrt(a_ii) block, then the observation entries stay in global memory.
bool coarse_plan(int dim, const int* n_of_level, int top, bool top_is_fd_finest, int m, const int* nnz_of_level,
                 const int* g_rows_of_level, size_t elem, size_t limit, CoarsePlan* out)
{
    auto vol = [dim](long long s) { return dim == 3 ? s * s * s : s * s; };
    auto up = [](long long b, long long a) { return (b + a - 1) / a * a; };
    const long long n0 = vol(n_of_level[0]);
    for (int tight = 0; tight < 3; ++tight) {
        CoarsePlan p{};
        p.shared_z = (tight >= 1 && top > 0) ? 1 : 0;
        p.stage_ent = tight < 2 ? 1 : 0;
        long long o = 0;
        for (int l = 0; l < kCoarseMaxLevels; ++l) p.sa_off[l] = p.g_off[l] = p.gs_off[l] = -1;
        for (int l = 0; l <= top; ++l) {
            const long long sz = vol(n_of_level[l] + 2);
            p.x_off[l] = (int)o;
            o += (3 + coarse_slots(dim, l == top && top_is_fd_finest)) * sz;
            if (l == top && p.shared_z) continue;
            p.sa_off[l] = (int)o;
            o += sz;
        }
        long long bytes = up(o * (long long)elem, 16);
        p.ent_off = (int)bytes;
        if (p.stage_ent && m > 0) {
            for (int l = 0; l <= top; ++l) {
                p.ent0[l] = p.nent;
                p.nent += nnz_of_level[l];
            }
            bytes = up(bytes + 12LL * p.nent + 4LL * (top + 1) * (m + 1), 16);
        }
        // what follows the image
        long long z = 0;
        for (int l = 1; l <= top; ++l) {
            const long long n = n_of_level[l];
            z += (l == top && p.shared_z ? 1 : 2) * 4 * ((n + 3) / 4) * n * (dim == 3 ? n : 1);
        }
        const bool gain = n0 <= kCoarseGainMax;
        const long long lr = 8 * (5LL * (top + 1) * m + 2 * m + n0 + (gain ? 2 * n0 + m : n0)) + (long long)elem * m + 16;
        const long long tail = up(z * (long long)elem, 16) + lr;
        for (int l = 1; l <= top && m > 0; ++l) {
            const long long r = g_rows_of_level[l];
            const long long g = up(r * m * (long long)elem, 16) + up(4 * r, 16);
            if (bytes + g + tail > (long long)limit) break;
            p.g_off[l] = (int)bytes;
            p.gs_off[l] = (int)(bytes + up(r * m * (long long)elem, 16));
            bytes += g;
        }
        p.img_bytes = (int)bytes;
        long long zo = bytes / (long long)elem;
        for (int l = 1; l <= top; ++l) {
            const long long n = n_of_level[l], c = 4 * ((n + 3) / 4) * n * (dim == 3 ? n : 1);
            p.zf[l] = p.zb[l] = (int)zo;
            zo += c;
            if (l == top && p.shared_z) continue;
            p.zb[l] = (int)zo;
            zo += c;
        }
        p.lr_off = (int)up(zo * (long long)elem, 16);
        p.smem_bytes = (int)(p.lr_off + lr);
        if (p.smem_bytes <= (long long)limit) {
            *out = p;
            return true;
        }
    }
    return false;
}

__host__ __device__ inline int qoi_ctas(int n_qoi)
{
    const int c = (n_qoi + 1023) / 1024;
    return c < 1 ? 1 : (c > kQoiMaxCtas ? kQoiMaxCtas : c);
}

// F^T theta of every chain's finest grid, then step += 1, cycle += 1.  Up to 16 CTAs per
// chain: products and conversions are FP64, a few hundred cycles per warp and site each, so a
// QoI of thousands of sites takes several SMs (one CTA: 60 us for 16 641 sites, 16 CTAs:
// about 6 us).  The partial sums are added by the chain's last CTA in CTA order.
template <typename T>
__global__ void k_qoi_batch(const QoiJob<T>* __restrict__ jobs)
{
    __shared__ double part[256];
    pdl_launch_dependents();
    // the QoI sites and weights never change: the first kQoiPre of each thread are loaded
    // before the wait on the preceding launch, the state after it (same summation order)
    constexpr int kQoiPre = 4;
    const QoiJob<T> J = jobs[blockIdx.x];
    // the chain's own number of CTAs: its sum does not depend on the other chains of a launch
    const int nb = qoi_ctas(J.n_qoi);
    if ((int)blockIdx.y >= nb) return;
    const int t0 = blockIdx.y * blockDim.x + threadIdx.x, st = nb * blockDim.x;
    long long site[kQoiPre];
    double w[kQoiPre];
#pragma unroll
    for (int r = 0; r < kQoiPre; ++r) {
        const int t = t0 + r * st;
        site[r] = t < J.n_qoi ? J.q_site[t] : 0;
        w[r] = t < J.n_qoi ? J.q_w[t] : 0.0;
    }
    pdl_wait();
    double acc = 0.0;
#pragma unroll
    for (int r = 0; r < kQoiPre; ++r)
        if (t0 + r * st < J.n_qoi) acc += w[r] * (double)J.x[site[r]];
    for (int t = t0 + kQoiPre * st; t < J.n_qoi; t += st) acc += J.q_w[t] * (double)J.x[J.q_site[t]];
    part[threadIdx.x] = acc;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) part[threadIdx.x] += part[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x != 0) return;
    double q = part[0];
    if (nb > 1) {
        J.part[blockIdx.y] = q;
        __threadfence();
        if (atomicAdd(J.ticket, 1) != nb - 1) return;
        __threadfence();
        q = 0.0;
        for (int b = 0; b < nb; ++b) q += __ldcg(J.part + b);
        *J.ticket = 0;
    }
    CycleState* cs = J.cs;
    if (cs->qoi) cs->qoi[cs->step] = q;
    if (!isfinite(q)) atomicOr(&cs->status, kStatusNumeric);
    cs->step += 1;
    cs->cycle += 1;
}

__global__ void k_set_cycle_batch(CycleState* const* cs, int n, unsigned long long seed, unsigned long long cycle,
                                  int noise, double* qoi, long long n_steps)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    CycleState* s = cs[c];
    s->seed = seed;
    s->cycle = cycle;
    s->chain = (unsigned)c;
    s->noise = noise;
    s->qoi = qoi ? qoi + (long long)c * n_steps : nullptr;
    s->step = 0;
}

template <typename T>
cudaError_t coarse_prepare(int dim, size_t smem_bytes)
{
    if (dim == 2)
        return cudaFuncSetAttribute(k_coarse_cycle<T, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
    return cudaFuncSetAttribute(k_coarse_cycle<T, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
}

// writes the static image of one chain (set-up, on the stream given)
template <typename T>
cudaError_t coarse_image(const CoarseJob<T>* job, unsigned char* image, int dim, cudaStream_t st)
{
    if (dim == 2)
        k_coarse_image<T, 2><<<32, 256, 0, st>>>(job, image);
    else
        k_coarse_image<T, 3><<<32, 256, 0, st>>>(job, image);
    return cudaGetLastError();
}

template <typename T>
void launch_coarse(const CoarseJob<T>* jobs, int n, int dim, int threads, size_t smem_bytes, cudaStream_t st,
                   int& launches)
{
    const dim3 grid((unsigned)n), block((unsigned)(std::min(threads, dim == 2 ? coarse_max_threads<T, 2>() : coarse_max_threads<T, 3>()) + kHelp));
    if (dim == 2)
        launch_pdl(k_coarse_cycle<T, 2>, grid, block, smem_bytes, st, jobs);
    else
        launch_pdl(k_coarse_cycle<T, 3>, grid, block, smem_bytes, st, jobs);
    ++launches;
}

template <typename T>
void launch_qoi_batch(const QoiJob<T>* jobs, int n, int max_qoi, cudaStream_t st, int& launches)
{
    // chains along x: a batch may hold 65 536, one more than gridDim.y takes
    launch_pdl(k_qoi_batch<T>, dim3((unsigned)n, (unsigned)qoi_ctas(max_qoi)), dim3(256), 0, st, jobs);
    ++launches;
}

void launch_set_cycle_batch(CycleState* const* cs, int n, unsigned long long seed, unsigned long long cycle, int noise,
                            double* qoi, long long n_steps, cudaStream_t st)
{
    k_set_cycle_batch<<<(n + 127) / 128, 128, 0, st>>>(cs, n, seed, cycle, noise, qoi, n_steps);
}

template cudaError_t coarse_prepare<float>(int, size_t);
template cudaError_t coarse_prepare<double>(int, size_t);
template cudaError_t coarse_image<float>(const CoarseJob<float>*, unsigned char*, int, cudaStream_t);
template cudaError_t coarse_image<double>(const CoarseJob<double>*, unsigned char*, int, cudaStream_t);
template void launch_coarse<float>(const CoarseJob<float>*, int, int, int, size_t, cudaStream_t, int&);
template void launch_coarse<double>(const CoarseJob<double>*, int, int, int, size_t, cudaStream_t, int&);
template void launch_qoi_batch<float>(const QoiJob<float>*, int, int, cudaStream_t, int&);
template void launch_qoi_batch<double>(const QoiJob<double>*, int, int, cudaStream_t, int&);

}  // namespace mgmc
