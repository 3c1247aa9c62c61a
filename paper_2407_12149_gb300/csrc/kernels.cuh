// kernels.cuh -- launch wrappers of the V-cycle kernels (see kernels.cu).
#pragma once
#include "common.cuh"
#include "stencil.cuh"

namespace mgmc {

template <typename T>
void launch_sweep(const DevLevel<T>& L, const DevProblem& P, int dir, unsigned slot, cudaStream_t st, int& launches);
// dir < 0: only d_{l-1} = d_l - B^T theta (no correction)
template <typename T>
void launch_lowrank(const DevLevel<T>& L, const DevProblem& P, int dir, unsigned slot, bool dnext, cudaStream_t st,
                    int& launches);
template <typename T>
void launch_restrict(const DevLevel<T>& F, const DevLevel<T>& C, cudaStream_t st, int& launches);
// exact coarsest sample of the general path with the noise slot of the grid's visit
template <typename T>
void launch_coarsest_slot(const DevLevel<T>& L, const DevProblem& P, const double* chol, int n0, unsigned slot,
                          cudaStream_t st, int& launches);
// phases {code, grid, slot, flags} of the kernels that run several grids in one CTA, listed by
// the host from the cycle's recursion (coarse.cu; kernels.cu: k_cycle_small)
enum { kOpSweep = 0, kOpLowrank = 1, kOpRestrict = 2, kOpZero = 3, kOpCoarsest = 4, kOpProlong = 5 };
constexpr int kSmallCycleThreads = 512;
constexpr int kSmallMaxLevels = 16;   // grids 0..top held by the kernel (top < 16)
constexpr int kSmallMaxOps = 1024;    // phases staged in shared memory (later ones read from global)
constexpr int kSmallSharedN = 15;     // grids up to this size live in shared memory
constexpr int kSmallStageOps = 24;    // .. if the visit has at least as many phases
constexpr int kSmallPreN = 7;         // grids up to this size have their site normals drawn at the start
constexpr int kSmallMaxPre = 4096;    // normals drawn at the start, at most
// dynamic shared memory of the kernel: 227 KB less its static part
constexpr size_t kSmallArena = 232448 - 36 * 1024;
template <typename T>
cudaError_t cycle_small_prepare();
// gain: see setup.hpp (NULL: the coarsest grid is solved with the factor); ops' flags >> 8: 1 + the
// place of the phase's pre-drawn normals among the n_pre, 0 none.  zb: scratch of n^2 doubles for
// the largest 25-point grid held (the normals of a sweep)
template <typename T>
void launch_cycle_small(const DevLevel<T>* levels_dev, int top, const DevProblem& P, const double* chol,
                        const double* gain, int n0, const int4* ops, int n_ops, int n_pre, double* zb, cudaStream_t st,
                        int& launches);
template <typename T>
void launch_prolong(const DevLevel<T>& C, const DevLevel<T>& F, cudaStream_t st, int& launches);
// shared-memory plan of the coarse kernel (coarse.cu), offsets in elements of the path precision
constexpr int kCoarseMaxLevels = 8;   // grids it holds at most (their descriptors are staged)
constexpr int kCoarseGainMax = 64;    // coarsest unknowns up to which the gain matrix is used
struct CoarsePlan {
    int x_off[kCoarseMaxLevels];   // grid l's blocks: state, right-hand side, 1/a_ii, coefficients
    int sa_off[kCoarseMaxLevels];  // its sqrt(a_ii) block (-1: none)
    int zf[kCoarseMaxLevels];      // normals of the forward / backward sweep
    int zb[kCoarseMaxLevels];
    int g_off[kCoarseMaxLevels];   // byte offsets of the staged rows of G and their sites (-1: in global memory)
    int gs_off[kCoarseMaxLevels];
    int ent0[kCoarseMaxLevels];    // first staged observation entry
    int nent;                      // staged observation entries
    int stage_ent;                 // 0: the entries are read from global memory
    int ent_off;                   // byte offset of the entries
    int shared_z;                  // 1: the top grid's two sweeps share zf[top] = zb[top], no sqrt(a_ii) block
    int img_bytes;                 // the static image is the first img_bytes
    int lr_off;                    // byte offset of the low-rank area
    int smem_bytes;
    int pad;
};
// g_rows_of_level: rows of G of both directions together
bool coarse_plan(int dim, const int* n_of_level, int top, bool top_is_fd_finest, int m, const int* nnz_of_level,
                 const int* g_rows_of_level, size_t elem, size_t limit, CoarsePlan* out);
// dynamic shared memory the coarse kernel may use: 227 KB less its static part
constexpr size_t kCoarseSmemLimit = 232448 - 6144;
// one chain of a coarse-grid launch
template <typename T>
struct CoarseJob {
    const DevLevel<T>* levels;   // device descriptors of grids 0 .. L-1
    const DevProblem* P;
    const double* chol;          // Cholesky factor of the coarsest operator (n0 > kCoarseGainMax)
    const double* gain;          // [n0][2 n0 + m] rows [A~_0^-1 | A~_0^-1 B_0 Gamma^-1 | L_0^-T], or NULL
    const double* e0;            // [m][n0] columns of B_0 Gamma^-1 (n0 > kCoarseGainMax)
    const int4* ops;             // phases {code, grid, slot, flags}
    const unsigned char* image;  // static part of the shared memory (coarse_image)
    CoarsePlan plan;
    int n_ops;
    int top;
    int is_finest;
    int n0;
};
// one chain of a batched QoI launch
template <typename T>
struct QoiJob {
    const T* x;                  // finest-grid state
    int n_qoi;
    const long long* q_site;
    const double* q_w;
    CycleState* cs;
    double* part;                // [kQoiMaxCtas] partial sums
    int* ticket;                 // CTAs of the launch that have finished (0 between launches)
};
constexpr int kQoiMaxCtas = 16;
template <typename T>
void launch_qoi_batch(const QoiJob<T>* jobs, int n, int max_qoi, cudaStream_t st, int& launches);
void launch_set_cycle_batch(CycleState* const* cs, int n, unsigned long long seed, unsigned long long cycle, int noise,
                            double* qoi, long long n_steps, cudaStream_t st);

// the V-cycle of grids 0..top of n chains, one CTA each, with shared-memory state (coarse.cu)
template <typename T>
cudaError_t coarse_prepare(int dim, size_t smem_bytes);
template <typename T>
cudaError_t coarse_image(const CoarseJob<T>* job, unsigned char* image, int dim, cudaStream_t st);
template <typename T>
void launch_coarse(const CoarseJob<T>* jobs, int n, int dim, int threads, size_t smem_bytes, cudaStream_t st,
                   int& launches);
void launch_set_cycle(CycleState* cs, unsigned long long seed, unsigned long long cycle, unsigned chain, int noise,
                      double* qoi, cudaStream_t st);
template <typename T>
void launch_pack(const DevLevel<T>& L, T* dense, bool to_padded, cudaStream_t st);
// 2D dense user fields <-> padded finest-level states of many chains, one launch per
// kPackChunk chains; jobs[c] is the static part, dense[c] the caller's array
template <typename T>
struct PackJob {
    T* x;            // padded finest-level state
    int n;
    int pitch;
    long long base;
};
constexpr int kPackChunk = 256;
template <typename T>
void launch_pack_batch(const PackJob<T>* jobs, void* const* dense, int count, int max_n, bool to_padded,
                       cudaStream_t st);
template <typename T>
void launch_resid(const DevLevel<T>& L, const DevProblem& P, double* u, double* partial, int max_partial,
                  double* out, cudaStream_t st);

}  // namespace mgmc
