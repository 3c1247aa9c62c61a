// tc_conv.cuh -- 3x3 convolutions of channels-last BF16 images on the tcgen05 tensor
// cores without an im2col matrix (tc_conv.cu): the shifted pixels of a tap are a TMA box
// of the image itself, its out-of-range rows and columns the box's zero fill.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace mgmc {

// whether a layer can run here: whole 16-channel chunks on both sides (tcgen05's K = 16 stays
// inside a tap); the others take the im2col path
inline bool tc_conv_ok(int cin, int cout) { return cin % 16 == 0 && cout % 16 == 0; }

// status, wait_ns: as in tc_gemm_run (status not NULL)
// Y [P][cout] (BF16) = relu(conv(X [B][H][H][cin], W [cout][9 cin]) + bias), P = B H H, H a power of two >= 4
cudaError_t tc_conv_fwd(const __nv_bfloat16* X, int B, int H, int cin, const __nv_bfloat16* W, int cout,
                        const float* bias, __nv_bfloat16* Y, int* status, long long wait_ns, cudaStream_t st);
// dX [P][cin] (FP32) = sum over taps, in tap order, of the FP32 products dZ(shifted) [P][cout] Wt[tap cin ..][cout]^T
cudaError_t tc_conv_dgrad(const __nv_bfloat16* dZ, int B, int H, int cin, const __nv_bfloat16* Wt, int cout, float* dX,
                          int* status, long long wait_ns, cudaStream_t st);
// part [splits][9 cin][cout] (FP32) = X(shifted)^T dZ over `splits` ranges of k_per_split pixels (a multiple of 64)
cudaError_t tc_conv_wgrad(const __nv_bfloat16* X, const __nv_bfloat16* dZ, int B, int H, int cin, int cout, int splits,
                          long long k_per_split, float* part, int* status, long long wait_ns, cudaStream_t st);

}  // namespace mgmc
