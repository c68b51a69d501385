// Interface of the tensor-core GEMMs of the wave-packet transform (tc_gemm.cu).
#pragma once

#include "fga_internal.cuh"

namespace fga {

constexpr int TC_KB = 32;          // complex K per staged block
constexpr int TC_NC = 64;          // largest N tile (complex columns)
constexpr float TC_SB = 16384.0f;  // scale of the kernel matrices

// The kernel matrix of one axis, split to FP16 in the operand layout: ntile N tiles of nc rows, nkb K blocks.
struct KernelMatrix {
    int ny = 0, ntile = 0, nc = 0, nkb = 0;
    size_t bytes = 0;
    unsigned char *B = nullptr;   // DEVICE, 16-byte aligned
    double q0 = 0, dq = 0, p0 = 0, dp = 0, y0 = 0, dy = 0;
};
struct KernelMatrices {
    KernelMatrix ax[3];
    int nq = 0, np = 0;
    double k = 0;
};
// tile counts and bytes of an N x K kernel matrix
void tc_kernel_shape(int N, int K, KernelMatrix &X);
// evaluates the three axes' matrices
fga_status tc_kernel_matrices(const KernelMatrices &P, cudaStream_t s);
// C[z][m][n] = scale sum_k A[z][m][k] B[n][k] on the tensor cores (FP16 split, FP32 accumulation); row m of A and C at
// (m / rdiv) stride + m % rdiv; |Re|, |Im| of A bounded by (*amax) * amax_factor; *err set if a wait ran out
template <typename TA>
fga_status tc_cgemm(const TA *A, int64_t sAz, int64_t sAm, int64_t sAk, const KernelMatrix &X, float2 *C, int64_t sCz,
                    int64_t sCm, int64_t sCn, int rdiv, int Z, int64_t M, int N, float scale, const float *amax,
                    float amax_factor, int *err, cudaStream_t s);
fga_status tc_absmax(const double2 *x, int64_t n, float *out, cudaStream_t s);

}  // namespace fga
