// Launchers of the tensor-core (tcgen05) inference of the learned estimator.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <string>

#include "../../include/asse_learn.h"

namespace asse {

// fp32 parameters (asse_learn.h order) -> the packed BF16 operand images of
// W1 (HID x FEAT) and W2 (HID x HID) that the tensor-core kernel copies into
// shared memory.
cudaError_t launch_mlp_pack(const float *params, __nv_bfloat16 *w1p, __nv_bfloat16 *w2p, cudaStream_t s,
                            uint64_t *launches);

// y[i] = model(x[i]) for n row-major BF16 feature rows (16-byte aligned).
// Returns 0 when launched, else nonzero with the reason in *why.  A wait in
// the kernel that gives up sets *error to 1.
int launch_mlp_forward_tc(const __nv_bfloat16 *x, uint64_t n, const __nv_bfloat16 *w1p, const __nv_bfloat16 *w2p,
                          const float *params, float *y, int *error, cudaStream_t s, uint64_t *launches,
                          std::string *why);

// Where element (n, k) of W1 [ASSE_HID][ASSE_FEAT] and of W2 [ASSE_HID][ASSE_HID]
// lies in those images.
__host__ __device__ inline uint32_t mlp_w1p_at(uint32_t n, uint32_t k)
{
    return k / 16 * (ASSE_HID * 16) + n / 8 * 128 + k % 16 / 8 * 64 + n % 8 * 8 + k % 8;
}
__host__ __device__ inline uint32_t mlp_w2p_at(uint32_t n, uint32_t k)
{
    return n / 8 * (ASSE_HID * 8) + k / 8 * 64 + n % 8 * 8 + k % 8;
}

// Products of the training pass on the tensor cores (tcgen05):
// C[M][N] = sum_k A(m, k) B(n, k), operands addressed by strides (element
// (i, k) at p[i * si + k * sk]), N a multiple of 16 up to 256, the k range
// split over `splits` CTAs (more than one only with TE_ATOMIC), and a fused
// epilogue:
//   TE_BIAS_RELU      out = bf16(relu(C + bias[n]))
//   TE_BIAS_RELU_DOT  the same, and y[t][m] = the sum of out * w3[n] over column tile t (64 columns
//                     where N is a multiple of 64)
//   TE_RELU_GRAD      out = bf16(C) where act > 0, else 0, and outf[n] += its column sums
//   TE_ATOMIC         outf[m][n] += C (FP32 atomics)
// with row stride ld (a multiple of 8; out, act and outf 16-byte aligned).  A
// CTA whose bounded wait gave up sets *error to 1.
struct TcOperand {
    const __nv_bfloat16 *p;
    long si, sk;
};
enum { TE_BIAS_RELU = 0, TE_BIAS_RELU_DOT = 1, TE_RELU_GRAD = 2, TE_ATOMIC = 3 };
struct TcEpi {
    int kind;
    const float *bias;
    const float *w3;
    const __nv_bfloat16 *act;
    __nv_bfloat16 *out;
    float *outf;
    float *y;
    int ld;
};
struct TcProduct {
    TcOperand A, B;
    int M, N, K, splits;
    TcEpi epi;
};
// What a launch does besides (any of it null): n_zero floats at zero set to 0,
// *to = *from.
struct TcExtra {
    float *zero;
    uint32_t n_zero;
    float *to;
    const float *from;
};
// One launch of one product, or of two that do not depend on one another.
cudaError_t launch_tc_gemm(const TcProduct *products, int count, const TcExtra &extra, int *error, cudaStream_t s,
                           uint64_t *launches);

}  // namespace asse
