// Internal declarations of the surrogate's BF16 path.
#pragma once

#include <cuda_runtime.h>

#include "../../include/bvf_fno.h"
#include "bvf_internal.cuh"

namespace bvf {

// GELU with CUDA's erff, and its derivative Phi(s) + s phi(s)
__device__ __forceinline__ float gelu_exact(float s)
{
    return 0.5f * s * (1.0f + erff(s * 0.70710678118654752f));
}
__device__ __forceinline__ float gelu_grad(float s)
{
    return 0.5f * (1.0f + erff(s * 0.70710678118654752f)) +
           s * 0.39894228040143268f * expf(-0.5f * s * s);
}

// bvf_gemm with the rows of A and C and the columns of A taken apart, so that
// the axis order of the next product is a matter of addresses:
//   row r of A starts at (r / (ra ra2)) sam2 + (r / ra % ra2) sam1 + (r % ra) sam,
//   row r of C at        (r / rc) scm1 + (r % rc) scm,
//   column k of A lies at (k / ka) sak1 + (k % ka) sak, column n of C likewise
//   with nc, scn1, scn.
// ra = rc = ka = nc = 0: plain strides.
struct GemmX {
    bvf_gemm g;
    int ra = 0, ra2 = 1, rc = 0, ka = 0, nc = 0;
    long long sam1 = 0, sam2 = 0, scm1 = 0, sak1 = 0, scn1 = 0;
    int vec = 0;           // set by the launcher: float4 loads of A along k
};
cudaError_t launch_gemm_bf16(const GemmX &g, int *flag, cudaStream_t s);

// one row pass (see bvf_row_bf16.cu)
struct RowBf16 {
    const float *v;        // [B][cin][N]
    long long vb;          // sample stride of v
    int cin;
    const float *Wm;       // Wm(o, c) at o wso + c wsc
    int wso, wsc;
    const float *bias;     // [W] or NULL
    const float *S;        // [B][W][rows][2m], part-major pairs (NULL: no spectral term)
    const float *G;        // [2m][nx]
    float *pre;            // act 1: receives the pre-activation (or NULL); act 2: holds it
    int act;
    float *out;            // [B][W][N]
    int B, nx, rows, m, N, n_sm;
    int *flag;
};
bool row_bf16_fits(int width, int m, int nx);
cudaError_t launch_row_bf16(const RowBf16 &q, int width, cudaStream_t s);
// weight and bias gradient of a channel mix (see bvf_wgrad_bf16.cu)
struct WgradBf16 {
    const float *d;        // [B][O][N]
    const float *x;        // [B][C][N]
    int O, C;
    float *G;              // [O][C], added to
    float *g;              // [O], added to, or NULL
    int B, N;
    int *flag;
};
bool wgrad_fits(const WgradBf16 &q);      // rows of whole 16-byte pieces
cudaError_t launch_wgrad_bf16(const WgradBf16 &q, int n_sm, cudaStream_t s);
// one channel product (see bvf_row_bf16.cu)
struct ChanBf16 {
    const float *v;        // [B][K][N]
    int K, O;
    const float *Wm;       // Wm(o, c) at o wso + c wsc
    int wso, wsc;
    const float *bias;     // [O] or NULL
    float *pre;            // act 1: receives the pre-activation (or NULL); act 2: holds it
    int act;
    float *out;            // [B][O][N]
    int B, N;
    int *flag;
};
cudaError_t launch_chan_bf16(const ChanBf16 &q, int n_sm, cudaStream_t s);
cudaError_t launch_project_bf16(const float *v, const float *Q1, const float *q1, const float *Q2,
                                const float *q2, int width, int hidden, int c_out, float *out, int N,
                                int B, int n_sm, int *flag, cudaStream_t s);

}  // namespace bvf
