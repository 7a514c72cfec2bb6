// Forward x transform of real rows on the tensor cores, fed by TMA (see
// bvf_xfwd.cu); shared by the surrogate's FP32 and BF16 paths.
#pragma once

#include <cuda_runtime.h>

namespace bvf {

// D[i][j] = sum_x v[i][x] T[j][x] for every row i < R of v (nx per row)
struct XfwdArgs {
    const float *v;
    long long R;
    int nx, m;
    // TF32-split products (FP32 path): T[2 kx][x], T[2 kx + 1][x] = tx[kx nx + x],
    // out[i m + kx] = (D[i][2 kx], -D[i][2 kx + 1])
    const float2 *tx;
    float2 *out;
    // BF16 products: T[j][x] = F[x 2m + j], row i = (s, y) with ny values of y,
    // outw[s 2m ny + j ny + y] = D[i][j]
    const float *F;
    float *outw;
    int ny;
    int n_sm;
    int *flag;
};

// whether the TMA-fed kernel takes these rows: whole 16-byte pieces, nx >= 32,
// and the resident operand T plus a ring of three slots within shared memory
bool xfwd_fits(bool tf32, const float *v, long long R, int nx, int m);
// cudaErrorNotSupported: no tensor map could be made (the caller takes its
// other path)
cudaError_t launch_xfwd(bool tf32, const XfwdArgs &q, cudaStream_t s);

}  // namespace bvf
