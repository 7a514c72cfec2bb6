// BF16 path of the surrogate: inference and training of the Fourier neural
// operator (Li et al., ICLR 2021, Sec. 4; the network of include/bvf_fno.h)
// with every contraction on tcgen05 (BF16 operands, FP32 accumulation; row
// passes and projection: bvf_row_bf16.cu, forward x transform: bvf_xfwd.cu,
// weight gradients: bvf_wgrad_bf16.cu, y and z transforms and the general case:
// bvf_gemm_bf16.cu) and FP32 master weights.
//
// Layouts (per sample b, channel c, voxel p = (z ny + y) nx + x):
//   volumes  [b][c][p];
//   spectra  [b][c][ky][kx][part][kz] with ky, kz the 2m signed slots, kx in
//            0 .. m-1, part 0 = real, 1 = imaginary (8 m^3 floats per channel).
// Forward transform of a layer (the kept modes of rfftn), three products:
//   x: rows (b, c, z, y) x nx  ->  [part][kx]      (cos, -sin)
//   y: rows (b, c, z, kx) x [part][y]  ->  [part][ky]   (e^{-i theta} as a
//      real 2 x 2 block)
//   z: rows (b, c, ky, kx) x [part][z]  ->  [part][kz]
// each reading and writing its neighbours' axis order; the inverse (irfftn of
// the kept half spectrum) is the same chain backwards with e^{+i theta} and,
// on x, the weights c(kx)/N (c = 1 for kx = 0, 2 otherwise); its x stage runs
// in one pass with the layer's channel mix (bvf_row_bf16.cu).  The mode mix (per mode a
// W x W complex matrix) is a small SIMT kernel.
//
// Backward (gradients of the loss below): the adjoint of the inverse is the
// forward transform with the weights c(kx)/N, the adjoint of the forward
// transform is the inverse without them, the mix's adjoints take conj(R);
// weight and bias gradients are sums over the batch and the voxels (split,
// added atomically).  GELU's derivative is
// applied in the product epilogue from the stored pre-activation.
//
// Loss of a batch: the mean over samples of the relative L2 error
// ||out_0 - target|| / ||target|| of output channel 0, plus, when the net has
// a second output channel, el_weight times the mean squared error of that
// channel's spatial mean against the sample's transmission target.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "bvf_fno_bf16.cuh"
#include "bvf_xfwd.cuh"

using bvf::ChanBf16;
using bvf::GemmX;
using bvf::launch_gemm_bf16;
using bvf::RowBf16;
using bvf::WgradBf16;

namespace {

constexpr double kPi = 3.14159265358979323846;

int b16_fail(int code, const std::string &msg)
{
    bvf::set_context_free_error(msg.c_str());
    return code;
}

int b16_cuda(cudaError_t e, const std::string &where)
{
    // reported here: the next call's launches must not find it pending
    (void)cudaGetLastError();
    return b16_fail(e == cudaErrorMemoryAllocation ? BVF_E_NOMEM : BVF_E_CUDA,
                    where + ": " + cudaGetErrorString(e));
}

#define BCK(call, where)                                   \
    do {                                                   \
        cudaError_t e_ = (call);                           \
        if (e_ != cudaSuccess) return b16_cuda(e_, where); \
    } while (0)

__host__ __device__ __forceinline__ int slot_freq(int j, int m) { return j < m ? j : j - 2 * m; }

// spectrum position of mode (kz, ky, kx), part, in a channel's 8 m^3 floats
__device__ __forceinline__ int spec_pos(int kz, int ky, int kx, int part, int m)
{
    return ((ky * m + kx) * 2 + part) * (2 * m) + kz;
}

// Y[b][o][mode] = sum_c R[mode][c][o] X[b][c][mode]  (R: [kz][ky][kx][c][o][2])
__global__ void k_mix_fwd(const float *__restrict__ X, const float *__restrict__ R, int B, int W,
                          int m, float *__restrict__ Y)
{
    const int modes = 4 * m * m * m, S = 8 * m * m * m;
    const long long n = (long long)B * modes * W;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        const int o = (int)(t % W);
        const int mode = (int)((t / W) % modes);
        const int b = (int)(t / ((long long)W * modes));
        const int kx = mode % m, ky = (mode / m) % (2 * m), kz = mode / (2 * m * m);
        const int pr = spec_pos(kz, ky, kx, 0, m), pi = spec_pos(kz, ky, kx, 1, m);
        const float *Rm = R + (size_t)mode * W * W * 2;
        float yr = 0.0f, yi = 0.0f;
        for (int c = 0; c < W; ++c) {
            const float *xc = X + ((size_t)b * W + c) * S;
            const float xr = xc[pr], xi = xc[pi];
            const float rr = Rm[((size_t)c * W + o) * 2], ri = Rm[((size_t)c * W + o) * 2 + 1];
            yr = fmaf(rr, xr, fmaf(-ri, xi, yr));
            yi = fmaf(rr, xi, fmaf(ri, xr, yi));
        }
        float *yo = Y + ((size_t)b * W + o) * S;
        yo[pr] = yr;
        yo[pi] = yi;
    }
}

// dX[b][c][mode] = sum_o conj(R[mode][c][o]) dY[b][o][mode]
__global__ void k_mix_adj(const float *__restrict__ dY, const float *__restrict__ R, int B, int W,
                          int m, float *__restrict__ dX)
{
    const int modes = 4 * m * m * m, S = 8 * m * m * m;
    const long long n = (long long)B * modes * W;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(t % W);
        const int mode = (int)((t / W) % modes);
        const int b = (int)(t / ((long long)W * modes));
        const int kx = mode % m, ky = (mode / m) % (2 * m), kz = mode / (2 * m * m);
        const int pr = spec_pos(kz, ky, kx, 0, m), pi = spec_pos(kz, ky, kx, 1, m);
        const float *Rc = R + ((size_t)mode * W + c) * W * 2;
        float xr = 0.0f, xi = 0.0f;
        for (int o = 0; o < W; ++o) {
            const float *yo = dY + ((size_t)b * W + o) * S;
            const float yr = yo[pr], yi = yo[pi];
            const float rr = Rc[2 * o], ri = Rc[2 * o + 1];
            xr = fmaf(rr, yr, fmaf(ri, yi, xr));
            xi = fmaf(rr, yi, fmaf(-ri, yr, xi));
        }
        float *xc = dX + ((size_t)b * W + c) * S;
        xc[pr] = xr;
        xc[pi] = xi;
    }
}

// dR[mode][c][o] += sum_b dY[b][o][mode] conj(X[b][c][mode])
__global__ void k_mix_dR(const float *__restrict__ dY, const float *__restrict__ X, int B, int W,
                         int m, float *__restrict__ dR)
{
    const int modes = 4 * m * m * m, S = 8 * m * m * m;
    const long long n = (long long)modes * W * W;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        const int o = (int)(t % W);
        const int c = (int)((t / W) % W);
        const int mode = (int)(t / ((long long)W * W));
        const int kx = mode % m, ky = (mode / m) % (2 * m), kz = mode / (2 * m * m);
        const int pr = spec_pos(kz, ky, kx, 0, m), pi = spec_pos(kz, ky, kx, 1, m);
        float gr = 0.0f, gi = 0.0f;
        for (int b = 0; b < B; ++b) {
            const float *yo = dY + ((size_t)b * W + o) * S;
            const float *xc = X + ((size_t)b * W + c) * S;
            const float yr = yo[pr], yi = yo[pi], xr = xc[pr], xi = xc[pi];
            gr = fmaf(yr, xr, fmaf(yi, xi, gr));
            gi = fmaf(yi, xr, fmaf(-yr, xi, gi));
        }
        dR[t * 2] += gr;
        dR[t * 2 + 1] += gi;
    }
}

// ------------------------------------------------------- tiled mode mix
// The mix and its adjoints move a layer's spectral weights (W x W complex per
// mode, 56.6 MB at width 32, m 12) and do little else.  A block takes KZ modes
// of one (ky, kx), which lie together in the spectra: their spectra of all
// samples and channels sit in shared memory, the weights of a mode stream
// through once for the whole batch, and results leave as they came in.  One
// thread per output that fetched every operand itself took 65 us (mix), 215
// (adjoint) and 235 (weight gradient) a layer at batch 4; now 49, and 98 for
// both adjoints.  Sums run in the same order as there.
//
// spectra tile: [b * W + c][part][KZ], channel rows padded by one float
struct MixTile {
    int B, W, m, KZ, pitch;
    __host__ __device__ MixTile(int B_, int W_, int m_, int kz) : B(B_), W(W_), m(m_), KZ(kz)
    {
        pitch = 2 * kz + 1;
    }
    __host__ __device__ size_t bytes() const { return (size_t)B * W * pitch * sizeof(float); }
};
// copy the tile of modes kz0 .. kz0 + n - 1 at (ky, kx) = yx between a spectrum
// array and shared memory
__device__ __forceinline__ void tile_io(float *tile, const MixTile &t, float *X, int yx, int kz0,
                                        int n, bool store)
{
    const int S2 = 2 * t.m;
    const size_t S = (size_t)8 * t.m * t.m * t.m;
    for (int e = threadIdx.x; e < t.B * t.W * 2 * t.KZ; e += blockDim.x) {
        const int z = e % t.KZ, part = e / t.KZ % 2, bc = e / (2 * t.KZ);
        if (z >= n) continue;
        float *x = X + bc * S + ((size_t)yx * 2 + part) * S2 + kz0 + z;
        float *p = tile + bc * t.pitch + part * t.KZ + z;
        if (store)
            *x = *p;
        else
            *p = *x;
    }
}

// Y[b][o][mode] = sum_c R[mode][c][o] X[b][c][mode]: 16 lanes take two outputs
// each (W / 2 in passes), for BT samples at a time
template <int BT>
__global__ void __launch_bounds__(256) k_mix_fwd_tile(float *X, const float *R, MixTile t, float *Y)
{
    extern __shared__ float s_mix[];
    float *sx = s_mix, *sy = s_mix + t.bytes() / sizeof(float);
    const int yx = blockIdx.x, kz0 = blockIdx.y * t.KZ, n = min(t.KZ, 2 * t.m - kz0);
    tile_io(sx, t, X, yx, kz0, n, false);
    __syncthreads();
    const int W = t.W, lane = threadIdx.x & 15, groups = blockDim.x >> 4;
    for (int w = threadIdx.x >> 4; w < n * (W / 32 + (W % 32 != 0)); w += groups) {
        const int z = w % n, o2 = w / n * 16 + lane;          // output pair
        if (2 * o2 >= W) continue;
        const size_t mode = (size_t)(kz0 + z) * 2 * t.m * t.m + yx;
        const float4 *r = reinterpret_cast<const float4 *>(R + mode * W * W * 2) + o2;
        for (int b0 = 0; b0 < t.B; b0 += BT) {
            float2 y0[BT], y1[BT];
#pragma unroll
            for (int b = 0; b < BT; ++b) y0[b] = y1[b] = make_float2(0.0f, 0.0f);
#pragma unroll 8
            for (int c = 0; c < W; ++c) {
                const float4 q = r[c * (W / 2)];
#pragma unroll
                for (int b = 0; b < BT; ++b) {
                    if (b0 + b >= t.B) break;
                    const float *x = sx + ((b0 + b) * W + c) * t.pitch + z;
                    const float xr = x[0], xi = x[t.KZ];
                    y0[b].x = fmaf(q.x, xr, fmaf(-q.y, xi, y0[b].x));
                    y0[b].y = fmaf(q.x, xi, fmaf(q.y, xr, y0[b].y));
                    y1[b].x = fmaf(q.z, xr, fmaf(-q.w, xi, y1[b].x));
                    y1[b].y = fmaf(q.z, xi, fmaf(q.w, xr, y1[b].y));
                }
            }
#pragma unroll
            for (int b = 0; b < BT; ++b) {
                if (b0 + b >= t.B) break;
                float *y = sy + ((b0 + b) * W + 2 * o2) * t.pitch + z;
                y[0] = y0[b].x;
                y[t.KZ] = y0[b].y;
                y[t.pitch] = y1[b].x;
                y[t.pitch + t.KZ] = y1[b].y;
            }
        }
    }
    __syncthreads();
    tile_io(sy, t, Y, yx, kz0, n, true);
}

// dX[b][c][mode] = sum_o conj(R[mode][c][o]) dY[b][o][mode] and
// dR[mode][c][o] = sum_b dY[b][o][mode] conj(X[b][c][mode]): a warp brings one
// mode's weights into shared memory (rows padded), sums its lanes' channels
// over the outputs, and writes the mode's weight gradient.  dX replaces X in
// its tile.
__global__ void __launch_bounds__(256) k_mix_bwd_tile(float *dY, float *X, const float *R, MixTile t,
                                                      float *dR, float *dX)
{
    extern __shared__ float s_mix[];
    const int W = t.W, tile = (int)(t.bytes() / sizeof(float));
    float *sy = s_mix, *sx = sy + tile, *sd = sx + tile;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int rp = W + 1;
    float2 *sr = reinterpret_cast<float2 *>(s_mix + (3 * tile + 1) / 2 * 2) + warp * W * rp;
    const int yx = blockIdx.x, kz0 = blockIdx.y * t.KZ, n = min(t.KZ, 2 * t.m - kz0);
    tile_io(sy, t, dY, yx, kz0, n, false);
    tile_io(sx, t, X, yx, kz0, n, false);
    __syncthreads();
    for (int z = warp; z < n; z += warps) {
        const size_t mode = (size_t)(kz0 + z) * 2 * t.m * t.m + yx;
        const float4 *r = reinterpret_cast<const float4 *>(R + mode * W * W * 2);
        float4 *g = reinterpret_cast<float4 *>(dR + mode * W * W * 2);
        __syncwarp();
#pragma unroll 4
        for (int e = lane; e < W * W / 2; e += 32) {
            const float4 q = r[e];
            const int c = e / (W / 2), o = 2 * (e - c * (W / 2));
            sr[c * rp + o] = make_float2(q.x, q.y);
            sr[c * rp + o + 1] = make_float2(q.z, q.w);
            float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            for (int b = 0; b < t.B; ++b) {
                const float *x = sx + (b * W + c) * t.pitch + z, *y = sy + (b * W + o) * t.pitch + z;
                const float xr = x[0], xi = x[t.KZ];
                const float yr = y[0], yi = y[t.KZ], zr = y[t.pitch], zi = y[t.pitch + t.KZ];
                a.x = fmaf(yr, xr, fmaf(yi, xi, a.x));
                a.y = fmaf(yi, xr, fmaf(-yr, xi, a.y));
                a.z = fmaf(zr, xr, fmaf(zi, xi, a.z));
                a.w = fmaf(zi, xr, fmaf(-zr, xi, a.w));
            }
            g[e] = a;
        }
        __syncwarp();
        for (int c = lane; c < W; c += 32)
            for (int b = 0; b < t.B; ++b) {
                float xr = 0.0f, xi = 0.0f;
#pragma unroll 8
                for (int o = 0; o < W; ++o) {
                    const float *y = sy + (b * W + o) * t.pitch + z;
                    const float yr = y[0], yi = y[t.KZ];
                    const float2 w = sr[c * rp + o];
                    xr = fmaf(w.x, yr, fmaf(w.y, yi, xr));
                    xi = fmaf(w.x, yi, fmaf(-w.y, yr, xi));
                }
                float *d = sd + (b * W + c) * t.pitch + z;
                d[0] = xr;
                d[t.KZ] = xi;
            }
    }
    __syncthreads();
    tile_io(sd, t, dX, yx, kz0, n, true);
}

// modes of a tile: as many of the 2m as leave room for two blocks per SM (`per`
// tiles and `extra` bytes a block), 0 if not even one fits
constexpr size_t kMixSmem = 110 * 1024;
inline int mix_modes(int B, int W, int m, int per, size_t extra)
{
    for (int kz = 2 * m; kz >= 1; kz = kz > 8 ? (kz + 1) / 2 : kz - 1)
        if (per * MixTile(B, W, m, kz).bytes() + extra <= kMixSmem) return kz;
    return 0;
}

// a kernel's shared-memory limit, raised once per process
template <auto Kernel>
cudaError_t mix_smem()
{
    static std::atomic<int> done{0};
    if (done.load(std::memory_order_acquire)) return cudaSuccess;
    const cudaError_t e =
        cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMixSmem);
    if (e == cudaSuccess) done.store(1, std::memory_order_release);
    return e;
}

// out[c] += sum over samples and voxels of x[b][c][p]
__global__ void k_chan_sum(const float *__restrict__ x, int B, int C, int N, float *__restrict__ out)
{
    const int c = blockIdx.y;
    float acc = 0.0f;
    for (int b = 0; b < B; ++b) {
        const float *xc = x + ((size_t)b * C + c) * N;
        const int step = gridDim.x * blockDim.x, t = blockIdx.x * blockDim.x + threadIdx.x;
        if (N % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0) {
            // four 16-byte loads in flight
            const float4 *x4 = reinterpret_cast<const float4 *>(xc);
            const int n4 = N / 4;
            for (int p = t; p < n4; p += 4 * step) {
                float4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    v[u] = p + u * step < n4 ? __ldg(x4 + p + u * step)
                                             : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                for (int u = 0; u < 4; ++u) acc += (v[u].x + v[u].y) + (v[u].z + v[u].w);
            }
        } else {
            for (int p = t; p < N; p += step) acc += xc[p];
        }
    }
    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    __shared__ float sh[32];
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        float v = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0f;
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) atomicAdd(out + c, v);
    }
}

// per sample: [0] sum (out0 - y)^2, [1] sum y^2, [2] sum out1 (FP64)
__global__ void k_loss_sums(const float *__restrict__ out, const float *__restrict__ y, int c_out,
                            int N, double *__restrict__ sums)
{
    const int b = blockIdx.y;
    const float *o0 = out + (size_t)b * c_out * N, *yb = y + (size_t)b * N;
    double e = 0.0, t = 0.0, s1 = 0.0;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < N; p += gridDim.x * blockDim.x) {
        const double d = (double)o0[p] - yb[p];
        e += d * d;
        t += (double)yb[p] * yb[p];
        if (c_out > 1) s1 += o0[N + p];
    }
    for (int o = 16; o; o >>= 1) {
        e += __shfl_xor_sync(0xffffffffu, e, o);
        t += __shfl_xor_sync(0xffffffffu, t, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(sums + 3 * b, e);
        atomicAdd(sums + 3 * b + 1, t);
        atomicAdd(sums + 3 * b + 2, s1);
    }
}

// d loss / d out for the loss of the file header (scale = 1 / batch)
__global__ void k_loss_grad(const float *__restrict__ out, const float *__restrict__ y,
                            const float *__restrict__ el, const double *__restrict__ sums, int B,
                            int c_out, int N, float el_weight, float *__restrict__ dout)
{
    // blockIdx.x: sample and channel, whose factor is the same for every voxel:
    // one thread's work, since FP64 is slow on this part (59 us at 64 x 64 x 96,
    // batch 4, with every thread making it; now 28)
    const int b = blockIdx.x / c_out, k = blockIdx.x % c_out;
    __shared__ bool s_on;
    __shared__ double s_f;
    if (threadIdx.x == 0) {
        const double *s = sums + 3 * b;
        bool on = false;
        double f = 0.0;
        if (k == 0) {
            const double rel = sqrt(s[0] / s[1]);
            on = rel > 0.0;
            if (on) f = 1.0 / (rel * s[1] * B);
        } else if (k == 1 && el) {
            f = 2.0 * el_weight * (s[2] / N - el[b]) / ((double)N * B);
        }
        s_on = on;
        s_f = f;
    }
    __syncthreads();
    const bool on = s_on;
    const double f = s_f;
    const float *o = out + (size_t)blockIdx.x * N, *yb = y + (size_t)b * N;
    float *d = dout + (size_t)blockIdx.x * N;
    for (int p = blockIdx.y * blockDim.x + threadIdx.x; p < N; p += gridDim.y * blockDim.x)
        d[p] = k == 0 ? (on ? (float)(((double)o[p] - yb[p]) * f) : 0.0f) : (float)f;
}

// sum of n floats into *out (FP64)
__global__ void k_sum(const float *__restrict__ x, size_t n, double *__restrict__ out)
{
    double acc = 0.0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        acc += x[i];
    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(out, acc);
}

__global__ void k_adam(float *__restrict__ w, const float *__restrict__ g, float *__restrict__ m1,
                       float *__restrict__ m2, size_t n, float lr, float b1, float b2, float eps,
                       float c1, float c2)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float a = b1 * m1[i] + (1.0f - b1) * gi;
        const float v = b2 * m2[i] + (1.0f - b2) * gi * gi;
        m1[i] = a;
        m2[i] = v;
        w[i] -= lr * (a / c1) / (sqrtf(v / c2) + eps);
    }
}

inline unsigned grid_for(long long n)
{
    long long b = (n + 255) / 256;
    return (unsigned)std::max(1LL, std::min(b, 152LL * 32));
}

}  // namespace

struct bvf_fno_bf16 {
    bvf_fno_dims d{};
    int nx = 0, ny = 0, nz = 0, N = 0, Bmax = 0;
    size_t n_w = 0;
    float *w = nullptr, *g = nullptr, *m1 = nullptr, *m2 = nullptr;
    long long adam_t = 0;
    // stage matrices: forward x (plain, weighted c/N), y, z; inverse z, y, x (weighted, plain)
    float *Fx = nullptr, *Fxw = nullptr, *Fy = nullptr, *Fz = nullptr;
    float *Gz = nullptr, *Gy = nullptr, *Gxw = nullptr, *Gx = nullptr;
    std::vector<float *> v, s, X;       // L+1 volumes, L-1 pre-activations, L spectra
    float *pre1 = nullptr, *h = nullptr, *out = nullptr;
    float *w1 = nullptr, *w2 = nullptr, *S1 = nullptr, *S2 = nullptr;
    float *dv = nullptr, *dv2 = nullptr, *dh = nullptr, *dout = nullptr;
    double *sums = nullptr;
    int *flag = nullptr;
    std::vector<void *> all;
    int n_sm = 152;
    int ksplit = 1;                     // K split of the voxel-sum products
};

namespace {

size_t layer_floats(const bvf_fno_dims &d)
{
    const size_t m = d.modes, W = d.width;
    return (2 * m) * (2 * m) * m * W * W * 2 + W * W + W;      // R, W, b
}

struct Off {
    size_t Wp, bp, lay0, lf, Q1, q1, Q2, q2;
};
Off offsets(const bvf_fno_dims &d)
{
    Off o{};
    o.Wp = 0;
    o.bp = (size_t)d.width * d.c_in;
    o.lay0 = o.bp + d.width;
    o.lf = layer_floats(d);
    o.Q1 = o.lay0 + (size_t)d.n_layers * o.lf;
    o.q1 = o.Q1 + (size_t)d.hidden * d.width;
    o.Q2 = o.q1 + d.hidden;
    o.q2 = o.Q2 + (size_t)d.c_out * d.hidden;
    return o;
}

template <typename P>
int dalloc(bvf_fno_bf16 *t, P **p, size_t n, const char *what)
{
    cudaError_t e = cudaMalloc((void **)p, n * sizeof(P));
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return b16_fail(BVF_E_NOMEM, std::string("bvf_fno_bf16_create: ") + what);
    }
    t->all.push_back(*p);
    return BVF_OK;
}

// stage matrices in FP64, rounded once to FP32
void build_matrices(int nx, int ny, int nz, int m, std::vector<std::vector<float>> &out)
{
    const double N = (double)nx * ny * nz;
    auto wk = [&](int kx) { return (kx == 0 ? 1.0 : 2.0) / N; };
    std::vector<float> Fx((size_t)nx * 2 * m), Fxw(Fx.size()), Gx((size_t)2 * m * nx), Gxw(Gx.size());
    for (int x = 0; x < nx; ++x)
        for (int kx = 0; kx < m; ++kx) {
            const double ph = 2.0 * kPi * kx * x / nx, c = std::cos(ph), s = std::sin(ph);
            Fx[(size_t)x * 2 * m + kx] = (float)c;
            Fx[(size_t)x * 2 * m + m + kx] = (float)(-s);
            Fxw[(size_t)x * 2 * m + kx] = (float)(wk(kx) * c);
            Fxw[(size_t)x * 2 * m + m + kx] = (float)(-wk(kx) * s);
            Gx[(size_t)kx * nx + x] = (float)c;
            Gx[(size_t)(m + kx) * nx + x] = (float)(-s);
            Gxw[(size_t)kx * nx + x] = (float)(wk(kx) * c);
            Gxw[(size_t)(m + kx) * nx + x] = (float)(-wk(kx) * s);
        }
    // complex stage along an axis of length n over the 2m slots, forward
    // (e^{-i theta}, K = [part][n] -> N = [part][slot]) and inverse
    // (e^{+i theta}, K = [part][slot] -> N = [part][n])
    auto axis = [&](int n, std::vector<float> &F, std::vector<float> &G) {
        const int S = 2 * m;
        F.assign((size_t)2 * n * 2 * S, 0.0f);
        G.assign((size_t)2 * S * 2 * n, 0.0f);
        for (int q = 0; q < n; ++q)
            for (int j = 0; j < S; ++j) {
                const double th = 2.0 * kPi * slot_freq(j, m) * q / n, c = std::cos(th), s = std::sin(th);
                // forward: re' = a cos + b sin, im' = b cos - a sin
                F[(size_t)q * 2 * S + j] = (float)c;
                F[(size_t)q * 2 * S + S + j] = (float)(-s);
                F[(size_t)(n + q) * 2 * S + j] = (float)s;
                F[(size_t)(n + q) * 2 * S + S + j] = (float)c;
                // inverse: re' = a cos - b sin, im' = b cos + a sin
                G[(size_t)j * 2 * n + q] = (float)c;
                G[(size_t)j * 2 * n + n + q] = (float)s;
                G[(size_t)(S + j) * 2 * n + q] = (float)(-s);
                G[(size_t)(S + j) * 2 * n + n + q] = (float)c;
            }
    };
    std::vector<float> Fy, Gy, Fz, Gz;
    axis(ny, Fy, Gy);
    axis(nz, Fz, Gz);
    out = {Fx, Fxw, Fy, Fz, Gz, Gy, Gxw, Gx};
}

// C[rows][N] = A[rows][K] B[K][N] (all row-major, B shared)
bvf_gemm rowmajor(const float *A, const float *B, float *C, long long rows, int K, int N)
{
    bvf_gemm g{};
    g.A = A;
    g.sam = K;
    g.sak = 1;
    g.B = B;
    g.sbk = N;
    g.sbn = 1;
    g.C = C;
    g.scm = N;
    g.scn = 1;
    g.M = (int)rows;
    g.N = N;
    g.K = K;
    g.batch = 1;
    g.ksplit = 1;
    g.alpha = 1.0f;
    return g;
}

int gemm(bvf_fno_bf16 *t, const GemmX &x, cudaStream_t s, const char *what)
{
    BCK(launch_gemm_bf16(x, t->flag, s), what);
    return BVF_OK;
}
int gemm(bvf_fno_bf16 *t, const bvf_gemm &g, cudaStream_t s, const char *what)
{
    GemmX x;
    x.g = g;
    return gemm(t, x, s, what);
}

// Between the stages of a transform the axes change places.  Each product
// reads and writes its neighbours' order directly (GemmX): with separate
// permutes every stage's output was read and written once more, 1.56 of 28.2
// ms of a forward at 240 x 240 x 200 and 2.05 of 17.3 ms of a gradient at
// 64 x 64 x 96, batch 4.

// forward transform of BC real volumes -> BC spectra (weighted: the x stage
// carries c(kx)/N, the adjoint of the inverse)
int spec_fwd(bvf_fno_bf16 *t, const float *in, long long BC, bool weighted, float *S, cudaStream_t s)
{
    const int nx = t->nx, ny = t->ny, nz = t->nz, m = t->d.modes;
    int rc;
    // x: rows (bc, z, y) -> w1 [bc][z][part][kx][y]
    const long long rows = BC * nz * ny;
    cudaError_t e = cudaErrorNotSupported;
    if (bvf::xfwd_fits(false, in, rows, nx, m)) {
        bvf::XfwdArgs q{};
        q.v = in;
        q.R = rows;
        q.nx = nx;
        q.m = m;
        q.F = weighted ? t->Fxw : t->Fx;
        q.outw = t->w1;
        q.ny = ny;
        q.n_sm = t->n_sm;
        q.flag = t->flag;
        e = bvf::launch_xfwd(false, q, s);
        if (e != cudaErrorNotSupported) BCK(e, "spectral x");
    }
    GemmX x;
    x.g = rowmajor(in, weighted ? t->Fxw : t->Fx, t->w1, BC * nz * ny, nx, 2 * m);
    x.rc = ny;
    x.scm1 = 2LL * m * ny;
    x.g.scm = 1;
    x.g.scn = ny;
    if (e == cudaErrorNotSupported && (rc = gemm(t, x, s, "spectral x")) != BVF_OK) return rc;
    // y: rows (bc, kx, z), K (part, y) -> w2 [bc][part][ky][kx][z]
    x = GemmX();
    x.g = rowmajor(t->w1, t->Fy, t->w2, BC * nz * m, 2 * ny, 4 * m);
    x.ra = nz;
    x.ra2 = m;
    x.g.sam = 2LL * m * ny;
    x.sam1 = ny;
    x.sam2 = 2LL * m * ny * nz;
    x.ka = ny;
    x.sak1 = (long long)m * ny;
    x.rc = m * nz;
    x.scm1 = 4LL * m * m * nz;
    x.g.scm = 1;
    x.g.scn = (long long)m * nz;
    if ((rc = gemm(t, x, s, "spectral y")) != BVF_OK) return rc;
    // z: rows (bc, ky, kx), K (part, z) -> S [bc][ky][kx][part][kz]
    x = GemmX();
    x.g = rowmajor(t->w2, t->Fz, S, BC * 2 * m * m, 2 * nz, 4 * m);
    x.ra = 2 * m * m;
    x.g.sam = nz;
    x.sam2 = 4LL * m * m * nz;
    x.ka = nz;
    x.sak1 = 2LL * m * m * nz;
    return gemm(t, x, s, "spectral z");
}

// the z and y stages of the inverse transform of BC spectra: what its x stage
// reads, w2 [bc][z][y][part][kx]
int spec_inv_zy(bvf_fno_bf16 *t, const float *S, long long BC, cudaStream_t s)
{
    const int ny = t->ny, nz = t->nz, m = t->d.modes;
    // z: rows (bc, ky, kx) -> w1 [bc][ky][kx][part][z]
    const int rc = gemm(t, rowmajor(S, t->Gz, t->w1, BC * 2 * m * m, 4 * m, 2 * nz), s, "inverse z");
    if (rc != BVF_OK) return rc;
    // y: rows (bc, z, kx), K (part, ky)
    GemmX x;
    x.g = rowmajor(t->w1, t->Gy, t->w2, BC * nz * m, 4 * m, 2 * ny);
    x.ra = m;
    x.ra2 = nz;
    x.g.sam = 2LL * nz;
    x.sam1 = 1;
    x.sam2 = 4LL * m * m * nz;
    x.ka = 2 * m;
    x.g.sak = 2LL * m * nz;
    x.sak1 = nz;
    x.rc = m;
    x.scm1 = 2LL * m * ny;
    x.g.scm = 1;
    x.nc = ny;
    x.g.scn = 2 * m;
    x.scn1 = m;
    return gemm(t, x, s, "inverse y");
}

// channel mix out[b][o][p] (+)= sum_c Wt[o][c] in[b][c][p] (Wt row-major [O][C])
bvf_gemm chan(const float *in, int C, const float *Wt, float *out, int O, int N, int B)
{
    bvf_gemm g{};
    g.A = in;
    g.sam = 1;
    g.sak = N;
    g.sab = (long long)C * N;
    g.B = Wt;
    g.sbk = 1;
    g.sbn = C;
    g.sbb = 0;
    g.C = out;
    g.scm = 1;
    g.scn = N;
    g.scb = (long long)O * N;
    g.M = N;
    g.N = O;
    g.K = C;
    g.batch = B;
    g.ksplit = 1;
    g.alpha = 1.0f;
    return g;
}

// weight gradient G[o][c] += sum_{b,p} d[b][o][p] x[b][c][p]
bvf_gemm wgrad(const float *d, int O, const float *x, int C, float *G, int N, int B, int ksplit)
{
    bvf_gemm g{};
    g.A = d;
    g.sam = N;
    g.sak = 1;
    g.sab = (long long)O * N;
    g.B = x;
    g.sbk = 1;
    g.sbn = N;
    g.sbb = (long long)C * N;
    g.C = G;
    g.scm = C;
    g.scn = 1;
    g.scb = 0;
    g.M = O;
    g.N = C;
    g.K = N;
    g.batch = B;
    g.ksplit = std::max(2, ksplit);   // the batch shares G: always the atomic path
    g.alpha = 1.0f;
    g.beta = 1.0f;
    return g;
}

int chan_sum(const float *x, int B, int C, int N, float *out, cudaStream_t s)
{
    k_chan_sum<<<dim3(std::min(64, (N + 255) / 256), C), 256, 0, s>>>(x, B, C, N, out);
    BCK(cudaGetLastError(), "channel sum");
    return BVF_OK;
}

// G += d x^T and g += the sums of d over the batch's points.  Volumes whose
// rows are no whole 16-byte pieces take a general product and separate sums.
int weight_grad(bvf_fno_bf16 *t, int batch, const float *dd, int O, const float *x, int C, float *G,
                float *g, cudaStream_t s)
{
    const WgradBf16 q{dd, x, O, C, G, g, batch, t->N, t->flag};
    if (bvf::wgrad_fits(q)) {
        BCK(bvf::launch_wgrad_bf16(q, t->n_sm, s), "weight gradient");
        return BVF_OK;
    }
    const int rc = gemm(t, wgrad(dd, O, x, C, G, t->N, batch, t->ksplit), s, "weight gradient");
    return rc != BVF_OK ? rc : chan_sum(dd, batch, O, t->N, g, s);
}

// Y = R X per mode
int mix_forward(bvf_fno_bf16 *t, int batch, float *X, const float *Rw, float *Y, cudaStream_t s)
{
    const int W = t->d.width, m = t->d.modes, kz = mix_modes(batch, W, m, 2, 0);
    if (!kz) {
        k_mix_fwd<<<grid_for((long long)batch * 4 * m * m * m * W), 256, 0, s>>>(X, Rw, batch, W, m, Y);
    } else {
        const MixTile tile(batch, W, m, kz);
        const dim3 grid(2 * m * m, (2 * m + kz - 1) / kz);
        const size_t smem = 2 * tile.bytes();
        if (batch == 1) {
            BCK(mix_smem<k_mix_fwd_tile<1>>(), "mix");
            k_mix_fwd_tile<1><<<grid, 256, smem, s>>>(X, Rw, tile, Y);
        } else {
            BCK(mix_smem<k_mix_fwd_tile<4>>(), "mix");
            k_mix_fwd_tile<4><<<grid, 256, smem, s>>>(X, Rw, tile, Y);
        }
    }
    BCK(cudaGetLastError(), "mix");
    return BVF_OK;
}

// dR = dY conj(X) summed over the batch, dX = conj(R) dY (gR starts at zero)
int mix_backward(bvf_fno_bf16 *t, int batch, float *dY, float *X, const float *Rw, float *gR,
                 float *dX, cudaStream_t s)
{
    const int W = t->d.width, m = t->d.modes;
    const int warps = W <= 32 ? 8 : 2;                    // a warp holds one mode's weights
    const size_t wb = (size_t)warps * W * (W + 1) * sizeof(float2) + 16;
    const int kz = mix_modes(batch, W, m, 3, wb);
    const MixTile tile(batch, W, m, kz ? kz : 1);
    const size_t smem = 3 * tile.bytes() + wb;
    if (!kz) {                                            // a batch too large for a tile
        k_mix_dR<<<grid_for((long long)4 * m * m * m * W * W), 256, 0, s>>>(dY, X, batch, W, m, gR);
        k_mix_adj<<<grid_for((long long)batch * 4 * m * m * m * W), 256, 0, s>>>(dY, Rw, batch, W, m, dX);
    } else {
        BCK(mix_smem<k_mix_bwd_tile>(), "d mix");
        k_mix_bwd_tile<<<dim3(2 * m * m, (2 * m + kz - 1) / kz), 32 * warps, smem, s>>>(dY, X, Rw, tile,
                                                                                      gR, dX);
    }
    BCK(cudaGetLastError(), "d mix");
    return BVF_OK;
}

// One row pass over `batch` samples: out = act(Inv_x(w2) + mix of v + bias)
// with the channel weights Wm(o, c) at o wso + c wsc (v has cin channels); G
// the x stage's matrix, NULL for no spectral term.  act as in bvf_gemm.  Rows
// too long for shared memory take the two products, with the sum through
// `out`.
int row_pass(bvf_fno_bf16 *t, int batch, const float *v, int cin, const float *Wm, int wso, int wsc,
             const float *bias, const float *G, int act, float *pre, float *out, cudaStream_t s)
{
    const int W = t->d.width, m = t->d.modes, N = t->N;
    if (bvf::row_bf16_fits(W, m, t->nx)) {
        RowBf16 q{v, (long long)cin * N, cin, Wm, wso, wsc, bias, G ? t->w2 : nullptr, G, pre, act,
                  out, batch, t->nx, t->ny * t->nz, m, N, t->n_sm, t->flag};
        BCK(bvf::launch_row_bf16(q, W, s), "row pass");
        return BVF_OK;
    }
    if (G) {
        const int rc = gemm(t, rowmajor(t->w2, G, out, (long long)batch * W * t->nz * t->ny, 2 * m,
                                        t->nx), s, "inverse x");
        if (rc != BVF_OK) return rc;
    }
    bvf_gemm g = chan(v, cin, Wm, out, W, N, batch);
    g.sbk = wsc;
    g.sbn = wso;
    g.beta = G ? 1.0f : 0.0f;
    g.bias = bias;
    g.bias_mode = bias ? 1 : 0;
    g.act = act;
    g.C_pre = pre;
    return gemm(t, g, s, "pointwise");
}

// out = act(Wm v + bias), K input and O output channels (Wm(o, c) at o wso + c wsc)
int chan_pass(bvf_fno_bf16 *t, int batch, const float *v, int K, const float *Wm, int wso, int wsc,
              const float *bias, int act, float *pre, float *out, int O, cudaStream_t s)
{
    const ChanBf16 q{v, K, O, Wm, wso, wsc, bias, pre, act, out, batch, t->N, t->flag};
    BCK(bvf::launch_chan_bf16(q, t->n_sm, s), "channel product");
    return BVF_OK;
}

// forward pass of `batch` samples into `out` ([batch][c_out][N]); with `keep`
// every activation the backward pass needs is kept, without it (inference)
// the pre-activations are not written
int forward(bvf_fno_bf16 *t, int batch, const float *in, float *out, bool keep, cudaStream_t s)
{
    const bvf_fno_dims &d = t->d;
    const int W = d.width, N = t->N, L = d.n_layers, m = d.modes;
    const Off o = offsets(d);
    const float *w = t->w;
    int rc;
    if ((rc = row_pass(t, batch, in, d.c_in, w + o.Wp, d.c_in, 1, w + o.bp, nullptr, 0, nullptr,
                       t->v[0], s)) != BVF_OK)
        return rc;
    for (int l = 0; l < L; ++l) {
        const float *lw = w + o.lay0 + l * o.lf;
        const float *R = lw, *Wl = lw + (size_t)4 * m * m * m * W * W * 2, *bl = Wl + (size_t)W * W;
        if ((rc = spec_fwd(t, t->v[l], (long long)batch * W, false, t->X[l], s)) != BVF_OK) return rc;
        if ((rc = mix_forward(t, batch, t->X[l], R, t->S1, s)) != BVF_OK) return rc;
        if ((rc = spec_inv_zy(t, t->S1, (long long)batch * W, s)) != BVF_OK) return rc;
        const int act = l < L - 1;
        if ((rc = row_pass(t, batch, t->v[l], W, Wl, W, 1, bl, t->Gxw, act,
                           act && keep ? t->s[l] : nullptr, t->v[l + 1], s)) != BVF_OK)
            return rc;
    }
    if (!keep) {
        BCK(bvf::launch_project_bf16(t->v[L], w + o.Q1, w + o.q1, w + o.Q2, w + o.q2, W, d.hidden,
                                     d.c_out, out, N, batch, t->n_sm, t->flag, s),
            "projection");
        return BVF_OK;
    }
    if ((rc = chan_pass(t, batch, t->v[L], W, w + o.Q1, W, 1, w + o.q1, 1, t->pre1, t->h, d.hidden,
                        s)) != BVF_OK)
        return rc;
    return chan_pass(t, batch, t->h, d.hidden, w + o.Q2, d.hidden, 1, w + o.q2, 0, nullptr, out,
                     d.c_out, s);
}

// loss and gradient into t->g (zeroed first); h_loss on the host
int gradient(bvf_fno_bf16 *t, int batch, const float *in, const float *target, const float *el,
             double el_weight, double *h_loss, cudaStream_t s)
{
    const bvf_fno_dims &d = t->d;
    const int W = d.width, N = t->N, L = d.n_layers, m = d.modes, H = d.hidden;
    const Off o = offsets(d);
    int rc = forward(t, batch, in, t->out, true, s);
    if (rc != BVF_OK) return rc;
    BCK(cudaMemsetAsync(t->sums, 0, 3 * sizeof(double) * batch, s), "loss");
    k_loss_sums<<<dim3(std::min(64, (N + 255) / 256), batch), 256, 0, s>>>(t->out, target, d.c_out,
                                                                          N, t->sums);
    k_loss_grad<<<dim3(batch * d.c_out, std::min(256, (N + 255) / 256)), 256, 0, s>>>(
        t->out, target, d.c_out > 1 ? el : nullptr, t->sums, batch, d.c_out, N, (float)el_weight,
        t->dout);
    BCK(cudaGetLastError(), "loss");
    BCK(cudaMemsetAsync(t->g, 0, t->n_w * sizeof(float), s), "gradient");
    float *G = t->g;
    const float *w = t->w;
    // projection
    if ((rc = chan_pass(t, batch, t->dout, d.c_out, w + o.Q2, 1, H, nullptr, 2, t->pre1, t->dh, H,
                        s)) != BVF_OK)                 // dh -> d pre1
        return rc;
    if ((rc = weight_grad(t, batch, t->dout, d.c_out, t->h, H, G + o.Q2, G + o.q2, s)) != BVF_OK)
        return rc;
    if ((rc = weight_grad(t, batch, t->dh, H, t->v[L], W, G + o.Q1, G + o.q1, s)) != BVF_OK)
        return rc;
    if ((rc = chan_pass(t, batch, t->dh, H, w + o.Q1, 1, W, nullptr, 0, nullptr, t->dv, W, s)) !=
        BVF_OK)
        return rc;
    // Fourier layers, top down; ds holds d(pre-activation) of layer l
    float *ds = t->dv, *dn = t->dv2;
    for (int l = L - 1; l >= 0; --l) {
        const float *lw = w + o.lay0 + l * o.lf;
        float *gl = G + o.lay0 + l * o.lf;
        const float *R = lw, *Wl = lw + (size_t)4 * m * m * m * W * W * 2;
        float *gR = gl, *gW = gl + (size_t)4 * m * m * m * W * W * 2, *gb = gW + (size_t)W * W;
        if ((rc = weight_grad(t, batch, ds, W, t->v[l], W, gW, gb, s)) != BVF_OK) return rc;
        if ((rc = spec_fwd(t, ds, (long long)batch * W, true, t->S1, s)) != BVF_OK) return rc;
        if ((rc = mix_backward(t, batch, t->S1, t->X[l], R, gR, t->S2, s)) != BVF_OK) return rc;
        // dn = d v_l; for l > 0 it becomes d s_{l-1} = d v_l GELU'(s_{l-1})
        if ((rc = spec_inv_zy(t, t->S2, (long long)batch * W, s)) != BVF_OK) return rc;
        if ((rc = row_pass(t, batch, ds, W, Wl, 1, W, nullptr, t->Gx, l > 0 ? 2 : 0,
                           l > 0 ? t->s[l - 1] : nullptr, dn, s)) != BVF_OK)
            return rc;
        std::swap(ds, dn);
    }
    // lift
    if ((rc = weight_grad(t, batch, ds, W, in, d.c_in, G + o.Wp, G + o.bp, s)) != BVF_OK) return rc;
    if (h_loss) {
        std::vector<double> h(3 * batch);
        BCK(cudaMemcpyAsync(h.data(), t->sums, h.size() * sizeof(double), cudaMemcpyDeviceToHost, s),
            "loss");
        std::vector<float> e(batch);
        if (d.c_out > 1 && el)
            BCK(cudaMemcpyAsync(e.data(), el, batch * sizeof(float), cudaMemcpyDeviceToHost, s), "loss");
        BCK(cudaStreamSynchronize(s), "loss");
        double loss = 0.0;
        for (int b = 0; b < batch; ++b) {
            loss += std::sqrt(h[3 * b] / h[3 * b + 1]) / batch;
            if (d.c_out > 1 && el) {
                const double dm = h[3 * b + 2] / N - e[b];
                loss += el_weight * dm * dm / batch;
            }
        }
        *h_loss = loss;
    }
    return BVF_OK;
}

}  // namespace

extern "C" {

int bvf_fno_bf16_create(bvf_fno_bf16 **out, const bvf_fno_dims *d, const float *h_weights, size_t n,
                        int nx, int ny, int nz, int max_batch)
{
    if (!out) return b16_fail(BVF_E_ARG, "bvf_fno_bf16_create: out is NULL");
    *out = nullptr;
    if (!d || !h_weights || bvf_fno_weight_count(d) == 0 || n != bvf_fno_weight_count(d))
        return b16_fail(BVF_E_ARG, "bvf_fno_bf16_create: bad dims or weight count");
    const int m = d->modes;
    if (nx < 1 || ny < 1 || nz < 1 || m > nx / 2 || 2 * m > ny || 2 * m > nz || max_batch < 1 ||
        (long long)nx * ny * nz * max_batch * std::max(d->hidden, d->width) >= (1LL << 31))
        return b16_fail(BVF_E_ARG, "bvf_fno_bf16_create: grid too small for the modes, or too large");
    bvf_fno_bf16 *t = new (std::nothrow) bvf_fno_bf16;
    if (!t) return b16_fail(BVF_E_NOMEM, "bvf_fno_bf16_create: host allocation");
    t->d = *d;
    t->nx = nx;
    t->ny = ny;
    t->nz = nz;
    t->N = nx * ny * nz;
    t->Bmax = max_batch;
    t->n_w = n;
    auto fail = [&](int rc) {
        bvf_fno_bf16_destroy(t);
        return rc;
    };
    const size_t N = t->N, B = max_batch, W = d->width, H = d->hidden, S = 8 * (size_t)m * m * m;
    int rc = BVF_OK;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&t->n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return fail(b16_fail(BVF_E_CUDA, "bvf_fno_bf16_create: device"));
    for (float **p : {&t->w, &t->g, &t->m1, &t->m2})
        if ((rc = dalloc(t, p, n, "weights")) != BVF_OK) return fail(rc);
    std::vector<std::vector<float>> mats;
    build_matrices(nx, ny, nz, m, mats);
    float **mp[8] = {&t->Fx, &t->Fxw, &t->Fy, &t->Fz, &t->Gz, &t->Gy, &t->Gxw, &t->Gx};
    for (int i = 0; i < 8; ++i) {
        if ((rc = dalloc(t, mp[i], mats[i].size(), "stage matrices")) != BVF_OK) return fail(rc);
        if (cudaMemcpy(*mp[i], mats[i].data(), mats[i].size() * sizeof(float),
                       cudaMemcpyHostToDevice) != cudaSuccess)
            return fail(b16_fail(BVF_E_CUDA, "bvf_fno_bf16_create: copy"));
    }
    t->v.resize(d->n_layers + 1);
    t->s.resize(std::max(0, d->n_layers - 1));
    t->X.resize(d->n_layers);
    for (auto &p : t->v)
        if ((rc = dalloc(t, &p, B * W * N, "activations")) != BVF_OK) return fail(rc);
    for (auto &p : t->s)
        if ((rc = dalloc(t, &p, B * W * N, "activations")) != BVF_OK) return fail(rc);
    for (auto &p : t->X)
        if ((rc = dalloc(t, &p, B * W * S, "spectra")) != BVF_OK) return fail(rc);
    const size_t ws = std::max({B * W * nz * ny * 2 * m, B * W * nz * m * 4 * m,
                                B * W * 2 * m * m * 4 * m, B * W * 2 * m * m * 2 * nz,
                                B * W * nz * m * 2 * ny});
    if ((rc = dalloc(t, &t->pre1, B * H * N, "projection")) != BVF_OK ||
        (rc = dalloc(t, &t->h, B * H * N, "projection")) != BVF_OK ||
        (rc = dalloc(t, &t->dh, B * H * N, "projection")) != BVF_OK ||
        (rc = dalloc(t, &t->out, B * d->c_out * N, "output")) != BVF_OK ||
        (rc = dalloc(t, &t->dout, B * d->c_out * N, "output")) != BVF_OK ||
        (rc = dalloc(t, &t->w1, ws, "work")) != BVF_OK ||
        (rc = dalloc(t, &t->w2, ws, "work")) != BVF_OK ||
        (rc = dalloc(t, &t->S1, B * W * S, "spectra")) != BVF_OK ||
        (rc = dalloc(t, &t->S2, B * W * S, "spectra")) != BVF_OK ||
        (rc = dalloc(t, &t->dv, B * W * N, "gradients")) != BVF_OK ||
        (rc = dalloc(t, &t->dv2, B * W * N, "gradients")) != BVF_OK ||
        (rc = dalloc(t, &t->sums, 3 * B, "loss")) != BVF_OK ||
        (rc = dalloc(t, &t->flag, 1, "flag")) != BVF_OK)
        return fail(rc);
    if (cudaMemcpy(t->w, h_weights, n * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(t->m1, 0, n * sizeof(float)) != cudaSuccess ||
        cudaMemset(t->m2, 0, n * sizeof(float)) != cudaSuccess ||
        cudaMemset(t->flag, 0, sizeof(int)) != cudaSuccess)
        return fail(b16_fail(BVF_E_CUDA, "bvf_fno_bf16_create: initial copies"));
    // voxel sums of the weight gradients: enough K-split blocks to fill the GPU
    t->ksplit = (int)std::max<long long>(1, std::min<long long>(256, (long long)N / 4096));
    *out = t;
    return BVF_OK;
}

int bvf_fno_bf16_destroy(bvf_fno_bf16 *t)
{
    if (!t) return BVF_OK;
    cudaDeviceSynchronize();
    for (void *p : t->all) cudaFree(p);
    delete t;
    return BVF_OK;
}

int bvf_fno_bf16_forward(bvf_fno_bf16 *t, int batch, const float *d_in, float *d_out, void *stream)
{
    if (!t || !d_in || !d_out || batch < 1 || batch > t->Bmax)
        return b16_fail(BVF_E_ARG, "bvf_fno_bf16_forward: bad argument");
    return forward(t, batch, d_in, d_out, false, static_cast<cudaStream_t>(stream));
}

int bvf_fno_bf16_gradient(bvf_fno_bf16 *t, int batch, const float *d_in, const float *d_target,
                          const float *d_el, double el_weight, float *d_grad, double *h_loss,
                          void *stream)
{
    if (!t || !d_in || !d_target || batch < 1 || batch > t->Bmax || !(el_weight >= 0.0) ||
        (t->d.c_out > 1 && el_weight > 0.0 && !d_el))
        return b16_fail(BVF_E_ARG, "bvf_fno_bf16_gradient: bad argument");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int rc = gradient(t, batch, d_in, d_target, d_el, el_weight, h_loss, s);
    if (rc != BVF_OK) return rc;
    if (d_grad)
        BCK(cudaMemcpyAsync(d_grad, t->g, t->n_w * sizeof(float), cudaMemcpyDeviceToDevice, s),
            "bvf_fno_bf16_gradient: copy");
    return BVF_OK;
}

int bvf_fno_bf16_adam(bvf_fno_bf16 *t, int batch, const float *d_in, const float *d_target,
                      const float *d_el, double el_weight, double lr, double *h_loss, void *stream)
{
    if (!t || !(lr > 0.0)) return b16_fail(BVF_E_ARG, "bvf_fno_bf16_adam: bad argument");
    int rc = bvf_fno_bf16_gradient(t, batch, d_in, d_target, d_el, el_weight, nullptr, h_loss, stream);
    if (rc != BVF_OK) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const double b1 = 0.9, b2 = 0.999;
    ++t->adam_t;
    const float c1 = (float)(1.0 - std::pow(b1, (double)t->adam_t));
    const float c2 = (float)(1.0 - std::pow(b2, (double)t->adam_t));
    k_adam<<<grid_for((long long)t->n_w), 256, 0, s>>>(t->w, t->g, t->m1, t->m2, t->n_w, (float)lr,
                                                      (float)b1, (float)b2, 1e-8f, c1, c2);
    BCK(cudaGetLastError(), "bvf_fno_bf16_adam");
    return BVF_OK;
}

int bvf_fno_bf16_weights(bvf_fno_bf16 *t, float *h_weights)
{
    if (!t || !h_weights) return b16_fail(BVF_E_ARG, "bvf_fno_bf16_weights: bad argument");
    BCK(cudaDeviceSynchronize(), "bvf_fno_bf16_weights");
    BCK(cudaMemcpy(h_weights, t->w, t->n_w * sizeof(float), cudaMemcpyDeviceToHost),
        "bvf_fno_bf16_weights");
    return BVF_OK;
}

int bvf_fno_mean(const float *d_x, size_t n, double *h_mean, void *stream)
{
    if (!d_x || !h_mean || n == 0) return b16_fail(BVF_E_ARG, "bvf_fno_mean: bad argument");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    double *d = nullptr;
    BCK(cudaMallocAsync((void **)&d, sizeof(double), s), "bvf_fno_mean");
    double h = 0.0;
    cudaError_t e = cudaMemsetAsync(d, 0, sizeof(double), s);
    if (e == cudaSuccess) {
        k_sum<<<grid_for((long long)n), 256, 0, s>>>(d_x, n, d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFreeAsync(d, s);
    BCK(e, "bvf_fno_mean");
    *h_mean = h / (double)n;
    return BVF_OK;
}

int bvf_fno_bf16_synchronize(bvf_fno_bf16 *t, void *stream)
{
    if (!t) return b16_fail(BVF_E_ARG, "bvf_fno_bf16_synchronize: NULL");
    BCK(cudaStreamSynchronize(static_cast<cudaStream_t>(stream)), "bvf_fno_bf16_synchronize");
    int f = 0;
    BCK(cudaMemcpy(&f, t->flag, sizeof(int), cudaMemcpyDeviceToHost), "bvf_fno_bf16_synchronize");
    if (f) {
        cudaMemset(t->flag, 0, sizeof(int));
        return b16_fail(BVF_E_CUDA, "bvf_fno_bf16: a bounded wait for the tensor cores ran out");
    }
    return BVF_OK;
}

}  // extern "C"
