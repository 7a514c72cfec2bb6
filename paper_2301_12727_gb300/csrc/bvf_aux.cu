// Auxiliary kernels: index-range scan, pressure / amplitude-phase read-out,
// Rayleigh-Sommerfeld bowl field (Sec. 2.3), BHTE + CEM43 step (Sec. 2.4),
// and the E_L reductions (Sec. 2.4, Eq. 2).
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>
#include <cmath>

#include "bvf_stencil.cuh"
#include "bvf_tma.cuh"

namespace bvf {

namespace {

constexpr int kThreads = 256;

inline unsigned blocks_for(size_t n, int per_block = kThreads, unsigned cap = 152u * 16u)
{
    size_t b = (n + per_block - 1) / per_block;
    return (unsigned)(b < cap ? (b ? b : 1) : cap);
}

// element q of a dense array in one with row pitch r.pitch
__device__ __forceinline__ size_t in_rows(size_t q, Rows r)
{
    if (r.pitch == r.nx) return q;
    const unsigned row = (unsigned)q / r.nx;
    return (size_t)row * r.pitch + ((unsigned)q - row * r.nx);
}

// f(q, i) for the n elements q of a dense array, i the same element of one whose
// rows lie r.pitch apart: a thread each, or a warp per row where they do.
template <class F>
__device__ __forceinline__ void for_rows(size_t n, Rows r, F f)
{
    if (r.pitch == r.nx) {
        for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n;
             q += (size_t)gridDim.x * blockDim.x)
            f(q, q);
        return;
    }
    const size_t rows = n / r.nx, step = (size_t)gridDim.x * (blockDim.x / 32);
    for (size_t row = blockIdx.x * (size_t)(blockDim.x / 32) + (threadIdx.x >> 5); row < rows; row += step) {
        const size_t q = row * r.nx, i = row * r.pitch;
#pragma unroll 4
        for (unsigned x = threadIdx.x & 31; x < r.nx; x += 32) f(q + x, i + x);
    }
}

// out[q] = f(i) likewise, four values of a row in flight
template <class F>
__device__ __forceinline__ void rows_out(float *out, size_t n, Rows r, F f)
{
    if (r.pitch == r.nx) {
        for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n;
             q += (size_t)gridDim.x * blockDim.x)
            out[q] = f(q);
        return;
    }
    const size_t rows = n / r.nx, step = (size_t)gridDim.x * (blockDim.x / 32);
    for (size_t row = blockIdx.x * (size_t)(blockDim.x / 32) + (threadIdx.x >> 5); row < rows; row += step) {
        const size_t q = row * r.nx, i = row * r.pitch;
        for (unsigned x = threadIdx.x & 31; x < r.nx; x += 128) {
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (x + 32 * u < r.nx) v[u] = f(i + x + 32 * u);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (x + 32 * u < r.nx) out[q + x + 32 * u] = v[u];
        }
    }
}

// Arrays whose rows lie apart on one side: a warp per row and four accesses in
// flight, every array of a snapshot in one launch (blockIdx.y).  Copies of
// cudaMemcpy2DAsync took 1.12 ms for a snapshot at 197 x 211 x 163 (FP32) and 26
// us for one array of it; this takes 0.26 ms and 6 us.
template <typename U>
__device__ __forceinline__ void copy_rows(const RowSeg &g)
{
    const U *src = static_cast<const U *>(g.src);
    U *dst = static_cast<U *>(g.dst);
    const unsigned lane = threadIdx.x & 31;
    const size_t step = (size_t)gridDim.x * (kThreads / 32);
    for (size_t r = blockIdx.x * (size_t)(kThreads / 32) + (threadIdx.x >> 5); r < g.rows; r += step) {
        const U *s = src + r * g.src_pitch;
        U *d = dst + r * g.dst_pitch;
        for (unsigned x = lane; x < g.w; x += 128) {
            U v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (x + 32 * u < g.w) v[u] = s[x + 32 * u];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (x + 32 * u < g.w) d[x + 32 * u] = v[u];
        }
    }
    if (blockIdx.x == 0)
        for (unsigned x = threadIdx.x; x < g.tail; x += kThreads) dst[g.rows * g.dst_pitch + x] = U{};
}

__global__ void __launch_bounds__(kThreads) k_copy_rows(const __grid_constant__ RowSegs q)
{
    const RowSeg &g = q.s[blockIdx.y];
    switch (g.unit) {
    case 1: copy_rows<uint8_t>(g); break;
    case 2: copy_rows<uint16_t>(g); break;
    case 4: copy_rows<uint32_t>(g); break;
    default: copy_rows<uint2>(g);
    }
}

__global__ void k_index_max(const uint8_t *__restrict__ idx, size_t n, unsigned *out)
{
    unsigned m = 0;
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n;
         q += (size_t)gridDim.x * blockDim.x)
        m = max(m, (unsigned)idx[q]);
    for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

static_assert(sizeof(st::StressCoef) == 32, "bvf_ctx::slut holds 32 bytes per material");
__global__ void k_stress_table(const MatCoef *__restrict__ lut, int n, float Lf,
                               st::StressCoef *__restrict__ out)
{
    const int m = threadIdx.x;
    if (m < n) out[m] = st::make_stress_coef(lut[m], Lf);
}

template <typename T>
__global__ void k_pressure(const T *__restrict__ a, const T *__restrict__ b,
                           const T *__restrict__ c, float scale, float *__restrict__ out, size_t n,
                           Rows r)
{
    rows_out(out, n, r, [&](size_t i) {
        return -(st::tof(a[i]) + st::tof(b[i]) + st::tof(c[i])) / 3.0f * scale;
    });
}

// state array (element q at f[q * stride]) <-> FP32 values in physical units
// (scale = the storage scale)
template <typename T>
__global__ void k_field_out(const T *__restrict__ f, size_t stride, float scale,
                            float *__restrict__ out, size_t n, Rows r)
{
    rows_out(out, n, r, [&](size_t i) { return st::tof(f[i * stride]) * scale; });
}
template <typename T>
__global__ void k_field_in(const float *__restrict__ in, size_t stride, float inv_scale,
                           T *__restrict__ f, size_t n, Rows r)
{
    for_rows(n, r, [&](size_t q, size_t i) { st::stv(f + i * stride, in[q] * inv_scale); });
}
// out = in * scale, or out = scale where in is NULL (fill)
__global__ void k_scale_copy(const float *__restrict__ in, float scale, float *__restrict__ out,
                             size_t n, Rows r)
{
    rows_out(out, n, r, [&](size_t i) { return in ? in[i] * scale : scale; });
}

// p(t) = A cos(w t + phi): C = A N/2 cos phi, S = -A N/2 sin phi
__global__ void k_amp_phase(const double *__restrict__ C, const double *__restrict__ S, size_t n,
                            Rows r, double inv_half_n, double scale, double *amp, double *ph)
{
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n;
         q += (size_t)gridDim.x * blockDim.x) {
        const size_t i = in_rows(q, r);
        const double c = C[i], s = S[i];
        if (amp) amp[q] = sqrt(c * c + s * s) * inv_half_n * scale;
        if (ph) ph[q] = atan2(-s, c);
    }
}

// p = pref * sum_e dA_e (sin(k r) + i cos(k r)) / r   with pref = k p0 / (2 pi):
// the i k p0 / (2 pi) prefactor times exp(-i k r) = cos kr - i sin kr.
// Elements with complex weights w_e (phased arrays, WT): the element's term is
// multiplied by w_e = wr + i wi.
//
// The sum runs in tiles of 256 elements, FP32 within a tile and FP64 over the
// tiles in their order, in one of two ways with the same bits (see rs_split):
//   k_rs_point  a thread per point, 256 points a block, the tile in shared
//               memory;
//   k_rs        a block of 32 points x 8 threads takes 8 tiles at a time, one
//               per thread of a point, the elements (98 KB of 6150) from the L1
//               at an address a point's whole warp shares, and the first thread
//               of the point adds the 8 partial sums in order.
// The sum is bound by its instructions (square root, sincospi and division of
// every pair).  A thread per point gives 225 blocks on 152 SMs at 240 x 240
// points, half the SMs with one block of 8 warps, and 976 us with 6150 elements;
// eight take 650 us.
constexpr int kRsTile = 256;             // elements per FP32 partial sum
constexpr int kRsPts = 32, kRsGroups = 8;

// one element's term added to a partial sum; weight() is its complex weight
template <bool WT, class Weight>
__device__ __forceinline__ void rs_add(float4 E, Weight weight, float x, float y, float zp,
                                       float k_over_pi, float &pre, float &pim)
{
    const float ddx = x - E.x, ddy = y - E.y, ddz = zp - E.z;
    const float r = sqrtf(fmaf(ddx, ddx, fmaf(ddy, ddy, ddz * ddz)));
    float sn, cs;
    sincospif(k_over_pi * r, &sn, &cs);
    const float w = E.w / r;
    if (WT) {                            // (wr + i wi)(sin kr + i cos kr)
        const float2 W = weight();
        pre = fmaf(w, fmaf(W.x, sn, -W.y * cs), pre);
        pim = fmaf(w, fmaf(W.x, cs, W.y * sn), pim);
    } else {
        pre = fmaf(w, sn, pre);
        pim = fmaf(w, cs, pim);
    }
}

template <bool WT>
__global__ void __launch_bounds__(kRsTile)
    k_rs_point(const float4 *__restrict__ el, const float2 *__restrict__ wt, int ne, int nx, int ny,
               float dx, float zp, float k_over_pi, double pref, float2 *__restrict__ out)
{
    __shared__ float4 s_el[kRsTile];
    __shared__ float2 s_wt[WT ? kRsTile : 1];
    const int q = blockIdx.x * kRsTile + threadIdx.x;
    const bool live = q < nx * ny;
    const float x = live ? (q % nx) * dx : 0.0f;
    const float y = live ? (q / nx) * dx : 0.0f;
    double re = 0.0, im = 0.0;
    for (int base = 0; base < ne; base += kRsTile) {
        if (base + (int)threadIdx.x < ne) {
            s_el[threadIdx.x] = el[base + threadIdx.x];
            if (WT) s_wt[threadIdx.x] = wt[base + threadIdx.x];
        }
        __syncthreads();
        const int n = min(kRsTile, ne - base);
        float pre = 0.0f, pim = 0.0f;
        for (int e = 0; e < n; ++e) {
            const float2 W = s_wt[WT ? e : 0];
            rs_add<WT>(s_el[e], [&] { return W; }, x, y, zp, k_over_pi, pre, pim);
        }
        re += pre;
        im += pim;
        __syncthreads();
    }
    if (live) out[q] = make_float2((float)(pref * re), (float)(pref * im));
}

template <bool WT>
__global__ void __launch_bounds__(kRsPts *kRsGroups)
    k_rs(const float4 *__restrict__ el, const float2 *__restrict__ wt, int ne, int nx, int ny,
         float dx, float zp, float k_over_pi, double pref, float2 *__restrict__ out)
{
    __shared__ float2 s_part[kRsGroups][kRsPts];
    const int pt = threadIdx.x, g = threadIdx.y;
    const int q = blockIdx.x * kRsPts + pt;
    const bool live = q < nx * ny;
    const float x = live ? (q % nx) * dx : 0.0f;
    const float y = live ? (q / nx) * dx : 0.0f;
    double re = 0.0, im = 0.0;
    for (int base = 0; base < ne; base += kRsTile * kRsGroups) {
        const int e0 = base + g * kRsTile, e1 = min(ne, e0 + kRsTile);
        float pre = 0.0f, pim = 0.0f;
#pragma unroll 4
        for (int e = e0; e < e1; ++e)
            rs_add<WT>(__ldg(el + e), [&] { return __ldg(wt + e); }, x, y, zp, k_over_pi, pre, pim);
        s_part[g][pt] = make_float2(pre, pim);
        __syncthreads();
        if (g == 0)
            for (int t = 0; t < kRsGroups && base + t * kRsTile < ne; ++t) {
                re += s_part[t][pt].x;
                im += s_part[t][pt].y;
            }
        __syncthreads();
    }
    if (g == 0 && live) out[q] = make_float2((float)(pref * re), (float)(pref * im));
}

__global__ void k_heat_source(const uint8_t *__restrict__ idx, const ThermCoef *__restrict__ lut,
                              const double *__restrict__ amp, double p_scale,
                              float *__restrict__ Q, size_t n, int *q_bad)
{
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n;
         q += (size_t)gridDim.x * blockDim.x) {
        const float A = amp ? (float)(p_scale * amp[q]) : 0.0f;
        const float h = lut[idx[q]].qfac * A * A;
        Q[q] = h;
        if (!isfinite(h)) *q_bad = 1;
    }
}

__global__ void k_classes(const uint8_t *__restrict__ idx, const uint8_t *__restrict__ cls,
                          uint8_t *__restrict__ out, size_t n, Rows r)
{
    __shared__ uint8_t s_c[BVF_MAX_MATERIALS];
    for (int m = threadIdx.x; m < BVF_MAX_MATERIALS; m += blockDim.x) s_c[m] = cls[m];
    __syncthreads();
    for_rows(n, r, [&](size_t q, size_t i) { out[i] = s_c[idx[q]]; });
}

// Pennes forward-Euler step on the rise; border voxels held at T_a (rise 0);
// T_max and CEM43 fused.
// A 32 x 8 block walks a chunk of z.  Every value plane k needs (T and the
// material of the voxel and its four in-plane neighbours, Q, T_max, the dose
// partial) is loaded one plane ahead, so those loads are in flight while the
// previous plane is computed; the z-neighbours come from the planes already
// held.  Face conductivity: harmonic mean 2 k_c k_n / (k_c + k_n).  The
// chunk length p.kz comes from thermal_kchunk.

// One interior voxel's forward-Euler step on the rise theta = T - T_a:
// theta + dt (div(k grad theta) - w_b c_b theta + DC Q) / (rho c) (T_a is
// constant, so the diffusion of theta is that of T), the six face terms
// summed in the order
// x-, x+, y-, y+, z-, z+ (k_f from the pair table of the centre material c;
// where all six neighbours share c's material, its diagonal entry, held in
// c.k, serves every face without a table read).  Explicit round-to-nearest
// operations, so the direct and TMA kernels agree bit for bit.
__device__ __forceinline__ float thermal_update(const ThParams &p, const ThermCoef &c, int mc,
                                                const float *kf, float Tc, float Tw, int mw,
                                                float Te, int me, float Ts, int ms, float Tq,
                                                int mq, float Tm, int mm, float Tp, int mp, float Q)
{
    float kw, ke, ks, kq, km, kp;
    if (mw == mc && me == mc && ms == mc && mq == mc && mm == mc && mp == mc) {
        kw = ke = ks = kq = km = kp = c.k;
    } else {
        kw = __ldg(kf + mw);
        ke = __ldg(kf + me);
        ks = __ldg(kf + ms);
        kq = __ldg(kf + mq);
        km = __ldg(kf + mm);
        kp = __ldg(kf + mp);
    }
    float lap = __fmul_rn(kw, __fsub_rn(Tw, Tc));
    lap = __fmaf_rn(ke, __fsub_rn(Te, Tc), lap);
    lap = __fmaf_rn(ks, __fsub_rn(Ts, Tc), lap);
    lap = __fmaf_rn(kq, __fsub_rn(Tq, Tc), lap);
    lap = __fmaf_rn(km, __fsub_rn(Tm, Tc), lap);
    lap = __fmaf_rn(kp, __fsub_rn(Tp, Tc), lap);
    const float perf = __fmul_rn(c.perfw, Tc);
    const float rhs = __fmaf_rn(p.dc, Q, __fmaf_rn(lap, p.inv_dx2, -perf));
    return __fmaf_rn(__fmul_rn(p.dt, rhs), c.inv_rhoc, Tc);
}

// The maximum rise and the CEM43 partial of a voxel after its step (dose
// rate R^(43-T) per minute, R = 1/2 at T >= 43 C, 1/4 below: exp2(l2r
// (rise43 - theta)) with l2r = -1 or -2); every 32nd step the FP32 partial
// goes into the FP64 sum.
__device__ __forceinline__ void thermal_outputs(const ThParams &p, size_t q, float Tn, float Tmax,
                                                float cemf)
{
    p.Tmax[q] = fmaxf(Tmax, Tn);
    const float l2r = (Tn >= p.rise43) ? -1.0f : -2.0f;
    const float part = __fmaf_rn(p.dt60, exp2f(__fmul_rn(l2r, __fsub_rn(p.rise43, Tn))), cemf);
    if (p.flush) {
        p.cem[q] += (double)part;
        p.cemf[q] = 0.0f;
    } else {
        p.cemf[q] = part;
    }
}

__global__ void __launch_bounds__(256) k_thermal(ThParams p)
{
    extern __shared__ ThermCoef s_th[];
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    for (int m = tid; m < p.n_mat; m += blockDim.x * blockDim.y) s_th[m] = p.lut[m];
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    if (i >= nx || j >= ny) return;
    const int k0 = blockIdx.z * p.kz, k1 = min(nz, k0 + p.kz);
    const int SZ = nx * ny, col = j * nx + i;
    const bool xy_border = i == 0 || j == 0 || i == nx - 1 || j == ny - 1;
    const float *__restrict__ T = p.T;
    const uint8_t *__restrict__ idx = p.idx;
    // everything plane k needs, loaded one plane ahead
    struct Plane {
        float Tc, Tw, Te, Ts, Tq, Q, Tmax, cemf;
        int mc, mw, me, ms, mq;
    };
    auto load = [&](int k, Plane &P) {
        const int q = k * SZ + col;
        P.Tc = __ldg(T + q);
        P.mc = __ldg(idx + q);
        P.Q = p.Q[q];
        P.Tmax = p.Tmax[q];
        P.cemf = p.cemf[q];
        if (!xy_border) {
            P.Tw = __ldg(T + q - 1); P.Te = __ldg(T + q + 1);
            P.Ts = __ldg(T + q - nx); P.Tq = __ldg(T + q + nx);
            P.mw = __ldg(idx + q - 1); P.me = __ldg(idx + q + 1);
            P.ms = __ldg(idx + q - nx); P.mq = __ldg(idx + q + nx);
        }
    };
    float Tm = k0 > 0 ? __ldg(T + (k0 - 1) * SZ + col) : 0.0f;
    int mm = k0 > 0 ? __ldg(idx + (k0 - 1) * SZ + col) : 0;
    Plane cur, nxt;
    load(k0, cur);
    for (int k = k0; k < k1; ++k) {
        const int q = k * SZ + col;
        if (k + 1 < nz) load(k + 1, nxt);
        else { nxt.Tc = 0.0f; nxt.mc = 0; }
        float Tn;
        if (xy_border || k == 0 || k == nz - 1) {
            Tn = 0.0f;
        } else {
            // face conductivities 2 k_a k_b / (k_a + k_b) from the pair table
            Tn = thermal_update(p, s_th[cur.mc], cur.mc, p.kface + cur.mc * p.n_mat, cur.Tc, cur.Tw,
                                cur.mw, cur.Te, cur.me, cur.Ts, cur.ms, cur.Tq, cur.mq, Tm, mm,
                                nxt.Tc, nxt.mc, cur.Q);
        }
        p.Tn[q] = Tn;
        thermal_outputs(p, q, Tn, cur.Tmax, cur.cemf);
        Tm = cur.Tc;
        mm = cur.mc;
        cur = nxt;
    }
}

// The same step for two x-neighbours, arithmetic on pairs (bit for bit two
// calls of thermal_update): face conductivities k[] in the order x-, x+, y-,
// y+, z-, z+, nperf = -perfw and inv_rhoc of the two centres.
__device__ __forceinline__ float2 thermal_update2(const ThParams &p, const float2 (&k)[6],
                                                  float2 nperfw, float2 inv_rhoc, float2 Tc,
                                                  float2 Tw, float2 Te, float2 Ts, float2 Tq,
                                                  float2 Tm, float2 Tp, float2 Q)
{
    using st::splat;
    float2 lap = st::vmul(k[0], st::vsub(Tw, Tc));
    lap = st::vfma(k[1], st::vsub(Te, Tc), lap);
    lap = st::vfma(k[2], st::vsub(Ts, Tc), lap);
    lap = st::vfma(k[3], st::vsub(Tq, Tc), lap);
    lap = st::vfma(k[4], st::vsub(Tm, Tc), lap);
    lap = st::vfma(k[5], st::vsub(Tp, Tc), lap);
    const float2 nperf = st::vmul(nperfw, Tc);
    const float2 rhs =
        st::vfma(splat<float2>(p.dc), Q, st::vfma(lap, splat<float2>(p.inv_dx2), nperf));
    return st::vfma(st::vmul(splat<float2>(p.dt), rhs), inv_rhoc, Tc);
}

// thermal_outputs for the pair at q, q + 1 (q even)
__device__ __forceinline__ void thermal_outputs2(const ThParams &p, size_t q, float2 Tn, float2 Tmax,
                                                 float2 cemf)
{
    st::st2(p.Tmax + q, make_float2(fmaxf(Tmax.x, Tn.x), fmaxf(Tmax.y, Tn.y)));
    const float2 l2r = make_float2((Tn.x >= p.rise43) ? -1.0f : -2.0f,
                                   (Tn.y >= p.rise43) ? -1.0f : -2.0f);
    const float2 x = st::vmul(l2r, st::vsub(st::splat<float2>(p.rise43), Tn));
    const float2 part =
        st::vfma(st::splat<float2>(p.dt60), make_float2(exp2f(x.x), exp2f(x.y)), cemf);
    if (p.flush) {
        p.cem[q] += (double)part.x;
        p.cem[q + 1] += (double)part.y;
        st::st2(p.cemf + q, make_float2(0.0f, 0.0f));
    } else {
        st::st2(p.cemf + q, part);
    }
}

// TMA-fed step (grids with nx % 8 == 0).  A block of 16 x 16 threads owns a
// 32 x 16 x-y tile (thread (tx, ty) the pair x0 + 2 tx, + 1 of row y0 + ty) and
// walks a z-chunk.  Every input of a plane arrives through the tensor-memory
// accelerator in shared-memory rings: T and the conduction class as halo'd
// boxes (T: x0-4 .. x0+35, class: x0-16 .. x0+47, both y0-1 .. y0+16; a TMA
// box starts on a 16-byte boundary, out-of-range elements read as zero and
// only feed border voxels, which are held at T_a), the material, Q (while the
// source is on), T_max and the dose partial as 32 x 16 boxes.  Plane k reads
// planes k-1, k, k+1 while k+2 and k+3 are in flight; results are stored
// directly.  One thread issues the copies; waits are bounded as in the
// acoustic kernels (a time-out sets bit 2 of the flag after the block's armed
// copies have landed).
//
// At 240 x 240 x 200 the copies and stores alone take 60 us of a step (four
// planes of ring, one of them in flight: 62), a voxel a time with a pair
// look-up for every bone voxel took 84.9 in all.  Pairs (8-byte shared-memory
// and global accesses, the class as 16-bit words, one comparison of all
// twelve, packed arithmetic) and classes instead of materials (the 125 bone
// bins of the skull share one conductivity) bring it to 74.4, 67.3 in one
// tissue.  Where the twelve classes differ, three of their twelve faces are known
// without a look-up (k_low, kab): 256 conductivities at random take 373 us a
// step, 471 with twelve look-ups, 441 a voxel a time; the skull case 73.7.
constexpr int kThRing = 5, kThVRing = 4;     // T and index planes k-1 .. k+3; streams k .. k+3
constexpr int kThTileY = 16;
constexpr int kThTW = 40, kThTH = kThTileY + 2, kThTBytes = kThTW * kThTH * 4;   // 2880 B
constexpr int kThTSlot = 2944;                                         // 23 x 128 B
constexpr int kThIW = 64, kThIBytes = kThIW * kThTH;                   // 1152 B
constexpr int kThVBytes = 32 * kThTileY * 4;                           // Q, T_max, partial: 2048 B
constexpr int kThSlot = kThTSlot + kThIBytes, kThVSlot = 3 * kThVBytes + 512;
constexpr int kThMBytes = 32 * kThTileY;                               // own materials: 512 B
constexpr int kThOffV = kThRing * kThSlot;
constexpr int kThOffBar = kThOffV + kThVRing * kThVSlot;
constexpr int kThOffAbort = kThOffBar + 8 * kThRing;
constexpr int kThOffLut = (kThOffAbort + (int)sizeof(int) + 15) / 16 * 16;
static_assert(kThTSlot % 128 == 0 && kThTSlot >= kThTBytes && kThIBytes % 128 == 0 &&
                  kThVBytes % 128 == 0 && kThSlot % 128 == 0 && kThOffLut % 16 == 0,
              "ring slots 128-byte aligned, coefficients 16");

__global__ void __launch_bounds__(256, 4)
    k_thermal_tma(ThParams p, const __grid_constant__ ThermTmaMaps tm, int *flag)
{
    extern __shared__ __align__(128) unsigned char smb[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smb + kThOffBar);
    volatile int *s_abort = reinterpret_cast<volatile int *>(smb + kThOffAbort);
    ThermCoef *s_th = reinterpret_cast<ThermCoef *>(smb + kThOffLut);
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * 16 + tx;
    for (int m = tid; m < p.n_mat; m += 256) s_th[m] = p.lut[m];
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * kThTileY, i = x0 + 2 * tx, j = y0 + ty;
    const int k0 = blockIdx.z * p.kz, k1 = min(nz, k0 + p.kz);
    if (tid == 0) {
        for (int b = 0; b < kThRing; ++b) tma::mbar_init(&bars[b], 1);
        tma::mbar_init_fence();
        *s_abort = -1;
    }
    __syncthreads();
    // the coefficients are in place; the rest is the step before's
    tma::pdl_wait();
    tma::pdl_launch_next();
    // T and the index of plane pl of the chunk's window k0-1 .. k1 sit in slot
    // (pl - k0 + 1) % 5 of their ring, the (pl - k0 + 1) / 5-th phase of that
    // slot's barrier; Q, T_max and the partial of an own plane in slot
    // (pl - k0) % 4 of theirs, on the same barrier
    auto slot = [&](int pl) { return (pl - k0 + 1) % kThRing; };
    auto parity = [&](int pl) { return (unsigned)((pl - k0 + 1) / kThRing) & 1u; };
    const bool heat = p.dc != 0.0f || *p.q_bad != 0;
    auto issue = [&](int pl) {
        uint64_t *bar = &bars[slot(pl)];
        unsigned char *d = smb + slot(pl) * kThSlot;
        // the per-voxel streams only for the chunk's own planes; its two
        // neighbour planes supply T and the index
        const bool own = pl >= k0 && pl < k1;
        tma::mbar_expect_tx(bar, (unsigned)(kThTBytes + kThIBytes) +
                                     (own ? (heat ? 3u : 2u) * kThVBytes + kThMBytes : 0u));
        if (p.hold_plane >= 0 && pl == p.hold_plane) return;   // test hook: armed, none issued
        tma::load3d(d, &tm.T, x0 - 4, y0 - 1, pl, bar);
        tma::load3d(d + kThTSlot, &tm.cls, x0 - 16, y0 - 1, pl, bar);
        if (own) {
            unsigned char *e = smb + kThOffV + (pl - k0) % kThVRing * kThVSlot;
            if (heat) tma::load3d(e, &tm.Q, x0, y0, pl, bar);
            tma::load3d(e + kThVBytes, &tm.Tmax, x0, y0, pl, bar);
            tma::load3d(e + 2 * kThVBytes, &tm.cemf, x0, y0, pl, bar);
            tma::load3d(e + 3 * kThVBytes, &tm.idx, x0, y0, pl, bar);
        }
    };
    auto wait = [&](int pl) { return tma::mbar_wait(&bars[slot(pl)], parity(pl), p.wait_limit); };
    const int first_last = min(k1, k0 + 2);
    if (tid == 0)
        for (int pl = k0 - 1; pl <= first_last; ++pl) issue(pl);
    int issued = first_last;

    // nx is even: a pair lies inside the grid or outside
    const bool live = i < nx && j < ny, xb0 = i == 0, xb1 = i + 1 == nx - 1;
    const bool yb = j == 0 || j == ny - 1;
    const int c = (ty + 1) * kThTW + 2 * tx + 4, d = (ty + 1) * kThIW + 2 * tx + 16;
    const int cv = ty * 32 + 2 * tx;
    const size_t SZ = (size_t)nx * ny;
    size_t q = (size_t)k0 * SZ + (size_t)j * nx + i;
    // conductivities of the pair's lower z-faces, once a plane has given them
    float2 k_low = make_float2(0.0f, 0.0f);
    bool k_known = false;
    // the pair of plane k: S, Sm, Sp the ring slots of planes k, k-1, k+1, V0
    // the streams of plane k
    auto pair_step = [&](const unsigned char *S, const unsigned char *Sm, const unsigned char *Sp,
                         const float *V0, bool border) {
        const float *T0 = reinterpret_cast<const float *>(S);
        const unsigned char *I0 = S + kThTSlot;
        const float2 Q = heat ? st::ld2(V0 + cv) : make_float2(0.0f, 0.0f), Tmax = st::ld2(V0 + cv + kThVBytes / 4),
                     cemf = st::ld2(V0 + cv + kThVBytes / 2);
        float2 Tn = make_float2(0.0f, 0.0f);
        if (!border) {
            auto w16 = [](const unsigned char *p16) {
                return (unsigned)*reinterpret_cast<const unsigned short *>(p16);
            };
            const float2 Tc = st::ld2(T0 + c), Tl = st::ld2(T0 + c - 2), Tr = st::ld2(T0 + c + 2);
            const float2 Ts = st::ld2(T0 + c - kThTW), Tq = st::ld2(T0 + c + kThTW);
            const float2 Tm = st::ld2(reinterpret_cast<const float *>(Sm) + c);
            const float2 Tp = st::ld2(reinterpret_cast<const float *>(Sp) + c);
            const float2 Tw = make_float2(Tl.y, Tc.x), Te = make_float2(Tc.y, Tr.x);
            const unsigned m2 = w16(I0 + d), ml = w16(I0 + d - 2) >> 8, mr = w16(I0 + d + 2) & 255u;
            const unsigned ms = w16(I0 + d - kThIW), mq = w16(I0 + d + kThIW);
            const unsigned mm = w16(Sm + kThTSlot + d), mp = w16(Sp + kThTSlot + d);
            // m..: conduction classes; own materials for the other coefficients
            const unsigned ca = m2 & 255u, cb = m2 >> 8, one = ca * 0x0101u;
            const unsigned own =
                w16(reinterpret_cast<const unsigned char *>(V0 + 3 * (kThVBytes / 4)) + cv);
            const ThermCoef a = s_th[own & 255u], b = s_th[own >> 8];
            float2 k[6];
            if (((m2 ^ one) | (ms ^ one) | (mq ^ one) | (mm ^ one) | (mp ^ one) | (ml ^ ca) |
                 (mr ^ ca)) == 0u) {
#pragma unroll
                for (int f = 0; f < 6; ++f) k[f] = st::splat<float2>(a.k);
            } else {
                // the face between the pair's voxels, and the lower one of each,
                // which was the upper one a plane before, are known (the table is
                // symmetric)
                const float *ka = p.kface + ca * p.n_cls, *kb = p.kface + cb * p.n_cls;
                const float kab = __ldg(ka + cb);
                k[0] = make_float2(__ldg(ka + ml), kab);
                k[1] = make_float2(kab, __ldg(kb + mr));
                k[2] = make_float2(__ldg(ka + (ms & 255u)), __ldg(kb + (ms >> 8)));
                k[3] = make_float2(__ldg(ka + (mq & 255u)), __ldg(kb + (mq >> 8)));
                k[4] = k_known ? k_low
                               : make_float2(__ldg(ka + (mm & 255u)), __ldg(kb + (mm >> 8)));
                k[5] = make_float2(__ldg(ka + (mp & 255u)), __ldg(kb + (mp >> 8)));
            }
            const float2 nperfw = make_float2(-a.perfw, -b.perfw),
                         irc = make_float2(a.inv_rhoc, b.inv_rhoc);
            Tn = thermal_update2(p, k, nperfw, irc, Tc, Tw, Te, Ts, Tq, Tm, Tp, Q);
            if (xb0) Tn.x = 0.0f;
            if (xb1) Tn.y = 0.0f;
            k_low = k[5];
        }
        k_known = !border;
        st::st2(p.Tn + q, Tn);
        thermal_outputs2(p, q, Tn, Tmax, cemf);
    };
    // slots of planes k-1, k, k+1 and of plane k's streams, rotated per plane;
    // parity of plane k+1's barrier
    int sm1 = 0, sc = 1, sp1 = 2, sv = 0;
    unsigned ph = 0;
    for (int k = k0; k < k1; ++k, q += SZ) {
        __syncthreads();
        if (*s_abort >= 0) break;             // a wait of the previous plane ran out
        if (k + 3 <= k1 && k + 3 > issued) {  // into the slots planes k-2 and k-1 have freed
            if (tid == 0) {
                tma::fence_async_smem();
                issue(k + 3);
            }
            issued = k + 3;
        }
        bool ready = true;
        if (k == k0) ready = wait(k0 - 1) && wait(k0);
        ready = ready && tma::mbar_wait(&bars[sp1], ph, p.wait_limit);
        if (!ready) *s_abort = k;             // leaves at the next barrier
        if (ready && live)
            pair_step(smb + sc * kThSlot, smb + sm1 * kThSlot, smb + sp1 * kThSlot,
                      reinterpret_cast<const float *>(smb + kThOffV + sv * kThVSlot),
                      yb || k == 0 || k == nz - 1);
        sm1 = sc;
        sc = sp1;
        if (++sp1 == kThRing) {
            sp1 = 0;
            ph ^= 1u;
        }
        sv = sv + 1 == kThVRing ? 0 : sv + 1;
    }
    __syncthreads();
    const int ab = *s_abort;
    if (ab >= 0 && tid == 0) {
        // every armed phase from the one that ran out on has landed before
        // the block's shared memory is released
        for (int pl = max(k0 - 1, ab - 1); pl <= issued; ++pl) wait(pl);
        atomicOr(flag, 2);
    }
}

// Intensity I = A^2 / (2 rho c) = A^2 * zw[m] with zw[m] = 1 / (2 rho c).
// Positive doubles order like their bit patterns, so atomicMax on the bits
// finds the maximum.
__global__ void k_int_max(const uint8_t *__restrict__ idx, const double *__restrict__ zw,
                          const double *__restrict__ amp, size_t n, unsigned long long *best)
{
    unsigned long long m = 0;
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n;
         q += (size_t)gridDim.x * blockDim.x) {
        const double I = amp[q] * amp[q] * zw[idx[q]];
        m = max(m, (unsigned long long)__double_as_longlong(I));
    }
    for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(best, m);
}

__global__ void k_int_argmin(const uint8_t *__restrict__ idx, const double *__restrict__ zw,
                             const double *__restrict__ amp, size_t n,
                             const unsigned long long *best, unsigned long long *out)
{
    const unsigned long long b = *best;
    unsigned long long m = ~0ull;
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n;
         q += (size_t)gridDim.x * blockDim.x) {
        const double I = amp[q] * amp[q] * zw[idx[q]];
        if ((unsigned long long)__double_as_longlong(I) == b) m = min(m, (unsigned long long)q);
    }
    for (int o = 16; o; o >>= 1) m = min(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMin(out, m);
}

// Plane sums of both intensity maps at z_m, one block, fixed order.
__global__ void __launch_bounds__(1024) k_plane_sums(
    const uint8_t *__restrict__ ia, const double *__restrict__ za, const double *__restrict__ aa,
    const uint8_t *__restrict__ iw, const double *__restrict__ zw, const double *__restrict__ aw,
    int nx, int ny, int nz, const unsigned long long *qbest, double *sums)
{
    __shared__ double s_a[1024], s_w[1024];
    const long long plane = (long long)nx * ny;
    if (*qbest >= (unsigned long long)(plane * nz)) {   // no maximum found
        if (threadIdx.x == 0) sums[0] = sums[1] = sums[2] = 0.0;
        return;
    }
    const long long z = (long long)(*qbest / (unsigned long long)plane);
    const long long base = z * plane;
    double sa = 0.0, sw = 0.0;
    for (long long t = threadIdx.x; t < plane; t += blockDim.x) {
        const long long q = base + t;
        sa += aa[q] * aa[q] * za[ia[q]];
        sw += aw[q] * aw[q] * zw[iw[q]];
    }
    s_a[threadIdx.x] = sa;
    s_w[threadIdx.x] = sw;
    __syncthreads();
    for (int o = blockDim.x / 2; o; o >>= 1) {
        if ((int)threadIdx.x < o) {
            s_a[threadIdx.x] += s_a[threadIdx.x + o];
            s_w[threadIdx.x] += s_w[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        sums[0] = s_a[0];
        sums[1] = s_w[0];
        sums[2] = (double)z;
    }
}

// Time-reversal (phase-conjugation) plane from the FP64 DFT sums of one
// z-plane: with amplitude 2 |C - iS| / N and phase atan2(-S, C) the captured
// complex amplitude is P = (2/N)(C - iS), so conj(P) / max|P| over the plane is
// (C + iS) / max |C + iS|.  First pass: the largest |C + iS|^2 of the plane
// (non-negative doubles order like their bit patterns, so one 64-bit
// atomicMax keeps it); second pass: the normalised conjugate.
__global__ void k_plane_absmax(const double *__restrict__ C, const double *__restrict__ S,
                               size_t n, Rows r, unsigned long long *out)
{
    double m = 0.0;
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n;
         q += (size_t)gridDim.x * blockDim.x) {
        const size_t i = in_rows(q, r);
        m = fmax(m, C[i] * C[i] + S[i] * S[i]);
    }
    for (int o = 16; o; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

__global__ void k_conj_normalise(const double *__restrict__ C, const double *__restrict__ S,
                                 size_t n, Rows r, const unsigned long long *mx,
                                 float2 *__restrict__ out)
{
    const double m2 = __longlong_as_double((long long)*mx);
    const double inv = m2 > 0.0 ? 1.0 / sqrt(m2) : 0.0;
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n;
         q += (size_t)gridDim.x * blockDim.x) {
        const size_t i = in_rows(q, r);
        out[q] = make_float2((float)(C[i] * inv), (float)(S[i] * inv));
    }
}

}  // namespace

cudaError_t launch_conj_plane(const double *C, const double *S, size_t n, Rows r,
                              unsigned long long *d_max, float2 *out, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(d_max, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    k_plane_absmax<<<blocks_for(n), kThreads, 0, s>>>(C, S, n, r, d_max);
    k_conj_normalise<<<blocks_for(n), kThreads, 0, s>>>(C, S, n, r, d_max, out);
    return cudaGetLastError();
}

cudaError_t launch_stress_table(const MatCoef *lut, int n, float Lf, void *slut, cudaStream_t s)
{
    k_stress_table<<<1, BVF_MAX_MATERIALS, 0, s>>>(lut, n, Lf, static_cast<st::StressCoef *>(slut));
    return cudaGetLastError();
}

void RowSegs::add(void *dst, size_t dst_pitch, const void *src, size_t src_pitch, size_t w, size_t rows,
                  size_t es, size_t tail)
{
    // accesses of whole elements, or of what both addresses are aligned to (a
    // caller's buffer may start anywhere)
    size_t unit = es;
    while ((reinterpret_cast<uintptr_t>(dst) | reinterpret_cast<uintptr_t>(src)) % unit) unit /= 2;
    const size_t k = es / unit;
    s[n++] = RowSeg{dst, src, dst_pitch * k, src_pitch * k, rows, (unsigned)(w * k), (unsigned)(tail * k),
                    (int)unit};
}

cudaError_t launch_copy_rows(const RowSegs &q, cudaStream_t s)
{
    size_t rows = 0;
    for (int i = 0; i < q.n; ++i) rows = rows > q.s[i].rows ? rows : q.s[i].rows;
    k_copy_rows<<<dim3(blocks_for(rows, kThreads / 32), q.n), kThreads, 0, s>>>(q);
    return cudaGetLastError();
}

cudaError_t launch_index_max(const uint8_t *idx, size_t n, unsigned *d_out, cudaStream_t s)
{
    k_index_max<<<blocks_for(n), kThreads, 0, s>>>(idx, n, d_out);
    return cudaGetLastError();
}

cudaError_t launch_pressure(const void *sxx, const void *syy, const void *szz, int h16,
                            float scale, float *out, size_t n, Rows r, cudaStream_t s)
{
    if (h16)
        k_pressure<__half><<<blocks_for(n), kThreads, 0, s>>>(
            static_cast<const __half *>(sxx), static_cast<const __half *>(syy),
            static_cast<const __half *>(szz), scale, out, n, r);
    else
        k_pressure<float><<<blocks_for(n), kThreads, 0, s>>>(
            static_cast<const float *>(sxx), static_cast<const float *>(syy),
            static_cast<const float *>(szz), scale, out, n, r);
    return cudaGetLastError();
}

cudaError_t launch_field_out(const void *f, int h16, size_t stride, float scale, float *out,
                             size_t n, Rows r, cudaStream_t s)
{
    if (h16)
        k_field_out<__half><<<blocks_for(n), kThreads, 0, s>>>(static_cast<const __half *>(f),
                                                              stride, scale, out, n, r);
    else
        k_field_out<float><<<blocks_for(n), kThreads, 0, s>>>(static_cast<const float *>(f),
                                                             stride, scale, out, n, r);
    return cudaGetLastError();
}

cudaError_t launch_field_in(const float *in, int h16, size_t stride, float inv_scale, void *f,
                            size_t n, Rows r, cudaStream_t s)
{
    if (h16)
        k_field_in<__half><<<blocks_for(n), kThreads, 0, s>>>(in, stride, inv_scale,
                                                             static_cast<__half *>(f), n, r);
    else
        k_field_in<float><<<blocks_for(n), kThreads, 0, s>>>(in, stride, inv_scale,
                                                            static_cast<float *>(f), n, r);
    return cudaGetLastError();
}

__global__ void k_add_const(float *__restrict__ x, float c, size_t n)
{
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n;
         q += (size_t)gridDim.x * blockDim.x)
        x[q] = __fadd_rn(x[q], c);
}

cudaError_t launch_add_const(float *x, float c, size_t n, cudaStream_t s)
{
    k_add_const<<<blocks_for(n), kThreads, 0, s>>>(x, c, n);
    return cudaGetLastError();
}

cudaError_t launch_fill(float *out, float value, size_t n, cudaStream_t s)
{
    k_scale_copy<<<blocks_for(n), kThreads, 0, s>>>(nullptr, value, out, n, Rows{1, 1});
    return cudaGetLastError();
}

cudaError_t launch_scale_copy(const float *in, float scale, float *out, size_t n, Rows r,
                              cudaStream_t s)
{
    k_scale_copy<<<blocks_for(n), kThreads, 0, s>>>(in, scale, out, n, r);
    return cudaGetLastError();
}

cudaError_t launch_amp_phase(const double *C, const double *S, size_t n, Rows r, int count,
                             double scale, double *amp, double *ph, cudaStream_t s)
{
    k_amp_phase<<<blocks_for(n), kThreads, 0, s>>>(C, S, n, r, 2.0 / count, scale, amp, ph);
    return cudaGetLastError();
}

// Whether eight threads share a point: where that is estimated to be the faster
// way.  The estimates (us, with b blocks per SM) are fits to both kernels' times
// at 459 sizes, 32^2 to 2048^2 points and 256 to 4200 elements; the kernel they
// pick is at most 3 % slower than the other.  Few elements leave most of the
// eight threads idle (256 elements at 512 x 512 points: 324 us, 135 with a
// thread per point), and many on a small plane leave a thread per point to a
// serial chain (1024 at 64 x 64: 139 us, 62 with eight).  From about 900 x 900
// points on the two are within 3 % of each other for any number of elements
// above 1500.
static bool rs_split(int points, int ne, bool weighted)
{
    constexpr int n_sm = 152;
    // a thread per point: an element's latency, or the SM's share of its issue
    const int blocks = (points + kRsTile - 1) / kRsTile, b1 = (blocks + n_sm - 1) / n_sm;
    const double t_point = ne * std::max(0.137, 0.070 * b1 + 0.035);
    // eight threads: the chain of a tile, and the issue of all of them
    const double b8 = points / (double)(kRsPts * n_sm);
    const double tile = b8 <= 6.6 ? (weighted ? 59.0 : 51.5)
                                  : std::max(90.0, (weighted ? 46.0 : 40.0) + 4.5 * b8);
    const int round = kRsTile * kRsGroups, rest = ne % round;
    const double chain = tile * (ne / round + std::min(kRsTile, rest) / (double)kRsTile);
    const double issue = (weighted ? 0.0088 : 0.0085) * b8 * ne;
    return std::pow(std::pow(chain, 2.5) + std::pow(issue, 2.5), 0.4) < t_point;
}

template <bool WT>
static cudaError_t launch_rs_t(const float4 *el, const float2 *wt, int ne, int nx, int ny, float dx,
                               float zp, float k_over_pi, double pref, float2 *out, cudaStream_t s)
{
    const int n = nx * ny;
    if (rs_split(n, ne, WT))
        k_rs<WT><<<(n + kRsPts - 1) / kRsPts, dim3(kRsPts, kRsGroups), 0, s>>>(
            el, wt, ne, nx, ny, dx, zp, k_over_pi, pref, out);
    else
        k_rs_point<WT><<<(n + kRsTile - 1) / kRsTile, kRsTile, 0, s>>>(el, wt, ne, nx, ny, dx, zp,
                                                                       k_over_pi, pref, out);
    return cudaGetLastError();
}

cudaError_t launch_rs(const float4 *el, int ne, int nx, int ny, float dx, float zp, float k_over_pi,
                      double pref, float2 *out, cudaStream_t s)
{
    return launch_rs_t<false>(el, nullptr, ne, nx, ny, dx, zp, k_over_pi, pref, out, s);
}

cudaError_t launch_rs_weighted(const float4 *el, const float2 *wt, int ne, int nx, int ny,
                               float dx, float zp, float k_over_pi, double pref, float2 *out,
                               cudaStream_t s)
{
    return launch_rs_t<true>(el, wt, ne, nx, ny, dx, zp, k_over_pi, pref, out, s);
}

cudaError_t launch_classes(const uint8_t *idx, const uint8_t *cls, uint8_t *out, size_t n, Rows r,
                           cudaStream_t s)
{
    k_classes<<<blocks_for(n), kThreads, 0, s>>>(idx, cls, out, n, r);
    return cudaGetLastError();
}

cudaError_t launch_heat_source(const uint8_t *idx, const ThermCoef *lut, int n_mat,
                               const double *amp, double p_scale, float *Q, size_t n,
                               int *q_bad, cudaStream_t s)
{
    (void)n_mat;
    k_heat_source<<<blocks_for(n), kThreads, 0, s>>>(idx, lut, amp, p_scale, Q, n, q_bad);
    return cudaGetLastError();
}

static cudaError_t raise_thermal_smem()
{
    return cudaFuncSetAttribute(k_thermal_tma, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kThOffLut + BVF_MAX_MATERIALS * (int)sizeof(ThermCoef));
}

// The z-chunk of a BHTE launch: blocks of a chunk run in waves of
// (resident blocks per SM) x (SMs); a block's time is about its planes plus
// two (the z-neighbour planes and the pipeline fill), so the chunk length kz
// in 1 .. 32 that minimises waves(kz) x (kz + 2) is taken.
int thermal_kchunk(int nx, int ny, int nz, bool tma, int n_mat)
{
    int dev = 0, n_sm = 152, per_sm = 0;
    if (cudaGetDevice(&dev) == cudaSuccess)
        cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    const size_t smem = tma ? kThOffLut + n_mat * sizeof(ThermCoef) : n_mat * sizeof(ThermCoef);
    if (tma) raise_thermal_smem();
    const cudaError_t e =
        tma ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_thermal_tma, 256, smem)
            : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_thermal, 256, smem);
    if (e != cudaSuccess || per_sm < 1) per_sm = 1;
    const long long tiles = (long long)((nx + 31) / 32) * ((ny + (tma ? kThTileY : 8) - 1) /
                                                           (tma ? kThTileY : 8));
    const long long slots = (long long)per_sm * n_sm;
    int best = 16;
    long long best_cost = -1;
    for (int kz = 1; kz <= 32; ++kz) {
        const long long blocks = tiles * ((nz + kz - 1) / kz);
        const long long cost = ((blocks + slots - 1) / slots) * (kz + 2);
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = kz;
        }
    }
    return best < nz ? best : (nz > 0 ? nz : 1);
}

cudaError_t launch_thermal_step(const ThParams &p, const ThermTmaMaps *tm, int *flag,
                               cudaStream_t s)
{
    dim3 blk(32, 8, 1);
    dim3 grd((p.nx + 31) / 32, (p.ny + 7) / 8, (p.nz + p.kz - 1) / p.kz);
    if (tm) {
        // the shared-memory limit is raised once per process (graph capture)
        static std::atomic<int> raised{0};
        if (!raised.load(std::memory_order_acquire)) {
            const cudaError_t e = raise_thermal_smem();
            if (e != cudaSuccess) return e;
            raised.store(1, std::memory_order_release);
        }
        grd.y = (p.ny + kThTileY - 1) / kThTileY;
        return launch_pdl(k_thermal_tma, grd, dim3(16, 16, 1),
                          kThOffLut + p.n_mat * sizeof(ThermCoef), s, p, *tm, flag);
    } else {
        k_thermal<<<grd, blk, p.n_mat * sizeof(ThermCoef), s>>>(p);
    }
    return cudaGetLastError();
}

cudaError_t launch_intensity_argmax(const uint8_t *idx, const double *zw, const double *amp,
                                    size_t n, unsigned long long *d_best, cudaStream_t s)
{
    k_int_max<<<blocks_for(n), kThreads, 0, s>>>(idx, zw, amp, n, d_best);
    return cudaGetLastError();
}

cudaError_t launch_intensity_argmin_index(const uint8_t *idx, const double *zw,
                                          const double *amp, size_t n,
                                          const unsigned long long *d_best,
                                          unsigned long long *d_idx, cudaStream_t s)
{
    k_int_argmin<<<blocks_for(n), kThreads, 0, s>>>(idx, zw, amp, n, d_best, d_idx);
    return cudaGetLastError();
}

cudaError_t launch_plane_sums(const uint8_t *idx_a, const double *za, const double *amp_a,
                              const uint8_t *idx_w, const double *zw, const double *amp_w,
                              int nx, int ny, int nz, const unsigned long long *d_idx,
                              double *d_sums, cudaStream_t s)
{
    k_plane_sums<<<1, 1024, 0, s>>>(idx_a, za, amp_a, idx_w, zw, amp_w, nx, ny, nz, d_idx, d_sums);
    return cudaGetLastError();
}

}  // namespace bvf
