// Fused row passes of the surrogate's BF16 path on the fifth-generation
// tensor cores (BF16 operands, FP32 accumulation in TMEM; the network of
// include/bvf_fno.h, Li et al., ICLR 2021, Sec. 4):
//
//   k_row_bf16      one Fourier layer's output, or its backward, in one pass:
//     out[o][p] = act( sum_j G[j][x] S[o][row][j] + sum_c Wm(o, c) v[c][p] + b[o] )
//     the real inverse transform along x of the row's spectrum S (or, in the
//     backward pass, the adjoint of the forward one) plus the channel mix;
//     act: none, GELU (the pre-activation kept when asked), or times GELU'
//     of a stored pre-activation.  Without S it is the lift.
//   k_project_bf16  both layers of the projection with the hidden
//     activations in shared memory.
//   k_chan_bf16     one layer of the projection with its activations kept
//     (training), and the backward products.
//
// What they replace are separate products (bvf_gemm_bf16.cu) with the volume
// between them in HBM.  At 240 x 240 x 200, width 32, a layer took 904 us for
// the inverse (1.5 GB written) and 2040 us for the mix (1.5 GB read twice
// over, 1.5 GB written), the projection 6806 + 2151 us around 5.9 GB of
// hidden activations; now 690 us a layer and 1793 us.  Every product keeps its
// operands' rounding and its order of K steps, and the two sums of a layer
// meet in FP32 in the epilogue as they did through memory, so the results are
// the separate products' bit for bit.
//
// Waits are bounded as in the other tensor-core kernels: a block whose wait
// runs out issues nothing more, waits (bounded) for the products in flight,
// frees its tensor memory, sets bit 2 of the flag and ends.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "bvf_fno_bf16.cuh"
#include "bvf_tc.cuh"
#include "bvf_tma.cuh"

namespace bvf {

namespace {

constexpr int kSmemCap = 200 * 1024;

// Points of a tile: 128 consecutive x of one (z, y) row, or, where a row is
// shorter than 65 points, RP whole rows (RP <= 4).  With several rows the
// spectral operand is block diagonal: row r of the tile has its own JP
// columns of K, zero for the other rows' points.
struct RowBLayout {
    int RP, nxt, JP, KS, sA, sT, sW, sS, sb, bar, tmem, bytes;
    __host__ __device__ RowBLayout(int width, int kc, int m, int nx, bool spec)
    {
        RP = nx > 64 ? 1 : (nx > 32 ? 2 : 4);
        nxt = nx > 64 ? (nx + 127) / 128 : 1;
        JP = spec ? (2 * m + 15) / 16 * 16 : 0;
        KS = RP * JP;
        sA = 0;                                   // [128][kc]
        sT = sA + 128 * kc * 2;                   // [nxt][128][KS]
        sW = sT + nxt * 128 * KS * 2;             // [width][kc]
        sS = sW + width * kc * 2;                 // [width][KS]
        sb = sS + width * KS * 2;
        bar = (sb + width * 4 + 15) & ~15;
        tmem = bar + 16;
        bytes = tmem + 16;
    }
};

// e / d by multiplication (d >= 1, e d < 2^30)
struct SmallDiv {
    unsigned d, f;
    __device__ explicit SmallDiv(unsigned d_) : d(d_), f((0x80000000u + d_ - 1) / d_) {}
    __device__ unsigned quot(unsigned e) const { return __umulhi(2 * e, f); }
};

// W output channels; input channels padded to KC (a multiple of 16); RP rows a
// tile; SPEC: with a spectral term (the lift has none).  The products of a
// tile run under the epilogue of the tile before it: two accumulator sets in
// tensor memory, one barrier a tile.  With the products waited for in turn,
// and divisions for the row, branches and 64-bit address products for every
// output (80 instructions an output, two thirds of the issue slots), a layer
// took 1179 us at 240 x 240 x 200, width 32, the last one (no GELU) 845 and the
// lift 787; now 690, 592 and 331.  Bound by issue under a GELU, by its reads
// and writes (433 us at 6.8 TB/s) without.
template <int W, int KC, int RP, bool SPEC>
struct RowBShape {
    static constexpr int kSet = SPEC ? 2 * W : W;            // columns of a set
    static constexpr int kCols = 2 * kSet <= 32 ? 32 : (2 * kSet <= 64 ? 64 : (2 * kSet <= 128 ? 128 : 256));
    static constexpr int kBlocks = SPEC ? (kCols <= 128 ? 3 : 2) : 4;
};

template <int W, int KC, int RP, bool SPEC>
__global__ void __launch_bounds__(256, (RowBShape<W, KC, RP, SPEC>::kBlocks))
    k_row_bf16(const __grid_constant__ RowBf16 q)
{
    static_assert(W % 16 == 0 && KC % 16 == 0, "tile shape");
    using Shape = RowBShape<W, KC, RP, SPEC>;
    extern __shared__ __align__(128) unsigned char sm[];
    const int nx = q.nx, m = q.m, rows = q.rows, N = q.N;
    const RowBLayout L(W, KC, m, nx, SPEC);
    const int JP = L.JP, KS = L.KS, nxt = L.nxt;
    unsigned char *sA = sm + L.sA, *sT = sm + L.sT, *sW = sm + L.sW, *sS = sm + L.sS;
    float *sb = reinterpret_cast<float *>(sm + L.sb);
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + L.bar);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(sm + L.tmem);
    const int tid = threadIdx.x, warp = tid >> 5, pt = tid & 127, half = tid >> 7;
    // this thread's point: row lr of the tile, x (of the first tile)
    const int lr = RP > 1 ? pt / nx : 0, px = pt - lr * nx;
    // block constants: the channel weights, the x table, the zero columns of S
    for (int e = tid; e < W * (KC / 2); e += 256) {
        const int o = e / (KC / 2), c = 2 * (e - o * (KC / 2));
        const float w0 = c < q.cin ? q.Wm[o * q.wso + c * q.wsc] : 0.0f;
        const float w1 = c + 1 < q.cin ? q.Wm[o * q.wso + (c + 1) * q.wsc] : 0.0f;
        *reinterpret_cast<uint32_t *>(sW + tc::kmaj_off16(o, c & ~7, KC) + (c & 7) * 2) =
            tc::pack_bf16(w0, w1);
    }
    if (SPEC) {
        for (int e = tid; e < nxt * 128 * (KS / 2); e += 256) {
            const int t = e / (128 * (KS / 2)), r = e - t * 128 * (KS / 2);
            const int xl = r / (KS / 2), k = 2 * (r - xl * (KS / 2));
            const int xr = RP > 1 ? xl / nx : 0, x = RP > 1 ? xl - xr * nx : 128 * t + xl;
            const int kr = k / JP, j = k - kr * JP;
            const bool on = xr < RP && kr == xr && x < nx;
            const float g0 = on && j < 2 * m ? q.G[j * nx + x] : 0.0f;
            const float g1 = on && j + 1 < 2 * m ? q.G[(j + 1) * nx + x] : 0.0f;
            *reinterpret_cast<uint32_t *>(sT + t * 128 * KS * 2 + tc::kmaj_off16(xl, k & ~7, KS) +
                                          (k & 7) * 2) = tc::pack_bf16(g0, g1);
        }
        for (int e = tid; e < W * (KS / 2); e += 256) {
            const int o = e / (KS / 2), k = 2 * (e - o * (KS / 2));
            if (k % JP >= 2 * m)
                *reinterpret_cast<uint32_t *>(sS + tc::kmaj_off16(o, k & ~7, KS) + (k & 7) * 2) = 0u;
        }
    }
    for (int o = tid; o < W; o += 256) sb[o] = q.bias ? q.bias[o] : 0.0f;
    if (tid == 0) {
        tma::mbar_init(bar, 1);
        tma::mbar_init_fence();
    }
    if (warp == 0) {
        tc::alloc(tslot, Shape::kCols);
        tc::relinquish();
    }
    tma::fence_async_smem();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = *tslot;
    const uint32_t idesc = tc::idesc_bf16(128, W);
    constexpr int CH = KC / 2;                       // channels a thread stages
    constexpr uint32_t SBO = (KC / 8) * 128;
    const uint32_t sbo_s = (uint32_t)(KS / 8) * 128;
    const int groups = (rows + RP - 1) / RP;         // row groups of a sample

    struct Pos {
        int b, g, t;                                 // sample, row group, tile of the row
    };
    auto next = [&](Pos p) {
        if (++p.t == nxt) {
            p.t = 0;
            for (p.g += gridDim.x; p.g >= groups; p.g -= groups) ++p.b;
        }
        return p;
    };
    // this thread's point of a tile: whether there is one, and its index
    auto point = [&](const Pos &p, long long &at) {
        const int row = p.g * RP + lr, x = RP > 1 ? px : 128 * p.t + pt;
        at = (long long)row * nx + x;
        return RP > 1 ? (lr < RP && row < rows) : x < nx;
    };
    // loaded one tile (channels) or one row group (spectral pairs) ahead of staging
    float xv[CH];
    const bool full = q.cin == KC;
    auto load_v = [&](const Pos &p) {
        long long at;
        const bool ok = point(p, at);
        const float *src = q.v + p.b * q.vb + (long long)(half * CH) * N + at;
        if (full) {
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                xv[c] = ok ? tma::ld_stream(src) : 0.0f;
                src += N;
            }
        } else {
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                xv[c] = ok && half * CH + c < q.cin ? tma::ld_stream(src) : 0.0f;
                src += N;
            }
        }
    };
    constexpr int PRE = SPEC ? (W * RP * 16 + 255) / 256 : 1;   // pairs per thread at m = 16
    float2 pre[PRE];
    const SmallDiv by_rm((unsigned)(RP * (SPEC ? m : 1))), by_m((unsigned)(SPEC ? m : 1));
    auto load_s = [&](const Pos &p) {
        const int row0 = p.g * RP;
        const float *src = q.S + ((long long)p.b * W * rows + row0) * (2 * m);
#pragma unroll
        for (int i = 0; i < PRE; ++i) {
            const int e = tid + i * 256;
            pre[i] = make_float2(0.0f, 0.0f);
            if (e < W * RP * m) {
                const int o = by_rm.quot(e), r = e - o * RP * m;   // r: pair of the o's RP rows
                if (RP == 1 || row0 + (int)by_m.quot(r) < rows)
                    pre[i] = tma::ld_stream(
                        reinterpret_cast<const float2 *>(src + (long long)o * rows * (2 * m)) + r);
            }
        }
    };
    auto stage = [&](const Pos &p) {
#pragma unroll
        for (int c8 = 0; c8 < CH / 8; ++c8)
            *reinterpret_cast<uint4 *>(sA + tc::kmaj_off16(pt, half * CH + 8 * c8, KC)) =
                make_uint4(tc::pack_bf16(xv[8 * c8], xv[8 * c8 + 1]),
                           tc::pack_bf16(xv[8 * c8 + 2], xv[8 * c8 + 3]),
                           tc::pack_bf16(xv[8 * c8 + 4], xv[8 * c8 + 5]),
                           tc::pack_bf16(xv[8 * c8 + 6], xv[8 * c8 + 7]));
        if (SPEC && p.t == 0) {
#pragma unroll
            for (int i = 0; i < PRE; ++i) {
                const int e = tid + i * 256;
                if (e < W * RP * m) {
                    const int o = by_rm.quot(e), r = e - o * RP * m;
                    const int kr = RP == 1 ? 0 : by_m.quot(r), k = kr * JP + 2 * (r - kr * m);
                    *reinterpret_cast<uint32_t *>(sS + tc::kmaj_off16(o, k & ~7, KS) + (k & 7) * 2) =
                        tc::pack_bf16(pre[i].x, pre[i].y);
                }
            }
        }
        tma::fence_async_smem();
        tc::fence_before();
    };
    // thread 0, after a barrier behind stage(): both sums of a tile into a set
    auto issue = [&](const Pos &p, int set) {
        const uint32_t ta = tbase + (uint32_t)(set * Shape::kSet);
        tc::fence_after();
        if (SPEC)
            for (int ks = 0; ks < KS / 16; ++ks)
                tc::mma_f16(ta, tc::smem_desc(sT + p.t * 128 * KS * 2 + ks * 256, 128, sbo_s),
                            tc::smem_desc(sS + ks * 256, 128, sbo_s), idesc, ks > 0);
#pragma unroll
        for (int ks = 0; ks < KC / 16; ++ks)
            tc::mma_f16(ta + (SPEC ? W : 0), tc::smem_desc(sA + ks * 256, 128, SBO),
                        tc::smem_desc(sW + ks * 256, 128, SBO), idesc, ks > 0);
        tc::commit(bar);
    };
    // ACT: 0 none, 1 GELU, 2 times GELU' of the stored value, 3 GELU, value kept
    auto epilogue = [&](auto act, const Pos &p, int set) {
        constexpr int ACT = decltype(act)::value;
        long long at;
        const bool ok = point(p, at);
        const int o0 = half * (W / 2);
        const uint32_t ta = tbase + (uint32_t)(set * Shape::kSet + o0) +
                            ((uint32_t)(32 * (warp & 3)) << 16);
        at += ((long long)p.b * W + o0) * N;
        float *op = q.out + at;
        float *pp = ACT >= 2 ? q.pre + at : nullptr;
#pragma unroll 1
        for (int c0 = 0; c0 < W / 2; c0 += 8) {
            float d[8], s[8], pv[8];
            tc::ld8(ta + (SPEC ? W : 0) + c0, d);
            if (SPEC) tc::ld8(ta + c0, s);
            if (ACT == 2 && ok) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    pv[i] = tma::ld_stream(pp);
                    pp += N;
                }
            }
            tc::wait_ld();
            if (ok) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    float v = SPEC ? __fadd_rn(s[i], d[i]) : d[i];
                    v = __fadd_rn(v, sb[o0 + c0 + i]);
                    if (ACT == 3) {
                        *pp = v;
                        pp += N;
                    }
                    if (ACT == 1 || ACT == 3) v = gelu_exact(v);
                    if (ACT == 2) v *= gelu_grad(pv[i]);
                    *op = v;
                    op += N;
                }
            }
            __syncwarp();            // the next tensor-memory load is warp-wide
        }
    };
    // weights and tables are in place: the rest depends on earlier kernels
    tma::pdl_wait();
    tma::pdl_launch_next();
    Pos cur{0, (int)blockIdx.x, 0};
    for (; cur.g >= groups; cur.g -= groups) ++cur.b;     // gridDim.x <= B groups
    load_v(cur);
    if (SPEC) load_s(cur);
    stage(cur);
    __syncthreads();
    if (tid == 0) issue(cur, 0);
    Pos nxtp = next(cur);
    if (nxtp.b < q.B) {
        load_v(nxtp);
        if (SPEC && nxtp.t == 0) load_s(nxtp);
    }
    int phase = 0;
    bool gave_up = false;
    while (cur.b < q.B) {
        // the products of cur: their operands and the other accumulators are free
        const bool ready =
            __all_sync(0xffffffffu, tma::mbar_wait(bar, phase & 1, tma::kWaitLimit));
        tc::fence_after();
        const bool more = nxtp.b < q.B;
        if (more && ready) stage(nxtp);
        gave_up = __syncthreads_or(!ready) != 0;
        if (gave_up) break;
        Pos after = nxtp;
        if (more) {
            if (tid == 0) issue(nxtp, (phase + 1) & 1);
            after = next(nxtp);
            if (after.b < q.B) {
                load_v(after);
                if (SPEC && after.t == 0) load_s(after);
            }
        }
        const int set = phase & 1;
        if (!SPEC || q.act == 0)
            epilogue(std::integral_constant<int, 0>{}, cur, set);
        else if (q.act == 2)
            epilogue(std::integral_constant<int, 2>{}, cur, set);
        else if (q.pre)
            epilogue(std::integral_constant<int, 3>{}, cur, set);
        else
            epilogue(std::integral_constant<int, 1>{}, cur, set);
        tc::fence_before();
        cur = nxtp;
        nxtp = after;
        ++phase;
    }
    if (gave_up && tid == 0) {
        tma::mbar_wait(bar, phase & 1, tma::kWaitLimit);
        atomicOr(q.flag, 2);
    }
    tc::fence_after();
    __syncthreads();
    if (warp == 0) tc::dealloc(tbase, Shape::kCols);
}

// ---------------------------------------------------------------- projection
// out[k][p] = q2[k] + sum_j Q2[k][j] GELU(q1[j] + sum_c Q1[j][c] v[c][p]) on
// 128-point tiles: the first product into TMEM, GELU and rounding to BF16 into
// shared memory, the second product over the first one's columns of TMEM.
struct ProjBLayout {
    int HP, ncols, sA, sB, sH, sQ, sq1, sq2, bar, tmem, bytes;
    __host__ __device__ ProjBLayout(int width, int hidden)
    {
        HP = (hidden + 15) & ~15;
        ncols = 32;
        while (ncols < HP) ncols *= 2;
        sA = 0;                              // [128][width]
        sB = sA + 128 * width * 2;           // [HP][width]
        sH = sB + HP * width * 2;            // [128][HP]
        sQ = sH + 128 * HP * 2;              // [16][HP]
        sq1 = sQ + 16 * HP * 2;
        sq2 = sq1 + HP * 4;
        bar = (sq2 + 8 * 4 + 15) & ~15;
        tmem = bar + 16;
        bytes = tmem + 16;
    }
};

template <int W>
__global__ void __launch_bounds__(256, 3)
    k_project_bf16(const float *v, const float *__restrict__ Q1,
                   const float *__restrict__ q1, const float *__restrict__ Q2,
                   const float *__restrict__ q2, int hidden, int c_out, float *__restrict__ out,
                   int N, int B, int *flag)
{
    extern __shared__ __align__(128) unsigned char sm[];
    const ProjBLayout L(W, hidden);
    const int HP = L.HP;
    unsigned char *sA = sm + L.sA, *sB = sm + L.sB, *sH = sm + L.sH, *sQ = sm + L.sQ;
    float *sq1 = reinterpret_cast<float *>(sm + L.sq1), *sq2 = reinterpret_cast<float *>(sm + L.sq2);
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + L.bar);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(sm + L.tmem);
    const int tid = threadIdx.x, warp = tid >> 5, pt = tid & 127, half = tid >> 7;
    for (int e = tid; e < HP * (W / 2); e += 256) {
        const int j = e / (W / 2), c = 2 * (e - j * (W / 2));
        const bool on = j < hidden;
        *reinterpret_cast<uint32_t *>(sB + tc::kmaj_off16(j, c & ~7, W) + (c & 7) * 2) =
            tc::pack_bf16(on ? Q1[j * W + c] : 0.0f, on ? Q1[j * W + c + 1] : 0.0f);
    }
    for (int e = tid; e < 16 * (HP / 2); e += 256) {
        const int k = e / (HP / 2), j = 2 * (e - k * (HP / 2));
        const float a = k < c_out && j < hidden ? Q2[k * hidden + j] : 0.0f;
        const float c = k < c_out && j + 1 < hidden ? Q2[k * hidden + j + 1] : 0.0f;
        *reinterpret_cast<uint32_t *>(sQ + tc::kmaj_off16(k, j & ~7, HP) + (j & 7) * 2) =
            tc::pack_bf16(a, c);
    }
    for (int j = tid; j < HP; j += 256) sq1[j] = j < hidden ? q1[j] : 0.0f;
    if (tid < 8) sq2[tid] = tid < c_out ? q2[tid] : 0.0f;
    if (tid == 0) {
        tma::mbar_init(bar, 1);
        tma::mbar_init_fence();
    }
    if (warp == 0) {
        tc::alloc(tslot, L.ncols);
        tc::relinquish();
    }
    tma::fence_async_smem();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = *tslot;
    const uint32_t id1 = tc::idesc_bf16(128, HP), id2 = tc::idesc_bf16(128, 16);
    constexpr uint32_t SBO = (W / 8) * 128;
    const uint32_t sbo_h = (uint32_t)(HP / 8) * 128;
    constexpr int CH = W / 2;
    const int per = (N + 127) / 128, tiles = per * B;      // tiles of one sample, of the batch
    float xv[CH];
    auto load = [&](int tile) {
        const int b = tile / per, p = (tile - b * per) * 128 + pt;
        const float *src = v + (long long)b * W * N + p;
#pragma unroll
        for (int c = 0; c < CH; ++c)
            xv[c] = p < N ? tma::ld_stream(src + (long long)(half * CH + c) * N) : 0.0f;
    };
    tma::pdl_wait();
    tma::pdl_launch_next();
    if ((int)blockIdx.x < tiles) load(blockIdx.x);
    int phase = 0;
    bool gave_up = false;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
#pragma unroll
        for (int c8 = 0; c8 < CH / 8; ++c8)
            *reinterpret_cast<uint4 *>(sA + tc::kmaj_off16(pt, half * CH + 8 * c8, W)) =
                make_uint4(tc::pack_bf16(xv[8 * c8], xv[8 * c8 + 1]),
                           tc::pack_bf16(xv[8 * c8 + 2], xv[8 * c8 + 3]),
                           tc::pack_bf16(xv[8 * c8 + 4], xv[8 * c8 + 5]),
                           tc::pack_bf16(xv[8 * c8 + 6], xv[8 * c8 + 7]));
        tma::fence_async_smem();
        tc::fence_before();
        __syncthreads();
        if (tid == 0) {
            tc::fence_after();
#pragma unroll
            for (int ks = 0; ks < W / 16; ++ks)
                tc::mma_f16(tbase, tc::smem_desc(sA + ks * 256, 128, SBO),
                            tc::smem_desc(sB + ks * 256, 128, SBO), id1, ks > 0);
            tc::commit(bar);
        }
        if (tile + (int)gridDim.x < tiles) load(tile + gridDim.x);
        bool ready = __all_sync(0xffffffffu, tma::mbar_wait(bar, phase & 1, tma::kWaitLimit));
        tc::fence_after();
        if (ready) {
            for (int c0 = 32 * half; c0 < HP; c0 += 64) {      // HP is a multiple of 16
                float r[32];
                tc::ld32(tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0, r);
                tc::wait_ld();
#pragma unroll
                for (int i = 0; i < 32; i += 8) {
                    if (c0 + i >= HP) break;
                    uint32_t u[4];
#pragma unroll
                    for (int h = 0; h < 4; ++h)
                        u[h] = tc::pack_bf16(gelu_exact(__fadd_rn(r[i + 2 * h], sq1[c0 + i + 2 * h])),
                                             gelu_exact(__fadd_rn(r[i + 2 * h + 1],
                                                                  sq1[c0 + i + 2 * h + 1])));
                    *reinterpret_cast<uint4 *>(sH + tc::kmaj_off16(pt, c0 + i, HP)) =
                        make_uint4(u[0], u[1], u[2], u[3]);
                }
            }
        }
        tma::fence_async_smem();
        tc::fence_before();
        gave_up = __syncthreads_or(!ready) != 0;
        if (gave_up) break;
        ++phase;
        if (tid == 0) {
            tc::fence_after();
            for (int ks = 0; ks < HP / 16; ++ks)
                tc::mma_f16(tbase, tc::smem_desc(sH + ks * 256, 128, sbo_h),
                            tc::smem_desc(sQ + ks * 256, 128, sbo_h), id2, ks > 0);
            tc::commit(bar);
        }
        ready = __all_sync(0xffffffffu, tma::mbar_wait(bar, phase & 1, tma::kWaitLimit));
        tc::fence_after();
        if (ready && !half) {
            float r[8];
            tc::ld8(tbase + ((uint32_t)(32 * warp) << 16), r);
            tc::wait_ld();
            const int b = tile / per, p = (tile - b * per) * 128 + pt;
            if (p < N) {
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (k < c_out)
                        out[((long long)b * c_out + k) * N + p] = __fadd_rn(r[k], sq2[k]);
            }
        }
        tc::fence_before();
        gave_up = __syncthreads_or(!ready) != 0;
        if (gave_up) break;
        ++phase;
    }
    if (gave_up && tid == 0) {
        tma::mbar_wait(bar, phase & 1, tma::kWaitLimit);
        atomicOr(flag, 2);
    }
    tc::fence_after();
    __syncthreads();
    if (warp == 0) tc::dealloc(tbase, L.ncols);
}

// ------------------------------------------------------------ channel product
// out[o][p] = act( sum_c Wm(o, c) v[c][p] + b[o] ) on 128-point tiles, any K up
// to 256 input and N up to 256 output channels: the projection's two layers
// and their backward products when their activations are kept.  All of K is
// staged at once (16 channels per thread in flight), the weights once per
// block.  As separate products of one tile a block the four took 1244, 397,
// 1244 and 397 us at 64 x 64 x 96, batch 4; now 371, 189, 466 (two special
// functions for each of 201 million values) and 205.
struct ChanBLayout {
    int KP, NP, ncols, sA, sB, sb, bar, tmem, bytes;
    __host__ __device__ ChanBLayout(int K, int N)
    {
        KP = (K + 15) & ~15;
        NP = (N + 15) & ~15;
        ncols = 32;
        while (ncols < NP) ncols *= 2;
        sA = 0;                              // [128][KP]
        sB = sA + 128 * KP * 2;              // [NP][KP]
        sb = sB + NP * KP * 2;
        bar = (sb + NP * 4 + 15) & ~15;
        tmem = bar + 16;
        bytes = tmem + 16;
    }
};

__global__ void __launch_bounds__(256, 3) k_chan_bf16(const __grid_constant__ ChanBf16 q)
{
    extern __shared__ __align__(128) unsigned char sm[];
    const ChanBLayout L(q.K, q.O);
    const int KP = L.KP, NP = L.NP, N = q.N;
    unsigned char *sA = sm + L.sA, *sB = sm + L.sB;
    float *sb = reinterpret_cast<float *>(sm + L.sb);
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + L.bar);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(sm + L.tmem);
    const int tid = threadIdx.x, warp = tid >> 5, pt = tid & 127, half = tid >> 7;
    for (int e = tid; e < NP * (KP / 2); e += 256) {
        const int o = e / (KP / 2), c = 2 * (e - o * (KP / 2));
        const float w0 = o < q.O && c < q.K ? q.Wm[o * q.wso + c * q.wsc] : 0.0f;
        const float w1 = o < q.O && c + 1 < q.K ? q.Wm[o * q.wso + (c + 1) * q.wsc] : 0.0f;
        *reinterpret_cast<uint32_t *>(sB + tc::kmaj_off16(o, c & ~7, KP) + (c & 7) * 2) =
            tc::pack_bf16(w0, w1);
    }
    for (int o = tid; o < NP; o += 256) sb[o] = q.bias && o < q.O ? q.bias[o] : 0.0f;
    if (tid == 0) {
        tma::mbar_init(bar, 1);
        tma::mbar_init_fence();
    }
    if (warp == 0) {
        tc::alloc(tslot, L.ncols);
        tc::relinquish();
    }
    tma::fence_async_smem();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = *tslot;
    const uint32_t idesc = tc::idesc_bf16(128, NP);
    const uint32_t sbo = (uint32_t)(KP / 8) * 128;
    const int per = (N + 127) / 128, tiles = per * q.B;
    tma::pdl_wait();
    tma::pdl_launch_next();
    // 16 channels of this thread's point: c0 + 16 half ..
    float xv[16];
    auto load = [&](int tile, int c0) {
        const int b = tile / per, p = (tile - b * per) * 128 + pt, ch = c0 + 16 * half;
        const float *src = q.v + ((long long)b * q.K + ch) * N + p;
#pragma unroll
        for (int c = 0; c < 16; ++c)
            xv[c] = p < N && ch + c < q.K ? tma::ld_stream(src + (long long)c * N) : 0.0f;
    };
    // ACT: 0 none, 1 GELU (the value kept when asked), 2 times GELU' of the kept one
    auto epilogue = [&](auto act, int tile) {
        constexpr int ACT = decltype(act)::value;
        const int b = tile / per, p = (tile - b * per) * 128 + pt;
        const bool keep = ACT == 1 && q.pre;
#pragma unroll 1
        for (int c0 = 16 * half; c0 < NP; c0 += 32) {
            const int n = p < N ? min(16, q.O - c0) : 0;
            const long long at = ((long long)b * q.O + c0) * N + p;
            float r[16], pv[16];
            tc::ld16(tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0, r);
            if (ACT == 2) {
                const float *pp = q.pre + at;
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    if (i < n) pv[i] = tma::ld_stream(pp);
                    pp += N;
                }
            }
            tc::wait_ld();
            float *op = q.out + at, *pp = ACT == 1 ? q.pre + at : nullptr;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                if (i < n) {
                    float v = q.bias ? __fadd_rn(r[i], sb[c0 + i]) : r[i];
                    if (ACT == 1) {
                        if (keep) *pp = v;
                        v = gelu_exact(v);
                    } else if (ACT == 2) {
                        v *= gelu_grad(pv[i]);
                    }
                    *op = v;
                }
                op += N;
                if (ACT == 1) pp += N;
            }
            __syncwarp();            // the next tensor-memory load is warp-wide
        }
    };
    if ((int)blockIdx.x < tiles) load(blockIdx.x, 0);
    int phase = 0;
    bool gave_up = false;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        for (int c0 = 0; c0 < KP; c0 += 32) {
            const int ch = c0 + 16 * half;
            if (ch < KP) {                       // KP is a multiple of 16
                *reinterpret_cast<uint4 *>(sA + tc::kmaj_off16(pt, ch, KP)) =
                    make_uint4(tc::pack_bf16(xv[0], xv[1]), tc::pack_bf16(xv[2], xv[3]),
                               tc::pack_bf16(xv[4], xv[5]), tc::pack_bf16(xv[6], xv[7]));
                *reinterpret_cast<uint4 *>(sA + tc::kmaj_off16(pt, ch + 8, KP)) =
                    make_uint4(tc::pack_bf16(xv[8], xv[9]), tc::pack_bf16(xv[10], xv[11]),
                               tc::pack_bf16(xv[12], xv[13]), tc::pack_bf16(xv[14], xv[15]));
            }
            if (c0 + 32 < KP) load(tile, c0 + 32);
        }
        tma::fence_async_smem();
        tc::fence_before();
        __syncthreads();
        if (tid == 0) {
            tc::fence_after();
            for (int ks = 0; ks < KP / 16; ++ks)
                tc::mma_f16(tbase, tc::smem_desc(sA + ks * 256, 128, sbo),
                            tc::smem_desc(sB + ks * 256, 128, sbo), idesc, ks > 0);
            tc::commit(bar);
        }
        if (tile + (int)gridDim.x < tiles) load(tile + gridDim.x, 0);
        const bool ready = __all_sync(0xffffffffu, tma::mbar_wait(bar, phase & 1, tma::kWaitLimit));
        tc::fence_after();
        if (ready) {
            if (q.act == 0)
                epilogue(std::integral_constant<int, 0>{}, tile);
            else if (q.act == 2)
                epilogue(std::integral_constant<int, 2>{}, tile);
            else
                epilogue(std::integral_constant<int, 1>{}, tile);
        }
        tc::fence_before();
        gave_up = __syncthreads_or(!ready) != 0;
        if (gave_up) break;
        ++phase;
    }
    if (gave_up && tid == 0) {
        tma::mbar_wait(bar, phase & 1, tma::kWaitLimit);
        atomicOr(q.flag, 2);
    }
    tc::fence_after();
    __syncthreads();
    if (warp == 0) tc::dealloc(tbase, L.ncols);
}

// the shared-memory limit, raised once per process and kernel to the cap, so
// that later launches make no other runtime call
template <auto Kernel>
cudaError_t raise_smem()
{
    static std::atomic<int> done{0};
    if (done.load(std::memory_order_acquire)) return cudaSuccess;
    const cudaError_t e =
        cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
    if (e == cudaSuccess) done.store(1, std::memory_order_release);
    return e;
}

int blocks_per_sm(int bytes, int ncols, int most = 3)
{
    return std::max(1, std::min({most, (227 * 1024) / (bytes + 1024), 512 / ncols}));
}

template <int W, int KC, int RP, bool SPEC>
cudaError_t launch_row_k(const RowBf16 &q, const RowBLayout &L, cudaStream_t s)
{
    using Shape = RowBShape<W, KC, RP, SPEC>;
    const cudaError_t e = raise_smem<k_row_bf16<W, KC, RP, SPEC>>();
    if (e != cudaSuccess) return e;
    const int items = q.B * ((q.rows + RP - 1) / RP);
    const int grid = std::min(items, q.n_sm * blocks_per_sm(L.bytes, Shape::kCols, Shape::kBlocks));
    if (SPEC) return launch_pdl(k_row_bf16<W, KC, RP, SPEC>, grid, 256, L.bytes, s, q);
    // the lift reads weights that an optimiser step just before it may have
    // written: an ordinary launch
    k_row_bf16<W, KC, RP, SPEC><<<grid, 256, L.bytes, s>>>(q);
    return cudaGetLastError();
}

template <int W, int KC, bool SPEC>
cudaError_t launch_row_w(const RowBf16 &q, cudaStream_t s)
{
    const RowBLayout L(W, KC, q.m, q.nx, SPEC);
    if (L.RP == 1) return launch_row_k<W, KC, 1, SPEC>(q, L, s);
    if (L.RP == 2) return launch_row_k<W, KC, 2, SPEC>(q, L, s);
    return launch_row_k<W, KC, 4, SPEC>(q, L, s);
}

}  // namespace

bool row_bf16_fits(int width, int m, int nx)
{
    return RowBLayout(width, width, m, nx, true).bytes <= kSmemCap;
}

cudaError_t launch_row_bf16(const RowBf16 &q, int width, cudaStream_t s)
{
    // the lift's 1 .. 16 input channels fill one K step; a layer has W
    if (!q.S) {
        switch (width) {
        case 16: return launch_row_w<16, 16, false>(q, s);
        case 32: return launch_row_w<32, 16, false>(q, s);
        case 48: return launch_row_w<48, 16, false>(q, s);
        default: return launch_row_w<64, 16, false>(q, s);
        }
    }
    switch (width) {
    case 16: return launch_row_w<16, 16, true>(q, s);
    case 32: return launch_row_w<32, 32, true>(q, s);
    case 48: return launch_row_w<48, 48, true>(q, s);
    default: return launch_row_w<64, 64, true>(q, s);
    }
}

cudaError_t launch_chan_bf16(const ChanBf16 &q, int n_sm, cudaStream_t s)
{
    const ChanBLayout L(q.K, q.O);
    const cudaError_t e = raise_smem<k_chan_bf16>();
    if (e != cudaSuccess) return e;
    const int grid = std::min((q.N + 127) / 128 * q.B, n_sm * blocks_per_sm(L.bytes, L.ncols));
    return launch_pdl(k_chan_bf16, grid, 256, L.bytes, s, q);
}

cudaError_t launch_project_bf16(const float *v, const float *Q1, const float *q1, const float *Q2,
                                const float *q2, int width, int hidden, int c_out, float *out, int N,
                                int B, int n_sm, int *flag, cudaStream_t s)
{
    const ProjBLayout L(width, hidden);
    const int tiles = (N + 127) / 128 * B;
    const int grid = std::min(tiles, n_sm * blocks_per_sm(L.bytes, L.ncols));
    cudaError_t e = cudaSuccess;
#define BVF_PROJ(WW)                                                                             \
    e = raise_smem<k_project_bf16<WW>>();                                                          \
    if (e == cudaSuccess)                                                                          \
        e = launch_pdl(k_project_bf16<WW>, grid, 256, L.bytes, s, v, Q1, q1, Q2, q2, hidden, c_out, \
                       out, N, B, flag);
    switch (width) {
    case 16: BVF_PROJ(16) break;
    case 32: BVF_PROJ(32) break;
    case 48: BVF_PROJ(48) break;
    default: BVF_PROJ(64) break;
    }
#undef BVF_PROJ
    return e;
}

}  // namespace bvf
