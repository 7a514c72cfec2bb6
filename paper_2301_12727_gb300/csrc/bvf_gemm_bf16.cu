// BF16 tensor-core product on the fifth-generation tensor cores (tcgen05):
// C = alpha A B + beta C (+ bias) (-> GELU), FP32 in and out, BF16 operands,
// FP32 accumulation in tensor memory.  The y and z transforms of the surrogate's
// BF16 path and of its training run on it, and every other contraction where a
// kernel of its own does not take the shape, as calls on strided views.
//
// A block of 128 threads computes a 128 x BN tile of C:
//   * K runs in chunks of 64; the chunk's A (128 x 64) and B (BN x 64) tiles
//     are read from their strided FP32 arrays, rounded to BF16 and written to
//     shared memory K-major with a 128-byte swizzle (without one the eight
//     pieces of a row share their banks), two stages deep, so the threads stage chunk c+1 while the
//     tensor cores multiply chunk c;
//   * thread 0 issues four tcgen05.mma.kind::f16 (K = 16 each) per chunk into
//     the TMEM accumulator and commits them to the stage's mbarrier;
//   * the epilogue reads the accumulator with tcgen05.ld (warp w holds rows
//     32 w .. 32 w + 31) and applies alpha, beta, the bias and GELU (keeping
//     the pre-activation when asked), or adds into C atomically when K is
//     split over several blocks.
// Waits are bounded: a block whose wait runs out stops issuing products,
// waits (bounded) for those in flight, frees its tensor memory, sets bit 2 of
// the flag and ends.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>

#include "bvf_fno_bf16.cuh"
#include "bvf_tc.cuh"
#include "bvf_tma.cuh"

namespace bvf {

namespace {

constexpr int GK = 64;                 // K chunk (BF16 elements): 128 bytes per row
constexpr int GSEG = GK / 8;           // 16-byte core-matrix rows per tile row and chunk
// NS shared-memory stages of GK-wide K chunks: two overlap the staging of a
// chunk with the products of the previous one; products of a single chunk
// (K <= GK) take one, so twice as many blocks fit per SM.
template <int BN, int NS>
struct GemmLayout {
    static constexpr int A_BYTES = 128 * GK * 2;
    static constexpr int B_BYTES = BN * GK * 2;
    static constexpr int STAGE = A_BYTES + B_BYTES;
    static constexpr int off_bar = NS * STAGE;
    static constexpr int off_tmem = off_bar + 16;
    static constexpr int off_rows = off_tmem + 16;     // [128] row starts of A, then of C
    static constexpr int bytes = off_rows + 2 * 128 * 8;
    static_assert(NS * STAGE >= 4 * 32 * 33 * 4, "the epilogue's transpose buffers fit the stages");
};

using tc::pack_bf16;

// Rows [0, rows) x K-chunk [k0, k0 + GK) of an FP32 operand (element (r, k) at
// src[start(r) + kof(k)]; zero for r >= valid or k >= K) written as BF16,
// K-major, swizzled.  Where k is contiguous (kc), consecutive threads
// take consecutive 8-element pieces of one row, otherwise consecutive rows,
// so the global reads are coalesced in both layouts.  vec: the pieces load
// as two float4 (aligned rows, four-element groups never straddle K or a part
// of it); four pieces are in flight per thread, against eight floats of one:
// the staging is bound by the latency of its loads.  own: the row a thread
// takes of a 128-row tile where k is not contiguous.
template <class Start, class Kof>
__device__ __forceinline__ void stage_tile(unsigned char *dst, const float *src,
                                           Start start, Kof kof, bool kc, bool vec, int rows,
                                           int valid, int k0, int K, int tid, int own)
{
    const int segs = rows * GSEG;
    if (vec) {
        constexpr int U = 4;
        for (int s0 = tid; s0 < segs; s0 += 128 * U) {
            float4 v[U][2];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int s = s0 + 128 * u, r = s / GSEG, k = k0 + (s % GSEG) * 8;
                const bool on = s < segs && r < valid;
                const float *row = src + (on ? start(r) : 0);
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    v[u][h] = (on && k + 4 * h < K)
                                  ? *reinterpret_cast<const float4 *>(row + kof(k + 4 * h))
                                  : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int s = s0 + 128 * u;
                if (s < segs)
                    *reinterpret_cast<uint4 *>(dst + tc::sw128_off(s / GSEG, s % GSEG)) =
                        make_uint4(pack_bf16(v[u][0].x, v[u][0].y), pack_bf16(v[u][0].z, v[u][0].w),
                                   pack_bf16(v[u][1].x, v[u][1].y), pack_bf16(v[u][1].z, v[u][1].w));
            }
        }
        return;
    }
#pragma unroll 2
    for (int s = tid; s < segs; s += 128) {
        int r, k8;
        if (kc) {
            r = s / GSEG;
            k8 = (s % GSEG) * 8;
        } else {
            r = rows == 128 ? own : s % rows;
            k8 = (s / rows) * 8;
        }
        float v[8];
        const bool on = r < valid;
        const float *row = src + (on ? start(r) : 0);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int k = k0 + k8 + j;
            v[j] = (on && k < K) ? row[kof(k)] : 0.0f;
        }
        *reinterpret_cast<uint4 *>(dst + tc::sw128_off(r, k8 >> 3)) =
            make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]),
                       pack_bf16(v[6], v[7]));
    }
}

template <int BN, int NS>
__global__ void __launch_bounds__(128) k_gemm_bf16(const __grid_constant__ GemmX gx, int *flag)
{
    const bvf_gemm &g = gx.g;
    extern __shared__ __align__(1024) unsigned char sm[];
    using Lay = GemmLayout<BN, NS>;
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + Lay::off_bar);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(sm + Lay::off_tmem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.x * 128, n0 = blockIdx.y * BN;
    const int b = blockIdx.z / g.ksplit, split = blockIdx.z % g.ksplit;
    const int n_chunks = (g.K + GK - 1) / GK;
    const int per = (n_chunks + g.ksplit - 1) / g.ksplit;
    const int c_begin = split * per, c_end = min(n_chunks, c_begin + per);
    const float *A = g.A + (long long)b * g.sab;
    const float *B = g.B + (long long)b * g.sbb + (long long)n0 * g.sbn;
    const int va = min(128, g.M - m0), vb = min(BN, g.N - n0);
    // where the tile's rows start in A and C
    long long *s_ar = reinterpret_cast<long long *>(sm + Lay::off_rows), *s_cr = s_ar + 128;
    {
        const int r = m0 + tid;
        s_ar[tid] = gx.ra ? (r / (gx.ra * gx.ra2)) * gx.sam2 + (r / gx.ra % gx.ra2) * gx.sam1 +
                                (r % gx.ra) * g.sam
                          : (long long)r * g.sam;
        s_cr[tid] = gx.rc ? (r / gx.rc) * gx.scm1 + (r % gx.rc) * g.scm : (long long)r * g.scm;
    }
    // Where rows ra apart are neighbours in memory (the inverse y transform: kx
    // runs fastest through the rows, z through A) the threads take the tile's
    // rows in A's order, so a warp's loads touch 4 lines instead of 32: at 64 x
    // 64 x 96, batch 4, that product took 104 us, at 240 x 240 x 200 192 us; with
    // that and the plain stores below 46 and 114.
    int own = tid;
    if (gx.ra > 0 && gx.ra < 128 && gx.sam1 == 1 && g.sam != 1) {
        const int q = 128 / gx.ra, rem = 128 % gx.ra, big = rem * (q + 1);
        const int t = tid - big;
        own = tid < big ? tid / (q + 1) + (tid % (q + 1)) * gx.ra : rem + t / q + (t % q) * gx.ra;
    }
    auto a_row = [&](int r) { return s_ar[r]; };
    auto a_col = [&](int k) -> long long {
        return gx.ka ? (k < gx.ka ? k * g.sak : gx.sak1 + (k - gx.ka) * g.sak) : k * g.sak;
    };
    auto b_row = [&](int r) { return (long long)r * g.sbn; };
    auto b_col = [&](int k) { return (long long)k * g.sbk; };
    if (tid == 0) {
        tma::mbar_init(&bar[0], 1);
        tma::mbar_init(&bar[1], 1);
        tma::mbar_init_fence();
    }
    if (warp == 0) {
        tc::alloc(tslot, BN);
        tc::relinquish();
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    tma::pdl_wait();
    tma::pdl_launch_next();
    const uint32_t tbase = *tslot;
    const uint32_t idesc = tc::idesc_bf16(128, BN);

    bool bad = false;
    int nc = 0;                             // chunks whose products were issued
    for (int c = c_begin; c < c_end; ++c, ++nc) {
        const int st = nc % NS;
        unsigned char *sa = sm + st * Lay::STAGE, *sb = sa + Lay::A_BYTES;
        if (nc >= NS) {                     // the products of chunk nc - NS read this stage
            const bool ok = tma::mbar_wait(&bar[st], ((nc - NS) / NS) & 1, tma::kWaitLimit);
            if (__syncthreads_or(!ok)) {
                bad = true;
                break;
            }
        }
        stage_tile(sa, A, a_row, a_col, g.sak == 1, gx.vec & 1, 128, va, c * GK, g.K, tid, own);
        stage_tile(sb, B, b_row, b_col, g.sbk == 1, gx.vec & 2, BN, vb, c * GK, g.K, tid, tid);
        tma::fence_async_smem();
        tc::fence_before();
        __syncthreads();
        if (tid == 0) {
            tc::fence_after();
#pragma unroll
            for (int ks = 0; ks < GK / 16; ++ks) {
                // 32 bytes of each row per K step of 16
                tc::mma_f16(tbase, tc::smem_desc_sw(sa + 32 * ks, 1024, tc::kSwizzle128),
                            tc::smem_desc_sw(sb + 32 * ks, 1024, tc::kSwizzle128), idesc, (nc > 0 || ks > 0) ? 1 : 0);
            }
            tc::commit(&bar[st]);
        }
    }
    if (!bad && nc > 0) {                   // the last commit covers every earlier product
        const int last = nc - 1;
        const bool ok = tma::mbar_wait(&bar[last % NS], (last / NS) & 1, tma::kWaitLimit);
        bad = __syncthreads_or(!ok) != 0;
    }
    if (bad) {
        if (tid == 0) {
            const int last = nc - 1;
            if (last >= 0) tma::mbar_wait(&bar[last % NS], (last / NS) & 1, tma::kWaitLimit);
            atomicOr(flag, 2);
        }
    } else {
        tc::fence_after();
        // element (mm, n) of the tile: alpha, beta C, bias, activation, store
        auto finish = [&](int mm, int n, float acc) {
            const long long nn = gx.nc && n >= gx.nc ? gx.scn1 + (n - gx.nc) * g.scn : n * g.scn;
            const long long at = (long long)b * g.scb + s_cr[mm - m0] + nn;
            float *cp = g.C + at;
            float *pp = g.C_pre ? g.C_pre + at : nullptr;
            float v = g.alpha * acc;
            if (g.ksplit > 1) {
                if (nc > 0) atomicAdd(cp, v);
                return;
            }
            if (g.beta != 0.0f) v = fmaf(g.beta, *cp, v);
            if (g.bias_mode == 1) v += g.bias[n];
            else if (g.bias_mode == 2) v += g.bias[mm];
            if (g.act == 1) {
                if (pp) *pp = v;
                v = gelu_exact(v);
            } else if (g.act == 2) {
                v *= gelu_grad(*pp);
            }
            *cp = v;
        };
        // Thread `lane` of a warp holds row warp * 32 + lane of the tile.  With
        // the columns of C contiguous (scn == 1) each warp transposes its
        // 32 x 32 block through shared memory (the stage buffers, free now
        // that every product has completed) so that a warp's stores cover 32
        // consecutive columns of one row; otherwise (rows contiguous) it
        // stores straight from the accumulator row.
        const bool by_rows = g.scn == 1 && g.ksplit == 1;
        // A plain product is stored without the choices of finish(): 32 copies of
        // those do not fit the instruction cache (4.6 of 12 cycles between a
        // warp's instructions in the inverse y product were spent on it).
        const bool plain = g.alpha == 1.0f && g.ksplit == 1 && g.beta == 0.0f && g.bias_mode == 0 &&
                           g.act == 0;
        float *wbuf = reinterpret_cast<float *>(sm) + warp * (32 * 33);
        const int m = m0 + warp * 32 + lane;
#pragma unroll 1
        for (int c0 = 0; c0 < BN; c0 += 32) {
            __syncwarp();                   // the tensor-memory load is warp-wide
            float r[32];
            if (nc > 0) {
                tc::ld32(tbase + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, r);
                tc::wait_ld();
            } else {
#pragma unroll
                for (int i = 0; i < 32; ++i) r[i] = 0.0f;
            }
            if (by_rows) {
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 32; ++i) wbuf[lane * 33 + i] = r[i];
                __syncwarp();
                const int n = n0 + c0 + lane;
                if (plain) {
                    float *cp = g.C + (long long)b * g.scb +
                                (gx.nc && n >= gx.nc ? gx.scn1 + (n - gx.nc) : n);
                    if (n < g.N)
#pragma unroll 4
                        for (int i = 0; i < min(32, g.M - m0 - warp * 32); ++i)
                            cp[s_cr[warp * 32 + i]] = wbuf[i * 33 + lane];
                    continue;
                }
#pragma unroll 1
                for (int i = 0; i < 32; ++i) {
                    const int mm = m0 + warp * 32 + i;
                    if (mm < g.M && n < g.N) finish(mm, n, wbuf[i * 33 + lane]);
                }
            } else if (plain) {
                if (m >= g.M) continue;
                int n = n0 + c0;
                float *cp = g.C + (long long)b * g.scb + s_cr[m - m0];
                float *at = cp + (gx.nc && n >= gx.nc ? gx.scn1 + (n - gx.nc) * g.scn : n * g.scn);
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    if (n < g.N) *at = r[i];
                    ++n;
                    at = gx.nc && n == gx.nc ? cp + gx.scn1 : at + g.scn;
                }
            } else {
                if (m >= g.M) continue;
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const int n = n0 + c0 + i;
                    if (n < g.N) finish(m, n, r[i]);
                }
            }
        }
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::dealloc(tbase, BN);
}

template <int BN, int NS>
cudaError_t launch_gemm_ns(const GemmX &x, int *flag, cudaStream_t s)
{
    const bvf_gemm &g = x.g;
    const dim3 grid((g.M + 127) / 128, (g.N + BN - 1) / BN, g.batch * g.ksplit);
    // the shared-memory limit is raised once per process, so that later
    // launches make no other runtime call (a forward can be recorded in a graph)
    static std::atomic<int> raised{0};
    if (!raised.load(std::memory_order_acquire)) {
        const cudaError_t e = cudaFuncSetAttribute(
            k_gemm_bf16<BN, NS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
            GemmLayout<BN, NS>::bytes);
        if (e != cudaSuccess) return e;
        raised.store(1, std::memory_order_release);
    }
    return launch_pdl(k_gemm_bf16<BN, NS>, grid, 128, GemmLayout<BN, NS>::bytes, s, x, flag);
}

// one stage when the product is a single K chunk
template <int BN>
cudaError_t launch_gemm_t(const GemmX &x, int *flag, cudaStream_t s)
{
    const int per_split = ((x.g.K + GK - 1) / GK + x.g.ksplit - 1) / x.g.ksplit;
    return per_split <= 1 ? launch_gemm_ns<BN, 1>(x, flag, s) : launch_gemm_ns<BN, 2>(x, flag, s);
}

}  // namespace

// BN: the smallest tile width of 32, 64, 128, 256 that holds N (256 beyond),
// at most 64 for a single-chunk product
cudaError_t launch_gemm_bf16(const GemmX &gx, int *flag, cudaStream_t s)
{
    GemmX x = gx;
    const bvf_gemm &g = x.g;
    auto al4 = [](long long v) { return v % 4 == 0; };
    auto al16 = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
    x.vec = (g.sak == 1 && g.K % 4 == 0 && al16(g.A) && al4(g.sam) && al4(g.sab) && al4(x.sam1) &&
             al4(x.sam2) && al4(x.ka) && al4(x.sak1))
                ? 1
                : 0;
    if (g.sbk == 1 && g.K % 4 == 0 && al16(g.B) && al4(g.sbn) && al4(g.sbb)) x.vec |= 2;
    if (g.N <= 32) return launch_gemm_t<32>(x, flag, s);
    // a single-chunk product restages its small A tile per N tile but keeps
    // 64 TMEM columns per block, so up to 8 blocks share an SM's 512
    const int per_split = ((g.K + GK - 1) / GK + g.ksplit - 1) / g.ksplit;
    if (g.N <= 64 || per_split <= 1) return launch_gemm_t<64>(x, flag, s);
    if (g.N <= 128) return launch_gemm_t<128>(x, flag, s);
    return launch_gemm_t<256>(x, flag, s);
}

}  // namespace bvf

extern "C" int bvf_gemm_bf16(const bvf_gemm *g, int *d_flag, void *stream)
{
    if (!g || !g->A || !g->B || !g->C || !d_flag || g->M < 1 || g->N < 1 || g->K < 0 ||
        g->batch < 1 || g->ksplit < 1 || g->batch * g->ksplit > 65535 ||
        (g->bias_mode != 0 && !g->bias) || g->bias_mode < 0 || g->bias_mode > 2 || g->act < 0 ||
        g->act > 2 || (g->act == 2 && !g->C_pre) ||
        (g->ksplit > 1 && (g->bias_mode != 0 || g->act != 0 || g->beta != 1.0f))) {
        bvf::set_context_free_error("bvf_gemm_bf16: bad argument");
        return BVF_E_ARG;
    }
    bvf::GemmX x;
    x.g = *g;
    const cudaError_t e = bvf::launch_gemm_bf16(x, d_flag, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) {
        bvf::set_context_free_error(cudaGetErrorString(e));
        return BVF_E_CUDA;
    }
    return BVF_OK;
}
