// Weight and bias gradients of a channel mix (BF16 path, training) in one pass
// over the volumes:
//   G[o][c] += sum_{b, p} bf16(d[b][o][p]) bf16(x[b][c][p])
//   g[o]    += sum_{b, p} d[b][o][p]                        (when asked)
//
// A contraction over millions of points into a few small tiles, so bound by
// reading d and x once (402 MB, 59 us at 6.8 TB/s, for 32 x 32 channels at 64 x
// 64 x 96, batch 4).  Blocks take 64-point chunks of the whole batch in turn, so
// that together they read one stretch of each row at a time; a chunk's rows (o
// of d, then c of x) are loaded one or two chunks ahead, 32 bytes a thread and
// row piece, summed for the bias, rounded to BF16 and written to one of two
// swizzled stages, and only rows that exist are staged: the rows up to the
// product's 128 stay zero from the start.  The accumulator stays in tensor
// memory until the block's last chunk and is then added to G.
// As general products (one 128-row tile staged per chunk with its zero rows,
// loads waited for chunk by chunk) and separate sums the layer's pair took 212
// and 35 us, the hidden layer's 264 and 113; now 75 and 139 (155 and 158 with a
// run of chunks per block, one chunk ahead, and G added to value by value).
//
// Waits are bounded as in the other tensor-core kernels.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

#include "bvf_fno_bf16.cuh"
#include "bvf_tc.cuh"
#include "bvf_tma.cuh"

namespace bvf {

namespace {

constexpr int kWgK = 64;                 // points per chunk: 128 bytes of BF16

struct WgLayout {
    int CP, ncols, stage, bar, tmem, bytes;
    __host__ __device__ explicit WgLayout(int C)
    {
        CP = (C + 15) & ~15;
        ncols = 32;
        while (ncols < CP) ncols *= 2;
        // 8-row groups of 1 KB: d's 128 rows, then x's
        stage = 128 * 128 + CP * 128;
        bar = 2 * stage;
        tmem = bar + 16;
        bytes = tmem + 16;
    }
};

// ITEMS: row pieces (8 points) of a chunk per thread
template <int ITEMS>
__global__ void __launch_bounds__(256, ITEMS <= 2 ? 4 : 2)
    k_wgrad_bf16(const __grid_constant__ WgradBf16 q)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    const WgLayout L(q.C);
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + L.bar);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(sm + L.tmem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int o0 = blockIdx.y * 128, no = min(128, q.O - o0), pieces = (no + q.C) * 8;
    const int N = q.N;
    for (int e = tid; e < 2 * L.stage / 16; e += 256)
        reinterpret_cast<uint4 *>(sm)[e] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) {
        tma::mbar_init(&bar[0], 1);
        tma::mbar_init(&bar[1], 1);
        tma::mbar_init_fence();
    }
    if (warp == 0) {
        tc::alloc(tslot, L.ncols);
        tc::relinquish();
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = *tslot;
    const uint32_t idesc = tc::idesc_bf16(128, L.CP);
    // this block's chunks: every gridDim.x-th of the batch's, so that the
    // blocks together read one stretch of each row at a time
    const int per = (N + kWgK - 1) / kWgK, all = per * q.B;
    const int n = (int)blockIdx.x < all ? (all - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
    int lb = blockIdx.x / per, lc = blockIdx.x - lb * per;                  // next chunk to load
    constexpr int AHEAD = ITEMS <= 2 ? 2 : 1;
    float4 v[AHEAD][ITEMS][2];
    float acc[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) acc[i] = 0.0f;
    auto load_next = [&](float4 (&v)[ITEMS][2]) {
        if (lb >= q.B) return;
        const float *d = q.d + ((long long)lb * q.O + o0) * N + lc * kWgK;
        const float *x = q.x + (long long)lb * q.C * N + lc * kWgK;
        const int left = N - lc * kWgK;              // a multiple of 4
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const int e = tid + 256 * i, r = e >> 3, k = (e & 7) * 8;
            const float *src = (r < no ? d + (long long)r * N : x + (long long)(r - no) * N) + k;
#pragma unroll
            for (int h = 0; h < 2; ++h)
                v[i][h] = e < pieces && k + 4 * h < left
                              ? tma::ld_stream(reinterpret_cast<const float4 *>(src + 4 * h))
                              : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        for (lc += gridDim.x; lc >= per; lc -= per) ++lb;
    };
    tma::pdl_wait();
    tma::pdl_launch_next();
#pragma unroll
    for (int u = 0; u < AHEAD; ++u) load_next(v[u]);
    bool gave_up = false;
    int c = 0;
    while (c < n && !gave_up) {
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
            if (c >= n) break;
            const int st = c & 1;
            unsigned char *sa = sm + st * L.stage, *sb = sa + 128 * 128;
            // the products that read this stage two chunks ago are done
            bool ok = true;
            if (c >= 2)
                ok = __all_sync(0xffffffffu,
                                tma::mbar_wait(&bar[st], ((c - 2) >> 1) & 1, tma::kWaitLimit));
            if (ok) {
#pragma unroll
                for (int i = 0; i < ITEMS; ++i) {
                    const int e = tid + 256 * i, r = e >> 3;
                    if (e >= pieces) continue;
                    const float4 a = v[u][i][0], b = v[u][i][1];
                    acc[i] += ((a.x + a.y) + (a.z + a.w)) + ((b.x + b.y) + (b.z + b.w));
                    unsigned char *dst = r < no ? sa + tc::sw128_off(r, e & 7) : sb + tc::sw128_off(r - no, e & 7);
                    *reinterpret_cast<uint4 *>(dst) =
                        make_uint4(tc::pack_bf16(a.x, a.y), tc::pack_bf16(a.z, a.w),
                                   tc::pack_bf16(b.x, b.y), tc::pack_bf16(b.z, b.w));
                }
            }
            load_next(v[u]);
            tma::fence_async_smem();
            tc::fence_before();
            if (__syncthreads_or(!ok)) {
                gave_up = true;
                break;
            }
            if (tid == 0) {
                tc::fence_after();
#pragma unroll
                for (int ks = 0; ks < kWgK / 16; ++ks)
                    tc::mma_f16(tbase, tc::smem_desc_sw(sa + 32 * ks, 1024, tc::kSwizzle128),
                                tc::smem_desc_sw(sb + 32 * ks, 1024, tc::kSwizzle128), idesc,
                                c > 0 || ks > 0);
                tc::commit(&bar[st]);
            }
            ++c;
        }
    }
    // the last commit covers every earlier product
    bool ready = !gave_up;
    if (c > 0) {
        const bool ok = tma::mbar_wait(&bar[(c - 1) & 1], ((c - 1) >> 1) & 1, tma::kWaitLimit);
        ready = __syncthreads_or(!ok) == 0 && ready;
    }
    tc::fence_after();
    if (!ready) {
        if (tid == 0) atomicOr(q.flag, 2);
    } else if (c > 0) {
        const int o = 32 * (warp & 3) + lane;
        // four columns an addition where rows of G start on 16 bytes
        const bool vec = q.C % 4 == 0 && (reinterpret_cast<uintptr_t>(q.G) & 15) == 0;
        for (int k0 = 16 * (warp >> 2); k0 < L.CP; k0 += 32) {
            float r[16];
            tc::ld16(tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)k0, r);
            tc::wait_ld();
            if (o < no) {
#pragma unroll
                for (int k = 0; k < 16; k += 4) {
                    float *at = q.G + (long long)(o0 + o) * q.C + k0 + k;
                    if (vec) {
                        if (k0 + k < q.C)
                            asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(at),
                                         "f"(r[k]), "f"(r[k + 1]), "f"(r[k + 2]), "f"(r[k + 3])
                                         : "memory");
                    } else {
#pragma unroll
                        for (int h = 0; h < 4; ++h)
                            if (k0 + k + h < q.C) atomicAdd(at + h, r[k + h]);
                    }
                }
            }
            __syncwarp();
        }
        if (q.g) {
            // eight neighbouring lanes hold the pieces of one row
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                float s = acc[i];
                for (int w = 4; w; w >>= 1) s += __shfl_xor_sync(0xffffffffu, s, w);
                const int r = (tid + 256 * i) >> 3;
                if ((tid & 7) == 0 && r < no) atomicAdd(q.g + o0 + r, s);
            }
        }
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::dealloc(tbase, L.ncols);
}

template <int ITEMS>
cudaError_t launch_items(const WgradBf16 &q, int n_sm, cudaStream_t s)
{
    const WgLayout L(q.C);
    static std::atomic<int> raised{0};
    if (!raised.load(std::memory_order_acquire)) {
        const cudaError_t e = cudaFuncSetAttribute(
            k_wgrad_bf16<ITEMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, WgLayout(256).bytes);
        if (e != cudaSuccess) return e;
        raised.store(1, std::memory_order_release);
    }
    const int per = std::max(1, std::min({ITEMS <= 2 ? 4 : 2, 512 / L.ncols,
                                          (227 * 1024) / (L.bytes + 1024)}));
    const int oy = (q.O + 127) / 128;
    // eight chunks a block at least, so that adding its tile to G stays small
    const long long chunks = (long long)((q.N + kWgK - 1) / kWgK) * q.B;
    const int grid = (int)std::max<long long>(
        1, std::min<long long>((chunks + 7) / 8, std::max(1, n_sm * per / oy)));
    return launch_pdl(k_wgrad_bf16<ITEMS>, dim3(grid, oy), 256, L.bytes, s, q);
}

}  // namespace

bool wgrad_fits(const WgradBf16 &q)
{
    auto al16 = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
    return q.N % 4 == 0 && q.C <= 256 && al16(q.d) && al16(q.x) && (std::min(q.O, 128) + q.C) <= 384;
}

cudaError_t launch_wgrad_bf16(const WgradBf16 &q, int n_sm, cudaStream_t s)
{
    const int rows = std::min(q.O, 128) + q.C;
    if (rows <= 64) return launch_items<2>(q, n_sm, s);
    if (rows <= 128) return launch_items<4>(q, n_sm, s);
    if (rows <= 192) return launch_items<6>(q, n_sm, s);
    return launch_items<12>(q, n_sm, s);
}

}  // namespace bvf
