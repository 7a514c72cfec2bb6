// Forward x transform of the surrogate's volumes, D = v T^T over 128-row
// tiles (tcgen05), for rows that TMA can fetch:
//
//   - TMA keeps a ring of [128 rows][32 x] boxes (128-byte swizzle) in flight,
//     so the bytes on their way do not depend on registers or on how far the
//     compiler lets loads run ahead;
//   - each thread reads 16 values of its row (conflict-free through the
//     swizzle), splits them into TF32 head and remainder, or rounds them to
//     BF16, and stores them to tensor memory, where the product takes its A
//     operand from: no second pass of A through shared memory and no proxy
//     fence;
//   - products run two chunks behind the staging, and a tile's results are
//     written behind the wait that frees its last chunk's A buffer.
//
// Per K step the split takes two products: A_hi [T_hi | T_lo] (T_lo lies right
// behind T_hi, one operand of 2 NB rows) and A_lo T_hi into the second half;
// the halves are added when they are read.
//
// What it replaces staged A through registers and shared memory in chunks of
// 16: 475 us a layer at 240 x 240 x 200, width 32, m = 13 (FP32 path), and the
// general product, 490 us (BF16 path), for 1.47 GB read (217 us at 6.8 TB/s).
// Now 298 and 272 us (FP32, BF16), and 42 instead of 112 at 64 x 64 x 96, batch
// 4.  Loading four chunks ahead in registers instead gave nothing (479 us): what
// bound it was the round trip of each chunk through the barrier, and shared
// memory twice.
//
// Waits are bounded: a block whose wait runs out issues nothing more, waits
// (bounded) for its copies and products in flight, frees its tensor memory,
// sets bit 2 of the flag and ends.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>

#include "bvf_internal.cuh"
#include "bvf_tc.cuh"
#include "bvf_tma.cuh"
#include "bvf_xfwd.cuh"

namespace bvf {

namespace {

constexpr int kXc = 32;                        // x per chunk: one 128-byte swizzle row
constexpr int kSlot = 128 * kXc * 4;
constexpr int kSmemCap = 200 * 1024;

struct XfLayout {
    int nch, nxp, slots, sB, bar, tmem, bytes;
    __host__ __device__ XfLayout(bool tf, int nb, int nx, int slots_) : slots(slots_)
    {
        // two chunks at least: a tile's accumulator is read before the next but
        // one tile's first product
        nch = nx <= kXc ? 2 : (nx + kXc - 1) / kXc;
        nxp = nch * kXc;
        sB = slots * kSlot;
        bar = sB + (tf ? 2 * nb * nxp * 4 : nb * nxp * 2);
        tmem = bar + (slots + 2) * 8;
        bytes = tmem + 16;
    }
};

// the deepest ring that lets two blocks share an SM, or, where T is too
// large for that, the deepest that fits one
int pick_slots(bool tf, int nb, int nx)
{
    const int half = (227 * 1024 - 2 * 1024) / 2;
    for (int s = 5; s >= 3; --s)
        if (XfLayout(tf, nb, nx, s).bytes <= half) return s;
    for (int s = 6; s >= 3; --s)
        if (XfLayout(tf, nb, nx, s).bytes <= kSmemCap) return s;
    return 0;
}

__device__ __forceinline__ void load2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%2, %3}], [%4];" ::"r"(tma::saddr(dst)),
                 "l"(map), "r"(x), "r"(y), "r"(tma::saddr(bar))
                 : "memory");
}

template <bool TF, int NB>      // NB: T rows, 16 or 32
__global__ void __launch_bounds__(256, 2)
    k_xfwd(const __grid_constant__ CUtensorMap map, const __grid_constant__ XfwdArgs q, int slots)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    const XfLayout L(TF, NB, q.nx, slots);
    const int nx = q.nx, m = q.m, nch = L.nch, nxp = L.nxp;
    unsigned char *sB = sm + L.sB;
    uint64_t *full = reinterpret_cast<uint64_t *>(sm + L.bar), *done = full + slots;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(sm + L.tmem);
    const int tid = threadIdx.x, warp = tid >> 5, half = tid >> 7;
    constexpr int SET = TF ? 2 * NB : NB;            // accumulator columns of a tile
    constexpr int ABUF = TF ? 2 * kXc : kXc / 2;     // A columns of a chunk
    constexpr int NEED = 2 * (SET + ABUF), NCOLS = NEED <= 64 ? 64 : (NEED <= 128 ? 128 : 256);
    // T, resident, K-major
    if (TF) {
        for (int e = tid; e < NB * nxp; e += 256) {
            const int j = e / nxp, x = e - j * nxp;
            float val = 0.0f;
            if (j < 2 * m && x < nx) {
                const float2 c = q.tx[(long long)(j >> 1) * nx + x];
                val = (j & 1) ? c.y : c.x;
            }
            const uint32_t h = __float_as_uint(val) & 0xFFFFE000u, off = tc::kmaj_off(j, x, nxp);
            *reinterpret_cast<uint32_t *>(sB + off) = h;
            *reinterpret_cast<uint32_t *>(sB + NB * nxp * 4 + off) =
                __float_as_uint(val - __uint_as_float(h));
        }
    } else {
        for (int e = tid; e < NB * (nxp / 2); e += 256) {
            const int j = e / (nxp / 2), x = 2 * (e - j * (nxp / 2));
            const float a = j < 2 * m && x < nx ? q.F[(long long)x * 2 * m + j] : 0.0f;
            const float b = j < 2 * m && x + 1 < nx ? q.F[(long long)(x + 1) * 2 * m + j] : 0.0f;
            *reinterpret_cast<uint32_t *>(sB + tc::kmaj_off16(j, x & ~7, nxp) + (x & 7) * 2) =
                tc::pack_bf16(a, b);
        }
    }
    if (tid == 0) {
        for (int i = 0; i < slots + 2; ++i) tma::mbar_init(full + i, 1);
        tma::mbar_init_fence();
    }
    if (warp == 0) {
        tc::alloc(tslot, NCOLS);
        tc::relinquish();
    }
    tma::fence_async_smem();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = *tslot, abase = tbase + 2 * SET;
    const uint32_t idesc = TF ? tc::idesc_tf32(128, NB) : tc::idesc_bf16(128, NB);
    const uint32_t idesc2 = TF ? tc::idesc_tf32(128, 2 * NB) : 0u;
    const uint32_t sbo = (uint32_t)(nxp / (TF ? 4 : 8)) * 128;
    const int row = 32 * (warp & 3) + (tid & 31);    // this thread's row of a tile
    const uint32_t lanes = (uint32_t)(32 * (warp & 3)) << 16;

    const int tiles = (int)((q.R + 127) / 128);
    const int my = (int)blockIdx.x < tiles ? (tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
    const int total = my * nch;
    int lk = 0, lch = 0, lslot = 0;                  // thread 0: next chunk to copy
    auto copy_next = [&]() {
        if (lk >= my) return;
        tma::mbar_expect_tx(full + lslot, kSlot);
        load2d(sm + lslot * kSlot, &map, lch * kXc, ((int)blockIdx.x + lk * (int)gridDim.x) * 128,
               full + lslot);
        if (++lch == nch) {
            lch = 0;
            ++lk;
        }
        if (++lslot == slots) lslot = 0;
    };
    tma::pdl_wait();
    tma::pdl_launch_next();
    if (tid == 0)
        for (int i = 0; i < slots; ++i) copy_next();
    int slot = 0, turn = 0;                          // ring position of chunk gc
    int sk = 0, sch = 0;                             // its tile of this block, its chunk
    int ek = 0, ech = 0;                             // of the chunk two behind
    int gc = 0;
    bool gave_up = false;
    for (; gc < total + 2; ++gc) {
        const int st = gc & 1;
        // the products that read this A buffer two chunks ago are done, and
        // this chunk has arrived
        bool ok = true;
        if (gc >= 2) ok = tma::mbar_wait(&done[st], ((gc - 2) >> 1) & 1, tma::kWaitLimit);
        if (gc < total) ok = tma::mbar_wait(&full[slot], turn & 1, tma::kWaitLimit) && ok;
        ok = __all_sync(0xffffffffu, ok);
        tc::fence_after();
        if (gc < total && ok) {
            const unsigned char *src = sm + slot * kSlot + row * 128;
            float v[16];
#pragma unroll
            for (int p = 0; p < 4; ++p)
                *reinterpret_cast<float4 *>(v + 4 * p) =
                    *reinterpret_cast<const float4 *>(src + (((4 * half + p) ^ (row & 7)) << 4));
            const uint32_t ta = abase + lanes + (uint32_t)(st * ABUF);
            if (TF) {
                uint32_t h[16], l[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    h[i] = __float_as_uint(v[i]) & 0xFFFFE000u;
                    l[i] = __float_as_uint(v[i] - __uint_as_float(h[i]));
                }
                tc::st16(ta + 16 * half, h);
                tc::st16(ta + 32 + 16 * half, l);
            } else {
                uint32_t u[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) u[i] = tc::pack_bf16(v[2 * i], v[2 * i + 1]);
                tc::st8(ta + 8 * half, u);
            }
            tc::wait_st();
        }
        tc::fence_before();
        if (__syncthreads_or(!ok)) {
            gave_up = true;
            break;
        }
        if (gc < total) {
            if (tid == 0) {
                const uint32_t ta = abase + (uint32_t)(st * ABUF);
                const uint32_t td = tbase + (uint32_t)(SET * (sk & 1));
                tc::fence_after();
                if (TF) {
#pragma unroll
                    for (int ks = 0; ks < kXc / 8; ++ks) {
                        const uint64_t b = tc::smem_desc(sB + (sch * (kXc / 8) + ks) * 256, 128, sbo);
                        tc::mma_ta(td, ta + 8 * ks, b, idesc2, sch > 0 || ks > 0);
                        tc::mma_ta(td + NB, ta + 32 + 8 * ks, b, idesc, 1);
                    }
                } else {
#pragma unroll
                    for (int ks = 0; ks < kXc / 16; ++ks)
                        tc::mma_f16_ta(td, ta + 8 * ks,
                                    tc::smem_desc(sB + (sch * (kXc / 16) + ks) * 256, 128, sbo),
                                    idesc, sch > 0 || ks > 0);
                }
                tc::commit(&done[st]);
                copy_next();                         // every thread has read this slot
            }
            if (++sch == nch) {
                sch = 0;
                ++sk;
            }
            if (++slot == slots) {
                slot = 0;
                ++turn;
            }
        }
        if (gc >= 2 && ++ech == nch) {               // a whole tile is done
            const long long i = ((long long)blockIdx.x + (long long)ek * gridDim.x) * 128 + row;
            const uint32_t td = tbase + lanes + (uint32_t)(SET * (ek & 1) + half * (NB / 2));
            ech = 0;
            ++ek;
#pragma unroll
            for (int c0 = 0; c0 < NB / 2; c0 += 8) {
                float r[8], r2[8];
                tc::ld8(td + (uint32_t)c0, r);
                if (TF) tc::ld8(td + (uint32_t)(NB + c0), r2);
                tc::wait_ld();
                if (i < q.R) {
                    const int j0 = half * (NB / 2) + c0;
                    if (TF) {
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (j0 / 2 + k < m)
                                q.out[i * m + j0 / 2 + k] = make_float2(
                                    r[2 * k] + r2[2 * k], -(r[2 * k + 1] + r2[2 * k + 1]));
                    } else {
                        const long long sl = i / q.ny;
                        float *o = q.outw + sl * (2LL * m * q.ny) + (i - sl * q.ny) +
                                   (long long)j0 * q.ny;
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            if (j0 + k < 2 * m) *o = r[k];
                            o += q.ny;
                        }
                    }
                }
                __syncwarp();            // the next tensor-memory load is warp-wide
            }
        }
        tc::fence_before();
    }
    // after a time-out: the copies and products in flight end first
    if (gave_up && tid == 0) {
        const int last = std::min(gc, total) - 1;
        if (last >= 0) tma::mbar_wait(&done[last & 1], (last >> 1) & 1, tma::kWaitLimit);
        for (int c = gc; c < std::min(total, gc + slots); ++c)
            tma::mbar_wait(&full[c % slots], (c / slots) & 1, tma::kWaitLimit);
        atomicOr(q.flag, 2);
    }
    tc::fence_after();
    __syncthreads();
    if (warp == 0) tc::dealloc(tbase, NCOLS);
}

bool encode_rows(CUtensorMap *map, const float *v, int nx, long long R)
{
    static const auto enc = []() -> PFN_cuTensorMapEncodeTiled_v12000 {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult r;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault,
                                             &r) == cudaSuccess &&
            r == cudaDriverEntryPointSuccess)
            return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
        return nullptr;
    }();
    if (!enc) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)nx, (cuuint64_t)R};
    const cuuint64_t strides[1] = {(cuuint64_t)nx * 4};
    const cuuint32_t box[2] = {kXc, 128}, estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float *>(v), dims, strides, box,
               estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <bool TF, int NB>
cudaError_t launch_k(const CUtensorMap &map, const XfwdArgs &q, cudaStream_t s)
{
    static std::atomic<int> raised{0};
    if (!raised.load(std::memory_order_acquire)) {
        const cudaError_t e = cudaFuncSetAttribute(
            k_xfwd<TF, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
        if (e != cudaSuccess) return e;
        raised.store(1, std::memory_order_release);
    }
    const int slots = pick_slots(TF, NB, q.nx);
    const XfLayout L(TF, NB, q.nx, slots);
    const long long tiles = (q.R + 127) / 128;
    const int per = 2 * (L.bytes + 1024) <= 228 * 1024 ? 2 : 1;
    const int grid = (int)std::min<long long>(tiles, (long long)q.n_sm * per);
    return launch_pdl(k_xfwd<TF, NB>, grid, 256, L.bytes, s, map, q, slots);
}

}  // namespace

bool xfwd_fits(bool tf32, const float *v, long long R, int nx, int m)
{
    return nx >= kXc && nx % 4 == 0 && reinterpret_cast<uintptr_t>(v) % 16 == 0 && 2 * m <= 32 &&
           R < (1LL << 31) - 128 && pick_slots(tf32, 2 * m <= 16 ? 16 : 32, nx) > 0;
}

cudaError_t launch_xfwd(bool tf32, const XfwdArgs &q, cudaStream_t s)
{
    CUtensorMap map;
    if (!encode_rows(&map, q.v, q.nx, q.R)) return cudaErrorNotSupported;
    if (tf32)
        return 2 * q.m <= 16 ? launch_k<true, 16>(map, q, s) : launch_k<true, 32>(map, q, s);
    return 2 * q.m <= 16 ? launch_k<false, 16>(map, q, s) : launch_k<false, 32>(map, q, s);
}

}  // namespace bvf
