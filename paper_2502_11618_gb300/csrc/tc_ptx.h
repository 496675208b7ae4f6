// PTX wrappers and the unrolled MMA issue of one pipeline stage, shared by the tensor-core
// convolutions (conv_tc.cu, conv_split.cu).
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include "lnr_internal.h"

namespace lnr {
namespace {

constexpr long long kWaitCycles = 4000000000ll;  // ~2 s at 2 GHz
constexpr long long kStallWaitCycles = 2000000ll;  // ~1 ms: the timeout tests' wait
constexpr int kMmaWarps = 4;
constexpr int kHaloW = 130;  // staged pixels per halo row

// ------------------------------------------------------------- PTX wrappers ----

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// One bounded try: the thread may sleep in the barrier until the phase completes, for at
// most the suspend-time hint (10 ms), instead of spinning and taking issue slots from the
// epilogue warps of its scheduler.
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(10000000u)
        : "memory");
    return ok != 0;
}
// Bounded wait for the phase of parity `parity`: false after `limit` cycles (~2 s by default).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, long long limit = kWaitCycles) {
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try(bar, parity))
        if (clock64() - t0 > limit) return false;
    return true;
}

__device__ __forceinline__ void tma_2d(uint32_t dst, const CUtensorMap* m, uint32_t bar, int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"((uint64_t)m), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma_4d(uint32_t dst, const CUtensorMap* m, uint32_t bar, int c0, int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
        "l"((uint64_t)m), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma_5d(uint32_t dst, const CUtensorMap* m, uint32_t bar, int c0, int c1, int c2, int c3,
                                       int c4) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(dst),
        "l"((uint64_t)m), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void mma_fp8(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
template <bool IN8>
__device__ __forceinline__ void mma_op(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    if (IN8) mma_fp8(d, a, b, idesc, acc);
    else mma_bf16(d, a, b, idesc, acc);
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// 16 consecutive FP32 columns of this warp's 32 TMEM lanes (one lane per thread).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// UMMA shared-memory descriptor of a K-major, swizzled operand tile.
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t sbo, uint32_t swz) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(sbo >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)swz << 61);
}

__device__ __forceinline__ void named_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// n contiguous bytes into shared memory.  A TMA box moves about one of its rows per cycle,
// whatever their length: rows of 32 bytes come at 25 bytes per cycle and SM, rows of 64 at 50
// (measured), a contiguous copy at the L2's rate.  Weights are therefore laid out as shared
// memory holds them, swizzle included.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t n, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(n), "r"(bar)
                 : "memory");
}

// 32 bytes to a 32-byte-aligned global address in one store.
__device__ __forceinline__ void st_32b(void* dst, uint4 a, uint4 b) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(a.x), "r"(a.y), "r"(a.z),
                 "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
                 : "memory");
}

// 16 TMEM columns of this warp's lanes into r without waiting; tmem_wait16 completes it.
__device__ __forceinline__ void tmem_ld16_async(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
// Waits for every TMEM load this thread issued; r is threaded through so that no use of
// it can be scheduled before the wait.
__device__ __forceinline__ void tmem_wait16(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
}

// High bits of a swizzled K-major UMMA descriptor (everything but the start address).
__device__ __forceinline__ uint64_t sdesc_hi(uint32_t sbo, uint32_t swz) {
    return ((uint64_t)1 << 16) | ((uint64_t)(sbo >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)swz << 61);
}

// ---- MMA issue of one pipeline stage, fully unrolled ----
//
// One thread issues about one tcgen05.mma per 50-110 cycles; loop control and descriptor
// arithmetic with run-time bounds made that several times slower.  The issue sequence of a
// stage is therefore unrolled at compile time over taps, K steps (NK MMAs of 32 bytes of
// K) and the issuer's rows / units, so that every descriptor is a per-stage base plus a
// constant.

// Work split of a tile among its MMA-issuing threads: standard tiles give each of
// issuers(R) threads consecutive output rows; parity tiles give each of up to MAXI threads
// consecutive (row, y class) units.
template <int R, int PAR, int MAXI = kMmaWarps>
struct IssueSplit {
    static constexpr int NY = PAR == 4 ? 2 : 1;
    static constexpr int units = PAR == 0 ? R : NY * R;
    static constexpr int issuers = PAR == 0 ? (R >= 2 && MAXI >= 2 ? 2 : 1) : (units < MAXI ? units : MAXI);
    static constexpr int per = units / issuers;
};

// Staged rows of an operand: bytes per pixel, bytes of one x-parity plane (skip operand of
// the decoder's concat convs), UMMA swizzle type.
struct StageGeom {
    uint32_t pitch, plane, swz;
};

struct IssueCtx {
    int g;           // issuer index
    int px, py;      // parity class of the tile (PAR 1 and 2)
    uint32_t N;      // output channels
    uint32_t idesc;  // instruction descriptor for N columns
};

__device__ __forceinline__ uint32_t idesc_n(uint32_t idesc, uint32_t n) {
    return (idesc & ~(0x3Fu << 17)) | ((n >> 3) << 17);
}

// COARSE_FIRST: a stage of the nearest-upsampled operand may be a tile's first (`first`).
template <int R, int PAR, bool IN8, int NK, int MAXI = kMmaWarps, bool COARSE_FIRST = false>
__device__ __forceinline__ void issue_stage(const IssueCtx& q, int sg, uint32_t a0, uint32_t b0, const StageGeom& s,
                                            uint32_t d0, bool first) {
    using Sp = IssueSplit<R, PAR, MAXI>;
    constexpr int PER = Sp::per;
    const uint32_t N = q.N;
    const uint32_t pitch16 = s.pitch >> 4, row16 = kHaloW * pitch16, btap = N * pitch16;
    const uint64_t hi = sdesc_hi(8 * s.pitch, s.swz);
    if (PAR == 0) {
        // Halo row h shifted by kx feeds output rows r = h - ky, ky = 0..2; the rows of one
        // halo row go into one MMA (accumulators adjacent in TMEM, weight blocks [kx][ky =
        // 2,1,0] adjacent in shared memory, N = rows * Cout <= 256).  In the stage's first
        // (kx, k) step every row is first touched alone (h = r), zeroing it on a tile's
        // first chunk, and the rest of that step covers h - r = 1, 2.
        const uint32_t d = d0 + (uint32_t)(q.g * PER) * N;
        const uint32_t a = a0 + (uint32_t)(q.g * PER) * row16;
        const uint32_t acc0 = first ? 0u : 1u;
#pragma unroll
        for (int kx = 0; kx < 3; ++kx)
#pragma unroll
            for (int k = 0; k < NK; ++k) {
                const uint32_t ak = a + (uint32_t)kx * pitch16 + 2 * k, bk = b0 + 2 * k;
                if (kx == 0 && k == 0) {
#pragma unroll
                    for (int r = 0; r < PER; ++r)
                        mma_op<IN8>(d + (uint32_t)r * N, hi | (uint64_t)(ak + (uint32_t)r * row16), hi | (uint64_t)(bk + 2 * btap),
                                    q.idesc, acc0);
#pragma unroll
                    for (int h = 1; h < PER + 2; ++h) {
                        const int rlo = h - 2 > 0 ? h - 2 : 0, rhi = h - 1 < PER - 1 ? h - 1 : PER - 1;
                        const int blk = 2 - (h - rlo);
                        mma_op<IN8>(d + (uint32_t)rlo * N, hi | (uint64_t)(ak + (uint32_t)h * row16),
                                    hi | (uint64_t)(bk + (uint32_t)blk * btap), idesc_n(q.idesc, (uint32_t)(rhi - rlo + 1) * N), 1u);
                    }
                } else {
#pragma unroll
                    for (int h = 0; h < PER + 2; ++h) {
                        const int rlo = h - 2 > 0 ? h - 2 : 0, rhi = h < PER - 1 ? h : PER - 1;
                        const int blk = kx * 3 + 2 - (h - rlo);
                        mma_op<IN8>(d + (uint32_t)rlo * N, hi | (uint64_t)(ak + (uint32_t)h * row16),
                                    hi | (uint64_t)(bk + (uint32_t)blk * btap), idesc_n(q.idesc, (uint32_t)(rhi - rlo + 1) * N), 1u);
                    }
                }
            }
    } else {
        constexpr int NY = Sp::NY, NX = PAR >= 2 ? 2 : 1;
        const uint32_t plane16 = s.plane >> 4;
        const uint32_t id2 = idesc_n(q.idesc, 2 * N);
        const int u0 = q.g * PER;
        if (sg == 0) {
            // skip operand: the fine pixel of class cx at tap (ky, kx) is x-offset dxf = cx +
            // kx - 1 from 2X, i.e. plane dxf & 1, staged column 1 + (dxf >> 1).  With both x
            // classes in the tile, dxf = 0 and 1 serve both classes with weight blocks
            // (ky, dxf) and (ky, dxf + 1), adjacent in shared memory, into the unit's two
            // adjacent accumulators [cx = 1, cx = 0]: one MMA of 2N columns.
#pragma unroll
            for (int ky = 0; ky < 3; ++ky)
#pragma unroll
                for (int k = 0; k < NK; ++k)
#pragma unroll
                    for (int uu = 0; uu < PER; ++uu) {
                        const int u = u0 + uu;
                        const int r = u / NY, cy = PAR == 4 ? u - r * NY : q.py;
                        const uint32_t du = d0 + (uint32_t)(u * NX) * N;
                        const uint32_t ar = a0 + (uint32_t)((PAR == 4 ? cy : 0) + ky + 2 * r) * row16 + 2 * k;
                        auto A = [&](int dxf) {
                            return hi | (uint64_t)(ar + (uint32_t)(dxf & 1) * plane16 + (uint32_t)(1 + (dxf >> 1)) * pitch16);
                        };
                        const uint32_t bk = b0 + (uint32_t)(3 * ky) * btap + 2 * k;
                        const uint32_t init = (first && ky == 0 && k == 0) ? 0u : 1u;
                        if (NX == 2) {
                            mma_op<IN8>(du, A(0), hi | (uint64_t)bk, id2, init);
                            mma_op<IN8>(du, A(1), hi | (uint64_t)(bk + btap), id2, 1u);
                            mma_op<IN8>(du + N, A(-1), hi | (uint64_t)bk, q.idesc, 1u);
                            mma_op<IN8>(du, A(2), hi | (uint64_t)(bk + 2 * btap), q.idesc, 1u);
                        } else {
                            mma_op<IN8>(du, A(q.px - 1), hi | (uint64_t)bk, q.idesc, init);
                            mma_op<IN8>(du, A(q.px), hi | (uint64_t)(bk + btap), q.idesc, 1u);
                            mma_op<IN8>(du, A(q.px + 1), hi | (uint64_t)(bk + 2 * btap), q.idesc, 1u);
                        }
                    }
        } else {
            // nearest-upsampled operand: class (cx, cy) reads coarse rows cy - 1 + j (j = 0,
            // 1) and columns dxc in {cx - 1, cx}, each with the sum of the 3x3 taps that land
            // on that coarse pixel (blocks per (cy, j): [cx=1 dxc=+1][cx=1 dxc=0][cx=0 dxc=0]
            // [cx=0 dxc=-1]); dxc = 0 serves both x classes with one MMA of 2N columns.
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int k = 0; k < NK; ++k)
#pragma unroll
                    for (int uu = 0; uu < PER; ++uu) {
                        const int u = u0 + uu;
                        const int r = u / NY, cy = PAR == 4 ? u - r * NY : q.py;
                        const uint32_t du = d0 + (uint32_t)(u * NX) * N;
                        const uint32_t ar = a0 + (uint32_t)(r + cy + j) * row16 + 2 * k;
                        const uint32_t bj = b0 + (uint32_t)((PAR == 4 ? 8 * cy : 0) + 4 * j) * btap + 2 * k;
                        if (NX == 2 && COARSE_FIRST && first && j == 0 && k == 0) {
                            // the MMA of both classes starts the two accumulators
                            mma_op<IN8>(du, hi | (uint64_t)(ar + pitch16), hi | (uint64_t)(bj + btap), id2, 0u);
                            mma_op<IN8>(du, hi | (uint64_t)(ar + 2 * pitch16), hi | (uint64_t)bj, q.idesc, 1u);
                            mma_op<IN8>(du + N, hi | (uint64_t)ar, hi | (uint64_t)(bj + 3 * btap), q.idesc, 1u);
                        } else if (NX == 2) {
                            mma_op<IN8>(du, hi | (uint64_t)(ar + 2 * pitch16), hi | (uint64_t)bj, q.idesc, 1u);
                            mma_op<IN8>(du, hi | (uint64_t)(ar + pitch16), hi | (uint64_t)(bj + btap), id2, 1u);
                            mma_op<IN8>(du + N, hi | (uint64_t)ar, hi | (uint64_t)(bj + 3 * btap), q.idesc, 1u);
                        } else {
                            // one class: cx = 1 uses blocks 0, 1 at columns +1, 0; cx = 0 blocks 2, 3 at 0, -1
                            const uint32_t c1 = q.px ? 2 * pitch16 : pitch16;
                            const uint32_t bb = bj + (q.px ? 0u : 2 * btap);
                            mma_op<IN8>(du, hi | (uint64_t)(ar + c1), hi | (uint64_t)bb, q.idesc, 1u);
                            mma_op<IN8>(du, hi | (uint64_t)(ar + c1 - pitch16), hi | (uint64_t)(bb + btap), q.idesc, 1u);
                        }
                    }
        }
    }
}

// ------------------------------------------------------------------ host side ----

// cuTensorMapEncodeTiled through the runtime's driver entry-point lookup, so that the
// library links no driver library and loads on machines without one.
static CUresult encode_tiled(CUtensorMap* m, CUtensorMapDataType dt, cuuint32_t rank, void* addr, const cuuint64_t* dims,
                             const cuuint64_t* strides, const cuuint32_t* box, const cuuint32_t* es,
                             CUtensorMapInterleave il, CUtensorMapSwizzle sw, CUtensorMapL2promotion l2,
                             CUtensorMapFloatOOBfill oob) {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    }();
    if (!fn) return CUDA_ERROR_NOT_SUPPORTED;
    return fn(m, dt, rank, addr, dims, strides, box, es, il, sw, l2, oob);
}

// Byte `off` of a block of rows of `pitch` bytes (32, 64 or 128) where the TMA and UMMA swizzle
// of that row length puts it: the 16-byte chunk index XOR address bits 7 and up.
inline uint32_t swizzled(uint32_t off, uint32_t pitch) {
    const uint32_t mask = pitch == 128 ? 7u : pitch == 64 ? 3u : 1u;
    return off ^ (((off >> 7) & mask) << 4);
}

inline CUtensorMapSwizzle swizzle_pitch(uint32_t pitch) {
    return pitch == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : pitch == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
}

inline uint32_t align_up(uint32_t v, uint32_t a) { return (v + a - 1) / a * a; }

}  // namespace
}  // namespace lnr
