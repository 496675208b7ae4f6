// U-Net 3x3 convolutions on the 5th-generation tensor cores (tcgen05 + TMEM), fed by TMA
// (Fig. 1; Sec. 3, "U-Net Reconstruction").
//
// Each convolution is an implicit GEMM: D[128 output pixels][Cout] += A[pixels][K] B[Cout][K]^T
// with K = 9 taps x input channels.  A tile of A is one TMA box of the NHWC activation
// tensor shifted by the tap; out-of-image rows and columns are zero-filled by TMA, which
// gives the convolution's zero padding for free.  Weights are K-major [Cout][tap][Cin].
//
// Fusions:
//  - encoder convs below the bottleneck also write the 2x2 max-pooled output (the tile is
//    2 rows x 64 pixels, so every pooling quad lies in one tile);
//  - the first decoder conv of each level reads the skip tensor and the nearest-2x-
//    upsampled deeper tensor directly, never materialising the concatenation: its output
//    tile is 128 pixels of one parity class (x mod 2, y mod 2), for which the upsampled
//    operand of every tap is a plain row of the coarse tensor and the skip operand a
//    stride-2 row of the fine one (a 5-D TMA view);
//  - the last decoder conv applies the 1x1 head and the sigmoid in its epilogue.
//
// Kernel structure (persistent, one CTA per SM, 6 warps):
//  warp 0   TMA producer: A and B tiles into an S-stage shared-memory ring;
//  warp 1   MMA issuer: tcgen05.mma kind::f16 (BF16 in, FP32 accumulate) into one of two
//           TMEM accumulators, tcgen05.commit to free ring stages and publish results;
//  warps 2-5 epilogue: tcgen05.ld, bias, ReLU, BF16 store (+ pool / head).
// Every mbarrier wait is bounded (about 2 s); a wait that runs out sets an error word and
// the CTA drains its copies, frees its TMEM and exits.
#include <cuda_fp8.h>

#include <cstdlib>
#include <type_traits>
#include <cstring>

#include "tc_ptx.h"

namespace lnr {
namespace {

constexpr int kThreads = 192;
// halo kernel: producer warp, MMA-issuing warps (one per independent unit of a parity tile
// of the decoder's concat convs, at most kMmaWarps; two for standard tiles, whose rows split
// between two issuers), then EPI epilogue warps.  Each issuer owns disjoint accumulators.
// An issuing thread shares its scheduler with the epilogue warps of its TMEM lane quarter,
// so small-N convolutions, whose MMAs are short, are issued from several threads.
__host__ __device__ constexpr int halo_mma_warps(int par, int r) {
    return par == 0 ? 2 : ((par == 4 ? 2 : 1) * r < kMmaWarps ? (par == 4 ? 2 : 1) * r : kMmaWarps);
}
// Epilogue warps, chosen per layer: 4 (one per TMEM lane quarter), 8 or 12 (two or three per
// quarter: more latency hiding for TMEM loads, stores and the fused head's dot products, at
// 128 registers per thread).  12 for standard tiles and for tiles of two parity classes and
// at most two rows, whose two issuers leave room for them.
__host__ __device__ constexpr int halo_threads(int par, int r, int epi) { return 32 * (1 + halo_mma_warps(par, r) + epi); }
constexpr int kXchStride = 33;                   // floats per row of the pooling exchange

struct Seg {
    CUtensorMap a;   // activation view of this K segment's source
    CUtensorMap b;   // weight view with box {kc, N}
    int kind;        // 0: same-resolution source (2x64 tiles); 1: skip, parity tiles; 2: coarse, parity tiles
    int kc;          // channels per K chunk: 16, 32 or 64
    int nchunk;      // chunks per tap
    int koff;        // K offset of the segment inside one tap
    uint32_t bytes;  // A + B bytes of one chunk
    uint32_t swz;    // UMMA layout type of the chunk (SW32 = 6, SW64 = 4, SW128 = 2)
    uint32_t sbo;    // bytes between 8-row core-matrix groups
};

struct Params {
    Seg seg[2];
    int nseg;
    int parity;       // 1: decoder parity tiles, 0: 2 x 64 pixel tiles
    int W, H, B, N, cin_pad;
    int tiles_x, tiles_y, ntiles;
    int stages;
    uint32_t stage_bytes, a_region, xch_bytes, tmem_cols, idesc;
    const float* bias;
    __nv_bfloat16* out;
    __nv_bfloat16* pool_out;
    const float* head_w;
    const float* head_b;
    float* head_out;
    int head_o;
    int* err;
};

struct TileCoord {
    int n, x0, y0;    // standard tiles: image, first column, first row
    int cx0, cy, px, py;  // parity tiles: first coarse column, coarse row, parity
};

__device__ __forceinline__ TileCoord decode(const Params& p, int t) {
    TileCoord c{};
    const int tx = t % p.tiles_x;
    int r = t / p.tiles_x;
    const int ty = r % p.tiles_y;
    r /= p.tiles_y;
    if (p.parity) {
        const int par = r & 3;
        c.n = r >> 2;
        c.px = par & 1;
        c.py = par >> 1;
        c.cx0 = tx * 128;
        c.cy = ty;
    } else {
        c.n = r;
        c.x0 = tx * 64;
        c.y0 = ty * 2;
    }
    return c;
}

__global__ void __launch_bounds__(kThreads, 1) k_conv_tc(const __grid_constant__ Params p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* const gbase = smem_raw + (base - raw);
    const int S = p.stages;
    float* xch = reinterpret_cast<float*>(gbase + S * p.stage_bytes);
    const uint32_t bars = base + S * p.stage_bytes + p.xch_bytes;
    auto full = [&](int s) { return bars + 8u * s; };
    auto empty = [&](int s) { return bars + 8u * (S + s); };
    auto tfull = [&](int b) { return bars + 8u * (2 * S + b); };
    auto tempty = [&](int b) { return bars + 8u * (2 * S + 2 + b); };
    const uint32_t drain = bars + 8u * (2 * S + 4);
    const uint32_t tslot = bars + 8u * (2 * S + 5);
    volatile int* flag = reinterpret_cast<volatile int*>(gbase + (tslot - base) + 4);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(tfull(b), 1);
            mbar_init(tempty(b), 4);
        }
        mbar_init(drain, 1);
        *flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(tslot, p.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(gbase + (tslot - base));

    if (warp == 0 && lane == 0) {
        // ------------------------------------------------------------ producer --
        int use = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
            const TileCoord c = decode(p, t);
            for (int tap = 0; tap < 9 && ok; ++tap) {
                const int ky = tap / 3, kx = tap % 3;
                for (int sg = 0; sg < p.nseg && ok; ++sg) {
                    const Seg& s = p.seg[sg];
                    for (int cc = 0; cc < s.nchunk; ++cc) {
                        const int st = use % S;
                        if (!mbar_wait(empty(st), ((use / S) & 1) ^ 1)) { ok = false; break; }
                        const uint32_t a_dst = base + st * p.stage_bytes, b_dst = a_dst + p.a_region;
                        mbar_expect_tx(full(st), s.bytes);
                        const int cb = cc * s.kc;
                        if (s.kind == 0) {
                            tma_4d(a_dst, &s.a, full(st), cb, c.x0 + kx - 1, c.y0 + ky - 1, c.n);
                        } else if (s.kind == 1) {
                            const int dxf = c.px + kx - 1;
                            tma_5d(a_dst, &s.a, full(st), cb, dxf & 1, c.cx0 + (dxf >> 1), 2 * c.cy + c.py + ky - 1, c.n);
                        } else {
                            tma_4d(a_dst, &s.a, full(st), cb, c.cx0 + ((c.px + kx - 1) >> 1), c.cy + ((c.py + ky - 1) >> 1),
                                   c.n);
                        }
                        tma_2d(b_dst, &s.b, full(st), tap * p.cin_pad + s.koff + cb, 0);
                        ++use;
                    }
                }
            }
        }
        if (!ok) atomicExch(p.err, 1);
        // no copy may still be in flight when the CTA exits
        for (int k = use > S ? use - S : 0; k < use; ++k) mbar_wait(full(k % S), (k / S) & 1);
    } else if (warp == 1 && lane == 0) {
        // ----------------------------------------------------------------- MMA --
        int use = 0, tcount = 0;
        bool ok = true, issued = false;
        for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x, ++tcount) {
            const int b = tcount & 1;
            if (!mbar_wait(tempty(b), ((tcount >> 1) & 1) ^ 1)) { ok = false; break; }
            tc_fence_after();
            const uint32_t d = tmem + (uint32_t)(b * p.N);
            uint32_t acc = 0;
            for (int tap = 0; tap < 9 && ok; ++tap)
                for (int sg = 0; sg < p.nseg && ok; ++sg) {
                    const Seg& s = p.seg[sg];
                    for (int cc = 0; cc < s.nchunk; ++cc) {
                        const int st = use % S;
                        if (!mbar_wait(full(st), (use / S) & 1)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t a_addr = base + st * p.stage_bytes, b_addr = a_addr + p.a_region;
                        for (int k = 0; k < s.kc / 16; ++k) {
                            mma_bf16(d, sdesc(a_addr + 32u * k, s.sbo, s.swz), sdesc(b_addr + 32u * k, s.sbo, s.swz),
                                     p.idesc, acc);
                            acc = 1;
                        }
                        issued = true;
                        mma_commit(empty(st));
                        ++use;
                    }
                }
            if (ok) mma_commit(tfull(b));
        }
        if (!ok) atomicExch(p.err, 2);
        if (issued) {  // every MMA issued has completed before TMEM is released
            mma_commit(drain);
            mbar_wait(drain, 0);
        }
    } else if (warp >= 2) {
        // ------------------------------------------------------------ epilogue --
        const int q = warp & 3;          // TMEM lane quarter this warp may access
        const int m = 32 * q + lane;     // tile row of this thread
        const bool leader = threadIdx.x == 64;
        const int Wh = p.W >> 1, Hh = p.H >> 1;
        int tcount = 0;
        for (int t = blockIdx.x; t < p.ntiles; t += gridDim.x, ++tcount) {
            const int b = tcount & 1;
            if (leader && !mbar_wait(tfull(b), (tcount >> 1) & 1)) *flag = 1;
            named_sync(1, 128);
            if (*flag) break;
            tc_fence_after();
            const TileCoord c = decode(p, t);
            int x, y;
            if (p.parity) {
                x = 2 * (c.cx0 + m) + c.px;
                y = 2 * c.cy + c.py;
            } else {
                x = c.x0 + (m & 63);
                y = c.y0 + (m >> 6);
            }
            const bool valid = x < p.W && y < p.H;
            const size_t pix = ((size_t)c.n * p.H + y) * p.W + x;
            float h[4] = {0.f, 0.f, 0.f, 0.f};
            const uint32_t trow = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * p.N);
            for (int c0 = 0; c0 < p.N; c0 += 16) {
                float v[16];
                tmem_ld16(trow + c0, v);
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] = fmaxf(v[j] + __ldg(p.bias + c0 + j), 0.f);
                if (p.head_out) {
                    for (int o = 0; o < p.head_o; ++o) {
                        float s = 0.f;
#pragma unroll
                        for (int j = 0; j < 16; ++j) s = fmaf(__ldg(p.head_w + o * p.N + c0 + j), v[j], s);
                        h[o] += s;
                    }
                } else if (valid) {
                    uint4 pk[2];
                    uint32_t* pw = reinterpret_cast<uint32_t*>(pk);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        __nv_bfloat162 b2 = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
                        pw[j] = *reinterpret_cast<uint32_t*>(&b2);
                    }
                    uint4* dst = reinterpret_cast<uint4*>(p.out + pix * p.N + c0);
                    dst[0] = pk[0];
                    dst[1] = pk[1];
                }
                if (p.pool_out) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) xch[m * kXchStride + j] = v[j];
                    named_sync(1, 128);
                    if (m < 64 && (m & 1) == 0 && valid) {
                        uint4 pk[2];
                        uint32_t* pw = reinterpret_cast<uint32_t*>(pk);
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            float a0 = fmaxf(fmaxf(xch[m * kXchStride + 2 * j], xch[(m + 1) * kXchStride + 2 * j]),
                                             fmaxf(xch[(m + 64) * kXchStride + 2 * j], xch[(m + 65) * kXchStride + 2 * j]));
                            float a1 = fmaxf(fmaxf(xch[m * kXchStride + 2 * j + 1], xch[(m + 1) * kXchStride + 2 * j + 1]),
                                             fmaxf(xch[(m + 64) * kXchStride + 2 * j + 1],
                                                   xch[(m + 65) * kXchStride + 2 * j + 1]));
                            __nv_bfloat162 b2 = __floats2bfloat162_rn(a0, a1);
                            pw[j] = *reinterpret_cast<uint32_t*>(&b2);
                        }
                        const size_t pp = ((size_t)c.n * Hh + (y >> 1)) * Wh + (x >> 1);
                        uint4* dst = reinterpret_cast<uint4*>(p.pool_out + pp * p.N + c0);
                        dst[0] = pk[0];
                        dst[1] = pk[1];
                    }
                    named_sync(1, 128);
                }
            }
            if (p.head_out && valid) {
                for (int o = 0; o < p.head_o; ++o) {
                    const float z = h[o] + __ldg(p.head_b + o);
                    p.head_out[pix * p.head_o + o] = 1.0f / (1.0f + expf(-z));
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(tempty(b));
        }
        if (leader && *flag) atomicExch(p.err, 3);
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, p.tmem_cols);
    }
}

// ================================================================ halo kernel ==
//
// The same convolution with the input staged ONCE per tile and K chunk: a tile is R output
// rows x 128 columns (or, for the decoder's first conv, R coarse rows x 128 coarse columns
// of one parity class).  For every K chunk of ck channels the producer loads the input
// halo -- R+2 rows x 130 pixels (or the parity-class rows) -- with one TMA box whose
// innermost extent is the whole chunk (32, 64 or 128 bytes per pixel, swizzled), plus the
// chunk's weights for all 9 taps.  The tensor cores apply the swizzle from absolute
// shared-memory address bits, as TMA does, so each tap is just the halo's start address
// shifted by whole pixels and rows: the 9 taps x R rows of MMAs all read the halo that was
// fetched once.  The R accumulators of a tile sit side by side in TMEM (R*N columns,
// double-buffered).  2x2 pooling needs no shared-memory exchange: a thread owns one column
// of R rows and its horizontal neighbour is the adjacent lane.

// Weights come as one contiguous copy per chunk, not as TMA boxes of 32- or 64-byte rows, and
// the upsampled operand of a single y class stages only the R + 1 rows that it reads: the 1080p
// decoder convs with 128 and 256 input channels were bound by TMA's row rate.  Eight 1080p
// views 4618 -> 4416 us, one 648 -> 594, four 720p views in FP8 1049 -> 947 (whole frames).

constexpr int kHaloMaxN = 256;  // output channels of one halo-kernel launch, at most

struct HSeg {
    CUtensorMap a;   // kind 0/2: 4-D {C, W, H, N}, box {ck, 130, rows, 1}; kind 1: 5-D, box {ck, 1, 130, rows, 1}
    const uint8_t* w;  // weights [chunk][block][N][ck], each chunk as shared memory holds it
    int kind;        // 0: same-resolution source; 1: skip (parity tiles); 2: coarse (parity tiles)
    uint32_t w_chunk;  // bytes of a chunk in memory (9 blocks, or 16 for the coarse operand)
    uint32_t w_bytes;  // bytes staged per chunk (coarse: all blocks for 4 classes, else the tile's y class's 8)
    uint32_t w_sel;    // offset of the second y class's blocks when only one's are staged, else 0
    int ck;          // channels per chunk (16, 32 or 64): 32, 64 or 128 bytes per pixel
    int rows;        // halo rows staged
    int nchunk;      // K chunks of this segment
    uint32_t pitch;  // bytes per staged pixel (= ck * 2)
    uint32_t plane;  // bytes of one staged plane (rows x 130 pixels, 1024-aligned)
    uint32_t a_bytes, b_off, bytes;  // A bytes per chunk, B offset in the stage, A + B bytes
    uint32_t swz;    // UMMA layout type (SW128 = 2, SW64 = 4, SW32 = 6)
};

struct HParams {
    HSeg seg[2];
    int nseg;
    int R, parity, W, H, B, N;  // parity: parity classes per tile (0 = standard tiles)
    int wmax;                   // standard tiles: output rows per MMA (N = wmax * Cout <= 256)
    int nmma;                   // MMA-issuing threads in use (<= kMmaWarps, <= accumulators per tile)
    int tiles_x, tiles_y, ntiles;
    int stages;
    uint32_t stage_bytes, tmem_cols, idesc;
    void* out;                  // NHWC output, BF16 or (out_fp8) E4M3
    void* pool_out;             // 2x2 max-pooled output, same type, or null
    int out_fp8, pool_fp8;      // output / pooled output stored as E4M3 (else BF16)
    float inv_out;              // E4M3 output: value * inv_out is stored
    float* head_out;
    int head_o;
    int* err;
    // TMA-store epilogue (ostage = 1): per epilogue warp a staging area of ost_warp bytes at
    // ost_off from the 1024-aligned base: (pool ? 2 : 1) rows of 32 pixels x N channels,
    // then (pool) 16 pooled pixels, every part 1024-aligned; rows split into boxes of
    // orow_b bytes (<= 128, swizzle mask omask), pooled rows into prow_b (pmask)
    CUtensorMap omap;    // output: 4-D {N, W, H, B} box {orow_b/e, 32, 1, 1}; parity: 5-D {N, 2, W/2, H, B}
    CUtensorMap pmap;    // pooled output: 4-D {N, W/2, H/2, B} box {prow_b/e, 16, 1, 1}
    int ostage;
    uint32_t stg_bytes;                             // epilogue staging bytes (TMA stores)
    int ost_nbuf;                                   // staging buffers per warp (1 or 2, used in turn)
    uint32_t ost_off, ost_warp, ost_unit, ost_row, ost_pool;  // offset, bytes per warp, per buffer, row part, pool part
    uint32_t orow_b, omask, prow_b, pmask;
    // Per-output-channel epilogue constants, read through the constant cache (the kernel's
    // parameter bank) rather than shared memory, whose bandwidth the MMAs' operand reads
    // already use up: bias, accumulator scale (E4M3 operands, else 1), and the fused head's
    // weights [4][N] (zero past head_o) followed by its 4 biases.
    // stall = 1 makes the MMA issuer first wait on a barrier that nothing arrives on, giving
    // up after kStallWaitCycles (the timeout test's switch); every other wait gives up after
    // kWaitCycles, so the stalled launch ends within a few seconds.
    int stall;
    int tbufs;  // TMEM accumulator buffers: 2 (the epilogue of a tile overlaps the next tile's
                // MMAs) or 1 (tiles of up to 512 accumulator columns; each weight stage feeds more MMAs)
    alignas(16) float cbias[kHaloMaxN];
    alignas(16) float cscale[kHaloMaxN];
    alignas(16) float chead[4 * kHaloMaxN + 4];
};

// 16 channels of one pixel as E4M3 of v * inv (16 bytes, saturating).
__device__ __forceinline__ void st_fp8x16(uint8_t* dst, const float* v, float inv) {
    uint4 pk;
    uint16_t* ph = reinterpret_cast<uint16_t*>(&pk);
#pragma unroll
    for (int j = 0; j < 8; ++j)
        ph[j] = __nv_cvt_float2_to_fp8x2(make_float2(v[2 * j] * inv, v[2 * j + 1] * inv), __NV_SATFINITE, __NV_E4M3);
    *reinterpret_cast<uint4*>(dst) = pk;
}

// ReLU of 16 values, rounded to BF16 and packed two per word (lower half the even element).
// The conversion applies the ReLU (cvt.rn.relu.bf16x2.f32): the same BF16 values as
// rounding fmaxf(v, 0), in 8 instructions instead of 16 + 8.
__device__ __forceinline__ void relu_bf16x16(const float* v, uint4 (&pk)[2]) {
    uint32_t* pw = reinterpret_cast<uint32_t*>(pk);
#pragma unroll
    for (int j = 0; j < 8; ++j) asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(pw[j]) : "f"(v[2 * j + 1]), "f"(v[2 * j]));
}
// Bias + ReLU of 16 FP32 accumulator columns as BF16 pairs; keep = false gives zeros.
__device__ __forceinline__ void bias_relu_bf16x16(const uint32_t (&u)[16], const float* bias, bool keep, uint4 (&pk)[2]) {
    float f[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) f[j] = __uint_as_float(u[j]) + bias[j];
    relu_bf16x16(f, pk);
    if (!keep) pk[0] = pk[1] = make_uint4(0u, 0u, 0u, 0u);
}
// 32 packed bytes to a 32-byte-aligned global address.
__device__ __forceinline__ void st_pk32(void* dst, const uint4 (&pk)[2]) { st_32b(dst, pk[0], pk[1]); }
// ReLU of 16 values, stored as 16 BF16 channels (32 bytes, 32-byte aligned).
__device__ __forceinline__ void st_relu_bf16x16(__nv_bfloat16* dst, const float* v) {
    uint4 pk[2];
    relu_bf16x16(v, pk);
    st_32b(dst, pk[0], pk[1]);
}
__device__ __forceinline__ void relu16(float (&f)[16]) {
#pragma unroll
    for (int j = 0; j < 16; ++j) f[j] = fmaxf(f[j], 0.f);
}

// 16 channels as E4M3 of v * inv (one 16-byte chunk, saturating).
__device__ __forceinline__ uint4 pack_fp8x16(const float* v, float inv) {
    uint4 pk;
    uint16_t* ph = reinterpret_cast<uint16_t*>(&pk);
#pragma unroll
    for (int j = 0; j < 8; ++j)
        ph[j] = __nv_cvt_float2_to_fp8x2(make_float2(v[2 * j] * inv, v[2 * j + 1] * inv), __NV_SATFINITE, __NV_E4M3);
    return pk;
}

// Packed FP32 pair (lo, hi) and its fused multiply-add d = a * b + c, lane by lane (IEEE fma).
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    return (uint64_t)__float_as_uint(lo) | ((uint64_t)__float_as_uint(hi) << 32);
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// Epilogue staging for TMA stores: 16 bytes at byte `off` of a 1024-aligned staging box
// whose rows are swizzled like TMA's 32/64/128-byte modes (16-byte chunk index XOR address
// bits 7-9, `mask` = 1, 3 or 7), so that a warp writing one row per lane hits distinct banks.
__device__ __forceinline__ void sts_swz(uint32_t buf, uint32_t off, uint4 v, uint32_t mask) {
    const uint32_t a = buf + off;
    const uint32_t ph = a ^ (((a >> 7) & mask) << 4);
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(ph), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// 16 bytes at an already swizzled shared-memory address.
__device__ __forceinline__ void sts16(uint32_t a, uint4 v) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* m, uint32_t src, int c0, int c1, int c2, int c3) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"((uint64_t)m),
                 "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
                 : "memory");
}
__device__ __forceinline__ void tma_store_5d(const CUtensorMap* m, uint32_t src, int c0, int c1, int c2, int c3, int c4) {
    asm volatile("cp.async.bulk.tensor.5d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5, %6}], [%1];" ::"l"((uint64_t)m),
                 "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// every committed store has finished reading its shared-memory source
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// all but the most recent committed store have finished reading their sources
__device__ __forceinline__ void bulk_wait_read1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
// every committed store is complete
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// PAR = 0: standard tiles of R rows x 128 columns.  PAR = 1, 2 or 4: the decoder's first
// conv; a tile is R coarse rows x 128 coarse columns and PAR of the four parity classes
// (x mod 2, y mod 2) of the fine pixels above them: 1 class, both x classes of one y
// class, or all four.  The tile's PAR*R accumulators share every staged halo and weight.
template <int R, int PAR, bool IN8, int EPI>
__global__ void __launch_bounds__(halo_threads(PAR, R, EPI), 1) k_conv_halo(const __grid_constant__ HParams p) {
    constexpr int MW = halo_mma_warps(PAR, R);
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* const gbase = smem_raw + (base - raw);
    const int S = p.stages;
    const uint32_t stg = base + S * p.stage_bytes;  // epilogue staging (TMA stores), 1024-aligned
    const uint32_t bars = stg + p.stg_bytes;
    auto full = [&](int s) { return bars + 8u * s; };
    auto empty = [&](int s) { return bars + 8u * (S + s); };
    auto tfull = [&](int b) { return bars + 8u * (2 * S + b); };
    auto tempty = [&](int b) { return bars + 8u * (2 * S + 2 + b); };
    const uint32_t drain = bars + 8u * (2 * S + 4);
    const uint32_t tslot = bars + 8u * (2 * S + 5);
    const uint32_t never = bars + 8u * (2 * S + 6);  // no thread ever arrives on it
    volatile int* flag = reinterpret_cast<volatile int*>(gbase + (tslot - base) + 4);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int N = p.N;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), p.nmma);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(tfull(b), p.nmma);
            mbar_init(tempty(b), EPI);
        }
        mbar_init(drain, p.nmma);
        mbar_init(never, 1);
        *flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(tslot, p.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(gbase + (tslot - base));
    // Tile sequence: blockIdx.x, + gridDim.x, ...
    auto tile_live = [&](int t) { return t < p.ntiles; };

    // tile t -> image n, first column x0 and first row y0 (coarse for parity tiles) and the
    // parity class (px, py); parity is the fastest index so that the four classes of a
    // region run back to back and share its halo in L2
    // (for PAR 1 and 2, px / py are the tile's class; PAR 4 covers every class)
    auto tile_of = [&](int t, int& n, int& x0, int& y0, int& px, int& py) {
        px = py = 0;
        if (PAR == 1) {
            px = t & 1;
            py = (t >> 1) & 1;
            t >>= 2;
        } else if (PAR == 2) {
            py = t & 1;
            t >>= 1;
        }
        const int tx = t % p.tiles_x;
        t /= p.tiles_x;
        const int ty = t % p.tiles_y;
        n = t / p.tiles_y;
        x0 = tx * 128;
        y0 = ty * R;
    };

    if (warp == 0 && lane == 0) {
        // ------------------------------------------------------------ producer --
        int use = 0;
        int st = 0;         // stage of this use (use % S, kept incrementally)
        uint32_t ph = 1u;   // parity that the stage's empty barrier must reach
        bool ok = true;
        for (int t = blockIdx.x; tile_live(t) && ok; t += gridDim.x) {
            int n, x0, y0, px, py;
            tile_of(t, n, x0, y0, px, py);
            for (int sg = 0; sg < p.nseg && ok; ++sg) {
                const HSeg& s = p.seg[sg];
                for (int cc = 0; cc < s.nchunk; ++cc) {
                    if (!mbar_wait(empty(st), ph)) { ok = false; break; }
                    const uint32_t a_dst = base + st * p.stage_bytes;
                    mbar_expect_tx(full(st), s.bytes);
                    const int c = cc * s.ck;
                    if (PAR && sg == 0) {
                        const int fy = PAR == 4 ? 2 * y0 - 1 : 2 * y0 + py - 1;  // first staged fine row
                        tma_5d(a_dst, &s.a, full(st), c, 0, x0 - 1, fy, n);
                        tma_5d(a_dst + s.plane, &s.a, full(st), c, 1, x0 - 1, fy, n);
                    } else {
                        // (the upsampled operand of one y class from its first row on)
                        tma_4d(a_dst, &s.a, full(st), c, x0 - 1, y0 - 1 + (PAR == 1 || PAR == 2 ? py : 0), n);
                    }
                    bulk_load(a_dst + s.b_off, s.w + (size_t)cc * s.w_chunk + (uint32_t)py * s.w_sel, s.w_bytes, full(st));
                    ++use;
                    if (++st == S) {
                        st = 0;
                        ph ^= 1u;
                    }
                }
            }
        }
        if (!ok) atomicExch(p.err, 5);
        for (int k = use > S ? use - S : 0; k < use; ++k) mbar_wait(full(k % S), (k / S) & 1);
    } else if (warp >= 1 && warp <= MW && lane == 0 && warp - 1 < p.nmma) {
        // ----------------------------------------------------------------- MMA --
        // Issuer g owns work units [a_lo, a_hi] of every tile: standard tiles one output row
        // each; parity tiles one (row, y class) each, owning the accumulators of its NX x
        // classes (adjacent in TMEM, cx = 1 first).  Descriptors are built once per stage;
        // every tap, row and K step only adds a constant to the start-address field
        // (address >> 4, 14 bits).
        IssueCtx q;
        q.g = warp - 1;
        q.N = (uint32_t)N;
        q.idesc = p.idesc;
        int tcount = 0;
        int st = 0;        // stage (use % S, kept incrementally)
        uint32_t ph = 0u;  // parity that the stage's full barrier must reach
        bool ok = !p.stall || mbar_wait(never, 0, kStallWaitCycles), issued = false;
        for (int t = blockIdx.x; tile_live(t) && ok; t += gridDim.x, ++tcount) {
            int n, x0, y0, px, py;
            tile_of(t, n, x0, y0, px, py);
            q.px = px;
            q.py = py;
            const int b = p.tbufs == 2 ? (tcount & 1) : 0;
            const int u = p.tbufs == 2 ? (tcount >> 1) : tcount;  // uses of buffer b so far
            if (!mbar_wait(tempty(b), (u & 1) ^ 1)) { ok = false; break; }
            tc_fence_after();
            constexpr int NACC = R * (PAR == 0 ? 1 : PAR);
            const uint32_t d0 = tmem + (uint32_t)(b * NACC * N);
            for (int sg = 0; sg < p.nseg && ok; ++sg) {
                const HSeg& s = p.seg[sg];
                const StageGeom geo{s.pitch, s.plane, s.swz};
                const int nk = (int)(s.pitch >> 5);  // one MMA per 32 bytes of K (16 BF16 or 32 E4M3)
                for (int cc = 0; cc < s.nchunk; ++cc) {
                    if (!mbar_wait(full(st), ph)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t stage0 = (base + st * p.stage_bytes) >> 4, b0 = stage0 + (s.b_off >> 4);
                    const uint32_t a0 =
                        (PAR == 1 || PAR == 2) && sg == 1 ? stage0 - (uint32_t)py * kHaloW * (s.pitch >> 4) : stage0;
                    switch (nk) {
                        case 1: issue_stage<R, PAR, IN8, 1>(q, sg, a0, b0, geo, d0, sg == 0 && cc == 0); break;
                        case 2: issue_stage<R, PAR, IN8, 2>(q, sg, a0, b0, geo, d0, sg == 0 && cc == 0); break;
                        default: issue_stage<R, PAR, IN8, 4>(q, sg, a0, b0, geo, d0, sg == 0 && cc == 0); break;
                    }
                    issued = true;
                    mma_commit(empty(st));
                    if (++st == S) {
                        st = 0;
                        ph ^= 1u;
                    }
                }
            }
            if (ok) mma_commit(tfull(b));
        }
        if (!ok) atomicExch(p.err, 6);
        // every issuer arrives (the barrier counts them all); the wait makes sure every MMA
        // issued has completed before TMEM is released
        (void)issued;
        mma_commit(drain);
        mbar_wait(drain, 0);
    } else if (warp > MW) {
        // ------------------------------------------------------------ epilogue --
        const int q = warp & 3;
        const int m = 32 * q + lane;
        constexpr int NE = EPI / 4;                   // warps per TMEM lane quarter
        const int eh = (warp - MW - 1) >> 2;  // which of them this warp is
        const bool leader = threadIdx.x == 32 * (MW + 1);
        const int Wh = p.W >> 1, Hh = p.H >> 1;
        const bool pool = p.pool_out != nullptr;
        // bias (+ per-channel scale of E4M3 operands) and ReLU of 16 accumulator columns
        auto act16 = [&](const uint32_t (&u)[16], int c, float (&f)[16]) {
            const float4* b4 = reinterpret_cast<const float4*>(p.cbias + c);
            const float4* s4 = reinterpret_cast<const float4*>(p.cscale + c);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 bv = b4[j];
                const float bb[4] = {bv.x, bv.y, bv.z, bv.w};
                if (IN8) {
                    const float4 sv = s4[j];
                    const float ss[4] = {sv.x, sv.y, sv.z, sv.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) f[4 * j + i] = fmaxf(fmaf(__uint_as_float(u[4 * j + i]), ss[i], bb[i]), 0.f);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) f[4 * j + i] = fmaxf(__uint_as_float(u[4 * j + i]) + bb[i], 0.f);
                }
            }
        };
        // the same before the ReLU: BF16 outputs take the ReLU in their conversion
        // (relu_bf16x16); E4M3 outputs and the head apply relu16 first
        auto pre16 = [&](const uint32_t (&u)[16], int c, float (&f)[16]) {
            const float4* b4 = reinterpret_cast<const float4*>(p.cbias + c);
            const float4* s4 = reinterpret_cast<const float4*>(p.cscale + c);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 bv = b4[j];
                const float bb[4] = {bv.x, bv.y, bv.z, bv.w};
                if (IN8) {
                    const float4 sv = s4[j];
                    const float ss[4] = {sv.x, sv.y, sv.z, sv.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) f[4 * j + i] = fmaf(__uint_as_float(u[4 * j + i]), ss[i], bb[i]);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) f[4 * j + i] = __uint_as_float(u[4 * j + i]) + bb[i];
                }
            }
        };
        int tcount = 0;
        int oc = 0;  // rows (row pairs) this warp has staged: selects the staging buffer
        for (int t = blockIdx.x; tile_live(t); t += gridDim.x, ++tcount) {
            const int b = p.tbufs == 2 ? (tcount & 1) : 0;
            const int u = p.tbufs == 2 ? (tcount >> 1) : tcount;
            if (leader && !mbar_wait(tfull(b), u & 1)) *flag = 1;
            named_sync(1, 32 * EPI);
            if (*flag) break;
            tc_fence_after();
            int n, x0, y0, px, py;
            tile_of(t, n, x0, y0, px, py);
            // Never taken (the loop bound keeps t < ntiles), but kept: with this exit in the
            // loop body nvcc allocates the epilogue's registers without spills (ptxas: the
            // R = 8, 12-warp instance spills 80 bytes without it, none with it).
            if (t >= p.ntiles) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(tempty(b));
                continue;
            }
            constexpr int NCE = PAR == 0 ? 1 : PAR;
            const uint32_t trow = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * NCE * R * N);
            if (pool) {
                // rows in pairs (pairs alternate between the quarter's warps): both rows
                // stored, their 2x2 maximum pooled with the lane holding the next column
                for (int r = 2 * eh; r < R; r += 2 * NE) {
                    const int x = x0 + m, y = y0 + r;
                    const bool v0 = x < p.W && y < p.H, v1 = x < p.W && y + 1 < p.H;
                    const uint32_t wb = stg + (uint32_t)(warp - MW - 1) * p.ost_warp +
                                        (uint32_t)(oc % p.ost_nbuf) * p.ost_unit;
                    if (p.ostage) {  // the store that last used this staging buffer has read it
                        if (lane == 0) {
                            if (p.ost_nbuf > 1) bulk_wait_read1();
                            else bulk_wait_read();
                        }
                        __syncwarp();
                    }
                    for (int c0 = 0; c0 < N; c0 += 16) {
                        uint32_t u0[16], u1[16];
                        tmem_ld16_async(trow + (uint32_t)(r * N + c0), u0);
                        tmem_ld16_async(trow + (uint32_t)((r + 1) * N + c0), u1);
                        tmem_wait16(u0);
                        tmem_wait16(u1);
                        // the 2x2 maximum before the ReLU gives the same pooled values
                        float f0[16], f1[16], pm[16];
                        pre16(u0, c0, f0);
                        pre16(u1, c0, f1);
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const float a = fmaxf(f0[j], f1[j]);
                            pm[j] = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, 1));
                        }
                        if (p.out_fp8) {
                            relu16(f0);
                            relu16(f1);
                        }
                        if (p.pool_fp8) relu16(pm);
                        if (p.ostage) {
                            const uint32_t eo = p.out_fp8 ? 1u : 2u, epb = p.pool_fp8 ? 1u : 2u;
                            auto stage_row = [&](uint32_t buf, const float* f) {
                                if (p.out_fp8) {
                                    const uint32_t cb = (uint32_t)c0 * eo;
                                    sts_swz(buf, (cb / p.orow_b) * 32u * p.orow_b + (uint32_t)lane * p.orow_b + cb % p.orow_b,
                                            pack_fp8x16(f, p.inv_out), p.omask);
                                } else {
                                    uint4 pk[2];
                                    relu_bf16x16(f, pk);
#pragma unroll
                                    for (int h2 = 0; h2 < 2; ++h2) {
                                        const uint32_t cb = (uint32_t)(c0 + 8 * h2) * eo;
                                        sts_swz(buf, (cb / p.orow_b) * 32u * p.orow_b + (uint32_t)lane * p.orow_b + cb % p.orow_b,
                                                pk[h2], p.omask);
                                    }
                                }
                            };
                            stage_row(wb, f0);
                            stage_row(wb + p.ost_row, f1);
                            if ((m & 1) == 0) {
                                const uint32_t pb = wb + p.ost_pool, i = (uint32_t)lane >> 1;
                                if (p.pool_fp8) {
                                    const uint32_t cb = (uint32_t)c0;
                                    sts_swz(pb, (cb / p.prow_b) * 16u * p.prow_b + i * p.prow_b + cb % p.prow_b,
                                            pack_fp8x16(pm, p.inv_out), p.pmask);
                                } else {
                                    uint4 pk[2];
                                    relu_bf16x16(pm, pk);
#pragma unroll
                                    for (int h2 = 0; h2 < 2; ++h2) {
                                        const uint32_t cb = (uint32_t)(c0 + 8 * h2) * epb;
                                        sts_swz(pb, (cb / p.prow_b) * 16u * p.prow_b + i * p.prow_b + cb % p.prow_b, pk[h2],
                                                p.pmask);
                                    }
                                }
                            }
                            continue;
                        }
                        const size_t e0 = (((size_t)n * p.H + y) * p.W + x) * N + c0;
                        const size_t e1 = e0 + (size_t)p.W * N;
                        const size_t ep = (((size_t)n * Hh + (y >> 1)) * Wh + (x >> 1)) * N + c0;
                        if (p.out_fp8) {
                            if (v0) st_fp8x16(static_cast<uint8_t*>(p.out) + e0, f0, p.inv_out);
                            if (v1) st_fp8x16(static_cast<uint8_t*>(p.out) + e1, f1, p.inv_out);
                        } else {
                            if (v0) st_relu_bf16x16(static_cast<__nv_bfloat16*>(p.out) + e0, f0);
                            if (v1) st_relu_bf16x16(static_cast<__nv_bfloat16*>(p.out) + e1, f1);
                        }
                        if ((m & 1) == 0 && v1) {
                            if (p.pool_fp8) st_fp8x16(static_cast<uint8_t*>(p.pool_out) + ep, pm, p.inv_out);
                            else st_relu_bf16x16(static_cast<__nv_bfloat16*>(p.pool_out) + ep, pm);
                        }
                    }
                    if (p.ostage) {  // both rows and the pooled row leave by TMA (clipped at the image edges)
                        fence_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            const uint32_t eo = p.out_fp8 ? 1u : 2u, epb = p.pool_fp8 ? 1u : 2u;
                            const int X = x0 + 32 * q;
                            for (uint32_t sb = 0; sb * p.orow_b < (uint32_t)N * eo; ++sb) {
                                const int ch = (int)(sb * p.orow_b / eo);
                                tma_store_4d(&p.omap, wb + sb * 32u * p.orow_b, ch, X, y, n);
                                tma_store_4d(&p.omap, wb + p.ost_row + sb * 32u * p.orow_b, ch, X, y + 1, n);
                            }
                            for (uint32_t sb = 0; sb * p.prow_b < (uint32_t)N * epb; ++sb)
                                tma_store_4d(&p.pmap, wb + p.ost_pool + sb * 16u * p.prow_b, (int)(sb * p.prow_b / epb), X >> 1,
                                             y >> 1, n);
                            bulk_commit();
                        }
                        ++oc;
                    }
                }
            } else if (PAR == 0 && N == 32 && p.head_out) {
                // fused 1x1 head on 32 channels: the next row's TMEM loads are in flight while
                // this row's bias, ReLU, dot products and sigmoid run
                uint32_t ua[16], ub[16];
                if (eh < R) {
                    tmem_ld16_async(trow + (uint32_t)(eh * 32), ua);
                    tmem_ld16_async(trow + (uint32_t)(eh * 32 + 16), ub);
                }
                for (int a = eh; a < R; a += NE) {
                    tmem_wait16(ua);
                    tmem_wait16(ub);
                    float f0[16], f1[16];
                    act16(ua, 0, f0);
                    act16(ub, 16, f1);
                    if (a + NE < R) {
                        tmem_ld16_async(trow + (uint32_t)((a + NE) * 32), ua);
                        tmem_ld16_async(trow + (uint32_t)((a + NE) * 32 + 16), ub);
                    }
                    const int x = x0 + m, y = y0 + a;
                    float h[4];
#pragma unroll
                    for (int o = 0; o < 4; ++o) {
                        const float4* w4 = reinterpret_cast<const float4*>(p.chead + o * 32);
                        uint64_t acc = 0;
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const float4 wv = w4[j];
                            const float* f = j < 4 ? f0 + 4 * j : f1 + 4 * (j - 4);
                            acc = fma2(pack2(wv.x, wv.y), pack2(f[0], f[1]), acc);
                            acc = fma2(pack2(wv.z, wv.w), pack2(f[2], f[3]), acc);
                        }
                        h[o] = __uint_as_float((uint32_t)acc) + __uint_as_float((uint32_t)(acc >> 32));
                    }
                    if (x < p.W && y < p.H) {
                        const size_t pix = ((size_t)n * p.H + y) * p.W + x;
#pragma unroll
                        for (int o = 0; o < 4; ++o) {
                            if (o >= p.head_o) break;
                            p.head_out[pix * p.head_o + o] = __frcp_rn(1.0f + __expf(-(h[o] + p.chead[4 * 32 + o])));
                        }
                    }
                }
            } else {
                for (int a = eh; a < NCE * R; a += NE) {
                    int x, y;
                    bool v;
                    if (PAR) {
                        // accumulator a: unit a / NX = (row, y class), x class 1 before 0
                        constexpr int NYE = PAR == 4 ? 2 : 1, NXE = PAR >= 2 ? 2 : 1;
                        const int u = a / NXE, r = u / NYE;
                        const int cpx = NXE == 2 ? 1 - (a & 1) : px;
                        const int cpy = PAR == 4 ? u - r * NYE : py;
                        x = 2 * (x0 + m) + cpx;
                        y = 2 * (y0 + r) + cpy;
                        v = (x0 + m) < Wh && (y0 + r) < Hh;
                    } else {
                        x = x0 + m;
                        y = y0 + a;
                        v = x < p.W && y < p.H;
                    }
                    const size_t pix = ((size_t)n * p.H + y) * p.W + x;
                    float h[4] = {0.f, 0.f, 0.f, 0.f};
                    const uint32_t wb = stg + (uint32_t)(warp - MW - 1) * p.ost_warp +
                                        (uint32_t)(oc % p.ost_nbuf) * p.ost_unit;
                    if (p.ostage) {  // the store that last used this staging buffer has read it
                        if (lane == 0) {
                            if (p.ost_nbuf > 1) bulk_wait_read1();
                            else bulk_wait_read();
                        }
                        __syncwarp();
                    }
                    for (int c0 = 0; c0 < N; c0 += 32) {
                        uint32_t u0[16], u1[16];
                        const bool two = c0 + 16 < N;
                        tmem_ld16_async(trow + (uint32_t)(a * N + c0), u0);
                        if (two) tmem_ld16_async(trow + (uint32_t)(a * N + c0 + 16), u1);
                        tmem_wait16(u0);
                        if (two) tmem_wait16(u1);
                        float f0[16], f1[16];
                        pre16(u0, c0, f0);
                        if (two) pre16(u1, c0 + 16, f1);
                        if (p.out_fp8 || p.head_out) {
                            relu16(f0);
                            if (two) relu16(f1);
                        }
                        if (p.ostage) {
                            const uint32_t eo = p.out_fp8 ? 1u : 2u;
                            for (int hf = 0; hf < (two ? 2 : 1); ++hf) {
                                const float* f = hf ? f1 : f0;
                                const int cf = c0 + 16 * hf;
                                if (p.out_fp8) {
                                    const uint32_t cb = (uint32_t)cf;
                                    sts_swz(wb, (cb / p.orow_b) * 32u * p.orow_b + (uint32_t)lane * p.orow_b + cb % p.orow_b,
                                            pack_fp8x16(f, p.inv_out), p.omask);
                                } else {
                                    uint4 pk[2];
                                    relu_bf16x16(f, pk);
#pragma unroll
                                    for (int h2 = 0; h2 < 2; ++h2) {
                                        const uint32_t cb = (uint32_t)(cf + 8 * h2) * eo;
                                        sts_swz(wb, (cb / p.orow_b) * 32u * p.orow_b + (uint32_t)lane * p.orow_b + cb % p.orow_b,
                                                pk[h2], p.omask);
                                    }
                                }
                            }
                        } else if (p.head_out) {
                            // 1x1 head: 4 outputs (zero weights past head_o), channel pairs
                            // accumulated with packed FP32x2 fused multiply-adds
#pragma unroll
                            for (int o = 0; o < 4; ++o) {
                                const float4* w4 = reinterpret_cast<const float4*>(p.chead + o * N + c0);
                                uint64_t acc = 0;  // (0.f, 0.f)
#pragma unroll
                                for (int j = 0; j < 8; ++j) {
                                    if (j >= 4 && !two) break;
                                    const float4 wv = w4[j];
                                    const float* f = j < 4 ? f0 + 4 * j : f1 + 4 * (j - 4);
                                    acc = fma2(pack2(wv.x, wv.y), pack2(f[0], f[1]), acc);
                                    acc = fma2(pack2(wv.z, wv.w), pack2(f[2], f[3]), acc);
                                }
                                h[o] += __uint_as_float((uint32_t)acc) + __uint_as_float((uint32_t)(acc >> 32));
                            }
                        } else if (v) {
                            if (p.out_fp8) {
                                uint8_t* d8 = static_cast<uint8_t*>(p.out) + pix * N + c0;
                                if (two)  // 32 E4M3 channels in one 32-byte store (N is a multiple of 32)
                                    st_32b(d8, pack_fp8x16(f0, p.inv_out), pack_fp8x16(f1, p.inv_out));
                                else
                                    st_fp8x16(d8, f0, p.inv_out);
                            } else {
                                st_relu_bf16x16(static_cast<__nv_bfloat16*>(p.out) + pix * N + c0, f0);
                                if (two) st_relu_bf16x16(static_cast<__nv_bfloat16*>(p.out) + pix * N + c0 + 16, f1);
                            }
                        }
                    }
                    if (p.head_out && v) {
#pragma unroll
                        for (int o = 0; o < 4; ++o) {
                            if (o >= p.head_o) break;
                            p.head_out[pix * p.head_o + o] = __frcp_rn(1.0f + __expf(-(h[o] + p.chead[4 * N + o])));
                        }
                    }
                    if (p.ostage) {  // the row leaves by TMA (clipped at the image edges)
                        fence_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            const uint32_t eo = p.out_fp8 ? 1u : 2u;
                            for (uint32_t sb = 0; sb * p.orow_b < (uint32_t)N * eo; ++sb) {
                                const int ch = (int)(sb * p.orow_b / eo);
                                if (PAR)  // x = 2 X + cx: the 5-D view {N, 2, W/2, H, B}
                                    tma_store_5d(&p.omap, wb + sb * 32u * p.orow_b, ch, x & 1, x0 + 32 * q, y, n);
                                else
                                    tma_store_4d(&p.omap, wb + sb * 32u * p.orow_b, ch, x0 + 32 * q, y, n);
                            }
                            bulk_commit();
                        }
                        ++oc;
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(tempty(b));
        }
        if (p.ostage && lane == 0) bulk_wait_all();  // no store may outlive the staging
        if (leader && *flag) atomicExch(p.err, 7);
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, p.tmem_cols);
    }
}

// ================================================================ fused level 0 ==
//
// The encoder's two full-resolution convolutions in one pass.  A tile is R output rows x
// kFuseW output columns of the second conv.  The first conv (on the 16-channel BF16 input,
// staged with one TMA box per tile and issued like a standard halo tile) is computed for
// the tile and its one-pixel border: R + 2 rows x 128 columns.  Its epilogue applies bias and ReLU, rounds to BF16 and writes zero outside the
// image (the second conv's zero padding).  It stores the result in shared memory, in the
// swizzled K-major layout of a staged halo, so the second conv is issued on it exactly like
// on a TMA-loaded halo (issue_stage).  The second conv's epilogue writes its output (the
// skip tensor) and the 2x2 max-pooled output.  The first conv's output never reaches
// global memory.  The MMA rows 126 and 127 of the second conv read border columns that are
// never written; their results are discarded (accumulator rows are independent).
//
// Warps: 0 producer (both weight sets once, then one input halo per tile into an S-stage
// ring), 1-2 MMA issuers (each takes half the rows of both convs), 3-10 the first epilogue
// (two per TMEM lane quarter, alternate rows), 11-18 the second epilogue (two per quarter,
// alternate row pairs).  The first conv's accumulators are single-buffered, the second
// conv's and the shared-memory activations double-buffered.

constexpr int kFuseW = 126;                 // output columns per tile
constexpr int kFuseThreads = 32 * 19;
constexpr int kFuseMaxN = 32;

struct FParams {
    CUtensorMap in;   // network input 4-D {16, W, H, B}, box {16, 130, R + 4, 1}, 32-byte swizzle
    const uint8_t *w1, *w2;  // weights of the two convs, as shared memory holds them (blocks [kx][ky = 2, 1, 0])
    uint32_t w1_bytes, w2_bytes;
    int W, H, B;
    int N1, N2;
    int tiles_x, tiles_y, ntiles, stages;
    uint32_t in_bytes, in_stage, w1_off, w2_off, in_off, act_off, act_bytes;
    uint32_t pitch1, swz1, smask1;  // second conv's staged pixel: N1 x 2 bytes, UMMA layout, swizzle mask
    uint32_t tmem_cols, idesc1, idesc2;
    __nv_bfloat16* out;
    void* pool_out;
    int pool8;
    float inv_pool;
    int* err;
    alignas(16) float b1[kFuseMaxN];
    alignas(16) float b2[kFuseMaxN];
};

template <int R>
__global__ void __launch_bounds__(kFuseThreads, 1) k_enc0_fused(const __grid_constant__ FParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* const gbase = smem_raw + (base - raw);
    const int S = p.stages;
    const uint32_t w1s = base + p.w1_off, w2s = base + p.w2_off, ins = base + p.in_off, acts = base + p.act_off;
    const uint32_t bars = acts + 2 * p.act_bytes;
    auto in_full = [&](int s) { return bars + 8u * s; };
    auto in_empty = [&](int s) { return bars + 8u * (S + s); };
    const uint32_t wbar = bars + 8u * (2 * S);
    const uint32_t a_full = bars + 8u * (2 * S + 1), a_empty = bars + 8u * (2 * S + 2);
    auto act_full = [&](int b) { return bars + 8u * (2 * S + 3 + b); };
    auto act_empty = [&](int b) { return bars + 8u * (2 * S + 5 + b); };
    auto b_full = [&](int b) { return bars + 8u * (2 * S + 7 + b); };
    auto b_empty = [&](int b) { return bars + 8u * (2 * S + 9 + b); };
    const uint32_t drain = bars + 8u * (2 * S + 11);
    const uint32_t tslot = bars + 8u * (2 * S + 12);
    volatile int* flag = reinterpret_cast<volatile int*>(gbase + (tslot - base) + 4);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int N1 = p.N1, N2 = p.N2;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(in_full(s), 1);
            mbar_init(in_empty(s), 2);
        }
        mbar_init(wbar, 1);
        mbar_init(a_full, 2);
        mbar_init(a_empty, 8);
        for (int b = 0; b < 2; ++b) {
            mbar_init(act_full(b), 1);
            mbar_init(act_empty(b), 2);
            mbar_init(b_full(b), 2);
            mbar_init(b_empty(b), 8);
        }
        mbar_init(drain, 2);
        flag[0] = 0;
        flag[1] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(tslot, p.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(gbase + (tslot - base));
    const uint32_t accA = tmem, accB = tmem + (uint32_t)((R + 2) * N1);
    auto tile_of = [&](int t, int& n, int& x0, int& y0) {
        const int tx = t % p.tiles_x;
        t /= p.tiles_x;
        y0 = (t % p.tiles_y) * R;
        n = t / p.tiles_y;
        x0 = tx * kFuseW;
    };

    if (warp == 0 && lane == 0) {
        // ------------------------------------------------------------ producer --
        bool ok = true;
        mbar_expect_tx(wbar, p.w1_bytes + p.w2_bytes);
        bulk_load(w1s, p.w1, p.w1_bytes, wbar);
        bulk_load(w2s, p.w2, p.w2_bytes, wbar);
        int use = 0, st = 0;
        uint32_t ph = 1u;
        for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
            int n, x0, y0;
            tile_of(t, n, x0, y0);
            if (!mbar_wait(in_empty(st), ph)) { ok = false; break; }
            mbar_expect_tx(in_full(st), p.in_bytes);
            tma_4d(ins + st * p.in_stage, &p.in, in_full(st), 0, x0 - 2, y0 - 2, n);
            ++use;
            if (++st == S) { st = 0; ph ^= 1u; }
        }
        if (!ok) atomicExch(p.err, 5);
        mbar_wait(wbar, 0);
        for (int k = use > S ? use - S : 0; k < use; ++k) mbar_wait(in_full(k % S), (k / S) & 1);
    } else if ((warp == 1 || warp == 2) && lane == 0) {
        // ----------------------------------------------------------------- MMA --
        // A(k) for the k-th tile of this CTA as soon as the first epilogue has read A(k-1);
        // then B(k-1) once its activations are in shared memory.
        IssueCtx qa{warp - 1, 0, 0, (uint32_t)N1, p.idesc1}, qb{warp - 1, 0, 0, (uint32_t)N2, p.idesc2};
        const StageGeom h1{32, 0, 6};  // the 16-channel input
        const StageGeom h2{p.pitch1, 0, p.swz1};
        bool ok = mbar_wait(wbar, 0);
        int st = 0;
        uint32_t ph = 0u;
        for (int t = blockIdx.x, k = 0; ok; t += gridDim.x, ++k) {
            const bool have = t < p.ntiles;
            if (have) {
                if (!mbar_wait(in_full(st), ph) || !mbar_wait(a_empty, (k & 1) ^ 1)) { ok = false; break; }
                tc_fence_after();
                issue_stage<R + 2, 0, false, 1>(qa, 0, (ins + st * p.in_stage) >> 4, w1s >> 4, h1, accA, true);
                mma_commit(in_empty(st));
                mma_commit(a_full);
                if (++st == S) { st = 0; ph ^= 1u; }
            }
            if (k >= 1) {
                const int kb = k - 1, ab = kb & 1;
                if (!mbar_wait(act_full(ab), (kb >> 1) & 1) || !mbar_wait(b_empty(ab), ((kb >> 1) & 1) ^ 1)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t a0 = (acts + ab * p.act_bytes) >> 4, d0 = accB + (uint32_t)(ab * R * N2);
                if (p.pitch1 == 64) issue_stage<R, 0, false, 2>(qb, 0, a0, w2s >> 4, h2, d0, true);
                else issue_stage<R, 0, false, 1>(qb, 0, a0, w2s >> 4, h2, d0, true);
                mma_commit(act_empty(ab));
                mma_commit(b_full(ab));
            }
            if (!have) break;
        }
        if (!ok) atomicExch(p.err, 6);
        mma_commit(drain);
        mbar_wait(drain, 0);
    } else if (warp >= 3 && warp <= 10) {
        // ---------------------------------------- first epilogue: activations -> smem --
        const int q = warp & 3, m = 32 * q + lane, half = (warp - 3) >> 2;
        const bool leader = threadIdx.x == 32 * 3;
        for (int t = blockIdx.x, k = 0; t < p.ntiles; t += gridDim.x, ++k) {
            const int ab = k & 1;
            if (leader && (!mbar_wait(a_full, k & 1) || !mbar_wait(act_empty(ab), ((k >> 1) & 1) ^ 1))) flag[0] = 1;
            named_sync(1, 256);
            if (flag[0]) break;
            tc_fence_after();
            int n, x0, y0;
            tile_of(t, n, x0, y0);
            const int x = x0 - 1 + m;
            const uint32_t buf = acts + ab * p.act_bytes;
            for (int r = half; r < R + 2; r += 2) {
                const int y = y0 - 1 + r;
                const bool inside = x >= 0 && x < p.W && y >= 0 && y < p.H;
                const uint32_t trow = accA + ((uint32_t)(32 * q) << 16) + (uint32_t)(r * N1);
                // the pixel's 32 or 64 bytes lie in one 128-byte line: one swizzle pattern
                const uint32_t a = buf + (uint32_t)(r * kHaloW + m) * p.pitch1;
                const uint32_t sx = ((a >> 7) & p.smask1) << 4;
                // both 16-column halves of the row in flight before one wait (N1 is 16 or 32)
                uint32_t u0[16], u1[16];
                tmem_ld16_async(trow, u0);
                if (N1 > 16) tmem_ld16_async(trow + 16u, u1);
                tmem_wait16(u0);
                uint4 pk[2];
                bias_relu_bf16x16(u0, p.b1, inside, pk);
                sts16(a ^ sx, pk[0]);
                sts16((a + 16) ^ sx, pk[1]);
                if (N1 > 16) {
                    tmem_wait16(u1);
                    bias_relu_bf16x16(u1, p.b1 + 16, inside, pk);
                    sts16((a + 32) ^ sx, pk[0]);
                    sts16((a + 48) ^ sx, pk[1]);
                }
            }
            tc_fence_before();
            fence_async_smem();  // the tensor cores read these activations
            __syncwarp();
            if (lane == 0) mbar_arrive(a_empty);
            named_sync(1, 256);
            if (leader) mbar_arrive(act_full(ab));
        }
        if (leader && flag[0]) atomicExch(p.err, 7);
    } else if (warp >= 11) {
        // ------------------------------------------------ second epilogue: global stores --
        const int q = warp & 3, m = 32 * q + lane, half = (warp - 11) >> 2;
        const bool leader = threadIdx.x == 32 * 11;
        const int Wh = p.W >> 1, Hh = p.H >> 1;
        for (int t = blockIdx.x, k = 0; t < p.ntiles; t += gridDim.x, ++k) {
            const int ab = k & 1;
            if (leader && !mbar_wait(b_full(ab), (k >> 1) & 1)) flag[1] = 1;
            named_sync(2, 256);
            if (flag[1]) break;
            tc_fence_after();
            int n, x0, y0;
            tile_of(t, n, x0, y0);
            const int x = x0 + m;
            const bool vx = m < kFuseW && x < p.W;
            const uint32_t tb = accB + ((uint32_t)(32 * q) << 16) + (uint32_t)(ab * R * N2);
            for (int r = 2 * half; r < R; r += 4) {
                const int y = y0 + r;
                for (int c0 = 0; c0 < N2; c0 += 16) {
                    uint32_t u0[16], u1[16];
                    tmem_ld16_async(tb + (uint32_t)(r * N2 + c0), u0);
                    tmem_ld16_async(tb + (uint32_t)((r + 1) * N2 + c0), u1);
                    tmem_wait16(u0);
                    tmem_wait16(u1);
                    // ReLU is applied by the BF16 conversions; the 2x2 maximum is taken before
                    // it, which gives the same pooled values (ReLU is monotone)
                    float f0[16], f1[16], pm[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        f0[j] = __uint_as_float(u0[j]) + p.b2[c0 + j];
                        f1[j] = __uint_as_float(u1[j]) + p.b2[c0 + j];
                        const float a = fmaxf(f0[j], f1[j]);
                        pm[j] = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, 1));
                    }
                    uint4 pk[2];
                    if (vx && y < p.H) {
                        relu_bf16x16(f0, pk);
                        st_pk32(p.out + (((size_t)n * p.H + y) * p.W + x) * N2 + c0, pk);
                    }
                    if (vx && y + 1 < p.H) {
                        relu_bf16x16(f1, pk);
                        st_pk32(p.out + (((size_t)n * p.H + y + 1) * p.W + x) * N2 + c0, pk);
                    }
                    if (vx && (m & 1) == 0 && y + 1 < p.H) {
                        const size_t pp = (((size_t)n * Hh + (y >> 1)) * Wh + (x >> 1)) * N2 + c0;
                        if (p.pool8) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) pm[j] = fmaxf(pm[j], 0.f);
                            st_fp8x16(static_cast<uint8_t*>(p.pool_out) + pp, pm, p.inv_pool);
                        } else {
                            relu_bf16x16(pm, pk);
                            st_pk32(static_cast<__nv_bfloat16*>(p.pool_out) + pp, pk);
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(b_empty(ab));
        }
        if (leader && flag[1]) atomicExch(p.err, 7);
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, p.tmem_cols);
    }
}

// ------------------------------------------------------------------ host side ----

// Chunk width of a K segment of C channels (C a multiple of 16): the largest of 64, 32, 16
// that is at most ckmax and divides C.
int seg_ck(int C, int ckmax) {
    int ck = std::min(C, ckmax);
    while (C % ck) ck >>= 1;
    return ck;
}

CUtensorMapSwizzle swizzle_for(int kc) {
    return kc == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : kc == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
}
uint32_t umma_layout_for(int kc) { return kc == 64 ? 2u : kc == 32 ? 4u : 6u; }

bool encode(CUtensorMap* m, int rank, const void* ptr, const cuuint64_t* dims, const cuuint64_t* strides_bytes,
            const cuuint32_t* box, int kc) {
    cuuint32_t es[5] = {1, 1, 1, 1, 1};
    CUresult r = encode_tiled(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(ptr), dims,
                                        strides_bytes, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_for(kc),
                                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

}  // namespace

bool tc_available() { return true; }

// Channels a layer's first source carries in the tensor-core layout (the RGBDA input is
// padded to 16 so that every K chunk is one 32-byte MMA step).
static int tc_c0(const ConvLayer& L) { return L.cin0 == 5 ? 16 : L.cin0; }

static cudaError_t prepare_halo_weights(ConvLayer& L, int ckmax);

cudaError_t tc_prepare_layer(ConvLayer& L, lnr_precision p) {
    if (p != LNR_BF16) return cudaErrorNotSupported;
    const int c0 = tc_c0(L), cin = L.cin0 + L.cin1, cpad = c0 + L.cin1;
    std::vector<__nv_bfloat16> w((size_t)L.cout * 9 * cpad, __float2bfloat16(0.f));
    for (int co = 0; co < L.cout; ++co)
        for (int ci = 0; ci < cin; ++ci) {
            const int k = ci < L.cin0 ? ci : c0 + (ci - L.cin0);
            for (int t = 0; t < 9; ++t)
                w[((size_t)co * 9 + t) * cpad + k] = __float2bfloat16(L.wf[((size_t)co * cin + ci) * 9 + t]);
        }
    if (L.wtc) cudaFree(L.wtc);
    L.wtc = nullptr;
    cudaError_t e = cudaMalloc(&L.wtc, w.size() * 2);
    if (e != cudaSuccess) return e;
    e = cudaMemcpy(L.wtc, w.data(), w.size() * 2, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return e;
    for (int ck : {16, 32, 64}) {
        e = prepare_halo_weights(L, ck);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

static void tc_conv_generic(const ConvLayer& L, const void* src0, const void* src1, void* out, void* pool_out,
                            const float* head_w, const float* head_b, float* head_out, int B, int W, int H, int head_o,
                            cudaStream_t st, TcState& tc) {
    Params p;
    std::memset(&p, 0, sizeof(p));
    const int N = L.cout;
    const int c0 = tc_c0(L), cpad = c0 + L.cin1;
    p.N = N;
    p.W = W;
    p.H = H;
    p.B = B;
    p.cin_pad = cpad;
    p.parity = L.cin1 > 0;
    const cuuint64_t Ktot = 9ull * cpad;
    auto set_seg = [&](Seg& s, int kind, const void* src, int C, int koff, int Ws, int Hs) {
        s.kind = kind;
        s.kc = seg_ck(C, 64);
        s.nchunk = C / s.kc;
        s.koff = koff;
        s.swz = umma_layout_for(s.kc);
        s.sbo = 16u * s.kc;  // 8 rows x (kc x 2 bytes)
        s.bytes = (uint32_t)(128 + N) * s.kc * 2;
        const cuuint64_t eb = 2;
        if (kind == 1) {
            cuuint64_t dims[5] = {(cuuint64_t)C, 2, (cuuint64_t)Ws / 2, (cuuint64_t)Hs, (cuuint64_t)B};
            cuuint64_t str[4] = {C * eb, 2 * C * eb, (cuuint64_t)Ws * C * eb, (cuuint64_t)Hs * Ws * C * eb};
            cuuint32_t box[5] = {(cuuint32_t)s.kc, 1, 128, 1, 1};
            if (!encode(&s.a, 5, src, dims, str, box, s.kc)) tc.host_err = 4;
        } else {
            cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)Ws, (cuuint64_t)Hs, (cuuint64_t)B};
            cuuint64_t str[3] = {C * eb, (cuuint64_t)Ws * C * eb, (cuuint64_t)Hs * Ws * C * eb};
            cuuint32_t box[4] = {(cuuint32_t)s.kc, kind == 0 ? 64u : 128u, kind == 0 ? 2u : 1u, 1};
            if (!encode(&s.a, 4, src, dims, str, box, s.kc)) tc.host_err = 4;
        }
        cuuint64_t wd[2] = {Ktot, (cuuint64_t)N};
        cuuint64_t ws_[1] = {Ktot * eb};
        cuuint32_t wb[2] = {(cuuint32_t)s.kc, (cuuint32_t)N};
        if (!encode(&s.b, 2, L.wtc, wd, ws_, wb, s.kc)) tc.host_err = 4;
    };
    if (p.parity) {
        p.nseg = 2;
        set_seg(p.seg[0], 1, src0, c0, 0, W, H);
        set_seg(p.seg[1], 2, src1, L.cin1, c0, W / 2, H / 2);
        p.tiles_x = (W / 2 + 127) / 128;
        p.tiles_y = H / 2;
        p.ntiles = B * 4 * p.tiles_y * p.tiles_x;
    } else {
        p.nseg = 1;
        set_seg(p.seg[0], 0, src0, c0, 0, W, H);
        p.tiles_x = (W + 63) / 64;
        p.tiles_y = (H + 1) / 2;
        p.ntiles = B * p.tiles_y * p.tiles_x;
    }
    int kc_max = 0;
    for (int i = 0; i < p.nseg; ++i) kc_max = std::max(kc_max, p.seg[i].kc);
    p.a_region = (uint32_t)(128 * kc_max * 2);
    const uint32_t b_region = (uint32_t)((N * kc_max * 2 + 1023) & ~1023);
    p.stage_bytes = p.a_region + b_region;
    p.xch_bytes = pool_out ? (uint32_t)((128 * kXchStride * 4 + 1023) & ~1023) : 0;
    const uint32_t budget = 220 * 1024 - p.xch_bytes;
    p.stages = std::min<int>(8, budget / p.stage_bytes);
    uint32_t cols = 32;
    while (cols < 2u * N) cols <<= 1;
    p.tmem_cols = cols;
    p.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    p.bias = L.b32;
    p.out = static_cast<__nv_bfloat16*>(out);
    p.pool_out = static_cast<__nv_bfloat16*>(pool_out);
    p.head_w = head_w;
    p.head_b = head_b;
    p.head_out = head_out;
    p.head_o = head_o;
    p.err = tc.err;
    const size_t smem = 1024 + (size_t)p.stages * p.stage_bytes + p.xch_bytes + 8 * (2 * p.stages + 6) + 16;
    const int grid = std::min(p.ntiles, tc.num_sms);
    if (tc.host_err || !L.wtc) return;
    tc_allow_smem((const void*)k_conv_tc);
    k_conv_tc<<<grid, kThreads, smem, st>>>(p);
    count_launch();
}

// ---- halo kernel host side ----

static int ck_index(int ck) { return ck == 16 ? 0 : ck == 32 ? 1 : 2; }


// Weight blocks of one K chunk of segment sg of the halo kernel, as 9-bit tap masks (bit
// 3 * ky + kx); a block holds the sum of its taps' weights.
//  - standard convs: single taps ordered [kx][ky = 2, 1, 0], so that the blocks of one kx
//    and consecutive output rows form one contiguous B operand;
//  - decoder concat convs, skip operand: single taps [ky][kx];
//  - decoder concat convs, nearest-upsampled operand: for output class (cx, cy) the 3x3
//    taps fall on only 2 x 2 coarse pixels (coarse offset ((c + k - 1) >> 1) per axis), so
//    the conv of the upsampled tensor is a 2x2 conv of the coarse one with summed taps.
//    Blocks per (cy, j = coarse row cy - 1 + j): [cx=1 dxc=+1][cx=1 dxc=0][cx=0 dxc=0]
//    [cx=0 dxc=-1], 16 per chunk.
std::vector<uint16_t> halo_blocks(const ConvLayer& L, int sg) {
    std::vector<uint16_t> b;
    if (!L.cin1) {
        for (int j = 0; j < 9; ++j) b.push_back((uint16_t)(1u << ((2 - j % 3) * 3 + j / 3)));
    } else if (sg == 0) {
        for (int t = 0; t < 9; ++t) b.push_back((uint16_t)(1u << t));
    } else {
        const int cls[4][2] = {{1, 1}, {1, 0}, {0, 0}, {0, -1}};  // (cx, dxc)
        for (int cy = 0; cy < 2; ++cy)
            for (int j = 0; j < 2; ++j)
                for (const auto& c : cls) {
                    uint16_t m = 0;
                    for (int ky = 0; ky < 3; ++ky)
                        for (int kx = 0; kx < 3; ++kx)
                            if (((cy + ky - 1) >> 1) == cy - 1 + j && ((c[0] + kx - 1) >> 1) == c[1])
                                m |= (uint16_t)(1u << (3 * ky + kx));
                    b.push_back(m);
                }
    }
    return b;
}

// Original input channel of padded channel ch of a layer (-1 for the RGBDA padding).
static int halo_src(const ConvLayer& L, int ch) {
    const int c0 = tc_c0(L);
    if (ch < c0) return ch < L.cin0 ? ch : -1;
    return L.cin0 + (ch - c0);
}

// Weights of the halo kernel for chunks of at most ckmax channels: every K segment's
// chunks in turn, each chunk [block][N][ck] with ck = seg_ck(C_segment, ckmax), swizzled like
// the halo rows, so that one contiguous copy stages it.  value(n, src, mask) gives the (summed)
// weight of output n, original input channel src over the taps in mask; enc(v) its stored bytes.
template <class T, class Value, class Enc>
static cudaError_t halo_weights(const ConvLayer& L, int ckmax, Value value, Enc enc, void*& dst) {
    const int c0 = tc_c0(L), N = L.cout;
    const int segC[2] = {c0, L.cin1}, segOff[2] = {0, c0};
    const int nseg = L.cin1 ? 2 : 1;
    std::vector<T> w;
    for (int sg = 0; sg < nseg; ++sg) {
        const int ck = seg_ck(segC[sg], ckmax);
        const uint32_t pitch = (uint32_t)(ck * sizeof(T));
        const std::vector<uint16_t> blk = halo_blocks(L, sg);
        for (int cc = 0; cc < segC[sg] / ck; ++cc) {
            const size_t at = w.size();
            w.resize(at + blk.size() * N * ck);
            uint32_t off = 0;
            for (uint16_t m : blk)
                for (int n = 0; n < N; ++n)
                    for (int e = 0; e < ck; ++e, off += sizeof(T)) {
                        const int src = halo_src(L, segOff[sg] + cc * ck + e);
                        w[at + swizzled(off, pitch) / sizeof(T)] = enc(src >= 0 ? value(n, src, m) : 0.f);
                    }
        }
    }
    if (dst) cudaFree(dst);
    dst = nullptr;
    cudaError_t e = cudaMalloc(&dst, w.size() * sizeof(T));
    if (e != cudaSuccess) return e;
    return cudaMemcpy(dst, w.data(), w.size() * sizeof(T), cudaMemcpyHostToDevice);
}

// Sum of f(t) over the taps t in mask, in double, rounded once to float.
template <class F>
static float tap_sum(uint16_t mask, F f) {
    double acc = 0.0;
    for (int t = 0; t < 9; ++t)
        if (mask >> t & 1) acc += (double)f(t);
    return (float)acc;
}

static cudaError_t prepare_halo_weights(ConvLayer& L, int ckmax) {
    const int cin = L.cin0 + L.cin1;
    return halo_weights<__nv_bfloat16>(
        L, ckmax,
        [&](int n, int src, uint16_t m) { return tap_sum(m, [&](int t) { return L.wf[((size_t)n * cin + src) * 9 + t]; }); },
        [](float v) { return __float2bfloat16(v); }, L.wh[ck_index(ckmax)]);
}

// E4M3 weights of an FP8 layer: w * (scale of the input segment the channel comes from),
// divided by a per-output-channel scale so that each channel's largest stored |w| (after
// tap sums) maps to 448.
cudaError_t tc_prepare_fp8(ConvLayer& L) {
    const int cin = L.cin0 + L.cin1, N = L.cout, c0 = tc_c0(L);
    std::vector<float> sw(N, 0.f);
    auto scaled = [&](int n, int src, uint16_t m) {
        const float sc = src < L.cin0 ? L.in_scale[0] : L.in_scale[1];
        return tap_sum(m, [&](int t) { return L.wf[((size_t)n * cin + src) * 9 + t]; }) * sc;
    };
    const int segC[2] = {c0, L.cin1}, segOff[2] = {0, c0};
    for (int n = 0; n < N; ++n) {
        float mx = 0.f;
        for (int sg = 0; sg < (L.cin1 ? 2 : 1); ++sg)
            for (uint16_t m : halo_blocks(L, sg))
                for (int ch = segOff[sg]; ch < segOff[sg] + segC[sg]; ++ch) {
                    const int src = halo_src(L, ch);
                    if (src >= 0) mx = std::max(mx, std::fabs(scaled(n, src, m)));
                }
        sw[n] = std::max(mx, 1e-30f) / 448.0f;
    }
    cudaError_t e;
    for (int i = 0; i < 3; ++i) {
        const int ck = 32 << i;
        e = halo_weights<__nv_fp8_storage_t>(
            L, ck, [&](int n, int src, uint16_t m) { return scaled(n, src, m) / sw[n]; },
            [](float v) { return __nv_cvt_float_to_fp8(v, __NV_SATFINITE, __NV_E4M3); }, L.wh8[i]);
        if (e != cudaSuccess) return e;
    }
    if (L.wscale8) cudaFree(L.wscale8);
    L.wscale8 = nullptr;
    if ((e = cudaMalloc(&L.wscale8, 4 * N)) != cudaSuccess) return e;
    L.fp8 = true;
    L.wscale8_h = sw;
    return cudaMemcpy(L.wscale8, sw.data(), 4 * N, cudaMemcpyHostToDevice);
}

// Weight blocks staged per chunk: 9, or for the nearest-upsampled operand of a decoder
// concat conv 16 (all four classes) or the 8 of the tile's y class.
static int halo_bload(int kind, int P) { return kind == 2 ? (P == 4 ? 16 : 8) : 9; }

// Parity-class tiles stack the two x classes along N (MMAs of 2N columns, at most 256).
static bool halo_parity_ok(const ConvLayer& L, int P) { return P == 1 || (P >= 2 && 2 * L.cout <= 256); }

// Bytes of one pipeline stage of the halo kernel for a layer at tile height R, P parity
// classes per tile (decoder concat convs) and chunks of at most ckmax channels: a bound.  The
// upsampled operand of a single y class is staged in R + 1 rows and counted with R + 2, as it was
// when the rules that choose a tile were measured.
static uint32_t halo_stage_bytes(const ConvLayer& L, int R, int P, int ckmax, int esize = 2) {
    const int segC[2] = {tc_c0(L), L.cin1};
    uint32_t st = 0;
    for (int sg = 0; sg < (L.cin1 ? 2 : 1); ++sg) {
        const int ck = seg_ck(segC[sg], ckmax);
        const int kind1 = L.cin1 && sg == 0;
        const uint32_t rows = kind1 ? 2 * R + (P == 4 ? 2 : 1) : R + 2, pitch = (uint32_t)(esize * ck);
        const uint32_t plane = align_up(rows * kHaloW * pitch, 1024);
        const int kind = L.cin1 ? (sg == 0 ? 1 : 2) : 0;
        const int bl = halo_bload(kind, P);
        st = std::max(st, align_up((kind1 ? 2 : 1) * plane + (uint32_t)bl * L.cout * pitch, 1024));
    }
    return st;
}

// Default halo tile of a layer: the most pixels per tile (P parity classes x R rows x 128
// columns) whose P*R*N accumulator columns fit TMEM twice (even R when the layer pools),
// then the widest chunk (64, then 32 channels) that leaves two pipeline stages; 16-channel
// chunks only as a last resort.  LNR_CONV_TMEM1=1: tiles whose accumulators fit TMEM once
// (single-buffered), for tests of that variant.
void halo_default(const ConvLayer& L, int& R, int& P, int& ckmax) {
    const int N = L.cout;
    static const int nbuf = [] {
        const char* e = getenv("LNR_CONV_TMEM1");
        return e && atoi(e) == 1 ? 1 : 2;
    }();
    const int Ps[3] = {4, 2, 1};
    for (int pass = 0; pass < 2; ++pass)
        for (int area = 8; area >= 1; area /= 2)
            for (int pi = 0; pi < (L.cin1 ? 3 : 1); ++pi) {
                const int pp = L.cin1 ? Ps[pi] : 1;
                if (area % pp) continue;
                const int r = area / pp;
                if (nbuf * area * N > 512 || (L.pool && (r & 1)) || (L.cin1 && !halo_parity_ok(L, pp))) continue;
                const int cks[2] = {64, 32};
                for (int i = 0; i < (pass ? 1 : 2); ++i) {
                    const int ck = pass ? 16 : cks[i];
                    if (halo_stage_bytes(L, r, pp, ck) * 2 <= 220u * 1024u) {
                        R = r;
                        P = L.cin1 ? pp : 0;
                        ckmax = ck;
                        return;
                    }
                }
            }
    R = 1;
    P = L.cin1 ? 1 : 0;
    ckmax = 16;
}

// Tile of an untuned launch for a layer at (B, W, H): rows R, parity classes P and epilogue
// warps E.  The chunk width CK and whether the classes run alone (P = 1) or in pairs stay as
// halo_default chose them: they fix the order in which an accumulator's products are added,
// so the results do not depend on the choice made here.
//  - When halo_default's tile gives every SM at most one tile, it stays: smaller tiles would
//    shorten a frame that has the GPU to itself (256x256: 243 -> 217 us of kernel time), but
//    take more SM time in all, and frames of several contexts or streams share the SMs
//    (three contexts: 100.9 -> 103.0 us per frame).
//  - Else the tile with the least ceil(tiles / SMs) * (accumulators per tile + 1): every tile
//    costs its accumulators plus about one more for its halo rows and hand-overs, and tiles
//    are handed out in whole waves.  Ties go to the larger tile.
//  - TMEM holds two tiles' accumulators (the epilogue overlaps the next tile's MMAs) unless
//    that leaves fewer than 4 in a concat conv or 2 in another one, i.e. N >= 128 or 256;
//    then one tile's (each staged weight block feeds twice the pixels: decoder level 2 of a
//    1080p view, N = 128: 109 us with two buffers, 75 us with one).
//  - 12 epilogue warps for narrow outputs without pooling (N <= 32: the first conv of 8 1080p
//    views 328 -> 316 us, the last with its head 328 -> 309 us), else 8.
//  - Stores go straight to global memory: staging them in shared memory for TMA costs the
//    pipeline a stage or the epilogue a copy, and lost in every layer but two that it left
//    unchanged (first conv of a 1080p view: 72 us staged, 54 us direct).
// False when no tile fits.
bool halo_pick(const ConvLayer& L, int esize, int ck, int B, int W, int H, int num_sms, int& R, int& P, int& E) {
    const int N = L.cout, p_default = P;
    E = !L.cin1 && !L.pool && N <= 32 ? 12 : 8;
    auto tiles_of = [&](int r, int pp) {
        const int w = L.cin1 ? W / 2 : W, h = L.cin1 ? H / 2 : H;
        return (long)B * ((w + 127) / 128) * ((h + r - 1) / r) * (pp ? 4 / pp : 1);
    };
    if (tiles_of(R, P) <= num_sms) return 2 * halo_stage_bytes(L, R, P, ck, esize) <= 220u * 1024u;
    long best = -1;
    int best_area = 0;
    const int Ps[3] = {4, 2, 1};
    for (int pi = 0; pi < (L.cin1 ? 3 : 1); ++pi)
        for (int r = 8; r >= 1; r /= 2) {
            const int pp = L.cin1 ? Ps[pi] : 0, area = r * (pp ? pp : 1);
            if (L.cin1 && ((pp == 1) != (p_default == 1) || !halo_parity_ok(L, pp))) continue;
            const bool single = N * (L.cin1 ? 4 : 2) > 256;
            if (area * N > (single ? 512 : 256) || (L.pool && (r & 1))) continue;
            if (2 * halo_stage_bytes(L, r, pp, ck, esize) > 220u * 1024u) continue;
            const long cost = (tiles_of(r, pp) + num_sms - 1) / num_sms * (area + 1);
            if (best < 0 || cost < best || (cost == best && area > best_area)) {
                best = cost;
                best_area = area;
                R = r;
                P = pp;
            }
        }
    return best >= 0;
}

// Shared-memory staging of the TMA-store epilogue, bytes per epilogue warp: (pool ? 2 : 1)
// rows of 32 pixels x N channels of eo bytes, then (pool) 16 pooled pixels of ep bytes, every
// part 1024-aligned; 0 when the layout has no matching TMA swizzle (row bytes not a power of
// two >= 32).
static uint32_t halo_ostage_warp(int N, bool pool, uint32_t eo, uint32_t ep) {
    auto pow2 = [](uint32_t v) { return v >= 32 && (v & (v - 1)) == 0; };
    if (!pow2((uint32_t)N * eo) || (pool && !pow2((uint32_t)N * ep))) return 0;
    const uint32_t row = align_up(32u * N * eo, 1024);
    return (pool ? 2 : 1) * row + (pool ? align_up(16u * N * ep, 1024) : 0);
}

// Element encoding of one halo-kernel launch: BF16 or E4M3 operands, BF16 or E4M3 output.
struct HaloTypes {
    bool in8 = false, out8 = false, pool8 = false;
    float inv_out = 1.f;
    const float* cscale = nullptr;  // host, per-output-channel accumulator scale (E4M3 operands), or null
};

// head_wh, head_bh: host copies of the fused head's weights [head_o][N] and biases.
bool tc_conv_halo(const ConvLayer& L, const void* src0, const void* src1, void* out, void* pool_out,
                  const float* head_wh, const float* head_bh, float* head_out, int B, int W, int H, int head_o, int R,
                  int P, int ckmax, int O, int E, cudaStream_t st, const HaloTypes& ty, TcState& tc) {
    const int esize = ty.in8 ? 1 : 2;
    if (L.cout > kHaloMaxN || (int)L.bf.size() < L.cout || (head_out && (head_o > 4 || !head_wh || !head_bh)))
        return false;
    if (ty.in8 && ckmax < 32) return false;
    const void* whp = ty.in8 ? L.wh8[ckmax == 32 ? 0 : ckmax == 64 ? 1 : 2] : L.wh[ck_index(ckmax)];
    if (!whp) return false;
    const uint8_t* wh = static_cast<const uint8_t*>(whp);
    HParams p;
    std::memset(&p, 0, sizeof(p));
    p.ost_nbuf = 1;
    const int N = L.cout, c0 = tc_c0(L);
    if (!L.cin1) P = 0;
    else if ((P != 1 && P != 2 && P != 4) || !halo_parity_ok(L, P)) return false;
    const int NC = P ? P : 1;
    if ((R != 1 && R != 2 && R != 4 && R != 8) || NC * R * N > 512 || (L.pool && (R & 1))) return false;
    p.N = N; p.W = W; p.H = H; p.B = B; p.R = R;
    p.parity = P;
    p.wmax = std::max(1, std::min(3, 256 / N));
    // two issuers for standard tiles (each takes half the rows and windows within it); for
    // the decoder concat convs one per (row, y class) unit, up to four
    p.nmma = P ? std::min(kMmaWarps, (P == 4 ? 2 : 1) * R) : (R >= 2 ? 2 : 1);
    const cuuint64_t eb = (cuuint64_t)esize;
    const CUtensorMapDataType dt = ty.in8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    size_t w_off = 0;  // bytes into wh
    uint32_t stage = 0;
    auto set_seg = [&](HSeg& s, int kind, const void* src, int C, int Ws, int Hs) -> bool {
        s.kind = kind;
        s.ck = seg_ck(C, ckmax);
        s.pitch = (uint32_t)s.ck * esize;
        s.swz = s.pitch == 128 ? 2u : s.pitch == 64 ? 4u : 6u;
        s.rows = kind == 1 ? 2 * R + (P == 4 ? 2 : 1) : kind == 2 && P != 4 ? R + 1 : R + 2;
        s.nchunk = C / s.ck;
        const uint32_t planes = kind == 1 ? 2 : 1;
        s.plane = align_up((uint32_t)s.rows * kHaloW * s.pitch, 1024);
        s.a_bytes = planes * (uint32_t)s.rows * kHaloW * s.pitch;
        s.b_off = planes * s.plane;
        const uint32_t blk_bytes = (uint32_t)N * s.pitch;
        s.w = wh + w_off;
        s.w_chunk = (kind == 2 ? 16u : 9u) * blk_bytes;
        s.w_bytes = (uint32_t)halo_bload(kind, P) * blk_bytes;
        s.w_sel = kind == 2 && P != 4 ? 8u * blk_bytes : 0u;
        const uint32_t b_bytes = s.w_bytes;
        s.bytes = s.a_bytes + b_bytes;
        stage = std::max(stage, align_up(s.b_off + b_bytes, 1024));
        cuuint32_t es[5] = {1, 1, 1, 1, 1};
        bool ok;
        if (kind == 1) {
            cuuint64_t dims[5] = {(cuuint64_t)C, 2, (cuuint64_t)Ws / 2, (cuuint64_t)Hs, (cuuint64_t)B};
            cuuint64_t str[4] = {C * eb, 2 * C * eb, (cuuint64_t)Ws * C * eb, (cuuint64_t)Hs * Ws * C * eb};
            cuuint32_t box[5] = {(cuuint32_t)s.ck, 1, (cuuint32_t)kHaloW, (cuuint32_t)s.rows, 1};
            ok = encode_tiled(&s.a, dt, 5, const_cast<void*>(src), dims, str, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              swizzle_pitch(s.pitch), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
        } else {
            cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)Ws, (cuuint64_t)Hs, (cuuint64_t)B};
            cuuint64_t str[3] = {C * eb, (cuuint64_t)Ws * C * eb, (cuuint64_t)Hs * Ws * C * eb};
            cuuint32_t box[4] = {(cuuint32_t)s.ck, (cuuint32_t)kHaloW, (cuuint32_t)s.rows, 1};
            ok = encode_tiled(&s.a, dt, 4, const_cast<void*>(src), dims, str, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              swizzle_pitch(s.pitch), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
        }
        w_off += (size_t)s.nchunk * s.w_chunk;
        return ok;
    };
    bool ok;
    if (p.parity) {
        p.nseg = 2;
        ok = set_seg(p.seg[0], 1, src0, c0, W, H);
        ok = set_seg(p.seg[1], 2, src1, L.cin1, W / 2, H / 2) && ok;
        p.tiles_x = (W / 2 + 127) / 128;
        p.tiles_y = (H / 2 + R - 1) / R;
        p.ntiles = B * (4 / P) * p.tiles_y * p.tiles_x;
    } else {
        p.nseg = 1;
        ok = set_seg(p.seg[0], 0, src0, c0, W, H);
        p.tiles_x = (W + 127) / 128;
        p.tiles_y = (H + R - 1) / R;
        p.ntiles = B * p.tiles_y * p.tiles_x;
    }
    p.stage_bytes = stage;
    // epilogue warps: 12 for standard tiles and for tiles of two parity classes and at most
    // two rows (the decoder's full- and quarter-resolution concat convs)
    const int epi = E == 4 ? 4 : (E == 12 && (P == 0 || (P == 2 && R <= 2))) ? 12 : 8;
    // epilogue stores through staging + TMA (no fused head: its outputs are per-pixel floats)
    uint32_t stg_total = 0;
    if (O) {
        if (head_out) return false;
        const uint32_t eo = ty.out8 ? 1u : 2u, epb = ty.pool8 ? 1u : 2u;
        p.ost_unit = halo_ostage_warp(N, pool_out != nullptr, eo, epb);
        if (!p.ost_unit) return false;
        p.ostage = 1;
        p.ost_nbuf = O >= 2 ? 2 : 1;
        p.ost_warp = p.ost_nbuf * p.ost_unit;
        p.ost_row = align_up(32u * N * eo, 1024);
        p.ost_pool = (pool_out ? 2u : 1u) * p.ost_row;
        p.orow_b = std::min<uint32_t>((uint32_t)N * eo, 128u);
        p.prow_b = std::min<uint32_t>((uint32_t)N * epb, 128u);
        p.omask = p.orow_b == 128 ? 7u : p.orow_b == 64 ? 3u : 1u;
        p.pmask = p.prow_b == 128 ? 7u : p.prow_b == 64 ? 3u : 1u;
        stg_total = epi * p.ost_warp;
        cuuint32_t es[5] = {1, 1, 1, 1, 1};
        const CUtensorMapDataType odt = ty.out8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
        const cuuint64_t ro = (cuuint64_t)N * eo;
        if (P) {  // fine pixel x = 2 X + cx
            cuuint64_t dims[5] = {(cuuint64_t)N, 2, (cuuint64_t)W / 2, (cuuint64_t)H, (cuuint64_t)B};
            cuuint64_t str[4] = {ro, 2 * ro, (cuuint64_t)W * ro, (cuuint64_t)H * W * ro};
            cuuint32_t box[5] = {p.orow_b / eo, 1, 32, 1, 1};
            ok = ok && encode_tiled(&p.omap, odt, 5, out, dims, str, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                    swizzle_pitch(p.orow_b), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
        } else {
            cuuint64_t dims[4] = {(cuuint64_t)N, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
            cuuint64_t str[3] = {ro, (cuuint64_t)W * ro, (cuuint64_t)H * W * ro};
            cuuint32_t box[4] = {p.orow_b / eo, 32, 1, 1};
            ok = ok && encode_tiled(&p.omap, odt, 4, out, dims, str, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                    swizzle_pitch(p.orow_b), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
        }
        if (pool_out) {
            const CUtensorMapDataType pdt = ty.pool8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
            const cuuint64_t rp = (cuuint64_t)N * epb, Wh = (cuuint64_t)(W >> 1), Hh = (cuuint64_t)(H >> 1);
            cuuint64_t dims[4] = {(cuuint64_t)N, Wh, Hh, (cuuint64_t)B};
            cuuint64_t str[3] = {rp, Wh * rp, Hh * Wh * rp};
            cuuint32_t box[4] = {p.prow_b / epb, 16, 1, 1};
            ok = ok && encode_tiled(&p.pmap, pdt, 4, pool_out, dims, str, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                    swizzle_pitch(p.prow_b), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
        }
    }
    p.stg_bytes = stg_total;
    if (stg_total + 2 * p.stage_bytes > 220u * 1024u) return false;  // staging + two pipeline stages must fit
    p.stages = std::min<int>(8, (int)((220u * 1024u - stg_total) / p.stage_bytes));
    if (p.stages < 2) return false;
    if (!ok) {
        tc.host_err = 4;
        return true;
    }
    p.tbufs = 2 * NC * R * N <= 512 ? 2 : 1;
    uint32_t cols = 32;
    while (cols < (uint32_t)(p.tbufs * NC * R * N)) cols <<= 1;
    p.tmem_cols = cols;
    // D = FP32; operands BF16 (format 1, kind::f16) or E4M3 (format 0, kind::f8f6f4)
    p.idesc = (1u << 4) | (ty.in8 ? 0u : (1u << 7) | (1u << 10)) | ((uint32_t)(N >> 3) << 17) |
              ((uint32_t)(128 >> 4) << 24);
    for (int i = 0; i < N; ++i) {
        p.cbias[i] = L.bf[i];
        p.cscale[i] = ty.cscale ? ty.cscale[i] : 1.0f;
    }
    if (head_out)
        for (int o = 0; o < head_o; ++o) {
            for (int i = 0; i < N; ++i) p.chead[o * N + i] = head_wh[o * N + i];
            p.chead[4 * N + o] = head_bh[o];
        }
    p.out = out;
    p.pool_out = pool_out;
    p.out_fp8 = ty.out8;
    p.pool_fp8 = ty.pool8;
    p.inv_out = ty.inv_out;
    p.head_out = head_out;
    p.head_o = head_o;
    p.err = tc.err;
    const size_t smem = 1024 + (size_t)p.stages * p.stage_bytes + stg_total + 8 * (2 * p.stages + 7) + 16;
    p.stall = tc_stall_once();
    const int grid = std::min(p.ntiles, tc.num_sms);
    auto launch = [&](void (*kern)(HParams), int threads) {
        tc_allow_smem((const void*)kern);
        kern<<<grid, threads, smem, st>>>(p);
        count_launch();
        if (cudaGetLastError() != cudaSuccess) tc.host_err = 9;  // a launch that did not start: reported, never silent
    };
    auto pick4 = [&](auto par, auto ep) {
        constexpr int PP = decltype(par)::value, EE = decltype(ep)::value;
        if (ty.in8) {
            switch (R) {
                case 1: launch(k_conv_halo<1, PP, true, EE>, halo_threads(PP, 1, EE)); break;
                case 2: launch(k_conv_halo<2, PP, true, EE>, halo_threads(PP, 2, EE)); break;
                case 4: launch(k_conv_halo<4, PP, true, EE>, halo_threads(PP, 4, EE)); break;
                default: launch(k_conv_halo<8, PP, true, EE>, halo_threads(PP, 8, EE)); break;
            }
        } else {
            switch (R) {
                case 1: launch(k_conv_halo<1, PP, false, EE>, halo_threads(PP, 1, EE)); break;
                case 2: launch(k_conv_halo<2, PP, false, EE>, halo_threads(PP, 2, EE)); break;
                case 4: launch(k_conv_halo<4, PP, false, EE>, halo_threads(PP, 4, EE)); break;
                default: launch(k_conv_halo<8, PP, false, EE>, halo_threads(PP, 8, EE)); break;
            }
        }
    };
    auto pick = [&](auto par) {
        if (epi == 8) pick4(par, std::integral_constant<int, 8>{});
        else pick4(par, std::integral_constant<int, 4>{});
    };
    switch (P) {
        case 0:
            if (epi == 12) pick4(std::integral_constant<int, 0>{}, std::integral_constant<int, 12>{});
            else pick(std::integral_constant<int, 0>{});
            break;
        case 1: pick(std::integral_constant<int, 1>{}); break;
        case 2:
            if (epi == 12) {  // R is 1 or 2 here
                if (ty.in8) {
                    if (R == 1) launch(k_conv_halo<1, 2, true, 12>, halo_threads(2, 1, 12));
                    else launch(k_conv_halo<2, 2, true, 12>, halo_threads(2, 2, 12));
                } else {
                    if (R == 1) launch(k_conv_halo<1, 2, false, 12>, halo_threads(2, 1, 12));
                    else launch(k_conv_halo<2, 2, false, 12>, halo_threads(2, 2, 12));
                }
            } else {
                pick(std::integral_constant<int, 2>{});
            }
            break;
        default: pick(std::integral_constant<int, 4>{}); break;
    }
    return true;
}

// The fused level-0 encoder (k_enc0_fused): the first conv L0 on the 8-channel input and the
// second conv L1 with its 2x2 pooled output.  R output rows per tile (2 or 4).  Returns false
// when the pair or the types do not fit it (the caller then runs the two convs apart).
bool tc_enc0_fused(const ConvLayer& L0, const ConvLayer& L1, const void* in, void* out, void* pool_out, int B, int W,
                   int H, int R, cudaStream_t st, const HaloTypes& ty1, TcState& tc) {
    const int N1 = L0.cout, N2 = L1.cout;
    if (L0.cin0 != 5 || L0.cin1 || L1.cin0 != N1 || L1.cin1 || !L1.pool || !pool_out || (N1 != 16 && N1 != 32) ||
        (N2 != 16 && N2 != 32) || (R != 2 && R != 4) || ty1.in8 || ty1.out8)
        return false;
    const void* w1 = L0.wh[0];
    const void* w2 = L1.wh[ck_index(N1)];
    if (!w1 || !w2 || (int)L0.bf.size() < N1 || (int)L1.bf.size() < N2) return false;
    FParams p;
    std::memset(&p, 0, sizeof(p));
    p.W = W; p.H = H; p.B = B; p.N1 = N1; p.N2 = N2;
    p.tiles_x = (W + kFuseW - 1) / kFuseW;
    p.tiles_y = (H + R - 1) / R;
    p.ntiles = B * p.tiles_x * p.tiles_y;
    p.pitch1 = (uint32_t)N1 * 2;
    p.swz1 = p.pitch1 == 64 ? 4u : 6u;
    p.smask1 = p.pitch1 == 64 ? 3u : 1u;
    p.in_bytes = (uint32_t)(R + 4) * kHaloW * 32;
    p.in_stage = align_up(p.in_bytes, 1024);
    const uint32_t w1b = 9u * N1 * 32, w2b = 9u * N2 * p.pitch1;
    p.w1 = static_cast<const uint8_t*>(w1);
    p.w2 = static_cast<const uint8_t*>(w2);
    p.w1_bytes = w1b;
    p.w2_bytes = w2b;
    p.w1_off = 0;
    p.w2_off = align_up(w1b, 1024);
    p.in_off = p.w2_off + align_up(w2b, 1024);
    p.act_bytes = align_up((uint32_t)(R + 2) * kHaloW * p.pitch1, 1024);
    const uint32_t budget = 220u * 1024u;
    const uint32_t fixed = p.in_off + 2 * p.act_bytes;
    if (fixed + 2 * p.in_stage > budget) return false;
    p.stages = std::min<int>(4, (int)((budget - fixed) / p.in_stage));
    p.act_off = p.in_off + (uint32_t)p.stages * p.in_stage;
    uint32_t cols = 32;
    while (cols < (uint32_t)((R + 2) * N1 + 2 * R * N2)) cols <<= 1;
    if (cols > 512) return false;
    p.tmem_cols = cols;
    p.idesc1 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N1 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    p.idesc2 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N2 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    for (int i = 0; i < N1; ++i) p.b1[i] = L0.bf[i];
    for (int i = 0; i < N2; ++i) p.b2[i] = L1.bf[i];
    p.out = static_cast<__nv_bfloat16*>(out);
    p.pool_out = pool_out;
    p.pool8 = ty1.pool8 ? 1 : 0;
    p.inv_pool = ty1.inv_out;
    p.err = tc.err;
    cuuint32_t es[5] = {1, 1, 1, 1, 1};
    bool ok;
    {
        cuuint64_t dims[4] = {16, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
        cuuint64_t str[3] = {32, (cuuint64_t)W * 32, (cuuint64_t)H * W * 32};
        cuuint32_t box[4] = {16, (cuuint32_t)kHaloW, (cuuint32_t)(R + 4), 1};
        ok = encode_tiled(&p.in, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(in), dims, str, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
    if (!ok) {
        tc.host_err = 4;
        return true;
    }
    const size_t smem = 1024 + (size_t)p.act_off + 2 * p.act_bytes + 8 * (2 * p.stages + 14) + 16;
    const int grid = std::min(p.ntiles, tc.num_sms);
    auto launch = [&](void (*kern)(FParams)) {
        tc_allow_smem((const void*)kern);
        kern<<<grid, kFuseThreads, smem, st>>>(p);
        count_launch();
        if (cudaGetLastError() != cudaSuccess) tc.host_err = 9;
    };
    if (R == 2) launch(k_enc0_fused<2>);
    else launch(k_enc0_fused<4>);
    return true;
}

// The fused level-0 encoder for the pair (L0, L1) at a precision: only with BF16 operands
// for both (FP8 mode keeps them BF16 by its policy); the pooled output stores E4M3 when its
// consumer reads E4M3.
bool tc_fused_enc0(const ConvLayer& L0, const ConvLayer& L1, lnr_precision prec, const void* in, void* out,
                   void* pool_out, int B, int W, int H, int R, cudaStream_t st, TcState& tc) {
    HaloTypes ty;
    if (prec == LNR_FP8) {
        if (L0.fp8 || L1.fp8) return false;
        ty.out8 = !L1.out_bf16;
        ty.pool8 = !L1.pool_bf16;
        ty.inv_out = 1.0f / L1.out_scale;
    }
    return tc_enc0_fused(L0, L1, in, out, pool_out, B, W, H, R, st, ty, tc);
}

// Whether a test's environment switch asks for one kernel variant everywhere: the untuned
// choices then step aside.
bool tc_variant_forced() {
    static const bool forced = getenv("LNR_CONV_KERNEL") || getenv("LNR_CONV_EPI") || getenv("LNR_CONV_TMA_STORE") ||
                               getenv("LNR_CONV_TMEM1");
    return forced;
}

void tc_conv(const ConvLayer& L, lnr_precision prec, const void* src0, const void* src1, void* out, void* pool_out,
             const float* head_w, const float* head_b, const float* head_wh, const float* head_bh, float* head_out, int B,
             int W, int H, int head_o, cudaStream_t st, TcState& tc, const TcConfig* force) {
    static const int forced = [] {
        const char* e = getenv("LNR_CONV_KERNEL");
        return (e && !strcmp(e, "generic")) ? 2 : (e && !strcmp(e, "halo")) ? 3 : 0;
    }();
    // LNR_CONV_EPI=4|8|12: epilogue warps of the untuned halo kernel (default 8; 12 applies
    // to standard tiles, the concat convs keep 8)
    static const int epi = [] {
        const char* e = getenv("LNR_CONV_EPI");
        const int v = e ? atoi(e) : 8;
        return v == 4 || v == 12 ? v : 8;
    }();
    const bool fp8 = prec == LNR_FP8;
    HaloTypes ty;
    if (fp8) {
        ty.in8 = L.fp8;
        ty.out8 = head_out == nullptr && !L.out_bf16;
        ty.pool8 = !L.pool_bf16;
        ty.inv_out = 1.0f / L.out_scale;
        ty.cscale = L.fp8 ? L.wscale8_h.data() : nullptr;
    }
    TcConfig cfg;
    const auto& table = fp8 ? L.tuned8 : L.tuned;
    if (force) {
        cfg = *force;
    } else if (!forced || fp8) {
        auto it = table.find({W, H});
        if (it != table.end()) cfg = it->second;
        else if (L.cout >= 256 && !fp8) cfg.mode = 2;  // B traffic per 128-row tile favours the generic kernel there
    } else if (forced == 2) {
        cfg.mode = 2;
    }
    if (fp8 && cfg.mode == 2) cfg.mode = 0;  // the generic kernel is BF16 only
    if (cfg.mode != 2) {
        int R = cfg.R, P = cfg.P, CK = cfg.CK;
        if (cfg.mode == 0) {
            halo_default(L, R, P, CK);
            if (ty.in8) CK = std::max(32, CK);
            int E = 8;
            if (!tc_variant_forced() && halo_pick(L, ty.in8 ? 1 : 2, CK, B, W, H, tc.num_sms, R, P, E) &&
                tc_conv_halo(L, src0, src1, out, pool_out, head_wh, head_bh, head_out, B, W, H, head_o, R, P, CK, 0, E, st,
                             ty, tc))
                return;
            // a forced variant (tests): TMA-store epilogue where it fits next to two pipeline stages
            // LNR_CONV_TMA_STORE=0: direct stores; =1: one staging buffer per warp
            static const int tma_store = [] {
                const char* e = getenv("LNR_CONV_TMA_STORE");
                return e ? atoi(e) : 2;
            }();
            if (tma_store > 0)
                for (int nbuf = std::min(tma_store, 2); nbuf >= 1; --nbuf)
                    if (tc_conv_halo(L, src0, src1, out, pool_out, head_wh, head_bh, head_out, B, W, H, head_o, R, P, CK, nbuf,
                                     epi, st, ty, tc))
                        return;
        }
        if (tc_conv_halo(L, src0, src1, out, pool_out, head_wh, head_bh, head_out, B, W, H, head_o, R, P, CK, cfg.O,
                         cfg.mode == 0 ? epi : cfg.E, st, ty, tc))
            return;
        if (fp8) {  // no fallback for FP8: record and skip
            tc.host_err = 8;
            return;
        }
    }
    tc_conv_generic(L, src0, src1, out, pool_out, head_w, head_b, head_out, B, W, H, head_o, st, tc);
}

// Every valid kernel configuration of a layer: the generic kernel, and the halo kernel over
// tile heights, parity classes per tile and chunk widths that fit TMEM (double-buffered
// accumulators, or single-buffered ones for tiles of up to 512 accumulator columns) and at
// least two pipeline stages.
std::vector<TcConfig> tc_candidates(const ConvLayer& L, lnr_precision prec) {
    std::vector<TcConfig> out;
    const bool in8 = prec == LNR_FP8 && L.fp8;
    if (prec != LNR_FP8) {
        TcConfig g;
        g.mode = 2;
        out.push_back(g);
    }
    const int N = L.cout, esize = in8 ? 1 : 2;
    const int Ps[3] = {1, 2, 4};
    for (int r : {1, 2, 4, 8})
        for (int pi = 0; pi < (L.cin1 ? 3 : 1); ++pi) {
            const int P = L.cin1 ? Ps[pi] : 0, NC = P ? P : 1;
            if (NC * r * N > 512 || (L.pool && (r & 1)) || (L.cin1 && !halo_parity_ok(L, P))) continue;
            int last_ck[2] = {-1, -1};
            for (int ck : {16, 32, 64, 128}) {
                if (ck * esize > 128 || (in8 && ck < 32)) continue;
                // skip chunk widths that give the same per-segment chunks as a smaller one
                const int c0 = seg_ck(tc_c0(L), ck), c1 = L.cin1 ? seg_ck(L.cin1, ck) : 0;
                if (c0 == last_ck[0] && c1 == last_ck[1]) continue;
                last_ck[0] = c0;
                last_ck[1] = c1;
                const uint32_t sb = halo_stage_bytes(L, r, P, ck, esize);
                if (sb * 2 > 220u * 1024u) continue;
                for (int e : {4, 8, 12}) {
                    if (e == 12 && P && !(P == 2 && r <= 2)) continue;  // 12 epilogue warps: see the launch
                    TcConfig c;
                    c.mode = 1;
                    c.R = r;
                    c.P = P;
                    c.CK = ck;
                    c.E = e;
                    out.push_back(c);
                    // the same tile with the TMA-store epilogue, where its staging fits
                    const bool fp8 = prec == LNR_FP8;
                    const uint32_t eo = fp8 && !L.out_bf16 ? 1u : 2u, ep = fp8 && !L.pool_bf16 ? 1u : 2u;
                    const uint32_t wst = L.head ? 0u : halo_ostage_warp(N, L.pool, eo, ep);
                    for (int nbuf = 1; nbuf <= 2; ++nbuf)
                        if (wst && sb * 2 + (uint32_t)e * nbuf * wst <= 220u * 1024u) {
                            c.O = nbuf;
                            out.push_back(c);
                        }
                }
            }
        }
    return out;
}

// LNR_TEST_STALL_ONCE=1: the MMA issuers of the first halo or FP32 convolution of the process
// wait on a barrier nothing arrives on and give up after ~1 ms; the others then give up after ~2 s
// (the tests of the bounded waits and LNR_E_TIMEOUT).
int tc_stall_once() {
    static std::atomic<int> left{[] {
        const char* e = getenv("LNR_TEST_STALL_ONCE");
        return e && atoi(e) == 1 ? 1 : 0;
    }()};
    return left.load(std::memory_order_relaxed) ? left.exchange(0) : 0;
}

void tc_allow_smem(const void* kernel) {
    static std::mutex mu;
    static std::set<std::pair<int, const void*>> done;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return;
    std::lock_guard<std::mutex> g(mu);
    if (done.count({dev, kernel})) return;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) == cudaSuccess)
        done.insert({dev, kernel});
}

cudaError_t TcState::ensure(int sms) {
    num_sms = sms;
    if (err) return cudaSuccess;
    const cudaError_t e = cudaHostAlloc(reinterpret_cast<void**>(&err), sizeof(int), cudaHostAllocPortable);
    if (e == cudaSuccess) *err = 0;
    return e;
}

void TcState::release() {
    if (err) cudaFreeHost(err);
    err = nullptr;
}

int TcState::take_host() {
    const int code = host_err;
    host_err = 0;
    return code;
}

int TcState::take() {
    int code = take_host();
    if (!err) return code;
    if (!code) code = *static_cast<volatile int*>(err);
    *static_cast<volatile int*>(err) = 0;
    return code;
}

}  // namespace lnr
