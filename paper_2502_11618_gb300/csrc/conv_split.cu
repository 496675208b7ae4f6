// FP32 U-Net convolutions on the tensor cores (Fig. 1; Sec. 3, "U-Net Reconstruction").
//
// The tensor cores multiply BF16 operands exactly and add the products in FP32.  Every FP32
// value v, activation or weight, is therefore stored as three BF16 numbers
//     v = hi + mid + lo,   hi = v to kHiBits significant bits, mid = BF16(v - hi),
//                          lo = BF16(v - hi - mid)
// (together 24 significant bits), and a product of two of them as the six partial products
// hi hi, hi mid, mid hi, hi lo, lo hi, mid mid; the dropped ones are near 2^-26 of the
// product on average and at most 2^-22 of it.  (Parts have BF16's exponents: below about
// 2^-110 a value's lowest bits are lost.)  A convolution takes the MMAs of six BF16 ones, and these bound it: a tile's
// operand reads from shared memory (32 + n / 4 cycles an MMA of n columns) and the loads that
// share its bandwidth.
//
// The accumulator is the inexact part.  A tcgen05.mma rounds the sum of 16 products and the
// accumulator toward zero (measured on this GPU: that model gives 99.6 % of the results bit
// for bit), where an FP32 fused multiply-add rounds to nearest.  Two things keep the results
// more accurate than a chain of FP32 multiply-adds:
//  - the MMAs of one K chunk (16 channels x 9 taps) go into a fresh accumulator, the small
//    partial products first and the hi hi products last, so that at most 9 of its roundings
//    are at the size of the result; the epilogue warps add the chunks' accumulators in
//    registers, in FP32 rounded to nearest, while the MMAs of the next chunk run into the
//    other half of TMEM;
//  - hi has 7 bits and not BF16's 8, so that products have 14 and more of the sums are exact.
// Errors against a 64-bit network (relative 2-norm) depend on cloud, pose and weights.  Of six
// pairs of frames with FP32 multiply-adds on the same inputs (the worst 2.5e-7 against 5.3e-7, the
// best 7.5e-8 against 1.3e-7) these have 0.36 to 0.58 of the error.  Logits of a 264x136 view,
// net 32-64-128, three seeds each, for other weights than He-normal ones (5.6e-7 to 8.8e-7 against
// 6.1e-7 to 1.2e-6): pairs of taps that cancel to a thousandth 1.3e-6 against 3.0e-6; log-normal
// magnitudes (sigma 3) 2.2e-7 to 9.4e-7 against 2.2e-7 to 8.8e-7; all positive, where truncations
// add up, 2.0e-7 to 2.6e-7 against 2.0e-7 to 2.1e-7; layers scaled by 2^-100 and 2^100 in turn as
// unscaled.
//
// Measured on a 1080p view with the 4-level net (before: CUDA-core kernels, bound by their
// shared-memory operand reads): all convolutions 19.0 -> 2.4 ms.  Level 0: 107, 227 and 211
// us (the first near its DRAM floor: 400 MB out), 128-channel layers 140 us with the tensor
// pipe's front end 75 % busy, the concat convs 354 to 510 us.
//
// Tiles, operand staging and the MMA sequence of one stage are those of the halo kernel of
// conv_tc.cu: R output rows x 128 columns (or R coarse rows x 128 coarse columns of 2 or 4
// parity classes for the decoder's concat convs), the input halo staged once per chunk and
// part, taps as descriptor offsets into it.  Wide outputs are split into tiles of at most
// 128 channels.
//
// Activations lie in planes of 16 channels, [image][part][channels / 16][H][W][16]: a warp of
// the epilogue (32 pixels) writes a contiguous kilobyte, and a staged row is contiguous.
//
// Warps: 0 producer (TMA); 1-2 MMA issuers (half the rows or units each; one issuer for all
// was 10 % slower); 3-10 epilogue, two per TMEM lane quarter, each with half the tile's
// channels.  Two rings in shared memory: planes of the input halo, used in the order lo, mid,
// hi, and weight sets of a chunk (hi, mid, lo of all taps; 4 slots, so that the next chunk's
// first set is there when a chunk ends).  Holding the planes and passing the weights instead
// was slower (128 channels: 178 against 141 us).  Every wait is bounded, as in conv_tc.cu.
#include <cstring>
#include <type_traits>

#include "tc_ptx.h"

namespace lnr {
namespace {

constexpr int kEpi = 8;           // epilogue warps
constexpr int kIssuers = 2;       // MMA-issuing warps, at most
constexpr int kSplitThreads = 32 * (1 + kIssuers + kEpi);
constexpr int kBSlots = 4;        // weight sets: a chunk's three and the next one's first
constexpr float kMaxAct = 3.3e38f;  // its leading part is still finite; larger activations (infinite, past FP32) count as it
constexpr uint32_t kSmemBudget = 225u * 1024u;

struct SSeg {
    CUtensorMap a;   // 4-D {16, W, H, images} box {16, 130, rows, 1}; the concat convs' skip operand 5-D {16, 2, W/2, H, images}
    const uint8_t* w;  // weights [n tile][chunk][hi, mid, lo][block][Nt][16], each set as shared memory holds it
    int nchunk;      // chunks of 16 channels; part q of chunk cc of image n is image (3 n + q) nchunk + cc
    uint32_t w_set, w_sel;  // bytes of a set; offset of the second y class's blocks when only one's are staged
    uint32_t plane;         // bytes of one x-parity plane of a staged halo
    uint32_t a_bytes, b_bytes;
};

struct SParams {
    SSeg seg[2];
    int nseg;
    int packed;      // the network input: 16 channels hi5 | mid5 | lo5 | 0, one chunk, one plane
    int W, H, N;
    int ntn, tiles_x, tiles_y, ntiles;  // channel tiles, tiles
    int a_slots;
    uint32_t a_slot, b_slot, tmem_cols, idesc;
    __nv_bfloat16* out;       // [image][hi, mid, lo][N / 16][H][W][16], or null
    __nv_bfloat16* pool_out;  // 2x2 max-pooled output, the same layout, or null
    // The last conv's share of the 1x1 head instead of out: sums over its warps' channels,
    // [image][head part][4 outputs][H][W], parts of NT / 2 channels
    float* logits;
    int head_o;
    int* err;
    int stall;  // 1: the MMA issuers first wait on a barrier nothing arrives on, for ~1 ms (tests)
    alignas(16) float bias[256];
    alignas(16) float head[4 * 256];  // the head's weights [4][N], zero past its outputs
};

// 16 or 8 channels' three BF16 parts, each written as one 32- or 16-byte store; `part`
// elements lie between the parts.  The values are finite and at most kMaxAct.
template <int NV>
__device__ __forceinline__ void st_split(__nv_bfloat16* dst, size_t part, const float* v) {
    uint32_t w[3][NV / 2];
#pragma unroll
    for (int j = 0; j < NV / 2; ++j) {
        constexpr uint32_t drop = 24 - kHiBits;
        const uint32_t ha = (__float_as_uint(v[2 * j]) + (1u << (drop - 1))) & ~((1u << drop) - 1);
        const uint32_t hb = (__float_as_uint(v[2 * j + 1]) + (1u << (drop - 1))) & ~((1u << drop) - 1);
        const float ra = v[2 * j] - __uint_as_float(ha), rb = v[2 * j + 1] - __uint_as_float(hb);
        const __nv_bfloat162 m = __floats2bfloat162_rn(ra, rb);
        const uint32_t mw = *reinterpret_cast<const uint32_t*>(&m);
        const __nv_bfloat162 l =
            __floats2bfloat162_rn(ra - __uint_as_float(mw << 16), rb - __uint_as_float(mw & 0xffff0000u));
        w[0][j] = __byte_perm(ha, hb, 0x7632);  // the upper halves: both have 16 zero bits below
        w[1][j] = mw;
        w[2][j] = *reinterpret_cast<const uint32_t*>(&l);
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        __nv_bfloat16* d = dst + q * part;
        if (NV == 16) {
            st_32b(d, make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]),
                   make_uint4(w[q][NV / 2 - 4], w[q][NV / 2 - 3], w[q][NV / 2 - 2], w[q][NV / 2 - 1]));
        } else {
            *reinterpret_cast<uint4*>(d) = make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
        }
    }
}

// 8 TMEM columns of this warp's lanes; tmem_wait8 completes the load.
__device__ __forceinline__ void tmem_ld8_async(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait8(uint32_t (&r)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
                 :
                 : "memory");
}

// PAR = 0: R output rows x 128 columns.  PAR = 2 or 4: R coarse rows x 128 coarse columns of
// both x classes of one y class, or of all four classes.  NT output channels per tile.
template <int R, int PAR, int NT>
__global__ void __launch_bounds__(kSplitThreads, 1) k_conv_split(const __grid_constant__ SParams p) {
    using Sp = IssueSplit<R, PAR, kIssuers>;
    constexpr int NACC = R * (PAR == 0 ? 1 : PAR);   // accumulators per tile
    constexpr int NH = NT / 2;                       // channels of one epilogue warp
    constexpr int G = NH >= 16 ? 16 : 8;             // channels per TMEM load
    constexpr StageGeom kGeo{32, 0, 6};              // 16 BF16 channels per staged pixel
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* const gbase = smem_raw + (base - raw);
    const int SA = p.a_slots;
    const uint32_t a_ring = base, b_ring = base + SA * p.a_slot, bars = b_ring + kBSlots * p.b_slot;
    auto a_full = [&](int s) { return bars + 8u * s; };
    auto a_empty = [&](int s) { return bars + 8u * (SA + s); };
    auto b_full = [&](int s) { return bars + 8u * (2 * SA + s); };
    auto b_empty = [&](int s) { return bars + 8u * (2 * SA + kBSlots + s); };
    auto t_full = [&](int b) { return bars + 8u * (2 * SA + 2 * kBSlots + b); };
    auto t_empty = [&](int b) { return bars + 8u * (2 * SA + 2 * kBSlots + 2 + b); };
    const uint32_t drain = bars + 8u * (2 * SA + 2 * kBSlots + 4);
    const uint32_t tslot = bars + 8u * (2 * SA + 2 * kBSlots + 5);
    const uint32_t never = bars + 8u * (2 * SA + 2 * kBSlots + 6);  // p.stall's barrier
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < SA; ++s) {
            mbar_init(a_full(s), 1);
            mbar_init(a_empty(s), Sp::issuers);
        }
        for (int s = 0; s < kBSlots; ++s) {
            mbar_init(b_full(s), 1);
            mbar_init(b_empty(s), Sp::issuers);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(t_full(b), Sp::issuers);
            mbar_init(t_empty(b), kEpi);
        }
        mbar_init(drain, Sp::issuers);
        mbar_init(never, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(tslot, p.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(gbase + (tslot - base));

    // tile -> image n, first column and row (coarse for parity tiles), y class, channel tile;
    // the channel tiles and y classes of a region run side by side and share its halo in L2
    auto tile_of = [&](int t, int& n, int& x0, int& y0, int& py, int& nt) {
        nt = t % p.ntn;
        t /= p.ntn;
        py = 0;
        if (PAR == 2) {
            py = t & 1;
            t >>= 1;
        }
        x0 = (t % p.tiles_x) * 128;
        t /= p.tiles_x;
        y0 = (t % p.tiles_y) * R;
        n = t / p.tiles_y;
    };

    if (warp == 0 && lane == 0) {
        // ------------------------------------------------------------ producer --
        int ua = 0, ub = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
            int n, x0, y0, py, nt;
            tile_of(t, n, x0, y0, py, nt);
            for (int sg = 0; sg < p.nseg && ok; ++sg) {
                const SSeg& s = p.seg[sg];
                auto load_a = [&](int img) {
                    const int as = ua % SA;
                    if (!mbar_wait(a_empty(as), ((ua / SA) & 1) ^ 1)) return false;
                    const uint32_t dst = a_ring + as * p.a_slot;
                    mbar_expect_tx(a_full(as), s.a_bytes);
                    if (PAR && sg == 0) {
                        const int fy = PAR == 4 ? 2 * y0 - 1 : 2 * y0 + py - 1;  // first staged fine row
                        tma_5d(dst, &s.a, a_full(as), 0, 0, x0 - 1, fy, img);
                        tma_5d(dst + s.plane, &s.a, a_full(as), 0, 1, x0 - 1, fy, img);
                    } else {
                        tma_4d(dst, &s.a, a_full(as), 0, x0 - 1, y0 - 1 + py, img);
                    }
                    ++ua;
                    return true;
                };
                auto load_b = [&](int cc, int v) {
                    const int bs = ub % kBSlots;
                    if (!mbar_wait(b_empty(bs), ((ub / kBSlots) & 1) ^ 1)) return false;
                    mbar_expect_tx(b_full(bs), s.b_bytes);
                    bulk_load(b_ring + bs * p.b_slot,
                              s.w + (size_t)((nt * s.nchunk + cc) * 3 + v) * s.w_set + (uint32_t)py * s.w_sel, s.b_bytes, b_full(bs));
                    ++ub;
                    return true;
                };
                for (int cc = 0; cc < s.nchunk && ok; ++cc) {
                    if (p.packed) {
                        ok = load_a(n) && load_b(cc, 2) && load_b(cc, 1) && load_b(cc, 0);
                        continue;
                    }
                    for (int i = 0; i < 3 && ok; ++i)  // planes lo, mid, hi; weight sets hi, mid, lo
                        ok = load_a((3 * n + 2 - i) * s.nchunk + cc) && load_b(cc, i);
                }
            }
        }
        if (!ok) atomicExch(p.err, 5);
        // no copy may still be in flight when the CTA exits
        for (int k = ua > SA ? ua - SA : 0; k < ua; ++k) mbar_wait(a_full(k % SA), (k / SA) & 1);
        for (int k = ub > kBSlots ? ub - kBSlots : 0; k < ub; ++k) mbar_wait(b_full(k % kBSlots), (k / kBSlots) & 1);
    } else if (warp >= 1 && warp <= Sp::issuers && lane == 0) {
        // ----------------------------------------------------------------- MMA --
        IssueCtx q;
        q.g = warp - 1;
        q.px = 0;
        q.N = NT;
        q.idesc = p.idesc;
        // Slots and phases of the rings are kept incrementally, so that a step costs this thread
        // little beside its MMAs.
        int k = 0;                 // chunks issued
        uint32_t ub = 0;           // next use of the weight ring
        uint32_t as = 0, aph = 0;  // slot and phase of the plane ring
        bool ok = !p.stall || mbar_wait(never, 0, kStallWaitCycles);
        for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
            int n, x0, y0, nt;
            tile_of(t, n, x0, y0, q.py, nt);
            for (int sg = 0; sg < (PAR ? 2 : 1) && ok; ++sg) {
                StageGeom geo = kGeo;
                geo.plane = PAR ? p.seg[0].plane : 0;
                // the upsampled operand of one y class is staged from its first row on
                const uint32_t a_back = PAR == 2 && sg == 1 ? (uint32_t)q.py * kHaloW * 2u : 0u;
                const int nchunk = p.seg[sg].nchunk;
                for (int cc = 0; cc < nchunk; ++cc, ++k) {
                    const int b = k & 1;
                    if (!mbar_wait(t_empty(b), ((k >> 1) & 1) ^ 1)) { ok = false; break; }
                    const uint32_t d0 = tmem + (uint32_t)(b * NACC * NT);
                    // Steps of a chunk (plane x weight set), the hi hi products last: lo hi, mid hi, mid
                    // mid, hi mid, hi lo, hi hi.  The network input has hi, mid and lo in one plane; its
                    // weight sets (lo), (mid), (hi) follow in turn.
                    const int steps = p.packed ? 3 : 6;
                    const uint32_t set = p.packed ? 0x24u : 0x250u;   // 2 bits a step: weight set, in load order
                    const uint32_t a_done = p.packed ? 0x4u : 0x25u;  // 1 bit a step: last use of the plane
                    const uint32_t b_done = p.packed ? 0x7u : 0x38u;  // last use of the weight set
#pragma unroll 1
                    for (int v = 0; v < steps; ++v) {
                        const uint32_t u = ub + ((set >> (2 * v)) & 3u), bs = u % kBSlots;
                        if (!mbar_wait(a_full((int)as), aph) || !mbar_wait(b_full((int)bs), (u / kBSlots) & 1u)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        issue_stage<R, PAR, false, 1, kIssuers, true>(q, sg, ((a_ring + as * p.a_slot) >> 4) - a_back,
                                                                      (b_ring + bs * p.b_slot) >> 4, geo, d0, v == 0);
                        if ((b_done >> v) & 1u) mma_commit(b_empty((int)bs));
                        if ((a_done >> v) & 1u) {
                            mma_commit(a_empty((int)as));
                            if (++as == (uint32_t)SA) {
                                as = 0;
                                aph ^= 1u;
                            }
                        }
                    }
                    if (!ok) break;
                    ub += 3;
                    mma_commit(t_full(b));
                }
            }
        }
        if (!ok) atomicExch(p.err, 6);
        mma_commit(drain);  // every MMA issued has completed before TMEM is released
        mbar_wait(drain, 0);
    } else if (warp > kIssuers) {
        // ------------------------------------------------------------ epilogue --
        const int q = warp & 3, m = 32 * q + lane;
        const int half = (warp - kIssuers - 1) >> 2;  // which half of the tile's channels
        const int Wh = p.W >> 1, Hh = p.H >> 1;
        int chunks = p.seg[0].nchunk;
        if (p.nseg > 1) chunks += p.seg[1].nchunk;
        int k = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
            int n, x0, y0, py, nt;
            tile_of(t, n, x0, y0, py, nt);
            const int ch = nt * NT + half * NH;
            float acc[NACC][NH];
#pragma unroll
            for (int j = 0; j < NH; j += 4) {
                const float4 bv = *reinterpret_cast<const float4*>(p.bias + ch + j);
#pragma unroll
                for (int a = 0; a < NACC; ++a) {
                    acc[a][j] = bv.x;
                    acc[a][j + 1] = bv.y;
                    acc[a][j + 2] = bv.z;
                    acc[a][j + 3] = bv.w;
                }
            }
            for (int cc = 0; cc < chunks; ++cc, ++k) {
                const int b = k & 1;
                if (lane == 0) ok = mbar_wait(t_full(b), (k >> 1) & 1);
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) break;
                tc_fence_after();
                const uint32_t tb = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * NACC * NT + half * NH);
#pragma unroll
                for (int a = 0; a < NACC; ++a)
#pragma unroll
                    for (int c = 0; c < NH; c += G) {
                        if constexpr (G == 16) {
                            uint32_t u[16];
                            tmem_ld16_async(tb + (uint32_t)(a * NT + c), u);
                            tmem_wait16(u);
#pragma unroll
                            for (int j = 0; j < 16; ++j) acc[a][c + j] += __uint_as_float(u[j]);
                        } else {
                            uint32_t u[8];
                            tmem_ld8_async(tb + (uint32_t)(a * NT + c), u);
                            tmem_wait8(u);
#pragma unroll
                            for (int j = 0; j < 8; ++j) acc[a][c + j] += __uint_as_float(u[j]);
                        }
                    }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(t_empty(b));
            }
            if (!ok) break;
#pragma unroll
            for (int a = 0; a < NACC; ++a)
#pragma unroll
                // an activation past the largest value with a finite leading part counts as that
                for (int j = 0; j < NH; ++j) acc[a][j] = fminf(fmaxf(acc[a][j], 0.f), kMaxAct);
#pragma unroll
            for (int a = 0; a < NACC; ++a) {
                int x, y;
                bool in;
                if (PAR) {
                    // accumulator a: unit a / 2 = (row, y class), x class 1 before 0
                    const int u = a / 2, r = PAR == 4 ? u / 2 : u, cy = PAR == 4 ? u % 2 : py;
                    x = 2 * (x0 + m) + 1 - (a & 1);
                    y = 2 * (y0 + r) + cy;
                    in = x0 + m < Wh && y0 + r < Hh;
                } else {
                    x = x0 + m;
                    y = y0 + a;
                    in = x < p.W && y < p.H;
                }
                const size_t P = (size_t)p.H * p.W, at = (size_t)y * p.W + x;
                if (p.logits) {
                    float z[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int j = 0; j < NH; j += 4)
#pragma unroll
                        for (int o = 0; o < 4; ++o) {
                            const float4 w = *reinterpret_cast<const float4*>(p.head + o * p.N + ch + j);
                            z[o] = fmaf(w.x, acc[a][j], z[o]);
                            z[o] = fmaf(w.y, acc[a][j + 1], z[o]);
                            z[o] = fmaf(w.z, acc[a][j + 2], z[o]);
                            z[o] = fmaf(w.w, acc[a][j + 3], z[o]);
                        }
                    float* d = p.logits + ((size_t)n * (p.N / NH) + ch / NH) * 4 * P + at;
                    if (in) {
#pragma unroll
                        for (int o = 0; o < 4; ++o)
                            if (o < p.head_o) d[o * P] = z[o];
                    }
                } else if (in) {
#pragma unroll
                    for (int c = 0; c < NH; c += G)
                        st_split<G>(p.out + (((size_t)n * 3 * p.N / 16 + (ch + c) / 16) * P + at) * 16 + (ch + c) % 16,
                                    (size_t)p.N * P, &acc[a][c]);
                }
                if (PAR == 0 && NACC >= 2 && (a & 1) && p.pool_out) {
                    // 2x2 maximum with the row above and the lane holding the next column
#pragma unroll
                    for (int j = 0; j < NH; ++j) {
                        const float v = fmaxf(acc[a - 1][j], acc[a][j]);
                        acc[a - 1][j] = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
                    }
                    if (in && (m & 1) == 0) {
                        const size_t Pp = (size_t)Hh * Wh, pat = (size_t)(y >> 1) * Wh + (x >> 1);
#pragma unroll
                        for (int c = 0; c < NH; c += G)
                            st_split<G>(p.pool_out + (((size_t)n * 3 * p.N / 16 + (ch + c) / 16) * Pp + pat) * 16 + (ch + c) % 16,
                                        (size_t)p.N * Pp, &acc[a - 1][c]);
                    }
                }
            }
        }
        if (!ok && lane == 0) atomicExch(p.err, 7);
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, p.tmem_cols);
    }
}

// ------------------------------------------------------------------ host side ----

// Output channels per tile: the largest power of two that divides N, up to 128, or 64 for the
// concat convs, whose tiles then have twice the pixels (weights, which every tile loads from
// L2, are most of what those load), and for the first conv, whose single plane passes its
// held weight sets.
int tile_channels(const ConvLayer& L) {
    int nt = L.cin1 || L.cin0 == 5 ? 64 : 128;
    while (L.cout % nt) nt >>= 1;
    return nt;
}

// Cycles of one MMA of M = 128, K = 16 and n columns: the larger of its shared-memory operand
// reads and its math (measured; conv_tc.cu issues the same MMAs).
int mma_cycles(int n) { return std::max(32 + n / 4, n / 2); }

uint32_t skip_rows(int R, int P) { return 2 * R + (P == 4 ? 2 : 1); }
uint32_t plain_rows(int R, int P) { return P == 2 ? R + 1 : R + 2; }  // of the upsampled operand, or of a plain conv
uint32_t a_slot_bytes(int R, int P) {
    const uint32_t plain = align_up(plain_rows(R, P) * kHaloW * 32, 1024);
    return P ? std::max(plain, 2 * align_up(skip_rows(R, P) * kHaloW * 32, 1024)) : plain;
}
uint32_t b_slot_bytes(int P, int NT) { return align_up((P == 4 ? 16u : 9u) * NT * 32, 1024); }

// Cycles of a tile: per chunk the larger of its MMAs (all taps, parts and weight sets) and of
// loading its three input planes and weight sets from L2 at kLoadRate bytes per cycle.
constexpr int kLoadRate = 24;
long tile_cycles(const ConvLayer& L, int R, int P, int NT) {
    const bool packed = L.cin0 == 5;
    const int six = packed ? 3 : 6;
    const long w9 = 9l * NT * 32, row = kHaloW * 32;
    if (P) {
        const int units = R * (P == 4 ? 2 : 1);
        const long skip = six * units * 3l * (2 * mma_cycles(2 * NT) + 2 * mma_cycles(NT));
        const long coarse = six * units * 2l * (mma_cycles(2 * NT) + 2 * mma_cycles(NT));
        const long skip_b = 3 * (2 * skip_rows(R, P) * row + w9);
        const long coarse_b = 3 * (plain_rows(R, P) * row + (P == 4 ? 16l : 8l) * NT * 32);
        return L.cin0 / 16 * std::max(skip, skip_b / kLoadRate) + L.cin1 / 16 * std::max(coarse, coarse_b / kLoadRate);
    }
    const int issuers = std::min(R >= 2 ? 2 : 1, kIssuers), per = R / issuers;
    long c = 0;
    for (int h = 0; h < per + 2; ++h) {
        const int lo = std::max(h - 2, 0), hi = std::min(h, per - 1);
        c += mma_cycles((hi - lo + 1) * NT);
    }
    const long mma = 3l * issuers * c * six, bytes = (packed ? 1 : 3) * (R + 2) * row + 3 * w9;
    return (packed ? 1 : L.cin0 / 16) * std::max(mma, bytes / kLoadRate);
}

// Tile (R rows, P parity classes) with the least time over the waves of tiles; ties go to the
// larger tile.  On a frame that fills the GPU that is the largest that two accumulator halves
// of TMEM hold (R x P x NT = 256); a 128 x 128 layer gets one or two rows, since with more
// most SMs would have no tile.
void pick_tile(const ConvLayer& L, int NT, int B, int W, int H, int num_sms, int& R, int& P) {
    long best = -1;
    int best_area = 0;
    for (int pp : {4, 2})
        for (int r = 8; r >= 1; r /= 2) {
            const int par = L.cin1 ? pp : 0, area = r * (par ? par : 1);
            if (area * NT > 256 || (L.pool && r < 2) || (par && area > 8)) continue;
            if (2 * a_slot_bytes(r, par) + kBSlots * b_slot_bytes(par, NT) > kSmemBudget) continue;
            const int w = par ? W / 2 : W, h = par ? H / 2 : H;
            const long tiles = (long)B * ((w + 127) / 128) * ((h + r - 1) / r) * (par ? 4 / par : 1) * (L.cout / NT);
            // ~2000 cycles to start a tile's first chunk and store its results
            const long cost = (tiles + num_sms - 1) / num_sms * (tile_cycles(L, r, par, NT) + 2000);
            if (best < 0 || cost < best || (cost == best && area > best_area)) {
                best = cost;
                best_area = area;
                R = r;
                P = par;
            }
        }
}

void launch(void (*kern)(SParams), const SParams& p, int grid, size_t smem, cudaStream_t st, TcState& tc) {
    tc_allow_smem((const void*)kern);
    kern<<<grid, kSplitThreads, smem, st>>>(p);
    count_launch();
    if (cudaGetLastError() != cudaSuccess) tc.host_err = 9;
}

}  // namespace

// Split weights of a layer: per K segment [channel tile][chunk][hi, mid, lo][block][NT][16], blocks
// as for the halo kernel (taps of the concat convs' upsampled operand summed in double).  The
// network input's 16 channels are hi5 | mid5 | lo5 | 0: its weight sets are hi on all three
// parts, mid on hi and mid, lo on hi.
cudaError_t split_prepare_layer(ConvLayer& L) {
    const int NT = tile_channels(L), cin = L.cin0 + L.cin1;
    const bool packed = L.cin0 == 5;
    std::vector<__nv_bfloat16> w;
    for (int sg = 0; sg < (L.cin1 ? 2 : 1); ++sg) {
        const std::vector<uint16_t> blk = halo_blocks(L, sg);
        const int chunks = packed ? 1 : (sg ? L.cin1 : L.cin0) / 16, off = sg ? L.cin0 : 0;
        const size_t set = blk.size() * NT * 16;
        size_t at = w.size();
        w.resize(at + (size_t)(L.cout / NT) * chunks * 3 * set, __float2bfloat16(0.f));
        for (int nt = 0; nt < L.cout / NT; ++nt)
            for (int cc = 0; cc < chunks; ++cc, at += 3 * set)
                for (size_t j = 0; j < blk.size(); ++j)
                    for (int n = 0; n < NT; ++n) {
                        const float* wf = &L.wf[((size_t)(nt * NT + n) * cin + off + 16 * cc) * 9];
                        __nv_bfloat16* d = &w[at + (j * NT + n) * 16];
                        const int swz = (n >> 2 & 1) * 8;  // the 32-byte swizzle: halves swap in every other 128 bytes
                        for (int e = 0; e < (packed ? 5 : 16); ++e) {
                            double v = 0.0;
                            for (int t = 0; t < 9; ++t)
                                if (blk[j] >> t & 1) v += (double)wf[e * 9 + t];
                            const float hi = split_hi((float)v);
                            const __nv_bfloat16 mid = __float2bfloat16((float)(v - (double)hi));
                            const __nv_bfloat16 lo =
                                __float2bfloat16((float)(v - (double)hi - (double)__bfloat162float(mid)));
                            d[e ^ swz] = __float2bfloat16(hi);
                            d[set + (e ^ swz)] = mid;
                            d[2 * set + (e ^ swz)] = lo;
                            if (packed) {
                                d[(e + 5) ^ swz] = d[(e + 10) ^ swz] = d[e ^ swz];
                                d[set + ((e + 5) ^ swz)] = mid;
                            }
                        }
                    }
    }
    if (L.wsplit) cudaFree(L.wsplit);
    L.wsplit = nullptr;
    cudaError_t e = cudaMalloc(&L.wsplit, w.size() * 2);
    if (e != cudaSuccess) return e;
    return cudaMemcpy(L.wsplit, w.data(), w.size() * 2, cudaMemcpyHostToDevice);
}

int split_head_parts(const ConvLayer& L) { return 2 * (L.cout / tile_channels(L)); }

void conv_split(const ConvLayer& L, const void* src0, const void* src1, void* out, void* pool_out, float* logits,
                const float* head_wh, int head_o, int B, int W, int H, cudaStream_t st, TcState& tc) {
    SParams p;
    std::memset(&p, 0, sizeof(p));
    const int N = L.cout, NT = tile_channels(L), num_sms = tc.num_sms;
    int R = 0, P = 0;
    pick_tile(L, NT, B, W, H, num_sms, R, P);
    p.packed = L.cin0 == 5;
    p.W = W;
    p.H = H;
    p.N = N;
    p.ntn = N / NT;
    p.nseg = P ? 2 : 1;
    const CUtensorMapDataType dt = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    const CUtensorMapSwizzle sw = CU_TENSOR_MAP_SWIZZLE_32B;
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    const uint8_t* wp = static_cast<const uint8_t*>(L.wsplit);  // its sets are multiples of 256 bytes
    bool ok = wp != nullptr;
    auto map = [&](CUtensorMap* m, int rank, const void* ptr, const cuuint64_t* dims, const cuuint64_t* str,
                   const cuuint32_t* box) {
        ok = ok && encode_tiled(m, dt, rank, const_cast<void*>(ptr), dims, str, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
                                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    for (int sg = 0; sg < p.nseg; ++sg) {
        SSeg& s = p.seg[sg];
        const bool skip = P && sg == 0;
        const int Ws = sg ? W / 2 : W, Hs = sg ? H / 2 : H;
        s.nchunk = p.packed ? 1 : (sg ? L.cin1 : L.cin0) / 16;
        s.w_set = (sg ? 16u : 9u) * NT * 32;
        s.w_sel = sg && P != 4 ? 8u * NT * 32 : 0u;
        s.b_bytes = s.w_sel ? s.w_sel : s.w_set;
        s.w = wp;
        wp += (size_t)(N / NT) * s.nchunk * 3 * s.w_set;
        const cuuint64_t images = (cuuint64_t)B * (p.packed ? 1 : 3 * s.nchunk), px = 32;
        const cuuint32_t rows = skip ? skip_rows(R, P) : plain_rows(R, P);
        s.plane = align_up(rows * kHaloW * 32, 1024);
        s.a_bytes = (skip ? 2 : 1) * rows * kHaloW * 32;
        const void* src = sg ? src1 : src0;
        if (skip) {
            cuuint64_t dims[5] = {16, 2, (cuuint64_t)Ws / 2, (cuuint64_t)Hs, images};
            cuuint64_t str[4] = {px, 2 * px, (cuuint64_t)Ws * px, (cuuint64_t)Hs * Ws * px};
            cuuint32_t box[5] = {16, 1, (cuuint32_t)kHaloW, rows, 1};
            map(&s.a, 5, src, dims, str, box);
        } else {
            cuuint64_t dims[4] = {16, (cuuint64_t)Ws, (cuuint64_t)Hs, images};
            cuuint64_t str[3] = {px, (cuuint64_t)Ws * px, (cuuint64_t)Hs * Ws * px};
            cuuint32_t box[4] = {16, (cuuint32_t)kHaloW, rows, 1};
            map(&s.a, 4, src, dims, str, box);
        }
    }
    p.tiles_x = ((P ? W / 2 : W) + 127) / 128;
    p.tiles_y = ((P ? H / 2 : H) + R - 1) / R;
    p.ntiles = B * p.tiles_x * p.tiles_y * (P ? 4 / P : 1) * p.ntn;
    p.a_slot = a_slot_bytes(R, P);
    p.b_slot = b_slot_bytes(P, NT);
    p.a_slots = std::min<int>(6, (int)((kSmemBudget - kBSlots * p.b_slot) / p.a_slot));
    uint32_t cols = 32;
    while (cols < 2u * R * (P ? P : 1) * NT) cols <<= 1;
    p.tmem_cols = cols;
    // D = FP32, A and B = BF16, N and M
    p.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NT >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    p.out = static_cast<__nv_bfloat16*>(out);
    p.pool_out = static_cast<__nv_bfloat16*>(pool_out);
    p.logits = logits;
    p.head_o = head_o;
    if (logits)
        for (int i = 0; i < head_o * N; ++i) p.head[i] = head_wh[i];
    p.err = tc.err;
    p.stall = tc_stall_once();
    for (int i = 0; i < N; ++i) p.bias[i] = L.bf[i];
    if (!ok) {
        tc.host_err = 4;
        return;
    }
    const size_t smem = 1024 + (size_t)p.a_slots * p.a_slot + (size_t)kBSlots * p.b_slot +
                        8 * (2 * p.a_slots + 2 * kBSlots + 7);
    const int grid = std::min(p.ntiles, num_sms);
    auto go = [&](auto r, auto par, auto nt) {
        launch(k_conv_split<decltype(r)::value, decltype(par)::value, decltype(nt)::value>, p, grid, smem, st, tc);
    };
    using std::integral_constant;
    auto tile = [&](auto nt) {
        constexpr int T = decltype(nt)::value;
        const integral_constant<int, 1> r1{};
        const integral_constant<int, 2> r2{};
        const integral_constant<int, 4> r4{};
        const integral_constant<int, 8> r8{};
        const integral_constant<int, 0> p0{};
        if (P == 0) {
            if (R == 1) return go(r1, p0, nt);
            if (R == 2) return go(r2, p0, nt);
            if constexpr (4 * T <= 256)
                if (R == 4) return go(r4, p0, nt);
            if constexpr (8 * T <= 256) return go(r8, p0, nt);
        } else if (P == 2) {
            if (R == 1) return go(r1, r2, nt);
            if constexpr (4 * T <= 256)
                if (R == 2) return go(r2, r2, nt);
            if constexpr (8 * T <= 256) return go(r4, r2, nt);
        } else {
            if constexpr (4 * T <= 256)
                if (R == 1) return go(r1, r4, nt);
            if constexpr (8 * T <= 256) return go(r2, r4, nt);
        }
        tc.host_err = 8;
    };
    switch (NT) {
        case 16: return tile(integral_constant<int, 16>{});
        case 32: return tile(integral_constant<int, 32>{});
        case 64: return tile(integral_constant<int, 64>{});
        default: return tile(integral_constant<int, 128>{});
    }
}

}  // namespace lnr
