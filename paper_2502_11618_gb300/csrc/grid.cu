// Uniform-grid build on the device (Sec. 1; Sec. 3, "Point Cloud Projection"): the only
// preprocessing of the cloud.  Points are counting-sorted by linear cell id, stably, by
// a least-significant-digit radix sort on 8-bit digits; each sorted point then stores its
// FP32 offset to its cell's FP64 origin and its packed colour.
//
// Compiled with --fmad=false: every FP64 step below is one IEEE operation, rounded on
// its own, so the offsets match an FP64 host computation bit for bit.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "lnr_internal.h"

namespace lnr {
namespace {

constexpr int kThreads = 256;
constexpr int kItems = 16;
constexpr int kTile = kThreads * kItems;  // keys per radix tile
constexpr int kWarps = kThreads / 32;

// ---- bounds ----
//
// FP64 arithmetic runs at two lanes per SM and clock here, so every kernel of the build keeps
// it to the operations whose roundings matter; minima and maxima are taken on the doubles'
// bits, mapped so that signed integers order as the (finite) doubles do.

constexpr int kBoxThreads = 384;  // a multiple of 3: the coordinates a thread reads are all of one axis

__device__ __forceinline__ long long order_bits(long long b) { return b ^ ((b >> 63) & 0x7fffffffffffffffll); }

__global__ void k_bbox_init(long long* __restrict__ box) {
    if (threadIdx.x < 6) box[threadIdx.x] = threadIdx.x < 3 ? 0x7fffffffffffffffll : -0x7fffffffffffffffll - 1;
}

// box[0..2], box[3..5]: minimum and maximum per axis (ordered bits).  Bound by reading the
// coordinates: 20M points, 480 MB, 255 us with FP64 minima, 72 us so.
__global__ void __launch_bounds__(kBoxThreads) k_bbox(const long long* __restrict__ xyz, uint64_t n3,
                                                      long long* __restrict__ box) {
    const uint64_t stride = (uint64_t)gridDim.x * kBoxThreads;  // a multiple of 3
    long long lo = 0x7fffffffffffffffll, hi = -0x7fffffffffffffffll - 1;
    uint64_t i = (uint64_t)blockIdx.x * kBoxThreads + threadIdx.x;
    for (; i + 3 * stride < n3; i += 4 * stride) {
        long long v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = __ldg(xyz + i + k * stride);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const long long o = order_bits(v[k]);
            lo = min(lo, o);
            hi = max(hi, o);
        }
    }
    for (; i < n3; i += stride) {
        const long long o = order_bits(__ldg(xyz + i));
        lo = min(lo, o);
        hi = max(hi, o);
    }
    __shared__ long long slo[kBoxThreads], shi[kBoxThreads];
    slo[threadIdx.x] = lo;
    shi[threadIdx.x] = hi;
    __syncthreads();
    for (int w = kBoxThreads / 2; w >= 3; w >>= 1) {  // 192, 96, ..., 3: multiples of 3
        if (threadIdx.x < w) {
            slo[threadIdx.x] = min(slo[threadIdx.x], slo[threadIdx.x + w]);
            shi[threadIdx.x] = max(shi[threadIdx.x], shi[threadIdx.x + w]);
        }
        __syncthreads();
    }
    if (threadIdx.x < 3) {
        atomicMin(box + threadIdx.x, slo[threadIdx.x]);
        atomicMax(box + 3 + threadIdx.x, shi[threadIdx.x]);
    }
}

// ---- cell of a point ----

struct GridFrame {
    double g0[3], cell, inv;  // inv = 1 / cell
    int dim[3];
    int log2_cell;            // cell = 2^log2_cell, where it is a power of two (dividing is a change of exponent)
    int divide;               // 1 / cell is not a normal number: always divide
};

// Cell index of coordinate x along an axis: floor((x - g0) / cell), clamped to [0, dim).  The
// quotient is taken as a product with 1 / cell (a change of exponent for a power of two), at
// most 3 units of 2^-53 of itself away from the correctly rounded one, and its floor is read
// off the upper 32 bits of the product's mantissa.  Within 2^-16 of a whole number, where the
// two could differ, and past 2^13 cells, where those bits resolve no 2^-16, the division is made.
template <bool POWER>
__device__ __forceinline__ int cell_index(double x, double g0, const GridFrame& f, int dim) {
    const double d = __dsub_rn(x, g0);
    const double q = POWER ? d : __dmul_rn(d, f.inv);
    const uint32_t top = (uint32_t)__double2hiint(q);
    if (top >> 31) return 0;
    const int e = (int)(top >> 20) - 1023 - (POWER ? f.log2_cell : 0);
    const uint32_t m = 0x80000000u | __funnelshift_l((uint32_t)__double2loint(q), top, 11);
    if (POWER) return e < 0 ? 0 : e > 30 ? dim - 1 : min((int)(m >> (31 - e)), dim - 1);
    const uint32_t frac = e < 0 ? (e == -1 ? m : 0x40000000u) : m << (e + 1);  // of the quotient (e = -2 or less: far from 1)
    if (e > 12 || f.divide || frac > 0xffff0000u || (e >= 0 && frac < 0x10000u)) {
        const double k = floor(__ddiv_rn(d, f.cell));
        return k > 0.0 ? (k < (double)(dim - 1) ? (int)k : dim - 1) : 0;
    }
    return e < 0 ? 0 : min((int)(m >> (31 - e)), dim - 1);
}

// Origin of cell k along axis a, from the table og (axis after axis) when there is one.
__device__ __forceinline__ double cell_origin(const GridFrame& f, const double* __restrict__ og, int a, int k) {
    if (og) return __ldg(og + (a > 0 ? f.dim[0] : 0) + (a > 1 ? f.dim[1] : 0) + k);
    return __dadd_rn(f.g0[a], __dmul_rn((double)k, f.cell));
}

// The double rounded to FP32 (to nearest, ties to even).  The conversion instruction shares
// the FP64 pipe's rate; normal results are rounded on the integer units.
__device__ __forceinline__ float round_f32(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int e = (int)(b >> 52 & 0x7ff) - 1023;
    if (e < -126 || e > 126) return __double2float_rn(v);  // zero, subnormal or near overflow
    const unsigned long long m = b & 0xfffffffffffffull;
    const uint32_t low = (uint32_t)m & 0x1fffffffu, head = (uint32_t)(m >> 29);
    const uint32_t up = low > 0x10000000u || (low == 0x10000000u && (head & 1u)) ? 1u : 0u;
    return __uint_as_float(((uint32_t)(b >> 32) & 0x80000000u) | (((uint32_t)(e + 127) << 23) + head + up));
}

// Cell id of every point and the histogram of its lowest digit per radix tile.  Bound by the
// FP64 pipe (one operation per SM and cycle): 20M points 2296 us with three divisions a point
// and a global count per cell, 247 us with 6 operations (268 with cells of 0.3 m), 123 us with 3
// (POWER: the cell is a power of two).
template <bool POWER>
__global__ void __launch_bounds__(kThreads) k_cell_id(const double* __restrict__ xyz, uint64_t n, const GridFrame f,
                                                      uint32_t* __restrict__ cid, uint32_t* __restrict__ hist,
                                                      uint32_t nblocks) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const uint64_t base = (uint64_t)blockIdx.x * kTile;
#pragma unroll 4
    for (int k = 0; k < kItems; ++k) {
        const uint64_t i = base + (uint64_t)k * kThreads + threadIdx.x;
        if (i < n) {
            int64_t c[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) c[a] = cell_index<POWER>(__ldg(xyz + 3 * i + a), f.g0[a], f, f.dim[a]);
            const uint32_t id = (uint32_t)((c[2] * f.dim[1] + c[1]) * f.dim[0] + c[0]);
            cid[i] = id;
            atomicAdd(&h[id & 255u], 1u);
        }
    }
    __syncthreads();
    hist[(uint64_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// ---- device-wide exclusive scan of uint32 (3 phases, recursive on the block sums) ----

constexpr int kScanItems = 8;
constexpr int kScanTile = kThreads * kScanItems;

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* total) {
    __shared__ uint32_t warp_sum[kWarps];
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < kWarps ? warp_sum[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < kWarps) warp_sum[lane] = w;
    }
    __syncthreads();
    uint32_t base = warp ? warp_sum[warp - 1] : 0;
    *total = warp_sum[kWarps - 1];
    __syncthreads();
    return base + x - v;
}

__global__ void k_scan_reduce(const uint32_t* __restrict__ in, uint64_t n, uint32_t* __restrict__ bsum) {
    uint64_t base = (uint64_t)blockIdx.x * kScanTile;
    uint32_t s = 0;
    for (int k = 0; k < kScanItems; ++k) {
        uint64_t i = base + (uint64_t)k * kThreads + threadIdx.x;
        if (i < n) s += in[i];
    }
    uint32_t tot;
    block_exclusive_scan(s, &tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void k_scan_apply(const uint32_t* __restrict__ in, uint64_t n, uint32_t* __restrict__ out,
                             const uint32_t* __restrict__ boff) {
    uint64_t base = (uint64_t)blockIdx.x * kScanTile + (uint64_t)threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    uint32_t s = 0;
    for (int k = 0; k < kScanItems; ++k) {
        uint64_t i = base + k;
        v[k] = i < n ? in[i] : 0;
        s += v[k];
    }
    uint32_t tot;
    uint32_t run = block_exclusive_scan(s, &tot) + (boff ? boff[blockIdx.x] : 0);
    for (int k = 0; k < kScanItems; ++k) {
        uint64_t i = base + k;
        if (i < n) out[i] = run;
        run += v[k];
    }
}

// Exclusive scan of n values; tmp must hold scan_tmp_words(n) words.
size_t scan_tmp_words(uint64_t n) {
    size_t w = 0;
    while (n > (uint64_t)kScanTile) {
        n = (n + kScanTile - 1) / kScanTile;
        w += 2 * n;
    }
    return w + 1;
}

void scan_exclusive(const uint32_t* in, uint32_t* out, uint64_t n, uint32_t* tmp, cudaStream_t st) {
    if (n == 0) return;
    if (n <= (uint64_t)kScanTile) {
        k_scan_apply<<<1, kThreads, 0, st>>>(in, n, out, nullptr);
        return;
    }
    uint64_t nb = (n + kScanTile - 1) / kScanTile;
    uint32_t* bsum = tmp;
    uint32_t* boff = tmp + nb;
    k_scan_reduce<<<(unsigned)nb, kThreads, 0, st>>>(in, n, bsum);
    scan_exclusive(bsum, boff, nb, tmp + 2 * nb, st);
    k_scan_apply<<<(unsigned)nb, kThreads, 0, st>>>(in, n, out, boff);
}

// ---- stable LSD radix sort of (cell id, point index) -----------------------------------

__global__ void k_radix_hist(const uint32_t* __restrict__ keys, uint64_t n, int shift,
                             uint32_t* __restrict__ hist, uint32_t nblocks) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    uint64_t base = (uint64_t)blockIdx.x * kTile;
    for (int k = 0; k < kItems; ++k) {
        uint64_t i = base + (uint64_t)k * kThreads + threadIdx.x;
        if (i < n) atomicAdd(&h[(keys[i] >> shift) & 255u], 1u);
    }
    __syncthreads();
    hist[(uint64_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// Stable scatter: warp w of a tile owns keys [w*512, (w+1)*512) of the tile and walks them
// 32 at a time in order, so ranks among equal digits follow the input order.  The tile is put
// in digit order in shared memory first, so that its runs of equal digits leave as contiguous
// pieces (20M points, the pass with scattered digits: 293 -> 206 us), and lanes of one digit
// are found with eight ballots, not match_any, whose time grows with the distinct values (206
// -> 131 us).  Bound by the integer pipe (65 %).
__global__ void __launch_bounds__(kThreads) k_radix_scatter(
    const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin, uint32_t* __restrict__ kout,
    uint32_t* __restrict__ vout, const uint32_t* __restrict__ offs, uint64_t n, int shift,
    uint32_t nblocks) {
    __shared__ uint32_t wcnt[kWarps][256];
    __shared__ uint32_t delta[256];  // global position - position in the tile, per digit
    __shared__ uint32_t sk[kTile], sv[kTile];
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int d = threadIdx.x; d < kWarps * 256; d += kThreads) (&wcnt[0][0])[d] = 0;
    __syncthreads();
    const uint64_t tile0 = (uint64_t)blockIdx.x * kTile;
    uint64_t base = tile0 + (uint64_t)warp * (kItems * 32);
    uint32_t key[kItems], val[kItems], rank[kItems];
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        uint64_t i = base + (uint64_t)r * 32 + lane;
        key[r] = i < n ? kin[i] : 0u;
        val[r] = i < n ? (vin ? vin[i] : (uint32_t)i) : 0u;
    }
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        uint64_t i = base + (uint64_t)r * 32 + lane;
        const bool valid = i < n;
        const uint32_t d = (key[r] >> shift) & 255u;
        uint32_t peers = __ballot_sync(0xffffffffu, valid);  // valid lanes of the same digit
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const uint32_t ones = __ballot_sync(0xffffffffu, (d >> b) & 1u);
            peers &= (d >> b) & 1u ? ones : ~ones;
        }
        const uint32_t old = wcnt[warp][d];
        __syncwarp();
        if (valid && lane == __ffs(peers) - 1) wcnt[warp][d] = old + __popc(peers);
        __syncwarp();
        rank[r] = old + __popc(peers & lt);
    }
    __syncthreads();
    {
        uint32_t d = threadIdx.x, run = 0, total;
        for (int w = 0; w < kWarps; ++w) run += wcnt[w][d];
        const uint32_t start = block_exclusive_scan(run, &total);
        run = start;
        for (int w = 0; w < kWarps; ++w) {
            uint32_t c = wcnt[w][d];
            wcnt[w][d] = run;
            run += c;
        }
        delta[d] = offs[(uint64_t)d * nblocks + blockIdx.x] - start;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        uint64_t i = base + (uint64_t)r * 32 + lane;
        if (i < n) {
            const uint32_t p = wcnt[warp][(key[r] >> shift) & 255u] + rank[r];
            sk[p] = key[r];
            sv[p] = val[r];
        }
    }
    __syncthreads();
    const uint32_t count = (uint32_t)min((uint64_t)kTile, n - tile0);
    for (uint32_t p = threadIdx.x; p < count; p += kThreads) {
        const uint32_t k = sk[p], to = delta[(k >> shift) & 255u] + p;
        kout[to] = k;
        vout[to] = sv[p];
    }
}

// First sorted position of every cell: cell_start[c] = number of keys below c, c = 0..C.  Two
// warps of a block find the keys of its cells, 32 probes a step, then each thread its cell's
// inside them.
__global__ void __launch_bounds__(kThreads) k_cell_bounds(const uint32_t* __restrict__ key, uint64_t n, uint64_t C,
                                                          uint32_t* __restrict__ cell_start) {
    __shared__ uint64_t ends[2];
    const uint64_t c0 = (uint64_t)blockIdx.x * kThreads;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < 2) {
        const uint64_t c = c0 + warp * (uint64_t)kThreads;
        uint64_t lo = 0, hi = n;  // keys before lo are below c, keys from hi on are not
        while (lo < hi) {
            const uint64_t step = (hi - lo + 31) / 32, at = lo + step * lane + (step - 1);
            const uint32_t below = __ballot_sync(0xffffffffu, at < hi && __ldg(key + min(at, n - 1)) < c);
            const int k = __popc(below);  // the first k probes are below c
            const uint64_t next = lo + step * k;
            hi = min(hi, next + step - 1);
            lo = min(next, hi);
        }
        if (lane == 0) ends[warp] = lo;
    }
    __syncthreads();
    const uint64_t c = c0 + threadIdx.x;
    if (c > C) return;
    uint64_t lo = ends[0], hi = ends[1];
    while (lo < hi) {
        const uint64_t mid = (lo + hi) / 2;
        if (__ldg(key + mid) < c) lo = mid + 1;
        else hi = mid;
    }
    cell_start[c] = (uint32_t)lo;
}

// Origins of the cells' rows along the three axes (dx + dy + dz values).
__global__ void k_origins(const GridFrame f, double* __restrict__ og) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, n = f.dim[0] + f.dim[1] + f.dim[2];
    if (i >= n) return;
    const int a = i < f.dim[0] ? 0 : i < f.dim[0] + f.dim[1] ? 1 : 2;
    const int k = i - (a > 0 ? f.dim[0] : 0) - (a > 1 ? f.dim[1] : 0);
    og[i] = __dadd_rn(f.g0[a], __dmul_rn((double)k, f.cell));
}

// Colour and scanner of every point in one word: the final gather then touches one sector for
// them instead of two.
__global__ void k_pack_rgbs(const uint8_t* __restrict__ rgb, const uint8_t* __restrict__ scan, uint64_t n,
                            uint32_t* __restrict__ out) {
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = (uint32_t)rgb[3 * i] | ((uint32_t)rgb[3 * i + 1] << 8) | ((uint32_t)rgb[3 * i + 2] << 16) |
             ((scan ? (uint32_t)scan[i] : 0u) << 24);
}

// Sorted points: FP32 offsets to their cells' FP64 origins, and colours.  key and val (cell
// and index of the point at each position) may lie in two of the output arrays: a thread reads
// its position's before it writes there.  Bound by gathering 24 + 4 bytes from random points,
// for which DRAM reads 173 (3.6 GB in all at 20M points): 552 us (667 with the origins in FP64
// per point and colours in separate bytes).
__global__ void __launch_bounds__(kThreads) k_offsets(const double* __restrict__ xyz, const uint32_t* __restrict__ rgbs_in,
                                                      const uint32_t* key, const uint32_t* val, uint64_t n,
                                                      const GridFrame f, const double* __restrict__ og, float* ox, float* oy,
                                                      float* oz, uint32_t* rgbs) {
    const uint64_t pos = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (pos >= n) return;
    const uint32_t id = __ldcs(key + pos), row = id / (uint32_t)f.dim[0], k = row / (uint32_t)f.dim[1];
    const int c[3] = {(int)(id - row * (uint32_t)f.dim[0]), (int)(row - k * (uint32_t)f.dim[1]), (int)k};
    // everything but the colours passes through L2 first to leave, so that the colours (4 bytes
    // a point against 24) can stay there across the gather
    const uint64_t p = __ldcs(val + pos);
    const double v[3] = {__ldcs(xyz + 3 * p), __ldcs(xyz + 3 * p + 1), __ldcs(xyz + 3 * p + 2)};
    const uint32_t col = __ldg(rgbs_in + p);
    float o[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) o[a] = round_f32(__dsub_rn(v[a], cell_origin(f, og, a, c[a])));
    __stcs(ox + pos, o[0]);
    __stcs(oy + pos, o[1]);
    __stcs(oz + pos, o[2]);
    __stcs(rgbs + pos, col);
}

}  // namespace

// Bounds of the cloud; box: device, 6 words.
cudaError_t grid_bbox(const double* xyz, uint64_t n, long long* box, double out[6], cudaStream_t st) {
    k_bbox_init<<<1, 32, 0, st>>>(box);
    const uint64_t blocks = (3 * n + kBoxThreads - 1) / kBoxThreads;
    k_bbox<<<(unsigned)std::min<uint64_t>(blocks, 152 * 5), kBoxThreads, 0, st>>>(
        reinterpret_cast<const long long*>(xyz), 3 * n, box);
    long long h[6];
    cudaError_t e = cudaMemcpyAsync(h, box, sizeof(h), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    for (int a = 0; a < 6; ++a) {
        const long long b = h[a] ^ ((h[a] >> 63) & 0x7fffffffffffffffll);
        std::memcpy(&out[a], &b, 8);
    }
    return cudaGetLastError();
}

// Sort the loaded cloud into the grid described by c->g0 / c->dims / c->cell.  The only
// temporaries are the histograms (2 KiB per 4096 points): up to kKeepTmp bytes of them stay
// with the context for its next build (allocating and freeing 16 bytes a point, as the sort's
// own buffers would take, cost 0.3 ms of a 20M-point build).
constexpr size_t kKeepTmp = 64u << 20;
cudaError_t grid_build(lnr_ctx* c, cudaStream_t st) {
    const uint64_t n = c->n;
    const int64_t C = c->ncells;
    cudaError_t e;
    GridFrame f;
    for (int a = 0; a < 3; ++a) {
        f.g0[a] = c->g0[a];
        f.dim[a] = c->dims[a];
    }
    f.cell = c->cell;
    f.inv = 1.0 / c->cell;
    int ex;
    f.divide = !std::isnormal(f.inv);
    // The change of exponent needs normal cells (a zero's exponent field stands for 2^-1023, the
    // size of a subnormal cell) that leave an overflown difference past every index.
    const bool power = std::frexp(c->cell, &ex) == 0.5 && !f.divide && std::isnormal(c->cell) && ex <= 900;
    f.log2_cell = ex - 1;
    const uint64_t nblocks = (n + kTile - 1) / kTile, nog = (uint64_t)c->dims[0] + c->dims[1] + c->dims[2];
    const bool table = nog <= 65536;
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t hb = up(4 * 256 * nblocks), sb = up(4 * scan_tmp_words(256 * nblocks)), ob = up(8 * (table ? nog : 1));
    if ((e = c->grid_tmp.ensure(2 * hb + sb + ob)) || (e = c->cell_start.ensure(4 * (C + 1))) || (e = c->ox.ensure(4 * n)) ||
        (e = c->oy.ensure(4 * n)) || (e = c->oz.ensure(4 * n)) || (e = c->rgbs.ensure(4 * n)))
        return e;
    uint8_t* at = c->grid_tmp.as<uint8_t>();
    uint32_t *hist = reinterpret_cast<uint32_t*>(at), *hscan = reinterpret_cast<uint32_t*>(at + hb),
             *stmp = reinterpret_cast<uint32_t*>(at + 2 * hb);
    double* og = table ? reinterpret_cast<double*>(at + 2 * hb + sb) : nullptr;
    // the sort's keys and values alternate between the four arrays that its result goes to
    uint32_t *kin = c->ox.as<uint32_t>(), *kout = c->oy.as<uint32_t>(), *vspare = c->oz.as<uint32_t>(),
             *vout = c->rgbs.as<uint32_t>(), *vin = nullptr;
    if (og) k_origins<<<(unsigned)((nog + 255) / 256), 256, 0, st>>>(f, og);
    (power ? k_cell_id<true> : k_cell_id<false>)<<<(unsigned)nblocks, kThreads, 0, st>>>(c->xyz.as<double>(), n, f, kin, hist, (uint32_t)nblocks);
    int bits = 1;
    while (bits < 32 && ((uint64_t)1 << bits) < (uint64_t)C) ++bits;
    for (int shift = 0; shift < bits; shift += 8) {
        if (shift) k_radix_hist<<<(unsigned)nblocks, kThreads, 0, st>>>(kin, n, shift, hist, (uint32_t)nblocks);
        scan_exclusive(hist, hscan, 256 * nblocks, stmp, st);
        k_radix_scatter<<<(unsigned)nblocks, kThreads, 0, st>>>(kin, vin, kout, vout, hscan, n, shift, (uint32_t)nblocks);
        std::swap(kin, kout);
        uint32_t* nv = vout;
        vout = vin ? vin : vspare;
        vin = nv;
    }
    k_cell_bounds<<<(unsigned)(((uint64_t)C + kThreads) / kThreads), kThreads, 0, st>>>(kin, n, (uint64_t)C,
                                                                                       c->cell_start.as<uint32_t>());
    k_offsets<<<(unsigned)((n + kThreads - 1) / kThreads), kThreads, 0, st>>>(
        c->xyz.as<double>(), c->rgbs_in.as<uint32_t>(), kin, vin, n, f, og, c->ox.as<float>(), c->oy.as<float>(),
        c->oz.as<float>(), c->rgbs.as<uint32_t>());
    e = cudaStreamSynchronize(st);
    if (c->grid_tmp.bytes > kKeepTmp) c->grid_tmp.release();
    if (e == cudaSuccess) e = cudaGetLastError();
    return e;
}

// rgbs[i] = r | g << 8 | b << 16 | scanner << 24 of every point (scan may be null: 0).
cudaError_t pack_rgbs(const uint8_t* rgb, const uint8_t* scan, uint64_t n, uint32_t* out, cudaStream_t st) {
    k_pack_rgbs<<<(unsigned)((n + kThreads - 1) / kThreads), kThreads, 0, st>>>(rgb, scan, n, out);
    const cudaError_t e = cudaStreamSynchronize(st);
    return e == cudaSuccess ? cudaGetLastError() : e;
}

// exported for the raster translation unit
void scan_exclusive_u32(const uint32_t* in, uint32_t* out, uint64_t n, uint32_t* tmp, cudaStream_t st) {
    scan_exclusive(in, out, n, tmp, st);
}
size_t scan_tmp_words_u32(uint64_t n) { return scan_tmp_words(n); }

}  // namespace lnr
