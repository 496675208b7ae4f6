// U-Net reconstruction (Fig. 1; Sec. 3, "U-Net Reconstruction"): encoder of two 3x3
// convolutions + ReLU per level with 2x2 max pooling between levels, decoder of nearest
// 2x upsampling, concatenation [skip, upsampled] and two 3x3 convolutions + ReLU, then a
// 1x1 head with a sigmoid.  Batch norm after the encoder convolutions is folded into them
// when the weights are loaded.
//
// This file holds the layer orchestration shared by every precision and the FP32 path's head.
// Pooling, upsampling and concatenation are fused into the convolutions (conv_split.cu in
// FP32, conv_tc.cu in BF16 and FP8): nothing but conv outputs is written.
#include <atomic>
#include <cmath>
#include <cuda_bf16.h>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "lnr_internal.h"

namespace lnr {
namespace {

// End of the FP32 path's 1x1 head: out[q][o] = 1 / (1 + exp(-(b[o] + sum of the parts' sums))),
// from the last conv's partial sums [image][part][4][pixel].  One thread per pixel.  Reading
// the sums (24 bytes per pixel of a 32-channel net with 3 outputs) in place of the features
// (128) took this launch on a 1080p view from 686 us, read a channel at a time, to 22 us.
__global__ void __launch_bounds__(256) k_head_f32(const float* __restrict__ z, int parts, const float* __restrict__ b,
                                                  int O, float* __restrict__ out, int64_t P, int64_t npx) {
    for (int64_t q = blockIdx.x * (int64_t)256 + threadIdx.x; q < npx; q += (int64_t)gridDim.x * 256) {
        const float* zp = z + q / P * parts * 4 * P + q % P;
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            if (o >= O) break;
            float s = __ldg(zp + o * P);
            for (int k = 1; k < parts; ++k) s += __ldg(zp + (4 * k + o) * P);
            out[q * O + o] = 1.0f / (1.0f + expf(-(s + __ldg(b + o))));
        }
    }
}

// Activation buffer slots: for level l, 4*l + {0: first conv out, 1: skip, 2: pooled, 3: decoder out}.
inline int slot(int l, int k) { return 4 * l + k; }

}  // namespace

int unet_in_kind(lnr_precision p) { return p == LNR_FP32 ? 3 : 1; }
// Bytes per pixel of the network-input buffer: 16 BF16 channels, or 8 FP32 ones (the layout
// of the stage taps at every precision).
size_t unet_in_bytes_per_px(lnr_precision) { return 32; }

// Bytes of an activation: three BF16 parts (conv_split.cu) for the FP32 network.
static size_t elem_bytes(lnr_precision p) { return p == LNR_FP32 ? 6 : 2; }

// Elements of a level's activation buffer k.  The FP32 network writes its decoder outputs over
// the level's skip tensor, which no later conv reads, so that its 6 bytes per value take about
// the memory that 4 took with a buffer of their own (the FP8 calibration reads the other
// precisions' outputs after the frame).
static size_t slot_elems(const Unet& u, int B, int W, int H, lnr_precision p, int l, int k) {
    if (k == 3 && p == LNR_FP32) return 0;
    if (k == 2) return (size_t)B * (W >> (l + 1)) * (H >> (l + 1)) * u.ch[l];
    return (size_t)B * (W >> l) * (H >> l) * u.ch[l];
}

// Activation buffers of the forward pass (the network input and output are counted with the
// frame's raster buffers): four per level, each at most the level's size (+ 256 bytes).
size_t unet_act_bytes(const Unet& u, int B, int W, int H, lnr_precision p) {
    size_t tot = 0;
    for (int l = 0; l < u.levels; ++l) {
        if (p != LNR_FP32) {
            tot += (slot_elems(u, B, W, H, p, l, 0) * elem_bytes(p) + 256) * 4;
            continue;
        }
        for (int k = 0; k < 4; ++k) tot += slot_elems(u, B, W, H, p, l, k) * elem_bytes(p) + 256;
    }
    return tot;
}

// Ensure the activation buffers of the workspace for (B, W, H); a reallocation bumps the
// workspace's allocation generation (captured graphs must be rebuilt).
cudaError_t unet_ensure(const Unet& u, Workspace& ws, lnr_precision p) {
    const size_t e = elem_bytes(p);
    cudaError_t err;
    for (int l = 0; l < u.levels; ++l) {
        for (int k = 0; k < 4; ++k) {
            const size_t n = slot_elems(u, ws.B, ws.W, ws.H, p, l, k);
            if (!n && k == 3) continue;
            const void* before = ws.act[slot(l, k)].p;
            if ((err = ws.act[slot(l, k)].ensure(n * e + 256))) return err;
            if (before != ws.act[slot(l, k)].p) ws.alloc_gen++;
        }
    }
    return cudaSuccess;
}

// One convolution launch of the forward pass: layer, sources, outputs, resolution.
struct ConvCall {
    int layer;
    const void* src0;
    const void* src1;
    void* out;
    void* pool;
    const float* head_w;   // device
    const float* head_b;
    const float* head_wh;  // host copies
    const float* head_bh;
    float* head_out;
    int W, H;
};

// The forward pass as a list of convolution launches (encoder: conv, conv (+pool) per
// level; decoder: concat conv, conv (+head on the last)); buffers from the workspace.
static std::vector<ConvCall> unet_plan(const Unet& u, Workspace& ws, lnr_precision p, const void* in, float* out) {
    std::vector<ConvCall> calls;
    const int L = u.levels;
    int ci = 0;
    const void* x = in;
    for (int l = 0; l < L; ++l) {
        const int W = ws.W >> l, H = ws.H >> l;
        void* t = ws.act[slot(l, 0)].p;
        void* s = ws.act[slot(l, 1)].p;
        void* pl = (l < L - 1) ? ws.act[slot(l, 2)].p : nullptr;
        calls.push_back({ci, x, nullptr, t, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, W, H});
        calls.push_back({ci + 1, t, nullptr, s, pl, nullptr, nullptr, nullptr, nullptr, nullptr, W, H});
        ci += 2;
        x = pl;
    }
    const void* deep = ws.act[slot(L - 1, 1)].p;
    for (int l = L - 2; l >= 0; --l) {
        const int W = ws.W >> l, H = ws.H >> l;
        void* t = ws.act[slot(l, 0)].p;
        void* d = ws.act[slot(l, p == LNR_FP32 ? 1 : 3)].p;
        const void* skip = ws.act[slot(l, 1)].p;
        calls.push_back({ci, skip, deep, t, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, W, H});
        const bool fuse_head = (l == 0) && p != LNR_FP32;
        calls.push_back({ci + 1, t, nullptr, d, nullptr, fuse_head ? u.head_w : nullptr, fuse_head ? u.head_b : nullptr,
                         fuse_head ? u.head_wh.data() : nullptr, fuse_head ? u.head_bh.data() : nullptr,
                         fuse_head ? out : nullptr, W, H});
        ci += 2;
        deep = d;
    }
    return calls;
}

static void run_call(const Unet& u, const ConvCall& k, Workspace& ws, lnr_precision p, cudaStream_t st,
                     const TcConfig* force) {
    const ConvLayer& L = u.convs[k.layer];
    if (p == LNR_FP32)
        conv_split(L, k.src0, k.src1, k.out, k.pool,
                   k.layer + 1 == (int)u.convs.size() ? static_cast<float*>(k.out) : nullptr, u.head_wh.data(), u.out_ch,
                   ws.B, k.W, k.H, st, ws.tc);
    else
        tc_conv(L, p, k.src0, k.src1, k.out, k.pool, k.head_w, k.head_b, k.head_wh, k.head_bh, k.head_out, ws.B, k.W, k.H,
                u.out_ch, st, ws.tc, force);
}

// Rows per tile of the fused level-0 encoder for B images at the layer resolution (W, H), or
// 0 to run the first two convs apart: the autotuner's choice, else LNR_CONV_FUSE0=0|2|4
// (tests), else 4 rows where its tiles (4 rows x 126 columns) number at least 300, about two
// for every SM of the chip.  There it beats the two convs apart (one view: 1920x1080 77
// against 111 us, 640x360 19 against 27; same results bit for bit); a 256x256 view has 192
// tiles in two uneven waves and a third of its columns idle: it takes 152 CTAs for 12.6 us
// where the convs apart take 64 CTAs for 19, which frames sharing the GPU pay for.
static int fuse_rows(const Unet& u, lnr_precision p, int B, int W, int H) {
    if (p == LNR_FP32 || u.convs.size() < 2) return 0;
    static const int forced = [] {
        const char* e = getenv("LNR_CONV_FUSE0");
        const int v = e ? atoi(e) : -1;
        return v == 0 || v == 2 || v == 4 ? v : -1;
    }();
    const auto& table = p == LNR_FP8 ? u.convs[0].tuned8 : u.convs[0].tuned;
    auto it = table.find({W, H});
    if (it != table.end() && it->second.F) return it->second.F;
    if (forced >= 0) return forced;
    if (it != table.end() || tc_variant_forced()) return 0;
    return (int64_t)B * ((H + 3) / 4) * ((W + 125) / 126) >= 300 ? 4 : 0;
}

void unet_forward(const lnr_ctx* c, Workspace& ws, lnr_precision p, const void* in, float* out,
                  cudaStream_t st, cudaEvent_t* layer_ev) {
    const Unet& u = c->unet;
    if (unet_ensure(u, ws, p) != cudaSuccess) return;
    int ev = 0;
    if (layer_ev) cudaEventRecord(layer_ev[ev++], st);
    const std::vector<ConvCall> calls = unet_plan(u, ws, p, in, out);
    for (size_t i = 0; i < calls.size(); ++i) {
        const ConvCall& k = calls[i];
        if (k.layer == 0 && i + 1 < calls.size() && ws.allow_fuse) {
            const int R = fuse_rows(u, p, ws.B, k.W, k.H);
            const ConvCall& k1 = calls[i + 1];
            if (R && tc_fused_enc0(u.convs[0], u.convs[1], p, k.src0, k1.out, k1.pool, ws.B, k.W, k.H, R, st, ws.tc)) {
                ++i;  // both convs done
                if (layer_ev) cudaEventRecord(layer_ev[ev++], st);
                if (layer_ev) cudaEventRecord(layer_ev[ev++], st);
                continue;
            }
        }
        run_call(u, k, ws, p, st, nullptr);
        if (layer_ev) cudaEventRecord(layer_ev[ev++], st);
    }
    if (p == LNR_FP32) {
        const void* deep = calls.back().out;
        size_t npx = (size_t)ws.B * ws.W * ws.H;
        const unsigned grid = (unsigned)std::min<size_t>((npx + 255) / 256, (size_t)c->num_sms * 8);
        k_head_f32<<<grid, 256, 0, st>>>((const float*)deep, split_head_parts(u.convs.back()), u.head_b, u.out_ch, out,
                                         (int64_t)ws.W * ws.H, (int64_t)npx);
        count_launch();
        if (layer_ev) cudaEventRecord(layer_ev[ev++], st);
    }
}

// FP8 policy.  Headroom of the static activation scales over the calibration frames'
// largest magnitudes, and the convolutions that keep BF16 operands: the full-resolution
// encoder convs (the first reads the BF16 RGBDA image) and every decoder conv at full and
// half resolution (the last one's features feed the output head).  E4M3's three mantissa
// bits cost the most accuracy there: on 16 1080p views keeping the second encoder conv in
// BF16 raised the minimum PSNR by 0.8 dB, and on a small frame with other weights the
// decoder's level-1 convs decided whether the 38 dB bar held.  Scale headroom between 2
// and 64 changed nothing measurable (E4M3 is floating point).  LNR_FP8_HEADROOM and
// LNR_FP8_BF16_LAYERS (comma-separated indices in network order, replacing the default
// set) override them for measurements.
constexpr float kFp8Headroom = 8.0f;

static float fp8_headroom() {
    const char* e = getenv("LNR_FP8_HEADROOM");
    const float v = e ? (float)atof(e) : kFp8Headroom;
    return v >= 1.0f && v <= 1e4f ? v : kFp8Headroom;
}

static bool fp8_layer_bf16(int layer, int level, bool decoder) {
    static const char* env = getenv("LNR_FP8_BF16_LAYERS");
    if (!env) return decoder ? level <= 1 : level == 0;
    static const std::vector<int> keep = [] {
        std::vector<int> v;
        for (const char* p = env; p && *p;) {
            v.push_back(atoi(p));
            p = strchr(p, ',');
            if (p) ++p;
        }
        return v;
    }();
    for (int k : keep)
        if (k == layer) return true;
    return false;
}

__global__ void k_amax_bf16(const __nv_bfloat16* __restrict__ x, size_t n, unsigned* __restrict__ out) {
    float m = 0.f;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        m = fmaxf(m, fabsf(__bfloat162float(x[i])));
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));  // non-negative floats order as integers
}

// FP8 calibration, after a BF16 forward pass on ws: the largest magnitude of every
// convolution's output gives that tensor's E4M3 scale (amax / 448); each layer's E4M3
// weights then fold in the scales of its inputs.  The first conv keeps BF16 operands (its
// input is the RGBDA image) and writes E4M3.
lnr_status unet_calibrate_fp8(lnr_ctx* c, Workspace& ws) {
    Unet& u = c->unet;
    const void* in = ws.act[4 * kMaxUnetLevels].p;
    const std::vector<ConvCall> calls = unet_plan(u, ws, LNR_BF16, in, ws.out.as<float>());
    unsigned* d_amax = nullptr;
    cudaError_t e = cudaMalloc(&d_amax, sizeof(unsigned) * calls.size());
    if (e != cudaSuccess) return cuda_fail(c, e, "calibration");
    cudaMemsetAsync(d_amax, 0, sizeof(unsigned) * calls.size(), ws.stream);
    for (size_t i = 0; i < calls.size(); ++i) {
        const ConvCall& k = calls[i];
        if (k.head_out) continue;  // the last conv's features go straight into the head
        const size_t n = (size_t)ws.B * k.W * k.H * u.convs[k.layer].cout;
        k_amax_bf16<<<1024, 256, 0, ws.stream>>>(static_cast<const __nv_bfloat16*>(k.out), n, d_amax + i);
    }
    std::vector<unsigned> h(calls.size());
    e = cudaMemcpyAsync(h.data(), d_amax, sizeof(unsigned) * calls.size(), cudaMemcpyDeviceToHost, ws.stream);
    if (!e) e = cudaStreamSynchronize(ws.stream);
    cudaFree(d_amax);
    if (e != cudaSuccess) return cuda_fail(c, e, "calibration");
    // Buffers are reused across levels (an encoder and a decoder conv of one level write
    // the same slot), so the producer of an input is the LAST earlier call that wrote it.
    std::vector<float> sc(calls.size());
    for (size_t i = 0; i < calls.size(); ++i) {
        float a;
        std::memcpy(&a, &h[i], 4);
        // headroom of 8x over the calibration view's maximum: other views may see larger
        // activations, and E4M3 keeps its relative precision over a wide exponent range, so
        // the margin costs almost nothing while clipping would cost a lot
        sc[i] = std::max(a, 1e-6f) * fp8_headroom() / 448.0f;
        u.convs[calls[i].layer].out_scale = sc[i];
        u.convs[calls[i].layer].out_bf16 = false;
    }
    auto producer = [&](size_t i, const void* buf) -> int {
        for (size_t j = i; j-- > 0;)
            if (calls[j].out == buf || (calls[j].pool && calls[j].pool == buf)) return (int)j;
        return -1;  // the BF16 input image
    };
    // BF16 operands for the first conv (the BF16 input image) and the last one (its
    // features feed the output head directly) -- optionally the whole full-resolution
    // decoder level; E4M3 everywhere else.  A producer writes BF16 for a BF16 consumer.
    for (size_t i = 0; i < calls.size(); ++i) {
        const ConvCall& k = calls[i];
        ConvLayer& L = u.convs[k.layer];
        L.pool_bf16 = false;
        const int p0 = producer(i, k.src0);
        const bool bf16 = p0 < 0 || k.head_out || fp8_layer_bf16(k.layer, L.level, k.layer >= 2 * u.levels);
        L.fp8 = !bf16;
        if (bf16) {
            for (const void* src : {k.src0, k.src1}) {
                if (!src) continue;
                const int pj = producer(i, src);
                if (pj < 0) continue;
                if (calls[pj].out == src) u.convs[calls[pj].layer].out_bf16 = true;
                else u.convs[calls[pj].layer].pool_bf16 = true;
            }
        }
    }
    for (size_t i = 0; i < calls.size(); ++i) {
        const ConvCall& k = calls[i];
        ConvLayer& L = u.convs[k.layer];
        if (!L.fp8) continue;
        L.in_scale[0] = sc[producer(i, k.src0)];
        const int p1 = k.src1 ? producer(i, k.src1) : -1;
        L.in_scale[1] = p1 >= 0 ? sc[p1] : 1.f;
        if ((e = tc_prepare_fp8(L)) != cudaSuccess) return cuda_fail(c, e, "FP8 weights");
        L.fp8 = true;
    }
    // the weights' copies, from pageable memory on the legacy stream, are done before any frame
    // on the context's stream reads them
    if ((e = cudaStreamSynchronize(nullptr)) != cudaSuccess) return cuda_fail(c, e, "FP8 weights");
    u.fp8_ready = true;
    c->unet_gen++;
    return LNR_OK;
}

// Autotuner: for every tensor-core convolution of the forward pass at the workspace's
// (B, W, H), time each candidate kernel configuration (CUDA events, `reps` launches after a
// warm-up launch) on the layer's real buffers and keep the fastest for that layer
// resolution.  Contents of the buffers do not matter: the kernels are data-independent.
lnr_status unet_autotune(lnr_ctx* c, Workspace& ws, lnr_precision p, int reps) {
    Unet& u = c->unet;
    if (p == LNR_FP32) return LNR_OK;
    cudaError_t e = unet_ensure(u, ws, p);
    if (e != cudaSuccess) return cuda_fail(c, e, "autotune buffers");
    cudaStream_t st = ws.stream;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const void* in = ws.act[4 * kMaxUnetLevels].p;
    // LNR_TUNE_LOG=1: each layer's choice on stderr; =2: also every candidate's time
    static const int log = [] {
        const char* v = getenv("LNR_TUNE_LOG");
        return v ? std::max(1, atoi(v)) : 0;
    }();
    const std::vector<ConvCall> calls = unet_plan(u, ws, p, in, ws.out.as<float>());
    std::vector<float> best_ms(calls.size(), 0.f);
    for (size_t ci = 0; ci < calls.size(); ++ci) {
        const ConvCall& k = calls[ci];
        ConvLayer& L = u.convs[k.layer];
        float best = 1e30f;
        TcConfig best_cfg;
        for (const TcConfig& cfg : tc_candidates(L, p)) {
            run_call(u, k, ws, p, st, &cfg);  // warm-up (and first-use set-up)
            cudaEventRecord(e0, st);
            for (int r = 0; r < reps; ++r) run_call(u, k, ws, p, st, &cfg);
            cudaEventRecord(e1, st);
            if ((e = cudaEventSynchronize(e1)) != cudaSuccess) break;
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (ws.tc.take()) continue;  // a configuration that failed is never chosen
            if (log >= 2)
                fprintf(stderr, "  candidate layer %d: mode %d R %d P %d ck %d O %d E %d  %.1f us\n", k.layer, cfg.mode,
                        cfg.R, cfg.P, cfg.CK, cfg.O, cfg.E, 1e3 * ms / reps);
            if (ms < best) {
                best = ms;
                best_cfg = cfg;
            }
        }
        if (e != cudaSuccess) break;
        best_ms[ci] = best;
        (p == LNR_FP8 ? L.tuned8 : L.tuned)[{k.W, k.H}] = best_cfg;
        if (log)
            fprintf(stderr, "autotune layer %d %dx%d: mode %d R %d P %d ck %d O %d E %d  %.1f us\n", k.layer, k.W, k.H,
                    best_cfg.mode, best_cfg.R, best_cfg.P, best_cfg.CK, best_cfg.O, best_cfg.E, 1e3 * best / reps);
    }
    // the first two convs fused, against the two best separate configurations
    if (e == cudaSuccess && calls.size() >= 2 && calls[0].layer == 0 && calls[1].layer == 1) {
        const ConvCall &k0 = calls[0], &k1 = calls[1];
        auto& entry = (p == LNR_FP8 ? u.convs[0].tuned8 : u.convs[0].tuned)[{k0.W, k0.H}];
        entry.F = 0;
        float best = best_ms[0] + best_ms[1];
        for (int R : {2, 4}) {
            if (!tc_fused_enc0(u.convs[0], u.convs[1], p, k0.src0, k1.out, k1.pool, ws.B, k0.W, k0.H, R, st, ws.tc)) continue;
            cudaEventRecord(e0, st);
            for (int r = 0; r < reps; ++r)
                tc_fused_enc0(u.convs[0], u.convs[1], p, k0.src0, k1.out, k1.pool, ws.B, k0.W, k0.H, R, st, ws.tc);
            cudaEventRecord(e1, st);
            if ((e = cudaEventSynchronize(e1)) != cudaSuccess) break;
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (ws.tc.take()) continue;
            if (log) fprintf(stderr, "autotune fused layers 0+1 %dx%d: R %d  %.1f us (apart %.1f us)\n", k0.W, k0.H, R,
                             1e3 * ms / reps, 1e3 * (best_ms[0] + best_ms[1]) / reps);
            if (ms < best) {
                best = ms;
                entry.F = R;
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (e != cudaSuccess) return cuda_fail(c, e, "autotune");
    c->unet_gen++;  // captured graphs hold the old kernel choices
    return LNR_OK;
}

// Convert the host weights (already batch-norm folded) to the device layouts.
lnr_status unet_prepare(lnr_ctx* c) {
    Unet& u = c->unet;
    // Each layer's layouts are converted on the host: up to eight threads take one at a time.
    std::vector<cudaError_t> err(u.convs.size(), cudaSuccess);
    std::atomic<size_t> next{0};
    auto work = [&] {
        cudaSetDevice(c->device);
        for (size_t i; (i = next++) < u.convs.size();) {
            ConvLayer& L = u.convs[i];
            try {
                if (L.b32) cudaFree(L.b32);
                L.b32 = nullptr;
                if ((err[i] = cudaMalloc(&L.b32, L.cout * 4)) != cudaSuccess) continue;
                if ((err[i] = cudaMemcpy(L.b32, L.bf.data(), L.cout * 4, cudaMemcpyHostToDevice)) != cudaSuccess) continue;
                if ((err[i] = split_prepare_layer(L)) != cudaSuccess) continue;
                if (tc_available()) err[i] = tc_prepare_layer(L, LNR_BF16);
            } catch (const std::bad_alloc&) {
                err[i] = cudaErrorMemoryAllocation;
            }
        }
    };
    std::vector<std::thread> threads;
    try {
        while (threads.size() + 1 < std::min<size_t>(8, u.convs.size())) threads.emplace_back(work);
    } catch (const std::exception&) {  // fewer threads, then
    }
    work();
    for (auto& t : threads) t.join();
    for (cudaError_t e : err)
        if (e != cudaSuccess) return cuda_fail(c, e, "U-Net weight upload");
    if (u.head_w) cudaFree(u.head_w);
    if (u.head_b) cudaFree(u.head_b);
    u.head_w = u.head_b = nullptr;
    cudaError_t e;
    if ((e = cudaMalloc(&u.head_w, u.head_wh.size() * 4)) || (e = cudaMalloc(&u.head_b, u.head_bh.size() * 4)))
        return cuda_fail(c, e, "U-Net head upload");
    cudaMemcpy(u.head_w, u.head_wh.data(), u.head_wh.size() * 4, cudaMemcpyHostToDevice);
    cudaMemcpy(u.head_b, u.head_bh.data(), u.head_bh.size() * 4, cudaMemcpyHostToDevice);
    e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return cuda_fail(c, e, "U-Net upload");
    return LNR_OK;
}

}  // namespace lnr
