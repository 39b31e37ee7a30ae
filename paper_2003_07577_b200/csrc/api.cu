// C ABI of libebs: host-side validation, kernel selection, launches.  See include/ebs.h.
#include <string.h>

#include "ebs_internal.cuh"

namespace ebs {

static thread_local char g_cuda_error[256] = "";

int check_cuda(cudaError_t e) {
    if (e == cudaSuccess) return EBS_OK;
    strncpy(g_cuda_error, cudaGetErrorString(e), sizeof(g_cuda_error) - 1);
    g_cuda_error[sizeof(g_cuda_error) - 1] = '\0';
    return EBS_ERR_CUDA;
}

const ConvVariant* conv_popc_variant(int w_bits, int a_bits, int variant) {
    switch (w_bits) {
        case 1: return conv_popc_variant_w1(a_bits, variant);
        case 2: return conv_popc_variant_w2(a_bits, variant);
        case 3: return conv_popc_variant_w3(a_bits, variant);
        case 4: return conv_popc_variant_w4(a_bits, variant);
        case 5: return conv_popc_variant_w5(a_bits, variant);
        case 6: return conv_popc_variant_w6(a_bits, variant);
        case 7: return conv_popc_variant_w7(a_bits, variant);
        case 8: return conv_popc_variant_w8(a_bits, variant);
        default: return nullptr;
    }
}

const ConvVariant* conv_mma_variant(int w_bits, int a_bits, int variant) {
    if (w_bits < 1 || w_bits > 8) return nullptr;
    switch (a_bits) {
        case 1: return conv_mma_variant_a1(variant);
        case 2: return conv_mma_variant_a2(variant);
        case 3: return conv_mma_variant_a3(variant);
        case 4: return conv_mma_variant_a4(variant);
        case 5: return conv_mma_variant_a5(variant);
        case 6: return conv_mma_variant_a6(variant);
        case 7: return conv_mma_variant_a7(variant);
        case 8: return conv_mma_variant_a8(variant);
        default: return nullptr;
    }
}

unsigned long long conv_umma_timeouts() {
    return conv_umma_tile_timeouts() +
           conv_umma_strip_timeouts() + conv_umma_resident_timeouts() + conv_umma_pipe_timeouts() + fused_net_timeouts();
}

// Polls a bounded device-side wait makes before it gives up (about 40 ns each), and test flags; process-wide,
// changed only by ebs_test_set_device_wait.
static unsigned g_wait_limit = 1u << 20;
static int g_test_flags = 0;
static long long g_check_shrink = 0;      // range-checked build, tests only: result extents declared this much too short

// Range-checked build only: the device words the kernels record their first out-of-range index in.
#ifdef EBS_CHECKED
static __device__ unsigned long long g_check_words[4];
static unsigned long long* check_status_words() {
    void* ptr = nullptr;
    return cudaGetSymbolAddress(&ptr, g_check_words) == cudaSuccess ? static_cast<unsigned long long*>(ptr) : nullptr;
}
#else
static unsigned long long* check_status_words() { return nullptr; }
#endif

static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

static int out_dim(int in, int pad, int k, int stride) {
    const int span = in + 2 * pad - k;
    return span < 0 ? 0 : span / stride + 1;
}

static int validate_desc(const ebs_conv_desc* d) {
    if (!d) return EBS_ERR_INVALID_ARG;
    if (d->c_in <= 0 || d->c_out <= 0 || d->kh <= 0 || d->kw <= 0 || d->stride_h <= 0 || d->stride_w <= 0 ||
        d->pad_h < 0 || d->pad_w < 0)
        return EBS_ERR_INVALID_ARG;
    if (d->w_bits < 1 || d->w_bits > 8 || d->a_bits < 1 || d->a_bits > 8) return EBS_ERR_INVALID_ARG;
    if (d->kh > 255 || d->kw > 255 || d->c_in > (1 << 20) || d->c_out > (1 << 20)) return EBS_ERR_UNSUPPORTED;
    if (!(d->w_scale > 0.0f) || !(d->a_scale > 0.0f)) return EBS_ERR_INVALID_ARG;
    // largest |acc| = c_in*kh*kw * 2^(w_bits-1) * (2^a_bits - 1) must fit int32
    const long long s = (long long)d->c_in * d->kh * d->kw;
    if (d->w_levels != 0 && d->w_levels != 1) return EBS_ERR_INVALID_ARG;
    const long long wmax = d->w_levels ? (1LL << d->w_bits) - 1 : (1LL << (d->w_bits - 1));   // largest |weight level|
    const long long worst = s * wmax * ((1LL << d->a_bits) - 1);
    if (worst >= (1LL << 31)) return EBS_ERR_OVERFLOW;
    return EBS_OK;
}

static int sm_count() {
    int dev = 0, n = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 148;
}

// Picks the tile variant: tile_c from c_out, then the largest pixel tile that still gives every SM
// about two CTAs; problems too small for that use the small tile.
static int choose_variant(int w_bits, int a_bits, int P, int Co, bool want_packed, int sms) {
    const int tc_idx = Co <= 16 ? 0 : (Co <= 32 ? 1 : 2);
    for (int tp_idx = 2; tp_idx >= 0; --tp_idx) {
        const ConvVariant* v = conv_popc_variant(w_bits, a_bits, tc_idx * 3 + tp_idx);
        const long long ctas = (long long)((P + v->tile_p - 1) / v->tile_p) * ((Co + v->tile_c - 1) / v->tile_c);
        if (ctas >= 2LL * sms) return tc_idx * 3 + tp_idx;
    }
    const ConvVariant* v1 = conv_popc_variant(w_bits, a_bits, tc_idx * 3);
    const long long ctas1 = (long long)((P + v1->tile_p - 1) / v1->tile_p) * ((Co + v1->tile_c - 1) / v1->tile_c);
    if (ctas1 >= sms) return tc_idx * 3;
    // the small tile has 16 channels: a packed output word needs all 32 channels of a word in one CTA
    if (want_packed && Co > 16) return tc_idx * 3;
    return CONV_VARIANT_SMALL;
}

// The tensor-pipe kernels keep a table of the reduction words in shared memory, masks of valid taps
// in 32-bit words and word offsets in int: layers outside those limits use the popcount kernels.
static bool mma_path_supported(const ConvParams& p, const ebs_conv_desc* d) {
    const long long x_words = (long long)p.N * p.H * p.W * p.CW * d->a_bits;
    return p.KK <= CONV_MMA_MAX_KK && d->kh <= 32 && d->kw <= 32 && x_words < (1LL << 31);
}

// Tensor-pipe variant: tile_c from c_out; the largest warp tile that still gives every SM about a
// dozen warps (smaller layers need more, smaller tiles to hide latency).
static int choose_mma_variant(int w_bits, int a_bits, int P, int Co, int sms) {
    const int tc_idx = Co <= 16 ? 0 : (Co <= 32 ? 1 : 2);
    for (int cls = 0; cls < 2; ++cls) {
        const ConvVariant* v = conv_mma_variant(w_bits, a_bits, cls * 3 + tc_idx);
        const long long ctas = (long long)((P + v->tile_p - 1) / v->tile_p) * ((Co + v->tile_c - 1) / v->tile_c);
        if (ctas * (v->threads / 32) >= 12LL * sms) return cls * 3 + tc_idx;
    }
    return 6 + tc_idx;
}

// The persistent pipeline kernel covers layers of strides up to 2 whose strip fits.  It pays off when the layer has at least
// 64 output channels and enough outputs to fill the GPU.  Returns the pipeline variant (0..2: channel tiles of 64, 128
// and 256) or -1.
static int choose_pipe_variant(const ConvParams& p) {
    // (layers with few input channels too: the kernel spends a whole 32-channel word per tap on them, and is still
    // six times faster on an ImageNet stem, 3 -> 64 channels 7x7 stride 2, than the tap-folding per-tap kernels)
    if (p.Co < 64 || (long long)p.P * p.Co < (1LL << 20) || p.w_levels) return -1;
    // Ragged channel groups leave the lean epilogues only as packed planes; with 32-bit results the tile kernel's epilogue is
    // up to twice as fast (48 -> 77 3x3 at 28x28, batch 128: 44 us against 83).
    if ((p.Co & 31) != 0 && (p.acc || p.y)) return -1;
    // The widest channel tile that does not add much to the padding of the narrowest: a wide tile expands the activations
    // fewer times (512 -> 224 1x1 at 28x28, batch 256: 119, 66 and 44 us with 64, 128 and 256 channels; 256 -> 300 at
    // 14x14: 31, 20, 21; 192 -> 192 3x3 at 28x28: 123, 201, 134).
    auto padded = [&](int v) { return (p.Co + (64 << v) - 1) / (64 << v) * (64 << v); };
    if (padded(2) * 8 <= padded(0) * 9 && conv_umma_pipe_applies(p, 2)) return 2;
    if (padded(1) * 4 <= padded(0) * 5 && conv_umma_pipe_applies(p, 1)) return 1;
    return conv_umma_pipe_applies(p, 0) ? 0 : -1;
}

// Layers that do not fill the GPU several times over run on the tile kernel, with the channel tile of the smallest
// estimate (32, 64 or 128; wider never was the fastest).  Measured against the other families on ResNet-18/50 shapes it is
// ahead up to about three rounds of 128-channel tiles on all SMs -- 128 -> 128 3x3 at 28x28, batch 32: 9.6 against
// 14.1 us; 512 -> 512 3x3 at 7x7, batch 1: 7.8 against 17.7 us -- and behind the persistent pipeline kernel beyond (64 -> 64
// 1x1 at 56x56, batch 256: 93 against 66 us).  Returns the variant or -1.
static int choose_tile_variant(const ConvParams& p) {
    int pick = -1;
    float best = 0.0f;
    for (int v = 1; v <= 3; ++v) {
        if (v > 1 && (16 << (v - 1)) >= p.Co) break;          // a narrower tile already covers every channel
        const float c = conv_umma_cost(p, v);
        if (c >= 0.0f && (pick < 0 || c < best)) { pick = v; best = c; }
    }
    return pick;
}
static bool tile_kernel_pays(const ConvParams& p, int sms) {
    const long long tiles = (long long)((p.P + 127) / 128) * ((p.Co + 127) / 128);
    return tiles <= 3LL * sms;
}

// Layers of up to three rounds of tiles that the pipeline kernel is ahead on all the same: packed planes only, and a reduction deep
// enough that its expansion, shared by up to 512 accumulators and overlapped with the epilogue, counts for more than its longer way from
// launch to result.  Measured on the ResNet-18/50 shapes at batch 8 to 256 (us, tile and pipeline kernel; a round = one 128 x 128 tile an SM):
//  * strided k x k, 256 channels on, 1.2 rounds on: 256 -> 256 3x3 stride 2 at 28x28, batch 64 21.8 and 19.2; 512 -> 512 at 14x14, batch 256 75.8
//    and 52.2 (128 channels: 22.4 and 22.0; stride 1 stays: 512 -> 512 at 7x7, batch 256 47.4 and 55.1);
//  * 1x1 of 1024 channels on from 1.2 rounds, of 256 on from two: 2048 -> 512 at 7x7, batch 128 18.4 and 15.5; 1024 -> 256 at 14x14, batch 64 11.4
//    and 11.0; 256 -> 64 at 56x56, batch 16 9.0 and 7.6; with per-channel terms of 2048 and 512: batch 128 20.1 and 18.4; 512 -> 128 at 28x28, batch 64
//    16.4 and 15.1 (1024 -> 256, batch 64: 13.2 and 13.8; 256 -> 64: 10.5 and 10.4);
//  * 1x1 of 5 to 7 planes without terms.  Words by tensor copies: 512 channels on from 0.6 rounds, 256 on from 1.5, any from two: 512 -> 128 at 28x28,
//    batch 16, 7 planes 10.1 and 7.6; 512 -> 256, 2.2 rounds 21.0 and 12.7; 256 -> 512, 5 planes, 1.6 rounds 9.4 and 8.2; 192 -> 256, 6 planes, 2.8
//    rounds 9.2 and 8.4 (256 -> 256, 6 planes, 1.3 rounds: 5.4 and 6.9; 256 -> 1024, 7 planes, 1.35: 6.3 and 7.4).  Where a pixel is no whole 16
//    bytes, so that they come 8 or 4 bytes a lane: 128 output channels on from 2.5 rounds: 160 -> 256, 7 planes, 2.8 rounds 16.9 and 10.3; 96 -> 512, 5
//    planes 12.2 and 8.6 (608 -> 64, 7 planes, 1.6 rounds: 11.1 and 17.1; 1056 -> 128, 5 planes, 1.3: 15.0 and 18.6; 96 -> 128, 2.2: 7.0 and 7.6).
static bool pipe_before_tile(const ConvParams& p, int sms) {
    if (!p.packed_next || p.acc || p.y || p.w_levels) return false;
    const double rounds = (double)((p.P + 127) / 128) * ((p.Co + 127) / 128) / sms;
    const bool terms = p.ch_scale || p.ch_bias || p.residual || p.res_packed;
    if (p.kh * p.kw > 1) return (p.sh > 1 || p.sw > 1) && p.CW >= 8 && rounds >= 1.2;
    if (!terms && p.sh == 1 && p.sw == 1 && p.x_words >= 5 && p.x_words <= 7) {
        if (!conv_umma_pipe_copies(p, choose_pipe_variant(p))) return rounds >= 2.5 && p.Co >= 128;
        return rounds >= 2.0 || (rounds >= 1.5 && p.CW >= 8 && p.Co >= 128) || (rounds >= 0.6 && p.CW >= 16);
    }
    return (rounds >= 1.2 && p.CW >= (terms ? 64 : 32)) || (rounds >= 2.0 && p.CW >= (terms ? 16 : 8));
}

// What a layer that the tile kernel fits only in its per-tap form runs on instead of it; -1: nothing is better.  The per-tap
// form expands 128 pixels for every (tap, word), whatever the channels and bits, and its epilogue for 32-bit results and
// weight levels takes long beside a short reduction; the warp-level kernels' time grows with the plane pairs.
static int choose_beside_tap_form(const ConvParams& p, const ebs_conv_desc* d, int sms) {
    constexpr int MS_BASE = NUM_CONV_VARIANTS + NUM_CONV_MMA_VARIANTS + NUM_CONV_UMMA_VARIANTS + NUM_CONV_STRIP_VARIANTS +
                            NUM_CONV_RESIDENT_VARIANTS;
    const int mma = NUM_CONV_VARIANTS + choose_mma_variant(d->w_bits, d->a_bits, p.P, p.Co, sms);
    const bool words32 = p.acc || p.y;
    auto strip = [&](int v) { return p.kh * p.kw > 1 && conv_mma_strip_applies(p, v); };
    // at most 32 channels leave most of an accumulator empty (64 -> 16 3x3 at 200x224, two images: 10-13 us by strip, 25)
    if (p.Co <= 32) return strip(p.Co <= 16 ? 0 : 1) ? MS_BASE + (p.Co <= 16 ? 0 : 1) : mma;
    if (p.KK <= 18 && p.Co * p.CW <= 256) {
        // few pixels (64 -> 64 3x3 at 16x224: 6.9 against 8.5 us), or 32-bit results of not too many channels (64 -> 64 at 200x224,
        // two images: 29 against 34; 16 -> 48: 12 against 28; 64 -> 96: 43 either way; 8 -> 128 behind the per-tap warp-level
        // kernel); the 16-channel tile cannot pack, and is the faster one for the results
        const bool results = words32 && p.Co <= 96 && p.Co * p.CW <= 128;
        if ((p.P < (1 << 13) || (results && p.packed_next)) && strip(2)) return MS_BASE + 2;
        if (results && !p.packed_next && strip(0)) return MS_BASE;
    }
    // no strip at all: the per-tap warp-level kernel while there are few plane pairs (3 -> 64 3x3 at 200x224, 32-bit results: 16-20
    // against 28 us up to four bits, 38 against 29 at six; 64 -> 64 3x3 stride 3, two bits: 18 against 22, four bits: 23 and 22)
    if ((words32 || p.w_levels) && p.KK * (d->w_bits + d->a_bits) <= 72) return mma;
    return -1;
}

// Layers with 32-bit results and a short reduction: the tile kernel's epilogue through shared memory takes longer than those of
// the warp-level kernels.  Returns the variant of the faster one, or -1.  (us at 4 bits, accumulators and planes, this choice
// against the tile kernel.)
static int choose_for_results(const ConvParams& p, const ebs_conv_desc* d, int sms) {
    constexpr int MS_BASE = NUM_CONV_VARIANTS + NUM_CONV_MMA_VARIANTS + NUM_CONV_UMMA_VARIANTS + NUM_CONV_STRIP_VARIANTS +
                            NUM_CONV_RESIDENT_VARIANTS;
    if (!p.acc && !p.y) return -1;
    const int tile = p.Co <= 16 ? 0 : 1;
    const long long outputs = (long long)p.P * p.Co;
    if (conv_mma_strip_applies(p, tile)) {
        // 1x1: 64 -> 64 at 32x32, batch 1: 4.0 and 5.9; 128 -> 256 stride 2 at 28x28: 4.3 and 6.2; 64 -> 64 at 56x56, batch 16: 9.2 and
        // 15.7.  k x k: 64 -> 64 3x3 at 32x32, batch 1: 5.4 and 6.5; 32 -> 64 at 28x28, batch 32: 8.3 and 9.5; 32 -> 32 5x5 at
        // 32x32, batch 8: 6.9 and 7.6; not on many pixels of two words (64 -> 64 3x3 at 28x28, batch 32: 12.0 and 10.0).
        const bool shallow = p.kh * p.kw == 1 ? p.Co <= 256 && outputs <= (1LL << 22)
                                              : (p.Co * p.CW <= 64 && p.KK <= 25) || (p.Co <= 64 && p.KK <= 18 && p.P <= (1 << 14));
        return shallow ? MS_BASE + tile : -1;
    }
    // strided k x k with few plane pairs: 16 -> 32 3x3 stride 2 at 32x32, batch 128: 8.9 and 9.4, 2 bits 8.1 and 10.1 (8 bits: 13.6 and
    // 9.6); 32 -> 64 at 28x28, batch 4: 6.9 and 7.5
    const bool few_pairs = (p.sh > 1 || p.sw > 1) && p.kh * p.kw > 1 && !p.w_levels && p.Co <= 64 && outputs <= (1LL << 20) &&
                           p.KK * (d->w_bits + d->a_bits) <= 72;
    return few_pairs ? NUM_CONV_VARIANTS + choose_mma_variant(d->w_bits, d->a_bits, p.P, p.Co, sms) : -1;
}

// A validated, fully decided launch: nothing has been enqueued when conv_plan returns.
struct ConvPlan {
    ConvParams p;
    const ConvVariant* v;
    dim3 grid;
    int variant;
};

// byte_acts: packed_x holds the activations as unpacked u8 NHWC codes instead of bit planes (ebs_conv2d_i8).
static int conv_plan(const void* packed_x, int n, int h, int w, const void* packed_w, const ebs_conv_desc* d,
                     const ebs_epilogue* epi, int32_t* acc_out, float* y_out, void* packed_next, int variant,
                     ConvPlan* plan, bool byte_acts = false) {
    int rc = validate_desc(d);
    if (rc) return rc;
    if (!packed_x || !packed_w || n <= 0 || h <= 0 || w <= 0) return EBS_ERR_INVALID_ARG;
    if (!acc_out && !y_out && !packed_next) return EBS_ERR_INVALID_ARG;
    if (!aligned16(packed_x) || !aligned16(packed_w) || !aligned16(acc_out) || !aligned16(y_out) ||
        !aligned16(packed_next))
        return EBS_ERR_INVALID_ARG;
    if (h > 32000 || w > 32000) return EBS_ERR_UNSUPPORTED;
    const int Ho = out_dim(h, d->pad_h, d->kh, d->stride_h), Wo = out_dim(w, d->pad_w, d->kw, d->stride_w);
    if (Ho <= 0 || Wo <= 0) return EBS_ERR_INVALID_ARG;
    const long long P = (long long)n * Ho * Wo, in_pixels = (long long)n * h * w;
    if (P >= (1LL << 31) || in_pixels >= (1LL << 31) || P * d->c_out >= (1LL << 40)) return EBS_ERR_OVERFLOW;
    if (packed_next) {
        if (!epi || epi->next_a_bits < 1 || epi->next_a_bits > 8 || !(epi->next_a_scale > 0.0f))
            return EBS_ERR_INVALID_ARG;
    }
    if (epi) {
        if (epi->y_layout != EBS_NCHW && epi->y_layout != EBS_NHWC) return EBS_ERR_INVALID_ARG;
        if (!aligned16(epi->residual_dev) || !aligned16(epi->res_packed_dev)) return EBS_ERR_INVALID_ARG;
        if (epi->res_packed_dev && (epi->res_bits < 1 || epi->res_bits > 8)) return EBS_ERR_INVALID_ARG;
    }
    constexpr int STRIP_BASE = NUM_CONV_VARIANTS + NUM_CONV_MMA_VARIANTS + NUM_CONV_UMMA_VARIANTS;
    constexpr int RES_BASE = STRIP_BASE + NUM_CONV_STRIP_VARIANTS;
    constexpr int MS_BASE = RES_BASE + NUM_CONV_RESIDENT_VARIANTS;
    constexpr int PIPE_BASE = MS_BASE + NUM_CONV_MMA_STRIP_VARIANTS;
    if (variant >= PIPE_BASE + NUM_CONV_PIPE_VARIANTS) return EBS_ERR_INVALID_ARG;

    ConvParams& p = plan->p;
    memset(&p, 0, sizeof(p));
    p.x = static_cast<const uint32_t*>(packed_x);
    p.w = static_cast<const uint32_t*>(packed_w);
    p.w8 = static_cast<const uint8_t*>(packed_w) + packed_weight_plane_bytes(*d);
    p.Co16 = (d->c_out + 15) & ~15;
    p.N = n; p.H = h; p.W = w; p.CW = (d->c_in + 31) / 32;
    p.Co = d->c_out; p.Ho = Ho; p.Wo = Wo; p.CWo = (d->c_out + 31) / 32;
    p.kh = d->kh; p.kw = d->kw; p.sh = d->stride_h; p.sw = d->stride_w; p.ph = d->pad_h; p.pw = d->pad_w;
    p.x_words = byte_acts ? 8 : d->a_bits;
    p.KK = d->kh * d->kw * p.CW;
    p.P = (int)P;
    p.acc = acc_out; p.y = y_out; p.packed_next = static_cast<uint32_t*>(packed_next);
    p.S = d->w_scale * d->a_scale;       // one rounded fp32 multiply
    p.next_bits = 1;
    p.one = 1.0f;
    p.w_levels = d->w_levels;
    p.acc_bound = (long long)d->c_in * d->kh * d->kw * (d->w_levels ? (1LL << d->w_bits) - 1 : 1LL << (d->w_bits - 1)) *
                  (byte_acts ? 255 : (1LL << d->a_bits) - 1);
    p.fold = d->c_in <= 4 ? 8 : (d->c_in <= 8 ? 4 : (d->c_in <= 16 ? 2 : 1));
    p.fold_bits = 32 / p.fold;
    p.wait_limit = g_wait_limit;
    p.test_flags = g_test_flags;
    p.lim_x = byte_acts ? in_pixels * p.CW * 8 : in_pixels * p.CW * d->a_bits;
    p.lim_w = (long long)(packed_weight_plane_bytes(*d) / 4);
    p.lim_w8 = (long long)d->kh * d->kw * p.CW * p.Co16 * 32;
    p.lim_out = P * d->c_out - g_check_shrink;
    p.lim_pn = packed_next && epi ? P * p.CWo * epi->next_a_bits : 0;
    p.check_status = check_status_words();
    if (epi) {
        p.ch_scale = epi->ch_scale_dev; p.ch_bias = epi->ch_bias_dev; p.residual = epi->residual_dev;
        p.res_packed = static_cast<const uint32_t*>(epi->res_packed_dev); p.res_bits = epi->res_bits; p.res_scale = epi->res_scale;
        p.relu = epi->relu ? 1 : 0;
        p.y_nchw = epi->y_layout == EBS_NCHW;
        if (packed_next) { p.next_bits = epi->next_a_bits; p.inv_next = 1.0f / epi->next_a_scale; }
    }
    // the tcgen05 kernels walk any reduction length; word offsets are int
    const bool umma_ok = (long long)n * h * w * p.CW * (byte_acts ? 8 : d->a_bits) < (1LL << 31);
    const bool mma_ok = umma_ok && mma_path_supported(p, d);
    if (byte_acts) {
        // the context path exists in the persistent pipeline kernels only: whole 32-channel words of byte codes
        if ((d->c_in & 31) != 0 || d->w_levels || !umma_ok) return EBS_ERR_UNSUPPORTED;
        int pick = -1;
        for (int v = 2; v >= 0 && pick < 0; --v)
            if ((p.Co % (64 << v) == 0 || v == 0) && conv_umma_pipe_applies(p, v)) pick = v;
        if (pick < 0) return EBS_ERR_UNSUPPORTED;
        const ConvVariant* bv = conv_umma_pipe_variant(0, pick);
        if (!bv) return EBS_ERR_UNSUPPORTED;
        plan->v = bv;
        plan->grid = dim3(1, 1, 1);
        return EBS_OK;
    }
    if (variant == -2) {
        variant = choose_variant(d->w_bits, d->a_bits, p.P, p.Co, packed_next != nullptr, sm_count());
    } else if (variant < 0) {
        const bool small = tile_kernel_pays(p, sm_count()) && !pipe_before_tile(p, sm_count());
        const int tile = umma_ok && (p.Co > 16 || p.KK >= 18) ? choose_tile_variant(p) : -1;
        const int pipe = umma_ok && !(small && tile >= 0) ? choose_pipe_variant(p) : -1;
        // few channels on many pixels: the warp-level strip kernel (16 -> 16 3x3 at 32x32, batch 128: 7.1 us, the tile kernel,
        // whose accumulator is then mostly empty, 22; 32 -> 32 at 16x16: 7.2 against 8.3)
        const bool few = p.Co <= 32 && p.CW <= 2 && d->kh * d->kw > 1 && (long long)p.P > 128LL * sm_count();
        const int results = mma_ok ? choose_for_results(p, d, sm_count()) : -1;
        const int beside = mma_ok && tile >= 0 && conv_umma_tap_form(p) ? choose_beside_tap_form(p, d, sm_count()) : -1;
        if (pipe >= 0) variant = PIPE_BASE + pipe;
        else if (mma_ok && few && p.Co <= 16 && conv_mma_strip_applies(p, 0)) variant = MS_BASE;
        else if (mma_ok && few && conv_mma_strip_applies(p, 1)) variant = MS_BASE + 1;
        else if (results >= 0) variant = results;
        else if (beside >= 0) variant = beside;
        else if (tile >= 0) variant = NUM_CONV_VARIANTS + NUM_CONV_MMA_VARIANTS + tile;
        else if (mma_ok && p.Co <= 16 && d->kh * d->kw > 1 && conv_mma_strip_applies(p, 0)) variant = MS_BASE;
        else variant = mma_ok ? NUM_CONV_VARIANTS + choose_mma_variant(d->w_bits, d->a_bits, p.P, p.Co, sm_count())
                              : choose_variant(d->w_bits, d->a_bits, p.P, p.Co, packed_next != nullptr, sm_count());
    }
    constexpr int MMA_BASE = NUM_CONV_VARIANTS, UMMA_BASE = MMA_BASE + NUM_CONV_MMA_VARIANTS;
    const bool warp_level = (variant >= MMA_BASE && variant < UMMA_BASE) || (variant >= MS_BASE && variant < PIPE_BASE);
    if (variant >= NUM_CONV_VARIANTS && !(warp_level ? mma_ok : umma_ok)) return EBS_ERR_UNSUPPORTED;
    if (variant >= PIPE_BASE) {
        if (!conv_umma_pipe_applies(p, variant - PIPE_BASE)) return EBS_ERR_UNSUPPORTED;
    } else if (variant >= MS_BASE) {
        if (!conv_mma_strip_applies(p, variant - MS_BASE)) return EBS_ERR_UNSUPPORTED;
    } else if (variant >= RES_BASE) {
        if (!conv_umma_resident_applies(p, variant - RES_BASE)) return EBS_ERR_UNSUPPORTED;
    } else if (variant >= STRIP_BASE) {
        if (!conv_umma_strip_applies(p, variant - STRIP_BASE)) return EBS_ERR_UNSUPPORTED;
    } else if (variant >= UMMA_BASE) {
        if (!conv_umma_applies(p, variant - UMMA_BASE)) return EBS_ERR_UNSUPPORTED;
    }
    const ConvVariant* v =
        variant >= PIPE_BASE ? conv_umma_pipe_variant(d->a_bits, variant - PIPE_BASE) :
        variant >= MS_BASE ? conv_mma_strip_variant(d->a_bits, variant - MS_BASE) :
        variant >= RES_BASE ? conv_umma_resident_variant(d->a_bits, variant - RES_BASE) :
        variant >= STRIP_BASE ? conv_umma_strip_variant(d->a_bits, variant - STRIP_BASE) :
        variant >= UMMA_BASE ? conv_umma_variant(d->a_bits, variant - UMMA_BASE) :
        variant >= MMA_BASE ? conv_mma_variant(d->w_bits, d->a_bits, variant - MMA_BASE)
                            : conv_popc_variant(d->w_bits, d->a_bits, variant);
    if (!v) return EBS_ERR_UNSUPPORTED;
    if (packed_next && (v->tile_c % 32) != 0 && v->tile_c < p.Co) return EBS_ERR_UNSUPPORTED;
    const long long gx = (P + v->tile_p - 1) / v->tile_p, gy = (p.Co + v->tile_c - 1) / v->tile_c;
    if (gy > 65535) return EBS_ERR_UNSUPPORTED;
    plan->v = v;
    plan->variant = variant;
    plan->grid = dim3((unsigned)gx, (unsigned)gy, 1);
    return EBS_OK;
}

static int conv_launch(const ConvPlan& plan, void* stream) {
    const int rc = plan.v->launch(plan.p, plan.grid, static_cast<cudaStream_t>(stream));
    if (rc) return rc;
    return check_cuda(cudaGetLastError());
}

static int conv_impl(const void* packed_x, int n, int h, int w, const void* packed_w, const ebs_conv_desc* d,
                     const ebs_epilogue* epi, int32_t* acc_out, float* y_out, void* packed_next, void* stream,
                     int variant) {
    ConvPlan plan;
    const int rc = conv_plan(packed_x, n, h, w, packed_w, d, epi, acc_out, y_out, packed_next, variant, &plan);
    if (rc) return rc;
    return conv_launch(plan, stream);
}

}  // namespace ebs

using namespace ebs;

extern "C" {

int ebs_version(void) { return 100; }

const char* ebs_status_string(int status) {
    switch (status) {
        case EBS_OK: return "ok";
        case EBS_ERR_INVALID_ARG: return "invalid argument";
        case EBS_ERR_UNSUPPORTED: return "unsupported configuration";
        case EBS_ERR_OVERFLOW: return "accumulator or index would overflow";
        case EBS_ERR_CUDA: return "CUDA runtime error";
        case EBS_ERR_TIMEOUT: return "device-side wait timed out";
        case EBS_ERR_SCRATCH_TOO_SMALL: return "request exceeds the built-in scratch of the no-allocation call";
        default: return "unknown status";
    }
}

const char* ebs_last_cuda_error(void) { return g_cuda_error; }

int ebs_conv_out_shape(const ebs_conv_desc* d, int h, int w, int* h_out, int* w_out) {
    int rc = validate_desc(d);
    if (rc) return rc;
    if (h <= 0 || w <= 0 || !h_out || !w_out) return EBS_ERR_INVALID_ARG;
    const int Ho = out_dim(h, d->pad_h, d->kh, d->stride_h), Wo = out_dim(w, d->pad_w, d->kw, d->stride_w);
    if (Ho <= 0 || Wo <= 0) return EBS_ERR_INVALID_ARG;
    *h_out = Ho;
    *w_out = Wo;
    return EBS_OK;
}

size_t ebs_packed_weight_bytes(const ebs_conv_desc* d) {
    if (validate_desc(d)) return 0;
    return packed_weight_plane_bytes(*d) + packed_weight_image_bytes(*d);
}

size_t ebs_packed_weight_plane_bytes(const ebs_conv_desc* d) {
    if (validate_desc(d)) return 0;
    return packed_weight_plane_bytes(*d);
}

size_t ebs_packed_act_bytes(int n, int h, int w, int c, int a_bits) {
    if (n <= 0 || h <= 0 || w <= 0 || c <= 0 || a_bits < 1 || a_bits > 8) return 0;
    return (size_t)n * h * w * ((c + 31) / 32) * a_bits * sizeof(uint32_t);
}

int ebs_pack_weights(const void* w_dev, int dtype, int layout, const ebs_conv_desc* d, void* packed_w_dev,
                     void* stream) {
    int rc = validate_desc(d);
    if (rc) return rc;
    if (!w_dev || !packed_w_dev || !aligned16(w_dev) || !aligned16(packed_w_dev)) return EBS_ERR_INVALID_ARG;
    if (dtype != EBS_F32 && dtype != EBS_I8_CODES) return EBS_ERR_INVALID_ARG;
    if (layout != EBS_NCHW && layout != EBS_NHWC) return EBS_ERR_INVALID_ARG;
    return launch_pack_weights(w_dev, dtype, layout, *d, 1.0f / d->w_scale, static_cast<uint32_t*>(packed_w_dev),
                               static_cast<cudaStream_t>(stream));
}

static int validate_pack_acts(const void* x_dev, int dtype, int layout, int n, int c, int h, int w, int a_bits,
                              float a_scale, const void* packed_x_dev) {
    if (!x_dev || !packed_x_dev || n <= 0 || c <= 0 || h <= 0 || w <= 0) return EBS_ERR_INVALID_ARG;
    if (a_bits < 1 || a_bits > 8) return EBS_ERR_INVALID_ARG;
    if (dtype != EBS_F32 && dtype != EBS_U8_CODES) return EBS_ERR_INVALID_ARG;
    if (layout != EBS_NCHW && layout != EBS_NHWC) return EBS_ERR_INVALID_ARG;
    if (dtype == EBS_F32 && !(a_scale > 0.0f)) return EBS_ERR_INVALID_ARG;
    if (!aligned16(x_dev) || !aligned16(packed_x_dev)) return EBS_ERR_INVALID_ARG;
    if ((long long)n * h * w >= (1LL << 31)) return EBS_ERR_OVERFLOW;
    return EBS_OK;
}

int ebs_pack_acts(const void* x_dev, int dtype, int layout, int n, int c, int h, int w, int a_bits, float a_scale,
                  void* packed_x_dev, void* stream) {
    const int rc = validate_pack_acts(x_dev, dtype, layout, n, c, h, w, a_bits, a_scale, packed_x_dev);
    if (rc) return rc;
    const float inv = dtype == EBS_F32 ? 1.0f / a_scale : 1.0f;
    return launch_pack_acts(x_dev, dtype, layout, n, c, h, w, a_bits, inv, static_cast<uint32_t*>(packed_x_dev),
                            static_cast<cudaStream_t>(stream));
}

int ebs_pack_acts_s2d(const void* x_dev, int n, int c, int h, int w, int offset, int a_bits, void* packed_x_dev,
                      void* stream) {
    if (!x_dev || !packed_x_dev || n <= 0 || c <= 0 || h <= 0 || w <= 0) return EBS_ERR_INVALID_ARG;
    if (a_bits < 1 || a_bits > 8 || (offset != 0 && offset != 1)) return EBS_ERR_INVALID_ARG;
    if (4 * c > 32 || (h & 1) || (w & 1)) return EBS_ERR_UNSUPPORTED;
    if (!aligned16(packed_x_dev)) return EBS_ERR_INVALID_ARG;
    if (h > 32000 || w > 32000 || (long long)n * h * w >= (1LL << 31)) return EBS_ERR_OVERFLOW;
    return launch_pack_acts_s2d(x_dev, n, c, h, w, offset, a_bits, static_cast<uint32_t*>(packed_x_dev),
                                static_cast<cudaStream_t>(stream));
}

int ebs_conv2d_mixed(const void* packed_x_dev, int n, int h, int w, const void* packed_w_dev,
                     const ebs_conv_desc* desc, const ebs_epilogue* epi, int32_t* acc_out_dev, float* y_out_dev,
                     void* packed_next_dev, void* stream) {
    return conv_impl(packed_x_dev, n, h, w, packed_w_dev, desc, epi, acc_out_dev, y_out_dev, packed_next_dev,
                     stream, -1);
}

int ebs_conv2d_i8(const void* x_codes_dev, int n, int h, int w, const void* packed_w_dev, const ebs_conv_desc* desc,
                  const ebs_epilogue* epi, int32_t* acc_out_dev, float* y_out_dev, void* packed_next_dev, void* stream) {
    ConvPlan plan;
    const int rc = conv_plan(x_codes_dev, n, h, w, packed_w_dev, desc, epi, acc_out_dev, y_out_dev, packed_next_dev, -1,
                             &plan, true);
    if (rc) return rc;
    return conv_launch(plan, stream);
}

int ebs_num_conv_variants(void) {
    return NUM_CONV_VARIANTS + NUM_CONV_MMA_VARIANTS + NUM_CONV_UMMA_VARIANTS + NUM_CONV_STRIP_VARIANTS +
           NUM_CONV_RESIDENT_VARIANTS + NUM_CONV_MMA_STRIP_VARIANTS + NUM_CONV_PIPE_VARIANTS;
}

const char* ebs_conv_variant_family(int variant) {
    int v = variant;
    if (v < 0) return "";
    if (v < NUM_CONV_VARIANTS) return "popc";
    v -= NUM_CONV_VARIANTS;
    if (v < NUM_CONV_MMA_VARIANTS) return "mma";
    v -= NUM_CONV_MMA_VARIANTS;
    if (v < NUM_CONV_UMMA_VARIANTS) return "umma";
    v -= NUM_CONV_UMMA_VARIANTS;
    if (v < NUM_CONV_STRIP_VARIANTS) return "umma_strip";
    v -= NUM_CONV_STRIP_VARIANTS;
    if (v < NUM_CONV_RESIDENT_VARIANTS) return "umma_resident";
    v -= NUM_CONV_RESIDENT_VARIANTS;
    if (v < NUM_CONV_MMA_STRIP_VARIANTS) return "mma_strip";
    v -= NUM_CONV_MMA_STRIP_VARIANTS;
    if (v < NUM_CONV_PIPE_VARIANTS) return "umma_pipe";
    return "";
}

int ebs_conv_variant_applies(const ebs_conv_desc* desc, int n, int h, int w, const ebs_epilogue* epi, int want_acc,
                             int want_y, int want_packed_next, int variant) {
    // the validation and selection of a launch with stand-in buffers (aligned, never dereferenced): nothing is enqueued
    void* fake = reinterpret_cast<void*>(static_cast<uintptr_t>(256));
    ConvPlan plan;
    return conv_plan(fake, n, h, w, fake, desc, epi, want_acc ? static_cast<int32_t*>(fake) : nullptr,
                     want_y ? static_cast<float*>(fake) : nullptr, want_packed_next ? fake : nullptr, variant, &plan);
}

int ebs_test_conv_route(const ebs_conv_desc* desc, int n, int h, int w, const ebs_epilogue* epi, int want_acc, int want_y,
                        int want_packed_next, int variant, int* route) {
    void* fake = reinterpret_cast<void*>(static_cast<uintptr_t>(256));
    if (!route) return EBS_ERR_INVALID_ARG;
    ConvPlan plan;
    const int rc = conv_plan(fake, n, h, w, fake, desc, epi, want_acc ? static_cast<int32_t*>(fake) : nullptr,
                             want_y ? static_cast<float*>(fake) : nullptr, want_packed_next ? fake : nullptr, variant, &plan);
    if (rc) return rc;
    memset(route, 0, 10 * sizeof(int));
    route[0] = plan.variant;
    const int pipe = plan.variant - (ebs_num_conv_variants() - NUM_CONV_PIPE_VARIANTS);
    if (pipe >= 0) conv_umma_pipe_route(plan.p, pipe, route + 1);
    return EBS_OK;
}

int ebs_test_set_device_wait(unsigned int limit, int skip_mma) {
    g_wait_limit = limit == 0 ? (1u << 20) : limit;
    g_test_flags = skip_mma == 2 ? 2 : skip_mma == 3 ? 4 : skip_mma ? 1 : 0;
    return EBS_OK;
}

int ebs_check_device_status(void) {
    static long long seen = 0;
    const long long now = (long long)conv_umma_timeouts();
    const bool fresh = now > seen;
    seen = now;
    return fresh ? EBS_ERR_TIMEOUT : EBS_OK;
}

int ebs_checked_build(void) {
#ifdef EBS_CHECKED
    return 1;
#else
    return 0;
#endif
}

int ebs_checked_status(int* site, long long* index, long long* limit, int clear) {
#ifdef EBS_CHECKED
    unsigned long long w[4] = {0, 0, 0, 0};
    if (cudaDeviceSynchronize() != cudaSuccess) return EBS_ERR_CUDA;
    if (cudaMemcpyFromSymbol(w, g_check_words, sizeof(w)) != cudaSuccess) return EBS_ERR_CUDA;
    if (site) *site = (int)(w[0] >> 48);
    if (index) *index = (long long)w[1];
    if (limit) *limit = (long long)w[2];
    if (clear) {
        const unsigned long long z[4] = {0, 0, 0, 0};
        if (cudaMemcpyToSymbol(g_check_words, z, sizeof(z)) != cudaSuccess) return EBS_ERR_CUDA;
    }
    return w[0] ? 1 : 0;
#else
    (void)site; (void)index; (void)limit; (void)clear;
    return EBS_ERR_UNSUPPORTED;
#endif
}

int ebs_test_checked_shrink(long long elements) {
#ifdef EBS_CHECKED
    if (elements < 0) return EBS_ERR_INVALID_ARG;
    g_check_shrink = elements;
    return EBS_OK;
#else
    (void)elements;
    return EBS_ERR_UNSUPPORTED;
#endif
}

long long ebs_device_wait_timeouts(void) { return (long long)conv_umma_timeouts(); }

int ebs_conv2d_mixed_variant(const void* packed_x_dev, int n, int h, int w, const void* packed_w_dev,
                             const ebs_conv_desc* desc, const ebs_epilogue* epi, int32_t* acc_out_dev,
                             float* y_out_dev, void* packed_next_dev, void* stream, int variant) {
    return conv_impl(packed_x_dev, n, h, w, packed_w_dev, desc, epi, acc_out_dev, y_out_dev, packed_next_dev,
                     stream, variant);
}

int ebs_dequant(const int32_t* acc_dev, size_t n_pixels, int c_out, float scale, const float* ch_scale_dev,
                const float* ch_bias_dev, int relu, float* y_dev, void* stream) {
    if (!acc_dev || !y_dev || n_pixels == 0 || c_out <= 0) return EBS_ERR_INVALID_ARG;
    if (!aligned16(acc_dev) || !aligned16(y_dev)) return EBS_ERR_INVALID_ARG;
    if (n_pixels >= ((size_t)1 << 40) / (size_t)c_out) return EBS_ERR_OVERFLOW;
    return launch_dequant(acc_dev, n_pixels, c_out, scale, ch_scale_dev, ch_bias_dev, relu ? 1 : 0, y_dev,
                          static_cast<cudaStream_t>(stream));
}

int ebs_search_weight_forward(const float* w_dev, size_t n, const int* bits, const float* coeff, int n_cand,
                              float* w_hat_dev, void* scratch_dev, void* stream) {
    if (!w_dev || !w_hat_dev || !scratch_dev || n == 0) return EBS_ERR_INVALID_ARG;
    if (!aligned16(w_dev) || !aligned16(w_hat_dev) || !aligned16(scratch_dev)) return EBS_ERR_INVALID_ARG;
    return launch_search_weights(w_dev, n, bits, coeff, n_cand, w_hat_dev, scratch_dev, static_cast<cudaStream_t>(stream));
}

int ebs_search_act_forward(const float* x_dev, size_t n, float alpha, const int* bits, const float* coeff, int n_cand,
                           float* x_hat_dev, void* stream) {
    if (!x_dev || !x_hat_dev || n == 0 || !(alpha > 0.0f)) return EBS_ERR_INVALID_ARG;
    if (!aligned16(x_dev) || !aligned16(x_hat_dev)) return EBS_ERR_INVALID_ARG;
    return launch_search_acts(x_dev, n, alpha, bits, coeff, n_cand, x_hat_dev, static_cast<cudaStream_t>(stream));
}

float ebs_combined_scale(float w_scale, float a_scale) { return w_scale * a_scale; }        // one rounded fp32 multiply
float ebs_reciprocal_step(float step) { return 1.0f / step; }                               // one rounded fp32 division

double ebs_expected_flops(double macs, const int* bits_w, const float* coeff_w, int n_w, const int* bits_x,
                          const float* coeff_x, int n_x) {
    if (!bits_w || !coeff_w || !bits_x || !coeff_x || n_w < 1 || n_x < 1 || !(macs >= 0.0)) return -1.0;
    double m = 0.0, k = 0.0;
    for (int i = 0; i < n_w; ++i) m += (double)coeff_w[i] * bits_w[i];
    for (int j = 0; j < n_x; ++j) k += (double)coeff_x[j] * bits_x[j];
    return macs * m * k;
}

int ebs_fused_plan_upload(const ebs_fused_layer* layers_host, int n_layers, void* layers_dev, void* stream) {
    if (!layers_host || !layers_dev || n_layers < 1 || n_layers > 4096) return EBS_ERR_INVALID_ARG;
    return fused_plan_upload(layers_host, n_layers, layers_dev, static_cast<cudaStream_t>(stream));
}

int ebs_resnet_cifar_forward(const unsigned char* images_dev, int n, int img_h, int img_w, const void* layers_dev,
                             int n_layers, const ebs_fused_head* head_host, float* logits_dev, unsigned char* trace_dev,
                             long long trace_stride, void* stream) {
    if (!images_dev || !layers_dev || !head_host || !logits_dev || n < 1 || n_layers < 1) return EBS_ERR_INVALID_ARG;
    if (img_h < 1 || img_w < 1 || (img_h + 2) * (img_w + 2) > 1156) return EBS_ERR_UNSUPPORTED;
    if (!head_host->w8 || head_host->c_in < 1 || head_host->c_in > 64 || head_host->c_out < 1 || head_host->c_out > 256)
        return EBS_ERR_INVALID_ARG;
    return launch_fused_resnet(images_dev, n, img_h, img_w, layers_dev, n_layers, head_host, logits_dev, trace_dev,
                               trace_stride, g_wait_limit, g_test_flags, static_cast<cudaStream_t>(stream));
}

int ebs_global_avgpool(const float* y_dev, int n, int hw, int c, float* out_dev, void* stream) {
    if (!y_dev || !out_dev || n <= 0 || hw <= 0 || c <= 0) return EBS_ERR_INVALID_ARG;
    if ((long long)n * c >= (1LL << 31)) return EBS_ERR_OVERFLOW;
    return launch_avgpool(y_dev, n, hw, c, out_dev, static_cast<cudaStream_t>(stream));
}

int ebs_maxpool_packed(const void* packed_x_dev, int n, int h, int w, int c, int a_bits, int k, int stride, int pad,
                       void* packed_out_dev, void* stream) {
    if (!packed_x_dev || !packed_out_dev || n <= 0 || h <= 0 || w <= 0 || c <= 0) return EBS_ERR_INVALID_ARG;
    if (a_bits < 1 || a_bits > 8 || k < 1 || stride < 1 || pad < 0 || pad >= k) return EBS_ERR_INVALID_ARG;
    if (!aligned16(packed_x_dev) || !aligned16(packed_out_dev) || packed_x_dev == packed_out_dev) return EBS_ERR_INVALID_ARG;
    const int ho = out_dim(h, pad, k, stride), wo = out_dim(w, pad, k, stride);
    if (ho <= 0 || wo <= 0) return EBS_ERR_INVALID_ARG;
    if ((long long)n * h * w * ((c + 31) / 32) * a_bits >= (1LL << 31)) return EBS_ERR_OVERFLOW;
    return launch_maxpool_packed(static_cast<const uint32_t*>(packed_x_dev), n, h, w, c, a_bits, k, stride, pad, ho, wo,
                                 static_cast<uint32_t*>(packed_out_dev), static_cast<cudaStream_t>(stream));
}

static size_t round256(size_t v) { return (v + 255) & ~(size_t)255; }

size_t ebs_host_workspace_bytes(const ebs_conv_desc* d, int n, int h, int w, int dtype, int next_a_bits) {
    if (validate_desc(d) || n <= 0 || h <= 0 || w <= 0) return 0;
    const int Ho = out_dim(h, d->pad_h, d->kh, d->stride_h), Wo = out_dim(w, d->pad_w, d->kw, d->stride_w);
    if (Ho <= 0 || Wo <= 0) return 0;
    const size_t elems_in = (size_t)n * h * w * d->c_in, outs = (size_t)n * Ho * Wo * d->c_out;
    size_t total = round256(elems_in * (dtype == EBS_F32 ? 4 : 1));
    total += round256(ebs_packed_act_bytes(n, h, w, d->c_in, d->a_bits));
    total += round256(outs * 4) * 2;                                   // acc and y
    if (next_a_bits >= 1 && next_a_bits <= 8) total += round256(ebs_packed_act_bytes(n, Ho, Wo, d->c_out, next_a_bits));
    return total;
}

int ebs_conv2d_mixed_host(const void* x_host, int dtype, int layout, int n, int h, int w, const void* packed_w_dev,
                          const ebs_conv_desc* d, const ebs_epilogue* epi, void* workspace_dev, size_t workspace_bytes,
                          int32_t* acc_out_host, float* y_out_host, void* packed_next_host, void* stream) {
    int rc = validate_desc(d);
    if (rc) return rc;
    if (!x_host || !workspace_dev || !aligned16(workspace_dev) || n <= 0 || h <= 0 || w <= 0) return EBS_ERR_INVALID_ARG;
    if (dtype != EBS_F32 && dtype != EBS_U8_CODES) return EBS_ERR_INVALID_ARG;
    if (!acc_out_host && !y_out_host && !packed_next_host) return EBS_ERR_INVALID_ARG;
    if (packed_next_host && (!epi || epi->next_a_bits < 1 || epi->next_a_bits > 8)) return EBS_ERR_INVALID_ARG;
    const int next_bits = packed_next_host ? epi->next_a_bits : 0;
    const size_t need = ebs_host_workspace_bytes(d, n, h, w, dtype, next_bits);
    if (need == 0 || workspace_bytes < need) return EBS_ERR_INVALID_ARG;
    const int Ho = out_dim(h, d->pad_h, d->kh, d->stride_h), Wo = out_dim(w, d->pad_w, d->kw, d->stride_w);
    const size_t elems_in = (size_t)n * h * w * d->c_in, outs = (size_t)n * Ho * Wo * d->c_out;
    cudaStream_t st = static_cast<cudaStream_t>(stream);

    char* ws = static_cast<char*>(workspace_dev);
    void* x_dev = ws;                 ws += round256(elems_in * (dtype == EBS_F32 ? 4 : 1));
    void* px_dev = ws;                ws += round256(ebs_packed_act_bytes(n, h, w, d->c_in, d->a_bits));
    int32_t* acc_dev = (int32_t*)ws;  ws += round256(outs * 4);
    float* y_dev = (float*)ws;        ws += round256(outs * 4);
    void* pn_dev = ws;

    // every argument check of the two device calls comes first: an error return means nothing was enqueued
    // (and, for the caller that shares one scratch between calls, that the scratch was not touched)
    rc = validate_pack_acts(x_dev, dtype, layout, n, d->c_in, h, w, d->a_bits, d->a_scale, px_dev);
    if (rc) return rc;
    ConvPlan plan;
    rc = conv_plan(px_dev, n, h, w, packed_w_dev, d, epi, acc_out_host ? acc_dev : nullptr,
                   y_out_host ? y_dev : nullptr, packed_next_host ? pn_dev : nullptr, -1, &plan);
    if (rc) return rc;

    rc = check_cuda(cudaMemcpyAsync(x_dev, x_host, elems_in * (dtype == EBS_F32 ? 4 : 1), cudaMemcpyHostToDevice, st));
    if (rc) return rc;
    rc = ebs_pack_acts(x_dev, dtype, layout, n, d->c_in, h, w, d->a_bits, d->a_scale, px_dev, stream);
    if (rc) return rc;
    rc = conv_launch(plan, stream);
    if (rc) return rc;
    if (acc_out_host) {
        rc = check_cuda(cudaMemcpyAsync(acc_out_host, acc_dev, outs * 4, cudaMemcpyDeviceToHost, st));
        if (rc) return rc;
    }
    if (y_out_host) {
        rc = check_cuda(cudaMemcpyAsync(y_out_host, y_dev, outs * 4, cudaMemcpyDeviceToHost, st));
        if (rc) return rc;
    }
    if (packed_next_host) {
        rc = check_cuda(cudaMemcpyAsync(packed_next_host, pn_dev, ebs_packed_act_bytes(n, Ho, Wo, d->c_out, next_bits),
                                        cudaMemcpyDeviceToHost, st));
        if (rc) return rc;
    }
    return EBS_OK;
}

}  // extern "C"
