// Whole-network kernel for basic-block CIFAR ResNets: one CTA carries one image through every layer
// with its activations resident in shared memory.
//
// The activation codes of an image live in shared memory as BYTES, already in the un-swizzled K-major strip layout the
// tcgen05 operand descriptors read ([16-byte half][frame pixel][16 bytes] per 32-channel word, frame = zero-padded
// image), so between layers there is no bit-to-byte expansion, no global traffic and no launch.  Per layer
//   1. the weight byte image (the second part of an ebs_pack_weights buffer) arrives in one of two shared buffers by
//      cp.async.bulk while earlier layers run,
//   2. the MMAs -- every 128-row tile of the frame x every tap x every 32-channel word, a tap being a shifted
//      descriptor -- go into tensor-memory accumulators (tile t at columns 32 t or 64 t),
//   3. the epilogue runs the fp32 steps out of tensor memory (scale, per-channel scale/shift, shortcut, ReLU, requantize:
//      the same individually rounded operations as the per-layer kernels) and writes the codes as bytes at frame
//      position f + Wp + 1 of the destination strip: outputs that do not exist (frame columns >= Wo, rows >= Ho) land
//      exactly on padding positions and are written as zero.
// What bounds it is the chain from layer to layer, so the layers overlap as a wavefront and nothing waits for a whole
// layer: 16 epilogue warps take (tile, channel group) units as their accumulators complete, two warps issue MMAs, one
// fetches weights, layer records and per-channel terms ahead.  In a run of 3x3 stride-1 layers of one geometry the MMAs of
// tile t need the codes of tiles 0 .. t + 1 of the layer before, and no strip or accumulator is overwritten earlier than
// that same order allows; where the geometry changes, the next layer waits for all tiles.  (With the phases of a layer one
// after the other between block barriers a layer took 5.5 us whatever its size.)
// Layers with at most 16 input channels would leave half of every MMA's 32 reduction bytes empty: their strips hold 16 bytes
// a pixel, and an MMA takes two taps -- the distance between the two 16-byte halves of an operand row is a descriptor
// field, here the distance between the taps.  The loader re-lays their weights accordingly (5 MMAs a tile instead of 9; an
// MMA costs 41-50 clocks of operand reads and issue however narrow it is).
// A unit is the 16 channels that fill one 16-byte half of a pixel's row (channels 8 i + 4 h + e of a 32-channel word), so
// its codes leave in one 16-byte store and its identity shortcut is one 16-byte load.
// Stride-2 3x3 layers are computed at stride 1 and subsampled in the epilogue (4x the MMAs of two or three
// layers, no phase logic); a 1x1 stride-2 projection runs on a subsampled copy of its input laid out in the
// output frame, keeps its accumulators in tensor memory, and the next layer's epilogue adds them as the
// shortcut.  The identity shortcut is read from the destination strip (the block input) just before it is
// overwritten in place.  After the last block: average pooling (pixels added in order), 8-bit
// quantization, and the classifier as a plain integer dot product, a warp per class.
// Every wait is bounded; on a timeout the CTA sets its abort flag, every role leaves its loop, tensor memory is freed.
#include <type_traits>

#include "conv_frame.cuh"

namespace ebs {

constexpr int FUSED_EPI_WARPS = 16, FUSED_ISSUER_WARP = 16, FUSED_ISSUERS = 2, FUSED_LOADER_WARP = 18;
constexpr int FUSED_THREADS = 20 * 32;                 // (warp 19 has no role)
constexpr int FUSED_MAX_TILES = 10;                    // 320 accumulator columns of at least 32
constexpr int FUSED_RING = 4;                          // layer records and terms in shared memory
constexpr int FUSED_ACT_PIX = 1360;                    // pixels an activation strip holds (34 x 34 frame + halo, 128-row tiles)
constexpr int FUSED_ACT_BYTES = FUSED_ACT_PIX * 32;    // one 32-channel word
constexpr int FUSED_W_BYTES = 37 * 1024;               // largest weight image (3x3 64->64)
constexpr int FUSED_SMEM = 3 * FUSED_ACT_BYTES + 2 * FUSED_W_BYTES + 1024;
constexpr int FUSED_PACKED_W = 20 * 1024;             // where a narrow layer's re-laid weights lie in its weight buffer (raw: <= 18.4 KB)
constexpr int FUSED_HOLD_COL = 320;                    // accumulator columns of a held projection

using FusedLayer = ebs_fused_layer;
using FusedHead = ebs_fused_head;

__device__ __forceinline__ uint8_t* strip_ptr(uint8_t* acts, int buf) { return acts + buf * FUSED_ACT_BYTES; }
// A strip holds one 32-channel word of up to 1360 frame pixels or two words of up to 680: pixels per word.
__host__ __device__ inline int strip_cap(int channels) { return channels > 32 ? FUSED_ACT_PIX / 2 : FUSED_ACT_PIX; }

// What the roles derive from a layer record.
struct FusedGeom {
    int cw, co16, Ho, Wo, Hf, Wf, frame, tiles, acc_stride, units;   // units: epilogue units per tile (1, 2 or 4)
};
__device__ __forceinline__ FusedGeom fused_geom(const FusedLayer& L) {
    FusedGeom g;
    g.cw = (L.c_in + 31) >> 5;
    g.co16 = (L.c_out + 15) & ~15;
    g.Ho = L.stride == 2 ? L.h_in / 2 : L.h_in;
    g.Wo = L.stride == 2 ? L.w_in / 2 : L.w_in;
    // frame in which the MMAs run: the padded input for a 3x3 layer, the padded OUTPUT frame for the projection
    g.Hf = L.k == 3 ? L.h_in + 2 : g.Ho + 2;
    g.Wf = L.k == 3 ? L.w_in + 2 : g.Wo + 2;
    g.frame = g.Hf * g.Wf;
    g.tiles = (g.frame + UMMA_M - 1) / UMMA_M;
    g.acc_stride = g.co16 > 32 ? g.co16 : 32;
    g.units = L.c_out <= 16 ? 1 : (L.c_out <= 32 ? 2 : 4);
    return g;
}
// Layer `L` can follow `P` tile by tile: same frame, stride 1, reads what P writes, nothing to clear or copy.
__device__ __forceinline__ bool fused_follows(const FusedLayer& P, const FusedLayer& L) {
    return L.k == 3 && P.k == 3 && P.stride == 1 && !P.hold && !L.hold && L.stride == 1 && !L.zero_dst && L.h_in == P.h_in &&
           L.w_in == P.w_in && L.src == P.dst && L.c_out == P.c_out;
}

struct FusedTerms {                                     // per-channel terms in the order the epilogue reads them
    float cs[64], cb[64], pcs[64], pcb[64];             // of the layer, and of the held projection
};

__device__ __forceinline__ void tmem_ld4_issue(uint32_t taddr, uint32_t (&v)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld4_wait(uint32_t (&a)[4], uint32_t (&b)[4], uint32_t (&c)[4], uint32_t (&d)[4]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;\n"
                 : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]),
                   "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]), "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]) :: "memory");
}
// What the units of a layer share.
struct FusedUnitEnv {
    uint64_t S2, PS2, rs2, one2, inv2;
    int out_bits, c_out, cap_out;
    uint8_t* dst;                                       // destination strip
    const uint8_t* res;                                 // strip of the identity shortcut
    const FusedTerms* T;
};
__device__ __forceinline__ uint64_t fused_value(uint64_t w, float s0, float s1, float b0, float b1, uint64_t one2) {
    return f32x2_add_one(f32x2_mul_rn(w, f32x2_pack(s0, s1)), one2, f32x2_pack(b0, b1));
}
__device__ __forceinline__ uint64_t fused_pair(uint32_t a, uint32_t b) { return f32x2_pack((float)(int)a, (float)(int)b); }
// Bytes 2 j and 2 j + 1 of a register as fp32, exactly (2^23 + byte, minus 2^23).
__device__ __forceinline__ uint64_t fused_byte_pair(uint32_t r, int j, uint64_t one2) {
    const float lo = __uint_as_float(__byte_perm(r, 0x4B000000u, 0x7540u + 2u * (uint32_t)j)), hi = __uint_as_float(__byte_perm(r, 0x4B000000u, 0x7541u + 2u * (uint32_t)j));
    return f32x2_add_one(f32x2_pack(lo, hi), one2, f32x2_pack(-8388608.0f, -8388608.0f));
}
__device__ __forceinline__ void fused_code(uint64_t w, const FusedUnitEnv& E, uint32_t& m0, uint32_t& m1) {
    code_pair<0>(f32x2_mul_rn(w, E.inv2), E.out_bits, m0, m1);
}
// The fp32 values of a unit's 16 channels at this thread's pixel, two to a register: wide layers w[2 e + j] = word 4 hf + e of
// the 32-channel group, its bytes 2 j and 2 j + 1 (channels 8 i + 4 hf + e); narrow ones (all 16 channels in one unit) w[b] =
// channels b and 8 + b.  RES: 0 none, 1 identity shortcut, 2 held projection.  Straight-line code for each form: a unit is
// some 200 instructions, and branching through all forms cost ten times their issue time in instruction fetch.
template <bool NARROW, int RES>
__device__ __forceinline__ void fused_unit_values(const FusedUnitEnv& E, uint32_t trow, int un, int target, uint64_t (&w)[8]) {
    const int grp = un >> 1, hf = un & 1;
    const FusedTerms& T = *E.T;
    uint32_t resw[8];
    if constexpr (NARROW) {
        uint32_t v[16], pv[16];
        tmem_ld16_issue(trow, v);
        if constexpr (RES == 2) tmem_ld16_issue(trow + FUSED_HOLD_COL, pv);
        if constexpr (RES == 1) {
            const uint4 a = *reinterpret_cast<const uint4*>(E.res + target * 16);
            resw[0] = a.x; resw[1] = a.y; resw[2] = a.z; resw[3] = a.w;
        }
        tmem_ld16_wait(v);
        if constexpr (RES == 2) tmem_ld16_wait(pv);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 s4 = *reinterpret_cast<const float4*>(&T.cs[4 * q]), b4 = *reinterpret_cast<const float4*>(&T.cb[4 * q]);
            w[2 * q] = fused_value(f32x2_mul_rn(fused_pair(v[2 * q], v[8 + 2 * q]), E.S2), s4.x, s4.y, b4.x, b4.y, E.one2);
            w[2 * q + 1] = fused_value(f32x2_mul_rn(fused_pair(v[2 * q + 1], v[9 + 2 * q]), E.S2), s4.z, s4.w, b4.z, b4.w, E.one2);
            if constexpr (RES == 2) {
                const float4 ps = *reinterpret_cast<const float4*>(&T.pcs[4 * q]), pb = *reinterpret_cast<const float4*>(&T.pcb[4 * q]);
                w[2 * q] = f32x2_add_one(w[2 * q], E.one2, fused_value(f32x2_mul_rn(fused_pair(pv[2 * q], pv[8 + 2 * q]), E.PS2), ps.x, ps.y, pb.x, pb.y, E.one2));
                w[2 * q + 1] = f32x2_add_one(w[2 * q + 1], E.one2, fused_value(f32x2_mul_rn(fused_pair(pv[2 * q + 1], pv[9 + 2 * q]), E.PS2), ps.z, ps.w, pb.z, pb.w, E.one2));
            }
        }
        if constexpr (RES == 1) {
#pragma unroll
            for (int b = 0; b < 8; ++b) w[b] = f32x2_add_one(w[b], E.one2, f32x2_mul_rn(E.rs2, fused_byte_pair(resw[b & 3], b >> 2, E.one2)));
        }
    } else {
        uint32_t v[4][4], pv[4][4];
        const uint32_t tc = trow + (uint32_t)(32 * grp + 4 * hf);
#pragma unroll
        for (int i = 0; i < 4; ++i) tmem_ld4_issue(tc + 8u * i, v[i]);
        if constexpr (RES == 2) {
#pragma unroll
            for (int i = 0; i < 4; ++i) tmem_ld4_issue(tc + FUSED_HOLD_COL + 8u * i, pv[i]);
        }
        if constexpr (RES == 1) {
            const uint4 a = *reinterpret_cast<const uint4*>(E.res + grp * E.cap_out * 32 + hf * E.cap_out * 16 + target * 16);
            resw[0] = a.x; resw[1] = a.y; resw[2] = a.z; resw[3] = a.w;
        }
        tmem_ld4_wait(v[0], v[1], v[2], v[3]);
        if constexpr (RES == 2) tmem_ld4_wait(pv[0], pv[1], pv[2], pv[3]);
        const int t0 = grp * 32 + 16 * hf;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float4 s4 = *reinterpret_cast<const float4*>(&T.cs[t0 + 4 * e]), b4 = *reinterpret_cast<const float4*>(&T.cb[t0 + 4 * e]);
            w[2 * e] = fused_value(f32x2_mul_rn(fused_pair(v[0][e], v[1][e]), E.S2), s4.x, s4.y, b4.x, b4.y, E.one2);
            w[2 * e + 1] = fused_value(f32x2_mul_rn(fused_pair(v[2][e], v[3][e]), E.S2), s4.z, s4.w, b4.z, b4.w, E.one2);
            if constexpr (RES == 2) {
                const float4 ps = *reinterpret_cast<const float4*>(&T.pcs[t0 + 4 * e]), pb = *reinterpret_cast<const float4*>(&T.pcb[t0 + 4 * e]);
                w[2 * e] = f32x2_add_one(w[2 * e], E.one2, fused_value(f32x2_mul_rn(fused_pair(pv[0][e], pv[1][e]), E.PS2), ps.x, ps.y, pb.x, pb.y, E.one2));
                w[2 * e + 1] = f32x2_add_one(w[2 * e + 1], E.one2, fused_value(f32x2_mul_rn(fused_pair(pv[2][e], pv[3][e]), E.PS2), ps.z, ps.w, pb.z, pb.w, E.one2));
            }
            if constexpr (RES == 1) {
                w[2 * e] = f32x2_add_one(w[2 * e], E.one2, f32x2_mul_rn(E.rs2, fused_byte_pair(resw[e], 0, E.one2)));
                w[2 * e + 1] = f32x2_add_one(w[2 * e + 1], E.one2, f32x2_mul_rn(E.rs2, fused_byte_pair(resw[e], 1, E.one2)));
            }
        }
    }
}
// First and second channel of register i of a unit.
__device__ __forceinline__ int fused_channel(bool narrow, int un, int i) {
    return narrow ? i : 32 * (un >> 1) + 4 * (un & 1) + (i >> 1) + 16 * (i & 1);       // (the second one is 8 further)
}
// Codes of a unit to its 16 bytes of a pixel in the destination strip.
template <bool NARROW, int RES>
__device__ __forceinline__ void fused_unit_codes(const FusedUnitEnv& E, uint32_t trow, int un, int target, bool valid, bool in_frame,
                                                 uint8_t* trace) {
    uint64_t w[8];
    fused_unit_values<NARROW, RES>(E, trow, un, target, w);
    const int grp = un >> 1, hf = un & 1;
    uint8_t* at = E.dst + grp * E.cap_out * 32 + hf * E.cap_out * 16 + target * 16;
    const uint32_t z = valid ? 0xFFFFFFFFu : 0u;
    uint32_t words[4];
    if constexpr (NARROW) {                              // 16 bytes a pixel: word j = channels j, 8 + j, 4 + j, 12 + j
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            uint32_t m[4];
            fused_code(w[e], E, m[0], m[1]);
            fused_code(w[4 + e], E, m[2], m[3]);
            words[e] = join_codes(m, k256_of(__uint_as_float((uint32_t)E.one2))) & z;
        }
        if (E.c_out & 15) {                              // channels past c_out
#pragma unroll
            for (int e = 0; e < 4; ++e)
                words[e] &= (e < E.c_out ? 0xFFu : 0u) | (e + 8 < E.c_out ? 0xFF00u : 0u) | (e + 4 < E.c_out ? 0xFF0000u : 0u) | (e + 12 < E.c_out ? 0xFF000000u : 0u);
        }
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            uint32_t m[4];
            fused_code(w[2 * e], E, m[0], m[1]);
            fused_code(w[2 * e + 1], E, m[2], m[3]);
            words[e] = join_codes(m, k256_of(__uint_as_float((uint32_t)E.one2))) & z;
        }
        if (E.c_out & 31) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int c = 32 * grp + 4 * hf + e;
                words[e] &= (c < E.c_out ? 0xFFu : 0u) | (c + 8 < E.c_out ? 0xFF00u : 0u) | (c + 16 < E.c_out ? 0xFF0000u : 0u) | (c + 24 < E.c_out ? 0xFF000000u : 0u);
            }
        }
    }
    if (in_frame) *reinterpret_cast<uint4*>(at) = make_uint4(words[0], words[1], words[2], words[3]);
    if (trace && valid) {
#pragma unroll 1
        for (int i = 0; i < 16; ++i) {
            const int e = i & 3, byte = i >> 2, c = NARROW ? 8 * (byte & 1) + 4 * (byte >> 1) + e : 32 * grp + 8 * byte + 4 * hf + e;
            if (c < E.c_out) trace[c] = at[e * 4 + byte];
        }
    }
}
// fp32 results of the last layer's unit for pooling: [pixel][c_out].
template <bool NARROW, int RES>
__device__ __forceinline__ void fused_unit_pool(const FusedUnitEnv& E, uint32_t trow, int un, int target, bool valid, bool relu, float* row) {
    uint64_t w[8];
    fused_unit_values<NARROW, RES>(E, trow, un, target, w);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        float y0 = __uint_as_float((uint32_t)w[i]), y1 = __uint_as_float((uint32_t)(w[i] >> 32));
        if (relu) { y0 = y0 > 0.0f ? y0 : 0.0f; y1 = y1 > 0.0f ? y1 : 0.0f; }
        const int c = fused_channel(NARROW, un, i);
        if (valid && c < E.c_out) row[c] = y0;
        if (valid && c + 8 < E.c_out) row[c + 8] = y1;
    }
}

__global__ void __launch_bounds__(FUSED_THREADS, 1)
fused_resnet_kernel(const uint8_t* __restrict__ images, int img_h, int img_w, const FusedLayer* __restrict__ layers,
                    int n_layers, const FusedHead head, float one, float* __restrict__ logits, uint8_t* __restrict__ trace,
                    long long trace_stride, unsigned limit, int test_flags) {
    extern __shared__ uint8_t dyn_smem[];
    __shared__ __align__(8) uint64_t w_full[2], w_raw[2], w_free[2], rec_full[FUSED_RING], rec_free[FUSED_RING];
    __shared__ __align__(8) uint64_t acc_full[FUSED_MAX_TILES], ep_done[FUSED_MAX_TILES], hold_full, copy_ready, epi_sync;
    __shared__ __align__(16) FusedTerms s_terms[FUSED_RING];
    __shared__ __align__(16) FusedLayer s_rec[FUSED_RING];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ int fc_codes[64];

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int img = blockIdx.x;
    uint8_t* base = dyn_smem + ((1024u - (smem_u32(dyn_smem) & 1023u)) & 1023u);
    uint8_t* acts = base;                                        // three strips
    uint8_t* wbuf = base + 3 * FUSED_ACT_BYTES;                  // two weight images
    volatile int* abortp = &abort_flag;
    const bool skip_mma = (test_flags & 1) != 0;                 // test hook: issue nothing, so that waits run out

    if (tid == 0) {
        abort_flag = 0;
        for (int i = 0; i < 2; ++i) {
            mbar_init(&w_full[i], 1);
            mbar_init(&w_raw[i], 1);
            mbar_init(&w_free[i], FUSED_ISSUERS);
        }
        for (int i = 0; i < FUSED_RING; ++i) {
            mbar_init(&rec_full[i], 1);
            mbar_init(&rec_free[i], FUSED_EPI_WARPS + FUSED_ISSUERS);
        }
        for (int i = 0; i < FUSED_MAX_TILES; ++i) {
            // Every issuing warp and every epilogue warp arrives once per tile and layer, also where another one has the
            // work, once it has waited for what its turn waits for: so no barrier can run a phase ahead of a warp that has
            // not looked at it yet, and parities suffice.
            mbar_init(&acc_full[i], FUSED_ISSUERS);
            mbar_init(&ep_done[i], FUSED_EPI_WARPS);
        }
        mbar_init(&hold_full, FUSED_ISSUERS);
        mbar_init(&copy_ready, FUSED_EPI_WARPS);
        mbar_init(&epi_sync, FUSED_EPI_WARPS);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == FUSED_ISSUER_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_slot)),
                     "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (warp != FUSED_LOADER_WARP) {                             // (the loader goes ahead)
        constexpr int NT = FUSED_THREADS - 32;
        const int i0 = warp > FUSED_LOADER_WARP ? tid - 32 : tid;
        // all strips start as zeros (padding positions are never written with anything else)
        for (int i = i0; i < 3 * FUSED_ACT_BYTES / 16; i += NT) reinterpret_cast<uint4*>(acts)[i] = make_uint4(0, 0, 0, 0);
        asm volatile("bar.sync 1, %0;\n" ::"n"(FUSED_THREADS - 32) : "memory");
        // the image: u8 NHWC, 3 channels -> bytes of strip 0 in the padded frame (channel c is byte 4c of word 0)
        const int Wp = img_w + 2, pixels = img_h * img_w;
        const uint8_t* src = images + (size_t)img * pixels * 3;
#pragma unroll 2
        for (int pix = i0; pix < pixels; pix += NT) {
            const int h = pix / img_w, w = pix - h * img_w;
            const uint32_t r = src[pix * 3], g = src[pix * 3 + 1], b = src[pix * 3 + 2];
            uint32_t* dst = reinterpret_cast<uint32_t*>(strip_ptr(acts, 0) + ((h + 1) * Wp + (w + 1)) * 16);
            dst[0] = r; dst[1] = g; dst[2] = b;                   // words 0..2 of the first 16-byte half: channels 0, 1, 2
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        asm volatile("bar.sync 1, %0;\n" ::"n"(FUSED_THREADS - 32) : "memory");
    }
    const uint32_t tmem_base = tmem_slot;
    float* pool_scratch = reinterpret_cast<float*>(strip_ptr(acts, 0));      // [pixels][c_out] of the last layer

    if (warp == FUSED_LOADER_WARP) {
        // =========================== records, terms, weights ===========================
        const float *hold_cs = nullptr, *hold_cb = nullptr;
        int n_raw[2] = {0, 0};
        for (int li = 0; li < n_layers; ++li) {
            const int slot = li & (FUSED_RING - 1), use = li / FUSED_RING;
            if (use > 0 && !mbar_wait_bounded_warp(&rec_free[slot], (uint32_t)((use - 1) & 1), abortp, limit)) break;
            for (int i = lane; i < (int)(sizeof(FusedLayer) / 4); i += 32)
                reinterpret_cast<uint32_t*>(&s_rec[slot])[i] = __ldg(reinterpret_cast<const uint32_t*>(layers + li) + i);
            __syncwarp();
            const FusedLayer& L = s_rec[slot];
            FusedTerms& T = s_terms[slot];
            for (int c = lane; c < 64; c += 32) {
                const int at = L.c_out <= 16 ? (c < 16 ? (c & 7) * 2 + (c >> 3) : c) : (c & 32) + (c & 7) * 4 + ((c & 31) >> 3);
                const bool in = c < L.c_out;
                T.cs[at] = (L.ch_scale && in) ? __ldg(L.ch_scale + c) : 1.0f;    // identities: x * 1, x + (-0)
                T.cb[at] = (L.ch_bias && in) ? __ldg(L.ch_bias + c) : -0.0f;
                T.pcs[at] = (hold_cs && in) ? __ldg(hold_cs + c) : 1.0f;
                T.pcb[at] = (hold_cb && in) ? __ldg(hold_cb + c) : -0.0f;
            }
            hold_cs = L.hold ? L.ch_scale : nullptr;
            hold_cb = L.hold ? L.ch_bias : nullptr;
            __syncwarp();
            if (lane == 0) mbar_arrive(&rec_full[slot]);
            if (li >= 2 && !mbar_wait_bounded_warp(&w_free[li & 1], (uint32_t)(((li >> 1) - 1) & 1), abortp, limit)) break;
            const int co16 = (L.c_out + 15) & ~15, taps = L.k * L.k;
            uint8_t* raw = wbuf + (li & 1) * FUSED_W_BYTES;
            uint64_t* bar = L.c_in <= 16 ? &w_raw[li & 1] : &w_full[li & 1];
            if (lane == 0) {
                const uint32_t bytes = (uint32_t)(taps * ((L.c_in + 31) >> 5) * co16 * 32);
                mbar_arrive_expect_tx(bar, bytes);
                bulk_copy_g2s(raw, L.w8, bytes, bar);
            }
            __syncwarp();
            if (L.c_in <= 16) {
                // 16 bytes a tap and row -- word j = channels j, 8 + j, 4 + j, 12 + j -- two taps to a 32-byte row, rows
                // swizzled as in the image
                const int uses = n_raw[li & 1]++;
                if (!mbar_wait_bounded_warp(bar, (uint32_t)(uses & 1), abortp, limit)) break;
                for (int e = lane; e < ((taps + 1) & ~1) * co16; e += 32) {
                    const int t = e / co16, row = e - t * co16, sw = (row >> 2) & 1;
                    uint4 v = make_uint4(0, 0, 0, 0);                 // the partner of an odd last tap
                    if (t < taps) {
                        const uint4* src = reinterpret_cast<const uint4*>(raw + (t * co16 + row) * 32);
                        const uint4 lo = src[sw], hi = src[sw ^ 1];
                        v = make_uint4(__byte_perm(lo.x, hi.x, 0x5410), __byte_perm(lo.y, hi.y, 0x5410), __byte_perm(lo.z, hi.z, 0x5410),
                                       __byte_perm(lo.w, hi.w, 0x5410));
                    }
                    reinterpret_cast<uint4*>(raw + FUSED_PACKED_W + ((t >> 1) * co16 + row) * 32)[(t & 1) ^ sw] = v;
                }
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&w_full[li & 1]);
            }
        }
    } else if (warp >= FUSED_ISSUER_WARP && warp < FUSED_ISSUER_WARP + FUSED_ISSUERS) {
        // =========================== MMAs ===========================
        const int k_iss = warp - FUSED_ISSUER_WARP;
        const uint32_t leader = elect_one() ? 1u : 0u;
        uint32_t par = 0u;                               // bit t: parity of the number of layers that used tile t so far
        int prev = -1, prev_tiles = 0, n_copies = 0;     // the last layer with an epilogue
        bool ok = true;
        for (int li = 0; li < n_layers && ok; ++li) {
            const int slot = li & (FUSED_RING - 1);
            if (!mbar_wait_bounded_warp(&rec_full[slot], (uint32_t)((li / FUSED_RING) & 1), abortp, limit)) break;
            const FusedLayer& L = s_rec[slot];
            const FusedGeom g = fused_geom(L);
            // (the record before it is still in the ring: this warp has not released it while it is compared)
            const bool wave = prev >= 0 && prev == li - 1 && fused_follows(s_rec[prev & (FUSED_RING - 1)], L);
            if (!mbar_wait_bounded_warp(&w_full[li & 1], (uint32_t)((li >> 1) & 1), abortp, limit)) break;
            if (L.k == 1) {                              // the subsampled copy of its input
                if (!mbar_wait_bounded_warp(&copy_ready, (uint32_t)(n_copies & 1), abortp, limit)) break;
                ++n_copies;
            }
            const int cap_in = uni(strip_cap(L.c_in));
            const bool narrow = uni(L.c_in) <= 16;
            // (narrow: the field for the distance between the halves is added per MMA)
            const uint64_t da0 = umma_desc_interleaved(smem_u32(strip_ptr(acts, L.k == 1 ? L.dst : L.src)), narrow ? 0u : (uint32_t)(cap_in * 16));
            const uint64_t db0 = umma_desc_sw32(smem_u32(wbuf + (li & 1) * FUSED_W_BYTES + (narrow ? FUSED_PACKED_W : 0)));
            const uint32_t idesc = umma_idesc_i8(g.co16);
            const uint64_t step = (uint64_t)((g.co16 * 32) >> 4);
            const int k = uni(L.k), cw = uni(g.cw), tiles = uni(g.tiles), Wf = uni(g.Wf), hold = uni(L.hold);
            const uint32_t tm0 = uni(tmem_base + (uint32_t)(L.hold ? FUSED_HOLD_COL : 0)), tm_step = uni((uint32_t)g.acc_stride);
            int waited = 0;                              // tiles of the layer before that are known to be finished
            auto wait_tiles = [&](int upto) {
                for (; waited < upto; ++waited)
                    if (!mbar_wait_bounded_warp(&ep_done[waited], ((par >> waited) & 1u) ^ 1u, abortp, limit)) return false;
                return true;
            };
            for (int t = 0; t < tiles; ++t) {
                const int need = wave ? min(prev_tiles, (t * UMMA_M + UMMA_M + Wf) / UMMA_M + 1) : prev_tiles;
                if (!wait_tiles(need)) { ok = false; break; }
                if ((t & (FUSED_ISSUERS - 1)) != k_iss) {
                    if (!hold && leader) mbar_arrive(&acc_full[t]);
                    continue;
                }
                if (skip_mma) continue;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                if (elect_one()) {
                    const uint32_t tm = tm0 + (uint32_t)t * tm_step;
                    const uint64_t da_t = da0 + (uint64_t)(t * UMMA_M);
                    uint64_t db = db0;
                    if (narrow) {
                        // taps in pairs (the ninth alone): operand row = 16 bytes at the first tap, 16 at the second
                        constexpr uint64_t LBO1 = 1ull << 16;
                        if (k == 3) {
                            const uint64_t w = (uint64_t)Wf;
                            umma_i8(tm, da_t + LBO1, db, idesc, 0u);
                            umma_i8(tm, da_t + 2 + ((w - 2) << 16), db + step, idesc, 1u);
                            umma_i8(tm, da_t + w + 1 + LBO1, db + 2 * step, idesc, 1u);
                            umma_i8(tm, da_t + 2 * w + LBO1, db + 3 * step, idesc, 1u);
                            umma_i8(tm, da_t + 2 * w + 2 + LBO1, db + 4 * step, idesc, 1u);
                        } else {
                            umma_i8(tm, da_t + (uint64_t)(Wf + 1) + LBO1, db, idesc, 0u);
                        }
                    } else if (k == 3) {
                        const uint64_t bs = step * (uint64_t)cw;              // weight tiles are ordered [tap][word]
                        for (int wd = 0; wd < cw; ++wd, db += step) {
                            const uint64_t r0 = da_t + (uint64_t)(wd * cap_in * 2), r1 = r0 + (uint64_t)Wf, r2 = r1 + (uint64_t)Wf;
                            umma_i8(tm, r0, db, idesc, wd > 0 ? 1u : 0u);
                            umma_i8(tm, r0 + 1, db + bs, idesc, 1u);
                            umma_i8(tm, r0 + 2, db + 2 * bs, idesc, 1u);
                            umma_i8(tm, r1, db + 3 * bs, idesc, 1u);
                            umma_i8(tm, r1 + 1, db + 4 * bs, idesc, 1u);
                            umma_i8(tm, r1 + 2, db + 5 * bs, idesc, 1u);
                            umma_i8(tm, r2, db + 6 * bs, idesc, 1u);
                            umma_i8(tm, r2 + 1, db + 7 * bs, idesc, 1u);
                            umma_i8(tm, r2 + 2, db + 8 * bs, idesc, 1u);
                        }
                    } else {
                        for (int wd = 0; wd < cw; ++wd, db += step)
                            umma_i8(tm, da_t + (uint64_t)(wd * cap_in * 2 + Wf + 1), db, idesc, wd > 0 ? 1u : 0u);
                    }
                }
                __syncwarp();
                if (!hold) umma_commit_pred(leader, &acc_full[t]);
            }
            if (!ok || !wait_tiles(prev_tiles)) break;   // (every phase of these barriers is waited for, so that parities stay in step)
            if (L.hold) {
                if (!skip_mma) umma_commit_pred(leader, &hold_full);
            } else {
                prev = li;
                prev_tiles = tiles;
                par ^= (1u << tiles) - 1u;
            }
            umma_commit_pred(leader, &w_free[li & 1]);
            __syncwarp();
            // the slot before this one is not looked at any more
            if (li > 0 && lane == 0) mbar_arrive(&rec_free[(li - 1) & (FUSED_RING - 1)]);
        }
        // the last commits have arrived before the block ends
        if (ok && n_layers > 0 && !*abortp) mbar_wait_bounded_warp(&w_free[(n_layers - 1) & 1], (uint32_t)(((n_layers - 1) >> 1) & 1), abortp, limit);
    } else if (warp < FUSED_EPI_WARPS) {
        // =========================== epilogue ===========================
        const int quarter = warp & 3, quad = warp >> 2;
        uint32_t par = 0u;
        int turn = 0, n_sync = 0, n_hold = 0;            // turn: units dealt so far, modulo 4
        bool ok = true;
        auto all_epilogue_warps = [&]() {
            __syncwarp();
            if (lane == 0) mbar_arrive(&epi_sync);
            const bool good = mbar_wait_bounded_warp(&epi_sync, (uint32_t)(n_sync & 1), abortp, limit);
            ++n_sync;
            return good;
        };
        for (int li = 0; li < n_layers && ok; ++li) {
            const int slot = li & (FUSED_RING - 1);
            if (!mbar_wait_bounded_warp(&rec_full[slot], (uint32_t)((li / FUSED_RING) & 1), abortp, limit)) break;
            const FusedLayer& L = s_rec[slot];
            const FusedTerms& T = s_terms[slot];
            const FusedGeom g = fused_geom(L);
            uint8_t* dst_strip = L.dst >= 0 ? strip_ptr(acts, L.dst) : nullptr;
            const int cap_out = strip_cap(L.c_out);
            if (dst_strip && (L.zero_dst || L.k == 1)) {
                // the strip's old contents have no reader left once every warp is here (its units waited for the MMAs)
                if (!all_epilogue_warps()) break;
                for (int i = tid; i < FUSED_ACT_BYTES / 16; i += FUSED_EPI_WARPS * 32) reinterpret_cast<uint4*>(dst_strip)[i] = make_uint4(0, 0, 0, 0);
                if (!all_epilogue_warps()) break;
            }
            if (L.k == 1) {
                // projection: its input is the stride-2 subsample of strip src, copied into strip dst in the output frame
                const int Wp_in = L.w_in + 2, cap_in = strip_cap(L.c_in);
                const uint8_t* src_strip = strip_ptr(acts, L.src);
                const int hshift = L.c_in <= 16 ? 0 : 1;         // 16-byte halves of a pixel and word: one or two
                for (int e = tid; e < (g.Ho * g.Wo * g.cw) << hshift; e += FUSED_EPI_WARPS * 32) {
                    const int hf = e & hshift, rest = e >> hshift, wd = rest % g.cw, pix = rest / g.cw;
                    const int ho = pix / g.Wo, wo = pix - ho * g.Wo;
                    const uint8_t* s = src_strip + wd * cap_in * 32 + hf * cap_in * 16 + ((2 * ho + 1) * Wp_in + 2 * wo + 1) * 16;
                    uint8_t* d = dst_strip + wd * cap_in * 32 + hf * cap_in * 16 + ((ho + 1) * g.Wf + wo + 1) * 16;
                    *reinterpret_cast<uint4*>(d) = *reinterpret_cast<const uint4*>(s);
                }
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&copy_ready);
                // its MMAs: before anything may overwrite the copy, and before the next layer reads their accumulators
                if (!mbar_wait_bounded_warp(&hold_full, (uint32_t)(n_hold & 1), abortp, limit)) break;
                ++n_hold;
            } else {
                const int units = g.units, ushift = units == 1 ? 0 : (units == 2 ? 1 : 2), Wp_out = g.Wo + 2;
                const bool to_pool = L.dst < 0, relu = L.relu != 0, two = L.stride == 2;
                const int Wf = g.Wf, Ho = g.Ho, Wo = g.Wo, frame = g.frame;
                const float rcp_w = __frcp_rn((float)Wf);
                FusedUnitEnv E;
                E.S2 = f32x2_pack(L.S, L.S);
                E.rs2 = f32x2_pack(L.res_step, L.res_step);
                E.one2 = f32x2_pack(one, one);
                E.inv2 = f32x2_pack(L.out_inv_step, L.out_inv_step);
                E.out_bits = L.out_bits;
                const float PS = L.res == 2 ? s_rec[(li - 1) & (FUSED_RING - 1)].S : 0.0f;
                E.PS2 = f32x2_pack(PS, PS);
                E.c_out = L.c_out;
                E.cap_out = cap_out;
                E.dst = dst_strip;
                E.res = strip_ptr(acts, L.res_buf);
                E.T = &T;
                uint8_t* tr = trace && L.trace_off >= 0 ? trace + (size_t)img * trace_stride + L.trace_off : nullptr;
                const int res = uni(L.res);
                const bool narrow = uni(L.c_out) <= 16;
                const int total = g.tiles << ushift;
                if (L.src == (to_pool ? 0 : L.dst)) {    // writes over its own input: only after the last MMA
                    for (int t = 0; t < g.tiles && ok; ++t) ok = mbar_wait_bounded_warp(&acc_full[t], (par >> t) & 1u, abortp, limit);
                    if (!ok) break;
                }
                // One loop over the tiles per form, so that a unit is straight-line code: with the choice of form (a jump through
                // a table) and the layer's fields read per unit, what preceded the arithmetic took longer than it.
                const int tiles = g.tiles, c_out = L.c_out;
                const uint32_t acc_stride = (uint32_t)g.acc_stride, trow0 = tmem_base + ((uint32_t)(quarter * 32) << 16);
                auto run = [&](auto narrow_t, auto res_t, auto pool_t) {
                    constexpr bool NARROW = decltype(narrow_t)::value, POOL = decltype(pool_t)::value;
                    constexpr int RES = decltype(res_t)::value;
#pragma unroll 1
                    for (int t = 0; t < tiles; ++t) {
                        const int f = t * UMMA_M + quarter * 32 + lane;
                        const int hp = __float2int_rd(__fmul_rn((float)f + 0.5f, rcp_w)), wp = f - hp * Wf;   // (exact: f < 2^20)
                        // does this frame row have an output, and where does it go in the destination frame
                        const int ho = two ? hp >> 1 : hp, wo = two ? wp >> 1 : wp;
                        const bool valid = f < frame && !(two && ((hp | wp) & 1)) && ho < Ho && wo < Wo;
                        const int target = two ? (ho + 1) * Wp_out + wo + 1 : f + Wf + 1;
                        const bool in_frame = f < frame && (!two || valid);          // stride 1 also writes the zeros of the padding
                        // the unit of this tile that is this warp's, if any: at most one, there are as many groups of warps as units
                        const int un = (quad - turn - (t << ushift)) & 3;
                        const bool work = un < units && __any_sync(0xffffffffu, in_frame);
                        if (!mbar_wait_bounded_warp(&acc_full[t], (par >> t) & 1u, abortp, limit)) return false;
                        if (work) {
                            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                            const uint32_t trow = trow0 + (uint32_t)t * acc_stride;
                            if constexpr (POOL) fused_unit_pool<NARROW, RES>(E, trow, un, target, valid, relu, pool_scratch + (ho * Wo + wo) * c_out);
                            else fused_unit_codes<NARROW, RES>(E, trow, un, target, valid, in_frame, tr ? tr + (size_t)(ho * Wo + wo) * c_out : nullptr);
                            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                        }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&ep_done[t]);
                    }
                    return true;
                };
                auto by_res = [&](auto narrow_t, auto pool_t) {
                    if (res == 0) return run(narrow_t, std::integral_constant<int, 0>{}, pool_t);
                    if (res == 1) return run(narrow_t, std::integral_constant<int, 1>{}, pool_t);
                    return run(narrow_t, std::integral_constant<int, 2>{}, pool_t);
                };
                using True = std::true_type;
                using False = std::false_type;
                if (to_pool) ok = narrow ? by_res(True{}, True{}) : by_res(False{}, True{});
                else ok = narrow ? by_res(True{}, False{}) : by_res(False{}, False{});
                if (!ok) break;
                turn = (turn + total) & 3;
                par ^= (1u << g.tiles) - 1u;
            }
            __syncwarp();
            // (a held projection's record is read once more by the layer after it)
            if (ok && lane == 0) {
                if (li > 0) mbar_arrive(&rec_free[(li - 1) & (FUSED_RING - 1)]);
            }
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    // ---- pooling, 8-bit quantization, classifier
    if (!abort_flag && n_layers > 0) {
        const FusedLayer& L = s_rec[(n_layers - 1) & (FUSED_RING - 1)];
        const FusedGeom g = fused_geom(L);
        const int hw = g.Ho * g.Wo, C = L.c_out;
        if (tid < C && tid < 64) {
            float acc = 0.0f;
#pragma unroll 8
            for (int p = 0; p < hw; ++p) acc = __fadd_rn(acc, pool_scratch[p * C + tid]);
            const float m = __fmul_rn(acc, 1.0f / (float)hw);
            fc_codes[tid] = quantize_act_code(m, head.a_inv_step, 255);
        }
        __syncthreads();
        const int co16 = (head.c_out + 15) & ~15;
        for (int o = warp; o < head.c_out; o += FUSED_THREADS / 32) {
            int acc = 0;
            for (int c = lane; c < head.c_in; c += 32) {
                const int wd = c >> 5, cc = c & 31, j = 4 * (cc & 7) + (cc >> 3);      // byte 4b + i of the row
                const int jj = j ^ (((o >> 2) & 1) << 4);                                 // halves swapped for these rows
                acc += (int)(int8_t)head.w8[((size_t)wd * co16 + o) * 32 + jj] * fc_codes[c];
            }
            acc = __reduce_add_sync(0xffffffffu, acc);
            if (lane == 0) {
                float y = __fmul_rn((float)acc, head.S);
                if (head.ch_scale) y = __fmul_rn(y, __ldg(head.ch_scale + o));
                if (head.ch_bias) y = __fadd_rn(y, __ldg(head.ch_bias + o));
                logits[(size_t)img * head.c_out + o] = y;
            }
        }
    }

    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == FUSED_ISSUER_WARP) {                             // (the block's memory is its own until this warp leaves)
        if (abort_flag != 0) {
            giveup_drain();
            if (lane == 0) atomicAdd(&g_umma_timeouts, 1ull);
        }
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

// Limits of the kernel for one layer; returns EBS_OK or the reason it cannot run.
static int check_layer(const FusedLayer& L, const FusedLayer* prev) {
    if (!L.w8 || (L.k != 1 && L.k != 3) || (L.stride != 1 && L.stride != 2)) return EBS_ERR_INVALID_ARG;
    if (L.c_in < 1 || L.c_in > 64 || L.c_out < 1 || L.c_out > 64 || L.h_in < 1 || L.w_in < 1) return EBS_ERR_UNSUPPORTED;
    if (L.k == 1 && (L.stride != 2 || !L.hold)) return EBS_ERR_UNSUPPORTED;        // 1x1 only as the strided projection
    if (L.stride == 2 && ((L.h_in | L.w_in) & 1)) return EBS_ERR_UNSUPPORTED;
    if (L.src < 0 || L.src > 2 || L.dst < -1 || L.dst > 2 || (L.hold && L.dst < 0)) return EBS_ERR_INVALID_ARG;
    if (L.res < 0 || L.res > 2 || (L.res == 1 && (L.res_buf < 0 || L.res_buf > 2))) return EBS_ERR_INVALID_ARG;
    if (L.res == 2 && (!prev || !prev->hold || prev->c_out != L.c_out)) return EBS_ERR_INVALID_ARG;
    if (L.dst >= 0 && !L.hold && (L.out_bits < 1 || L.out_bits > 8 || !(L.out_inv_step > 0.0f))) return EBS_ERR_INVALID_ARG;
    const int Ho = L.stride == 2 ? L.h_in / 2 : L.h_in, Wo = L.stride == 2 ? L.w_in / 2 : L.w_in;
    const int Hf = L.k == 3 ? L.h_in + 2 : Ho + 2, Wf = L.k == 3 ? L.w_in + 2 : Wo + 2;
    const int tiles = (Hf * Wf + UMMA_M - 1) / UMMA_M, co16 = (L.c_out + 15) & ~15, cw = (L.c_in + 31) >> 5;
    if (tiles * UMMA_M + 2 * Wf + 2 > strip_cap(L.c_in)) return EBS_ERR_UNSUPPORTED;          // rows the MMAs read
    if (L.dst >= 0 && !L.hold && (Ho + 2) * (Wo + 2) + Wo + 3 > strip_cap(L.c_out)) return EBS_ERR_UNSUPPORTED;   // rows written
    if ((L.hold ? FUSED_HOLD_COL : 0) + tiles * (co16 > 32 ? co16 : 32) > (L.hold ? 512 : FUSED_HOLD_COL)) return EBS_ERR_UNSUPPORTED;
    if (L.k * L.k * cw * co16 * 32 > FUSED_W_BYTES) return EBS_ERR_UNSUPPORTED;
    if (L.dst < 0 && Ho * Wo * L.c_out * 4 > FUSED_ACT_BYTES) return EBS_ERR_UNSUPPORTED;
    if ((reinterpret_cast<uintptr_t>(L.w8) & 15u) != 0) return EBS_ERR_INVALID_ARG;
    return EBS_OK;
}

int fused_plan_upload(const void* layers_host, int n_layers, void* layers_dev, cudaStream_t st) {
    const FusedLayer* L = static_cast<const FusedLayer*>(layers_host);
    for (int i = 0; i < n_layers; ++i) {
        const int rc = check_layer(L[i], i > 0 ? &L[i - 1] : nullptr);
        if (rc) return rc;
    }
    if (L[0].c_in > 4 || L[0].src != 0) return EBS_ERR_UNSUPPORTED;                   // the image goes to strip 0, <= 4 channels
    if (L[n_layers - 1].dst != -1 || L[n_layers - 1].c_out > 64) return EBS_ERR_INVALID_ARG;
    return check_cuda(cudaMemcpyAsync(layers_dev, layers_host, (size_t)n_layers * sizeof(FusedLayer), cudaMemcpyHostToDevice, st));
}

int launch_fused_resnet(const uint8_t* images, int n, int img_h, int img_w, const void* layers_dev, int n_layers,
                        const void* head_host, float* logits, uint8_t* trace, long long trace_stride, unsigned wait_limit, int test_flags,
                        cudaStream_t st) {
    static bool attr_set[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        if (check_cuda(cudaFuncSetAttribute(fused_resnet_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FUSED_SMEM)))
            return EBS_ERR_CUDA;
        attr_set[dev] = true;
    }
    FusedHead head;
    memcpy(&head, head_host, sizeof(head));
    fused_resnet_kernel<<<n, FUSED_THREADS, FUSED_SMEM, st>>>(images, img_h, img_w, static_cast<const FusedLayer*>(layers_dev),
                                                               n_layers, head, 1.0f, logits, trace, trace_stride, wait_limit, test_flags);
    return check_cuda(cudaGetLastError());
}

unsigned long long fused_net_timeouts() {
    unsigned long long v = 0;
    cudaMemcpyFromSymbol(&v, g_umma_timeouts, sizeof(v));
    return v;
}

int fused_layer_bytes() { return (int)sizeof(FusedLayer); }
int fused_head_bytes() { return (int)sizeof(FusedHead); }

}  // namespace ebs

