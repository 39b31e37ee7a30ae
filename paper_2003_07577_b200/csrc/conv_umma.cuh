// Shared pieces of the tcgen05 convolution kernels (sm_100a): mbarrier, descriptor and tensor-memory wrappers, and the
// general epilogue out of tensor memory.
//
// The arithmetic of all of them: the plane-pair sum of the binary decomposition,
//     sum_m sum_k c_m 2^(m+k) * bitcount(AND(activation plane k, weight plane m)),
// regroups channel by channel into (sum_k 2^k a_k) * (sum_m c_m 2^m w_m): the expanders merge the planes of a packed word
// back into one byte per channel (the activation code as u8; the weight code as two's-complement s8, prepared once by
// ebs_pack_weights), and ONE int8 MMA per reduction word then retires all Wb*Ab plane pairs of its 32 channels into one
// int32 accumulator per output in tensor memory.  Operands stay bit planes in global memory; bytes exist only in shared
// memory.
//
// Every wait on an mbarrier is bounded; on a timeout the CTA raises a shared abort flag, all its
// loops end, it records the event in a device counter, frees its tensor memory and returns.
#pragma once

#include "ebs_internal.cuh"

namespace ebs {

constexpr int UMMA_M = 128;             // pixels per CTA = TMEM lanes
constexpr unsigned UMMA_WAIT_LIMIT = 1u << 20;

static __device__ unsigned long long g_umma_timeouts = 0ull;   // CTAs that gave up waiting (0 in a healthy run)

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
// Bounded wait of a whole warp for the phase with the given parity; false = gave up (or another warp already had).  The outcome is a
// vote: lanes that left a loop at a poll of their own while others went on would meet those neither at the next __syncwarp
// nor at the block's barrier.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                                  unsigned limit = UMMA_WAIT_LIMIT) {
    const uint32_t addr = smem_u32(bar);
    for (unsigned it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done) : "r"(addr), "r"(parity) : "memory");
        if (__all_sync(0xffffffffu, done != 0)) return true;
        if (__any_sync(0xffffffffu, *abort_flag != 0)) return false;
        __nanosleep(it < 8 ? 40 : 200);   // leave the issue slots to the warps that have work
    }
    *abort_flag = 1;
    return false;
}
// The same wait for one thread, or for warps that vote on the outcome themselves (weight producer): no sleep between polls (the
// try_wait itself suspends the thread for a while), so that they react as soon as the barrier flips.
__device__ __forceinline__ bool mbar_wait_bounded_hot(uint64_t* bar, uint32_t parity, volatile int* abort_flag, unsigned limit) {
    const uint32_t addr = smem_u32(bar);
    for (unsigned it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done) : "r"(addr), "r"(parity) : "memory");
        if (done) return true;
        if (*abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}

// What a CTA that gave up does before it frees its memory: copies into its shared memory and MMAs that were started may still
// be under way, and nothing waits for them any more (64 us; either takes a few).
__device__ __forceinline__ void giveup_drain() {
#pragma unroll 1
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
}

// Shared-memory matrix descriptor: K-major operand, 32-byte swizzle, rows of 32 bytes (K = 32 int8),
// 8-row groups 256 bytes apart.
__device__ __forceinline__ uint64_t umma_desc_sw32(uint32_t smem_addr) {
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr >> 4) & 0x3FFFu);     // start address, 16-byte units
    d |= (uint64_t)1u << 16;                         // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(256u >> 4) << 32;                // stride byte offset between 8-row groups
    d |= (uint64_t)1u << 46;                         // descriptor version of this architecture
    d |= (uint64_t)6u << 61;                         // layout type: 32-byte swizzle
    return d;
}

// Instruction descriptor: D = s32, A = u8 (activations), B = s8 (weights), both K-major, M = 128.
__host__ __device__ constexpr uint32_t umma_idesc_i8(int n) {
    return (2u << 4) | (0u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(UMMA_M >> 4) << 24);
}

__device__ __forceinline__ void umma_i8(uint32_t tmem_d, uint64_t desc_a, uint64_t desc_b, uint32_t idesc,
                                        uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}\n"
        :: "r"(tmem_d), "l"(desc_a), "l"(desc_b), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

// Address of 16-byte chunk c (0/1) of row `row` in a 32-byte-swizzled tile (tile base 256-byte aligned).
__device__ __forceinline__ uint8_t* sw32_chunk(uint8_t* tile, int row, int c) {
    return tile + row * 32 + ((c ^ ((row >> 2) & 1)) << 4);
}

// The two halves of a tensor-memory load: issue, and later wait.  The wait names the destination registers
// as read-write operands so that no use of them is scheduled before it.
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld16_wait(uint32_t (&v)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;\n"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                   "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
                 :: "memory");
}

// Four integers -> four bytes a | b << 8 | c << 16 | d << 24, each saturated to 0 .. 255.
__device__ __forceinline__ uint32_t pack_sat_u8x4(int a, int b, int c, int d) {
    uint32_t hi, out;
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;\n" : "=r"(hi) : "r"(d), "r"(c), "r"(0));
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;\n" : "=r"(out) : "r"(b), "r"(a), "r"(hi));
    return out;
}

// Epilogue straight out of tensor memory.  Warp w reads TMEM lanes 32 * (w % 4) .. + 31: thread `lane`
// of it owns the accumulators of one pixel row (global output pixel gp; pvalid false = row without an
// output).  Warps w and w + 4 split the channels when the tile is wide enough.  The thread stores the
// accumulators, applies the fp32 steps and packs the requantized codes of its pixel into plane words.
// AFFINE = false compiles the straight-line path without per-channel terms and shortcuts (layers that have
// them then take the general path); kernels that are built in both forms pick the form on the host, so the
// extra registers of the terms do not lower the occupancy of layers without them.
template <int TILE_N, bool AFFINE = false>
__device__ __forceinline__ void umma_epilogue(const ConvParams& p, uint32_t tmem_base, int warp, int gp, bool pvalid,
                                              int wsum_row, int co0) {
    constexpr int EPI_WARPS = TILE_N >= 64 ? 8 : 4;
    constexpr int COLS_PER_WARP = TILE_N >= 64 ? TILE_N / 2 : TILE_N;
    if (warp < EPI_WARPS) {
        const bool want_y = p.y != nullptr, want_q = p.packed_next != nullptr;
        const int qmax = (1 << p.next_bits) - 1;
        const bool vec_ok = (p.Co & 3) == 0;                        // 16-byte aligned groups of four channels
        const uint32_t trow = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
        const int hw = p.Ho * p.Wo;
        const int img = pvalid ? gp / hw : 0, rem = pvalid ? gp - img * hw : 0;
        const int cbeg = (warp >> 2) * COLS_PER_WARP;
        // Common case -- the whole channel tile exists, channels in aligned groups of four, no per-channel
        // terms, no shortcut, NHWC: straight-line code, 32 channels (one packed output word) per round.
        const bool terms_aligned = (((uintptr_t)p.ch_scale | (uintptr_t)p.ch_bias) & 15u) == 0;
        const bool no_terms = !p.ch_scale && !p.ch_bias && !p.residual && !p.res_packed;
        if (COLS_PER_WARP % 32 == 0 && co0 + TILE_N <= p.Co && vec_ok && !p.y_nchw &&
            (AFFINE ? terms_aligned : no_terms)) {
            const int nb = want_q ? p.next_bits : 0;
            const float S = p.S, inv_next = p.inv_next;
            const bool relu = p.relu != 0, w_levels = p.w_levels != 0;
            // 16 channels of this thread's pixel: store, fp32 steps, requantize, shift their plane bits into `planes`
            uint32_t resw[8];                                   // shortcut planes of the current 32-channel word
            auto process16 = [&](uint32_t (&v)[16], int cbase, uint32_t (&planes)[8]) {
                if (w_levels) {
#pragma unroll
                    for (int e = 0; e < 16; ++e) v[e] = (uint32_t)(2 * (int)v[e] + wsum_row);
                }
                const size_t o = (size_t)gp * p.Co + co0 + cbase;
                if (p.acc && pvalid) {
#pragma unroll
                    for (int gq = 0; gq < 4; ++gq)
                        *reinterpret_cast<int4*>(p.acc + o + 4 * gq) =
                            make_int4((int)v[4 * gq], (int)v[4 * gq + 1], (int)v[4 * gq + 2], (int)v[4 * gq + 3]);
                }
                if (want_y || want_q) {
                    float y[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) y[e] = __fmul_rn((float)(int)v[e], S);
                    if (AFFINE && p.ch_scale) {                 // the same 16 values for every lane: broadcast vector loads
#pragma unroll
                        for (int gq = 0; gq < 4; ++gq) {
                            const float4 t = __ldg(reinterpret_cast<const float4*>(p.ch_scale + co0 + cbase) + gq);
                            y[4 * gq] = __fmul_rn(y[4 * gq], t.x); y[4 * gq + 1] = __fmul_rn(y[4 * gq + 1], t.y);
                            y[4 * gq + 2] = __fmul_rn(y[4 * gq + 2], t.z); y[4 * gq + 3] = __fmul_rn(y[4 * gq + 3], t.w);
                        }
                    }
                    if (AFFINE && p.ch_bias) {
#pragma unroll
                        for (int gq = 0; gq < 4; ++gq) {
                            const float4 t = __ldg(reinterpret_cast<const float4*>(p.ch_bias + co0 + cbase) + gq);
                            y[4 * gq] = __fadd_rn(y[4 * gq], t.x); y[4 * gq + 1] = __fadd_rn(y[4 * gq + 1], t.y);
                            y[4 * gq + 2] = __fadd_rn(y[4 * gq + 2], t.z); y[4 * gq + 3] = __fadd_rn(y[4 * gq + 3], t.w);
                        }
                    }
                    if (AFFINE && p.residual && pvalid) {
#pragma unroll
                        for (int gq = 0; gq < 4; ++gq) {
                            const float4 t = __ldg(reinterpret_cast<const float4*>(p.residual + o) + gq);
                            y[4 * gq] = __fadd_rn(y[4 * gq], t.x); y[4 * gq + 1] = __fadd_rn(y[4 * gq + 1], t.y);
                            y[4 * gq + 2] = __fadd_rn(y[4 * gq + 2], t.z); y[4 * gq + 3] = __fadd_rn(y[4 * gq + 3], t.w);
                        }
                    }
                    if (AFFINE && p.res_packed) {               // shortcut codes from packed planes: bit i of a nibble -> byte i
                        const int sh = cbase & 16;
#pragma unroll
                        for (int gq = 0; gq < 4; ++gq) {
                            uint32_t c4r = 0u;
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                if (j >= p.res_bits) break;
                                c4r |= ((((resw[j] >> (sh + 4 * gq)) & 0xFu) * 0x00204081u) & 0x01010101u) << j;
                            }
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                y[4 * gq + e] = __fadd_rn(y[4 * gq + e],
                                                          __fmul_rn(p.res_scale, (float)((c4r >> (8 * e)) & 0xFFu)));
                        }
                    }
                    if (relu) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) y[e] = y[e] > 0.0f ? y[e] : 0.0f;
                    }
                    if (want_y && pvalid) {
#pragma unroll
                        for (int gq = 0; gq < 4; ++gq)
                            *reinterpret_cast<float4*>(p.y + o + 4 * gq) =
                                make_float4(y[4 * gq], y[4 * gq + 1], y[4 * gq + 2], y[4 * gq + 3]);
                    }
                    if (want_q) {
#pragma unroll
                        for (int gq = 3; gq >= 0; --gq) {
                            // codes of four channels as bytes: floor(y / step + 0.5), at most qmax; the pack
                            // instruction saturates at 0 (negative values, and NaN converts to 0)
                            int q[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                q[e] = min(__float2int_rd(__fadd_rn(__fmul_rn(y[4 * gq + e], inv_next), 0.5f)), qmax);
                            const uint32_t c4 = pack_sat_u8x4(q[0], q[1], q[2], q[3]);
                            // plane j of the four codes -> the top nibble of a product, shifted into the plane word
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                if (j >= nb) break;
                                const uint32_t bits = j <= 4 ? (c4 & (0x01010101u << j)) * (0x10204080u >> j)
                                                             : ((c4 >> j) & 0x01010101u) * 0x10204080u;
                                planes[j] = __funnelshift_l(bits, planes[j], 4);
                            }
                        }
                    }
                }
            };
            // the load of the next 16 channels is in flight while the current ones are processed; the upper
            // half of a 32-channel word comes first because the plane words grow by shifting left
            uint32_t va[16], vb[16];
            tmem_ld16_issue(trow + (uint32_t)(cbeg + 16), va);     // whole warp, also for rows past the end
#pragma unroll 1
            for (int c0 = cbeg; c0 < cbeg + COLS_PER_WARP; c0 += 32) {
                uint32_t planes[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
                if (AFFINE && p.res_packed) {
                    const uint32_t* rw = p.res_packed + ((size_t)gp * p.CWo + ((co0 + c0) >> 5)) * p.res_bits;
#pragma unroll
                    for (int j = 0; j < 8; ++j) resw[j] = (pvalid && j < p.res_bits) ? __ldg(rw + j) : 0u;
                }
                tmem_ld16_wait(va);
                tmem_ld16_issue(trow + (uint32_t)c0, vb);
                process16(va, c0 + 16, planes);
                tmem_ld16_wait(vb);
                if (c0 + 32 < cbeg + COLS_PER_WARP) tmem_ld16_issue(trow + (uint32_t)(c0 + 48), va);
                process16(vb, c0, planes);
                if (want_q && pvalid) {
                    uint32_t* dst = p.packed_next + ((size_t)gp * p.CWo + ((co0 + c0) >> 5)) * nb;
                    if (nb == 4) {
                        *reinterpret_cast<uint4*>(dst) = make_uint4(planes[0], planes[1], planes[2], planes[3]);
                    } else if (nb == 8) {
                        *reinterpret_cast<uint4*>(dst) = make_uint4(planes[0], planes[1], planes[2], planes[3]);
                        *reinterpret_cast<uint4*>(dst + 4) = make_uint4(planes[4], planes[5], planes[6], planes[7]);
                    } else if (nb == 2) {
                        *reinterpret_cast<uint2*>(dst) = make_uint2(planes[0], planes[1]);
                    } else {
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            if (j >= nb) break;
                            dst[j] = planes[j];
                        }
                    }
                }
            }
            return;
        }
        uint32_t planes[8];
#pragma unroll 1
        for (int c0 = cbeg; c0 < cbeg + COLS_PER_WARP; c0 += 16) {
            uint32_t v[16];
            tmem_ld16(trow + (uint32_t)c0, v);                       // whole warp, also for rows past the end
            if (p.w_levels) {
#pragma unroll
                for (int e = 0; e < 16; ++e) v[e] = (uint32_t)(2 * (int)v[e] + wsum_row);
            }
            if ((c0 & 31) == 0) {
#pragma unroll
                for (int j = 0; j < 8; ++j) planes[j] = 0u;
            }
#pragma unroll
            for (int gq = 0; gq < 4; ++gq) {                          // four channels at a time
                const int co = co0 + c0 + 4 * gq;
                uint32_t code4 = 0u;
                float yv[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int a = (int)v[4 * gq + e];
                    float y = __fmul_rn((float)a, p.S);
                    if (co + e < p.Co) {
                        if (p.ch_scale) y = __fmul_rn(y, __ldg(p.ch_scale + co + e));
                        if (p.ch_bias) y = __fadd_rn(y, __ldg(p.ch_bias + co + e));
                        if (p.residual && pvalid) y = __fadd_rn(y, __ldg(p.residual + (size_t)gp * p.Co + co + e));
                        if (p.res_packed && pvalid) y = __fadd_rn(y, packed_residual(p, gp, co + e));
                    }
                    if (p.relu && !(y > 0.0f)) y = 0.0f;
                    yv[e] = y;
                    if (want_q && co + e < p.Co) code4 |= (uint32_t)quantize_act_code(y, p.inv_next, qmax) << (8 * e);
                }
                if (pvalid && co < p.Co) {
                    const size_t o = (size_t)gp * p.Co + co;
                    if (p.acc) {
                        if (vec_ok) *reinterpret_cast<int4*>(p.acc + o) =
                            make_int4((int)v[4 * gq], (int)v[4 * gq + 1], (int)v[4 * gq + 2], (int)v[4 * gq + 3]);
                        else
                            for (int e = 0; e < 4 && co + e < p.Co; ++e) p.acc[o + e] = (int)v[4 * gq + e];
                    }
                    if (want_y) {
                        if (p.y_nchw) {
                            for (int e = 0; e < 4 && co + e < p.Co; ++e)
                                p.y[((size_t)img * p.Co + co + e) * hw + rem] = yv[e];
                        } else if (vec_ok) {
                            *reinterpret_cast<float4*>(p.y + o) = make_float4(yv[0], yv[1], yv[2], yv[3]);
                        } else {
                            for (int e = 0; e < 4 && co + e < p.Co; ++e) p.y[o + e] = yv[e];
                        }
                    }
                }
                if (want_q) {
                    const int nib_pos = ((c0 & 16) >> 2) + gq;          // which nibble of the 32-channel word
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (j < p.next_bits)
                            planes[j] |= ((((code4 >> j) & 0x01010101u) * 0x01020408u) >> 24) << (4 * nib_pos);
                }
            }
            const bool word_done = ((c0 & 16) != 0) || (c0 + 16 >= TILE_N);
            if (want_q && word_done && pvalid) {
                const int cwg = (co0 + c0) >> 5;
                if (cwg < p.CWo) {
                    uint32_t* dst = p.packed_next + ((size_t)gp * p.CWo + cwg) * p.next_bits;
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (j < p.next_bits) dst[j] = planes[j];
                }
            }
        }
    }
}

constexpr int UMMA_EXPANDERS = 256;     // threads of warps 0-7
constexpr int UMMA_THREADS = UMMA_EXPANDERS + 32;

}  // namespace ebs
