// What the strip-addressed tcgen05 kernels (conv_umma_pipe.cuh, conv_umma_tile.cuh) share: the frame of outputs with its
// phase images and tap shifts, the transposes between plane words and channel bytes, and small PTX wrappers.
#pragma once

#include "conv_umma_strip.cuh"

namespace ebs {

constexpr int FRAME_MAX_TAPS = 64, FRAME_MAX_PHASES = 4;
constexpr int FRAME_MAX_CW = 1024;                 // 32-channel words of a pixel: as far as the tile and the pipeline kernel are tested

// Exact unsigned division by a run-time constant (Granlund and Montgomery, "Division by Invariant Integers using
// Multiplication", 1994): q = (t + ((n - t) >> s1)) >> s2, t = mulhi(m, n).
struct FastDiv {
    uint32_t m, s1, s2;
};
inline FastDiv make_fastdiv(uint32_t d) {
    FastDiv f{};
    uint32_t l = 0;
    while ((1ull << l) < d) ++l;
    f.m = (uint32_t)(((1ull << 32) * ((1ull << l) - d)) / d + 1);
    f.s1 = l < 1 ? l : 1;
    f.s2 = l > 1 ? l - 1 : 0;
    return f;
}
__device__ __forceinline__ uint32_t fastdiv(uint32_t n, const FastDiv& f) {
    const uint32_t t = __umulhi(f.m, n);
    return (t + ((n - t) >> f.s1)) >> f.s2;
}

// Frame of a layer's outputs (see conv_umma_pipe.cuh: one addressing scheme for all strides), computed on the host.
struct FrameGeom {
    int Wq, Hq, frame;                 // frame of one image and pixels of all images
    FastDiv div_img, div_row;          // by Hq * Wq and by Wq
    int q0r, q0s;                      // smallest tap quotients (<= 0)
    int taps, n_ph, max_shift, max_ph_taps;
    int ph_a[FRAME_MAX_PHASES], ph_b[FRAME_MAX_PHASES];
    int ph_rows[FRAME_MAX_PHASES], ph_cols[FRAME_MAX_PHASES], ph_shift[FRAME_MAX_PHASES];   // a phase's taps: rows x cols
                                       // consecutive shifts (row pitch Wq) from ph_shift on
    int ph_tap0[FRAME_MAX_PHASES + 1]; // tap slots of phase i: [ph_tap0[i], ph_tap0[i + 1])
    short tap_shift[FRAME_MAX_TAPS];   // per tap slot: shift inside the strip, in pixels
    short tap_id[FRAME_MAX_TAPS];      // per tap slot: r * kw + s (tile index in the weight byte image)
};

inline int floordiv_int(int a, int b) { return (a >= 0) ? a / b : -((-a + b - 1) / b); }

// False when the layer is outside the scheme (stride above 2, more than 64 taps, ...).
inline bool frame_geometry(const ConvParams& p, FrameGeom& g) {
    const int taps = p.kh * p.kw;
    if (p.sh > 2 || p.sw > 2 || taps > FRAME_MAX_TAPS || p.kh > 16 || p.kw > 16) return false;
    if (p.CW > FRAME_MAX_CW) return false;
    g.q0r = floordiv_int(-p.ph, p.sh);
    g.q0s = floordiv_int(-p.pw, p.sw);
    const int qr_max = floordiv_int(p.kh - 1 - p.ph, p.sh), qs_max = floordiv_int(p.kw - 1 - p.pw, p.sw);
    g.Hq = p.Ho + qr_max - g.q0r;
    g.Wq = p.Wo + qs_max - g.q0s;
    const long long frame = (long long)p.N * g.Hq * g.Wq;
    if (frame >= (1LL << 31) - 4096) return false;
    g.frame = (int)frame;
    g.div_img = make_fastdiv((uint32_t)(g.Hq * g.Wq));
    g.div_row = make_fastdiv((uint32_t)g.Wq);
    g.max_shift = (qr_max - g.q0r) * g.Wq + (qs_max - g.q0s);
    if (g.max_shift > 30000) return false;
    g.taps = taps;
    g.n_ph = 0;
    g.max_ph_taps = 0;
    int slot = 0;
    for (int a = 0; a < p.sh; ++a)
        for (int b = 0; b < p.sw; ++b) {
            const int first = slot;
            for (int r = 0; r < p.kh; ++r) {
                const int qr = floordiv_int(r - p.ph, p.sh);
                if ((r - p.ph) - p.sh * qr != a) continue;
                for (int s = 0; s < p.kw; ++s) {
                    const int qs = floordiv_int(s - p.pw, p.sw);
                    if ((s - p.pw) - p.sw * qs != b) continue;
                    g.tap_shift[slot] = (short)((qr - g.q0r) * g.Wq + (qs - g.q0s));
                    g.tap_id[slot] = (short)(r * p.kw + s);
                    ++slot;
                }
            }
            if (slot > first) {
                g.ph_a[g.n_ph] = a;
                g.ph_b[g.n_ph] = b;
                g.ph_tap0[g.n_ph] = first;
                g.ph_shift[g.n_ph] = g.tap_shift[first];
                g.ph_cols[g.n_ph] = 1;                       // (r = stride q + a: the quotients of a phase are consecutive)
                while (first + g.ph_cols[g.n_ph] < slot && g.tap_shift[first + g.ph_cols[g.n_ph]] == g.tap_shift[first] + g.ph_cols[g.n_ph] &&
                       g.tap_id[first + g.ph_cols[g.n_ph]] / p.kw == g.tap_id[first] / p.kw) ++g.ph_cols[g.n_ph];
                g.ph_rows[g.n_ph] = (slot - first) / g.ph_cols[g.n_ph];
                ++g.n_ph;
                if (slot - first > g.max_ph_taps) g.max_ph_taps = slot - first;
            }
        }
    g.ph_tap0[g.n_ph] = slot;
    return true;
}

// NW plane words of one (pixel, 32-channel word) item -> eight registers of four channel bytes (row byte 4b + i = channel
// 8i + b).  With v_k = rotl(w_k, k), register b is rotr(t_b, b) where byte position (b + k) & 7 of t_b holds plane k.  The
// eight t_b pick the planes in eight cyclic orders, and orders that agree modulo 2 (modulo 4) share their pairs (quads)
// of planes: one bit-select per pair and parity, one per quad and residue, one per register - 24 selects for eight
// planes where a merge per (register, plane) takes 64.
__device__ __forceinline__ uint32_t bit_select(uint32_t a, uint32_t b, uint32_t m) { return (a & m) | (b & ~m); }

template <int NW>
__device__ __forceinline__ void planes_to_bytes(const uint32_t (&w)[NW], uint32_t (&r)[8]) {
    uint32_t v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = k < NW ? __funnelshift_l(w[k < NW ? k : 0], w[k < NW ? k : 0], k) : 0u;
    if constexpr (NW == 1) {
#pragma unroll
        for (int bb = 0; bb < 8; ++bb) {
            const uint32_t t = v[0] & (0x01010101u << bb);
            r[bb] = __funnelshift_r(t, t, bb);
        }
    } else {
        // pairs: plane 2j on the even bit positions and plane 2j + 1 on the odd ones (parity 0), or the reverse
        uint32_t pr[4][2];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            pr[j][0] = bit_select(v[2 * j], v[2 * j + 1], 0x55555555u);
            pr[j][1] = bit_select(v[2 * j + 1], v[2 * j], 0x55555555u);
        }
        if constexpr (NW == 2) {
#pragma unroll
            for (int bb = 0; bb < 8; ++bb) {
                const uint32_t t = pr[0][bb & 1] & ((0x01010101u << bb) | (0x01010101u << ((bb + 1) & 7)));
                r[bb] = __funnelshift_r(t, t, bb);
            }
        } else {
            // quads: the pair 2i on the positions = c, c + 1 (mod 4), the pair 2i + 1 on the other two
            uint32_t qd[2][4];
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const uint32_t m2 = c == 0 ? 0x33333333u : c == 1 ? 0x66666666u : c == 2 ? 0xCCCCCCCCu : 0x99999999u;
                    qd[i][c] = bit_select(pr[2 * i][c & 1], pr[2 * i + 1][c & 1], m2);
                }
#pragma unroll
            for (int bb = 0; bb < 8; ++bb) {
                const uint32_t m3 = 0x01010101u * (uint32_t)(((0x0Fu << bb) | (0x0Fu >> (8 - bb))) & 0xFFu);
                const uint32_t t = bit_select(qd[0][bb & 3], qd[1][bb & 3], m3);   // planes 0-3 on positions bb .. bb + 3
                r[bb] = __funnelshift_r(t, t, bb);
            }
        }
    }
}

// Eight registers of four channel bytes (byte i of register b = channel 8i + b) -> plane words: the mirror image of
// planes_to_bytes.  With c_b = rotl(bytes_b, b), plane j is rotr(t_j, j) where byte position (b + j) & 7 of t_j comes from
// register b; the pair and quad selects are shared between the planes (16 + nb selects where a merge per (plane,
// register) takes 8 * nb).
__device__ __forceinline__ void bytes_to_planes(const uint32_t (&cr)[8], int nb, uint32_t (&planes)[8]) {
    uint32_t pr[4][2], qd[2][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        pr[j][0] = bit_select(cr[2 * j], cr[2 * j + 1], 0x55555555u);
        pr[j][1] = bit_select(cr[2 * j + 1], cr[2 * j], 0x55555555u);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint32_t m2 = c == 0 ? 0x33333333u : c == 1 ? 0x66666666u : c == 2 ? 0xCCCCCCCCu : 0x99999999u;
            qd[i][c] = bit_select(pr[2 * i][c & 1], pr[2 * i + 1][c & 1], m2);
        }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (j >= nb) break;
        const uint32_t m3 = 0x01010101u * (uint32_t)(((0x0Fu << j) | (0x0Fu >> (8 - j))) & 0xFFu);
        const uint32_t t = bit_select(qd[0][j & 3], qd[1][j & 3], m3);
        planes[j] = __funnelshift_r(t, t, j);
    }
}

// tcgen05.mma with both descriptors given as (low word, high word): the start-address field sits in the low word, so
// an operand is moved by a 32-bit addition.  The whole warp executes the call with the same operands and the
// instruction is predicated on `leader` (non-zero in one lane): with the issue loop free of divergent branches its
// address arithmetic stays warp-uniform, which measured faster than a loop run by one thread alone.
__device__ __forceinline__ void umma_i8_split(uint32_t leader, uint32_t tmem_d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo,
                                              uint32_t b_hi, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "setp.ne.b32 q, %7, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::i8 [%0], da, db, %5, p;\n\t}\n"
        :: "r"(tmem_d), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate), "r"(leader)
        : "memory");
}
// Address of the same shared-memory object in the CTA of the given rank of this cluster.
__device__ __forceinline__ uint32_t cluster_addr(const void* ptr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(smem_u32(ptr)), "r"(rank));
    return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_address) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];\n" ::"r"(cluster_address) : "memory");
}
// Bounded wait on a barrier another CTA of the cluster arrives on.
__device__ __forceinline__ bool mbar_wait_cluster_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag, unsigned limit) {
    const uint32_t addr = smem_u32(bar);
    for (unsigned it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done) : "r"(addr), "r"(parity) : "memory");
        if (__all_sync(0xffffffffu, done != 0)) return true;
        if (__any_sync(0xffffffffu, *abort_flag != 0)) return false;
    }
    *abort_flag = 1;
    return false;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// The same value in every lane, known to the compiler to be so: what the issuing warps feed into descriptors and loop
// bounds has to live in uniform registers, or every MMA moves four operands there first (130 clocks an MMA instead of 40).
__device__ __forceinline__ int uni(int v) { return __shfl_sync(0xffffffffu, v, 0); }
__device__ __forceinline__ uint32_t uni(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }
// True in one lane of a converged warp, always the same one.
__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(r));
    return r != 0;
}
__device__ __forceinline__ void umma_commit_pred(uint32_t leader, uint64_t* bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "setp.ne.b32 q, %1, 0;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}\n"
        ::"r"(smem_u32(bar)), "r"(leader) : "memory");
}

// Two fp32 values in one 64-bit register for the packed fp32 instructions (one issue slot for two results; each lane is
// an individually rounded IEEE operation, identical to the scalar instruction).
__device__ __forceinline__ uint64_t f32x2_pack(float lo, float hi) {
    return ((uint64_t)__float_as_uint(hi) << 32) | (uint64_t)__float_as_uint(lo);
}
__device__ __forceinline__ uint64_t f32x2_mul_rn(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// Two rounded additions in one instruction, as multiply-adds by one: `one2` holds 1.0f twice, passed in at run time.  A
// packed addition behind a packed product comes out of the assembler as one fused operation, which changes codes at ties;
// a product by a run-time value cannot be folded that way.
__device__ __forceinline__ uint64_t f32x2_add_one(uint64_t a, uint64_t one2, uint64_t b) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(one2), "l"(b));
    return d;
}

// Global loads of what an earlier launch in the stream wrote, for kernels that may start before that launch has ended
// (programmatic dependent launch): neither through the read-only path (its data must not change while the kernel runs) nor
// movable across the wait for the earlier launch.
__device__ __forceinline__ uint32_t ld_dep(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 ld_dep(const uint2* p) {
    uint2 v;
    asm volatile("ld.global.v2.u32 {%0, %1}, [%2];\n" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ uint4 ld_dep(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld_dep(const float* p) { return __uint_as_float(ld_dep(reinterpret_cast<const uint32_t*>(p))); }
__device__ __forceinline__ float4 ld_dep(const float4* p) {
    const uint4 v = ld_dep(reinterpret_cast<const uint4*>(p));
    return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
}
// NW packed words in the widest loads their alignment (4 * NW bytes) allows.
template <int NW>
__device__ __forceinline__ void ld_dep_words(const uint32_t* src, uint32_t (&dst)[NW]) {
    if constexpr (NW % 4 == 0) {
#pragma unroll
        for (int i = 0; i < NW / 4; ++i) {
            const uint4 t = ld_dep(reinterpret_cast<const uint4*>(src) + i);
            dst[4 * i] = t.x; dst[4 * i + 1] = t.y; dst[4 * i + 2] = t.z; dst[4 * i + 3] = t.w;
        }
    } else if constexpr (NW % 2 == 0) {
#pragma unroll
        for (int i = 0; i < NW / 2; ++i) {
            const uint2 t = ld_dep(reinterpret_cast<const uint2*>(src) + i);
            dst[2 * i] = t.x; dst[2 * i + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < NW; ++i) dst[i] = ld_dep(src + i);
    }
}
// The same for a run-time number of words (1 .. 8; the others become 0).
__device__ __forceinline__ void ld_dep_planes(const uint32_t* src, int n, uint32_t (&dst)[8]) {
#pragma unroll
    for (int j = 0; j < 8; ++j) dst[j] = 0u;
    if ((n & 3) == 0) {
        const uint4 t = ld_dep(reinterpret_cast<const uint4*>(src));
        dst[0] = t.x; dst[1] = t.y; dst[2] = t.z; dst[3] = t.w;
        if (n == 8) {
            const uint4 u = ld_dep(reinterpret_cast<const uint4*>(src) + 1);
            dst[4] = u.x; dst[5] = u.y; dst[6] = u.z; dst[7] = u.w;
        }
    } else if ((n & 1) == 0) {
        const uint2 t = ld_dep(reinterpret_cast<const uint2*>(src));
        dst[0] = t.x; dst[1] = t.y;
        if (n == 6) {
            const uint2 u = ld_dep(reinterpret_cast<const uint2*>(src) + 1), w = ld_dep(reinterpret_cast<const uint2*>(src) + 2);
            dst[2] = u.x; dst[3] = u.y; dst[4] = w.x; dst[5] = w.y;
        }
    } else {
#pragma unroll
        for (int j = 0; j < 7; ++j)
            if (j < n) dst[j] = ld_dep(src + j);
    }
}

// Bounded wait for a whole warp: the outcome is a vote, so that the loops around it stay warp-uniform for the compiler.
__device__ __forceinline__ bool mbar_wait_bounded_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag, unsigned limit) {
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
    }
    *abort_flag = 1;
    return false;
}

// Four requantized codes -> one register, channel order as in planes_to_bytes.
// k256 = 256, unknown to the compiler: the first step as multiply-adds, which the logic pipe has no part in.
__device__ __forceinline__ uint32_t join_codes(const uint32_t (&m)[4], uint32_t k256) {
    return __byte_perm(m[1] * k256 + m[0], m[3] * k256 + m[2], 0x5410);
}
__device__ __forceinline__ uint32_t k256_of(float one) { return (__float_as_uint(one) & 0x00800000u) >> 15; }
// Codes of a pair of values w = fl(y / step), nb planes.  t = fl(w + 1/2) / 2^nb is clamped to [0, 1] by the addition itself
// (the scaling is exact; NaN becomes 0).  Its product with the denormal 2^nb * 2^-149, rounded down, is floor(t * 2^nb) units
// of 2^-149: the register then holds that integer, and one packed instruction serves both values.  What is clamped above comes
// out as 2^nb: with the plane count in the code (NB = 1..7) codes_to_planes spreads that bit over the planes, else (NB = 0: nb
// counted at run time; 8) it is brought down to 2^nb - 1 here.
template <int NB>
__device__ __forceinline__ void code_pair(uint64_t w, int nb, uint32_t& lo, uint32_t& hi) {
    const int n = NB == 0 ? nb : NB;
    const float down = __uint_as_float((uint32_t)(127 - n) << 23), half = 0.5f * down;
    float a, b;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;\n" : "=f"(a) : "f"(__uint_as_float((uint32_t)w)), "f"(down), "f"(half));
    asm("fma.rn.sat.f32 %0, %1, %2, %3;\n" : "=f"(b) : "f"(__uint_as_float((uint32_t)(w >> 32))), "f"(down), "f"(half));
    uint64_t d;
    const uint64_t up2 = ((uint64_t)(1u << n) << 32) | (uint64_t)(1u << n);
    asm("mul.rm.f32x2 %0, %1, %2;\n" : "=l"(d) : "l"(f32x2_pack(a, b)), "l"(up2));
    lo = (uint32_t)d;
    hi = (uint32_t)(d >> 32);
    if constexpr (NB == 0 || NB == 8) {
        lo = min(lo, (1u << n) - 1u);
        hi = min(hi, (1u << n) - 1u);
    }
}
// Code registers of code_pair<NB> -> plane words.
template <int NB>
__device__ __forceinline__ void codes_to_planes(const uint32_t (&cr)[8], int nb, uint32_t (&planes)[8]) {
    if constexpr (NB == 0 || NB == 8) {
        bytes_to_planes(cr, nb, planes);
    } else {
        bytes_to_planes(cr, NB + 1, planes);
#pragma unroll
        for (int j = 0; j < NB; ++j) planes[j] |= planes[NB];
    }
}
// Byte i of a register as fp32, exactly, without the conversion pipe: 2^23 + byte, minus 2^23.
__device__ __forceinline__ float byte_to_float(uint32_t w, int i) {
    return __fadd_rn(__uint_as_float(__byte_perm(w, 0x4B000000u, 0x7540u + (uint32_t)i)), -8388608.0f);
}

// Per-channel terms: identities (x * 1, x + (-0)) where a layer has no such term or the channel does not exist.
__device__ __forceinline__ float term_at(const float* t, int co, int Co, float identity) {
    return t && co < Co ? ld_dep(t + co) : identity;
}

// Tensor memory -> registers in fragments: 16 rows x 32 columns, lane l holds columns 8 o + 2 (l % 4) + {0, 1}, o = 0..3, of rows
// l / 4 (v[4 o], v[4 o + 1]) and l / 4 + 8 (v[4 o + 2], v[4 o + 3]).
__device__ __forceinline__ void tmem_ld_frag_issue(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
}
// A warp's fragments <-> pixels, through 1 KB of shared memory of its own: row i of 32 bytes = pixel i of the group, in two
// 16-byte halves (e = 0, 1: byte registers 2 q + e of planes_to_bytes, q = 0..3), swapped in every other run of four rows so
// that eight rows hit different banks.  A fragment register t[r][e] of lane l belongs to pixel l / 4 + 8 r and q = l % 4, which
// is how the matrix loads and stores place them.  As a transposition by shuffles the same took 40 instructions instead of 4 (with
// one instruction for two codes' floors in code_pair: 128 -> 512 1x1 at 28x28, batch 16, terms and packed shortcut, 12.3 -> 11.0
// us; 64 -> 64 3x3 at 56x56, batch 64, 29.9 -> 28.0).
struct FragRows {
    uint32_t own;                                        // half 0 of the row of this lane's pixel (half 1: own ^ 16)
    __device__ __forceinline__ explicit FragRows(uint32_t smem) {
        const uint32_t lane = threadIdx.x & 31u;
        own = smem + lane * 32u + ((lane & 4u) << 2);
    }
    __device__ __forceinline__ void put_frag(const uint32_t (&t)[4][2]) const {
#pragma unroll
        for (int e = 0; e < 2; ++e)
            asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};\n" ::"r"(own ^ (16u * e)), "r"(t[0][e]),
                         "r"(t[1][e]), "r"(t[2][e]), "r"(t[3][e]) : "memory");
    }
    __device__ __forceinline__ void get_frag(uint32_t (&t)[4][2]) const {
#pragma unroll
        for (int e = 0; e < 2; ++e)
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n" : "=r"(t[0][e]), "=r"(t[1][e]),
                         "=r"(t[2][e]), "=r"(t[3][e]) : "r"(own ^ (16u * e)) : "memory");
    }
    __device__ __forceinline__ void put_row(const uint32_t (&c)[8]) const {
#pragma unroll
        for (int e = 0; e < 2; ++e)
            asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n" ::"r"(own ^ (16u * e)), "r"(c[e]), "r"(c[2 + e]), "r"(c[4 + e]),
                         "r"(c[6 + e]) : "memory");
    }
    __device__ __forceinline__ void get_row(uint32_t (&c)[8]) const {
#pragma unroll
        for (int e = 0; e < 2; ++e)
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(c[e]), "=r"(c[2 + e]), "=r"(c[4 + e]), "=r"(c[6 + e])
                         : "r"(own ^ (16u * e)) : "memory");
    }
};
// Where the terms of a group's channel lie in the 32 floats that a lane reads eight of, at 8 (l % 4): channel 8 o + 2 q + e.
__device__ __forceinline__ int frag_term_at(int channel) { return ((channel & 7) >> 1) * 8 + (channel >> 3) * 2 + (channel & 1); }

// Shortcut of a group in fragments.  RES = 1: fp32 values, res[8 r + 2 o + e] = pixel l / 4 + 8 r, channel 8 o + 2 q + e;
// RES = 2: byte o of rb[r][e] = code of that pixel and channel.
// 1024 accumulators (lo / hi: pixels 0-15 / 16-31 of the group) -> requantized codes t (byte o of t[r][e]), and the fp32 values
// at y[r] + 8 o where VALUES and the pointer is not null.  Every fp32 step is rounded on its own, in the library's order; products
// and sums are packed two to an instruction (f32x2_add_one).  A lane needs the terms of eight channels for its four pixels
// (cs, cb: entries of frag_term_at).  The ReLU is applied to the values only: the quantizer's clamp at zero gives the same codes.
template <int RES, int NB, bool VALUES>
__device__ __forceinline__ void terms_codes_frag(const uint32_t (&lo)[16], const uint32_t (&hi)[16], float S, float one, const float2* cs,
                                                 const float2* cb, const float (&res)[32], const uint32_t (&rb)[4][2], float res_scale,
                                                 float inv_next, int nb, bool relu, float* const (&y)[4], uint32_t (&t)[4][2]) {
    const uint32_t k256 = k256_of(one);
    const uint64_t S2 = f32x2_pack(S, S), one2 = f32x2_pack(one, one), inv2 = f32x2_pack(inv_next, inv_next), rs2 = f32x2_pack(res_scale, res_scale);
    const uint64_t bias2 = f32x2_pack(-8388608.0f, -8388608.0f);
#pragma unroll
    for (int o = 3; o >= 0; --o) {
        const float2 s = cs[o], b = cb[o];
        const uint64_t s2 = f32x2_pack(s.x, s.y), b2 = f32x2_pack(b.x, b.y);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const uint32_t a0 = r < 2 ? lo[4 * o + 2 * (r & 1)] : hi[4 * o + 2 * (r & 1)];
            const uint32_t a1 = r < 2 ? lo[4 * o + 2 * (r & 1) + 1] : hi[4 * o + 2 * (r & 1) + 1];
            uint64_t w = f32x2_mul_rn(f32x2_pack((float)(int)a0, (float)(int)a1), S2);
            w = f32x2_add_one(f32x2_mul_rn(w, s2), one2, b2);
            if (RES == 1) w = f32x2_add_one(w, one2, f32x2_pack(res[8 * r + 2 * o], res[8 * r + 2 * o + 1]));
            if (RES == 2) {
                // a byte as fp32, exactly, without the conversion pipe: 2^23 + byte, minus 2^23
                const uint64_t m = ((uint64_t)__byte_perm(rb[r][1], 0x4B000000u, 0x7540u + (uint32_t)o) << 32) |
                                   (uint64_t)__byte_perm(rb[r][0], 0x4B000000u, 0x7540u + (uint32_t)o);
                uint64_t v;
                asm("add.rn.f32x2 %0, %1, %2;\n" : "=l"(v) : "l"(m), "l"(bias2));
                w = f32x2_add_one(w, one2, f32x2_mul_rn(rs2, v));
            }
            if constexpr (VALUES) {
                if (y[r]) {
                    float2 v = make_float2(__uint_as_float((uint32_t)w), __uint_as_float((uint32_t)(w >> 32)));
                    if (relu) {
                        v.x = v.x > 0.f ? v.x : 0.f;
                        v.y = v.y > 0.f ? v.y : 0.f;
                    }
                    *reinterpret_cast<float2*>(y[r] + 8 * o) = v;
                }
            }
            uint32_t m0, m1;
            code_pair<NB>(f32x2_mul_rn(w, inv2), nb, m0, m1);
            t[r][0] = o == 3 ? m0 : t[r][0] * k256 + m0;
            t[r][1] = o == 3 ? m1 : t[r][1] * k256 + m1;
        }
    }
}
// Byte registers of a pixel's codes -> plane words.
template <int NB>
__device__ __forceinline__ void row_to_planes(uint32_t (&c)[8], int nb, uint32_t (&planes)[8]) {
#pragma unroll
    for (int bb = 0; bb < 8; ++bb) c[bb] = __funnelshift_l(c[bb], c[bb], bb);
    codes_to_planes<NB>(c, nb, planes);
}

// Codes of the 32 values of a pixel's group -> eight registers (register bb: channels bb, 8 + bb, 16 + bb, 24 + bb).  value2(i, b):
// the fp32 images of channels 8 i + 2 b and 8 i + 2 b + 1, one after the other in the registers that tensor memory was read
// into: pairs taken eight channels apart, as the code registers join them, cost a move per value (64 -> 64 3x3 at 56x56, batch 256,
// 47.8 -> 45.2 us; 64 -> 256 1x1, 8 planes out, 95.3 -> 90.3).
template <int NB, class V>
__device__ __forceinline__ void pair_codes32(V value2, float one, float inv_next, int nb, uint32_t (&cr)[8]) {
    const uint32_t k256 = k256_of(one);
    const uint64_t inv2 = f32x2_pack(inv_next, inv_next);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        uint32_t m0[4], m1[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) code_pair<NB>(f32x2_mul_rn(value2(i, b), inv2), nb, m0[i], m1[i]);
        const uint32_t c0 = join_codes(m0, k256), c1 = join_codes(m1, k256);
        cr[2 * b] = __funnelshift_l(c0, c0, 2 * b);
        cr[2 * b + 1] = __funnelshift_l(c1, c1, 2 * b + 1);
    }
}
// Two fp32 values to a register: yy[i][b] = channels 8 i + 2 b and 8 i + 2 b + 1.
__device__ __forceinline__ void value_codes32(const uint64_t (&yy)[4][4], float one, float inv_next, int nb, uint32_t (&cr)[8]) {
    pair_codes32<0>([&](int i, int b) { return yy[i][b]; }, one, inv_next, nb, cr);
}
__device__ __forceinline__ void store_values32(const uint64_t (&yy)[4][4], bool relu, float* dst) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        float t[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const uint64_t w = yy[q >> 1][2 * (q & 1) + (e >> 1)];   // channel 4 q + e
            t[e] = __uint_as_float((e & 1) ? (uint32_t)(w >> 32) : (uint32_t)w);
            if (relu) t[e] = t[e] > 0.f ? t[e] : 0.f;
        }
        *reinterpret_cast<float4*>(dst + 4 * q) = make_float4(t[0], t[1], t[2], t[3]);
    }
}

// 32 accumulators of one pixel and 32-channel group -> eight registers of requantized codes of a layer without per-channel terms and
// shortcut.  SMALL: accumulators below 2^23 taken as they are (pipe_small_accumulators).
template <int NB, bool SMALL = false>
__device__ __forceinline__ void plain_codes32(const uint32_t (&v)[32], float S, float one, float inv_next, uint32_t (&cr)[8]) {
    const uint64_t S2 = f32x2_pack(S, S);
    auto value = [](uint32_t a) { return SMALL ? __uint_as_float(a) : (float)(int)a; };
    pair_codes32<NB>([&](int i, int b) { return f32x2_mul_rn(f32x2_pack(value(v[8 * i + 2 * b]), value(v[8 * i + 2 * b + 1])), S2); },
                     one, inv_next, NB, cr);
}

// Zero bits behind the last `left` channels of a group that is not whole.
__device__ __forceinline__ void mask_planes(uint32_t (&planes)[8], int left) {
#pragma unroll
    for (int j = 0; j < 8; ++j) planes[j] &= (1u << left) - 1u;
}

// A group's plane words in the widest stores their alignment (4 * nb bytes) allows.
__device__ __forceinline__ void store_plane_words(const uint32_t (&planes)[8], int nb, uint32_t* dst) {
    if (nb == 4) {
        *reinterpret_cast<uint4*>(dst) = make_uint4(planes[0], planes[1], planes[2], planes[3]);
    } else if (nb == 8) {
        *reinterpret_cast<uint4*>(dst) = make_uint4(planes[0], planes[1], planes[2], planes[3]);
        *reinterpret_cast<uint4*>(dst + 4) = make_uint4(planes[4], planes[5], planes[6], planes[7]);
    } else if (nb == 2) {
        *reinterpret_cast<uint2*>(dst) = make_uint2(planes[0], planes[1]);
    } else if (nb == 6) {
        *reinterpret_cast<uint2*>(dst) = make_uint2(planes[0], planes[1]);
        *reinterpret_cast<uint2*>(dst + 2) = make_uint2(planes[2], planes[3]);
        *reinterpret_cast<uint2*>(dst + 4) = make_uint2(planes[4], planes[5]);
    } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (j >= nb) break;
            dst[j] = planes[j];
        }
    }
}

}  // namespace ebs
