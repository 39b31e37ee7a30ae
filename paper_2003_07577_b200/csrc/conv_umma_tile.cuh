// One thread block per (128 frame pixels, channel tile, share of the reduction): the tcgen05 kernel for layers that do not
// fill the GPU with the pipeline kernel's super-tiles -- small batches, the deep 7x7 and 14x14 layers, odd channel
// counts -- and for the paper's weight levels.
//
// Arithmetic and addressing are those of conv_umma_pipe.cuh: planes of a packed word merged back into one byte per
// channel, one int8 MMA of 128 pixels x N channels x 32 channels of a tap, phase images and tap shifts inside a strip
// that is expanded once.  What bounds such a layer is latency: a launch, a round trip for the packed words, the chain of
// MMAs onto one accumulator (about 50 clocks each at N = 64) and the epilogue, with most SMs idle.  Hence
//  * the reduction is split over the CTAs of a cluster (up to 8) by input-channel words; each accumulates its share in its
//    own tensor memory, the copy engine brings the partial sums together in distributed shared memory and every CTA of the
//    cluster finishes its part of the pixels (exact: integer sums);
//  * all of a CTA's operands are in flight at once where they fit (100 KB, so that two CTAs share an SM and one's epilogue
//    runs under the other's MMAs), weight tiles by bulk copies of one warp, packed words by the expanders;
//  * the launch may begin while its predecessor in the stream finishes (programmatic dependent launch): barriers, tables
//    and tensor memory are set up before the wait.
// Roles (10 warps): warps 0-7 expand and later run the epilogue, warp 8 issues the MMAs, warp 9 fetches weights.
// Three forms: 1 = packed planes only, no per-channel terms, reduction not split, whole 32-channel words: out of tensor
// memory with a thread per pixel; 2 = the same with per-channel terms and shortcut; 0 = everything else: the sums go
// through shared memory and a warp finishes 32 channels of a pixel at a time (coalesced stores; the codes go back into
// shared memory as bytes and a thread packs the 32 channels of a pixel).
// TAP: the per-tap form (tap_geometry), a kernel of its own because its addresses cost the strip layers 0.4 us a launch where
// both were compiled into one.
// Weight levels (w_levels): the window sum of the codes is one more accumulator column, an MMA against a tile of ones.
// Every wait on an mbarrier is bounded as in the other tcgen05 kernels.  The two cluster barriers of a split launch have no
// limit of their own: every thread of every CTA reaches both whether it gave up or not, after bounded waits only.
#pragma once

#include <type_traits>

#include "conv_frame.cuh"

namespace ebs {

constexpr int TILE_WORKERS = 256, TILE_ISSUER = 8, TILE_PRODUCER = 9, TILE_THREADS = 320;
constexpr int TILE_SLOTS = 2;                       // (pixel, word) items an expander handles per stage
constexpr int TILE_MAX_STAGES = 16, TILE_MAX_SPLIT = 8;
constexpr int TILE_SMEM_SHARED = 104 * 1024, TILE_SMEM_MAX = 216 * 1024;   // two CTAs / one CTA per SM

struct TileGeom : FrameGeom {
    int per_tap;                       // 1: per-tap form (tap_geometry)
    FastDiv div_cw, div_kw;            // per-tap form: reduction word -> tap and channel word, tap -> row and column
    int tile_n, n_ptiles, n_ctiles, split;
    int S, SP, kw;                     // strip pixels, rounded up to 8; words per stage
    int n_words, words;                // reduction words: input-channel words (per-tap form: times taps), and those of a CTA (the
                                       // last of a cluster may have fewer)
    int a_word_bytes, b_off, stage_bytes, n_stages;
    int tmem_cols, smem_bytes, part_pitch, xch_off;   // xch_off: where a cluster's CTAs put their sums, from the stages on
    float cost;                        // estimated clocks of the launch
    bool ok;
};

inline int tile_round_up(int v, int m) { return (v + m - 1) / m * m; }

// Whether a layer has no strip: one that the expanders cannot hold (3x3 taps on more than 189 pixels of width, 5x5 on more than
// 91) or no phases in the frame scheme (strides above 2, more than 64 taps).
inline bool tile_tap_form(const ConvParams& p, FrameGeom& g) {
    return !frame_geometry(p, g) || UMMA_M + g.max_shift > TILE_SLOTS * TILE_WORKERS;
}
// The per-tap form for such layers.  The frame is the outputs
// themselves and every (tap, word) pair is a word of the reduction with a strip of its own, the 128 input pixels that the
// tap reads, expanded anew for every tap; the weight byte image has the pairs in that order.
inline bool tap_geometry(const ConvParams& p, FrameGeom& g) {
    g = FrameGeom{};
    const long long frame = (long long)p.N * p.Ho * p.Wo;
    if (frame >= (1LL << 31) - 4096 || p.CW > FRAME_MAX_CW) return false;
    g.Wq = p.Wo;
    g.Hq = p.Ho;
    g.frame = (int)frame;
    g.div_img = make_fastdiv((uint32_t)(g.Hq * g.Wq));
    g.div_row = make_fastdiv((uint32_t)g.Wq);
    g.taps = g.n_ph = g.max_ph_taps = g.ph_rows[0] = g.ph_cols[0] = g.ph_tap0[1] = 1;
    return true;
}

// Geometry for a channel tile of tile_n and a split of the reduction (0: the split with the smallest estimate).
inline TileGeom tile_geometry(const ConvParams& p, int tile_n, int sms, int split_req) {
    TileGeom g{};
    if (tile_tap_form(p, g)) {
        if (!tap_geometry(p, g)) return g;
        g.per_tap = 1;
        g.div_cw = make_fastdiv((uint32_t)p.CW);
        g.div_kw = make_fastdiv((uint32_t)p.kw);
    }
    g.n_words = p.CW * (g.per_tap ? p.kh * p.kw : 1);
    g.tile_n = tile_n;
    g.S = UMMA_M + g.max_shift;
    g.SP = tile_round_up(g.S, 8);
    g.n_ptiles = (g.frame + UMMA_M - 1) / UMMA_M;
    g.n_ctiles = (p.Co + tile_n - 1) / tile_n;
    if (g.n_ctiles > 65535) return g;
    g.tmem_cols = 32;
    while (g.tmem_cols < tile_n + (p.w_levels ? 16 : 0)) g.tmem_cols *= 2;
    if (g.tmem_cols > 512) return g;
    g.part_pitch = (tile_n + (p.w_levels ? 1 : 0) + 3) / 4 * 4 + 4;
    const int b_tile = tile_n * 32;
    TileGeom best{};
    for (int split = 1; split <= TILE_MAX_SPLIT; split *= 2) {
        if (split_req && split != split_req) continue;
        // A CTA holds its tensor memory while it waits for the others of its cluster, so clusters take at most a quarter of
        // it: no mix of resident blocks can then keep a member from starting (at most three of this kernel fit an SM).
        if (split > g.n_words || (split > 1 && g.tmem_cols > 128)) break;
        TileGeom c = g;
        c.words = (g.n_words + split - 1) / split;
        c.split = (g.n_words + c.words - 1) / c.words;
        if (c.split != split) continue;                        // a rank without words
        c.kw = TILE_SLOTS * TILE_WORKERS / c.S;
        if (c.kw > 4) c.kw = 4;
        if (c.kw > c.words) c.kw = c.words;
        // the strip of a word: two halves of SP x 16 bytes, skewed so that lanes on consecutive words hit different banks
        auto stage = [&](int kw) {
            c.a_word_bytes = c.SP * 32 + (kw == 4 ? 32 : kw == 3 ? 48 : 64);
            c.b_off = tile_round_up(kw * c.a_word_bytes, 256);
            return c.b_off + kw * c.max_ph_taps * b_tile;
        };
        const int fixed = 1024 + 512 + (split == 1 ? 0 : UMMA_M * c.part_pitch * 4);
        while (c.kw > 1 && 3 * stage(c.kw) + fixed > TILE_SMEM_SHARED) --c.kw;
        c.stage_bytes = stage(c.kw);
        const int chunks = c.n_ph * ((c.words + c.kw - 1) / c.kw);
        // the sums lie over the stages; those that the CTAs of a cluster send each other lie behind them (in `fixed`)
        const int part = UMMA_M * c.part_pitch * 4;
        const int need = chunks < 2 ? 1 : 2;
        int budget = TILE_SMEM_SHARED;
        if (need * c.stage_bytes + fixed > budget || part + fixed > budget) budget = TILE_SMEM_MAX;
        c.n_stages = (budget - fixed) / c.stage_bytes;
        if (c.n_stages > chunks) c.n_stages = chunks;
        if (c.n_stages > TILE_MAX_STAGES) c.n_stages = TILE_MAX_STAGES;
        if (c.n_stages < need) continue;
        const int body = c.n_stages * c.stage_bytes > part ? c.n_stages * c.stage_bytes : part;
        c.xch_off = body;
        c.smem_bytes = body + fixed;
        if (c.smem_bytes > TILE_SMEM_MAX) continue;
        // Estimate of the launch, fitted to about 1000 measured (layer, channel tile, split) points: the serial chain of a
        // CTA is the longer of its MMAs and its expansion plus an epilogue per channel, or the exchange of the sums; from
        // about 1.2 CTAs per SM on time grows with their number.  Of 140 other layers it picks a channel tile within 5% of the
        // fastest for 94% (1.1% off in the geometric mean, 43% with the slowest).
        const double ctas = (double)c.n_ptiles * c.n_ctiles * split;
        if (split == TILE_MAX_SPLIT && ctas > sms / 2) continue;   // (more clusters of eight than GPCs run at once: slower)
        const double mma = (double)c.words * c.taps * (17.0 + 0.34 * tile_n + (p.w_levels ? 20.0 : 0.0));
        const int cols = tile_n < tile_round_up(p.Co, 32) ? tile_n : tile_round_up(p.Co, 32);
        const double tail = split == 1 ? 21.0 * cols : 1610.0 + 114.0 * cols / split;
        double expand = 1.26 * c.words * c.n_ph * c.S, load = ctas / (1.21 * sms);
        if (c.per_tap) {                                       // a stage has one MMA per word: its waits dominate, and two CTAs on an
            expand = chunks * (1150.0 + 200.0 * c.kw);         // SM hide them (fitted to 50 layers x 4 channel tiles)
            load = ctas / ((split == 1 && c.smem_bytes <= TILE_SMEM_SHARED ? 1.6 : 1.0) * sms);
        }
        c.cost = (float)((86.0 + (mma > expand ? mma : expand) + tail) * (load > 1.0 ? load : 1.0));
        c.ok = true;
        if (!best.ok || c.cost < best.cost) best = c;
    }
    return best;
}

template <int AB, int FORM, bool TAP>
__global__ void __launch_bounds__(TILE_THREADS, 2) conv_umma_tile_kernel(const ConvParams p, const TileGeom g) {
    extern __shared__ uint8_t dyn_smem[];
    __shared__ __align__(8) uint64_t full[TILE_MAX_STAGES], empty[TILE_MAX_STAGES], acc_full, xch_full;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ int gp_s[UMMA_M];                         // output pixel of every row, -1: none
    __shared__ int s_tap_id[FRAME_MAX_TAPS];
    __shared__ __align__(16) float s_terms[FORM == 2 ? 512 : 4];   // FORM 2: scale and shift of the channel tile, frag_term_at order

    // (read from lane 0, so that the compiler knows the role branches to be warp-uniform and keeps the issuing warp's
    // descriptors in uniform registers)
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int rank = (int)blockIdx.z, split = g.split;   // cluster of `split` CTAs along z
    const int f0 = (int)blockIdx.x * UMMA_M, co0 = (int)blockIdx.y * g.tile_n;
    const int N = g.tile_n, b_tile = N * 32, KW = g.kw, NST = g.n_stages, SP = g.SP, S = g.S;
    uint8_t* ones = dyn_smem + ((1024u - (smem_u32(dyn_smem) & 1023u)) & 1023u);   // w_levels: 16 rows of ones
    uint8_t* stages = ones + 512;                        // [NST] x { KW strips, KW * taps weight tiles }; later the partial sums
    volatile int* abortp = &abort_flag;
    const unsigned limit = p.wait_limit;
    const int w0 = rank * g.words, nw = min(g.words, g.n_words - w0);
    const int nwg = (nw + KW - 1) / KW, nchunks = g.n_ph * nwg;

    if (tid == 0) {
        abort_flag = 0;
        for (int s = 0; s < NST; ++s) {
            mbar_init(&full[s], 8 + 1);                  // expander warps and the weight producer
            mbar_init(&empty[s], 1);
        }
        mbar_init(&acc_full, 1);
        mbar_init(&xch_full, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (tid < FRAME_MAX_TAPS) s_tap_id[tid] = g.tap_id[tid];
    if (p.w_levels && tid < 128) reinterpret_cast<uint32_t*>(ones)[tid] = 0x01010101u;
    if (warp == TILE_ISSUER) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_slot)),
                     "r"((uint32_t)g.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = tmem_slot;
    // The next launch may start its own set-up from here on: this CTA has its tensor memory, so nothing it still needs can
    // be taken by a CTA that waits for it.  Global memory is touched only behind the wait for the previous launch.
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    if (split > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::: "memory");   // this CTA runs: its memory may be written

    if (warp < 8) {
        // =========================== expanders ===========================
        int slot_q[TILE_SLOTS], slot_dst[TILE_SLOTS], slot_f[TILE_SLOTS];
#pragma unroll
        for (int j = 0; j < TILE_SLOTS; ++j) {
            const int e = tid + j * TILE_WORKERS;
            const int s = e / KW, q = e - s * KW;         // consecutive lanes: consecutive words of one pixel
            slot_q[j] = s < S ? q : -1;
            slot_f[j] = f0 + s;
            slot_dst[j] = q * g.a_word_bytes + s * 16;
        }
        const uint32_t* src[TILE_SLOTS];
        auto phase_pointers = [&](int ph) {
#pragma unroll
            for (int j = 0; j < TILE_SLOTS; ++j) {
                src[j] = nullptr;                        // padding, past the batch, or no item: zero bytes
                const int f = slot_f[j];
                if (slot_q[j] < 0 || f >= g.frame) continue;
                const uint32_t n = fastdiv((uint32_t)f, g.div_img);
                const uint32_t rem = (uint32_t)f - n * (uint32_t)(g.Hq * g.Wq);
                const uint32_t hq = fastdiv(rem, g.div_row), wq = rem - hq * (uint32_t)g.Wq;
                const int h = p.sh * ((int)hq + g.q0r) + g.ph_a[ph], w = p.sw * ((int)wq + g.q0s) + g.ph_b[ph];
                if ((unsigned)h < (unsigned)p.H && (unsigned)w < (unsigned)p.W)
                    src[j] = p.x + (size_t)((((int)n * p.H + h) * p.W + w) * p.CW + w0 + slot_q[j]) * AB;
            }
        };
        // TAP: first input pixel of a slot's window; its image, -1: none
        int slot_h[TILE_SLOTS], slot_w[TILE_SLOTS], slot_img[TILE_SLOTS];
        auto window_starts = [&]() {
#pragma unroll
            for (int j = 0; j < TILE_SLOTS; ++j) {
                const uint32_t f = (uint32_t)slot_f[j], n = fastdiv(f, g.div_img), rem = f - n * (uint32_t)(g.Hq * g.Wq);
                const uint32_t ho = fastdiv(rem, g.div_row), wo = rem - ho * (uint32_t)g.Wq;
                slot_h[j] = p.sh * (int)ho - p.ph;
                slot_w[j] = p.sw * (int)wo - p.pw;
                slot_img[j] = slot_q[j] >= 0 && slot_f[j] < g.frame ? (int)n : -1;
            }
        };
        // TAP: packed words of reduction word q of this CTA for slot j, null: zero bytes
        auto tap_item = [&](int j, int q) -> const uint32_t* {
            if (slot_img[j] < 0 || q >= nw) return nullptr;
            const uint32_t kk = (uint32_t)(w0 + q), tap = fastdiv(kk, g.div_cw), r = fastdiv(tap, g.div_kw);
            const int h = slot_h[j] + (int)r, w = slot_w[j] + (int)(tap - r * (uint32_t)p.kw);
            if ((unsigned)h >= (unsigned)p.H || (unsigned)w >= (unsigned)p.W) return nullptr;
            return p.x + (size_t)(((slot_img[j] * p.H + h) * p.W + w) * p.CW + (int)(kk - tap * (uint32_t)p.CW)) * AB;
        };
        constexpr int SETS = AB <= 4 ? 4 : 3;            // packed words of SETS - 1 chunks in flight
        uint32_t words[SETS][TILE_SLOTS][AB];
        int ld_ph = 0, ld_wg = 0;
        auto load_next = [&](int set) {
            if (!TAP && ld_wg == 0 && ld_ph > 0) phase_pointers(ld_ph);
#pragma unroll
            for (int j = 0; j < TILE_SLOTS; ++j) {
                const uint32_t* a;
                bool in;
                if constexpr (TAP) {
                    a = tap_item(j, ld_wg * KW + slot_q[j]);
                    in = a != nullptr;
                } else {
                    a = src[j] + (size_t)ld_wg * KW * AB;
                    in = src[j] != nullptr && ld_wg * KW + slot_q[j] < nw;
                }
                if (in && EBS_IN_RANGE(p, CHK_UT_X, (a - p.x) + AB - 1, p.lim_x)) {
                    ld_dep_words<AB>(a, words[set][j]);
                } else {
#pragma unroll
                    for (int k = 0; k < AB; ++k) words[set][j][k] = 0u;
                }
            }
            if (++ld_wg == nwg) { ld_wg = 0; ++ld_ph; }
        };
        if constexpr (TAP) window_starts();
        else phase_pointers(0);
        asm volatile("griddepcontrol.wait;\n" ::: "memory");
#pragma unroll
        for (int u = 0; u < SETS - 1; ++u)
            if (u < nchunks) load_next(u);
        bool ok = true;
        int st = 0;
        uint32_t round = 0;
        for (int c0 = 0; c0 < nchunks && ok; c0 += SETS) {
#pragma unroll
            for (int u = 0; u < SETS; ++u) {
                if (c0 + u >= nchunks) break;
                if (c0 + u + SETS - 1 < nchunks) load_next((u + SETS - 1) % SETS);
                if (round > 0 && !mbar_wait_bounded(&empty[st], (round - 1) & 1u, abortp, limit)) { ok = false; break; }
                uint8_t* A = stages + st * g.stage_bytes;
#pragma unroll
                for (int j = 0; j < TILE_SLOTS; ++j) {
                    if (slot_q[j] < 0) continue;
                    uint32_t r[8];
                    planes_to_bytes<AB>(words[u][j], r);
                    uint8_t* dst = A + slot_dst[j];
                    if (!EBS_IN_RANGE(p, CHK_UT_STAGE, (dst + SP * 16 + 15) - stages, NST * g.stage_bytes)) continue;
                    *reinterpret_cast<uint4*>(dst) = make_uint4(r[0], r[1], r[2], r[3]);
                    *reinterpret_cast<uint4*>(dst + SP * 16) = make_uint4(r[4], r[5], r[6], r[7]);
                }
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&full[st]);
                if (++st == NST) { st = 0; ++round; }
            }
        }
        // under the last MMAs: this thread's output pixel, the per-channel terms and the first shortcut values
        const int row = (warp & 3) * 32 + lane, f = f0 + row;
        int gp = -1;
        if (f < g.frame) {
            const uint32_t n = fastdiv((uint32_t)f, g.div_img);
            const uint32_t rem = (uint32_t)f - n * (uint32_t)(g.Hq * g.Wq);
            const uint32_t hq = fastdiv(rem, g.div_row), wq = rem - hq * (uint32_t)g.Wq;
            if ((int)hq < p.Ho && (int)wq < p.Wo) gp = ((int)n * p.Ho + (int)hq) * p.Wo + (int)wq;
        }
        if constexpr (FORM == 0) {
            if (warp < 4) gp_s[row] = gp;
            if (ok) mbar_wait_bounded(&acc_full, 0u, abortp, limit);
        } else {
            // =========================== epilogue, a thread per pixel ===========================
            const bool pvalid = gp >= 0;
            const size_t gpz = pvalid ? gp : 0;
            const int half = (warp >> 2) * 32;               // this warp's first group of 32 channels; every other one is its own
            const bool mine = half < N && co0 + half < p.Co;
            int gr[4];                                       // FORM 2: output pixels of the four rows of this lane's fragments
            if constexpr (FORM == 2) {
                if (tid < N) {                               // channel tid of the tile
                    const int at = (tid & ~31) + frag_term_at(tid & 31);
                    s_terms[at] = term_at(p.ch_scale, co0 + tid, p.Co, 1.0f);
                    s_terms[256 + at] = term_at(p.ch_bias, co0 + tid, p.Co, -0.0f);
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) gr[r] = __shfl_sync(0xffffffffu, gp, (lane >> 2) + 8 * r);
            }
            // the rest with the kind of shortcut and the plane count as constants of the code
            auto finish = [&](auto nb_tag, auto res_tag) {
                constexpr int NB = decltype(nb_tag)::value, RES = decltype(res_tag)::value;
                uint32_t rw[8];
                float res[32];
                auto load_shortcut = [&](int c0) {
                    if constexpr (RES == 1) {
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const float2* r2 = reinterpret_cast<const float2*>(p.residual + (size_t)max(gr[r], 0) * p.Co + co0 + c0 + 2 * (lane & 3));
#pragma unroll
                            for (int o = 0; o < 4; ++o) {
                                const uint2 t = ld_dep(reinterpret_cast<const uint2*>(r2 + 4 * o));
                                res[8 * r + 2 * o] = __uint_as_float(t.x); res[8 * r + 2 * o + 1] = __uint_as_float(t.y);
                            }
                        }
                    } else if constexpr (RES == 2) {
                        ld_dep_planes(p.res_packed + (gpz * p.CWo + ((co0 + c0) >> 5)) * p.res_bits, p.res_bits, rw);
                    }
                };
                if (mine) load_shortcut(half);
                if (ok) mbar_wait_bounded(&acc_full, 0u, abortp, limit);
                asm volatile("bar.sync 1, 256;\n" ::: "memory");
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                if (__any_sync(0xffffffffu, abort_flag != 0) || !__any_sync(0xffffffffu, pvalid)) return;
                const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);
                const FragRows rows(smem_u32(stages) + (uint32_t)warp * 1024u);   // (every MMA has read its operands)
#pragma unroll 1
                for (int c0 = half; c0 < N && co0 + c0 < p.Co; c0 += 64) {
                    uint32_t v[32], cr[8], planes[8];
                    uint32_t (&lo)[16] = *reinterpret_cast<uint32_t(*)[16]>(&v[0]);
                    uint32_t (&hi)[16] = *reinterpret_cast<uint32_t(*)[16]>(&v[16]);
                    if constexpr (FORM == 2) {
                        uint32_t rb[4][2], t[4][2];
                        tmem_ld_frag_issue(trow + (uint32_t)c0, lo);
                        tmem_ld_frag_issue(trow + (16u << 16) + (uint32_t)c0, hi);
                        if constexpr (RES == 2) {
                            uint32_t rbyte[8];
                            planes_to_bytes<8>(rw, rbyte);
                            rows.put_row(rbyte);
                            __syncwarp();
                            rows.get_frag(rb);
                            __syncwarp();                    // the codes take the place of the shortcut's
                        }
                        tmem_ld16_wait(lo);
                        tmem_ld16_wait(hi);
                        float* const none[4] = {nullptr, nullptr, nullptr, nullptr};
                        terms_codes_frag<RES, NB, false>(lo, hi, p.S, p.one, reinterpret_cast<const float2*>(s_terms + c0) + 4 * (lane & 3),
                                                         reinterpret_cast<const float2*>(s_terms + 256 + c0) + 4 * (lane & 3), res, rb,
                                                         p.res_scale, p.inv_next, NB, false, none, t);
                        rows.put_frag(t);
                        if (c0 + 64 < N && co0 + c0 + 64 < p.Co) load_shortcut(c0 + 64);
                        __syncwarp();
                        rows.get_row(cr);
                        __syncwarp();                        // (the next group's codes take their place)
                        row_to_planes<NB>(cr, NB, planes);
                    } else {
                        tmem_ld16_issue(trow + (uint32_t)c0, lo);
                        tmem_ld16_issue(trow + (uint32_t)(c0 + 16), hi);
                        tmem_ld16_wait(lo);
                        tmem_ld16_wait(hi);
                        plain_codes32<NB>(v, p.S, p.one, p.inv_next, cr);
                        codes_to_planes<NB>(cr, NB, planes);
                    }
                    if (p.Co - co0 - c0 < 32) mask_planes(planes, p.Co - co0 - c0);
                    uint32_t* dst = p.packed_next + (gpz * p.CWo + ((co0 + c0) >> 5)) * NB;
                    if (pvalid && EBS_IN_RANGE(p, CHK_UT_PN, (dst - p.packed_next) + NB - 1, p.lim_pn)) store_plane_words(planes, NB, dst);
                }
            };
            auto with_planes = [&](auto res_tag) {
                switch (p.next_bits) {
                    case 1: finish(std::integral_constant<int, 1>{}, res_tag); break;
                    case 2: finish(std::integral_constant<int, 2>{}, res_tag); break;
                    case 3: finish(std::integral_constant<int, 3>{}, res_tag); break;
                    case 4: finish(std::integral_constant<int, 4>{}, res_tag); break;
                    case 5: finish(std::integral_constant<int, 5>{}, res_tag); break;
                    case 6: finish(std::integral_constant<int, 6>{}, res_tag); break;
                    case 7: finish(std::integral_constant<int, 7>{}, res_tag); break;
                    default: finish(std::integral_constant<int, 8>{}, res_tag); break;
                }
            };
            if (FORM == 2 && p.residual) with_planes(std::integral_constant<int, FORM == 2 ? 1 : 0>{});
            else if (FORM == 2 && p.res_packed) with_planes(std::integral_constant<int, FORM == 2 ? 2 : 0>{});
            else with_planes(std::integral_constant<int, 0>{});
        }
    } else if (warp == TILE_ISSUER) {
        // =========================== issuer ===========================
        const bool levels = p.w_levels != 0;
        const bool skip_mma = (p.test_flags & 1) != 0;   // test hook: issue nothing, so that waits run out
        const uint32_t leader = elect_one() ? 1u : 0u;
        const uint64_t da0 = umma_desc_interleaved(smem_u32(stages), (uint32_t)(SP * 16)), db0 = umma_desc_sw32(smem_u32(stages + g.b_off));
        const uint32_t da_hi = (uint32_t)(da0 >> 32), db_hi = (uint32_t)(db0 >> 32), ones_lo = (uint32_t)umma_desc_sw32(smem_u32(ones));
        const uint32_t idesc = umma_idesc_i8(N), word16 = (uint32_t)g.a_word_bytes >> 4, bt16 = (uint32_t)b_tile >> 4;
        int st = 0, ph = 0, wg = 0;
        uint32_t round = 0;
        // its waits start with the data's: polls counted while the previous launch still runs would make a slow predecessor
        // look like a stage that never fills
        asm volatile("griddepcontrol.wait;\n" ::: "memory");
        for (int c = 0; c < nchunks; ++c) {
            if (!mbar_wait_bounded_warp(&full[st], round & 1u, abortp, limit)) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            if (!skip_mma) {
                // The taps of a phase are a rectangle of shifts, walked by additions; the weight tiles lie in the same order.
                const int nq = min(KW, nw - wg * KW), rows = g.ph_rows[ph], cols = g.ph_cols[ph];
                const uint32_t stage16 = (uint32_t)(st * g.stage_bytes) >> 4;
                uint32_t a_word = (uint32_t)da0 + stage16 + (uint32_t)g.ph_shift[ph], b_lo = (uint32_t)db0 + stage16;
                uint32_t accu = c == 0 ? 0u : 1u;
                if (elect_one()) {
                    for (int q = 0; q < nq; ++q, a_word += word16) {
                        uint32_t a_row = a_word;
                        for (int r = 0; r < rows; ++r, a_row += (uint32_t)g.Wq) {
                            if (cols == 3 && !levels) {
                                umma_i8_split(1u, tmem, a_row, da_hi, b_lo, db_hi, idesc, accu);
                                umma_i8_split(1u, tmem, a_row + 1u, da_hi, b_lo + bt16, db_hi, idesc, 1u);
                                umma_i8_split(1u, tmem, a_row + 2u, da_hi, b_lo + 2u * bt16, db_hi, idesc, 1u);
                                b_lo += 3u * bt16;
                                accu = 1u;
                                continue;
                            }
                            for (int s = 0; s < cols; ++s, b_lo += bt16) {
                                umma_i8_split(1u, tmem, a_row + (uint32_t)s, da_hi, b_lo, db_hi, idesc, accu);
                                if (levels) umma_i8_split(1u, tmem + (uint32_t)N, a_row + (uint32_t)s, da_hi, ones_lo, db_hi, umma_idesc_i8(16), accu);
                                accu = 1u;
                            }
                        }
                    }
                }
                __syncwarp();
                umma_commit_pred(leader, &empty[st]);
                if (c == nchunks - 1) umma_commit_pred(leader, &acc_full);
            }
            __syncwarp();
            if (++st == NST) { st = 0; ++round; }
            if (++wg == nwg) { wg = 0; ++ph; }
        }
    } else {
        // =========================== weight tiles ===========================
        asm volatile("griddepcontrol.wait;\n" ::: "memory");
        const uint32_t bytes = (uint32_t)min(N, p.Co16 - co0) * 32u;
        int st = 0, ph = 0, wg = 0;
        uint32_t round = 0;
        for (int c = 0; c < nchunks; ++c) {
            if (round > 0) {
                const bool got = mbar_wait_bounded_hot(&empty[st], (round - 1) & 1u, abortp, limit);
                if (!__all_sync(0xffffffffu, got)) break;
            }
            const int nq = min(KW, nw - wg * KW), t0 = g.ph_tap0[ph], ntaps = g.ph_tap0[ph + 1] - t0, n = nq * ntaps;
            if (lane == 0) mbar_arrive_expect_tx(&full[st], bytes * (uint32_t)n);
            __syncwarp();
            uint8_t* B = stages + st * g.stage_bytes + g.b_off;
            for (int i = lane; i < n; i += 32) {
                const int q = i / ntaps, ts = t0 + (i - q * ntaps);
                const size_t at = ((size_t)(s_tap_id[ts] * p.CW + w0 + wg * KW + q) * p.Co16 + co0) * 32;
                // (a copy skipped by the range-checked build leaves its barrier incomplete: the CTA gives up at its wait)
                if (EBS_IN_RANGE(p, CHK_UT_W8, at + bytes - 1, p.lim_w8)) bulk_copy_g2s(B + i * b_tile, p.w8 + at, bytes, &full[st]);
            }
            if (++st == NST) { st = 0; ++round; }
            if (++wg == nwg) { wg = 0; ++ph; }
        }
    }

    if constexpr (FORM == 0) {
        // =========================== epilogue through shared memory ===========================
        // A worker's TMEM row -> a row of sums [128][part_pitch] over the stages (every MMA has finished).  In a cluster each CTA
        // finishes 128 / split rows; the copy engine carries every CTA's block of those rows to it ([split][128 / split] rows
        // behind the stages), rows past the frame excepted: 1.7 us for eight CTAs and 64 channels, where reading the peers' sums
        // from the finishing threads took 2.5 and pushing them with thread stores 3.8.
        const int pitch = g.part_pitch, rows = UMMA_M / split;
        int* dump = reinterpret_cast<int*>(stages);
        int* part = reinterpret_cast<int*>(stages + (split == 1 ? 0 : g.xch_off));
        auto block_bytes = [&](int r) { return (uint32_t)(min(max(g.frame - f0 - r * rows, 0), rows) * pitch * 4); };
        // This CTA finishes rows rank * 128 / split ..; a warp takes 32 channels of four pixels at a time, a lane four
        // channels of one of them (16-byte accesses; with a channel a lane the same work took five times the instructions).
        const int groups = (N + 31) >> 5, grp = warp & (groups - 1), rstep = 8 / groups;
        const int sub = lane & 7, col = grp * 32 + 4 * sub, co = co0 + col, live = col < N ? min(max(p.Co - co, 0), 4) : 0;
        const int nb = p.next_bits, qmax = (1 << nb) - 1, word = (co0 >> 5) + grp, hw = p.Ho * p.Wo;
        const bool vec = (p.Co & 3) == 0;            // then live is 0 or 4 and every access is aligned
        float cs[4], cb[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            cs[i] = i < live ? term_at(p.ch_scale, co + i, p.Co, 1.0f) : 1.0f;
            cb[i] = i < live ? term_at(p.ch_bias, co + i, p.Co, -0.0f) : -0.0f;
        }
        __syncwarp();
        if (split > 1) asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");   // every CTA of the cluster runs
        if (warp < 8 && !__any_sync(0xffffffffu, abort_flag != 0)) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);
            int* row = dump + ((warp & 3) * 32 + lane) * pitch;
            const int cols = N + (p.w_levels ? 1 : 0);
#pragma unroll 1
            for (int c0 = (warp >> 2) * 16; c0 < cols; c0 += 32) {
                uint32_t v[16];
                tmem_ld16(trow + (uint32_t)c0, v);
                if (c0 < N) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) *reinterpret_cast<uint4*>(row + c0 + 4 * i) = make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                } else {
                    row[N] = (int)v[0];                  // the window sum
                }
            }
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        }
        __syncthreads();
        if (split > 1) {
            if (warp == 0 && abort_flag == 0) {
                if (lane == 0) mbar_arrive_expect_tx(&xch_full, (uint32_t)split * block_bytes(rank));
                __syncwarp();
                const bool mute = (p.test_flags & 2) != 0 && rank == 0;
                if (lane < split && block_bytes(lane) != 0u && !mute)
                    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                                     cluster_addr(part + rank * rows * pitch, (uint32_t)lane)),
                                 "r"(smem_u32(dump + lane * rows * pitch)), "r"(block_bytes(lane)), "r"(cluster_addr(&xch_full, (uint32_t)lane))
                                 : "memory");
            }
            __syncwarp();
            if (warp < 8 && !mbar_wait_bounded_warp(&xch_full, 0u, abortp, limit)) giveup_drain();
            __syncthreads();
            // (no CTA may end while the copies out of its memory are under way: every peer reports that it has received all, or
            // has given up and waited for its own)
            asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
        }
        if (warp < 8 && abort_flag == 0) {
            const int off = min(col, N - 4);
#pragma unroll 1
            for (int r0 = (warp / groups) * 4; r0 < rows; r0 += rstep * 4) {
                const int r = r0 + (lane >> 3), gp = gp_s[rank * rows + r];
                int* sums = part + r * pitch;
                int a[4] = {0, 0, 0, 0}, wsum = 0;
#pragma unroll
                for (int i = 0; i < TILE_MAX_SPLIT; ++i) {   // exact: integer partial sums of the cluster's CTAs
                    if (i < split) {
                        const int4 t = *reinterpret_cast<const int4*>(sums + i * rows * pitch + off);
                        a[0] += t.x; a[1] += t.y; a[2] += t.z; a[3] += t.w;
                        if (p.w_levels) wsum += sums[i * rows * pitch + N];
                    }
                }
                if (p.w_levels) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) a[i] = 2 * a[i] + wsum;
                }
                const bool out = gp >= 0 && live > 0;
                const size_t o = (size_t)(gp < 0 ? 0 : gp) * p.Co + co;
                if (p.acc && out && EBS_IN_RANGE(p, CHK_UT_ACC, o + live - 1, p.lim_out)) {
                    if (vec) *reinterpret_cast<int4*>(p.acc + o) = make_int4(a[0], a[1], a[2], a[3]);
                    else
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (i < live) p.acc[o + i] = a[i];
                }
                float y[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) y[i] = __fadd_rn(__fmul_rn(__fmul_rn((float)a[i], p.S), cs[i]), cb[i]);
                if (p.residual && out) {
                    if (vec) {
                        const float4 t = ld_dep(reinterpret_cast<const float4*>(p.residual + o));
                        y[0] = __fadd_rn(y[0], t.x); y[1] = __fadd_rn(y[1], t.y); y[2] = __fadd_rn(y[2], t.z); y[3] = __fadd_rn(y[3], t.w);
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (i < live) y[i] = __fadd_rn(y[i], ld_dep(p.residual + o + i));
                    }
                }
                if (p.res_packed && out) {
                    const uint32_t* rw = p.res_packed + ((size_t)gp * p.CWo + word) * p.res_bits;
                    uint32_t code4 = 0u;                 // plane j of the four channels -> bit j of four bytes
#pragma unroll 1
                    for (int j = 0; j < p.res_bits; ++j)
                        code4 |= ((((ld_dep(rw + j) >> (4 * sub)) & 0xFu) * 0x00204081u) & 0x01010101u) << j;
#pragma unroll
                    for (int i = 0; i < 4; ++i) y[i] = __fadd_rn(y[i], __fmul_rn(p.res_scale, byte_to_float(code4, i)));
                }
                if (p.relu) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) y[i] = y[i] > 0.0f ? y[i] : 0.0f;
                }
                if (p.y && out && EBS_IN_RANGE(p, CHK_UT_Y, o + live - 1, p.lim_out)) {
                    if (p.y_nchw) {
                        const int img = gp / hw;
                        float* dst = p.y + ((size_t)img * p.Co + co) * hw + (gp - img * hw);
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (i < live) dst[(size_t)i * hw] = y[i];
                    } else if (vec) {
                        *reinterpret_cast<float4*>(p.y + o) = make_float4(y[0], y[1], y[2], y[3]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (i < live) p.y[o + i] = y[i];
                    }
                }
                if (p.packed_next) {                     // the four codes as bytes over the start of the group's sums
                    uint32_t code4 = 0u;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (i < live) code4 |= (uint32_t)quantize_act_code(y[i], p.inv_next, qmax) << (8 * i);
                    __syncwarp();                        // every lane of these rows has read its sums
                    reinterpret_cast<uint32_t*>(sums + grp * 32)[sub] = code4;
                }
            }
            if (p.packed_next) {
                asm volatile("bar.sync 1, 256;\n" ::: "memory");
                // a thread per (pixel, 32-channel word): 32 code bytes in channel order -> plane words
                for (int e = tid; e < rows * groups; e += TILE_WORKERS) {
                    const int r = e / groups, gi = e - r * groups, gp = gp_s[rank * rows + r], wd = (co0 >> 5) + gi;
                    if (gp < 0 || wd >= p.CWo) continue;
                    const uint4* src4 = reinterpret_cast<const uint4*>(part + r * pitch + gi * 32);
                    const uint4 lo = src4[0], hi = src4[1];
                    const uint32_t n[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                    uint32_t cr[8], planes[8];
#pragma unroll
                    for (int bb = 0; bb < 8; ++bb) {     // register bb: channels bb, 8 + bb, 16 + bb, 24 + bb
                        const uint32_t sel = 0x0040u + 0x11u * (uint32_t)(bb & 3);
                        const uint32_t c4 = __byte_perm(__byte_perm(n[bb >> 2], n[2 + (bb >> 2)], sel), __byte_perm(n[4 + (bb >> 2)], n[6 + (bb >> 2)], sel), 0x5410);
                        cr[bb] = __funnelshift_l(c4, c4, bb);
                    }
                    bytes_to_planes(cr, nb, planes);
                    uint32_t* dst = p.packed_next + ((size_t)gp * p.CWo + wd) * nb;
                    if (EBS_IN_RANGE(p, CHK_UT_PN, (dst - p.packed_next) + nb - 1, p.lim_pn)) store_plane_words(planes, nb, dst);
                }
            }
        }
        __syncwarp();
        if (split > 1) asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    }

    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == TILE_ISSUER) {                           // (the block's memory is its own until this warp leaves)
        if (abort_flag != 0) {
            giveup_drain();
            if (lane == 0) atomicAdd(&g_umma_timeouts, 1ull);
        }
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"((uint32_t)g.tmem_cols) : "memory");
    }
}

int tile_sm_count();

// Whether the epilogue can run a thread per pixel (forms 1 and 2): packed planes only; an fp32 shortcut is read in whole
// 32-channel groups.
inline bool tile_thread_epilogue(const ConvParams& p, int tile_n) {
    return p.packed_next && !p.acc && !p.y && !p.w_levels && (tile_n & 31) == 0 && !(p.residual && (p.res_packed || (p.Co & 31) != 0));
}

template <int AB, int FORM, bool TAP>
int launch_conv_umma_tile_form(const ConvParams& p, const TileGeom& g, cudaStream_t st) {
    auto kern = conv_umma_tile_kernel<AB, FORM, TAP>;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, TILE_SMEM_MAX);
        attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)g.n_ptiles, (unsigned)g.n_ctiles, (unsigned)g.split);
    cfg.blockDim = dim3(TILE_THREADS, 1, 1);
    cfg.dynamicSmemBytes = (size_t)g.smem_bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = (unsigned)g.split;
    cfg.attrs = attr;
    cfg.numAttrs = g.split > 1 ? 2 : 1;
    return check_cuda(cudaLaunchKernelEx(&cfg, kern, p, g));
}

template <int AB, int TILE_N>
int launch_conv_umma_tile(const ConvParams& p, dim3 /*grid*/, cudaStream_t st) {
    const TileGeom g = tile_geometry(p, TILE_N, tile_sm_count(), p.tile_split);
    if (!g.ok) return EBS_ERR_UNSUPPORTED;                    // the geometry does not apply: nothing is launched
    const bool terms = p.ch_scale || p.ch_bias || p.residual || p.res_packed;
    const int form = g.split > 1 || !tile_thread_epilogue(p, TILE_N) ? 0 : terms ? 2 : 1;
    if (g.per_tap)
        return form == 0 ? launch_conv_umma_tile_form<AB, 0, true>(p, g, st) :
               form == 1 ? launch_conv_umma_tile_form<AB, 1, true>(p, g, st) : launch_conv_umma_tile_form<AB, 2, true>(p, g, st);
    return form == 0 ? launch_conv_umma_tile_form<AB, 0, false>(p, g, st) :
           form == 1 ? launch_conv_umma_tile_form<AB, 1, false>(p, g, st) : launch_conv_umma_tile_form<AB, 2, false>(p, g, st);
}

constexpr int NUM_TILE_VARIANTS = 5;           // TILE_N = 16, 32, 64, 128, 256

// One translation unit per activation bit count (conv_umma_tile_a1.cu .. a8.cu).
#define EBS_DEFINE_TILE_ROW(AB)                                                                            \
    const ConvVariant* conv_umma_variant_a##AB(int variant) {                                              \
        static const ConvVariant row[NUM_TILE_VARIANTS] = {                                                \
            ConvVariant{&launch_conv_umma_tile<AB, 16>, UMMA_M, 16, TILE_THREADS},                         \
            ConvVariant{&launch_conv_umma_tile<AB, 32>, UMMA_M, 32, TILE_THREADS},                         \
            ConvVariant{&launch_conv_umma_tile<AB, 64>, UMMA_M, 64, TILE_THREADS},                         \
            ConvVariant{&launch_conv_umma_tile<AB, 128>, UMMA_M, 128, TILE_THREADS},                       \
            ConvVariant{&launch_conv_umma_tile<AB, 256>, UMMA_M, 256, TILE_THREADS}};                      \
        return variant < 0 || variant >= NUM_TILE_VARIANTS ? nullptr : &row[variant];                      \
    }                                                                                                      \
    unsigned long long conv_umma_timeouts_a##AB() {                                                        \
        unsigned long long v = 0;                                                                          \
        cudaMemcpyFromSymbol(&v, g_umma_timeouts, sizeof(v));                                              \
        return v;                                                                                          \
    }

}  // namespace ebs
