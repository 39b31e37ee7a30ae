// Persistent, warp-specialised bit-plane convolution on the tcgen05 tensor cores for every layer
// geometry the ResNet stacks contain: stride-1 k x k, strided k x k, and 1 x 1 at any stride.
//
// Arithmetic (Eq. 13-14 regrouped channel by channel): the planes of a packed
// word are merged back into one byte per channel and one int8 MMA per (tap, reduction word) retires
// all Wb*Ab plane pairs of its 32 channels.  What this kernel adds:
//
//  * One addressing scheme for all strides.  Write a tap offset as r - pad_h = stride_h * qr + a with
//    0 <= a < stride_h (likewise s - pad_w = stride_w * qs + b).  The input pixels with row parity a and
//    column parity b form a "phase" image X_ab[i][j] = X[stride_h * i + a][stride_w * j + b], and tap
//    (r, s) of output (ho, wo) reads X_ab[ho + qr][wo + qs]: a stride-1 access.  Outputs are numbered in
//    a frame of Hq x Wq pixels per image (Hq = Ho + max qr - min qr, likewise Wq) and a tap becomes a
//    constant shift (qr - min qr) * Wq + (qs - min qs) inside the strip of frame pixels a CTA expands to
//    bytes.  Stride 1 has one phase (the frame is the zero-padded input); a 3x3 stride-2 layer has
//    four, a strided 1x1 layer one (only the pixels it reads).  Every input pixel is expanded once per
//    CTA and tile, whatever the stride and however many taps read it.
//  * Super-tiles: a CTA owns m_sub x 128 consecutive frame pixels x TILE_N channels with one
//    accumulator per 128 pixels in tensor memory, so a weight tile fetched into shared memory feeds
//    m_sub MMAs and the halo of the strip is shared.
//  * Weights stay resident in shared memory when all (tap, word) tiles of a channel tile fit, else they
//    stream through the stage ring by cp.async.bulk, a stage ahead of the MMAs.
//  * Roles (20 warps, 28 where the 256-channel tile leaves as packed planes without per-channel terms): warps 0-7 expand (packed words ->
//    byte strips; the words arrive in a ring of shared memory, one to three passes ahead: by the expanders' own cp.async, or, in
//    pointwise layers of 3, 5, 6 or 7 planes whose pixels are whole 16 bytes, by tensor copies that warp 11 issues), warps 8-9
//    issue the MMAs (two warps when a tile has an even number of accumulators: each owns the accumulators of one
//    parity, so that one's waits and addresses run while the other issues), warp 10 fetches weight
//    tiles (every lane one tile of a ring slot), warps 12 on (eight, or sixteen) run the epilogue out of tensor memory while the
//    next tile's MMAs fill the other accumulator set.
//  * Bit <-> byte transposes by rotate and bit-select: with v_k = rotl(w_k, k) the byte register of
//    channels {b, 8+b, 16+b, 24+b} is rotr(t_b, b), byte position (b+k) & 7 of t_b taken from v_k; the
//    selects of plane pairs and quads are shared between the eight registers (planes_to_bytes), and the
//    epilogue packs requantized codes into plane words with the mirrored tree (bytes_to_planes).
//  * PAIR form (the 256-channel tile on a cluster of two CTAs): one MMA of M = 256 per (tap, word) over
//    both CTAs' shared and tensor memory (cta_group::2), each CTA fetching the weight rows of half the
//    channel tile; see the kernel.  Every copy into shared memory is a plain per-CTA copy; the MMAs' completion is
//    signalled to both CTAs by one tcgen05.commit each.
//
// Every wait on an mbarrier is bounded (ConvParams::wait_limit polls); on a timeout the CTA raises a
// shared abort flag, all its loops end, it records the event in a device counter, frees its tensor
// memory and returns.  The single-CTA forms use no clusters.
#pragma once

#include <cuda.h>
#include <math.h>

#include <type_traits>

#include "conv_frame.cuh"

namespace ebs {

constexpr int PIPE_EXPANDERS = 256;
// Warps 8 and 9 issue the MMAs, warp 10 fetches weights, warp 11 packed words where they come by tensor copies, warps 12 on run the
// epilogue.
constexpr int PIPE_ISSUER_WARP = 8, PIPE_ISSUERS = 2, PIPE_PRODUCER_WARP = 10, PIPE_FETCH_WARP = 11, PIPE_EPI_WARP0 = 12;
// Epilogue warps: sixteen where the 256-channel tile leaves as packed planes without per-channel terms.  These layers wait for the
// epilogue's instructions; eight warps issue in 60% of the cycles and sixteen, of 80 or 88 registers each, in 80% (64 -> 256 1x1 at
// 56x56, batch 256, 4 planes: 91.4 -> 78.1 us; 256 -> 1024 at 14x14: 31.0 -> 28.8).  Narrower tiles wait for their expanders, and the
// warps only poll beside them (512 -> 128 at 28x28: 32.9 and 35.0); terms and 32-bit results take more registers.
__host__ __device__ constexpr int pipe_epi_warps(int tile_n, bool affine, int form, bool pair) {
    return tile_n == 256 && !affine && form != 0 && !pair ? 16 : 8;
}
__host__ __device__ constexpr int pipe_threads(int epi_warps) { return (PIPE_EPI_WARP0 + epi_warps) * 32; }
constexpr int PIPE_THREADS = pipe_threads(8);
constexpr int PIPE_SLOTS = 2;                      // (pixel, word) items an expander thread handles per stage
constexpr int PIPE_MAX_ITEMS = PIPE_SLOTS * PIPE_EXPANDERS;
constexpr int PIPE_MAX_TAPS = FRAME_MAX_TAPS, PIPE_MAX_STAGES = 4;
constexpr int PIPE_MAX_BSLOTS = 32;                // weight tiles in flight when the weights stream
// Passes of packed words in the expanders' ring, where shared memory leaves room for them (8 planes: three passes measured the same);
// two at least.
__host__ __device__ constexpr int pipe_raw_depth(int words) { return words <= 4 ? 4 : words < 8 ? 3 : 2; }
constexpr int PIPE_MAX_RAW = 4;                    // slots of packed words that arrive by tensor copies
constexpr int PIPE_SMEM_MAX = 225 * 1024;          // dynamic; layers with per-channel terms or shortcuts: PIPE_SMEM_TERMS less, for the
constexpr int PIPE_SMEM_TERMS = 11 * 1024;         // epilogue warps' terms and matrix rows (FragRows, static)

// What one slot of the weight ring holds of a phase with rows x cols taps: whole words, or whole rows of taps of one word,
// or a part of a row, so that the MMAs of a slot are straight runs along the taps.  cap: tiles a slot has room for.
struct PipeSlot {
    int words, rows, cols;
};
inline PipeSlot pipe_slot(int rows, int cols, int cap) {
    PipeSlot s;
    s.cols = cols < cap ? cols : cap;
    s.rows = cols > cap ? 1 : rows * cols <= cap ? rows : cap / cols;
    s.words = rows * cols <= cap ? cap / (rows * cols) : 1;
    return s;
}

// Launch geometry, computed on the host and passed to the kernel by value.
struct PipeGeom : FrameGeom {
    int m_sub, tile_pix;               // accumulators per super-tile; 128 * m_sub
    int n_ptiles, n_ctiles;
    int S, SP;                         // strip pixels (tile_pix + largest tap shift), rounded up to 8
    int ks, nsub, kss, nwg;            // words per expander pass; passes per stage; words per stage = ks * nsub;
                                       // word groups (stages per tile and phase) = ceil(CW / kss)
    int nchunks;                       // chunks per tile = n_ph * nwg (phase-major)
    int n_stages, a_word_bytes, a_stage_bytes, stage_bytes;
    int raw_bytes, rows_bytes;         // ring of packed words; rows of planes on their way out (pipe_rows_apply)
    int raw_words, raw_slots, raw_slot_bytes;   // words of a pixel in a slot of that ring (a multiple of ks)
    int ring_full;                     // by cp.async: 1: the ring has its full depth, in slots of PIPE_MAX_ITEMS items, 0: two slots of the strip's size
    int tma;                           // 1: a slot arrives by a tensor copy (one box; two where a tile has 512 pixels), 0: by the expanders' own cp.async
    int linear_in, linear_out;         // a frame pixel is the input pixel, the output pixel, of the same number
    int b_resident, b_total_bytes;
    PipeSlot slot[FRAME_MAX_PHASES];   // of each phase
    int b_slots, b_group;              // streamed weights: ring of slots of b_group (tap, word) tiles of TILE_N x 32 bytes
    int nbuf, tmem_cols, smem_bytes;
    int pair;                          // 1: two CTAs of a cluster share every MMA (256 pixels x 256 channels, half a weight tile each)
    int grid_x, grid_y;
    bool ok;
};

// Kernel form for a layer: 0 = every output mode; 1 = packed planes only (the usual layer of a network: its epilogue holds nothing
// but the lean group, or the group with per-channel terms); 2 = form 1 with the planes of two neighbouring groups passing through
// shared memory.  What else is compiled into a kernel costs the path that runs: with two epilogue forms in one kernel layers were
// 15-25% slower.
inline bool pipe_packed_only(const ConvParams& p) {
    return p.packed_next && !p.acc && !p.y && !p.y_nchw && !p.w_levels && !(p.residual && (p.res_packed || (p.Co & 31) != 0));
}
// Form 2.  A group's planes are 4 * nb bytes of its pixel; with 32 lanes storing their own pixel's planes, 5 or 7 planes are as many
// single-word stores of 32 sectors each and 6 planes three half-width ones.  As rows of two groups in shared memory they leave in
// runs of 8-byte stores, four lanes to a pixel.  us, direct and through rows: 64 -> 256 1x1 at 56x56, batch 256, 5 planes 185 and 84 (held back
// in registers until four groups filled wide stores: 99), 6 planes 113 and 84, 7 planes 264 and 88 (104); 256 -> 1024 at 14x14, 3
// planes 47 and 29, 6 planes 50 and 31; 256 -> 128 at 56x56, 5 planes 94 and 68, 6 planes 70 and 68.  Even counts that fill one or two 16-byte
// stores are faster direct (4 planes: 73 and 80; 8 planes: 90 and 101), 3 planes in the 128-channel tile too (60 and 64).
inline bool pipe_rows_apply(const ConvParams& p, int tile_n) {
    const int nb = p.next_bits;
    return tile_n >= 128 && pipe_packed_only(p) && (p.Co & 63) == 0 && ((nb >= 5 && nb <= 7) || (nb == 3 && tile_n == 256));
}
inline bool pipe_has_terms(const ConvParams& p) { return p.ch_scale || p.ch_bias || p.residual || p.res_packed; }
inline int pipe_rows_bytes(const ConvParams& p, int tile_n, bool pair) {
    return !pair && pipe_rows_apply(p, tile_n) ? pipe_epi_warps(tile_n, pipe_has_terms(p), 2, false) * 32 * 8 * p.next_bits : 0;
}

// The geometry with packed words by tensor copies (copies) or by cp.async; see pipe_geometry.
inline PipeGeom pipe_geometry_with(const ConvParams& p, int tile_n, int sms, int m_sub_req, bool pair, bool copies) {
    PipeGeom g{};
    if (pair && (tile_n != 256 || (p.Co % 256) != 0 || sms < 2)) return g;
    const int pw = pair ? 2 : 1;                               // CTAs that share a pixel pair-tile
    g.pair = pair ? 1 : 0;
    sms /= pw;                                                 // the unit that takes work items: a CTA, or a pair
    if (p.w_levels || (tile_n != 64 && tile_n != 128 && tile_n != 256)) return g;
    if (!frame_geometry(p, g)) return g;
    const int taps = g.taps, max_shift = g.max_shift, max_ph_taps = g.max_ph_taps;
    const long long frame = g.frame;
    g.n_ctiles = (p.Co + tile_n - 1) / tile_n;
    const int b_tile = tile_n * 32 / pw;                       // a pair: each CTA holds the rows of half the channels
    g.b_total_bytes = p.CW * taps * b_tile;
    const int deep = p.CW * taps;                               // MMAs per accumulator and tile
    // candidates for the super-tile, largest first: it must leave the strip within the expanders' items and give
    // the SMs enough tiles; a deep reduction prefers the widest accumulator set even without double buffering
    const int m_cap = 512 / tile_n;                             // accumulators that fit in tensor memory at all
    int m_sub = 0;
    for (int m = m_cap; m >= 1; m >>= 1) {
        if (m_sub_req && m != m_sub_req) continue;
        const int nb = (2 * m * tile_n <= 512) ? 2 : 1;
        if (nb == 1 && deep < 64 && !m_sub_req) continue;        // shallow reductions want the epilogue overlapped
        if (m * UMMA_M + max_shift > PIPE_MAX_ITEMS) continue;
        const long long pt = (frame + (long long)m * UMMA_M * pw - 1) / ((long long)m * UMMA_M * pw);
        // Expander lanes run over the words of a pass first: with one word a pass every lane of a load reads a line of its
        // own, which for pixels of about a line or more, expanded for one tap only, costs more than the larger strip saves (256 -> 64
        // 1x1 at 56x56, batch 128: 4 bits 40.3 -> 36.6 us with half the pixels and two words, 5 bits 56.1 -> 40.7).  Over 42
        // layers of 64 channels the gain is 1.00-1.38 from 24 words a pixel on and would be 1.00-1.11 below.
        if (!m_sub_req && m > 1 && taps == 1 && m * UMMA_M > PIPE_MAX_ITEMS / 2 && p.CW > 2 && p.CW * p.x_words >= 24) continue;
        if (!m_sub_req && m > 1 && pt * g.n_ctiles < (deep >= 64 ? 1LL : 2LL) * sms) continue;
        m_sub = m;
        break;
    }
    if (!m_sub) return g;
    g.m_sub = m_sub;
    g.tile_pix = m_sub * UMMA_M;
    g.nbuf = (2 * m_sub * tile_n <= 512) ? 2 : 1;
    g.tmem_cols = g.nbuf * m_sub * tile_n;
    if (g.tmem_cols < 32) g.tmem_cols = 32;
    g.n_ptiles = (int)((frame + (long long)g.tile_pix * pw - 1) / ((long long)g.tile_pix * pw));   // pair-tiles for a pair
    g.S = g.tile_pix + max_shift;
    g.SP = (g.S + 7) & ~7;
    g.a_word_bytes = g.SP * 32 + 64;                           // sized with the largest skew; fixed once ks is known
    if (g.SP * 16 >= (1 << 18)) return g;
    // weights resident when they leave room for at least two activation stages
    const int smem_max = PIPE_SMEM_MAX - (pipe_has_terms(p) ? PIPE_SMEM_TERMS : 0);
    g.linear_in = taps == 1 && p.sh == 1 && p.sw == 1 && p.ph == 0 && p.pw == 0;
    g.linear_out = g.Hq == p.Ho && g.Wq == p.Wo;
    g.rows_bytes = pipe_rows_bytes(p, tile_n, pair);
    if (copies && (!g.linear_in || pair || p.x_words < 3 || p.x_words == 4 || p.x_words == 8 || p.CW * p.x_words % 4 != 0)) return g;
    // A slot of the ring of packed words: a pass of the strip, or what a tensor copy brings, whole 16 bytes of every pixel (2 or 4 words).
    // Two slots are enough where shared memory is short: the ring gets its full depth only where that displaces neither resident weights nor
    // words of a pass.  us with the full ring throughout, and so: 512 -> 256 1x1 at 28x28, batch 256, 7 planes in and out 82.3 and
    // 53.7; 256 -> 128 at 56x56 140 and 79.8; 512 -> 128 at 28x28, 5 planes 53.3 and 32.7; strided 608 -> 2048 1x1 at 58x29, 5 planes 534 and 281; 128 ->
    // 128 3x3 at 28x28, batch 64, 7 planes and terms 25.6 and 17.9.  A third stage instead of the deeper ring: 224 -> 64 3x3 stride 2 259 and 356.
    auto slot_words = [&](int k) {
        int u = k;
        while (copies && u % (p.x_words == 6 ? 2 : 4) != 0) u += k;
        return u;
    };
    auto slot_bytes = [&](int k) { return ((copies ? g.tile_pix : g.S) * slot_words(k) * p.x_words * 4 + 127) & ~127; };
    const int budget = smem_max - 2048 - g.rows_bytes;
    int ks = PIPE_MAX_ITEMS / g.S;
    if (ks > 4) ks = 4;
    if (ks > p.CW) ks = p.CW;
    if (ks < 1) return g;
    const int full_ring = pipe_raw_depth(p.x_words) * PIPE_MAX_ITEMS * p.x_words * 4;
    // Streamed weights go through a ring of their own (slots of a few consecutive (tap, word) tiles), so that copies are
    // in flight all the time (a stage-sized unit would leave the copy engine idle while a stage's MMAs run).
    auto stage_bytes = [&](int k) { return (k * g.a_word_bytes + 255) & ~255; };
    // Weights stay resident beside two stages of whole passes; a layer of several taps, whose weight traffic is the larger, keeps them beside
    // stages of one word too (1184 -> 320 1x1, 7 planes: 391 us streamed, 648 resident with one word a pass).
    auto beside = [&](int b_bytes, int k, int words, int ring) { return b_bytes + 2 * stage_bytes(words) + ring <= budget; };
    g.b_resident = g.b_total_bytes <= 160 * 1024 && (beside(g.b_total_bytes, ks, slot_words(ks), 2 * slot_bytes(ks)) ||
                                                     (taps > 1 && beside(g.b_total_bytes, 1, slot_words(1), 2 * slot_bytes(1))));
    const int b_bytes = g.b_resident ? g.b_total_bytes : 96 * 1024 / pw, avail = budget - b_bytes;
    while (ks > 1 && !beside(b_bytes, ks, slot_words(ks), 2 * slot_bytes(ks))) --ks;
    if (!beside(b_bytes, ks, slot_words(ks), 2 * slot_bytes(ks))) return g;
    // A stage is filled in nsub expander passes of ks words: the waits, addresses and commits of a stage cost an issuing
    // warp a thousand clocks, to be spread over some forty MMAs (64 -> 64 3x3 at 56x56, batch 256: 55.6 us with a word a
    // stage, 18 MMAs, 50.3 with two; 256 -> 256 3x3 stride 2 at 28x28: 65.1 and 49.9).
    int nsub = slot_words(ks) / ks;                            // (a stage holds whole slots)
    if (nsub > 4) return g;
    auto short_of = [&](int mmas) { return nsub < 4 && ks * nsub * taps * m_sub < mmas && ks * nsub < p.CW; };
    const int ring = full_ring > 2 * slot_bytes(ks) ? full_ring : 2 * slot_bytes(ks);
    while (short_of(40) && beside(b_bytes, ks, ks * 2 * nsub, ring)) nsub *= 2;
    // (a single word of nine taps is too short a stage even so: 128 -> 128 3x3 at 28x28, batch 256, 6 planes: 44.7 and 43.1; from some 32 MMAs
    // on the third stage and the deeper ring are worth more: 672 -> 2048 3x3 886 and 910, 896 -> 256 1x1 63.5 and 74.2)
    while (taps > 1 && short_of(32) && beside(b_bytes, ks, ks * 2 * nsub, 2 * slot_bytes(ks))) nsub *= 2;
    // Skew between the word tiles of a pass: the 8 lanes of a quarter warp store 16 bytes each for ks words of 8 / ks
    // pixels; a skew of 128 / ks bytes (48 for three words) puts them on eight different 16-byte bank groups.
    g.a_word_bytes = g.SP * 32 + (ks == 4 ? 32 : ks == 3 ? 48 : 64);
    g.ks = ks;
    g.nsub = nsub;
    g.kss = ks * nsub;
    g.nwg = (p.CW + g.kss - 1) / g.kss;
    g.nchunks = g.n_ph * g.nwg;
    g.a_stage_bytes = stage_bytes(g.kss);
    g.stage_bytes = g.a_stage_bytes;
    const int st_cap = g.b_resident ? PIPE_MAX_STAGES : (pair ? PIPE_MAX_STAGES : 3);
    g.tma = copies;
    g.raw_words = slot_words(ks);
    g.raw_slot_bytes = slot_bytes(ks);
    const int reserve = beside(b_bytes, ks, g.kss, ring) ? ring : 2 * g.raw_slot_bytes;
    g.n_stages = (avail - reserve) / g.stage_bytes;
    if (g.n_stages > st_cap) g.n_stages = st_cap;
    if (!g.b_resident) {
        // a slot holds up to 32 KB of consecutive tiles (one wait and one commit per slot, not per MMA); where three do not fit beside the
        // stages (a CTA pair reserves half as much for them), fewer stages make room, then smaller slots
        auto weight_slots = [&](int most) {
            g.b_group = 1;
            for (int i = 0; i < g.n_ph; ++i) {
                const PipeSlot sl = g.slot[i] = pipe_slot(g.ph_rows[i], g.ph_cols[i], most);
                if (sl.words * sl.rows * sl.cols > g.b_group) g.b_group = sl.words * sl.rows * sl.cols;
            }
            g.b_slots = (budget - reserve - g.n_stages * g.stage_bytes) / (g.b_group * b_tile);
            return g.b_slots >= 3;
        };
        int most = 32768 / b_tile > g.kss * max_ph_taps ? g.kss * max_ph_taps : 32768 / b_tile;
        while (!weight_slots(most)) {
            if (g.n_stages > 2) --g.n_stages;
            else if (most > 1) most >>= 1;
            else return g;
        }
        if (g.b_slots > PIPE_MAX_BSLOTS) g.b_slots = PIPE_MAX_BSLOTS;
    }
    const int fixed = (g.b_resident ? g.b_total_bytes : g.b_slots * g.b_group * b_tile) + g.rows_bytes + 1024;
    const int left = smem_max - fixed - g.n_stages * g.stage_bytes;
    g.ring_full = !copies && left >= full_ring;
    if (g.ring_full) g.raw_slot_bytes = PIPE_MAX_ITEMS * p.x_words * 4;
    g.raw_slots = copies ? (left / g.raw_slot_bytes < PIPE_MAX_RAW ? left / g.raw_slot_bytes : PIPE_MAX_RAW) : g.ring_full ? pipe_raw_depth(p.x_words) : 2;
    g.raw_bytes = g.raw_slots * g.raw_slot_bytes;
    g.smem_bytes = fixed + g.n_stages * g.stage_bytes + g.raw_bytes;
    if (g.b_resident) {                                        // a CTA keeps one channel tile
        g.grid_y = g.n_ctiles;
        long long gx = sms / g.n_ctiles;
        if (gx < 1) gx = 1;
        if (gx > g.n_ptiles) gx = g.n_ptiles;
        g.grid_x = (int)gx * pw;
    } else {
        g.grid_y = 1;
        const long long items = (long long)g.n_ptiles * g.n_ctiles;
        g.grid_x = (int)(items < sms ? items : sms) * pw;
    }
    g.ok = g.n_stages >= 2 && g.smem_bytes <= smem_max && g.grid_y <= 65535 && g.n_ctiles <= 65535;
    return g;
}

// m_sub_req = 0: chosen here.  Returns ok = false when the kernel does not apply.
// Packed words come by tensor copies where the strip is a run of input pixels and a thread's own words are no whole 16 bytes (3, 5, 6, 7
// planes): cp.async then moves 8 or 4 bytes a lane, which 5 to 7 planes wait for.  A copy takes whole 16 bytes of every pixel (2 or 4
// words), and its box at most 256 pixels and 256 words.  us, by cp.async and by tensor copies: 512 -> 128 1x1 at 28x28, batch 256, 7 planes
// 74.3 and 41.1 (6 planes 49.0 and 37.0); 256 -> 64 at 56x56, 5 planes 68.9 and 57.6; 1024 -> 256 at 14x14, 7 planes 37.0 and 26.8; 256 ->
// 128, 3 planes 65.9 and 63.4.  With 1, 2, 4 and 8 planes, whose items are fetched in whole, it made no difference (256 -> 64, 4 planes: 57.2
// and 57.5 in one form of the loop).  copies = false: by cp.async in every layer; a layer that applies does so either way.
inline PipeGeom pipe_geometry(const ConvParams& p, int tile_n, int sms, int m_sub_req = 0, bool pair = false, bool copies = true) {
    const PipeGeom g = pipe_geometry_with(p, tile_n, sms, m_sub_req, pair, false);
    if (!copies || !g.ok) return g;
    const PipeGeom t = pipe_geometry_with(p, tile_n, sms, m_sub_req, pair, true);
    return t.ok && t.b_resident == g.b_resident ? t : g;
}

// umma_i8_split for a CTA pair: M = 256 over the two CTAs' tensor memory, issued by the even CTA; the commit arrives on the
// barrier at this offset in both CTAs.
__device__ __forceinline__ void umma_i8_split_pair(uint32_t leader, uint32_t tmem_d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo,
                                                   uint32_t b_hi, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "setp.ne.b32 q, %7, 0;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::i8 [%0], da, db, %5, p;\n\t}\n"
        :: "r"(tmem_d), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate), "r"(leader)
        : "memory");
}
// Completion of the pair's MMAs issued so far, signalled to the barrier at this offset in both CTAs: one commit on the
// issuing (even) CTA's barrier and one on the odd CTA's, whose address in the cluster window is passed in.
__device__ __forceinline__ void umma_commit_pred_pair(uint32_t leader, uint64_t* bar, uint32_t peer_delta) {
    const uint32_t own = smem_u32(bar);
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "setp.ne.b32 q, %2, 0;\n\t"
        "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t"
        "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%1];\n\t}\n"
        ::"r"(own), "r"(own + peer_delta), "r"(leader) : "memory");
}

// One 32-channel group of the plain epilogue with 32-bit results: 32 accumulators of this thread's pixel -> stores, fp32
// steps, requantized codes -> plane words.
// The float -> int conversion issues at an eighth of the fp32 rate on this machine (16 results per clock and SM against
// 128 fp32 operations) and was what bounded the epilogue, so the floor and the clamp are done with an fp32 addition and
// integer min / max instead (see below); the fp32 steps run as packed two-lane instructions.
template <bool WANT_Q>
__device__ __forceinline__ void pipe_group32(const ConvParams& p, uint32_t (&v)[32], size_t o, bool pvalid, float S,
                                             float inv_next, int nb, uint32_t* dst) {
    if (p.acc && pvalid && EBS_IN_RANGE(p, CHK_PIPE_ACC, o + 31, p.lim_out)) {
#pragma unroll
        for (int gq = 0; gq < 8; ++gq)
            *reinterpret_cast<int4*>(p.acc + o + 4 * gq) =
                make_int4((int)v[4 * gq], (int)v[4 * gq + 1], (int)v[4 * gq + 2], (int)v[4 * gq + 3]);
    }
    // y = fl(float(acc) * S) for the 32 channels, two to a register: yy[i][b] = channels 8 i + 2 b and 8 i + 2 b + 1
    uint64_t yy[4][4];
    const uint64_t S2 = f32x2_pack(S, S);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int b = 0; b < 4; ++b)
            yy[i][b] = f32x2_mul_rn(f32x2_pack((float)(int)v[8 * i + 2 * b], (float)(int)v[8 * i + 2 * b + 1]), S2);
    if (p.y && pvalid && EBS_IN_RANGE(p, CHK_PIPE_Y, o + 31, p.lim_out)) store_values32(yy, p.relu != 0, p.y + o);
    if (WANT_Q) {
        // The clamp at zero of the quantizer makes an explicit ReLU redundant here: a negative y gives
        // floor(y / step + 0.5) <= 0 and is clamped to code 0, exactly what max(y, 0) would give.
        uint32_t cr[8];
        value_codes32(yy, p.one, inv_next, nb, cr);
        uint32_t planes[8];
        bytes_to_planes(cr, nb, planes);
        if (pvalid && EBS_IN_RANGE(p, CHK_PIPE_PN, (dst - p.packed_next) + nb - 1, p.lim_pn)) store_plane_words(planes, nb, dst);
    }
}

// Planes on their way out of a form-2 kernel: a row of 2 * NB words per pixel of the warp, two neighbouring groups of 32 channels.
template <int NB>
__device__ __forceinline__ void pipe_row_put(uint32_t rows, int second, const uint32_t (&planes)[8]) {
    const uint32_t at = rows + (threadIdx.x & 31u) * (8u * NB) + (uint32_t)second * (4u * NB);
    if constexpr (NB % 2 == 0) {
#pragma unroll
        for (int k = 0; k < NB; k += 2) asm volatile("st.shared.v2.u32 [%0], {%1, %2};\n" ::"r"(at + 4 * k), "r"(planes[k]), "r"(planes[k + 1]) : "memory");
    } else {
#pragma unroll
        for (int k = 0; k < NB; ++k) asm volatile("st.shared.u32 [%0], %1;\n" ::"r"(at + 4 * k), "r"(planes[k]) : "memory");
    }
}
// Both groups of every row are there: the rows leave, four lanes to a pixel.  gp: this lane's output pixel, -1: none; word: the first
// group's channel word.
template <int NB>
__device__ __forceinline__ void pipe_rows_leave(const ConvParams& p, uint32_t rows, int gp, int word) {
    const int lane = (int)(threadIdx.x & 31), q = lane & 3;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int px = 8 * i + (lane >> 2), to = __shfl_sync(0xffffffffu, gp, px);
        uint32_t* out = p.packed_next + ((size_t)max(to, 0) * p.CWo + word) * NB + 2 * q;
        const uint32_t from = rows + (uint32_t)(px * (8 * NB) + 8 * q);
#pragma unroll
        for (int r = 0; 4 * r < NB; ++r) {
            if (to >= 0 && q + 4 * r < NB && EBS_IN_RANGE(p, CHK_PIPE_PN, (out - p.packed_next) + 8 * r + 1, p.lim_pn)) {
                uint32_t x, y;
                asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];\n" : "=r"(x), "=r"(y) : "r"(from + 32 * r) : "memory");
                *reinterpret_cast<uint2*>(out + 8 * r) = make_uint2(x, y);
            }
        }
    }
    __syncwarp();                                            // (the next pair of groups takes their place)
}

// The same group when only packed planes are asked for (a chained network: no accumulator and no fp32 output): the
// four channels of a byte register go from accumulator to code in one short chain, so that nothing but the 32
// accumulators and the finished code registers is alive at a time -- the general form above keeps the 32 fp32 images
// as well, which at 96 registers costs spills and the parallelism of the instruction stream.
template <int NB, bool SMALL>
__device__ __forceinline__ void pipe_group32_packed(const uint32_t (&v)[32], float S, float inv_next, const ConvParams& p, uint32_t (&planes)[8]) {
    uint32_t cr[8];
    plain_codes32<NB, SMALL>(v, S, p.one, inv_next, cr);
    codes_to_planes<NB>(cr, NB, planes);
}

// Epilogue of a layer with per-channel terms and / or a shortcut (a folded batch normalisation, the second convolution of a
// residual block): NHWC, packed planes and / or fp32 out.  The warp walks its (accumulator, 32-channel group) units; the next
// unit's accumulators, shortcut and terms are requested before the current one is packed and stored.  The accumulators are
// loaded as fragments (terms_codes_frag), so that a lane reads the terms of eight channels instead of 32, and the codes -- and
// the codes of a packed shortcut the other way -- pass through shared memory as matrices (FragRows).  terms: 64 floats of the
// warp's own, rows: 1 KB.  VALUES: fp32 output may be wanted too, stored from the fragments (whole 32-byte sectors).
template <int TILE_N, bool ROWS, bool VALUES, int NB, int RES>
__device__ __forceinline__ void pipe_epilogue_terms_nb(const ConvParams& p, const FrameGeom& g, uint32_t tmem_set, int m_sub, int vwarp,
                                                    int f0, int co0, float* terms, const FragRows& rows, uint32_t out_rows) {
    const int lane = (int)(threadIdx.x & 31), quad = lane & 3;
    const int at = frag_term_at(lane);
    const uint32_t trow = tmem_set + ((uint32_t)((vwarp & 3) * 32) << 16);
    constexpr int COLS = TILE_N / 2;
    const int cbeg = (vwarp >> 2) * COLS, cend = COLS == 32 ? cbeg + 32 : min(cbeg + COLS, p.Co - co0);   // (cend: groups start below)
    if (co0 + cbeg >= p.Co) return;
    const int nb = NB > 0 ? NB : p.next_bits;                // (a constant where only planes are written)
    float res[32], t_scale, t_bias;
    uint32_t rw[8];
    int gp = 0, gr[4];                                       // output pixels of this lane's row and of its fragment's four rows
    bool pvalid = false;
    uint32_t lo[16], hi[16];
    auto locate = [&](int j) {
        const int f = f0 + j * UMMA_M;
        pvalid = false;
        gp = 0;
        if (f < g.frame) {
            const uint32_t n = fastdiv((uint32_t)f, g.div_img);
            const uint32_t rem = (uint32_t)f - n * (uint32_t)(g.Hq * g.Wq);
            const uint32_t hq = fastdiv(rem, g.div_row), wq = rem - hq * (uint32_t)g.Wq;
            if ((int)hq < p.Ho && (int)wq < p.Wo) {
                pvalid = true;
                gp = ((int)n * p.Ho + (int)hq) * p.Wo + (int)wq;
            }
        }
        if constexpr (RES == 1 || VALUES) {
#pragma unroll
            for (int r = 0; r < 4; ++r) gr[r] = __shfl_sync(0xffffffffu, pvalid ? gp : -1, (lane >> 2) + 8 * r);
        }
    };
    auto request = [&](int c) {                              // c: first channel of the unit
        const bool in = c + lane < p.Co;
        t_scale = p.ch_scale && in ? __ldg(p.ch_scale + c + lane) : 1.0f;
        t_bias = p.ch_bias && in ? __ldg(p.ch_bias + c + lane) : -0.0f;
        if constexpr (RES == 1) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float2* r2 = reinterpret_cast<const float2*>(p.residual + (size_t)max(gr[r], 0) * p.Co + c + 2 * quad);
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                    const float2 t = __ldg(r2 + 4 * o);
                    res[8 * r + 2 * o] = t.x; res[8 * r + 2 * o + 1] = t.y;
                }
            }
        } else if constexpr (RES == 2) {
            ld_dep_planes(p.res_packed + ((size_t)gp * p.CWo + (c >> 5)) * p.res_bits, p.res_bits, rw);
        }
    };
    auto load = [&](int j, int c0) {
        tmem_ld_frag_issue(trow + (uint32_t)(j * TILE_N + c0), lo);
        tmem_ld_frag_issue(trow + (16u << 16) + (uint32_t)(j * TILE_N + c0), hi);
    };
    // (the next unit's accumulators are requested early only where the registers hold them)
    constexpr bool EARLY = !VALUES && !ROWS;
    locate(0);
    request(co0 + cbeg);
    if (EARLY) load(0, cbeg);
    int j = 0, c0 = cbeg;
#pragma unroll 1
    while (true) {
        const int c = co0 + c0;
        const bool ok = pvalid, some = __any_sync(0xffffffffu, ok);   // (none: 32 frame pixels without an output)
        const size_t gpz = gp;
        const int cn = c0 + 32 < cend ? c0 + 32 : cbeg, jn = c0 + 32 < cend ? j : j + 1;
        __syncwarp();                                        // every lane has read the unit before
        terms[at] = t_scale;
        terms[32 + at] = t_bias;
        uint32_t rb[4][2], t[4][2];
        if (!EARLY) load(j, c0);
        if constexpr (RES == 2) {
            uint32_t rbyte[8];
            planes_to_bytes<8>(rw, rbyte);
            rows.put_row(rbyte);
        }
        __syncwarp();
        if constexpr (RES == 2) {
            rows.get_frag(rb);
            __syncwarp();                                    // the codes take the place of the shortcut's
        }
        tmem_ld16_wait(lo);
        tmem_ld16_wait(hi);
        if (some) {
            float* y[4];
            if constexpr (VALUES) {
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const size_t o = (size_t)max(gr[r], 0) * p.Co + c + 2 * quad;
                    y[r] = p.y && gr[r] >= 0 && EBS_IN_RANGE(p, CHK_PIPE_Y, o + 25, p.lim_out) ? p.y + o : nullptr;
                }
            }
            terms_codes_frag<RES, NB, VALUES>(lo, hi, p.S, p.one, reinterpret_cast<const float2*>(terms) + 4 * quad,
                                              reinterpret_cast<const float2*>(terms + 32) + 4 * quad, res, rb, p.res_scale, p.inv_next,
                                              nb, p.relu != 0, y, t);
            if (!VALUES || p.packed_next) rows.put_frag(t);
        }
        if (jn < m_sub) {
            if (EARLY) load(jn, cn);
            if (jn != j) locate(jn);
            request(co0 + cn);
        }
        __syncwarp();
        if (some && (!VALUES || p.packed_next)) {
            uint32_t cr[8], planes[8];
            rows.get_row(cr);
            row_to_planes<NB>(cr, nb, planes);
            if (p.Co - c < 32) mask_planes(planes, p.Co - c);
            if constexpr (ROWS) {
                pipe_row_put<NB>(out_rows, (c >> 5) & 1, planes);
                if (c & 32) pipe_rows_leave<NB>(p, out_rows, ok ? (int)gpz : -1, (c >> 5) - 1);
            } else {
                uint32_t* dst = p.packed_next + (gpz * p.CWo + (c >> 5)) * nb;
                if (ok && EBS_IN_RANGE(p, CHK_PIPE_PN, (dst - p.packed_next) + nb - 1, p.lim_pn)) store_plane_words(planes, nb, dst);
            }
        }
        if (jn >= m_sub) break;
        j = jn;
        c0 = cn;
    }
}

// Plain epilogue with 32-bit results (no per-channel terms, no shortcut, NHWC, c_out a multiple of 32; without such results:
// pipe_epilogue_packed_nb) of one 128-pixel accumulator.  vwarp 0..7: TMEM lane quarter vwarp % 4, channel half vwarp / 4.
template <int TILE_N>
__device__ __forceinline__ void pipe_epilogue_plain(const ConvParams& p, uint32_t tmem_acc, int vwarp, int gp, bool pvalid,
                                                      int co0) {
    const uint32_t trow = tmem_acc + ((uint32_t)((vwarp & 3) * 32) << 16);
    constexpr int COLS = TILE_N / 2;
    const int cbeg = (vwarp >> 2) * COLS;
    const bool want_q = p.packed_next != nullptr;
    const int nb = want_q ? p.next_bits : 0;
    const float S = p.S, inv_next = p.inv_next;
    uint32_t v[32];
#pragma unroll 1
    for (int c0 = cbeg; c0 < cbeg + COLS; c0 += 32) {
        if (co0 + c0 >= p.Co) break;
        uint32_t (&lo)[16] = *reinterpret_cast<uint32_t(*)[16]>(&v[0]);
        uint32_t (&hi)[16] = *reinterpret_cast<uint32_t(*)[16]>(&v[16]);
        tmem_ld16_issue(trow + (uint32_t)c0, lo);
        tmem_ld16_issue(trow + (uint32_t)(c0 + 16), hi);
        tmem_ld16_wait(lo);
        tmem_ld16_wait(hi);
        const size_t o = (size_t)gp * p.Co + co0 + c0;
        uint32_t* dst = p.packed_next + ((size_t)gp * p.CWo + ((co0 + c0) >> 5)) * nb;
        if (want_q) {
            pipe_group32<true>(p, v, o, pvalid, S, inv_next, nb, dst);
        } else {
            pipe_group32<false>(p, v, o, pvalid, S, inv_next, nb, dst);
        }
    }
}

// Packed-only epilogue without per-channel terms of one 128-pixel accumulator: nothing but the lean
// group, for the kernel forms that are launched only for such layers.  A last group of fewer than 32 channels writes zero bits behind them.
template <int TILE_N, bool ROWS, bool SMALL, int EPI_WARPS, int NB>
__device__ __forceinline__ void pipe_epilogue_packed_nb(const ConvParams& p, uint32_t tmem_acc, int vwarp, int gp, bool pvalid,
                                                       int co0, uint32_t out_rows) {
    const uint32_t trow = tmem_acc + ((uint32_t)((vwarp & 3) * 32) << 16);
    constexpr int COLS = TILE_N * 4 / EPI_WARPS;
    const int cbeg = (vwarp >> 2) * COLS;
    const float S = p.S, inv_next = p.inv_next;
    uint32_t v[32];
    uint32_t* dst = p.packed_next + ((size_t)gp * p.CWo + ((co0 + cbeg) >> 5)) * NB;
#pragma unroll 1
    for (int c0 = cbeg; c0 < cbeg + COLS; c0 += 32, dst += NB) {
        if (co0 + c0 >= p.Co) break;
        uint32_t (&lo)[16] = *reinterpret_cast<uint32_t(*)[16]>(&v[0]);
        uint32_t (&hi)[16] = *reinterpret_cast<uint32_t(*)[16]>(&v[16]);
        tmem_ld16_issue(trow + (uint32_t)c0, lo);
        tmem_ld16_issue(trow + (uint32_t)(c0 + 16), hi);
        tmem_ld16_wait(lo);
        tmem_ld16_wait(hi);
        uint32_t planes[8];
        pipe_group32_packed<NB, SMALL>(v, S, inv_next, p, planes);
        if constexpr (ROWS) {
            pipe_row_put<NB>(out_rows, (c0 >> 5) & 1, planes);
            if (c0 & 32) pipe_rows_leave<NB>(p, out_rows, pvalid ? gp : -1, (co0 + c0 - 32) >> 5);
        } else {
            if (p.Co - co0 - c0 < 32) mask_planes(planes, p.Co - co0 - c0);
            if (pvalid && EBS_IN_RANGE(p, CHK_PIPE_PN, (dst - p.packed_next) + NB - 1, p.lim_pn)) store_plane_words(planes, NB, dst);
        }
    }
}

// The plane count as a constant of the code: with run-time counts every group ran through a dozen branches (plane loops,
// store widths), which cost the epilogue warps more in instruction fetch than their arithmetic.
#define EBS_PIPE_EACH_NB(CALL)                                                                                    \
    if constexpr (ROWS) {                                                                                         \
        switch (p.next_bits) {                                                                                    \
            case 3: { constexpr int NB = 3; CALL; } break;                                                        \
            case 5: { constexpr int NB = 5; CALL; } break;                                                        \
            case 6: { constexpr int NB = 6; CALL; } break;                                                        \
            default: { constexpr int NB = 7; CALL; } break;                                                       \
        }                                                                                                         \
    } else {                                                                                                      \
        switch (p.next_bits) {                                                                                    \
            case 1: { constexpr int NB = 1; CALL; } break;                                                        \
            case 2: { constexpr int NB = 2; CALL; } break;                                                        \
            case 3: { constexpr int NB = 3; CALL; } break;                                                        \
            case 4: { constexpr int NB = 4; CALL; } break;                                                        \
            case 5: { constexpr int NB = 5; CALL; } break;                                                        \
            case 6: { constexpr int NB = 6; CALL; } break;                                                        \
            case 7: { constexpr int NB = 7; CALL; } break;                                                        \
            default: { constexpr int NB = 8; CALL; } break;                                                       \
        }                                                                                                         \
    }
template <int TILE_N, bool ROWS, bool SMALL, int EPI_WARPS>
__device__ __forceinline__ void pipe_epilogue_packed_g(const ConvParams& p, uint32_t tmem_acc, int vwarp, int gp, bool pvalid, int co0,
                                                       uint32_t out_rows) {
    EBS_PIPE_EACH_NB((pipe_epilogue_packed_nb<TILE_N, ROWS, SMALL, EPI_WARPS, NB>(p, tmem_acc, vwarp, gp, pvalid, co0, out_rows)))
}

template <int TILE_N, bool ROWS, bool VALUES>
__device__ __forceinline__ void pipe_epilogue_terms(const ConvParams& p, const FrameGeom& g, uint32_t tmem_set, int m_sub, int vwarp,
                                                    int f0, int co0, float* terms, const FragRows& rows, uint32_t out_rows) {
    auto run = [&](auto res_tag) {
        constexpr int RES = decltype(res_tag)::value;
        if constexpr (VALUES) pipe_epilogue_terms_nb<TILE_N, false, true, 0, RES>(p, g, tmem_set, m_sub, vwarp, f0, co0, terms, rows, out_rows);
        else EBS_PIPE_EACH_NB((pipe_epilogue_terms_nb<TILE_N, ROWS, false, NB, RES>(p, g, tmem_set, m_sub, vwarp, f0, co0, terms, rows, out_rows)))
    };
    if (p.residual) run(std::integral_constant<int, 1>{});
    else if (p.res_packed) run(std::integral_constant<int, 2>{});
    else run(std::integral_constant<int, 0>{});
}

template <int AB, int TILE_N, bool AFFINE, int FORM, bool PAIR = false, bool SMALL = false>
__global__ void __launch_bounds__(pipe_threads(pipe_epi_warps(TILE_N, AFFINE, FORM, PAIR)), 1) conv_umma_pipe_kernel(const ConvParams p, const PipeGeom g, const __grid_constant__ CUtensorMap words) {
    constexpr int EPI_WARPS = pipe_epi_warps(TILE_N, AFFINE, FORM, PAIR);
    constexpr bool ROWS = FORM == 2;                           // two groups' planes leave together through rows in shared memory
    // PAIR: the two CTAs of a cluster work as one.  Each expands its own 128 * m_sub pixels and holds the weight rows of
    // half the channel tile; the even CTA issues MMAs of M = 256 (cta_group::2) that read both CTAs' shared memory and
    // write both CTAs' tensor memory, so a weight byte is fetched from L2 once per 256 pixels instead of once per 128.
    // The odd CTA's issuing warp only reports to the even CTA when its stages, weight slots and accumulators are ready.
    constexpr int B_ROWS = PAIR ? TILE_N / 2 : TILE_N;
    constexpr int B_TILE_BYTES = B_ROWS * 32;
    static_assert(!PAIR || TILE_N == 256, "a CTA pair works on 256-channel tiles");
    __shared__ __align__(8) uint64_t st_peer[PAIR ? PIPE_MAX_STAGES : 1], bs_peer[PAIR ? PIPE_MAX_BSLOTS : 1], acc_peer[2], b_peer;
    const int crank = PAIR ? (int)(blockIdx.x & 1u) : 0;       // rank in the pair (cluster of 2 along x)
    const int bx = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x, gx = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
    extern __shared__ uint8_t dyn_smem[];
    __shared__ __align__(8) uint64_t st_full[PIPE_MAX_STAGES], st_empty[PIPE_MAX_STAGES], acc_full[2], acc_empty[2], b_full;
    __shared__ __align__(8) uint64_t bs_full[PIPE_MAX_BSLOTS], bs_empty[PIPE_MAX_BSLOTS];   // streamed weight tiles
    __shared__ __align__(8) uint64_t raw_full[PIPE_MAX_RAW], raw_empty[PIPE_MAX_RAW];       // packed words by tensor copies
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ __align__(16) float s_terms[AFFINE ? EPI_WARPS : 1][64];
    __shared__ __align__(128) uint8_t s_rows[AFFINE ? EPI_WARPS : 1][AFFINE ? 1024 : 16];
    __shared__ int s_tap_id[PIPE_MAX_TAPS];             // (in shared memory: indexed at run time by single threads)

    // (the warp number read from lane 0, so that the compiler knows the role branches to be warp-uniform: the issuing warps' waits
    // and addresses then take two thirds of the time)
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    if (tid < PIPE_MAX_TAPS) s_tap_id[tid] = (int)g.tap_id[tid];
    const int NST = g.n_stages, KS = g.ks, KSS = g.kss, NSUB = g.nsub, SP = g.SP, S = g.S;
    const int nchunks = g.nchunks, nwg = g.nwg;
    const bool resident = g.b_resident != 0;
    uint8_t* base = dyn_smem + ((1024u - (smem_u32(dyn_smem) & 1023u)) & 1023u);
    uint8_t* b_res = base;                                               // resident: [CW][tap slots][TILE_N][32]; else the ring of tiles
    uint8_t* stages = base + (resident ? g.b_total_bytes : g.b_slots * g.b_group * B_TILE_BYTES);   // [NST] x [KS][2][SP][16]
    uint8_t* raw = stages + g.n_stages * g.stage_bytes;                  // ring of packed words, then the rows of planes
    const int NBS = g.b_slots, GB = g.b_group;
    // Streamed weights: every CTA of a channel tile reads the same weight tiles, and CTAs that start together would ask
    // the same few L2 slices for the same tile at the same time.  Integer accumulation is exact in any order, so each
    // CTA starts its walk over the word groups at a different one.
    const int wg_rot = resident ? 0 : bx % nwg;
    volatile int* abortp = &abort_flag;
    const unsigned wait_limit = p.wait_limit;

    // work items of this CTA: (pixel super-tile, channel tile)
    const int n_items = resident ? g.n_ptiles : g.n_ptiles * g.n_ctiles;
    const int my_items = (bx < n_items) ? (n_items - 1 - bx) / gx + 1 : 0;
    auto item_of = [&](int it, int& ptile, int& ctile) {
        const int idx = bx + it * gx;
        if (resident) { ptile = idx; ctile = (int)blockIdx.y; }
        else { ptile = idx / g.n_ctiles; ctile = idx - ptile * g.n_ctiles; }
    };

    // Issuing warps: the tensor pipe needs 49, 65 and 129 clocks for an MMA of 64, 128 and 256 channels (operands from shared
    // memory) and one warp can issue that fast, but its waits and addresses between the runs of MMAs cannot hide, so with two
    // or four accumulators per tile two warps share the work, each owning the accumulators of one parity -- MMAs of different warps never touch the same accumulator, so
    // no order between the warps is needed.  One accumulator: one issuing warp.
    const int n_iss = (g.m_sub & 1) == 0 ? PIPE_ISSUERS : 1;
    if (tid == 0) {
        abort_flag = 0;
        for (int s = 0; s < PIPE_MAX_STAGES; ++s) {
            mbar_init(&st_full[s], (PIPE_EXPANDERS / 32) * g.nsub);  // every expander warp arrives once per pass
            mbar_init(&st_empty[s], n_iss);                         // every issuing warp commits its own MMAs
        }
        for (int s = 0; s < PIPE_MAX_BSLOTS; ++s) {
            mbar_init(&bs_full[s], 1);
            mbar_init(&bs_empty[s], n_iss);
        }
        mbar_init(&acc_full[0], n_iss);
        mbar_init(&acc_full[1], n_iss);
        mbar_init(&acc_empty[0], EPI_WARPS);
        mbar_init(&acc_empty[1], EPI_WARPS);
        mbar_init(&b_full, 1);
        for (int s = 0; s < PIPE_MAX_RAW; ++s) {
            mbar_init(&raw_full[s], 1);
            mbar_init(&raw_empty[s], PIPE_EXPANDERS / 32);
        }
        if constexpr (PAIR) {
            for (int s = 0; s < PIPE_MAX_STAGES; ++s) mbar_init(&st_peer[s], 1);
            for (int s = 0; s < PIPE_MAX_BSLOTS; ++s) mbar_init(&bs_peer[s], 1);
            mbar_init(&acc_peer[0], 1);
            mbar_init(&acc_peer[1], 1);
            mbar_init(&b_peer, 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == PIPE_ISSUER_WARP) {
        if constexpr (PAIR) {                                 // the same warp of both CTAs, the same slot address
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_slot)),
                         "r"((uint32_t)g.tmem_cols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_slot)),
                         "r"((uint32_t)g.tmem_cols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if constexpr (PAIR) cluster_sync_all();                   // the other CTA's barriers exist before anything arrives on them
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem_base = tmem_slot;

    // Registers follow the roles (warpgroups of four warps: 0-7 expanders, 8-11 issuers / producer / no role, then the
    // epilogue): each role's branch opens with a setmaxnreg executed by all four warps of its warpgroups, and the
    // assembler allocates each branch for its own count.  With 96 registers in eight epilogue warps the epilogue spilled and its
    // instruction stream lost its parallelism (wide 1x1 layers 15-20% slower); the expanders, whose words wait in shared memory, need 40
    // for up to four planes.  The increase waits in hardware until the CTA's pool has the registers, so the counts must fit
    // into what the launch allots: checked at compile time.  (The middle role spilled at 56, which cost the GEMM a fifth.)
    constexpr bool MANY = EPI_WARPS == 16, WIDE_ITEMS = AB == 0 || AB > 4;
    constexpr int REG_LAUNCH = MANY ? 72 : 96, REG_MID = 64;
    constexpr int REG_EXP = !MANY ? 64 : WIDE_ITEMS ? 48 : 40, REG_EPI = !MANY ? 144 : WIDE_ITEMS ? 80 : 88;
    static_assert(8 * REG_EXP + 4 * REG_MID + EPI_WARPS * REG_EPI <= (PIPE_EPI_WARP0 + EPI_WARPS) * REG_LAUNCH, "setmaxnreg: the roles' registers exceed the CTA's pool");
    static_assert(PIPE_EPI_WARP0 == 12, "role layout changed: revisit the register split");
    if (warp < 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(REG_EXP));
        // =========================== expanders ===========================
        // An even number of words per pass: a thread takes two adjacent words of one pixel, so that for an odd plane count
        // its 2 * AB packed words still start on an 8-byte boundary and load as pairs.  Otherwise items tid and tid + 256.
        constexpr int NW = AB == 0 ? 8 : AB;                  // words of one (pixel, 32-channel word) item; AB = 0: byte codes
        constexpr int UNIT = NW % 4 == 0 ? 16 : NW % 2 == 0 ? 8 : 4, UNITS = NW * 4 / UNIT;
        constexpr uint32_t RAW_PASS = PIPE_MAX_ITEMS * NW * 4;
        const bool paired = (NW & 1) != 0 && (KS & 1) == 0 && (p.CW & 1) == 0;
        int item_pix[PIPE_SLOTS];                             // strip pixel, -1: no item
        uint32_t item_dst[PIPE_SLOTS], item_q[PIPE_SLOTS], item_at[PIPE_SLOTS];   // item_at: its words in a slot of the ring
#pragma unroll
        for (int j = 0; j < PIPE_SLOTS; ++j) {
            const int e = paired ? 2 * tid + j : tid + j * PIPE_EXPANDERS;
            const int s = e / KS, q = e - s * KS;            // consecutive lanes: consecutive words of one pixel
            item_pix[j] = s < S ? s : -1;
            item_q[j] = (uint32_t)q * (NW * 4);
            item_dst[j] = (uint32_t)(q * g.a_word_bytes + s * 16);
            item_at[j] = smem_u32(raw) + (s < S ? (uint32_t)((s * g.raw_words + q) * (NW * 4)) : 0u);
        }
        // Fetching runs RD - 1 passes ahead of the expansion, also across tile boundaries: cp.async brings a thread's own items into
        // its places of the ring, so that no barrier is needed and one loop body serves every pass.  (With the words in flight in
        // registers the body existed once per set, 19 KB of code beside the epilogue's, and 90-140 of a warp's 200 instructions a pass
        // were addresses: 256 -> 64 1x1 at 56x56, batch 256, 4 bits, 72.0 us against 54.5 with this ring; 4096^3 GEMM, packed, 85 and 73.)
        const uint8_t* src[PIPE_SLOTS];                       // words of the item's pixel, at its word position
        uint32_t lim[PIPE_SLOTS];                             // bytes of a pixel's words from there on; 0: no pixel (padding, past the batch), zero bytes
        int ld_it = 0, ld_ph = 0, ld_left = 0;
        const uint32_t px_bytes = (uint32_t)p.CW * (NW * 4), step = (uint32_t)KS * (NW * 4), wrap = (uint32_t)(nwg * KSS) * (NW * 4);
        const uint32_t first = (uint32_t)(wg_rot * KSS) * (NW * 4);
        uint32_t ld_off = first;
        uint32_t raw_w = 0, raw_r = 0;
        auto locate = [&]() {
            int ptile, ctile;
            item_of(ld_it, ptile, ctile);
            const int f0 = (PAIR ? 2 * ptile + crank : ptile) * g.tile_pix;
            const int dh = p.sh * g.q0r + g.ph_a[ld_ph], dw = p.sw * g.q0s + g.ph_b[ld_ph];
#pragma unroll
            for (int j = 0; j < PIPE_SLOTS; ++j) {
                const uint32_t f = (uint32_t)(f0 + item_pix[j]);
                bool in = item_pix[j] >= 0 && (int)f < g.frame;
                uint32_t pix = f;
                if (!g.linear_in) {
                    const uint32_t n = fastdiv(f, g.div_img), rem = f - n * (uint32_t)(g.Hq * g.Wq);
                    const uint32_t hq = fastdiv(rem, g.div_row), wq = rem - hq * (uint32_t)g.Wq;
                    const int h = p.sh * (int)hq + dh, w = p.sw * (int)wq + dw;
                    in = in && (unsigned)h < (unsigned)p.H && (unsigned)w < (unsigned)p.W;
                    pix = (n * p.H + h) * p.W + w;
                }
                src[j] = reinterpret_cast<const uint8_t*>(p.x) + item_q[j];
                if (in) src[j] += (size_t)pix * px_bytes;
                lim[j] = in ? px_bytes - item_q[j] : 0u;
            }
            ld_left = nwg * NSUB;
            ld_off = first;
            if (++ld_ph == g.n_ph) { ld_ph = 0; ++ld_it; }
        };
        auto fetch = [&](uint32_t raw_last, uint32_t raw_pass) {
            if (ld_left == 0) locate();
            --ld_left;
#pragma unroll
            for (int j = 0; j < PIPE_SLOTS; ++j) {
                if (paired && j > 0) break;
                if (item_pix[j] < 0) continue;
                const uint8_t* a = src[j] + ld_off;
                bool real = ld_off < lim[j];                  // (a ragged last group: words past the pixel's, which feed no MMA)
                if (real && !EBS_IN_RANGE(p, CHK_PIPE_X, (reinterpret_cast<const uint32_t*>(a) - p.x) + (paired ? 2 : 1) * NW - 1, p.lim_x)) real = false;
                if (paired) {
#pragma unroll
                    for (int u = 0; u < NW; ++u)
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(item_at[j] + raw_w + 8 * u), "l"(a + 8 * u), "r"(real ? 8 : 0) : "memory");
                } else {
#pragma unroll
                    for (int u = 0; u < UNITS; ++u) {
                        const uint32_t dst = item_at[j] + raw_w + (uint32_t)(u * UNIT);
                        if constexpr (UNIT == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(a + 16 * u), "r"(real ? 16 : 0) : "memory");
                        else asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(dst), "l"(a + UNIT * u), "n"(UNIT), "r"(real ? UNIT : 0) : "memory");
                    }
                }
            }
            raw_w = raw_w == raw_last ? 0u : raw_w + raw_pass;
            ld_off += step;
            if (ld_off == wrap) ld_off = 0;
        };
        const int total = my_items * nchunks * NSUB;           // expander passes
        const uint32_t st0 = smem_u32(stages), pass_bytes = (uint32_t)(KS * g.a_word_bytes);
        uint32_t at = st0, full = smem_u32(&st_full[0]);
        const uint32_t half = (uint32_t)SP * 16;
        const int parts = g.raw_words / KS;                    // passes of a slot
        int st = 0, sub = 0, part = 0, slot = 0;
        uint32_t raw_par = 0u;
        uint32_t par = 1u;                                      // (a fresh barrier lets a wait for the phase before its first pass)
        // (a loop each for tensor copies, the full ring and two slots: the fetching chosen at run time cost 3 us of 54, the ring's size and
        // depth in registers up to 6% of strided layers: 128 -> 128 3x3 at 56x56, batch 256, 1 plane 46.8 and 49.8)
        auto passes = [&](auto form) {
            constexpr bool TMA = decltype(form)::value == 0, FULL = decltype(form)::value == 1;
            constexpr int RD = FULL ? pipe_raw_depth(NW) : 2;   // passes in the ring
            const uint32_t raw_pass = FULL ? RAW_PASS : (uint32_t)g.raw_slot_bytes, raw_last = (RD - 1) * raw_pass;
#pragma unroll 1
            for (int gi = TMA ? 0 : 1 - RD; gi < total; ++gi) {
                if constexpr (!TMA) {
                    if (gi + RD - 1 < total) fetch(raw_last, raw_pass);
                    asm volatile("cp.async.commit_group;\n" ::: "memory");
                    if (gi < 0) continue;
                }
                if (sub == 0) {                                     // the MMAs that read this stage one round ago must be done
                    if (!mbar_wait_bounded(&st_empty[st], par, abortp, wait_limit)) break;
                }
                if constexpr (!TMA) {
                    asm volatile("cp.async.wait_group %0;\n" ::"n"(RD - 1) : "memory");
                } else if (part == 0) {
                    if (!mbar_wait_bounded(&raw_full[slot], raw_par, abortp, wait_limit)) break;
                }
                uint32_t w[PIPE_SLOTS][NW];
#pragma unroll
                for (int j = 0; j < PIPE_SLOTS; ++j)
#pragma unroll
                    for (int u = 0; u < UNITS; ++u) {
                        const uint32_t a = item_at[j] + raw_r + (uint32_t)(u * UNIT);
                        if constexpr (UNIT == 16) asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(w[j][4 * u]), "=r"(w[j][4 * u + 1]), "=r"(w[j][4 * u + 2]), "=r"(w[j][4 * u + 3]) : "r"(a) : "memory");
                        else if constexpr (UNIT == 8) asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];\n" : "=r"(w[j][2 * u]), "=r"(w[j][2 * u + 1]) : "r"(a) : "memory");
                        else asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(w[j][u]) : "r"(a) : "memory");
                    }
                if constexpr (!TMA) {
                    raw_r = raw_r == raw_last ? 0u : raw_r + raw_pass;
                }
#pragma unroll
                for (int j = 0; j < PIPE_SLOTS; ++j) {
                    if (item_pix[j] < 0) continue;
                    uint32_t r[8];
                    if constexpr (AB == 0) {
                        // byte codes, channel c in byte c of the item: only the order changes (row byte 4b + i = channel 8i + b, the
                        // order of the weight image): register b takes byte b % 4 of words b / 4, 2 + b / 4, ...
#pragma unroll
                        for (int bb = 0; bb < 8; ++bb) {
                            const uint32_t sel = 0x0040u + 0x11u * (uint32_t)(bb & 3);          // byte (bb & 3) of both operands
                            const uint32_t lo = __byte_perm(w[j][bb >> 2], w[j][2 + (bb >> 2)], sel);
                            const uint32_t hi = __byte_perm(w[j][4 + (bb >> 2)], w[j][6 + (bb >> 2)], sel);
                            r[bb] = __byte_perm(lo, hi, 0x5410);
                        }
                    } else {
                        planes_to_bytes<NW>(w[j], r);
                    }
                    const uint32_t dst = at + item_dst[j];
                    if (!EBS_IN_RANGE(p, CHK_PIPE_STAGE, (long long)(dst + half + 15u) - st0, NST * g.stage_bytes) ||
                        !EBS_IN_RANGE(p, CHK_PIPE_STAGE, (long long)dst - st0, NST * g.stage_bytes))
                        continue;
                    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n" ::"r"(dst), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
                    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n" ::"r"(dst + half), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
                }
                // every lane makes its bytes visible to the tensor core's proxy, then one lane arrives for the warp (32 arrivals on one
                // barrier word would be served one after the other)
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                __syncwarp();
                if ((tid & 31) == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(full) : "memory");
                if constexpr (TMA) {
                    raw_r += step;
                    if (++part == parts) {                          // this warp has used its words of the slot: only here, so that the next
                        part = 0;                                   // copy cannot overtake loads that are still under way
                        if ((tid & 31) == 0) mbar_arrive(&raw_empty[slot]);
                        if (++slot == g.raw_slots) { slot = 0; raw_par ^= 1u; }
                        raw_r = (uint32_t)(slot * g.raw_slot_bytes);
                    }
                }
                at += pass_bytes;
                if (++sub == NSUB) {
                    sub = 0;
                    full += 8u;
                    if (++st == NST) { st = 0; par ^= 1u; full = smem_u32(&st_full[0]); }
                    at = st0 + (uint32_t)(st * g.stage_bytes);
                }
            }
        };
        if (NW >= 3 && NW != 4 && NW != 8 && g.tma) passes(std::integral_constant<int, 0>{});
        else if (g.ring_full) passes(std::integral_constant<int, 1>{});
        else passes(std::integral_constant<int, 2>{});
        asm volatile("cp.async.wait_all;\n" ::: "memory");
    } else if (warp < PIPE_EPI_WARP0) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(REG_MID));
      if (PAIR && crank == 1 && warp < PIPE_PRODUCER_WARP) {
        // =========================== the odd CTA of a pair: reports ===========================
        // One warp follows this CTA's own barriers in the order the even CTA's issuing warps wait for them and passes
        // each completion on with one arrival on the even CTA's barrier of the same name.
        if (warp == PIPE_ISSUER_WARP) {
            const bool lane0 = (tid & 31) == 0;
            const uint32_t r_st = cluster_addr(&st_peer[0], 0), r_bs = cluster_addr(&bs_peer[0], 0);
            const uint32_t r_acc = cluster_addr(&acc_peer[0], 0), r_b = cluster_addr(&b_peer, 0);
            bool ok = true;
            if (my_items > 0 && resident) {
                ok = mbar_wait_bounded_warp(&b_full, 0u, abortp, wait_limit);
                if (ok && lane0) mbar_arrive_cluster(r_b);
            }
            int st = 0, bs = 0;
            uint32_t st_round = 0, bs_round = 0;
            for (int it = 0; it < my_items && ok; ++it) {
                const int buf = g.nbuf == 2 ? (it & 1) : 0;
                const int use = g.nbuf == 2 ? (it >> 1) : it;
                if (use > 0) {
                    if (!mbar_wait_bounded_warp(&acc_empty[buf], (uint32_t)((use - 1) & 1), abortp, wait_limit)) break;
                    if (lane0) mbar_arrive_cluster(r_acc + 8u * (uint32_t)buf);
                }
                int ph = 0, wg = 0;
                for (int c = 0; c < nchunks && ok; ++c) {
                    if (!mbar_wait_bounded_warp(&st_full[st], st_round & 1u, abortp, wait_limit)) { ok = false; break; }
                    if (lane0) mbar_arrive_cluster(r_st + 8u * (uint32_t)st);
                    if (!resident) {
                        const int wgr = wg + wg_rot >= nwg ? wg + wg_rot - nwg : wg + wg_rot;
                        const int words = min(KSS, p.CW - wgr * KSS);
                        const int rows = g.ph_rows[ph], cols = g.ph_cols[ph];
                        const PipeSlot sl = g.slot[ph];
                        for (int q = 0, r = 0, s = 0; q < words;) {
                            if ((s += sl.cols) >= cols) { s = 0; if ((r += sl.rows) >= rows) { r = 0; q += sl.words; } }
                            if (!mbar_wait_bounded_warp(&bs_full[bs], bs_round & 1u, abortp, wait_limit)) { ok = false; break; }
                            if (lane0) mbar_arrive_cluster(r_bs + 8u * (uint32_t)bs);
                            if (++bs == NBS) { bs = 0; ++bs_round; }
                        }
                    }
                    __syncwarp();
                    if (++st == NST) { st = 0; ++st_round; }
                    if (++wg == nwg) { wg = 0; ++ph; }
                }
            }
        }
      } else if (warp >= PIPE_ISSUER_WARP && warp < PIPE_ISSUER_WARP + n_iss) {
        // =========================== issuers ===========================
        const int k_iss = warp - PIPE_ISSUER_WARP;                // this warp owns the accumulators k_iss, k_iss + n_iss, ...
        // The issuing thread is a pipeline stage of its own: every address is advanced by additions (descriptor start
        // addresses are in 16-byte units), a handful of instructions per MMA.
        constexpr uint32_t IDESC = PAIR ? (umma_idesc_i8(TILE_N) & ~(0x1Fu << 24)) | ((256u >> 4) << 24) : umma_idesc_i8(TILE_N);
        constexpr uint32_t BT16 = B_TILE_BYTES >> 4;
        const bool skip_mma = (p.test_flags & 1) != 0;            // test hook: issue nothing, so that waits run out
        bool ok = my_items == 0 || !resident || mbar_wait_bounded_warp(&b_full, 0u, abortp, wait_limit);
        if (PAIR && ok && my_items > 0 && resident) ok = mbar_wait_cluster_warp(&b_peer, 0u, abortp, wait_limit);
        const uint64_t da_ring = umma_desc_interleaved(smem_u32(stages), (uint32_t)(SP * 16));
        const uint64_t db_res = umma_desc_sw32(smem_u32(b_res));   // resident tiles, or slot 0 of the ring
        const uint32_t da_lo = (uint32_t)da_ring, da_hi = (uint32_t)(da_ring >> 32);
        const uint32_t db_lo = (uint32_t)db_res, db_hi = (uint32_t)(db_res >> 32);
        const uint32_t stage16 = (uint32_t)(g.stage_bytes >> 4), word16 = (uint32_t)(g.a_word_bytes >> 4);
        const int m_sub = g.m_sub, my_acc = m_sub / n_iss;        // accumulators k_iss, k_iss + n_iss, ... of a tile
        const uint32_t a_first = (uint32_t)(uni(k_iss) * UMMA_M), a_step = (uint32_t)(n_iss * UMMA_M);
        const uint32_t d_first = (uint32_t)(uni(k_iss) * TILE_N), d_step = (uint32_t)(n_iss * TILE_N), b_first = uni(db_lo);
        const uint32_t leader = elect_one() ? 1u : 0u;
        // `steps` rows of `cols` taps (or `steps` words of a 1 x 1 layer), into every accumulator of this warp: straight-line
        // code for the tap rows and accumulator counts that occur, run by one elected lane.  (Behind a test of the lane number
        // instead of elect.sync every MMA moves its operands to uniform registers on its own: 64 -> 64 3x3 at 56x56, batch 256
        // takes 75 us instead of 62.)
        auto issue_n = [&](auto cols_tag, auto acc_tag, int steps, uint32_t d0, uint32_t a, uint32_t a_inc, uint32_t b, uint32_t b_inc,
                           uint32_t accu) {
            constexpr int COLS = decltype(cols_tag)::value, ACC = decltype(acc_tag)::value;
            if (elect_one()) {
#pragma unroll 1
                for (int i = 0; i < steps; ++i, a += a_inc, b += b_inc) {
#pragma unroll
                    for (int s = 0; s < COLS; ++s) {
#pragma unroll
                        for (int j = 0; j < ACC; ++j) {
                            const uint32_t d = d0 + (uint32_t)j * d_step, al = a + (uint32_t)s + (uint32_t)j * a_step, bl = b + (uint32_t)s * BT16;
                            if constexpr (PAIR) umma_i8_split_pair(1u, d, al, da_hi, bl, db_hi, IDESC, s > 0 ? 1u : accu);
                            else umma_i8_split(1u, d, al, da_hi, bl, db_hi, IDESC, s > 0 ? 1u : accu);
                        }
                    }
                    accu = 1u;
                }
            }
            __syncwarp();
        };
        auto issue = [&](int steps, int cols, uint32_t d0, uint32_t a, uint32_t a_inc, uint32_t b, uint32_t b_inc, uint32_t accu) {
            auto with = [&](auto acc_tag) {
                if (cols == 1) issue_n(std::integral_constant<int, 1>{}, acc_tag, steps, d0, a, a_inc, b, b_inc, accu);
                else if (cols == 2) issue_n(std::integral_constant<int, 2>{}, acc_tag, steps, d0, a, a_inc, b, b_inc, accu);
                else if (cols == 3) issue_n(std::integral_constant<int, 3>{}, acc_tag, steps, d0, a, a_inc, b, b_inc, accu);
                else for (int i = 0; i < steps; ++i, accu = 1u)
                    issue_n(std::integral_constant<int, 1>{}, acc_tag, cols, d0, a + (uint32_t)i * a_inc, 1u, b + (uint32_t)i * b_inc, BT16, accu);
            };
            if (my_acc == 1) with(std::integral_constant<int, 1>{});
            else with(std::integral_constant<int, 2>{});
        };
        // (a pair: the odd CTA's shared window lies at a fixed distance from this one's in the cluster window)
        const uint32_t peer_delta = PAIR ? cluster_addr(&abort_flag, 1) - smem_u32(&abort_flag) : 0u;
        auto mma_commit = [peer_delta](uint32_t ld, uint64_t* bar) {
            if constexpr (PAIR) umma_commit_pred_pair(ld, bar, peer_delta);
            else umma_commit_pred(ld, bar);
        };
        int st = 0, bs = 0;
        uint32_t st_round = 0, bs_round = 0;
        for (int it = 0; it < my_items && ok; ++it) {
            const int buf = g.nbuf == 2 ? (it & 1) : 0;
            const int use = g.nbuf == 2 ? (it >> 1) : it;          // how often this accumulator set was used before
            if (use > 0) {                                          // its epilogue must have drained it
                if (!mbar_wait_bounded_warp(&acc_empty[buf], (uint32_t)((use - 1) & 1), abortp, wait_limit)) break;
                if (PAIR && !mbar_wait_cluster_warp(&acc_peer[buf], (uint32_t)((use - 1) & 1), abortp, wait_limit)) break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint32_t tmem_d = tmem_base + (uint32_t)(buf * m_sub * TILE_N);
            int ph = 0, wg = 0;
            for (int c = 0; c < nchunks; ++c) {
                if (!mbar_wait_bounded_warp(&st_full[st], st_round & 1u, abortp, wait_limit)) { ok = false; break; }
                if (PAIR && !mbar_wait_cluster_warp(&st_peer[st], st_round & 1u, abortp, wait_limit)) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                if (!skip_mma) {
                    const int wgr = uni(wg + wg_rot >= nwg ? wg + wg_rot - nwg : wg + wg_rot);
                    const int words = min(KSS, p.CW - wgr * KSS), rows = uni(g.ph_rows[ph]), cols = uni(g.ph_cols[ph]);
                    const uint32_t a0 = uni(da_lo + (uint32_t)st * stage16 + (uint32_t)g.ph_shift[ph]) + a_first;
                    const uint32_t d0 = uni(tmem_d) + d_first;
                    uint32_t accu = c == 0 ? 0u : 1u;              // the first MMA into each accumulator of a tile overwrites it
                    if (resident) {
                        const uint32_t b0 = b_first + (uint32_t)((wgr * KSS) * g.taps + uni(g.ph_tap0[ph])) * BT16;
                        if (rows * cols == 1) {
                            issue(words, 1, d0, a0, word16, b0, (uint32_t)g.taps * BT16, accu);
                        } else {
                            for (int q = 0; q < words; ++q, accu = 1u)
                                issue(rows, cols, d0, a0 + (uint32_t)q * word16, (uint32_t)g.Wq, b0 + (uint32_t)(q * g.taps) * BT16,
                                      (uint32_t)cols * BT16, accu);
                        }
                    } else {
                        // streamed weights, slot by slot
                        const PipeSlot sl = g.slot[ph];
                        for (int q = 0; q < words && ok; q += sl.words) {
                            for (int r = 0; r < rows && ok; r += sl.rows) {
                                for (int s = 0; s < cols; s += sl.cols) {
                                    if (!mbar_wait_bounded_warp(&bs_full[bs], bs_round & 1u, abortp, wait_limit)) { ok = false; break; }
                                    if (PAIR && !mbar_wait_cluster_warp(&bs_peer[bs], bs_round & 1u, abortp, wait_limit)) { ok = false; break; }
                                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                                    const int nq = min(sl.words, words - q), nr = min(sl.rows, rows - r), ns = min(sl.cols, cols - s);
                                    uint32_t b_lo = uni(db_lo + (uint32_t)(bs * GB) * BT16), a_lo = a0 + (uint32_t)q * word16 + (uint32_t)(r * g.Wq + s);
                                    if (rows * cols == 1) {
                                        issue(nq, 1, d0, a_lo, word16, b_lo, BT16, accu);
                                    } else {
                                        for (int i = 0; i < nq; ++i, a_lo += word16, b_lo += (uint32_t)(nr * ns) * BT16, accu = 1u)
                                            issue(nr, ns, d0, a_lo, (uint32_t)g.Wq, b_lo, (uint32_t)ns * BT16, accu);
                                    }
                                    accu = 1u;
                                    mma_commit(leader, &bs_empty[bs]);
                                    if (++bs == NBS) { bs = 0; ++bs_round; }
                                }
                            }
                        }
                        if (!ok) break;
                    }
                    mma_commit(leader, &st_empty[st]);
                    if (c == nchunks - 1) mma_commit(leader, &acc_full[buf]);
                }
                __syncwarp();
                if (++st == NST) { st = 0; ++st_round; }
                if (++wg == nwg) { wg = 0; ++ph; }
            }
        }
    } else if (warp == PIPE_PRODUCER_WARP) {
        // =========================== weight tiles ===========================
        // The whole warp runs the loops with uniform control flow and every lane issues the copy of one tile of a slot
        // (its own address arithmetic, side by side with the other lanes'): a single lane working through the tiles one
        // after the other retired an instruction every dozen clocks and needed about 360 clocks per tile -- more than
        // the two MMAs that consume a 256-channel tile -- which bounded every layer whose weights stream.
        const int lane = tid & 31;
        if (my_items > 0) {
            if (resident) {                                      // all tiles of this CTA's channel tile, once
                const int co0 = (int)blockIdx.y * TILE_N + crank * B_ROWS;   // a pair: this CTA's half of the channel tile
                const uint32_t rows = (uint32_t)min(B_ROWS, p.Co16 - co0);
                const int total_tiles = p.CW * g.taps;
                if (lane == 0) mbar_arrive_expect_tx(&b_full, rows * 32u * (uint32_t)total_tiles);
                __syncwarp();
                for (int t = lane; t < total_tiles; t += 32) {
                    const int cw = t / g.taps, ts = t - cw * g.taps;
                    if (EBS_IN_RANGE(p, CHK_PIPE_W8, ((long long)(s_tap_id[ts] * p.CW + cw) * p.Co16 + co0) * 32 + rows * 32 - 1, p.lim_w8))
                        bulk_copy_g2s(b_res + t * B_TILE_BYTES,
                                      p.w8 + ((size_t)(s_tap_id[ts] * p.CW + cw) * p.Co16 + co0) * 32, rows * 32u, &b_full);
                }
            } else {
                int bs = 0;
                uint32_t bs_round = 0;
                bool ok = true;
                for (int it = 0; it < my_items && ok; ++it) {
                    int ptile, ctile;
                    item_of(it, ptile, ctile);
                    const int co0 = ctile * TILE_N + crank * B_ROWS;
                    const uint32_t bytes = (uint32_t)min(B_ROWS, p.Co16 - co0) * 32u;
                    int ph = 0, wg = -1;
                    for (int c = 0; c < nchunks && ok; ++c) {
                        if (++wg == nwg) { wg = 0; ++ph; }
                        const int wgr = wg + wg_rot >= nwg ? wg + wg_rot - nwg : wg + wg_rot;
                        const int words = min(KSS, p.CW - wgr * KSS);
                        const int rows = g.ph_rows[ph], cols = g.ph_cols[ph], t0 = g.ph_tap0[ph];
                        const PipeSlot sl = g.slot[ph];
                        int q0 = 0, r0 = 0, s0 = 0;
                        while (q0 < words) {
                            if (bs_round > 0) {                     // the MMAs that read this slot one round ago must be done
                                const bool free = mbar_wait_bounded_hot(&bs_empty[bs], (bs_round - 1) & 1u, abortp, wait_limit);
                                if (!__all_sync(0xffffffffu, free)) { ok = false; break; }
                            }
                            const int nr = min(sl.rows, rows - r0), ns = min(sl.cols, cols - s0), n = min(sl.words, words - q0) * nr * ns;
                            if (lane == 0) mbar_arrive_expect_tx(&bs_full[bs], bytes * (uint32_t)n);
                            __syncwarp();
                            if (lane < n) {                          // tile of the slot: word-major, rows, taps of a row
                                const int per = nr * ns, w = per == 1 ? lane : lane / per, t = lane - w * per, rr = nr == 1 ? 0 : t / ns;
                                const int q = q0 + w, ts = t0 + (r0 + rr) * cols + s0 + (t - rr * ns);
                                const size_t src = ((size_t)(s_tap_id[ts] * p.CW + wgr * KSS + q) * p.Co16 + co0) * 32;
                                // (a copy skipped by the range-checked build leaves its barrier incomplete: the CTA then gives
                                // up at its bounded wait, which is reported as well)
                                if (EBS_IN_RANGE(p, CHK_PIPE_W8, src + bytes - 1, p.lim_w8))
                                    bulk_copy_g2s(b_res + (bs * GB + lane) * B_TILE_BYTES, p.w8 + src, bytes, &bs_full[bs]);
                            }
                            if (++bs == NBS) { bs = 0; ++bs_round; }
                            if ((s0 += sl.cols) >= cols) { s0 = 0; if ((r0 += sl.rows) >= rows) { r0 = 0; q0 += sl.words; } }
                        }
                    }
                }
            }
        }
      } else if (warp == PIPE_FETCH_WARP && g.tma) {
        // =========================== packed words by tensor copies ===========================
        const int per_stage = KSS / g.raw_words, slot_words = g.raw_words * p.x_words, rows = min(g.tile_pix, 256);
        const uint32_t leader = elect_one() ? 1u : 0u;
        int slot = 0;
        uint32_t par = 1u;
        bool ok = true;
        for (int it = 0; it < my_items && ok; ++it) {
            int ptile, ctile;
            item_of(it, ptile, ctile);
            for (int wg = 0; wg < nwg && ok; ++wg) {
                const int wgr = wg + wg_rot >= nwg ? wg + wg_rot - nwg : wg + wg_rot;
                for (int i = 0; i < per_stage; ++i) {
                    if (!mbar_wait_bounded_warp(&raw_empty[slot], par, abortp, wait_limit)) { ok = false; break; }
                    if (leader) {
                        mbar_arrive_expect_tx(&raw_full[slot], (uint32_t)g.raw_slot_bytes);
                        for (int y = 0; y < g.tile_pix; y += rows)
                            asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(
                                             smem_u32(raw) + (uint32_t)(slot * g.raw_slot_bytes + y * slot_words * 4)),
                                         "l"(reinterpret_cast<uint64_t>(&words)), "r"((wgr * per_stage + i) * slot_words), "r"(ptile * g.tile_pix + y),
                                         "r"(smem_u32(&raw_full[slot])) : "memory");
                    }
                    __syncwarp();
                    if (++slot == g.raw_slots) { slot = 0; par ^= 1u; }
                }
            }
        }
      }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(REG_EPI));
        // =========================== epilogue ===========================
        const int half = (warp - PIPE_EPI_WARP0) >> 2;           // which share of the channels
        const int vwarp = (warp & 3) + 4 * half;                 // TMEM lane quarter = warp % 4 (hardware rule), share of the channels
        const int row = (warp & 3) * 32 + (tid & 31);
        const uint32_t out_rows = smem_u32(raw) + (uint32_t)g.raw_bytes + (uint32_t)((warp - PIPE_EPI_WARP0) * 256 * p.next_bits);   // (form 2)
        const bool plain_ok = !AFFINE && !p.ch_scale && !p.ch_bias && !p.residual && !p.res_packed && !p.y_nchw &&
                              (p.Co & 31) == 0;
        // layers with per-channel terms or a shortcut and without integer output (the layers of a network)
        const bool affine_ok = AFFINE && !p.acc && !p.y_nchw && (p.Co & 31) == 0 && !(p.residual && p.res_packed);
        for (int it = 0; it < my_items; ++it) {
            const int buf = g.nbuf == 2 ? (it & 1) : 0;
            const int use = g.nbuf == 2 ? (it >> 1) : it;
            if (!mbar_wait_bounded(&acc_full[buf], (uint32_t)(use & 1), abortp, wait_limit)) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            int ptile, ctile;
            item_of(it, ptile, ctile);
            const int co0 = ctile * TILE_N;
            if (AFFINE && (FORM != 0 || affine_ok)) {
                if constexpr (AFFINE)
                    pipe_epilogue_terms<TILE_N, ROWS, FORM == 0>(p, g, tmem_base + (uint32_t)(buf * g.m_sub * TILE_N), g.m_sub, vwarp,
                                                                  (PAIR ? 2 * ptile + crank : ptile) * g.tile_pix + row, co0,
                                                                  s_terms[warp - PIPE_EPI_WARP0], FragRows(smem_u32(s_rows[warp - PIPE_EPI_WARP0])), out_rows);
            } else for (int j = 0; j < g.m_sub; ++j) {
                const int f = (PAIR ? 2 * ptile + crank : ptile) * g.tile_pix + j * UMMA_M + row;
                bool pvalid = false;
                int gp = 0;
                if (g.linear_out) {
                    pvalid = f < g.frame;
                    gp = pvalid ? f : 0;
                } else if (f < g.frame) {
                    const uint32_t n = fastdiv((uint32_t)f, g.div_img);
                    const uint32_t rem = (uint32_t)f - n * (uint32_t)(g.Hq * g.Wq);
                    const uint32_t hq = fastdiv(rem, g.div_row), wq = rem - hq * (uint32_t)g.Wq;
                    pvalid = (int)hq < p.Ho && (int)wq < p.Wo;
                    gp = ((int)n * p.Ho + (int)hq) * p.Wo + (int)wq;
                }
                if (!__any_sync(0xffffffffu, pvalid)) continue;   // 32 frame pixels without an output
                const uint32_t tmem_acc = tmem_base + (uint32_t)((buf * g.m_sub + j) * TILE_N);
                if constexpr (FORM != 0) {
                    if constexpr (!AFFINE) pipe_epilogue_packed_g<TILE_N, ROWS, SMALL, EPI_WARPS>(p, tmem_acc, vwarp, gp, pvalid, co0, out_rows);
                } else {
                    if (plain_ok) pipe_epilogue_plain<TILE_N>(p, tmem_acc, vwarp, gp, pvalid, co0);
                    else umma_epilogue<TILE_N, AFFINE>(p, tmem_acc, vwarp, gp, pvalid, 0, co0);
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncwarp();
            if ((tid & 31) == 0) mbar_arrive(&acc_empty[buf]);
        }
    }

    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if constexpr (PAIR) {
        if (abort_flag != 0) giveup_drain();
        __syncwarp();
        cluster_sync_all();                                   // neither CTA leaves while the other may still arrive on its barriers
    }
    if (warp == PIPE_ISSUER_WARP) {                           // (the block's memory is its own until this warp leaves)
        if (abort_flag != 0) {
            giveup_drain();
            if ((tid & 31) == 0) atomicAdd(&g_umma_timeouts, 1ull);
        }
        __syncwarp();
        if constexpr (PAIR)
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"((uint32_t)g.tmem_cols)
                         : "memory");
        else
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"((uint32_t)g.tmem_cols)
                         : "memory");
    }
}

int pipe_sm_count();

// Tensor map of the packed words of all pixels, for boxes of one slot of the ring.  False: the driver has none, or refused it.
bool pipe_words_map(const ConvParams& p, const PipeGeom& g, CUtensorMap* map);

template <int AB, int TILE_N, int FORM, bool AFFINE, bool SMALL>
int launch_conv_umma_pipe_kernel(const ConvParams& p, const PipeGeom& g, const CUtensorMap& words, cudaStream_t st) {
    auto kern = conv_umma_pipe_kernel<AB, TILE_N, AFFINE, FORM, false, SMALL>;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, PIPE_SMEM_MAX - (AFFINE ? PIPE_SMEM_TERMS : 0));
        attr_set[dev] = true;
    }
    kern<<<dim3((unsigned)g.grid_x, (unsigned)g.grid_y, 1), pipe_threads(pipe_epi_warps(TILE_N, AFFINE, FORM, false)), g.smem_bytes, st>>>(p, g, words);
    return EBS_OK;
}

// Accumulators below 2^23 in a layer without per-channel terms need no conversion to fp32: the integer a, read as fp32, is the
// denormal a * 2^-149, its product with S * 2^75 is rounded as that of float(a) with S and scaled by 2^-74, and 1 / step carries the
// 2^74 back.  A negative one reads as a NaN or a negative value and becomes code 0, which any negative value does.  One of seven
// instructions an output (64 -> 256 1x1 at 56x56, batch 256, 4 planes: 78.1 -> 74.0 us; 64 -> 64 3x3: 47.3 -> 46.1).
inline bool pipe_small_accumulators(const ConvParams& p) {
    auto moderate = [](float v) { return v >= 0x1p-50f && v <= 0x1p+50f; };
    return p.acc_bound < (1LL << 23) && moderate(p.S) && moderate(p.inv_next);
}

template <int AB, int TILE_N, int FORM>
int launch_conv_umma_pipe_form(const ConvParams& p, const PipeGeom& g, const CUtensorMap& words, cudaStream_t st) {
    if (pipe_has_terms(p)) return launch_conv_umma_pipe_kernel<AB, TILE_N, FORM, true, false>(p, g, words, st);
    if constexpr (FORM != 0) {
        if (pipe_small_accumulators(p)) {
            ConvParams q = p;
            q.S = ldexpf(p.S, 75);
            q.inv_next = ldexpf(p.inv_next, 74);
            return launch_conv_umma_pipe_kernel<AB, TILE_N, FORM, false, true>(q, g, words, st);
        }
    }
    return launch_conv_umma_pipe_kernel<AB, TILE_N, FORM, false, false>(p, g, words, st);
}

// The CTA-pair form: clusters of two CTAs along x; packed-only whole tiles (form 1) or every output mode (form 0),
// no per-channel terms.
template <int AB, int FORM>
int launch_conv_umma_pipe_pair_form(const ConvParams& p, const PipeGeom& g, cudaStream_t st) {
    static bool attr_set[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    auto kern = conv_umma_pipe_kernel<AB, 256, false, FORM, true>;
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, PIPE_SMEM_MAX);
        attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)g.grid_x, (unsigned)g.grid_y, 1);
    cfg.blockDim = dim3(PIPE_THREADS, 1, 1);
    cfg.dynamicSmemBytes = (size_t)g.smem_bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, p, g, CUtensorMap{}) == cudaSuccess ? EBS_OK : EBS_ERR_CUDA;
}

inline bool pipe_pair_request_ok(const ConvParams& p) {
    return !p.ch_scale && !p.ch_bias && !p.residual && !p.res_packed && !p.w_levels && (p.Co % 256) == 0;
}

template <int AB>
int launch_conv_umma_pipe_pair(const ConvParams& p, dim3 /*grid*/, cudaStream_t st) {
    if (!pipe_pair_request_ok(p)) return EBS_ERR_UNSUPPORTED;
    const PipeGeom g = pipe_geometry(p, 256, pipe_sm_count(), p.pipe_m_sub, true);
    if (!g.ok) return EBS_ERR_UNSUPPORTED;
    if (pipe_packed_only(p)) return launch_conv_umma_pipe_pair_form<AB, 1>(p, g, st);
    return launch_conv_umma_pipe_pair_form<AB, 0>(p, g, st);
}

template <int AB, int TILE_N>
int launch_conv_umma_pipe(const ConvParams& p, dim3 /*grid*/, cudaStream_t st) {
    PipeGeom g = pipe_geometry(p, TILE_N, pipe_sm_count(), p.pipe_m_sub);
    if (!g.ok) return EBS_ERR_UNSUPPORTED;                    // the geometry does not apply: nothing is launched
    CUtensorMap words{};
    if (g.tma && !pipe_words_map(p, g, &words)) g = pipe_geometry(p, TILE_N, pipe_sm_count(), p.pipe_m_sub, false, false);   // by cp.async
    if (pipe_packed_only(p)) {
        if constexpr (TILE_N >= 128) {
            if (pipe_rows_apply(p, TILE_N)) return launch_conv_umma_pipe_form<AB, TILE_N, 2>(p, g, words, st);
        }
        return launch_conv_umma_pipe_form<AB, TILE_N, 1>(p, g, words, st);
    }
    return launch_conv_umma_pipe_form<AB, TILE_N, 0>(p, g, words, st);
}

constexpr int NUM_UMMA_PIPE_VARIANTS = 4;          // TILE_N = 64, 128, 256; 256 on a CTA pair

// One translation unit per activation bit count (conv_umma_pipe_a1.cu .. a8.cu): its three channel tiles and
// its share of the give-up counter.
#define EBS_DEFINE_PIPE_ROW(AB)                                                                             \
    const ConvVariant* conv_umma_pipe_variant_a##AB(int variant) {                                          \
        static const ConvVariant row[NUM_UMMA_PIPE_VARIANTS] = {                                            \
            ConvVariant{&launch_conv_umma_pipe<AB, 64>, UMMA_M, 64, PIPE_THREADS},                          \
            ConvVariant{&launch_conv_umma_pipe<AB, 128>, UMMA_M, 128, PIPE_THREADS},                        \
            ConvVariant{&launch_conv_umma_pipe<AB, 256>, UMMA_M, 256, PIPE_THREADS},                        \
            ConvVariant{&launch_conv_umma_pipe_pair<AB>, UMMA_M, 256, PIPE_THREADS}};                       \
        if (variant < 0 || variant >= NUM_UMMA_PIPE_VARIANTS) return nullptr;                               \
        return &row[variant];                                                                               \
    }                                                                                                       \
    unsigned long long conv_umma_pipe_timeouts_a##AB() {                                                    \
        unsigned long long v = 0;                                                                           \
        cudaMemcpyFromSymbol(&v, g_umma_timeouts, sizeof(v));                                               \
        return v;                                                                                           \
    }

}  // namespace ebs
