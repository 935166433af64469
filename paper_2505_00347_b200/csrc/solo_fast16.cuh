// Sixteen elements per thread: the streamlined step for the plain step (2/3/4/8-bit states, blocks of
// 64, 128, 256 or 2048, fp32 or bf16 parameters; no L2 term in the gradient, no AdaBelief, base from the
// p-quantile, xi drawn: MODES = 0).  The other instantiations: MODES = 1 reads the L2 term, AdaBelief, a fixed base and no dither from
// the arguments; MODES = 3 is the plain step with stochastic rounding of the first moment (Eq. 5), MODES = 4 the plain step
// with a baseline second-moment codebook (a fixed level table instead of the logarithmic levels: no quantile, no draws, nearest
// level), both fixed at compile time; MODES = 2 reads all of them, for the combinations.  What an instantiation leaves out costs
// twice, in branches and in places of the instruction cache: MODES = 1 read as MODES = 2 is 11 % slower, Eq. 5 took 295 us as
// MODES = 2 and takes 260 (4/2 bit, 2^26 elements; 8/8 bit 388 and 319), dynamic exponent for both moments 219 and 209.
//
// Same arithmetic, element for element, as solo_step_fast_kernel (solo_fast.cuh), in packed pairs of
// binary32 (F2): the kernel is bound by instruction issue and a packed operation gives two results per issue
// slot.  2^27 elements, block 128: 2/3 bit 436 -> 416 us, 4/4 bit 491 -> 455 us, 2/2 bit 429 -> 395 us, with the
// L2 term 596 -> 508 us.  What changes is the work split.  A CTA of 128 threads owns a tile of 2048 consecutive elements, a thread
// sixteen of them, a block of 64 / 128 / 256 elements G = 4 / 8 / 16 consecutive lanes, a warp eight,
// four or two blocks; a block of 2048 the whole CTA (G = 128).  The per-thread work that does not depend on the element count (waiting for the
// staged inputs, addressing, the level tables, the exchange with the first warp, the rounds of the
// selection) is spent once per sixteen elements instead of once per eight.
//
// Resources are cut for seven or eight resident CTAs per SM (ctas16): at most 72 or 64 registers per thread
// and one input stage of 13.6 KB (15 KB of shared memory in all; 23 KB for blocks of 64); with 8-bit states six or seven CTAs,
// at most 80 or 72 registers and up to 39 KB.  The stage is read only
// before the tile's first CTA barrier, so the copies of the CTA's next tile are issued right after
// that barrier and land while the tile's second half (per-block scalars, random draws,
// quantization) runs.  Parameters stay in the stage until the update of their four elements needs
// them.
//
// Shared-memory banks: a thread's sixteen parameters are 64 consecutive bytes of the staged tile, so
// the eight lanes that one 128-bit shared-memory access serves hit only two groups of four banks (a
// four-way conflict; gradients, 32 bytes per thread: two-way).  Lanes 4..7 of every group of eight
// therefore take the two halves of their sixteen elements in the other order (`sw`): their accesses
// fall on the other banks, which halves the conflicts of the parameters and removes those of the
// gradients.  Everything that is tied to an element's position (its codes, its Philox draw, where
// its parameter is stored) follows the swap; nothing else depends on the order.
//
// 8-bit states: codes of fixed codebooks by one cell look-up and one comparison (solo_lut8.cuh), alpha^k from a table
// of the code's low bits that the block's lanes double bit by bit.  Against the eight-per-thread kernel's eight-step
// searches and eight-factor chains (2^27 elements): 8/8 bit 886 -> 496 us, block 256 947 -> 502, 8/4 bit 816 -> 418; against the
// general kernel: dynamic exponent for both moments 1754 -> 417 us, Eq. 5 2356 -> 763.  With two fixed codebooks the
// kernel is bound by shared-memory wavefronts (83 % of their peak: six look-ups per element, two to four
// different words per bank each).
//
// This kernel processes full tiles of 16-byte aligned tensors only; every other tile is left to
// a second launch with StepArgs::only_partial set: of solo_step_fast_kernel, or of the general kernel
// where that one has no path (Eq. 5, the baseline codebooks).
#pragma once

#include "solo_dispatch.h"
#include "solo_fast.cuh"
#include "solo_lut8.cuh"

namespace solo {

constexpr int EPT16 = 16;               // elements per thread
static_assert(CTA16 * EPT16 == TILE, "same tile as the other kernels");

// Resident CTAs per SM an instantiation is compiled for: eight (64 registers), seven (72) for 4-bit first moments
// and for blocks of 256, which spill more at 64 (2^27 elements: 2/3 bit at block 128 380 us at seven, 367 us at
// eight; 4/4 bit 422 and 421 us; 4/4 bit at block 256 432 and 434 us).  8-bit states, whose tables fill the shared
// memory: seven, six where the modes' tables come on top (8/8 bit five 516, six 498, seven 496 us; Eq. 5 four 830, five
// 799, six 763 us, read from the arguments; Eq. 5 alone and a codebook alone have the same number and were not timed with others).
template <int BM, int BV, int G, int MODES>
constexpr int ctas16() { return BM == 8 || BV == 8 ? (MODES >= 2 ? 6 : 7) : BM == 4 || G >= 16 ? 7 : 8; }

// What the first rounds of Philox4x32-10 leave of the counter's words that are the same for a whole tile: (position, high word,
// step, 4 * stream) differ in the position's low word only, which reaches half of the second round and all of the third.
// Computed per tensor by the thread that walks (draw_keys): a call is 18 wide multiplications instead of 20, and no thread looks up its
// tensor's stream (2^26 elements: 2/3 bit 183.5 -> 181.7 us, bf16 parameters stochastically rounded 240 -> 236).
struct DrawKeys {
    uint32_t k2, k3, k4, k6;
};
__device__ __forceinline__ DrawKeys draw_keys(const uint32_t (&rk)[20], uint32_t ctr_hi, uint32_t step, uint32_t stream4) {
    const uint64_t p1 = (uint64_t)0xCD9E8D57u * step;
    const uint64_t p0 = (uint64_t)0xD2511F53u * ((uint32_t)(p1 >> 32) ^ ctr_hi ^ rk[0]);
    return {stream4 ^ rk[1], (uint32_t)p1 ^ rk[2], (uint32_t)(p0 >> 32) ^ rk[3], (uint32_t)p0 ^ rk[5]};
}
// philox_rk(c0, ctr_hi, step, stream4 + purpose, rk, out)
__device__ __forceinline__ void philox_keys(uint32_t c0, const DrawKeys& k, uint32_t purpose, const uint32_t (&rk)[20], uint32_t (&out)[4]) {
    constexpr uint64_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
    uint64_t p0 = M0 * c0;
    uint64_t p1 = M1 * ((uint32_t)(p0 >> 32) ^ k.k2 ^ purpose);
    c0 = (uint32_t)(p1 >> 32) ^ k.k3;
    uint32_t c1 = (uint32_t)p1, c2 = (uint32_t)p0 ^ k.k4;
    p0 = M0 * c0;
    p1 = M1 * c2;
    c0 = (uint32_t)(p1 >> 32) ^ c1 ^ rk[4];
    c2 = (uint32_t)(p0 >> 32) ^ k.k6;
    c1 = (uint32_t)p1;
    uint32_t c3 = (uint32_t)p0;
#pragma unroll
    for (int r = 3; r < 10; ++r) {
        p0 = M0 * c0;
        p1 = M1 * c2;
        c0 = (uint32_t)(p1 >> 32) ^ c1 ^ rk[2 * r];
        c2 = (uint32_t)(p0 >> 32) ^ c3 ^ rk[2 * r + 1];
        c1 = (uint32_t)p1;
        c3 = (uint32_t)p0;
    }
    out[0] = c0; out[1] = c1; out[2] = c2; out[3] = c3;
}

// Which kernels take a tile's keys from its description; the others draw from the counters as they are.  Blocks of 64: the keys
// gain nothing there (2^24 elements, fp32: 1.00) and cost the modes that are read from the arguments 2 to 3 %.  Modes read from the
// arguments with bf16 parameters, blocks of 128 and 256: the keys cost steps with a fixed base, which have little else to do, up to 4 %
// (2^25 elements, block 128, 8/4 bit 105.2 us, without 100.1, 3/4 bit 108.0 and 103.6) and the other modes up to 3 % (AdaBelief, 2/2 bit
// 117.0 and 113.5; 2/3 bit alone is faster with them, 120.0 and 122.1).  But with 4-bit first moments the kernel spills more without
// (4/2 bit, fixed base, 99.6 and 104.3), and blocks of 2048 are 2 to 5 % slower without.
template <int BM, bool PBF, int G, int MODES>
constexpr bool DRAW_KEYS = G != 4 && !(PBF && MODES == 1 && BM != 4 && G <= 16);

// G: lanes per block (4, 8, 16 or 128 for blocks of 64, 128, 256 or 2048 elements); NG = 128 / G blocks per tile.
template <int BM, int BV, bool PBF, int G>
struct Fast16Shared {
    static constexpr int NG = CTA16 / G;
    static constexpr int LG = G < 32 ? G : 32;                       // lanes that build a block's level tables,
    static constexpr int NT = CTA16 / LG;                            // and how many there are: a block of 2048 has one per warp
    // G = 4: sorted keys of the threads, one column per thread: row j holds the (j+2)-th smallest key, row 15 a
    // sentinel above every key
    uint32_t sort[G == 4 ? 16 : 1][G == 4 ? CTA16 : 1];
    // per block: K_v second-moment levels alpha^k Delta_v and K_m first-moment levels y_k Delta_m.
    // Two arrays, so that the four blocks of a warp occupy distinct banks (up to eight levels).  2-bit
    // moments: the sixteen pairs of levels instead, so that one look-up serves two elements; four lanes
    // per block spend more on building sixteen pairs than they save (2/2 bit at block 64 on 2^27 elements:
    // 346 us with single levels, 380 us with pairs).
    static constexpr bool PAIRS = G >= 8;
    // 8-bit second moments: alpha^k for the low TB bits of the code, sixteen entries per lane of the block
    // (eight words of padding put the blocks of a warp on different banks); the factors of the bits above
    // are multiplied on per element.  With G = 16 that is all eight bits, and Delta_v is in the table.  8-bit first
    // moments: the codebook itself, scaled per element.
    static constexpr int TB = BV != 8 ? BV : G == 4 ? 6 : G == 8 ? 7 : 8;
    static constexpr int TAB8 = (1 << TB) + (G == 128 ? 64 : 8);
    alignas(16) float tab_v[NT][BV == 8 ? TAB8 : BV == 2 && PAIRS ? 32 : 1 << BV];
    alignas(8) float tab_m[BM == 8 ? 1 : NT][BM == 8 ? 2 : BM == 2 && PAIRS ? 32 : 1 << BM];
    alignas(16) unsigned char lut_m[BM == 8 ? LUT8_M_BYTES : 16];        // cells of the signed codebook (solo_lut8.cuh)
    // 8-bit baseline second-moment codebook, in the place of tab_v, which it has no use for
    struct Codebook8 {
        unsigned char lut[LUT8_V_BYTES];
        float y[256], mid[256];              // mid[255]: +infinity
    };
    static_assert(BV != 8 || sizeof(Codebook8) <= sizeof(float) * NT * TAB8, "fits the table's place");
    __device__ Codebook8& v8() { return *reinterpret_cast<Codebook8*>(&tab_v[0][0]); }
    // Blocks of 2048: what the four warps exchange, the histogram and the list of the selection (select_cta16)
    struct Cta {
        uint32_t m[4], v[4], lo[4], failed[4];   // per warp: maxima of |m^| and v^, minimum of v^, gave up on the tile's inputs
        uint32_t hist[256], list[512], fill;
    };
    alignas(16) unsigned char cta_bytes[G == 128 ? sizeof(Cta) : 16];
    __device__ Cta& cta() { return *reinterpret_cast<Cta*>(cta_bytes); }
    // Exchange with the first warp.  One copy is enough: xin is written before the tile's first
    // barrier and read between its two barriers, xout is written between the barriers and read
    // after the second, and nobody writes either again before passing those barriers.
    uint4 xin[NG];                       // per block: bits of Delta_m', Delta_v', x_p; .w != 0: the block's warp skips the tile
    float4 xout[NG];                     // per block: vanishing Delta_v' (1 or 0), 1/Delta_v', 1/log2(alpha'), rounding limit
    // per 3-bit moment and warp: the packed codes of the warp's 512 elements, for 128-bit stores
    static constexpr int N3 = (BM == 3 ? 1 : 0) + (BV == 3 ? 1 : 0);
    alignas(16) uint32_t cout[N3 > 0 ? N3 : 1][N3 > 0 ? 4 : 1][N3 > 0 ? 48 : 4];   // (a token array without 3-bit codes)
    struct Stage {
        alignas(16) unsigned char p[TILE * (PBF ? 2 : 4)];   // 2048 parameters
        alignas(16) unsigned char g[TILE * 2];                // 2048 bf16 gradients
        uint32_t cm[64 * BM + 4];        // packed codes of the tile: 256 * bits bytes, from a 16-byte boundary
        uint32_t cv[64 * BV + 4];
        float sc[3][NG >= 4 ? NG + 4 : 8];   // Delta_m, Delta_v, alpha of the tile's blocks, from a 16-byte boundary
    };
    alignas(16) Stage stage;
    alignas(8) unsigned long long mbar;      // the stage's copies
    // The CTA's walk over the tiles (see produce_tile16): kept here and not in registers, because one thread uses it
    alignas(8) unsigned long long mbar_steal;
    alignas(16) uint4 steal;                 // answer of the last request for another CTA's tiles
    static constexpr bool KEYS = G != 4;     // some kernel with this layout has DRAW_KEYS
    struct Walk {
        char* p;                             // tensor: its parameters, gradients, first block
        const char* g;
        int64_t jb0;
        uint64_t ctr0;                       // its place in the random stream
        uint32_t stream4, ctr_hi;
        alignas(16) DrawKeys keys[KEYS ? 2 : 1];     // for the high word of ctr0, and for the one after
        int tensor, t_lo, t_hi, full_tiles;  // tensor: tiles [t_lo, t_hi), the first full_tiles of them full
        int tile, tile_end;                  // last tile handed out; end of the tiles taken
        uint32_t phase;                      // parity of mbar_steal's next phase
        bool unanswered;                     // the wait for an answer ran out: it may still come
        bool gave_up;                        // some thread waited in vain for a copy: the CTA takes no further tile
    } walk;
    struct Desc {
        char* p;                             // the tile's parameters, gradients, first block
        const char* g;
        int64_t jb;
        int tile, valid;                     // valid 0: no tile left
        uint32_t ctr, ctr_hi;                // stream position of its first element (element index / 8); ctr_hi and
        uint32_t stream4;                    // stream4 are left out with DRAW_KEYS
        alignas(16) DrawKeys keys[KEYS ? 2 : 1];     // [1]: of the elements behind a change of the high word
    };
    alignas(16) Desc desc[2];                 // written for the next tile between the two barriers of this one
};

__device__ __forceinline__ void bar_sync16(int id) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(CTA16) : "memory");
}

// Byte offsets (8 * pair of codes) of the eight pairs among sixteen 2-bit codes in one word, for a table of
// float pairs; see CodeOffsets.
struct PairOffsets2 {
    uint32_t even, odd;
    __device__ __forceinline__ explicit PairOffsets2(uint32_t c) : even(c & 0x0F0F0F0Fu), odd(c & 0xF0F0F0F0u) {}
    __device__ __forceinline__ uint32_t operator()(int j) const {
        const uint32_t w = (j & 1) ? odd : even;
        uint32_t top;
        asm("mul.lo.u32 %0, %1, %2;" : "=r"(top) : "r"(w), "r"(1u << (28 - 4 * j)));
        return top >> 25;
    }
};

// The thread's sixteen BITS-bit codes as two words of eight codes each, from the tile's staged
// code words (thread t owns bytes [2 * BITS * t, 2 * BITS * (t + 1)) of them).  sw = 1: the two
// words are exchanged (h[0] then holds elements 8..15).
template <int BITS>
__device__ __forceinline__ void load_codes16(const uint32_t* st, int tid, uint32_t sw, uint32_t (&h)[BITS == 8 ? 4 : 2]) {
    if constexpr (BITS == 8) {                                    // four codes per word
        const uint4 c = reinterpret_cast<const uint4*>(st)[tid];
        h[0] = sw ? c.z : c.x; h[1] = sw ? c.w : c.y;
        h[2] = sw ? c.x : c.z; h[3] = sw ? c.y : c.w;
    } else if constexpr (BITS == 2) {
        const uint32_t c = __funnelshift_r(st[tid], st[tid], 16u * sw);
        h[0] = c & 0xFFFFu; h[1] = c >> 16;
    } else if constexpr (BITS == 4) {
        const uint2 c = reinterpret_cast<const uint2*>(st)[tid];
        h[0] = sw ? c.y : c.x; h[1] = sw ? c.x : c.y;
    } else {
        static_assert(BITS == 3, "2, 3 or 4 bits");
        const int cw = (6 * tid) >> 2, cs = ((6 * tid) & 3) * 8;  // 48 bits from byte 6 * tid; cs is 0 or 16
        const uint32_t w0 = st[cw], w1 = st[cw + 1];
        const uint32_t c32 = __funnelshift_r(w0, w1, cs);         // bits 0..31
        const uint32_t c16 = (w1 >> cs) & 0xFFFFu;                // bits 32..47
        const uint32_t lo = c32 & 0xFFFFFFu, hi = (c32 >> 24) | (c16 << 8);
        h[0] = sw ? hi : lo; h[1] = sw ? lo : hi;
    }
}
// The reverse, to the tile's codes in global memory (`tile_codes`: their first byte).  3-bit codes
// (48 bits per thread) go through `stage` (48 words of the warp) so that twelve lanes store the
// warp's 192 bytes as 128-bit words.
template <int BITS>
__device__ __forceinline__ void store_codes16(uint8_t* tile_codes, uint32_t* stage, int tid, const uint32_t (&h)[BITS == 8 ? 4 : 2]) {
    if constexpr (BITS == 8) {
        __stcs(reinterpret_cast<uint4*>(tile_codes) + tid, make_uint4(h[0], h[1], h[2], h[3]));
    } else if constexpr (BITS == 2) {
        __stcs(reinterpret_cast<uint32_t*>(tile_codes) + tid, h[0] | (h[1] << 16));
    } else if constexpr (BITS == 4) {
        __stcs(reinterpret_cast<uint2*>(tile_codes) + tid, make_uint2(h[0], h[1]));
    } else {
        const int lane = tid & 31, warp = tid >> 5;
        unsigned short* const half = reinterpret_cast<unsigned short*>(stage) + 3 * lane;
        half[0] = (unsigned short)h[0];
        half[1] = (unsigned short)((h[0] >> 16) | (h[1] << 8));
        half[2] = (unsigned short)(h[1] >> 8);
        __syncwarp();
        // the warp's 192 bytes: 128-bit words where the tile's codes start on a 16-byte boundary, else
        // (3-bit codes of 64-element blocks, 24 bytes each, from an odd block on) 64-bit words
        uint8_t* const dst = tile_codes + warp * 192;
        if ((reinterpret_cast<uintptr_t>(tile_codes) & 15u) == 0) {
            if (lane < 12) __stcs(reinterpret_cast<uint4*>(dst) + lane, reinterpret_cast<const uint4*>(stage)[lane]);
        } else {
            if (lane < 24) __stcs(reinterpret_cast<uint2*>(dst) + lane, reinterpret_cast<const uint2*>(stage)[lane]);
        }
        __syncwarp();
    }
}

// Batcher's odd-even merge sort of sixteen keys without the one exchange that only orders key[13], key[14], as a
// list, so that other work can be issued between its exchanges.
__device__ constexpr unsigned char SORT16_PAIRS[62][2] = {
    {0, 1}, {2, 3}, {0, 2}, {1, 3}, {1, 2}, {4, 5}, {6, 7}, {4, 6}, {5, 7}, {5, 6},
    {0, 4}, {2, 6}, {2, 4}, {1, 5}, {3, 7}, {3, 5}, {1, 2}, {3, 4}, {5, 6},
    {8, 9}, {10, 11}, {8, 10}, {9, 11}, {9, 10}, {12, 13}, {14, 15}, {12, 14}, {13, 15}, {13, 14},
    {8, 12}, {10, 14}, {10, 12}, {9, 13}, {11, 15}, {11, 13}, {9, 10}, {11, 12}, {13, 14},
    {0, 8}, {4, 12}, {4, 8}, {2, 10}, {6, 14}, {6, 10}, {2, 4}, {6, 8}, {10, 12},
    {1, 9}, {5, 13}, {5, 9}, {3, 11}, {7, 15}, {7, 11}, {3, 5}, {7, 9}, {11, 13},
    {1, 2}, {3, 4}, {5, 6}, {7, 8}, {9, 10}, {11, 12}};

// Thresholds of the 8-bit codebooks below the cell of r (solo_lut8.cuh); |r| < 1 + 1/64 or NaN.
__device__ __forceinline__ uint32_t cell8_m(const unsigned char* lut, float r) {
    const uint32_t t = __float_as_uint(fmaxf(fabsf(r), 0x1p-22f)) ^ ((__float_as_uint(r) >> 3) & 0x10000000u);
    // (negative values: exponent bit 5 cleared.  Written so that the positive cells follow the negative ones.)
    return lut[(t >> 17) - LUT8_M_BASE];
}
__device__ __forceinline__ uint32_t cell8_v(const unsigned char* lut, float r) {
    return lut[(__float_as_uint(fmaxf(r, 0x1p-23f)) >> 16) - LUT8_V_BASE];
}
// Four codes to a word.
__device__ __forceinline__ uint32_t pack8(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    return __byte_perm(__byte_perm(a, b, 0x0040u), __byte_perm(c, d, 0x0040u), 0x5410u);
}

// A block's scale for its reciprocal: a vanishing one (below TINY; its codes are zeroed) counts as TINY, so that no ratio exceeds 1
// and the ratios index the cell tables; a NaN stays one.  On the pattern: a selection of 0 instead made 4/4 bit at block 2048
// spill twice as much (ragged set 5411 -> 5821 us).
__device__ __forceinline__ float at_least_tiny(uint32_t scale) {
    return __uint_as_float(max(scale, 0x0D800000u));
}

// Minimum / maximum over the calling lane's group of G lanes.  The shuffle-and-compare steps serve
// all groups of the warp at once; for groups of eight measured faster here than the full-mask reductions
// over a transformed value that solo_fast.cuh uses for its groups of sixteen (four REDUX plus selects for
// four groups): 294 vs 284 Gparams/s on the 7B set.
template <int G>
__device__ __forceinline__ uint32_t group_min16(uint32_t x) {
#pragma unroll
    for (int d = 1; d < G; d <<= 1) x = min(x, __shfl_xor_sync(0xffffffffu, x, d));
    return x;
}
template <int G>
__device__ __forceinline__ uint32_t group_max16(uint32_t x) {
#pragma unroll
    for (int d = 1; d < G; d <<= 1) x = max(x, __shfl_xor_sync(0xffffffffu, x, d));
    return x;
}

// Minimum of 31-bit keys over the calling lane's group.  Groups of sixteen: one full-mask minimum and one
// maximum serve both groups of the warp, the upper group's keys going in complemented (vx = ~0 there, else 0).
template <int G>
__device__ __forceinline__ uint32_t group_min31(uint32_t x, uint32_t vx) {
    if constexpr (G == 32) {
        return __reduce_min_sync(0xffffffffu, x);
    } else if constexpr (G == 16) {
        const uint32_t lo = __reduce_min_sync(0xffffffffu, x ^ vx);
        const uint32_t up = __reduce_max_sync(0xffffffffu, x ^ vx);
        return (vx ? up : lo) ^ vx;
    } else {
        return group_min16<G>(x);
    }
}

// How many of the four predicates of each of the group's lanes hold.
template <int G>
__device__ __forceinline__ int group_count4(bool p0, bool p1, bool p2, bool p3, int lane) {
    const uint32_t b0 = __ballot_sync(0xffffffffu, p0), b1 = __ballot_sync(0xffffffffu, p1);
    const uint32_t b2 = __ballot_sync(0xffffffffu, p2), b3 = __ballot_sync(0xffffffffu, p3);
    if constexpr (G == 32) {
        return (__popc(b0) + __popc(b1)) + (__popc(b2) + __popc(b3));
    } else if constexpr (G == 16) {
        const uint32_t sel = (lane & 16) ? 0x7632u : 0x5410u;
        return __popc(__byte_perm(b0, b1, sel)) + __popc(__byte_perm(b2, b3, sel));
    } else {
        static_assert(G == 8, "groups of four select by pops");
        // the byte of each ballot that holds the group
        const uint32_t sel = 0x40u + 0x11u * ((uint32_t)lane >> 3);
        return __popc(__byte_perm(__byte_perm(b0, b1, sel), __byte_perm(b2, b3, sel), 0x5410u));
    }
}

// The rank-th smallest (1-based) of the values that the G lanes of a group hold, one each: the lanes sort
// them among themselves (bitonic network over shuffles, every stage ascending, the first of each merge against the mirrored
// lane) and read the lane of that rank.
template <int G>
__device__ __forceinline__ uint32_t lanes_rank(uint32_t x, int rank, int lane) {
#pragma unroll
    for (int size = 2; size <= G; size <<= 1) {
#pragma unroll
        for (int d = size >> 1; d >= 1; d >>= 1) {
            const uint32_t y = __shfl_xor_sync(0xffffffffu, x, 2 * d == size ? size - 1 : d);
            x = (y < x) != ((lane & d) != 0) ? y : x;
        }
    }
    return __shfl_sync(0xffffffffu, x, (lane & ~(G - 1)) + rank - 1);
}

// Drops the head of a sorted list if it is at most t and n < rem (`p`, `go`: the same as predicates).  Groups of eight: the entries
// move up by predicated additions of `zero` (StepArgs::only_partial), which the compiler does not know: an addition goes to any of the integer pipes at
// one warp a cycle, a selection to one that takes a warp every other cycle (2^26 elements, 2/3 bit 186.7 -> 183.5 us, 3/3 bit 204.3 ->
// 201; bf16 parameters, 2/2 bit, 249 -> 240).  Groups of sixteen and the CTA's selections are faster (4/4 bit 220 us against 232).
template <int G>
__device__ __forceinline__ void list_drop(uint32_t (&l)[4], const bool p, const bool go, const int n, const int rem, const uint32_t t,
                                          const uint32_t zero) {
    if constexpr (G == 8) {
        asm("{\n\t.reg .pred g, p;\n\tsetp.lt.s32 g, %4, %5;\n\tsetp.le.and.u32 p, %0, %6, g;\n\t@p add.u32 %0, %1, %7;\n\t@p add.u32 %1, %2, %7;\n\t"
            "@p add.u32 %2, %3, %7;\n\t@p add.u32 %3, %7, %8;\n\t}"
            : "+r"(l[0]), "+r"(l[1]), "+r"(l[2]), "+r"(l[3]) : "r"(n), "r"(rem), "r"(t), "r"(zero), "n"(KEY_MAX));
    } else if (p && go) {
        l[0] = l[1]; l[1] = l[2]; l[2] = l[3]; l[3] = KEY_MAX;
    }
}

// k-th smallest (1-based, duplicates counted) of the 16 * G keys of a group of G lanes; each lane holds its
// sixteen as four sorted lists l[q][0..3].  A round: T = the smallest second key among the group's 4 * G
// lists; every list whose head is at most T drops it.  The n keys dropped are at most every key that stays, so
// the rank sought becomes k - n.  Of uniformly spread keys a round drops as many as one draws until
// two fall into the same list (about 7.6 of 32 lists), so rank 13 takes two or three rounds, each serving
// all groups of the warp, where popping one minimum per round took twelve and needed all sixteen keys
// of a lane in order (62 exchanges; four lists of four: 20).  When n reaches the rank, the key sought is
// among the heads: the same rounds follow over the lanes' sorted heads, then the lanes sort one value each.
// ROUNDS rounds are laid out in line, the others loop.  Every loop ends: a round drops at least one key (the
// loops are bounded by k all the same).
template <int G, int ROUNDS>
__device__ __forceinline__ uint32_t select_rank16(uint32_t (&l)[4][4], const int k, const int lane, const uint32_t zero) {
    const uint32_t vx = G == 16 && (lane & 16) ? 0xFFFFFFFFu : 0u;
    int rem = k;
    auto round = [&]() {
        const uint32_t t = group_min31<G>(min(min(l[0][1], l[1][1]), min(l[2][1], l[3][1])), vx);
        bool p[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) p[q] = l[q][0] <= t;
        const int n = group_count4<G>(p[0], p[1], p[2], p[3], lane);
        const bool go = n < rem;
#pragma unroll
        for (int q = 0; q < 4; ++q) list_drop<G>(l[q], p[q], go, n, rem, t, zero);
        if (go) rem -= n;
        return go;
    };
    bool go = true;
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) go = round();
#pragma unroll 1
    for (int it = 0; it < k && __any_sync(0xffffffffu, go); ++it) go = round();
    uint32_t h[4] = {l[0][0], l[1][0], l[2][0], l[3][0]};
    cswap(h[0], h[1]); cswap(h[2], h[3]); cswap(h[0], h[2]); cswap(h[1], h[3]); cswap(h[1], h[2]);
    const uint32_t gmask = (G == 32 ? 0xFFFFFFFFu : (1u << (G & 31)) - 1u) << (lane & ~(G - 1));
    auto head_round = [&]() {
        const uint32_t t = group_min31<G>(h[1], vx);
        const bool p = h[0] <= t;
        const int n = __popc(__ballot_sync(0xffffffffu, p) & gmask);
        go = n < rem;
        list_drop<G>(h, p, go, n, rem, t, zero);
        if (go) rem -= n;
    };
    head_round();
    head_round();
#pragma unroll 1
    for (int it = 0; it < k && __any_sync(0xffffffffu, go); ++it) head_round();
    return lanes_rank<G>(h[0], rem, lane);
}

__device__ __forceinline__ void sort_list4(uint32_t (&l)[4]) {
    cswap(l[0], l[1]); cswap(l[2], l[3]); cswap(l[0], l[2]); cswap(l[1], l[3]); cswap(l[1], l[2]);
}

// A block of 2048: k-th smallest (1-based, duplicates counted) of the CTA's keys, sixteen per thread; lo and hi are the
// smallest and the largest.  Returns it in every lane of the first warp (anything in the others).
// With the eight-per-thread kernel's eleven-bit levels and five barriers each (2^27 elements) 2/2 bit took 602 us, 4/4 bit
// 655, 8/8 bit 1028; here 491, 594, 667 (dynamic exponent for both moments, no selection: 1304 in the general
// kernel, 438).  What is left is the wait for the first warp (barrier stalls 2.3 per issue).
// The block's own range of key values is cut into 256 bins; every warp scans the histogram for itself, so that no
// barrier is needed to publish the bin that holds the rank.  The bin's keys (a tenth of the block lies
// in the lowest level of the last step's codes, so often two hundred of them side by side) are collected, up to 512, and
// ranked by the first warp alone (select_rank16).  A fuller bin is cut again.  hist and fill are zero on entry and on exit.
// All threads of the CTA, converged; three barriers in the usual case.
template <class Cta>
__device__ __forceinline__ uint32_t select_cta16(const uint32_t (&key)[EPT16], const int k, Cta& c, const uint32_t lo,
                                                 const uint32_t hi, const int tid) {
    const int lane = tid & 31, warp = tid >> 5;
    if (hi == lo) return lo;                                      // (uniform)
    int bits = 32 - __clz(hi - lo), shift = max(bits - 8, 0);     // keys of interest: base <= key < base + 2^bits
    uint32_t base = lo, kk = (uint32_t)k, cnt;
    const uint32_t hist = smem_u32(c.hist);
    // (all keys of the first histogram, without a branch around each: 8/8 bit 349 -> 313 us on 2^26 elements)
#pragma unroll
    for (int i = 0; i < EPT16; ++i)
        asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(hist + (((key[i] - lo) >> shift) << 2)) : "memory");
    __syncthreads();
    for (;;) {
        const uint4 h0 = reinterpret_cast<const uint4*>(c.hist)[2 * lane], h1 = reinterpret_cast<const uint4*>(c.hist)[2 * lane + 1];
        const uint32_t h[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
        const uint32_t mine = ((h[0] + h[1]) + (h[2] + h[3])) + ((h[4] + h[5]) + (h[6] + h[7]));
        uint32_t incl = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += t;
        }
        const int src = __ffs(__ballot_sync(0xffffffffu, kk <= incl)) - 1;      // the lane that holds the rank
        uint32_t run = incl - mine, below = run, bin = 8u * (uint32_t)lane;     // keys in the bins before the one that holds it
#pragma unroll
        for (int j = 0; j < 7; ++j) {
            run += h[j];
            if (run < kk) {
                below = run;
                ++bin;
            }
        }
        bin = __shfl_sync(0xffffffffu, bin, src);
        kk -= __shfl_sync(0xffffffffu, below, src);
        cnt = c.hist[bin];
        base += bin << shift;
        bits = shift;
        if (shift == 0 || cnt <= 512u) break;
        __syncthreads();                                          // every warp has read the histogram
        c.hist[tid] = 0u;
        c.hist[tid + CTA16] = 0u;
        __syncthreads();
        shift = max(bits - 8, 0);
#pragma unroll
        for (int i = 0; i < EPT16; ++i) {
            const uint32_t d = key[i] - base;
            asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %1, %2;\n\t@p red.shared.add.u32 [%0], 1;\n\t}"
                         ::"r"(hist + ((d >> shift) << 2)), "r"(d), "r"(1u << bits) : "memory");
        }
        __syncthreads();
    }
    uint32_t x = base;
    if (bits > 0) {
        const uint32_t width = 1u << bits;
        uint32_t mine = 0;
#pragma unroll
        for (int i = 0; i < EPT16; ++i)                           // if (key[i] - base < width) ++mine;
            asm("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %1, %2;\n\t@p add.u32 %0, %0, 1;\n\t}" : "+r"(mine) : "r"(key[i] - base), "r"(width));
        uint32_t incl = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += t;
        }
        uint32_t at = lane == 31 ? atomicAdd(&c.fill, incl) : 0u;
        at = smem_u32(c.list) + 4u * (__shfl_sync(0xffffffffu, at, 31) + incl - mine);
#pragma unroll
        for (int i = 0; i < EPT16; ++i) {
            // if (key[i] - base < width) c.list[at++] = key[i];
            asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %1, %2;\n\t@p st.shared.u32 [%0], %3;\n\t@p add.u32 %0, %0, 4;\n\t}"
                         : "+r"(at) : "r"(key[i] - base), "r"(width), "r"(key[i]) : "memory");
        }
    }
    __syncthreads();
    c.hist[tid] = 0u;                                             // (next counted into after the next tile's barriers)
    c.hist[tid + CTA16] = 0u;
    if (tid == CTA16 - 1) c.fill = 0u;
    if (bits > 0 && warp == 0) {
        uint32_t l[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t j = (uint32_t)(lane + 32 * (4 * q + i));
                l[q][i] = j < cnt ? c.list[j] : KEY_MAX;
            }
            sort_list4(l[q]);
        }
        x = select_rank16<32, 2>(l, (int)kk, lane, 0u);
    }
    return x;
}

// Four lanes per block: k-th smallest of the 64 keys, each lane's sixteen sorted, by popping one minimum per round
// from exactly one lane (the lowest whose head equals it), k - 1 times.  With rank 7 (p = 0.1) six rounds over
// two-step minima beat the batch rounds of select_rank16, whose lists collide sooner with fewer lanes (2/2 bit,
// 2^27 elements: 328 us against 370 us).  `col`: the lane's column of Fast16Shared::sort.
__device__ __forceinline__ uint32_t select_pops4(const uint32_t (&key)[EPT16], const int k, uint32_t* const col, const int lane) {
#pragma unroll
    for (int j = 1; j < EPT16; ++j) col[(j - 1) * CTA16] = key[j];
    const uint32_t self = 1u << lane;
    const uint32_t le = (self | (self - 1u)) & (15u << (lane & ~3));
    uint32_t head = key[0];
    int off = 0;
    auto pop = [&]() {
        const uint32_t tgt = group_min16<4>(head);
        const uint32_t nxt = col[off];
        const uint32_t upto = __ballot_sync(0xffffffffu, head == tgt) & le;
        // if (upto == self) { head = nxt; off += CTA16; }
        asm("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, %2, %3;\n\t@p mov.u32 %0, %4;\n\t@p add.s32 %1, %1, %5;\n\t}"
            : "+r"(head), "+r"(off) : "r"(upto), "r"(self), "r"(nxt), "n"(CTA16));
    };
    if (k == 7) {                                                 // p = 0.1
#pragma unroll
        for (int r = 0; r < 6; ++r) pop();
    } else {
#pragma unroll 1
        for (int r = 1; r < k; ++r) {
            pop();
            off = min(off, 15 * CTA16);                           // (row 15: the sentinel)
        }
    }
    return group_min16<4>(head);
}

// Bulk copies of one full tile's inputs into the stage (one thread; a bulk copy is a warp-wide
// instruction, so copies issued by many lanes would be serialised lane by lane).  The per-block
// scalars are copied from the 16-byte boundary at or below the first.
// `extra_tx`: bytes announced on top of what is copied (test hook: the wait for this tile then runs out).
template <int BM, int BV, bool PBF, int G>
__device__ __forceinline__ void issue_tile_copy16(const StepArgs& a, Fast16Shared<BM, BV, PBF, G>& s, const char* pt,
                                                  const char* gt, int64_t jb_tile, uint32_t extra_tx) {
    constexpr int NG = CTA16 / G;
    typename Fast16Shared<BM, BV, PBF, G>::Stage& st = s.stage;
    const uint32_t bar = smem_u32(&s.mbar);
    // byte offsets of the tile's codes (2 * G * bits bytes per block); only 3-bit codes in blocks of 64
    // (24 bytes) can start 8 bytes off a 16-byte boundary: they are copied from the boundary below, with
    // 16 bytes more (the state's arrays carry that slack), and read with an offset
    const int64_t bm0 = jb_tile * (2 * G * BM), bv0 = jb_tile * (2 * G * BV);
    const uint32_t bytes_m = 256 * BM + ((bm0 & 15) ? 16u : 0u), bytes_v = 256 * BV + ((bv0 & 15) ? 16u : 0u);
    // (a single block's scalar lies within the 16 bytes that start at the boundary)
    const uint32_t bytes_s = NG < 4 ? 16u : (NG + ((jb_tile & 3) ? 4u : 0u)) * 4u;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                 "r"((uint32_t)(TILE * (PBF ? 2 : 4) + TILE * 2) + bytes_m + bytes_v + 3u * bytes_s + extra_tx)
                 : "memory");
    bulk_copy(st.p, pt, TILE * (PBF ? 2 : 4), bar);
    bulk_copy(st.g, gt, TILE * 2, bar);
    bulk_copy(st.cm, a.codes_m + (bm0 & ~(int64_t)15), bytes_m, bar);
    bulk_copy(st.cv, a.codes_v + (bv0 & ~(int64_t)15), bytes_v, bar);
    const int64_t j0 = jb_tile & ~(int64_t)3;
    bulk_copy(st.sc[0], a.scale_m + j0, bytes_s, bar);
    bulk_copy(st.sc[1], a.scale_v + j0, bytes_s, bar);
    bulk_copy(st.sc[2], a.alpha + j0, bytes_s, bar);
}

// Asks the hardware for the tiles of a CTA of this grid that has not started yet: that CTA is cancelled and its
// number written to s.steal, or the answer says that none is left.  One thread; at most one request in flight.
template <class Shared>
__device__ __forceinline__ void steal_request(Shared& s) {
    const uint32_t bar = smem_u32(&s.mbar_steal);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");         // the last answer has been read
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], 16;" ::"r"(bar) : "memory");
    asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];"
                 ::"r"(smem_u32(&s.steal)), "r"(bar) : "memory");
}
// The answer: the number of the CTA whose tiles are ours now, or -1.
template <class Shared>
__device__ __forceinline__ int steal_answer(Shared& s, int* status) {
    if (!mbar_wait(smem_u32(&s.mbar_steal), s.walk.phase)) {
        atomicOr(status, 2);                                            // (its tiles, if it was cancelled, are not stepped)
        s.walk.unanswered = true;
        return -1;
    }
    s.walk.phase ^= 1u;
    int cta;
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b128 h;\n\tld.shared.b128 h, [%1];\n\t"
        "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, h;\n\tmov.b32 %0, -1;\n\t"
        "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %0, h;\n\t}"
        : "=r"(cta) : "r"(smem_u32(&s.steal)) : "memory");
    return cta;
}

// Finds the CTA's next full tile, issues the copies of its inputs and describes it in `d` (one thread).
// A CTA owns a.share consecutive tiles of the launch; when they are done it takes over those of a CTA that
// has not started (requested when it began on its own, so the answer is there), until none is left.  The SMs
// so end together whatever their speed, a CTA sets up once for many shares, and inputs are copied ahead across
// tensors and shares.  One share per resident CTA (a static walk) left 5 % of the SM cycles idle at the launch's
// end and SMs with fewer CTAs before it: LLaMA layers 2357 -> 2170 us, GPT-125M-shaped set 432 -> 390 us, ragged set
// 3418 -> 3200 us, 2^24 elements 60 -> 55 us (bursts of ten steps; for seconds on end, at the power limit, the
// GPT-125M-shaped set takes 416 us and the ragged one 3480).
// A CTA that waited in vain for a copy ends here: it takes in the answer to its last request, so that nothing writes to its
// shared memory any more, and asks for no other.  What it then leaves unstepped (and has reported in the status word) is
// the rest of its share and at most the one that answer brought, however many CTAs have not started yet.
template <int BM, int BV, bool PBF, int G, int MODES>
__device__ __forceinline__ void produce_tile16(const StepArgs& a, Fast16Shared<BM, BV, PBF, G>& s, typename Fast16Shared<BM, BV, PBF, G>::Desc& d) {
    using Shared = Fast16Shared<BM, BV, PBF, G>;
    constexpr int NG = CTA16 / G, PSZ = PBF ? 2 : 4;
    constexpr bool DRAWS = MODES != 4 || PBF, KEYS = DRAW_KEYS<BM, PBF, G, MODES>;
    typename Fast16Shared<BM, BV, PBF, G>::Walk& w = s.walk;
    int tile_end = w.tile_end, tile = w.gave_up ? tile_end : w.tile;
    for (;;) {
        if (++tile >= tile_end) {
            const int cta = steal_answer(s, a.status);
            if (cta < 0 || w.gave_up) {                                  // (one request is under way as long as there are tiles)
                d.valid = 0;
                return;
            }
            steal_request(s);
            tile = (int)a.tile_first + cta * a.share;
            tile_end = (int)min((int64_t)tile + a.share, a.total_tiles);
            w.tile_end = tile_end;
            if (tile < w.t_lo || tile >= w.t_hi) {
                w.tensor = (a.num_tensors > 1 ? find_tensor(a.tile_start, a.num_tensors, tile) : 0) - 1;
                w.t_hi = tile;
            }
        }
        if (tile >= w.t_hi) {
            int tensor = w.tensor, t_hi;
            do {
                ++tensor;
                t_hi = (int)__ldg(a.tile_start + tensor + 1);
            } while (tile >= t_hi);
            const int64_t n = __ldg(a.numel + tensor);
            char* const pb = (char*)(a.param_list ? a.param_list[tensor] : a.param_single);
            const char* const gb = (const char*)(a.grad_list ? a.grad_list[tensor] : a.grad_single);
            const bool aligned = ((((uintptr_t)pb) | ((uintptr_t)gb)) & 15u) == 0;
            const bool skip = a.numel_check != nullptr && __ldg(a.numel_check + tensor) != n;   // reported by the other launch
            w.tensor = tensor;
            w.t_lo = (int)__ldg(a.tile_start + tensor);
            w.t_hi = t_hi;
            w.full_tiles = aligned && !skip ? (int)(n / TILE) : 0;
            w.jb0 = __ldg(a.block_start + tensor);
            w.p = pb;
            w.g = gb;
            if constexpr (DRAWS) {
                const Origin org = origin_of(a, tensor);
                w.ctr0 = org.ctr0;
                w.stream4 = org.stream * 4u;
                w.ctr_hi = (uint32_t)(org.ctr0 >> 32);
                if constexpr (KEYS) {
                    w.keys[0] = draw_keys(a.rk, w.ctr_hi, a.step32, w.stream4);
                    w.keys[1] = draw_keys(a.rk, w.ctr_hi + 1u, a.step32, w.stream4);
                }
            }
        }
        if (tile - w.t_lo < w.full_tiles) break;
        tile = min(w.t_hi, tile_end) - 1;                                // the rest of the tensor is left to the other launch
    }
    w.tile = tile;
    const int tin = tile - w.t_lo;
    d.p = w.p + (int64_t)tin * (TILE * PSZ);
    d.g = w.g + (int64_t)tin * (TILE * 2);
    d.jb = w.jb0 + (int64_t)tin * NG;
    if constexpr (DRAWS) {
        const uint64_t ctr = w.ctr0 + (uint64_t)(uint32_t)tin * (TILE / 8);
        d.ctr = (uint32_t)ctr;
        if constexpr (KEYS) {
            if ((uint32_t)(ctr >> 32) != w.ctr_hi) {
                w.ctr_hi = (uint32_t)(ctr >> 32);
                w.keys[0] = draw_keys(a.rk, w.ctr_hi, a.step32, w.stream4);
                w.keys[1] = draw_keys(a.rk, w.ctr_hi + 1u, a.step32, w.stream4);
            }
            d.keys[0] = w.keys[0];
            d.keys[1] = w.keys[1];
        } else {
            d.ctr_hi = (uint32_t)(ctr >> 32);
            d.stream4 = w.stream4;
        }
    }
    d.tile = tile;
    d.valid = 1;
    issue_tile_copy16<BM, BV, PBF, G>(a, s, d.p, d.g, d.jb, tile + 1 == a.debug_stall_tile_p1 ? 16u : 0u);
}

// Per-block scalars of the tile's sixteen blocks (one block per calling thread, tid = 0..15), from
// what the blocks' lanes left in xin: stores Delta_m', Delta_v', alpha' of the blocks whose warp did not
// skip the tile and leaves what Eq. 6 needs in xout.
template <int KV, class Shared>
__device__ __forceinline__ void block_scalars16(const StepArgs& a, Shared& s, const int64_t jb_tile, const int tid,
                                                const bool fixed_base, const bool vtab) {
    const uint4 in = s.xin[tid];
    const float dm_new = __uint_as_float(in.x), dv_new = __uint_as_float(in.y);
    const bool zero_m = dm_new < TINY, zero_v = dv_new < TINY;
    const float inv_dv = __frcp_rn(at_least_tiny(in.y));
    const float rho = fminf(fmaxf(__uint_as_float(in.z) * inv_dv, RHO_MIN), RHO_MAX);
    const float lam = log2_sp(rho) * (1.0f / (float)(KV - 1));
    // (a baseline codebook has no base: the array keeps its initial 1/2)
    const float al_new = vtab ? 0.5f : fixed_base ? a.fixed_alpha : exp2_sp(lam);
    const float inv_lambda = __frcp_rn(log2_sp(al_new));
    const float guard = __fmaf_rn(fabsf(inv_lambda), LG2_ABS, LG2_REL * (float)(KV + 1));
    s.xout[tid] = make_float4(zero_v ? 1.0f : 0.0f, inv_dv, inv_lambda, 0.5f - guard);
    if (in.w == 0u) {
        const int64_t j = jb_tile + tid;
        a.scale_m[j] = zero_m ? 0.0f : dm_new;
        a.scale_v[j] = zero_v ? 0.0f : dv_new;
        a.alpha[j] = zero_v ? 0.5f : al_new;
    }
}

// One full tile.  DECAY: the parameter is multiplied by 1 - lr * wd (false: that factor is 1).
//
// Order of the work, chosen so that at most the two moments and the sort keys (48 registers) are
// live at once: (A) inputs, Eq. 2-3; (B) the parameter update, parameters read from the stage four
// at a time; (C) the first moment's scale and codes (each thread divides for itself: the scale is
// known to all eight lanes after the maximum); (D) the sorted lists and the selection rounds; (E) the
// exchange with the first warp, the thread's two Philox blocks meanwhile, the second moment's codes, the stores.
template <int BM, int BV, bool PBF, int G, bool DECAY, int MODES, bool SR>
__device__ __forceinline__ void fast16_tile(const StepArgs& a, Fast16Shared<BM, BV, PBF, G>& s, const float* s_y, const float* s_mid,
                                            const float4* s_mid4, const float* s_yv, const float4* s_nv,
                                            const float2* s_yg, const float4* s_br,
                                            const uint32_t fill, bool& failed) {
    using Shared = Fast16Shared<BM, BV, PBF, G>;
    constexpr int KM = 1 << BM, KV = 1 << BV, NG = Shared::NG;    // G lanes per block, NG blocks per tile
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int gl = tid & (G - 1), grp = tid / G;
    const uint32_t sw = ((uint32_t)tid >> 2) & 1u;               // 1: this thread takes elements 8..15 first (see the top of the file)
    // PLAIN: the step of the paper as it stands (no L2 term in the gradient, no AdaBelief, base from the
    // p-quantile, xi drawn), with Eq. 5 (MODES 3) or a baseline codebook (MODES 4) or without; the other
    // instantiations read these modes from the arguments, MODES 2 also Eq. 5 and the baseline codebooks
    constexpr bool PLAIN = MODES == 0 || MODES >= 3;
    // bf16 parameters: how they are rounded is a property of the instantiation where the update is tried by approximations (see there)
    constexpr bool BY_ROUNDING = PBF && ROUNDING_INSTANCES<G, MODES>;
    static_assert(BY_ROUNDING || !SR, "other instantiations read it from the arguments");
    const bool l2 = !PLAIN && a.l2, belief = !PLAIN && a.belief;
    // baseline codebook for the second moment: levels s_yv, nearest level by the midpoints in s_nv
    const bool vtab = MODES == 4 || (MODES == 2 && a.tables_v != nullptr);
    const bool fixed_base = MODES == 4 || (!PLAIN && (a.fixed_alpha > 0.0f || vtab));   // no quantile to find
    const bool round_v = MODES != 4 && (PLAIN || (a.round_v && !vtab));
    const bool round_m = MODES == 3 || (MODES == 2 && a.round_m);   // Eq. 5 instead of Eq. 1 for the first moment

    const typename Shared::Desc& desc = s.desc[fill & 1u];
    char* const pt = desc.p;
    const int64_t jb_tile = desc.jb;

    // ---- (A) inputs from the stage ----
    // Copy number f completes phase f of the stage's mbarrier (parity f & 1).  The copy for this tile
    // was issued after the first barrier of the tile before it (every thread had read the stage by then).
    if (!mbar_wait(smem_u32(&s.mbar), fill & 1u, failed ? 1 : MBAR_POLLS)) {
        if (!failed) atomicOr(a.status, 2);
        failed = true;
        s.walk.gave_up = true;
    }
    // A warp in which any lane gave up leaves the tile alone: it stores nothing, flags its blocks
    // for the first warp (which stores the per-block scalars), and only keeps the CTA's barriers and, if it is
    // the first warp, the other warps' scalars going.  It is the CTA's last tile (produce_tile16).
    // A block of 2048 spans the CTA, which leaves the tile as a whole (below).
    const bool gave_up = __any_sync(0xffffffffu, failed);
    if (G != 128 && gave_up) {
        if (gl == 0) s.xin[grp] = make_uint4(0u, 0u, 0u, 1u);
        bar_sync16(1);
        if (tid == 32) produce_tile16<BM, BV, PBF, G, MODES>(a, s, s.desc[(fill + 1u) & 1u]);
        if (tid < NG) block_scalars16<KV>(a, s, jb_tile, tid, fixed_base, vtab);
        bar_sync16(2);
        return;
    }

    const typename Shared::Stage& st = s.stage;
    F2 mh[EPT16 / 2], vh[EPT16 / 2];                              // elements 2j, 2j + 1 (in the thread's order)
    auto mh_at = [&](int i) { return (i & 1) ? mh[i >> 1].hi() : mh[i >> 1].lo(); };
    auto vh_at = [&](int i) { return (i & 1) ? vh[i >> 1].hi() : vh[i >> 1].lo(); };
    uint32_t mx_v = 0;
    float mx_m_f = 0.0f;
    {
        uint32_t cm[BM == 8 ? 4 : 2], cv[BV == 8 ? 4 : 2];        // eight codes per word, 8-bit: four
        // (word offsets of codes that do not start on a 16-byte boundary: 0 or 2, see issue_tile_copy16)
        load_codes16<BM>(st.cm + ((int)((jb_tile * (2 * G * BM)) & 15) >> 2), tid, sw, cm);
        load_codes16<BV>(st.cv + ((int)((jb_tile * (2 * G * BV)) & 15) >> 2), tid, sw, cv);
        const int so = (int)(jb_tile & 3) + grp;
        const float dm = st.sc[0][so], dv = st.sc[1][so], al = st.sc[2][so];

        // per-block level tables (Eq. 2), built by the block's G lanes
        constexpr int LG = Shared::LG;
        const int tl = tid & (LG - 1), tt = tid / LG;             // lane among the table's, its number
        float* const tab_vf = s.tab_v[tt];
        float* const tab_mf = s.tab_m[BM == 8 ? 0 : tt];
        float a2[BV];
        {
            a2[0] = al;
#pragma unroll
            for (int i = 1; i < BV; ++i) a2[i] = a2[i - 1] * a2[i - 1];
            auto level_v = [&](uint32_t k) { return (vtab ? s_yv[k] : pow_sm<BV>(a2, k)) * dv; };
            if constexpr (BV == 8) {
                // entries 2 tl, 2 tl + 1 from the bits that tell the lanes apart, then doubled bit by bit: entry q is
                // entry (q without its top bit) times the top bit's factor, as in the chain of pow_sm
                if (!vtab) {
                    constexpr int LB = LG == 4 ? 3 : LG == 8 ? 4 : LG == 16 ? 5 : 6;      // bits of 2 tl + 1
                    constexpr int DB = Shared::TB - LB;
                    float f[LB];
#pragma unroll
                    for (int i = 0; i < LB; ++i) f[i] = a2[i];
                    F2 e[1 << DB];
                    e[0] = F2::pack(pow_sm<LB>(f, (uint32_t)(2 * tl)), pow_sm<LB>(f, (uint32_t)(2 * tl + 1)));
#pragma unroll
                    for (int b = 0; b < DB; ++b)
#pragma unroll
                        for (int i = 0; i < (1 << b); ++i) e[i + (1 << b)] = mul2(e[i], F2::dup(a2[LB + b]));
#pragma unroll
                    for (int i = 0; i < (1 << DB); ++i) {
                        const F2 t = Shared::TB == 8 ? mul2(e[i], F2::dup(dv)) : e[i];
                        *reinterpret_cast<float2*>(tab_vf + 2 * tl + (i << LB)) = make_float2(t.lo(), t.hi());
                    }
                }
            } else if constexpr (BV == 2 && Shared::PAIRS) {
#pragma unroll
                for (int r0 = 0; r0 < 16; r0 += LG)
                    if (r0 + tl < 16)
                        *reinterpret_cast<float2*>(tab_vf + 2 * (r0 + tl)) = make_float2(level_v((r0 + tl) & 3), level_v((r0 + tl) >> 2));
            } else {
#pragma unroll
                for (int r0 = 0; r0 < KV; r0 += LG)
                    if (r0 + tl < KV) tab_vf[r0 + tl] = level_v(r0 + tl);
            }
            if constexpr (BM == 8) {
            } else if constexpr (BM == 2 && Shared::PAIRS) {
#pragma unroll
                for (int r0 = 0; r0 < 16; r0 += LG)
                    if (r0 + tl < 16)
                        *reinterpret_cast<float2*>(tab_mf + 2 * (r0 + tl)) = make_float2(s_y[(r0 + tl) & 3] * dm, s_y[(r0 + tl) >> 2] * dm);
            } else {
#pragma unroll
                for (int r0 = 0; r0 < KM; r0 += LG)
                    if (r0 + tl < KM) tab_mf[r0 + tl] = s_y[r0 + tl] * dm;
            }
        }
        __syncwarp();

        // Eq. 2, Eq. 3
        const char* const tab_v = reinterpret_cast<const char*>(tab_vf);
        const char* const tab_m = reinterpret_cast<const char*>(tab_mf);
        const PairOffsets2 om16(cm[0] | (cm[1] << 16)), ov16(cv[0] | (cv[1] << 16));   // used for 2-bit codes only
        const CodeOffsets<BM> om4a(cm[0], cm[1]), om4b(cm[BM == 8 ? 2 : 1], cm[BM == 8 ? 3 : 1]);
        const CodeOffsets<BV> ov4a(cv[0], cv[1]), ov4b(cv[BV == 8 ? 2 : 1], cv[BV == 8 ? 3 : 1]);
        const unsigned char* const sgb = st.g + 32 * tid;
        const uint4* const sg[2] = {reinterpret_cast<const uint4*>(sgb + 16u * sw),
                                    reinterpret_cast<const uint4*>(sgb + 16u - 16u * sw)};
        const F2 beta1 = F2::dup(a.beta1), omb1 = F2::dup(a.omb1), beta2 = F2::dup(a.beta2), omb2 = F2::dup(a.omb2);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint4 gw = *sg[h];
            const uint32_t gg[4] = {gw.x, gw.y, gw.z, gw.w};
            F2 g2[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) g2[k] = F2::pack(__uint_as_float(gg[k] << 16), __uint_as_float(gg[k] & 0xffff0000u));
            if (l2) {                                             // Adam: the decay term joins the gradient
                F2 p2[4];
                if constexpr (PBF) {
                    const uint4 pw = reinterpret_cast<const uint4*>(st.p)[2 * tid + ((uint32_t)h ^ sw)];
                    const uint32_t pin[4] = {pw.x, pw.y, pw.z, pw.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) p2[k] = F2::pack(__uint_as_float(pin[k] << 16), __uint_as_float(pin[k] & 0xffff0000u));
                } else {
                    const float4* const ph = reinterpret_cast<const float4*>(st.p + 64 * tid + 32u * ((uint32_t)h ^ sw));
                    const float4 pa = ph[0], pb = ph[1];
                    p2[0] = F2::pack(pa.x, pa.y); p2[1] = F2::pack(pa.z, pa.w);
                    p2[2] = F2::pack(pb.x, pb.y); p2[3] = F2::pack(pb.z, pb.w);
                }
                const F2 wd = F2::dup(a.weight_decay);
#pragma unroll
                for (int k = 0; k < 4; ++k) g2[k] = fma2(wd, p2[k], g2[k]);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int j = 4 * h + k;                          // pair of elements 2j, 2j + 1
                auto code_m = [&](int i) {
                    const char* const t = BM == 8 ? reinterpret_cast<const char*>(s_y) : tab_m;
                    return *reinterpret_cast<const float*>(t + (i < 8 ? om4a(i) : om4b(i - 8)));
                };
                auto code_v = [&](int i) {
                    if constexpr (BV == 8) {
                        const uint32_t o = i < 8 ? ov4a(i) : ov4b(i - 8);
                        if (vtab) return *reinterpret_cast<const float*>(reinterpret_cast<const char*>(s.v8().y) + o);
                        float x = *reinterpret_cast<const float*>(tab_v + (o & ((4u << Shared::TB) - 4u)));
#pragma unroll
                        for (int b = Shared::TB; b < 8; ++b) x = x * ((o >> (b + 2)) & 1u ? a2[b] : 1.0f);
                        return x;
                    } else {
                        return *reinterpret_cast<const float*>(tab_v + (i < 8 ? ov4a(i) : ov4b(i - 8)));
                    }
                };
                F2 mt, vt;
                if constexpr (BM == 2 && Shared::PAIRS) mt = F2::load(tab_m + om16(j));
                else mt = F2::pack(code_m(2 * j), code_m(2 * j + 1));
                if constexpr (BV == 2 && Shared::PAIRS) vt = F2::load(tab_v + ov16(j));
                else vt = F2::pack(code_v(2 * j), code_v(2 * j + 1));
                if constexpr (BM == 8) mt = mul2(mt, F2::dup(dm));
                if constexpr (BV == 8) {
                    if (Shared::TB < 8 || vtab) vt = mul2(vt, F2::dup(dv));
                }
                mh[j] = fma2(beta1, mt, mul2(omb1, g2[k]));
                if (belief) {                                     // AdaBelief: (g - m^)^2, plus eps
                    const F2 sig = fma2(mh[j], F2::dup(-1.0f), g2[k]);      // g - m^, one rounding
                    vh[j] = add2(fma2(beta2, vt, mul2(omb2, mul2(sig, sig))), F2::dup(a.eps));
                } else {
                    vh[j] = fma2(beta2, vt, mul2(omb2, mul2(g2[k], g2[k])));
                }
                mx_m_f = max_abs_nan(max_abs_nan(mx_m_f, mh[j].lo()), mh[j].hi());
                mx_v = max(max(mx_v, __float_as_uint(vh[j].lo())), __float_as_uint(vh[j].hi()));
            }
        }
    }

    const uint32_t tmx_v = mx_v;                                  // the thread's own maximum
    uint32_t mx_m = __float_as_uint(mx_m_f), mn_v = 0u;
    if constexpr (G == 128) {
        // maxima (and the minimum of v^, for the selection) over the CTA through shared memory
        typename Shared::Cta& c = s.cta();
        mn_v = __float_as_uint(vh_at(0));
#pragma unroll
        for (int i = 1; i < EPT16; ++i) mn_v = min(mn_v, __float_as_uint(vh_at(i)));
        mx_m = __reduce_max_sync(0xffffffffu, mx_m);
        mx_v = __reduce_max_sync(0xffffffffu, mx_v);
        mn_v = __reduce_min_sync(0xffffffffu, mn_v);
        if (lane == 0) {
            c.m[warp] = mx_m;
            c.v[warp] = mx_v;
            c.lo[warp] = mn_v;
            c.failed[warp] = gave_up ? 1u : 0u;
        }
        __syncthreads();
        const uint4 m4 = *reinterpret_cast<const uint4*>(c.m), v4 = *reinterpret_cast<const uint4*>(c.v);
        const uint4 l4 = *reinterpret_cast<const uint4*>(c.lo), f4 = *reinterpret_cast<const uint4*>(c.failed);
        if (f4.x | f4.y | f4.z | f4.w) {
            if (tid == 32) produce_tile16<BM, BV, PBF, G, MODES>(a, s, s.desc[(fill + 1u) & 1u]);
            bar_sync16(2);
            return;
        }
        mx_m = max(max(m4.x, m4.y), max(m4.z, m4.w));
        mx_v = max(max(v4.x, v4.y), max(v4.z, v4.w));
        mn_v = min(min(l4.x, l4.y), min(l4.z, l4.w));
    }

    // ---- (B) Adam(W) update, four (fp32) or eight (bf16) elements at a time ----
    // bf16 parameters: correctly rounded square root and division (see solo_fast.cuh), rounded to nearest even or
    // with the element's Philox draw (purpose 2, one block per eight elements)
    // The draws of the thread's eight elements `half` (0: the first in its own order).  Positions in the stream count eights of
    // elements; a tensor starts at a multiple of eight of them, so that the thread's two share the high word.
    auto draw8 = [&](uint32_t half, uint32_t purpose, uint32_t (&out)[4]) {
        const uint32_t c0 = desc.ctr + 2u * (uint32_t)tid;
        if constexpr (DRAW_KEYS<BM, PBF, G, MODES>) {
            const DrawKeys k = desc.keys[c0 < desc.ctr ? 1 : 0];
            philox_keys(c0 + half, k, purpose, a.rk, out);
        } else {
            philox_rk(c0 + half, desc.ctr_hi + (c0 < desc.ctr ? 1u : 0u), a.step32, desc.stream4 + purpose, a.rk, out);
        }
    };
    if constexpr (!PBF) {
        // the thread's first eight elements (in its own order) at `sp[0]`, the others at `sp[1]`
        const unsigned char* const spb = st.p + 64 * tid;
        char* const gpb = pt + 64 * tid;
        const float4* const sp[2] = {reinterpret_cast<const float4*>(spb + 32u * sw),
                                     reinterpret_cast<const float4*>(spb + 32u - 32u * sw)};
        float4* const gp[2] = {reinterpret_cast<float4*>(gpb + 32u * sw), reinterpret_cast<float4*>(gpb + 32u - 32u * sw)};
        const F2 isb = F2::dup(a.inv_sqrt_bc2), eps = F2::dup(a.eps), lr = F2::dup(a.step_size), decay = F2::dup(a.decay);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 pv = sp[q >> 1][q & 1];
            F2 p[2] = {F2::pack(pv.x, pv.y), F2::pack(pv.z, pv.w)};
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const F2 m = mh[2 * q + k], v = vh[2 * q + k];
                const F2 den = fma2(F2::pack(sqrt_approx(v.lo()), sqrt_approx(v.hi())), isb, eps);
                // with the negated reciprocal every product has its sign turned, so that the quotient comes
                // out negated and no operand needs a negation: -q0 = m (-1/den), -q1 = (m - den q0)(-1/den) - q0
                const F2 nrc = F2::pack(rcp_approx(-den.lo()), rcp_approx(-den.hi()));
                const F2 nq0 = mul2(m, nrc);
                const F2 nq1 = fma2(fma2(den, nq0, m), nrc, nq0);
                p[k] = fma2(lr, nq1, DECAY ? mul2(p[k], decay) : p[k]);
            }
            __stcs(gp[q >> 1] + (q & 1), make_float4(p[0].lo(), p[0].hi(), p[1].lo(), p[1].hi()));
        }
    } else {
        const uint4* const sp = reinterpret_cast<const uint4*>(st.p) + 2 * tid;
        // An update by approximations is within 5.25 * 2^-23 of the IEEE operations': the square root and the reciprocal 2^-23 each, the
        // denominator's, the first quotient's and the last rounding 2^-24 each, the same of the IEEE square root, denominator and quotient,
        // a subnormal v^ that is taken as zero 2^-25.  The residual step takes the reciprocal's error and the first quotient's out
        // again (then 3.75), but not where the remainder is near the smallest subnormal number: |m^| below 2^-126.  Made smaller and larger
        // by 6 * 2^-23 (5.5 are left after the factors' own roundings) and rounded to bf16, both results are the same pattern unless
        // a rounding boundary lies between them; and then the IEEE update's too, every operation on the way being monotone.  A
        // boundary lies there for 1.8e-4 to 3.7e-4 times |update / result| of the elements: one warp (512 elements) in some eight where
        // updates are as large as the parameters, in some ten thousand where they are a thousandth of them.  Such a warp, and values or hyper-parameters out of
        // these ranges, go the long way below.  (LLaMA layer, 2/2 bit: the long way for all 689 us, this 624.)
        // Where updates are as large as the parameters, rounding to nearest, which costs less to
        // begin with, then loses (3/3 bit, mixed gradients: up to 17 %), and so does a codebook that decodes small moments as zero:
        // stochastic rounding with the logarithmic levels only, and of blocks of 128 and 2048, which have a kernel per rounding: one kernel
        // for both spilled 108 bytes a thread instead of 24 (nearest) and 48 (2/3 bit, block 128) and cost rounding to nearest up to 4 %
        // (2^25 elements, 3/4 bit, block 128: 124.3 us; without the bracket 119.5, this 116.9).  Blocks of 64 and 256 have one kernel for both
        // without the bracket, whose registers cost rounding to nearest 2 to 8 % and 1 to 4 % there.
        // A quotient below 2^-126 is rounded otherwise than in the IEEE update, which shows in results below 2^-99 |step_size| <=
        // 2^-80 only (in others it is lost against the parameter).
        // A thread whose first moments are all zero has exact results on every way (quotients of zero, with the sign of the IEEE
        // ones) and is not looked at for small ones: rows of zero weights and gradients take one pass.  A warp that has small results of another
        // kind does not try the pairwise sequence, whose look they would fail as well.  (2^25 weights and gradients of zero, 2/2 bit,
        // block 128: stochastic, in three passes 313 us, this 104; to nearest 206 and 100.)
        const bool moves = !BY_ROUNDING || mx_m_f != 0.0f;
        bool done = false, small = false;
        if (SR) {
            bool usual = tmx_v < 0x4D000000u && mx_m_f < 0x1p20f && a.eps < 0x1p30f && a.inv_sqrt_bc2 < 0x1p30f &&
                         (a.step_size == 0.0f || fabsf(a.step_size) > 0x1p-100f) && fabsf(a.step_size) < 0x1p19f;
            if (a.eps < a.inv_sqrt_bc2 * 0x1p-38f) {                  // (a subnormal v^ would show)
                uint32_t least = 0xFFFFFFFFu;
#pragma unroll
                for (int i = 0; i < EPT16; ++i) least = min(least, __float_as_uint(vh_at(i)) - 1u);
                usual = usual && least >= 0x007FFFFFu;
            }
            if (__all_sync(0xffffffffu, usual)) {
                const F2 isb = F2::dup(a.inv_sqrt_bc2), eps = F2::dup(a.eps), decay = F2::dup(a.decay);
                const F2 lr_lo = F2::dup(a.step_size * (1.0f - 0x1.8p-21f)), lr_hi = F2::dup(a.step_size * (1.0f + 0x1.8p-21f));
                uint32_t differ = 0u, all = 0xFFFFFFFFu, some = 0u;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t he = (uint32_t)h ^ sw;
                    const uint4 pw = sp[he];
                    const uint32_t pin[4] = {pw.x, pw.y, pw.z, pw.w};
                    uint32_t wp[4], pp[4];
                    draw8(he, 2u, wp);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const F2 m = mh[4 * h + k], v = vh[4 * h + k];
                        const F2 den = fma2(F2::pack(sqrt_approx(v.lo()), sqrt_approx(v.hi())), isb, eps);
                        const F2 nrc = F2::pack(rcp_approx(-den.lo()), rcp_approx(-den.hi()));
                        const F2 nq0 = mul2(m, nrc);
                        const F2 nq1 = fma2(fma2(den, nq0, m), nrc, nq0);
                        F2 pd = F2::pack(__uint_as_float(pin[k] << 16), __uint_as_float(pin[k] & 0xffff0000u));
                        if (DECAY) pd = mul2(pd, decay);
                        const F2 r1 = fma2(lr_lo, nq1, pd), r2 = fma2(lr_hi, nq1, pd);
                        // (bf16_sr of what is no NaN)
                        const uint32_t dl = wp[k] & 0xFFFFu, dh = wp[k] >> 16;
                        pp[k] = __byte_perm(__float_as_uint(r1.lo()) + dl, __float_as_uint(r1.hi()) + dh, 0x7632u);
                        const uint32_t o2 = __byte_perm(__float_as_uint(r2.lo()) + dl, __float_as_uint(r2.hi()) + dh, 0x7632u);
                        differ |= pp[k] ^ o2;
                    }
                    all &= (pp[0] & pp[1]) & (pp[2] & pp[3]);
                    some |= (pin[0] | pin[1]) | (pin[2] | pin[3]);
                    __stcs(reinterpret_cast<uint4*>(pt) + 2 * tid + he, make_uint4(pp[0], pp[1], pp[2], pp[3]));
                }
                // Results below 2^-63 (exponent bit 6 is set from there to 2) and parameters from 2 up are looked at more closely: the
                // former for subnormal quotients, the latter for NaN, which the short form of the stochastic rounding does not know.
                done = !__any_sync(0xffffffffu, differ != 0u || (moves && (~all & 0x20002000u) != 0u) || (some & 0x40004000u) != 0u);
                if (!done) {
                    bool redo = differ != 0u, tiny = false;
#pragma unroll 1
                    for (int i = 0; i < EPT16; ++i) {
                        tiny |= (reinterpret_cast<const unsigned short*>(pt)[EPT16 * tid + i] & 0x7FFFu) < 0x1800u;
                        redo |= (reinterpret_cast<const unsigned short*>(st.p)[EPT16 * tid + i] & 0x7FFFu) > 0x7F80u;
                    }
                    small = __any_sync(0xffffffffu, moves && tiny);
                    done = !small && !__any_sync(0xffffffffu, redo);
                }
            }
        }
        if (!done) {
            // The exact pairwise sequence where its scaling holds: v^ < 2^27, |m^| < 2^20 (a NaN compares false), usual
            // hyper-parameters (this kernel runs with eps >= 1e-12 > 2^-40 only); the IEEE operations otherwise.  A quotient
            // below 2^-126 is not rounded to the subnormal grid before it is multiplied, which shows in results below
            // 2^-99 |step_size| <= 2^-80 only (in others it is lost against the parameter): a warp that gets one takes the IEEE
            // operations instead, the parameters being in the stage still.  Two looks: exponent bit 6 is set in all results
            // from 2^-63 to 2 (one operation per four of them), whatever lacks it is compared.  The two passes one after the other,
            // and not two sides of a branch per half: LLaMA layer, 2/2 bit, 757 -> 716 us (one loop around both 747, and 2/2 bit with Eq. 5
            // spilled: 659 -> 723 us on 2^27 elements, as it is 646).
            bool exact = !small && __all_sync(0xffffffffu, tmx_v < 0x4D000000u && mx_m_f < 0x1p20f && a.eps < 0x1p30f && a.inv_sqrt_bc2 < 0x1p30f &&
                                                     fabsf(a.step_size) > 0x1p-40f && fabsf(a.step_size) < 0x1p19f);
            auto load8 = [&](int h, float (&p)[8]) {
                const uint4 pw = sp[(uint32_t)h ^ sw];
                const uint32_t pin[4] = {pw.x, pw.y, pw.z, pw.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    p[2 * k] = __uint_as_float(pin[k] << 16);
                    p[2 * k + 1] = __uint_as_float(pin[k] & 0xffff0000u);
                }
            };
            auto store8 = [&](int h, const float (&p)[8]) {             // returns the conjunction of the patterns
                const uint32_t he = (uint32_t)h ^ sw;
                uint32_t pp[4];
                if (BY_ROUNDING ? SR : a.param_sr) {
                    uint32_t wp[4];
                    draw8(he, 2u, wp);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        pp[k] = bf16_sr(p[2 * k], wp[k] & 0xFFFFu) | (bf16_sr(p[2 * k + 1], wp[k] >> 16) << 16);
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const __nv_bfloat162 h2 = __floats2bfloat162_rn(p[2 * k], p[2 * k + 1]);
                        pp[k] = *reinterpret_cast<const uint32_t*>(&h2);
                    }
                }
                __stcs(reinterpret_cast<uint4*>(pt) + 2 * tid + he, make_uint4(pp[0], pp[1], pp[2], pp[3]));
                return (pp[0] & pp[1]) & (pp[2] & pp[3]);
            };
            if (exact) {
                uint32_t all = 0xFFFFFFFFu;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float p[8];
                    load8(h, p);
                    const F2 nisb = F2::dup(-a.inv_sqrt_bc2 * 0x1p-50f), eps = F2::dup(a.eps), lr = F2::dup(a.step_size * 0x1p-64f);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int j = 4 * h + k;
                        const F2 den = fma2(neg_sqrt2(mul2(vh[j], F2::dup(-0x1p100f))), nisb, eps);
                        const F2 nq = neg_div2(mul2(mh[j], F2::dup(0x1p64f)), den);
                        F2 pj = F2::pack(p[2 * k], p[2 * k + 1]);
                        pj = fma2(lr, nq, DECAY ? mul2(pj, F2::dup(a.decay)) : pj);
                        p[2 * k] = pj.lo();
                        p[2 * k + 1] = pj.hi();
                    }
                    all &= store8(h, p);
                }
                if (__any_sync(0xffffffffu, moves && (~all & 0x20002000u) != 0u)) {
                    uint32_t least = 0x7FFFu;                         // of the patterns stored, signs off
#pragma unroll 1
                    for (int i = 0; i < EPT16; ++i)
                        least = min(least, reinterpret_cast<const unsigned short*>(pt)[EPT16 * tid + i] & 0x7FFFu);
                    exact = !__any_sync(0xffffffffu, moves && least < 0x1800u);        // 2^-79: no result below 2^-80 was rounded up to it
                }
            }
            if (!exact) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float p[8];
                    load8(h, p);
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const int i = 8 * h + k;
                        const float den = __fmaf_rn(__fsqrt_rn(vh_at(i)), a.inv_sqrt_bc2, a.eps);
                        p[k] = __fmaf_rn(-a.step_size, __fdiv_rn(mh_at(i), den), DECAY ? p[k] * a.decay : p[k]);
                    }
                    store8(h, p);
                }
            }
        }
    }

    // ---- (C) first moment: block scale, nearest level (Eq. 1), see fast_tile ----
    if constexpr (G != 128) mx_m = group_max16<G>(mx_m);
    uint32_t om[BM == 8 ? 4 : 2] = {};                            // eight codes per word, 8-bit: four
    const float dm_new = __uint_as_float(mx_m);
    const float inv_m = __frcp_rn(at_least_tiny(mx_m));
    // code = number of midpoints below r, each comparison as the saturation of (r - mid) * 2^100 on the FMA
    // pipe (exactly 0 or 1, see fast_tile).  The codes of elements 2j and 2j + 1 are accumulated side by side
    // in one pair of binary32 (eight 2- or 3-bit codes per pair, at most 21 bits each: exact).
    constexpr float BIG = 0x1p100f;
    const float n0 = BM == 8 ? 0.0f : -s_mid[0] * BIG, n1 = BM == 8 ? 0.0f : -s_mid[1] * BIG, n2 = BM == 8 ? 0.0f : -s_mid[2] * BIG;
    float n3[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if constexpr (BM == 3) {
#pragma unroll
        for (int k = 0; k < 4; ++k) n3[k] = -s_mid[3 + k] * BIG;
    }
    // 4-bit: the same comparisons in two levels of three: mid[3], mid[7], mid[11] give the quarter s of
    // the codebook, the three midpoints inside it come from a table row addressed by s (s_mid4, scaled
    // like n0..n2); code = 4 s + their count.  Four codes (12 bits each half) per accumulator.
    float nq[3] = {0.0f, 0.0f, 0.0f};
    if constexpr (BM == 4) {
        nq[0] = -s_mid[3] * BIG; nq[1] = -s_mid[7] * BIG; nq[2] = -s_mid[11] * BIG;
    }
    constexpr int CPA = BM == 4 ? 4 : 8;                          // codes per accumulator
    F2 omf[EPT16 / CPA];
#pragma unroll
    for (int k = 0; k < EPT16 / CPA; ++k) omf[k] = F2::dup(0.0f);
    const F2 inv_m2 = F2::dup(inv_m);
    auto quant_m = [&](int j) {                                   // call with j = 7, 6, ..., 0
        const F2 r = mul2(mh[j], inv_m2);
        if constexpr (BM == 8) {
            // midpoints below the cell of r, plus one if r is above the cell's own
            uint32_t q0 = cell8_m(s.lut_m, r.lo()), q1 = cell8_m(s.lut_m, r.hi());
            q0 += r.lo() > s_mid[q0] ? 1u : 0u;
            q1 += r.hi() > s_mid[q1] ? 1u : 0u;
            const uint32_t two = __byte_perm(q0, q1, 0x0040u);
            om[j >> 1] = (j & 1) ? two : __byte_perm(two, om[j >> 1], 0x5410u);
            return;
        }
        F2& acc = omf[2 * j / CPA];
        const F2 up = F2::dup((float)(KM * KM));
        auto step = [&](float n) {
            return F2::pack(__saturatef(__fmaf_rn(r.lo(), BIG, n)), __saturatef(__fmaf_rn(r.hi(), BIG, n)));
        };
        if constexpr (BM <= 3) {
            acc = fma2(acc, up, step(n0));
            acc = add2(acc, step(n1));
            acc = add2(acc, step(n2));
            if constexpr (BM == 3) {
#pragma unroll
                for (int k = 0; k < 4; ++k) acc = add2(acc, step(n3[k]));
            }
        } else {
            const F2 c0 = step(nq[0]), c1 = step(nq[1]), c2 = step(nq[2]);
            // 2^23 + 16 s: the low bits of the pattern are the byte offset of row s
            const F2 sq = add2(add2(c0, c1), c2);
            const F2 t = fma2(sq, F2::dup(16.0f), F2::dup(8388608.0f));
            auto row_at = [&](float o) {
                return *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(s_mid4) + (__float_as_uint(o) & 0x30u));
            };
            const float4 ra = row_at(t.lo()), rb = row_at(t.hi());
            auto inner = [&](float na, float nb) {
                return F2::pack(__saturatef(__fmaf_rn(r.lo(), BIG, na)), __saturatef(__fmaf_rn(r.hi(), BIG, nb)));
            };
            acc = fma2(acc, up, fma2(sq, F2::dup(4.0f), inner(ra.x, rb.x)));
            acc = add2(acc, inner(ra.y, rb.y));
            acc = add2(acc, inner(ra.z, rb.z));
        }
    };
    // 8-bit codes of a block with a NaN or infinite scale: every comparison with a NaN is false (code 0), zeros are code
    // 127 (the cell tables know no NaN)
    auto special_m8 = [&]() {
#pragma unroll
        for (int i = 0; i < 4; ++i) om[BM == 8 ? i : 0] = 0u;
#pragma unroll
        for (int i = EPT16 - 1; i >= 0; --i) {
            const float r = mh_at(i) * inv_m;
            om[BM == 8 ? i >> 2 : 0] = (om[BM == 8 ? i >> 2 : 0] << 8) + (r == r ? 127u : 0u);
        }
    };
    auto quant_m_done = [&]() {
        if constexpr (BM == 8) {
            if (!(dm_new < __int_as_float(0x7f800000))) special_m8();
            if (dm_new < TINY) {
#pragma unroll
                for (int i = 0; i < 4; ++i) om[BM == 8 ? i : 0] = 0u;
            }
            return;
        }
        uint32_t half[EPT16 / CPA];
#pragma unroll
        for (int k = 0; k < EPT16 / CPA; ++k) half[k] = (uint32_t)__fmaf_rn(omf[k].hi(), (float)KM, omf[k].lo());
        if constexpr (BM <= 3) {
            om[0] = half[0];
            om[1] = half[1];
        } else {
            om[0] = half[0] | (half[1] << 16);
            om[1] = half[2] | (half[3] << 16);
        }
        if (dm_new < TINY) { om[0] = 0; om[1] = 0; }             // vanishing block: all codes 0
    };
    if (round_m) {
        // Eq. 5: q = number of levels y_1 .. y_{K-2} that r reaches (the lower end of its bracket), plus
        // one when the element's draw u (Philox purpose 1) falls below (r - y_q) / (y_{q+1} - y_q).
        // "r >= y" is counted on the FMA pipe as the saturation of t - y'*2^100 with t = r*2^100 and y'
        // the binary32 just below y (exactly 0 or 1: two distinct binary32 near a level differ by far
        // more than 2^-100); the level 0 as the saturation of t*2^100 + 1 (t = +-0: 1; else |t*2^100| >=
        // 2^51, or infinite).  NaN counts nowhere and is never below anything: code 0.  In pairs where a packed
        // operation exists (4/2 bit, 2^27 elements: 601 -> 582 us).
        uint32_t wm[8];
        {
            uint32_t w4[4];
            draw8(sw, 1u, w4);
#pragma unroll
            for (int i = 0; i < 4; ++i) wm[i] = w4[i];
            draw8(sw ^ 1u, 1u, w4);
#pragma unroll
            for (int i = 0; i < 4; ++i) wm[4 + i] = w4[i];
        }
        constexpr int Z = KM / 2 - 1;                             // index of the level 0
        float nb[BM >= 4 ? 3 : KM - 2];                           // nb[j - 1]: threshold of level j, BM == 4: of levels 4, 8, 12
        if constexpr (BM == 8) {
        } else if constexpr (BM == 4) {
            const float4 c4 = s_br[4];
            nb[0] = c4.x; nb[1] = c4.y; nb[2] = c4.z;
        } else {
            const float4 ba = s_br[0];
            nb[0] = ba.x; nb[1] = ba.y;
            if constexpr (BM == 3) {
                const float4 bb = s_br[1];
                nb[2] = ba.z; nb[3] = ba.w; nb[4] = bb.x; nb[5] = bb.y;
            }
        }
        F2 accm[EPT16 / CPA];                                     // codes of elements 2j and 2j + 1 side by side, as above
#pragma unroll
        for (int k = 0; k < EPT16 / CPA; ++k) accm[k] = F2::dup(0.0f);
#pragma unroll
        for (int j = EPT16 / 2 - 1; j >= 0; --j) {
            float d[2];                                           // the 16-bit draws of elements 2j, 2j + 1 as binary32
            halves_to_float(wm[j], d[0], d[1]);
            if constexpr (BM == 8) {
#pragma unroll
                for (int e = 1; e >= 0; --e) {
                    // levels reached below the cell of r, plus the cell's own
                    const float re = mh_at(2 * j + e) * inv_m;
                    uint32_t q = cell8_m(s.lut_m, re);
                    q += re >= s_yg[q + 1].x ? 1u : 0u;
                    const float2 yg = s_yg[q];
                    const float frac = (re - yg.x) * yg.y;
                    q += d[e] < frac * 65536.0f ? 1u : 0u;
                    om[j >> 1] = (om[j >> 1] << 8) + q;
                }
                continue;
            }
            const F2 r = mul2(mh[j], inv_m2), t = mul2(r, F2::dup(BIG));
            auto reached = [&](float na, float nb2) { return F2::pack(__saturatef(t.lo() + na), __saturatef(t.hi() + nb2)); };
            F2 qf;
            if constexpr (BM == 4) {
                const F2 sq = add2(add2(reached(nb[0], nb[0]), reached(nb[1], nb[1])), reached(nb[2], nb[2]));
                const F2 o = fma2(sq, F2::dup(16.0f), F2::dup(8388608.0f));
                // row s: thresholds of levels 4s+1, 4s+2, 4s+3 (.w: the factor of t for the third,
                // 2^100 where that level is 0)
                auto row_at = [&](float x) {
                    return *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(s_br) + (__float_as_uint(x) & 0x30u));
                };
                const float4 ra = row_at(o.lo()), rb = row_at(o.hi());
                qf = fma2(sq, F2::dup(4.0f), reached(ra.x, rb.x));
                qf = add2(qf, reached(ra.y, rb.y));
                qf = add2(qf, F2::pack(__saturatef(__fmaf_rn(t.lo(), ra.w, ra.z)), __saturatef(__fmaf_rn(t.hi(), rb.w, rb.z))));
            } else {
                qf = F2::pack(__saturatef(__fmaf_rn(t.lo(), BIG, 1.0f)), __saturatef(__fmaf_rn(t.hi(), BIG, 1.0f)));   // level 0
#pragma unroll
                for (int l = 1; l <= KM - 2; ++l)
                    if (l != Z) qf = add2(qf, reached(nb[l - 1], nb[l - 1]));
            }
            // the bracket's lower level (negated) and the reciprocal of its width, from the pair table
            const F2 o8 = fma2(qf, F2::dup(8.0f), F2::dup(8388608.0f));
            auto pair_at = [&](float x) {
                return *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(s_yg) + (__float_as_uint(x) & 0xF8u));
            };
            const float2 ya = pair_at(o8.lo()), yb = pair_at(o8.hi());
            const F2 f = mul2(mul2(add2(r, F2::pack(ya.x, yb.x)), F2::pack(ya.y, yb.y)), F2::dup(65536.0f));
            const F2 code = add2(qf, F2::pack(d[0] < f.lo() ? 1.0f : 0.0f, d[1] < f.hi() ? 1.0f : 0.0f));     // u = d / 2^16 < frac
            accm[2 * j / CPA] = fma2(accm[2 * j / CPA], F2::dup((float)(KM * KM)), code);
        }
        uint32_t half[EPT16 / CPA];
#pragma unroll
        for (int k = 0; k < EPT16 / CPA; ++k) half[k] = (uint32_t)__fmaf_rn(accm[k].hi(), (float)KM, accm[k].lo());
        if constexpr (BM == 8) {
            // (an infinite scale: r is +-0, level 127 exactly, or NaN)
            if (!(dm_new < __int_as_float(0x7f800000))) special_m8();
        } else if constexpr (BM == 4) {
            om[0] = half[0] | (half[1] << 16);
            om[1] = half[EPT16 / CPA - 2] | (half[EPT16 / CPA - 1] << 16);
        } else {
            om[0] = half[0];
            om[1] = half[1];
        }
        if (dm_new < TINY) {                                      // vanishing block: all codes 0
#pragma unroll
            for (int i = 0; i < (BM == 8 ? 4 : 2); ++i) om[i] = 0u;
        }
    }

    // ---- (D) second moment: block scale and the p-quantile ----
    if constexpr (G != 128) mx_v = group_max16<G>(mx_v);
    uint32_t x_p;
    uint32_t w[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};             // 16 halfwords: the draws of the 16 elements
    if (fixed_base) {
        // every block keeps the given base: no quantile to find
        if (!round_m) {
#pragma unroll
            for (int j = EPT16 / 2 - 1; j >= 0; --j) quant_m(j);
            quant_m_done();
        }
        x_p = 0u;
    } else {
        // the keys are sorted with the first moment's FMA-pipe work issued between the ALU-pipe exchanges
        if constexpr (G == 4) {
            uint32_t key[EPT16];
#pragma unroll
            for (int i = 0; i < EPT16; ++i) key[i] = __float_as_uint(vh_at(i));
#pragma unroll
            for (int k = 0; k < 62; ++k) {
                cswap(key[SORT16_PAIRS[k][0]], key[SORT16_PAIRS[k][1]]);
                if (!round_m && ((k & 7) == 7 || k == 61)) quant_m(7 - (k >> 3));
            }
            cswap(key[13], key[14]);
            if (!round_m) quant_m_done();
            x_p = select_pops4(key, a.k_full, &s.sort[0][tid], lane);
        } else if constexpr (G == 128) {
            if (!round_m) {
#pragma unroll
                for (int j = EPT16 / 2 - 1; j >= 0; --j) quant_m(j);
                quant_m_done();
            }
            uint32_t key[EPT16];
#pragma unroll
            for (int i = 0; i < EPT16; ++i) key[i] = __float_as_uint(vh_at(i));
            x_p = select_cta16(key, a.k_full, s.cta(), mn_v, mx_v, tid);
        } else {
            uint32_t l[4][4];
#pragma unroll
            for (int i = 0; i < EPT16; ++i) l[i >> 2][i & 3] = __float_as_uint(vh_at(i));
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                cswap(l[q][0], l[q][1]); cswap(l[q][2], l[q][3]);
                if (!round_m) quant_m(7 - 2 * q);
                cswap(l[q][0], l[q][2]); cswap(l[q][1], l[q][3]);
                if (!round_m) quant_m(6 - 2 * q);
                cswap(l[q][1], l[q][2]);
            }
            if (!round_m) quant_m_done();
            x_p = select_rank16<G, G == 16 ? 3 : 2>(l, a.k_full, lane, (uint32_t)a.only_partial);
        }
    }

    // ---- (E) per-block scalars by the first warp; the next tile's copies start meanwhile ----
    auto draw = [&]() {
        if (round_v) {
            uint32_t w4[4];
            draw8(sw, 0u, w4);
#pragma unroll
            for (int i = 0; i < 4; ++i) w[i] = w4[i];
            draw8(sw ^ 1u, 0u, w4);
#pragma unroll
            for (int i = 0; i < 4; ++i) w[4 + i] = w4[i];
        }
    };
    // (a block of 2048: the other warps draw while the first one selects)
    if (G == 128 && warp != 0) draw();
    if (gl == 0) s.xin[grp] = make_uint4(mx_m, mx_v, x_p, 0u);
    bar_sync16(1);
    // every thread has read what it needs from the stage
    if (tid == 32) produce_tile16<BM, BV, PBF, G, MODES>(a, s, s.desc[(fill + 1u) & 1u]);
    if (tid < NG) block_scalars16<KV>(a, s, jb_tile, tid, fixed_base, vtab);
    // meanwhile every thread draws: Philox4x32-10 on the counters of its two groups of eight elements,
    // (ctr, step, 4 * stream) and (ctr + 1, ...), in its own order.  (Between the selection's rounds, where the draws
    // once hid the shuffles' latency, they gain nothing with 28 to 32 resident warps; here they fill the wait for
    // the first warp: bf16 parameters 536 -> 528 us, 4/4 bit 407 -> 402 us on 2^27 elements.)
    if (G != 128) draw();
    bar_sync16(2);
    if (G == 128 && warp == 0) draw();
    const float4 sc = s.xout[grp];

    // second moment: Eq. 6, see fast_tile
    uint32_t ov[BV == 8 ? 4 : 2];
    if (vtab) {
        // Eq. 1 on the fixed codebook: code = number of midpoints below r, counted like the first
        // moment's (saturated multiply-adds, exactly 0 or 1 each: r and a midpoint, if they differ at all,
        // differ by far more than 2^-100, the smallest midpoint of these codebooks being about 1e-4)
        const float inv = sc.y;
        if constexpr (BV == 8) {
            // (a NaN falls into the first cell, as a zero does: code 0)
            const typename Shared::Codebook8& cb = s.v8();
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                uint32_t q[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float r = vh_at(4 * k + i) * inv;
                    q[i] = cell8_v(cb.lut, r);
                    q[i] += r > cb.mid[q[i]] ? 1u : 0u;
                }
                ov[k] = pack8(q[0], q[1], q[2], q[3]);
            }
        } else if constexpr (BV <= 3) {
            const float4 na = s_nv[0], nb = s_nv[1];
            float acc[2] = {0.0f, 0.0f};                         // eight codes, at most 24 bits: exact
#pragma unroll
            for (int i = EPT16 - 1; i >= 0; --i) {
                const float r = vh_at(i) * inv;
                float& c = acc[i >> 3];
                c = __fmaf_rn(c, (float)KV, __saturatef(__fmaf_rn(r, BIG, na.x)));
                c += __saturatef(__fmaf_rn(r, BIG, na.y));
                c += __saturatef(__fmaf_rn(r, BIG, na.z));
                if constexpr (BV == 3) {
                    c += __saturatef(__fmaf_rn(r, BIG, na.w));
                    c += __saturatef(__fmaf_rn(r, BIG, nb.x));
                    c += __saturatef(__fmaf_rn(r, BIG, nb.y));
                    c += __saturatef(__fmaf_rn(r, BIG, nb.z));
                }
            }
            ov[0] = (uint32_t)acc[0];
            ov[1] = (uint32_t)acc[1];
        } else {
            // sixteen levels in two steps of three comparisons, as for 4-bit first moments: row 3 holds
            // the midpoints 3, 7, 11, rows 4..7 the three midpoints inside each quarter
            const float4 nq4 = s_nv[3];
            float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};            // four codes each
#pragma unroll
            for (int i = EPT16 - 1; i >= 0; --i) {
                const float r = vh_at(i) * inv;
                const float c0 = __saturatef(__fmaf_rn(r, BIG, nq4.x));
                const float c1 = __saturatef(__fmaf_rn(r, BIG, nq4.y));
                const float c2 = __saturatef(__fmaf_rn(r, BIG, nq4.z));
                const float t = __fmaf_rn(c2, 16.0f, __fmaf_rn(c1, 16.0f, __fmaf_rn(c0, 16.0f, 8388608.0f)));
                const float4 row = *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(s_nv + 4) + (__float_as_uint(t) & 0x30u));
                float code = __fmaf_rn((c0 + c1) + c2, 4.0f, __saturatef(__fmaf_rn(r, BIG, row.x)));
                code += __saturatef(__fmaf_rn(r, BIG, row.y));
                code += __saturatef(__fmaf_rn(r, BIG, row.z));
                acc[i >> 2] = __fmaf_rn(acc[i >> 2], 16.0f, code);
            }
            ov[0] = (uint32_t)acc[0] | ((uint32_t)acc[1] << 16);
            ov[1] = (uint32_t)acc[2] | ((uint32_t)acc[3] << 16);
        }
        if (sc.x != 0.0f) {                                       // vanishing block: all codes 0
#pragma unroll
            for (int i = 0; i < (BV == 8 ? 4 : 2); ++i) ov[i] = 0u;
        }
    } else {
        const float inv = sc.y, il = sc.z, lim = sc.w;
        constexpr float KM1 = (float)(KV - 1);
        constexpr float MAGIC = 12582912.0f;
        const float ils = il * (1.0f / KM1);
        // xi = (d + 1/2) / 2^16 - 1/2 (exact), scaled like t; zero without the dither
        const F2 xs1 = F2::dup(round_v ? (float)(0x1p-16 / (KV - 1)) : 0.0f);
        const F2 xs0 = F2::dup(round_v ? (float)((-0.5 + 0x1p-17) / (KV - 1)) : 0.0f);
        const F2 inv2 = F2::dup(inv);
        // codes of elements 2j and 2j + 1 side by side in one pair of binary32, as for the first moment
        constexpr int CPA = BV >= 4 ? 4 : 8;
        float worst = 0.0f;
        F2 acc[EPT16 / CPA];
#pragma unroll
        for (int k = 0; k < EPT16 / CPA; ++k) acc[k] = F2::dup(0.0f);
#pragma unroll
        for (int j = EPT16 / 2 - 1; j >= 0; --j) {
            float d0, d1;                                         // the 16-bit draws of elements 2j, 2j + 1 as binary32
            halves_to_float(w[j], d0, d1);
            const F2 x = fma2(F2::pack(d0, d1), xs1, xs0);
            const F2 r = mul2(vh[j], inv2);
            const F2 ts = F2::pack(__saturatef(__fmaf_rn(lg2_approx(r.lo()), ils, x.lo())),
                                   __saturatef(__fmaf_rn(lg2_approx(r.hi()), ils, x.hi())));
            const F2 u = fma2(ts, F2::dup(KM1), F2::dup(MAGIC));  // the codes, rounded, in the low bits
            const F2 q = add2(u, F2::dup(-MAGIC));
            const F2 off = fma2(ts, F2::dup(-KM1), q);            // their distance from what was rounded
            worst = fmaxf(fmaxf(worst, fabsf(off.lo())), fabsf(off.hi()));
            if constexpr (BV == 8) {                              // (a byte each)
                const uint32_t two = __byte_perm(__float_as_uint(u.lo()), __float_as_uint(u.hi()), 0x0040u);
                ov[j >> 1] = (j & 1) ? two : __byte_perm(two, ov[j >> 1], 0x5410u);
            } else {
                acc[2 * j / CPA] = fma2(acc[2 * j / CPA], F2::dup((float)(KV * KV)), q);
            }
        }
        if constexpr (BV != 8) {
            uint32_t half[EPT16 / CPA];
#pragma unroll
            for (int k = 0; k < EPT16 / CPA; ++k) half[k] = (uint32_t)__fmaf_rn(acc[k].hi(), (float)KV, acc[k].lo());
            ov[0] = BV <= 3 ? half[0] : half[0] | (half[1] << 16);
            ov[1] = BV <= 3 ? half[1] : half[EPT16 / CPA - 2] | (half[EPT16 / CPA - 1] << 16);
        }
        if (__any_sync(0xffffffffu, worst > lim)) {
            // too close to a rounding boundary for the approximate logarithm somewhere in the warp:
            // the exact sequence for all sixteen
            const float x1 = round_v ? 0x1p-16f : 0.0f, x0 = round_v ? -0.5f + 0x1p-17f : 0.0f;
#pragma unroll
            for (int i = 0; i < (BV == 8 ? 4 : 2); ++i) ov[i] = 0u;
#pragma unroll
            for (int j = EPT16 / 2 - 1; j >= 0; --j) {
                float d[2];
                halves_to_float(w[j], d[0], d[1]);
#pragma unroll
                for (int e = 1; e >= 0; --e) {
                    const int i = 2 * j + e;
                    const float r = vh_at(i) * inv;
                    uint32_t q = KV - 1;
                    if (!(r < TINY)) {
                        float t = __fmaf_rn(log2_sp(r), il, __fmaf_rn(d[e], x1, x0));
                        t = fminf(fmaxf(t, 0.0f), KM1);
                        q = (uint32_t)__float2int_rn(t);
                    }
                    uint32_t& o = ov[BV == 8 ? i >> 2 : i >> 3];
                    o = (o << BV) + q;
                }
            }
        }
        if (sc.x != 0.0f) {                                       // vanishing block: all codes 0
#pragma unroll
            for (int i = 0; i < (BV == 8 ? 4 : 2); ++i) ov[i] = 0u;
        }
    }

    // ---- store the codes ----
    uint32_t om_e[BM == 8 ? 4 : 2], ov_e[BV == 8 ? 4 : 2];        // back to element order
#pragma unroll
    for (int i = 0; i < (BM == 8 ? 4 : 2); ++i) om_e[i] = sw ? om[i ^ (BM == 8 ? 2 : 1)] : om[i];
#pragma unroll
    for (int i = 0; i < (BV == 8 ? 4 : 2); ++i) ov_e[i] = sw ? ov[i ^ (BV == 8 ? 2 : 1)] : ov[i];
    store_codes16<BM>(a.codes_m + jb_tile * (2 * G * BM), s.cout[0][BM == 3 ? warp : 0], tid, om_e);
    store_codes16<BV>(a.codes_v + jb_tile * (2 * G * BV), s.cout[(BM == 3 && BV == 3) ? 1 : 0][BV == 3 ? warp : 0], tid, ov_e);
}

template <int BM, int BV, bool PBF, int G, int MODES, bool SR>
__global__ void __launch_bounds__(CTA16, ctas16<BM, BV, G, MODES>()) solo_step_fast16_kernel(const __grid_constant__ StepArgs a) {
    constexpr int KM = 1 << BM;
    constexpr bool EXT = MODES >= 2, EQ5 = MODES == 2 || MODES == 3;
    using Shared = Fast16Shared<BM, BV, PBF, G>;
    extern __shared__ __align__(16) unsigned char fast16_smem[];
    Shared& s = *reinterpret_cast<Shared*>(fast16_smem);
    __shared__ float s_y[KM];
    __shared__ float s_mid[KM];
    __shared__ float2 s_yg[EQ5 ? KM : 1];                    // Eq. 5: see the set-up below
    __shared__ float4 s_br[EQ5 ? (BM == 4 ? 5 : 2) : 1];
    __shared__ float s_yv[(MODES == 2 || MODES == 4) && BV != 8 ? 1 << BV : 1];               // baseline second-moment codebook: its levels,
    __shared__ float4 s_nv[MODES == 2 || MODES == 4 ? 8 : 1];                     // its midpoints times -2^100 (rows as the tile function reads them)
    __shared__ float4 s_mid4[4];             // 4-bit first moments: per quarter of the codebook, its three inner midpoints times -2^100
    const int tid = threadIdx.x;
    pdl_wait();
    pdl_release();
    for (int i = tid; i < KM; i += CTA16) {
        s_y[i] = a.tables[i];
        s_mid[i] = i < KM - 1 ? a.tables[KM + i] : __int_as_float(0x7f800000);
    }
    if constexpr (BM == 8) {
        const uint4* const src = reinterpret_cast<const uint4*>(g_lut8_m[MODES == 3 || (MODES == 2 && a.round_m) ? 1 : 0].q);
        for (int i = tid; i < LUT8_M_BYTES / 16; i += CTA16) reinterpret_cast<uint4*>(s.lut_m)[i] = src[i];
    }
    if (BM == 4 && tid < 4)
        s_mid4[tid] = make_float4(-a.tables[KM + 4 * tid] * 0x1p100f, -a.tables[KM + 4 * tid + 1] * 0x1p100f,
                                  -a.tables[KM + 4 * tid + 2] * 0x1p100f, 0.0f);
    if constexpr (EXT) {
        if (MODES == 3 || (MODES == 2 && a.round_m)) {
            // Eq. 5: per level q <= K-2 the pair (y_q, 1 / (y_{q+1} - y_q)); thresholds of "r >= y_j" as
            // -y'_j * 2^100, y'_j the binary32 just below y_j (rows as the tile function reads them:
            // 2- and 3-bit, levels 1..6 in rows 0, 1; 4-bit, row s = levels 4s+1..4s+3 and row 4 = levels
            // 4, 8, 12).  The level 0 is compared another way; a level past K-2 gets -infinity: never reached.
            const float* const yk = a.tables;
            if constexpr (BM == 8) {                              // (the pair past the last bracket is never reached)
                for (int i = tid; i < KM; i += CTA16)
                    s_yg[i] = i < KM - 1 ? make_float2(yk[i], a.tables[2 * KM - 1 + i]) : make_float2(__int_as_float(0x7f800000), 0.0f);
            }
            auto below = [&](int j) {
                const float y = yk[j];
                return -__uint_as_float(__float_as_uint(y) + (y < 0.0f ? 1u : 0xFFFFFFFFu)) * 0x1p100f;
            };
            if (BM != 8 && tid < KM - 1) s_yg[tid] = make_float2(-yk[tid], a.tables[2 * KM - 1 + tid]);
            if (BM <= 3 && tid < 2) {
                float t4[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int j = 4 * tid + k + 1;
                    t4[k] = j <= KM - 2 && j != KM / 2 - 1 ? below(j) : 0.0f;
                }
                s_br[tid] = make_float4(t4[0], t4[1], t4[2], t4[3]);
            }
            if (BM == 4 && tid < 4) {
                const int j = 4 * tid + 1;
                const bool zero3 = j + 2 == KM / 2 - 1;            // the row's third level is the level 0
                s_br[tid] = make_float4(below(j), below(j + 1),
                                        zero3 ? 1.0f : j + 2 <= KM - 2 ? below(j + 2) : -__int_as_float(0x7f800000),
                                        zero3 ? 0x1p100f : 1.0f);
            }
            if (BM == 4 && tid == 4) s_br[4] = make_float4(below(4), below(8), below(12), 0.0f);
        }
        if (MODES == 4 || (MODES == 2 && a.tables_v != nullptr)) {
            constexpr int KV = 1 << BV;
            const float* const midv = a.tables_v + KV;            // KV - 1 midpoints
            if constexpr (BV == 8) {
                typename Shared::Codebook8& cb = s.v8();
                for (int i = tid; i < KV; i += CTA16) {
                    cb.y[i] = a.tables_v[i];
                    cb.mid[i] = i < KV - 1 ? midv[i] : __int_as_float(0x7f800000);
                }
                const uint4* const src = reinterpret_cast<const uint4*>(g_lut8_v[a.v_kind - 1].q);
                for (int i = tid; i < LUT8_V_BYTES / 16; i += CTA16) reinterpret_cast<uint4*>(cb.lut)[i] = src[i];
            } else if (tid < KV) {
                s_yv[tid] = a.tables_v[tid];
            }
            if (BV != 8 && tid < 2) {                                         // rows 0, 1: midpoints 0..7 (rows of 3 or 7 are padded)
                float m4[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) m4[k] = 4 * tid + k < KV - 1 ? -midv[4 * tid + k] * 0x1p100f : 0.0f;
                s_nv[tid] = make_float4(m4[0], m4[1], m4[2], m4[3]);
            }
            if (BV == 4 && tid == 3)
                s_nv[3] = make_float4(-midv[3] * 0x1p100f, -midv[7] * 0x1p100f, -midv[11] * 0x1p100f, 0.0f);
            if (BV == 4 && tid >= 4 && tid < 8)
                s_nv[tid] = make_float4(-midv[4 * (tid - 4)] * 0x1p100f, -midv[4 * (tid - 4) + 1] * 0x1p100f,
                                        -midv[4 * (tid - 4) + 2] * 0x1p100f, 0.0f);
        }
    }
    if constexpr (G == 4) s.sort[15][tid] = KEY_MAX;              // never overwritten
    if constexpr (G == 128) {
        s.cta().hist[tid] = 0u;
        s.cta().hist[tid + CTA16] = 0u;
        if (tid == 0) s.cta().fill = 0u;
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s.mbar)) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s.mbar_steal)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    if (tid == 32) {
        s.walk.phase = 0;
        s.walk.gave_up = s.walk.unanswered = false;
        s.walk.t_lo = s.walk.t_hi = -1;
        s.walk.tile = (int)a.tile_first + (int)blockIdx.x * a.share - 1;
        s.walk.tile_end = (int)min((int64_t)s.walk.tile + 1 + a.share, a.total_tiles);
        s.walk.tensor = (a.num_tensors > 1 ? find_tensor(a.tile_start, a.num_tensors, s.walk.tile + 1) : 0) - 1;
        steal_request(s);
        produce_tile16<BM, BV, PBF, G, MODES>(a, s, s.desc[0]);
    }
    __syncthreads();

    bool failed = false;          // this thread waited in vain for a copy: it stores nothing
    uint32_t fill = 0;            // number of the tile, and of the copy it waits for
    const bool decay = a.decay != 1.0f;
    for (; s.desc[fill & 1u].valid; ++fill) {
        if (decay)
            fast16_tile<BM, BV, PBF, G, true, MODES, SR>(a, s, s_y, s_mid, s_mid4, s_yv, s_nv, s_yg, s_br, fill, failed);
        else
            fast16_tile<BM, BV, PBF, G, false, MODES, SR>(a, s, s_y, s_mid, s_mid4, s_yv, s_nv, s_yg, s_br, fill, failed);
    }
    // A thread that gave up on a copy waits once more, again bounded, for the last one that was issued,
    // so that no copy is still writing to the stage when the CTA's shared memory is released; likewise for an answer.
    if (failed && fill > 0) mbar_wait(smem_u32(&s.mbar), (fill - 1u) & 1u);
    if (tid == 32 && s.walk.unanswered) mbar_wait(smem_u32(&s.mbar_steal), s.walk.phase);
}

}  // namespace solo
