// Cell tables of the 8-bit codebooks (Appendix A), computed by the compiler.
//
// The nearest of 256 levels is a count of midpoints, an eight-step search with a dependent shared-memory look-up
// per step.  Here the binary32 number line is cut into cells of equal exponent and leading mantissa bits, narrow
// enough that no cell holds more than one midpoint: a cell's byte is the number of midpoints below the cell, and
// one comparison with the next midpoint gives the code exactly.
#pragma once

#include <stdint.h>

namespace solo {

constexpr double pow2c(int e) { return e < 0 ? 0.5 * pow2c(e + 1) : e > 0 ? 2.0 * pow2c(e - 1) : 1.0; }

// Levels of the 8-bit codebooks, the same arithmetic as the tables a state carries: the midpoint of fraction cell j
// of [0.1, 1] scaled by 10^-E, as one binary64 division.
constexpr float de8_level(int E, int F, int j) {
    double ten = 10.0;
    for (int i = 0; i < E; ++i) ten *= 10.0;
    const double two = (double)(1 << (F + 1));
    return (float)((two + 9.0 * (double)(2 * j + 1)) / (ten * two));
}

struct Levels8 {
    float y[256];
};
constexpr Levels8 signed_de8() {
    Levels8 t{};
    int n = 0;
    for (int E = 6; E >= 0; --E)                              // positive levels 128..254, smallest decade first
        for (int j = 0; j < (1 << (6 - E)); ++j) t.y[128 + n++] = de8_level(E, 6 - E, j);
    for (int k = 0; k < 127; ++k) t.y[k] = -t.y[254 - k];
    t.y[127] = 0.0f;
    t.y[255] = 1.0f;
    return t;
}
constexpr Levels8 unsigned8(int kind) {                       // 1 dynamic exponent, 2 linear, 3 linear without zero
    Levels8 t{};
    if (kind == 1) {
        int n = 1;
        for (int E = 6; E >= 0; --E)
            for (int j = 0; j < (1 << (7 - E)); ++j) t.y[n++] = de8_level(E, 7 - E, j);
        t.y[0] = 0.0f;
        t.y[255] = 1.0f;
    } else {
        for (int k = 0; k < 256; ++k) t.y[k] = kind == 2 ? (float)((double)k / 255.0) : (float)((double)(k + 1) / 256.0);
    }
    return t;
}

// Signed values |r| <= 1 (and one rounding above): six mantissa bits, magnitudes below 2^-22 in the first cell of
// their sign.  index(r) = pattern of max(|r|, 2^-22), for negative r with exponent bit 5 cleared, shifted right by
// 17, from LUT8_M_BASE on; cells of [1, 1 + 1/64) included.
constexpr int LUT8_M_OCTAVES = 22, LUT8_M_CELLS = LUT8_M_OCTAVES * 64 + 1;
constexpr uint32_t LUT8_M_BASE = (0x34800000u ^ 0x10000000u) >> 17;      // 2^-22, negative
constexpr int LUT8_M_POS = (int)((0x34800000u >> 17) - LUT8_M_BASE);     // first cell of the positive values
constexpr int LUT8_M_BYTES = (LUT8_M_POS + LUT8_M_CELLS + 15) / 16 * 16;
// Unsigned values: seven mantissa bits, values below 2^-23 in the first cell.
constexpr int LUT8_V_OCTAVES = 23, LUT8_V_CELLS = LUT8_V_OCTAVES * 128 + 1;
constexpr uint32_t LUT8_V_BASE = 0x34000000u >> 16;
constexpr int LUT8_V_BYTES = (LUT8_V_CELLS + 15) / 16 * 16;

template <int BYTES>
struct alignas(16) Lut8 {
    unsigned char q[BYTES];
    bool exact;                                               // no cell holds two thresholds
};

// thr[0..n): ascending thresholds; a cell's byte is the number of them below every value of the cell.
constexpr Lut8<LUT8_M_BYTES> make_lut8_m(const float (&thr)[256], int n) {
    Lut8<LUT8_M_BYTES> t{};
    t.exact = true;
    int below = 0, upto = 0;
    for (int c = 0; c < LUT8_M_CELLS; ++c) {                  // positive cells [lo, hi), ascending
        const double step = pow2c(c / 64 - LUT8_M_OCTAVES) / 64.0;
        const double lo = step * (64 + c % 64), hi = lo + step;
        while (below < n && thr[below] < lo) ++below;
        upto = below;
        while (upto < n && thr[upto] < hi) ++upto;
        if (upto > below + 1) t.exact = false;
        t.q[LUT8_M_POS + c] = (unsigned char)below;
    }
    below = 0;
    for (int c = LUT8_M_CELLS - 1; c >= 0; --c) {             // negative cells (-hi, -lo], ascending
        const double step = pow2c(c / 64 - LUT8_M_OCTAVES) / 64.0;
        const double lo = step * (64 + c % 64), hi = lo + step;
        while (below < n && thr[below] <= -hi) ++below;
        upto = below;
        while (upto < n && thr[upto] <= -lo) ++upto;
        if (upto > below + 1) t.exact = false;
        t.q[c] = (unsigned char)below;
    }
    return t;
}
constexpr Lut8<LUT8_M_BYTES> lut8_m_nearest() {
    const Levels8 l = signed_de8();
    float mid[256] = {};
    for (int k = 0; k < 255; ++k) mid[k] = 0.5f * (l.y[k] + l.y[k + 1]);
    return make_lut8_m(mid, 255);
}
constexpr Lut8<LUT8_M_BYTES> lut8_m_bracket() {               // Eq. 5: levels 1..254 that are reached
    const Levels8 l = signed_de8();
    float thr[256] = {};
    for (int k = 1; k <= 254; ++k) thr[k - 1] = l.y[k];
    return make_lut8_m(thr, 254);
}
constexpr Lut8<LUT8_V_BYTES> lut8_v(int kind) {
    const Levels8 l = unsigned8(kind);
    Lut8<LUT8_V_BYTES> t{};
    t.exact = true;
    int below = 0, upto = 0;
    for (int c = 0; c < LUT8_V_CELLS; ++c) {
        const double step = pow2c(c / 128 - LUT8_V_OCTAVES) / 128.0;
        const double lo = step * (128 + c % 128), hi = lo + step;
        while (below < 255 && 0.5f * (l.y[below] + l.y[below + 1]) < lo) ++below;
        upto = below;
        while (upto < 255 && 0.5f * (l.y[upto] + l.y[upto + 1]) < hi) ++upto;
        if (upto > below + 1) t.exact = false;
        t.q[c] = (unsigned char)below;
    }
    return t;
}

static __device__ const Lut8<LUT8_M_BYTES> g_lut8_m[2] = {lut8_m_nearest(), lut8_m_bracket()};
static __device__ const Lut8<LUT8_V_BYTES> g_lut8_v[3] = {lut8_v(1), lut8_v(2), lut8_v(3)};
static_assert(lut8_m_nearest().exact && lut8_m_bracket().exact && lut8_v(1).exact && lut8_v(2).exact && lut8_v(3).exact,
              "cells narrower than the spacing of the thresholds");

}  // namespace solo
