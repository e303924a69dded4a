// On-chip pieces of the binary-polynomial product (cm_gf2.cu says what the
// transform is): basis conversions of packed bits and the levels of the
// additive transform on a tile in shared memory.  Every function is one
// thread's part of a phase; phases are separated by barriers in the kernels.
#pragma once
#include "gf2.cuh"

namespace cm {
namespace gf {

enum ConvKind : int { kConvA = 0, kConvB = 1, kConvBInv = 2 };

constexpr int kMinLg = 15;  // shortest and longest transform, log2 bits
constexpr int kMaxLg = 25;
// lengths with a second shape, last-pass tiles of 2^12 words, for few operands
constexpr int kFewMinLg = 22, kFewMaxLg = 24;
constexpr int kMaxLev = 18;  // levels of one pass

// One level of a pass over tiles.  A tile word address has NB bits: NFREE
// point / column bits below FMAX positions that end as the components x_0 ..
// of the field; the level's index bit sits at position p, and the elements
// have 2^f components (positions NFREE .. NFREE + f - 1).
struct Lev {
    uint32_t p, f, missing;
    uint32_t base[2];     // twiddle at point bits 0: operand a, operand b
    uint32_t pad[3];
    uint32_t lut[64];     // twiddle contribution of address bits 0..3 [0], 4..7 [16], 8..12 [32]
    uint32_t ext[16];     // of the point bits that number the tiles
    uint32_t lanes[32];   // of the point bits inside a word: component j's lane pattern
};

struct alignas(16) Pass {
    uint32_t nlev, npre;      // levels; those before the word bits change places with point bits
    uint32_t next;            // bits of the tile number
    uint32_t xp[5];           // address bit that changes places with word bit b
    uint32_t extpos[16];      // word-index bit of each bit of the tile number
    uint32_t glut[3][32];     // tile element number (5 bits each) -> word index in the array
    uint32_t alut[3][32];     // -> tile word address
    uint32_t xlut[2][16];     // number of a 32-word block (4 bits each) -> the address bits outside xp
    Lev lev[kMaxLev];
};

// Bank swizzle: a warp that skips one of the five low address bits reaches
// address bit 5 instead; flipping the bank where bit 5 is set keeps its 32
// words in 32 banks.
CM_HD uint32_t phys(uint32_t a) { return a ^ ((a & 32u) ? 31u : 0u); }

CM_HD uint32_t lut3(const uint32_t (*t)[32], uint32_t e) {
    return t[0][e & 31u] | t[1][(e >> 5) & 31u] | t[2][e >> 10];
}

// ---------------------------------------------------------------------------
// Conversion of 256 bits (8 words) to the novel basis: stages (top, sh), each
// adding the upper half of a block of 2^(top+1) bits, 2^sh higher, to the
// lower half.  kConvB is the stage's transposed inverse on the bit-reversed
// array (the wrapped terms stay in the lower half), kConvBInv undoes kConvB.
template <int TOP, int SH, int KIND>
CM_HD void conv_stage(uint32_t (&x)[8]) {
    constexpr int H = 1 << TOP, S = 1 << SH;
    if constexpr (TOP < 5) {
        constexpr uint32_t low = TOP == 0 ? 0x55555555u : TOP == 1 ? 0x33333333u : TOP == 2 ? 0x0F0F0F0Fu
                                 : TOP == 3 ? 0x00FF00FFu : 0x0000FFFFu;  // lower halves
        // positions H - S .. H - 1 of the lower halves
        constexpr uint32_t endlo = low & ~((low >> S) & low);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            uint32_t v = x[i];
            if (KIND == kConvA) v ^= (v & (endlo << H)) >> (H - S);
            if (KIND == kConvB) v ^= (v & endlo) >> (H - S);
            v ^= (((v & ~low) >> H) << S) & low;
            if (KIND == kConvBInv) v ^= (v & endlo) >> (H - S);
            x[i] = v;
        }
    } else {
        constexpr int HW = H / 32;
#pragma unroll
        for (int b = 0; b < 8; b += 2 * HW) {
            auto wrap = [&](int o) {  // low S bits of the half at o from its top S bits
                if constexpr (S < 32) x[o] ^= x[o + HW - 1] >> (32 - S);
                else {
                    uint32_t t[S / 32];
#pragma unroll
                    for (int i = 0; i < S / 32; ++i) t[i] = x[o + HW - S / 32 + i];
#pragma unroll
                    for (int i = 0; i < S / 32; ++i) x[o + i] ^= t[i];
                }
            };
            if (KIND == kConvA) wrap(b + HW);
            if (KIND == kConvB) wrap(b);
#pragma unroll
            for (int i = 0; i < HW; ++i) {
                if constexpr (S < 32) {
                    uint32_t t = x[b + HW + i] << S;
                    if (i > 0) t |= x[b + HW + i - 1] >> (32 - S);
                    x[b + i] ^= t;
                } else if (i >= S / 32) {
                    x[b + i] ^= x[b + HW + i - S / 32];
                }
            }
            if (KIND == kConvBInv) wrap(b);
        }
    }
}

template <int KIND>
CM_HD void conv8(uint32_t (&x)[8]) {
    if constexpr (KIND == kConvBInv) {
        conv_stage<1, 0, KIND>(x);
        conv_stage<3, 2, KIND>(x);
        conv_stage<2, 0, KIND>(x);
        conv_stage<3, 1, KIND>(x);
        conv_stage<5, 4, KIND>(x);
        conv_stage<7, 6, KIND>(x);
        conv_stage<6, 4, KIND>(x);
        conv_stage<7, 5, KIND>(x);
        conv_stage<4, 0, KIND>(x);
        conv_stage<5, 1, KIND>(x);
        conv_stage<6, 2, KIND>(x);
        conv_stage<7, 3, KIND>(x);
    } else {
        conv_stage<7, 3, KIND>(x);
        conv_stage<6, 2, KIND>(x);
        conv_stage<5, 1, KIND>(x);
        conv_stage<4, 0, KIND>(x);
        conv_stage<7, 5, KIND>(x);
        conv_stage<6, 4, KIND>(x);
        conv_stage<7, 6, KIND>(x);
        conv_stage<5, 4, KIND>(x);
        conv_stage<3, 1, KIND>(x);
        conv_stage<2, 0, KIND>(x);
        conv_stage<3, 2, KIND>(x);
        conv_stage<1, 0, KIND>(x);
    }
}

// Conversion stages above the first ones of a length: (block bit, shift bit)
// pairs in rows, in order for kConvA / kConvB.
struct Stages {
    int n;
    uint8_t top[16], sh[16];
};

// ---------------------------------------------------------------------------
// Levels.

// Tile word address of unit u of a level: u's bits over the address bits other
// than p and the components.
template <int NFREE>
CM_HD uint32_t unit_addr(uint32_t u, uint32_t p, uint32_t f) {
    if (p < (uint32_t)NFREE) {
        const uint32_t lo = u & ((1u << (NFREE - 1)) - 1u), hi = u >> (NFREE - 1);
        const uint32_t below = lo & ((1u << p) - 1u);
        return below | ((lo ^ below) << 1) | (hi << (NFREE + f));
    }
    const uint32_t lo = u & ((1u << NFREE) - 1u);
    uint32_t hi = u >> NFREE;
    const uint32_t q = p - NFREE - f;  // p's place among the positions above the components
    const uint32_t below = hi & ((1u << q) - 1u);
    hi = below | ((hi ^ below) << 1);
    return lo | (hi << (NFREE + f));
}

CM_HD uint32_t twiddle(const Lev &v, uint32_t base, uint32_t a) {
    return base ^ v.lut[a & 15u] ^ v.lut[16 + ((a >> 4) & 15u)] ^ v.lut[32 + (a >> 8)];
}

// Bit-sliced twiddle words of one unit: element e in every lane, plus the lane
// patterns of the point bits inside the word.
template <int F>
CM_HD void spread(const Lev &v, uint32_t e, bool lanes, uint32_t *t) {
#pragma unroll
    for (int j = 0; j < (1 << F); ++j) t[j] = (uint32_t)((int32_t)(e << (31 - j)) >> 31);
    if (lanes) {
#pragma unroll
        for (int j = 0; j < (1 << F); ++j) t[j] ^= v.lanes[j];
    }
}

// Forward: (f0, f1) -> (f0 + c f1, f0 + (c + 1) f1); a missing level (its index
// bit becomes the component x_F) f0 + u f1 beside f1.
// Inverse: (p0, p1) -> (p0 + c (p0 + p1), p0 + p1); a missing level undoes itself.
template <int NFREE, int F, bool INV>
CM_HD void level_unit(uint32_t *sm, const Lev &v, uint32_t base, bool lanes, uint32_t u) {
    const uint32_t a = unit_addr<NFREE>(u, v.p, F);
    uint32_t *s0 = sm + phys(a), *s1 = sm + phys(a | (1u << v.p));
    uint32_t x0[1 << F], x1[1 << F], t[1 << F], o[1 << F];
    spread<F>(v, twiddle(v, base, a), lanes, t);
    // every load of a unit comes before its first store: the two halves' addresses
    // are unrelated to the compiler, which would otherwise chain them
    if (v.missing || !INV) {
#pragma unroll
        for (int j = 0; j < (1 << F); ++j) x1[j] = s1[j << NFREE];
        mul<F>(x1, t, o);
#pragma unroll
        for (int j = 0; j < (1 << F); ++j) x0[j] = s0[j << NFREE] ^ o[j];
#pragma unroll
        for (int j = 0; j < (1 << F); ++j) s0[j << NFREE] = x0[j];
        if (!v.missing) {
#pragma unroll
            for (int j = 0; j < (1 << F); ++j) s1[j << NFREE] = x0[j] ^ x1[j];
        }
    } else {
#pragma unroll
        for (int j = 0; j < (1 << F); ++j) {
            x0[j] = s0[j << NFREE];
            x1[j] = s1[j << NFREE];
        }
#pragma unroll
        for (int j = 0; j < (1 << F); ++j) x1[j] ^= x0[j];
        mul<F>(x1, t, o);
#pragma unroll
        for (int j = 0; j < (1 << F); ++j) {
            s0[j << NFREE] = x0[j] ^ o[j];
            s1[j << NFREE] = x1[j];
        }
    }
}

// Thread tid of nt: one level over the whole tile of 2^NB words.
template <int NB, int NFREE, int FMAX, bool INV>
CM_HD void level(uint32_t *sm, const Lev &v, uint32_t base, bool lanes, uint32_t tid, uint32_t nt) {
    const uint32_t units = 1u << (NB - 1 - v.f);
    switch (v.f) {
        case 0: for (uint32_t u = tid; u < units; u += nt) level_unit<NFREE, 0, INV>(sm, v, base, lanes, u); break;
        case 1: for (uint32_t u = tid; u < units; u += nt) level_unit<NFREE, 1, INV>(sm, v, base, lanes, u); break;
        case 2: for (uint32_t u = tid; u < units; u += nt) level_unit<NFREE, 2, INV>(sm, v, base, lanes, u); break;
        case 3: for (uint32_t u = tid; u < units; u += nt) level_unit<NFREE, 3, INV>(sm, v, base, lanes, u); break;
        case 4:
            if constexpr (FMAX >= 4)
                for (uint32_t u = tid; u < units; u += nt) level_unit<NFREE, 4, INV>(sm, v, base, lanes, u);
            break;
        default:
            if constexpr (FMAX >= 5)
                for (uint32_t u = tid; u < units; u += nt) level_unit<NFREE, 5, INV>(sm, v, base, lanes, u);
    }
}

// The tile's contribution to each level's twiddle (thread i: level i).
CM_HD uint32_t ext_twiddle(const Lev &v, uint32_t base, uint32_t tile) {
    for (int b = 0; tile; ++b, tile >>= 1)
        if (tile & 1u) base ^= v.ext[b];
    return base;
}

CM_HD uint32_t tile_base(const Pass &P, uint32_t tile) {
    uint32_t g = 0;
    for (uint32_t b = 0; b < P.next; ++b) g |= ((tile >> b) & 1u) << P.extpos[b];
    return g;
}

// Address of word l of 32-word block u of the bit transposition.
CM_HD uint32_t xpose_addr(const Pass &P, uint32_t u, uint32_t l) {
    uint32_t a = P.xlut[0][u & 15u] | P.xlut[1][u >> 4];
#pragma unroll
    for (int b = 0; b < 5; ++b) a |= ((l >> b) & 1u) << P.xp[b];
    return a;
}

}  // namespace gf
}  // namespace cm
