// Bit-sliced arithmetic in the tower GF(2) < GF(2^2) < ... < GF(2^32).
//
// GF(2^(2h)) = GF(2^h)[x] / (x^2 + x + c), c of trace 1 (the c of each step is
// the one whose multiplication matrix has the fewest ones, found by search),
// so an element of 2^LW bits is stored in the basis of products of the five
// generators: bit j of the element belongs to the product of the x_b over the
// set bits b of j.  Bit-sliced: word j of an array of 2^LW words holds bit j of
// 32 elements, one a lane, and a product of 32 pairs is a fixed network of
// AND / XOR on words (Karatsuba at every step of the tower, which the three-
// input LOP3 merges further).  It needs no table, no carry and no data-
// dependent branch; the ALU pipe is its only resource.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace cm {
namespace gf {

#define CM_HD __host__ __device__ __forceinline__

// x_(lw)^2 = x_(lw) + kC[lw], kC[lw] in GF(2^(2^lw))
constexpr uint32_t kC[5] = {1u, 2u, 12u, 240u, 43520u};

// Product of two elements of 2^lw bits (host tables, compile-time matrices).
constexpr uint32_t gmul(uint32_t a, uint32_t b, int lw) {
    if (lw == 0) return a & b;
    const int h = 1 << (lw - 1);
    const uint32_t m = (1u << h) - 1u;
    const uint32_t a0 = a & m, a1 = a >> h, b0 = b & m, b1 = b >> h;
    const uint32_t p0 = gmul(a0, b0, lw - 1), p2 = gmul(a1, b1, lw - 1), p1 = gmul(a0 ^ a1, b0 ^ b1, lw - 1);
    return (p0 ^ gmul(p2, kC[lw - 1], lw - 1)) | ((p1 ^ p0) << h);
}

// Row i of the matrix of multiplication by kC[LW]: the input bits output bit i sums.
template <int LW>
struct CRows {
    uint32_t r[1 << LW];
    constexpr CRows() : r{} {
        for (int j = 0; j < (1 << LW); ++j) {
            const uint32_t col = gmul(1u << j, kC[LW], LW);
            for (int i = 0; i < (1 << LW); ++i)
                if ((col >> i) & 1u) r[i] |= 1u << j;
        }
    }
};

// Three-input forms the compiler does not always find.
CM_HD uint32_t xor3(uint32_t a, uint32_t b, uint32_t c) {
#ifdef __CUDA_ARCH__
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0x96;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
#else
    return a ^ b ^ c;
#endif
}
CM_HD uint32_t and_xor(uint32_t a, uint32_t b, uint32_t c) {  // (a & b) ^ c
#ifdef __CUDA_ARCH__
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0x6A;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
#else
    return (a & b) ^ c;
#endif
}
CM_HD uint32_t xor_and(uint32_t a, uint32_t b, uint32_t c) {  // (a ^ b) & c
#ifdef __CUDA_ARCH__
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0x28;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
#else
    return (a ^ b) & c;
#endif
}

// o = a b on 2^LW words each.
template <int LW>
CM_HD void mul(const uint32_t *a, const uint32_t *b, uint32_t *o) {
    if constexpr (LW == 0) {
        o[0] = a[0] & b[0];
    } else if constexpr (LW == 1) {  // x_0^2 = x_0 + 1: five operations
        const uint32_t p0 = a[0] & b[0], s = b[0] ^ b[1];
        o[0] = and_xor(a[1], b[1], p0);
        o[1] = xor_and(a[0], a[1], s) ^ p0;
    } else {
        constexpr int H = 1 << (LW - 1);
        constexpr CRows<LW - 1> C{};
        uint32_t sa[H], sb[H], p0[H], p2[H], p1[H];
#pragma unroll
        for (int i = 0; i < H; ++i) {
            sa[i] = a[i] ^ a[H + i];
            sb[i] = b[i] ^ b[H + i];
        }
        mul<LW - 1>(a, b, p0);
        mul<LW - 1>(a + H, b + H, p2);
        mul<LW - 1>(sa, sb, p1);
#pragma unroll
        for (int i = 0; i < H; ++i) {
            o[H + i] = p1[i] ^ p0[i];
            uint32_t v = p0[i], w = 0;
            bool half = false;  // w holds a term waiting for a second
#pragma unroll
            for (int j = 0; j < H; ++j)
                if ((C.r[i] >> j) & 1u) {
                    if (half) v = xor3(v, w, p2[j]);
                    w = p2[j];
                    half = !half;
                }
            o[i] = half ? v ^ w : v;
        }
    }
}

}  // namespace gf
}  // namespace cm
