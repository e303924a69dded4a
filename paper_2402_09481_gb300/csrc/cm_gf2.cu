// Middle products as binary polynomials: additive transforms over a cross-
// section of Frobenius orbits.
//
// z_i = sum_t a_t b_(t+i) (mod 2) is the transpose of multiplication by the
// polynomial A(X) = sum a_t X^t over GF(2).  With E the map from 2^k
// coefficients to the values at 2^k / w points of GF(2^w) (one point from each
// Frobenius orbit; the values at the others are their squares, so the w bits
// of each value are all there is), multiplication is E^-1 (E a . E p), and its
// transpose E^T ((E a) . (E^-T b)): three transforms over k bits an operand,
// where a number-theoretic transform carries 32- or 64-bit words for each bit.
//
// Points.  beta_i is the Cantor basis (D. Cantor 1989), s_i the polynomial that
// vanishes on span(beta_0 .. beta_(i-1)); s_i(beta_(i+j)) = beta_j.  In the
// basis X_j = prod s_i^(bit i of j) (Lin, Chung, Han 2014) level i takes
// f = f0 + s_i f1 to its values on a coset and the next one: f0 + c f1 and
// f0 + (c + 1) f1 with c = s_i there.  All points lie in beta_k + span(beta_i,
// i < k).  Frobenius maps beta_i to beta_i + beta_(i-1), so the orbit of a point
// meets the points whose beta_(k - 2^j) coordinates are 0 exactly once (the
// cross-section of Li, Chen, Kuo, Cheng, Yang 2018, for a power-of-two set):
// the "missing" levels i = k - 2^j keep one value of the two, f0 + c f1 with
// c = x_j + u, which is an element of the field twice as large with x_j
// coefficient f1.  The first levels so run on single bits, the last on 16- or
// 32-bit elements; the data are 2^k bits throughout.
//
// Transposition.  Under <u, v> = coefficient of the top basis product in u v,
// multiplications are self-adjoint, and E^-T on the bit-reversed b turns out to
// be the same levels with c and c + 1 exchanged and u + 1 for u; E^T is its
// inverse.  The conversion to the basis X_j is stages of XORs (von zur Gathen,
// Gerhard 1996: division by s_(2^t) = X^(2^(2^t)) + X), transposed the same way.
// Point bits run complemented in both operands, so that values meet in place.
//
// Passes, for arrays of packed bits in natural order (index bits 0..4 inside a
// word):
//   k_gf_rows   (k > 16) input bits -> conversion across rows of 2^16 bits
//   k_gf_units  conversion of each row down to units of 256 bits
//   k_gf_cols   (k > 18) levels k-1 .. lo on tiles of 2^13 words, both operands
//   k_gf_mid    256-bit conversions, levels lo-1 .. 0, product, and back
// and the inverses of the first three on the product.  One product of 2^25 bits,
// us: rows 35.5 (inverse 20.7), units 18.5 (12), cols 23.5 (18.5), mid 84.5; the
// call 198, two summed integer products of 2^24 before it 545.  Past 2^25 bits
// k_gf_fwd and k_gf_sum / k_gf_sum2 stand in for k_gf_mid (2^28: 449 and 282 us
// of 1431; integer transforms 10650).  Levels are bit-sliced
// (gf2.cuh): a thread holds whole elements, one component a register, 32 of
// them a word.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include "cm_ctx.h"
#include "cm_gf2.h"
#include "cm_internal.h"

namespace cm {
namespace gf {

namespace {

// How an operand block's words lie in the source: word w of the array, inside
// [w0[i], w0[i] + n[i]), is the 32 bits from bit sh[i] of source word
// p[i] + dir w (in reversed order when dir < 0).  The two pieces are the bits
// before and after b's cyclic wrap; words w >= zero (a) or < zero (b) are 0, and
// the few others (at the pieces' ends) are read bit by bit.
struct Lin {
    const uint32_t *p[2];
    uint32_t sh[2], w0[2], n[2], zero;
    bool back;
};

__device__ __forceinline__ Lin lin_of(const InOp &o, bool is_b, int lg) {
    Lin l;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(o.map.src);
    const int64_t N = 1ll << lg, nw = N >> 5;
    l.w0[0] = l.w0[1] = l.n[0] = l.n[1] = l.sh[0] = l.sh[1] = 0;
    l.p[0] = l.p[1] = src;
    l.back = is_b || o.map.mode == kReverse;
    if (!is_b) {
        const uint64_t left = o.map.len > o.base ? o.map.len - o.base : 0, bits = left < o.lim ? left : o.lim;
        l.zero = (uint32_t)(((int64_t)bits + 31 < N ? (int64_t)bits + 31 : N) >> 5);
        l.n[0] = (uint32_t)((int64_t)bits < N ? (int64_t)bits >> 5 : nw);
        const int64_t c = l.back ? (int64_t)o.map.off - (int64_t)o.base - 31 : (int64_t)o.base;
        l.sh[0] = (uint32_t)c & 31u;
        l.p[0] = src + (c >> 5);
    } else {
        const int64_t top = (int64_t)o.base + N;  // word w: positions top - 32 - 32 w ..
        const int64_t z = top - (int64_t)o.map.len, cut = top + (int64_t)o.map.off - (int64_t)o.map.srclen;
        l.zero = z > 0 ? (uint32_t)(z >> 5) : 0u;               // words wholly past the end
        const int64_t full = z > 0 ? (z + 31) >> 5 : 0;         // first word wholly inside
        const int64_t e1 = cut > 0 ? cut >> 5 : 0;              // words [full, e1) lie past the wrap
        const int64_t b0 = cut > 0 ? (cut + 31) >> 5 : 0;       // words [b0, nw) before it
        for (int i = 0; i < 2; ++i) {
            int64_t w0 = i ? full : (full > b0 ? full : b0), w1 = i ? (e1 < nw ? e1 : nw) : nw;
            l.w0[i] = (uint32_t)(w0 < nw ? w0 : nw);
            l.n[i] = w1 > w0 ? (uint32_t)(w1 - w0) : 0u;
            const int64_t c = top - 32 + (int64_t)o.map.off - (i ? (int64_t)o.map.srclen : 0);
            l.sh[i] = (uint32_t)c & 31u;
            l.p[i] = src + (c >> 5);
        }
    }
    return l;
}

// Words at(0) .. at(N - 1) (~0: none) of an operand block's array of 2^lg bits:
// all the loads first, so that they are in flight together.
template <int N, class F>
__device__ __forceinline__ void in_words(const InOp &o, const Lin &l, bool is_b, int lg, F at, uint32_t (&v)[N]) {
    uint32_t lo[N], hi[N], sh[N];
    bool slow = false;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const uint32_t w = at(i);
        const bool in0 = w - l.w0[0] < l.n[0], in1 = w - l.w0[1] < l.n[1];
        const uint32_t *p = (in1 ? l.p[1] : l.p[0]) + (l.back ? -(int64_t)w : (int64_t)w);
        sh[i] = in1 ? l.sh[1] : l.sh[0];
        lo[i] = hi[i] = 0;
        if (in0 || in1) {
            lo[i] = __ldg(p);
            if (sh[i]) hi[i] = __ldg(p + 1);
        } else {
            slow |= w != ~0u && (is_b ? w >= l.zero : w < l.zero);
        }
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
        v[i] = __funnelshift_r(lo[i], hi[i], sh[i]);
        if (l.back) v[i] = __brev(v[i]);
    }
    if (slow) {
#pragma unroll 1
        for (int i = 0; i < N; ++i) {
            const uint32_t w = at(i);
            if (w == ~0u || w - l.w0[0] < l.n[0] || w - l.w0[1] < l.n[1] || !(is_b ? w >= l.zero : w < l.zero)) continue;
            uint32_t r = 0;
            for (uint32_t b = 0; b < 32; ++b) {
                const uint64_t j = 32ull * w + b;
                const uint64_t k = is_b ? o.base + (1ull << lg) - 1 - j : o.base + j;
                if (is_b || j < o.lim) r |= (uint32_t)o.map.get(k) << b;
            }
#pragma unroll
            for (int t = 0; t < N; ++t)
                if (t == i) v[t] = r;
        }
    }
}

__device__ __forceinline__ InOp in_op(const Ops &q, uint32_t o) {
    if (q.in) return q.in[o];
    InOp r = o < q.na ? q.a0 : q.b0;
    r.base += o < q.na ? q.astep * o : q.bstep * (o - q.na);
    return r;
}

__device__ __forceinline__ OutOp out_op(const Ops &q, uint32_t o) {
    if (q.out) return q.out[o];
    OutOp r = q.z0;
    const uint64_t done = q.zstep * o;
    r.z += done >> 6;
    r.m -= done;
    if (o + 1 < q.nz && r.m > q.zstep) r.m = q.zstep;
    return r;
}

// Word w of the product's array goes, reversed, to its place in z.
__device__ __forceinline__ void out_word(const OutOp &o, bool bad, int lg, uint64_t w, uint32_t v) {
    const uint64_t i = (1ull << (lg - 5)) - 1 - w;
    if (i >= 2 * ((o.m + 63) >> 6)) return;
    v = bad ? 0u : __brev(v);
    const uint64_t at = 32 * i;
    if (at >= o.m) v = 0u;
    else if (o.m - at < 32) v &= (1u << (uint32_t)(o.m - at)) - 1u;
    reinterpret_cast<uint32_t *>(o.z)[i] = v;
}

__device__ __forceinline__ bool constant_input(const OutOp &o, bool tell) {
    const bool bad = o.pre && (o.pre[0] == 0u || o.pre[1] == 0u);
    if (bad && tell) atomicOr(o.status, kFlagPrecond);
    return bad;
}

// ---------------------------------------------------------------------------
// Conversion across rows.  The stages "add row 2^j below, 2^j bits higher" of a
// column stripe need the 2^r - 1 bits to its left, so a warp holds 32 columns
// (words), lanes 16..31 its stripe and lanes 0..15 the words before it; rows sit
// in registers, five row bits at a time, and the shifts are shuffles.  Left of
// column 0 the stages are continued on the row's other end:
//   kConvA     bits shifted past the row's end (hi) return as hi X to the start
//              of their row and as hi to the next one;
//   kConvBInv  the words before column 0 are X end + (row above's end);
//   kConvB     its inverse: they are the row above's end alone.
// A CTA has 512 rows of stripes (2^r rows each); the whole-row stages that
// follow (kConvBInv: precede) run in shared memory, and from r = 4 on the first
// four levels of the transform with them: their twiddles are the same for every
// length and column, so they are one fixed map of 16 rows (first_levels).
constexpr int kRowsThreads = 512;
constexpr int kRowsSmem = 4 * 512 * (32 + 16);

// Unit (stripe, row) of register i of warp w in a round over row bits b .. b + 4.
template <int B>
__device__ __forceinline__ uint32_t row_unit(uint32_t w, int i) {
    return (w & ((1u << B) - 1u)) | ((uint32_t)i << B) | ((w >> B) << (B + 5));
}

// Stages of row bits HI - 1 .. LO (those below r) on registers that hold row
// bits B .. B + 4.
template <int B, int HI, int LO>
__device__ __forceinline__ void row_shift_stages(uint32_t (&x)[32], uint32_t lane, int r) {
#pragma unroll
    for (int j = HI - 1; j >= LO; --j) {
        if (j >= r) continue;
        const int s = 1 << j, bit = 1 << (j - B);
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if (!(i & bit)) {
                const uint32_t y = x[i | bit];
                if (s < 32) {
                    uint32_t p = __shfl_up_sync(0xFFFFFFFFu, y, 1);
                    if (lane == 0) p = 0;
                    x[i] ^= __funnelshift_l(p, y, s);
                } else {
                    const uint32_t p = __shfl_up_sync(0xFFFFFFFFu, y, s >> 5);
                    x[i] ^= lane >= (uint32_t)(s >> 5) ? p : 0u;
                }
            }
    }
}

// All shift stages: x in the layout of the first round on entry, row bits 0..4
// in registers on return.  xch: 512 x 32 words.  RC = max(r, 5).
template <int RC>
__device__ __forceinline__ void row_shifts(uint32_t (&x)[32], uint32_t *xch, uint32_t warp, uint32_t lane, int r) {
    if constexpr (RC > 5) {
        row_shift_stages<RC - 5, RC, RC - 5>(x, lane, r);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 32; ++i) xch[row_unit<RC - 5>(warp, i) * 32 + lane] = x[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 32; ++i) x[i] = xch[row_unit<0>(warp, i) * 32 + lane];
        row_shift_stages<0, RC - 5, 0>(x, lane, r);
    } else {
        row_shift_stages<0, 5, 0>(x, lane, r);
    }
}

// Row i of multiplication by C in GF(2^4): the input bits output bit i sums.
template <uint32_t C>
struct Rows4 {
    uint32_t r[4];
    constexpr Rows4() : r{} {
        for (int j = 0; j < 4; ++j)
            for (int i = 0; i < 4; ++i) r[i] |= ((gmul(1u << j, C, 2) >> i) & 1u) << j;
    }
};

// f * C in GF(2^4), bit-sliced.
template <uint32_t C>
__device__ __forceinline__ void times4(const uint32_t (&f)[4], uint32_t (&o)[4]) {
    constexpr Rows4<C> M{};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        o[i] = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if ((M.r[i] >> j) & 1u) o[i] ^= f[j];
    }
}

// Levels lg - 1 .. lg - 4 on 16 words whose number's bits 3 .. 0 are those index
// bits.  KIND 0: a, 1: b, 2: b's inverse.  Levels lg - 1, lg - 2 and lg - 4 are
// missing ones (components x_0, x_1, x_2); the twiddles are beta_1 .. beta_4 with
// the point bit of level lg - 3 (build_pass computes the same for the other
// lengths' tables).
template <int KIND>
__device__ __forceinline__ void first_levels(uint32_t (&x)[16]) {
    auto missing1 = [&]() {
        if (KIND == 0) return;  // u = 0
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] ^= x[i + 8];
    };
    auto missing2 = [&]() {
        if (KIND == 0) return;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            x[i] ^= x[i + 4];
            x[i + 8] ^= x[i + 12];
        }
    };
    auto level3 = [&]() {
#pragma unroll
        for (int b0 = 0; b0 < 2; ++b0) {
            uint32_t f[4], o[4];
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const int at = b0 + 8 * (w & 1) + 4 * (w >> 1);
                f[w] = KIND == 2 ? x[at] ^ x[at + 2] : x[at + 2];
            }
            times4<KIND == 0 ? 0xBu : 0xAu>(f, o);
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const int at = b0 + 8 * (w & 1) + 4 * (w >> 1);
                x[at] ^= o[w];
                x[at + 2] = KIND == 2 ? f[w] : x[at] ^ f[w];
            }
        }
    };
    auto missing4 = [&]() {
#pragma unroll
        for (int b1 = 0; b1 < 2; ++b1) {
            uint32_t f[4], o[4];
#pragma unroll
            for (int w = 0; w < 4; ++w) f[w] = x[2 * b1 + 8 * (w & 1) + 4 * (w >> 1) + 1];
            if (b1) times4<KIND == 0 ? 0xEu : 0xFu>(f, o);
            else times4<KIND == 0 ? 0xCu : 0xDu>(f, o);
#pragma unroll
            for (int w = 0; w < 4; ++w) x[2 * b1 + 8 * (w & 1) + 4 * (w >> 1)] ^= o[w];
        }
    };
    if (KIND == 2) {
        missing4();
        level3();
        missing2();
        missing1();
    } else {
        missing1();
        missing2();
        level3();
        missing4();
    }
}

// X e_row + e_(row - 1), word c (e_row at e + row * ld).
__device__ __forceinline__ uint32_t row_before(const uint32_t *e, uint32_t row, uint32_t c, uint32_t ld) {
    uint32_t v = e[row * ld + c] << 1;
    if (c) v |= e[row * ld + c - 1] >> 31;
    if (row) v ^= e[(row - 1) * ld + c];
    return v;
}

// One whole-row stage (top, sh) on sm[512][CW].
template <int KIND, int CW>
__device__ __forceinline__ void row_whole_stage(uint32_t *sm, uint32_t top, uint32_t sh) {
    constexpr int LC = CW == 32 ? 5 : 4;
    constexpr uint32_t NG = kRowsThreads >> LC;
    const uint32_t c = threadIdx.x & (CW - 1u), g = threadIdx.x >> LC;
    const uint32_t H = 1u << top, s = 1u << sh;
    auto bulk = [&]() {
        __syncthreads();
#pragma unroll
        for (uint32_t i = 0; i < 256; i += NG) {
            const uint32_t u = i + g, v = u & (H - 1u), row = v | ((u ^ v) << 1);
            if (v >= s) sm[row * CW + c] ^= sm[(row + H - s) * CW + c];
        }
    };
    auto wrapped = [&]() {
        __syncthreads();
        for (uint32_t u = g; u < (512u >> (top + 1)) * s; u += NG) {
            const uint32_t row = ((u >> sh) << (top + 1)) + (KIND == kConvA ? H : 0u) + (u & (s - 1u));
            sm[row * CW + c] ^= sm[(row + H - s) * CW + c];
        }
    };
    if (KIND == kConvBInv) {
        bulk();
        wrapped();
    } else {
        wrapped();
        bulk();
    }
}

// The stages that convert k index bits from `base` on, in kConvA's order: the
// shifts of the top k - q of them (q the largest power of two below k), then
// those bits and the lower q among themselves.
constexpr void conv_list(int base, int k, Stages *s) {
    if (k <= 1) return;
    int t = 0;
    while ((2 << t) < k) ++t;
    const int q = 1 << t, r = k - q;
    for (int j = r - 1; j >= 0; --j) {
        s->top[s->n] = (uint8_t)(base + q + j);
        s->sh[s->n++] = (uint8_t)(base + j);
    }
    conv_list(base + q, r, s);
    conv_list(base, q, s);
}
template <int BITS>
struct StageList {
    Stages s;
    constexpr StageList() : s{} { conv_list(0, BITS, &s); }
};

// All whole-row stages: RC > 5 rows' list is known at compile time.
template <int KIND, int CW, int RC>
__device__ __forceinline__ void row_whole_stages(uint32_t *sm, const Stages &st) {
    if constexpr (RC > 5) {
        constexpr StageList<RC> L{};
#pragma unroll
        for (int n = 0; n < L.s.n; ++n) {
            const int q = KIND == kConvBInv ? L.s.n - 1 - n : n;
            row_whole_stage<KIND, CW>(sm, L.s.top[q], L.s.sh[q]);
        }
    } else {
        for (int n = 0; n < st.n; ++n) {
            const int q = KIND == kConvBInv ? st.n - 1 - n : n;
            row_whole_stage<KIND, CW>(sm, st.top[q], st.sh[q]);
        }
    }
    __syncthreads();
}

template <int RC, bool INV>
__global__ void __launch_bounds__(kRowsThreads, 2) k_gf_rows(const __grid_constant__ Ops q, int lg,
                                                          const __grid_constant__ Stages st, uint32_t *__restrict__ data) {
    extern __shared__ __align__(16) uint32_t sm[];
    uint32_t *xch = sm, *side = sm + 512 * 32;  // side: 2^r x 16 words past the row's end
    constexpr int B0 = RC - 5;                  // first round's lowest row bit
    const int r = lg - 16, S = 9 - r;           // 2^S stripes a CTA (128 in all)
    const uint32_t R = 1u << r, groups = S < 7 ? 128u >> S : 1u;
    const uint32_t grp = blockIdx.x % groups, op = blockIdx.x / groups;
    uint32_t *arr = data + ((uint64_t)op << (lg - 5));
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const bool first = grp == 0, is_b = op >= q.na;
    uint32_t x[32];
    if (!INV) {
        const InOp in = in_op(q, op);
        const Lin lin = lin_of(in, is_b, lg);
        // phase 0 (a's first stripe): the row's last words, then zeros its shifts
        // run into; phase 1: the stripes
        for (int phase = first && !is_b ? 0 : 1; phase < 2; ++phase) {
            __syncthreads();
            for (int i0 = 0; i0 < 32; i0 += 8) {
                uint32_t v[8];
                in_words<8>(in, lin, is_b, lg, [&](int i) -> uint32_t {
                    const uint32_t u = row_unit<B0>(warp, i0 + i), row = u & (R - 1u), stripe = (grp << S) + (u >> r);
                    const uint32_t at = row * 2048u + 16 * stripe + lane - 16;  // b: on into the row above
                    if (phase == 0) return u < R && lane < 16 ? row * 2048u + 2032u + lane : ~0u;
                    return stripe < 128 && (16 * stripe + lane >= 16 || (is_b && row)) ? at : ~0u;
                }, v);
#pragma unroll
                for (int i = 0; i < 8; ++i) xch[row_unit<B0>(warp, i0 + i) * 32 + lane] = v[i];
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 32; ++i) x[i] = xch[row_unit<B0>(warp, i) * 32 + lane];
            row_shifts<RC>(x, xch, warp, lane, r);
            if (phase == 1) break;
            __syncthreads();
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const uint32_t u = row_unit<0>(warp, i);
                if (lane >= 16 && u < R) side[u * 16 + lane - 16] = x[i];
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if (lane >= 16) sm[row_unit<0>(warp, i) * 16 + lane - 16] = x[i];
        __syncthreads();
        const uint32_t c = threadIdx.x & 15u;
        if (first && !is_b)
            for (uint32_t u = threadIdx.x >> 4; u < R; u += 32) sm[u * 16 + c] ^= row_before(side, u, c, 16);
        if (is_b) row_whole_stages<kConvB, 16, RC>(sm, st);
        else row_whole_stages<kConvA, 16, RC>(sm, st);
        if (r >= 4) {
            const uint32_t g = threadIdx.x >> 4, row = g & (R / 16 - 1u), sl = g >> (r - 4), stripe = (grp << S) + sl;
            uint32_t y[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) y[k] = sm[(sl * R + row + k * (R / 16)) * 16 + c];
            if (is_b) first_levels<1>(y);
            else first_levels<0>(y);
#pragma unroll
            for (int k = 0; k < 16; ++k) arr[(uint64_t)(row + k * (R / 16)) * 2048u + stripe * 16u + c] = y[k];
        } else {
            for (uint32_t u = threadIdx.x >> 4; u < 512; u += 32) {
                const uint32_t row = u & (R - 1u), stripe = (grp << S) + (u >> r);
                if (stripe < 128) arr[(uint64_t)row * 2048u + stripe * 16u + c] = sm[u * 16 + c];
            }
        }
    } else {
        const OutOp out = out_op(q, op);
        const bool bad = constant_input(out, first && threadIdx.x == 0);
        if (r >= 4) {
#pragma unroll
            for (uint32_t g = warp; g < 32; g += 16) {
                const uint32_t row = g & (R / 16 - 1u), sl = g >> (r - 4), col = (16u * ((grp << S) + sl) + lane - 16u) & 2047u;
                uint32_t y[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) y[k] = arr[(uint64_t)(row + k * (R / 16)) * 2048u + col];
                first_levels<2>(y);
#pragma unroll
                for (int k = 0; k < 16; ++k) sm[(sl * R + row + k * (R / 16)) * 32 + lane] = y[k];
            }
        } else {
#pragma unroll 8
            for (uint32_t u = warp; u < 512; u += 16) {
                const uint32_t row = u & (R - 1u), stripe = ((grp << S) + (u >> r)) & 127u;
                sm[u * 32 + lane] = arr[(uint64_t)row * 2048u + ((16u * stripe + lane - 16u) & 2047u)];
            }
        }
        row_whole_stages<kConvBInv, 32, RC>(sm, st);
#pragma unroll
        for (int i = 0; i < 32; ++i) x[i] = sm[row_unit<B0>(warp, i) * 32 + lane];
        if (first && lane < 16) {
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const uint32_t u = row_unit<B0>(warp, i);
                if (u < R) x[i] = row_before(sm, u, lane, 32);
            }
        }
        row_shifts<RC>(x, xch, warp, lane, r);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if (lane >= 16) sm[row_unit<0>(warp, i) * 16 + lane - 16] = x[i];
        __syncthreads();
        const uint32_t c = threadIdx.x & 15u;
        for (uint32_t u = threadIdx.x >> 4; u < 512; u += 32) {
            const uint32_t row = u & (R - 1u), stripe = (grp << S) + (u >> r);
            if (stripe < 128) out_word(out, bad, lg, (uint64_t)row * 2048u + stripe * 16u + c, sm[u * 16 + c]);
        }
    }
}

// ---------------------------------------------------------------------------
// Conversion of rows of 2^(8 + UB) bits to 256-bit units (UB = 8, or 7 for
// transforms of 2^15): the same stages as across rows, units for rows and 8
// words for columns.  16 threads have a unit's 8 words and the 8 words before
// (kConvB, kConvBInv) or past (kConvA) it, 32 units in registers; the whole-unit
// stages are the shifts of the upper four unit bits in shared memory, then four
// bits' conversion in registers, twice.  Bound by instruction issue (about 55 a
// word; stages between barriers on a unit a thread took 150).  In place; for
// lg <= 16 the row is the whole operand, read from the inputs or written to z.
constexpr int kUnitsThreads = 256;

// Conversion of the 4 index bits of 16 registers.
template <int KIND, int TOP, int SH>
__device__ __forceinline__ void conv4_stage(uint32_t (&x)[16]) {
    constexpr int H = 1 << TOP, S = 1 << SH;
    auto wrap = [&]() {
#pragma unroll
        for (int b = 0; b < 16; b += 2 * H)
#pragma unroll
            for (int v = 0; v < S; ++v) {
                const int o = b + (KIND == kConvA ? H : 0);
                x[o + v] ^= x[o + H - S + v];
            }
    };
    if (KIND != kConvBInv) wrap();
#pragma unroll
    for (int b = 0; b < 16; b += 2 * H)
#pragma unroll
        for (int v = S; v < H; ++v) x[b + v] ^= x[b + H + v - S];
    if (KIND == kConvBInv) wrap();
}

template <int KIND>
__device__ __forceinline__ void conv4(uint32_t (&x)[16]) {
    if (KIND == kConvBInv) {
        conv4_stage<KIND, 1, 0>(x);
        conv4_stage<KIND, 3, 2>(x);
        conv4_stage<KIND, 2, 0>(x);
        conv4_stage<KIND, 3, 1>(x);
    } else {
        conv4_stage<KIND, 3, 1>(x);
        conv4_stage<KIND, 2, 0>(x);
        conv4_stage<KIND, 3, 2>(x);
        conv4_stage<KIND, 1, 0>(x);
    }
}

// Conversion of 3 index bits (the upper ones when UB = 7) of 8 registers, every
// second of 16.
template <int KIND>
__device__ __forceinline__ void conv3(uint32_t (&x)[8]) {
    // stages (2, 0), then (1, 0) of the lower two bits
    auto st = [&](int H, int S) {
        if (KIND != kConvBInv)
            for (int b = 0; b < 8; b += 2 * H)
                for (int v = 0; v < S; ++v) x[b + (KIND == kConvA ? H : 0) + v] ^= x[b + (KIND == kConvA ? H : 0) + H - S + v];
        for (int b = 0; b < 8; b += 2 * H)
            for (int v = S; v < H; ++v) x[b + v] ^= x[b + H + v - S];
        if (KIND == kConvBInv)
            for (int b = 0; b < 8; b += 2 * H)
                for (int v = 0; v < S; ++v) x[b + v] ^= x[b + H - S + v];
    };
    if (KIND == kConvBInv) {
        st(2, 1);
        st(4, 1);
    } else {
        st(4, 1);
        st(2, 1);
    }
}

// Shift stages HI - 1 .. LO of the unit bits B .. B + 4 in registers.
template <int B, int HI, int LO>
__device__ __forceinline__ void unit_shift_stages(uint32_t (&x)[32], uint32_t c16) {
#pragma unroll
    for (int j = HI - 1; j >= LO; --j) {
        const int s = 1 << j, bit = 1 << (j - B);
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if (!(i & bit)) {
                const uint32_t y = x[i | bit];
                if (s < 32) {
                    uint32_t p = __shfl_up_sync(0xFFFFFFFFu, y, 1, 16);
                    if (c16 == 0) p = 0;
                    x[i] ^= __funnelshift_l(p, y, s);
                } else {
                    const uint32_t p = __shfl_up_sync(0xFFFFFFFFu, y, s >> 5, 16);
                    x[i] ^= c16 >= (uint32_t)(s >> 5) ? p : 0u;
                }
            }
    }
}

// Whole-unit stages on S[unit * 8 + word].  tid: of the row's 2^(UB - 1) threads.
template <int KIND, int UB>
__device__ __forceinline__ void unit_whole_stages(uint32_t *S, uint32_t tid) {
    constexpr uint32_t TPR = 1u << (UB - 1), NU = 1u << UB;
    const uint32_t c = tid & 7u, g = tid >> 3;
    auto shifts = [&](int top, int sh) {  // of the upper bits, by the lower four
        const uint32_t H = 1u << top, s = 1u << sh;
        auto bulk = [&]() {
            __syncthreads();
#pragma unroll
            for (uint32_t i = 0; i < NU / 2; i += TPR / 8) {
                const uint32_t u = i + g, v = u & (H - 1u), t = v | ((u ^ v) << 1);
                if (v >= s) S[t * 8 + c] ^= S[(t + H - s) * 8 + c];
            }
        };
        auto wrap = [&]() {
            __syncthreads();
            for (uint32_t u = g; u < (NU >> (top + 1)) * s; u += TPR / 8) {
                const uint32_t t = ((u >> sh) << (top + 1)) + (KIND == kConvA ? H : 0u) + (u & (s - 1u));
                S[t * 8 + c] ^= S[(t + H - s) * 8 + c];
            }
        };
        if (KIND != kConvBInv) wrap();
        bulk();
        if (KIND == kConvBInv) wrap();
    };
    auto upper = [&]() {  // conversion of the upper UB - 4 bits
        __syncthreads();
        if (UB == 8) {
            uint32_t x[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = S[(16 * i + g) * 8 + c];
            conv4<KIND>(x);
#pragma unroll
            for (int i = 0; i < 16; ++i) S[(16 * i + g) * 8 + c] = x[i];
        } else {
            for (uint32_t k = g; k < 16; k += TPR / 8) {
                uint32_t x[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) x[i] = S[(16 * i + k) * 8 + c];
                conv3<KIND>(x);
#pragma unroll
                for (int i = 0; i < 8; ++i) S[(16 * i + k) * 8 + c] = x[i];
            }
        }
    };
    auto lower = [&]() {  // of the lower four
        __syncthreads();
        for (uint32_t h = g; h < NU / 16; h += TPR / 8) {
            uint32_t x[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = S[(16 * h + i) * 8 + c];
            conv4<KIND>(x);
#pragma unroll
            for (int i = 0; i < 16; ++i) S[(16 * h + i) * 8 + c] = x[i];
        }
    };
    if (KIND == kConvBInv) {
        lower();
        upper();
#pragma unroll
        for (int j = 0; j < UB - 4; ++j) shifts(4 + j, j);
    } else {
#pragma unroll
        for (int j = UB - 5; j >= 0; --j) shifts(4 + j, j);
        upper();
        lower();
    }
    __syncthreads();
}

// The shift stages of a row in S through the exchange buffer E[unit * 16 + c16].
template <int KIND, int UB>
__device__ __forceinline__ void unit_shifts(uint32_t *S, uint32_t *E, uint32_t tid, uint32_t (&x)[32]) {
    const uint32_t c16 = tid & 15u, tu = tid >> 4;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        const uint32_t u = tu | (uint32_t)i << (UB - 5), at = u * 8 + c16;
        if (KIND == kConvA) x[i] = c16 < 8 ? S[at] : 0u;
        else if (KIND == kConvB) x[i] = at >= 8 ? S[at - 8] : 0u;
        else x[i] = c16 >= 8 ? S[at - 8] : row_before(S, u, c16, 8);
    }
    unit_shift_stages<UB - 5, UB, UB - 5>(x, c16);
#pragma unroll
    for (int i = 0; i < 32; ++i) E[(tu | (uint32_t)i << (UB - 5)) * 16 + c16] = x[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 32; ++i) x[i] = E[((uint32_t)i | tu << 5) * 16 + c16];
    unit_shift_stages<0, UB - 5, 0>(x, c16);
}

// KIND is the same in a CTA: kConvA and kConvB rows (ra and rb of them) have CTAs
// of their own.
template <int KIND, int UB>
__device__ __forceinline__ void units_row(const Ops &q, int lg, uint32_t row, bool in_range, uint32_t *S, uint32_t *E,
                                          uint32_t tid, uint32_t *__restrict__ data) {
    constexpr uint32_t TPR = 1u << (UB - 1), NW = 8u << UB;
    uint32_t *arr = data + (uint64_t)row * NW;
    const uint32_t op = (uint32_t)(((uint64_t)row << (UB + 8)) >> lg);
    const uint32_t c16 = tid & 15u, tu = tid >> 4;
    uint32_t x[32];
    if (in_range) {
        if (KIND != kConvBInv && lg <= 16) {
            const InOp in = in_op(q, op);
            const Lin lin = lin_of(in, KIND == kConvB, lg);
            for (uint32_t i = 0; i < NW / TPR; i += 8) {
                uint32_t v[8];
                in_words<8>(in, lin, KIND == kConvB, lg, [&](int k) -> uint32_t { return (i + k) * TPR + tid; }, v);
#pragma unroll
                for (int k = 0; k < 8; ++k) S[(i + k) * TPR + tid] = v[k];
            }
        } else {
#pragma unroll
            for (uint32_t i = tid; i < NW / 4; i += TPR) reinterpret_cast<uint4 *>(S)[i] = reinterpret_cast<const uint4 *>(arr)[i];
        }
    }
    __syncthreads();
    if (KIND == kConvBInv) unit_whole_stages<KIND, UB>(S, tid);
    unit_shifts<KIND, UB>(S, E, tid, x);
    if (KIND == kConvA) {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 32; ++i) E[((uint32_t)i | tu << 5) * 16 + c16] = x[i];
        __syncthreads();
        for (uint32_t w = tid; w < NW; w += TPR) {
            const uint32_t u = w >> 3, c = w & 7u;
            S[w] = E[u * 16 + c] ^ row_before(E + 8, u, c, 16);
        }
    } else {  // all of S has been read
        if (c16 >= 8)
#pragma unroll
            for (int i = 0; i < 32; ++i) S[((uint32_t)i | tu << 5) * 8 + c16 - 8] = x[i];
    }
    if (KIND != kConvBInv) unit_whole_stages<KIND, UB>(S, tid);
    else __syncthreads();
    if (!in_range) return;
    if (KIND == kConvBInv && lg <= 16) {
        const OutOp out = out_op(q, op);
        const bool bad = constant_input(out, tid == 0);
        for (uint32_t w = tid; w < NW; w += TPR) out_word(out, bad, lg, w, S[w]);
    } else {
#pragma unroll
        for (uint32_t i = tid; i < NW / 4; i += TPR) reinterpret_cast<uint4 *>(arr)[i] = reinterpret_cast<const uint4 *>(S)[i];
    }
}

template <bool INV, int UB>
__global__ void __launch_bounds__(kUnitsThreads, 4) k_gf_units(const __grid_constant__ Ops q, int lg, uint32_t ra,
                                                               uint32_t rb, uint32_t *__restrict__ data) {
    constexpr uint32_t TPR = 1u << (UB - 1), NW = 8u << UB, RPC = kUnitsThreads / TPR;
    extern __shared__ __align__(16) uint32_t sm[];
    const uint32_t mine = threadIdx.x / TPR, tid = threadIdx.x % TPR, ca = (ra + RPC - 1) / RPC;
    uint32_t *S = sm + mine * 3 * NW, *E = S + NW;
    if (INV || blockIdx.x >= ca) {
        const uint32_t k = (INV ? blockIdx.x : blockIdx.x - ca) * RPC + mine;
        units_row<INV ? kConvBInv : kConvB, UB>(q, lg, INV ? k : ra + k, k < (INV ? ra : rb), S, E, tid, data);
    } else {
        const uint32_t k = blockIdx.x * RPC + mine;
        units_row<kConvA, UB>(q, lg, k, k < ra, S, E, tid, data);
    }
}

// ---------------------------------------------------------------------------
// Level passes.

__device__ __forceinline__ void load_pass(Pass *P, const Pass *__restrict__ g) {
    uint4 *d = reinterpret_cast<uint4 *>(P);
    const uint4 *s = reinterpret_cast<const uint4 *>(g);
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < sizeof(Pass) / 16; i += blockDim.x) d[i] = __ldg(s + i);
}

// Levels lg - 1 .. lo: fields up to GF(2^16), twiddles that depend on the tile's
// own bits only.  In place; grid: tiles of every array.  Two operands of 2^25: 23.5
// us, most of it the loads' and stores' latency (seven levels; the first four, on
// single bits to GF(16), have constant twiddles and run with the row conversion).
constexpr int kColsThreads = 256;

template <bool INV>
__global__ void __launch_bounds__(kColsThreads, 3) k_gf_cols(int lg, uint32_t na, const Pass *__restrict__ table,
                                                          uint32_t *__restrict__ data) {
    __shared__ __align__(16) uint32_t sm[8192];
    __shared__ Pass P;
    const uint32_t tile = blockIdx.x & ((1u << (lg - 18)) - 1u), op = blockIdx.x >> (lg - 18);
    load_pass(&P, table);
    __syncthreads();
    uint32_t *arr = data + ((uint64_t)op << (lg - 5)) + tile_base(P, tile);
    const uint32_t which = INV || op >= na;
#pragma unroll
    for (uint32_t e = 4 * threadIdx.x; e < 8192; e += 4 * kColsThreads) {
        const uint4 v = *reinterpret_cast<const uint4 *>(arr + lut3(P.glut, e));
        sm[phys(lut3(P.alut, e))] = v.x;
        sm[phys(lut3(P.alut, e + 1))] = v.y;
        sm[phys(lut3(P.alut, e + 2))] = v.z;
        sm[phys(lut3(P.alut, e + 3))] = v.w;
    }
    __syncthreads();
    for (uint32_t l = 0; l < P.nlev; ++l) {
        const Lev &v = P.lev[INV ? P.nlev - 1 - l : l];
        level<13, 9, 4, INV>(sm, v, v.base[which], false, threadIdx.x, kColsThreads);
        __syncthreads();
    }
    for (uint32_t e = 4 * threadIdx.x; e < 8192; e += 4 * kColsThreads) {
        uint4 v;
        v.x = sm[phys(lut3(P.alut, e))];
        v.y = sm[phys(lut3(P.alut, e + 1))];
        v.z = sm[phys(lut3(P.alut, e + 2))];
        v.w = sm[phys(lut3(P.alut, e + 3))];
        *reinterpret_cast<uint4 *>(arr + lut3(P.glut, e)) = v;
    }
}

// The word bits change places with five point bits: a warp transposes 32 x 32
// bit blocks by shuffles (word l of a block in lane l), three instructions a
// step: exchange, rotate to the other half, merge (bytes: permute).
template <int NB>
__device__ void transpose_bits(uint32_t *sm, const Pass &P, uint32_t warp, uint32_t nwarp) {
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t keep[3], rot[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const uint32_t m = b == 0 ? 0x55555555u : b == 1 ? 0x33333333u : 0x0F0F0F0Fu;
        const bool up = (lane >> b) & 1u;
        keep[b] = up ? ~m : m;
        rot[b] = up ? 32u - (1u << b) : 1u << b;
    }
    const uint32_t sel3 = (lane & 8u) ? 0x3715u : 0x6240u, sel4 = (lane & 16u) ? 0x3276u : 0x5410u;
    const uint32_t la = xpose_addr(P, 0, lane);
#pragma unroll 4
    for (uint32_t u = warp; u < (1u << (NB - 5)); u += nwarp) {
        uint32_t *at = sm + phys(la | P.xlut[0][u & 15u] | P.xlut[1][u >> 4]);
        uint32_t v = *at;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, v, 1 << b);
            v = (v & keep[b]) | (__funnelshift_l(y, y, rot[b]) & ~keep[b]);
        }
        v = __byte_perm(v, __shfl_xor_sync(0xFFFFFFFFu, v, 8), sel3);
        v = __byte_perm(v, __shfl_xor_sync(0xFFFFFFFFu, v, 16), sel4);
        *at = v;
    }
}

template <int NB, int KIND>
__device__ void load_tile(uint32_t *sm, const Pass &P, const uint32_t *__restrict__ arr, uint32_t tid, uint32_t nt) {
#pragma unroll 4
    for (uint32_t e = 8 * tid; e < (1u << NB); e += 8 * nt) {
        const uint32_t *g = arr + lut3(P.glut, e);
        const uint4 u = *reinterpret_cast<const uint4 *>(g), v = *reinterpret_cast<const uint4 *>(g + 4);
        uint32_t x[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
        conv8<KIND>(x);
#pragma unroll
        for (int i = 0; i < 8; ++i) sm[phys(lut3(P.alut, e + i))] = x[i];
    }
}

template <int NB>
__device__ void store_tile(const uint32_t *sm, const Pass &P, uint32_t *__restrict__ arr, uint32_t tid, uint32_t nt) {
    for (uint32_t e = 8 * tid; e < (1u << NB); e += 8 * nt) {
        uint32_t x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = sm[phys(lut3(P.alut, e + i))];
        conv8<kConvBInv>(x);
        uint32_t *g = arr + lut3(P.glut, e);
        *reinterpret_cast<uint4 *>(g) = make_uint4(x[0], x[1], x[2], x[3]);
        *reinterpret_cast<uint4 *>(g + 4) = make_uint4(x[4], x[5], x[6], x[7]);
    }
}

template <int NB, int FMAX>
struct MidShape {
    static constexpr int NFREE = NB - FMAX;
    // one thread a unit of the longest elements in each operand's tile
    static constexpr int HALF = 1 << (NB - 1 - FMAX);
    static constexpr int SMEM1 = 4 << NB;
};

template <int NB, int FMAX>
__device__ void inverse_levels(uint32_t *sm, const Pass &P, const uint32_t *base, int nt) {
    for (int l = (int)P.nlev - 1; l >= 0; --l) {
        level<NB, NB - FMAX, FMAX, true>(sm, P.lev[l], base[l], l >= (int)P.npre, threadIdx.x, (uint32_t)nt);
        __syncthreads();
        if (l == (int)P.npre) {
            transpose_bits<NB>(sm, P, threadIdx.x >> 5, (uint32_t)nt >> 5);
            __syncthreads();
        }
    }
}

// One pair of tiles: both forward transforms, the product, the inverse
// transform in place of b's tile.  The ALU pipe bounds it; a thread holds one
// unit of 2 x 32 words.  PAR: half the threads on each operand, for few tiles
// (a tile's own time counts); else one operand after the other on half as many
// threads, so that three CTAs of an SM fill each other's gaps.  2^25: 84.5 us (91
// before a unit's loads came before its stores), 46% of the ALU rate: 128 tiles
// have two warps a scheduler, the inverse one, and the first stall is instruction
// fetch (a product of GF(2^32) elements is about a thousand instructions in line).  Both operands' units in one
// thread, sharing the twiddle sums, took 120 for 91 (255 registers).
template <int NB, int FMAX, bool PAR>
__global__ void __launch_bounds__((PAR ? 2 : 1) * MidShape<NB, FMAX>::HALF, PAR ? 1 : 384 / MidShape<NB, FMAX>::HALF)
k_gf_mid(int lg, const Pass *__restrict__ table,
                                                                         const uint32_t *__restrict__ A,
                                                                         uint32_t *__restrict__ B) {
    using S = MidShape<NB, FMAX>;
    constexpr int NT = (PAR ? 2 : 1) * S::HALF, W = 1 << FMAX;
    extern __shared__ __align__(16) uint32_t sm[];
    __shared__ Pass P;
    __shared__ uint32_t base[2][kMaxLev];
    const int lgt = lg - 5 - NB;
    const uint32_t tile = blockIdx.x & ((1u << lgt) - 1u), pair = blockIdx.x >> lgt;
    load_pass(&P, table);
    __syncthreads();
    const uint64_t off = ((uint64_t)pair << (lg - 5)) + tile_base(P, tile);
    for (uint32_t i = threadIdx.x; i < 2 * P.nlev; i += NT) {
        const uint32_t l = i >> 1, o = i & 1u;
        base[o][l] = ext_twiddle(P.lev[l], P.lev[l].base[o], tile);
    }
    const uint32_t op = PAR ? threadIdx.x >= S::HALF : 0u, tid = threadIdx.x - op * S::HALF;
    uint32_t *mine = sm + op * (1u << NB);
    if (PAR ? op : false) load_tile<NB, kConvB>(mine, P, B + off, tid, S::HALF);
    else load_tile<NB, kConvA>(mine, P, A + off, tid, S::HALF);
    if (!PAR) load_tile<NB, kConvB>(sm + (1u << NB), P, B + off, tid, S::HALF);
    __syncthreads();
    for (uint32_t k = 0; k < (PAR ? 1u : 2u) * P.nlev; ++k) {
        const uint32_t o = PAR ? op : k >= P.nlev, l = k - (PAR ? 0u : o * P.nlev);
        uint32_t *t = sm + o * (1u << NB);
        if (l == P.npre) {
            transpose_bits<NB>(PAR ? sm : t, P, threadIdx.x >> 5, NT >> 5);
            if (PAR) transpose_bits<NB>(sm + (1u << NB), P, threadIdx.x >> 5, NT >> 5);
            __syncthreads();
        }
        level<NB, S::NFREE, FMAX, false>(t, P.lev[l], base[o][l], l >= P.npre, tid, S::HALF);
        __syncthreads();
    }
    uint32_t *sb = sm + (1u << NB);
    for (uint32_t u = threadIdx.x; u < (1u << S::NFREE); u += NT) {
        uint32_t a[W], b[W], o[W];
        const uint32_t at = phys(u);
#pragma unroll
        for (int j = 0; j < W; ++j) {
            a[j] = sm[at + (j << S::NFREE)];
            b[j] = sb[at + (j << S::NFREE)];
        }
        mul<FMAX>(a, b, o);
#pragma unroll
        for (int j = 0; j < W; ++j) sb[at + (j << S::NFREE)] = o[j];
    }
    __syncthreads();
    inverse_levels<NB, FMAX>(sb, P, base[1], NT);
    store_tile<NB>(sb, P, B + off, threadIdx.x, NT);
}

// Several blocks: the forward half alone, tile words to H in tile order (449 us in
// the 2^28 product; ALU pipe) ...
__global__ void __launch_bounds__(128) k_gf_fwd(int lg, uint32_t na, const Pass *__restrict__ table,
                                                const uint32_t *__restrict__ data, uint32_t *__restrict__ hat) {
    __shared__ __align__(16) uint32_t sm[8192];
    __shared__ Pass P;
    __shared__ uint32_t base[kMaxLev];
    const uint32_t tile = blockIdx.x & ((1u << (lg - 18)) - 1u), op = blockIdx.x >> (lg - 18);
    const bool is_b = op >= na;
    load_pass(&P, table);
    __syncthreads();
    if (threadIdx.x < P.nlev)
        base[threadIdx.x] = ext_twiddle(P.lev[threadIdx.x], P.lev[threadIdx.x].base[is_b], tile);
    const uint32_t *arr = data + ((uint64_t)op << (lg - 5)) + tile_base(P, tile);
    if (is_b) load_tile<13, kConvB>(sm, P, arr, threadIdx.x, 128);
    else load_tile<13, kConvA>(sm, P, arr, threadIdx.x, 128);
    __syncthreads();
    for (uint32_t l = 0; l < P.nlev; ++l) {
        if (l == P.npre) {
            transpose_bits<13>(sm, P, threadIdx.x >> 5, 4);
            __syncthreads();
        }
        level<13, 8, 5, false>(sm, P.lev[l], base[l], l >= P.npre, threadIdx.x, 128);
        __syncthreads();
    }
    uint4 *o = reinterpret_cast<uint4 *>(hat + ((uint64_t)op << (lg - 5)) + ((uint64_t)tile << 13));
    for (uint32_t i = threadIdx.x; i < 2048; i += 128) o[i] = reinterpret_cast<const uint4 *>(sm)[i];
}

// ... and a window's sum of products with the inverse: window w adds a's block
// i times b's block i + w over i < nin.  One thread a point word (32 elements).
__device__ __forceinline__ void load32(uint32_t (&v)[32], const uint32_t *p) {
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __ldg(p + (j << 8));
}

__global__ void __launch_bounds__(256) k_gf_sum(int lg, uint32_t na, uint32_t nin, const Pass *__restrict__ table,
                                                const uint32_t *__restrict__ hat, uint32_t *__restrict__ out) {
    __shared__ __align__(16) uint32_t sm[8192];
    __shared__ Pass P;
    __shared__ uint32_t base[kMaxLev];
    const uint32_t tile = blockIdx.x & ((1u << (lg - 18)) - 1u), win = blockIdx.x >> (lg - 18);
    load_pass(&P, table);
    __syncthreads();
    if (threadIdx.x < P.nlev)
        base[threadIdx.x] = ext_twiddle(P.lev[threadIdx.x], P.lev[threadIdx.x].base[1], tile);
    const uint32_t at = phys(threadIdx.x);
    const uint32_t *ha = hat + ((uint64_t)tile << 13) + at;
    const uint32_t *hb = ha + ((uint64_t)(na + win) << (lg - 5));
    uint32_t acc[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) acc[j] = 0;
    for (uint32_t i = 0; i < nin; ++i) {
        uint32_t a[32], b[32], o[32];
        load32(a, ha);
        load32(b, hb);
        mul<5>(a, b, o);
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] ^= o[j];
        ha += 1ull << (lg - 5);
        hb += 1ull << (lg - 5);
    }
#pragma unroll
    for (int j = 0; j < 32; ++j) sm[at + (j << 8)] = acc[j];
    __syncthreads();
    inverse_levels<13, 5>(sm, P, base, 256);
    store_tile<13>(sm, P, out + ((uint64_t)win << (lg - 5)) + tile_base(P, tile), threadIdx.x, 256);
}

// Two windows at a time: a_0, a_1 (blocks i, i + 1) and B_0, B_1, B_2 (blocks
// i + w ..) give w and w + 1 with three products for four,
//   a_0 B_0 + a_1 B_1 = a_0 (B_0 + B_1) + (a_0 + a_1) B_1,
//   a_0 B_1 + a_1 B_2 = a_1 (B_1 + B_2) + (a_0 + a_1) B_1,
// and both inverses run together, one on each half of the threads.  ALU pipe; the
// two-source extraction of 2^30 bits (64 + 89 blocks) 10.2 -> 9.2 ms against
// k_gf_sum for each window.
__global__ void __launch_bounds__(256) k_gf_sum2(int lg, uint32_t na, uint32_t nb, uint32_t nin, uint32_t nz,
                                                 const Pass *__restrict__ table, const uint32_t *__restrict__ hat,
                                                 uint32_t *__restrict__ out) {
    extern __shared__ __align__(16) uint32_t sm[];
    __shared__ Pass P;
    __shared__ uint32_t base[kMaxLev];
    const uint32_t tile = blockIdx.x & ((1u << (lg - 18)) - 1u), win = 2 * (blockIdx.x >> (lg - 18));
    load_pass(&P, table);
    __syncthreads();
    if (threadIdx.x < P.nlev)
        base[threadIdx.x] = ext_twiddle(P.lev[threadIdx.x], P.lev[threadIdx.x].base[1], tile);
    const uint32_t at = phys(threadIdx.x);
    const uint32_t *h0 = hat + ((uint64_t)tile << 13) + at;
    auto block = [&](uint32_t k) { return h0 + ((uint64_t)k << (lg - 5)); };
    uint32_t w0[32], w1[32], a[32], b[32], o[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) w0[j] = w1[j] = 0;
#pragma unroll 1
    for (uint32_t i = 0; i < nin; i += 2) {
        const bool odd = i + 1 == nin;  // no a_1
        const uint32_t last = nb - 1, k0 = i + win, k1 = k0 + 1 < last ? k0 + 1 : last, k2 = k0 + 2 < last ? k0 + 2 : last;
        const uint32_t *a0 = block(i), *a1 = block(i + 1), *b0 = block(na + k0), *b1 = block(na + k1), *b2 = block(na + k2);
#pragma unroll 1
        for (int t = 0; t < (odd ? 2 : 3); ++t) {
            // t = 0: (a_0 + a_1) B_1 to both; 1: a_0 (B_0 + B_1) to w; 2: a_1 (B_1 + B_2) to w + 1
            load32(a, t == 2 ? a1 : a0);
            if (t == 0 && !odd) {
#pragma unroll
                for (int j = 0; j < 32; ++j) a[j] ^= __ldg(a1 + (j << 8));
            }
            load32(b, b1);
            if (t) {
                const uint32_t *bx = t == 1 ? b0 : b2;
#pragma unroll
                for (int j = 0; j < 32; ++j) b[j] ^= __ldg(bx + (j << 8));
            }
            mul<5>(a, b, o);
            const uint32_t m0 = t == 2 ? 0u : ~0u, m1 = t == 1 ? 0u : ~0u;
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                w0[j] ^= o[j] & m0;
                w1[j] ^= o[j] & m1;
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        sm[at + (j << 8)] = w0[j];
        sm[8192 + at + (j << 8)] = w1[j];
    }
    __syncthreads();
    const uint32_t h = threadIdx.x >> 7, tid = threadIdx.x & 127u;
    uint32_t *mine = sm + 8192 * h;
    for (int l = (int)P.nlev - 1; l >= 0; --l) {
        level<13, 8, 5, true>(mine, P.lev[l], base[l], l >= (int)P.npre, tid, 128);
        __syncthreads();
        if (l == (int)P.npre) {
            transpose_bits<13>(mine, P, tid >> 5, 4);
            __syncthreads();
        }
    }
    if (win + h < nz) store_tile<13>(mine, P, out + ((uint64_t)(win + h) << (lg - 5)) + tile_base(P, tile), tid, 128);
}

// The operands of a dense product as plain bits: a_t at bit 256 + t, b_k at bit k,
// zeros around; z cleared.
__global__ void __launch_bounds__(256) k_gf_tc_prep(const __grid_constant__ Ops q, int lg, uint32_t aw, uint32_t bw,
                                                    uint32_t zw, uint32_t *__restrict__ a, uint32_t *__restrict__ b,
                                                    uint32_t *__restrict__ z) {
    const uint32_t i = blockIdx.x * 256 + threadIdx.x, nw = 1u << (lg - 5);
    uint32_t v[1];
    let_next_start();
    if (i < aw) {
        in_words<1>(q.a0, lin_of(q.a0, false, lg), false, lg, [&](int) -> uint32_t { return i - 8 < nw ? i - 8 : ~0u; }, v);
        a[i] = v[0];
    }
    if (i < bw) {
        in_words<1>(q.b0, lin_of(q.b0, true, lg), true, lg, [&](int) -> uint32_t { return i < nw ? nw - 1 - i : ~0u; }, v);
        b[i] = __brev(v[0]);
    }
    if (i < zw) z[i] = 0;
}

__global__ void __launch_bounds__(256) k_gf_same(const SameOp *__restrict__ ops) {
    const SameOp o = ops[blockIdx.x];
    const uint64_t words = (o.n + 63) >> 6;
    bool any1 = false, any0 = false;
    for (uint64_t w = (uint64_t)blockIdx.y * 256 + threadIdx.x; w < words; w += (uint64_t)gridDim.y * 256) {
        const uint64_t mask = o.n - 64 * w < 64 ? (1ull << (o.n - 64 * w)) - 1 : ~0ull, v = __ldg(o.x + w) & mask;
        any1 |= v != 0;
        any0 |= v != mask;
    }
    any1 = __syncthreads_or(any1);
    any0 = __syncthreads_or(any0);
    if (threadIdx.x == 0) {
        if (any1) atomicOr(o.flags, 1u);
        if (any0) atomicOr(o.flags + 1, 1u);
    }
}

Stages stages_of(int bits) {
    Stages s;
    memset(&s, 0, sizeof(s));
    conv_list(0, bits, &s);
    return s;
}

struct Scope {  // tracing, when there is a context
    alignas(ProfScope) unsigned char mem[sizeof(ProfScope)];
    ProfScope *p = nullptr;
    Scope(cm_ctx *c, const char *name, cudaStream_t st) {
        if (c) p = new (mem) ProfScope(c, name, st);
    }
    ~Scope() {
        if (p) p->~ProfScope();
    }
};

template <int RC>
cudaError_t rows_launch_r(bool inv, const Ops &q, int lg, uint32_t ops, uint32_t *data, cudaStream_t st) {
    cudaError_t e = inv ? smem_attr_once<k_gf_rows<RC, true>>(kRowsSmem) : smem_attr_once<k_gf_rows<RC, false>>(kRowsSmem);
    if (e != cudaSuccess) return e;
    const int r = lg - 16;
    const Stages s = stages_of(r);
    const uint32_t grid = ops * (r > 2 ? 128u >> (9 - r) : 1u);
    if (inv) k_gf_rows<RC, true><<<grid, kRowsThreads, kRowsSmem, st>>>(q, lg, s, data);
    else k_gf_rows<RC, false><<<grid, kRowsThreads, kRowsSmem, st>>>(q, lg, s, data);
    return cudaGetLastError();
}

cudaError_t rows_launch(cm_ctx *c, bool inv, const Ops &q, int lg, uint32_t ops, uint32_t *data, cudaStream_t st) {
    Scope ps(c, inv ? "k_gf_rows_inv" : "k_gf_rows", st);
    switch (lg - 16) {
        case 6: return rows_launch_r<6>(inv, q, lg, ops, data, st);
        case 7: return rows_launch_r<7>(inv, q, lg, ops, data, st);
        case 8: return rows_launch_r<8>(inv, q, lg, ops, data, st);
        case 9: return rows_launch_r<9>(inv, q, lg, ops, data, st);
        default: return rows_launch_r<5>(inv, q, lg, ops, data, st);
    }
}

template <int UB>
cudaError_t units_launch_ub(bool inv, const Ops &q, int lg, uint32_t na, uint32_t nb, uint32_t *data, cudaStream_t st) {
    constexpr uint32_t RPC = kUnitsThreads >> (UB - 1);
    constexpr int smem = (int)(RPC * 3 * (8u << UB) * 4);
    cudaError_t e = inv ? smem_attr_once<k_gf_units<true, UB>>(smem) : smem_attr_once<k_gf_units<false, UB>>(smem);
    if (e != cudaSuccess) return e;
    const uint32_t ra = na << (lg - 8 - UB), rb = nb << (lg - 8 - UB), grid = (ra + RPC - 1) / RPC + (rb + RPC - 1) / RPC;
    if (inv) k_gf_units<true, UB><<<grid, kUnitsThreads, smem, st>>>(q, lg, ra, rb, data);
    else k_gf_units<false, UB><<<grid, kUnitsThreads, smem, st>>>(q, lg, ra, rb, data);
    return cudaGetLastError();
}

// Forward: na arrays of a, nb of b; inverse: na arrays.
cudaError_t units_launch(cm_ctx *c, bool inv, const Ops &q, int lg, uint32_t na, uint32_t nb, uint32_t *data,
                         cudaStream_t st) {
    Scope ps(c, inv ? "k_gf_units_inv" : "k_gf_units", st);
    return lg == 15 ? units_launch_ub<7>(inv, q, lg, na, nb, data, st) : units_launch_ub<8>(inv, q, lg, na, nb, data, st);
}

template <int NB, int FMAX>
cudaError_t mid_launch(int nsm, int lg, uint32_t pairs, const Pass *table, const uint32_t *A, uint32_t *B,
                       cudaStream_t st) {
    using S = MidShape<NB, FMAX>;
    const uint32_t grid = pairs << (lg - 5 - NB);
    cudaError_t e;
    if (grid <= (uint32_t)nsm) {
        if ((e = smem_attr_once<k_gf_mid<NB, FMAX, true>>(2 * S::SMEM1)) != cudaSuccess) return e;
        k_gf_mid<NB, FMAX, true><<<grid, 2 * S::HALF, 2 * S::SMEM1, st>>>(lg, table, A, B);
    } else {
        if ((e = smem_attr_once<k_gf_mid<NB, FMAX, false>>(2 * S::SMEM1)) != cudaSuccess) return e;
        k_gf_mid<NB, FMAX, false><<<grid, S::HALF, 2 * S::SMEM1, st>>>(lg, table, A, B);
    }
    return cudaGetLastError();
}

}  // namespace

void build_tables(Pass *t) {
    for (int lg = kMinLg; lg <= kMaxLg; ++lg) {
        Pass *p = t + 2 * (lg - kMinLg);
        memset(p, 0, 2 * sizeof(Pass));
        build_passes(lg, false, p, p + 1);
    }
    for (int lg = kFewMinLg; lg <= kFewMaxLg; ++lg) {
        Pass *p = t + kFewTables + 2 * (lg - kFewMinLg);
        memset(p, 0, 2 * sizeof(Pass));
        build_passes(lg, true, p, p + 1);
    }
}

static bool summed(const Product &p, const Ops &q) { return p.nin > 1 || (!q.in && q.nz > 1); }

uint64_t product_scratch(const Product &p, const Ops &q) {
    const uint64_t arr = 1ull << (p.lg - 3);
    return (q.na + q.nb) * arr * (summed(p, q) ? 2 : 1);
}

uint32_t product_launches(const Product &p, const Ops &q) {
    const Shape s = shape_of(p.lg);
    return 2 + (s.colr ? 2 : 0) + (s.two ? 2 : 0) + (summed(p, q) ? 2 : 1);
}

cudaError_t launch_same(const SameOp *ops, uint32_t count, cudaStream_t st) {
    k_gf_same<<<dim3(count, 8), 256, 0, st>>>(ops);
    return cudaGetLastError();
}

cudaError_t launch_tc_prep(const Ops &q, const TcShape &s, uint32_t *a, uint32_t *b, uint64_t *z, uint64_t m,
                           cudaStream_t st) {
    const uint64_t zw = 2 * ((m + 63) / 64);
    uint64_t n = s.a_words > s.b_words ? s.a_words : s.b_words;
    if (zw > n) n = zw;
    int lg = 5;
    while ((1ull << lg) < 32 * n) ++lg;
    k_gf_tc_prep<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(q, lg, (uint32_t)s.a_words, (uint32_t)s.b_words, (uint32_t)zw, a,
                                                              b, reinterpret_cast<uint32_t *>(z));
    return cudaGetLastError();
}

cudaError_t launch_product(cm_ctx *c, int nsm, const Product &p, const Ops &q, const Pass *tables, void *scratch,
                           cudaStream_t st) {
    const bool sum = summed(p, q);
    // Few operands: last-pass tiles of 2^12 words, one level more in the column
    // passes, while one SM each holds them all: such a tile's pass is a chain of
    // levels with one warp a scheduler, half as long in its forward half on half
    // the words (one product of 2^24, us: k_gf_mid 84.0 -> 68.1, the column passes
    // 31.9 -> 36.2, the call 167 -> 158).  Not for more: 4096 mixed instances,
    // k_gf_mid 7.06 ms, 9.11 with these tiles.
    const bool few = !sum && p.lg >= kFewMinLg && p.lg <= kFewMaxLg && (uint64_t)q.na << (p.lg - 17) <= (uint64_t)nsm;
    const Shape s = shape_of(p.lg, few);
    const Pass *mid = tables + (few ? kFewTables + 2 * (p.lg - kFewMinLg) : 2 * (p.lg - kMinLg)), *col = mid + 1;
    const uint32_t ops = q.na + q.nb;
    uint32_t *data = static_cast<uint32_t *>(scratch);
    uint32_t *B = data + ((uint64_t)q.na << (p.lg - 5));
    cudaError_t e = cudaSuccess;
    if (s.colr && (e = rows_launch(c, false, q, p.lg, ops, data, st)) != cudaSuccess) return e;
    if ((e = units_launch(c, false, q, p.lg, q.na, q.nb, data, st)) != cudaSuccess) return e;
    if (s.two) {
        Scope ps(c, "k_gf_cols", st);
        k_gf_cols<false><<<ops << (p.lg - 18), kColsThreads, 0, st>>>(p.lg, q.na, col, data);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    uint32_t *out = B;
    if (sum) {
        uint32_t *hat = data + ((uint64_t)ops << (p.lg - 5));
        {
            Scope ps(c, "k_gf_fwd", st);
            k_gf_fwd<<<ops << (p.lg - 18), 128, 0, st>>>(p.lg, q.na, mid, data, hat);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        out = data;  // the operands' arrays are free again: na + nb >= nz of them
        Scope ps(c, "k_gf_sum", st);
        if (q.nz > 1) {
            if ((e = smem_attr_once<k_gf_sum2>(65536)) != cudaSuccess) return e;
            k_gf_sum2<<<(q.nz + 1) / 2 << (p.lg - 18), 256, 65536, st>>>(p.lg, q.na, q.nb, p.nin, q.nz, mid, hat, out);
        } else {
            k_gf_sum<<<1 << (p.lg - 18), 256, 0, st>>>(p.lg, q.na, p.nin, mid, hat, out);
        }
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    } else {
        Scope ps(c, "k_gf_mid", st);
        switch (s.nb) {
            case 10: e = mid_launch<10, 4>(nsm, p.lg, q.na, mid, data, B, st); break;
            case 11: e = mid_launch<11, 5>(nsm, p.lg, q.na, mid, data, B, st); break;
            case 12: e = mid_launch<12, 5>(nsm, p.lg, q.na, mid, data, B, st); break;
            default: e = mid_launch<13, 5>(nsm, p.lg, q.na, mid, data, B, st);
        }
        if (e != cudaSuccess) return e;
    }
    if (s.two) {
        Scope ps(c, "k_gf_cols_inv", st);
        k_gf_cols<true><<<q.nz << (p.lg - 18), kColsThreads, 0, st>>>(p.lg, 0, col, out);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if ((e = units_launch(c, true, q, p.lg, q.nz, 0, out, st)) != cudaSuccess) return e;
    if (s.colr) e = rows_launch(c, true, q, p.lg, q.nz, out, st);
    return e;
}

}  // namespace gf
}  // namespace cm
