// Many inputs under one Toeplitz seed: Z = toep(y) X over GF(2) as a dense
// blocked matrix product (Eq. toep-ext / Eq. toep applied to `count` inputs).
//
// The seed is expanded once into T, the m x n Toeplitz matrix of Eq. toep as
// packed bit rows (T[i][j] = y[(i - j) mod (n + m - 1)], zero-padded to whole
// tiles).  Exact engines multiply T by the packed inputs:
//
//  * kImma: INT8 tensor cores (mma.sync m16n8k32, s8 x s8 -> s32).  Operand
//    fragments are built in registers from the packed bits (4 bits -> 4 bytes of
//    0/1 by one multiply and one mask); the int32 accumulators hold exact
//    counts <= n, and the epilogue keeps bit 0 (mod 2).  sm_103a has no
//    tcgen05 integer kind, so this is the warp-level MMA.
//  * kGf2: CUDA cores.  Over GF(2) a dot product of bit vectors is the parity of
//    popcount(AND); the kernel accumulates XOR(T_word AND X_word) (one LOP3 per
//    32 bit-products) and takes the parity once per output.
//
//  * kBmma: binary tensor cores (mma.sync m16n8k256, b1 x b1 -> s32 with
//    AND-POPC): popcount(row AND column) over 256 bits per instruction from
//    the packed words; exact int32 counts, bit 0 kept.
//
//  * kF4: e2m1 tensor cores (cm_ss_f4.cu): the default from 2^30 bit products on,
//    n <= 2^14 (65536 inputs of 4096 bits, m = 2048: 0.235 ms, kGf2 1.31 ms).
//
// All give identical bits; below that the default picks the fastest of the first
// three on the first call of a shape (timed on that call) and remembers it.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <map>
#include <mutex>
#include <tuple>
#include <utility>
#include <vector>

#include "cm.h"
#include "cm_ctx.h"
#include "cm_internal.h"
#include "cm_ss_f4.h"

namespace cm {
namespace {

constexpr int kSsRows = 64;     // output rows per CTA tile
constexpr int kSsKw = 32;       // 32-bit words of K per smem chunk (1024 bits)
constexpr int kImCols = 128;    // IMMA engine: instances per CTA tile

// T bit rows: word w (32-bit) of row i holds bits j = 32 w .. 32 w + 31.
__global__ void k_toep_rows(const uint64_t *__restrict__ y, uint64_t n, uint64_t m, uint32_t *T,
                            uint32_t rows_pad, uint32_t words_pad) {
    const uint64_t N = n + m - 1;
    const uint64_t total = (uint64_t)rows_pad * words_pad;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t i = t / words_pad, w = t - i * words_pad;
        uint32_t v = 0;
        if (i < m) {
            for (int b = 0; b < 32; ++b) {
                const uint64_t j = 32 * w + b;
                if (j >= n) break;
                const uint64_t k = (i + N - (j % N)) % N;  // (i - j) mod N
                v |= (uint32_t)((__ldg(y + (k >> 6)) >> (k & 63)) & 1ull) << b;
            }
        }
        T[t] = v;
    }
}

// 32-bit word w of instance c (zero past the instance's words).
__device__ __forceinline__ uint32_t x_word(const uint64_t *X, uint64_t wx, uint64_t c, uint64_t w) {
    if (w >= 2 * wx) return 0u;
    const uint64_t v = __ldg(X + c * wx + (w >> 1));
    return (w & 1) ? (uint32_t)(v >> 32) : (uint32_t)v;
}

// ---------------------------------------------------------------------------
// GF(2) engine: thread tile 16 rows x CPT instances, XOR-of-AND accumulators.
// CTA: 8 warps = 4 row groups (16 rows each, 64 rows) x 2 instance groups of
// 32 CPT instances.  CPT = 4 holds 64 accumulators (2 CTAs per SM by
// registers); CPT = 2 holds 32 and fits more CTAs; the autotuner picks.
// ---------------------------------------------------------------------------
template <int CPT>
__global__ void __launch_bounds__(256)
k_ss_gf2(const uint32_t *__restrict__ T, uint32_t words_pad, const uint64_t *__restrict__ X, uint64_t wx,
         uint64_t count, uint64_t *__restrict__ Z, uint64_t wz) {
    constexpr int COLS = 64 * CPT;  // instances per CTA
    __shared__ __align__(16) uint32_t sT[kSsKw][kSsRows + 4];  // [w][row], rows padded (16-B aligned)
    __shared__ __align__(16) uint32_t sX[kSsKw][COLS];         // [w][col]
    __shared__ uint16_t sOut[COLS][4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rg = warp & 3, cg = warp >> 2;
    const uint32_t row0 = blockIdx.x * kSsRows;
    const uint64_t col0 = (uint64_t)blockIdx.y * COLS;
    uint32_t acc[16][CPT];
#pragma unroll
    for (int r = 0; r < 16; ++r)
#pragma unroll
        for (int c = 0; c < CPT; ++c) acc[r][c] = 0u;
    for (uint32_t w0 = 0; w0 < words_pad; w0 += kSsKw) {
        // coalesced reads of T rows; the row padding spreads the transposed stores
        for (int e = threadIdx.x; e < kSsKw * kSsRows; e += 256) {
            const int r = e / kSsKw, w = e % kSsKw;
            sT[w][r] = __ldg(T + (uint64_t)(row0 + r) * words_pad + w0 + w);
        }
        for (int cc = threadIdx.x; cc < COLS; cc += 256) {
            const uint64_t c = col0 + cc;
            for (int w = 0; w < kSsKw; w += 2) {
                uint64_t v = 0;
                if (c < count && (w0 + w) / 2 < wx) v = __ldg(X + c * wx + (w0 + w) / 2);
                sX[w][cc] = (uint32_t)v;
                sX[w + 1][cc] = (uint32_t)(v >> 32);
            }
        }
        __syncthreads();
#pragma unroll 4
        for (int w = 0; w < kSsKw; ++w) {
            uint32_t xv[CPT];
            if constexpr (CPT == 4) {
                const uint4 x4 = *reinterpret_cast<const uint4 *>(&sX[w][cg * 128 + lane * 4]);
                xv[0] = x4.x; xv[1] = x4.y; xv[2] = x4.z; xv[3] = x4.w;
            } else {
                const uint2 x2 = *reinterpret_cast<const uint2 *>(&sX[w][cg * 64 + lane * 2]);
                xv[0] = x2.x; xv[1] = x2.y;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint4 t4 = *reinterpret_cast<const uint4 *>(&sT[w][rg * 16 + q * 4]);
                const uint32_t tv[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int c = 0; c < CPT; ++c) acc[q * 4 + r][c] ^= tv[r] & xv[c];
            }
        }
        __syncthreads();
    }
    // parity of each accumulator: 16 row bits per instance per thread
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        uint32_t bits = 0;
#pragma unroll
        for (int r = 0; r < 16; ++r) bits |= (uint32_t)(__popc(acc[r][c]) & 1) << r;
        sOut[cg * 32 * CPT + lane * CPT + c][rg] = (uint16_t)bits;
    }
    __syncthreads();
    for (int cc = threadIdx.x; cc < COLS; cc += 256) {
        const uint64_t c = col0 + cc;
        if (c < count) {
            const uint64_t word = (uint64_t)sOut[cc][0] | ((uint64_t)sOut[cc][1] << 16) |
                                  ((uint64_t)sOut[cc][2] << 32) | ((uint64_t)sOut[cc][3] << 48);
            Z[c * wz + (row0 >> 6)] = word;
        }
    }
}

// ---------------------------------------------------------------------------
// INT8 tensor-core engine: warp tile 32 rows x 32 instances (2 x 4 m16n8k32).
// ---------------------------------------------------------------------------
// 4 bits -> 4 bytes of 0/1 (bit k of b lands at bit 8k; the shifted copies do
// not overlap, so no carries).
__device__ __forceinline__ uint32_t expand4(uint32_t b) { return (b * 0x00204081u) & 0x01010101u; }

__global__ void __launch_bounds__(256)
k_ss_imma(const uint32_t *__restrict__ T, uint32_t words_pad, const uint64_t *__restrict__ X, uint64_t wx,
          uint64_t count, uint64_t *__restrict__ Z, uint64_t wz) {
    __shared__ __align__(16) uint32_t sT[kSsRows][kSsKw + 1];   // [row][w], padded
    __shared__ __align__(16) uint32_t sX[kImCols][kSsKw + 1];   // [col][w], padded
    __shared__ uint8_t sPar[kImCols][kSsRows];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int wr = warp & 1, wc = warp >> 1;  // warp tile: rows wr*32 .., cols wc*32 ..
    const uint32_t row0 = blockIdx.x * kSsRows;
    const uint64_t col0 = (uint64_t)blockIdx.y * kImCols;
    int acc[2][4][4];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[a][b][k] = 0;
    for (uint32_t w0 = 0; w0 < words_pad; w0 += kSsKw) {
        for (int e = threadIdx.x; e < kSsKw * kSsRows; e += 256) {
            const int r = e / kSsKw, w = e % kSsKw;
            sT[r][w] = __ldg(T + (uint64_t)(row0 + r) * words_pad + w0 + w);
        }
        for (int e = threadIdx.x; e < kSsKw * kImCols; e += 256) {
            const int cc = e / kSsKw, w = e % kSsKw;
            const uint64_t c = col0 + cc;
            sX[cc][w] = c < count ? x_word(X, wx, c, w0 + w) : 0u;
        }
        __syncthreads();
#pragma unroll 2
        for (int w = 0; w < kSsKw; ++w) {  // one k32 step per 32-bit word
            uint32_t afr[2][4], bfr[4][2];
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const uint32_t lo = sT[wr * 32 + a * 16 + g][w], hi = sT[wr * 32 + a * 16 + g + 8][w];
                afr[a][0] = expand4((lo >> (4 * t)) & 0xFu);
                afr[a][1] = expand4((hi >> (4 * t)) & 0xFu);
                afr[a][2] = expand4((lo >> (16 + 4 * t)) & 0xFu);
                afr[a][3] = expand4((hi >> (16 + 4 * t)) & 0xFu);
            }
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const uint32_t xv = sX[wc * 32 + b * 8 + g][w];
                bfr[b][0] = expand4((xv >> (4 * t)) & 0xFu);
                bfr[b][1] = expand4((xv >> (16 + 4 * t)) & 0xFu);
            }
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    asm volatile(
                        "mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
                        "{%8,%9}, {%0,%1,%2,%3};"
                        : "+r"(acc[a][b][0]), "+r"(acc[a][b][1]), "+r"(acc[a][b][2]), "+r"(acc[a][b][3])
                        : "r"(afr[a][0]), "r"(afr[a][1]), "r"(afr[a][2]), "r"(afr[a][3]), "r"(bfr[b][0]),
                          "r"(bfr[b][1]));
        }
        __syncthreads();
    }
    // mod-2 epilogue: accumulator (row g / g+8, cols 2t, 2t+1) -> parity bytes
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int r = wr * 32 + a * 16 + g, cc = wc * 32 + b * 8 + 2 * t;
            sPar[cc][r] = (uint8_t)(acc[a][b][0] & 1);
            sPar[cc + 1][r] = (uint8_t)(acc[a][b][1] & 1);
            sPar[cc][r + 8] = (uint8_t)(acc[a][b][2] & 1);
            sPar[cc + 1][r + 8] = (uint8_t)(acc[a][b][3] & 1);
        }
    __syncthreads();
    // pack: one warp per instance column at a time, 64 rows -> one word
    for (int cc = warp; cc < kImCols; cc += 8) {
        const uint32_t lo = __ballot_sync(0xffffffffu, sPar[cc][lane]);
        const uint32_t hi = __ballot_sync(0xffffffffu, sPar[cc][32 + lane]);
        const uint64_t c = col0 + cc;
        if (lane == 0 && c < count) Z[c * wz + (row0 >> 6)] = ((uint64_t)hi << 32) | lo;
    }
}

// ---------------------------------------------------------------------------
// Binary tensor-core engine: mma.sync m16n8k256 b1 x b1 -> s32 with AND-POPC,
// i.e. popcount(row AND column) over 256 bits per instruction, straight from
// the packed words (no byte expansion).  The counts are exact in int32 (at
// most n) and the epilogue keeps bit 0.  Thread t of a quad holds, per row or
// column, the words w + t and w + 4 + t of a 256-bit step in both operands, so
// A and B cover the same bits of K in the same order and the popcount is the
// dot product whatever the register's bit order.
// CTA: ROWS x 128 instances, 8 warps of (ROWS / 2) rows x 32 instances.
// ---------------------------------------------------------------------------
constexpr int kBmPad = 4;  // row stride 36 words: fragment loads hit 32 distinct banks

template <int ROWS>
__global__ void __launch_bounds__(256)
k_ss_bmma(const uint32_t *__restrict__ T, uint32_t rows_pad, uint32_t words_pad, const uint64_t *__restrict__ X,
          uint64_t wx, uint64_t count, uint64_t *__restrict__ Z, uint64_t wz) {
    constexpr int WM = ROWS / 2, AT = WM / 16;  // warp rows, 16-row A tiles per warp
    static_assert(kImCols * ROWS <= ROWS * (kSsKw + kBmPad) * 4, "parity bytes reuse the T tile");
    __shared__ __align__(16) uint32_t sT[ROWS][kSsKw + kBmPad];
    __shared__ __align__(16) uint32_t sX[kImCols][kSsKw + kBmPad];
    auto sPar = reinterpret_cast<uint8_t (*)[ROWS]>(&sT[0][0]);  // after the last K chunk
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int wr = warp & 1, wc = warp >> 1;  // warp tile: rows wr * WM .., instances wc * 32 ..
    const uint32_t row0 = blockIdx.x * ROWS;
    const uint64_t col0 = (uint64_t)blockIdx.y * kImCols;
    int acc[AT][4][4];
#pragma unroll
    for (int a = 0; a < AT; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[a][b][k] = 0;
    for (uint32_t w0 = 0; w0 < words_pad; w0 += kSsKw) {
        // 16-byte loads: T rows (words_pad is a multiple of kSsKw), X instances (wx u64 words each)
        for (int e = threadIdx.x; e < ROWS * (kSsKw / 4); e += 256) {
            const int r = e / (kSsKw / 4), q = e % (kSsKw / 4);
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (row0 + r < rows_pad)
                v = __ldg(reinterpret_cast<const uint4 *>(T + (uint64_t)(row0 + r) * words_pad + w0) + q);
            *reinterpret_cast<uint4 *>(&sT[r][4 * q]) = v;
        }
        for (int e = threadIdx.x; e < kImCols * (kSsKw / 4); e += 256) {
            const int cc = e / (kSsKw / 4), q = e % (kSsKw / 4);
            const uint64_t c = col0 + cc, u = w0 / 2 + 2 * q;  // first u64 word of this 16 bytes
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (c < count) {
                const uint64_t *src = X + c * wx + u;
                const uint64_t lo = u < wx ? __ldg(src) : 0ull, hi = u + 1 < wx ? __ldg(src + 1) : 0ull;
                v = make_uint4((uint32_t)lo, (uint32_t)(lo >> 32), (uint32_t)hi, (uint32_t)(hi >> 32));
            }
            *reinterpret_cast<uint4 *>(&sX[cc][4 * q]) = v;
        }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kSsKw; w += 8) {  // one k256 step per 8 words
            uint32_t afr[AT][4], bfr[4][2];
#pragma unroll
            for (int a = 0; a < AT; ++a) {
                const int r = wr * WM + a * 16 + g;
                afr[a][0] = sT[r][w + t];
                afr[a][1] = sT[r + 8][w + t];
                afr[a][2] = sT[r][w + 4 + t];
                afr[a][3] = sT[r + 8][w + 4 + t];
            }
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int cc = wc * 32 + b * 8 + g;
                bfr[b][0] = sX[cc][w + t];
                bfr[b][1] = sX[cc][w + 4 + t];
            }
#pragma unroll
            for (int a = 0; a < AT; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    asm volatile(
                        "mma.sync.aligned.m16n8k256.row.col.s32.b1.b1.s32.and.popc {%0,%1,%2,%3}, "
                        "{%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                        : "+r"(acc[a][b][0]), "+r"(acc[a][b][1]), "+r"(acc[a][b][2]), "+r"(acc[a][b][3])
                        : "r"(afr[a][0]), "r"(afr[a][1]), "r"(afr[a][2]), "r"(afr[a][3]), "r"(bfr[b][0]),
                          "r"(bfr[b][1]));
        }
        __syncthreads();
    }
    // mod-2 epilogue: accumulator (row g / g + 8, instances 2t, 2t + 1) -> parity bytes
#pragma unroll
    for (int a = 0; a < AT; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int r = wr * WM + a * 16 + g, cc = wc * 32 + b * 8 + 2 * t;
            sPar[cc][r] = (uint8_t)(acc[a][b][0] & 1);
            sPar[cc + 1][r] = (uint8_t)(acc[a][b][1] & 1);
            sPar[cc][r + 8] = (uint8_t)(acc[a][b][2] & 1);
            sPar[cc + 1][r + 8] = (uint8_t)(acc[a][b][3] & 1);
        }
    __syncthreads();
    // pack: one warp per (instance, 64-row word) at a time
    for (int e = warp; e < kImCols * (ROWS / 64); e += 8) {
        const int cc = e / (ROWS / 64), h = e % (ROWS / 64);
        const uint32_t lo = __ballot_sync(0xffffffffu, sPar[cc][64 * h + lane]);
        const uint32_t hi = __ballot_sync(0xffffffffu, sPar[cc][64 * h + 32 + lane]);
        const uint64_t c = col0 + cc, zw = (row0 >> 6) + h;
        if (lane == 0 && c < count && zw < wz) Z[c * wz + zw] = ((uint64_t)hi << 32) | lo;
    }
}

// CM_ENGINE_AUTO takes the tcgen05 engine for this many bit products or more.
// Measured, us a call, CUDA cores / tcgen05 (n x m x count): 4096 x 2048 x 65536
// 1309 / 232, 8000 x 6000 x 300 169 / 44, 4096 x 2048 x 300 59 / 28, 1000 x 300 x
// 4096 (2^30.2) 22.3 / 16.6; below, either is launch latency.  So it is however few
// the inputs or the rows: 16384 x 65536 x 1 (a 512 MB matrix) 2708 / 270 and x 64
// 2753 / 283, 4096 x 4096 x 64 76 / 35, 1024 x 1024 x 1024 31.8 / 24.2, 4096 x 64 x
// 16384 42.9 / 32.2; over 208 shapes from 2^30 to 2^37 the ratio was 0.07 to 0.76.
constexpr double kSsF4Min = 1073741824.0;

std::mutex g_engine_mu;
// (n, m, engine asked for) -> the variant the first call of that shape timed fastest
std::map<std::tuple<uint64_t, uint64_t, int>, int> g_engine_choice;

// shapes whose last CM_ENGINE_AUTO call was long enough for the tcgen05 engine
std::map<std::pair<uint64_t, uint64_t>, int> g_engine_wide;

// Engine variants the autotuner times: the INT8 engine, the GF(2) engine
// with 4 or 2 instances per thread, and the binary engine with 64- or 128-row
// tiles.
constexpr int kVarImma = 0, kVarGf2x4 = 1, kVarGf2x2 = 2, kVarBmma64 = 3, kVarBmma128 = 4, kVarF4 = 5;
inline int engine_of(int var) {
    if (var == kVarF4) return CM_ENGINE_F4;
    return var == kVarImma ? CM_ENGINE_IMMA : (var >= kVarBmma64 ? CM_ENGINE_BMMA : CM_ENGINE_GF2);
}

cm_status launch_variant(int var, const uint32_t *T, uint32_t rows_pad, uint32_t words_pad,
                         const uint64_t *X, uint64_t wx, uint64_t count, uint64_t *Z, uint64_t wz,
                         cm_ctx *ctx, cudaStream_t st) {
    if (var == kVarGf2x4) {
        dim3 grid(rows_pad / kSsRows, (unsigned)((count + 255) / 256));
        ProfScope ps(ctx, "k_ss_gf2", st);
        k_ss_gf2<4><<<grid, 256, 0, st>>>(T, words_pad, X, wx, count, Z, wz);
    } else if (var == kVarGf2x2) {
        dim3 grid(rows_pad / kSsRows, (unsigned)((count + 127) / 128));
        ProfScope ps(ctx, "k_ss_gf2", st);
        k_ss_gf2<2><<<grid, 256, 0, st>>>(T, words_pad, X, wx, count, Z, wz);
    } else if (var == kVarBmma64 || var == kVarBmma128) {
        const int rows = var == kVarBmma64 ? 64 : 128;
        dim3 grid((rows_pad + rows - 1) / rows, (unsigned)((count + kImCols - 1) / kImCols));
        ProfScope ps(ctx, "k_ss_bmma", st);
        if (var == kVarBmma64)
            k_ss_bmma<64><<<grid, 256, 0, st>>>(T, rows_pad, words_pad, X, wx, count, Z, wz);
        else
            k_ss_bmma<128><<<grid, 256, 0, st>>>(T, rows_pad, words_pad, X, wx, count, Z, wz);
    } else {
        dim3 grid(rows_pad / kSsRows, (unsigned)((count + kImCols - 1) / kImCols));
        ProfScope ps(ctx, "k_ss_imma", st);
        k_ss_imma<<<grid, 256, 0, st>>>(T, words_pad, X, wx, count, Z, wz);
    }
    return cudaGetLastError() == cudaSuccess ? CM_OK : CM_EDEVICE;
}

}  // namespace
}  // namespace cm

using namespace cm;

extern "C" cm_status cm_batch_toeplitz_shared_seed(cm_ctx *ctx, const uint64_t *y, uint64_t n, uint64_t m,
                                                   const uint64_t *X, uint64_t count, uint64_t *Z,
                                                   int engine, cm_stream stream) {
    if (!ctx || !y || !X || !Z || n == 0 || m == 0 || count == 0) return CM_EINVAL;
    if (engine != CM_ENGINE_AUTO && engine != CM_ENGINE_IMMA && engine != CM_ENGINE_GF2 && engine != CM_ENGINE_BMMA &&
        engine != CM_ENGINE_F4)
        return CM_EINVAL;
    if (n > (1ull << 24) || m > (1ull << 24) || (n * m) > (1ull << 34) || count > (1ull << 31))
        return CM_EINVAL;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CM_EDEVICE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (engine == CM_ENGINE_F4 && n > kSsF4MaxN) return CM_EINVAL;
    if (engine == CM_ENGINE_F4 ||
        (engine == CM_ENGINE_AUTO && n <= kSsF4MaxN && ss_f4_bytes(n, m) <= ctx->budget &&
         (double)n * (double)m * (double)count >= kSsF4Min)) {
        const uint64_t tb = ss_f4_bytes(n, m);
        if (tb > ctx->budget) return CM_ENOMEM;
        void *Tf = nullptr;
        if (cudaMallocFromPoolAsync(&Tf, tb, ctx->pool, st) == cudaSuccess) {
            cudaError_t e;
            {
                ProfScope ps(ctx, "k_ss_f4_rows", st);
                e = launch_ss_f4_rows(y, n, m, Tf, ctx->nsm, st);
            }
            if (e == cudaSuccess) {
                ProfScope ps(ctx, "k_ss_f4", st);
                e = launch_ss_f4(Tf, n, m, X, count, Z, ctx->d_status, ctx->nsm, st);
            }
            cudaFreeAsync(Tf, st);
            if (engine == CM_ENGINE_AUTO) {
                std::lock_guard<std::mutex> lock(g_engine_mu);
                g_engine_wide[{n, m}] = kVarF4;
            }
            return e == cudaSuccess ? CM_OK : CM_EDEVICE;
        }
        cudaGetLastError();
        if (engine == CM_ENGINE_F4) return CM_ENOMEM;
    }
    const uint32_t rows_pad = (uint32_t)((m + kSsRows - 1) / kSsRows * kSsRows);
    const uint32_t words_pad = (uint32_t)((n + 32 * kSsKw - 1) / (32 * kSsKw) * kSsKw);
    const uint64_t wx = (n + 63) / 64, wz = (m + 63) / 64;
    const size_t tbytes = (size_t)rows_pad * words_pad * sizeof(uint32_t);
    if (tbytes > ctx->budget) return CM_ENOMEM;
    void *Tv = nullptr;
    if (cudaMallocFromPoolAsync(&Tv, tbytes, ctx->pool, st) != cudaSuccess) {
        cudaGetLastError();
        return CM_ENOMEM;
    }
    uint32_t *T = static_cast<uint32_t *>(Tv);
    cm_status s = CM_OK;
    {
        ProfScope ps(ctx, "k_toep_rows", st);
        const uint64_t total = (uint64_t)rows_pad * words_pad;
        uint64_t blocks = (total + 255) / 256;
        if (blocks > (uint64_t)ctx->nsm * 16) blocks = (uint64_t)ctx->nsm * 16;
        k_toep_rows<<<(unsigned)blocks, 256, 0, st>>>(y, n, m, T, rows_pad, words_pad);
        if (cudaGetLastError() != cudaSuccess) s = CM_EDEVICE;
    }
    // candidates of the engine asked for; the first call of a shape times them
    // on its own data and later calls take the fastest
    std::vector<int> cand;
    if (engine == CM_ENGINE_AUTO || engine == CM_ENGINE_IMMA) cand.push_back(kVarImma);
    if (engine == CM_ENGINE_AUTO || engine == CM_ENGINE_GF2) {
        cand.push_back(kVarGf2x4);
        cand.push_back(kVarGf2x2);
    }
    if (engine == CM_ENGINE_AUTO || engine == CM_ENGINE_BMMA) {
        cand.push_back(kVarBmma64);
        cand.push_back(kVarBmma128);
    }
    int var = cand[0];
    if (s == CM_OK && cand.size() > 1) {
        std::lock_guard<std::mutex> lock(g_engine_mu);
        if (engine == CM_ENGINE_AUTO) g_engine_wide.erase({n, m});
        const auto key = std::make_tuple(n, m, engine);
        auto it = g_engine_choice.find(key);
        if (it != g_engine_choice.end()) {
            var = it->second;
        } else {
            float best = 1e30f;
            cudaEvent_t e0, e1;
            cudaEventCreate(&e0);
            cudaEventCreate(&e1);
            for (int v : cand) {
                launch_variant(v, T, rows_pad, words_pad, X, wx, count, Z, wz, ctx, st);  // warm-up
                cudaEventRecord(e0, st);
                s = launch_variant(v, T, rows_pad, words_pad, X, wx, count, Z, wz, ctx, st);
                cudaEventRecord(e1, st);
                cudaEventSynchronize(e1);
                float ms = 0.f;
                cudaEventElapsedTime(&ms, e0, e1);
                if (s != CM_OK) break;
                if (ms < best) {
                    best = ms;
                    var = v;
                }
            }
            cudaEventDestroy(e0);
            cudaEventDestroy(e1);
            if (s == CM_OK) g_engine_choice[key] = var;
        }
    }
    if (s == CM_OK) s = launch_variant(var, T, rows_pad, words_pad, X, wx, count, Z, wz, ctx, st);
    cudaFreeAsync(Tv, st);
    return s;
}

extern "C" int cm_shared_seed_engine(uint64_t n, uint64_t m) {
    std::lock_guard<std::mutex> lock(g_engine_mu);
    if (g_engine_wide.count({n, m})) return CM_ENGINE_F4;
    auto it = g_engine_choice.find(std::make_tuple(n, m, (int)CM_ENGINE_AUTO));
    if (it == g_engine_choice.end()) return CM_ENGINE_AUTO;
    return engine_of(it->second);
}
