// Short products (K + m - 1 <= 2^13) in one launch without a transform.
//
// Each CTA makes 32 output bits: its warps share the words of a; a lane that
// holds a word of a and the 63 bits of b it meets adds a & (b >> j) to
// accumulator j, one funnel shift and one LOP3 for 32 bit products.  The 32
// accumulators are reduced across the warp by halving exchanges (each step
// sends the half another lane keeps), so that lane j ends with the parity word
// of output j.  At most 2^23.4 bit products over a few hundred CTAs: the call is
// launch latency and one chain of loads, where the one-CTA transform ran 40
// barriers on one SM (n = 4096, m = 2048: 18.5 -> 4.8 us a call, host included).
#include <cuda_runtime.h>
#include <stdint.h>

#include "cm_gf2.h"
#include "cm_internal.h"

namespace cm {
namespace gf {

namespace {

constexpr int kDenseWarps = 4;

// Bits idx .. idx + cnt - 1 of src (cnt <= 32), touching only their words.
__device__ __forceinline__ uint32_t bits_at(const uint32_t *src, uint32_t idx, uint32_t cnt) {
    const uint32_t w = idx >> 5, sh = idx & 31u;
    const uint32_t lo = cnt ? __ldg(src + w) : 0u, hi = sh + cnt > 32 ? __ldg(src + w + 1) : 0u;
    return __funnelshift_r(lo, hi, sh) & (cnt < 32 ? (1u << cnt) - 1u : ~0u);
}

// The operands as 32-bit numbers: a_t = x[n - 1 - t] (back) or x[t], 0 past n;
// b_k = y[(k + off) mod len_y] for k < len (at most one wrap).
struct DenseArgs {
    const uint32_t *x, *y;
    uint32_t n, len_y, off, len, K, m;
    bool back;
};

__device__ __forceinline__ uint32_t a_word(const DenseArgs &q, uint32_t t) {
    const uint32_t left = q.n > t ? q.n - t : 0u, cnt = left < 32 ? left : 32u;
    if (!q.back) return bits_at(q.x, t, cnt);
    return cnt ? __brev(bits_at(q.x, left - cnt, cnt)) >> (32 - cnt) : 0u;
}

__device__ __forceinline__ uint32_t b_word(const DenseArgs &q, uint32_t k) {
    const uint32_t left = q.len > k ? q.len - k : 0u, want = left < 32 ? left : 32u;
    uint32_t idx = k + q.off;
    if (idx >= q.len_y) idx -= q.len_y;
    const uint32_t run = q.len_y > idx ? q.len_y - idx : 0u, c1 = want < run ? want : run;
    uint32_t v = bits_at(q.y, idx, c1);
    if (c1 < want) v |= bits_at(q.y, 0, want - c1) << c1;
    return v;
}

__global__ void __launch_bounds__(32 * kDenseWarps) k_gf_dense(const __grid_constant__ DenseArgs q, bool check, 
                                                               uint32_t *__restrict__ z, uint32_t *status,
                                                               uint32_t *pre) {
    const uint32_t K = q.K, m = q.m;
    __shared__ uint32_t part[kDenseWarps], seen1[kDenseWarps], seen0[kDenseWarps];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, i0 = 32 * blockIdx.x;
    uint32_t acc[32], any1 = 0, any0 = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) acc[j] = 0;
    for (uint32_t t = 32 * threadIdx.x; t < K; t += 32 * 32 * kDenseWarps) {
        const uint32_t av = a_word(q, t), b0 = b_word(q, t + i0), b1 = b_word(q, t + i0 + 32);
        any1 |= av;
        any0 |= ~av & (K - t < 32 ? (1u << (K - t)) - 1u : ~0u);
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] ^= av & __funnelshift_r(b0, b1, j);
    }
    // lane l keeps accumulators whose index agrees with l in the bits done so far
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const bool up = lane & s;
#pragma unroll
        for (int j = 0; j < s; ++j) {
            const uint32_t send = up ? acc[j] : acc[j + s];
            acc[j] = (up ? acc[j + s] : acc[j]) ^ __shfl_xor_sync(0xFFFFFFFFu, send, s);
        }
    }
    const uint32_t word = __ballot_sync(0xFFFFFFFFu, __popc(acc[0]) & 1);
    if (check) {
        any1 = __ballot_sync(0xFFFFFFFFu, any1 != 0);
        any0 = __ballot_sync(0xFFFFFFFFu, any0 != 0);
    }
    if (lane == 0) {
        part[warp] = word;
        seen1[warp] = any1;
        seen0[warp] = any0;
    }
    __syncthreads();
    if (threadIdx.x) return;
    uint32_t v = 0;
    any1 = any0 = 0;
#pragma unroll
    for (int w = 0; w < kDenseWarps; ++w) {
        v ^= part[w];
        any1 |= seen1[w];
        any0 |= seen0[w];
    }
    if (pre && blockIdx.x == 0) {
        pre[0] = any1;
        pre[1] = any0;
    }
    if (check && !(any1 && any0)) {  // a constant Dodis et al. input
        v = 0;
        if (blockIdx.x == 0) atomicOr(status, kFlagPrecond);
    }
    if (i0 >= m) v = 0;  // the upper half of the last word
    else if (m - i0 < 32) v &= (1u << (m - i0)) - 1u;
    z[blockIdx.x] = v;
}

}  // namespace

cudaError_t launch_dense(const BitMap &a, const BitMap &b, uint32_t K, uint32_t m, bool check, uint64_t *z,
                         uint32_t *status, uint32_t *pre, cudaStream_t st) {
    DenseArgs q;
    q.x = reinterpret_cast<const uint32_t *>(a.src);
    q.y = reinterpret_cast<const uint32_t *>(b.src);
    q.n = (uint32_t)a.srclen;
    q.back = a.mode == kReverse;
    q.len_y = (uint32_t)b.srclen;
    q.off = (uint32_t)b.off;
    q.len = (uint32_t)b.len;
    q.K = K;
    q.m = m;
    k_gf_dense<<<2 * ((m + 63) / 64), 32 * kDenseWarps, 0, st>>>(q, check, reinterpret_cast<uint32_t *>(z), status, pre);
    return cudaGetLastError();
}

}  // namespace gf
}  // namespace cm
