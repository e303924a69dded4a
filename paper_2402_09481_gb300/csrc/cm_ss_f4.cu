// Many inputs under one Toeplitz seed on the 5th-generation tensor cores:
// Z = toep(y) X as an e2m1 product with 0 / 1 operands (tcgen05.mma kind::mxf4,
// every block scale 1, float accumulators in tensor memory), parities in the
// epilogue.
//
// sm_103a has no integer tcgen05 kind, but counts are exact in float: a bit is
// 0.5 (nibble 1, so that a shift and a mask make eight elements), products are
// 0.25, and the epilogue adds 2^21, whose unit in the last place is 0.25: bit 0
// of the word is the count's parity.
//
// A CTA makes 256 inputs x 224 outputs: two accumulators of 128 x 224 and 64
// columns of scales fill tensor memory; 256 columns of K a stage, three stages.
//   warps 4..11  input bits -> nibbles, swizzled to shared memory (a shift and a
//                mask per eight elements)
//   warp 12      bulk copies of the matrix, expanded once per call into the
//                swizzled order of its shared-memory tiles (28 KB a stage)
//   warp 13      issues the MMAs (2 x 4 of 128 x 224 x 64 a stage)
//   warps 0..3   accumulators -> parity words, 28 bytes a row
// Elements lie along K in the order the cheap expansion gives (bit q + 4 b of a
// 32-bit word at nibble b of word q) in both operands.  Shared-memory traffic
// bounds it (operands in and, for two MMAs, out again: 37 KB per step of K = 64).
// 65536 inputs of 4096 bits, m = 2048: 232 us, 4.7 PFLOP/s (the CUDA-core engine,
// AND / XOR on words: 1309 us; an e4m3 form of this kernel: 369 us; input loads a
// row a lane instead of eight rows a warp: 305 us).
//
// Every wait has a limit, after which the kernel records CM_FLAG_TIMEOUT and
// ends.
#include <cuda_runtime.h>
#include <stdint.h>

#include "cm_internal.h"
#include "cm_ss_f4.h"
#include "tc05.cuh"

namespace cm {

using namespace tc;

namespace {

constexpr int kStages = 3, kChunk = 256;              // K elements a stage: rows of 128 bytes
constexpr int kInBytes = 256 * 128, kTileBytes = kRows * 128;
constexpr int kStageBytes = kInBytes + kTileBytes;
constexpr int kSmem = kStages * kStageBytes + 1024;   // 1 KB to align
constexpr int kF4Threads = 14 * 32;

__global__ void __launch_bounds__(kF4Threads, 1) k_ss_f4(const uint8_t *__restrict__ T, uint32_t chunks, uint32_t pblocks,
                                                       const uint64_t *__restrict__ X, uint64_t n, uint64_t wx,
                                                       uint64_t count, uint64_t *__restrict__ Z,
                                                       uint64_t wz, uint64_t units, uint32_t *status) {
    extern __shared__ uint8_t raw[];
    __shared__ __align__(8) uint64_t bars[2 * kStages + 2];
    __shared__ uint32_t tmem_at;
    __shared__ volatile uint32_t dead;
    uint8_t *base = raw + ((1024u - (saddr(raw) & 1023u)) & 1023u);
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
    const uint32_t full = saddr(bars), empty = saddr(bars + kStages), accfull = saddr(bars + 2 * kStages),
                   accempty = accfull + 8;
    if (threadIdx.x == 0) {
        dead = 0;
        for (int s = 0; s < kStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full + 8 * s), "r"(257));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(empty + 8 * s), "r"(1));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(accfull), "r"(1));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(accempty), "r"(128));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 13) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(saddr(&tmem_at)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_at;
    if (warp < 4) set_scales(tmem, warp);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

    if (warp >= 4 && warp < 12) {
        // rows 8 i + lane / 4 of the warp's 32, 64-bit word lane % 4 of a stage's
        // four: a load touches 8 rows' sectors, a store 8 distinct 16-byte pieces
        const uint32_t r0 = (warp - 4) * 32 + (lane >> 2), q = lane & 3u;
        uint32_t it = 0;
        bool ok = true;
        for (uint64_t u = blockIdx.x; u < units && ok; u += gridDim.x) {
            const uint64_t c0 = u / pblocks * 256 + r0;
            const uint64_t *row = X + c0 * wx + q;
            auto load = [&](uint32_t k, uint64_t (&w)[4]) {
                const uint64_t j = 4ull * k + q;
                const uint64_t keep = j + 1 < wx ? ~0ull : j < wx ? ((n & 63) ? (1ull << (n & 63)) - 1 : ~0ull) : 0ull;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    w[i] = keep && c0 + 8 * i < count ? __ldg(row + 8 * i * wx + 4ull * k) & keep : 0ull;
            };
            uint64_t w[4], nx[4];
            load(0, w);
            for (uint32_t k = 0; k < chunks; ++k, ++it) {
                if (k + 1 < chunks) load(k + 1, nx);
                const uint32_t s = it % kStages, ph = (it / kStages) & 1u;
                if (!(ok = wait(empty + 8 * s, ph ^ 1u, &dead))) break;
                uint8_t *dst = base + s * kStageBytes + r0 * 128;
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint32_t b = (uint32_t)(w[i] >> (32 * h));
                        *reinterpret_cast<uint4 *>(dst + i * 1024 + (((2 * q + h) ^ (r0 & 7u)) << 4)) =
                            nibbles(b);
                    }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                arrive(full + 8 * s);
#pragma unroll
                for (int i = 0; i < 4; ++i) w[i] = nx[i];
            }
        }
    } else if (warp == 12 && lane == 0) {
        uint32_t it = 0;
        bool ok = true;
        for (uint64_t u = blockIdx.x; u < units && ok; u += gridDim.x) {
            const uint8_t *src = T + (u % pblocks) * (uint64_t)chunks * kTileBytes;
            for (uint32_t k = 0; k < chunks; ++k, ++it) {
                const uint32_t s = it % kStages, ph = (it / kStages) & 1u;
                if (!(ok = wait(empty + 8 * s, ph ^ 1u, &dead))) break;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full + 8 * s), "r"(kTileBytes) : "memory");
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                        saddr(base + s * kStageBytes + kInBytes)),
                    "l"(src + (uint64_t)k * kTileBytes), "r"(kTileBytes), "r"(full + 8 * s)
                    : "memory");
            }
        }
    } else if (warp == 13 && lane == 0) {
        uint32_t it = 0, acc = 0;
        bool ok = true;
        for (uint64_t u = blockIdx.x; u < units && ok; u += gridDim.x, ++acc) {
            if (!(ok = wait(accempty, (acc & 1u) ^ 1u, &dead))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (uint32_t k = 0; k < chunks; ++k, ++it) {
                const uint32_t s = it % kStages, ph = (it / kStages) & 1u;
                if (!(ok = wait(full + 8 * s, ph, &dead))) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t at = saddr(base + s * kStageBytes);
                const uint64_t a = operand(at), a2 = operand(at + kInBytes / 2), b = operand(at + kInBytes);
#pragma unroll
                for (int q = 0; q < 4; ++q) {  // 32 bytes of K: 2 units of the descriptor's address
                    mma(tmem, a + 2 * q, b + 2 * q, tmem + kScaleCol, k || q);
                    mma(tmem + kRows, a2 + 2 * q, b + 2 * q, tmem + kScaleCol, k || q);
                }
                commit(empty + 8 * s);
            }
            if (ok) commit(accfull);
        }
    } else if (warp < 4) {
        uint32_t acc = 0;
        for (uint64_t u = blockIdx.x; u < units; u += gridDim.x, ++acc) {
            if (!wait_warp(accfull, acc & 1u, &dead)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t pb = u % pblocks;
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                const uint64_t c = u / pblocks * 256 + h * 128 + threadIdx.x;
                uint32_t word[7];
#pragma unroll
                for (int q = 0; q < 7; ++q) {
                    word[q] = parities(tmem + ((warp * 32u) << 16) + kRows * h + 32 * q);
                }
                if (c < count) {
                    uint32_t *row = reinterpret_cast<uint32_t *>(Z + c * wz);
#pragma unroll
                    for (int q = 0; q < 7; ++q)
                        if (7 * pb + q < 2 * wz) row[7 * pb + q] = word[q];  // rows past m are 0 in the matrix
                    if (7 * pb + 7 < 2 * wz && pb + 1 == pblocks) row[7 * pb + 7] = 0;
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            arrive(accempty);
        }
    }
    __syncwarp();
    if (dead) __nanosleep(1000000);  // copies and MMAs still in flight end by themselves
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && dead) atomicOr(status, kFlagTimeout);
    if (warp == 13) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
    }
}

// The matrix in tile order: block (p, k) holds rows 224 p .. of the Toeplitz
// matrix, columns 256 k .. as nibbles, rows of 128 bytes with their 16-byte pieces
// exchanged by row mod 8.  One thread a row's 32 columns.
__global__ void __launch_bounds__(256) k_ss_f4_rows(const uint32_t *__restrict__ y, uint64_t n, uint64_t m, uint32_t chunks,
                                                    uint8_t *__restrict__ T, uint64_t total) {
    const uint64_t N = n + m - 1;
    for (uint64_t t = (uint64_t)blockIdx.x * 256 + threadIdx.x; t < total; t += (uint64_t)gridDim.x * 256) {
        const uint32_t g = (uint32_t)(t & 7u);
        const uint64_t rr = t >> 3, blk = rr / kRows, p = blk / chunks, k = blk - p * chunks;
        const uint32_t r = (uint32_t)(rr - blk * kRows);
        const uint64_t i = kRows * p + r, j0 = (uint64_t)kChunk * k + 32 * g;
        uint32_t w = 0;  // bit t: y[(i - j0 - t) mod N]
        if (i < m && j0 < n) {
            const uint32_t cnt = n - j0 < 32 ? (uint32_t)(n - j0) : 32u;
            int64_t lo = (int64_t)i - (int64_t)j0 - (int64_t)(cnt - 1);  // ascending run lo .. lo + cnt - 1
            uint32_t v = 0;
            if (lo >= 0 || lo + (int64_t)cnt <= 0) {
                if (lo < 0) lo += (int64_t)N;
                const uint32_t sh = (uint32_t)lo & 31u;
                const uint32_t a = __ldg(y + (lo >> 5)), b = sh + cnt > 32 ? __ldg(y + (lo >> 5) + 1) : 0u;
                v = __funnelshift_r(a, b, sh);
            } else {
                for (uint32_t b = 0; b < cnt; ++b) {
                    int64_t q = lo + b;
                    if (q < 0) q += (int64_t)N;
                    v |= ((__ldg(y + (q >> 5)) >> (q & 31)) & 1u) << b;
                }
            }
            w = __brev(v) >> (32 - cnt);
            if (cnt < 32) w &= (1u << cnt) - 1u;
        }
        uint8_t *row = T + blk * kTileBytes + r * 128;
        *reinterpret_cast<uint4 *>(row + ((g ^ (r & 7u)) << 4)) = nibbles(w);
    }
}

__global__ void __launch_bounds__(256) k_ss_f4_pack(const uint32_t *__restrict__ G, uint64_t gw, uint64_t m, uint32_t chunks,
                                                    uint8_t *__restrict__ T, uint64_t total) {
    for (uint64_t t = (uint64_t)blockIdx.x * 256 + threadIdx.x; t < total; t += (uint64_t)gridDim.x * 256) {
        const uint32_t g = (uint32_t)(t & 7u);
        const uint64_t rr = t >> 3, blk = rr / kRows, p = blk / chunks, k = blk - p * chunks;
        const uint32_t r = (uint32_t)(rr - blk * kRows);
        const uint64_t i = kRows * p + r, j = 8 * k + g;
        const uint32_t w = i < m && j < gw ? __ldg(G + i * gw + j) : 0u;
        *reinterpret_cast<uint4 *>(T + blk * kTileBytes + r * 128 + ((g ^ (r & 7u)) << 4)) = nibbles(w);
    }
}

}  // namespace

uint64_t ss_f4_bytes(uint64_t n, uint64_t m) {
    return (m + kRows - 1) / kRows * ((n + kChunk - 1) / kChunk) * kTileBytes;
}

cudaError_t launch_ss_f4_rows(const uint64_t *y, uint64_t n, uint64_t m, void *T, int nsm, cudaStream_t st) {
    const uint64_t total = ss_f4_bytes(n, m) / 16;
    const uint64_t blocks = (total + 255) / 256, cap = (uint64_t)nsm * 16;
    k_ss_f4_rows<<<(unsigned)(blocks < cap ? blocks : cap), 256, 0, st>>>(
        reinterpret_cast<const uint32_t *>(y), n, m, (uint32_t)((n + kChunk - 1) / kChunk), static_cast<uint8_t *>(T), total);
    return cudaGetLastError();
}

cudaError_t launch_ss_f4_pack(const uint32_t *G, uint64_t gw, uint64_t n, uint64_t m, void *T, int nsm, cudaStream_t st) {
    const uint64_t total = ss_f4_bytes(n, m) / 16, blocks = (total + 255) / 256, cap = (uint64_t)nsm * 16;
    k_ss_f4_pack<<<(unsigned)(blocks < cap ? blocks : cap), 256, 0, st>>>(
        G, gw, m, (uint32_t)((n + kChunk - 1) / kChunk), static_cast<uint8_t *>(T), total);
    return cudaGetLastError();
}

cudaError_t launch_ss_f4(const void *T, uint64_t n, uint64_t m, const uint64_t *X, uint64_t count, uint64_t *Z,
                         uint32_t *status, int nsm, cudaStream_t st) {
    cudaError_t e = smem_attr_once<k_ss_f4>(kSmem);
    if (e != cudaSuccess) return e;
    const uint64_t pblocks = (m + kRows - 1) / kRows, units = (count + 255) / 256 * pblocks;
    k_ss_f4<<<(unsigned)(units < (uint64_t)nsm ? units : nsm), kF4Threads, kSmem, st>>>(
        static_cast<const uint8_t *>(T), (uint32_t)((n + kChunk - 1) / kChunk), (uint32_t)pblocks, X, n, (n + 63) / 64, count,
        Z, (m + 63) / 64, units, status);
    return cudaGetLastError();
}

}  // namespace cm
