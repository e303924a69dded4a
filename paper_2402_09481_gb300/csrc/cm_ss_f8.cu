// Many inputs under one Toeplitz seed on the 5th-generation tensor cores:
// Z = toep(y) X as an e4m3 product with 0 / 1 operands (tcgen05.mma
// kind::f8f6f4, float accumulators in tensor memory), parities in the epilogue.
//
// sm_103a has no integer tcgen05 kind, but counts are exact in float: an input
// bit is 2^-6 (byte 0x08, so that a shift and a mask make four elements), a
// matrix bit 1.0 (0x38), and the epilogue adds 2^17, whose unit in the last
// place is 2^-6: bit 0 of the word is the count's parity.
//
// A CTA makes 256 inputs x 256 outputs: two accumulators of 128 x 256 (all 512
// columns of tensor memory), 128 columns of K a stage, three stages.
//   warps 4..11  one input row a thread: 128 bits -> 128 bytes, swizzled to
//                shared memory (16 shift/mask pairs per 32 bits)
//   warp 12      bulk copies of the matrix, expanded once per call into the
//                swizzled order of its shared-memory tiles (32 KB a stage)
//   warp 13      issues the MMAs (2 x 4 of 128 x 256 x 32 a stage)
//   warps 0..3   accumulators -> parity words, 32 bytes a row
// Elements lie along K in the order the cheap expansion gives (bit q + 8 b of a
// 32-bit word at byte 4 q + b) in both operands.  Shared-memory traffic bounds
// it (operands in, operands out for two MMAs: about 40 KB per 284 cycles of
// MMA at the e4m3 rate).  65536 inputs of 4096 bits, m = 2048: 369 us, 3.0 PFLOP/s
// (the CUDA-core engine, AND / XOR on words: 1309 us).
//
// Every wait has a limit, after which the kernel records CM_FLAG_TIMEOUT and
// ends.
#include <cuda_runtime.h>
#include <stdint.h>

#include "cm_internal.h"
#include "cm_ss_f8.h"

namespace cm {

namespace {

constexpr int kStages = 3, kChunk = 128;
constexpr int kTileBytes = 256 * kChunk;                 // one operand's stage
constexpr int kSmem = kStages * 2 * kTileBytes + 1024;   // 1 KB to align
constexpr int kF8Threads = 14 * 32;
constexpr uint64_t kWaitNs = 2000000000ull;

__device__ __forceinline__ uint32_t saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t now_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok;
}

// False when the wait ran out (here or, through `dead`, in another warp).
__device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity, volatile uint32_t *dead) {
    if (try_wait(bar, parity)) return true;
    const uint64_t t0 = now_ns();
    while (!try_wait(bar, parity)) {
        if (*dead) return false;
        if (now_ns() - t0 > kWaitNs) {
            *dead = 1;
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ void arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Shared-memory operand descriptor: K-major rows of 128 bytes, 128-byte
// swizzle, 1024 bytes between groups of 8 rows.
__device__ __forceinline__ uint64_t operand(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}

// e4m3 x e4m3 -> f32, M = 128, N = 256, both operands K-major.
constexpr uint32_t kInstr = (1u << 4) | ((256u >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, bool add) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}" ::"r"(d),
        "l"(a), "l"(b), "r"(kInstr), "r"((uint32_t)add)
        : "memory");
}

__device__ __forceinline__ void commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__global__ void __launch_bounds__(kF8Threads, 1) k_ss_f8(const uint8_t *__restrict__ T, uint32_t chunks, uint32_t pblocks,
                                                       const uint64_t *__restrict__ X, uint64_t n, uint64_t wx,
                                                       uint64_t count, uint64_t *__restrict__ Z, uint64_t m,
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

    if (warp >= 4 && warp < 12) {
        const uint32_t r = threadIdx.x - 128;  // input row of the CTA's 256
        uint32_t it = 0;
        bool ok = true;
        for (uint64_t u = blockIdx.x; u < units && ok; u += gridDim.x) {
            const uint64_t c = u / pblocks * 256 + r;
            const uint64_t *row = X + c * wx;
            auto load = [&](uint32_t k, uint64_t (&w)[2]) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const uint64_t j = 2ull * k + i;
                    w[i] = c < count && j < wx ? __ldg(row + j) : 0ull;
                    if (j < wx && n - 64 * j < 64) w[i] &= (1ull << (n - 64 * j)) - 1;
                }
            };
            uint64_t w[2], nx[2];
            load(0, w);
            for (uint32_t k = 0; k < chunks; ++k, ++it) {
                if (k + 1 < chunks) load(k + 1, nx);
                const uint32_t s = it % kStages, ph = (it / kStages) & 1u;
                if (!(ok = wait(empty + 8 * s, ph ^ 1u, &dead))) break;
                uint8_t *dst = base + s * 2 * kTileBytes + r * 128;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint32_t b = (uint32_t)(w[j >> 2] >> (32 * ((j >> 1) & 1)));
                    uint4 v;
                    if (j & 1) v = make_uint4((b >> 1) & 0x08080808u, (b >> 2) & 0x08080808u, (b >> 3) & 0x08080808u, (b >> 4) & 0x08080808u);
                    else v = make_uint4((b << 3) & 0x08080808u, (b << 2) & 0x08080808u, (b << 1) & 0x08080808u, b & 0x08080808u);
                    *reinterpret_cast<uint4 *>(dst + ((j ^ (r & 7u)) << 4)) = v;
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                arrive(full + 8 * s);
                w[0] = nx[0];
                w[1] = nx[1];
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
                        saddr(base + (s * 2 + 1) * kTileBytes)),
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
                const uint64_t a = operand(saddr(base + s * 2 * kTileBytes)), a2 = operand(saddr(base + s * 2 * kTileBytes + kTileBytes / 2)),
                               b = operand(saddr(base + (s * 2 + 1) * kTileBytes));
#pragma unroll
                for (int q = 0; q < 4; ++q) {  // 32 bytes of K: 2 units of the descriptor's address
                    mma(tmem, a + 2 * q, b + 2 * q, k || q);
                    mma(tmem + 256, a2 + 2 * q, b + 2 * q, k || q);
                }
                commit(empty + 8 * s);
            }
            if (ok) commit(accfull);
        }
    } else if (warp < 4) {
        uint32_t acc = 0;
        for (uint64_t u = blockIdx.x; u < units; u += gridDim.x, ++acc) {
            if (!wait(accfull, acc & 1u, &dead)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t pb = u % pblocks;
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                const uint64_t c = u / pblocks * 256 + h * 128 + threadIdx.x;
                uint32_t word[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    uint32_t v[32];
                    const uint32_t at = tmem + ((warp * 32u) << 16) + 256 * h + 32 * q;
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
                          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                        : "r"(at));
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    uint32_t o = 0;
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        o = __funnelshift_r(o, __float_as_uint(__uint_as_float(v[j]) + 131072.0f), 1);
                    word[q] = o;
                }
                if (c < count) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const uint64_t w = 4 * pb + q;
                        uint64_t v = (uint64_t)word[2 * q + 1] << 32 | word[2 * q];
                        if (w < wz) {
                            if (m - 64 * w < 64) v &= (1ull << (m - 64 * w)) - 1;
                            Z[c * wz + w] = v;
                        }
                    }
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

// The matrix in tile order: block (p, k) holds rows 256 p .. of the Toeplitz
// matrix, columns 128 k .. as bytes, rows of 128 with their 16-byte pieces
// exchanged by row mod 8.  One thread a row's 32 columns.
__global__ void __launch_bounds__(256) k_ss_f8_rows(const uint32_t *__restrict__ y, uint64_t n, uint64_t m, uint32_t chunks,
                                                    uint8_t *__restrict__ T, uint64_t total) {
    const uint64_t N = n + m - 1;
    for (uint64_t t = (uint64_t)blockIdx.x * 256 + threadIdx.x; t < total; t += (uint64_t)gridDim.x * 256) {
        const uint32_t g = (uint32_t)(t & 3u), r = (uint32_t)(t >> 2) & 255u;
        const uint64_t blk = t >> 10, p = blk / chunks, k = blk - p * chunks;
        const uint64_t i = 256 * p + r, j0 = 128 * k + 32 * g;
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
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint4 v;
            v.x = ((w >> (4 * h)) & 0x01010101u) * 0x38u;
            v.y = ((w >> (4 * h + 1)) & 0x01010101u) * 0x38u;
            v.z = ((w >> (4 * h + 2)) & 0x01010101u) * 0x38u;
            v.w = ((w >> (4 * h + 3)) & 0x01010101u) * 0x38u;
            *reinterpret_cast<uint4 *>(row + (((2 * g + h) ^ (r & 7u)) << 4)) = v;
        }
    }
}

}  // namespace

uint64_t ss_f8_bytes(uint64_t n, uint64_t m) {
    return (m + 255) / 256 * ((n + kChunk - 1) / kChunk) * kTileBytes;
}

cudaError_t launch_ss_f8_rows(const uint64_t *y, uint64_t n, uint64_t m, void *T, int nsm, cudaStream_t st) {
    const uint64_t total = ss_f8_bytes(n, m) / 32;
    const uint64_t blocks = (total + 255) / 256, cap = (uint64_t)nsm * 16;
    k_ss_f8_rows<<<(unsigned)(blocks < cap ? blocks : cap), 256, 0, st>>>(
        reinterpret_cast<const uint32_t *>(y), n, m, (uint32_t)((n + kChunk - 1) / kChunk), static_cast<uint8_t *>(T), total);
    return cudaGetLastError();
}

cudaError_t launch_ss_f8(const void *T, uint64_t n, uint64_t m, const uint64_t *X, uint64_t count, uint64_t *Z,
                         uint32_t *status, int nsm, cudaStream_t st) {
    cudaError_t e = smem_attr_once<k_ss_f8>(kSmem);
    if (e != cudaSuccess) return e;
    const uint64_t pblocks = (m + 255) / 256, units = (count + 255) / 256 * pblocks;
    k_ss_f8<<<(unsigned)(units < (uint64_t)nsm ? units : nsm), kF8Threads, kSmem, st>>>(
        static_cast<const uint8_t *>(T), (uint32_t)((n + kChunk - 1) / kChunk), (uint32_t)pblocks, X, n, (n + 63) / 64, count,
        Z, m, (m + 63) / 64, units, status);
    return cudaGetLastError();
}

}  // namespace cm
