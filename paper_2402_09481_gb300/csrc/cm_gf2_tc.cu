// One extraction as a dense product on the 5th-generation tensor cores: 2^17 .. 2^22
// terms, while the longest chain of stages leaves it ahead of the transforms (to about
// 2^19.2 terms where K and m are alike, further for a short or a narrow product).
//
// z_(224 c + i) = sum_u b_(u + 224 c) a_(u - i), i < 224: a product of two bit
// matrices, rows of windows of b 224 apart and rows of shifts of a, whose outputs
// are z in order.  K m products cost what m / 224 inputs of K bits cost in the
// shared-seed product (cm_ss_f4.cu has the number format); here both operands are
// expanded from bits on the way into shared memory.
//
// A CTA makes 256 x 224 outputs over a share of the terms, and its parities are
// XORed into z (cleared by the launch before, which also lays the operands out as
// plain bits): at these lengths one share an SM fills the GPU with a few dozen
// stages each, where a transform has fewer tiles than SMs.
//   warps 4..11   b's windows (256 rows): 32-bit aligned, 64 bits a lane
//   warps 12..18  a's shifts (224 rows): funnel shifts
//   warp 19       MMAs; warps 0..3 parities and XORs
// About 0.7 us a stage after 12 us of launches, set-up and parities: n = 300007,
// m = 150001 29.4 us (integer transforms 47).
// Every wait has a limit, after which the kernel records CM_FLAG_TIMEOUT at gave_up
// and ends (stall, for tests: the accumulators' wait runs out).
#include <cuda_runtime.h>
#include <stdint.h>

#include "cm_gf2.h"
#include "cm_internal.h"
#include "tc05.cuh"

namespace cm {
namespace gf {

using namespace tc;

namespace {

constexpr int kStages = 3, kInBytes = 256 * 128, kTileBytes = kRows * 128, kStageBytes = kInBytes + kTileBytes;
constexpr int kSmem = kStages * kStageBytes + 1024;  // 1 KB to align
constexpr int kTcThreads = 20 * 32;

__global__ void __launch_bounds__(kTcThreads, 1) k_gf_tc(const uint32_t *a, const uint32_t *b, uint32_t chunks, uint32_t rows, uint32_t splits, uint32_t per,
                                                         uint32_t *__restrict__ z, uint64_t m,
                                                         const uint32_t *__restrict__ pre, uint32_t *status,
                                                         uint32_t *gave_up, bool stall) {
    extern __shared__ uint8_t raw[];
    __shared__ __align__(8) uint64_t bars[2 * kStages + 1];
    __shared__ uint32_t tmem_at;
    __shared__ volatile uint32_t dead;
    uint8_t *base = raw + ((1024u - (saddr(raw) & 1023u)) & 1023u);
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
    const uint32_t full = saddr(bars), empty = saddr(bars + kStages), done = saddr(bars + 2 * kStages);
    const uint32_t blk = blockIdx.x / splits, k0 = (blockIdx.x % splits) * per,
                   n = k0 >= chunks ? 0u : chunks - k0 < per ? chunks - k0 : per;
    if (threadIdx.x == 0) {
        dead = 0;
        for (int s = 0; s < kStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full + 8 * s), "r"(15));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(empty + 8 * s), "r"(1));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(done), "r"(1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 19) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(saddr(&tmem_at)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_at;
    if (warp < 4) set_scales(tmem, warp);
    wait_for_previous();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

    if (warp >= 4 && warp < 19) {
        // rows 8 i + lane / 4 of the warp's 32, 64-bit piece lane % 4 of a stage's 256
        const bool shifts = warp >= 12;
        const uint32_t r0 = (shifts ? warp - 12 : warp - 4) * 32 + (lane >> 2), q = lane & 3u;
        const uint32_t *src[4];
        uint32_t sh[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t r = r0 + 8 * i, c = 256 * blk + r < rows ? 256 * blk + r : rows - 1;  // rows past the last: any
            const uint32_t bit = shifts ? 256u + 64 * q - r : 0u;  // a has 256 zero bits in front
            src[i] = (shifts ? a + (bit >> 5) : b + 7 * c + 2 * q) + 8ull * k0;
            sh[i] = bit & 31u;
        }
        auto load = [&](uint32_t k, uint32_t (&w)[4][2]) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t *p = src[i] + 8 * k;
                const uint32_t w0 = __ldca(p), w1 = __ldca(p + 1), w2 = shifts ? __ldca(p + 2) : 0u;
                w[i][0] = __funnelshift_r(w0, w1, sh[i]);
                w[i][1] = __funnelshift_r(w1, w2, sh[i]);
            }
        };
        uint32_t w[4][2], nx[4][2];
        if (n) load(0, w);
        for (uint32_t k = 0; k < n; ++k) {
            if (k + 1 < n) load(k + 1, nx);
            const uint32_t s = k % kStages, ph = (k / kStages) & 1u;
            if (!wait_warp(empty + 8 * s, ph ^ 1u, &dead)) break;
            uint8_t *dst = base + s * kStageBytes + (shifts ? kInBytes : 0) + r0 * 128;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    *reinterpret_cast<uint4 *>(dst + i * 1024 + (((2 * q + h) ^ (r0 & 7u)) << 4)) = nibbles(w[i][h]);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) arrive(full + 8 * s);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                w[i][0] = nx[i][0];
                w[i][1] = nx[i][1];
            }
        }
    } else if (warp == 19 && lane == 0 && n) {
        bool ok = true;
        for (uint32_t k = 0; k < n; ++k) {
            const uint32_t s = k % kStages, ph = (k / kStages) & 1u;
            if (!(ok = wait(full + 8 * s, ph, &dead))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t at = saddr(base + s * kStageBytes);
            const uint64_t d0 = operand(at), d1 = operand(at + kInBytes / 2), e = operand(at + kInBytes);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                mma(tmem, d0 + 2 * j, e + 2 * j, tmem + kScaleCol, k || j);
                mma(tmem + kRows, d1 + 2 * j, e + 2 * j, tmem + kScaleCol, k || j);
            }
            commit(empty + 8 * s);
        }
        if (ok && !stall) commit(done);
    } else if (warp < 4 && n) {
        const bool bad = pre && (pre[0] == 0u || pre[1] == 0u);
        if (bad && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(status, kFlagPrecond);
        if (wait_warp(done, 0, &dead)) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                const uint32_t c = 256 * blk + h * 128 + threadIdx.x;
#pragma unroll 1
                for (int q = 0; q < 7; ++q) {
                    uint32_t v = parities(tmem + ((warp * 32u) << 16) + kRows * h + 32 * q);
                    const uint64_t at = 32ull * (7ull * c + q);
                    if (c >= rows || at >= m || bad) v = 0u;
                    else if (m - at < 32) v &= (1u << (uint32_t)(m - at)) - 1u;
                    if (v) atomicXor(z + 7ull * c + q, v);
                }
            }
        }
    }
    __syncwarp();
    if (dead) __nanosleep(1000000);  // MMAs still in flight end by themselves
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && dead) atomicOr(gave_up, kFlagTimeout);
    if (warp == 19) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
    }
}

}  // namespace

TcShape tc_shape(uint64_t K, uint64_t m, int nsm) {
    TcShape s;
    s.rows = (m + kRows - 1) / kRows;
    s.chunks = (K + kRows - 1 + 255) / 256;
    const uint64_t blocks = (s.rows + 255) / 256;
    uint64_t splits = (uint64_t)nsm / blocks;
    if (splits < (s.chunks + 63) / 64) splits = (s.chunks + 63) / 64;  // counts of at most 2^14
    if (splits < 1) splits = 1;
    if (splits > s.chunks) splits = s.chunks;
    s.per = (s.chunks + splits - 1) / splits;
    s.splits = (s.chunks + s.per - 1) / s.per;
    s.a_words = 8 + 8 * s.chunks + 4;
    s.b_words = 7 * (s.rows - 1) + 8 * s.chunks + 4;
    s.stages = s.per * ((blocks * s.splits + (uint64_t)nsm - 1) / (uint64_t)nsm);
    return s;
}

cudaError_t launch_tc(const TcShape &s, const uint32_t *a, const uint32_t *b, uint64_t *z, uint64_t m,
                      const uint32_t *pre, uint32_t *status, uint32_t *gave_up, bool stall, bool dependent,
                      cudaStream_t st) {
    cudaError_t e = smem_attr_once<k_gf_tc>(kSmem);
    if (e != cudaSuccess) return e;
    const uint64_t blocks = (s.rows + 255) / 256;
    return launch_after(dependent, k_gf_tc, (uint32_t)(blocks * s.splits), kTcThreads, kSmem, st, a, b, (uint32_t)s.chunks,
                        (uint32_t)s.rows, (uint32_t)s.splits, (uint32_t)s.per, reinterpret_cast<uint32_t *>(z), m, pre,
                        status, gave_up, stall);
}

}  // namespace gf
}  // namespace cm
