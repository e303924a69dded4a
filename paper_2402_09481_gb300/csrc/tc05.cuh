// tcgen05 pieces of the exact 0 / 1 products (cm_ss_f4.cu, cm_gf2_tc.cu): bounded
// mbarrier waits, shared-memory operands of 128-byte rows, kind::mxf4 MMAs of
// 128 x 224 x 64 with every block scale 1, and parity words out of tensor memory.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace cm {
namespace tc {

constexpr int kRows = 224;                 // outputs (N) of an accumulator
constexpr uint32_t kScaleCol = 2 * kRows;  // tensor memory columns of scales
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

// The same for a warp whose lanes go on together (__syncwarp, tcgen05.ld): one answer
// for all, so that where a wait runs out no lane stays behind in a loop the others left.
__device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, volatile uint32_t *dead) {
    return __all_sync(0xFFFFFFFFu, wait(bar, parity, dead));
}

__device__ __forceinline__ void arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Shared-memory operand descriptor: K-major rows of 128 bytes, 128-byte
// swizzle, 1024 bytes between groups of 8 rows.
__device__ __forceinline__ uint64_t operand(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}

// e2m1 x e2m1 -> f32, ue8m0 scales, M = 128, N = 224, both operands K-major.
constexpr uint32_t kInstr = (1u << 7) | (1u << 10) | ((uint32_t)(kRows >> 3) << 17) | (1u << 23) | ((128u >> 4) << 24);

__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t scale, bool add) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%5], [%5], p;\n}" ::"r"(d),
        "l"(a), "l"(b), "r"(kInstr), "r"((uint32_t)add), "r"(scale)
        : "memory");
}

__device__ __forceinline__ void commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// Every scale 1.0 (127), whatever row and block it is read for (warps 0..3).
__device__ __forceinline__ void set_scales(uint32_t tmem, uint32_t warp) {
#pragma unroll 1
    for (uint32_t c = 0; c < 64; c += 8)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(
                         tmem + ((warp * 32u) << 16) + kScaleCol + c),
                     "r"(0x7F7F7F7Fu)
                     : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Parities of 32 columns of a lane's row: products are 0.25 each, so adding 2^21
// leaves the count's parity in bit 0.
__device__ __forceinline__ uint32_t parities(uint32_t at) {
    uint32_t v[32];
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
        o = __funnelshift_r(o, __float_as_uint(__uint_as_float(v[j]) + 2097152.0f), 1);
    return o;
}

// 32 bits -> 32 nibbles: bit q + 4 b at nibble b of word q.
__device__ __forceinline__ uint4 nibbles(uint32_t b) {
    return make_uint4(b & 0x11111111u, (b >> 1) & 0x11111111u, (b >> 2) & 0x11111111u, (b >> 3) & 0x11111111u);
}

}  // namespace tc
}  // namespace cm
