// Launch interface of the binary-polynomial product (cm_gf2.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "cm.h"
#include "gf2_plan.h"
#include "ntt_device.cuh"

struct cm_ctx;

namespace cm {
namespace gf {

// The tensor-core product starts as a programmatic dependent of the launch that
// lays out its operands: barriers, tensor memory and scales are ready when those
// are.  (Launching the transforms' kernels this way measured slower, 199 -> 216 us
// at 2^25: a kernel's early CTAs crowd the SMs that happen to be free.)
#ifdef __CUDACC__
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class K, class... A>
cudaError_t launch_after(bool dependent, K kern, uint32_t grid, uint32_t block, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}
// Dependent launches may be used on st (not under stream capture, where the
// graphs of a batch keep plain edges).
inline bool may_depend(cudaStream_t st) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(st, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone;
}
#endif

// One operand block: bit j of its array is map(base + j) for j < lim (a), or
// map(base + 2^lg - 1 - j) (b, reversed; lim unused).
struct InOp {
    BitMap map;
    uint64_t base, lim;
};

// One output window: m bits to z (words past m written 0); zero, with the
// status flag set, when the Dodis et al. flags at pre (if any) report a
// constant input.
struct OutOp {
    uint64_t *z;
    uint64_t m;
    const uint32_t *pre;
    uint32_t *status;
};

// The operand blocks and windows of one launch sequence.  Blocks 0 .. na - 1
// are a's, then nb of b.  A single extraction generates them from one pair of
// maps and fixed steps; a batch lists them in device memory (in / out).
struct Ops {
    const InOp *in;
    const OutOp *out;
    InOp a0, b0;
    OutOp z0;
    uint64_t astep, bstep, zstep;  // zstep a multiple of 64
    uint32_t na, nb, nz;
};

// A transform length and the blocks over it.  nin > 1 or nz > 1 (generated ops
// only): window w sums the products of a's block i with b's block i + w.
struct Product {
    int lg;
    uint32_t nin;  // products summed per window (1: pair i gives window i)
};

// Scratch bytes of a product over `ops`.
uint64_t product_scratch(const Product &p, const Ops &ops);
// Enqueue it; scratch holds product_scratch bytes.  tables: device Pass tables
// (2 per length from kMinLg on: mid, col).  c: context for tracing (may be null).
cudaError_t launch_product(cm_ctx *c, int nsm, const Product &p, const Ops &ops, const Pass *tables, void *scratch,
                           cudaStream_t st);

// Dodis et al. flags of `count` listed inputs (x bits, pairs of zeroed words):
// flags[0] set by a 1 bit, flags[1] by a 0 bit.
struct SameOp {
    const uint64_t *x;
    uint64_t n;
    uint32_t *flags;
};
cudaError_t launch_same(const SameOp *ops, uint32_t count, cudaStream_t st);
// Kernel launches of a product.
uint32_t product_launches(const Product &p, const Ops &ops);

// z = the m outputs of K terms, K + m - 1 <= 2^13, in one launch (cm_gf2_dense.cu);
// check: a is a Dodis et al. input, all of it; pre (may be null): its flags,
// pre[0] == 0 without a 1 bit, pre[1] == 0 without a 0 bit.
constexpr int kDenseMaxLg = 13;
cudaError_t launch_dense(const BitMap &a, const BitMap &b, uint32_t K, uint32_t m, bool check, uint64_t *z,
                         uint32_t *status, uint32_t *pre, cudaStream_t st);

// Dense product on the tensor cores (cm_gf2_tc.cu): the shape of K terms and m
// outputs (stages: the longest CTA chain's, the time's measure), the operands as
// plain bits (a after 256 zero bits; b in order) with z cleared, the product.
// status: the Dodis et al. flag; gave_up: CM_FLAG_TIMEOUT when a bounded wait ran
// out (z is then undefined); stall: make one run out.
struct TcShape {
    uint64_t rows, chunks, splits, per, a_words, b_words, stages;
};
TcShape tc_shape(uint64_t K, uint64_t m, int nsm);
cudaError_t launch_tc_prep(const Ops &q, const TcShape &s, uint32_t *a, uint32_t *b, uint64_t *z, uint64_t m,
                           cudaStream_t st);
cudaError_t launch_tc(const TcShape &s, const uint32_t *a, const uint32_t *b, uint64_t *z, uint64_t m,
                      const uint32_t *pre, uint32_t *status, uint32_t *gave_up, bool stall, bool dependent,
                      cudaStream_t st);

// Host image of the device tables.
constexpr int kFewTables = 2 * (kMaxLg - kMinLg + 1);  // where the few-operand shapes' begin
constexpr int kTables = kFewTables + 2 * (kFewMaxLg - kFewMinLg + 1);
void build_tables(Pass *t);  // kTables entries

}  // namespace gf
}  // namespace cm
