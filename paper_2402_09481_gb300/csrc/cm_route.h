// How one extraction runs: as binary polynomials (cm_gf2.cu) or as the block
// list of the integer transforms (cm_api.cu).
#pragma once
#include <vector>

#include "cm_ctx.h"
#include "cm_gf2.h"
#include "cm_internal.h"

namespace cm {

struct Route {
    bool gf = false, dense = false, tc = false;
    gf::TcShape shape;
    gf::Product prod;
    gf::Ops ops;  // pointers filled in by enqueue_route
    int kind;
    uint64_t n, m;
    std::vector<Block> bl;
    uint64_t need = 0, tmp_off = 0, pre_off = 0;  // scratch bytes; offsets in it
};

// The context's options leave the choice of transform to the library.
bool gf_allowed(const cm_ctx *ctx);
// The operands' maps and the transform length(s) of (kind, n, m), valid arguments.
void gf_maps(int kind, uint64_t n, uint64_t m, gf::Ops *q);
void gf_shape(int kind, uint64_t n, uint64_t m, gf::Product *p, gf::Ops *q);

// z's words overlap an operand's.  The dense forms' CTAs read the operands while
// others write z; the transforms' launches have read them before the last one
// writes, so such calls keep to those.
inline bool in_place(int kind, uint64_t n, uint64_t m, const uint64_t *x, const uint64_t *y, const uint64_t *z) {
    const uint64_t yb = kind == CM_TOEPLITZ ? n + m - 1 : kind == CM_CIRCULANT ? n + 1 : n;
    auto meets = [&](const uint64_t *p, uint64_t bits) {
        const uintptr_t a = (uintptr_t)p, b = (uintptr_t)z;
        return a < b + 8 * ((m + 63) / 64) && b < a + 8 * ((bits + 63) / 64);
    };
    return meets(x, n) || meets(y, yb);
}

// CM_EINVAL for invalid arguments, CM_ENOMEM when no form fits `budget`.
cm_status make_route(const cm_ctx *ctx, int kind, uint64_t n, uint64_t m, uint64_t budget, bool in_place, Route *r);
// gave_up: where a bounded wait that runs out (tc) is recorded, for callers that
// report it themselves; null: the context's status.
cm_status enqueue_route(cm_ctx *ctx, Route &r, const uint64_t *x, const uint64_t *y, uint64_t *z, void *scratch,
                        cudaStream_t st, uint32_t *gave_up = nullptr);

// Kernel launches of a route.
uint32_t route_launches(const Route &r);

}  // namespace cm
