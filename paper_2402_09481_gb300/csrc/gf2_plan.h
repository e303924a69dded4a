// Host tables of the binary-polynomial transform (cm_gf2.cu).
#pragma once
#include "gf2_tile.cuh"

namespace cm {
namespace gf {

// Cantor basis beta_0 = 1, beta_i^2 + beta_i = beta_(i-1) of GF(2^32).
void cantor_basis(uint32_t beta[32]);

// Shape of the transform of 2^lg bits.
struct Shape {
    int lg;
    int fmax;       // log2 components at the points: 4 (lg = 15) or 5
    int nb, nfree;  // tile of the last pass: 2^nb words, 2^nfree point words
    int lo;         // index bits below lo are handled in the last pass
    bool two;       // a column pass over index bits lo .. lg - 1 comes first
    int tiles;      // tiles of the last pass (and of the column pass)
    int colr;       // index bits above 16 (rows of the first conversion), 0 if lg <= 16
};
// few: the smaller tiles for few operands (lg of kFewMinLg .. kFewMaxLg).
Shape shape_of(int lg, bool few = false);

// Fill the pass tables: mid always, col when two.
void build_passes(int lg, bool few, Pass *mid, Pass *col);

}  // namespace gf
}  // namespace cm
