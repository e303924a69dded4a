// Host tables of the binary-polynomial transform: the Cantor basis and, for
// every length, the levels of its two passes (which index bit sits where in a
// tile, and each level's twiddles).  cm_gf2.cu explains the transform.
#include "gf2_plan.h"

#include <string.h>

#include <vector>

namespace cm {
namespace gf {

void cantor_basis(uint32_t beta[32]) {
    // y -> y^2 + y over the 32 unit vectors, reduced by their highest bits
    uint32_t val[32], comb[32];
    bool have[32] = {};
    for (int i = 0; i < 32; ++i) {
        uint32_t e = 1u << i, c = e, v = gmul(e, e, 5) ^ e;
        while (v) {
            const int h = 31 - __builtin_clz(v);
            if (!have[h]) {
                have[h] = true;
                val[h] = v;
                comb[h] = c;
                break;
            }
            v ^= val[h];
            c ^= comb[h];
        }
    }
    beta[0] = 1;
    for (int i = 1; i < 32; ++i) {
        uint32_t t = beta[i - 1], y = 0;
        while (t) {
            const int h = 31 - __builtin_clz(t);
            t ^= val[h];  // solvable for every beta_i, i < 31
            y ^= comb[h];
        }
        beta[i] = y & ~1u;  // y and y + 1 both solve it
    }
}

Shape shape_of(int lg, bool few) {
    Shape s;
    s.lg = lg;
    s.fmax = lg < 16 ? 4 : 5;
    s.two = lg > 18;
    s.nb = few ? 12 : lg >= 18 ? 13 : lg - 5;
    s.nfree = s.nb - s.fmax;
    // components whose index bit is at least lo come with the tile from above it
    s.lo = !s.two ? lg : few ? 13 : lg <= 21 ? 15 : 14;
    s.tiles = 1 << (lg - 5 - s.nb);
    s.colr = lg > 16 ? lg - 16 : 0;
    return s;
}

static int missing_of(int lg, int i) {  // j with i = lg - 2^j, else -1
    for (int j = 0; j < 5; ++j)
        if (lg - (1 << j) == i) return j;
    return -1;
}

// Levels hi .. lo (index bits, downwards) on tiles holding the index bits of
// `in` (each >= 5); word bits 0..4 take part when lo == 0.
static void build_pass(int lg, int nb, int nfree, int fmax, const std::vector<int> &in, int hi, int lo,
                       const uint32_t *beta, Pass *P) {
    memset(P, 0, sizeof(*P));
    int at[32], lane[32];  // index bit -> address position / word bit (-1: elsewhere)
    for (int i = 0; i < 32; ++i) at[i] = lane[i] = -1;
    uint32_t used = 0;
    for (int i : in) {
        const int j = missing_of(lg, i);
        if (j >= 0 && j < fmax) {
            at[i] = nfree + j;
            used |= 1u << at[i];
        }
    }
    for (int i : in)
        if (at[i] < 0) {
            int pos = 0;
            while ((used >> pos) & 1u) ++pos;
            at[i] = pos;
            used |= 1u << pos;
        }
    // tile element numbers run over the tile's index bits in order
    for (int t = 0; t < 3; ++t)
        for (int e = 0; e < 32; ++e)
            for (int b = 0; b < 5; ++b)
                if (((e >> b) & 1) && 5 * t + b < nb) {
                    P->glut[t][e] |= 1u << (in[5 * t + b] - 5);
                    P->alut[t][e] |= 1u << at[in[5 * t + b]];
                }
    // the other word bits of the index number the tiles
    std::vector<int> ext;
    for (int i = 5; i < lg; ++i)
        if (at[i] < 0) ext.push_back(i);
    P->next = (uint32_t)ext.size();
    for (size_t b = 0; b < ext.size(); ++b) P->extpos[b] = (uint32_t)(ext[b] - 5);
    for (int b = 0; b < 5; ++b) lane[b] = b;
    int n = 0;
    P->npre = 0;
    for (int i = hi; i >= lo; --i) {
        if (i == 4) {  // the word bits change places with five point bits
            P->npre = (uint32_t)n;
            uint32_t taken = 0;
            for (int b = 0; b < 5; ++b) {
                const int j = missing_of(lg, b);
                if (j >= 0) taken |= 1u << (P->xp[b] = (uint32_t)(nfree + j));
            }
            for (int b = 0; b < 5; ++b)
                if (missing_of(lg, b) < 0) {
                    int pos = 0;
                    while ((taken >> pos) & 1u) ++pos;
                    taken |= 1u << (P->xp[b] = (uint32_t)pos);
                }
            int bit = 0;
            for (int pos = 0; pos < nb; ++pos)
                if (!((taken >> pos) & 1u)) {
                    for (int e = 0; e < 16; ++e)
                        if ((e >> (bit & 3)) & 1) P->xlut[bit >> 2][e] |= 1u << pos;
                    ++bit;
                }
            for (int b = 0; b < 5; ++b) {
                int old = 5;
                while (at[old] != (int)P->xp[b]) ++old;
                at[old] = -1;
                lane[b] = -1;
                lane[old] = b;
                at[b] = (int)P->xp[b];
            }
        }
        Lev &v = P->lev[n++];
        const int j = missing_of(lg, i);
        v.p = (uint32_t)at[i];
        v.missing = j >= 0;
        int f = 0;  // components formed before this level
        for (int q = 0; q < 5; ++q) f += lg - (1 << q) > i;
        v.f = (uint32_t)f;
        uint32_t base = beta[lg - i];
        for (int t = i + 1; t < lg; ++t) {
            if (missing_of(lg, t) >= 0) continue;
            const uint32_t c = beta[t - i];
            base ^= c;
            if (at[t] >= 0) {
                const int tab = at[t] < 4 ? 0 : at[t] < 8 ? 16 : 32, bit = at[t] < 4 ? at[t] : at[t] < 8 ? at[t] - 4 : at[t] - 8;
                for (int e = 0; e < (tab == 32 ? 32 : 16); ++e)
                    if ((e >> bit) & 1) v.lut[tab + e] ^= c;
            } else if (lane[t] >= 0) {
                static const uint32_t pat[5] = {0xAAAAAAAAu, 0xCCCCCCCCu, 0xF0F0F0F0u, 0xFF00FF00u, 0xFFFF0000u};
                for (int w = 0; w < 32; ++w)
                    if ((c >> w) & 1u) v.lanes[w] ^= pat[lane[t]];
            } else {
                for (size_t b = 0; b < ext.size(); ++b)
                    if (ext[b] == t) v.ext[b] = c;
            }
        }
        if (j >= 0) {
            base ^= 1u << (1 << j);  // the twiddle less its x_j
            v.base[0] = base;
            v.base[1] = base ^ 1u;
        } else {
            v.base[0] = base ^ 1u;
            v.base[1] = base;
        }
    }
    P->nlev = (uint32_t)n;
    if (lo > 4) P->npre = P->nlev;
}

void build_passes(int lg, bool few, Pass *mid, Pass *col) {
    const Shape s = shape_of(lg, few);
    uint32_t beta[32];
    cantor_basis(beta);
    std::vector<int> in;
    for (int i = 5; i < s.lo; ++i) in.push_back(i);
    for (int i = s.lo; i < lg; ++i)
        if (missing_of(lg, i) >= 0) in.push_back(i);
    build_pass(lg, s.nb, s.nfree, s.fmax, in, s.two ? s.lo - 1 : lg - 1, 0, beta, mid);
    if (s.two) {
        std::vector<int> cin;
        const int rows = lg - s.lo;
        for (int i = 5; i < 5 + 13 - rows; ++i) cin.push_back(i);
        for (int i = s.lo; i < lg; ++i) cin.push_back(i);
        // from 2^20 on the row conversion does the first four levels (first_levels)
        build_pass(lg, 13, 9, 4, cin, lg >= 20 ? lg - 5 : lg - 1, s.lo, beta, col);
    }
}

}  // namespace gf
}  // namespace cm
