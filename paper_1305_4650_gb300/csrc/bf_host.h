// Host helpers shared by the plan code (bf_api.cu) and the allocation-free apply (bf_noalloc.cu).
#pragma once

#include <cmath>

#include "../../include/bf.h"
#include "bf_device.cuh"

namespace bfl {

// Upper bounds over X x Y of the linear part and of the root part of |Phi| (their sum bounds |Phi|).
inline void phase_bounds(int d, int kind, const bf_params *p, double *lin, double *root)
{
    double mx[3], my[3], xy = 0.0, q2 = 0.0;
    for (int k = 0; k < d; ++k) {
        mx[k] = std::fmax(std::fabs(p->x_lo[k]), std::fabs(p->x_lo[k] + p->x_w[k]));
        my[k] = std::fmax(std::fabs(p->y_lo[k]), std::fabs(p->y_lo[k] + p->y_w[k]));
        xy += mx[k] * my[k];
        q2 += my[k] * my[k];
    }
    *lin = *root = 0.0;
    switch (kind) {
    case BF_PHASE_DOT: *lin = xy; break;
    case BF_PHASE_GENRADON: *lin = xy; *root = std::sqrt(q2); break;   // a_k(x) <= 1
    case BF_PHASE_HYPRADON: *root = mx[0] * std::sqrt(my[0] * my[0] + my[1] * my[1] * mx[1] * mx[1]); break;
    default:
        for (int k = 0; k < d; ++k) *lin += 1.0 + my[k] * my[k] / (k + 2.0);
    }
    *lin *= std::fabs(p->phase_scale);
    *root *= std::fabs(p->phase_scale);
}

// Upper bound of |Phi| over X x Y.  The mixed path rounds to integers by adding
// 1.5 * 2^23, which is exact only below 2^22 cycles (kept under 2^21 here).
inline double phase_bound(int d, int kind, const bf_params *p)
{
    double lin, root;
    phase_bounds(d, kind, p, &lin, &root);
    return lin + root;
}

// 1.5 * 2^23 G with G the smallest power of two for which every term of the sum of squares
// under the root, and the sum, is at most 2^21 G: the terms rounded to multiples of G
// (Ph::quant) then add without rounding, and differ by a multiple of G that FP32 holds from
// the square of any integer next to the root.
inline float sqrt_grid(int d, int kind, const bf_params *p)
{
    double lin, root;
    phase_bounds(d, kind, p, &lin, &root);
    int e = -60;
    while (std::ldexp(1.0, e + 21) < root * root) ++e;
    return (float)std::ldexp(1.5, e + 23);
}

// tiles of 2^{dk} pairs per CTA of a k-level pass, np_cta pairs per CTA
inline int tiles_of(int64_t npts, int64_t np_cta, int d, int k)
{
    const int64_t np = npts < np_cta ? npts : np_cta;
    const int T = (int)(np >> (d * k));
    return T < 1 ? 1 : T;
}

// KArgs::corner of a plan: Lobatto nodes and grid points at the lower corners of their boxes.
// The first level must be a column level.  tc_levels runs every column level in a pass of its
// own kind, with the general first step.
inline int corner_of(int d, int q, int m, const bf_params *p, int lobatto, bool tc)
{
    if (d == 3 && p->node_kind == 0)
        return (p->src_off == 0.0 && m >= 1 ? bfk::LEAF_SRC : 0) | (p->tgt_off == 0.0 ? bfk::LEAF_TGT : 0);
    if (!lobatto || d != 2 || !(q & 1)) return 0;
    const bool src = p->src_off == 0.0 && m >= 1 && !(tc && p->tc_levels);
    return (src ? bfk::CORNER_SRC : 0) | (p->tgt_off == 0.0 ? bfk::CORNER_TGT : 0);
}

// The forward schedule: column passes of at most kmax levels (first step in the first, switch
// in the last), then row passes (last step in the last); rem_first puts the short pass of a run
// of levels first.  With a corner the first (last) level costs nothing, so a pass of that level
// alone would only move the weights: the short pass then goes to the other end of the run.
template <class Fn>
void each_pass(int L, int m, int kmax, bool rem_first, int corner, Fn fn)
{
    auto run = [&](int l, int end, bool first, auto flags, int row) {
        const int rem = (end - l) % kmax, l_first = l;
        while (l < end) {
            int k = end - l < kmax ? end - l : kmax;
            if (first && rem && l == l_first) k = rem;
            fn(row, l, k, flags(l, k));
            l += k;
        }
    };
    if (m == 0) {
        fn(0, 0, 0, bfk::F_INIT | bfk::F_SWITCH);
    } else {
        const bool lone = (corner & bfk::CORNER_SRC) && m > 1 && m % kmax == 1 && kmax > 1;
        run(0, m, rem_first && !lone,
            [&](int l, int k) { return (l == 0 ? bfk::F_INIT : 0) | (l + k == m ? bfk::F_SWITCH : 0); }, 0);
    }
    const bool lone = (corner & bfk::CORNER_TGT) && (L - m) % kmax == 1 && kmax > 1;
    run(m, L, rem_first || lone, [&](int l, int k) { return l + k == L ? bfk::F_FINAL : 0; }, 1);
}

}  // namespace bfl
