// Host helpers shared by the plan code (bf_api.cu) and the allocation-free apply (bf_noalloc.cu).
#pragma once

#include <cmath>

#include "../../include/bf.h"
#include "bf_device.cuh"
#include "bf_launch.h"

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

// Lower bound over X x Y of the root part of |Phi| (0 for the kinds without a root).
inline double root_floor(int d, int kind, const bf_params *p)
{
    double nx[3], ny[3], q2 = 0.0;   // distances of the intervals from 0
    auto gap = [](double lo, double w) { return lo > 0.0 ? lo : (lo + w < 0.0 ? -(lo + w) : 0.0); };
    for (int k = 0; k < d; ++k) {
        nx[k] = gap(p->x_lo[k], p->x_w[k]);
        ny[k] = gap(p->y_lo[k], p->y_w[k]);
        q2 += ny[k] * ny[k];
    }
    const double s = std::fabs(p->phase_scale);
    if (kind == BF_PHASE_GENRADON) return s * std::sqrt(q2) / 3.0;   // a_k(x) >= 1/3
    if (kind == BF_PHASE_HYPRADON) return s * nx[0] * std::sqrt(ny[0] * ny[0] + ny[1] * ny[1] * nx[1] * nx[1]);
    return 0.0;
}

// Whether the mixed precisions keep the rounding error of the sums under the root (PMIXW; the
// kernels of get_fns(..., wide)).  With the common grid G of sqrt_grid, G < 2^-20 R^2 for
// roots up to R, a sum is good to about 2^-23 G and a root x to 2^-44 R^2 / x; below
// x = 2^-10.5 R, where the terms are smaller than G/2 and FP32 holds them relative to themselves,
// the error falls again.  The grid serves plans where that is at most 6e-8 cycles (2^-24, the spacing of
// the FP32 numbers below 1 that the reduced phase is made of): roots up to 724 cycles whatever the
// domain, and any root of a domain away from the origin (hyperbolic Radon, tau in [1, 2): up to 4.5
// times the smallest one).  NumPy restatement, worst error over all roots, grid and exact sums:
// R = 724 3.8e-8 and 2.7e-8, 5.7e3 2.3e-7 and 2.9e-8, 3.3e4 1.2e-6 and 3.0e-8, 1.5e6 6.0e-5 and 4.2e-8.
inline bool wide_root(int d, int kind, const bf_params *p)
{
    if (p->precision == BF_PREC_FP64 || (kind != BF_PHASE_GENRADON && kind != BF_PHASE_HYPRADON)) return false;
    double lin, root;
    phase_bounds(d, kind, p, &lin, &root);
    const double x = std::fmax(root_floor(d, kind, p), std::exp2(-10.5) * root);
    return std::exp2(-44.0) * root * root > 6e-8 * x;
}

// 1.5 * 2^23 G with G the smallest power of two for which every term of the sum of squares
// under the root, and the sum, is at most 2^21 G: the terms rounded to multiples of G
// (Ph::quant) then add without rounding.  0 for wide roots: the terms stay as they are.
inline float sqrt_grid(int d, int kind, const bf_params *p)
{
    if (wide_root(d, kind, p)) return 0.0f;
    double lin, root;
    phase_bounds(d, kind, p, &lin, &root);
    int e = 0;
    const double m = std::frexp(root * root, &e);   // root^2 = m 2^e, m in [1/2, 1) (or 0)
    e = (m == 0.5 ? e - 1 : e) - 21;
    return (float)std::ldexp(1.5, (m > 0.0 && e > -60 ? e : -60) + 23);
}

// tiles of 2^{dk} pairs per CTA of a k-level pass, np_cta pairs per CTA
inline int tiles_of(int64_t npts, int64_t np_cta, int d, int k)
{
    const int64_t np = npts < np_cta ? npts : np_cta;
    const int T = (int)(np >> (d * k));
    return T < 1 ? 1 : T;
}

// Pairs per CTA of the single-RHS forward passes.  FP64 at d = 2 puts two tiles in a CTA (whole
// warps of its FP64 instructions: Fourier phase N = 256 6.10 ms, with one tile 7.12), one where
// the grid of single tiles leaves SMs idle: hyperbolic Radon N = 32, q = 8 1.63 -> 0.87 ms.
inline int64_t single_pairs(const PassFns *f, int d, int64_t npts)
{
    const int64_t tile = (int64_t)1 << (d * f->kmax);
    return f->np > tile && npts / tile <= sm_count() ? tile : f->np;
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
