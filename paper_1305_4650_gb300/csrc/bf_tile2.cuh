// Single-RHS forward passes for d = 2: the tiles, the in-place update and the node formulas
// of Tile (bf_device.cuh), with three savings.
//
// 1. Parts.  A phase of a pair is the sum of one part per source coordinate plus a root and a
//    sincos (Ph::add, Ph::fin2).  The r modulation phases of the four children of an output
//    pair have only 2q distinct parts per coordinate (and q for the output), so a column level
//    first writes those 6q parts of every output pair to shared memory and evaluates each
//    phase from two of them: 3 additions instead of a double-float product, an exact sum and
//    its reduction per phase.  The parts of level i+1 and the geometry they need are computed
//    beside the stages of level i, so a level has two barriers.  The switch has one target per
//    item and keeps the parts of coordinate 0 in registers; the row levels evaluate the four
//    children of a target node together, from two parts per coordinate.
// 2. Lobatto nodes of odd q (LB).  The end nodes of a child box are nodes of its parent: two of
//    the q columns of M_h are unit vectors (triv), so their products are one addition or none.
// 3. Grid points at box corners (LB and offset 0; KArgs::corner).  A leaf's point is its last
//    node, so the phase factors of the first step cancel and its weight is g at that node; the
//    points of the four leaves of a level-1 source box are four of its nodes, where the factors
//    of the first merge cancel as well.  The first pass starts from those values at level 1,
//    level 1 has four non-zero nodes per input, and the transposed statements hold for the
//    last two levels: the target values are sums of weights of level L - 1 at four nodes.
//
// Measured (generalized Radon, q = 5, one right-hand side): N = 1024 5.28 -> 3.69 ms, N = 128
// 100 -> 60 us; hyperbolic Radon N = 512 with 16 right-hand sides (TileMR, the same three
// points) 8.24 -> 6.10 ms; the largest share is point 3, which leaves 8 of 10 levels at
// N = 1024, two of them with a third of the factors.
//
// Bound: in the mixed precisions the FP32 pipe and issue (one phase is about 26 FP32 operations
// with its sincos, a special-function one and 9 integer ones); in FP64 the FP64 pipe.
#pragma once

namespace bfk {

// parent node that child node u of half h coincides with, or -1 (Lobatto nodes, odd q, in
// descending order: node 0 at +1/2, q - 1 at -1/2)
template <int Q, bool LB>
__host__ __device__ constexpr int triv(int h, int u)
{
    if (!LB) return -1;
    if (h == 0) return u == Q - 1 ? Q - 1 : (u == 0 ? (Q - 1) / 2 : -1);
    return u == 0 ? 0 : (u == Q - 1 ? (Q - 1) / 2 : -1);
}

// acc += M[h][t][u] v with compile-time h, t, u: two scalar FMAs whose coefficient is a
// kernel-parameter operand (a packed FMA needs the coefficient pair in registers first and
// measured 1% slower), nothing or an addition for the unit columns
template <int Q, bool LB, class MS, class C>
__device__ __forceinline__ void mmac(C &acc, const MS &ms, int h, int t, int u, C v)
{
    if (triv<Q, LB>(h, u) < 0)
        cfma(acc, ms.M[h][t][u], v);
    else if (triv<Q, LB>(h, u) == t)
        acc = madd(acc, v);
}

template <int Q, class P, int K, bool LB>
struct Tile2 {
    using R = typename P::R;
    using C = typename P::C;
    using TL = Tile<2, Q, P, K>;
    using PH = Ph<P, 2, K>;
    using PH2 = Ph2<P, 2, K>;
    using V = typename PH2::V;                                 // two lanes of R
    using Part = typename PH::Part;
    using Part2 = typename PH2::Part;
    using FT = typename TL::FT;
    static constexpr int D = 2, NC = 4, RR = Q * Q;
    static constexpr int MID = (Q - 1) / 2, END = Q - 1;       // the nodes that stay with CORNER_*
    static constexpr int QE = (Q + 1) & ~1;                    // row of q parts, padded to whole lane pairs
    static constexpr int NCMP = PH::NCMP;
    static constexpr int PROW = NCMP * QE;                     // numbers of one row: [component][QE]
    static constexpr int PSTR = 6 * PROW;                      // numbers of one pair: [coordinate][child 0, child 1, output]

    // bytes of n arrays of r complex numbers per pair (W, the stage scratch), rounded up to the 16 bytes
    // that the geometry behind them is aligned to: one pair of odd q (a sharded apply of four
    // points) ends at 8 mod 16
    static __host__ __device__ constexpr size_t arrays(int np, int n)
    {
        return ((size_t)np * n * RR * sizeof(C) + 15) & ~(size_t)15;
    }

    // geometry of one output pair of a column level
    struct __align__(16) Geo {
        typename PH::T tA;   // features of the target box centre
        R sg;                // sign of the root's term
        int cb[2];           // coordinates of the parent source box
        int base;            // the merge block's first input slot in the CTA
        int pad;
    };
    // geometry of one merge block of a row level
    struct __align__(16) GeoR {
        int base;            // first input slot in the CTA
        int tcp;             // parent target box in the cache of node features
        int ca[2];           // coordinates of the parent target box (level l)
        int cb[2];           // coordinates of the parent source box (level l+1)
        int pad[2];
    };

    static __device__ __forceinline__ Part load1(const R *p)
    {
        Part o{};
        PH::each(o, [&](R &v, int c) { v = p[c * QE]; });
        return o;
    }
    static __device__ __forceinline__ void store1(R *p, Part o)
    {
        PH::each(o, [&](R &v, int c) { p[c * QE] = v; });
    }
    // two consecutive parts of a row (p aligned to a lane pair)
    static __device__ __forceinline__ Part2 load2(const R *p)
    {
        Part2 o{};
        PH::each(o, [&](V &v, int c) { v = *reinterpret_cast<const V *>(p + c * QE); });
        return o;
    }
    static __device__ __forceinline__ void store2(R *p, Part2 o)
    {
        PH::each(o, [&](V &v, int c) { *reinterpret_cast<V *>(p + c * QE) = v; });
    }
    static __device__ __forceinline__ Part lane(Part2 p, int j)
    {
        Part o{};
        R c[3] = {};
        PH::each(p, [&](V &v, int i) { c[i] = j ? v.y : v.x; });
        PH::each(o, [&](R &v, int i) { v = c[i]; });
        return o;
    }
    static __device__ __forceinline__ Part2 lanes(Part a, Part b)
    {
        Part2 o{};
        R ca[3] = {}, cb[3] = {};
        PH::each(a, [&](R &v, int i) { ca[i] = v; });
        PH::each(b, [&](R &v, int i) { cb[i] = v; });
        PH::each(o, [&](V &v, int i) { v.x = ca[i]; v.y = cb[i]; });
        return o;
    }

    // ---- phase tables (PM_BUILD, PM_TABLE; mixed precisions): one operand of the sincos per
    // factor, [phase of an item][item].  The blocks of levels that KArgs::corner shortens keep
    // their size; the missing factors are neither written nor read.
    static __device__ __forceinline__ int npr(const KArgs<P> &a) { return a.T << (D * a.k); }
    static __device__ __forceinline__ int64_t level_floats(const KArgs<P> &a) { return (int64_t)npr(a) * 5 * RR; }
    static __device__ __forceinline__ int64_t table_floats(const KArgs<P> &a, bool row)
    {
        int64_t f = a.k * level_floats(a);
        if (!row && (a.flags & F_SWITCH) && K != KIND_DOT && K != KIND_SEPARABLE) f += (int64_t)npr(a) * RR * RR;
        return f;
    }

    // Thread index for the work that runs beside a stage (geometry, parts and node features of the
    // next one): from the last thread down, after `used` items of other such work (4 per pair at
    // most, two rounds of the threads), so that where a small grid's CTA has more threads than the
    // stage has items, the two run on different warps instead of one after the other.
    static __device__ __forceinline__ int side(int used = 0)
    {
        int t = (int)blockDim.x - 1 - (int)threadIdx.x - used;
        if (used) {   // (0 at compile time where there is none)
            t += t < 0 ? (int)blockDim.x : 0;
            t += t < 0 ? (int)blockDim.x : 0;
        }
        return t;
    }

    // ---- column levels
    static __device__ __forceinline__ Geo pair_geo(const KArgs<P> &a, int l, int i, int j)
    {
        const int k = a.k, n = 1 << (D * k), nblk = n >> D, L = a.L;
        const int alpha = j & (NC - 1), beta = (j >> D) & (nblk - 1), tau = j >> (D * k);
        uint32_t Ap, Bstar, Apg, Bq;
        int base;
        TL::tile_of(a, tau, Ap, Bstar);
        TL::block_geo(Ap, Bstar, beta, i, k, Apg, Bq, base);
        const uint32_t Aa = (Apg << D) + alpha;
        int ca[DMAX], cbq[DMAX];
        morton_decode<D>(Aa, l + 1, ca);
        morton_decode<D>(Bq, L - l - 1, cbq);
        Geo g;
        g.cb[0] = cbq[0];
        g.cb[1] = cbq[1];
        g.base = tau * n + base;
        g.tA = tcenter<P, D, Q, K>(a, l + 1, Aa, ca);
        g.sg = PH::sign(a, g.tA);
        return g;
    }
    static __device__ __forceinline__ void geo_col(const KArgs<P> &a, Geo *G, int l, int i, int used = 0)
    {
        for (int j = side(used); j < npr(a); j += blockDim.x) G[j] = pair_geo(a, l, i, j);
    }
    // the q parts of one row: target features x and A of the row's coordinate, source entries
    // e[0..q); sp: the two nodes MID and END only; REV: in reverse order
    template <bool REV = false, class XF>
    static __device__ __forceinline__ void part_row(const KArgs<P> &a, const XF &x, const XF &A, bool first, const typename P::SE *e,
                                                    R *o, bool sp = false)
    {
        if constexpr (REV) {
#pragma unroll
            for (int j = 0; j < Q; ++j) store1(o + Q - 1 - j, PH::part_of(a, x, A, e[j], first));
            return;
        }
        if constexpr (LB) {
            if (sp) {
                store1(o + MID, PH::part_of(a, x, A, e[MID], first));
                store1(o + END, PH::part_of(a, x, A, e[END], first));
                return;
            }
        }
        const auto x2 = PH2::pack(x, x), A2 = PH2::pack(A, A);
#pragma unroll
        for (int j = 0; j + 1 < Q; j += 2) store2(o + j, PH2::part_of(a, x2, A2, e[j], e[j + 1], first));
        if constexpr (Q & 1) store1(o + Q - 1, PH::part_of(a, x, A, e[Q - 1], first));
    }
    // parts of the children's nodes (rows 0, 1 of both coordinates) of every output pair
    static __device__ __forceinline__ void parts_in(const KArgs<P> &a, const Geo *G, R *PT, int l, bool sp)
    {
        for (int it = side(); it < npr(a) * 4; it += blockDim.x) {
            const int c = it & 1, dim = (it >> 1) & 1, j = it >> 2;
            part_row(a, G[j].tA.x[dim], G[j].tA.A[dim], dim == 0, a.st[dim] + soff<Q>(a.L, l) + (2 * G[j].cb[dim] + c) * (Q + 2),
                     PT + j * PSTR + (dim * 3 + c) * PROW, sp);
        }
    }
    // the same for the first level of a pass, each item with its own geometry, which one item of a
    // pair keeps: one barrier and one chain of loads less than the geometry first
    static __device__ __forceinline__ void parts_first(const KArgs<P> &a, Geo *G, R *PT, int l, int i, bool sp)
    {
        for (int it = side(); it < npr(a) * 4; it += blockDim.x) {
            const int c = it & 1, dim = (it >> 1) & 1, j = it >> 2;
            const Geo g = pair_geo(a, l, i, j);
            if ((it & 3) == 0) G[j] = g;
            part_row(a, dim ? g.tA.x[1] : g.tA.x[0], dim ? g.tA.A[1] : g.tA.A[0], dim == 0,
                     a.st[dim] + soff<Q>(a.L, l) + (2 * (dim ? g.cb[1] : g.cb[0]) + c) * (Q + 2), PT + j * PSTR + (dim * 3 + c) * PROW, sp);
        }
    }
    // parts of the output box's nodes (row 2)
    static __device__ __forceinline__ void parts_out(const KArgs<P> &a, const Geo *G, R *PT, int l)
    {
        for (int it = side(); it < npr(a) * 2; it += blockDim.x) {
            const int dim = it & 1, j = it >> 1;
            part_row(a, G[j].tA.x[dim], G[j].tA.A[dim], dim == 0, a.st[dim] + soff<Q>(a.L, l + 1) + G[j].cb[dim] * (Q + 2),
                     PT + j * PSTR + (dim * 3 + 2) * PROW);
        }
    }
    // the q factors of a row of parts and one part of the other coordinate: o[j] = e^{2 pi i Phi}
    static __device__ __forceinline__ void phase_row(R sg, const R *p0, const Part &p1, C *o)
    {
        const Part2 p12 = PH2::dup(p1);
#pragma unroll
        for (int j = 0; j + 1 < Q; j += 2)
            TL::template ph2<PM_COMPUTE>(PH2::dup(sg), PH2::add(load2(p0 + j), p12), nullptr, nullptr, o[j], o[j + 1]);
        if constexpr (Q & 1) o[Q - 1] = TL::template ph<PM_COMPUTE>(sg, PH::add(load1(p0 + Q - 1), p1), nullptr);
    }

    template <class MS>
    static __device__ __forceinline__ void imac(C &acc, const MS &ms, int h, int t, int u, C v)
    {
        mmac<Q, LB>(acc, ms, h, t, u, v);
    }
    static __device__ __forceinline__ R sgn(const KArgs<P> &a, const Geo &g) { return K == KIND_HYPRADON ? g.sg : (R)a.sc.sgn; }

    // stage A: items (pair, c_1, t'_1): modulate the 2q inputs, contract dimension 0; SP: the
    // inputs' nodes MID and END of both dimensions only
    template <int PM, bool SP>
    static __device__ __forceinline__ void col_a(const KArgs<P> &a, const C *Wt, C *S, const Geo *G, const R *PT, int i, const FT &fa)
    {
        constexpr int QA = SP ? 2 : Q;
        const int tp = threadIdx.x % QA, hh = threadIdx.x / QA, chi = hh & 1, tq = SP ? (tp ? END : MID) : tp;
        const int step = blockDim.x / (2 * QA);
        if (hh >> 1 >= step) return;   // threads beyond a whole number of pairs
        for (int j = hh >> 1; j < npr(a); j += step) {
            const int it = j * 2 * Q + chi * Q + tq;
            const int base = G[j].base;
            const C *w0 = Wt + (base + ((2 * chi) << (D * i))) * RR + Q * tq;
            const C *w1 = Wt + (base + ((2 * chi + 1) << (D * i))) * RR + Q * tq;
            const R *p0 = PT + j * PSTR;
            Part2 P1{};
            V sg{};
            if constexpr (PM != PM_TABLE) {
                P1 = PH2::dup(load1(p0 + (3 + chi) * PROW + tq));
                sg = PH2::dup(sgn(a, G[j]));
            }
            C acc[Q];
#pragma unroll
            for (int t = 0; t < Q; ++t) acc[t] = czero<C>();
            // factors of node ta of child ca and node tb of child cb in one pair of lanes
            auto two = [&](int ca, int ta, int cb, int tb) {
                C E0, E1;
                Part2 pt{};
                if constexpr (PM != PM_TABLE) {
                    const R *ra = p0 + ca * PROW + ta, *rb = p0 + cb * PROW + tb;
                    pt = PH2::add(ca == cb && tb == ta + 1 && !(ta & 1) ? load2(ra) : lanes(load1(ra), load1(rb)), P1);
                }
                TL::template ph2<PM>(sg, pt, fa.at(ca * Q + ta, it), fa.at(cb * Q + tb, it), E0, E1);
                const C u0 = cmul(E0, (ca ? w1 : w0)[ta]), u1 = cmul(E1, (cb ? w1 : w0)[tb]);
#pragma unroll
                for (int t0 = 0; t0 < Q; ++t0) {
                    imac(acc[t0], a, ca, t0, ta, u0);
                    imac(acc[t0], a, cb, t0, tb, u1);
                }
            };
            if constexpr (SP) {
                two(0, MID, 0, END);
                two(1, MID, 1, END);
            } else {
#pragma unroll
                for (int cl = 0; cl < 2; ++cl)
#pragma unroll
                    for (int t0p = 0; t0p + 1 < Q; t0p += 2) two(cl, t0p, cl, t0p + 1);
                if constexpr (Q & 1) two(0, Q - 1, 1, Q - 1);   // the last nodes of both children
            }
            C *so = S + it * Q;
#pragma unroll
            for (int t = 0; t < Q; ++t) so[t] = acc[t];
        }
    }
    // stage B: items (pair, t_0): contract dimension 1 and c_1, demodulate
    template <int PM, bool SP>
    static __device__ __forceinline__ void col_b(const KArgs<P> &a, C *Wt, const C *S, const Geo *G, const R *PT, int i, const FT &fb)
    {
        const int tl = threadIdx.x % Q;
        for (int j = threadIdx.x / Q; j < npr(a); j += blockDim.x / Q) {
            const int it = j * Q + tl;
            const C *si = S + j * 2 * RR + tl;
            C acc[Q];
#pragma unroll
            for (int t = 0; t < Q; ++t) acc[t] = czero<C>();
#pragma unroll
            for (int chi = 0; chi < 2; ++chi)
#pragma unroll
                for (int tqp = 0; tqp < Q; ++tqp) {
                    if (SP && tqp != MID && tqp != END) continue;
                    const C v = si[(chi * Q + tqp) * Q];
#pragma unroll
                    for (int tq = 0; tq < Q; ++tq) imac(acc[tq], a, chi, tq, tqp, v);
                }
            C *wo = Wt + (G[j].base + ((j & (NC - 1)) << (D * i))) * RR + tl;
            const R *p1 = PT + j * PSTR + 5 * PROW;
            Part P0{};
            R sg{};
            if constexpr (PM != PM_TABLE) {
                P0 = load1(PT + j * PSTR + 2 * PROW + tl);
                sg = sgn(a, G[j]);
            }
            const Part2 P02 = PH2::dup(P0);
#pragma unroll
            for (int tq = 0; tq + 1 < Q; tq += 2) {
                C E0, E1;
                Part2 pt{};
                if constexpr (PM != PM_TABLE) pt = PH2::add(load2(p1 + tq), P02);
                TL::template ph2<PM>(PH2::dup(sg), pt, fb.at(tq, it), fb.at(tq + 1, it), E0, E1);
                wo[tq * Q] = cjmul(E0, acc[tq]);
                wo[(tq + 1) * Q] = cjmul(E1, acc[tq + 1]);
            }
            if constexpr (Q & 1) {
                Part pt{};
                if constexpr (PM != PM_TABLE) pt = PH::add(load1(p1 + Q - 1), P0);
                wo[(Q - 1) * Q] = cjmul(TL::template ph<PM>(sg, pt, fb.at(Q - 1, it)), acc[Q - 1]);
            }
        }
    }

    // first step and first merge with points at box corners: slot (block b, alpha) holds g of
    // the block's four leaves at nodes MID (upper half of a dimension) and END (lower half)
    static __device__ __forceinline__ void init_corner(const KArgs<P> &a, C *Wt, int rhs)
    {
        const int k = a.k, n = 1 << (D * k), nblk = n >> D, L = a.L;
        if (a.k == 1) {   // no level of this pass follows: the switch may read every node
            for (int j = threadIdx.x; j < a.T * n * RR; j += blockDim.x) Wt[j] = czero<C>();
            __syncthreads();
        }
        for (int it = threadIdx.x; it < a.T * n; it += blockDim.x) {
            const int c = it & (NC - 1), b = (it >> D) & (nblk - 1), tau = it >> (D * k);
            uint32_t Ap, Bstar;
            TL::tile_of(a, tau, Ap, Bstar);
            int cb[DMAX];
            morton_decode<D>((Bstar << (D * k)) + (it & (n - 1)), L, cb);
            const C v = a.g[(int64_t)rhs * a.npts + ((int64_t)cb[0] << L) + cb[1]];
            C *w = Wt + (tau * n + (b << D)) * RR + ((c & 1) ? MID : END) + ((c >> 1) ? MID : END) * Q;
#pragma unroll
            for (int al = 0; al < NC; ++al) w[al * RR] = v;
        }
    }
    // last merge and last step with points at box corners: tiles at level L - 1
    static __device__ __forceinline__ void final_corner(const KArgs<P> &a, const C *Wt, int rhs)
    {
        const int k = a.k, n = 1 << (D * k), nblk = n >> D, L = a.L;
        for (int it = threadIdx.x; it < a.T * n; it += blockDim.x) {
            const int al = it & (NC - 1), ra = (it >> D) & (nblk - 1), tau = it >> (D * k);
            uint32_t Ap, Bstar;
            TL::tile_of(a, tau, Ap, Bstar);
            int ca[DMAX];
            morton_decode<D>((((Ap << (D * (k - 1))) + digit_rev<D>(ra, k - 1)) << D) + al, L, ca);
            const C *w = Wt + (tau * n + ra) * RR + ((al & 1) ? MID : END) + ((al >> 1) ? MID : END) * Q;
            C acc = w[0];
#pragma unroll
            for (int c = 1; c < NC; ++c) acc = madd(acc, w[(c * nblk) * RR]);
            a.f[(int64_t)rhs * a.npts + ((int64_t)ca[0] << L) + ca[1]] = acc;
        }
    }

    // geometry of the pairs at the switch: (target box, source box) coordinates
    static __device__ __forceinline__ void geo_switch(const KArgs<P> &a, int4 *GS, int l)
    {
        const int k = a.k, n = 1 << (D * k);
        for (int j = side(); j < a.T * n; j += blockDim.x) {
            uint32_t Ap, Bstar;
            TL::tile_of(a, j >> (D * k), Ap, Bstar);
            int ca[DMAX], cb[DMAX];
            morton_decode<D>((Ap << (D * k)) + digit_rev<D>(j & (n - 1), k), l, ca);
            morton_decode<D>(Bstar, a.L - l, cb);
            GS[j] = make_int4(ca[0], ca[1], cb[0], cb[1]);
        }
    }
    // the switch: items (pair, s), all r sources in pairs of lanes: (t_0, t_0 + 1), and for odd
    // q the last t_0 of two consecutive t_1.  The parts of coordinate 0 stay in registers.
    template <int PM>
    static __device__ __forceinline__ void sw(const KArgs<P> &a, const C *Wt, C *S, const int4 *GS, int l, const FT &fs)
    {
        for (int it = threadIdx.x; it < npr(a) * RR; it += blockDim.x) {
            const int s = it % RR, j = it / RR;
            Part2 P0[(Q + 1) / 2];
            typename PH2::T t2{};
            V sg{};
            int4 g = make_int4(0, 0, 0, 0);
            if constexpr (PM != PM_TABLE) {
                g = GS[j];
                const int ca[DMAX] = {g.x, g.y, 0}, sk[DMAX] = {s % Q, s / Q, 0};
                const typename PH::T t = tpoint<P, D, Q, K>(a, l, ca, sk);
                t2 = PH2::dup(t);
                sg = PH2::dup(PH::sign(a, t));
#pragma unroll
                for (int t0 = 0; t0 < Q; t0 += 2)
                    P0[t0 / 2] = PH2::part(a, t2, sget<P, Q>(a, 0, l, g.z, t0), sget<P, Q>(a, 0, l, g.z, t0 + 1 < Q ? t0 + 1 : t0), 0);
            }
            C acc = czero<C>();
            const C *u = Wt + j * RR;
            auto two = [&](const Part2 &p, int ta, int tb) {
                C E0, E1;
                TL::template ph2<PM>(sg, p, fs.at(ta, it), fs.at(tb, it), E0, E1);
                cmac(acc, E0, u[ta]);
                cmac(acc, E1, u[tb]);
            };
#pragma unroll 1
            for (int t1 = 0; t1 + 1 < Q; t1 += 2) {
                Part2 pp{};   // coordinate 1: lanes t_1, t_1 + 1
                if constexpr (PM != PM_TABLE) pp = PH2::part(a, t2, sget<P, Q>(a, 1, l, g.w, t1), sget<P, Q>(a, 1, l, g.w, t1 + 1), 1);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const Part2 p1 = PH2::dup(lane(pp, h));
#pragma unroll
                    for (int t0 = 0; t0 + 1 < Q; t0 += 2)
                        two(PH2::add(P0[t0 / 2], p1), (t1 + h) * Q + t0, (t1 + h) * Q + t0 + 1);
                }
                if constexpr (Q & 1) two(PH2::add(PH2::dup(lane(P0[Q / 2], 0)), pp), t1 * Q + Q - 1, (t1 + 1) * Q + Q - 1);
            }
            if constexpr (Q & 1) {
                Part p1{};
                if constexpr (PM != PM_TABLE) p1 = PH::part(a, PH2::one(t2), sget<P, Q>(a, 1, l, g.w, Q - 1), 1);
                const Part2 p12 = PH2::dup(p1);
#pragma unroll
                for (int t0 = 0; t0 + 1 < Q; t0 += 2) two(PH2::add(P0[t0 / 2], p12), (Q - 1) * Q + t0, (Q - 1) * Q + t0 + 1);
                const Part pl = PH::add(lane(P0[Q / 2], 0), p1);
                cmac(acc, TL::template ph<PM>(sg.x, pl, fs.at(RR - 1, it)), u[RR - 1]);
            }
            S[it] = acc;
        }
    }

    // ---- row levels
    static __device__ __forceinline__ void geo_row(const KArgs<P> &a, GeoR *G, int l, int i)
    {
        const int k = a.k, n = 1 << (D * k), nblk = n >> D, L = a.L, nb = 1 << (D * i);
        for (int j = side(); j < a.T * nblk; j += blockDim.x) {
            const int beta = j & (nblk - 1), tau = j >> (D * (k - 1));
            uint32_t Ap, Bstar, Apg, Bq;
            int base, ca[DMAX], cb[DMAX];
            TL::tile_of(a, tau, Ap, Bstar);
            TL::block_geo(Ap, Bstar, beta, i, k, Apg, Bq, base);
            morton_decode<D>(Apg, l, ca);
            morton_decode<D>(Bq, L - l - 1, cb);
            G[j] = GeoR{tau * n + base, tau * nb + (int)digit_rev<D>(beta & (nb - 1), i), {ca[0], ca[1]}, {cb[0], cb[1]}, {0, 0}};
        }
    }
    // features of the nodes of the tiles' target boxes at level l = l0 + i (T 2^{Di} boxes x r)
    static __device__ __forceinline__ void node_cache(const KArgs<P> &a, typename PH::T *TC, int l, int i, int used = 0)
    {
        const int nb = 1 << (D * i);
        for (int j = side(used); j < a.T * nb * RR; j += blockDim.x) {
            const int t = j % RR, aloc = (j / RR) & (nb - 1), tau = (j / RR) >> (D * i);
            uint32_t Ap, Bstar;
            TL::tile_of(a, tau, Ap, Bstar);
            int ca[DMAX];
            morton_decode<D>((Ap << (D * i)) + aloc, l, ca);
            const int tk[DMAX] = {t % Q, t / Q, 0};
            TC[j] = tpoint<P, D, Q, K>(a, l, ca, tk);
        }
    }
    // the four children's factors at one target node: E[c], c = c_0 + 2 c_1
    template <int PM>
    static __device__ __forceinline__ void four(const KArgs<P> &a, const typename PH::T &t, const typename P::SE *s0,
                                                const typename P::SE *s1, const FT &ft, int j0, int it, C *E)
    {
        Part2 P0{}, P1{};
        V sg{};
        if constexpr (PM != PM_TABLE) {
            const typename PH2::T t2 = PH2::dup(t);
            sg = PH2::dup(PH::sign(a, t));
            P0 = PH2::part(a, t2, s0[0], s0[1], 0);   // lanes c_0 = 0, 1
            P1 = PH2::part(a, t2, s1[0], s1[1], 1);   // lanes c_1 = 0, 1
        }
        TL::template ph2<PM>(sg, PH2::add(P0, P1), ft.at(j0, it), ft.at(j0 + 3, it), E[0], E[3]);
        TL::template ph2<PM>(sg, PH2::add(P0, PH2::swap(P1)), ft.at(j0 + 2, it), ft.at(j0 + 1, it), E[2], E[1]);
    }
    // pre-modulation, in place: items (block, t), the block's four inputs at node t of the parent
    // box (conjugate factors; ADJ: the factors themselves)
    template <int PM, bool ADJ = false>
    static __device__ __forceinline__ void row_p(const KArgs<P> &a, C *Wt, const GeoR *G, const typename PH::T *TC, int l, int i,
                                                 const FT &fa)
    {
        for (int it = threadIdx.x; it < (npr(a) >> D) * RR; it += blockDim.x) {
            const int t = it % RR, b = it / RR;
            const GeoR g = G[b];
            typename P::SE s0[2], s1[2];
            typename PH::T tn{};
            if constexpr (PM != PM_TABLE) {
                tn = TC[g.tcp * RR + t];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    s0[h] = sget<P, Q>(a, 0, l, 2 * g.cb[0] + h, Q);
                    s1[h] = sget<P, Q>(a, 1, l, 2 * g.cb[1] + h, Q);
                }
            }
            C E[NC];
            four<PM>(a, tn, s0, s1, fa, 0, it, E);
            C *w = Wt + g.base * RR + t;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                C &x = w[(c << (D * i)) * RR];
                x = ADJ ? cmul(E[c], x) : cjmul(E[c], x);
            }
        }
    }
    // stage A: items (block, c, t_1): contract dimension 0 for both children alpha_0; SP: the
    // outputs' nodes MID and END only
    template <bool SP>
    static __device__ __forceinline__ void row_a(const KArgs<P> &a, const C *Wt, C *S, const GeoR *G, int i)
    {
        const int th = threadIdx.x % Q;
        for (int j = threadIdx.x / Q; j < npr(a); j += blockDim.x / Q) {
            const int it = j * Q + th, c = j & (NC - 1), b = j >> D;
            const C *w = Wt + (G[b].base + (c << (D * i))) * RR + th * Q;
            C z[2][Q];
#pragma unroll
            for (int s0 = 0; s0 < Q; ++s0) z[0][s0] = z[1][s0] = czero<C>();
#pragma unroll
            for (int t0 = 0; t0 < Q; ++t0) {
                const C u = w[t0];
#pragma unroll
                for (int s0 = 0; s0 < Q; ++s0) {
                    if (SP && s0 != MID && s0 != END) continue;
                    imac(z[0][s0], a, 0, t0, s0, u);
                    imac(z[1][s0], a, 1, t0, s0, u);
                }
            }
            C *so = S + it * 2 * Q;
#pragma unroll
            for (int s0 = 0; s0 < Q; ++s0) {
                if (SP && s0 != MID && s0 != END) continue;
                so[s0] = z[0][s0];
                so[Q + s0] = z[1][s0];
            }
        }
    }
    // stage B: items (pair, s_0): contract dimension 1 per child, post-modulate, sum over the
    // children.  TC: node features of the output boxes, null where no two pairs share a box.
    // M_1 is M_0 with both indices reversed, so a child alpha_1 = 1 reads and writes dimension 1
    // backwards and the coefficients are those of M_0 (compile-time operands).
    template <int PM, bool SP>
    static __device__ __forceinline__ void row_b(const KArgs<P> &a, C *Wt, const C *S, const GeoR *G, const typename PH::T *TC, int l,
                                                 int i, const FT &fb)
    {
        constexpr int QB = SP ? 2 : Q;
        const int sp = threadIdx.x % QB, s0 = SP ? (sp ? END : MID) : sp;
        if (threadIdx.x / QB >= blockDim.x / QB) return;   // threads beyond a whole number of pairs
        for (int pj = threadIdx.x / QB; pj < npr(a); pj += blockDim.x / QB) {
            const int it = pj * Q + s0, alpha = pj & (NC - 1), b = pj >> D;
            const int a0 = alpha & 1, a1 = alpha >> 1;
            const GeoR g = G[b];
            const C *si = S + b * NC * Q * 2 * Q + a0 * Q + s0 + (a1 ? (Q - 1) * 2 * Q : 0);
            const int ts = a1 ? -2 * Q : 2 * Q;
            C v[NC][QB];   // SP: nodes MID and END
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const C *sc = si + c * Q * 2 * Q;
                if constexpr (SP) {
                    v[c][0] = czero<C>();
#pragma unroll
                    for (int t1 = 0; t1 < Q; ++t1) imac(v[c][0], a, 0, t1, MID, sc[t1 * ts]);
                    v[c][1] = sc[(a1 ? MID : END) * ts];
                } else {
#pragma unroll
                    for (int s1 = 0; s1 < Q; ++s1) v[c][s1] = czero<C>();
#pragma unroll
                    for (int t1 = 0; t1 < Q; ++t1) {
                        const C zz = sc[t1 * ts];
#pragma unroll
                        for (int s1 = 0; s1 < Q; ++s1) imac(v[c][s1], a, 0, t1, s1, zz);
                    }
                }
            }
            typename P::SE e0[2], e1[2];
            if constexpr (PM != PM_TABLE) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    e0[h] = sget<P, Q>(a, 0, l, 2 * g.cb[0] + h, Q);
                    e1[h] = sget<P, Q>(a, 1, l, 2 * g.cb[1] + h, Q);
                }
            }
            C *wo = Wt + (g.base + (alpha << (D * i))) * RR + s0;
#pragma unroll
            for (int j = 0; j < QB; ++j) {
                const int s1 = SP ? (j ? END : MID) : (a1 ? Q - 1 - j : j);
                typename PH::T tS{};
                if constexpr (PM != PM_TABLE) {
                    if (TC) {
                        tS = TC[(g.tcp * NC + alpha) * RR + s1 * Q + s0];
                    } else {
                        const int ca[DMAX] = {2 * g.ca[0] + a0, 2 * g.ca[1] + a1, 0}, sk[DMAX] = {s0, s1, 0};
                        tS = tpoint<P, D, Q, K>(a, l + 1, ca, sk);
                    }
                }
                C E[NC];
                four<PM>(a, tS, e0, e1, fb, j * NC, it, E);
                C acc = cmul(E[0], v[0][j]);
                cmac(acc, E[3], v[3][j]);
                cmac(acc, E[2], v[2][j]);
                cmac(acc, E[1], v[1][j]);
                wo[s1 * Q] = acc;
            }
        }
    }

    // ====================================================================
    // Conjugate transposes for one right-hand side (mixed precisions): the same parts and
    // factors, the levels in reverse.  On entry to a level the slot of output alpha of a merge
    // block holds the level-(l+1) weights, on exit the slot of input c the level-l weights.

    // column level, stage A: items (pair alpha, t_1): re-modulate out_alpha at the nodes of B',
    // contract dimension 0 into both children c_0 -> S[pair][t_1][c_0][t'_0]; SP: nodes MID and
    // END of the children only
    template <bool SP>
    static __device__ __forceinline__ void col_adj_a(const KArgs<P> &a, const C *Wt, C *S, const Geo *G, const R *PT, int i)
    {
        const int th = threadIdx.x % Q;
        for (int j = threadIdx.x / Q; j < npr(a); j += blockDim.x / Q) {
            const C *w = Wt + (G[j].base + ((j & (NC - 1)) << (D * i))) * RR + th * Q;
            const R *pt = PT + j * PSTR;
            C E[Q], z[2][Q];
            phase_row(sgn(a, G[j]), pt + 2 * PROW, load1(pt + 5 * PROW + th), E);
#pragma unroll
            for (int s0 = 0; s0 < Q; ++s0) z[0][s0] = z[1][s0] = czero<C>();
#pragma unroll
            for (int t0 = 0; t0 < Q; ++t0) {
                const C u = cmul(E[t0], w[t0]);
#pragma unroll
                for (int s0 = 0; s0 < Q; ++s0) {
                    if (SP && s0 != MID && s0 != END) continue;
                    imac(z[0][s0], a, 0, t0, s0, u);
                    imac(z[1][s0], a, 1, t0, s0, u);
                }
            }
            C *so = S + (j * Q + th) * 2 * Q;
#pragma unroll
            for (int s0 = 0; s0 < Q; ++s0) {
                if (SP && s0 != MID && s0 != END) continue;
                so[s0] = z[0][s0];
                so[Q + s0] = z[1][s0];
            }
        }
    }
    // stage B: items (input pair c, t'_0): contract dimension 1 per output alpha, conjugate
    // modulation at the nodes of B_c, sum over alpha.  The rows of parts of children c_1 = 1 are
    // stored in reverse order (parts_in_adj), as dimension 1 runs backwards there (row_b).
    template <bool SP>
    static __device__ __forceinline__ void col_adj_b(const KArgs<P> &a, C *Wt, const C *S, const Geo *G, const R *PT, int i)
    {
        constexpr int QB = SP ? 2 : Q;
        const int sp = threadIdx.x % QB, s0 = SP ? (sp ? END : MID) : sp;
        if (threadIdx.x / QB >= blockDim.x / QB) return;   // threads beyond a whole number of pairs
        for (int j = threadIdx.x / QB; j < npr(a); j += blockDim.x / QB) {
            const int c0 = j & 1, c1 = (j >> 1) & 1, b0 = j & ~(NC - 1);
            C acc[QB];
#pragma unroll
            for (int e = 0; e < QB; ++e) acc[e] = czero<C>();
#pragma unroll 1
            for (int al = 0; al < NC; ++al) {
                const C *sc = S + (b0 + al) * Q * 2 * Q + c0 * Q + s0 + (c1 ? (Q - 1) * 2 * Q : 0);
                const int ts = c1 ? -2 * Q : 2 * Q;
                const R *pt = PT + (b0 + al) * PSTR;
                const R sg = sgn(a, G[b0 + al]);
                const Part P0 = load1(pt + c0 * PROW + s0);
                const R *p1 = pt + (3 + c1) * PROW;
                if constexpr (SP) {   // dimension-1 nodes MID and END: positions MID and (reversed) 0 or END
                    C v0 = czero<C>(), E0, E1;
#pragma unroll
                    for (int t1 = 0; t1 < Q; ++t1) imac(v0, a, 0, t1, MID, sc[t1 * ts]);
                    const C v1 = sc[(c1 ? MID : END) * ts];
                    TL::template ph2<PM_COMPUTE>(PH2::dup(sg), PH2::add(lanes(load1(p1 + MID), load1(p1 + (c1 ? 0 : END))), PH2::dup(P0)),
                                                 nullptr, nullptr, E0, E1);
                    acc[0] = madd(acc[0], cjmul(E0, v0));
                    acc[1] = madd(acc[1], cjmul(E1, v1));
                } else {
                    C v[Q], E[Q];
#pragma unroll
                    for (int e = 0; e < Q; ++e) v[e] = czero<C>();
#pragma unroll
                    for (int t1 = 0; t1 < Q; ++t1) {
                        const C zz = sc[t1 * ts];
#pragma unroll
                        for (int e = 0; e < Q; ++e) imac(v[e], a, 0, t1, e, zz);
                    }
                    phase_row(sg, p1, P0, E);
#pragma unroll
                    for (int e = 0; e < Q; ++e) acc[e] = madd(acc[e], cjmul(E[e], v[e]));
                }
            }
            C *wo = Wt + (G[j].base + ((j & (NC - 1)) << (D * i))) * RR + s0;
#pragma unroll
            for (int e = 0; e < QB; ++e) wo[(SP ? (e ? END : MID) : (c1 ? Q - 1 - e : e)) * Q] = acc[e];
        }
    }
    static __device__ __forceinline__ void parts_in_adj(const KArgs<P> &a, const Geo *G, R *PT, int l)
    {
        for (int it = side(); it < npr(a) * 4; it += blockDim.x) {
            const int c = it & 1, dim = (it >> 1) & 1, j = it >> 2;
            const typename P::SE *e = a.st[dim] + soff<Q>(a.L, l) + (2 * G[j].cb[dim] + c) * (Q + 2);
            R *o = PT + j * PSTR + (dim * 3 + c) * PROW;
            if (dim && c)
                part_row<true>(a, G[j].tA.x[1], G[j].tA.A[1], false, e, o);
            else
                part_row(a, G[j].tA.x[dim], G[j].tA.A[dim], dim == 0, e, o);
        }
    }
    // switch: u(t) = sum_s e^{-2 pi i Phi(x_s, y_t)} v(s); items (pair, t), q per thread.  As in
    // TileMR::switch_adj the sum runs over s_1, whose parts go to shared memory first (in the
    // space behind W, idle here).
    static constexpr int PSW = 2 * Q * NCMP * QE;   // [coordinate][t][component][s_0]
    static __device__ __forceinline__ void sw_adj(const KArgs<P> &a, C *Wt, R *PS, int l)
    {
        const int k = a.k, n = 1 << (D * k), np = npr(a);
        R *SG = PS + np * PSW;
        C acc[Q];
#pragma unroll
        for (int j = 0; j < Q; ++j) acc[j] = czero<C>();
#pragma unroll 1
        for (int s1 = 0; s1 < Q; ++s1) {
            if (s1) __syncthreads();   // the previous digit's parts have been used
            for (int it = threadIdx.x; it < np * 2 * Q; it += blockDim.x) {
                const int s0 = it % Q, dim = (it / Q) & 1, pr = it / (2 * Q);
                uint32_t Ap, Bstar;
                TL::tile_of(a, pr >> (D * k), Ap, Bstar);
                int ca[DMAX], cb[DMAX];
                morton_decode<D>((Ap << (D * k)) + digit_rev<D>(pr & (n - 1), k), l, ca);
                morton_decode<D>(Bstar, a.L - l, cb);
                const int sk[DMAX] = {s0, s1, 0};
                const typename PH::T tS = tpoint<P, D, Q, K>(a, l, ca, sk);
                const auto xf = dim ? tS.x[1] : tS.x[0];
                const auto Af = dim ? tS.A[1] : tS.A[0];
                const typename P::SE *e = a.st[dim] + soff<Q>(a.L, l) + (dim ? cb[1] : cb[0]) * (Q + 2);
                R *o = PS + pr * PSW + dim * Q * NCMP * QE + s0;
#pragma unroll
                for (int tt = 0; tt < Q; ++tt) store1(o + tt * NCMP * QE, PH::part_of(a, xf, Af, e[tt], dim == 0));
                if (dim == 0) SG[pr * Q + s0] = PH::sign(a, tS);
            }
            __syncthreads();
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                const int it = threadIdx.x + j * blockDim.x;
                if (it >= np * RR) continue;
                const int t = it % RR, pl = it / RR;
                const R *q0 = PS + pl * PSW + (t % Q) * NCMP * QE, *q1 = PS + pl * PSW + (Q + t / Q) * NCMP * QE;
                const C *v = Wt + pl * RR + s1 * Q;
#pragma unroll
                for (int s0 = 0; s0 + 1 < Q; s0 += 2) {
                    V sg = PH2::dup((R)a.sc.sgn);
                    if constexpr (K == KIND_HYPRADON) {
                        sg.x = SG[pl * Q + s0];
                        sg.y = SG[pl * Q + s0 + 1];
                    }
                    C E0, E1;
                    TL::template ph2<PM_COMPUTE>(sg, PH2::add(load2(q0 + s0), load2(q1 + s0)), nullptr, nullptr, E0, E1);
                    acc[j] = madd(acc[j], cjmul(E0, v[s0]));
                    acc[j] = madd(acc[j], cjmul(E1, v[s0 + 1]));
                }
                if constexpr (Q & 1) {
                    const R sg = K == KIND_HYPRADON ? SG[pl * Q + Q - 1] : (R)a.sc.sgn;
                    acc[j] = madd(acc[j], cjmul(TL::template ph<PM_COMPUTE>(sg, PH::add(load1(q0 + Q - 1), load1(q1 + Q - 1)), nullptr),
                                                v[Q - 1]));
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            const int it = threadIdx.x + j * blockDim.x;
            if (it < np * RR) Wt[it] = acc[j];
        }
        __syncthreads();
    }

    // row level, stage E: items (pair alpha, s): the products of out_alpha(s) with the conjugate
    // factors of the four inputs c -> X[block][c][alpha][s]; SP: nodes MID and END only
    template <bool SP>
    static __device__ __forceinline__ void row_adj_e(const KArgs<P> &a, const C *Wt, C *X, const GeoR *G, const typename PH::T *TC, int l,
                                                     int i)
    {
        constexpr int RS = SP ? 4 : RR;
        for (int it = threadIdx.x; it < npr(a) * RS; it += blockDim.x) {
            const int e = it % RS, j = it / RS, al = j & (NC - 1), b = j >> D;
            const int t = SP ? ((e & 1) ? END : MID) + ((e & 2) ? END : MID) * Q : e;
            const GeoR g = G[b];
            typename PH::T tS;
            if (TC) {
                tS = TC[(g.tcp * NC + al) * RR + t];
            } else {
                const int ca[DMAX] = {2 * g.ca[0] + (al & 1), 2 * g.ca[1] + (al >> 1), 0}, sk[DMAX] = {t % Q, t / Q, 0};
                tS = tpoint<P, D, Q, K>(a, l + 1, ca, sk);
            }
            typename P::SE s0[2], s1[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                s0[h] = sget<P, Q>(a, 0, l, 2 * g.cb[0] + h, Q);
                s1[h] = sget<P, Q>(a, 1, l, 2 * g.cb[1] + h, Q);
            }
            C E[NC];
            four<PM_COMPUTE>(a, tS, s0, s1, FT{nullptr, 0}, 0, 0, E);
            const C w = Wt[(g.base + (al << (D * i))) * RR + t];
            C *o = X + (b * NC * NC + al) * RR + t;
#pragma unroll
            for (int c = 0; c < NC; ++c) o[c * NC * RR] = cjmul(E[c], w);
        }
    }
    // stage A: items (input pair c, alpha_1, s_1): contract dimension 0 and alpha_0
    template <bool SP>
    static __device__ __forceinline__ void row_adj_a(const KArgs<P> &a, const C *X, C *S)
    {
        constexpr int QA = SP ? 2 : Q;
        const int tp = threadIdx.x % QA, hh = threadIdx.x / QA, ahi = hh & 1, sq = SP ? (tp ? END : MID) : tp;
        const int step = blockDim.x / (2 * QA);
        if (hh >> 1 >= step) return;   // threads beyond a whole number of pairs
        for (int j = hh >> 1; j < npr(a); j += step) {
            C acc[Q];
#pragma unroll
            for (int t = 0; t < Q; ++t) acc[t] = czero<C>();
#pragma unroll
            for (int al = 0; al < 2; ++al) {
                const C *xi = X + (j * NC + (al | (ahi << 1))) * RR + sq * Q;
#pragma unroll
                for (int s0 = 0; s0 < Q; ++s0) {
                    if (SP && s0 != MID && s0 != END) continue;
                    const C u = xi[s0];
#pragma unroll
                    for (int t0 = 0; t0 < Q; ++t0) imac(acc[t0], a, al, t0, s0, u);
                }
            }
            C *so = S + ((j * 2 + ahi) * Q + sq) * Q;
#pragma unroll
            for (int t = 0; t < Q; ++t) so[t] = acc[t];
        }
    }
    // stage B: items (input pair c, t_0): contract dimension 1 and alpha_1
    template <bool SP>
    static __device__ __forceinline__ void row_adj_b(const KArgs<P> &a, C *Wt, const C *S, const GeoR *G, int i)
    {
        const int tl = threadIdx.x % Q;
        for (int j = threadIdx.x / Q; j < npr(a); j += blockDim.x / Q) {
            C acc[Q];
#pragma unroll
            for (int t = 0; t < Q; ++t) acc[t] = czero<C>();
#pragma unroll
            for (int ahi = 0; ahi < 2; ++ahi)
#pragma unroll
                for (int sq = 0; sq < Q; ++sq) {
                    if (SP && sq != MID && sq != END) continue;
                    const C v = S[((j * 2 + ahi) * Q + sq) * Q + tl];
#pragma unroll
                    for (int tq = 0; tq < Q; ++tq) imac(acc[tq], a, ahi, tq, sq, v);
                }
            C *wo = Wt + (G[j >> D].base + ((j & (NC - 1)) << (D * i))) * RR + tl;
#pragma unroll
            for (int tq = 0; tq < Q; ++tq) wo[tq * Q] = acc[tq];
        }
    }

    static __host__ __device__ size_t col_adj_smem(int np) { return col_smem(np, false); }
    static __host__ __device__ size_t row_adj_smem(int np, int T, int k)
    {
        const size_t boxes = (size_t)T * ((((size_t)1 << (D * k)) - 1) / 3);   // levels 0 .. k-1 of the tiles
        return arrays(np, 3 + NC) + (size_t)k * (size_t)(np >> D) * sizeof(GeoR) + boxes * RR * sizeof(typename PH::T);
    }

    static __device__ __forceinline__ void col_pass_adj(const KArgs<P> &a, unsigned char *smem)
    {
        const int np = npr(a), rhs = blockIdx.y;
        C *Wt = reinterpret_cast<C *>(smem), *S = Wt + np * RR;
        Geo *G = reinterpret_cast<Geo *>(smem + arrays(np, 3));
        R *PT = reinterpret_cast<R *>(reinterpret_cast<int4 *>(G + 2 * np) + np);
        const bool skip0 = LB && (a.corner & CORNER_SRC) && (a.flags & F_INIT), sp1 = LB && (a.corner & CORNER_SRC);
        const int i0 = skip0 ? 1 : 0;
        TL::load_strided(a, Wt, rhs);
        __syncthreads();
        if (a.flags & F_SWITCH) {
            if constexpr (K == KIND_DOT || K == KIND_SEPARABLE)
                TL::template switch_sep<true>(a, Wt, S, a.l0 + a.k);
            else
                sw_adj(a, Wt, reinterpret_cast<R *>(S), a.l0 + a.k);
        }
        if (a.k > i0) {
            geo_col(a, G + ((a.k - 1) & 1) * np, a.l0 + a.k - 1, a.k - 1);
            __syncthreads();
            parts_out(a, G + ((a.k - 1) & 1) * np, PT, a.l0 + a.k - 1);
            __syncthreads();
        }
        for (int i = a.k - 1; i >= i0; --i) {
            const int l = a.l0 + i;
            const bool sp = sp1 && l == 1;
            Geo *Gi = G + (i & 1) * np, *Gn = G + (~i & 1) * np;
            if (LB && sp)
                col_adj_a<LB>(a, Wt, S, Gi, PT, i);
            else
                col_adj_a<false>(a, Wt, S, Gi, PT, i);
            parts_in_adj(a, Gi, PT, l);
            if (i > i0) geo_col(a, Gn, l - 1, i - 1, 4 * np);
            __syncthreads();
            if (LB && sp)
                col_adj_b<LB>(a, Wt, S, Gi, PT, i);
            else
                col_adj_b<false>(a, Wt, S, Gi, PT, i);
            if (i > i0) parts_out(a, Gn, PT, l - 1);
            __syncthreads();
        }
        if (skip0) {   // g of a leaf: the four outputs of its block (level 1) at the leaf's node
            const int k = a.k, n = 1 << (D * k), nblk = n >> D, L = a.L;
            for (int it = threadIdx.x; it < np; it += blockDim.x) {
                const int c = it & (NC - 1), b = (it >> D) & (nblk - 1), tau = it >> (D * k);
                uint32_t Ap, Bstar;
                TL::tile_of(a, tau, Ap, Bstar);
                int cb[DMAX];
                morton_decode<D>((Bstar << (D * k)) + (it & (n - 1)), L, cb);
                const C *w = Wt + (tau * n + (b << D)) * RR + ((c & 1) ? MID : END) + ((c >> 1) ? MID : END) * Q;
                C acc = w[0];
#pragma unroll
                for (int al = 1; al < NC; ++al) acc = madd(acc, w[al * RR]);
                a.gadj[(int64_t)rhs * a.npts + ((int64_t)cb[0] << L) + cb[1]] = acc;
            }
        } else if (a.flags & F_INIT) {
            TL::init_adj(a, Wt, rhs);
        } else {
            TL::store_contig(a, Wt, rhs);
        }
    }

    static __device__ __forceinline__ void row_pass_adj(const KArgs<P> &a, unsigned char *smem)
    {
        const int np = npr(a), rhs = blockIdx.y, nb = np >> D;
        C *Wt = reinterpret_cast<C *>(smem), *S = Wt + np * RR, *X = S + 2 * np * RR;
        GeoR *G = reinterpret_cast<GeoR *>(smem + arrays(np, 3 + NC));
        typename PH::T *TC = reinterpret_cast<typename PH::T *>(G + a.k * nb);
        auto tc = [&](int i) { return TC + a.T * (((1 << (D * i)) - 1) / 3) * RR; };   // nodes of level l0 + i
        const bool skip = LB && (a.corner & CORNER_TGT) && (a.flags & F_FINAL);
        const int lsp = LB && (a.corner & CORNER_TGT) ? a.L - 2 : -1;
        const int k1 = skip ? a.k - 1 : a.k;
        if (skip) {
            const int k = a.k, n = 1 << (D * k), nblk = n >> D, L = a.L;
            if (k == 1) {   // no level of this pass follows: the switch may read every node
                for (int j = threadIdx.x; j < np * RR; j += blockDim.x) Wt[j] = czero<C>();
                __syncthreads();
            }
            for (int it = threadIdx.x; it < np; it += blockDim.x) {
                const int al = it & (NC - 1), ra = (it >> D) & (nblk - 1), tau = it >> (D * k);
                uint32_t Ap, Bstar;
                TL::tile_of(a, tau, Ap, Bstar);
                int ca[DMAX];
                morton_decode<D>((((Ap << (D * (k - 1))) + digit_rev<D>(ra, k - 1)) << D) + al, L, ca);
                const C v = a.fadj[(int64_t)rhs * a.npts + ((int64_t)ca[0] << L) + ca[1]];
                C *w = Wt + (tau * n + ra) * RR + ((al & 1) ? MID : END) + ((al >> 1) ? MID : END) * Q;
#pragma unroll
                for (int c = 0; c < NC; ++c) w[(c * nblk) * RR] = v;
            }
        } else if (a.flags & F_FINAL) {
            TL::final_adj(a, Wt, rhs);
        } else {
            TL::load_strided(a, Wt, rhs);
        }
        for (int i = 0; i < k1; ++i) {
            geo_row(a, G + i * nb, a.l0 + i, i);
            node_cache(a, tc(i), a.l0 + i, i, np >> D);
        }
        __syncthreads();
        for (int i = k1 - 1; i >= 0; --i) {
            const int l = a.l0 + i;
            const GeoR *Gi = G + i * nb;
            if (LB && l == lsp) {
                row_adj_e<LB>(a, Wt, X, Gi, nullptr, l, i);
                __syncthreads();
                row_adj_a<LB>(a, X, S);
                __syncthreads();
                row_adj_b<LB>(a, Wt, S, Gi, i);
            } else {
                row_adj_e<false>(a, Wt, X, Gi, i + 1 < k1 ? tc(i + 1) : nullptr, l, i);
                __syncthreads();
                row_adj_a<false>(a, X, S);
                __syncthreads();
                row_adj_b<false>(a, Wt, S, Gi, i);
            }
            __syncthreads();
            row_p<PM_COMPUTE, true>(a, Wt, Gi, tc(i), l, i, FT{nullptr, 0});
            __syncthreads();
        }
        TL::store_contig(a, Wt, rhs);
    }

    // ---- shared memory of a CTA (bytes): W, twice that as stage scratch, then for a column
    // pass the geometry (two levels, and the switch's) and the parts, for a row pass the blocks'
    // geometry and the node features (two levels)
    static __host__ __device__ size_t col_smem(int np, bool tab)
    {
        return arrays(np, 3) + (size_t)np * ((tab ? 0 : PSTR * sizeof(R)) + 2 * sizeof(Geo) + sizeof(int4));
    }
    static __host__ __device__ size_t row_smem(int np, int T, int k, bool tab)
    {
        const size_t big = k > 0 ? (size_t)T << (D * (k - 1)) : 0, small = k > 1 ? (size_t)T << (D * (k - 2)) : 0;
        return arrays(np, 3) + (tab ? 0 : (big + small) * RR * sizeof(typename PH::T)) +
               2 * (size_t)(np >> D) * sizeof(GeoR);
    }

    template <int PM>
    static __device__ __forceinline__ void col_pass(const KArgs<P> &a, unsigned char *smem, R *tb)
    {
        const int np = npr(a), rhs = blockIdx.y;
        C *Wt = reinterpret_cast<C *>(smem), *S = Wt + np * RR;
        Geo *G = reinterpret_cast<Geo *>(smem + arrays(np, 3));
        int4 *GS = reinterpret_cast<int4 *>(G + 2 * np);
        R *PT = reinterpret_cast<R *>(GS + np);
        const int nlev = (int)level_floats(a);
        bool skip0 = false, sp1 = false;   // level 0 done by the first step; level 1 from four nodes
        if constexpr (LB) {
            skip0 = (a.corner & CORNER_SRC) && (a.flags & F_INIT);
            sp1 = a.corner & CORNER_SRC;
        }
        const int i0 = skip0 ? 1 : 0;
        if (PM != PM_COMPUTE && skip0) tb += nlev;
        if constexpr (PM == PM_TABLE)
            if (i0 < a.k) TL::prefetch_l2(tb, nlev);
        if (i0 < a.k) {
            if constexpr (PM == PM_TABLE)
                geo_col(a, G + (i0 & 1) * np, a.l0 + i0, i0);
            else
                parts_first(a, G + (i0 & 1) * np, PT, a.l0 + i0, i0, sp1 && a.l0 + i0 == 1);
        }
        if (skip0)
            init_corner(a, Wt, rhs);
        else if (a.flags & F_INIT)
            TL::init(a, Wt, rhs);
        else
            TL::load(a, Wt, rhs);
        if (i0 >= a.k && (a.flags & F_SWITCH)) geo_switch(a, GS, a.l0 + a.k);
        __syncthreads();
        for (int i = i0; i < a.k; ++i) {
            const int l = a.l0 + i;
            Geo *Gi = G + (i & 1) * np, *Gn = G + (~i & 1) * np;
            const FT fa{tb, np * 2 * Q}, fb{tb + (int64_t)np * 4 * RR, np * Q};
            if constexpr (PM != PM_COMPUTE) tb += nlev;
            if constexpr (PM == PM_TABLE) {   // the next level's blocks (or the switch's) while this level runs
                if (i + 1 < a.k)
                    TL::prefetch_l2(tb, nlev);
                else if (a.flags & F_SWITCH)
                    TL::prefetch_l2(tb, a.ftab_cta - (int64_t)a.k * nlev);
            }
            const bool sp = sp1 && l == 1;
            if (LB && sp)
                col_a<PM, LB>(a, Wt, S, Gi, PT, i, fa);
            else
                col_a<PM, false>(a, Wt, S, Gi, PT, i, fa);
            if constexpr (PM != PM_TABLE) parts_out(a, Gi, PT, l);
            if (i + 1 < a.k) geo_col(a, Gn, l + 1, i + 1, 2 * np);
            __syncthreads();
            if (LB && sp)
                col_b<PM, LB>(a, Wt, S, Gi, PT, i, fb);
            else
                col_b<PM, false>(a, Wt, S, Gi, PT, i, fb);
            if (i + 1 < a.k) {
                if constexpr (PM != PM_TABLE) parts_in(a, Gn, PT, l + 1, sp1 && l == 0);
            } else if (a.flags & F_SWITCH) {
                geo_switch(a, GS, l + 1);
            }
            __syncthreads();
        }
        if (a.flags & F_SWITCH) {
            if constexpr (K == KIND_DOT || K == KIND_SEPARABLE) {
                TL::template switch_sep<false>(a, Wt, S, a.l0 + a.k);
            } else {
                sw<PM>(a, Wt, S, GS, a.l0 + a.k, FT{tb, np * RR});
                __syncthreads();
                TL::store(a, S, rhs);
                return;
            }
        }
        TL::store(a, Wt, rhs);
    }

    template <int PM>
    static __device__ __forceinline__ void row_pass(const KArgs<P> &a, unsigned char *smem, R *tb)
    {
        const int np = npr(a), rhs = blockIdx.y;
        C *Wt = reinterpret_cast<C *>(smem), *S = Wt + np * RR;
        GeoR *G = reinterpret_cast<GeoR *>(smem + arrays(np, 3));
        const int big = a.k > 0 ? a.T << (D * (a.k - 1)) : 0;
        typename PH::T *T0 = reinterpret_cast<typename PH::T *>(G + 2 * (np >> D)), *T1 = T0 + big * RR;
        // level i's nodes: the larger buffer for the last level, alternating before it
        auto tc = [&](int i) { return ((a.k - 1 - i) & 1) ? T1 : T0; };
        const int nlev = (int)level_floats(a);
        // the last level is done by the last step; the one before it has four output nodes
        const bool skip = LB && (a.corner & CORNER_TGT) && (a.flags & F_FINAL);
        const int lsp = LB && (a.corner & CORNER_TGT) ? a.L - 2 : -1;
        const int k1 = skip ? a.k - 1 : a.k;
        if constexpr (PM == PM_TABLE)
            if (k1 > 0) TL::prefetch_l2(tb, nlev);
        TL::load(a, Wt, rhs);
        if (k1 > 0) {
            geo_row(a, G, a.l0, 0);
            if constexpr (PM != PM_TABLE) node_cache(a, tc(0), a.l0, 0, np >> D);
        }
        __syncthreads();
        for (int i = 0; i < k1; ++i) {
            const int l = a.l0 + i;
            GeoR *Gi = G + (i & 1) * (np >> D), *Gn = G + (~i & 1) * (np >> D);
            const FT fa{tb, (np >> D) * RR}, fb{tb + (int64_t)np * RR, np * Q};
            if constexpr (PM != PM_COMPUTE) tb += nlev;
            if constexpr (PM == PM_TABLE)   // the next level's blocks while this level runs
                if (i + 1 < k1) TL::prefetch_l2(tb, nlev);
            row_p<PM>(a, Wt, Gi, tc(i), l, i, fa);
            if (PM != PM_TABLE && i + 1 < a.k && l != lsp) node_cache(a, tc(i + 1), l + 1, i + 1);
            __syncthreads();
            if (LB && l == lsp)
                row_a<LB>(a, Wt, S, Gi, i);
            else
                row_a<false>(a, Wt, S, Gi, i);
            if (i + 1 < k1) geo_row(a, Gn, l + 1, i + 1);
            __syncthreads();
            if (LB && l == lsp)   // few nodes: their features are computed where they are used
                row_b<PM, LB>(a, Wt, S, Gi, nullptr, l, i, fb);
            else
                row_b<PM, false>(a, Wt, S, Gi, i + 1 < a.k ? tc(i + 1) : nullptr, l, i, fb);
            __syncthreads();
        }
        if (skip)
            final_corner(a, Wt, rhs);
        else if (a.flags & F_FINAL)
            TL::final_eval(a, Wt, rhs);
        else
            TL::store(a, Wt, rhs);
    }
};

}  // namespace bfk
