// Phase factors of the mixed precision, two at a time.
//
// sm_100 and later issue FP32 add, multiply and fused multiply-add on a pair of
// registers as one instruction (add/sub/mul/fma .f32x2).  The double-float
// evaluation of Phi and the sincos polynomial are long chains of such operations,
// so two independent phases (two lanes of a float2) take about the issue slots of
// one.  Every lane performs the operations of the scalar code in bf_device.cuh; where
// a caller sums the per-coordinate parts in another order than the scalar code, the
// two agree to FP32 rounding.
// Included by bf_device.cuh after the scalar phase code it builds on.
#pragma once

namespace bfk {

__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    float2 r;
    asm("{ .reg .b64 u, v, d; mov.b64 u, {%2, %3}; mov.b64 v, {%4, %5}; sub.rn.f32x2 d, u, v; mov.b64 {%0, %1}, d; }"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

struct df2 {
    float2 hi, lo;
};

__device__ __forceinline__ df2 two_sum2(float2 a, float2 b)
{
    const float2 s = add2(a, b);
    const float2 bb = sub2(s, a);
    return {s, add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}

__device__ __forceinline__ df2 fast_two_sum2(float2 a, float2 b)
{
    const float2 s = add2(a, b);
    return {s, sub2(b, sub2(s, a))};
}

__device__ __forceinline__ df2 df_mul_u2(const df2 &x, const df2 &y)
{
    const float2 p = mul2(x.hi, y.hi);
    float2 e = fma2(x.hi, y.hi, neg2(p));
    e = fma2(x.hi, y.lo, e);
    e = fma2(x.lo, y.hi, e);
    return {p, e};
}

__device__ __forceinline__ df2 df_add2(const df2 &x, const df2 &y)
{
    const df2 s = two_sum2(x.hi, y.hi);
    return fast_two_sum2(s.hi, add2(s.lo, add2(x.lo, y.lo)));
}

__device__ __forceinline__ float2 fround2(float2 x)
{
    const float2 M = dup2(12582912.0f);
    return sub2(add2(x, M), M);
}

// sqrt_frac of bf_device.cuh on both lanes
__device__ __forceinline__ float2 sqrt_frac2(float2 h, float2 l, float2 sg)
{
    const float2 M = dup2(12582912.0f);
    const float2 q = add2(h, l);
    const float2 r = mul2(sg, make_float2(rsqrt_approx(q.x), rsqrt_approx(q.y)));
    const float2 s = mul2(q, r);
    const float2 w = sub2(s, sub2(add2(s, M), M));
    const float2 res = add2(fma2(neg2(s), s, h), l);
    return fma2(dup2(0.5f), mul2(res, r), w);
}

__device__ __forceinline__ float2 df_frac2(const df2 &x) { return add2(sub2(x.hi, fround2(x.hi)), x.lo); }

__device__ __forceinline__ float2 df_mul_frac2(const df2 &x, const df2 &y)
{
    const float2 M = dup2(12582912.0f);
    const float2 n = sub2(fma2(x.hi, y.hi, M), M);
    const float2 f = fma2(x.hi, y.hi, neg2(n));
    return fma2(x.hi, y.lo, fma2(x.lo, y.hi, f));
}

// quad_reduce and quad_sincos of bf_device.cuh on both lanes
template <bool TWO>
__device__ __forceinline__ void quad_reduce2(float2 a, float2 b, float2 &r, int &j0, int &j1)
{
    const float2 M = dup2(12582912.0f);
    const float2 t = fma2(dup2(4.0f), TWO ? add2(a, b) : a, M);
    j0 = __float_as_int(t.x);
    j1 = __float_as_int(t.y);
    r = fma2(dup2(-0.25f), sub2(t, M), a);
    if (TWO) r = add2(r, b);
}
__device__ __forceinline__ void quad_sincos2(float2 r, int q0, int q1, float2 &s, float2 &c)
{
    const float2 u = mul2(r, r);
    float2 ps = fma2(u, dup2(SC_S3), dup2(SC_S2));
    ps = fma2(u, ps, dup2(SC_S1));
    ps = fma2(u, ps, dup2(SC_S0));
    const float2 sn = mul2(r, ps);
    float2 pc = fma2(u, dup2(SC_C3), dup2(SC_C2));
    pc = fma2(u, pc, dup2(SC_C1));
    const float2 cs = fma2(u, pc, dup2(1.0f));
    const float s0 = (q0 & 1) ? cs.x : sn.x, c0 = (q0 & 1) ? sn.x : cs.x;
    const float s1 = (q1 & 1) ? cs.y : sn.y, c1 = (q1 & 1) ? sn.y : cs.y;
    s.x = __int_as_float(__float_as_int(s0) ^ ((q0 & 2) << 30));
    s.y = __int_as_float(__float_as_int(s1) ^ ((q1 & 2) << 30));
    c.x = __int_as_float(__float_as_int(c0) ^ (((q0 + 1) & 2) << 30));
    c.y = __int_as_float(__float_as_int(c1) ^ (((q1 + 1) & 2) << 30));
}

// Ph<PMIXT> on two lanes: targets and sources are per lane (a shared one is duplicated)
template <class P, int D, int K> struct Ph2;

template <bool F, bool W, int D, int K>
struct Ph2<PMIXT<F, W>, D, K> {
    using PH = Ph<PMIXT<F, W>, D, K>;
    using V = float2;   // two lanes
    static __device__ __forceinline__ V dup(float a) { return dup2(a); }
    struct T { df2 x[D]; df2 A[D]; };
    struct Part { float2 f, h, l, g; };

    static __device__ __forceinline__ df2 pack(const df &a, const df &b) { return {make_float2(a.hi, b.hi), make_float2(a.lo, b.lo)}; }

    static __device__ __forceinline__ T dup(const typename PH::T &a) { return pair(a, a); }
    static __device__ __forceinline__ Part dup(const typename PH::Part &p)
    {
        return Part{dup2(p.f), dup2(p.h), dup2(p.l), dup2(p.g)};
    }
    static __device__ __forceinline__ typename PH::Part lane0(const Part &p)
    {
        return typename PH::Part{p.f.x, p.h.x, p.l.x, p.g.x};
    }

    // the target of lane 0
    static __device__ __forceinline__ typename PH::T one(const T &t)
    {
        typename PH::T o;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            o.x[k] = {t.x[k].hi.x, t.x[k].lo.x};
            o.A[k] = {t.A[k].hi.x, t.A[k].lo.x};
        }
        return o;
    }

    static __device__ __forceinline__ typename PH::Part lane1(const Part &p)
    {
        return typename PH::Part{p.f.y, p.h.y, p.l.y, p.g.y};
    }
    static __device__ __forceinline__ Part swap(const Part &p)
    {
        return Part{make_float2(p.f.y, p.f.x), make_float2(p.h.y, p.h.x), make_float2(p.l.y, p.l.x), make_float2(p.g.y, p.g.x)};
    }

    static __device__ __forceinline__ T pair(const typename PH::T &a, const typename PH::T &b)
    {
        T t;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            t.x[k] = pack(a.x[k], b.x[k]);
            t.A[k] = pack(a.A[k], b.A[k]);
        }
        return t;
    }

    // contribution of source coordinate k: entries e0 (lane 0) and e1 (lane 1)
    static __device__ __forceinline__ Part part(const KArgs<PMIXT<F, W>> &a, const T &t, const MixSE &e0, const MixSE &e1, int k)
    {
        return part_of(a, t.x[k], t.A[k], e0, e1, k == 0);
    }
    static __device__ __forceinline__ Part part_of(const KArgs<PMIXT<F, W>> &a, const df2 &x, const df2 &A, const MixSE &e0,
                                                   const MixSE &e1, bool first)
    {
        Part p{dup2(0.0f), dup2(0.0f), dup2(0.0f), dup2(0.0f)};
        const df2 y = {make_float2(e0.a.x, e1.a.x), make_float2(e0.a.y, e1.a.y)};
        const df2 y2 = {make_float2(e0.a.z, e1.a.z), make_float2(e0.a.w, e1.a.w)};
        if constexpr (K == KIND_DOT || K == KIND_GENRADON) p.f = df_mul_frac2(x, y);
        if constexpr (K == KIND_SEPARABLE) p.f = df_frac2(df_add2(x, y));
        if constexpr (PH::HAS_Q) {
            const df2 v = df_mul_u2(A, y2);
            p.h = sub2(add2(v.hi, dup2(a.sc.mg)), dup2(a.sc.mg));
            p.l = add2(sub2(v.hi, p.h), v.lo);
            p.l = add2(p.l, dup2(first ? 1e-30f : 0.0f));
        }
        return p;
    }
    static __device__ __forceinline__ Part add(const Part &u, const Part &v)
    {
        Part p{dup2(0.0f), dup2(0.0f), dup2(0.0f), dup2(0.0f)};
        if constexpr (PH::PAIR_F) {
            p.f = u.f;
            p.g = v.f;
        } else if constexpr (PH::HAS_F) {
            p.f = add2(u.f, v.f);
        }
        if constexpr (PH::HAS_Q) {
            p.h = add2(u.h, v.h);
            p.l = add2(u.l, v.l);
            if constexpr (W) p.l = add2(p.l, two_sum2(u.h, v.h).lo);
        }
        return p;
    }
    static __device__ __forceinline__ float2 sign(const KArgs<PMIXT<F, W>> &a, const T &t)
    {
        if constexpr (K == KIND_HYPRADON)
            return make_float2(copysignf(1.0f, t.x[0].hi.x), copysignf(1.0f, t.x[0].hi.y));
        else
            return dup2(a.sc.sgn);
    }
    static __device__ __forceinline__ void fin2(float2 sg, const Part &p, float2 &ra, float2 &rb)
    {
        ra = rb = dup2(0.0f);
        if constexpr (PH::HAS_F) ra = p.f;
        if constexpr (PH::PAIR_F) rb = p.g;
        if constexpr (PH::HAS_Q) (PH::HAS_F ? rb : ra) = sqrt_frac2(p.h, p.l, sg);
    }
    static __device__ __forceinline__ float2 fin(float2 sg, const Part &p)
    {
        float2 ra, rb;
        fin2(sg, p, ra, rb);
        return add2(ra, rb);
    }
};

// FP64: the same interface on pairs of doubles (two scalar evaluations; nothing is paired in
// the hardware), so that the d = 2 tile code serves both precisions
template <int D, int K>
struct Ph2<PF64, D, K> {
    using PH = Ph<PF64, D, K>;
    using V = double2;
    struct T { V x[D]; V A[D]; };
    struct Part { V f, q; };
    static __device__ __forceinline__ V pack(double a, double b) { return make_double2(a, b); }
    static __device__ __forceinline__ V dup(double a) { return make_double2(a, a); }
    static __device__ __forceinline__ T dup(const typename PH::T &a)
    {
        T t;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            t.x[k] = dup(a.x[k]);
            t.A[k] = dup(a.A[k]);
        }
        return t;
    }
    static __device__ __forceinline__ Part dup(const typename PH::Part &p) { return Part{dup(p.f), dup(p.q)}; }
    static __device__ __forceinline__ typename PH::Part lane0(const Part &p) { return typename PH::Part{p.f.x, p.q.x}; }
    static __device__ __forceinline__ typename PH::Part lane1(const Part &p) { return typename PH::Part{p.f.y, p.q.y}; }
    static __device__ __forceinline__ Part swap(const Part &p) { return Part{make_double2(p.f.y, p.f.x), make_double2(p.q.y, p.q.x)}; }
    static __device__ __forceinline__ typename PH::T one(const T &t)
    {
        typename PH::T o;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            o.x[k] = t.x[k].x;
            o.A[k] = t.A[k].x;
        }
        return o;
    }
    static __device__ __forceinline__ Part part_of(const KArgs<PF64> &a, const V &x, const V &A, const PF64::SE &e0,
                                                   const PF64::SE &e1, bool first)
    {
        const typename PH::Part p0 = PH::part_of(a, x.x, A.x, e0, first), p1 = PH::part_of(a, x.y, A.y, e1, first);
        return Part{make_double2(p0.f, p1.f), make_double2(p0.q, p1.q)};
    }
    static __device__ __forceinline__ Part part(const KArgs<PF64> &a, const T &t, const PF64::SE &e0, const PF64::SE &e1, int k)
    {
        return part_of(a, t.x[k], t.A[k], e0, e1, k == 0);
    }
    static __device__ __forceinline__ Part add(const Part &u, const Part &v)
    {
        Part p{};
        if constexpr (PH::HAS_F) p.f = make_double2(u.f.x + v.f.x, u.f.y + v.f.y);
        if constexpr (PH::HAS_Q) p.q = make_double2(u.q.x + v.q.x, u.q.y + v.q.y);
        return p;
    }
};

// e^{2 pi i Phi} on two lanes from the summed parts: lane 0 -> e0, lane 1 -> e1
template <class P, int D, int K>
__device__ __forceinline__ void expphase_part2(const KArgs<P> &a, const typename Ph2<P, D, K>::T &t,
                                               const typename Ph2<P, D, K>::Part &pt, float2 &e0, float2 &e1)
{
    using PH2 = Ph2<P, D, K>;
    float2 s, c;
    if constexpr (P::sfu) {
        const float2 fr = PH2::fin(PH2::sign(a, t), pt);
        sincos2pi_sfu(fr.x, s.x, c.x);
        sincos2pi_sfu(fr.y, s.y, c.y);
    } else {
        float2 ra, rb, r;
        int j0, j1;
        PH2::fin2(PH2::sign(a, t), pt, ra, rb);
        quad_reduce2<PH2::PH::TWO>(ra, rb, r, j0, j1);
        quad_sincos2(r, j0, j1, s, c);
    }
    e0 = make_float2(c.x, s.x);
    e1 = make_float2(c.y, s.y);
}

}  // namespace bfk
