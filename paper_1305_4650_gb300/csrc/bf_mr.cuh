// Multi-RHS forward passes for d = 2 (the batched right-hand sides of Section 1:
// one operator, several source vectors g).
//
// The phase factors of every step depend only on the geometry, not on g, so a CTA
// keeps up to MRMAX right-hand sides of its tiles in shared memory and splits each
// merge stage in two: all threads first evaluate the stage's phase factors once
// into a shared-memory cache, then apply them to every right-hand side.  The two
// interpolation stages of a merge exchange partial results through scratch; they
// run over the right-hand sides in chunks of rc, so the scratch holds rc of them.
// The switch keeps one accumulator per right-hand side in registers and evaluates
// each entry of the r x r phase matrix once.
//
// Shared memory (complex numbers, npr = pairs of the CTA):
//   W  [nr][npr][r]       weights of every right-hand side (in place, as in Tile)
//   S  [rc][2 npr r + ..] stage scratch (row scratch units padded, mr_pad)
//   PC [5 r npr + ..]     phase cache of the current stage (strides padded, mr_pad)
// Stages and accumulations are those of Tile2 (bf_tile2.cuh), in another order where lanes run over
// pairs or two outputs share an item.
//
// Phase tables (the precompute trade-off of Section 1.4).  A plan may keep every phase
// factor of its apply in device memory: PM_BUILD runs the phase stages only and writes
// each stage's cache (and the switch matrices) to the table, in the order PM_TABLE reads
// them back; PM_TABLE copies them into the cache instead of evaluating Phi, which turns
// the instruction-bound apply into a stream over the table.  The values are those the
// computing kernels (PM_COMPUTE) would produce, so the results are identical.
#pragma once

#include "bf_device.cuh"

namespace bfk {

constexpr int MRMAX = 16;   // right-hand sides held by one CTA

// ---- bulk copies (TMA engine) into shared memory, completed on an mbarrier
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// tiled bulk copy (TMA) of the 2-D box at element coordinates (x, y) of the tensor that
// `map` describes (a CUtensorMap in global memory) into shared memory, completed on bar;
// the box's rows land contiguously (x times the element size must be a multiple of 16 bytes)
__device__ __forceinline__ void bulk_tensor_2d_g2s(void *dst, const void *map, int x, int y, uint64_t *bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok)
                 : "r"(smem_u32(bar)), "r"(parity)
                 : "memory");
    return ok != 0;
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// wait for phase `parity` of an mbarrier; false after `limit` polls (the caller flags the error)
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity, int limit)
{
    for (int i = 0; i < limit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

constexpr int TS_MAXB = 16;          // table blocks per CTA and pass
constexpr int TS_POLLS = 1 << 16;    // polls of one wait before it is flagged

// Phase-table stream of a CTA (PM_TABLE): block j of the pass's table arrives in buffer
// j & 1 by one bulk copy, issued two blocks ahead of its use.
struct TabCtl {
    uint64_t bar[2];
    int64_t off[TS_MAXB + 1];   // block j of a tile group = complex numbers [off[j], off[j+1]) of its table
    int nblk;                   // blocks per tile group
    int total;                  // blocks of all the CTA's tile groups
};

template <class C>
struct TS {
    C *tb;          // PM_BUILD: write cursor; PM_TABLE: the pass's table in global memory
    C *buf[2];      // PM_TABLE: shared-memory buffers
    TabCtl *ctl;
    int j;          // PM_TABLE: next block to use
    int *err;       // set when a wait gives up
    int c0, cstep;  // PM_TABLE: the CTA's tile groups are c0, c0 + cstep, ...
    int64_t cstride;   // table complex numbers per tile group
};

// pairs per switch round and threads per CTA: the switch runs one thread per (pair, s)
template <int Q>
struct CfgMR {
    static constexpr int RR = Q * Q;
    static constexpr int PPR = RR <= 32 ? 16 : (RR <= 64 ? 8 : 4);
    static constexpr int NT = PPR * RR;
};
// CTAs per SM the register budget is cut for (FP64: one, its pipe needs few warps)
template <int Q, class P>
struct MinbMR {
    static constexpr int v = Q * Q <= 32 && !P::is_f64 ? 2 : 1;
};

// Padding (in complex numbers) of the shared-memory arrays read and written by the apply
// stages, so that the 64-bit accesses of a warp fall in distinct banks (32 banks of 4
// bytes), chosen per q by counting the wavefronts of every access pattern of the stages
// (TileMR::spread, gather) for 16 pairs; the phase-table layout stays compact.  Wavefronts
// without and with them: q = 3 1242 and 720, q = 4 5120 and 3264, q = 6 6360 and 4956,
// q = 8 33792 and 20736.
struct MRPad {
    int ca;   // column modulation: per (pair, chi) block of 2 r factors
    int cb;   // column demodulation: per pair (r factors)
    int rb;   // row post-modulation: per pair (4 r factors)
    int rs;   // row scratch: per (pair, t_1) unit of 2 q partial sums
};
__host__ __device__ constexpr MRPad mr_pad(int q)
{
    return q == 5   ? MRPad{7, 12, 1, 1}
           : q & 1  ? MRPad{1, 0, 1, 1}
           : q == 4 ? MRPad{1, 4, 8, 1}
           : q == 6 ? MRPad{1, 2, 8, 1}
           : q == 8 ? MRPad{1, 8, 8, 1}
                    : MRPad{1, 2, 2, 1};
}
// phase-cache entries per pair beyond 5 r (evaluating passes)
__host__ __device__ constexpr int mr_pc_extra(int q)
{
    return 2 * mr_pad(q).ca + mr_pad(q).cb > mr_pad(q).rb ? 2 * mr_pad(q).ca + mr_pad(q).cb : mr_pad(q).rb;
}
// scratch entries per right-hand side (2 r per pair, plus the padding: of the units of gather,
// or one entry per half of spread)
__host__ __device__ constexpr int64_t mr_s_stride(int q, int64_t npr)
{
    const int64_t pad = npr * q * mr_pad(q).rs;
    return 2 * npr * q * q + (pad > 2 ? pad : 2);
}
// complex numbers of the scratch S: rc right-hand sides, and at least the parts of a level
// (6 rows of up to three components of q, padded to even, and a sign per pair), which the
// phase stage keeps there
__host__ __device__ constexpr int64_t mr_s_size(int q, int64_t npr, int64_t rc)
{
    const int64_t st = rc * mr_s_stride(q, npr), pt = (npr * (18 * ((q + 1) & ~1) + 1) + 1) / 2;
    return ((st > pt ? st : pt) + 1) & ~(int64_t)1;
}

// LB: Lobatto nodes of odd q (unit columns of M, KArgs::corner; bf_tile2.cuh)
template <int Q, class P, int K, bool LB>
struct TileMR {
    static constexpr MRPad PAD = mr_pad(Q);
    static constexpr int D = 2, NC = 4, RR = Q * Q, NT = CfgMR<Q>::NT;
    using R = typename P::R;
    using C = typename P::C;
    using PH = Ph<P, 2, K>;
    using PH2 = Ph2<P, 2, K>;
    using TL = Tile<2, Q, P, K>;
    using T2 = Tile2<Q, P, K, LB>;
    static constexpr int MID = T2::MID, END = T2::END;
    // lane order of spread and gather: over the nodes first for even q, whose weights of a pair
    // (q^2 complex numbers) start in the same bank for every pair or every second one; over the
    // pairs first for odd q
    static constexpr bool NF = Q % 2 == 0;

    // geometry of one merge block of a row level (in S during the phase stage): the parent
    // target box (level l) and the parent source box (level l+1)
    struct __align__(16) GeoR {
        int ca[2];    // coordinates of the parent target box A_p
        int cbq[2];   // coordinates of the parent source box B_q
    };

    struct Ctx {
        int tile0;   // first tile of the CTA
        int rhs0;    // first right-hand side
        int nr;      // right-hand sides held (1..MRMAX)
        int npr;     // pairs held: T 2^{2k}
        int rc;      // right-hand sides per scratch chunk
        int lgp;     // log2(npr)
    };

    static __device__ __forceinline__ void tile_of(const KArgs<P> &a, const Ctx &x, int tau, uint32_t &Ap,
                                                   uint32_t &Bstar)
    {
        const uint32_t tile = (uint32_t)x.tile0 + (uint32_t)tau;
        const int sh = D * (a.L - a.l0 - a.k);
        Ap = tile >> sh;
        Bstar = tile & ((1u << sh) - 1u);
    }

    // the pass's first step also does level 0, its last step level L - 1 (KArgs::corner)
    static __device__ __forceinline__ bool skip_first(const KArgs<P> &a) { return LB && (a.corner & CORNER_SRC) && (a.flags & F_INIT); }
    static __device__ __forceinline__ bool skip_last(const KArgs<P> &a) { return LB && (a.corner & CORNER_TGT) && (a.flags & F_FINAL); }

    static __device__ __forceinline__ int block_base(int beta, int i)
    {
        const int ra = beta & ((1 << (D * i)) - 1);
        return ((beta >> (D * i)) << (D * (i + 1))) + ra;
    }

    // ---- phase-table stream (PM_TABLE)
    static __device__ void ts_issue(TS<C> &ts, int j)
    {
        TabCtl *c = ts.ctl;
        const int g = j / c->nblk, jj = j - g * c->nblk;
        const unsigned bytes = (unsigned)((c->off[jj + 1] - c->off[jj]) * (int64_t)sizeof(C));
        const C *src = ts.tb + (int64_t)(ts.c0 + g * ts.cstep) * ts.cstride + c->off[jj];
        mbar_expect_tx(&c->bar[j & 1], bytes);
        bulk_g2s(ts.buf[j & 1], src, bytes, &c->bar[j & 1]);
    }
    // block list of a tile group (sizes in complex numbers), barriers, the first two copies
    // of the stream over all the CTA's tile groups
    static __device__ void ts_setup(TS<C> &ts, const KArgs<P> &a, const Ctx &x, bool row)
    {
        if (threadIdx.x == 0) {
            TabCtl *c = ts.ctl;
            const int64_t npr = x.npr, r5 = 5 * RR * npr;
            int nb = 0;
            int64_t o = 0;
            auto add = [&](int64_t n) { c->off[nb++] = o; o += n; };
            if (!row) {
                if (skip_first(a))
                    o = RR * npr + r5;   // the blocks of the first step and of level 0 are not used
                else if (a.flags & F_INIT)
                    add(RR * npr);
                for (int i = skip_first(a) ? 1 : 0; i < a.k; ++i) add(r5);
                if ((a.flags & F_SWITCH) && K != KIND_DOT && K != KIND_SEPARABLE)
                    for (int th = 0; th < Q; ++th) add((int64_t)Q * RR * npr);
            } else {
                for (int i = 0; i < (skip_last(a) ? a.k - 1 : a.k); ++i) add(r5);
                if ((a.flags & F_FINAL) && !skip_last(a)) add((RR + 1) * npr);
            }
            c->off[nb] = o;
            c->nblk = nb;
            c->total = nb * ((a.ncta - ts.c0 + ts.cstep - 1) / ts.cstep);
            mbar_init(&c->bar[0], 1);
            mbar_init(&c->bar[1], 1);
            mbar_init_fence();
            for (int j = 0; j < 2 && j < c->total; ++j) ts_issue(ts, j);
        }
        ts.j = 0;
        __syncthreads();
    }
    // wait for the next block; a wait that gives up is flagged and waited for once more,
    // so no copy is left in flight (the results are then undefined, never a hang)
    static __device__ C *ts_acquire(TS<C> &ts)
    {
        const int j = ts.j;
        uint64_t *bar = &ts.ctl->bar[j & 1];
        if (!mbar_wait(bar, (unsigned)((j >> 1) & 1), TS_POLLS)) {
            if (ts.err) atomicExch(ts.err, 1);
            mbar_wait(bar, (unsigned)((j >> 1) & 1), TS_POLLS);
        }
        return ts.buf[j & 1];
    }
    // after the block's last reader (callers sync first): refill its buffer two blocks ahead
    static __device__ void ts_release(TS<C> &ts)
    {
        const int j = ts.j++;
        if (threadIdx.x == 0 && j + 2 < ts.ctl->total) {
            fence_proxy_async();
            ts_issue(ts, j + 2);
        }
    }

    // ---- phase-table store of n complex numbers (PM_BUILD; n even, 16-byte aligned blocks)
    static __device__ __forceinline__ void tab_store(C *dst, const C *src, int n)
    {
        const float4 *s4 = reinterpret_cast<const float4 *>(src);
        float4 *d4 = reinterpret_cast<float4 *>(dst);
        for (int j = threadIdx.x; j < (n >> 1); j += NT) __stcs(d4 + j, s4[j]);
    }

    // ---- CTA input: npr consecutive pairs per right-hand side (sharding mode 2: the pairs of
    // other ranks' source boxes read as zero)
    static __device__ void load(const KArgs<P> &a, const Ctx &x, C *W)
    {
        const int WS = x.npr * RR;
        const int64_t off = (int64_t)x.tile0 * ((int64_t)RR << (D * a.k));
        for (int j = threadIdx.x; j < x.nr * WS; j += NT) {
            const int rb = (j / RR) >> x.lgp, e = j - rb * WS;
            W[j] = a.shard_mode == 2 && !shard_owned<D>(a, (off + e) / RR)
                       ? czero<C>()
                       : __ldcg(a.win + (int64_t)(x.rhs0 + rb) * a.wstride + off + e);
        }
    }

    // ---- the same input by bulk copies (the TMA engine), one per right-hand side (npr r complex
    // numbers, contiguous in HBM and 16-byte aligned), completing on *bar; issued by thread 0
    // after the shared memory's previous generic accesses are ordered before the copies
    static __device__ void load_async(const KArgs<P> &a, const Ctx &x, C *W, uint64_t *bar)
    {
        if (threadIdx.x != 0) return;
        const unsigned bytes = (unsigned)(x.npr * RR * sizeof(C));
        const int64_t off = (int64_t)x.tile0 * ((int64_t)RR << (D * a.k));
        fence_proxy_async();
        mbar_expect_tx(bar, bytes * (unsigned)x.nr);
        for (int rb = 0; rb < x.nr; ++rb)
            bulk_g2s(W + rb * x.npr * RR, a.win + (int64_t)(x.rhs0 + rb) * a.wstride + off, bytes, bar);
    }
    // every thread: wait for those copies; a wait that gives up is flagged and waited for once
    // more, so no copy is left in flight (the results are then undefined, never a hang)
    static __device__ void wait_input(const KArgs<P> &a, uint64_t *bar, unsigned parity)
    {
        if (!mbar_wait(bar, parity, TS_POLLS)) {
            if (a.err) atomicExch(a.err, 1);
            mbar_wait(bar, parity, TS_POLLS);
        }
    }

    // ---- CTA output: tile slots are in digit-reversed order after k merges
    static __device__ void store(const KArgs<P> &a, const Ctx &x, const C *W)
    {
        // destination of each slot's pair, once per CTA (slots are in digit-reversed order)
        __shared__ int64_t poff[64];
        const int k = a.k, n = 1 << (D * k), WS = x.npr * RR;
        const int64_t Sstar = 1LL << (D * (a.L - a.l0 - k));
        for (int pl = threadIdx.x; pl < x.npr; pl += NT) {
            uint32_t Ap, Bstar;
            tile_of(a, x, pl >> (D * k), Ap, Bstar);
            poff[pl] = ((((int64_t)Ap << (D * k)) + digit_rev<D>(pl & (n - 1), k)) * Sstar + Bstar) * RR;
        }
        __syncthreads();
        for (int j = threadIdx.x; j < x.nr * WS; j += NT) {
            const int rb = (j / RR) >> x.lgp, e = j - rb * WS;
            const int pl = e / RR, t = e - pl * RR;
            a.wout[(int64_t)(x.rhs0 + rb) * a.wstride + poff[pl] + t] = W[j];
        }
    }

    // ---- init: PC[pair][t] = l_t(y) e^{-2pi i Phi(x0(X), y_t^B)} e^{2pi i Phi(x0(X), y)}, then W = PC g(y)
    static __device__ void init_factors(const KArgs<P> &a, const Ctx &x, C *PC)
    {
        const int k = a.k, n = 1 << (D * k), L = a.L, WS = x.npr * RR;
        const int cX[DMAX] = {0, 0, 0};
        const int ctr[DMAX] = {Q, Q, Q};
        const typename PH::T tX = tpoint<P, D, Q, K>(a, 0, cX, ctr);
        for (int it = threadIdx.x; it < WS; it += NT) {
            const int t = it % RR, pr = it / RR;
            const int tk[DMAX] = {t % Q, t / Q, 0};
            const R lag = a.lsrc[tk[0]] * a.lsrc[tk[1]];
            C e = czero<C>();
            if (lag != R(0)) {
                uint32_t Ap, Bstar;
                tile_of(a, x, pr >> (D * k), Ap, Bstar);
                int cb[DMAX];
                morton_decode<D>((Bstar << (D * k)) + (pr & (n - 1)), L, cb);
                const int pslot[DMAX] = {Q + 1, Q + 1, Q + 1};
                const C e1 = expphase<P, D, K>(a, tX, spoint<P, D, Q, K>(a, 0, cb, pslot));
                const C e0 = expphase<P, D, K>(a, tX, spoint<P, D, Q, K>(a, 0, cb, tk));
                e = cjmul(e0, e1);
                e.x *= lag;
                e.y *= lag;
            }
            PC[it] = e;
        }
    }
    template <int PM>
    static __device__ void init(const KArgs<P> &a, const Ctx &x, C *W, C *PC, const C *g, TS<C> &ts)
    {
        const int k = a.k, n = 1 << (D * k), L = a.L, WS = x.npr * RR;
        if constexpr (PM == PM_TABLE) PC = ts_acquire(ts);
        else init_factors(a, x, PC);
        __syncthreads();
        if constexpr (PM == PM_BUILD) {   // build: store the factors; no weights are touched
            tab_store(ts.tb, PC, WS);
            ts.tb += WS;
            __syncthreads();
        }
        if constexpr (PM != PM_BUILD) {
            // the grid point of a leaf box has a non-zero Lagrange value at few nodes (one
            // for points at box corners): zero the weights, then fill those nodes only
            __shared__ int nzt[QMAX * QMAX];
            __shared__ int nnz;
            if (threadIdx.x == 0) {
                int m = 0;
                for (int t = 0; t < RR; ++t)
                    if (a.lsrc[t % Q] * a.lsrc[t / Q] != R(0)) nzt[m++] = t;
                nnz = m;
            }
            float4 *w4 = reinterpret_cast<float4 *>(W);
            for (int j = threadIdx.x; j < (x.nr * WS * (int)sizeof(C)) / 16; j += NT) w4[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (sizeof(C) == 8 && (x.nr * WS & 1) && threadIdx.x == 0) W[x.nr * WS - 1] = czero<C>();   // one pair, odd q
            __syncthreads();
            for (int j = threadIdx.x; j < x.nr * x.npr * nnz; j += NT) {
                const int z = j % nnz, pr = (j / nnz) & (x.npr - 1), rb = (j / nnz) >> x.lgp;
                const int it = pr * RR + nzt[z];
                uint32_t Ap, Bstar;
                tile_of(a, x, pr >> (D * k), Ap, Bstar);
                int cb[DMAX];
                morton_decode<D>((Bstar << (D * k)) + (pr & (n - 1)), L, cb);
                const int64_t flat = ((int64_t)cb[0] << L) + cb[1];
                W[rb * WS + it] = cmul(PC[it], g[(int64_t)(x.rhs0 + rb) * a.npts + flat]);
            }
        }
        __syncthreads();
        if constexpr (PM == PM_TABLE) ts_release(ts);
    }

    // ---- first step and first merge, last merge and last step with points at box corners
    // (KArgs::corner; Tile2::init_corner, Tile2::final_corner)
    static __device__ void init_corner(const KArgs<P> &a, const Ctx &x, C *W, const C *g)
    {
        const int k = a.k, n = 1 << (D * k), nblk = n >> D, L = a.L, WS = x.npr * RR;
        if (a.k == 1) {   // no level of this pass follows: the switch may read every node
            for (int j = threadIdx.x; j < x.nr * WS; j += NT) W[j] = czero<C>();
            __syncthreads();
        }
        for (int it = threadIdx.x; it < x.nr * x.npr; it += NT) {
            const int pr = it & (x.npr - 1), rb = it >> x.lgp;
            const int c = pr & (NC - 1), b = (pr >> D) & (nblk - 1), tau = pr >> (D * k);
            uint32_t Ap, Bstar;
            tile_of(a, x, tau, Ap, Bstar);
            int cb[DMAX];
            morton_decode<D>((Bstar << (D * k)) + (pr & (n - 1)), L, cb);
            const C v = g[(int64_t)(x.rhs0 + rb) * a.npts + ((int64_t)cb[0] << L) + cb[1]];
            C *w = W + rb * WS + (tau * n + (b << D)) * RR + ((c & 1) ? MID : END) + ((c >> 1) ? MID : END) * Q;
#pragma unroll
            for (int al = 0; al < NC; ++al) w[al * RR] = v;
        }
        __syncthreads();
    }
    static __device__ void final_corner(const KArgs<P> &a, const Ctx &x, const C *W, C *f)
    {
        const int k = a.k, n = 1 << (D * k), nblk = n >> D, L = a.L, WS = x.npr * RR;
        for (int it = threadIdx.x; it < x.nr * x.npr; it += NT) {
            const int pr = it & (x.npr - 1), rb = it >> x.lgp;
            const int al = pr & (NC - 1), ra = (pr >> D) & (nblk - 1), tau = pr >> (D * k);
            uint32_t Ap, Bstar;
            tile_of(a, x, tau, Ap, Bstar);
            int ca[DMAX];
            morton_decode<D>((((Ap << (D * (k - 1))) + digit_rev<D>(ra, k - 1)) << D) + al, L, ca);
            const C *w = W + rb * WS + (tau * n + ra) * RR + ((al & 1) ? MID : END) + ((al >> 1) ? MID : END) * Q;
            C acc = w[0];
#pragma unroll
            for (int c = 1; c < NC; ++c) acc = madd(acc, w[(c * nblk) * RR]);
            f[(int64_t)(x.rhs0 + rb) * a.npts + ((int64_t)ca[0] << L) + ca[1]] = acc;
        }
    }

    // ---- the factors of a column level (l -> l+1), phase cache
    //   PA [alpha_0][pair alpha / 2][chi] blocks of PCA: [cl][t_1'][t_0']  e^{2 pi i Phi(x0(A_alpha), y_t'^{B_c})}, c = cl | chi << 1
    //   PB [pair alpha] blocks of PCB: [t_1][t_0]             e^{2 pi i Phi(x0(A_alpha), y_t^{B'})}
    // SP: the children's nodes MID and END of both dimensions only (level 1 with KArgs::corner)
    template <int PM> static constexpr int PCA = 2 * RR + (PM == PM_COMPUTE ? PAD.ca : 0);
    template <int PM> static constexpr int PCB = RR + (PM == PM_COMPUTE ? PAD.cb : 0);
    template <int PM> static constexpr int PRB = 4 * RR + (PM == PM_COMPUTE ? PAD.rb : 0);
    template <int PM>
    static __device__ __forceinline__ int pa_at(int npr, int pj, int chi)
    {
        return (pj & 1) * npr * PCA<PM> + ((pj >> 1) * 2 + chi) * PCA<PM>;
    }
    template <int PM, bool SP>
    static __device__ void col_phases(const KArgs<P> &a, const Ctx &x, C *S, C *PC, int l, int i)
    {
        const int k = a.k, n = 1 << (D * k), nblk = n >> D, L = a.L, nout = x.npr;
        C *PA = PC, *PB = PC + nout * 2 * PCA<PM>;
        // the parts of every output pair's nodes, once per level, into S (idle during the phase
        // stage): thread = (pair, coordinate, row of q parts), each with its own geometry
        R *PT = reinterpret_cast<R *>(S), *SG = PT + nout * T2::PSTR;
        for (int j = threadIdx.x; j < nout * 6; j += NT) {
            const int row = j % 3, dim = (j / 3) & 1, pA = j / 6;
            const int alpha = pA & (NC - 1), beta = (pA >> D) & (nblk - 1), tau = pA >> (D * k);
            uint32_t Ap, Bstar, Apg, Bq;
            int base;
            tile_of(a, x, tau, Ap, Bstar);
            TL::block_geo(Ap, Bstar, beta, i, k, Apg, Bq, base);
            const uint32_t Aa = (Apg << D) + alpha;
            int ca[DMAX], cbq[DMAX];
            morton_decode<D>(Aa, l + 1, ca);
            morton_decode<D>(Bq, L - l - 1, cbq);
            const typename PH::T tA = tcenter<P, D, Q, K>(a, l + 1, Aa, ca);
            const int cb = dim ? cbq[1] : cbq[0];
            const typename P::SE *e = a.st[dim] + (row < 2 ? soff<Q>(L, l) + (2 * cb + row) * (Q + 2) : soff<Q>(L, l + 1) + cb * (Q + 2));
            T2::part_row(a, dim ? tA.x[1] : tA.x[0], dim ? tA.A[1] : tA.A[0], dim == 0, e, PT + pA * T2::PSTR + (dim * 3 + row) * T2::PROW,
                         SP && row < 2);
            if (j % 6 == 0) SG[pA] = PH::sign(a, tA);
        }
        __syncthreads();
        // items (pair, g, t_1), q phases each: g < 4 modulations of child c_0 = g & 1, c_1 = g >> 1,
        // g = 4 the demodulation
        for (int it = threadIdx.x; it < nout * 5 * Q; it += NT) {
            const int tq = it % Q, g = (it / Q) % 5, pA = it / (5 * Q);
            const R *pt = PT + pA * T2::PSTR;
            const R *p0 = pt + (g < 4 ? g & 1 : 2) * T2::PROW;
            const typename PH::Part p1 = T2::load1(pt + (3 + (g >> 1)) * T2::PROW + tq);
            C *o = g < 4 ? PA + pa_at<PM>(nout, pA, g >> 1) + (g & 1) * RR + tq * Q : PB + pA * PCB<PM> + tq * Q;
            const R sg = K == KIND_HYPRADON ? SG[pA] : (R)a.sc.sgn;
            if (SP && g < 4) {
                if (tq == MID || tq == END)
                    TL::template ph2<PM_COMPUTE>(PH2::dup(sg), PH2::add(T2::lanes(T2::load1(p0 + MID), T2::load1(p0 + END)), PH2::dup(p1)),
                                                 nullptr, nullptr, o[MID], o[END]);
                continue;
            }
            T2::phase_row(sg, p0, p1, o);
        }
    }

    // ---- the factors of a row level (l -> l+1), phase cache
    //   PA [input pair c][t]                       e^{2 pi i Phi(x_t^{A_p}, y0(B_c))}
    //   PB [output pair alpha] blocks of PRB: [c][s] e^{2 pi i Phi(x_s^{A_alpha}, y0(B_c))}
    // SP: the child target boxes' nodes MID and END only
    template <int PM, bool SP>
    static __device__ void row_phases(const KArgs<P> &a, const Ctx &x, C *S, C *PC, int l, int i)
    {
        const int k = a.k, n = 1 << (D * k), nblk = n >> D, L = a.L, nout = x.npr;
        C *PA = PC, *PB = PC + nout * RR;
        // the blocks' geometry once per level, into S (idle during the phase stage)
        GeoR *GR = reinterpret_cast<GeoR *>(S);
        for (int j = threadIdx.x; j < (nout >> D); j += NT) {
            const int beta = j & (nblk - 1), tau = j >> (D * (k - 1));
            uint32_t Ap, Bstar, Apg, Bq;
            int base;
            tile_of(a, x, tau, Ap, Bstar);
            TL::block_geo(Ap, Bstar, beta, i, k, Apg, Bq, base);
            int ca[DMAX], cbq[DMAX];
            morton_decode<D>(Apg, l, ca);
            morton_decode<D>(Bq, L - l - 1, cbq);
            GR[j] = GeoR{{ca[0], ca[1]}, {cbq[0], cbq[1]}};
        }
        __syncthreads();
        // items (pair, s), the four factors at a child node, then (block, t), the four at a parent node
        constexpr int RP = SP ? 4 : RR;   // child nodes
        for (int it = threadIdx.x; it < nout * RP + (nout >> D) * RR; it += NT) {
            const bool post = it < nout * RP;
            const int jt = post ? it : it - nout * RP, pj = post ? jt / RP : jt / RR;
            const int t = SP && post ? ((jt & 1) ? END : MID) + ((jt & 2) ? END : MID) * Q : (post ? jt % RP : jt % RR);
            const GeoR g = GR[post ? pj >> D : pj];
            const int ca[DMAX] = {post ? 2 * g.ca[0] + (pj & 1) : g.ca[0], post ? 2 * g.ca[1] + ((pj >> 1) & 1) : g.ca[1], 0};
            const int tk[DMAX] = {t % Q, t / Q, 0};
            typename P::SE s0[2], s1[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                s0[h] = sget<P, Q>(a, 0, l, 2 * g.cbq[0] + h, Q);
                s1[h] = sget<P, Q>(a, 1, l, 2 * g.cbq[1] + h, Q);
            }
            C E[NC];
            T2::template four<PM_COMPUTE>(a, tpoint<P, D, Q, K>(a, post ? l + 1 : l, ca, tk), s0, s1, typename T2::FT{nullptr, 0}, 0, 0, E);
            C *o = post ? PB + pj * PRB<PM> + t : PA + pj * NC * RR + t;
#pragma unroll
            for (int c = 0; c < NC; ++c) o[c * RR] = E[c];
        }
    }

    // ---- The two data flows of a level, in place on the tile, in chunks of rc right-hand sides.
    // Factors come from pointer functions; CJ conjugates those of stage A, else those of stage B.
    // An item's digits other than its right-hand side depend on the thread only: every stage
    // has per <= NT items per right-hand side, NT / per of them run side by side, and the item
    // decoding and the pointers are computed once per level instead of once per item.
    //
    // Lanes run over the pairs first at odd q: with q = 5 and the paddings of mr_pad every access of
    // spread then takes the fewest wavefronts its bytes allow, those of gather 1.4 times that at most
    // (counted over the access patterns for 16 pairs; lanes over nodes first took 2.2 and 1.7
    // times, and shared-memory wavefronts are what these stages are bound by).  At even q pairs first
    // would put all lanes of a load of W into one bank (q = 4: 9280 wavefronts against 3264 with
    // lanes over nodes first).
    //
    // spread (column level; adjoint of a row level): out_j(t) = fB(j, t) sum_c sum_u M_c[t][u]
    // fA(j, c, u) in_c(u) for the four outputs j of a block, one dimension per stage.  A stage-A
    // item serves the two outputs j_0 = 0, 1 (SA: distance of their factors), which share the
    // inputs it reads.  SP: inputs at nodes MID and END only.
    template <bool SP, bool CJ, class MS, class FA, class FB>
    static __device__ __forceinline__ void spread(const MS &ms, const Ctx &x, int k, int i, C *W, C *S, int SA, FA fA, FB fB)
    {
        const int n = 1 << (D * k), nblk = n >> D, WS = x.npr * RR, SW = (int)mr_s_stride(Q, x.npr);
        constexpr int QA = SP ? 2 : Q;
        // stage A: items (rb, block and j_1, c_1, u_1): modulate the inputs, contract dimension 0
        const int perA = x.npr * QA, rA = NT / perA, a0 = (int)threadIdx.x % perA, rbA = (int)threadIdx.x / perA;
        const int tp = NF ? a0 % QA : a0 >> x.lgp, chi = NF ? (a0 / QA) & 1 : (a0 >> (x.lgp - 1)) & 1;
        const int pa = NF ? (a0 / (2 * QA)) << 1 : (a0 << 1) & (x.npr - 1), tq = SP ? (tp ? END : MID) : tp;
        const int SH = x.npr * RR + 1;   // scratch of the outputs with j_0 = 1
        const C *winA = W + (((pa >> (D * k)) << (D * k)) + block_base((pa >> D) & (nblk - 1), i) + (chi << (D * i + 1))) * RR + Q * tq;
        const C *phA = fA(pa, chi) + tq * Q;
        C *soA = S + ((pa + chi) * Q + tq) * Q;
        // stage B: items (rb, j, t_0): contract dimension 1 and the child bit c_1
        const int perB = x.npr * Q, rB = NT / perB, b0 = (int)threadIdx.x % perB, rbB = (int)threadIdx.x / perB;
        const int tl = NF ? b0 % Q : b0 >> x.lgp, pj = NF ? b0 / Q : b0 & (x.npr - 1);
        const C *siB = S + (pj & 1) * SH + (pj >> 1) * 2 * RR + tl;
        C *woB = W + (((pj >> (D * k)) << (D * k)) + block_base((pj >> D) & (nblk - 1), i) + ((pj & (NC - 1)) << (D * i))) * RR + tl;
        const C *phB = fB(pj) + tl;
        for (int r0 = 0; r0 < x.nr; r0 += x.rc) {
            const int nrc = min(x.rc, x.nr - r0);
            if (rbA < rA)
                for (int rb = rbA; rb < nrc; rb += rA) {
                    const C *w = winA + (r0 + rb) * WS;
                    C acc[2][Q];
#pragma unroll
                    for (int j = 0; j < Q; ++j) acc[0][j] = acc[1][j] = czero<C>();
#pragma unroll
                    for (int cl = 0; cl < 2; ++cl)
#pragma unroll
                        for (int t0p = 0; t0p < Q; ++t0p) {
                            if (SP && t0p != MID && t0p != END) continue;
                            const C v = w[(cl << (D * i)) * RR + t0p];
#pragma unroll
                            for (int j = 0; j < 2; ++j) {
                                const C e = phA[j * SA + fA.child(cl) + t0p];
                                const C u = CJ ? cjmul(e, v) : cmul(e, v);
#pragma unroll
                                for (int t0 = 0; t0 < Q; ++t0) mmac<Q, LB>(acc[j][t0], ms, cl, t0, t0p, u);
                            }
                        }
                    C *so = soA + rb * SW;
#pragma unroll
                    for (int j = 0; j < 2; ++j)
#pragma unroll
                        for (int t0 = 0; t0 < Q; ++t0) so[j * SH + t0] = acc[j][t0];
                }
            __syncthreads();
            if (rbB < rB)
                for (int rb = rbB; rb < nrc; rb += rB) {
                    const C *si = siB + rb * SW;
                    C acc[Q];
#pragma unroll
                    for (int j = 0; j < Q; ++j) acc[j] = czero<C>();
#pragma unroll
                    for (int ch = 0; ch < 2; ++ch)
#pragma unroll
                        for (int tqp = 0; tqp < Q; ++tqp) {
                            if (SP && tqp != MID && tqp != END) continue;
                            const C v = si[(ch * Q + tqp) * Q];
#pragma unroll
                            for (int t1 = 0; t1 < Q; ++t1) mmac<Q, LB>(acc[t1], ms, ch, t1, tqp, v);
                        }
                    C *wo = woB + (r0 + rb) * WS;
#pragma unroll
                    for (int t1 = 0; t1 < Q; ++t1) wo[t1 * Q] = CJ ? cmul(phB[t1 * Q], acc[t1]) : cjmul(phB[t1 * Q], acc[t1]);
                }
            __syncthreads();
        }
    }
    // gather (row level; adjoint of a column level): out_j(s) = sum_c fB(j, c, s) sum_t M_j[t][s]
    // fA(c, t) in_c(t); fB.at(c): distance of the factors of input c.  SP: outputs at nodes MID and
    // END only.
    template <bool SP, bool CJ, class MS, class FA, class FB>
    static __device__ __forceinline__ void gather(const MS &ms, const Ctx &x, int k, int i, C *W, C *S, FA fA, FB fB)
    {
        const int n = 1 << (D * k), nblk = n >> D, WS = x.npr * RR, SW = (int)mr_s_stride(Q, x.npr);
        constexpr int SU = 2 * Q + PAD.rs, QB = SP ? 2 : Q;
        // stage A: items (rb, c, t_1): modulate input c, contract dimension 0 for both bits j_0
        const int perA = x.npr * Q, rA = NT / perA, a0 = (int)threadIdx.x % perA, rbA = (int)threadIdx.x / perA;
        const int th = NF ? a0 % Q : a0 >> x.lgp, pin = NF ? a0 / Q : a0 & (x.npr - 1);
        const C *winA = W + (((pin >> (D * k)) << (D * k)) + block_base((pin >> D) & (nblk - 1), i) + ((pin & (NC - 1)) << (D * i))) * RR + th * Q;
        const C *phA = fA(pin) + th * Q;
        C *soA = S + (pin * Q + th) * SU;
        // stage B: items (rb, j, s_0): contract dimension 1 per input, modulate, sum over c.  M_1
        // is M_0 with both indices reversed: j_1 = 1 runs dimension 1 backwards, so the
        // coefficients are compile-time operands
        const int perB = x.npr * QB, rB = NT / perB, b0 = (int)threadIdx.x % perB, rbB = (int)threadIdx.x / perB;
        const int sp = NF ? b0 % QB : b0 >> x.lgp, s0 = SP ? (sp ? END : MID) : sp, pj = NF ? b0 / QB : b0 & (x.npr - 1), al = pj & (NC - 1), j0 = al & 1, j1 = al >> 1;
        const int rev = j1 ? -SU : SU, wst = j1 ? -Q : Q, first = j1 && !SP ? Q - 1 : 0;
        const C *siB = S + (pj - al) * Q * SU + j0 * Q + s0 + (j1 ? (Q - 1) * SU : 0);
        C *woB = W + (((pj >> (D * k)) << (D * k)) + block_base((pj >> D) & (nblk - 1), i) + (al << (D * i))) * RR + s0 + first * Q;
        const C *phB = fB(pj) + s0 + first * Q;
        for (int r0 = 0; r0 < x.nr; r0 += x.rc) {
            const int nrc = min(x.rc, x.nr - r0);
            if (rbA < rA)
                for (int rb = rbA; rb < nrc; rb += rA) {
                    const C *w = winA + (r0 + rb) * WS;
                    C z[2][Q];
#pragma unroll
                    for (int e = 0; e < Q; ++e) z[0][e] = z[1][e] = czero<C>();
#pragma unroll
                    for (int t0 = 0; t0 < Q; ++t0) {
                        const C u = CJ ? cjmul(phA[t0], w[t0]) : cmul(phA[t0], w[t0]);
#pragma unroll
                        for (int e = 0; e < Q; ++e) {
                            if (SP && e != MID && e != END) continue;
                            mmac<Q, LB>(z[0][e], ms, 0, t0, e, u);
                            mmac<Q, LB>(z[1][e], ms, 1, t0, e, u);
                        }
                    }
                    C *so = soA + rb * SW;
#pragma unroll
                    for (int e = 0; e < Q; ++e) {
                        if (SP && e != MID && e != END) continue;
                        so[e] = z[0][e];
                        so[Q + e] = z[1][e];
                    }
                }
            __syncthreads();
            if (rbB < rB)
                for (int rb = rbB; rb < nrc; rb += rB) {
                    C acc[QB];   // SP: nodes MID and END
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const C *si = siB + rb * SW + c * Q * SU;
                        const C *ph = phB + fB.at(c);
                        if constexpr (SP) {
                            C v = czero<C>();
#pragma unroll
                            for (int t1 = 0; t1 < Q; ++t1) mmac<Q, LB>(v, ms, 0, t1, MID, si[t1 * rev]);
                            const C e0 = ph[MID * Q], e1 = ph[END * Q], v1 = si[(j1 ? MID : END) * rev];
                            const C u0 = CJ ? cmul(e0, v) : cjmul(e0, v), u1 = CJ ? cmul(e1, v1) : cjmul(e1, v1);
                            acc[0] = c ? madd(acc[0], u0) : u0;
                            acc[1] = c ? madd(acc[1], u1) : u1;
                        } else {
                            C v[Q];
#pragma unroll
                            for (int e = 0; e < Q; ++e) v[e] = czero<C>();
#pragma unroll
                            for (int t1 = 0; t1 < Q; ++t1) {
                                const C zz = si[t1 * rev];
#pragma unroll
                                for (int e = 0; e < Q; ++e) mmac<Q, LB>(v[e], ms, 0, t1, e, zz);
                            }
#pragma unroll
                            for (int e = 0; e < Q; ++e) {
                                const C f = ph[e * wst], u = CJ ? cmul(f, v[e]) : cjmul(f, v[e]);
                                acc[e] = c ? madd(acc[e], u) : u;
                            }
                        }
                    }
                    C *wo = woB + (r0 + rb) * WS;
#pragma unroll
                    for (int e = 0; e < QB; ++e) wo[SP ? (e ? END : MID) * Q : e * wst] = acc[e];
                }
            __syncthreads();
        }
    }
    // factors of a column level for spread and for gather (its adjoint), of a row level for
    // gather and for spread (its adjoint)
    template <int PM> struct ColFA {
        const C *p;
        int npr;
        __device__ __forceinline__ const C *operator()(int pj, int chi) const { return p + pa_at<PM>(npr, pj, chi); }
        static __device__ __forceinline__ constexpr int child(int cl) { return cl * RR; }
    };
    struct ColAdjFB {
        const C *p;
        int npr;
        __device__ __forceinline__ const C *operator()(int pj) const
        {
            return p + pa_at<PM_COMPUTE>(npr, pj & ~3, (pj >> 1) & 1) + (pj & 1) * RR;
        }
        __device__ __forceinline__ int at(int al) const { return (al & 1) * npr * PCA<PM_COMPUTE> + (al >> 1) * 2 * PCA<PM_COMPUTE>; }
    };
    template <int PM> struct RowFB {
        const C *p;
        __device__ __forceinline__ const C *operator()(int pj) const { return p + pj * PRB<PM>; }
        static __device__ __forceinline__ constexpr int at(int c) { return c * RR; }
    };
    struct RowAdjFA {
        const C *p;
        __device__ __forceinline__ const C *operator()(int pj, int chi) const
        {
            return p + ((pj & ~3) + 2 * chi) * PRB<PM_COMPUTE> + (pj & 3) * RR;
        }
        static __device__ __forceinline__ constexpr int child(int cl) { return cl * PRB<PM_COMPUTE>; }
    };

    // ---- one column-form merge level (l -> l+1); ms.M holds the child->parent matrices
    template <int PM, bool SP, class MS>
    static __device__ void col_level(const KArgs<P> &a, const MS &ms, const Ctx &x, C *W, C *S, C *PC, int l, int i,
                                     TS<C> &ts, uint64_t *wbar = nullptr, unsigned wpar = 0)
    {
        const int nout = x.npr;
        if constexpr (PM == PM_TABLE) PC = ts_acquire(ts);
        else col_phases<PM, SP>(a, x, S, PC, l, i);
        __syncthreads();
        if (wbar) wait_input(a, wbar, wpar);   // the weights were copied in during the phase stage
        if constexpr (PM == PM_BUILD) {   // build: store the factors; no weights are touched
            tab_store(ts.tb, PC, 5 * RR * nout);
            ts.tb += 5 * RR * nout;
            __syncthreads();
        } else {
            const C *PA = PC, *PB = PC + nout * 2 * PCA<PM>;
            spread<SP, false>(ms, x, a.k, i, W, S, nout * PCA<PM>, ColFA<PM>{PA, nout}, [&](int pj) { return PB + pj * PCB<PM>; });
        }
        if constexpr (PM == PM_TABLE) ts_release(ts);
    }
    // its conjugate transpose (level l+1 -> l)
    template <bool SP>
    static __device__ void col_level_adj(const KArgs<P> &a, const Ctx &x, C *W, C *S, C *PC, int l, int i)
    {
        col_phases<PM_COMPUTE, SP>(a, x, S, PC, l, i);
        __syncthreads();
        const C *PA = PC, *PB = PC + x.npr * 2 * PCA<PM_COMPUTE>;
        gather<SP, false>(a, x, a.k, i, W, S, [&](int pj) { return PB + pj * PCB<PM_COMPUTE>; }, ColAdjFB{PA, x.npr});
    }

    // fn(rb) for the CTA's right-hand sides, rb a compile-time index of accumulators; a full CTA
    // runs without the checks
    template <class Fn>
    static __device__ __forceinline__ void each_rhs(const Ctx &x, Fn fn)
    {
        if (x.nr == MRMAX) {
#pragma unroll
            for (int rb = 0; rb < MRMAX; ++rb) fn(rb);
        } else {
#pragma unroll
            for (int rb = 0; rb < MRMAX; ++rb) {
                if (rb >= x.nr) break;
                fn(rb);
            }
        }
    }

    // ---- switch at level l: one thread per (pair, s), one accumulator per right-hand side;
    // rounds of whole pairs, results written back after every thread of the round has read.
    // Phase-table layout: q chunks (one per source digit t_1), each [pair][t_0][s], so a
    // chunk is one contiguous block (PM_TABLE plans have one round: npr <= PPR).
    template <int PM>
    static __device__ void switch_tiles(const KArgs<P> &a, const Ctx &x, C *W, int l, TS<C> &ts)
    {
        const int k = a.k, n = 1 << (D * k), L = a.L, WS = x.npr * RR;
        const int G = CfgMR<Q>::PPR;
        for (int p0 = 0; p0 < x.npr; p0 += G) {
            const int pl = p0 + (int)threadIdx.x / RR, s = (int)threadIdx.x % RR;
            const bool act = (int)threadIdx.x < G * RR && pl < x.npr;
            C acc[MRMAX];
#pragma unroll
            for (int rb = 0; rb < MRMAX; ++rb) acc[rb] = czero<C>();
            typename PH::T tS;
            int cb[DMAX] = {0, 0, 0};
            if (PM != PM_TABLE && act) {
                uint32_t Ap, Bstar;
                tile_of(a, x, pl >> (D * k), Ap, Bstar);
                const uint32_t A = (Ap << (D * k)) + digit_rev<D>(pl & (n - 1), k);
                int ca[DMAX];
                morton_decode<D>(A, l, ca);
                morton_decode<D>(Bstar, L - l, cb);
                const int sk[DMAX] = {s % Q, s / Q, 0};
                tS = tpoint<P, D, Q, K>(a, l, ca, sk);
            }
            const C *u = W + pl * RR;
#pragma unroll 1
            for (int th = 0; th < Q; ++th) {
                const C *chunk = nullptr;
                if constexpr (PM == PM_TABLE) chunk = ts_acquire(ts);
                if (act) {
                    C ev[Q];   // the factors of this digit t_1: two at a time (lanes t_0, t_0 + 1)
                    if constexpr (PM != PM_TABLE) {
                        const typename PH2::T tS2 = PH2::dup(tS);
                        const R sg = PH::sign(a, tS);
                        const typename PH::Part h1 = PH::part(a, tS, sget<P, Q>(a, 1, l, cb[1], th), 1);
                        const typename PH2::Part hp = PH2::dup(h1);
#pragma unroll
                        for (int t0 = 0; t0 + 1 < Q; t0 += 2)
                            TL::template ph2<PM_COMPUTE>(
                                PH2::dup(sg),
                                PH2::add(PH2::part(a, tS2, sget<P, Q>(a, 0, l, cb[0], t0), sget<P, Q>(a, 0, l, cb[0], t0 + 1), 0), hp),
                                nullptr, nullptr, ev[t0], ev[t0 + 1]);
                        if constexpr (Q & 1)
                            ev[Q - 1] = TL::template ph<PM_COMPUTE>(
                                sg, PH::add(PH::part(a, tS, sget<P, Q>(a, 0, l, cb[0], Q - 1), 0), h1), nullptr);
                    }
                    if constexpr (PM == PM_TABLE)
#pragma unroll
                        for (int t0 = 0; t0 < Q; ++t0) ev[t0] = chunk[(pl * Q + t0) * RR + s];
                    if constexpr (PM == PM_BUILD) {
#pragma unroll
                        for (int t0 = 0; t0 < Q; ++t0) __stcs(ts.tb + ((int64_t)th * x.npr * Q + pl * Q + t0) * RR + s, ev[t0]);
                    } else {
                        each_rhs(x, [&](int rb) {   // the q weights of a digit t_1 are adjacent: one pointer per right-hand side
                            const C *v = u + rb * WS + Q * th;
#pragma unroll
                            for (int t0 = 0; t0 < Q; ++t0) cmac(acc[rb], ev[t0], v[t0]);
                        });
                    }
                }
                if constexpr (PM == PM_TABLE) {
                    __syncthreads();
                    ts_release(ts);
                }
            }
            if constexpr (PM != PM_BUILD) {
                __syncthreads();
                if (act) {
#pragma unroll
                    for (int rb = 0; rb < MRMAX; ++rb)
                        if (rb < x.nr) W[rb * WS + pl * RR + s] = acc[rb];
                }
                __syncthreads();
            }
        }
        if constexpr (PM == PM_BUILD) ts.tb += (int64_t)x.npr * RR * RR;
    }

    // ---- conjugate transpose of the switch: u(t) = sum_s e^{-2 pi i Phi(x_s^A, y_t^B)} v(s); one
    // thread per (pair, t), one accumulator per right-hand side.  The sum runs over the digit
    // s_1: the parts of its q targets x_s (q per coordinate and target) go to PC first, the
    // targets in lane order, so a phase costs the addition of two of them.
    static __device__ void switch_adj(const KArgs<P> &a, const Ctx &x, C *W, C *PC, int l)
    {
        constexpr int QE = T2::QE, NCMP = T2::NCMP, PSW = 2 * Q * NCMP * QE;   // [coordinate][t][component][s_0]
        const int k = a.k, n = 1 << (D * k), L = a.L, WS = x.npr * RR;
        R *PT = reinterpret_cast<R *>(PC), *SG = PT + x.npr * PSW;
        for (int p0 = 0; p0 < x.npr; p0 += CfgMR<Q>::PPR) {
            const int pl = p0 + (int)threadIdx.x / RR, t = (int)threadIdx.x % RR;
            const bool act = (int)threadIdx.x < CfgMR<Q>::PPR * RR && pl < x.npr;
            C acc[MRMAX];
#pragma unroll
            for (int rb = 0; rb < MRMAX; ++rb) acc[rb] = czero<C>();
#pragma unroll 1
            for (int s1 = 0; s1 < Q; ++s1) {
                __syncthreads();   // the previous digit's (or round's) parts have been used
                for (int it = threadIdx.x; it < CfgMR<Q>::PPR * 2 * Q; it += NT) {
                    const int s0 = it % Q, dim = (it / Q) & 1, pr = p0 + it / (2 * Q);
                    if (pr >= x.npr) break;
                    uint32_t Ap, Bstar;
                    tile_of(a, x, pr >> (D * k), Ap, Bstar);
                    int ca[DMAX], cb[DMAX];
                    morton_decode<D>((Ap << (D * k)) + digit_rev<D>(pr & (n - 1), k), l, ca);
                    morton_decode<D>(Bstar, L - l, cb);
                    const int sk[DMAX] = {s0, s1, 0};
                    const typename PH::T tS = tpoint<P, D, Q, K>(a, l, ca, sk);
                    const auto xf = dim ? tS.x[1] : tS.x[0];
                    const auto Af = dim ? tS.A[1] : tS.A[0];
                    const typename P::SE *e = a.st[dim] + soff<Q>(L, l) + (dim ? cb[1] : cb[0]) * (Q + 2);
                    R *o = PT + pr * PSW + dim * Q * NCMP * QE + s0;
#pragma unroll
                    for (int tt = 0; tt < Q; ++tt) T2::store1(o + tt * NCMP * QE, PH::part_of(a, xf, Af, e[tt], dim == 0));
                    if (dim == 0) SG[pr * Q + s0] = PH::sign(a, tS);
                }
                __syncthreads();
                if (act) {
                    const R *q0 = PT + pl * PSW + (t % Q) * NCMP * QE, *q1 = PT + pl * PSW + (Q + t / Q) * NCMP * QE;
                    const C *v = W + pl * RR + s1 * Q;
                    C ev[Q];
#pragma unroll
                    for (int s0 = 0; s0 + 1 < Q; s0 += 2) {
                        typename PH2::V sg = PH2::dup((R)a.sc.sgn);
                        if constexpr (K == KIND_HYPRADON) {
                            sg.x = SG[pl * Q + s0];
                            sg.y = SG[pl * Q + s0 + 1];
                        }
                        TL::template ph2<PM_COMPUTE>(sg, PH2::add(T2::load2(q0 + s0), T2::load2(q1 + s0)), nullptr, nullptr, ev[s0], ev[s0 + 1]);
                    }
                    if constexpr (Q & 1) {
                        const R sg = K == KIND_HYPRADON ? SG[pl * Q + Q - 1] : (R)a.sc.sgn;
                        ev[Q - 1] = TL::template ph<PM_COMPUTE>(sg, PH::add(T2::load1(q0 + Q - 1), T2::load1(q1 + Q - 1)), nullptr);
                    }
                    each_rhs(x, [&](int rb) {
                        const C *w = v + rb * WS;
#pragma unroll
                        for (int s0 = 0; s0 < Q; ++s0) cjmac(acc[rb], ev[s0], w[s0]);
                    });
                }
            }
            __syncthreads();
            if (act) {
#pragma unroll
                for (int rb = 0; rb < MRMAX; ++rb)
                    if (rb < x.nr) W[rb * WS + pl * RR + t] = acc[rb];
            }
        }
        __syncthreads();
    }

    // ---- switch of a phase that is a sum over dimensions (Tile::switch_sep): the factors of both
    // dimensions (q x q per pair each; mr_s_size holds them for any rc) go to the scratch S, then
    // one sweep per dimension, in place.  ADJ: the conjugate transpose.
    template <bool ADJ>
    static __device__ void switch_sep(const KArgs<P> &a, const Ctx &x, C *W, C *S, int l)
    {
        const int k = a.k, n = 1 << (D * k), L = a.L, WS = x.npr * RR;
        for (int it = threadIdx.x; it < x.npr * 2 * RR; it += NT) {   // [pair][dim][s][t]
            const int t = it % Q, sd = (it / Q) % Q, dim = (it / RR) & 1, pr = it / (2 * RR);
            uint32_t Ap, Bstar;
            tile_of(a, x, pr >> (D * k), Ap, Bstar);
            int ca[DMAX], cb[DMAX];
            morton_decode<D>((Ap << (D * k)) + digit_rev<D>(pr & (n - 1), k), l, ca);
            morton_decode<D>(Bstar, L - l, cb);
            const int sk[DMAX] = {dim ? Q : sd, dim ? sd : Q, 0};
            const typename PH::T tS = tpoint<P, D, Q, K>(a, l, ca, sk);
            S[it] = TL::template ph<PM_COMPUTE>(
                PH::sign(a, tS),
                PH::part_of(a, dim ? tS.x[1] : tS.x[0], dim ? tS.A[1] : tS.A[0], sget<P, Q>(a, dim, l, dim ? cb[1] : cb[0], t), dim == 0),
                nullptr);
        }
        __syncthreads();
#pragma unroll
        for (int dim = 0; dim < 2; ++dim) {
            for (int it = threadIdx.x; it < x.nr * x.npr * Q; it += NT) {   // one line of q values
                const int o = it % Q, pr = (it / Q) & (x.npr - 1), rb = (it / Q) >> x.lgp;
                C *w = W + rb * WS + pr * RR + (dim ? o : o * Q);
                const C *e = S + (pr * 2 + dim) * RR;
                const int st = dim ? Q : 1;
                C v[Q];
#pragma unroll
                for (int u = 0; u < Q; ++u) v[u] = w[u * st];
#pragma unroll
                for (int s = 0; s < Q; ++s) {
                    C acc = czero<C>();
#pragma unroll
                    for (int u = 0; u < Q; ++u) {
                        if constexpr (ADJ)
                            acc = madd(acc, cjmul(e[u * Q + s], v[u]));
                        else
                            cmac(acc, e[s * Q + u], v[u]);
                    }
                    w[s * st] = acc;
                }
            }
            __syncthreads();
        }
    }

    // ---- one row-form merge level (l -> l+1); SP: the outputs' nodes MID and END only
    template <int PM, bool SP, class MS>
    static __device__ void row_level(const KArgs<P> &a, const MS &ms, const Ctx &x, C *W, C *S, C *PC, int l, int i,
                                     TS<C> &ts, uint64_t *wbar = nullptr, unsigned wpar = 0)
    {
        const int nout = x.npr;
        if constexpr (PM == PM_TABLE) PC = ts_acquire(ts);
        else row_phases<PM, SP>(a, x, S, PC, l, i);
        __syncthreads();
        if (wbar) wait_input(a, wbar, wpar);   // the weights were copied in during the phase stage
        if constexpr (PM == PM_BUILD) {   // build: store the factors; no weights are touched
            tab_store(ts.tb, PC, 5 * RR * nout);
            ts.tb += 5 * RR * nout;
            __syncthreads();
        } else {
            const C *PA = PC, *PB = PC + nout * RR;
            gather<SP, true>(ms, x, a.k, i, W, S, [&](int pj) { return PA + pj * RR; }, RowFB<PM>{PB});
        }
        if constexpr (PM == PM_TABLE) ts_release(ts);
    }
    // its conjugate transpose (level l+1 -> l); SP: inputs at nodes MID and END only
    template <bool SP>
    static __device__ void row_level_adj(const KArgs<P> &a, const Ctx &x, C *W, C *S, C *PC, int l, int i)
    {
        row_phases<PM_COMPUTE, SP>(a, x, S, PC, l, i);
        __syncthreads();
        const C *PA = PC, *PB = PC + x.npr * RR;
        spread<SP, true>(a, x, a.k, i, W, S, RR, RowAdjFA{PB}, [&](int pj) { return PA + pj * RR; });
    }

    // ---- final evaluation: PC[pair][t] = l_t(x) conj(e^{2pi i Phi(x_t, y0(Y))}), PC[pair][r] = e^{2pi i Phi(x, y0(Y))}
    static __device__ void final_factors(const KArgs<P> &a, const Ctx &x, C *PC)
    {
        const int k = a.k, n = 1 << (D * k), L = a.L;
        const int cY[DMAX] = {0, 0, 0};
        const int ctr[DMAX] = {Q, Q, Q};
        const typename PH::S sY = spoint<P, D, Q, K>(a, L, cY, ctr);
        for (int it = threadIdx.x; it < x.npr * (RR + 1); it += NT) {
            const int t = it % (RR + 1), pl = it / (RR + 1);
            C e = czero<C>();
            const R lag = t < RR ? a.ltgt[t % Q] * a.ltgt[t / Q] : R(1);
            if (lag != R(0)) {
                uint32_t Ap, Bstar;
                tile_of(a, x, pl >> (D * k), Ap, Bstar);
                int ca[DMAX];
                morton_decode<D>((Ap << (D * k)) + digit_rev<D>(pl & (n - 1), k), L, ca);
                const int tk[DMAX] = {t < RR ? t % Q : Q + 1, t < RR ? t / Q : Q + 1, 0};
                const C e0 = expphase<P, D, K>(a, tpoint<P, D, Q, K>(a, L, ca, tk), sY);
                if (t < RR) {
                    e.x = lag * e0.x;
                    e.y = -lag * e0.y;
                } else {
                    e = e0;
                }
            }
            PC[it] = e;
        }
    }
    template <int PM>
    static __device__ void final_eval(const KArgs<P> &a, const Ctx &x, const C *W, C *PC, C *f, TS<C> &ts)
    {
        const int k = a.k, n = 1 << (D * k), L = a.L, WS = x.npr * RR;
        if constexpr (PM == PM_TABLE) PC = ts_acquire(ts);
        else final_factors(a, x, PC);
        __syncthreads();
        if constexpr (PM == PM_BUILD) {   // build: store the factors; no weights are touched
            tab_store(ts.tb, PC, x.npr * (RR + 1));
            ts.tb += x.npr * (RR + 1);
            __syncthreads();
        }
        for (int j = threadIdx.x; PM != PM_BUILD && j < x.nr * x.npr; j += NT) {
            const int pl = j & (x.npr - 1), rb = j >> x.lgp;
            const C *pc = PC + pl * (RR + 1);
            const C *w = W + rb * WS + pl * RR;
            C acc = czero<C>();
            for (int t = 0; t < RR; ++t)
                if (a.ltgt[t % Q] * a.ltgt[t / Q] != R(0)) cmac(acc, pc[t], w[t]);
            uint32_t Ap, Bstar;
            tile_of(a, x, pl >> (D * k), Ap, Bstar);
            int ca[DMAX];
            morton_decode<D>((Ap << (D * k)) + digit_rev<D>(pl & (n - 1), k), L, ca);
            const int64_t flat = ((int64_t)ca[0] << L) + ca[1];
            f[(int64_t)(x.rhs0 + rb) * a.npts + flat] = cmul(pc[RR], acc);
        }
        if constexpr (PM == PM_TABLE) {   // the stream continues with the CTA's next tile group
            __syncthreads();
            ts_release(ts);
        }
    }

    // ---- adjoint pass input: the forward pass's outputs (strided pairs) into digit-reversed
    // slots; output: natural order, contiguous
    static __device__ void load_strided(const KArgs<P> &a, const Ctx &x, C *W)
    {
        __shared__ int64_t poff[64];
        const int k = a.k, n = 1 << (D * k), WS = x.npr * RR;
        const int64_t Sstar = 1LL << (D * (a.L - a.l0 - k));
        for (int pl = threadIdx.x; pl < x.npr; pl += NT) {
            uint32_t Ap, Bstar;
            tile_of(a, x, pl >> (D * k), Ap, Bstar);
            poff[pl] = ((((int64_t)Ap << (D * k)) + digit_rev<D>(pl & (n - 1), k)) * Sstar + Bstar) * RR;
        }
        __syncthreads();
        for (int j = threadIdx.x; j < x.nr * WS; j += NT) {
            const int rb = (j / RR) >> x.lgp, e = j - rb * WS;
            const int pl = e / RR, t = e - pl * RR;
            W[j] = __ldcg(a.win + (int64_t)(x.rhs0 + rb) * a.wstride + poff[pl] + t);
        }
    }
    static __device__ void store_contig(const KArgs<P> &a, const Ctx &x, const C *W)
    {
        const int WS = x.npr * RR;
        const int64_t off = (int64_t)x.tile0 * ((int64_t)RR << (D * a.k));
        for (int j = threadIdx.x; j < x.nr * WS; j += NT) {
            const int rb = (j / RR) >> x.lgp, e = j - rb * WS;
            a.wout[(int64_t)(x.rhs0 + rb) * a.wstride + off + e] = W[j];
        }
    }
    // ---- init^H: g(y) = sum_t conj(PC[pair][t]) w(t), PC as in init (slots in natural order)
    static __device__ void init_adj(const KArgs<P> &a, const Ctx &x, const C *W, C *PC)
    {
        const int k = a.k, n = 1 << (D * k), nblk = n >> D, L = a.L, WS = x.npr * RR;
        const bool corner = skip_first(a);
        if (!corner) {
            init_factors(a, x, PC);
            __syncthreads();
        }
        for (int it = threadIdx.x; it < x.nr * x.npr; it += NT) {
            const int pr = it & (x.npr - 1), rb = it >> x.lgp;
            uint32_t Ap, Bstar;
            tile_of(a, x, pr >> (D * k), Ap, Bstar);
            int cb[DMAX];
            morton_decode<D>((Bstar << (D * k)) + (pr & (n - 1)), L, cb);
            C acc = czero<C>();
            if (corner) {   // the four outputs of the block (level 1) at the leaf's node
                const int c = pr & (NC - 1), b = (pr >> D) & (nblk - 1), tau = pr >> (D * k);
                const C *w = W + rb * WS + (tau * n + (b << D)) * RR + ((c & 1) ? MID : END) + ((c >> 1) ? MID : END) * Q;
#pragma unroll
                for (int al = 0; al < NC; ++al) acc = madd(acc, w[al * RR]);
            } else {
                const C *w = W + rb * WS + pr * RR;
                for (int t = 0; t < RR; ++t)
                    if (a.lsrc[t % Q] * a.lsrc[t / Q] != R(0)) acc = madd(acc, cjmul(PC[pr * RR + t], w[t]));
            }
            a.gadj[(int64_t)(x.rhs0 + rb) * a.npts + ((int64_t)cb[0] << L) + cb[1]] = acc;
        }
    }
    // ---- final^H: w(t) = conj(PC[pair][t] PC[pair][r]) f(x), PC as in final_eval (slots in
    // digit-reversed order at level L; with a corner, level L - 1, the four inputs of a block)
    static __device__ void final_adj(const KArgs<P> &a, const Ctx &x, C *W, C *PC)
    {
        const int k = a.k, n = 1 << (D * k), nblk = n >> D, L = a.L, WS = x.npr * RR;
        const bool corner = skip_last(a);
        if (corner ? a.k == 1 : true)   // nodes beyond the four are read by no level of this pass
            for (int j = threadIdx.x; j < x.nr * WS; j += NT) W[j] = czero<C>();
        if (!corner) final_factors(a, x, PC);
        __syncthreads();
        if (corner) {
            for (int it = threadIdx.x; it < x.nr * x.npr; it += NT) {
                const int pr = it & (x.npr - 1), rb = it >> x.lgp;
                const int al = pr & (NC - 1), ra = (pr >> D) & (nblk - 1), tau = pr >> (D * k);
                uint32_t Ap, Bstar;
                tile_of(a, x, tau, Ap, Bstar);
                int ca[DMAX];
                morton_decode<D>((((Ap << (D * (k - 1))) + digit_rev<D>(ra, k - 1)) << D) + al, L, ca);
                const C v = a.fadj[(int64_t)(x.rhs0 + rb) * a.npts + ((int64_t)ca[0] << L) + ca[1]];
                C *w = W + rb * WS + (tau * n + ra) * RR + ((al & 1) ? MID : END) + ((al >> 1) ? MID : END) * Q;
#pragma unroll
                for (int c = 0; c < NC; ++c) w[(c * nblk) * RR] = v;
            }
        } else {
            for (int it = threadIdx.x; it < x.nr * x.npr; it += NT) {
                const int pl = it & (x.npr - 1), rb = it >> x.lgp;
                uint32_t Ap, Bstar;
                tile_of(a, x, pl >> (D * k), Ap, Bstar);
                int ca[DMAX];
                morton_decode<D>((Ap << (D * k)) + digit_rev<D>(pl & (n - 1), k), L, ca);
                const C *pc = PC + pl * (RR + 1);
                const C v = cjmul(pc[RR], a.fadj[(int64_t)(x.rhs0 + rb) * a.npts + ((int64_t)ca[0] << L) + ca[1]]);
                for (int t = 0; t < RR; ++t)
                    if (a.ltgt[t % Q] * a.ltgt[t / Q] != R(0)) W[rb * WS + pl * RR + t] = cjmul(pc[t], v);
            }
        }
        __syncthreads();
    }

    // shared memory of one CTA, bytes
    static __host__ __device__ size_t smem_bytes(int npr, int nr, int rc)
    {
        return sizeof(C) * ((size_t)npr * RR * (size_t)(nr + 5) + (size_t)mr_s_size(Q, npr, rc) +
                            (size_t)npr * mr_pc_extra(Q));
    }

    static __device__ __forceinline__ Ctx ctx(const KArgs<P> &a, int cta)
    {
        Ctx x;
        x.tile0 = (int)shard_cta<D>(a, (uint32_t)cta) * a.T;
        const int nb = P::is_f64 ? a.nb : MRMAX;   // (a compile-time number is worth 1% of the mixed passes)
        x.rhs0 = (int)blockIdx.y * nb;
        x.nr = min(nb, a.nrhs - x.rhs0);
        x.npr = a.T << (D * a.k);
        x.rc = a.rc;
        x.lgp = __ffs(x.npr) - 1;
        return x;
    }
};

// pass bodies shared by the per-pass kernels and the persistent batch kernel; ms is a
// kernel parameter holding M, so the interpolation reads its coefficients from the
// constant bank; ts carries the phase table (PM_BUILD, PM_TABLE)
// wbar (per-pass kernels): the input weights come by bulk copies that overlap the first
// level's phase stage (wpar: the mbarrier phase of this tile group); null: plain loads first
template <int Q, class P, int K, bool LB, int PM, class MS>
__device__ __forceinline__ bool col_pass_mr(const KArgs<P> &a, const MS &ms, const typename TileMR<Q, P, K, LB>::Ctx &x,
                                            unsigned char *sm, const typename P::C *g, TS<typename P::C> &ts,
                                            uint64_t *wbar = nullptr, unsigned wpar = 0)
{
    using C = typename P::C;
    using TM = TileMR<Q, P, K, LB>;
    const int WS = x.npr * TM::RR;
    C *W = reinterpret_cast<C *>(sm);
    C *S = W + x.nr * WS;
    C *PC = S + mr_s_size(Q, x.npr, x.rc);
    const bool async = wbar && !(a.flags & F_INIT) && a.k > 0 && a.shard_mode != 2;
    // KArgs::corner: level 0 is done by the first step, level 1 has four non-zero nodes per input
    const bool skip0 = TM::skip_first(a);
    if (skip0) {
        if constexpr (PM == PM_BUILD)
            ts.tb += (int64_t)6 * TM::RR * x.npr;   // the blocks of the first step and of level 0 stay unused
        else
            TM::init_corner(a, x, W, g);
    } else if (a.flags & F_INIT) {
        TM::template init<PM>(a, x, W, PC, g, ts);
    } else if (async) {
        TM::load_async(a, x, W, wbar);
    } else if (PM != PM_BUILD) {
        TM::load(a, x, W);
        __syncthreads();
    }
    for (int i = skip0 ? 1 : 0; i < a.k; ++i) {
        uint64_t *wb = async && i == 0 ? wbar : nullptr;
        if (LB && (a.corner & CORNER_SRC) && a.l0 + i == 1)
            TM::template col_level<PM, LB>(a, ms, x, W, S, PC, a.l0 + i, i, ts, wb, wpar);
        else
            TM::template col_level<PM, false>(a, ms, x, W, S, PC, a.l0 + i, i, ts, wb, wpar);
    }
    if (a.flags & F_SWITCH) {
        if constexpr (K == KIND_DOT || K == KIND_SEPARABLE) {   // evaluated, not tabled
            if constexpr (PM != PM_BUILD) TM::template switch_sep<false>(a, x, W, S, a.l0 + a.k);
        } else {
            TM::template switch_tiles<PM>(a, x, W, a.l0 + a.k, ts);
        }
    }
    if (PM != PM_BUILD) TM::store(a, x, W);
    return async;
}

template <int Q, class P, int K, bool LB, int PM, class MS>
__device__ __forceinline__ bool row_pass_mr(const KArgs<P> &a, const MS &ms, const typename TileMR<Q, P, K, LB>::Ctx &x,
                                            unsigned char *sm, typename P::C *f, TS<typename P::C> &ts,
                                            uint64_t *wbar = nullptr, unsigned wpar = 0)
{
    using C = typename P::C;
    using TM = TileMR<Q, P, K, LB>;
    const int WS = x.npr * TM::RR;
    C *W = reinterpret_cast<C *>(sm);
    C *S = W + x.nr * WS;
    C *PC = S + mr_s_size(Q, x.npr, x.rc);
    // KArgs::corner: the last step does the last level, and the level before it has four output nodes
    const bool skip = TM::skip_last(a);
    const int k1 = skip ? a.k - 1 : a.k;
    const bool async = wbar && k1 > 0 && a.shard_mode != 2;
    if (async) {
        TM::load_async(a, x, W, wbar);
    } else if (PM != PM_BUILD) {
        TM::load(a, x, W);
        __syncthreads();
    }
    for (int i = 0; i < k1; ++i) {
        uint64_t *wb = async && i == 0 ? wbar : nullptr;
        if (LB && (a.corner & CORNER_TGT) && a.l0 + i == a.L - 2)
            TM::template row_level<PM, LB>(a, ms, x, W, S, PC, a.l0 + i, i, ts, wb, wpar);
        else
            TM::template row_level<PM, false>(a, ms, x, W, S, PC, a.l0 + i, i, ts, wb, wpar);
    }
    if (skip) {
        if constexpr (PM != PM_BUILD) TM::final_corner(a, x, W, f);
    } else if (a.flags & F_FINAL)
        TM::template final_eval<PM>(a, x, W, PC, f, ts);
    else if (PM != PM_BUILD)
        TM::store(a, x, W);
    return async;
}

constexpr int TABCTL_BYTES = (int)((sizeof(TabCtl) + 15) / 16 * 16);

// largest table block of a pass (a level's 5 r factors per pair, or a switch chunk)
template <int Q>
__host__ __device__ constexpr int tab_blk_factor() { return Q > 5 ? Q : 5; }

// shared memory of a CTA: PM_TABLE puts the stream control and two block buffers first
template <int Q, class P, int K, bool LB, int PM>
__device__ __forceinline__ unsigned char *mr_setup(const KArgs<P> &a, const typename TileMR<Q, P, K, LB>::Ctx &x,
                                                   unsigned char *smem, TS<typename P::C> &ts, bool row)
{
    using C = typename P::C;
    ts.tb = nullptr;
    ts.ctl = nullptr;
    ts.buf[0] = ts.buf[1] = nullptr;
    ts.j = 0;
    ts.err = a.err;
    ts.c0 = (int)blockIdx.x;
    ts.cstep = (int)gridDim.x;
    ts.cstride = a.ptab_cta;
    if constexpr (PM != PM_TABLE) return smem;
    ts.tb = a.ptab;
    const int blk = tab_blk_factor<Q>() * Q * Q * x.npr;
    ts.ctl = reinterpret_cast<TabCtl *>(smem);
    ts.buf[0] = reinterpret_cast<C *>(smem + TABCTL_BYTES);
    ts.buf[1] = ts.buf[0] + blk;
    TileMR<Q, P, K, LB>::ts_setup(ts, a, x, row);
    return reinterpret_cast<unsigned char *>(ts.buf[1] + blk);
}

// Per-pass kernels.  A CTA runs tile groups blockIdx.x, blockIdx.x + gridDim.x, ... < a.ncta
// (one with a full grid; PM_TABLE launches as many CTAs as fit and streams the table of
// all its tile groups through one pipeline).
template <int Q, class P, int K, bool LB, int PM>
__global__ void __launch_bounds__(CfgMR<Q>::NT, MinbMR<Q, P>::v) k_col_pass_mr(const KArgs<P> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint64_t wbar;
    TS<typename P::C> ts;
    unsigned char *work = mr_setup<Q, P, K, LB, PM>(a, TileMR<Q, P, K, LB>::ctx(a, blockIdx.x), smem_raw, ts, false);
    if (PM == PM_COMPUTE && threadIdx.x == 0) {
        mbar_init(&wbar, 1);
        mbar_init_fence();
    }
    __syncthreads();
    unsigned it = 0;
    for (int c = blockIdx.x; c < a.ncta; c += gridDim.x, ++it) {
        if constexpr (PM == PM_BUILD) ts.tb = a.ptab + (int64_t)c * a.ptab_cta;
        col_pass_mr<Q, P, K, LB, PM>(a, a, TileMR<Q, P, K, LB>::ctx(a, c), work, a.g, ts, PM == PM_COMPUTE ? &wbar : nullptr,
                                 it & 1u);
        __syncthreads();
    }
}

template <int Q, class P, int K, bool LB, int PM>
__global__ void __launch_bounds__(CfgMR<Q>::NT, MinbMR<Q, P>::v) k_row_pass_mr(const KArgs<P> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint64_t wbar;
    TS<typename P::C> ts;
    unsigned char *work = mr_setup<Q, P, K, LB, PM>(a, TileMR<Q, P, K, LB>::ctx(a, blockIdx.x), smem_raw, ts, true);
    if (PM == PM_COMPUTE && threadIdx.x == 0) {
        mbar_init(&wbar, 1);
        mbar_init_fence();
    }
    __syncthreads();
    unsigned it = 0;
    for (int c = blockIdx.x; c < a.ncta; c += gridDim.x, ++it) {
        if constexpr (PM == PM_BUILD) ts.tb = a.ptab + (int64_t)c * a.ptab_cta;
        row_pass_mr<Q, P, K, LB, PM>(a, a, TileMR<Q, P, K, LB>::ctx(a, c), work, a.f, ts, PM == PM_COMPUTE ? &wbar : nullptr,
                                 it & 1u);
        __syncthreads();
    }
}

// Adjoint passes: the tiles of a forward pass, its steps conjugate-transposed in reverse order,
// for up to MRMAX right-hand sides per CTA.
template <int Q, class P, int K, bool LB>
__global__ void __launch_bounds__(CfgMR<Q>::NT, MinbMR<Q, P>::v) k_col_pass_mr_adj(const KArgs<P> a)
{
    using C = typename P::C;
    using TM = TileMR<Q, P, K, LB>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const typename TM::Ctx x = TM::ctx(a, blockIdx.x);
    C *W = reinterpret_cast<C *>(smem_raw), *S = W + x.nr * x.npr * TM::RR, *PC = S + mr_s_size(Q, x.npr, x.rc);
    TM::load_strided(a, x, W);
    __syncthreads();
    if (a.flags & F_SWITCH) {
        if constexpr (K == KIND_DOT || K == KIND_SEPARABLE)
            TM::template switch_sep<true>(a, x, W, S, a.l0 + a.k);
        else
            TM::switch_adj(a, x, W, PC, a.l0 + a.k);
    }
    for (int i = a.k - 1; i >= (TM::skip_first(a) ? 1 : 0); --i) {
        if (LB && (a.corner & CORNER_SRC) && a.l0 + i == 1)
            TM::template col_level_adj<LB>(a, x, W, S, PC, a.l0 + i, i);
        else
            TM::template col_level_adj<false>(a, x, W, S, PC, a.l0 + i, i);
    }
    if (a.flags & F_INIT)
        TM::init_adj(a, x, W, PC);
    else
        TM::store_contig(a, x, W);
}

template <int Q, class P, int K, bool LB>
__global__ void __launch_bounds__(CfgMR<Q>::NT, MinbMR<Q, P>::v) k_row_pass_mr_adj(const KArgs<P> a)
{
    using C = typename P::C;
    using TM = TileMR<Q, P, K, LB>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const typename TM::Ctx x = TM::ctx(a, blockIdx.x);
    C *W = reinterpret_cast<C *>(smem_raw), *S = W + x.nr * x.npr * TM::RR, *PC = S + mr_s_size(Q, x.npr, x.rc);
    if (a.flags & F_FINAL)
        TM::final_adj(a, x, W, PC);
    else
        TM::load_strided(a, x, W);
    __syncthreads();
    for (int i = (TM::skip_last(a) ? a.k - 1 : a.k) - 1; i >= 0; --i) {
        if (LB && (a.corner & CORNER_TGT) && a.l0 + i == a.L - 2)
            TM::template row_level_adj<LB>(a, x, W, S, PC, a.l0 + i, i);
        else
            TM::template row_level_adj<false>(a, x, W, S, PC, a.l0 + i, i);
    }
    TM::store_contig(a, x, W);
}

// ====================================================================== persistent batch
// Many independent problems in one launch.  A job is one pass of one problem for one
// block of up to MRMAX right-hand sides; its units are the pass's CTAs.  Jobs are
// ordered by pass index, so a unit only ever waits for units that come earlier in the
// queue: CTAs take units from a global counter in order, and before a unit of pass j
// starts, the CTA waits until every unit of the same problem's pass j-1 (same RHS
// block) has finished.  The unit that is earliest among the unfinished ones never
// waits, so the queue always advances.  A wait gives up after a time limit, sets the
// error flag and skips its unit; once the flag is set no unit waits or computes.

constexpr int BATCH_MAX = 256;          // problems per batch

struct BatchJob {
    int prob, desc;      // problem, descriptor (problem, pass) of the job
    int y;               // block of right-hand sides
    int ctas;            // CTAs of the pass (tile groups of T tiles)
    int per;             // CTAs per work unit, run one after another by one CTA
    int units, first;    // units of the job and index of its first unit in the queue
    int dep;             // job that must finish first (-1: none)
    int row, pad0, pad1, pad2;   // 1: row pass
};

template <class P>
struct BatchArgs {
    typename P::R M[2][QMAX][QMAX];   // child->parent matrices (the same for every problem)
    const KArgs<P> *__restrict__ desc;   // per (problem, pass); g and f come from the arrays below
    const BatchJob *jobs;
    int njobs, units;
    unsigned *ctr;                 // [njobs] finished units per job, [njobs] queue head
    int *err;                      // set when a wait times out
    unsigned long long *stats;     // [0] nanoseconds spent waiting, [1] waits
    unsigned long long wait_ns;    // time limit of one wait
    int dep_extra;                 // added to every wait's target (0; 1 only in the time-out self-test)
    const typename P::C *g[BATCH_MAX];
    typename P::C *f[BATCH_MAX];
};

__device__ __forceinline__ uint64_t globaltimer_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// wait (one thread) until *ctr >= target; 1 if given up (time limit or error flag)
__device__ __forceinline__ int wait_count(const unsigned *ctr, unsigned target, int *err, unsigned long long limit,
                                          unsigned long long *stats)
{
    const uint64_t t0 = globaltimer_ns();
    for (int n = 0;; ++n) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
        if (v >= target) {
            if (n > 0) {
                atomicAdd(&stats[0], (unsigned long long)(globaltimer_ns() - t0));
                atomicAdd(&stats[1], 1ull);
            }
            return 0;
        }
        if (*reinterpret_cast<volatile int *>(err)) return 1;
        if (globaltimer_ns() - t0 > limit) {
            atomicExch(err, 1);
            return 1;
        }
        __nanosleep(256);
    }
}

template <int Q, class P, int K, bool LB>
__global__ void __launch_bounds__(CfgMR<Q>::NT, MinbMR<Q, P>::v) k_batch_mr(const BatchArgs<P> b)
{
    using TM = TileMR<Q, P, K, LB>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_unit, s_job, s_skip;
    __shared__ uint64_t wbar;                                  // the units' input copies
    if (threadIdx.x == 0) {
        mbar_init(&wbar, 1);
        mbar_init_fence();
    }
    __syncthreads();
    unsigned wuse = 0;                                         // phases of wbar used so far
    for (;;) {
        if (threadIdx.x == 0) {
            const int u = (int)atomicAdd(&b.ctr[b.njobs], 1u);
            s_unit = u;
            if (u < b.units) {
                int lo = 0, hi = b.njobs - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (__ldg(&b.jobs[mid].first) <= u) lo = mid; else hi = mid - 1;
                }
                s_job = lo;
                int skip = *reinterpret_cast<volatile int *>(b.err);
                const int dep = __ldg(&b.jobs[lo].dep);
                if (!skip && dep >= 0)
                    skip = wait_count(&b.ctr[dep], (unsigned)(__ldg(&b.jobs[dep].units) + b.dep_extra), b.err, b.wait_ns,
                                      b.stats);
                s_skip = skip;
            }
        }
        __syncthreads();
        const int u = s_unit;
        if (u >= b.units) break;
        const BatchJob jb = b.jobs[s_job];
        if (!s_skip) {
            // the pass's arguments stay in global memory (read-only for the whole launch; the
            // kernel's shared memory is at the two-CTAs-per-SM limit)
            const KArgs<P> &a = b.desc[jb.desc];
            const int c0 = (u - jb.first) * jb.per;
            const int c1 = min(c0 + jb.per, jb.ctas);
            for (int c = c0; c < c1; ++c) {
                typename TM::Ctx x;
                x.tile0 = c * a.T;
                x.rhs0 = jb.y * MRMAX;
                x.nr = min(MRMAX, a.nrhs - x.rhs0);
                x.npr = a.T << (2 * a.k);
                x.rc = a.rc;
                x.lgp = __ffs(x.npr) - 1;
                TS<typename P::C> ts{};
                const bool used = jb.row ? row_pass_mr<Q, P, K, LB, PM_COMPUTE>(a, b, x, smem_raw, b.f[jb.prob], ts, &wbar, wuse & 1u)
                                         : col_pass_mr<Q, P, K, LB, PM_COMPUTE>(a, b, x, smem_raw, b.g[jb.prob], ts, &wbar, wuse & 1u);
                wuse += used ? 1u : 0u;
                __syncthreads();
            }
        }
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) atomicAdd(&b.ctr[s_job], 1u);
    }
}

}  // namespace bfk
