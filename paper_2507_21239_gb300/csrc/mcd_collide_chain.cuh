// mcd_collide_chain.cuh -- the mixed-precision collision chain of one cell,
// split over specialised warps.  Same method and arithmetic as cell_chain<1, ...>
// in mcd_collide.cuh (Zsom & Dullemond's representative-particle scheme, Summary
// of the mcdust paper), and the bits its builds have given: every rounding here is
// explicit, where pair_dv leaves the fusing of products to the compiler, and a dv
// below 1e-19 cm/s counts as 0.  What differs is who does what between which
// barriers.
//
// What bounds it: the serial chain of one event (choose i, form row i, choose
// j, apply the outcome, renew row and column i) on the heaviest cell; no pipe
// is near its peak.  Measured on GB300, one warp: a dependent FP32 operation 5
// cycles, a shuffle 25 (35 with its predicated add), a store to shared memory
// and a load of it by another lane 29, a block barrier of five warps 23, a
// ballot 25, an FP64 operation 65.  So as little as possible stays on the
// chain, and what stays runs in the warp that can do it in the fewest dependent
// steps:
//
//  * worker warps: thread k owns swarm k (group q of 32 swarms: warp q).  Workers
//    keep the row sums, form row i, the new row and column, and the prefixes
//    within each group (two exchanges through shared memory), and post those and
//    the groups' totals.  Their code is free of branches where the work lies.
//  * the choice warp finds i and j from the posted prefixes (lane s forms slot
//    s's prefix over the groups straight from the posted totals; choose()) and
//    says which outcome the event has.  One warp does this for all: done by
//    every worker warp, the same loads and additions compete for the issue slots
//    of the SM.  The two outcomes that do not depend on j (a partner lighter
//    than dm m_i is absorbed, or erodes i, in groups of total mass dm m_i) are
//    kept ready per swarm, new mass and swarm cache; other partners take the
//    general outcome in the lane that found j.
//  * while j is chosen the workers form the new row and column of the ready
//    outcome of the kind that came last, and (up to 256 swarms) the row sums they
//    lead to; if the event takes that outcome, the next choice's prefixes follow
//    at once.  Both ready outcomes together take longer than the choice: 100
//    swarms 0.92 against 0.90 us per event.
//  * the mass warp keeps the ready outcomes, masses and caches of the swarm that
//    has just changed.
//  * the clock warp sums the last event's new row (the fresh R_i), advances the
//    clock, tests it against t_end and draws the next block's random numbers,
//    one Philox round per event.
//
// Measured, heaviest cell, us per event (one thread per swarm with block-wide
// scans before -> now): 50 swarms 1.35 -> 0.85, 100: 1.40 -> 0.91, 200: 1.53 ->
// 0.98, 300: 1.69 -> 1.31, 400: 1.97 -> 1.47, 500: 2.01 -> 1.62.  (Without the
// row sums formed ahead 0.93 at 100 and 1.03 at 200; with them 1.56 at 400,
// where they compete with the choice for issue slots.)  Up to 256 swarms the
// shared matrix beats recomputing row i (200 swarms: 0.98 against 1.12); where the
// ready outcomes leave no room for the matrix (from about 290) recomputing in this
// layout beats the stored matrix in the block-scan layout (1.31 against 1.71).  Two groups per worker warp, to issue what does not
// depend on the swarm once per sub-partition, were slower at every size (200:
// 1.25, 400: 1.63): one warp's instructions issue in order, and two warps hide
// each other's latencies where two streams in one do not.
#pragma once
#include "mcd_collide.cuh"

namespace mcd {

// named barriers (0 is __syncthreads): count is the number of threads that
// arrive or wait.  The .aligned forms want the whole warp at one instruction;
// what precedes them may depend on the lane, so each brings the warp together first.
__device__ __forceinline__ void bar_sync(int id, int count)
{
    __syncwarp();
    asm volatile("barrier.cta.sync.aligned %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int count)
{
    __syncwarp();
    asm volatile("barrier.cta.arrive.aligned %0, %1;" ::"r"(id), "r"(count) : "memory");
}
// kBarNew: the new row posted (workers arrive; the clock warp waits); kBarRead:
// i's new cache read (workers arrive; the mass warp waits); kBarRates: prefixes
// of R posted, the fresh R_i, masses and caches too (workers and mass warp
// arrive; choice and clock warps wait); kBarI: i posted (the choice warp arrives;
// workers wait); kBarRow: prefixes of row i posted (workers arrive; the choice
// warp waits); kBarReady: the last swarm's ready outcomes stored (the mass warp
// arrives; workers wait); kBarEvent: outcome and verdict on the clock posted (all
// wait); kBarBuild: before a rebuild, the matrix entries of all workers and i's
// cache (workers wait; the mass warp arrives)
constexpr int kBarNew = 1, kBarRead = 2, kBarRates = 3, kBarI = 4, kBarRow = 5, kBarReady = 6, kBarEvent = 7,
              kBarBuild = 8;
constexpr int kChainRoles = 3;  // choice, mass and clock warps

// NW: slots for the groups' totals (a power of two).  Group q's total sits in
// slot q + NW - ng of ng groups, so the last slot always holds the last group's;
// the words before the first slot are zero.
template <int NW>
struct ChainShared {
    CellK<float> c;
    alignas(16) float ti[2 * NW];  // totals of the row sums, after NW zero words
    alignas(16) float tj[2 * NW];  // totals of row i
    alignas(16) float ys[32];      // the clock warp's partial sums of the new row
    alignas(16) Draw<float> ring[64];  // this block of 32 events' draws and the next one's
    double tn;                     // the clock after this event
    alignas(8) float2 at;          // a choice: the prefix below the bracketing group, and that group (as an int)
    alignas(8) int2 sel;           // x: i, -2 at the end; y: the fresh R_i of the last event's swarm (as a float)
    alignas(8) int2 pick;          // x: which of the ready outcomes (-1: no partner bracketed, -2: the end), y: the event crosses t_end
    int none;                      // MB > 1: the first waiting time is beyond t_end
    int ticket;                    // persistent CTAs: the queue entry taken
};

// the balanced sum of x, pairs counted from the last word down: ((x7 + x6) +
// (x5 + x4)) + ((x3 + x2) + (x1 + x0))
template <int NW>
__device__ __forceinline__ float tree_down(const float (&x)[NW])
{
    float s[NW];
#pragma unroll
    for (int q = 0; q < NW; ++q) s[q] = x[NW - 1 - q];
#pragma unroll
    for (int o = 1; o < NW; o *= 2)
#pragma unroll
        for (int q = 0; q < NW; q += 2 * o) s[q] += s[q + o];
    return s[0];
}

template <int NW>
__device__ __forceinline__ void load_words(const float *p, float (&x)[NW])  // p 16-byte aligned
{
#pragma unroll
    for (int q = 0; q < NW; q += 4) {
        const float4 v = *reinterpret_cast<const float4 *>(p + q);
        x[q] = v.x, x[q + 1] = v.y, x[q + 2] = v.z, x[q + 3] = v.w;
    }
}

// Choose element k with probability x_k / total from the posted prefixes: the
// first k whose inclusive prefix exceeds target = u * total (pf[k]: element k's
// prefix within its group of 32; t: the ng groups' totals).  Rp is element
// pend's value on top of its x (0); pend < 0 has Rp = 0.  Lane s forms slot s's
// inclusive prefix as a balanced sum over the slots below it (zero words stand
// for the absent ones): the sums that a Kogge-Stone scan over the groups forms,
// bit for bit.  The slot that brackets the target posts itself and what lies
// below it; then every lane tests its element of that group.  True in the one
// lane whose element k is chosen; false everywhere if nothing brackets the
// target (any false: sums that are not finite).  load(k) runs for every lane's
// k of the group as soon as the group is known, so that its loads overlap.
template <int NW, class F>
__device__ __forceinline__ bool choose(const float *t, const float *pf, float2 &at, float u, int pend, float Rp,
                                       int ng, int n, float &total, bool &any, int &k, F load)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, ls = lane & (NW - 1), first = NW - ng;
    float all[NW], mine[NW];
    load_words<NW>(t + NW, all);
    const float *const tl = t + 1 + ls;
#pragma unroll
    for (int q = 0; q < NW; ++q) mine[q] = tl[q];
    const float bs = tree_down<NW>(mine);
    const float below = __shfl_up_sync(FULL, bs, 1);
    const float tot = tree_down<NW>(all) + Rp;
    total = tot;
    float target = u * tot;
    if (target >= tot) target = tot * (float)(1.0 - 1e-7);
    const int g = ls - first;  // the group of this lane's slot
    const float hi = bs + ((pend >= 0 && g >= (pend >> 5)) ? Rp : 0.0f);
    const bool mine_in = target < hi && lane >= first && lane < NW;
    const unsigned in = __ballot_sync(FULL, mine_in);
    if (mine_in && (in & ((1u << lane) - 1u)) == 0u) at = make_float2(g > 0 ? below : 0.0f, __int_as_float(g));
    __syncwarp();
    any = in != 0u;
    const float2 a = at;
    const int q = any ? __float_as_int(a.y) : 0;
    const int kk = 32 * q + lane;
    k = min(kk, n - 1);
    const float wi = pf[kk];
    load(k);
    const float P = (a.x + wi) + ((pend >= 0 && kk >= pend) ? Rp : 0.0f);
    const bool over = P > target;
    const unsigned bal = __ballot_sync(FULL, over);
    // (a tree scan may leave lane 31's prefix an ulp below hi: then lane 31)
    return any && (bal & ((1u << lane) - 1u)) == 0u && (over || lane == 31);
}

// the random numbers of 32 events (lane l: event first + l), one Philox round
// at a time
struct PhiloxRounds {
    uint64_t c0, c1, c2, c3, k0, k1;
    __device__ __forceinline__ void start(uint64_t ev, uint64_t cell, uint64_t step, uint64_t seed, uint64_t disk)
    {
        c0 = ev, c1 = cell, c2 = step, c3 = kTagCollide, k0 = seed, k1 = disk;
    }
    __device__ __forceinline__ void round()
    {
        uint64_t h0, l0, h1, l1;
        mulhilo(kPhiloxM0, c0, h0, l0);
        mulhilo(kPhiloxM1, c2, h1, l1);
        const uint64_t n0 = h1 ^ c1 ^ k0, n2 = h0 ^ c3 ^ k1;
        c0 = n0, c1 = l1, c2 = n2, c3 = l0;
        k0 += kPhiloxW0, k1 += kPhiloxW1;
    }
    __device__ __forceinline__ U4 words() const { return U4{{c0, c1, c2, c3}}; }
    __device__ __forceinline__ Draw<float> draw(float sc) const { return make_draw(U4{{c0, c1, c2, c3}}, sc); }
};

// reciprocal and inverse square root through the special-function unit,
// flush-to-zero forms: the same bits as fdiv's reciprocal and rsqrtf for normal
// operands and results, without the rescaling code around them
__device__ __forceinline__ float rcp_ftz(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rsqrt_ftz(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

constexpr int kFlRenewed = 16;  // in Part<float>::fl: a cache formed by an event of this chain

// make_part<float> with every rounding explicit, so that the mass warp, the
// choice warp and the first build form the same bits
template <bool SEL>
__device__ __forceinline__ Part<float> make_part_rn(const CellK<float> &c, double m, float Mv, int renewed)
{
    Part<float> q;
    float mh, ml;
    split_f64(m, mh, ml);
    q.mh = mh;
    q.ml = ml;
    q.im = rcp_ftz(mh);
    q.Mv = Mv;
    q.gi = c.dm_t > 0.0f ? rcp_ftz(__fmul_rn(c.dm_t, mh)) : INFINITY;
    if (!SEL && c.kmode == 1) {  // the constant kernel: rates and outcomes take masses alone
        q.a = q.S = q.Sl = q.p = q.q = q.ad = 0.0f;
        q.fl = renewed;
        return q;
    }
    const bool stk = !pair_lt(mh, ml, c.msw_h, c.msw_l);
    const int cls = pair_lt(mh, ml, c.meta_h, c.meta_l) ? 0 : (pair_lt(mh, ml, c.mone_h, c.mone_l) ? 1 : 2);
    // x = cm m as a (hi, lo) pair, then a = cbrt(x) to about 2^-44: FP32 cube
    // root plus one Newton step on the residual x - a0^3 taken exactly
    const float xh = __fmul_rn(c.cm, mh);
    const float xl = __fmaf_rn(c.cm_lo, mh, __fmaf_rn(c.cm, ml, __fmaf_rn(c.cm, mh, -xh)));
    const float l3 = __fmul_rn(lg2_mufu(xh), 1.0f / 3.0f);
    const float a0 = ex2_mufu(l3), ia = ex2_mufu(-l3);  // ia: 1/a0 to a few ulp
    const float p2 = __fmul_rn(a0, a0), p2e = __fmaf_rn(a0, a0, -p2);  // a0^2 = p2 + p2e
    const float p3 = __fmul_rn(p2, a0), p3e = __fmaf_rn(p2, a0, -p3);  // p2 a0 = p3 + p3e
    const float res = __fadd_rn(__fmaf_rn(-p2e, a0, __fsub_rn(__fsub_rn(xh, p3), p3e)), xl);  // x - a0^3
    const float alo = __fmul_rn(res, __fmul_rn(__fmul_rn(ia, ia), 1.0f / 3.0f));
    q.a = a0;
    // S = Cst a^2 = Cst (p2 + p2e + 2 a0 alo) for Stokes drag, Cep a otherwise
    const float C = stk ? c.Cst : c.Cep, Cl = stk ? c.Cst_lo : c.Cep_lo, y = stk ? p2 : a0;
    const float yl = stk ? __fmaf_rn(__fmul_rn(2.0f, a0), alo, p2e) : alo;
    const float Sh = __fmul_rn(C, y);
    const float Se = __fmaf_rn(Cl, y, __fmaf_rn(C, yl, __fmaf_rn(C, y, -Sh)));
    q.S = __fadd_rn(Sh, Se);
    q.Sl = __fsub_rn(Se, __fsub_rn(q.S, Sh));
    q.p = rcp_ftz(__fmaf_rn(q.S, q.S, 1.0f));
    q.q = rcp_ftz(__fadd_rn(1.0f, q.S));
    // a - a_sw = cm (m - m_sw) / (a^2 + a a_sw + a_sw^2), m - m_sw from the pairs
    const float dsw = __fadd_rn(__fsub_rn(mh, c.msw_h), __fsub_rn(ml, c.msw_l));
    q.ad = stk ? __fmul_rn(__fmul_rn(c.cm, dsw), rcp_ftz(__fmaf_rn(a0, c.asw, __fmaf_rn(c.asw, c.asw, p2)))) : 0.0f;
    q.fl = cls | ((int)stk << 2) | renewed;
    return q;
}

// pair_dv<float> of N pairs (u, v) without a branch but the constant kernel's (the
// same for the whole cell; with every term formed for it too a 0D cell of 400 swarms
// took 6.1 ms to t = 100, now 3.9): every other case evaluated and selected, step by
// step for all N, so that the pairs fill each other's latencies.  Every rounding is explicit, so the bits depend
// neither on the store nor on the warp that forms them; they are pair_dv's,
// except that dv below 1e-19 cm/s (dv^2 no normal number) counts as 0.  EARLY:
// with early set, a pair of two swarms that no event of this chain has renewed
// takes the drift and settling terms' sum with the other product fused.  Neither
// rounding is the better one: it is kept so that runs of classes whose matrix fits
// into shared memory (up to 318 swarms) give the bits they always gave.
// COMMON (the first row sums, where a whole warp agrees): no v is a Stokes-law swarm,
// no pair in turbulence regime I and no swarm renewed, so a fifth of the terms is left out.
// SEL: the constant kernel is selected at the end, not branched to (MB > 1: the branch
// costs the event loop 4 % where registers are short; 64 swarms, 1 yr: 2.90 and 3.01 ms).
template <int N, bool EARLY, bool COMMON = false, bool SEL = false>
__device__ __forceinline__ void pair_flat(const PairK<float> &c, bool early, const Part<float> (&u)[N],
                                          const Part<float> (&v)[N], float (&dv)[N], float (&K)[N])
{
    typedef float T;
    T da[N], D[N], S1[N], S2[N], s[N], g1[N], t2[N], t3[N], coef[N], t0[N];
#define MCD_EACH _Pragma("unroll") for (int x = 0; x < N; ++x)
    if (!SEL && c.kmode == 1) {
        MCD_EACH dv[x] = (T)0, K[x] = c.Kc;
        return;
    }
    MCD_EACH
    {
        const T dm = fabsf(__fadd_rn(__fsub_rn(u[x].mh, v[x].mh), __fsub_rn(u[x].ml, v[x].ml)));
        const T den = __fmaf_rn(u[x].a, v[x].a, __fadd_rn(__fmul_rn(u[x].a, u[x].a), __fmul_rn(v[x].a, v[x].a)));
        da[x] = __fmul_rn(__fmul_rn(c.cm, dm), rcp_ftz(den));
    }
    MCD_EACH
    {
        S1[x] = fmaxf(u[x].S, v[x].S), S2[x] = fminf(u[x].S, v[x].S);
        s[x] = __fadd_rn(S1[x], S2[x]);
        if (!COMMON)
            g1[x] = __fmul_rn(__fmul_rn(c.vg2, __fmaf_rn(S1[x], S2[x], __fmul_rn(c.Se, s[x]))),
                              rcp_ftz(__fmul_rn(__fmul_rn(s[x], __fadd_rn(S1[x], c.Se)), __fadd_rn(S2[x], c.Se))));
    }
    MCD_EACH
    {
        const T A1 = __fmaf_rn((T)kYA, S1[x], S2[x]);
        const T num = __fmaf_rn(__fmul_rn(A1, __fmul_rn(S1[x], S1[x])), (T)(1.0 / (1.0 + kYA)),
                                __fmul_rn(__fmul_rn(S2[x], S2[x]), S2[x]));
        t2[x] = __fmul_rn(c.vg2, __fmaf_rn(__fmul_rn(2.0f, num), rcp_ftz(__fmul_rn(s[x], A1)),
                                           __fmaf_rn((T)(2.0 * kYA - 1.0), S1[x], -S2[x])));
        t3[x] = __fmul_rn(c.vg2, __fadd_rn(u[x].q, v[x].q));
    }
    MCD_EACH
    {
        const bool su = u[x].fl & 4, sv = !COMMON && (v[x].fl & 4);
        const T as = su || COMMON ? u[x].a : v[x].a, ads = su || COMMON ? u[x].ad : v[x].ad;
        const T D_st = __fmul_rn(__fmul_rn(c.Cst, __fadd_rn(u[x].a, v[x].a)), da[x]);
        const T D_mx = __fmul_rn(c.Cst, __fmaf_rn(as, ads, __fmul_rn(c.asw, da[x]))), D_ep = __fmul_rn(c.Cep, da[x]);
        D[x] = (su && sv) ? D_st : ((su || sv) ? D_mx : D_ep);
    }
    MCD_EACH
    {
        const int cls = max(u[x].fl & 3, v[x].fl & 3);
        const T pp = __fmul_rn(u[x].p, v[x].p);
        const T om = __fsub_rn(__fmaf_rn(-u[x].S, v[x].S, 1.0f),
                               __fadd_rn(__fmul_rn(u[x].S, v[x].Sl), __fmul_rn(u[x].Sl, v[x].S)));
        const T qv = __fmul_rn(u[x].q, v[x].q), qq = c.settle ? __fmul_rn(qv, qv) : 1.0f;
        const T Y = __fmaf_rn(__fmul_rn(c.e1, s[x]), s[x], __fmul_rn(__fmul_rn(c.e4, om), om)), pp2 = __fmul_rn(pp, pp);
        T Z = __fmaf_rn(c.oz2, qq, __fmul_rn(pp2, Y));
        if (EARLY && early && (COMMON || !((u[x].fl | v[x].fl) & kFlRenewed))) Z = __fmaf_rn(pp2, Y, __fmul_rn(c.oz2, qq));
        coef[x] = COMMON ? Z : __fadd_rn(Z, (cls == 0 && s[x] > 0.0f) ? g1[x] : 0.0f);
        t0[x] = __fmaf_rn(c.cbm, __fadd_rn(u[x].im, v[x].im), cls == 1 ? t2[x] : (cls == 2 ? t3[x] : 0.0f));
    }
    MCD_EACH
    {
        const T dv2 = __fmaf_rn(__fmul_rn(D[x], D[x]), coef[x], t0[x]);
        dv[x] = dv2 >= FLT_MIN ? __fmul_rn(dv2, rsqrt_ftz(dv2)) : 0.0f;
    }
    MCD_EACH
    {
        const T s2 = __fadd_rn(u[x].a, v[x].a);
        K[x] = __fmul_rn(__fmul_rn(__fmul_rn(c.pi, s2), s2), dv[x]);
        if (SEL) K[x] = c.kmode == 1 ? c.Kc : K[x], dv[x] = c.kmode == 1 ? 0.0f : dv[x];
    }
#undef MCD_EACH
}
template <bool EARLY, bool SEL = false>
__device__ __forceinline__ void pair_flat1(const PairK<float> &c, bool early, const Part<float> &u,
                                           const Part<float> &v, float &dv, float &K)
{
    const Part<float> uu[1] = {u}, vv[1] = {v};
    float d[1], k[1];
    pair_flat<1, EARLY, false, SEL>(c, early, uu, vv, d, k);
    dv = d[0];
    K = k[0];
}

// slots for the groups' totals of a chain launch with nsl swarm slots
inline int chain_slots(int nsl) { return nsl <= 128 ? 4 : (nsl <= 256 ? 8 : 16); }

// dynamic shared memory of a chain CTA with nsl swarm slots: caches, ready
// outcomes (two caches and masses per swarm and one place for a general
// outcome), masses with dm m, the tracer copy, the scans' rows, the posted new
// row, the prefixes, dv of row i, and the stored matrix (STORE == 1)
inline size_t collide_chain_smem_bytes(int nsl, bool tracer, int store, int rows, int W)
{
    size_t b = (size_t)nsl * (3 * sizeof(Part<float>) + 6 * sizeof(double) + (tracer ? sizeof(double) : 0) +
                              6 * sizeof(float)) +
               sizeof(Part<float>) + sizeof(double2) + 32 * chain_slots(nsl) * sizeof(float);
    if (store == 1) b += (size_t)rows * W * sizeof(float);
    return b;
}

// warps that share the first row sums of a chain launch without a stored matrix: a
// multiple of four, one sub-partition's worth over that would wait for the others
__host__ __device__ inline int chain_build_warps(int nsl) { return (nsl / 32 + kChainRoles) & ~3; }

// a swarm's cache or another's, field by field (no branch)
__device__ __forceinline__ Part<float> part_select(bool other, const Part<float> &o, const Part<float> &p)
{
    Part<float> r;
    r.a = other ? o.a : p.a, r.im = other ? o.im : p.im, r.Mv = p.Mv, r.gi = other ? o.gi : p.gi;
    r.S = other ? o.S : p.S, r.Sl = other ? o.Sl : p.Sl, r.p = other ? o.p : p.p, r.q = other ? o.q : p.q;
    r.mh = other ? o.mh : p.mh, r.ml = other ? o.ml : p.ml, r.ad = other ? o.ad : p.ad;
    r.fl = other ? o.fl : p.fl;
    return r;
}

// the outcomes of mass m that do not depend on the partner: a grouped partner
// of total mass dmm = dm m sticks, or erodes
template <class T>
__device__ __forceinline__ double ready_mass(const CellK<T> &c, double m, double dmm, bool erodes)
{
    if (!erodes) return m + dmm;
    const double me = m - c.chi * dmm;
    return dgt(me, c.m0) ? me : c.m0;
}

// inclusive prefix of x within the warp's group of 32, the sums of a
// Kogge-Stone scan bit for bit, by two exchanges through shared memory: four
// neighbours, then the sums of four at a stride of four.  xs: the group's rows
// (two of 64 words, the first 32 words of each zero)
__device__ __forceinline__ float group_prefix(float *xs, float x)
{
    const int lane = threadIdx.x & 31;
    float *const p = xs + 32 + lane, *const q = xs + 96 + lane;
    *p = x;
    __syncwarp();
    const float s4 = __fadd_rn(__fadd_rn(x, p[-1]), __fadd_rn(p[-2], p[-3]));
    *q = s4;
    __syncwarp();
    return __fadd_rn(__fadd_rn(__fadd_rn(s4, q[-4]), __fadd_rn(q[-8], q[-12])),
                     __fadd_rn(__fadd_rn(q[-16], q[-20]), __fadd_rn(q[-24], q[-28])));
}

// Cells of up to 64 swarms run several CTAs per SM: when the number was chosen,
// 32,768 light cells of 40 (64) swarms took 0.81 (1.26) ms with five (now 0.78, 1.14),
// 1.45 (1.92) ms with the two that fit without a register limit, while a heavy cell's
// event took 0.88 us against 0.80; seven spill (1.29 us), six too (48 swarms, 1 yr: 3.63
// ms against 3.03).
constexpr int kChainSmallCtas = 5;

// MB: resident CTAs per SM (cells of up to 64 swarms: many light cells run at
// once).  STORE, RAMP, TRACER as in cell_chain
template <int NW, int MB, int STORE, bool RAMP, bool TRACER>
__device__ __forceinline__ void chain_cell(const CollideArgs &A, const int64_t cell, const int64_t entry,
                                           ChainShared<NW> &sh, unsigned char *smem_raw)
{
    typedef float T;
    // the row sums a ready outcome leads to are formed ahead too, where the instructions fit
    // into the time that the choice of j takes
    constexpr bool AHEAD = NW <= 8 && MB == 1;
    constexpr int RW = 32 * NW;              // words of the posted new row
    const int nthr = blockDim.x, nsl = nthr - 32 * kChainRoles, ng = nsl >> 5;  // swarm slots (workers), groups
    Part<T> *parts = reinterpret_cast<Part<T> *>(smem_raw);
    Part<T> *ready = parts + nsl;  // [2][nsl]: grouped partner sticks, erodes; then a general outcome
    double2 *mm = reinterpret_cast<double2 *>(ready + 2 * nsl + 1);  // mass, dm m
    double2 *mready = mm + nsl;                                      // the same of ready
    double *qsh = reinterpret_cast<double *>(mready + 2 * nsl + 1);  // TRACER
    T *rn = reinterpret_cast<T *>(qsh + (TRACER ? nsl : 0));         // the last event's new row (zero beyond nsl)
    T *xs = rn + RW;                                                 // the scans' rows
    T *pf = xs + 4 * nsl;                                            // prefixes within the groups
    T *dvrow = pf + nsl;                                             // dv of row i
    T *Dm = dvrow + nsl;                                             // STORE == 1 (0: the first build's columns)
    const int W = A.dv_w;
    if constexpr (STORE == 2) Dm = reinterpret_cast<T *>(A.dvg) + (size_t)entry * A.dv_rows * W;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int n = A.cell_n[cell];
    if (n <= 0) {
        if (tid == 0) A.cell_events[cell] = 0;
        return;
    }
    if (n > nsl || (STORE && (n > A.dv_rows || n / 2 >= W))) {
        if (tid == 0) atomicOr(A.status, kStBadCell);
        return;
    }
    const int disk = A.cell_disk[cell];
    const int64_t off = A.cell_start[cell];
    {
        static_assert(sizeof(CellK<T>) % 4 == 0, "copied by words");
        const uint32_t *src = reinterpret_cast<const uint32_t *>(A.cellk + cell * kCellKBytes);
        for (int q = tid; q < (int)(sizeof(CellK<T>) / 4); q += nthr) reinterpret_cast<uint32_t *>(&sh.c)[q] = src[q];
    }
    if (tid < 2 * NW) sh.ti[tid] = sh.tj[tid] = 0.0f;
    for (int q = tid; q < RW + 4 * nsl; q += nthr) rn[q] = 0.0f;  // (and the scans' rows)
    __syncthreads();
    const CellK<T> &c = sh.c;
    const PairK<T> pc = pair_consts<T>(sh.c);
    const int k = tid;  // a worker's swarm
    const bool act = k < n;
    Part<T> pk;
    // the random stream is keyed by (seed, disk) and counted by
    // (event, disk-local cell, step, domain tag)
    const uint64_t dcell = (uint64_t)(cell - A.disks[disk].c_off);
    const uint64_t step = (uint64_t)A.state->step;
    const T sc = (T)c.sc;
    if (w == ng) {
        sh.ring[lane] = make_draw(philox((uint64_t)lane, dcell, step, kTagCollide, A.seed, (uint64_t)disk), sc);
    } else if (w < ng) {
        const int kc = act ? k : n - 1;
        const double mk = A.m[off + kc];
        // every mass the event loop can reach lies between the monomer mass and
        // the disk's dust mass, inside the split's range
        if (!mass_splits(mk)) atomicOr(A.status, kStBadCell);
        pk = make_part_rn<(MB > 1)>(c, mk, (T)(A.M[off + kc] * c.invVsc), 0);
        const double dmm = __dmul_rn(c.dm, mk);
        if (act) {
            mm[k] = make_double2(mk, dmm);
            if (TRACER) qsh[k] = A.q[off + k];
            parts[k] = pk;
        }
    }
    __syncthreads();

    const int reb = (int)(A.rebuild_every > 0 ? (A.rebuild_every < 0x7fffffff ? A.rebuild_every : 0x7fffffff)
                                              : 4 * (int64_t)n);
    int until_rebuild = reb;  // events left before the next full rebuild
    int64_t ev = 0;

    const bool early = A.early != 0;
    T *const xw = xs + 128 * w;
    Acc<T> R;
    R.zero();
    // row sums R_k += r_kj in j order, two at a time: from the stored matrix, from
    // columns formed by the warps that own no swarm, or from fresh entries (the same bits)
    auto add_stored = [&](int j0, int j1) {
        const int kc = act ? k : n - 1;
#pragma unroll 4
        for (int j = j0; j < j1; ++j) {
            const Part<T> pj = parts[j];
            const T dv = STORE != 0 ? Dm[sym_at(kc, j, n, W)] : Dm[(j - j0) * nsl + k];
            R.add(kern_of<T>(pc, pk.a, pj.a, dv) * weight<T>(pk, pj));
        }
    };
    auto fresh2 = [&](const Part<T> (&u)[2], const Part<T> (&o)[2], T (&dv)[2], T (&K)[2], bool first) {
        const int fl = min(o[0].fl & 3, o[1].fl & 3);
        if (first && fl && !((o[0].fl | o[1].fl) & 4))
            pair_flat<2, true, true>(pc, early, u, o, dv, K);
        else
            pair_flat<2, true>(pc, early, u, o, dv, K);
    };
    auto add_fresh = [&](int j0, int j1, bool first) {
        const Part<T> u[2] = {pk, pk};
        for (int j = j0; j < j1; j += 2) {
            const Part<T> o[2] = {parts[j], parts[min(j + 1, n - 1)]};
            T dv[2], K[2];
            fresh2(u, o, dv, K, first);
            R.add(K[0] * weight<T>(pk, o[0]));
            if (j + 1 < j1) R.add(K[1] * weight<T>(pk, o[1]));
        }
    };
    const bool swarms = 32 * w < n;  // (a worker warp with swarms)
    if constexpr (STORE != 0) {
        // every unordered pair once, in row order over all the CTA's threads (a row of a
        // small cell fills no warp), two at a time: pair t is offset t mod L of row t / L,
        // and the pairs half an even cell apart follow
        const int L = (n - 1) / 2 + 1, half = (n & 1) ? 0 : n / 2, pairs = n * L + half;
        const int step_r = nthr / L, step_d = nthr - step_r * L;
        int rr = tid / L, d = tid - rr * L, t = tid;
        if constexpr (MB > 1) {  // one at a time: two would spill registers
            for (; t < pairs; t += nthr) {
                const int row = t < n * L ? rr : t - n * L, o = t < n * L ? d : half;
                int j = row + o;
                if (j >= n) j -= n;
                T dv, K;
                pair_flat1<true, true>(pc, early, parts[row], parts[j], dv, K);
                Dm[row * W + o] = dv;
                rr += step_r, d += step_d;
                if (d >= L) d -= L, ++rr;
            }
        } else {
            while (t - lane < pairs) {  // (whole warps: they vote)
                int row[2], other[2], at2[2];
                bool in[2];
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    in[x] = t < pairs;
                    row[x] = !in[x] ? 0 : (t < n * L ? rr : t - n * L);
                    const int o = !in[x] ? 0 : (t < n * L ? d : half);
                    at2[x] = row[x] * W + o;
                    other[x] = row[x] + o;
                    if (other[x] >= n) other[x] -= n;
                    t += nthr, rr += step_r, d += step_d;
                    if (d >= L) d -= L, ++rr;
                }
                const Part<T> pr[2] = {parts[row[0]], parts[row[1]]}, pj[2] = {parts[other[0]], parts[other[1]]};
                T dv[2], K[2];
                const int cls = min(max(pr[0].fl & 3, pj[0].fl & 3), max(pr[1].fl & 3, pj[1].fl & 3));
                if (__all_sync(0xffffffffu, cls && !((pj[0].fl | pj[1].fl) & 4)))
                    pair_flat<2, true, true>(pc, early, pr, pj, dv, K);
                else
                    pair_flat<2, true>(pc, early, pr, pj, dv, K);
                if (in[0]) Dm[at2[0]] = dv[0];
                if (in[1]) Dm[at2[1]] = dv[1];
            }
        }
        __syncthreads();
        if (swarms) add_stored(0, n);
    } else {
        // the last columns by the warps without swarms, the others by their owners
        // (as many of them as leave every SM sub-partition the same number of warps).  4,096
        // cells of 300 swarms, collide of a 0.1-yr step: 2,004 -> 1,772 us, of 400: 3,187 ->
        // 2,650, with the terms that COMMON leaves out (the block kernel's shared half
        // matrix: 1,789; 400 swarms recomputing: 3,210).
        const int warps = chain_build_warps(nsl), busy = (n + 31) >> 5, idle = max(warps - busy, 0);
        const int cols = min(A.cols, n * idle / warps) & ~1, j0 = n - cols;
        if (swarms) {
            add_fresh(0, j0, true);
        } else if (w - busy < idle) {
            for (int j = j0 + 2 * (w - busy); j < n; j += 2 * idle) {
                const Part<T> o[2] = {parts[j], parts[j + 1]};
                for (int q = lane; q < 32 * busy; q += 32) {
                    const Part<T> u[2] = {parts[min(q, n - 1)], parts[min(q, n - 1)]};
                    T dv[2], K[2];
                    fresh2(u, o, dv, K, true);
                    Dm[(j - j0) * nsl + q] = dv[0];
                    Dm[(j + 1 - j0) * nsl + q] = dv[1];
                }
            }
        }
        __syncthreads();
        if (swarms) add_stored(j0, n);
    }
    T hi = act ? (T)R.hi() : (T)0;  // R_k for the next choice
    if constexpr (MB > 1) {
        if (w < ng) pf[k] = R.s, dvrow[k] = R.c;  // (kept there until the event loop: registers)
        // The first waiting time: most of many light cells have no event in a short step,
        // and need neither ready outcomes nor choices.  Collide of 32,768 cells of 32
        // swarms, with the pairs above in row order and R_k parked: a 0.001-yr step (no
        // events) 485 -> 260 us, a 0.1-yr one 557 -> 336, a 1-yr one 1,726 -> 1,620
        // (block-wide scans: 293, 342, 2,103).  In the one-CTA kernels the ready outcomes
        // are 3 % of a cell, and the branch costs the event loop as much.
        if (w < ng) {
            const T x = group_prefix(xw, hi);
            if (lane == 31) sh.ti[2 * NW - ng + w] = x;
        }
        __syncthreads();
        if (w == ng + 1) {
            T all[NW];
            load_words<NW>(sh.ti + NW, all);
            const T tot = tree_down<NW>(all);
            const double t_end = A.t_end_from_state ? A.state->t + A.state->dt : A.t_end_fixed;
            const bool none = tot > (T)0 && A.max_events > 0 && A.state->t + (double)fdiv(sh.ring[0].L, tot) >= t_end;
            if (lane == 0) {
                sh.none = none;
                if (none) {
                    A.cell_events[cell] = 0;
                    if (cell == A.log_cell) *A.log_n = 0;
                    if (A.Rtot) A.Rtot[cell] = (double)tot / c.sc;
                }
            }
        }
        __syncthreads();
        if (sh.none) {
            if (act && A.Rdump) A.Rdump[off + k] = R.value() / c.sc;
            return;
        }
    }
    if (w < ng) {
        const double2 mk = mm[act ? k : n - 1];
        for (int e = 0; e < 2; ++e) {
            const double mr = ready_mass(c, mk.x, mk.y, e != 0);
            const Part<T> pr = make_part_rn<(MB > 1)>(c, mr, pk.Mv, kFlRenewed);
            if (act) {
                ready[e * nsl + k] = pr;
                mready[e * nsl + k] = make_double2(mr, __dmul_rn(c.dm, mr));
            }
        }
    }

    if (w == ng) {  // ---- the choice warp ----
        const bool logging = (cell == A.log_cell);
        const bool group = c.dm > 0.0;
        // a grouped partner is lighter than dm m_i: with ratio dm well below 1 it is
        // also lighter than m_i / ratio, and the event erodes when it does not stick
        const bool eroding = c.dm < 1.0 && c.ratio * c.dm <= 0.5;
        const int gen = 2 * nsl;  // a general outcome's place among the ready ones
        int pend = -1;            // swarm whose fresh row sum rides on the next choice
        T vlo = (T)0, tot, tot2;
        int64_t left = A.max_events;  // events before the cap
        if constexpr (RAMP) {  // the ramp's foot as the plain FP64 evaluation forms it
            const mcd_disk_params &P = A.params[disk];
            vlo = (T)(P.v_frag * (1.0 - P.frag_ramp));
        }
        for (;;) {
            const Draw<T> dr = sh.ring[ev & 63];
            int i, j;
            bool any;
            bar_sync(kBarRates, nsl + 96);
            const T Rp = __int_as_float(sh.sel.y);
            const bool ihere = choose<NW>(sh.ti, pf, sh.at, dr.u1, pend, Rp, ng, n, tot, any, i, [](int) {});
            if (!(tot > (T)0) || left <= 0) {  // (uniform)
                if (lane == 0) {
                    if (left <= 0 && tot > (T)0 && !A.cap_stops) atomicOr(A.status, kStTimeout);
                    sh.pick.x = -2;
                    sh.sel.x = -2;
                }
                bar_arrive(kBarI, nsl + 32);
                bar_sync(kBarEvent, nthr);
                break;
            }
            if (any ? ihere : lane == 0) sh.sel.x = any ? i : n - 1;  // (no bracket, rates not finite: stay in bounds)
            bar_arrive(kBarI, nsl + 32);
            i = sh.sel.x;
            const double2 mmi = mm[i];
            const T Mvi = parts[i].Mv, mih = parts[i].mh;
            double mj, mst;
            T dvij;
            bar_sync(kBarRow, nsl + 32);
            const bool jhere = choose<NW>(sh.tj, pf, sh.at, dr.u2, -1, (T)0, ng, n, tot2, any, j, [&](int q) {
                mj = mm[q].x;
                dvij = dvrow[q];
                mst = mmi.x + (dgt(mmi.y, mj) ? mmi.y : mj);  // should it stick (the FP64 latency behind the choice)
            });
            T dvx = dvij;
            if constexpr (RAMP)  // inside the ramp: fragments as at v_frag with the ramp's probability
                if (pc.kmode != 1 && dvx < c.vfrag_t && !(dvx < vlo) && dr.u3 < fdiv(dvx - vlo, c.vfrag_t - vlo))
                    dvx = c.vfrag_t;
            const bool stick = pc.kmode == 1 || dvx < c.vfrag_t;
            const bool grouped = group && dgt(mmi.y, mj) && (stick || eroding);
            int kind = stick ? 0 : 2;
            double mnew = 0.0, qnew = 0.0;
            if (any ? jhere : lane == 0) sh.pick.x = any ? (grouped ? (stick ? i : nsl + i) : gen) : -1;
            if (jhere && (!grouped || TRACER || logging)) {
                if (!grouped) {
                    if (stick)
                        mnew = mst;
                    else if constexpr (RAMP)
                        mnew = outcome_ramp<T>(c, mmi.x, mj, mih, parts[j].mh, mmi.y, dvij, dr.u3, vlo, kind);
                    else
                        mnew = outcome<T>(c, mmi.x, mj, mih, parts[j].mh, mmi.y, dvij, dr.u3, kind);
                    ready[gen] = make_part_rn<(MB > 1)>(c, mnew, Mvi, kFlRenewed);
                    mready[gen] = make_double2(mnew, __dmul_rn(c.dm, mnew));
                } else {
                    mnew = ready_mass(c, mmi.x, mmi.y, !stick);  // (the mass warp may still be at work on mready)
                }
                if constexpr (TRACER)
                    qnew = tracer_update(mmi.x, mj, qsh[i], qsh[j], dgt(mmi.y, mj) ? mmi.y : mj, mnew, kind, c.chi);
            }
            bar_sync(kBarEvent, nthr);
            const int2 pick = sh.pick;
            if (pick.x < 0 || pick.y) {
                // nothing brackets j: the row's prefix sums are not finite
                if (pick.x < 0 && lane == 0) atomicOr(A.status, kStNaN);
                break;
            }
            if (TRACER || logging) {
                if (jhere) {
                    if constexpr (TRACER) qsh[i] = qnew;
                    if (logging && ev < A.log_cap) {
                        A.log_ijo[3 * ev] = i;
                        A.log_ijo[3 * ev + 1] = j;
                        A.log_ijo[3 * ev + 2] = kind;
                        A.log_t[ev] = sh.tn;
                        A.log_m[ev] = mnew;
                    }
                }
            }
            pend = i;
            ++ev;
            --left;
            if (--until_rebuild == 0) {
                pend = -1;
                until_rebuild = reb;
            }
        }
        if (lane == 0) {
            A.cell_events[cell] = ev;
            atomicAdd(&A.events_total[disk], (unsigned long long)ev);
            if (logging) *A.log_n = (unsigned long long)(ev < A.log_cap ? ev : A.log_cap);
            if (A.Rtot) A.Rtot[cell] = (double)tot / c.sc;
        }
        __syncwarp();
    } else if (w == ng + 1) {  // ---- the mass warp ----
        bar_arrive(kBarRates, nsl + 96);
        bar_arrive(kBarReady, nsl + 32);
        for (;;) {
            bar_sync(kBarEvent, nthr);
            const int2 pick = sh.pick;
            if (pick.x < 0 || pick.y) break;
            const int i = sh.sel.x;
            // i's new mass and cache
            if (lane < 3) reinterpret_cast<uint4 *>(parts + i)[lane] = reinterpret_cast<const uint4 *>(ready + pick.x)[lane];
            const T Mvi = ready[pick.x].Mv;
            const double2 mi = mready[pick.x];
            if (lane == 0) mm[i] = mi;
            if (--until_rebuild == 0) {
                bar_arrive(kBarBuild, nsl + 32);
                until_rebuild = reb;
            }
            bar_arrive(kBarRates, nsl + 96);
            // its ready outcomes: even lanes stick, odd lanes erode
            const double mnew = ready_mass(c, mi.x, mi.y, lane & 1), dmnew = __dmul_rn(c.dm, mnew);
            __syncwarp();
            const Part<T> pnew = make_part_rn<(MB > 1)>(c, mnew, Mvi, kFlRenewed);
            bar_sync(kBarRead, nsl + 32);
            if (lane < 2) {
                ready[lane * nsl + i] = pnew;
                mready[lane * nsl + i] = make_double2(mnew, dmnew);
            }
            bar_arrive(kBarReady, nsl + 32);
        }
    } else if (w > ng + 1) {  // ---- the clock warp ----
        const double t_end = A.t_end_from_state ? A.state->t + A.state->dt : A.t_end_fixed;
        double t = A.state->t;
        PhiloxRounds px;
        for (;;) {
            const T L = sh.ring[ev & 63].L;
            bar_sync(kBarNew, nsl + 32);
            T y[RW / 32], z[32], all[NW];
            load_words<RW / 32>(rn + lane * (RW / 32), y);
            sh.ys[lane] = tree_down<RW / 32>(y);
            __syncwarp();
            load_words<32>(sh.ys, z);
            const T Rp = tree_down<32>(z);
            if (lane == 0) sh.sel.y = __float_as_int(Rp);
            bar_sync(kBarRates, nsl + 96);
            load_words<NW>(sh.ti + NW, all);
            const T tot = tree_down<NW>(all) + Rp;
            if (!(tot > (T)0) || ev >= A.max_events) {
                bar_sync(kBarEvent, nthr);
                break;
            }
            t += (double)fdiv(L, tot);
            if (lane == 0) {
                sh.pick.y = t >= t_end;
                sh.tn = t;
            }
            // the next block's draws, one round per event of this block
            const int q = (int)(ev & 31);
            if (q == 0) px.start((uint64_t)((ev | 31) + 1 + lane), dcell, step, A.seed, (uint64_t)disk);
            if (q < 10) px.round();
            if (q == 10) sh.ring[((ev | 31) + 1 + lane) & 63] = px.draw(sc);
            bar_sync(kBarEvent, nthr);
            const int2 pick = sh.pick;
            if (pick.x < 0 || pick.y) break;
            ++ev;
        }
    } else {  // ---- the workers ----
        int pend = -1;  // swarm whose fresh row sum rides on the next choice
        if constexpr (MB > 1) {
            R.s = pf[k], R.c = dvrow[k];
            hi = act ? (T)R.hi() : (T)0;
        }
        bar_arrive(kBarNew, nsl + 32);
        int guess = 0;  // the kind of ready outcome that came last
        // hi is 0 for the swarm whose fresh sum rides on the next choice; what is put off
        // until the choice is under way: the event's entry of the
        // matrix, the updated R_k, and (took) the swarm's own new cache
        T dvn = (T)0;
        Acc<T> Rn = R;
        Part<T> us = pk;
        bool upd = false, took = false;
        int at = 0;
        for (;;) {
            // (1) row sums for the choice of i: the previous event's R_i (the sum of
            //     its new row) is folded in there
            T x = group_prefix(xw, hi);
            pf[k] = x;
            if (lane == 31) sh.ti[2 * NW - ng + w] = x;
            if (STORE != 0 && act && pend >= 0) Dm[at] = dvn;
            bar_arrive(kBarRates, nsl + 96);
            R.s = upd ? Rn.s : R.s;
            R.c = upd ? Rn.c : R.c;
            if (took) pk = us;  // (uniform)
            bar_sync(kBarI, nsl + 32);
            const int2 sel = sh.sel;
            const int i = max(sel.x, 0);
            // (2) row i (i meets k) and column i (k meets i) before the event
            const Part<T> pi = parts[i];
            at = STORE != 0 ? sym_at(i, act ? k : n - 1, n, W) : 0;
            T dvik, Kold;
            if constexpr (STORE != 0) {
                dvik = Dm[at];
                Kold = kern_of<T>(pc, pk.a, pi.a, dvik);
            } else {
                pair_flat1<true, (MB > 1)>(pc, early, pk, pi, dvik, Kold);
            }
            R.s = k == pend ? __int_as_float(sel.y) : R.s;
            R.c = k == pend ? (T)0 : R.c;
            if (sel.x < 0) {
                bar_sync(kBarReady, nsl + 32);
                bar_sync(kBarEvent, nthr);
                break;
            }
            dvrow[k] = dvik;
            x = group_prefix(xw, act ? Kold * weight<T>(pi, pk) : (T)0);
            pf[k] = x;
            if (lane == 31) sh.tj[2 * NW - ng + w] = x;
            bar_arrive(kBarRow, nsl + 32);
            const T colo = Kold * weight<T>(pk, pi);
            // (3) meanwhile, for the ready outcome of the kind that came last: the new
            //     row and column i, and the row sum they lead to
            //     (R_k += r_ki(new) - r_ki(old))
            bar_sync(kBarReady, nsl + 32);
            upd = act && k != i;
            const Part<T> o = ready[guess * nsl + i];
            us = part_select(k == i, o, pk);
            T dvs, Ks, rows, his;
            Acc<T> Rs;
            pair_flat1<false, (MB > 1)>(pc, false, us, o, dvs, Ks);
            // (here, not where they are used: the compiler would sink them behind the barrier)
            asm volatile("" : "+f"(Ks), "+f"(dvs));
            if constexpr (AHEAD) {
                rows = act ? Ks * weight<T>(o, us) : (T)0;
                Rs = R;
                Rs.update(Ks * weight<T>(us, o), colo);
                his = upd ? (T)Rs.hi() : (T)0;
                asm volatile("" : "+f"(rows), "+f"(his), "+f"(Rs.s), "+f"(Rs.c));
            }
            bar_sync(kBarEvent, nthr);
            const int2 pick = sh.pick;
            if (pick.x < 0 || pick.y) break;
            // (4) the outcome's new row and column i: taken over, or formed now; R_i afresh
            const bool rebuild = --until_rebuild == 0;
            const bool hit = pick.x == guess * nsl + i;
            took = AHEAD && hit;
            dvn = dvs;
            if (AHEAD && hit) {
                hi = his;
                rn[k] = rebuild ? (T)0 : rows;
                bar_arrive(kBarNew, nsl + 32);
                Rn = Rs;
            } else {
                const Part<T> pn = ready[pick.x];
                T Knew = Ks;
                pk = part_select(k == i, pn, pk);
                if (!hit) pair_flat1<false, (MB > 1)>(pc, false, pk, pn, dvn, Knew);
                rn[k] = act && !rebuild ? Knew * weight<T>(pn, pk) : (T)0;
                bar_arrive(kBarNew, nsl + 32);
                Rn = R;
                Rn.update(Knew * weight<T>(pk, pn), colo);
                hi = upd ? (T)Rn.hi() : (T)0;
                guess = pick.x < nsl ? 0 : (pick.x < 2 * nsl ? 1 : guess);
            }
            bar_arrive(kBarRead, nsl + 32);
            pend = i;
            if (rebuild) {
                if (took) pk = us;
                took = false;
                if (STORE != 0 && act) Dm[at] = dvn;
                bar_sync(kBarBuild, nsl + 32);
                R.zero();
                if (swarms && STORE != 0) add_stored(0, n);
                if (swarms && STORE == 0) add_fresh(0, n, false);
                Rn = R;
                pend = -1;
                until_rebuild = reb;
                hi = act ? (T)R.hi() : (T)0;
            }
        }
        if (act) {
            A.m[off + k] = mm[k].x;
            if (TRACER) A.q[off + k] = qsh[k];
            if (A.Rdump) A.Rdump[off + k] = R.value() / c.sc;
        }
    }
}

// One CTA per queue entry, or (qhead set) persistent CTAs that take entries
// by an atomic ticket until the queue is exhausted.
template <int NW, int MB, int STORE, bool RAMP, bool TRACER>
__global__ void __launch_bounds__(32 * ((MB > 1 ? 2 : NW) + kChainRoles), MB) k_collide_chain(CollideArgs A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ ChainShared<NW> sh;
    int64_t entry = blockIdx.x;
    for (;;) {
        if (A.qhead) {
            __syncthreads();  // the previous cell's shared data is no longer read
            if (threadIdx.x == 0) sh.ticket = atomicAdd(A.qhead, 1);
            __syncthreads();
            entry = sh.ticket;
        }
        if (entry >= A.n_queue) return;
        const int64_t cell = A.queue ? (int64_t)A.queue[entry] : entry;
        chain_cell<NW, MB, STORE, RAMP, TRACER>(A, cell, entry, sh, smem_raw);
        if (!A.qhead) return;
    }
}

// the variants' host entry point, one translation unit per (NW, MB); ops as in
// variant_op
template <int NW, int MB>
cudaError_t collide_chain_variant(int op, int store, bool ramp, bool tracer, unsigned grid, int nthr, size_t smem,
                                  cudaStream_t st, const CollideArgs *A, int *out);

template <int NW, int MB, int STORE>
cudaError_t collide_chain_store(int op, bool ramp, bool tracer, unsigned grid, int nthr, size_t smem, cudaStream_t st,
                                const CollideArgs *A, int *out)
{
    void (*ks[4])(CollideArgs) = {
        k_collide_chain<NW, MB, STORE, false, false>, k_collide_chain<NW, MB, STORE, true, false>,
        k_collide_chain<NW, MB, STORE, false, true>, k_collide_chain<NW, MB, STORE, true, true>};
    return variant_op(ks, op, ramp, tracer, grid, nthr, smem, st, A, out);
}

}  // namespace mcd
