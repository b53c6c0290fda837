// mcd_collide_chain64.cuh -- the FP64 collision chain of one cell, split over
// specialised warps: the same method as cell_chain in mcd_collide.cuh, in the
// division of work of mcd_collide_chain.cuh.
//
// What bounds it: the FP64 units.  One FP64 instruction of a warp holds its SM
// sub-partition's unit for 64 cycles whatever its lanes do, so an event costs
// the FP64 instructions of the busiest sub-partition, and what one lane alone
// needs (the clock, the outcome, a swarm's cache) costs as much as a whole row.
//  * worker warps (thread k owns swarm k) only form row i, the new row and
//    column and their weights, some 52 instructions per event, 40 of them the
//    new pair;
//  * prefixes and sums over a group of 32 swarms run in 64-bit integers at the
//    scale of the group's largest rate (group_prefix64): no FP64 instruction, and,
//    measured by the group's total, nearer to the exact sum than FP64 additions (7
//    to 9e-17 of it against 1.1 to 1.5e-16);
//  * the choice warp adds up the groups (lane l: group l), brackets i and j and
//    forms an outcome that depends on j; comparisons use the integer unit;
//  * the mass warp keeps the two outcomes that do not depend on j (a grouped
//    partner of total mass dm m_i sticks, or erodes) ready per swarm, mass and
//    cache, one reciprocal for all four of a cache's (a lane each);
//  * the clock warp advances the clock and draws the random numbers.
// Nothing is formed ahead of the choice of j: the unit would be held by the row
// of an outcome that a third of the events do not take.
//
// Measured, heaviest cell, us per event (every thread doing all of it with
// block-wide scans -> this): 20 swarms 6.7 -> 5.0, 100: 7.2 -> 5.4, 200: 9.9 ->
// 7.4, 300: 13.3 -> 9.4, 400: 16.6 -> 11.3, 512: 19.3 -> 13.3; recomputing row
// i 13.8 -> 11.6 at 200.  With powers of S and the terms of one swarm read from
// its cache, and the cache of a general outcome formed by the whole choice
// warp: 4.7, 5.1, 6.8 (200), 10.6 (400), 12.4 (512); recomputing 10.3 at 200.  Many light cells, which the units bound whatever the
// layout, take the same: 32,768 cells of 40 swarms 7.7 ms, of 64 14.7 ms.
#pragma once
#include "mcd_collide_chain.cuh"

namespace mcd {

// worker warps come first, then these: the mass warp's FP64 work falls to the
// sub-partition with the fewest workers where their number leaves one
constexpr int kRoleMass = 0, kRoleChoice = 1, kRoleClock = 2;

struct Chain64Shared {
    CellK<double> c;
    double tot[3][16];     // the groups' totals: the row sums, the last event's new row, row i
    Draw<double> ring[64]; // this block of 32 events' draws and the next one's
    double tn;             // the clock after this event
    double Rp;             // the fresh R_i of the last event's swarm
    int sel;               // i, -2 at the end
    int2 pick;             // x: which of the ready outcomes (-1: no partner bracketed, -2: the end), y: the event crosses t_end
    int ticket;            // persistent CTAs: the queue entry taken
};

// inclusive prefix of x >= 0 within the warp's group of 32 (a negative x, a row
// sum's rounding, counts as 0): 53-bit significands shifted to the scale of the
// group's largest, 2^-57 of it per unit (what lies below is cut off: a prefix
// ahead of the group's largest keeps that much of it, not of itself, and u, with 53
// bits, tells no more apart), added as integers, and the sum rounded to FP64
// once.  Five FP64 additions in a row would hold the unit for 320 cycles and
// round five times.  A sum with a value that is not finite is formed
// plainly.
__device__ __forceinline__ double group_prefix64(double x)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const long long b = __double_as_longlong(x);
    int e = (int)((unsigned)(b >> 52) & 0x7FFu);
    if (b < 0 && e != 0x7FF) e = 0;
    const int E = (int)__reduce_max_sync(FULL, (unsigned)e);
    if (E == 0x7FF) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        return x;
    }
    unsigned long long v = ((unsigned long long)b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
    v = e ? (v << 5) >> min(E - e, 63) : 0ull;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(FULL, v, o);
        v += lane >= o ? y : 0ull;
    }
    const int lz = __clzll((long long)v), ex = E + 6 - lz;
    const unsigned long long M = v << (lz & 63), mant = (M >> 11) + ((M >> 10) & 1ull);
    if (v == 0ull || ex <= 0) return 0.0;
    return ex >= 0x7FF ? (double)INFINITY : __longlong_as_double((long long)(((unsigned long long)(ex - 1) << 52) + mant));
}

// The groups' inclusive prefixes (lane l < NW) of t, and in lanes 16.. of y;
// total and (with y) the sum of y to every lane.
template <int NW>
__device__ __forceinline__ double group_totals(const double *t, const double *y, double &total, double &ysum)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, l = lane & 15;
    double x = lane < 16 ? t[l] : (y ? y[l] : 0.0);
#pragma unroll
    for (int o = 1; o < NW; o <<= 1) {
        const double z = __shfl_up_sync(FULL, x, o, 16);
        if (l >= o) x += z;
    }
    total = __shfl_sync(FULL, x, NW - 1);
    ysum = 0.0;
    if (y) {
        ysum = __shfl_sync(FULL, x, 16 + NW - 1);
        total += ysum;
    }
    return x;
}

// order and finiteness of sums of rates (not negative) on the integer unit
__device__ __forceinline__ bool lt_rate(double a, double b) { return __double_as_longlong(a) < __double_as_longlong(b); }
__device__ __forceinline__ bool finite_rate(double a)
{
    return ((unsigned)(__double_as_longlong(a) >> 52) & 0x7FFu) != 0x7FFu;
}

// positive (infinite too), not NaN
__device__ __forceinline__ bool positive(double x)
{
    const long long b = __double_as_longlong(x);
    return b > 0 && b <= 0x7FF0000000000000ll;
}

// Choose element k with probability x_k / total (pf[k]: element k's prefix
// within its group; bs: lane l's inclusive prefix of group totals; Rp: element
// pend's value on top of its x, pend < 0 has Rp = 0).  True in the one lane
// whose element is chosen; false everywhere (any false) if nothing brackets the
// target.  load(k) runs for every lane's k of the group.
template <class F>
__device__ __forceinline__ bool choose64(double bs, const double *pf, double u, int pend, double Rp, int ng, int n,
                                         double total, bool &any, int &k, F load)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, pg = pend >> 5;
    double target = u * total;
    if (!lt_rate(target, total)) target = total * (1.0 - 1e-7);
    const double hi = bs + (pend >= 0 && lane >= pg ? Rp : 0.0);
    const unsigned in = __ballot_sync(FULL, lane < ng && finite_rate(total) && lt_rate(target, hi));
    any = in != 0u;
    const int g = any ? __ffs(in) - 1 : 0;
    const double below = __shfl_up_sync(FULL, hi, 1);  // (the group below: the same sum as its upper end)
    const double rem = target - __shfl_sync(FULL, lane == 0 ? 0.0 : below, g);
    const int kk = 32 * g + lane;
    k = min(kk, n - 1);
    const double P = pf[kk] + (pg == g && pend >= 0 && kk >= pend ? Rp : 0.0);
    load(k);
    const bool over = lt_rate(rem, P);
    const unsigned bal = __ballot_sync(FULL, over);
    // (the group's total may round above its last prefix: then lane 31)
    return any && (bal & ((1u << lane) - 1u)) == 0u && (over || lane == 31);
}

// The cache of mass m in place, by a warp: lanes 4 e + f hold outcome e's mass
// (a general outcome: lanes f) and write its field f (from 1/(1+S^2), 1/(1+S),
// 1/m, 1/(dm m)), so that one reciprocal serves all of them; the same
// expressions as make_part<double>.
__device__ __forceinline__ void make_ready64(const CellK<double> &c, double m, double dmm, double Mv, Part<double> *dst,
                                             int f, bool store)
{
    const long long mb = __double_as_longlong(m);
    const bool stk = mb >= __double_as_longlong(c.m_sw);
    const int cls = mb < __double_as_longlong(c.m_eta) ? 0 : (mb < __double_as_longlong(c.m_one) ? 1 : 2);
    const bool flat = c.kmode == 1;  // the constant kernel: masses alone
    const double a = flat ? 0.0 : cbrt64(c.cm_d * m);
    const double S = (stk ? c.Cst * a : c.Cep) * a;
    const double S2 = S * S;
    double x = 1.0 + (f == 0 ? S2 : S);
    x = f == 2 ? m : (f == 3 ? dmm : x);
    double y = rcp64(x);
    if (f == 3 && !(__double_as_longlong(c.dm) > 0)) y = (double)INFINITY;
    const double z = y * (f == 2 ? c.cbm : y);  // (f == 3: not used)
    double ad = 0.0;
    if (__any_sync(0xffffffffu, stk && !flat))
        ad = stk ? c.cm_d * (m - c.m_sw) / ((a * a + c.asw * c.asw) + a * c.asw) : 0.0;
    if (!store) return;
    if (f == 0) {
        dst->P2 = z;
        dst->a = a;
        dst->S = S;
        dst->S2 = S2;
        dst->S3 = S2 * (S + S);
    } else if (f == 1) {
        dst->q = y;
        dst->qz = c.settle ? z * c.soz : c.soz;
        dst->mh = m;
    } else if (f == 2) {
        dst->im = y;
        dst->bm = z;
        dst->Mv = Mv;
        dst->ad = ad;
    } else {
        dst->gi = y;
        dst->fl = cls | ((int)stk << 2);
    }
}

// dynamic shared memory: caches, ready outcomes (two caches and masses per swarm
// and one place for a general outcome), masses with dm m, the tracer copy, the
// prefixes and dv of row i
inline size_t collide_chain64_smem_bytes(int nsl, bool tracer)
{
    return (size_t)nsl * (3 * sizeof(Part<double>) + (tracer ? 9 : 8) * sizeof(double)) + sizeof(Part<double>) +
           sizeof(double2);
}

// STORE: 0 recompute row i before every event, 2 the stored matrix in the
// workspace.  RAMP, TRACER as in cell_chain
template <int NW, int STORE, bool RAMP, bool TRACER>
__device__ __forceinline__ void chain64_cell(const CollideArgs &A, const int64_t cell, const int64_t entry,
                                             Chain64Shared &sh, unsigned char *smem_raw)
{
    typedef double T;
    const int nthr = blockDim.x, nsl = nthr - 32 * kChainRoles, ng = nsl >> 5;  // swarm slots (workers), groups
    Part<T> *parts = reinterpret_cast<Part<T> *>(smem_raw);
    Part<T> *ready = parts + nsl;  // [2][nsl]: grouped partner sticks, erodes; then a general outcome
    double2 *mm = reinterpret_cast<double2 *>(ready + 2 * nsl + 1);  // mass, dm m
    double2 *mready = mm + nsl;                                      // the same of ready
    T *pf = reinterpret_cast<T *>(mready + 2 * nsl + 1);             // prefixes within the groups
    T *dvrow = pf + nsl;                                             // dv of row i
    double *qsh = dvrow + nsl;                                       // TRACER
    const int W = A.dv_w;
    T *const Dm = STORE ? reinterpret_cast<T *>(A.dvg) + (size_t)entry * A.dv_rows * W : nullptr;
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
    if (tid < 48) (&sh.tot[0][0])[tid] = 0.0;
    __syncthreads();
    const CellK<T> &c = sh.c;
    const int k = tid;  // a worker's swarm
    const bool act = k < n;
    Part<T> pk;
    // the random stream is keyed by (seed, disk) and counted by
    // (event, disk-local cell, step, domain tag)
    const uint64_t dcell = (uint64_t)(cell - A.disks[disk].c_off);
    const uint64_t step = (uint64_t)A.state->step;
    const T sc = (T)c.sc;
    if (w == ng + kRoleClock) {
        sh.ring[lane] = make_draw(philox((uint64_t)lane, dcell, step, kTagCollide, A.seed, (uint64_t)disk), sc);
    } else if (w < ng) {
        const int kc = act ? k : n - 1;
        const double mk = A.m[off + kc];
        pk = make_part<T>(c, mk, (T)(A.M[off + kc] * c.invVsc));
        const double dmm = __dmul_rn(c.dm, mk);
        if (act) {
            mm[k] = make_double2(mk, dmm);
            if (TRACER) qsh[k] = A.q[off + k];
            parts[k] = pk;
        }
        for (int e = 0; e < 2; ++e) {
            const double mr = ready_mass(c, mk, dmm, e != 0);
            const Part<T> pr = make_part<T>(c, mr, pk.Mv);
            if (act) {
                ready[e * nsl + k] = pr;
                mready[e * nsl + k] = make_double2(mr, __dmul_rn(c.dm, mr));
            }
        }
    }
    __syncthreads();

    const int reb = (int)(A.rebuild_every > 0 ? (A.rebuild_every < 0x7fffffff ? A.rebuild_every : 0x7fffffff)
                                              : 4 * (int64_t)n);
    int until_rebuild = reb;  // events left before the next full rebuild
    int64_t ev = 0;

    if constexpr (STORE != 0) {
        // every unordered pair once (warp w takes rows w, w + ng + 3, ...; its lanes
        // consecutive offsets d, so the stores are consecutive words)
        for (int rr = w; rr < n; rr += ng + kChainRoles) {
            const Part<T> pr = parts[rr];
            const int dmax = (n - 1) / 2 + (((n & 1) == 0 && rr < n / 2) ? 1 : 0);
            for (int d = lane; d <= dmax; d += 32) {
                int j = rr + d;
                if (j >= n) j -= n;
                T K;
                Dm[rr * W + d] = pair_dv<T>(c, pr, parts[j], &K);
            }
        }
    }
    __syncthreads();

    if (w == ng + kRoleChoice) {  // ---- the choice warp ----
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
            T Rp, none;
            const T bi = group_totals<NW>(sh.tot[0], sh.tot[1], tot, Rp);
            const bool ihere = choose64(bi, pf, dr.u1, pend, Rp, ng, n, tot, any, i, [](int) {});
            if (!positive(tot) || left <= 0) {  // (uniform)
                if (lane == 0) {
                    if (left <= 0 && positive(tot) && !A.cap_stops) atomicOr(A.status, kStTimeout);
                    sh.pick.x = -2;
                    sh.sel = -2;
                    sh.Rp = Rp;
                }
                bar_arrive(kBarI, nsl + 32);
                bar_sync(kBarEvent, nthr);
                break;
            }
            if (any ? ihere : lane == 0) {
                sh.sel = any ? i : n - 1;  // (no bracket, rates not finite: stay in bounds)
                sh.Rp = Rp;
            }
            bar_arrive(kBarI, nsl + 32);
            i = sh.sel;
            const double2 mmi = mm[i];
            const T Mvi = parts[i].Mv;
            double mj, mst;
            T dvij;
            bar_sync(kBarRow, nsl + 32);
            const T bj = group_totals<NW>(sh.tot[2], nullptr, tot2, none);
            const bool jhere = choose64(bj, pf, dr.u2, -1, (T)0, ng, n, tot2, any, j, [&](int q) {
                mj = mm[q].x;
                dvij = dvrow[q];
                mst = mmi.x + (dgt(mmi.y, mj) ? mmi.y : mj);  // should it stick (the FP64 latency behind the choice)
            });
            T dvx = dvij;
            if constexpr (RAMP)  // inside the ramp: fragments as at v_frag with the ramp's probability
                if (c.kmode != 1 && dvx < c.vfrag && !(dvx < vlo) && dr.u3 < fdiv(dvx - vlo, c.vfrag - vlo))
                    dvx = c.vfrag;
            const bool stick = c.kmode == 1 || dgt(c.vfrag, dvx);
            const bool grouped = group && dgt(mmi.y, mj) && (stick || eroding);
            int kind = stick ? 0 : 2;
            double mnew = 0.0, qnew = 0.0;
            if (any ? jhere : lane == 0) sh.pick.x = any ? (grouped ? (stick ? i : nsl + i) : gen) : -1;
            if (jhere && (!grouped || TRACER || logging)) {
                if (!grouped) {
                    if (stick)
                        mnew = mst;
                    else if constexpr (RAMP)
                        mnew = outcome_ramp<T>(c, mmi.x, mj, (T)0, (T)0, mmi.y, dvij, dr.u3, vlo, kind);
                    else
                        mnew = outcome<T>(c, mmi.x, mj, (T)0, (T)0, mmi.y, dvij, dr.u3, kind);
                } else {
                    mnew = ready_mass(c, mmi.x, mmi.y, !stick);  // (the mass warp may still be at work on mready)
                }
                if constexpr (TRACER)
                    qnew = tracer_update(mmi.x, mj, qsh[i], qsh[j], dgt(mmi.y, mj) ? mmi.y : mj, mnew, kind, c.chi);
            }
            const unsigned gm = __ballot_sync(0xffffffffu, jhere && !grouped);
            if (gm) {  // the cache of a general outcome, by the whole warp
                const double m = __shfl_sync(0xffffffffu, mnew, __ffs(gm) - 1), dmm = __dmul_rn(c.dm, m);
                make_ready64(c, m, dmm, Mvi, ready + gen, lane & 3, lane < 4);
                if (lane == 0) mready[gen] = make_double2(m, dmm);
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
    } else if (w == ng + kRoleMass) {  // ---- the mass warp ----
        bar_arrive(kBarRates, nsl + 96);
        for (;;) {
            bar_sync(kBarEvent, nthr);
            const int2 pick = sh.pick;
            if (pick.x < 0 || pick.y) break;
            const int i = sh.sel;
            // i's new mass and cache
            if (lane < (int)(sizeof(Part<T>) / 16))
                reinterpret_cast<uint4 *>(parts + i)[lane] = reinterpret_cast<const uint4 *>(ready + pick.x)[lane];
            const T Mvi = ready[pick.x].Mv;
            const double2 mi = mready[pick.x];
            if (lane == 0) mm[i] = mi;
            if (--until_rebuild == 0) {
                bar_arrive(kBarBuild, nsl + 32);
                until_rebuild = reb;
            }
            bar_arrive(kBarRates, nsl + 96);
            // its ready outcomes: lanes 0..3 stick, 4..7 erode (the others repeat them)
            const int e = (lane >> 2) & 1;
            const double mnew = ready_mass(c, mi.x, mi.y, e), dmnew = __dmul_rn(c.dm, mnew);
            bar_sync(kBarRead, nsl + 32);
            make_ready64(c, mnew, dmnew, Mvi, ready + e * nsl + i, lane & 3, lane < 8);
            if (lane < 8 && (lane & 3) == 0) mready[e * nsl + i] = make_double2(mnew, dmnew);
        }
    } else if (w == ng + kRoleClock) {  // ---- the clock warp ----
        const double t_end = A.t_end_from_state ? A.state->t + A.state->dt : A.t_end_fixed;
        double t = A.state->t;
        PhiloxRounds px;
        for (;;) {
            const T L = sh.ring[ev & 63].L;
            bar_sync(kBarRates, nsl + 96);
            T tot, Rp;
            group_totals<NW>(sh.tot[0], sh.tot[1], tot, Rp);
            if (!positive(tot) || ev >= A.max_events) {
                bar_sync(kBarEvent, nthr);
                break;
            }
            t += fdiv(L, tot);
            if (lane == 0) {
                sh.pick.y = t >= t_end;
                sh.tn = t;
            }
            // the next block's draws, one round per event of this block
            const int q = (int)(ev & 31);
            if (q == 0) px.start((uint64_t)((ev | 31) + 1 + lane), dcell, step, A.seed, (uint64_t)disk);
            if (q < 10) px.round();
            if (q == 10) sh.ring[((ev | 31) + 1 + lane) & 63] = make_draw(px.words(), sc);
            bar_sync(kBarEvent, nthr);
            const int2 pick = sh.pick;
            if (pick.x < 0 || pick.y) break;
            ++ev;
        }
    } else {  // ---- the workers ----
        int pend = -1;  // swarm whose fresh row sum rides on the next choice
        Acc<T> R;
        // full build of the row sums: R_k = sum_j r_kj in j order, from the stored
        // matrix or from fresh entries
        auto build = [&]() {
            R.zero();
            const int kc = act ? k : n - 1;
#pragma unroll 2
            for (int j = 0; j < n; ++j) {
                const Part<T> pj = parts[j];
                T K;
                if constexpr (STORE != 0)
                    K = kern_of<T>(c, pk.a, pj.a, Dm[sym_at(kc, j, n, W)]);
                else
                    pair_dv<T>(c, pk, pj, &K);
                R.add(K * weight<T>(pk, pj));
            }
        };
        build();
        T hi = act ? R.hi() : (T)0;  // R_k for the next choice (0 for the swarm whose fresh sum rides on it)
        for (;;) {
            // (1) row sums for the choice of i
            T x = group_prefix64(hi);
            pf[k] = x;
            if (lane == 31) sh.tot[0][w] = x;
            bar_arrive(kBarRates, nsl + 96);
            bar_sync(kBarI, nsl + 32);
            const int sel = sh.sel, i = max(sel, 0);
            if (k == pend) R.set(sh.Rp);
            if (sel < 0) {
                bar_sync(kBarEvent, nthr);
                break;
            }
            // (2) row i (i meets k) and column i (k meets i) before the event
            const Part<T> pi = parts[i];
            const int at = STORE != 0 ? sym_at(i, act ? k : n - 1, n, W) : 0;
            T dvik, Kold;
            if constexpr (STORE != 0) {
                dvik = Dm[at];
                Kold = kern_of<T>(c, pk.a, pi.a, dvik);
            } else {
                dvik = pair_dv<T>(c, pk, pi, &Kold);
            }
            dvrow[k] = dvik;
            x = group_prefix64(act ? Kold * weight<T>(pi, pk) : (T)0);
            pf[k] = x;
            if (lane == 31) sh.tot[2][w] = x;
            bar_arrive(kBarRow, nsl + 32);
            const T colo = Kold * weight<T>(pk, pi);
            bar_sync(kBarEvent, nthr);
            const int2 pick = sh.pick;
            if (pick.x < 0 || pick.y) break;
            // (3) the new row and column i: R_k += r_ki(new) - r_ki(old); R_i afresh
            const Part<T> pn = ready[pick.x];
            if (k == i) pk = pn;
            bar_arrive(kBarRead, nsl + 32);
            T Knew;
            const T dvn = pair_dv<T>(c, pk, pn, &Knew);
            if (STORE != 0 && act) Dm[at] = dvn;
            if (act && k != i) R.update(Knew * weight<T>(pk, pn), colo);
            hi = act && k != i ? R.hi() : (T)0;
            const bool rebuild = --until_rebuild == 0;
            x = group_prefix64(act && !rebuild ? Knew * weight<T>(pn, pk) : (T)0);
            if (lane == 31) sh.tot[1][w] = x;
            pend = i;
            if (rebuild) {
                bar_sync(kBarBuild, nsl + 32);
                build();
                pend = -1;
                until_rebuild = reb;
                hi = act ? R.hi() : (T)0;
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
template <int NW, int STORE, bool RAMP, bool TRACER>
__global__ void __launch_bounds__(32 * (NW + kChainRoles)) k_collide_chain64(CollideArgs A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Chain64Shared sh;
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
        chain64_cell<NW, STORE, RAMP, TRACER>(A, cell, entry, sh, smem_raw);
        if (!A.qhead) return;
    }
}

// the variants' host entry point, one translation unit per NW; ops as in
// variant_op
template <int NW>
cudaError_t collide_chain64_variant(int op, int store, bool ramp, bool tracer, unsigned grid, int nthr, size_t smem,
                                    cudaStream_t st, const CollideArgs *A, int *out);

template <int NW, int STORE>
cudaError_t collide_chain64_store(int op, bool ramp, bool tracer, unsigned grid, int nthr, size_t smem,
                                  cudaStream_t st, const CollideArgs *A, int *out)
{
    void (*ks[4])(CollideArgs) = {k_collide_chain64<NW, STORE, false, false>, k_collide_chain64<NW, STORE, true, false>,
                                  k_collide_chain64<NW, STORE, false, true>, k_collide_chain64<NW, STORE, true, true>};
    return variant_op(ks, op, ramp, tracer, grid, nthr, smem, st, A, out);
}

}  // namespace mcd
