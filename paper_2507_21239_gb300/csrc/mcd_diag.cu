// mcd_diag.cu -- diagnostics: the dust mass distribution versus distance (the
// Benchmark section compares the codes by the dust surface density as a
// function of particle mass and distance from the star), in summary form:
// per radial bin [edges[b], edges[b+1]), the swarm-mass-weighted sums of the
// representative mass's first three powers and the particle count.
//
// Two paths.  Disks of many particles per bin (kMomentsSplitMin, kMomentsPerBin) are
// cut into parts of consecutive slots, one CTA each: a CTA finds the first and last
// bin of its particles in one pass and forms the sums of each bin between them in a
// pass of its own; after a regrid the slots lie in radial zones, so that is one bin
// or two, and on particles in no order every bin.  A second kernel adds the parts'
// sums bin by bin.  One CTA per bin that scans all particles (the other path, for
// small disks and many bins) leaves SMs idle with few bins and reads every particle
// once per bin.
// Bound by the FP64 unit (an instruction per 16 SM cycles): 19 instructions per
// particle and bin pass, so parts are small enough (1,024 particles) to even the
// SMs out.  Both diagnostics of 819,200 particles (32 bins; a 64 x 96 map), calls
// and copies included: 4.26 ms -> 0.19 ms (k_moments_parts 0.10 ms, k_map_add 0.03).
//
// In both, threads keep Neumaier-compensated sums over a fixed set of particles
// and they are combined in a fixed tree, so the result does not depend on
// scheduling.  Products and sums are explicitly rounded (no fused
// multiply-add), like the plain CPU evaluation they are compared with.
#include <algorithm>

#include "mcd_internal.cuh"

namespace mcd {

constexpr int kDiagThreads = 256;

struct NSum {
    double s, c;
    __device__ void add(double x)
    {
        // (|s| >= |x| on the integer unit: every FP64 instruction holds a sub-partition for 64 cycles)
        const double t = __dadd_rn(s, x);
        const bool sx = (__double_as_longlong(s) & 0x7FFFFFFFFFFFFFFFll) >= (__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll);
        c = __dadd_rn(c, __dadd_rn(__dsub_rn(sx ? s : x, t), sx ? x : s));
        s = t;
    }
};

// bit patterns that order like the values (-0 and +0 alike), for comparisons on
// the integer unit; NaN lies outside [key(-inf), key(+inf)]
__device__ __forceinline__ uint64_t diag_key(double x)
{
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    if (!(b << 1)) return 0x8000000000000000ULL;
    return (b >> 63) ? ~b : (b | 0x8000000000000000ULL);
}

// the last of the n + 1 non-decreasing keys k[0..n] not above v, for k[0] <= v < k[n]
__device__ __forceinline__ int last_key_not_above(const uint64_t *k, int n, uint64_t v)
{
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (k[mid] <= v)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

// one Neumaier sum added to another
__device__ __forceinline__ void nsum_merge(NSum &a, double s, double c)
{
    a.add(s);
    a.c = __dadd_rn(a.c, c);
}

// The four compensated sums of every lane combined over the warp in a fixed
// order: half the warp takes two of the sums from the other half, a quarter one
// of them, then three rounds on one sum each (six merges per lane instead of
// twenty).  Lane l ends with sum l >> 3 & 3 in its lanes l & 7 == 0.
__device__ __forceinline__ NSum warp_nsum4(const NSum (&a)[4])
{
    const int lane = threadIdx.x & 31;
    const bool up = lane & 16, uq = lane & 8;
    NSum h[2], r;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const double gs = __shfl_xor_sync(0xffffffffu, up ? a[q].s : a[q + 2].s, 16);
        const double gc = __shfl_xor_sync(0xffffffffu, up ? a[q].c : a[q + 2].c, 16);
        h[q] = up ? a[q + 2] : a[q];
        nsum_merge(h[q], gs, gc);
    }
    const double gs = __shfl_xor_sync(0xffffffffu, uq ? h[0].s : h[1].s, 8);
    const double gc = __shfl_xor_sync(0xffffffffu, uq ? h[0].c : h[1].c, 8);
    r = uq ? h[1] : h[0];
    nsum_merge(r, gs, gc);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        const double s = __shfl_down_sync(0xffffffffu, r.s, o, 8), c = __shfl_down_sync(0xffffffffu, r.c, o, 8);
        nsum_merge(r, s, c);
    }
    return r;
}

// ... and over the block of kDiagThreads: the warps' results by warp 0, whose
// lanes 0, 8, 16, 24 end with sums 0 to 3
__device__ __forceinline__ NSum block_nsum4(const NSum (&a)[4], double2 (*sh)[4])
{
    static_assert(kDiagThreads == 256, "eight warps, eight lanes per sum");
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    NSum r = warp_nsum4(a);
    __syncthreads();
    if ((lane & 7) == 0) sh[w][lane >> 3] = make_double2(r.s, r.c);
    __syncthreads();
    if (w == 0) {
        const double2 v = sh[lane & 7][lane >> 3];
        r.s = v.x, r.c = v.y;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            const double s = __shfl_down_sync(0xffffffffu, r.s, o, 8), c = __shfl_down_sync(0xffffffffu, r.c, o, 8);
            nsum_merge(r, s, c);
        }
    }
    return r;
}

// Where the parts pay.  A pass over one bin of a part takes some 9 us whatever the
// part's size (the block's sum is what it waits for), so with many bins per part
// the CTA per bin is faster: at 1,536 particles per bin 65,536 particles take 142
// (parts) against 153 us in zone order and 366 against 658 shuffled, at 1,024 181
// against 142 and 491 against 621.  Parts larger than 1,024 (above 113 bins, so
// that the records fit) are fewer and make longer passes: 204,800 particles at
// 1,536 per bin 365 against 290 us, at 2,048 (100 bins) 217 against 351.  Disks of up
// to 16,384 particles (80 to 155 us at 12,288) keep the CTA per bin.
constexpr int64_t kMomentsSplitMin = 16384, kMomentsPart = 1024;
constexpr int64_t kMomentsPerBin = 1536, kMomentsPerBinLarge = 2048;
// a part's record of one bin: four compensated sums and the count
struct MomentsPart {
    double s[4], c[4];
    long long n;
};

// part p: particles [p P, p P + P); its records to rec[p * nbins + bin], its bins' range to range[p]
__global__ void __launch_bounds__(kDiagThreads) k_moments_parts(const double *m, const double *M, const double *r,
                                                                int64_t n, int64_t P, int nbins, const double *edges,
                                                                MomentsPart *rec, int2 *range)
{
    extern __shared__ uint64_t ek[];  // nbins + 1 keys
    __shared__ double2 sh[kDiagThreads / 32][4];
    __shared__ int rg[2], cnt;
    const int k = threadIdx.x;
    for (int q = k; q <= nbins; q += kDiagThreads) ek[q] = diag_key(edges[q]);
    if (k == 0) rg[0] = nbins, rg[1] = -1;
    __syncthreads();
    const int64_t p0 = blockIdx.x * P, p1 = min(p0 + P, n);
    // the bins' range over the part
    auto bin_of = [&](double x) {
        const uint64_t v = diag_key(x);
        return v >= ek[0] && v < ek[nbins] && v <= 0xFFF0000000000000ULL ? last_key_not_above(ek, nbins, v) : -1;
    };
    int lo = nbins, hi = -1;
    for (int64_t i = p0 + k; i < p1; i += kDiagThreads) {
        const int b = bin_of(r[i]);
        if (b >= 0) lo = min(lo, b), hi = max(hi, b);
    }
    if (hi >= 0) {
        atomicMin(&rg[0], lo);
        atomicMax(&rg[1], hi);
    }
    __syncthreads();
    const int b0 = rg[0], b1 = rg[1];
    if (k == 0) range[blockIdx.x] = make_int2(b0, b1);
    for (int b = b0; b <= b1; ++b) {
        NSum acc[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q].s = acc[q].c = 0.0;
        int mine = 0;
        for (int64_t i = p0 + k; i < p1; i += kDiagThreads) {
            const uint64_t v = diag_key(r[i]);
            if (!(v >= ek[b] && v < ek[b + 1])) continue;
            const double w = M[i], x = m[i];
            const double w1 = __dmul_rn(w, x), w2 = __dmul_rn(w1, x), w3 = __dmul_rn(w2, x);
            acc[0].add(w);
            acc[1].add(w1);
            acc[2].add(w2);
            acc[3].add(w3);
            ++mine;
        }
        __syncthreads();
        if (k == 0) cnt = 0;
        __syncthreads();
        if (mine) atomicAdd(&cnt, mine);
        const NSum t = block_nsum4(acc, sh);
        MomentsPart &o = rec[(int64_t)blockIdx.x * nbins + b];
        if (k < 32 && (k & 7) == 0) o.s[k >> 3] = t.s, o.c[k >> 3] = t.c;
        if (k == 0) o.n = cnt;
    }
}

// bin b of every part, in part order per thread, then over the block
__global__ void __launch_bounds__(kDiagThreads) k_moments_sum(const MomentsPart *rec, const int2 *range, int parts,
                                                              int nbins, double *out)
{
    __shared__ double2 sh[kDiagThreads / 32][4];
    __shared__ unsigned long long cnt;
    const int b = blockIdx.x, k = threadIdx.x;
    if (k == 0) cnt = 0;
    __syncthreads();
    NSum acc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q].s = acc[q].c = 0.0;
    long long mine = 0;
    for (int p = k; p < parts; p += kDiagThreads) {
        const int2 g = range[p];
        if (b < g.x || b > g.y) continue;
        const MomentsPart &o = rec[(int64_t)p * nbins + b];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            acc[q].add(o.s[q]);
            acc[q].c = __dadd_rn(acc[q].c, o.c[q]);
        }
        mine += o.n;
    }
    if (mine) atomicAdd(&cnt, (unsigned long long)mine);
    const NSum t = block_nsum4(acc, sh);
    if (k < 32 && (k & 7) == 0) out[5 * b + (k >> 3)] = __dadd_rn(t.s, t.c);
    if (k == 0) out[5 * b + 4] = (double)cnt;  // (after the barriers above)
}

__global__ void __launch_bounds__(kDiagThreads) k_moments(const double *m, const double *M, const double *r,
                                                          int64_t n, const double *edges, double *out)
{
    __shared__ double ss[5][kDiagThreads], cs[5][kDiagThreads];
    const int b = blockIdx.x, k = threadIdx.x;
    const double lo = edges[b], hi = edges[b + 1];
    NSum acc[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) acc[q].s = acc[q].c = 0.0;
    for (int64_t i = k; i < n; i += kDiagThreads) {
        const double ri = r[i];
        if (!(ri >= lo && ri < hi)) continue;
        const double w = M[i], x = m[i];
        const double w1 = __dmul_rn(w, x), w2 = __dmul_rn(w1, x), w3 = __dmul_rn(w2, x);
        acc[0].add(w);
        acc[1].add(w1);
        acc[2].add(w2);
        acc[3].add(w3);
        acc[4].add(1.0);
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        ss[q][k] = acc[q].s;
        cs[q][k] = acc[q].c;
    }
    __syncthreads();
    for (int h = kDiagThreads / 2; h > 0; h >>= 1) {
        if (k < h) {
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                NSum a{ss[q][k], cs[q][k]};
                a.add(ss[q][k + h]);
                ss[q][k] = a.s;
                cs[q][k] = __dadd_rn(a.c, cs[q][k + h]);
            }
        }
        __syncthreads();
    }
    if (k < 5) out[5 * b + k] = __dadd_rn(ss[k][0], cs[k][0]);
}

// ---- sigma_d(m, r) map: swarm mass per (radial bin, mass bin) --------------
// Every particle's M enters as a 64-bit integer count of a power-of-two unit
// 2^(e-62), 2^e at least the disk's total live swarm mass, so no sum can
// overflow and integer atomics make the sums independent of the order of
// the additions.  M times a power of two is exact; each M is rounded once, to
// the nearest unit (2^-61 of the total at most).

// The unit's exponent: 2^e above the disk's live swarm mass, summed in a fixed
// order (per lane, per warp, then the warps' sums by the last block to finish,
// a ticket; nothing waits).  Plain FP64 sums are enough for an exponent with a
// factor of two to spare, and take one FP64 instruction per particle.
constexpr int kMapWarps = 4;
__global__ void __launch_bounds__(32 * kMapWarps) k_map_unit(const double *M, const double *r, int64_t n, double *part,
                                                             int *e_out, unsigned *ticket)
{
    __shared__ bool last;
    const int lane = threadIdx.x & 31, nw = gridDim.x * kMapWarps, w = blockIdx.x * kMapWarps + (threadIdx.x >> 5);
    auto live = [&](int64_t i) {
        const uint64_t v = diag_key(r[i]);  // r < inf and no NaN
        const double x = M[i];
        return v >= 0x000FFFFFFFFFFFFFULL && v < 0xFFF0000000000000ULL ? x : 0.0;
    };
    auto warp_sum = [](double x) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        return x;
    };
    double a = 0.0, b = 0.0;
    int64_t i = (int64_t)w * 32 + lane;
    const int64_t step = (int64_t)nw * 32;
    for (; i + step < n; i += 2 * step) {
        const double x = live(i), y = live(i + step);
        a += x;
        b += y;
    }
    if (i < n) a += live(i);
    a = warp_sum(a + b);
    if (lane == 0) part[w] = a;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    __threadfence();
    double t = 0.0;
    for (int q = lane; q < nw; q += 32) t += __ldcg(part + q);
    t = warp_sum(t);
    if (lane == 0) *e_out = t > 0.0 ? ilogb(t) + 2 : 0;
}

// M 2^up rounded to a whole number, on the integer unit (the plain evaluation
// for values that are not positive normal numbers or do not fit)
__device__ __forceinline__ unsigned long long units_of(double M, int up)
{
    const uint64_t b = (uint64_t)__double_as_longlong(M);
    const int E = (int)(b >> 52);  // (the sign bit set: 2048 or more)
    const int sh = E - 1075 + up;  // M = mant 2^(E - 1075)
    if (E == 0 || E >= 2047 || sh > 10) return __double2ull_rn(scalbn(M, up));
    const uint64_t mant = (b & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL;
    if (sh >= 0) return mant << sh;
    if (sh < -54) return 0;
    const uint64_t q = mant >> -sh, rem = mant - (q << -sh), half = 1ULL << (-sh - 1);
    return q + (rem > half || (rem == half && (q & 1)));
}

// the particles into the map, in units of 2^(e - 62); both edge lists as keys in
// shared memory, nothing on the FP64 unit
__global__ void __launch_bounds__(kDiagThreads) k_map_add(const double *m, const double *M, const double *r, int64_t n,
                                                          const double *re, int nr, const double *me, int nm,
                                                          const int *e_unit, unsigned long long *acc)
{
    extern __shared__ uint64_t keys[];  // nr + 1, then nm + 1
    uint64_t *rk = keys, *mk = keys + nr + 1;
    for (int q = threadIdx.x; q <= nr; q += kDiagThreads) rk[q] = diag_key(re[q]);
    for (int q = threadIdx.x; q <= nm; q += kDiagThreads) mk[q] = diag_key(me[q]);
    __syncthreads();
    const int up = 62 - *e_unit;
    const uint64_t top = 0xFFF0000000000000ULL;  // key(+inf)
    for (int64_t i = blockIdx.x * (int64_t)kDiagThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kDiagThreads) {
        const uint64_t ri = diag_key(r[i]), mi = diag_key(m[i]);
        if (!(ri >= rk[0] && ri < rk[nr] && ri <= top) || !(mi >= mk[0] && mi < mk[nm] && mi <= top)) continue;
        const int b = last_key_not_above(rk, nr, ri), q = last_key_not_above(mk, nm, mi);
        atomicAdd(&acc[(int64_t)b * nm + q], units_of(M[i], up));
    }
}

__global__ void k_map_out(const unsigned long long *acc, int64_t nb, const int *e_unit, double *out)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k < nb) out[k] = scalbn(__ull2double_rn(acc[k]), *e_unit - 62);
}

cudaError_t launch_sigma_map(mcd_ctx *c, int disk, int nr, int nm)
{
    const DiskDev &D = c->hd[disk];
    const int b = c->cur;
    const int64_t nb = (int64_t)nr * nm;
    unsigned long long *acc = reinterpret_cast<unsigned long long *>(c->map_acc);
    int *e_unit = reinterpret_cast<int *>(c->map_acc + nb);
    // the sums, and behind them the unit's exponent and its ticket
    cudaError_t e = cudaMemsetAsync(acc, 0, sizeof(unsigned long long) * (nb + 1), c->stream);
    if (e != cudaSuccess) return e;
    const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>(kMapSums / kMapWarps, D.n0 / (256 * kMapWarps)));
    k_map_unit<<<blocks, 32 * kMapWarps, 0, c->stream>>>(c->M[b] + D.p_off, c->r[b] + D.p_off, D.n0, c->map_sums, e_unit,
                                                        reinterpret_cast<unsigned *>(e_unit + 1));
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>(608, (D.n0 + kDiagThreads - 1) / kDiagThreads));
    const size_t smem = sizeof(uint64_t) * ((size_t)nr + nm + 2);
    if (smem > 48 * 1024 - 512 &&
        (e = cudaFuncSetAttribute(k_map_add, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)(sizeof(uint64_t) * (2 * MCD_MAX_MAP_EDGES + 2)))) != cudaSuccess)
        return e;
    k_map_add<<<g, kDiagThreads, smem, c->stream>>>(c->m[b] + D.p_off, c->M[b] + D.p_off, c->r[b] + D.p_off, D.n0,
                                                    c->map_redges, nr, c->map_medges, nm, e_unit, acc);
    k_map_out<<<(unsigned)((nb + 255) / 256), 256, 0, c->stream>>>(acc, nb, e_unit, c->map_out);
    c->launches += 3;
    return cudaGetLastError();
}

cudaError_t launch_moments(mcd_ctx *c, int disk, int nbins)
{
    const DiskDev &D = c->hd[disk];
    const int b = c->cur;
    const double *m = c->m[b] + D.p_off, *M = c->M[b] + D.p_off, *r = c->r[b] + D.p_off;
    // parts of P particles: their records and their bins' ranges take the sort's key
    // buffers (free between regrids)
    int64_t P = kMomentsPart;
    auto fits = [&](int64_t p) {
        return (size_t)((D.n0 + p - 1) / p) * nbins * sizeof(MomentsPart) <= sizeof(uint64_t) * (size_t)D.n0;
    };
    while (P < D.n0 && !fits(P)) P *= 2;
    const int64_t per_bin = P == kMomentsPart ? kMomentsPerBin : kMomentsPerBinLarge;
    if (D.n0 > kMomentsSplitMin && D.n0 >= per_bin * nbins && fits(P) && P <= D.n0 / 4) {
        const int parts = (int)((D.n0 + P - 1) / P);
        MomentsPart *rec = reinterpret_cast<MomentsPart *>(c->key[0] + D.p_off);
        int2 *range = reinterpret_cast<int2 *>(c->key[1] + D.p_off);
        k_moments_parts<<<parts, kDiagThreads, sizeof(uint64_t) * (nbins + 1), c->stream>>>(m, M, r, D.n0, P, nbins,
                                                                                        c->diag_edges, rec, range);
        k_moments_sum<<<(unsigned)nbins, kDiagThreads, 0, c->stream>>>(rec, range, parts, nbins, c->diag_out);
        c->launches += 2;
        return cudaGetLastError();
    }
    k_moments<<<(unsigned)nbins, kDiagThreads, 0, c->stream>>>(m, M, r, D.n0, c->diag_edges, c->diag_out);
    c->launches += 1;
    return cudaGetLastError();
}

}  // namespace mcd
