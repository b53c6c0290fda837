// mcd_transport.cu -- initial particles and particle transport (Summary of the
// mcdust paper: "transport in the vertical and radial directions" in a static
// power-law gas disk).
//
// Transport of one particle over dt (reading, Ciesla-type Monte Carlo
// diffusion): radial Ito step r += [v_r + (1/(r rho_g)) d(r D rho_g)/dr] dt
// + sqrt(2 D dt) xi_1 with v_r = -2 eta v_K St/(1+St^2), and an exact
// Ornstein-Uhlenbeck step in z with rate k = Omega (St + alpha) and
// stationary variance D/k, i.e. H_d = H_g sqrt(alpha/(alpha+St)).  Particles
// below r_in are removed (swarm mass accreted); beyond r_out reflected.
//
// One thread per particle slot over the structure-of-arrays state; reads
// r, z, m, M, id and writes r, z (about 44 algorithmic bytes per particle).
// The FP64 path evaluates everything in FP64; the mixed path evaluates the
// gas, drag and displacements in FP32 and adds them to FP64 positions.
#include <math.h>

#include <type_traits>

#include "mcd_internal.cuh"

namespace mcd {

__device__ __forceinline__ int find_disk(const DiskDev *disks, int nd, int64_t s)
{
    int lo = 0, hi = nd - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (disks[mid].p_off <= s) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// ---- initial state ---------------------------------------------------------------
__global__ void k_init(const mcd_disk_params *params, const DiskDev *disks, int nd, const double *Mswarm,
                       uint64_t seed, int64_t N, double *m, double *M, double *r, double *z, uint32_t *id)
{
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= N) return;
    int d = find_disk(disks, nd, s);
    const mcd_disk_params &P = params[d];
    int64_t k = s - disks[d].p_off;
    U4 x = philox((uint64_t)k, 0, 0, kTagInit, seed, (uint64_t)d);
    double u0 = u01d(x.x[0]), u1 = u01d(x.x[1]), u2 = u01d(x.x[2]);
    double e = 2.0 - P.p, rr;
    if (fabs(e) < 1e-12) {
        rr = P.r_in * exp(u0 * log(P.r_out / P.r_in));
    } else {
        double lo = pow(P.r_in, e), hi = pow(P.r_out, e);
        rr = pow(lo + u0 * (hi - lo), 1.0 / e);
    }
    double xi = sqrt(-2.0 * log(u1)) * cos(2.0 * kPI * u2);
    Gas<double> g = gas_at<double>(P, rr, 0.0);
    r[s] = rr;
    z[s] = g.H * xi;
    m[s] = monomer_mass(P);
    M[s] = Mswarm[d];
    id[s] = (uint32_t)k;
}

// ---- transport -------------------------------------------------------------------------
// (float)(ca m), the cube of the radius, without the FP64 unit: the product of
// two (hi, lo) pairs is good to 2^-47, so its rounding is the double product's
// but for a value that close to a tie
__device__ __forceinline__ float mass_x_ca(const DiskC<float> &P, double m)
{
    const float mh = d2f_int(m);
    const unsigned long long b = (unsigned long long)__double_as_longlong(m);
    const unsigned E = (unsigned)(b >> 52);
    if (E - 949u > 200u) return (float)(m * P.ca);
    // the part of m below mh: m's low bits as a signed count of 2^(E - 1075)
    const unsigned lo = (unsigned)b, up = ((lo >> 28) & 1u) & (((lo & 0x0FFFFFFFu) != 0u) | ((lo >> 29) & 1u));
    const float ml = __int2float_rn((int)(lo & 0x1FFFFFFFu) - (int)(up << 29)) * __uint_as_float((E - 948u) << 23);
    const float h = __fmul_rn(mh, P.ca_h);
    return __fadd_rn(h, __fmaf_rn(mh, P.ca_l, __fmaf_rn(ml, P.ca_h, __fmaf_rn(mh, P.ca_h, -h))));
}

// x^-(k/2) from 1/x, k >= 0 (a disk slope that is a multiple of one half)
__device__ __forceinline__ double inv_half_pow(double ix, int k)
{
    double y = (k & 1) ? sqrt(ix) : 1.0;
    for (int q = 0; q < (k >> 1); ++q) y *= ix;
    return y;
}

// FP64.  Bound by the FP64 unit (about two operations per SM and cycle), so the
// gas is formed from as few divisions, square roots and transcendental
// functions as it takes: reciprocals of r, Omega, c_s and rho shared by every
// quantity, slopes that are multiples of 1/2 without pow(), one expm1 or exp for both
// exponentials of the vertical step, sincospi.  819,200 particles: 0.84 ms ->
// 0.44 ms with both slopes multiples of 1/2, 0.57 with one pow(), 0.69 with two.
template <bool TABLE>
__device__ __forceinline__ void transport_fp64(const DiskC<double> &P, GasTab tab, double &r, double &z, double m,
                                               double dt, const U4 &x)
{
    const double r0 = r, z0 = z, ir = 1.0 / r0;
    double Sigma, T, p = P.p, q = P.q;
    if (TABLE && tab.n >= 2) {
        const GasKnot &K = tab.k[gas_segment(tab, r0)];
        const double dl = log(r0) - K.lnr;
        Sigma = exp(K.lnS - K.p * dl);
        T = exp(K.lnT - K.q * dl);
        p = K.p, q = K.q;
    } else {
        const double ix = ir * kAU;
        Sigma = P.sigma0 * (P.p2 >= 0 ? inv_half_pow(ix, P.p2) : pow(ix, P.p));
        T = P.T0 * (P.q2 >= 0 ? inv_half_pow(ix, P.q2) : pow(ix, P.q));
    }
    const double c2 = kKB * T / P.mump, cs = sqrt(c2), ics = 1.0 / cs;
    const double Om = sqrt(P.GM * ir * ir * ir), iOm = 1.0 / Om, iH = Om * ics;
    const double s2 = z0 * iH, D = P.alpha * c2 * iOm;
    const double rho_mid = Sigma * iH * (1.0 / 2.5066282746310002);
    const double rho = (P.tr_flags & MCD_TR_ST_MIDPLANE) ? rho_mid : rho_mid * exp(-0.5 * s2 * s2);  // (St's density)
    const double irho = 1.0 / rho, lambda = P.lamc * irho, vth = 1.5957691216057308 * cs;
    const double a = cbrt(P.ca * m);
    double St = a < 2.25 * lambda ? P.rho_s * a * irho * (ics * (1.0 / 1.5957691216057308)) * Om
                                  : 2.0 * P.rho_s * a * a / (4.5 * vth * lambda * rho) * Om;
    // 35 and more scale heights up (rho below 2^-930) 1/rho may be infinite where St is not
    if ((__double_as_longlong(rho) >> 52) < 93) St = P.rho_s * a / (rho * vth) * Om;
    const double rho_bm = sqrt(-2.0 * log(u01d(x.x[0])));
    double sn, cn;
    sincospi(2.0 * u01d(x.x[1]), &sn, &cn);
    if (P.tr_flags & MCD_TR_RADIAL) {
        const double vr = -(c2 * iOm * ir * (p + 0.5 * (3.0 + q))) * St / (1.0 + St * St);  // -2 eta v_K St / (1 + St^2)
        const double vD = D * ir * (1.0 - p - 0.5 * q + s2 * s2 * 0.5 * (3.0 - q));
        r = r0 + (vr + vD) * dt + sqrt(2.0 * D * dt) * (rho_bm * cn);
    }
    if (P.tr_flags & MCD_TR_VERTICAL) {
        const double sv = P.settle_form == 1 ? St / (1.0 + St) : St;
        const double k = Om * (sv + P.alpha), kdt = k * dt;
        double zs, v;  // z0 exp(-k dt) and 1 - exp(-2 k dt), from the exponential that keeps their digits
        if (kdt < 0.5) {
            const double em = expm1(-kdt);
            zs = z0 + z0 * em;
            v = -(em * (em + 2.0));
        } else {
            const double E = exp(-kdt);
            zs = z0 * E;
            v = (1.0 - E) * (1.0 + E);
        }
        z = zs + sqrt(D * v / k) * (rho_bm * sn);
    }
}

// Mixed: gas, drag and displacements in FP32, added to FP64 positions.  What
// bounds it is the FP64 unit too, as soon as anything but those two additions
// reaches it: the parameters come as floats (DiskC), conversions run on the
// integer unit (d2f_int, f2d_int), a^3 from a (hi, lo) split of the mass.
template <bool TABLE>
__device__ __forceinline__ void transport_mixed(const DiskC<float> &P, GasTab tab, double &r, double &z, double m,
                                                float dtf, const U4 &x)
{
    const float rho_bm = sqrtf(-2.0f * logf(u01f(x.x[0])));
    float sn, cs;
    sincospif(2.0f * u01f(x.x[1]), &sn, &cs);
    const float xi1 = rho_bm * cs, xi2 = rho_bm * sn;
    const double r0 = r, z0 = z;
    const float rf = d2f_int(r0), zf = d2f_int(z0);
    const Gas<float> g = gas_core<float>(P, TABLE ? tab : GasTab{nullptr, 0}, r0, rf, zf);
    const float rho_s = P.rho_s;
    float rho_st = g.rho, vth = g.vth, nu = g.nu, asw = g.asw;
    if (P.tr_flags & MCD_TR_ST_MIDPLANE) {
        const Gas<float> g0 = gas_core<float>(P, TABLE ? tab : GasTab{nullptr, 0}, r0, rf, 0.0f);
        rho_st = g0.rho, vth = g0.vth, nu = g0.nu, asw = g0.asw;
    }
    const float a = cbrtf(mass_x_ca(P, m));
    const float St = a < asw ? rho_s * a / (rho_st * vth) * g.Omega : 2.0f * rho_s * a * a / (9.0f * nu * rho_st) * g.Omega;
    if (P.tr_flags & MCD_TR_RADIAL) {
        float vr = -2.0f * g.etavk * St / (1.0f + St * St);
        float s2 = zf / g.H;
        float vD = g.D / rf * (1.0f - g.p - 0.5f * g.q + s2 * s2 * 0.5f * (3.0f - g.q));
        r = r0 + f2d_int((vr + vD) * dtf + sqrtf(2.0f * g.D * dtf) * xi1);
    }
    if (P.tr_flags & MCD_TR_VERTICAL) {
        float sv = P.settle_form == 1 ? St / (1.0f + St) : St;
        float k = g.Omega * (sv + P.alpha);
        float em1 = expm1f(-k * dtf);
        z = z0 + f2d_int(zf * em1 + sqrtf(g.D * (-expm1f(-2.0f * k * dtf)) / k) * xi2);
    }
}

// TABLE: some disk has a gas table (the variant without one reads none).
// One thread per particle slot.  819,200 particles, mixed: 61 us with every
// parameter converted per particle on the FP64 unit -> 33 us; what is left are 927
// instructions per warp that issue in 64 % of the cycles, no pipe above 43 % (ALU
// 43, FP64 40, FMA 33, special functions 14): the Philox block's 64-bit products,
// two powf, the IEEE divisions, the additions to FP64 positions, and loads waited for.
template <bool MIXED, bool TABLE>
__global__ void __launch_bounds__(256) k_transport(const DiskC<typename std::conditional<MIXED, float, double>::type> *consts,
                                                   const GasKnot *gas_knots, const int32_t *gas_n,
                                                   const int32_t *slot_disk, uint64_t seed, const StepState *state,
                                                   int64_t N, double *r, double *z, const double *m, const double *M,
                                                   const uint32_t *id, double *accreted)
{
    const int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= N) return;
    const int d = slot_disk[s];
    double rs = r[s], zs = z[s];
    const double ms = m[s];
    const uint32_t ids = id[s];
    if ((((unsigned)(__double_as_longlong(rs) >> 52)) & 0x7FFu) == 0x7FFu) return;  // not finite: removed
    const auto &P = consts[d];
    if (!P.moves) return;
    const U4 x = philox((uint64_t)ids, 0, (uint64_t)state->step, kTagTransport, seed, (uint64_t)d);
    const GasTab tab = TABLE ? gas_tab(gas_knots, gas_n, d) : GasTab{nullptr, 0};
    if constexpr (MIXED)
        transport_mixed<TABLE>(P, tab, rs, zs, ms, d2f_int(state->dt), x);
    else
        transport_fp64<TABLE>(P, tab, rs, zs, ms, state->dt, x);
    // rs < r_in, rs > r_out on the integer unit: bit patterns order like the values
    // against a positive edge (an rs that is not finite takes the comparison itself)
    const long long rb = __double_as_longlong(rs);
    const bool odd = (((unsigned)(rb >> 52)) & 0x7FFu) == 0x7FFu;
    const bool removed = odd ? rs < P.r_in : rb < __double_as_longlong(P.r_in);
    if (removed)
        rs = INFINITY;
    else if (odd ? rs > P.r_out : rb > __double_as_longlong(P.r_out))
        rs = 2.0 * P.r_out - rs;
    r[s] = rs;
    z[s] = zs;
    if (removed) atomicAdd(&accreted[d], M[s]);
}

__global__ void k_set_clock(StepState *st, double t, int set_t, double dt, int set_dt)
{
    if (set_t) st->t = t;
    if (set_dt) st->dt = dt;
}

__global__ void k_advance_clock(StepState *st, int add_dt_to_t)
{
    if (add_dt_to_t) st->t += st->dt;
    st->step += 1;
}

cudaError_t launch_init(mcd_ctx *c, const double *d_Mswarm)
{
    if (c->N == 0) return cudaSuccess;
    unsigned blocks = (unsigned)((c->N + 255) / 256);
    k_init<<<blocks, 256, 0, c->stream>>>(c->d_params, c->d_disks, c->n_disks, d_Mswarm, c->seed, c->N,
                                          c->m[c->cur], c->M[c->cur], c->r[c->cur], c->z[c->cur], c->id[c->cur]);
    c->launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_transport(mcd_ctx *c)
{
    if (c->N == 0) return cudaSuccess;
    unsigned blocks = (unsigned)((c->N + 255) / 256);
    int b = c->cur;
    auto go = [&](auto kernel) {
        if constexpr (std::is_invocable_v<decltype(kernel), const DiskC<float> *, const GasKnot *, const int32_t *,
                                          const int32_t *, uint64_t, const StepState *, int64_t, double *, double *,
                                          const double *, const double *, const uint32_t *, double *>)
            kernel<<<blocks, 256, 0, c->stream>>>(c->d_cf, c->gas_knots, c->gas_n, c->slot_disk, c->seed, c->state, c->N,
                                                  c->r[b], c->z[b], c->m[b], c->M[b], c->id[b], c->accreted);
        else
            kernel<<<blocks, 256, 0, c->stream>>>(c->d_cd, c->gas_knots, c->gas_n, c->slot_disk, c->seed, c->state, c->N,
                                                  c->r[b], c->z[b], c->m[b], c->M[b], c->id[b], c->accreted);
    };
    const bool mixed = c->prec == MCD_MIXED, table = c->gas_tables > 0;
    if (mixed)
        table ? go(k_transport<true, true>) : go(k_transport<true, false>);
    else
        table ? go(k_transport<false, true>) : go(k_transport<false, false>);
    c->launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_set_clock(mcd_ctx *c, double t, int set_t, double dt, int set_dt)
{
    k_set_clock<<<1, 1, 0, c->stream>>>(c->state, t, set_t, dt, set_dt);
    c->launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_advance_clock(mcd_ctx *c, int add_dt_to_t)
{
    k_advance_clock<<<1, 1, 0, c->stream>>>(c->state, add_dt_to_t);
    c->launches += 1;
    return cudaGetLastError();
}

}  // namespace mcd
