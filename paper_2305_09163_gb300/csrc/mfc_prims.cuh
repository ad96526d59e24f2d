// Conserved -> primitive recovery with the CFL rate, the six-equation model's
// pressure relaxation, and primitive -> conserved conversion (Sec. 2.1, 2.3).
#pragma once
#include "mfc_sweeps.cuh"

namespace mfc {

// Conserved -> primitive recovery per cell (prims_cell) and the CFL rate of a
// cell (cell_cfl_rate) live in mfc_cell.cuh, where the RK epilogue uses them too.

// Publish the CFL maximum and the non-physical count of a CTA of 8 warps: one
// ordered-bits atomic per CTA, exact and independent of scheduling.
__device__ __forceinline__ void publish_block_rate(const PrimArgs& a, double rate, int bad) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        rate = fmax(rate, __shfl_xor_sync(0xffffffffu, rate, o));
        bad += __shfl_xor_sync(0xffffffffu, bad, o);
    }
    __shared__ double srate[8];
    __shared__ int sbad[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) { srate[wid] = rate; sbad[wid] = bad; }
    __syncthreads();
    if (wid == 0) {
        const int nw = blockDim.x >> 5;
        rate = lane < nw ? srate[lane] : 0.0;
        bad = lane < nw ? sbad[lane] : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            rate = fmax(rate, __shfl_xor_sync(0xffffffffu, rate, o));
            bad += __shfl_xor_sync(0xffffffffu, bad, o);
        }
        if (lane == 0) {
            atomicMax(a.rate_max, (unsigned long long)__double_as_longlong(rate));
            if (bad) atomicAdd(a.bad, bad);
        }
    }
}

template <typename Real, int NF, int NDIM, bool RATE, bool SIX = false>
__global__ void __launch_bounds__(256) prims_kernel(const PrimArgs a) {
    using Lay = Layout<NF, NDIM>;
    constexpr int NS = Lay::NS;
    pdl_wait();
    const long long nc = a.g.ncell;
    double rate = 0.0;
    int bad = 0;
    Real* w = static_cast<Real*>(a.w);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nc;
         i += (long long)gridDim.x * blockDim.x) {
        double q[NS];
#pragma unroll
        for (int v = 0; v < NS; ++v) q[v] = __ldg(a.q + v * nc + i);
        Real wv[NS], c2;
        prims_cell<NF, NDIM, SIX>(q, a.e, wv, c2);
#pragma unroll
        for (int v = 0; v < NS; ++v) w[v * nc + i] = wv[v];
        if (RATE) {
            const double r = cell_cfl_rate<Real, NF, NDIM>(wv, c2, a.g, a.grid, a.grid_stride, i);
            if (__double2hiint(r) < 0) bad += 1;
            else rate = max_nonneg(rate, r);
        }
    }
    if (RATE) publish_block_rate(a, rate, bad);
}

// Six-equation model (Sec. 2.3): pressure relaxation of one cell's conserved
// state q[NQ] with infinite stiffness, in place, after a Runge-Kutta stage
// (Saurel, Petitpas & Berry 2009; Schmidmayer et al. 2020).  At fixed mass
// each phase's energy follows de_k = -p dv_k at the final pressure p, which for
// a stiffened gas gives the relaxed volume fraction
//     a_k(p) = (g_k - 1)(E_k0 + a_k0 p) / (g_k (p + pinf_k)),  E_k0 = a_k r_k e_k.
// The phases taking part are those with a_k0 > 0 and p_k0 + pinf_k > 0
// (E_k0 > a_k0 pinf_k); the others keep a_k0.  The relaxed pressure solves
// f(p) = sum_{taking part} a_k(p) - (1 - sum_{others} a_k0) = 0; on
// p > lo = -min pinf (over the phases taking part) f is convex and falls
// strictly from +inf to below zero, so the root is unique.
//  1. FP32 Newton from the pressure the mixture law gives for the total energy
//     with the old fractions (the root itself for a relaxed state): from the
//     left of the root Newton rises monotonically to it, from the right it
//     lands left of it unless it would leave the domain, when the step bisects
//     [lo, p] instead; at most 60 iterations, ending at a relative step of 2^-20;
//  2. two Newton steps with f in float-float arithmetic (f' in FP32 suffices:
//     its error only slows the quadratic convergence to a linear one with
//     factor ~1e-7), which bring p to ~1e-14 relative;
//  3. one Newton step with f in FP64, p1 = p0 - f(p0)/f'(p0), and the new fractions
//     a_k(p1) = a_k(p0) + a_k'(p0)(p1 - p0) (the second-order remainder is
//     below FP64 rounding): a fraction near 1 must be right to ~1e-16
//     absolute, since a trace phase's fraction is 1 minus it.  The correction is
//     ~1e-14 of a_k, so FP32 derivatives give it far below that;
//  4. in FP64 the pressure of the total energy with the mixture law of the
//     new fractions and every phase's energy reset to it.
// On GB300 an FP64 instruction costs the issue time of ~60 FP32 ones, and the
// relaxation is bound by them (44 per cell and stage with the recovery, two
// phases): the start of step 1 and the test E_k0 > a_k0 pinf_k, decided in FP64
// only where float-float cannot, take none.  STEADY (mixed form) keeps both and
// the derivatives of step 3 in FP64: there a trace fraction of ~1e-9 feeds FP32
// arithmetic that tells apart results one FP64 rounding of 1 away.  If no phase can
// relax the state is left as it is: the CFL check flags it.
__device__ __forceinline__ bool energy_above(double E, double x, double pinf, df Ed, df xd, df pinfd) {
    const unsigned big = (1023u + 120u) << 20;   // above 2^120 or not finite: float-float does not hold it
    if (((unsigned)__double2hiint(E) & 0x7FF00000u) < big && ((unsigned)__double2hiint(x) & 0x7FF00000u) < big) {
        const df d = df_add(Ed, df_neg(df_mul(xd, pinfd)));
        if (fabsf(d.hi) > 0x1p-40f * fabsf(Ed.hi)) return d.hi > 0.f;
    }
    return E > __dmul_rn(x, pinf);
}

template <int NF, int NDIM, bool STEADY>
__device__ __forceinline__ void relax6(const RelaxConst& c, const EosConst& e, double* q) {
    using Lay = Layout<NF, NDIM, true>;
    constexpr int IA = Lay::IA, II = Lay::II;
    double irho, eint;
    six_energy<NF, NDIM>(q, irho, eint);
    double a0[NF];
    df a0d[NF], E0d[NF];
    bool in[NF];
    double asum = 0.0;
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) {
        a0[k] = q[IA + k];
        asum += a0[k];
    }
    a0[NF - 1] = 1.0 - asum;
    double target = 1.0;
    float lo = 0.f;
    bool any = false;
#pragma unroll
    for (int k = 0; k < NF; ++k) {
        a0d[k] = df_from_double(a0[k]);
        E0d[k] = df_from_double(q[II + k]);
        in[k] = positive(a0[k]) && energy_above(q[II + k], a0[k], c.pinf[k], E0d[k], a0d[k], c.pinfd[k]);
        if (!in[k]) {
            target -= a0[k];
            continue;
        }
        lo = any ? fmaxf(lo, -c.pinff[k]) : -c.pinff[k];
        any = true;
    }
    if (any) {
        // 1. FP32 Newton from the mixture-law pressure (float-float: rho e - Pi cancels)
        float p;
        if constexpr (STEADY) {
            double G = e.G_N, P = e.P_N;
#pragma unroll
            for (int k = 0; k < NF - 1; ++k) {
                G = fma(q[IA + k], e.dG[k], G);
                P = fma(q[IA + k], e.dP[k], P);
            }
            p = (float)((eint - P) * rcp_nr(G));
        } else {
            df Pm = c.P_N;
            float Gm = c.G_N;
#pragma unroll
            for (int k = 0; k < NF - 1; ++k) {
                Pm = df_add(Pm, df_mul(a0d[k], c.dP[k]));
                Gm = fmaf(a0d[k].hi, c.dG[k], Gm);
            }
            p = df_add(df_from_double(eint), df_neg(Pm)).hi * rcp_approx(Gm);
        }
        if (!(p > lo)) p = lo + fmaxf(fabsf(lo), 1.f);
        const df targetd = df_from_double(target);
        float hi = INFINITY;
        for (int it = 0; it < 60; ++it) {
            float f = -targetd.hi, fp = 0.f;
#pragma unroll
            for (int k = 0; k < NF; ++k) {
                if (!in[k]) continue;
                const float t = rcp_approx(p + c.pinff[k]);
                f = fmaf(c.c1f[k] * fmaf(a0d[k].hi, p, E0d[k].hi), t, f);
                fp = fmaf(c.c1f[k] * fmaf(a0d[k].hi, c.pinff[k], -E0d[k].hi), t * t, fp);
            }
            if (f > 0.f) lo = p;
            else hi = p;
            float pn = p - f * rcp_approx(fp);
            if (!(pn > lo && pn < hi)) pn = 0.5f * (lo + (hi < INFINITY ? hi : p));
            const bool done = fabsf(pn - p) <= 0x1p-20f * fabsf(pn) || !(pn > lo && pn < hi);
            p = pn;
            if (done) break;
        }
        // 2. float-float Newton steps
        df pd = {p, 0.f};
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            df f = df_neg(targetd);
            float fp = 0.f;
#pragma unroll
            for (int k = 0; k < NF; ++k) {
                if (!in[k]) continue;
                const df num = df_add(E0d[k], df_mul(a0d[k], pd));
                const df den = df_add(pd, c.pinfd[k]);
                f = df_add(f, df_mul(c.c1d[k], df_div(num, den)));
                const float t = rcp_approx(den.hi);
                fp = fmaf(c.c1f[k] * fmaf(a0d[k].hi, c.pinff[k], -E0d[k].hi), t * t, fp);
            }
            pd = df_add(pd, {-(f.hi + f.lo) * rcp_approx(fp), 0.f});
        }
        // 3. one Newton step on f in FP64 and the fractions at its end (first order)
        const double p0 = df_to_double(pd);
        double ak[NF], f64 = -target;
        if constexpr (STEADY) {
            double dak[NF], fp64 = 0.0;
#pragma unroll
            for (int k = 0; k < NF; ++k) {
                ak[k] = a0[k];
                dak[k] = 0.0;
                if (!in[k]) continue;
                const double t = rcp_nr(p0 + c.pinf[k]);
                ak[k] = c.c1[k] * fma(a0[k], p0, q[II + k]) * t;
                dak[k] = c.c1[k] * fma(a0[k], c.pinf[k], -q[II + k]) * t * t;
                f64 += ak[k];
                fp64 += dak[k];
            }
            const double dp = df_widen(-(float)f64 * rcp_approx((float)fp64));
#pragma unroll
            for (int k = 0; k < NF - 1; ++k)
                if (in[k]) q[IA + k] = fma(dak[k], dp, ak[k]);
        } else {
            float dak[NF], fp = 0.f;
#pragma unroll
            for (int k = 0; k < NF; ++k) {
                ak[k] = a0[k];
                dak[k] = 0.f;
                if (!in[k]) continue;
                ak[k] = c.c1[k] * fma(a0[k], p0, q[II + k]) * rcp_nr(p0 + c.pinf[k]);
                const float t = rcp_approx(pd.hi + c.pinff[k]);
                dak[k] = c.c1f[k] * fmaf(a0d[k].hi, c.pinff[k], -E0d[k].hi) * t * t;
                f64 += ak[k];
                fp += dak[k];
            }
            // f' ~ 1/p leaves FP32 only for pressures beyond 1e30 (a phase energy that does
            // not belong to the cell's total energy): the fractions at p0 stand then
            const bool in_range = fabsf(fp) >= 0x1p-100f && fabsf(fp) <= 0x1p100f;
            const float dp = -narrow_rn(f64) * rcp_approx(fp);
#pragma unroll
            for (int k = 0; k < NF - 1; ++k)
                if (in[k]) q[IA + k] = ak[k] + df_widen(in_range ? dak[k] * dp : 0.f);
        }
    }
    // 4. the pressure of the total energy, the phase energies
    const double pressure = six_pressure<NF, NDIM>(q, e, eint);   // outside the test: the recovery takes it over
    if (any) {
        double an = 1.0;
#pragma unroll
        for (int k = 0; k < NF - 1; ++k) an -= q[IA + k];
#pragma unroll
        for (int k = 0; k < NF; ++k) q[II + k] = (k < NF - 1 ? q[IA + k] : an) * fma(c.G[k], pressure, c.P[k]);
    }
}

// Relaxation, primitive recovery and (RATE) the CFL rate of a stage's new state
// in one pass over it: the relaxed fractions and phase energies go back to q,
// the primitives to w.  In the epilogue of the last sweep the relaxation held up
// the sweep's barriers with 16 warps per SM (112x104x96 FP64: z sweep 700 us, then
// 44 us of recovery or 100 us of CFL pass; now 387 us and 137 or 151 us).
template <typename Real, int NF, int NDIM, bool RATE>
__global__ void __launch_bounds__(256) relax_prims_kernel(const PrimArgs a, const RelaxConst c) {
    using Lay = Layout<NF, NDIM, true>;
    constexpr int NS = Lay::NS, NQ = Lay::NQ, IA = Lay::IA, II = Lay::II;
    pdl_wait();
    const long long nc = a.g.ncell;
    double rate = 0.0;
    int bad = 0;
    double* qs = const_cast<double*>(a.q);
    Real* w = static_cast<Real*>(a.w);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nc;
         i += (long long)gridDim.x * blockDim.x) {
        double q[NQ];
#pragma unroll
        for (int v = 0; v < NQ; ++v) q[v] = qs[v * nc + i];
        relax6<NF, NDIM, sizeof(Real) == 4>(c, a.e, q);
#pragma unroll
        for (int v = IA; v < IA + NF - 1; ++v) qs[v * nc + i] = q[v];
#pragma unroll
        for (int v = II; v < II + NF; ++v) qs[v * nc + i] = q[v];
        Real wv[NS], c2;
        prims_cell<NF, NDIM, true>(q, a.e, wv, c2);   // shares 1/rho, energy and pressure with the relaxation
#pragma unroll
        for (int v = 0; v < NS; ++v) w[v * nc + i] = wv[v];
        if (RATE) {
            const double r = cell_cfl_rate<Real, NF, NDIM>(wv, c2, a.g, a.grid, a.grid_stride, i);
            if (__double2hiint(r) < 0) bad += 1;
            else rate = max_nonneg(rate, r);
        }
    }
    if (RATE) publish_block_rate(a, rate, bad);
}

// Primitive -> conserved (initial conditions), FP64.
template <int NF, int NDIM>
__global__ void __launch_bounds__(256) cons_kernel(Geometry g, EosConst e, const double* __restrict__ w,
                                                   double* __restrict__ q) {
    using Lay = Layout<NF, NDIM>;
    constexpr int NS = Lay::NS, IM = Lay::IM, IE = Lay::IE, IA = Lay::IA;
    const long long nc = g.ncell;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nc;
         i += (long long)gridDim.x * blockDim.x) {
        double s[NS];
#pragma unroll
        for (int v = 0; v < NS; ++v) s[v] = w[v * nc + i];
        double rho = s[0];
#pragma unroll
        for (int k = 1; k < NF; ++k) rho += s[k];
        double G = e.G_N, P = e.P_N;
#pragma unroll
        for (int k = 0; k < NF - 1; ++k) { G = fma(s[IA + k], e.dG[k], G); P = fma(s[IA + k], e.dP[k], P); }
        double ke = 0.0;
#pragma unroll
        for (int d = 0; d < NDIM; ++d) { ke = fma(s[IM + d], s[IM + d], ke); q[(IM + d) * nc + i] = rho * s[IM + d]; }
#pragma unroll
        for (int k = 0; k < NF; ++k) q[k * nc + i] = s[k];
        q[IE * nc + i] = fma(G, s[IE], P) + 0.5 * rho * ke;
#pragma unroll
        for (int k = 0; k < NF - 1; ++k) q[(IA + k) * nc + i] = s[IA + k];
    }
}

// Six-equation model: primitive (the five-equation variables, then the phase
// pressures p_k) -> conserved.  a_k r_k e_k = a_k (p_k + g_k pinf_k)/(g_k - 1)
// = a_k (G_k p_k + P_k), r E = sum_k a_k r_k e_k + r|u|^2/2; the primitive
// mixture-pressure row is not read.
template <int NF, int NDIM>
__global__ void __launch_bounds__(256) cons6_kernel(Geometry g, EosConst e, const double* __restrict__ w,
                                                    double* __restrict__ q) {
    using Lay = Layout<NF, NDIM, true>;
    constexpr int NQ = Lay::NQ, IM = Lay::IM, IE = Lay::IE, IA = Lay::IA, II = Lay::II;
    const long long nc = g.ncell;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nc;
         i += (long long)gridDim.x * blockDim.x) {
        double s[NQ];
#pragma unroll
        for (int v = 0; v < NQ; ++v) s[v] = w[v * nc + i];
        double rho = s[0];
#pragma unroll
        for (int k = 1; k < NF; ++k) rho += s[k];
        double ke = 0.0;
#pragma unroll
        for (int d = 0; d < NDIM; ++d) { ke = fma(s[IM + d], s[IM + d], ke); q[(IM + d) * nc + i] = rho * s[IM + d]; }
#pragma unroll
        for (int k = 0; k < NF; ++k) q[k * nc + i] = s[k];
        double aN = 1.0, esum = 0.0;
#pragma unroll
        for (int k = 0; k < NF - 1; ++k) {
            q[(IA + k) * nc + i] = s[IA + k];
            aN -= s[IA + k];
            const double E = s[IA + k] * fma(e.G_N + e.dG[k], s[II + k], e.P_N + e.dP[k]);
            q[(II + k) * nc + i] = E;
            esum += E;
        }
        const double EN = aN * fma(e.G_N, s[II + NF - 1], e.P_N);
        q[(II + NF - 1) * nc + i] = EN;
        q[IE * nc + i] = esum + EN + 0.5 * rho * ke;
    }
}

}  // namespace mfc
