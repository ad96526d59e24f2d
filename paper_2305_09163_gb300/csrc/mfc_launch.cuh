// Host-side launchers for the device templates.  Each translation unit
// instantiates them for one (arithmetic type, number of fluids) pair so the
// build compiles in parallel.
#pragma once
#include "mfc_device.cuh"

namespace mfc {

constexpr int kSweepThreads = 128;
constexpr int kElemThreads = 256;

// Chunks of kStreamThreads slots (edge cells) that one CTA of the x-stream
// kernel walks.  A CTA starts two slots early (both faces of its first cell), so
// k chunks finish 128 k - 2 slots; owning exactly that many leaves no nearly
// empty last chunk (2,048 owned slots took 17 chunks for the work of 16.02).
// Long runs save those two slots, short ones fill the chip: a launch of one
// chunk per CTA takes 10.7 us (1000 cells), a lone CTA's long walk ~6 us a chunk and
// four CTAs sharing an SM ~4.3 us for each, and with the fixed 16 chunks a 1000-cell row ran on one SM (79 us per launch) and a
// 65,000-cell block on half of them.  So k grows only once every SM has 16 CTAs to
// run, three to four times what it holds (five of the uniform two-fluid FP64 form, four
// of the others), where the walk's end is a small part; past 16 the two slots are 0.1%
// and nothing is left to save.
constexpr long long kStreamMaxChunks = 16;
constexpr long long kStreamMinBlocks = 152LL * 16;

inline long long stream_slots_per_block(long long total) {
    const long long chunks = (total + kStreamThreads - 3) / (kStreamThreads - 2);
    long long k = chunks / kStreamMinBlocks;
    if (k < 1) k = 1;
    if (k > kStreamMaxChunks) k = kStreamMaxChunks;
    return k * kStreamThreads - 2;
}

// Launch a kernel that begins with pdl_wait: it may be set up while the kernel
// ahead of it in the stream still ends, which hides the launch between them (8
// steps of a 1000-cell row 425 -> 355 us, with one memset and one copy per step
// fewer; five of a 301x201 plane 623 -> 530 us).
template <typename... P, typename... A>
cudaError_t launch_pdl(void (*kernel)(P...), unsigned blocks, int threads, size_t smem, cudaStream_t s, const A&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const cudaError_t rc = cudaLaunchKernelEx(&cfg, kernel, args...);
    if (rc != cudaSuccess) cudaGetLastError();   // reported here, not once more to whoever asks next
    return rc;
}

inline size_t stage_bytes_rt(int mask, int nq, size_t real_size) {
    return (size_t)nq * kStageSlots *
           (((mask & 1) ? real_size : 0) + ((mask & 2) ? sizeof(double) : 0) + ((mask & 4) ? sizeof(double) : 0));
}

// Launch one y/z stream kernel.  An entry built with staging (STAGE) gets its
// finish operands staged, dropping q0, then qs, then R from the staging while
// its shared memory would lower the number of CTAs resident per SM (the
// kernels are latency-bound: residency comes first).
template <typename Real, bool STAGE = false, typename Kernel>
cudaError_t launch_yz_stream(Kernel kernel, unsigned blocks, SweepArgs a, int nq, cudaStream_t s) {
    constexpr int threads = 32 * kRowsPerChunk;
    int mask = STAGE ? stage_mask(a) : 0;
    size_t dyn = 0;
    if (mask) {
        int occ0 = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ0, kernel, threads, 0);
        if (e != cudaSuccess) return e;
        for (; mask; mask &= ~(mask & 4 ? 4 : mask & 2 ? 2 : 1)) {
            dyn = stage_bytes_rt(mask, nq, sizeof(Real));
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
            if (e != cudaSuccess) return e;
            int occ = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, dyn);
            if (e != cudaSuccess) return e;
            if (occ >= occ0) break;
        }
        if (!mask) dyn = 0;
    }
    a.stage = mask;
    return launch_pdl(kernel, blocks, threads, dyn, s, a);
}

// SIX: the six-equation model (stream kernels, WENO5, uniform grids).
template <typename Real, int NF, bool LEARNED = false, int ORDER = 5, bool NONUNIF = false, bool SIX = false>
cudaError_t launch_sweep(SweepArgs a, int ndim, int dir, cudaStream_t s) {
    // FP64 x sweeps bounded to 4 CTAs per SM (128 registers): the stretched-grid,
    // six-equation and WENO3 variants, which take more when left unbounded; the
    // uniform WENO5 one fits 4 CTAs without a bound
    constexpr bool kBoundFp64 = NONUNIF || SIX || ORDER == 3;
    if (dir == 0) {
        const long long total = (long long)(a.g.n[0] + 2) * (a.g.ncell / a.g.n[0]);
        a.slots_per_block = stream_slots_per_block(total);
        const unsigned blocks = (unsigned)((total + a.slots_per_block - 1) / a.slots_per_block);
        if constexpr (LEARNED) {
            switch (ndim) {
                case 1: return launch_pdl(sweep_x_stream_learned_kernel<NF, 1>, blocks, kStreamThreads, 0, s, a);
                case 2: return launch_pdl(sweep_x_stream_learned_kernel<NF, 2>, blocks, kStreamThreads, 0, s, a);
                case 3: return launch_pdl(sweep_x_stream_learned_kernel<NF, 3>, blocks, kStreamThreads, 0, s, a);
                default: return cudaErrorInvalidValue;
            }
        } else if constexpr (sizeof(Real) == 8 && kBoundFp64) {
            switch (ndim) {
                case 1: return launch_pdl(sweep_x_stream_f64_kernel<NF, 1, ORDER, NONUNIF, SIX>, blocks, kStreamThreads, 0, s, a);
                case 2: return launch_pdl(sweep_x_stream_f64_kernel<NF, 2, ORDER, NONUNIF, SIX>, blocks, kStreamThreads, 0, s, a);
                case 3: return launch_pdl(sweep_x_stream_f64_kernel<NF, 3, ORDER, NONUNIF, SIX>, blocks, kStreamThreads, 0, s, a);
                default: return cudaErrorInvalidValue;
            }
        } else if constexpr (sizeof(Real) == 4 && !NONUNIF && !SIX) {
            switch (ndim) {
                case 1: return launch_pdl(sweep_x_stream_f32_kernel<NF, 1, ORDER>, blocks, kStreamThreads, 0, s, a);
                case 2: return launch_pdl(sweep_x_stream_f32_kernel<NF, 2, ORDER>, blocks, kStreamThreads, 0, s, a);
                case 3: return launch_pdl(sweep_x_stream_f32_kernel<NF, 3, ORDER>, blocks, kStreamThreads, 0, s, a);
                default: return cudaErrorInvalidValue;
            }
        } else {
            switch (ndim) {
                case 1: return launch_pdl(sweep_x_stream_kernel<Real, NF, 1, LEARNED, ORDER, NONUNIF, SIX>, blocks, kStreamThreads, 0, s, a);
                case 2: return launch_pdl(sweep_x_stream_kernel<Real, NF, 2, LEARNED, ORDER, NONUNIF, SIX>, blocks, kStreamThreads, 0, s, a);
                case 3: return launch_pdl(sweep_x_stream_kernel<Real, NF, 3, LEARNED, ORDER, NONUNIF, SIX>, blocks, kStreamThreads, 0, s, a);
                default: return cudaErrorInvalidValue;
            }
        }
    }
    const int t1 = (dir == 0) ? 1 : 0, t2 = (dir == 2) ? 1 : 2;
    if (NONUNIF || SIX || a.yz_stream) {   // non-uniform grids, six-equation model: the stream kernel only
        // y/z stream kernel, one CTA per 32 cells of the transverse plane and segment
        const unsigned blocks = (unsigned)((a.g.ncell / a.g.n[dir] + 31) / 32 * a.nseg);
        auto nq = [](int nd) { return 2 * NF + nd + (SIX ? NF : 0); };
        if constexpr (LEARNED) {
            switch (ndim * 4 + dir) {
                case 9: return launch_yz_stream<Real, true>(sweep_yz_stream_learned_kernel<NF, 2, 1>, blocks, a, nq(2), s);
                case 13: return launch_yz_stream<Real, true>(sweep_yz_stream_learned_kernel<NF, 3, 1>, blocks, a, nq(3), s);
                case 14: return launch_yz_stream<Real, true>(sweep_yz_stream_learned_kernel<NF, 3, 2>, blocks, a, nq(3), s);
                default: return cudaErrorInvalidValue;
            }
        } else if constexpr (sizeof(Real) == 8 && (kBoundFp64 || NF <= 2)) {
            switch (ndim * 4 + dir) {
                case 9: return launch_yz_stream<Real, !NONUNIF>(sweep_yz_stream_f64_kernel<NF, 2, 1, ORDER, NONUNIF, SIX>, blocks, a, nq(2), s);
                case 13: return launch_yz_stream<Real, !NONUNIF>(sweep_yz_stream_f64_kernel<NF, 3, 1, ORDER, NONUNIF, SIX>, blocks, a, nq(3), s);
                case 14: return launch_yz_stream<Real, !NONUNIF>(sweep_yz_stream_f64_kernel<NF, 3, 2, ORDER, NONUNIF, SIX>, blocks, a, nq(3), s);
                default: return cudaErrorInvalidValue;
            }
        } else if constexpr (sizeof(Real) == 8) {
            switch (ndim * 4 + dir) {
                case 9: return launch_yz_stream<Real, true>(sweep_yz_stream_f64b3_kernel<NF, 2, 1>, blocks, a, nq(2), s);
                case 13: return launch_yz_stream<Real, true>(sweep_yz_stream_f64b3_kernel<NF, 3, 1>, blocks, a, nq(3), s);
                case 14: return launch_yz_stream<Real, true>(sweep_yz_stream_f64b3_kernel<NF, 3, 2>, blocks, a, nq(3), s);
                default: return cudaErrorInvalidValue;
            }
        } else if constexpr (SIX && sizeof(Real) == 4) {
            switch (ndim * 4 + dir) {
                case 9: return launch_yz_stream<Real, true>(sweep_yz_stream_six32_kernel<NF, 2, 1, ORDER, NONUNIF>, blocks, a, nq(2), s);
                case 13: return launch_yz_stream<Real, true>(sweep_yz_stream_six32_kernel<NF, 3, 1, ORDER, NONUNIF>, blocks, a, nq(3), s);
                case 14: return launch_yz_stream<Real, true>(sweep_yz_stream_six32_kernel<NF, 3, 2, ORDER, NONUNIF>, blocks, a, nq(3), s);
                default: return cudaErrorInvalidValue;
            }
        } else if constexpr (sizeof(Real) == 4 && !NONUNIF) {
            switch (ndim * 4 + dir) {
                case 9: return launch_yz_stream<Real, true>(sweep_yz_stream_f32_kernel<NF, 2, 1, ORDER>, blocks, a, nq(2), s);
                case 13: return launch_yz_stream<Real, true>(sweep_yz_stream_f32_kernel<NF, 3, 1, ORDER>, blocks, a, nq(3), s);
                case 14: return launch_yz_stream<Real, true>(sweep_yz_stream_f32_kernel<NF, 3, 2, ORDER>, blocks, a, nq(3), s);
                default: return cudaErrorInvalidValue;
            }
        } else {
            switch (ndim * 4 + dir) {
                case 9: return launch_yz_stream<Real>(sweep_yz_stream_f32_nu_kernel<NF, 2, 1>, blocks, a, nq(2), s);
                case 13: return launch_yz_stream<Real>(sweep_yz_stream_f32_nu_kernel<NF, 3, 1>, blocks, a, nq(3), s);
                case 14: return launch_yz_stream<Real>(sweep_yz_stream_f32_nu_kernel<NF, 3, 2>, blocks, a, nq(3), s);
                default: return cudaErrorInvalidValue;
            }
        }
    }
    if constexpr (NONUNIF || SIX) return cudaErrorInvalidValue;
    const long long warps = (long long)((a.g.n[t1] + 31) / 32) * a.nseg * a.g.n[t2];
    const unsigned blocks = (unsigned)((warps * 32 + kSweepThreads - 1) / kSweepThreads);
    switch (ndim * 4 + dir) {
        case 9: sweep_kernel<Real, NF, 2, 1, LEARNED, ORDER><<<blocks, kSweepThreads, 0, s>>>(a); break;
        case 13: sweep_kernel<Real, NF, 3, 1, LEARNED, ORDER><<<blocks, kSweepThreads, 0, s>>>(a); break;
        case 14: sweep_kernel<Real, NF, 3, 2, LEARNED, ORDER><<<blocks, kSweepThreads, 0, s>>>(a); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

inline unsigned elem_blocks(long long n) {
    long long b = (n + kElemThreads - 1) / kElemThreads;
    const long long cap = 152LL * 16;
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (unsigned)b;
}

template <typename Real, int NF, bool SIX = false>
cudaError_t launch_prims(const PrimArgs& a, int ndim, bool rate, cudaStream_t s) {
    const unsigned blocks = elem_blocks(a.g.ncell);
    switch (ndim * 2 + (rate ? 1 : 0)) {
        case 2: return launch_pdl(prims_kernel<Real, NF, 1, false, SIX>, blocks, kElemThreads, 0, s, a);
        case 3: return launch_pdl(prims_kernel<Real, NF, 1, true, SIX>, blocks, kElemThreads, 0, s, a);
        case 4: return launch_pdl(prims_kernel<Real, NF, 2, false, SIX>, blocks, kElemThreads, 0, s, a);
        case 5: return launch_pdl(prims_kernel<Real, NF, 2, true, SIX>, blocks, kElemThreads, 0, s, a);
        case 6: return launch_pdl(prims_kernel<Real, NF, 3, false, SIX>, blocks, kElemThreads, 0, s, a);
        case 7: return launch_pdl(prims_kernel<Real, NF, 3, true, SIX>, blocks, kElemThreads, 0, s, a);
        default: return cudaErrorInvalidValue;
    }
}

// Six-equation model: relaxation and primitive recovery of a stage's new state.
template <typename Real, int NF>
cudaError_t launch_relax_prims(const PrimArgs& a, const RelaxConst& c, int ndim, bool rate, cudaStream_t s) {
    const unsigned blocks = elem_blocks(a.g.ncell);
    switch (ndim * 2 + (rate ? 1 : 0)) {
        case 2: return launch_pdl(relax_prims_kernel<Real, NF, 1, false>, blocks, kElemThreads, 0, s, a, c);
        case 3: return launch_pdl(relax_prims_kernel<Real, NF, 1, true>, blocks, kElemThreads, 0, s, a, c);
        case 4: return launch_pdl(relax_prims_kernel<Real, NF, 2, false>, blocks, kElemThreads, 0, s, a, c);
        case 5: return launch_pdl(relax_prims_kernel<Real, NF, 2, true>, blocks, kElemThreads, 0, s, a, c);
        case 6: return launch_pdl(relax_prims_kernel<Real, NF, 3, false>, blocks, kElemThreads, 0, s, a, c);
        case 7: return launch_pdl(relax_prims_kernel<Real, NF, 3, true>, blocks, kElemThreads, 0, s, a, c);
        default: return cudaErrorInvalidValue;
    }
}

// Characteristic boundary rates (cbc_rates_kernel): total = boundary cells.
template <typename Real, int NF>
cudaError_t launch_cbc(const SweepArgs& a, int ndim, long long total, cudaStream_t s) {
    const unsigned blocks = elem_blocks(total);
    switch (ndim) {
        case 1: cbc_rates_kernel<Real, NF, 1><<<blocks, kElemThreads, 0, s>>>(a, total); break;
        case 2: cbc_rates_kernel<Real, NF, 2><<<blocks, kElemThreads, 0, s>>>(a, total); break;
        case 3: cbc_rates_kernel<Real, NF, 3><<<blocks, kElemThreads, 0, s>>>(a, total); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <int NF>
cudaError_t launch_cons6(const Geometry& g, const EosConst& e, const double* w, double* q, int ndim,
                         cudaStream_t s) {
    const unsigned blocks = elem_blocks(g.ncell);
    switch (ndim) {
        case 1: cons6_kernel<NF, 1><<<blocks, kElemThreads, 0, s>>>(g, e, w, q); break;
        case 2: cons6_kernel<NF, 2><<<blocks, kElemThreads, 0, s>>>(g, e, w, q); break;
        case 3: cons6_kernel<NF, 3><<<blocks, kElemThreads, 0, s>>>(g, e, w, q); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <int NF>
cudaError_t launch_cons(const Geometry& g, const EosConst& e, const double* w, double* q, int ndim,
                        cudaStream_t s) {
    const unsigned blocks = elem_blocks(g.ncell);
    switch (ndim) {
        case 1: cons_kernel<NF, 1><<<blocks, kElemThreads, 0, s>>>(g, e, w, q); break;
        case 2: cons_kernel<NF, 2><<<blocks, kElemThreads, 0, s>>>(g, e, w, q); break;
        case 3: cons_kernel<NF, 3><<<blocks, kElemThreads, 0, s>>>(g, e, w, q); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// Host: the EOS constants of N stiffened-gas fluids (Sec. 2.1) as the kernels
// take them, relative to fluid N (whose fraction is 1 - sum of the others):
// Gamma_k = 1/(g_k - 1), Pi_k = g_k pinf_k/(g_k - 1), and for the six-equation
// model's frozen sound speed r c^2 = sum_k a_k g_k (p + pinf_k) the pairs
// (g_k, g_k pinf_k).  Every entry point builds its constants here.
inline EosConst make_eos_const(int N, const double* gamma, const double* pi_inf) {
    double G[3], P[3];
    for (int k = 0; k < N; ++k) {
        G[k] = 1.0 / (gamma[k] - 1.0);
        P[k] = gamma[k] * pi_inf[k] / (gamma[k] - 1.0);
    }
    EosConst e{};
    e.G_N = G[N - 1];
    e.P_N = P[N - 1];
    e.A_N = gamma[N - 1];
    e.B_N = gamma[N - 1] * pi_inf[N - 1];
    for (int k = 0; k < 2; ++k) {
        const bool on = k < N - 1;
        e.dG[k] = on ? G[k] - G[N - 1] : 0.0;
        e.dP[k] = on ? P[k] - P[N - 1] : 0.0;
        e.dA[k] = on ? gamma[k] - gamma[N - 1] : 0.0;
        e.dB[k] = on ? gamma[k] * pi_inf[k] - gamma[N - 1] * pi_inf[N - 1] : 0.0;
    }
    return e;
}

// Host: the six-equation relaxation's constants in the precisions it takes.
inline RelaxConst make_relax_const(int N, const double* gamma, const double* pi_inf, const EosConst& e) {
    RelaxConst c{};
    for (int k = 0; k < N; ++k) {
        c.pinf[k] = pi_inf[k];
        c.c1[k] = (gamma[k] - 1.0) / gamma[k];
        c.G[k] = k < N - 1 ? e.G_N + e.dG[k] : e.G_N;
        c.P[k] = k < N - 1 ? e.P_N + e.dP[k] : e.P_N;
        c.pinfd[k] = df_split(c.pinf[k]);
        c.c1d[k] = df_split(c.c1[k]);
        c.pinff[k] = (float)c.pinf[k];
        c.c1f[k] = c.c1d[k].hi;
    }
    c.P_N = df_split(e.P_N);
    c.G_N = (float)e.G_N;
    for (int k = 0; k < 2; ++k) {
        c.dP[k] = df_split(e.dP[k]);
        c.dG[k] = (float)e.dG[k];
    }
    return c;
}

// Host: cells per thread along direction dir of a marching sweep; halved while
// fewer than ~8 warps per SM would be resident.
inline int marching_segment(long long ncell, int n_dir) {
    const long long trans = ncell / n_dir;
    int L = 64;
    while (L > 8 && trans * ((n_dir + L - 1) / L) < 152LL * 4 * kSweepThreads) L /= 2;
    return L;
}

// Host: cells per segment of a y/z stream sweep.  A segment of L cells walks
// ceil((L + 2)/4) chunks of 4 edge cells, two of which a neighbour repeats, so
// only lengths 4 m - 2 (and what is left at the end) are taken: 128 cells took
// 33 chunks for the work of 32.5.  Long segments repeat fewer cells, short ones
// fill the chip, so the length with the smallest estimate is taken, in units of
// the time an SM with all its CTAs spends per chunk:
//     chunks of all CTAs / 152 SMs  +  tail * chunks of one CTA,
// each CTA charged a quarter of a chunk for its first rows.  The tail is what a
// CTA's walk adds when it does not overlap others: an SM holds 4 FP64 CTAs, and
// one alone takes 7.5 us per chunk where four share it at 4.15 us each; it holds
// 8 FP32 ones, 2.1 us against 0.55 us.  Measured over lengths 8-254 the estimate's
// choice is within 5% of the best one: FP64 y sweep of 64^3 97 -> 82 us, 100x90x77
// 234 -> 182, 600x500 98 -> 87, 128^3 577 -> 504, 256^3 3.76 -> 3.69 ms, against
// the former rule (lengths halved from 128 or 64 until ~8 warps per SM had work).
// The search ends where the tail alone, on top of the chunks that no length saves,
// is above the least estimate so far: 3-50 lengths for the usual sizes, 0.03-0.5 us
// of host time a launch (all lengths up to n_dir: 2.5 us for 1,000 cells, 250 us for
// 100,000).
inline int stream_segment(long long ncell, int n_dir, bool fp64) {
    const long long columns = (ncell / n_dir + 31) / 32;
    const double tail = fp64 ? 1.0 : 2.5, start = 0.25;
    const double floor = 0.25 * n_dir * (double)columns / 152.0 * (1.0 - 1e-12);
    int best = n_dir;
    double least = 0.0;
    for (int L = 2;; L += 4) {
        const int whole = n_dir / L, rest = n_dir % L;
        const double walk = (L + 2) / 4 + start;
        if (L > 2 && floor + tail * walk > least) break;
        const double all = (whole * walk + (rest ? (rest + 5) / 4 + start : 0.0)) * (double)columns;
        const double t = all / 152.0 + tail * walk;
        if (L == 2 || t < least) {
            least = t;
            best = L;
        }
        if (L >= n_dir) break;
    }
    return best;
}

// Explicitly instantiated in the mfc_inst_*.cu units.
#define MFC_DECLARE_INSTANCES(Real, NF)                                                         \
    extern template cudaError_t launch_sweep<Real, NF>(SweepArgs, int, int, cudaStream_t); \
    extern template cudaError_t launch_prims<Real, NF>(const PrimArgs&, int, bool, cudaStream_t); \
    extern template cudaError_t launch_cbc<Real, NF>(const SweepArgs&, int, long long, cudaStream_t);

MFC_DECLARE_INSTANCES(double, 1)
MFC_DECLARE_INSTANCES(double, 2)
MFC_DECLARE_INSTANCES(double, 3)
MFC_DECLARE_INSTANCES(float, 1)
MFC_DECLARE_INSTANCES(float, 2)
MFC_DECLARE_INSTANCES(float, 3)
extern template cudaError_t launch_sweep<float, 1, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<float, 2, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<float, 3, true>(SweepArgs, int, int, cudaStream_t);
// non-uniform grids (mfc_inst_*_nu_*.cu)
extern template cudaError_t launch_sweep<double, 1, false, 5, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<double, 2, false, 5, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<double, 3, false, 5, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<float, 1, false, 5, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<float, 2, false, 5, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<float, 3, false, 5, true>(SweepArgs, int, int, cudaStream_t);
// WENO3 (mfc_inst_*_w3_*.cu)
extern template cudaError_t launch_sweep<double, 1, false, 3>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<double, 2, false, 3>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<double, 3, false, 3>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<float, 1, false, 3>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<float, 2, false, 3>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<float, 3, false, 3>(SweepArgs, int, int, cudaStream_t);
// six-equation model (mfc_inst_*_six_*.cu; with a stretched grid or WENO3: mfc_inst_*_six_nu_*, *_six_w3_*)
extern template cudaError_t launch_sweep<double, 2, false, 5, true, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<double, 3, false, 5, true, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<float, 2, false, 5, true, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<float, 3, false, 5, true, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<double, 2, false, 3, false, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<double, 3, false, 3, false, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<float, 2, false, 3, false, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<float, 3, false, 3, false, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<double, 2, false, 5, false, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<double, 3, false, 5, false, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<float, 2, false, 5, false, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_sweep<float, 3, false, 5, false, true>(SweepArgs, int, int, cudaStream_t);
extern template cudaError_t launch_prims<double, 2, true>(const PrimArgs&, int, bool, cudaStream_t);
extern template cudaError_t launch_prims<double, 3, true>(const PrimArgs&, int, bool, cudaStream_t);
extern template cudaError_t launch_prims<float, 2, true>(const PrimArgs&, int, bool, cudaStream_t);
extern template cudaError_t launch_prims<float, 3, true>(const PrimArgs&, int, bool, cudaStream_t);
extern template cudaError_t launch_relax_prims<double, 2>(const PrimArgs&, const RelaxConst&, int, bool, cudaStream_t);
extern template cudaError_t launch_relax_prims<double, 3>(const PrimArgs&, const RelaxConst&, int, bool, cudaStream_t);
extern template cudaError_t launch_relax_prims<float, 2>(const PrimArgs&, const RelaxConst&, int, bool, cudaStream_t);
extern template cudaError_t launch_relax_prims<float, 3>(const PrimArgs&, const RelaxConst&, int, bool, cudaStream_t);
extern template cudaError_t launch_cons6<2>(const Geometry&, const EosConst&, const double*, double*, int, cudaStream_t);
extern template cudaError_t launch_cons6<3>(const Geometry&, const EosConst&, const double*, double*, int, cudaStream_t);
extern template cudaError_t launch_cons<1>(const Geometry&, const EosConst&, const double*, double*, int, cudaStream_t);
extern template cudaError_t launch_cons<2>(const Geometry&, const EosConst&, const double*, double*, int, cudaStream_t);
extern template cudaError_t launch_cons<3>(const Geometry&, const EosConst&, const double*, double*, int, cudaStream_t);

}  // namespace mfc
