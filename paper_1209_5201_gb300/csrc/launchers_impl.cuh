// Definitions of Launch<PREC>: lattice dispatch and launch geometry.
#pragma once

#include "k_aux.cuh"
#include "k_fluxes.cuh"
#include "k_init.cuh"
#include "k_step_cellwarp.cuh"
#include "k_step_cellwarp64.cuh"
#include "k_step_direct.cuh"
#include "k_step_staged.cuh"
#include "launchers.h"

namespace lbm {

template <int PREC>
struct Consts;
template <> struct Consts<LBM_FP64> {
    static const KConsts<double> &get(const SolverImpl &s) { return s.kd; }
};
template <> struct Consts<LBM_FP32> {
    static const KConsts<float> &get(const SolverImpl &s) { return s.kf; }
};
template <> struct Consts<LBM_BF16DEV> {
    static const KConsts<float> &get(const SolverImpl &s) { return s.kf; }
};
template <> struct Consts<LBM_BF16SHIFT> {
    static const KConsts<float> &get(const SolverImpl &s) { return s.kf; }
};

template <class C>
double weight_sum(const KConsts<C> &k) {
    double s = 0.0;
    for (int a = 0; a < k.Q; ++a) s += (double)k.w[a];
    return s;
}

inline int aux_blocks(long long n) {
    long long b = (n + kAuxThreads - 1) / kAuxThreads;
    if (b > 152 * 16) b = 152 * 16;
    return (int)(b < 1 ? 1 : b);
}

#define LBM_DISPATCH_Q(Q_, ...)                                 \
    switch (Q_) {                                               \
    case 17: { constexpr int QQ = 17; __VA_ARGS__; } break;     \
    case 25: { constexpr int QQ = 25; __VA_ARGS__; } break;     \
    case 37: { constexpr int QQ = 37; __VA_ARGS__; } break;     \
    default: return (int)cudaErrorInvalidValue;                 \
    }

// ---- direct kernel variants {BX, MINB, CS, RS} ----------------------------------
// RS: rows per block.  MINB < 0: the format's own choice (default_blocks).
struct DirectVariants {
    static constexpr int n = 9;
    static constexpr int v[n][4] = {{128, -1, 0, 1}, {128, 7, 0, 1}, {128, 6, 0, 1}, {256, 0, 0, 1},
                                    {128, 0, 1, 1}, {192, 0, 0, 1}, {128, 0, 0, 2}, {128, 5, 0, 1},
                                    {128, 0, 0, 1}};
};
// Blocks per SM that variant 0 asks the register allocator for, by what
// measured fastest untuned, us per step on 4096 x 2048 / 2050 x 1023 /
// 1000 x 500 with this request and with none: FP32 D2Q37 363 / 98.2 / 26.1 and
// 372 / 101.6 / 28.2 (5), D2Q25 247 / 67.9 / 16.5 and 254 / 73.7 / 21.2 (7),
// D2Q17 178 / 49.1 / 10.6 and 178 / 49.6 / 11.4 (7); BF16DEV D2Q37 293 / 83.9 /
// 24.2 and 392 / 111.5 / 28.1 (6), D2Q25 249 / 72.0 / 20.5 and 361 / 102.4 / 23.1
// (6), D2Q17 equal (7); BF16SHIFT D2Q37 236 / 69.0 / 19.3 and 307 / 87.6 / 21.8 (7),
// D2Q25 194 / 56.0 / 15.1 and 224 / 65.2 / 18.0 (7), D2Q17 equal (7).  FP64 is bound
// by its FP64 instructions: none is best throughout.
template <int Q, int PREC>
constexpr int default_blocks() {
    if (PREC == LBM_FP64) return 0;
    if (PREC == LBM_FP32) return Q == 37 ? 5 : 7;
    if (PREC == LBM_BF16DEV) return Q == 17 ? 7 : 6;
    return 7;
}

template <int Q, int PREC, int BX, int MINB, bool CS, int RS>
int launch_direct(SolverImpl &s, int src, int dst) {
    using S = typename Store<PREC>::S;
    const auto &k = Consts<PREC>::get(s);
    // blocks of BX columns never straddle two x-tiles
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(k.nt * ((k.tw + BX - 1) / BX), (s.p.Ny + RS - 1) / RS);
    cfg.blockDim = dim3(BX);
    cfg.stream = s.stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const S *fin = (const S *)s.f[src];
    S *fout = (S *)s.f[dst];
    const float *rin = s.rho[src];
    float *rout = s.rho[dst];
    auto go = [&](auto pc, auto iso2) {
        return (int)cudaLaunchKernelEx(
            &cfg, k_step_direct<Q, PREC, BX, MINB, CS, RS, decltype(pc)::value, decltype(iso2)::value>,
            fin, fout, rin, rout, k, s.kw);
    };
    // a pitch class: offsets as instruction immediates, else from the
    // constants; compiled for the one-row 128-column shapes of the 37-velocity
    // lattice and, for the others, for variant 0's
    auto by_pitch = [&](auto iso2) {
        if constexpr (BX == 128 && RS == 1 &&
                      (Q == 37 || (MINB == default_blocks<Q, PREC>() && !CS))) {
            constexpr int P0 = pitch_class(PREC, 0), P1 = pitch_class(PREC, 1),
                          P2 = pitch_class(PREC, 2);
            if (k.pitch == P0) return go(std::integral_constant<int, P0>{}, iso2);
            if (k.pitch == P1) return go(std::integral_constant<int, P1>{}, iso2);
            if (k.pitch == P2) return go(std::integral_constant<int, P2>{}, iso2);
        }
        return go(std::integral_constant<int, 0>{}, iso2);
    };
    // variant 0's shape also with the second-order isothermal equilibrium of the
    // 17- and 25-velocity lattices compiled in, us per step on 2050 x 1023 with
    // and without (the pitch in both): D2Q25 FP32 66.7 and 67.9, BF16DEV 57.7 and
    // 72.0, BF16SHIFT 48.1 and 56.0, FP64 792 and 1026; D2Q17 46.3 / 49.1, 43.0 / 50.0,
    // 38.7 / 45.2, 569 / 743.  (The fourth-order thermal one compiled in gained
    // nothing on D2Q37: FP32 366.7 against 363, BF16SHIFT 246 against 236.)
    if constexpr (Q != 37 && BX == 128 && RS == 1 && !CS && MINB == default_blocks<Q, PREC>())
        if (k.eq_order == 2 && !k.thermal && !k.const_tau) return by_pitch(std::true_type{});
    return by_pitch(std::false_type{});
}

// One lattice's direct-kernel variants (the 37-velocity ones, with their
// pitch-class instantiations, compile in a translation unit of their own).
template <int PREC, int Q>
int step_q(SolverImpl &s, int src, int dst, int variant) {
    using V = DirectVariants;
#define LBM_DIRECT_CASE(I)                                                                  \
    case I:                                                                                 \
        return launch_direct<Q, PREC, V::v[I][0],                                           \
                             (V::v[I][1] < 0 ? default_blocks<Q, PREC>() : V::v[I][1]),     \
                             (V::v[I][2] != 0), V::v[I][3]>(s, src, dst);
    switch (variant) {
        LBM_DIRECT_CASE(0)
        LBM_DIRECT_CASE(1)
        LBM_DIRECT_CASE(2)
        LBM_DIRECT_CASE(3)
        LBM_DIRECT_CASE(4)
        LBM_DIRECT_CASE(5)
        LBM_DIRECT_CASE(6)
        LBM_DIRECT_CASE(7)
        LBM_DIRECT_CASE(8)
    default: break;
    }
#undef LBM_DIRECT_CASE
    return (int)cudaErrorInvalidValue;
}

template <int PREC>
int Launch<PREC>::step(SolverImpl &s, int src, int dst, int variant) {
    switch (s.L.Q) {
    case 17: return step_q<PREC, 17>(s, src, dst, variant);
    case 25: return step_q<PREC, 25>(s, src, dst, variant);
    case 37: return step_q<PREC, 37>(s, src, dst, variant);
    default: break;
    }
    return (int)cudaErrorInvalidValue;
}

template <int PREC>
int Launch<PREC>::direct_variants() {
    // the last shape, no request, is FP64's variant 0
    return PREC == LBM_FP64 ? DirectVariants::n - 1 : DirectVariants::n;
}

template <int PREC>
bool Launch<PREC>::direct_repeats(int Q, int variant) {
    using V = DirectVariants;
    const int blocks = Q == 37   ? default_blocks<37, PREC>()
                       : Q == 25 ? default_blocks<25, PREC>()
                                 : default_blocks<17, PREC>();
    return variant > 0 && V::v[variant][0] == V::v[0][0] && V::v[variant][1] == blocks &&
           V::v[variant][2] == V::v[0][2] && V::v[variant][3] == V::v[0][3];
}

template <int PREC>
int Launch<PREC>::step_cellwarp(SolverImpl &s, int src, int dst) {
    using S = typename Store<PREC>::S;
    const auto &k = Consts<PREC>::get(s);
    const long long cells = (long long)s.p.Nx * s.p.Ny;
    if (cells > 0x7fffffffLL) return (int)cudaErrorInvalidValue;
    // programmatic dependent launch: a step's grid is launched while the
    // previous one runs and waits for it on the device (griddepcontrol.wait),
    // which hides the launch latency that dominates a step of a few thousand
    // cells
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cells);
    cfg.blockDim = dim3(32);
    cfg.stream = s.stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const S *fin = (const S *)s.f[src];
    S *fout = (S *)s.f[dst];
    if constexpr (PREC == LBM_FP64) {
        cfg.gridDim = dim3((unsigned)((cells + kCellWarps - 1) / kCellWarps));
        cfg.blockDim = dim3(32 * kCellWarps);
        LBM_DISPATCH_Q(s.L.Q, return (int)cudaLaunchKernelEx(&cfg, k_step_cellwarp64<QQ>, fin, fout,
                                                              k, s.lanes));
    } else {
        const float *rin = s.rho[src];
        float *rout = s.rho[dst];
        LBM_DISPATCH_Q(s.L.Q, return (int)cudaLaunchKernelEx(&cfg, k_step_cellwarp<QQ, PREC>, fin,
                                                              fout, rin, rout, k, s.kw));
    }
    return (int)cudaErrorInvalidValue;
}

// n steps of the one-warp-per-cell kernel from buffer src in one launch, or
// cudaErrorNotSupported where a launch per step it is: FP32 / BF16 storage, or
// more cells than resident warps.  Up to 64 cells run on one 16-CTA cluster
// (one cell per SM sub-partition: the FP64 chain of one cell is then a step's
// length, and the cluster barrier and a read of distributed shared memory are
// cheaper than the grid barrier and L2); more cells would queue on the
// cluster's FP64 units, so they spread over every SM.
template <int PREC>
int Launch<PREC>::steps_cellwarp(SolverImpl &s, int src, int n) {
    if constexpr (PREC != LBM_FP64) {
        return (int)cudaErrorNotSupported;
    } else {
        const long long cells = (long long)s.p.Nx * s.p.Ny;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        cfg.stream = s.stream;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        const double *fin = (const double *)s.f[src];
        double *fout = (double *)s.f[src ^ (n & 1)];
        if (cells <= kCellClusterCells && s.cell_cluster >= 0) {
            unsigned cl = 1;
            while (cl * kCellWarps < cells) cl *= 2;
            cfg.gridDim = dim3(cl);
            cfg.blockDim = dim3(32 * kCellWarps);
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = cl;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            LBM_DISPATCH_Q(s.L.Q, {
                auto kern = k_steps_cellwarp64_cluster<QQ>;
                if (s.cell_cluster == 0) {       // once per solver: does it schedule here?
                    cudaError_t e = cudaFuncSetAttribute(
                        kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
                    int fit = 0;
                    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&fit, kern, &cfg);
                    s.cell_cluster = e == cudaSuccess && fit >= 1 ? 1 : -1;
                    cudaGetLastError();          // not an error of the caller's
                }
                if (s.cell_cluster > 0)
                    return (int)cudaLaunchKernelEx(&cfg, kern, fin, fout, s.kd, s.lanes, n);
            });
        }
        const long long sms = s.sm_count;
        int warps = kCellWarps;              // per block: one block per SM
        while (warps * sms < cells) warps += kCellWarps;
        if (warps > kCellMaxWarps) return (int)cudaErrorNotSupported;
        cfg.gridDim = dim3((unsigned)((cells + warps - 1) / warps));
        cfg.blockDim = dim3(32 * warps);
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
        double *f0 = (double *)s.f[src], *f1 = (double *)s.f[src ^ 1];
        unsigned *bar = s.bar;
        int *err = s.derr;
        LBM_DISPATCH_Q(s.L.Q, {
            cudaError_t e =
                warps == kCellWarps
                    ? cudaLaunchKernelEx(&cfg, k_steps_cellwarp64_grid<QQ, kCellWarps>, f0, f1, s.kd,
                                         s.lanes, n, bar, err)
                    : cudaLaunchKernelEx(&cfg, k_steps_cellwarp64_grid<QQ, kCellMaxWarps>, f0, f1,
                                         s.kd, s.lanes, n, bar, err);
            if (e == cudaErrorCooperativeLaunchTooLarge) {
                cudaGetLastError();          // fewer SMs than the device has: a launch per step
                e = cudaErrorNotSupported;
            }
            return (int)e;
        });
        return (int)cudaErrorInvalidValue;
    }
}

// ---- TMA-staged kernel variants (tile TX x TY, ring of STAGES, CPT cells per
// consumer thread); the autotuner picks one per solver ------------------------
template <int PREC> struct Variants;
template <> struct Variants<LBM_FP32> {
    static constexpr int n = 4;
    static constexpr int v[n][4] = {{128, 2, 4, 1}, {128, 4, 2, 1}, {128, 4, 2, 2}, {64, 4, 4, 1}};
};
template <> struct Variants<LBM_FP64> {
    static constexpr int n = 2;
    static constexpr int v[n][4] = {{64, 2, 4, 1}, {64, 4, 2, 1}};
};
template <> struct Variants<LBM_BF16DEV> {
    static constexpr int n = 2;
    static constexpr int v[n][4] = {{128, 2, 4, 1}, {128, 4, 3, 1}};
};
// not built for BF16SHIFT (the direct kernel is the fast path of wide grids)
template <> struct Variants<LBM_BF16SHIFT> {
    static constexpr int n = 0;
    static constexpr int v[1][4] = {{0, 0, 0, 0}};
};

template <int Q, int PREC, int TX, int TY, int ST, int CPT>
int launch_staged(SolverImpl &s, int src, int dst) {
    using Cfg = StagedCfg<Q, PREC, TX, TY, ST, CPT>;
    using S = typename Store<PREC>::S;
    auto kern = k_step_staged<Q, PREC, TX, TY, ST, CPT>;
    int dev = 0;
    cudaGetDevice(&dev);
    static bool attr_set[64] = {false};
    if (dev < 64 && !attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             Cfg::kSmem);
        if (e != cudaSuccess) return (int)e;
        attr_set[dev] = true;
    }
    if (s.nt != 1) return (int)cudaErrorNotSupported;    // one x-tile grids only
    if (encode_tensor_maps(s, TX, TY)) return (int)cudaErrorInvalidValue;
    const int ntiles = ((s.p.Nx + TX - 1) / TX) * ((s.p.Ny + TY - 1) / TY);
    const int grid = ntiles < s.sm_count ? ntiles : s.sm_count;
    const auto &k = Consts<PREC>::get(s);
    kern<<<grid, Cfg::kThreads, Cfg::kSmem, s.stream>>>(
        s.tm_f[src], s.tm_r[src], (const S *)s.f[src], (S *)s.f[dst], s.rho[src], s.rho[dst],
        s.derr, k, s.kw);
    return (int)cudaGetLastError();
}

template <int PREC>
int Launch<PREC>::staged_variants() { return Variants<PREC>::n; }

template <int PREC>
int Launch<PREC>::step_staged(SolverImpl &s, int src, int dst, int variant) {
    using V = Variants<PREC>;
    if (variant < 0 || variant >= V::n) return (int)cudaErrorInvalidValue;
#define LBM_VARIANT_CASE(I)                                                              \
    case I:                                                                              \
        if constexpr (I < V::n) {                                                        \
            LBM_DISPATCH_Q(s.L.Q, return (launch_staged<QQ, PREC, V::v[I][0], V::v[I][1],  \
                                                        V::v[I][2], V::v[I][3]>(s, src, dst))); \
        }                                                                                \
        break;
    switch (variant) {
        LBM_VARIANT_CASE(0)
        LBM_VARIANT_CASE(1)
        LBM_VARIANT_CASE(2)
        LBM_VARIANT_CASE(3)
    default: break;
    }
#undef LBM_VARIANT_CASE
    return (int)cudaErrorInvalidValue;
}

template <int PREC>
int Launch<PREC>::init(SolverImpl &s, const double *rho, const double *ux, const double *uy,
                       const double *T, double *partials, int *nblocks) {
    using S = typename Store<PREC>::S;
    const auto &k = Consts<PREC>::get(s);
    *nblocks = (int)init_blocks(k);
    double *prev_u = s.prev, *prev_T = s.prev + (long long)s.p.Nx * s.p.Ny;
    LBM_DISPATCH_Q(s.L.Q, (k_init<QQ, PREC><<<*nblocks, kInitThreads, 0, s.stream>>>(
                               (S *)s.f[s.cur], s.rho[s.cur], k, rho, ux, uy, T, s.p.rho0,
                               s.p.noise_amp, s.p.seed, prev_u, prev_T, weight_sum(k),
                               partials)));
    return (int)cudaGetLastError();
}

template <int PREC>
int Launch<PREC>::plane_to_f64(SolverImpl &s, int a, double *out) {
    using S = typename Store<PREC>::S;
    const auto &k = Consts<PREC>::get(s);
    const long long n = (long long)s.p.Nx * s.p.Ny;
    LBM_DISPATCH_Q(s.L.Q, (k_plane_to_f64<QQ, PREC><<<aux_blocks(n), kAuxThreads, 0, s.stream>>>(
                               (const S *)s.f[s.cur], s.rho[s.cur], k, a, out)));
    return (int)cudaGetLastError();
}

template <int PREC>
int Launch<PREC>::plane_from_f64(SolverImpl &s, int a, const double *in) {
    using S = typename Store<PREC>::S;
    const auto &k = Consts<PREC>::get(s);
    const long long n = (long long)s.p.Nx * s.p.Ny;
    LBM_DISPATCH_Q(s.L.Q, (k_plane_from_f64<QQ, PREC><<<aux_blocks(n), kAuxThreads, 0, s.stream>>>(
                               (S *)s.f[s.cur], s.rho[s.cur], k, a, in)));
    return (int)cudaGetLastError();
}

template <int PREC>
int Launch<PREC>::macros(SolverImpl &s, double *rho, double *ux, double *uy, double *T,
                         int acc) {
    using S = typename Store<PREC>::S;
    const auto &k = Consts<PREC>::get(s);
    const long long n = (long long)s.p.Nx * s.p.Ny;
    LBM_DISPATCH_Q(s.L.Q, (k_macros<QQ, PREC><<<aux_blocks(n), kAuxThreads, 0, s.stream>>>(
                               (const S *)s.f[s.cur], s.rho[s.cur], k, rho, ux, uy, T, acc)));
    return (int)cudaGetLastError();
}

template <int PREC>
int Launch<PREC>::fluxes(SolverImpl &s, double *sxx, double *sxy, double *syy, double *qx,
                         double *qy) {
    using S = typename Store<PREC>::S;
    const auto &k = Consts<PREC>::get(s);
    dim3 grid((s.p.Nx + kFluxThreads - 1) / kFluxThreads, s.p.Ny);
    LatticeMoments lm = {};
    lm.h_tau = 0.5 / s.kd.tau_lat;
    lm.h_rho = 0.5 / s.kd.K;
    for (int a = 0; a < s.L.Q; ++a) {
        const double w = s.L.w[a], x2 = s.L.ex[a] * s.L.ex[a], y2 = s.L.ey[a] * s.L.ey[a];
        lm.m00 += w;
        lm.m20 += w * x2;
        lm.m40 += w * x2 * x2;
        lm.m22 += w * x2 * y2;
        lm.m60 += w * x2 * x2 * x2;
        lm.m42 += w * x2 * x2 * y2;
    }
    LBM_DISPATCH_Q(s.L.Q, (k_fluxes<QQ, PREC><<<grid, kFluxThreads, 0, s.stream>>>(
                               (const S *)s.f[s.cur], s.rho[s.cur], k, s.kw, s.kd, lm, sxx, sxy, syy, qx,
                               qy)));
    return (int)cudaGetLastError();
}

template <int PREC>
int Launch<PREC>::wall_mass(SolverImpl &s, double *m_in) {
    using S = typename Store<PREC>::S;
    const auto &k = Consts<PREC>::get(s);
    LBM_DISPATCH_Q(s.L.Q, (k_wall_mass<QQ, PREC><<<aux_blocks(2LL * s.p.Nx), kAuxThreads, 0,
                                                   s.stream>>>((const S *)s.f[s.cur],
                                                               s.rho[s.cur], k, m_in)));
    return (int)cudaGetLastError();
}

template <int PREC>
int Launch<PREC>::mass_partials(SolverImpl &s, double *partials, int nblocks) {
    using S = typename Store<PREC>::S;
    const auto &k = Consts<PREC>::get(s);
    LBM_DISPATCH_Q(s.L.Q, (k_mass_partials<QQ, PREC><<<nblocks, kAuxThreads, 0, s.stream>>>(
                               (const S *)s.f[s.cur], s.rho[s.cur], k, weight_sum(k), partials)));
    return (int)cudaGetLastError();
}

}  // namespace lbm
