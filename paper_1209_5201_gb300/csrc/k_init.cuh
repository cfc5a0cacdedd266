// Initial state of the single-domain solver.
#pragma once

#include "k_aux.cuh"
#include "k_step_direct.cuh"

namespace lbm {

// Initial state f~* = rho g^eq(u, T) of every cell, the fields of the first
// residual check (u_x and T of the stored state, prev_u / prev_T) and the mass
// (block partials, fixed grid and order), in one pass, bound by the one write
// of the state: D2Q37 4096 x 2048 FP32 290 us (212 at the copy rate), 918 us as
// initialisation, mass sum and read-out of the stored state one after another;
// BF16SHIFT 382 us after 639; a 1 x 500 FP64 column 22 us after 680.
// rho, ux, uy, T: FP64 device planes [Ny][Nx] (ux, uy, T may be NULL: u = 0, T = 1);
// rho NULL: rho0 (1 + amp (2U - 1)) at rest; wsum: FP64 sum of the weights.  One
// block per 128 columns of one row of a tile: no division per cell, stores as
// the step's (blocks that walk several rows wait for each row's density in
// turn: 440 - 550 us).
constexpr int kInitThreads = 128;

// blocks of k_init, one mass partial each: at most one per cell
template <class K>
__host__ __device__ __forceinline__ long long init_blocks(const K &k) {
    return (long long)k.nt * ((k.tw + kInitThreads - 1) / kInitThreads) * k.Ny;
}

template <int Q, int PREC>
__global__ void __launch_bounds__(kInitThreads)
k_init(typename Store<PREC>::S *f, float *rplane,
       const __grid_constant__ KConsts<typename Store<PREC>::C> k, const double *rho,
       const double *ux, const double *uy, const double *T, double rho0, double amp, uint64_t seed,
       double *prev_u, double *prev_T, double wsum, double *partials) {
    using S = typename Store<PREC>::S;
    using C = typename Store<PREC>::C;
    const int bpt = (k.tw + kInitThreads - 1) / kInitThreads, gx = k.nt * bpt;
    const int j = blockIdx.x / gx, bx = blockIdx.x - j * gx;
    const int t = bx / bpt, xl = (bx - t * bpt) * kInitThreads + threadIdx.x;
    const int w = tile_width(k, t);
    double mass[1] = {0.0};
    float sd = 0.0f, rd = 0.0f;              // FP32 / BF16: the cell's stored sum, its density
    if (xl < w) {
        const long long c = (long long)j * k.Nx + t * k.tw + xl;
        double r = rho0;
        if (rho) r = rho[c];
        else if (amp != 0.0) r = rho0 * (1.0 + amp * (2.0 * splitmix_u01(seed, (uint64_t)c) - 1.0));
        C o[Q];
        equilibrium_all<Q, C, Store<PREC>::shifted>((C)r, (C)(r - 1.0), ux ? (C)ux[c] : C(0),
                                                    uy ? (C)uy[c] : C(0), T ? (C)T[c] : C(1), k, o);
        S sv[Q];
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            C v = o[a];
            if constexpr (Store<PREC>::dev) v -= k.w[a] * (C)r;
            sv[a] = from_c<S>(v);
            o[a] = to_c(sv[a]);
        }
        float *rdst = Store<PREC>::dev ? rplane + rho_index(k, j, t * k.tw + xl) : nullptr;
        store_cell<Q, PREC, false, 0>(sv, (float)r, f, rplane, f + col_index(k, j, t * k.tw + xl),
                                      rdst, k, t, xl, w, j);
        double fl[4];
        cell_fields<Q, PREC, C>(o, (C)r, k, fl);
        prev_u[c] = fl[1];
        prev_T[c] = fl[3];
        if constexpr (PREC == LBM_FP64) {
            mass[0] = fl[0];
        } else {
#pragma unroll
            for (int a = 0; a < Q; ++a) sd += o[a];
            rd = (float)r;
        }
    }
    if constexpr (PREC == LBM_FP64) {
        block_sum<1>(mass, partials + blockIdx.x);
    } else {
        // as cell_mass, summed over the block: sum d, and sum w per cell
        // (BF16DEV: times the cell's density)
        double m = block_sum_f32(sd);
        if constexpr (Store<PREC>::dev) m += wsum * block_sum_f32(rd);
        else m += (double)max(0, min(kInitThreads, w - (bx - t * bpt) * kInitThreads));
        if (threadIdx.x == 0) partials[blockIdx.x] = m;
    }
}

}  // namespace lbm
