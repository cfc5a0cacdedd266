// Auxiliary kernels of a solver: initial state, conversions between the
// storage format and FP64 host planes, Eq. (3) macroscopic fields, the wall
// incoming mass of Eq. (12), and FP64 reductions.
#pragma once

#include "lbm_device.cuh"

namespace lbm {

constexpr int kAuxThreads = 256;

// SplitMix64 (Steele, Lea & Flood, OOPSLA 2014): first output of the stream
// seeded with seed XOR counter; top 53 bits as a double in [0, 1).
__device__ __forceinline__ double splitmix_u01(uint64_t seed, uint64_t k) {
    uint64_t z = (seed ^ k) + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z = z ^ (z >> 31);
    return (double)(z >> 11) * 0x1.0p-53;
}

// Equilibrium f~* = rho g^eq(u, T) (Eq. (4)) of every velocity, or its
// deviation w (rho g - 1) when SHIFT (drho = rho - 1 given separately so that
// it carries no cancellation error).
template <int Q, class C, bool SHIFT>
__device__ __forceinline__ void equilibrium_all(C rho, C drho, C ux, C uy, C T,
                                                const KConsts<C> &k, C (&o)[Q]) {
    // the equilibrium terms of a collision with omega = 1
    Collision<Q, C, SHIFT> col;
    const C u2 = ux * ux + uy * uy;
    col.set_omega(C(1));
    col.sx = k.r * ux;
    col.sy = k.r * uy;
    col.rho = rho;
    col.set_coefficients(u2, T - C(1), rho, drho / rho, k);
    o[0] = col.cw[0] * col.A0[0];
    PairLoop<1, Q>::run([&](auto ic) {
        constexpr int A = decltype(ic)::value;
        C P, R;
        col.template eq_pair<A>(P, R);
        o[A] = P + R;
        o[A + 1] = P - R;
    });
}

// Eq. (3) fields of a cell from its stored values v (deviations where the
// format stores them; BF16DEV: its density rc): rho, u_x, u_y and the kinetic
// temperature sum f |c - u|^2 / (2 rho), in the storage's compute type.
template <int Q, int PREC, class C>
__device__ __forceinline__ void cell_fields(const C (&sv)[Q], C rc, const KConsts<C> &k,
                                            double (&o)[4]) {
    using L = Lat<Q>;
    C s0 = 0, sx = 0, sy = 0, se = 0;
    if constexpr (PREC == LBM_FP64) {
        // FP64 instructions are the cost: sums and differences of opposite
        // pairs, and one reciprocal: about 115 of them instead of 175
        s0 = sv[0];
        PairLoop<1, Q>::run([&](auto ic) {
            constexpr int A = decltype(ic)::value;
            const C s = sv[A] + sv[A + 1], d = sv[A] - sv[A + 1];
            s0 += s;
            if constexpr (L::ex(A) != 0) sx += C(L::ex(A)) * d;
            if constexpr (L::ey(A) != 0) sy += C(L::ey(A)) * d;
            se += C(L::e2(A)) * s;
        });
    } else {
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            C v = sv[a];
            if constexpr (Store<PREC>::dev) v += k.w[a] * rc;
            s0 += v;
            sx += C(L::ex(a)) * v;
            sy += C(L::ey(a)) * v;
            se += C(L::e2(a)) * v;
        }
    }
    // shifted storage: the sums are of deviations; sum w = 1, sum e w = 0
    const C rh = Store<PREC>::shifted ? C(1) + s0 : s0;
    // rho D T = sum f |c - u|^2 = r^2 sum e^2 f - rho u^2
    if constexpr (PREC == LBM_FP64) {
        const C inv = __drcp_rn(rh), u = k.r * sx * inv, v = k.r * sy * inv;
        o[0] = rh;
        o[1] = u;
        o[2] = v;
        o[3] = 0.5 * (k.r2 * se * inv - (u * u + v * v));
    } else {
        const C u = k.r * sx / rh, v = k.r * sy / rh;
        if constexpr (Store<PREC>::shifted) se += k.e2w;
        const C e = k.r2 * se - rh * (u * u + v * v);
        o[0] = (double)rh;
        o[1] = (double)u;
        o[2] = (double)v;
        o[3] = (double)(e / (C(2) * rh));
    }
}

// sum of rho over a cell's stored values.  FP32 / BF16: the stored deviations
// are summed in FP32 (they are small, so its rounding is far below FP32
// resolution of the cell's mass) and the rest is added in FP64; FP64 storage
// sums in FP64.  wsum: FP64 sum of the weights (BF16DEV).
template <int Q, int PREC, class C>
__device__ __forceinline__ double cell_mass(const C (&sv)[Q], double wsum, float rc) {
    C sd = 0;
#pragma unroll
    for (int a = 0; a < Q; ++a) sd += sv[a];
    double s = (double)sd;
    if constexpr (Store<PREC>::shifted) s += 1.0;            // sum of the weights
    if constexpr (Store<PREC>::dev) s += wsum * (double)rc;
    return s;
}

// Block-level FP64 sum of NV values per thread (warp shuffle, then shared).
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double *out) {
    __shared__ double sh[32][NV];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < NV; ++i)
        for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_down_sync(0xffffffffu, v[i], o);
    if (lane == 0)
        for (int i = 0; i < NV; ++i) sh[wid][i] = v[i];
    __syncthreads();
    if (wid == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        for (int i = 0; i < NV; ++i) {
            double s = lane < nw ? sh[lane][i] : 0.0;
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            if (lane == 0) out[i] = s;
        }
    }
}

// Block sum of one FP32 value per thread to FP64 precision by error-free
// additions of float pairs (an FP64 add, or a conversion, takes a warp 64
// cycles); the result in thread 0.
__device__ __forceinline__ double block_sum_f32(float v) {
    __shared__ float sh[32][2];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float h = v, l = 0.0f;
    auto merge = [&](float h2, float l2) {
        float e;
        two_sum(h, h2, h, e);
        l = __fadd_rn(__fadd_rn(l, l2), e);
    };
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float h2 = __shfl_down_sync(0xffffffffu, h, o), l2 = __shfl_down_sync(0xffffffffu, l, o);
        merge(h2, l2);
    }
    __syncthreads();                         // sh may still be read by a call before
    if (lane == 0) sh[wid][0] = h, sh[wid][1] = l;
    __syncthreads();
    if (threadIdx.x != 0) return 0.0;
    for (int i = 1; i < (int)(blockDim.x + 31) / 32; ++i) merge(sh[i][0], sh[i][1]);
    return (double)h + (double)l;
}

// Velocity plane a of the stored state -> FP64 logical plane [Ny][Nx].
template <int Q, int PREC>
__global__ void k_plane_to_f64(const typename Store<PREC>::S *f, const float *rplane,
                               const __grid_constant__ KConsts<typename Store<PREC>::C> k,
                               int a, double *out) {
    const long long n = (long long)k.Nx * k.Ny;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
         c += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(c / k.Nx), x = (int)(c % k.Nx);
        const long long r = col_index(k, j, x) + (long long)a * k.pitch;
        double v = (double)to_c(f[r]);
        if constexpr (Store<PREC>::dev) v = (double)(to_c(f[r]) + k.w[a] * rplane[rho_index(k, j, x)]);
        if constexpr (Store<PREC>::shifted) v += (double)k.w[a];
        out[c] = v;
    }
}

// FP64 logical plane -> velocity plane a of the stored state (with images).
// BF16DEV needs the density plane written first (launch_rho_plane).
template <int Q, int PREC>
__global__ void k_plane_from_f64(typename Store<PREC>::S *f, const float *rplane,
                                 const __grid_constant__ KConsts<typename Store<PREC>::C> k,
                                 int a, const double *in) {
    using S = typename Store<PREC>::S;
    using C = typename Store<PREC>::C;
    const long long n = (long long)k.Nx * k.Ny;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
         c += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(c / k.Nx), x = (int)(c % k.Nx);
        C v = (C)in[c];
        if constexpr (Store<PREC>::dev) v -= k.w[a] * rplane[rho_index(k, j, x)];
        if constexpr (Store<PREC>::shifted) v = (C)(in[c] - (double)k.w[a]);
        store_pop<S>(f, k, a, j, x, from_c<S>(v));
    }
}

// Eq. (3) fields of every cell of the stored state; T is the kinetic
// temperature sum f |c - u|^2 / (2 rho).  Per-cell arithmetic in the storage's
// compute type (FP32 or FP64), outputs FP64.  Any output may be NULL.
// acc: add the fields to the outputs instead of writing them (acc == 1), or
// write them (acc == 0).
template <int Q, int PREC>
__global__ void k_macros(const typename Store<PREC>::S *f, const float *rplane,
                         const __grid_constant__ KConsts<typename Store<PREC>::C> k,
                         double *rho, double *ux, double *uy, double *T, int acc) {
    using C = typename Store<PREC>::C;
    const long long n = (long long)k.Nx * k.Ny;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
         c += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(c / k.Nx), x = (int)(c % k.Nx);
        const long long ro = col_index(k, j, x);
        C v[Q], rc = 0;
#pragma unroll
        for (int a = 0; a < Q; ++a) v[a] = to_c(f[ro + (long long)a * k.pitch]);
        if constexpr (Store<PREC>::dev) rc = rplane[rho_index(k, j, x)];
        double o[4];
        cell_fields<Q, PREC, C>(v, rc, k, o);
        double *out[4] = {rho, ux, uy, T};
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (out[i]) out[i][c] = acc ? out[i][c] + o[i] : o[i];
    }
}

// Numerator of Eq. (12) for every ghost column of both walls: m_in[w*Nx + x].
template <int Q, int PREC>
__global__ void k_wall_mass(const typename Store<PREC>::S *f, const float *rplane,
                            const __grid_constant__ KConsts<typename Store<PREC>::C> k,
                            double *m_in) {
    using L = Lat<Q>;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < 2 * k.Nx;
         t += gridDim.x * blockDim.x) {
        const int wall = t / k.Nx, xw = t % k.Nx;
        double m = 0.0;
#pragma unroll
        for (int b = 0; b < Q; ++b) {
            const int eyb = L::ey(b);
            if (wall == 0 ? !(eyb < 0) : !(eyb > 0)) continue;
            const int xs = wrap(xw - L::ex(b), k.Nx);
            const int depth = eyb < 0 ? -eyb : eyb;
            for (int kk = 0; kk < depth; ++kk) {
                const int row = wall == 0 ? kk : k.Ny - 1 - kk;
                double v = (double)to_c(f[col_index(k, row, xs) + (long long)b * k.pitch]);
                if constexpr (Store<PREC>::dev)
                    v += (double)k.w[b] * (double)rplane[rho_index(k, row, xs)];
                if constexpr (Store<PREC>::shifted) v += (double)k.w[b];
                m += v;
            }
        }
        m_in[t] = m;
    }
}

// Sum of rho over all cells: per-block partials (fixed grid, fixed order).  A
// block takes whole rows, several at a time where they are narrower than the
// block (one division per thread, none per cell).
template <int Q, int PREC>
__global__ void k_mass_partials(const typename Store<PREC>::S *f, const float *rplane,
                                const __grid_constant__ KConsts<typename Store<PREC>::C> k,
                                double wsum, double *partials) {
    using C = typename Store<PREC>::C;
    double acc[1] = {0.0};
    const int rows = k.Nx < (int)blockDim.x ? blockDim.x / k.Nx : 1;
    const int tr = rows > 1 ? threadIdx.x / k.Nx : 0, tx = threadIdx.x - tr * k.Nx;
    const int x0 = rows > 1 ? (tr < rows ? tx : k.Nx) : threadIdx.x;
    for (int j = blockIdx.x * rows + tr; j < k.Ny; j += gridDim.x * rows) {
        for (int x = x0; x < k.Nx; x += blockDim.x) {
            const typename Store<PREC>::S *cell = f + col_index(k, j, x);
            C v[Q];
#pragma unroll
            for (int a = 0; a < Q; ++a) v[a] = to_c(cell[(long long)a * k.pitch]);
            float rc = 0.0f;
            if constexpr (Store<PREC>::dev) rc = rplane[rho_index(k, j, x)];
            acc[0] += cell_mass<Q, PREC, C>(v, wsum, rc);
        }
    }
    block_sum<1>(acc, partials + blockIdx.x);
}

}  // namespace lbm
