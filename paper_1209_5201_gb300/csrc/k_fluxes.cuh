// Stress and heat flux of the distribution behind f~ (Sec. II).
//
// The stored state is post-collision f~*; the pre-collision f~ of the next
// step is what the pull of a step produces (Eq. (5) streaming with the Eq. (12)
// wall), so this kernel pulls exactly like k_step_direct and, instead of
// colliding, evaluates in FP64
//   f = (f~ + h f^eq) / (1 + h),  h = dt / (2 tau)      (definition of f~)
//   sigma_ij = sum (c_i - u_i)(c_j - u_j) f - rho T delta_ij
//   q_i      = 1/2 sum |c - u|^2 (c_i - u_i) f
// with T = 1 in an isothermal run.
//
// Bound by its FP64 instructions (64 cycles each per warp and SM sub-partition
// on GB300).  Forming f_a, its division and the central products velocity by
// velocity took about 1900 of them per cell; here 369 (counted, conversions too): the sums over the
// velocities are raw moments of f~ (sums and differences of opposite pairs,
// integer factors), f^eq enters through its moments alone - it is w_a times a
// polynomial in the integer velocity, so they are its 15 coefficients times
// the lattice's moments - and the shift by u is done once on the moments.
// D2Q37 FP32 1000 x 500: 355 us, 1281 before.
#pragma once

#include "k_aux.cuh"
#include "k_step_cellwarp64.cuh"             // rcp_cubic
#include "k_step_direct.cuh"

namespace lbm {

constexpr int kFluxThreads = 128;

// Lattice moments sum_a w_a e_ax^p e_ay^q in FP64 (symmetric in p and q), and
// h of a constant tau and h / rho of the mu = T law.
struct LatticeMoments { double m00, m20, m40, m22, m60, m42, h_tau, h_rho; };

// Raw moments up to third order, in units of the integer velocity: 1, x, y,
// xx, xy, yy, and x, y times |e|^2.
struct RawMoments {
    double n, x, y, xx, xy, yy, kx, ky;
};

// Moments of rho g^eq(u, T) / rho (Eq. (4), th = T - 1) on the lattice.
__device__ __forceinline__ RawMoments eq_moments(double ux, double uy, double th,
                                                 const KConsts<double> &k,
                                                 const LatticeMoments &m) {
    // g^eq = a00 + a01 c^2 + a02 c^4 + s (a10 + a11 c^2) + s^2 (a20 + a21 c^2) +
    // A3 s^3 + A4 s^4 (lbm_device.cuh) with s = e_x X + e_y Y and c^2 = r^2 |e|^2:
    // g_pq is the coefficient of e_x^p e_y^q; b_i = a_i1 r^2, b2 = a02 r^4
    const double X = k.r * ux, Y = k.r * uy, u2 = ux * ux + uy * uy;
    const double X2 = X * X, Y2 = Y * Y, XY = X * Y;
    double a00 = 1.0 - 0.5 * u2 - th, b0 = 0.5 * th, a10 = 1.0, a20 = 0.5;
    double g30 = 0.0, g12 = 0.0, g03 = 0.0, g21 = 0.0;
    double g40 = 0.0, g04 = 0.0, g22 = 0.0, g31 = 0.0, g13 = 0.0;
    if (k.eq_order >= 3) {
        const double b1 = 0.5 * k.r2 * th;
        a10 = 1.0 - 0.5 * u2 - 2.0 * th;
        g30 = X * (b1 + (1.0 / 6.0) * X2);
        g12 = X * (b1 + 0.5 * Y2);
        g03 = Y * (b1 + (1.0 / 6.0) * Y2);
        g21 = Y * (b1 + 0.5 * X2);
    }
    if (k.eq_order >= 4) {
        const double th2 = th * th, b21 = 0.25 * k.r2 * th, b2 = 0.125 * k.r2 * k.r2 * th2;
        a00 += 0.125 * u2 * u2 + th * u2 + th2;
        b0 -= 0.25 * th * u2 + th2;
        a20 -= 0.25 * u2 + 1.5 * th;
        g40 = b2 + X2 * (b21 + (1.0 / 24.0) * X2);
        g04 = b2 + Y2 * (b21 + (1.0 / 24.0) * Y2);
        g22 = 2.0 * b2 + b21 * (X2 + Y2) + 0.25 * X2 * Y2;
        g31 = XY * (2.0 * b21 + (1.0 / 6.0) * X2);
        g13 = XY * (2.0 * b21 + (1.0 / 6.0) * Y2);
    }
    b0 *= k.r2;
    const double g10 = a10 * X, g01 = a10 * Y, g11 = 2.0 * a20 * XY;
    const double g20 = b0 + a20 * X2, g02 = b0 + a20 * Y2;
    const double m4 = m.m40 + m.m22, m6 = m.m60 + m.m42, m42x2 = m.m42 + m.m42;
    RawMoments o;
    o.n = a00 * m.m00 + (g20 + g02) * m.m20 + (g40 + g04) * m.m40 + g22 * m.m22;
    o.x = g10 * m.m20 + g30 * m.m40 + g12 * m.m22;
    o.y = g01 * m.m20 + g03 * m.m40 + g21 * m.m22;
    o.xx = a00 * m.m20 + g20 * m.m40 + g02 * m.m22 + g40 * m.m60 + (g04 + g22) * m.m42;
    o.yy = a00 * m.m20 + g02 * m.m40 + g20 * m.m22 + g04 * m.m60 + (g40 + g22) * m.m42;
    o.xy = g11 * m.m22 + (g31 + g13) * m.m42;
    o.kx = g10 * m4 + g30 * m6 + g12 * m42x2;
    o.ky = g01 * m4 + g03 * m6 + g21 * m42x2;
    return o;
}

template <int Q, int PREC>
__global__ void __launch_bounds__(kFluxThreads)
k_fluxes(const typename Store<PREC>::S *__restrict__ fin, const float *__restrict__ rin,
         const __grid_constant__ KConsts<typename Store<PREC>::C> k,
         const __grid_constant__ KWall kw, const __grid_constant__ KConsts<double> kd,
         const __grid_constant__ LatticeMoments lm, double *sxx, double *sxy, double *syy,
         double *qx, double *qy) {
    using L = Lat<Q>;
    using C = typename Store<PREC>::C;
    __shared__ WallFills<PREC, kFluxThreads> s_fill;
    const int j = blockIdx.y;
    const int x0 = blockIdx.x * kFluxThreads;
    const int x = x0 + threadIdx.x;
    const bool bot = j < L::N, top = j >= k.Ny - L::N;
    if (bot || top) {
        wall_prologue<Q, PREC, kFluxThreads>(fin, rin, k, kw, bot ? 0 : 1, x0,
                                             min(kFluxThreads, k.Nx - x0) + 6, s_fill);
        __syncthreads();
    }
    if (x >= k.Nx) return;

    C fc[Q];
    const typename Store<PREC>::S *src = fin + col_index(k, j, x);
    const float *rsrc = Store<PREC>::dev ? rin + rho_index(k, j, x) : nullptr;
    if (bot || top) pull<Q, PREC, kFluxThreads, true, 0>(fin, rin, src, rsrc, k, kw, x, j, s_fill, fc);
    else pull<Q, PREC, kFluxThreads, false, 0>(fin, rin, src, rsrc, k, kw, x, j, s_fill, fc);

    // raw moments of f~ (shifted storage: of the deviations, then the weights')
    RawMoments m{(double)fc[0], 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    PairLoop<1, Q>::run([&](auto ic) {
        constexpr int A = decltype(ic)::value;
        constexpr double ex = L::ex(A), ey = L::ey(A), e2 = L::e2(A);
        const double fa = (double)fc[A], fb = (double)fc[A + 1], s = fa + fb, d = fa - fb;
        m.n += s;
        if constexpr (ex != 0) {
            m.x += ex * d;
            m.xx += (ex * ex) * s;
            m.kx += (e2 * ex) * d;
        }
        if constexpr (ey != 0) {
            m.y += ey * d;
            m.yy += (ey * ey) * s;
            m.ky += (e2 * ey) * d;
        }
        if constexpr (ex != 0 && ey != 0) m.xy += (ex * ey) * s;
    });
    if constexpr (Store<PREC>::shifted) {
        m.n += lm.m00;
        m.xx += lm.m20;
        m.yy += lm.m20;
    }
    const double r = kd.r, r2 = kd.r2, rho = m.n, inv = rcp_cubic(rho);
    const double ux = r * m.x * inv, uy = r * m.y * inv;
    const double u2 = ux * ux + uy * uy;
    const double T = kd.thermal ? 0.5 * (r2 * (m.xx + m.yy) * inv - u2) : 1.0;
    // tau / dt as the collision forms it; h = dt / (2 tau)
    double h;
    if (kd.const_tau) h = lm.h_tau;
    else if (kd.mu_is_one || !kd.thermal) h = lm.h_rho * rho;
    else h = 0.5 / (kd.K * inv * pow(T, kd.mu_m1));
    // moments of f = (f~ + h rho g^eq) / (1 + h), in units of c
    const RawMoments g = eq_moments(ux, uy, T - 1.0, kd, lm);
    const double i1 = rcp_cubic(1.0 + h), hr = h * rho, r3 = r2 * r;
    const double n = i1 * (m.n + hr * g.n);
    const double jx = i1 * r * (m.x + hr * g.x), jy = i1 * r * (m.y + hr * g.y);
    const double pxx = i1 * r2 * (m.xx + hr * g.xx), pyy = i1 * r2 * (m.yy + hr * g.yy);
    const double pxy = i1 * r2 * (m.xy + hr * g.xy);
    const double kx = i1 * r3 * (m.kx + hr * g.kx), ky = i1 * r3 * (m.ky + hr * g.ky);
    // ... shifted to the velocity u: sum (c - u)(c - u) f and sum |c - u|^2 (c - u) f
    const long long c = (long long)j * k.Nx + x;
    const double rt = rho * T, uj = ux * jx + uy * jy, tr = pxx + pyy;
    if (sxx) sxx[c] = pxx - ux * (2.0 * jx - n * ux) - rt;
    if (sxy) sxy[c] = pxy - ux * jy - uy * (jx - n * ux);
    if (syy) syy[c] = pyy - uy * (2.0 * jy - n * uy) - rt;
    const double w = 2.0 * uj - tr - u2 * n;
    if (qx) qx[c] = 0.5 * (kx + ux * w + u2 * jx) - (ux * pxx + uy * pxy);
    if (qy) qy[c] = 0.5 * (ky + uy * w + u2 * jy) - (ux * pxy + uy * pyy);
}

}  // namespace lbm
