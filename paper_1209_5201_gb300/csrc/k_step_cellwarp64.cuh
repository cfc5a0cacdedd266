// One-warp-per-cell time steps in FP64 (Eq. (5) with the Eq. (12) wall), for
// grids of a few thousand cells.
//
// What bounds them: GB300 has half an FP64 lane per cycle and SM sub-partition,
// so every FP64 warp instruction holds the sub-partition's FP64 unit for 64
// cycles (measured: dependent and independent DFMA chains alike, 1 to 32 lanes
// active).  A step of a small grid is the chain of one warp's FP64
// instructions times 64 cycles, whatever their lanes do, so a cell's update is
// written for the fewest FP64 instructions per warp:
//  * lane p carries the opposite pair (2p - 1, 2p), lane 0 the rest velocity:
//    one pass over at most 19 lanes, not two over 37 velocities;
//  * the moments are four dot products over Q, eight lanes each (the values
//    passed through shared memory): ceil(Q / 8) FMAs and three butterfly adds
//    for all four, not five adds for each;
//  * 1 / rho and 1 / (tau / dt + 1/2) (the latter as rho / (K + rho / 2)) are one
//    reciprocal in two lanes; u_x and u_y share instructions the same way;
//  * each lane forms the Eq. (4) coefficients of its own shell directly.
// D2Q37 thermal, order 4: 42 FP64 instructions per interior cell (about 110
// with one velocity per lane, two passes and whole-warp butterflies).
// Consecutive steps run in one launch: a launch per step reloads constants and
// addresses and cost 3.7 (64 cells, D2Q25) and 7.0 us (500 cells, D2Q37) per
// step with this update, 6.4 and 12.4 with the velocity-per-lane one; the
// many-step launches take 2.3 (one cluster) and 3.6 us (whole chip).
#pragma once

#include <type_traits>

#include "lbm_device.cuh"

namespace lbm {

constexpr int kCellWarps = 4;               // one warp on each SM sub-partition
constexpr int kCellMaxWarps = 28;           // warps (cells) per block: 72 registers a thread
constexpr int kCellClusterCells = 16 * kCellWarps;   // cells one 16-CTA cluster takes
constexpr int kCellErrTimeout = 2;

// 1 / x to within an ulp: the hardware's 20-bit estimate and one step of
// Chebyshev's third-order iteration r (1 + e + e^2), e = 1 - x r (its relative
// error is e^3 ~ 2^-60): three FP64 instructions, __drcp_rn about six.  Measured
// over [1e-30, 1e30]: error at most 0.508 ulp, another value than __drcp_rn's in
// 0.03 % of cases (0.19 % next to 1).
__device__ __forceinline__ double rcp_cubic(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = __fma_rn(-x, r, 1.0);
    return __fma_rn(__fma_rn(e, e, e), r, r);
}

// One lane's share of cell (x, j): its pair (a, b = a + 1), the addresses of
// its sources and its constants, all formed once.  Addr: how a population of
// the state is named; addr(a, row, column) gives it, ld(Addr) reads it.
template <int Q, class Addr>
struct CellLane {
    using L = Lat<Q>;
    static constexpr int NP = (Q - 1) / 2, KM = (Q + 7) / 8;
    static constexpr unsigned kAll = 0xffffffffu;
    int lane, a, b;
    bool mine, edge, fill_a, fill_b, one_col, term;
    int wall, from;                          // from: lane holding M_in of this lane's ghost column
    double cx, cy, x0, x1, x2, t1, t2, we, wo, cf;
    double mom[KM];
    Addr oa, ob, osp, ot[7];

    template <class AddrFn>
    __device__ __forceinline__ void init(const KConsts<double> &k, const CellLanes &c, int lane_,
                                         int cell, AddrFn &&addr) {
        lane = lane_;
        mine = lane <= NP;
        const int p = mine ? lane : 0;
        a = p ? 2 * p - 1 : 0;
        b = 2 * p;
        const int j = cell / k.Nx, x = cell - j * k.Nx;
        const int ex = c.ex[p], ey = c.ey[p];
        const bool bot = j < L::N, top = j >= k.Ny - L::N;       // warp-uniform
        edge = bot || top;
        wall = top ? 1 : 0;
        // sources beyond the wall (Ny >= 6: a row is near one wall at most)
        fill_a = j - ey < 0 || j - ey >= k.Ny;
        fill_b = j + ey < 0 || j + ey >= k.Ny;
        oa = addr(a, fill_a ? j : j - ey, wrap(x - ex, k.Nx));
        ob = addr(b, fill_b ? j : j + ey, wrap(x + ex, k.Nx));
        cx = c.cx[p], cy = c.cy[p], x0 = c.x0[p], x1 = c.x1[p], x2 = c.x2[p];
        t1 = c.t1[p], t2 = c.t2[p], we = c.we[p], wo = c.wo[p];
#pragma unroll
        for (int i = 0; i < KM; ++i) mom[i] = c.mom[lane >> 3][(lane & 7) + 8 * i];
        // wall rows: lane l < nterm carries the wall's l-th incoming term, at
        // the ghost columns x - 3 .. x + 3 (one column when Nx = 1); the fill
        // of velocity q comes from ghost column x - e_qx, the specular partner
        // from the same row, 2 e_qx columns back
        one_col = k.Nx == 1;
        term = edge && lane < c.nterm;
        cf = 0.0;
        from = 0;
        osp = oa;
        if (edge) {
            const int q = fill_b ? b : a, exq = fill_b ? -ex : ex;
            cf = fill_a || fill_b ? k.wcoef[wall][q] : 0.0;
            if (fill_a || fill_b) osp = addr(k.mirror[q], j, wrap(x - 2 * exq, k.Nx));
            if (!one_col) from = 4 * (3 - exq);
            const int tb = term ? c.tb[wall][lane] : 0, tk = term ? c.tk[wall][lane] : 0;
            const int tx = term ? c.tx[wall][lane] : 0;
            const int row = wall == 0 ? tk : k.Ny - 1 - tk;
#pragma unroll
            for (int t = 0; t < 7; ++t)
                if (t == 0 || !one_col) ot[t] = addr(tb, row, wrap(x - 3 + t - tx, k.Nx));
        }
    }

    // One step (explicit FMAs: every kernel below rounds alike): pull, collide; the pair's post-collision values in va, vb.
    // sf: the warp's 8 KM doubles of shared memory, zero past Q.
    template <class LoadFn>
    __device__ __forceinline__ void step(const KConsts<double> &k, const CellLanes &c, double *sf,
                                         double &va, double &vb, LoadFn &&ld) const {
        double fa = ld(oa), fb = ld(ob);
        if (edge) {
            // Eq. (12): M_in of the ghost columns, a fixed order of FP64 adds
            double m;
            if (one_col) {
                m = ld(ot[0]);
                if (!term) m = 0.0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(kAll, m, o);
            } else {
                // eight columns (the eighth zero) over 32 lanes: lanes exchange
                // half of their columns at each of three stages, 9 adds, not 35
                double v[8];
#pragma unroll
                for (int t = 0; t < 7; ++t) {
                    v[t] = ld(ot[t]);
                    if (!term) v[t] = 0.0;
                }
                v[7] = 0.0;
#pragma unroll
                for (int h = 4; h > 0; h >>= 1) {
                    const bool up = (lane & (4 * h)) != 0;
#pragma unroll
                    for (int i = 0; i < h; ++i) {
                        const double keep = up ? v[i + h] : v[i], send = up ? v[i] : v[i + h];
                        v[i] = keep + __shfl_xor_sync(kAll, send, 4 * h);
                    }
                }
                m = v[0];
                m += __shfl_xor_sync(kAll, m, 2);
                m += __shfl_xor_sync(kAll, m, 1);
            }
            m = __shfl_sync(kAll, m, from);
            double v = m * cf;
            if (!c.diffuse[wall])            // Eq. (9) with R = accom R_D + (1 - accom) R_S
                v = __fma_rn(k.accom[wall], v, (1.0 - k.accom[wall]) * ld(osp));
            if (fill_a) fa = v;
            if (fill_b) fb = v;
        }
        if (mine) {
            sf[b] = fb;
            sf[a] = fa;                      // lane 0: the same slot, the same value
        }
        __syncwarp();

        // Eq. (3): sum f, sum c_x f, sum c_y f, sum |c|^2 / 2 f in lanes 0, 8, 16, 24
        double acc = mom[0] * sf[lane & 7];
#pragma unroll
        for (int i = 1; i < KM; ++i) acc = __fma_rn(mom[i], sf[(lane & 7) + 8 * i], acc);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(kAll, acc, o);
        const double rho = __shfl_sync(kAll, acc, 0);
        const double jxy = __shfl_sync(kAll, acc, lane & 1 ? 16 : 8);
        const double e = __shfl_sync(kAll, acc, 24);

        // reciprocals, velocity, temperature, relaxation factor
        const bool joint = k.const_tau || k.mu_is_one || !k.thermal;
        double den = rho;
        if (joint && (lane & 1)) den = k.const_tau ? c.tau_half : __fma_rn(0.5, rho, k.K);
        const double r = rcp_cubic(den);
        const double inv = __shfl_sync(kAll, r, 0);
        const double u = jxy * inv;          // even lanes u_x, odd lanes u_y
        const double ux = __shfl_sync(kAll, u, 0), uy = __shfl_sync(kAll, u, 1);
        double u2 = u * u;
        u2 += __shfl_xor_sync(kAll, u2, 1);
        double th = 0.0;
        if (k.thermal) th = __fma_rn(-0.5, u2, __fma_rn(e, inv, -1.0));
        double om = __shfl_sync(kAll, r, 1);
        if (!joint) om = rcp_cubic(__fma_rn(k.K * inv, pow(1.0 + th, k.mu_m1), 0.5));
        else if (!k.const_tau) om = rho * om;

        // Eq. (4), even and odd part of the pair: 2E = 2 A0 + s^2 (2 A2 + 2 A4
        // s^2), O = s (A1 + A3 s^2); with Y = 1 - u^2 / 2 the theta-free parts
        // are 2 A0 = 1 + Y^2 (order 4) or 2 Y, A1 = Y (order >= 3) or 1,
        // 2 A2 = Y (order 4) or 1
        const double s = __fma_rn(cx, ux, cy * uy), s2 = s * s;
        const double Y = __fma_rn(-0.5, u2, 1.0);
        double E, O = s;
        if (k.eq_order >= 4) {
            double A0 = __fma_rn(Y, Y, 1.0), A2 = Y, A1 = Y;
            if (k.thermal) {
                A0 = __fma_rn(th, __fma_rn(x2, th, __fma_rn(x1, u2, x0)), A0);
                A1 = __fma_rn(t1, th, Y);
                A2 = __fma_rn(t2, th, Y);
            }
            E = __fma_rn(s2, __fma_rn(1.0 / 12.0, s2, A2), A0);
            O = s * __fma_rn(1.0 / 6.0, s2, A1);
        } else {
            double A0 = Y + Y, A1 = Y;
            if (k.thermal) {
                A0 = __fma_rn(th, x0, A0);
                if (k.eq_order == 3) A1 = __fma_rn(t1, th, Y);
            }
            E = __fma_rn(s, s, A0);
            if (k.eq_order == 3) O = s * __fma_rn(1.0 / 6.0, s2, A1);
        }
        const double orho = om * rho, omc = 1.0 - om;
        // (the pulled value, the largest term, is added last: one rounding at its size)
        const double P = (orho * we) * E, ow = orho * wo;
        va = __fma_rn(omc, fa, __fma_rn(ow, O, P));
        vb = __fma_rn(omc, fb, __fma_rn(-ow, O, P));
        __syncwarp();                        // every lane has read sf
    }
    // the pair into a state buffer, with the halo copies other kernels read
    __device__ __forceinline__ void store_images(double *f, const KConsts<double> &k, int cell,
                                                 double va, double vb) const {
        const int j = cell / k.Nx, x = cell - j * k.Nx;
        if (mine) store_pop<double>(f, k, a, j, x, va);
        if (mine && b) store_pop<double>(f, k, b, j, x, vb);
    }
};

// One step per launch (programmatic dependent launch; everything that does not
// depend on the state is formed before the wait on the previous step).
template <int Q>
__global__ void __launch_bounds__(32 * kCellWarps)
k_step_cellwarp64(const double *fin, double *fout, const __grid_constant__ KConsts<double> k,
                  const __grid_constant__ CellLanes c) {
    using Lane = CellLane<Q, long long>;
    __shared__ double s_f[kCellWarps][8 * Lane::KM];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cell = blockIdx.x * kCellWarps + warp;
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    if (cell >= k.Nx * k.Ny) return;         // no block barrier below
    double *sf = s_f[warp];
    if (lane < 8 * Lane::KM - Q) sf[Q + lane] = 0.0;
    Lane cl;
    cl.init(k, c, lane, cell, [&](int a, int row, int xc) {
        return col_index(k, row, xc) + (long long)a * k.pitch;
    });
    // the previous step's stores are visible from here on
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    double va, vb;
    cl.step(k, c, sf, va, vb, [&](long long o) { return __ldcg(fin + o); });
    cl.store_images(fout, k, cell, va, vb);
}

// Many steps per launch, the grid's cells on one cluster: the state stays in
// the CTAs' shared memory (cell c on CTA c / kCellWarps, two buffers), sources
// are read through distributed shared memory, one cluster barrier per step.
template <int Q>
__global__ void __launch_bounds__(32 * kCellWarps)
k_steps_cellwarp64_cluster(const double *fin, double *fout,
                           const __grid_constant__ KConsts<double> k,
                           const __grid_constant__ CellLanes c, int nsteps) {
    using Lane = CellLane<Q, uint32_t>;
    constexpr int QP = 8 * Lane::KM;
    __shared__ double s_f[kCellWarps][QP];
    __shared__ double s_st[2][kCellWarps][QP];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cell = blockIdx.x * kCellWarps + warp;         // one cluster: block = CTA rank
    const bool live = cell < k.Nx * k.Ny;
    double *sf = s_f[warp];
    if (lane < QP - Q) sf[Q + lane] = 0.0;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(&s_st[0][0][0]);
    constexpr uint32_t kBuf = kCellWarps * QP * 8u;
    Lane cl;
    double va = 0.0, vb = 0.0;
    if (live) {
        cl.init(k, c, lane, cell, [&](int a, int row, int xc) {
            const int src = row * k.Nx + xc;
            uint32_t out;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(out)
                         : "r"(base + (uint32_t)((src % kCellWarps) * QP + a) * 8u),
                           "r"((uint32_t)(src / kCellWarps)));
            return out;
        });
        const int j = cell / k.Nx, x = cell - j * k.Nx;
        const long long own = col_index(k, j, x);
        if (cl.mine) {
            s_st[0][warp][cl.b] = __ldcg(fin + own + (long long)cl.b * k.pitch);
            s_st[0][warp][cl.a] = __ldcg(fin + own + (long long)cl.a * k.pitch);
        }
    }
    for (int n = 0; n < nsteps; ++n) {
        // the sources of this step are in place, and every reader of the
        // buffer it writes is done
        asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;\n" ::: "memory");
        if (!live) continue;
        const uint32_t off = (n & 1) ? kBuf : 0u;
        cl.step(k, c, sf, va, vb, [&](uint32_t o) {
            double v;
            asm volatile("ld.shared::cluster.f64 %0, [%1];\n" : "=d"(v) : "r"(o + off));
            return v;
        });
        double *st = s_st[(n & 1) ^ 1][warp];
        if (cl.mine) {
            if (cl.b) st[cl.b] = vb;
            st[cl.a] = va;
        }
    }
    // no CTA leaves while another still reads its shared memory
    asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;\n" ::: "memory");
    if (live) cl.store_images(fout, k, cell, va, vb);
}

// Many steps per launch over the whole chip (a cooperative launch: every block
// is resident): the state alternates between the two buffers in global memory
// (L2), a grid barrier separates the steps.  bar: [0] arrivals, [1] blocks
// that have left, [2] a wait ran out; zero before and after every launch.
// Each wait is bounded (KConsts::wait_ns; 0: gives up at once, met or not): on
// expiry the error flag is set and every block leaves.  The halo copies are
// written by the last step only.
template <int Q, int MAXWARPS>
__global__ void __launch_bounds__(32 * MAXWARPS, 1)
k_steps_cellwarp64_grid(double *f0, double *f1, const __grid_constant__ KConsts<double> k,
                        const __grid_constant__ CellLanes c, int nsteps, unsigned *bar, int *err) {
    using Lane = CellLane<Q, int>;
    constexpr int QP = 8 * Lane::KM;
    __shared__ double s_f[MAXWARPS][QP];
    __shared__ int s_stop;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cell = blockIdx.x * (blockDim.x >> 5) + warp;
    const bool live = cell < k.Nx * k.Ny;
    double *sf = s_f[warp];
    if (lane < QP - Q) sf[Q + lane] = 0.0;
    if (threadIdx.x == 0) s_stop = 0;
    Lane cl;
    long long own = 0;
    if (live) {
        const int j = cell / k.Nx, x = cell - j * k.Nx;
        own = col_index(k, j, x);
        cl.init(k, c, lane, cell, [&](int a, int row, int xc) {
            return (int)(col_index(k, row, xc) + (long long)a * k.pitch);
        });
    }
    for (int n = 0; n < nsteps; ++n) {
        const double *src = (n & 1) ? f1 : f0;
        double *dst = (n & 1) ? f0 : f1;
        if (live) {
            double va, vb;
            cl.step(k, c, sf, va, vb, [&](int o) { return __ldcg(src + o); });
            if (n + 1 == nsteps) {
                cl.store_images(dst, k, cell, va, vb);
            } else if (cl.mine) {
                if (cl.b) dst[own + (long long)cl.b * k.pitch] = vb;
                dst[own + (long long)cl.a * k.pitch] = va;
            }
        }
        if (n + 1 == nsteps) break;
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned goal = gridDim.x * (unsigned)(n + 1);
            unsigned seen;
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(bar) : "memory");
            unsigned long long t0 = 0;
            for (int spin = 0;; ++spin) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(seen) : "l"(bar) : "memory");
                bool late = k.wait_ns == 0;
                if (!late && seen >= goal) break;
                if (late || (spin & 255) == 255) {
                    if (t0 == 0) t0 = global_ns();
                    late = late || global_ns() - t0 > k.wait_ns;
                    if (late) {
                        atomicOr(err, kCellErrTimeout);
                        atomicExch(bar + 2, 1u);
                    }
                    if (late || *(volatile unsigned *)(bar + 2)) {
                        s_stop = 1;
                        break;
                    }
                }
            }
        }
        __syncthreads();
        if (s_stop) break;
    }
    // the last block to leave clears the barrier for the next launch: every
    // block's arrivals (one that gave up has not seen its own counted) come
    // before its count here
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(bar + 1, 1u) == gridDim.x - 1) {
            __threadfence();
            bar[0] = bar[1] = bar[2] = 0u;
        }
    }
}

}  // namespace lbm
