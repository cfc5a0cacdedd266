// One-pass pull kernel of a full time step (Eq. (5) with the Eq. (12) wall).
//
// One thread per fluid cell (x, j); a block covers BX consecutive columns of
// one x-tile in RS consecutive rows (one in the fastest shapes), which each
// thread walks in order.  Every population is read once, straight from global
// memory at the source cell (x - e_ax, j - e_ay): within a tile the Q
// velocities of a row are consecutive segments and the x-halos hold the
// neighbouring tiles' columns, so a warp's 32 loads of one velocity are one
// contiguous (possibly 4..12-byte shifted) run and every source of a cell lies
// at a fixed offset ((a - e_ay Q) pitch - e_ax elements) from the cell's own
// element.  With the tile pitch a compile-time constant (PC, the pitch of
// wide grids) those offsets are immediates of the load and store
// instructions; otherwise they are per-velocity byte offsets added to the
// cell's address.  Blocks holding any of the N rows next to a wall first sum
// that wall's incoming mass M_in for the BX + 6 ghost columns their fill
// populations come from (fixed order, to FP64 precision).
#pragma once

#include <type_traits>

#include "lbm_device.cuh"

namespace lbm {

// Re-emissions of the ghost columns x0 - 3 + t, t in [0, ncols), one column
// per thread: s_fill[l][t] for the l-th outgoing velocity.
template <int PREC, int BX>
using WallFills = typename Store<PREC>::C[kMaxWallOut][BX + 6];
template <int Q, int PREC, int BX>
__device__ __forceinline__ void wall_prologue(const typename Store<PREC>::S *fin,
                                              const float *rin,
                                              const KConsts<typename Store<PREC>::C> &k,
                                              const KWall &kw, int wall, int x0, int ncols,
                                              WallFills<PREC, BX> &s_fill) {
    for (int t = threadIdx.x; t < ncols; t += BX)
        wall_column_fill<Q, PREC>(fin, rin, k, kw, wall, x0 - 3 + t, &s_fill[0][t], BX + 6);
}

// Pull of cell (x, j): src is the cell's own element (velocity 0) in its
// tile, rsrc its density (BF16DEV).  PC > 0: the tile pitch, a compile-time
// constant; PC = 0: the solver's pitch, offsets from the constants.
template <int Q, int PREC, int BX, bool WALL, int PC>
__device__ __forceinline__ void pull(const typename Store<PREC>::S *fin,
                                     const float *rin,
                                     const typename Store<PREC>::S *src,
                                     const float *rsrc,
                                     const KConsts<typename Store<PREC>::C> &k, const KWall &kw,
                                     int x, int j, const WallFills<PREC, BX> &s_fill,
                                     typename Store<PREC>::C (&f)[Q]) {
    using L = Lat<Q>;
    using S = typename Store<PREC>::S;
    using C = typename Store<PREC>::C;
    StaticFor<0, Q>::run([&](auto ac) {
        constexpr int a = decltype(ac)::value;
        const int sj = j - L::ey(a);
        bool wall_src = false;
        if constexpr (WALL && L::ey(a) > 0) wall_src = sj < 0;
        if constexpr (WALL && L::ey(a) < 0) wall_src = sj >= k.Ny;
        if (wall_src) {
            f[a] = s_fill[L::out_rank(a)][(int)threadIdx.x + 3 - L::ex(a)];
        } else {
            C v;
            if constexpr (PC > 0) {
                constexpr long long off = (long long)(a - L::ey(a) * Q) * PC - L::ex(a);
                v = to_c(ld_i<S, off * (long long)sizeof(S)>(src));
                if constexpr (Store<PREC>::dev) {
                    constexpr long long roff = -(long long)L::ey(a) * PC - L::ex(a);
                    v = dev_to_f(v, k.w[a], ld_i<float, roff * 4>(rsrc));
                }
            } else {
                v = to_c(ld_b(src, k.b_src[a]));
                if constexpr (Store<PREC>::dev) v = dev_to_f(v, k.w[a], ld_b(rsrc, k.b_rho[a]));
            }
            f[a] = v;
        }
    });
    if (WALL && !kw.diffuse[j < L::N ? 0 : 1]) {
        const int wall = j < L::N ? 0 : 1;
        StaticFor<0, Q>::run([&](auto ac) {
            constexpr int a = decltype(ac)::value;
            const int sj = j - L::ey(a);
            if (sj < 0 || sj >= k.Ny)
                f[a] = wall_mix<PREC>(f[a], k.accom[wall],
                                      specular_source<PREC>(fin, rin, k, a, L::ex(a), x, j));
        });
    }
}

// Store of population A of the cell whose own element is dst (velocity 0).
template <int PC, bool CS, int A, class S, class C>
__device__ __forceinline__ void store_one(S *dst, const KConsts<C> &k, S v) {
    if constexpr (PC > 0) {
        constexpr long long off = (long long)A * PC * (long long)sizeof(S);
        if constexpr (std::is_same<S, __nv_bfloat16>::value)
            st_i<off, CS>(reinterpret_cast<unsigned short *>(dst), __bfloat16_as_ushort(v));
        else
            st_i<off, CS>(dst, v);
    } else {
        if constexpr (std::is_same<S, __nv_bfloat16>::value)
            st_b<CS>(reinterpret_cast<unsigned short *>(dst), k.b_dst[A], __bfloat16_as_ushort(v));
        else
            st_b<CS>(dst, k.b_dst[A], v);
    }
}

// Store of a cell's Q values v (BF16DEV: and its density) in its own slots
// (dst: its element of velocity 0; rdst: its density) and, for the kPadL
// columns at either end of tile t (xl of w columns), the halo copies.  All
// values first, the copies behind one branch: a branch per velocity between
// the stores costs the 4096 x 2048 FP32 step 17 %.
template <int Q, int PREC, bool CS, int PC>
__device__ __forceinline__ void store_cell(const typename Store<PREC>::S (&v)[Q], float rho,
                                           typename Store<PREC>::S *__restrict__ fout,
                                           float *__restrict__ rout,
                                           typename Store<PREC>::S *__restrict__ dst,
                                           float *__restrict__ rdst,
                                           const KConsts<typename Store<PREC>::C> &k, int t, int xl,
                                           int w, int j) {
    using S = typename Store<PREC>::S;
    StaticFor<0, Q>::run([&](auto ac) {
        constexpr int A = decltype(ac)::value;
        store_one<PC, CS, A>(dst, k, v[A]);
    });
    if constexpr (Store<PREC>::dev) *rdst = rho;
    if (xl < kPadL || xl >= w - kPadL) {
        if (w >= 2 * kPadL) {
            // one copy, at the same offset from every velocity's slot: in the
            // previous tile's right halo (xl < kPadL) or the next tile's left
            // halo (with one tile: the periodic image x + Nx or x - Nx)
            long long d, dr;
            if (xl < kPadL) {
                const int tl = t == 0 ? k.nt - 1 : t - 1;
                const int wl = tile_width(k, tl);
                d = (tl - t) * k.tile_elems + wl;
                dr = (tl - t) * k.tile_rho + wl;
            } else {
                const int tr = t == k.nt - 1 ? 0 : t + 1;
                d = (tr - t) * k.tile_elems - w;
                dr = (tr - t) * k.tile_rho - w;
            }
            StaticFor<0, Q>::run([&](auto ac) {
                constexpr int A = decltype(ac)::value;
                store_one<PC, CS, A>(dst + d, k, v[A]);
            });
            if constexpr (Store<PREC>::dev) rdst[dr] = rho;
        } else {
            // a grid narrower than 2 kPadL: several images per column
            const long long rowq = (long long)j * k.Q;
#pragma unroll
            for (int a = 0; a < Q; ++a)
                store_halo_copies<S>(fout + (rowq + a) * k.pitch, k.tile_elems, k, t, xl, w, v[a]);
            if constexpr (Store<PREC>::dev)
                store_halo_copies<float>(rout + (long long)j * k.pitch, k.tile_rho, k, t, xl, w, rho);
        }
    }
}

// Collide the pulled values f of cell (x, j) — tile t, tile column xl of a
// tile of w columns — and store the result: its own slots (dst: its element
// of velocity 0; rdst: its density, BF16DEV) and, for the kPadL columns at
// either end of the tile, the halo copies.
template <int Q, int PREC, bool CS, int PC, bool ISO2>
__device__ __forceinline__ void collide_store(const typename Store<PREC>::C (&f)[Q],
                                              typename Store<PREC>::S *__restrict__ fout,
                                              float *__restrict__ rout,
                                              typename Store<PREC>::S *__restrict__ dst,
                                              float *__restrict__ rdst,
                                              const KConsts<typename Store<PREC>::C> &k, int t,
                                              int xl, int w, int x, int j, uint32_t seed) {
    using S = typename Store<PREC>::S;
    using C = typename Store<PREC>::C;
    const uint32_t hcell = Store<PREC>::sr ? sr_cell(seed, (uint32_t)j * (uint32_t)k.Nx + (uint32_t)x) : 0u;
    Collision<Q, C, Store<PREC>::shifted, ISO2> col;
    col.setup(f, k);
    C o[Q];
    o[0] = col.rest(f[0]);
    PairLoop<1, Q>::run([&](auto ic) {
        constexpr int A = decltype(ic)::value;
        col.template pair<A>(f[A], f[A + 1], o[A], o[A + 1]);
    });

    S v[Q];
    if constexpr (Store<PREC>::sr) {
        // BF16: the rest velocity alone, then each pair (a, a + 1) rounded by
        // one conversion (the same bits as store_rounded); BF16DEV first
        // takes w_a rho off, BF16SHIFT's collision output is the deviation
        const auto dv = [&](float oa, float wa) {
            if constexpr (Store<PREC>::dev) return f_to_dev(oa, wa, col.rho);
            else return oa;
        };
        const float v0 = dv(o[0], k.w[0]);
        const uint32_t d0 = bf16x2_rounded(v0, v0, sr_word(hcell, 0));   // upper: sr_bits(h, 0)
        v[0] = __ushort_as_bfloat16((unsigned short)(d0 >> 16));
        PairLoop<1, Q>::run([&](auto ic) {
            constexpr int A = decltype(ic)::value;
            const float va = dv(o[A], k.w[A]);
            const float vb = dv(o[A + 1], k.w[A + 1]);
            const uint32_t d = bf16x2_rounded(va, vb, sr_bits_pair(hcell, A));
            v[A] = __ushort_as_bfloat16((unsigned short)(d >> 16));
            v[A + 1] = __ushort_as_bfloat16((unsigned short)d);
        });
    } else {
#pragma unroll
        for (int a = 0; a < Q; ++a) v[a] = store_rounded<S>(o[a], 0u);
    }
    store_cell<Q, PREC, CS, PC>(v, (float)col.rho, fout, rout, dst, rdst, k, t, xl, w, j);
}

// BX threads per block (one row segment of a tile); MINB blocks per SM
// requested from the register allocator; CS: streaming stores; RS rows per
// block, walked in order (rows [RS blockIdx.y, RS blockIdx.y + RS)); PC: the
// tile pitch as a compile-time constant (0: the solver's); ISO2: the
// second-order isothermal equilibrium compiled in.  Grid: blockIdx.x
// = tile * ceil(tw / BX) + block of the tile.
template <int Q, int PREC, int BX, int MINB, bool CS, int RS, int PC, bool ISO2>
__global__ void __launch_bounds__(BX, MINB)
k_step_direct(const typename Store<PREC>::S *fin,
              typename Store<PREC>::S *__restrict__ fout, const float *rin,
              float *__restrict__ rout,
              const __grid_constant__ KConsts<typename Store<PREC>::C> k,
              const __grid_constant__ KWall kw) {
    using L = Lat<Q>;
    using C = typename Store<PREC>::C;
    // both walls' fills only where one block can hold rows of both
    __shared__ WallFills<PREC, BX> s_fill[RS > 1 ? 2 : 1];
    // launched with programmatic stream serialization: the next step's blocks
    // may take the places of finished ones, and everything before the wait
    // overlaps the previous step's last blocks
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    const int bpt = (k.tw + BX - 1) / BX;
    const int t = blockIdx.x / bpt, xl0 = (blockIdx.x - t * bpt) * BX;
    const int w = tile_width(k, t);
    if (xl0 >= w) return;                        // past the last tile's columns
    const int xl = xl0 + threadIdx.x, x = t * k.tw + xl;
    const int j0 = blockIdx.y * RS;
    const int j1 = min(k.Ny, j0 + RS);
    const bool bot = j0 < L::N, top = j1 > k.Ny - L::N;
    const int ncols = min(BX, w - xl0) + 6;
    // the previous step's stores are visible from here on (fin and rin, which it
    // writes, are not __restrict__: that would let loads move above the wait)
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    if (RS > 1) {
        if (bot) wall_prologue<Q, PREC, BX>(fin, rin, k, kw, 0, t * k.tw + xl0, ncols, s_fill[0]);
        if (top) wall_prologue<Q, PREC, BX>(fin, rin, k, kw, 1, t * k.tw + xl0, ncols, s_fill[RS > 1 ? 1 : 0]);
    } else if (bot || top) {
        wall_prologue<Q, PREC, BX>(fin, rin, k, kw, bot ? 0 : 1, t * k.tw + xl0, ncols, s_fill[0]);
    }
    if (bot || top) __syncthreads();
    // BF16: step count of the stochastic rounding (block 0 advances it)
    uint32_t seed = 0;
    if constexpr (Store<PREC>::sr)
        seed = step_count(fin, k, blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0);
    if (xl >= w) return;
    const long long pitch = PC > 0 ? PC : k.pitch;
    const long long cell0 = t * k.tile_elems + xl + kPadL;
    const long long rcell0 = t * k.tile_rho + xl + kPadL;
    for (int j = j0; j < j1; ++j) {
        const long long cell = cell0 + (long long)j * Q * pitch;
        const long long rcell = rcell0 + (long long)j * pitch;
        const float *rsrc = Store<PREC>::dev ? rin + rcell : nullptr;
        float *rdst = Store<PREC>::dev ? rout + rcell : nullptr;
        C f[Q];
        if (j < L::N || j >= k.Ny - L::N)
            pull<Q, PREC, BX, true, PC>(fin, rin, fin + cell, rsrc, k, kw, x, j,
                                        s_fill[RS > 1 && j >= L::N ? 1 : 0], f);
        else
            pull<Q, PREC, BX, false, PC>(fin, rin, fin + cell, rsrc, k, kw, x, j, s_fill[0], f);
        collide_store<Q, PREC, CS, PC, ISO2>(f, fout, rout, fout + cell, rdst, k, t, xl, w, x, j, seed);
    }
}

}  // namespace lbm
