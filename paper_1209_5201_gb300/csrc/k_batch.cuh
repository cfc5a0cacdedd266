// Batched chunk kernel: many independent single-column Couette instances
// (Nx = 1, each with its own lattice, height, Kn, wall speeds and wall
// temperatures) advanced together, `sub` chunks of `chunk` time steps per
// launch, with an FP64 steady-state residual after every check_every-th
// chunk of a slot.
//
// With Nx = 1 the pull of Eq. (5) only shifts in y: f_in(j, a) =
// f~*(j - e_ay, a).  A slot runs on a cluster of CL CTAs (CL = 1, 2, 4, 8 or
// 16): CTA `rank` owns rows [rank R, rank R + R), R =
// ceil(Ny / CL), and a cluster barrier with release / acquire semantics
// separates the steps.  When its rows fit (batch_uses_smem) the CTA keeps them in
// shared memory for the whole launch (loaded from the pool at the start, written
// back at the end; two buffers up to 256 rows, one ring per velocity up to 512:
// SmemState) and pulls the <= 3 rows it needs from each neighbour through
// distributed shared memory (ld.shared::cluster); taller blocks keep the state in
// global memory (L2-resident, two buffers) and read it with ld.global.cg.
//
// Row mapping inside a CTA: warp 0 of the bottom CTA owns the (up to) 32
// lowest rows and warp 0 (one CTA: warp 1) of the top CTA the 32 highest; each of
// those warps first sums its wall's incoming mass (numerator of Eq. (12)) to
// FP64 precision in a fixed order - the (velocity, row) terms of the wall's
// list, built on the host and carried in the slot descriptor - forms the
// normalised re-emission of every outgoing velocity once, and then updates its
// rows (branch-free: sources clamped into the slot, the wall's values selected
// afterwards).  The other rows never need a wall value, so no block barrier
// separates the wall sums from the bulk update (a full ring's first sums excepted:
// run_steps).  Every slot's arithmetic depends only on the slot itself, never on
// its cluster size, the slot index, the grid or other slots.
#pragma once

#include "batch_internal.h"
#include "lbm_device.cuh"

namespace lbm {

// A launch's time as its CTAs hold it: when this one began, LaunchBudget's limits
// and words, and from when on the words are read again (a read of host memory
// takes about 4 us: one per chunk cost a lone 4096-row column 0.5 %).
constexpr unsigned long long kLookNs = 300000ull;
struct LaunchTime {
    unsigned long long t0, base, more, look;
    volatile int *stopped;
    const volatile int *waiting;
};

// After chunk `done` of a slot's launch: whether another one ends in time (st->go).
// Out of line: once per chunk, and its registers are not the step loop's.
__device__ __noinline__ void launch_goes_on(LaunchTime &lt, SlotStatus *st, int sub, int done) {
    const unsigned long long el = global_ns() - lt.t0, end = el + el / (unsigned)done;
    if (done == sub) st->first_ns = (long long)el;
    bool go = end <= lt.base;
    if (!go && end <= lt.more) {
        go = true;
        if (el >= lt.look) {
            go = (*lt.stopped | *lt.waiting) == 0;
            lt.look = el + kLookNs;
        }
    }
    st->go = go && done < kMaxLaunchChunks;
}

// Shared per-step wall data of a slot: the re-emitted deviations of Eq. (12)
// per wall and velocity, the accommodation of each wall in FP32, and (state in
// global memory) the post-collision values of the 3 rows next to each wall,
// term[w][kk][a] at distance kk from wall w, which the next step's wall sum
// reads from here instead of from L2.
struct BatchWallShared {
    float fill[2][kMaxQ];
    float acc[2];
    float term[2][3][kMaxQ];
    int toff[2][kMaxTerm];     // where a state keeps each incoming term (its term_at)
};

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return r;
}

// Barrier of all threads of the slot's cluster, with release / acquire
// semantics at cluster scope: every global store of the cluster before it is
// visible to every thread of the cluster after it.  One CTA: the block barrier.
__device__ __forceinline__ void cluster_arrive() {
    // non-.aligned forms: correct even if a warp arrives diverged
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release;\n" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    asm volatile("barrier.cluster.wait.acquire;\n" ::: "memory");
}
__device__ __forceinline__ void slot_barrier(int CL) {
    if (CL == 1) {
        __syncthreads();
        return;
    }
    cluster_arrive();
    cluster_wait();
}

// Slots of a CTA's shared-memory state (SmemState).
constexpr int kRing = 512;
constexpr int kSmemBytes = kMaxQ * kRing * (int)sizeof(float);

// The shared-memory path serves every column whose CTAs' rows fit: three slots
// fewer than the ring has, or all of them on one CTA between diffuse walls.
__host__ __device__ inline bool batch_uses_smem(int Ny, int CL, bool diffuse) {
    return batch_rows_per_cta(Ny, CL) <= (CL == 1 && diffuse ? kRing : kRing - 3);
}

// Population a of the wall re-emission (Eq. (9) with R = accom R_D + (1 -
// accom) R_S): the diffuse part formed by the wall warp, plus the specular
// part (the mirrored velocity of the same row, `spec`, read only when accom <
// 1); both are deviations from w_a, so the mix is linear in them.
template <class SpecFn>
__device__ __forceinline__ float wall_value(const BatchWallShared &sw, int wall, int a,
                                            SpecFn &&spec) {
    const float acc = sw.acc[wall];
    float v = sw.fill[wall][a];
    if (acc != 1.0f) v = acc * v + (1.0f - acc) * spec();
    return v;
}

// Wall rows of a pull (EDGE): f[a] was loaded from the source row clamped into
// the slot; where the true source lies beyond a wall (e_y > j bottom, j - e_y
// >= Ny top) it is replaced by that wall's re-emission.  Without specular
// reflection the replacement is a predicated select, so the pull has no
// branch between its loads.
template <int Q, class MirrorFn>
__device__ __forceinline__ void apply_walls(const BatchWallShared &sw, int j, int Ny,
                                            float (&f)[Q], MirrorFn &&mirror) {
    using L = Lat<Q>;
    if (sw.acc[0] == 1.0f && sw.acc[1] == 1.0f) {
        StaticFor<0, Q>::run([&](auto ic) {
            constexpr int a = decltype(ic)::value;
            if constexpr (L::ey(a) > 0) f[a] = j - L::ey(a) < 0 ? sw.fill[0][a] : f[a];
            else if constexpr (L::ey(a) < 0) f[a] = j - L::ey(a) >= Ny ? sw.fill[1][a] : f[a];
        });
    } else {
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            const int sj = j - L::ey(a);
            if (sj < 0 || sj >= Ny)
                f[a] = wall_value(sw, sj < 0 ? 0 : 1, a, [&] { return mirror(a, L::ey(a)); });
        }
    }
}

// Slot state in global memory (pool), two buffers of [Q][Ny]; a step reads
// `src` and writes `dst`, rows of any CTA of the cluster.
struct GlobalState {
    static constexpr bool kTwoBuffers = false;   // (of shared memory)
    const float *src;
    float *dst;
    int Ny;
    float *stage;              // BatchWallShared::term of this CTA
    // population a of slot row `row` of the current state (coherent L2 read:
    // another SM may have written it)
    __device__ __forceinline__ float ld(int a, int row) const {
        return __ldcg(src + (long long)a * Ny + row);
    }
    __device__ __forceinline__ float ld_at(int a, int, int row) const { return ld(a, row); }
    // wall w's incoming term (a, kk) of the step just done (staged by store)
    __device__ __forceinline__ int term_off(int w, int a, int, int kk) const { return (w * 3 + kk) * kMaxQ + a; }
    __device__ __forceinline__ float term_at(int off) const { return stage[off]; }
    // f_in of row j (Eq. (5) pull with the Eq. (12) wall)
    template <int Q, bool EDGE>
    __device__ __forceinline__ void pull(const SlotDesc &d, const BatchWallShared &sw, int j,
                                         float (&f)[Q]) const {
        using L = Lat<Q>;
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            const int sj = j - L::ey(a);
            f[a] = ld(a, EDGE ? min(max(sj, 0), Ny - 1) : sj);
        }
        if constexpr (EDGE) apply_walls<Q>(sw, j, Ny, f, [&](int a, int) { return ld(d.k.mirror[a], j); });
    }
    template <int Q>
    __device__ __forceinline__ void store(int j, const float (&o)[Q]) const {
        using L = Lat<Q>;
#pragma unroll
        for (int a = 0; a < Q; ++a) dst[(long long)a * Ny + j] = o[a];
        // the velocities that stream into a wall from its 3 nearest rows
        if (j < 3) {
            StaticFor<0, Q>::run([&](auto ic) {
                constexpr int a = decltype(ic)::value;
                if constexpr (L::ey(a) < 0) stage[j * kMaxQ + a] = o[a];
            });
        } else if (j >= Ny - 3) {
            StaticFor<0, Q>::run([&](auto ic) {
                constexpr int a = decltype(ic)::value;
                if constexpr (L::ey(a) > 0) stage[(3 + Ny - 1 - j) * kMaxQ + a] = o[a];
            });
        }
    }
    __device__ __forceinline__ void flip() {
        const float *t = src;
        src = dst;
        dst = (float *)t;
    }
};

__device__ __forceinline__ float lds_f32(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];\n" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
template <int OFF>
__device__ __forceinline__ float lds_f32(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1+%2];\n" : "=f"(v) : "r"(addr), "n"(OFF) : "memory");
    return v;
}
template <int OFF>
__device__ __forceinline__ void sts_f32(uint32_t addr, float v) {
    asm volatile("st.shared.f32 [%0+%1], %2;\n" ::"r"(addr), "n"(OFF), "f"(v) : "memory");
}
// Load through the shared::cluster window (this CTA's or a neighbour's
// shared memory), without a compiler memory clobber: ordered only against the
// other volatile asm (the loads, stores and barriers of this file), so the
// constants read around it can stay in registers.
template <int OFF>
__device__ __forceinline__ float ldsc_f32_nc(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1+%2];\n" : "=f"(v) : "r"(addr), "n"(OFF));
    return v;
}
// shared::cluster address of the same location in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, unsigned rank) {
    uint32_t out;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(out) : "r"(addr), "r"(rank));
    return out;
}

// Slot state in the cluster's shared memory: rows of Q floats (row-major: a
// thread's Q populations are contiguous and Q is odd, so the 32 lanes of a warp,
// on 32 consecutive rows, hit 32 different banks).  lo / hi are the neighbours'
// shared memory (rows below / above) as shared::cluster addresses, 0 at the
// slot's ends.
//  * Two buffers of up to kRing / 2 rows (RING false): slot lr of a buffer is
//    local row lr; bulk rows read with compile-time offsets.
//  * One buffer of up to kRing rows (RING): every velocity is a ring that turns
//    by its e_y slots per step: after t steps of the launch local row lr is at slot
//    (lr - t e_y) mod kRing, so the value a row pulls and the value it stores for
//    that velocity share one slot, no other row touches it, and a step needs no
//    second buffer.  304 columns of 512 rows: 5.2 us per step, 6.45 with the
//    state in L2, whose bandwidth bounds a full GPU there; the slots' address
//    arithmetic costs 6 % where two buffers fit (a lone 128-row column 1.41 and
//    1.33 us).  What leaves a CTA stays readable in its slots during the step in
//    which what enters it is stored, if the ring has three slots beyond the rows
//    (a neighbour reads it then); on one CTA only its own walls read it, before
//    the step's barrier.
template <int Q, bool RING>
struct SmemState {
    static constexpr bool kTwoBuffers = !RING;
    uint32_t base;             // shared::cta address
    uint32_t lo, hi;           // shared::cluster addresses of the neighbours
    uint32_t self;             // shared::cluster address of this CTA
    int rpc, j0, Ny;           // rows per CTA, first row, rows of the slot
    int t;                     // RING: steps since the launch began; else: current buffer
    // slot of local row lr for a velocity of vertical component e, now
    __device__ __forceinline__ int slot_of(int lr, int e) const {
        if constexpr (RING) return (lr - e * t) & (kRing - 1);
        else return t * (kRing / 2) + lr;
    }
    __device__ __forceinline__ uint32_t slot_addr(int sl) const { return base + (uint32_t)(sl * Q) * 4u; }
    __device__ __forceinline__ void flip() {
        if constexpr (RING) ++t;
        else t ^= 1;
    }
    // population a (vertical component e) of slot row `row` of this CTA, now
    __device__ __forceinline__ float ld_at(int a, int e, int row) const {
        return lds_f32(slot_addr(slot_of(row - j0, e)) + (uint32_t)a * 4u);
    }
    // wall w's incoming term (a, kk), row kk from the wall of the current state:
    // local row, velocity and e_y packed
    __device__ __forceinline__ int term_off(int w, int a, int e, int kk) const {
        return ((w == 0 ? kk : Ny - 1 - kk) - j0) | (a << 16) | ((e + 4) << 24);
    }
    __device__ __forceinline__ float term_at(int off) const {
        return lds_f32(slot_addr(slot_of(off & 0xffff, (off >> 24) - 4)) + (uint32_t)((off >> 16) & 0xff) * 4u);
    }
    template <int Q_, bool EDGE>
    __device__ __forceinline__ void pull(const SlotDesc &d, const BatchWallShared &sw, int j,
                                         float (&f)[Q_]) const {
        using L = Lat<Q_>;
        if constexpr (!EDGE && !RING) {
            // every source row is one of this CTA's: offsets from row lr - 3
            const uint32_t r0 = slot_addr(slot_of(j - j0 - 3, 0));
            StaticFor<0, Q_>::run([&](auto ic) {
                constexpr int a = decltype(ic)::value;
                f[a] = lds_f32<((3 - L::ey(a)) * Q_ + a) * 4>(r0);
            });
            return;
        }
        uint32_t r[7];
        if constexpr (!EDGE) {
            StaticFor<0, 7>::run([&](auto ic) {
                constexpr int e = decltype(ic)::value - 3;
                r[e + 3] = slot_addr(slot_of(j - j0 - e, e));
            });
            StaticFor<0, Q_>::run([&](auto ic) {
                constexpr int a = decltype(ic)::value;
                f[a] = lds_f32<a * 4>(r[L::ey(a) + 3]);
            });
        } else {
            // source row clamped into the slot, then into this CTA or a
            // neighbour (selects, no branch): every load goes through the
            // shared::cluster window and all of them issue back to back
            StaticFor<0, 7>::run([&](auto ic) {
                constexpr int e = decltype(ic)::value - 3;
                const int l = min(max(j - e, 0), d.Ny - 1) - j0;
                const uint32_t bse = l < 0 ? lo : (l >= rpc ? hi : self);
                const int ln = l < 0 ? l + rpc : (l >= rpc ? l - rpc : l);
                r[e + 3] = bse + (uint32_t)(slot_of(ln, e) * Q) * 4u;
            });
            StaticFor<0, Q_>::run([&](auto ic) {
                constexpr int a = decltype(ic)::value;
                f[a] = ldsc_f32_nc<a * 4>(r[L::ey(a) + 3]);
            });
            apply_walls<Q_>(sw, j, d.Ny, f, [&](int a, int e) { return ld_at(d.k.mirror[a], -e, j); });
        }
    }
    template <int Q_>
    __device__ __forceinline__ void store(int j, const float (&o)[Q_]) const {
        using L = Lat<Q_>;
        if constexpr (RING) {
            uint32_t r[7];
            StaticFor<0, 7>::run([&](auto ic) {
                constexpr int e = decltype(ic)::value - 3;
                r[e + 3] = slot_addr(slot_of(j - j0 - e, e));
            });
            StaticFor<0, Q_>::run([&](auto ic) {
                constexpr int a = decltype(ic)::value;
                sts_f32<a * 4>(r[L::ey(a) + 3], o[a]);
            });
        } else {
            const uint32_t r = slot_addr((t ^ 1) * (kRing / 2) + j - j0);
            StaticFor<0, Q_>::run([&](auto ic) {
                constexpr int a = decltype(ic)::value;
                sts_f32<a * 4>(r, o[a]);
            });
        }
    }
};

// Numerator of Eq. (12) for `wall` summed by one full warp, and the normalised
// re-emission M_in g^w_a / D_w of each outgoing velocity (lane l: out_a[l]), as an
// FP32 deviation from w_a.  A step is as long as its wall warp: the update of
// its rows, this, and the barrier.  In FP64 (an add per butterfly stage, the
// conversions, the product) it took 1200 - 1550 cycles of a lone column's 3300 -
// 4900 per step, since every FP64 warp instruction takes 64 on GB300.  So the
// sum of the deviations runs in FP32 with error-free additions (Sum3: to far
// below FP64's rounding): every group of four lanes sums all terms, up to seven
// per lane, then two butterfly stages; and c0 + d c is evaluated in floats to what
// FP64 keeps of it (emit3).  terms(t, x) reads the incoming terms t[] of the
// current state; the wall rows belong to this CTA.
// The FP32 value of each re-emission is rounded stochastically (add_sr of
// its round-to-nearest value and the FP32 remainder), from the hash of the
// step and a counter beyond the slot's rows.
template <int Q>
constexpr int lane_terms() {
    int n = 0;                               // incoming terms per wall
    for (int a = 0; a < Q; ++a) n += Lat<Q>::ey(a) > 0 ? Lat<Q>::ey(a) : 0;
    return (n + 3) / 4;
}
template <int Q, class TermFn>
__device__ __forceinline__ void wall_fill_warp(const SlotDesc &d, int wall, int lane,
                                               float *fill, uint32_t step, TermFn &&terms) {
    constexpr int kLaneTerms = lane_terms<Q>();
    const int l = min(lane, d.nout - 1);
    const Emit3 ce = d.out_e[wall][l];
    // this lane's terms (lane & 3) + 4 i, all loads in flight; past the last
    // term the loads repeat it
    float x[kLaneTerms];
    int t[kLaneTerms];
#pragma unroll
    for (int i = 0; i < kLaneTerms; ++i) t[i] = min((lane & 3) + 4 * i, d.nterm - 1);
    terms(t, x);
    Sum3 sum;
#pragma unroll
    for (int i = 0; i < kLaneTerms; ++i) sum.add((lane & 3) + 4 * i < d.nterm ? x[i] : 0.0f);
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
        const float h = __shfl_xor_sync(0xffffffffu, sum.h, o), m = __shfl_xor_sync(0xffffffffu, sum.m, o),
                    r = __shfl_xor_sync(0xffffffffu, sum.l, o);
        sum.add(h, m, r);
    }
    float hi, lo;
    emit3(ce, sum, hi, lo);
    const uint32_t h = sr_cell(step, (uint32_t)(d.Ny + wall));
    if (lane < d.nout) fill[d.out_a[wall][l]] = add_sr(hi, lo, sr_bits32(h, lane));
    __syncwarp();
}

// Pull, collide and store row j (Eq. (5) with the Eq. (9)-(12) wall).  EDGE:
// the row is within 3 rows of its CTA's first or last row, so a source may lie
// beyond the slot's walls or in a neighbouring CTA; otherwise every source is
// one of this CTA's rows.
// PRECISE: conserving increments with stochastic rounding (the steady-state
// phase of a solve); otherwise the plain relaxation rounded to nearest.
// The two pulls share one collision and store: a step's loop then holds half the
// code, which an SM's instruction cache keeps: a lone 128-row D2Q37 column 1.33 us
// per step, 1.45 with a collision per pull (stochastic 1.78 and 1.83).
template <int Q, bool PRECISE, class State>
__device__ __forceinline__ void cell_update(const SlotDesc &d, const State &S, int j, bool edge,
                                            const BatchWallShared &sw, uint32_t step) {
    // the slot's constants live in shared memory; this compiler barrier keeps
    // them there (re-read per cell) instead of hoisted into registers for the
    // whole step loop, which spilled
    asm volatile("" ::: "memory");
    const KConsts<float> &k = d.k;
    float f[Q];
    if (edge) S.template pull<Q, true>(d, sw, j, f);
    else S.template pull<Q, false>(d, sw, j, f);
    Collision<Q, float, true> col;
    col.setup(f, k);
    // PRECISE: increments that conserve mass, momentum (and energy) in FP32,
    // added with stochastic rounding: random bits from the hash of the
    // request's step count and the row (the same however the column is split
    // or batched)
    float o[Q];
    if constexpr (PRECISE) {
        col.relax_conserving_sr(f, o, sr_cell(step, (uint32_t)j), k.thermal != 0);
    } else {
        o[0] = col.rest(f[0]);
        PairLoop<1, Q>::run([&](auto ic) {
            constexpr int A = decltype(ic)::value;
            col.template pair<A>(f[A], f[A + 1], o[A], o[A + 1]);
        });
    }
    S.template store<Q>(j, o);
}

// The chunk's time steps.  Warp 0 of the bottom CTA and warp 0 (one CTA: warp
// 1) of the top CTA own the wall blocks [j0, j0 + nb) and [j1 - nt, j1) and first
// form their wall's re-emission; every thread then updates its wall-block row (if any)
// and its share of the bulk rows [mb, me), handed out from the last thread
// down so that the wall warps get bulk rows last.
template <int Q, bool PRECISE, class State>
__device__ __forceinline__ void run_steps(const SlotDesc &d, State &S, BatchWallShared &sw,
                                          int chunk, int CL, int warp, int lane, int tid,
                                          int nth, int j0, int j1, int nb, int nt, int mb,
                                          int me, uint32_t step0) {
    constexpr int kLaneTerms = lane_terms<Q>();
    int jw = -1;
    // the top wall's warp: not the bottom wall's, and none of those that the
    // bulk rows of a full CTA with one wall fill
    const int wtop = nb > 0 ? 1 : 0;
    if (warp == 0 && nb > 0 && lane < nb) jw = j0 + lane;
    if (warp == wtop && nt > 0 && lane < nt) jw = j1 - nt + lane;
    const int jb = mb + (nth - 1 - tid);
    // a wall warp's incoming terms are rows of its own wall block
    const bool wall_warp = (warp == 0 && nb > 0) || (warp == wtop && nt > 0);
    const int wall = warp == 0 && nb > 0 ? 0 : 1;
    const int Ny = d.Ny;
    // the chunk's first wall sums read the state as loaded; later ones the
    // wall rows just written (staged in shared memory on the global path)
    if (wall_warp) {
        for (int t = lane; t < d.nterm; t += 32)
            sw.toff[wall][t] = S.term_off(wall, d.term_a[wall][t], d.term_ey[wall][t], d.term_row[wall][t]);
        wall_fill_warp<Q>(d, wall, lane, sw.fill[wall], step0, [&](const int (&t)[kLaneTerms], float (&x)[kLaneTerms]) {
#pragma unroll
            for (int i = 0; i < kLaneTerms; ++i) {
                const int kk = d.term_row[wall][t[i]];
                x[i] = S.ld_at(d.term_a[wall][t[i]], d.term_ey[wall][t[i]], wall == 0 ? kk : Ny - 1 - kk);
            }
        });
    }
    // A full ring (510 to 512 rows on one CTA) has no slot between what leaves
    // the column and what enters it.  Step t moves velocity e of row lr into slot
    // (lr - (t + 1) e) mod 512, where before it stood row lr - e; for lr - e < 0
    // or >= 512 that is row lr - e + 512 or - 512, one of the terms just read
    // (512 rows, e = 1: row 0 stores where row 511's term is; 510 rows, e = 3:
    // row 0 where row 509's is; 509 rows: no such row).  So every wall sum has
    // read its terms before any warp stores: here for the chunk's first step,
    // before the step's barrier for the others.
    if (!State::kTwoBuffers && CL == 1) __syncthreads();
    for (int step = 0; step < chunk; ++step) {
        const uint32_t gstep = step0 + (uint32_t)step;
        for (int it = jw >= 0 ? -1 : 0;; ++it) {
            const int j = it < 0 ? jw : jb + it * nth;
            if (it >= 0 && j >= me) break;
            // one path per warp: a warp with any row within 3 rows of its
            // CTA's ends takes the general (EDGE) path for all its rows, so
            // the collision is never executed twice by a diverged warp
            const bool edge = __any_sync(__activemask(), j < j0 + 3 || j >= j1 - 3);
            cell_update<Q, PRECISE>(d, S, j, edge, sw, gstep);
        }
        // The next step's wall sums read rows of their own warp alone, visible to
        // it after __syncwarp, so they run between arriving at the cluster barrier
        // and waiting on it; on one CTA before the block barrier, for afterwards
        // another warp may store to the slots (of a ring) of what has left the
        // column.  One copy of their code serves every case: a lone D2Q25 column
        // of 256 rows 1.07 us per step, 1.16 with a copy for each.
        __syncwarp();
        if (CL > 1) cluster_arrive();
        S.flip();
        if (wall_warp && step + 1 < chunk)
            wall_fill_warp<Q>(d, wall, lane, sw.fill[wall], gstep + 1u,
                              [&](const int (&t)[kLaneTerms], float (&x)[kLaneTerms]) {
                int off[kLaneTerms];
#pragma unroll
                for (int i = 0; i < kLaneTerms; ++i) off[i] = sw.toff[wall][t[i]];
#pragma unroll
                for (int i = 0; i < kLaneTerms; ++i) x[i] = S.term_at(off[i]);
            });
        if (CL > 1) cluster_wait();
        else __syncthreads();
    }
}

// The chunks of one launch for one slot on CTA `rank` of its CL-CTA cluster:
// d.sub of them, and then more while another one, as long as those so far,
// ends within the launch's time (LaunchBudget; fewer when the slot stops:
// converged, stagnated, non-finite or at max_steps); returns the chunks run.
// Results do not depend on how many chunks a launch runs: 128 mixed columns on
// 304 CTAs, whose tall one-CTA columns take 2.3 ms per chunk and clusters 0.2 -
// 0.7, 473 -> 414 ms to the last one's steady state.  chunks0 / steps0 are the slot's
// counters before the launch (read by every CTA before the first barrier);
// `part` the slot's per-chunk FP64 partial sums of the residual; `sm` the
// CTA's kSmemBytes of dynamic shared memory (used when its rows fit).  A
// residual check follows every check_every-th chunk of the slot's count, so
// the checks fall on the same steps whatever the number of chunks per launch.
template <int Q>
__device__ __forceinline__ int batch_slot(const SlotDesc &d, float *__restrict__ pool,
                                          SlotStatus *__restrict__ st, BatchWallShared &sw,
                                          int rank, int CL, int chunks0, long long steps0,
                                          int precise, double *__restrict__ part, float *sm,
                                          LaunchTime &lt) {
    using L = Lat<Q>;
    const int chunk = d.chunk_steps;
    const KConsts<float> &k = d.k;
    const int Ny = d.Ny;
    const int tid = threadIdx.x, nth = blockDim.x;
    const int warp = tid >> 5, lane = tid & 31;
    const int R = batch_rows_per_cta(Ny, CL);
    const int j0 = min(Ny, rank * R), j1 = min(Ny, j0 + R);
    const bool has_bot = rank == 0, has_top = rank == CL - 1;
    const int span = j1 - j0;
    // wall blocks: >= 3 rows each (every row that pulls from a wall), since
    // the host keeps Ny >= 6 and every CTA of a split >= 32 rows
    int nb = 0, nt = 0;
    if (has_bot && has_top) {
        nb = min(32, span / 2);
        nt = min(32, span - nb);
    } else if (has_bot) {
        nb = min(32, span);
    } else if (has_top) {
        nt = min(32, span);
    }
    const int mb = j0 + nb, me = j1 - nt;
    const bool smem = batch_uses_smem(Ny, CL, k.accom[0] == 1.0 && k.accom[1] == 1.0);

    // Change of the macroscopic fields since the last check (Eq. (3) moments
    // of the state after chunk ck, read through at(a, e_y, local row)), in the units of the accuracy the
    // solve is asked for: over the 32-row blocks of the column, the largest
    // change of a block's mean u_x divided by the wall speed u_ref, and for a
    // thermal lattice also the largest change of a block's mean T.  The block
    // means follow the smooth, slowly decaying modes that set the distance to
    // the steady state and average out the zero-mean noise of the stochastic
    // rounding.  Per 32-row block (one warp each) the changes, the mass and a
    // non-finite flag go to global memory, then one warp of CTA 0 combines
    // the blocks in a fixed order: the result does not depend on how the rows
    // were split across CTAs.  Returns whether the slot keeps running (the
    // same answer in every thread of the cluster).
    auto check = [&](auto &&at, int ck, long long steps_k) -> bool {
        float *prev_u = (float *)(pool + d.prev_off);
        float *prev_T = prev_u + Ny;
        const double r = (double)k.r;
        const int nwarps = nth >> 5;
        for (int c = j0 / kResidualChunk + warp; c * kResidualChunk < j1; c += nwarps) {
            const int j = c * kResidualChunk + lane;
            double acc[6] = {0, 0, 0, 0, 0, 0};
            if (j < j1) {
                // deviations d = f - w: rho = 1 + sum d, sum e w = 0, sum e^2 w = e2w
                double s0 = 0, sx = 0, sy = 0, se = (double)k.e2w;
#pragma unroll
                for (int a = 0; a < Q; ++a) {
                    const float *p = at(a, L::ey(a), j - j0);
                    const double fa = smem ? (double)*p : (double)__ldcg(p);
                    s0 += fa;
                    sx += L::ex(a) * fa;
                    sy += L::ey(a) * fa;
                    se += L::e2(a) * fa;
                }
                const double rh = 1.0 + s0;
                const double u = r * sx / rh, v = r * sy / rh;
                const double T = ((double)k.r2 * se - rh * (u * u + v * v)) / (2.0 * rh);
                const float uf = (float)u, Tf = (float)T;
                acc[0] = (double)uf - (double)prev_u[j];
                acc[2] = (double)Tf - (double)prev_T[j];
                acc[4] = rh;
                acc[5] = (!isfinite(u) || !isfinite(T)) ? 1.0 : 0.0;
                prev_u[j] = uf;
                prev_T[j] = Tf;
            }
#pragma unroll
            for (int i = 0; i < 6; ++i)
                for (int o = 16; o > 0; o >>= 1) acc[i] += __shfl_down_sync(0xffffffffu, acc[i], o);
            if (lane == 0) {
                // block means of the changes (the block's rows: whole blocks
                // except at the top of the column)
                const double nrow = (double)min(kResidualChunk, Ny - c * kResidualChunk);
                acc[0] = fabs(acc[0]) / nrow;
                acc[2] = fabs(acc[2]) / nrow;
                for (int i = 0; i < 6; ++i) part[c * 6 + i] = acc[i];
            }
        }
        slot_barrier(CL);                      // every chunk's partials written
        if (rank == 0) {
            double tot[6] = {0, 0, 0, 0, 0, 0};
            if (warp == 0) {
                const int nch = (Ny + kResidualChunk - 1) / kResidualChunk;
#pragma unroll
                for (int i = 0; i < 6; ++i) {
                    const bool mx = i == 0 || i == 2;
                    double v = 0.0;
                    for (int c = lane; c < nch; c += 32) v = mx ? fmax(v, part[c * 6 + i]) : v + part[c * 6 + i];
                    for (int o = 16; o > 0; o >>= 1) {
                        const double x = __shfl_down_sync(0xffffffffu, v, o);
                        v = mx ? fmax(v, x) : v + x;
                    }
                    tot[i] = v;
                }
            }
            if (tid == 0) {
                SlotStatus &s = *st;
                s.chunks = ck;
                s.steps = steps_k;
                s.checks += 1;
                s.mass = tot[4];
                double res = tot[0] / d.u_ref;
                if (k.thermal) res = fmax(res, tot[2]);
                if (s.precise == 0 && res <= d.precise_from && tot[5] == 0 && isfinite(res)) {
                    // close enough to the steady state for round-off to freeze:
                    // switch to conserving, stochastically rounded increments
                    // (the mass is restored below) and restart the
                    // convergence bookkeeping for the remaining approach
                    s.precise = 2;
                    s.checks = 0;
                    s.res = s.res_prev = 0.0;
                    s.err_est = 1e30;
                    s.best_res = 1e300;
                    s.since_best = 0;
                    if (s.steps >= d.max_steps) s.state = kSlotMaxSteps;
                } else {
                // geometric extrapolation of the remaining change: with a
                // per-check contraction q = res / res_prev < 1, the distance
                // to the steady state is about res q / (1 - q); q from the
                // last two checks, the slower of the two contractions
                const double q1 = s.res > 0 ? res / s.res : 1.0;
                const double q0 = s.res_prev > 0 ? s.res / s.res_prev : 1.0;
                const double q = fmax(q1, q0);
                const double prev_est = s.err_est;
                s.res_prev = s.res;
                s.res = res;
                s.err_est = (q < 0.999) ? res * q / (1.0 - q) : 1e30;
                if (res < s.best_res) { s.best_res = res; s.since_best = 0; }
                else s.since_best += 1;
                if (tot[5] > 0 || !isfinite(res)) s.state = kSlotNonFinite;
                else if (s.checks >= 4 && s.err_est <= d.tol && prev_est <= d.tol) s.state = kSlotConverged;
                // the change stopped shrinking below tol / 4: the column has
                // reached the noise of the stochastic rounding (the check
                // interval makes the slowest mode's decay visible, so a flat
                // change is noise, not slow convergence)
                else if (s.since_best >= 8 && s.best_res <= 0.25 * d.tol) s.state = kSlotConverged;
                else if (s.since_best >= 50) s.state = kSlotStagnated;
                else if (s.steps >= d.max_steps) s.state = kSlotMaxSteps;
                }
            }
        }
        slot_barrier(CL);                      // the new state visible to the cluster
        if (__ldcg(&st->precise) == 2) {
            // the round-to-nearest phase let the column's mass drift by its
            // systematic round-off: restore the admission mass, spread over
            // the cells as rest equilibrium (d_a += dm w_a, no momentum)
            const float dm = (float)((d.mass0 - __ldcg(&st->mass)) / (double)Ny);
            for (int j = j0 + tid; j < j1; j += nth)
#pragma unroll
                for (int a = 0; a < Q; ++a) {
                    float &v = *at(a, L::ey(a), j - j0);
                    v = __fmaf_rn(dm, k.w[a], v);
                }
            slot_barrier(CL);                  // every CTA read precise == 2 and corrected
            if (rank == 0 && tid == 0) st->precise = 1;
            precise = 1;
        }
        return __ldcg(&st->state) == kSlotRunning;
    };
    // after sub-chunk kk of this launch: a check when the slot's chunk count
    // calls for one, else the counters (and the max_steps stop)
    auto after_chunk = [&](auto &&at, int kk) -> bool {
        const int ck = chunks0 + kk;
        const long long steps_k = steps0 + (long long)kk * chunk;
        if (ck % d.check_every == 0) return check(at, ck, steps_k);
        if (rank == 0 && tid == 0) {
            st->chunks = ck;
            st->steps = steps_k;
            if (steps_k >= d.max_steps) st->state = kSlotMaxSteps;
        }
        return steps_k < d.max_steps;
    };

    // one more chunk in this launch?  (the same answer in every thread of the cluster)
    auto another = [&](int done) -> bool {
        if (done < d.sub) return true;
        if (rank == 0 && tid == 0) launch_goes_on(lt, st, d.sub, done);
        slot_barrier(CL);
        return __ldcg(&st->go) != 0;
    };
    // after chunk `done` of this launch: its check, then whether to go on
    auto go_on = [&](auto &&at, int done) -> bool {
        if (after_chunk(at, done)) return another(done);
        if (rank == 0 && tid == 0) *lt.stopped = 1;
        return false;
    };

    float *g_cur = pool + d.f_off + (d.cur ? (long long)Q * Ny : 0);
    float *g_oth = pool + d.f_off + (d.cur ? 0 : (long long)Q * Ny);
    if (tid < 2) sw.acc[tid] = (float)k.accom[tid];
    int done = 0;
    auto run_smem = [&](auto ring) {
        constexpr bool RING = decltype(ring)::value;
        // own rows into slots 0, 1, ... (t = 0)
        for (int i = tid; i < Q * span; i += nth) {
            const int a = i / span, r = i - a * span;
            sm[r * Q + a] = __ldcg(g_cur + (long long)a * Ny + j0 + r);
        }
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(sm);
        SmemState<Q, RING> S{base, 0u, 0u, map_rank(base, rank), R, j0, Ny, 0};
        if (rank > 0) S.lo = map_rank(base, rank - 1);
        if (rank < CL - 1) S.hi = map_rank(base, rank + 1);
        slot_barrier(CL);                      // every CTA loaded before any neighbour reads
        for (;;) {
            const uint32_t s0 = (uint32_t)(steps0 + (long long)done * chunk);
            if (precise) run_steps<Q, true>(d, S, sw, chunk, CL, warp, lane, tid, nth, j0, j1, nb, nt, mb, me, s0);
            else run_steps<Q, false>(d, S, sw, chunk, CL, warp, lane, tid, nth, j0, j1, nb, nt, mb, me, s0);
            ++done;
            // element of population a (vertical component e) of local row r
            const int t = S.t;
            auto at = [=](int a, int e, int r) -> float * {
                const int sl = RING ? (r - e * t) & (kRing - 1) : t * (kRing / 2) + r;
                return sm + sl * Q + a;
            };
            if (!go_on(at, done)) break;
        }
        // write the final state back to the pool buffer it came from
        StaticFor<0, Q>::run([&](auto ic) {
            constexpr int a = decltype(ic)::value;
            for (int r = tid; r < span; r += nth)
                g_cur[(long long)a * Ny + j0 + r] = sm[S.slot_of(r, L::ey(a)) * Q + a];
        });
    };
    if (smem && R <= kRing / 2) {
        run_smem(std::false_type{});
    } else if (smem) {
        run_smem(std::true_type{});
    } else {
        __syncthreads();
        GlobalState S{g_cur, g_oth, Ny, &sw.term[0][0][0]};
        for (;;) {
            const uint32_t s0 = (uint32_t)(steps0 + (long long)done * chunk);
            if (precise) run_steps<Q, true>(d, S, sw, chunk, CL, warp, lane, tid, nth, j0, j1, nb, nt, mb, me, s0);
            else run_steps<Q, false>(d, S, sw, chunk, CL, warp, lane, tid, nth, j0, j1, nb, nt, mb, me, s0);
            ++done;
            const float *src = S.src;
            auto at = [=](int a, int, int r) -> float * {
                return const_cast<float *>(src) + (long long)a * Ny + j0 + r;
            };
            if (!go_on(at, done)) break;
        }
    }
    return done;
}

}  // namespace lbm
