// Slot table of the batched / serving path, shared by the chunk kernel and
// the host runtime.
#pragma once

#include "float_pairs.h"
#include "lbm_internal.h"

namespace lbm {

// States of a slot (SlotStatus::state).
constexpr int kSlotIdle = 0;
constexpr int kSlotRunning = 1;
constexpr int kSlotConverged = 2;
constexpr int kSlotNonFinite = 3;
constexpr int kSlotMaxSteps = 4;
constexpr int kSlotStagnated = 5;
constexpr int kSlotCancelled = 6;         // set by the host; the kernel skips the slot

// Most velocities leaving one wall (e.n > 0): 15 for D2Q37.
constexpr int kMaxOut = 16;
// Most incoming terms per wall: 26 for D2Q37.
constexpr int kMaxTerm = 28;
// Chunks one launch runs for one slot: at most kMaxSub for certain (SlotDesc::
// sub), and more, up to kMaxLaunchChunks, while they fit the launch's time.
constexpr int kMaxSub = 16;
constexpr int kMaxLaunchChunks = 256;
// While nothing waits for its end, a launch goes on for about this long (ns):
// the host's work per launch is 20 - 50 us.
constexpr unsigned long long kMinLaunchNs = 2000000ull;
// How long a launch may last (device memory, uploaded with each launch).  Slots
// run further chunks up to `base`, the time the slowest of them takes for its
// own chunks anyway, and up to `more` as long as no slot has stopped in this
// launch (its result is read out at the launch's end) and the host has not
// raised its word (a request has arrived or is to be cancelled).
struct LaunchBudget {
    unsigned long long base, more;
    int stopped;              // set by the kernels
};
// Chunks per launch of a slot on a cluster of cl CTAs: about the factor by
// which the cluster shortens a step of a tall column, conservatively, so that
// a cluster slot is rarely the one a launch waits for.
inline int batch_sub_chunks(int cl) { return cl <= 2 ? 1 : cl / 2; }

struct SlotDesc {
    int Q;                    // 17, 25 or 37 (0: idle slot)
    int Ny;
    int cur;                  // buffer holding the current state (0 / 1)
    int check_every;          // residual every check_every chunks
    int chunk_steps;          // steps this slot runs per chunk launch
    int cl;                   // CTAs of the slot's cluster: 1, 2, 4, 8 or 16
    int sub;                  // chunks every launch runs (a cluster several, so that
                              // it keeps pace with one-CTA slots' launches); more
                              // follow while they fit the launch's time
    long long f_off;          // element offset of buffer 0 in the pool
    long long prev_off;       // element offset of the previous-check u_x, T
    double tol;               // target of the extrapolated distance to steady state
    long long max_steps;
    double u_ref;             // velocity scale of the change measure: max |u_wall|
    double mass0;             // the column's mass at admission (sum of rho)
    double precise_from;      // change per check below which the slot switches
                              // to stochastic rounding and conserving increments
    // initial state: u_x(y) = u0 + u1 (y - 1/2), T(y) = T0 + T1 y + T2 y (1 - y)
    // at rho = 1 (y = (j + 1/2) / Ny); rest: u0 = u1 = T1 = T2 = 0, T0 = 1
    double init_u0, init_u1, init_T0, init_T1, init_T2;
    // incoming terms of Eq. (12)'s numerator, built on the host: wall w (0
    // bottom, 1 top), term l < nterm is velocity term_a[w][l] at distance
    // term_row[w][l] from the wall
    int nterm;                // <= kMaxTerm
    int nout;                 // outgoing velocities per wall (e.n > 0), <= kMaxOut
    signed char term_a[2][32];
    signed char term_row[2][32];
    signed char term_ey[2][32];   // its e_y
    signed char out_a[2][kMaxOut];
    // its re-emission M_in g^w_a / D_w - w_a = c0 + d c with d the sum of the
    // incoming deviations, c = g^w_a / D_w and c0 = (the terms' weights) c - w_a
    Emit3 out_e[2][kMaxOut];
    KConsts<float> k;         // per-instance constants (Nx = 1, pitch = 1)
};

struct SlotStatus {
    long long steps;          // steps run since admission
    double res;               // last change over one check: max(L-inf |du_x| / u_ref,
                              // thermal: L-inf |dT|)
    double res_prev;          // change over the check before
    double err_est;           // extrapolated distance to the steady state (same units)
    double best_res;          // smallest change so far
    double mass;              // sum of rho (FP64) at the last check
    int state;                // kSlot*
    int checks;
    int since_best;           // checks without a new smallest residual
    int chunks;               // chunks run since admission
    long long first_ns;       // time the last launch's d.sub chunks took
    int go;                   // another chunk in this launch (shared by the cluster)
    int precise;              // 0: round-to-nearest collision; 1: conserving
                              // increments with stochastic rounding (2: switching)
};

// Cluster sizes of the slot classes.
constexpr int kBatchClasses = 5;
constexpr int kBatchClassCL[kBatchClasses] = {1, 2, 4, 8, 16};
// Tallest column a request may have.
constexpr int kMaxNy = 8192;
// Rows of the residual's partial sums (one warp each) and their most per slot.
constexpr int kResidualChunk = 32;
constexpr int kMaxResidualChunks = kMaxNy / kResidualChunk;

// Rows per CTA of a column of Ny rows on a cluster of CL CTAs: all of them on
// one CTA, else ceil(Ny / CL) rounded up to whole residual chunks, so that no
// chunk straddles two CTAs.
__host__ __device__ inline int batch_rows_per_cta(int Ny, int CL) {
    if (CL <= 1) return Ny;
    const int r = (Ny + CL - 1) / CL;
    return (r + kResidualChunk - 1) / kResidualChunk * kResidualChunk;
}
// A split is usable when every CTA, the last included, gets >= 32 rows.
__host__ __device__ inline bool batch_split_ok(int Ny, int CL) {
    if (CL == 1) return Ny >= 6;
    const int R = batch_rows_per_cta(Ny, CL);
    return (CL == 2 || CL == 4 || CL == 8 || CL == 16) && (CL - 1) * R + 32 <= Ny;
}
// The largest cluster a column of Ny rows may use: the smallest CL whose CTAs
// get at most `rows` rows each (max_cl if none does), reduced until the split
// is usable and fits the CTA budget.
inline int batch_cluster_size(int Ny, int rows, int max_ctas, int max_cl) {
    int cl = 1;
    while (cl < max_cl && batch_rows_per_cta(Ny, cl) > rows) cl *= 2;
    while (cl > 1 && (cl > max_ctas || !batch_split_ok(Ny, cl))) cl /= 2;
    return cl;
}

int preload_batch_kernels();
// 16 when the device can schedule a 16-CTA cluster of the chunk kernel (a
// non-portable size), else 8.
int batch_max_cluster();
// dbg: 8 device ints; dbg[0] != 0 records the first invalid descriptor or
// read-out offset a kernel met (and skipped).
// Chunks of the slots [slot0, slot0 + nlanes), each on a cluster of CL CTAs;
// waiting: the host's word (pinned memory), see LaunchBudget; part:
// kMaxResidualChunks x 6 FP64 residual partials per slot of the whole table.
int launch_batch_chunk(cudaStream_t st, SlotDesc *desc, SlotStatus *status, float *pool,
                       double *part, int slot0, int nlanes, int CL, long long pool_elems,
                       LaunchBudget *budget, const int *waiting, int *dbg);
int launch_batch_init(cudaStream_t st, SlotDesc *desc, float *pool, const int *slots, int n,
                      float rho0, int nslots, long long pool_elems, int *dbg);
int launch_batch_macros(cudaStream_t st, const SlotDesc *desc, const float *pool,
                        const int *slots, const long long *out_off, double *out, int n,
                        int nslots, long long pool_elems, long long out_elems, int *dbg);

}  // namespace lbm
