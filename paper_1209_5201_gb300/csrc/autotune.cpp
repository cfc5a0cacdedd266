// Tile / block-shape autotuner of the step kernel.
//
// Candidates: every variant of the one-pass direct kernel (variant 0's once, though the
// same request may be listed again) and of the TMA-staged one compiled for the solver's
// precision, which round alike; in FP64 also the one-warp-per-cell kernel.
// FP32 and BF16 grids take the latter by size alone (cellwarp_by_size).  Each runs
// `trial` steps after two warm-up steps, timed with CUDA events on the solver's
// stream; the fastest wins.
// Results are cached per (lattice, precision, order, Nx class, Ny class) for
// the life of the process and, when LBM_AUTOTUNE_CACHE names a file, across
// processes (one "key kernel variant ms" line per class).
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <mutex>
#include <string>

#include "launchers.h"
#include "lbm_internal.h"

namespace lbm {

namespace {

struct Choice {
    int kernel, variant;
    double ms;
};

std::mutex g_mu;
std::map<std::string, Choice> g_cache;
bool g_loaded = false;

int size_class(int n) {
    int c = 1;
    while (c < n) c <<= 1;
    return c;
}

std::string class_key(const SolverImpl &s) {
    char buf[128];
    std::snprintf(buf, sizeof buf, "Q%d_p%d_o%d_x%d_y%d", s.L.kind, s.p.precision, s.p.eq_order,
                  size_class(s.p.Nx), size_class(s.p.Ny));
    return buf;
}

void load_file_cache() {
    if (g_loaded) return;
    g_loaded = true;
    const char *path = std::getenv("LBM_AUTOTUNE_CACHE");
    if (!path) return;
    FILE *fh = std::fopen(path, "r");
    if (!fh) return;
    char key[100];
    Choice c;
    while (std::fscanf(fh, "%99s %d %d %lf", key, &c.kernel, &c.variant, &c.ms) == 4)
        g_cache[key] = c;
    std::fclose(fh);
}

void append_file_cache(const std::string &key, const Choice &c) {
    const char *path = std::getenv("LBM_AUTOTUNE_CACHE");
    if (!path) return;
    FILE *fh = std::fopen(path, "a");
    if (!fh) return;
    std::fprintf(fh, "%s %d %d %.6f\n", key.c_str(), c.kernel, c.variant, c.ms);
    std::fclose(fh);
}

// n steps by the launches lbm_solver_step makes: of the one-warp-per-cell kernel
// many steps in one where it has such a launch
int enqueue(SolverImpl &s, int kernel, int variant, int n) {
    while (n >= 2 && kernel == LBM_KERNEL_CELLWARP) {
        const int m = std::min(n, kLaunchSteps);
        const int e = launch_many_steps(s, m);
        if (e == (int)cudaErrorNotSupported) break;
        if (e) return LBM_ECUDA;
        s.cur ^= m & 1;
        n -= m;
    }
    for (int i = 0; i < n; ++i) {
        if (launch_step_variant(s, s.cur, s.cur ^ 1, kernel, variant)) return LBM_ECUDA;
        s.cur ^= 1;
    }
    return LBM_OK;
}

int time_candidate(SolverImpl &s, int kernel, int variant, int trial, double *ms) {
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return LBM_ECUDA;
    if (cudaEventCreate(&e1) != cudaSuccess) { cudaEventDestroy(e0); return LBM_ECUDA; }
    int rc = enqueue(s, kernel, variant, 2);
    cudaEventRecord(e0, s.stream);
    if (!rc) rc = enqueue(s, kernel, variant, trial);
    cudaEventRecord(e1, s.stream);
    float t = 0;
    if (!rc && cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&t, e0, e1) == cudaSuccess)
        *ms = t / trial;
    else
        rc = LBM_ECUDA;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return rc;
}

// Whether a tuned FP32 or BF16 grid takes the one-warp-per-cell kernel.  That
// kernel sums the moments in another order than the others, so the choice shows
// in the results (at FP32 round-off; in BF16 through the rounding of what is
// stored): it is made by size, not by a timing that differs from run to run, and
// the line is not moved with the kernels' speeds, for that would change the
// results of grids in use.  (Below it the one-thread kernels are the faster ones
// in FP32: D2Q37 60 x 60 4.0 us per step, one warp per cell 11.2; set_kernel
// takes either.)  Cells of a grid of fewer and of kWideColumns or more columns:
// a wide grid has more wall rows to its cells, whose warps sum the incoming mass
// of seven ghost columns first.
constexpr int kWideColumns = 120;
bool cellwarp_by_size(const SolverImpl &s) {
    struct Line { long long narrow, wide; };
    constexpr Line fp32[3] = {{6500, 4100}, {4800, 2200}, {0, 0}},
                   dev[3] = {{13000, 13000}, {9700, 9700}, {3700, 3700}},
                   shift[3] = {{11000, 11000}, {9000, 9000}, {2700, 2200}};
    if (s.p.precision == LBM_FP64) return false;
    const int i = s.L.Q == 37 ? 0 : s.L.Q == 25 ? 1 : 2;
    const Line l = s.p.precision == LBM_FP32 ? fp32[i] : s.p.precision == LBM_BF16DEV ? dev[i] : shift[i];
    return (long long)s.p.Nx * s.p.Ny <= (s.p.Nx < kWideColumns ? l.narrow : l.wide);
}

}  // namespace

int autotune_solver(SolverImpl &s, int trial) {
    const long long cells = (long long)s.p.Nx * s.p.Ny;
    const bool by_size = s.p.precision != LBM_FP64;
    const bool small = cellwarp_by_size(s);
    // a size class may straddle the line: an entry for each side
    const std::string key = class_key(s) + (small ? "_w" : "");
    {
        std::lock_guard<std::mutex> lk(g_mu);
        load_file_cache();
        auto it = g_cache.find(key);
        if (it != g_cache.end() &&
            (!by_size || small == (it->second.kernel == LBM_KERNEL_CELLWARP))) {
            s.p.kernel = it->second.kernel;
            s.variant = it->second.variant;
            s.tuned_ms = it->second.ms;
            return LBM_OK;
        }
    }
    // a valid state to step on; the caller re-initialises afterwards
    int rc = dispatch_init_rest(s);
    if (rc) return rc;
    Choice best{LBM_KERNEL_DIRECT, 0, 1e30};
    double ms = 0;
    const int nd = small ? 0 : direct_variant_count(s.p.precision);
    for (int v = 0; v < nd; ++v) {
        if (direct_variant_repeats(s, v)) continue;
        if ((rc = time_candidate(s, LBM_KERNEL_DIRECT, v, trial, &ms))) return rc;
        if (ms < best.ms) best = Choice{LBM_KERNEL_DIRECT, v, ms};
    }
    // the staged kernel: grids stored as one x-tile only
    const int nv = s.nt == 1 && !small ? staged_variant_count(s.p.precision) : 0;
    for (int v = 0; v < nv; ++v) {
        if ((rc = time_candidate(s, LBM_KERNEL_STAGED, v, trial, &ms))) return rc;
        if (ms < best.ms) best = Choice{LBM_KERNEL_STAGED, v, ms};
    }
    // one warp per cell: FP64, where it is timed on small grids (32 threads a cell)
    if (by_size ? small : cells <= 16 * kCellwarpAutoCells) {
        if ((rc = time_candidate(s, LBM_KERNEL_CELLWARP, 0, trial, &ms))) return rc;
        if (ms < best.ms) best = Choice{LBM_KERNEL_CELLWARP, 0, ms};
    }
    s.p.kernel = best.kernel;
    s.variant = best.variant;
    s.tuned_ms = best.ms;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        g_cache[key] = best;
        append_file_cache(key, best);
    }
    return dispatch_init_rest(s);
}

}  // namespace lbm
