// Host runtime behind the C ABI of include/dirac.h: grid handles, phase tables, launch planning,
// CUDA-graph replay of the step loop, observables and the autotuner.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/dirac.h"
#include "dirac_internal.cuh"
#include "rows.cuh"

using namespace dirac;

namespace {

thread_local std::string g_thread_err;

constexpr int kGraphBlocks = 32;   // step launches captured in one graph (even: parity returns)
constexpr int kObsBlocksMax = 1216;

struct Plan {
    int K = 1, P = 2, wpb = 4;
    int64_t strip_w = 0, nstrips = 0, nsegs = 0, seg_h = 0;
    const TileShape *tile = nullptr;  // 2-D small grids: the tile kernel's shape (tile_kernels.cuh); null: the row kernel
    int z_threads = 128;
    int64_t z_nsegs = 1, z_seg_h = 0;
    // 3-D: fused single-pass step (fused3d_kernels.cuh) instead of the x-y pass + z/phase pass
    int fused3d = 0, f_warps = 16;
    int64_t f_nstrips = 0, f_nytiles = 0, f_nzsegs = 0, f_zseg_h = 0;
    // two steps per fused pass (K = 2): 28-cell strips x tiles of one or two rows a warp, four of them halo
    int f2_warps = 16;
    int64_t f2_nstrips = 0, f2_nytiles = 0, f2_nzsegs = 0, f2_zseg_h = 0;
    // 3-D second-order step: three fused passes (strang3d_kernels.cuh) instead of eight single sweeps
    int s3_fused = 0, s3_warps = 16, s3_zfactor = 2;
    // 3-D second order as single sweeps with one-cell x shifts: C D C as one z-phase-z pass (seven launches a step)
    int s3_zpass = 0;
    struct XY {
        int64_t nstrips = 0, nytiles = 0, nzsegs = 0, zseg_h = 0;
    } s3_xy[2];  // x-y-x pass (half step) and x-y-x-x-y-x pass (two half steps)
    int64_t s3_z_nsegs = 1, s3_z_seg_h = 0;
};

}  // namespace

struct dirac_grid {
    dirac_config cfg{};
    cudaStream_t stream = nullptr;
    cudaStream_t cap_stream = nullptr;
    int fp32 = 0;
    int fx = 0;        // DIRAC_FX64: int64 fixed-point state q = psi 2^fx_shift
    int fx_shift = 0;
    size_t elem = 8;
    int64_t ncells = 0;
    void *psi[2] = {nullptr, nullptr};
    bool ext = false;  // psi[] are the caller's buffers (cfg.ext_state): never freed, not in device_bytes
    int cur = 0;
    void *table = nullptr;
    size_t table_cap = 0;  // bytes
    int table_full = 0;
    double *flux_part = nullptr;
    size_t flux_part_cap = 0;  // doubles
    size_t flux_used = 0;      // doubles of it that launches since the last fold write
    FluxFold flux{};           // and their places; empty between calls of dirac_step
    double *flux_dev = nullptr;
    unsigned *wait_err = nullptr;  // set by a step kernel whose bounded wait ran out
    std::vector<double> absorb;      // per-x-column damping factors (empty: none)
    std::vector<double> v_host;      // last potential set (for rebuilding the table)
    int v_layout = DIRAC_V_NONE;
    std::vector<double> avec;        // uniform vector potential: field integrals, 3 per step (empty: none)
    double *ucoef = nullptr;         // device: 12 doubles of U entries per step
    size_t ucoef_cap = 0;            // bytes
    // field varying in space and time (dirac_set_field): envelope integrals (4 per step; empty: none) on the host,
    // profiles a (3 per cell) and w (1 per cell), V dt per table entry and absorber factors on the device
    std::vector<double> fenv;
    double *fa_dev = nullptr, *fw_dev = nullptr, *fvdt_dev = nullptr, *fabs_dev = nullptr;
    size_t fa_bytes = 0, fw_bytes = 0, fvdt_bytes = 0, fabs_bytes = 0;
    bool tuning = false;             // autotune timing runs: table rows taken modulo its length
    int inject_stall = 0;            // DIRAC_INJECT_STALL set at creation: every step launch stalls one copy
    double *obs_partial = nullptr;
    double *obs_out = nullptr;
    double *host_obs = nullptr;  // pinned [8]
    double *density_tmp = nullptr;
    int obs_blocks = 0;
    int64_t step = 0;
    double dt = 0;
    int sm_count = 0;
    Plan plan;
    cudaGraphExec_t graph[2] = {nullptr, nullptr};
    int64_t graph_launches[2] = {0, 0};  // kernels in each
    int64_t launches = 0;
    size_t device_bytes = 0;
    std::string err;
};

namespace {

dirac_status fail(dirac_grid *g, dirac_status st, const std::string &msg) {
    if (g)
        g->err = msg;
    else
        g_thread_err = msg;
    return st;
}

dirac_status cuda_fail(dirac_grid *g, cudaError_t e, const char *where) {
    std::string msg = std::string(where) + ": " + cudaGetErrorName(e) + " (" + cudaGetErrorString(e) + ")";
    return fail(g, e == cudaErrorMemoryAllocation ? DIRAC_ERR_OOM : DIRAC_ERR_CUDA, msg);
}

#define CK(g, expr)                                            \
    do {                                                       \
        cudaError_t e_ = (expr);                               \
        if (e_ != cudaSuccess) return cuda_fail((g), e_, #expr); \
    } while (0)

int ndim_of(const dirac_grid *g) { return g->cfg.ndim; }
bool strang(const dirac_grid *g) { return g->cfg.splitting == DIRAC_STRANG; }
// Power-of-two scale the phase coefficients carry for the sweeps' 1/2 factors: 1/4 (2-D), 1/8 (3-D),
// 1/16 (2-D Strang: four sweeps per step).
// Power-of-two scale the phase coefficients carry for the sweeps' 1/2 factors: 1/4 (2-D), 1/8 (3-D),
// 1/16 (2-D Strang: four sweeps per step), 1/256 (3-D Strang: eight sweeps per step).
double scale_of(const dirac_grid *g) {
    // fixed-point 3-D second-order steps: the phase carries the first four halves, the last sweep the rest
    if (strang(g) && ndim_of(g) == 3 && g->fx) return 0.0625;
    if (strang(g)) return ndim_of(g) == 3 ? 1.0 / 256.0 : 0.0625;
    return ndim_of(g) == 3 ? 0.125 : 0.25;
}
int char_shift(const dirac_grid *g) { return g->cfg.char_shift > 1 ? g->cfg.char_shift : 1; }
// Step form: 0 2-D first order, 1 3-D first order, 2 2-D second order, 3 2-D first order with a vector potential,
// 4 2-D first order with char_shift > 1, 5 2-D second order with a vector potential, 6 3-D second order (any
// char_shift), 7 single-sweep launches with char_shift > 1 (3-D first order, 2-D second order), 8 single-sweep
// launches with a field varying in space and time (every dimension, splitting and char_shift).
int sweep_mode(const dirac_grid *g) {
    if (!g->fenv.empty()) return 8;
    if (strang(g)) return ndim_of(g) == 3 ? 6 : (char_shift(g) > 1 ? 7 : (g->avec.empty() ? 2 : 5));
    if (ndim_of(g) == 3) return char_shift(g) > 1 ? 7 : 1;
    if (char_shift(g) > 1) return 4;
    return g->avec.empty() ? 0 : 3;
}
int levels(const dirac_grid *g, int K) { return strang(g) ? 2 * K : K; }
// a uniform vector potential is set (2-D: mode 3; 3-D: the fused pass with the phase matrix)
bool field_on(const dirac_grid *g) { return !g->avec.empty(); }
// 3-D steps run as the fused single pass (chosen by the plan, or required by a vector potential)
bool cellfield_on(const dirac_grid *g) { return !g->fenv.empty(); }
bool fused_pass(const dirac_grid *g) {
    return ndim_of(g) == 3 && !strang(g) && char_shift(g) == 1 && !cellfield_on(g) && (g->plan.fused3d || field_on(g));
}
// 3-D second-order step as the x-y-x, z-phase-z, x-y-x passes
bool strang3d_fused(const dirac_grid *g) { return sweep_mode(g) == 6 && g->plan.s3_fused && char_shift(g) == 1; }
bool strang3d_zpass(const dirac_grid *g) {
    return sweep_mode(g) == 6 && !g->plan.s3_fused && g->plan.s3_zpass && char_shift(g) == 1;
}
// x halo cells of a strip (each side) for K steps per launch
int halo_of(const dirac_grid *g, int K) { return sweep_mode(g) == 4 ? char_shift(g) : levels(g, K); }
double cell_volume(const dirac_grid *g) {
    const double dx = g->cfg.dx;
    return ndim_of(g) == 3 ? dx * dx * dx : dx * dx;
}

// A graph holds the arguments of its launches: the plan, the buffers' addresses, the kind of the table, a fixed-point state's
// scale (which multiplies the flux).  Called wherever one of them changes.
void drop_graphs(dirac_grid *g) {
    for (auto &x : g->graph)
        if (x) {
            cudaGraphExecDestroy(x);
            x = nullptr;
        }
}

// Grows a device buffer of the grid to `bytes` (its contents are lost).  The new one is allocated before the old one is freed,
// so that a call that runs out of memory leaves the grid with the buffer that its next steps use.
template <typename T> dirac_status grow(dirac_grid *g, T *&dev, size_t &cap, size_t bytes) {
    if (bytes <= cap) return DIRAC_OK;
    T *fresh = nullptr;
    CK(g, cudaMalloc((void **)&fresh, bytes));
    if (dev) cudaFree(dev);
    g->device_bytes += bytes - cap;
    dev = fresh;
    cap = bytes;
    return DIRAC_OK;
}

dirac_status ensure_table(dirac_grid *g, size_t bytes) {
    if (bytes <= g->table_cap) return DIRAC_OK;
    dirac_status st = grow(g, g->table, g->table_cap, bytes);
    if (st == DIRAC_OK) drop_graphs(g);
    return st;
}

dirac_status upload_field_aux(dirac_grid *g);

dirac_status upload_table(dirac_grid *g, const double *V, int layout, int64_t count) {
    // with a vector potential the mass term lives in the U matrix and the table holds exp(-i V dt) alone
    const double mu = field_on(g) ? 0.0 : g->cfg.m * g->cfg.c * g->cfg.c * g->dt;
    const double scale = scale_of(g);
    const int64_t nentries = (layout == DIRAC_V_FULL) ? g->ncells : g->cfg.n[0];
    (void)count;
    const size_t bytes = (size_t)nentries * 4 * g->elem;
    dirac_status st = ensure_table(g, bytes);
    if (st != DIRAC_OK) return st;
    if (g->fx) {
        // round(p 2^62), p = the FP64 coefficient (which carries the 1/4): the phase product of the kernel
        std::vector<long long> h((size_t)nentries * 4);
#pragma omp parallel for schedule(static)
        for (int64_t e = 0; e < nentries; ++e) {
            const double v = (layout == DIRAC_V_NONE) ? 0.0 : V[e];
            double p[4];
            if (g->absorb.empty())
                phase_coeffs(mu, v, g->dt, scale, p);
            else
                phase_coeffs_masked(mu, v, g->dt, g->absorb[e % g->cfg.n[0]], scale, p);
            for (int k = 0; k < 4; ++k) h[e * 4 + k] = (long long)std::nearbyint(std::ldexp(p[k], 62));
        }
        CK(g, cudaMemcpyAsync(g->table, h.data(), bytes, cudaMemcpyHostToDevice, g->stream));
        CK(g, cudaStreamSynchronize(g->stream));
    } else if (g->fp32) {
        std::vector<float> h((size_t)nentries * 4);
#pragma omp parallel for schedule(static)
        for (int64_t e = 0; e < nentries; ++e) {
            const double v = (layout == DIRAC_V_NONE) ? 0.0 : V[e];
            const double a = g->absorb.empty() ? 1.0 : g->absorb[e % g->cfg.n[0]];
            double p[4];
            phase_coeffs(mu, v, g->dt, 1.0, p);
            float cu, su, cd, sd;
            if (a == 1.0) {
                round_unitary(p[0], p[1], cu, su);
                round_unitary(p[2], p[3], cd, sd);
            } else {
                cu = (float)(p[0] * a);
                su = (float)(p[1] * a);
                cd = (float)(p[2] * a);
                sd = (float)(p[3] * a);
            }
            h[e * 4 + 0] = cu * (float)scale;
            h[e * 4 + 1] = su * (float)scale;
            h[e * 4 + 2] = cd * (float)scale;
            h[e * 4 + 3] = sd * (float)scale;
        }
        CK(g, cudaMemcpyAsync(g->table, h.data(), bytes, cudaMemcpyHostToDevice, g->stream));
        CK(g, cudaStreamSynchronize(g->stream));
    } else {
        std::vector<double> h((size_t)nentries * 4);
#pragma omp parallel for schedule(static)
        for (int64_t e = 0; e < nentries; ++e) {
            const double v = (layout == DIRAC_V_NONE) ? 0.0 : V[e];
            if (g->absorb.empty())
                phase_coeffs(mu, v, g->dt, scale, &h[e * 4]);
            else
                phase_coeffs_masked(mu, v, g->dt, g->absorb[e % g->cfg.n[0]], scale, &h[e * 4]);
        }
        CK(g, cudaMemcpyAsync(g->table, h.data(), bytes, cudaMemcpyHostToDevice, g->stream));
        CK(g, cudaStreamSynchronize(g->stream));
    }
    if (g->table_full != (layout == DIRAC_V_FULL)) drop_graphs(g);
    g->table_full = (layout == DIRAC_V_FULL);
    return cellfield_on(g) ? upload_field_aux(g) : DIRAC_OK;
}

// Copies n doubles from the host to a device array of the grid, (re)allocating it to fit; n = 0 frees it.
dirac_status put_doubles(dirac_grid *g, double *&dev, size_t &bytes, const double *host, size_t n) {
    const size_t need = n * sizeof(double);
    if (need == 0) {
        if (dev) cudaFree(dev);
        g->device_bytes -= bytes;
        dev = nullptr;
        bytes = 0;
        return DIRAC_OK;
    }
    dirac_status st = grow(g, dev, bytes, need);
    if (st != DIRAC_OK) return st;
    CK(g, cudaMemcpyAsync(dev, host, need, cudaMemcpyHostToDevice, g->stream));
    CK(g, cudaStreamSynchronize(g->stream));
    return DIRAC_OK;
}

// The cell-field plan's per-entry V dt (host products V * dt, per x column or per cell as the potential was set) and
// absorber factors, refreshed whenever the potential, the absorber or the field changes.
dirac_status upload_field_aux(dirac_grid *g) {
    std::vector<double> vdt;
    if (g->v_layout != DIRAC_V_NONE) {
        vdt.resize(g->v_host.size());
        for (size_t e = 0; e < vdt.size(); ++e) vdt[e] = g->v_host[e] * g->dt;
    }
    dirac_status st = put_doubles(g, g->fvdt_dev, g->fvdt_bytes, vdt.data(), vdt.size());
    if (st != DIRAC_OK) return st;
    return put_doubles(g, g->fabs_dev, g->fabs_bytes, g->absorb.data(), g->absorb.size());
}

// Rows (or planes) per segment: the split of n rows that minimises a launch's time,
//   (rows + halo) x (full waves x row_time(resident) + row_time(the rest)),
// where each segment streams `halo` extra rows, `units` units of work per segment run `per_block` to a block, an SM
// holds `resident` blocks and row_time(b) is the time of one row with b blocks on an SM.  uneven: the part of a block
// that a launch loses at its end where its blocks differ (tiles cut by the grid's edge, the face's strip).
template <typename F>
int64_t pick_rows(int64_t n, int64_t units, int per_block, int64_t sms, int64_t resident, double halo, double uneven,
                  F row_time) {
    int64_t best_h = n;
    double best = 1e300;
    for (int64_t h = n; h >= 1;) {
        const int64_t segs = (n + h - 1) / h;
        const int64_t blocks = (units * segs + per_block - 1) / per_block;
        const int64_t per_sm = (blocks + sms - 1) / sms;  // on the fullest SM
        const int64_t waves = per_sm / resident, rest = per_sm % resident;
        const double t = ((double)h + halo) * (waves * row_time(resident) + (rest ? row_time(rest) : 0.0)) +
                         uneven * h * row_time(std::min(resident, per_sm));
        if (t < best * 0.999) {  // near ties: the longer segments
            best = t;
            best_h = h;
        }
        const int64_t next = (n + segs) / (segs + 1);  // the longest segment of one split more
        h = next < h ? next : h - 1;
    }
    return best_h;
}

// Time of one row of the 2-D step's row loop (microseconds) with w warps on an SM: a warp alone is bound by its chain
// of dependent instructions (lat), a full SM by the pipes (w x thr); in between the two add like independent delays.
// Fitted to measured launches (128^2 to 2048^2, segments of 1 to 64 rows); a fit within a quarter of the truth picks the
// segments, since the optimum is flat.  The launches of small grids were sized for few halo rows before (16 rows or
// more a segment): 256^2 FP64 42.5 us a step with 144 warps on the chip, 14.7 with 1152; FP32 13.6 -> 6.5.
struct RowTime {
    double lat, thr;
    double operator()(int64_t w) const { return std::sqrt(lat * lat + (w * thr) * (w * thr)); }
};
RowTime row_time_of(const dirac_grid *g, int K, int P) {
    const int mode = sweep_mode(g);
    const bool matrix = mode == 3 || mode == 5;
    // the second level of a second-order step has no phase (FP64: the phase is a third of the first's FP64 work)
    const double lv = strang(g) ? (g->fp32 || g->fx ? 1.5 : 2.0) * K : K;
    RowTime t = g->fx ? RowTime{1.03, 0.129} : (g->fp32 ? RowTime{0.5, 0.033} : RowTime{2.1, 0.31});
    // FP64, two points a lane: a row is one long chain whoever else runs (9.1 us a row of the second-order step with one block
    // on an SM, 11.5 with two), so a wave of short segments beats half a wave of long ones (1024^2 in a uniform field, second
    // order: 16 rows 292 us a step, 32 rows 381; 777 x 1000 11 rows 164, 22 rows 235)
    // (a shift step: 3.3 and 4.9)
    if (!g->fp32 && !g->fx && P == 2) t = mode == 4 ? RowTime{2.9, 0.24} : RowTime{5.0, 0.21};
    // (fixed point, four: 4.3 us a row; 1024^2 16 rows 98 us a step, 8 rows 74)
    if (g->fx && P == 4) t = RowTime{4.2, 0.116};
    t.lat *= lv * (matrix ? 1.4 : 1.0);
    t.thr *= lv * P * (matrix ? 1.7 : 1.0) * (!g->fp32 && !g->fx && P > 2 ? 1.4 : 1.0);
    return t;
}
// 4-warp blocks of the 2-D step resident on an SM (SweepMinBlocks; FP32 with one point a lane and one step fits five).
int resident_blocks(const dirac_grid *g, int K, int P) {
    if (sweep_mode(g) == 4) {
        // by their registers, [FP32][shift - 2][P - 1][field] (FP32 taken for four blocks, shift 4 at 2048^2 ran two waves of 32
        // rows, 77.5 us a step, where one of 64 takes 70.6)
        static const int blocks[2][3][2][2] = {{{{3, 3}, {2, 2}}, {{3, 2}, {2, 2}}, {{2, 2}, {2, 2}}},
                                               {{{4, 4}, {3, 2}}, {{4, 3}, {2, 2}}, {{3, 3}, {2, 2}}}};
        return blocks[g->fp32][char_shift(g) - 2][P - 1][field_on(g) ? 1 : 0];
    }
    if (P == 1) return g->fp32 && K == 1 ? 5 : 4;
    if (P == 4) return 2;
    return g->fp32 ? 4 : 2;
}

// Launch geometry for (K, P, warps per block): strips of 32P - 2K owned cells; segments for about `target` warps per
// SM, or, with target 0, by the row-time model above.
void make_plan(dirac_grid *g, int K, int P, int wpb, int target_warps_per_sm) {
    Plan &p = g->plan;
    p.tile = nullptr;
    p.K = K;
    p.P = P;
    p.wpb = wpb;
    const int64_t nx = g->cfg.n[0];
    const int64_t nr = (ndim_of(g) == 3) ? g->cfg.n[1] : g->cfg.n[2];
    const int64_t planes = (ndim_of(g) == 3) ? g->cfg.n[2] : 1;
    const int Lv = halo_of(g, K);
    p.strip_w = 32 * P - 2 * Lv;
    p.nstrips = (nx + p.strip_w - 1) / p.strip_w;
    const bool model = target_warps_per_sm == 0;
    const int64_t want = (int64_t)g->sm_count * (model ? 16 : target_warps_per_sm);
    if (model) {
        const RowTime rt = row_time_of(g, K, P);
        // a wave's blocks end apart: FP32 at 4096^2, k = 2, 165 G point-steps/s in one wave, 170-175 in two to four; at
        // 2048^2 145 in one, 130 in two; fixed point at 2048^2 33.7 in one, 32.8 in two; FP64 with two points a lane, second
        // order at 2048^2: 767 us a step in one wave of 61 rows, 805 in two of 30
        const double uneven = sweep_mode(g) == 4 ? 0.1 : (g->fp32 ? 0.2 : (!g->fx && P == 2 ? 0.0 : 0.1));
        p.seg_h = pick_rows(nr, p.nstrips * planes, wpb, g->sm_count, resident_blocks(g, K, P), 2.0 * Lv, uneven,
                            [&](int64_t blocks) { return rt(blocks * wpb); });
    } else {
        int64_t nsegs = std::max<int64_t>(1, want / std::max<int64_t>(1, p.nstrips * planes));
        // keep segments at least 8 levels' worth of rows so halo rows stay a small fraction
        const int64_t min_rows = std::max<int64_t>(8 * Lv, 16);
        nsegs = std::min<int64_t>(nsegs, std::max<int64_t>(1, nr / min_rows));
        p.seg_h = (nr + nsegs - 1) / nsegs;
    }
    p.seg_h = std::min(p.seg_h, kMaxSegRows);
    p.nsegs = (nr + p.seg_h - 1) / p.seg_h;
    // 3-D z pass: one thread per column, segments until ~target warps per SM
    if (ndim_of(g) == 3) {
        const int64_t ncol = g->cfg.n[0] * g->cfg.n[1];
        const int64_t nz = g->cfg.n[2];
        int64_t zs = std::max<int64_t>(1, want * 32 / std::max<int64_t>(1, ncol));
        zs = std::min<int64_t>(zs, std::max<int64_t>(1, nz / (ncol * nz < 32 * want * 32 ? 4 : 32)));  // small grids: short ones
        p.z_seg_h = (nz + zs - 1) / zs;
        p.z_nsegs = (nz + p.z_seg_h - 1) / p.z_seg_h;
        // fused pass: 30-cell strips x (warps - 2)-row tiles, z segments that fill whole waves (each carries two halo
        // planes and one plane's worth of start-up)
        p.f_nstrips = (g->cfg.n[0] + 29) / 30;
        p.f_nytiles = (g->cfg.n[1] + (p.f_warps - 2) - 1) / (p.f_warps - 2);
        const int64_t tiles = p.f_nstrips * p.f_nytiles;
        const auto whole = [](int64_t blocks) { return (double)blocks; };  // the passes: time as the blocks on an SM
        const int f_resident = !g->fp32 && p.f_warps == 8 ? 2 : 1;
        p.f_zseg_h = pick_rows(nz, tiles, 1, g->sm_count, f_resident, 3.0, 0.5, whole);
        p.f_nzsegs = (nz + p.f_zseg_h - 1) / p.f_zseg_h;
        // two steps per fused pass: 28-cell strips x (rows - 4)-row tiles, z segments as above (each carries two halo
        // planes a side).  FP32: 24 rows, two a warp, or 16, one a warp, where those fit a small grid better, whose planes take
        // 1.68 and 1.23 of the time (256^3: 219 us a step with 24, 271 with 16; 64^3 13.0 and 12.2); with the field's phase
        // matrices 16 rows; FP64 8 rows
        const bool two_rows = g->fp32 && !field_on(g);
        p.f2_nstrips = (g->cfg.n[0] + 27) / 28;
        double best = 1e300;
        for (int warps : {12, 16}) {
            if (!two_rows) warps = g->fp32 ? 16 : 8;
            const int64_t own = (warps == 12 ? 2 : 1) * warps - 4;
            const int64_t nytiles = (g->cfg.n[1] + own - 1) / own, tiles2 = p.f2_nstrips * nytiles;
            const int64_t h = pick_rows(nz, tiles2, 1, g->sm_count, 1, 5.0, 0.0, whole);
            const int64_t waves = (tiles2 * ((nz + h - 1) / h) + g->sm_count - 1) / g->sm_count;
            const double t = (warps == 12 ? 1.68 : 1.23) * (double)((h + 5) * waves);
            if (t < best) {
                best = t;
                p.f2_warps = warps;
                p.f2_nytiles = nytiles;
                p.f2_zseg_h = h;
            }
        }
        p.f2_nzsegs = (nz + p.f2_zseg_h - 1) / p.f2_zseg_h;
        // second-order passes: x-y-x(-x-y-x) blocks over (32 - 4 nh)-cell strips x (warps - 4 nh)-row tiles x
        // z segments (planes are independent; whole waves); z-phase-z columns x 2 plane parities
        // x z segments (~s3_zfactor x 1024 threads per SM, segments of at least 16 planes: four halo planes
        // each side)
        for (int nh = 1; nh <= 2; ++nh) {
            Plan::XY &q = p.s3_xy[nh - 1];
            const int own = 32 - 4 * nh, rows = p.s3_warps - 4 * nh;
            q.nstrips = (g->cfg.n[0] + own - 1) / own;
            q.nytiles = (g->cfg.n[1] + rows - 1) / rows;
            const int64_t tiles = q.nstrips * q.nytiles;
            q.zseg_h = pick_rows(nz, tiles, 1, g->sm_count, 1, 1.0, 0.5, whole);
            q.nzsegs = (nz + q.zseg_h - 1) / q.zseg_h;
        }
        int64_t zz = std::max<int64_t>(1, ((int64_t)p.s3_zfactor * 1024 * g->sm_count + ncol) / std::max<int64_t>(1, 2 * ncol));
        zz = std::min<int64_t>(zz, std::max<int64_t>(1, nz / (ncol * nz < 32 * 1024 * (int64_t)g->sm_count ? 8 : 16)));
        p.s3_z_seg_h = (nz + zz - 1) / zz;
        p.s3_z_nsegs = (nz + p.s3_z_seg_h - 1) / p.s3_z_seg_h;
    }
    drop_graphs(g);
}

int precision_index(const dirac_grid *g) { return g->fx ? 2 : (g->fp32 ? 1 : 0); }

// Launches of a tile shape's own step count (its remainders run with the same warps and rows).
void tile_plan(dirac_grid *g, const TileShape *t) {
    // the row kernel's (K, P) that a caller may ask for stands beside it, and is what dirac_get_info reports
    make_plan(g, t->steps, t->steps > 1 ? 2 : 1, 4, 0);
    g->plan.tile = t;
}

int64_t tiles_of(const dirac_grid *g, const TileShape &t) {
    const int H = levels(g, t.steps);
    const int64_t ox = 32 - 2 * H, oz = t.warps * t.rows - 2 * H;
    return ((g->cfg.n[0] + ox - 1) / ox) * ((g->cfg.n[2] + oz - 1) / oz);
}

// The tile shape for a 2-D grid, or null where the row kernel is faster: least modelled time a step.  The
// row kernel's time is taken as linear in its strips' cells (fitted from 128^2 to 4096^2), a launch of the tile kernel's as
// linear in the tiles on the fullest SM.  The lines cross, us a step with rows / tiles, at about: FP64 640^2 (512^2 30.2 /
// 28.4, 768^2 52.4 / 61), second order 900^2 (768^2 111 / 105, 1024^2 176 / 184), FP32 1900^2 (1024^2 9.5 / 6.0, 2048^2 21.2
// / 23), second order 1700^2 (1024^2 16.3 / 11.3, 1300^2 20.2 / 17), fixed point 768^2 (512^2 12.7 / 10.4, 1024^2 32.8 /
// 36.5), second order 700^2 (512^2 21.9 / 17.0, 768^2 32.3 / 35.4).
// With a uniform field (and an x-only table): FP64 350^2 (300^2 25.0 / 22.1, second order 45.8 / 33.6), FP32 1000^2 (300^2 6.6
// / 3.0), second order 1400^2 (300^2 10.9 / 5.1).
const TileShape *pick_tile(const dirac_grid *g) {
    const int mode = sweep_mode(g);
    const bool field = mode == 3 || mode == 5;
    if (ndim_of(g) != 2 || (mode != 0 && mode != 2 && !field) || g->inject_stall) return nullptr;
    if (g->cfg.n[0] >= (1 << 30) || g->cfg.n[2] >= (1 << 30)) return nullptr;  // the tile kernel's 32-bit coordinates
    static const double row[3][2][2] = {{{7.5, 7.8e-5}, {18.0, 1.5e-4}}, {{4.4, 4.0e-6}, {7.5, 7.0e-6}}, {{5.7, 2.67e-5}, {10.7, 3.9e-5}}};
    static const double frow[2][2][2] = {{{12.0, 1.31e-4}, {25.0, 2.1e-4}}, {{5.6, 8.2e-6}, {10.3, 1.25e-5}}};  // with a field
    const double *line = field ? frow[precision_index(g)][strang(g) ? 1 : 0] : row[precision_index(g)][strang(g) ? 1 : 0];
    const int64_t strip = g->fp32 ? 56 : 32 - 2 * levels(g, 1);
    double best = line[0] + line[1] * (double)((g->cfg.n[0] + strip - 1) / strip * strip * g->cfg.n[2]);
    const TileShape *pick = nullptr;
    int count = 0;
    const TileShape *t = tile_shapes(&count);
    for (; count > 0; --count, ++t) {
        if (!t->plan || t->precision != precision_index(g) || t->strang != (strang(g) ? 1 : 0) || t->field != (field ? 1 : 0)) continue;
        const int64_t per_sm = (tiles_of(g, *t) + g->sm_count - 1) / g->sm_count;
        const double us = (t->base + t->per_tile * (double)per_sm) / t->steps;
        if (us < best) {
            best = us;
            pick = t;
        }
    }
    return pick;
}

// Grid of the single-sweep kernels (grid-stride): up to 8 blocks of 256 threads per SM.
int axis_blocks(const dirac_grid *g) {
    const int64_t need = (g->ncells + 255) / 256;
    return (int)std::max<int64_t>(1, std::min<int64_t>(need, 8 * (int64_t)g->sm_count));
}

dirac_status ensure_flux_part(dirac_grid *g) {
    const int64_t planes = (ndim_of(g) == 3) ? g->cfg.n[2] : 1;
    size_t need = (size_t)8 * planes * std::max<int64_t>(g->plan.nsegs, 1);
    if (fused_pass(g)) {
        need = std::max(need, (size_t)(g->plan.f_nzsegs * g->plan.f_nytiles * g->plan.f_warps));
        if (g->plan.K == 2)
            need = std::max(need, (size_t)(2 * g->plan.f2_nzsegs * g->plan.f2_nytiles * g->plan.f2_warps));
    }
    if (g->plan.tile) need = std::max(need, (size_t)(levels(g, g->plan.K) * g->cfg.n[2]));
    if (sweep_mode(g) >= 6) need = std::max(need, (size_t)axis_blocks(g));
    if (strang3d_fused(g))
        for (int nh = 1; nh <= 2; ++nh) {
            const Plan::XY &q = g->plan.s3_xy[nh - 1];
            need = std::max(need, (size_t)(2 * nh * q.nzsegs * q.nytiles * g->plan.s3_warps));
        }
    // room for 32 launches between folds, within 4 MB (a launch that leaves more is folded by itself)
    need = std::max(need, std::min<size_t>(32 * need, (size_t)1 << 19));
    size_t bytes = g->flux_part_cap * sizeof(double);
    dirac_status st = grow(g, g->flux_part, bytes, need * sizeof(double));
    g->flux_part_cap = bytes / sizeof(double);
    return st;
}

// Folds what the launches since the last fold have left.
dirac_status fold_flux(dirac_grid *g, cudaStream_t s) {
    if (g->flux.count == 0) return DIRAC_OK;
    g->flux.part = g->flux_part;
    g->flux.flux_cum = g->flux_dev;
    g->flux.vol = cell_volume(g);
    cudaError_t e = launch_flux_fold(g->flux, s);
    g->flux.count = 0;
    g->flux_used = 0;
    if (e != cudaSuccess) return cuda_fail(g, e, "flux fold launch");
    g->launches++;
    return DIRAC_OK;
}

// A place for the flux partials of the next launch: `sums` sums (steps or x sweeps, in order) of n partials each.
dirac_status flux_place(dirac_grid *g, int sums, int64_t n, cudaStream_t s, double **part) {
    *part = g->flux_part;
    if (g->cfg.flux_face < 0) return DIRAC_OK;
    const size_t need = (size_t)sums * (size_t)n;
    if (g->flux.count + sums > kFluxEntries || g->flux_used + need > g->flux_part_cap) {
        dirac_status st = fold_flux(g, s);
        if (st != DIRAC_OK) return st;
    }
    if (need > g->flux_part_cap) return fail(g, DIRAC_ERR_STATE, "flux scratch too small");
    *part = g->flux_part + g->flux_used;
    for (int i = 0; i < sums; ++i) {
        g->flux.off[g->flux.count] = (unsigned)(g->flux_used + (size_t)i * n);
        g->flux.n[g->flux.count++] = (unsigned)n;
    }
    g->flux_used += need;
    return DIRAC_OK;
}

// Both state buffers lie on 32-byte boundaries (always, but for caller-owned ones).
int wide_state(const dirac_grid *g) {
    return ((reinterpret_cast<uintptr_t>(g->psi[0]) | reinterpret_cast<uintptr_t>(g->psi[1])) & 31u) == 0;
}

// One block of work: K steps (2-D) or one step (3-D), from psi[parity] to psi[parity ^ 1] (2-D) or back
// to psi[parity] (3-D).  Enqueued on s.  K_override > 0 runs that many steps with P from the plan.
dirac_status enqueue_block(dirac_grid *g, int parity, int K, cudaStream_t s, int64_t step0) {
    const Plan &p = g->plan;
    const bool flux = g->cfg.flux_face >= 0;
    const int64_t planes = (ndim_of(g) == 3) ? g->cfg.n[2] : 1;
    SweepArgs a{};
    a.in = g->psi[parity];
    a.out = g->psi[parity ^ 1];
    a.wide = wide_state(g);
    a.table = g->table;
    a.nx = g->cfg.n[0];
    a.nr = (ndim_of(g) == 3) ? g->cfg.n[1] : g->cfg.n[2];
    a.nplanes = planes;
    a.strip_w = 32 * p.P - 2 * halo_of(g, K);
    a.nstrips = (a.nx + a.strip_w - 1) / a.strip_w;
    a.nsegs = p.nsegs;
    a.seg_h = p.seg_h;
    a.flux_face = flux ? g->cfg.flux_face : -1;
    a.err = g->wait_err;
    a.periodic = g->cfg.boundary == DIRAC_BC_PERIODIC;
    a.full_table = g->table_full;
    a.ucoef = g->ucoef;
    a.ucoef_n = (int64_t)(g->avec.size() / 3);
    a.step0 = step0;
    a.inject_stall = g->inject_stall;
    a.flux_unit = g->fx ? std::ldexp(1.0, -2 * g->fx_shift) : 1.0;
    const int mode = sweep_mode(g);
    if (mode == 6) {
        // 3-D second-order step (Sec. 2.4): A(1) B(2) A(1) C(2) D C(2) A(1) B(2) A(1), cells moved per sweep in
        // parentheses.  Each sweep doubles the state and the table carries 1/256, so the state entering the
        // four x sweeps is 1, 4, 1/8 and 1/2 times the true state (flux scale 1/2 over its square).
        static const int axes[8] = {0, 1, 0, 2, 2, 0, 1, 0};
        static const double fscale[8] = {0.5, 0, 0.5 / 16.0, 0, 0, 0.5 * 64.0, 0, 0.5 * 4.0};
        // fixed point: the phase carries only the first four halves (1/16), so the state entering the last
        // two x sweeps is 2 and 8 times the true one, and the last sweep divides by 16 with rounding
        static const double fscale_fx[8] = {0.5, 0, 0.5 / 16.0, 0, 0, 0.5 / 4.0, 0, 0.5 / 64.0};
        const int blocks = axis_blocks(g);
        const int64_t K = char_shift(g);  // c dt / 4 = K dx: x sweeps move K cells, y and z sweeps 2 K
        const bool zpass = strang3d_zpass(g);
        int par = parity;
        for (int q = 0; q < 8; ++q) {
            const int ax = axes[q];
            if (zpass && q == 3) {
                // C D C in one pass: the same sums in the same order as sweeps 3 and 4, so the same bits
                cudaError_t e = launch_strang_z(g->psi[par], g->psi[par ^ 1], g->table, g->cfg.n[0], g->cfg.n[1],
                                                g->cfg.n[2], a.periodic, g->table_full, field_on(g) ? g->ucoef : nullptr,
                                                a.ucoef_n, step0, g->plan.s3_z_nsegs, g->plan.s3_z_seg_h,
                                                g->fx ? 2 : (g->fp32 ? 1 : 0), s);
                if (e != cudaSuccess) return cuda_fail(g, e, "3-D second-order z-phase-z pass launch");
                g->launches++;
                par ^= 1;
                ++q;  // sweep 4 is done too
                continue;
            }
            if (ax == 0) {
                dirac_status st = flux_place(g, 1, blocks, s, &a.flux_part);
                if (st != DIRAC_OK) return st;
            }
            cudaError_t e = launch_axis(g->psi[par], g->psi[par ^ 1], g->table, g->cfg.n[0], g->cfg.n[1], g->cfg.n[2], ax,
                                        ax == 0 ? K : 2 * K, a.periodic, g->table_full, q == 3 ? 1 : 0,
                                        ax == 0 ? a.flux_face : -1, (g->fx ? fscale_fx[q] : fscale[q]) * a.flux_unit,
                                        a.flux_part, q == 3 ? a.ucoef : nullptr,
                                        q == 3 ? a.ucoef_n : 0, step0,
                                        g->fx ? DIRAC_FX64 : (g->fp32 ? DIRAC_FP32 : DIRAC_FP64),
                                        (g->fx && q == 7) ? 4 : 0, blocks, s);
            if (e != cudaSuccess) return cuda_fail(g, e, "3-D second-order sweep launch");
            g->launches++;
            par ^= 1;
        }
        return DIRAC_OK;
    }
    if (mode == 8) {
        // a field varying in space and time as single-sweep launches: the sweeps of the grid's step form (shift K),
        // the phase epilogue of its z sweep forming U(At(i)) exp(-i V~(i)) per cell from the profiles and this step's
        // envelope integrals (Sec. 2.3, Eqs. sol_dis_4, field_dis1, field_dis2).  Each sweep doubles the state; the
        // phase carries the halves.  First order 2-D: x z+phase; 3-D: x y z+phase; second order 2-D: x z+phase z x;
        // 3-D: A B A C+phase C A B A (x moving K cells, y and z 2 K), flux scales as for the single-sweep plans.
        struct Sw {
            int axis, phase;
            double fscale;
        };
        static const Sw lie2[2] = {{0, 0, 0.5}, {2, 1, 0.0}};
        static const Sw lie3[3] = {{0, 0, 0.5}, {1, 0, 0.0}, {2, 1, 0.0}};
        static const Sw strang2[4] = {{0, 0, 0.5}, {2, 1, 0.0}, {2, 0, 0.0}, {0, 0, 2.0}};
        static const Sw strang3[8] = {{0, 0, 0.5},        {1, 0, 0.0}, {0, 0, 0.5 / 16.0}, {2, 1, 0.0},
                                      {2, 0, 0.0}, {0, 0, 0.5 * 64.0}, {1, 0, 0.0}, {0, 0, 0.5 * 4.0}};
        const bool s3 = strang(g) && ndim_of(g) == 3;
        const Sw *seq = strang(g) ? (s3 ? strang3 : strang2) : (ndim_of(g) == 3 ? lie3 : lie2);
        const int nseq = strang(g) ? (s3 ? 8 : 4) : (ndim_of(g) == 3 ? 3 : 2);
        const int64_t K = char_shift(g);
        const int64_t nrows = (int64_t)(g->fenv.size() / 4);
        const double *F = &g->fenv[4 * (size_t)(step0 % nrows)];
        const int blocks = axis_blocks(g);
        const int prec = g->fp32 ? DIRAC_FP32 : DIRAC_FP64;
        int par = parity;
        for (int q = 0; q < nseq; ++q) {
            const Sw &w = seq[q];
            const int64_t sh = (s3 && w.axis != 0) ? 2 * K : K;
            cudaError_t e;
            if (w.phase) {
                AxisArgs z{};
                z.in = g->psi[par];
                z.out = g->psi[par ^ 1];
                z.table = g->table;
                z.nx = g->cfg.n[0];
                z.ny = g->cfg.n[1];
                z.nz = g->cfg.n[2];
                z.shift = sh;
                z.periodic = a.periodic;
                z.flux_face = -1;
                z.fa = g->fa_dev;
                z.fw = g->fw_dev;
                z.fvdt = g->fvdt_dev;
                z.fvdt_full = g->v_layout == DIRAC_V_FULL;
                z.fabs = g->fabs_dev;
                for (int d = 0; d < 4; ++d) z.fenv[d] = F[d];
                z.fmu = g->cfg.m * g->cfg.c * g->cfg.c * g->dt;
                z.fscale_phase = scale_of(g);
                e = launch_axis_cellfield(z, prec, blocks, s);
            } else {
                if (w.axis == 0) {
                    dirac_status st = flux_place(g, 1, blocks, s, &a.flux_part);
                    if (st != DIRAC_OK) return st;
                }
                e = launch_axis(g->psi[par], g->psi[par ^ 1], g->table, g->cfg.n[0], g->cfg.n[1], g->cfg.n[2], w.axis,
                                sh, a.periodic, g->table_full, 0, w.axis == 0 ? a.flux_face : -1, w.fscale,
                                a.flux_part, nullptr, 0, step0, prec, 0, blocks, s);
            }
            if (e != cudaSuccess) return cuda_fail(g, e, "cell-field sweep launch");
            g->launches++;
            par ^= 1;
        }
        return DIRAC_OK;
    }
    if (mode == 7) {
        // characteristic shift K > 1 as single-sweep launches (Sec. 2.3: c dt = K dx per sweep), each sweep doubling
        // the state and the table carrying the halves: 3-D first order x(K) y(K) z(K)+phase over dt = K dx / c, the
        // state entering the x sweep at its true size (flux scale 1/2); 2-D second order x(K) z(K)+phase z(K) x(K)
        // over dt = 2 K dx / c, the state entering the second x sweep at half its true size (flux scale 2)
        struct Sw {
            int axis, phase;
            double fscale;
        };
        static const Sw lie3[3] = {{0, 0, 0.5}, {1, 0, 0.0}, {2, 1, 0.0}};
        static const Sw strang2[4] = {{0, 0, 0.5}, {2, 1, 0.0}, {2, 0, 0.0}, {0, 0, 2.0}};
        const Sw *seq = ndim_of(g) == 3 ? lie3 : strang2;
        const int nseq = ndim_of(g) == 3 ? 3 : 4;
        const int blocks = axis_blocks(g);
        int par = parity;
        for (int q = 0; q < nseq; ++q) {
            const Sw &w = seq[q];
            if (w.axis == 0) {
                dirac_status st = flux_place(g, 1, blocks, s, &a.flux_part);
                if (st != DIRAC_OK) return st;
            }
            cudaError_t e = launch_axis(g->psi[par], g->psi[par ^ 1], g->table, g->cfg.n[0], g->cfg.n[1], g->cfg.n[2],
                                        w.axis, char_shift(g), a.periodic, g->table_full, w.phase,
                                        w.axis == 0 ? a.flux_face : -1, w.fscale, a.flux_part,
                                        w.phase ? a.ucoef : nullptr, w.phase ? a.ucoef_n : 0, step0,
                                        g->fp32 ? DIRAC_FP32 : DIRAC_FP64, 0, blocks, s);
            if (e != cudaSuccess) return cuda_fail(g, e, "characteristic-shift sweep launch");
            g->launches++;
            par ^= 1;
        }
        return DIRAC_OK;
    }
    if (mode == 1 && fused_pass(g)) {
        cudaError_t e;
        a.nplanes = 1;
        if (K == 2) {
            a.nsegs = p.f2_nzsegs * p.f2_nytiles * p.f2_warps;  // flux parts per step of the fused pass
            dirac_status st = flux_place(g, 2, a.nsegs, s, &a.flux_part);
            if (st != DIRAC_OK) return st;
            e = launch_fused3d(a, g->fx ? 2 : g->fp32, p.f2_warps, 2, g->cfg.n[1], g->cfg.n[2], p.f2_nstrips, p.f2_nytiles,
                               p.f2_nzsegs, p.f2_zseg_h, s);
        } else {
            a.nsegs = p.f_nzsegs * p.f_nytiles * p.f_warps;  // flux parts of the fused pass
            dirac_status st = flux_place(g, 1, a.nsegs, s, &a.flux_part);
            if (st != DIRAC_OK) return st;
            e = launch_fused3d(a, g->fx ? 2 : g->fp32, p.f_warps, 1, g->cfg.n[1], g->cfg.n[2], p.f_nstrips, p.f_nytiles,
                               p.f_nzsegs, p.f_zseg_h, s);
        }
        if (e != cudaSuccess) return cuda_fail(g, e, "fused 3-D step launch");
        g->launches++;
        return DIRAC_OK;
    }
    if (p.tile && !(p.tile->field && g->table_full)) {  // (a field over a full table: the row kernel of the same K)
        a.strip_w = 32 - 2 * levels(g, K);
        a.nstrips = (a.nx + a.strip_w - 1) / a.strip_w;
        dirac_status st = flux_place(g, levels(g, K), a.nr, s, &a.flux_part);
        if (st != DIRAC_OK) return st;
        cudaError_t e = launch_tile(a, *p.tile, K, g->sm_count, s);
        if (e != cudaSuccess) return cuda_fail(g, e, "tile kernel launch");
        g->launches++;
        return DIRAC_OK;
    }
    dirac_status st = flux_place(g, mode == 4 ? 1 : levels(g, K), a.nsegs * planes, s, &a.flux_part);
    if (st != DIRAC_OK) return st;
    cudaError_t e = mode == 4 ? launch_shift(a, g->fp32, char_shift(g), p.P, p.wpb, s)
                    : g->fx   ? launch_sweep_fx(a, mode, K, p.P, p.wpb, s)
                    : g->fp32 ? launch_sweep_f32(a, mode, K, p.P, p.wpb, s)
                              : launch_sweep_f64(a, mode, K, p.P, p.wpb, s);
    if (e != cudaSuccess) return cuda_fail(g, e, "sweep kernel launch");
    g->launches++;
    if (ndim_of(g) == 3) {
        ZArgs z{};
        z.in = g->psi[parity ^ 1];
        z.out = g->psi[parity];
        z.table = g->table;
        z.nx = g->cfg.n[0];
        z.ny = g->cfg.n[1];
        z.nz = g->cfg.n[2];
        z.nsegs = p.z_nsegs;
        z.seg_h = p.z_seg_h;
        z.periodic = a.periodic;
        z.full_table = g->table_full;
        e = g->fx ? launch_zphase_fx(z, p.z_threads, s)
            : g->fp32 ? launch_zphase_f32(z, p.z_threads, s) : launch_zphase_f64(z, p.z_threads, s);
        if (e != cudaSuccess) return cuda_fail(g, e, "z-phase kernel launch");
        g->launches++;
    }
    return DIRAC_OK;
}

// A run of m >= 1 second-order 3-D steps as fused passes (Sec. 2.4): x-y-x, then m z-phase-z passes
// separated by m - 1 x-y-x-x-y-x passes, then x-y-x; 2m + 1 launches from psi[parity], ending in
// psi[parity ^ 1].  Each sweep doubles the state and the table carries 1/256, so the states entering a step's
// four x sweeps are 1, 4, 1/8 and 1/2 times the true state (flux scale 1/2 over its square).
dirac_status enqueue_strang3d_run(dirac_grid *g, int parity, int64_t m, cudaStream_t s, int64_t step0) {
    const Plan &p = g->plan;
    const bool flux = g->cfg.flux_face >= 0;
    const int64_t ny = g->cfg.n[1], nz = g->cfg.n[2];
    static const double first_half[4] = {0.5, 0.5 / 16.0, 0.0, 0.0};
    static const double second_half[4] = {0.5 * 64.0, 0.5 * 4.0, 0.0, 0.0};
    static const double both_halves[4] = {0.5 * 64.0, 0.5 * 4.0, 0.5, 0.5 / 16.0};
    // fixed point: the phase carries the first four halves (1/16), so the states entering a step's x sweeps are
    // 1, 4, 2 and 8 times the true state and the step's last x sweep is followed by the division by 16
    static const double first_half_fx[4] = {0.5, 0.5 / 16.0, 0.0, 0.0};
    static const double second_half_fx[4] = {0.5 / 4.0, 0.5 / 64.0, 0.0, 0.0};
    static const double both_halves_fx[4] = {0.5 / 4.0, 0.5 / 64.0, 0.5, 0.5 / 16.0};
    const int prec = g->fx ? 2 : g->fp32;
    const double funit = g->fx ? std::ldexp(1.0, -2 * g->fx_shift) : 1.0;
    SweepArgs a{};
    a.table = g->table;
    a.nx = g->cfg.n[0];
    a.nplanes = 1;
    a.flux_face = flux ? g->cfg.flux_face : -1;
    a.err = g->wait_err;
    a.periodic = g->cfg.boundary == DIRAC_BC_PERIODIC;
    const double *ucoef = field_on(g) ? g->ucoef : nullptr;
    const int64_t ucoef_n = (int64_t)(g->avec.size() / 3);
    int par = parity;
    // ends_step: the pass's last sweep ends a step (fixed point: divide by 16 there)
    auto xy = [&](int nh, const double *fs, bool ends_step) -> dirac_status {
        const Plan::XY &q = p.s3_xy[nh - 1];
        a.in = g->psi[par];
        a.out = g->psi[par ^ 1];
        a.wide = wide_state(g);
        a.nsegs = q.nzsegs * q.nytiles * p.s3_warps;  // flux parts per x sweep
        dirac_status st = flux_place(g, 2 * nh, a.nsegs, s, &a.flux_part);
        if (st != DIRAC_OK) return st;
        double fsu[4];
        for (int i = 0; i < 4; ++i) fsu[i] = fs[i] * funit;
        const int rmid = (g->fx && nh == 2) ? 4 : 0, rend = (g->fx && ends_step) ? 4 : 0;
        cudaError_t e = launch_strang_xy(a, prec, p.s3_warps, nh, ny, nz, q.nstrips, q.nytiles, q.nzsegs, q.zseg_h,
                                         fsu, rmid, rend, s);
        if (e != cudaSuccess) return cuda_fail(g, e, "3-D second-order x-y-x pass launch");
        g->launches++;
        par ^= 1;
        return DIRAC_OK;
    };
    dirac_status st = xy(1, g->fx ? first_half_fx : first_half, false);
    for (int64_t i = 0; i < m && st == DIRAC_OK; ++i) {
        cudaError_t e = launch_strang_z(g->psi[par], g->psi[par ^ 1], g->table, a.nx, ny, nz, a.periodic, g->table_full,
                                        ucoef, ucoef_n, step0 + i, p.s3_z_nsegs, p.s3_z_seg_h, prec, s);
        if (e != cudaSuccess) return cuda_fail(g, e, "3-D second-order z-phase-z pass launch");
        g->launches++;
        par ^= 1;
        const bool last = i + 1 == m;
        st = xy(last ? 1 : 2, last ? (g->fx ? second_half_fx : second_half) : (g->fx ? both_halves_fx : both_halves), last);
    }
    return st;
}

int block_flips(const dirac_grid *g) {
    if (sweep_mode(g) == 6)  // eight sweeps per step: parity returns; seven with the z-phase-z pass: it flips
        return strang3d_zpass(g) ? 1 : 0;  // (fused runs: enqueue_strang3d_run)
    if (sweep_mode(g) == 7) return ndim_of(g) == 3 ? 1 : 0;  // three or four single sweeps
    if (sweep_mode(g) == 8) return (ndim_of(g) == 3 && !strang(g)) ? 1 : 0;  // two, three, four or eight sweeps
    return (ndim_of(g) == 3 && !fused_pass(g)) ? 0 : 1;
}

dirac_status get_graph(dirac_grid *g, int parity, cudaGraphExec_t *out) {
    if (g->graph[parity]) {
        *out = g->graph[parity];
        return DIRAC_OK;
    }
    CK(g, cudaStreamBeginCapture(g->cap_stream, cudaStreamCaptureModeRelaxed));
    int par = parity;
    const int64_t l0 = g->launches;
    dirac_status st = DIRAC_OK;
    if (strang3d_fused(g)) {
        st = enqueue_strang3d_run(g, par, kGraphBlocks, g->cap_stream, 0);
    } else {
        for (int b = 0; b < kGraphBlocks && st == DIRAC_OK; ++b) {
            st = enqueue_block(g, par, g->plan.K, g->cap_stream, 0);
            par ^= block_flips(g);
        }
    }
    if (st == DIRAC_OK) st = fold_flux(g, g->cap_stream);
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamEndCapture(g->cap_stream, &graph);
    g->graph_launches[parity] = g->launches - l0;
    g->launches = l0;  // captured, not launched
    if (st != DIRAC_OK) {
        if (graph) cudaGraphDestroy(graph);
        return st;
    }
    if (e != cudaSuccess) return cuda_fail(g, e, "cudaStreamEndCapture");
    cudaGraphExec_t exec = nullptr;
    e = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) return cuda_fail(g, e, "cudaGraphInstantiate");
    g->graph[parity] = exec;
    *out = exec;
    return DIRAC_OK;
}

dirac_status run_steps(dirac_grid *g, int64_t nsteps) {
    g->flux.count = 0;  // nothing is left over but by a call that failed
    g->flux_used = 0;
    const int K = (ndim_of(g) == 3) ? (fused_pass(g) ? g->plan.K : 1) : g->plan.K;
    int64_t blocks = nsteps / K;
    int64_t rem = nsteps % K;
    const bool field = field_on(g) || cellfield_on(g);
    if (field_on(g) && !g->tuning && g->step + nsteps > (int64_t)(g->avec.size() / 3))
        return fail(g, DIRAC_ERR_ARG, "the vector-potential table ends before step " + std::to_string(g->step + nsteps));
    if (cellfield_on(g) && !g->tuning && g->step + nsteps > (int64_t)(g->fenv.size() / 4))
        return fail(g, DIRAC_ERR_ARG, "the field's table ends before step " + std::to_string(g->step + nsteps));
    int64_t t = g->step;  // step index of the next launch (selects the field's table row)
    if (strang3d_fused(g)) {
        // runs of kGraphBlocks steps from the captured graph (2 kGraphBlocks + 1 launches, parity flips), then
        // the rest as one run
        int64_t left = nsteps;
        if (g->cfg.use_graphs && !field)
            while (left >= kGraphBlocks) {
                cudaGraphExec_t ex = nullptr;
                dirac_status st = get_graph(g, g->cur, &ex);
                if (st != DIRAC_OK) return st;
                CK(g, cudaGraphLaunch(ex, g->stream));
                g->launches += g->graph_launches[g->cur];
                g->cur ^= 1;
                left -= kGraphBlocks;
                t += kGraphBlocks;
            }
        if (left > 0) {
            dirac_status st = enqueue_strang3d_run(g, g->cur, left, g->stream, t);
            if (st != DIRAC_OK) return st;
            g->cur ^= 1;
        }
        g->step += nsteps;
        return fold_flux(g, g->stream);
    }
    // launches with a field take their step index as an argument: no graph replay
    if (g->cfg.use_graphs && !field && blocks >= kGraphBlocks) {
        while (blocks >= kGraphBlocks) {
            cudaGraphExec_t ex = nullptr;
            dirac_status st = get_graph(g, g->cur, &ex);
            if (st != DIRAC_OK) return st;
            CK(g, cudaGraphLaunch(ex, g->stream));
            g->launches += g->graph_launches[g->cur];
            blocks -= kGraphBlocks;
            // kGraphBlocks is even: parity unchanged
        }
    }
    for (int64_t b = 0; b < blocks; ++b) {
        dirac_status st = enqueue_block(g, g->cur, K, g->stream, t);
        if (st != DIRAC_OK) return st;
        g->cur ^= block_flips(g);
        t += K;
    }
    while (rem > 0) {
        // the tile kernel and the FP32 one of four steps have launches of two and one besides
        const int kk = rem >= 2 && K == 4 ? 2 : 1;
        dirac_status st = enqueue_block(g, g->cur, kk, g->stream, t);
        if (st != DIRAC_OK) return st;
        g->cur ^= block_flips(g);
        t += kk;
        rem -= kk;
    }
    g->step += nsteps;
    return fold_flux(g, g->stream);
}

void release(dirac_grid *g) {
    if (!g) return;
    if (g->stream || g->cap_stream) cudaStreamSynchronize(g->stream);
    drop_graphs(g);
    if (!g->ext)
        for (auto &p : g->psi)
            if (p) cudaFree(p);
    if (g->table) cudaFree(g->table);
    if (g->ucoef) cudaFree(g->ucoef);
    for (double *p : {g->fa_dev, g->fw_dev, g->fvdt_dev, g->fabs_dev})
        if (p) cudaFree(p);
    if (g->flux_part) cudaFree(g->flux_part);
    if (g->flux_dev) cudaFree(g->flux_dev);
    if (g->wait_err) cudaFree(g->wait_err);
    if (g->obs_partial) cudaFree(g->obs_partial);
    if (g->obs_out) cudaFree(g->obs_out);
    if (g->density_tmp) cudaFree(g->density_tmp);
    if (g->host_obs) cudaFreeHost(g->host_obs);
    if (g->cap_stream) cudaStreamDestroy(g->cap_stream);
    delete g;
}

void set_fx_shift(dirac_grid *g, int shift) {
    if (g->fx_shift != shift) drop_graphs(g);
    g->fx_shift = shift;
}

// DIRAC_FX64 state in: the complex128 state is copied to the idle ping-pong buffer, its discrete L2 norm A
// (square root of the sum of |psi_c|^2 over all cells and components) reduced there, the shift chosen as
// S = 60 - e in 2-D, 59 - e in 3-D, with A = m 2^e, m in [0.5, 1): each sweep (with its 1/2) and the phase
// do not raise the discrete norm, so after j of the step's sweeps (without the 1/2) a component is at most
// 2^j A, and every sum of a step stays below 2^62 (the two-component sums below 2^62.5); and the state
// encoded as q = round(psi 2^S) into the current buffer.
dirac_status fx_load_state(dirac_grid *g, const void *psi, int on_device) {
    const size_t bytes = (size_t)g->ncells * 8 * g->elem;
    double *tmp = static_cast<double *>(g->psi[g->cur ^ 1]);
    if (!(on_device && psi == tmp))
        CK(g, cudaMemcpyAsync(tmp, psi, bytes, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, g->stream));
    ObsArgs o{};
    o.psi = tmp;
    o.scale = 1.0;
    o.nx = g->cfg.n[0];
    o.ny = g->cfg.n[1];
    o.nz = g->cfg.n[2];
    o.dx = g->cfg.dx;
    o.face = -1;
    o.partial = g->obs_partial;
    o.out = g->obs_out;
    CK(g, launch_observables(o, DIRAC_FP64, g->obs_blocks, g->stream));
    CK(g, cudaMemcpyAsync(g->host_obs, g->obs_out, sizeof(double), cudaMemcpyDeviceToHost, g->stream));
    CK(g, cudaStreamSynchronize(g->stream));
    const double sumsq = g->host_obs[0];
    if (!std::isfinite(sumsq)) return fail(g, DIRAC_ERR_NONFINITE, "dirac_set_state: state holds NaN or Inf");
    int e = 0;
    if (sumsq > 0) std::frexp(std::sqrt(sumsq), &e);
    set_fx_shift(g, (ndim_of(g) == 3 ? (strang(g) ? 57 : 59) : 60) - e);
    CK(g, launch_fx_encode(tmp, static_cast<long long *>(g->psi[g->cur]), g->ncells * 8, g->fx_shift, g->stream));
    return DIRAC_OK;
}

void default_plan(dirac_grid *g) {
    const int k = g->cfg.steps_per_launch, pp = g->cfg.points_per_lane;
    if (sweep_mode(g) >= 7) {  // single-sweep launches, one step per block
        g->plan.fused3d = 0;
        g->plan.s3_fused = 0;
        g->plan.s3_zpass = 0;
        make_plan(g, 1, 1, 4, 8);
        return;
    }
    if (ndim_of(g) == 3 && g->fx) {
        // fixed point, first order: points_per_lane 0 = the fused single pass (one step per pass), 1, 2 or 4 =
        // the x-y pass + z/phase pass with that P; second order: points_per_lane 1 = eight single sweeps, 0 or 2 =
        // the fused passes (bandwidth-bound integer sweeps: the passes move a seventh of the single sweeps' bytes),
        // 4 = single x and y sweeps with one z-phase-z pass
        // (64^3 and 96^3 the two passes with P = 1 are faster, 32.0 and 61 us a step against 40.3 and 74; the autotuner finds
        // them)
        g->plan.fused3d = pp > 0 ? 0 : 1;
        g->plan.f_warps = 8;  // two blocks an SM (fused3d_kernels.cuh)
        g->plan.s3_fused = (strang(g) && pp != 1 && pp != 4) ? 1 : 0;
        g->plan.s3_zpass = (strang(g) && pp == 4) ? 1 : 0;
        g->plan.s3_warps = 32;  // measured at 384^3: 12.5 G point-steps/s against 10.5 with 16-warp blocks (fewer
                                // recomputed halo rows outweigh the int64 x-y-x-x-y-x pass's small spill at 64 registers)
        make_plan(g, 1, pp > 0 ? pp : 1, 4, 16);
        return;
    }
    if (ndim_of(g) == 3) {
        // points_per_lane 0: the fused single-pass step; 1, 2 or 4: the x-y pass + z/phase pass with that P.  FP64, bound by
        // its pipe, recomputes no halo rows in the two passes, whose one point a lane splits its sums over both pipes: the
        // library's choice from about 60^3 (64^3 60.5 us a step against 74.3 fused, 256^3 1798 against 2217, 384^3 5999
        // against 6956)
        const bool two64 = !g->fp32 && !strang(g) && !field_on(g) && k == 0 && pp == 0 && g->ncells > 200000;
        g->plan.fused3d = pp > 0 || two64 ? 0 : 1;
        // FP64: 8-warp blocks, two on an SM (fused3d_kernels.cuh); FP32: 16, short y extents 8 (6-row tiles waste fewer
        // halo rows)
        g->plan.f_warps = !g->fp32 || g->cfg.n[1] <= 12 ? 8 : 16;
        // second-order step: points_per_lane 1 = eight single-sweep launches, 2 = the three fused passes, 4 = x and
        // y single sweeps with one z-phase-z pass, 0 = library choice (fused passes for FP32 storage, which is
        // bandwidth-bound; for FP64, which is bound by the FP64 pipe and would recompute the x-y-x pass's halo
        // cells, single x and y sweeps with the z-phase-z pass: 3.06 against 2.95 G point-steps/s at 384^3)
        g->plan.s3_fused = (pp == 1 || pp == 4) ? 0 : (pp == 2 ? 1 : (g->fp32 ? 1 : 0));
        g->plan.s3_zpass = (pp == 4 || (pp == 0 && !g->fp32)) ? 1 : 0;
        g->plan.s3_warps = 32;  // measured at 384^3: 24 owned rows of 32 beat 8 of 16 (more recomputed halo rows)
        // first-order fused pass: steps_per_launch 1 or 2 (temporal block); library choice two in FP32
        // storage (bandwidth-bound), one in FP64 (bound by the FP64 pipe: the second step's halo would cost)
        int K3 = 1;
        if (!strang(g) && (pp == 0 || field_on(g))) K3 = k == 2 ? 2 : (k == 1 ? 1 : (g->fp32 ? 2 : 1));
        // FP64 two-pass plan: 32 warps an SM of segments (8.75 against 8.2 G at 256^3 with 16)
        make_plan(g, K3, pp > 0 ? pp : (two64 ? 1 : 2), 4, g->fp32 ? 16 : 32);
        return;
    }
    if (sweep_mode(g) == 4) {
        // FP64, K = 2, no field: one point a lane and 24 warps an SM of segments, whose sweeps fill the FP64 and the
        // integer pipe (9.4 against 8.7 G point-steps/s at 2048^2); elsewhere two (with the field's phase matrix
        // 4.5 against 4.2 G)
        const bool one = !g->fp32 && char_shift(g) == 2 && !field_on(g);
        const int P = pp == 1 || pp == 2 ? pp : (one ? 1 : 2);
        make_plan(g, 1, P, 4, 0);
        return;
    }
    const int mode = sweep_mode(g);
    if (k == 0 && pp == 0) {
        if (const TileShape *t = pick_tile(g)) {
            tile_plan(g, t);
            return;
        }
    }
    if (g->fx) {
        // one cell per lane (128 registers: four blocks per SM) and enough segments to fill them
        int K = k > 0 ? k : 1, P = pp > 0 ? pp : 1;
        if (!sweep_supported_fx(mode, K, P)) {
            K = 1;
            P = 1;
        }
        make_plan(g, K, P, 4, 0);
        return;
    }
    // FP64: one point a lane, 16 warps an SM (four blocks of 128 registers): the sweeps' pairs split over the FP64 and
    // the integer pipe need warps to overlap (2048^2: 13.9 against 10.8 G with two points and 8 warps; second order
    // 7.1 against 5.5; in a laser field 7.7 against 6.6)
    // FP32: four steps a launch (2048^2 20.8 us a step against 25.1 with two, 4096^2 70.6 against 87.2, where two move twice
    // the bytes)
    int K = g->fp32 ? (pp == 0 || pp == 2 ? 4 : 2) : 1, P = g->fp32 ? 2 : 1;
    // with a field FP32 first order two (2048^2 43.9 us a step against 61.0 with one, 1000 x 777 12.0 and 17.0, 300^2 6.8 and
    // 9.0; the kernels of four would not fit the registers), else one
    if (mode == 3 || mode == 5) K = mode == 3 && g->fp32 && (pp == 0 || pp == 2) ? 2 : 1;
    if (mode == 2) K = g->fp32 ? 2 : 1;  // FP32 second order: two steps per pass with the history in shared memory
    if (k > 0) K = k;
    if (mode == 0 && g->fp32 && K == 1) P = 1;  // one step a launch: 84.9 against 76.8 G at 2048^2
    if (pp > 0) P = pp;
    if (!sweep_supported(g->fp32, mode, K, P)) P = sweep_supported(g->fp32, mode, K, 4) ? 4 : 2;
    if (!sweep_supported(g->fp32, mode, K, P)) {
        K = 1;
        P = 2;
    }
    make_plan(g, K, P, 4, 0);
}

}  // namespace

namespace dirac {
// FP32 representation of (cos t, -sin t): among the float neighbours of the rounded values, the pair
// whose squared modulus is closest to 1 (keeps the FP32 phase step unitary to ~1e-9 instead of ~1e-7).
void round_unitary(double c, double s, float &cf, float &sf) {
    const float c0 = (float)c, s0 = (float)s;
    const float cs[3] = {nextafterf(c0, -2.f), c0, nextafterf(c0, 2.f)};
    const float ss[3] = {nextafterf(s0, -2.f), s0, nextafterf(s0, 2.f)};
    double best = 1e300;
    cf = c0;
    sf = s0;
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) {
            const double dc = cs[i], ds = ss[j];
            const double err = std::fabs(dc * dc + ds * ds - 1.0);
            const double dist = std::fabs(dc - c) + std::fabs(ds - s);
            const double key = err + 1e-3 * dist;
            if (key < best) {
                best = key;
                cf = cs[i];
                sf = ss[j];
            }
        }
}

// Phase coefficients of Eq. sol_dis_4 at A = 0 for potential energy v, pre-scaled by 2^-d:
// components 1,2: exp(-i (m c^2 dt + v dt)), components 3,4: exp(-i (v dt - m c^2 dt)).
void phase_coeffs(double mu, double v, double dt, double scale, double out[4]) {
    const double vdt = v * dt;
    const double t_up = mu + vdt;
    const double t_dn = vdt - mu;
    out[0] = std::cos(t_up) * scale;
    out[1] = -std::sin(t_up) * scale;
    out[2] = std::cos(t_dn) * scale;
    out[3] = -std::sin(t_dn) * scale;
}


void phase_coeffs_masked(double mu, double v, double dt, double a, double scale, double out[4]) {
    const double vdt = v * dt;
    const double t_up = mu + vdt;
    const double t_dn = vdt - mu;
    out[0] = std::cos(t_up) * a * scale;
    out[1] = -std::sin(t_up) * a * scale;
    out[2] = std::cos(t_dn) * a * scale;
    out[3] = -std::sin(t_dn) * a * scale;
}

void u_entries(double mu, const double At[3], double out[12]) {
    const double A = std::sqrt(((mu * mu + At[0] * At[0]) + At[1] * At[1]) + At[2] * At[2]);
    const double sA = A > 0.0 ? std::sin(A) / A : 1.0;
    const double cA = std::cos(A);
    const double ax = At[0] * sA, ay = At[1] * sA, az = At[2] * sA, ms = mu * sA;
    const double e[12] = {cA, -ms,  cA, ms,     // Dup (components 1,2), Ddn (3,4)
                          0.0, az,  0.0, -az,   // Ez = i At_z s/A, -Ez
                          ay, ax,   -ay, ax};   // Ep = (i At_x + At_y) s/A, Em = (i At_x - At_y) s/A
    for (int i = 0; i < 12; ++i) out[i] = e[i];
}

// Records a message for dirac_last_error(NULL) on this thread (entry points without a grid).
dirac_status set_thread_error(dirac_status st, const std::string &msg) {
    g_thread_err = msg;
    return st;
}
}  // namespace dirac

extern "C" {

const char *dirac_version(void) { return "dirac-gb300 0.1 (sm_103a)"; }

void dirac_default_config(dirac_config *cfg) {
    if (!cfg) return;
    std::memset(cfg, 0, sizeof(*cfg));
    cfg->ndim = 2;
    cfg->n[0] = 256;
    cfg->n[1] = 1;
    cfg->n[2] = 256;
    cfg->dx = 10.0 / 8192.0;
    cfg->c = 137.0359895;
    cfg->m = 1.0;
    cfg->x_min[0] = -128 * cfg->dx;
    cfg->x_min[1] = 0.0;
    cfg->x_min[2] = -128 * cfg->dx;
    cfg->precision = DIRAC_FP64;
    cfg->boundary = DIRAC_BC_ZERO;
    cfg->flux_face = -1;
    cfg->stream = nullptr;
    cfg->device = 0;
    cfg->steps_per_launch = 0;
    cfg->use_graphs = 1;
    cfg->points_per_lane = 0;
    cfg->splitting = DIRAC_LIE;
}

const char *dirac_last_error(const dirac_grid *g) { return g ? g->err.c_str() : g_thread_err.c_str(); }

dirac_status dirac_create_grid(const dirac_config *cfg, dirac_grid **out) {
    if (!cfg || !out) return fail(nullptr, DIRAC_ERR_ARG, "dirac_create_grid: null argument");
    *out = nullptr;
    if (cfg->ndim != 2 && cfg->ndim != 3) return fail(nullptr, DIRAC_ERR_ARG, "ndim must be 2 or 3");
    for (int d = 0; d < 3; ++d)
        if (cfg->n[d] < 1 || cfg->n[d] > 0x7fffffff)
            return fail(nullptr, DIRAC_ERR_ARG, "grid sizes must be >= 1 and below 2^31");
    if (cfg->ndim == 2 && cfg->n[1] != 1) return fail(nullptr, DIRAC_ERR_ARG, "2-D grids (x-z plane) need n[1] == 1");
    if (!(cfg->dx > 0) || !(cfg->c > 0) || !std::isfinite(cfg->dx) || !std::isfinite(cfg->c) || !std::isfinite(cfg->m))
        return fail(nullptr, DIRAC_ERR_ARG, "dx and c must be finite and > 0, m finite");
    if (cfg->precision != DIRAC_FP64 && cfg->precision != DIRAC_FP32 && cfg->precision != DIRAC_FX64)
        return fail(nullptr, DIRAC_ERR_ARG, "precision must be DIRAC_FP64, DIRAC_FP32 or DIRAC_FX64");
    if (cfg->precision == DIRAC_FX64) {
        if (cfg->char_shift > 1)
            return fail(nullptr, DIRAC_ERR_ARG, "DIRAC_FX64 runs characteristic shift 1 (char_shift 0 or 1)");
        if (cfg->ndim == 3 && cfg->splitting == DIRAC_STRANG && (cfg->points_per_lane == 3 || cfg->points_per_lane > 4))
            return fail(nullptr, DIRAC_ERR_ARG,
                        "DIRAC_FX64 3-D second-order steps run as single sweeps (points_per_lane 1), single sweeps with "
                        "a z-phase-z pass (4) or fused passes (0, 2)");
        const int fmode = cfg->ndim == 3 ? 1 : (cfg->splitting == DIRAC_STRANG ? 2 : 0);
        const bool strang3 = cfg->ndim == 3 && cfg->splitting == DIRAC_STRANG;
        if (cfg->steps_per_launch > 2 || ((cfg->ndim == 3 || fmode == 2) && cfg->steps_per_launch > 1) ||
            (!strang3 && cfg->steps_per_launch > 0 && cfg->points_per_lane > 0 &&
             !sweep_supported_fx(fmode, cfg->steps_per_launch, cfg->points_per_lane)) ||
            (cfg->steps_per_launch == 2 && cfg->points_per_lane > 0 && cfg->points_per_lane != 2))
            return fail(nullptr, DIRAC_ERR_ARG,
                        "DIRAC_FX64 runs steps_per_launch 1 (points_per_lane 1, 2, 4) or, in 2-D, 2 (2)");
    }
    if (cfg->boundary != DIRAC_BC_ZERO && cfg->boundary != DIRAC_BC_PERIODIC)
        return fail(nullptr, DIRAC_ERR_ARG, "boundary must be DIRAC_BC_ZERO or DIRAC_BC_PERIODIC");
    if (cfg->flux_face != -1 && (cfg->flux_face < 1 || cfg->flux_face > cfg->n[0] - 1))
        return fail(nullptr, DIRAC_ERR_ARG, "flux_face must be -1 or in [1, nx-1]");
    const double ncells_d = (double)cfg->n[0] * (double)cfg->n[1] * (double)cfg->n[2];
    if (ncells_d > 4.0e10) return fail(nullptr, DIRAC_ERR_ARG, "grid too large");
    if (cfg->splitting != DIRAC_LIE && cfg->splitting != DIRAC_STRANG)
        return fail(nullptr, DIRAC_ERR_ARG, "splitting must be DIRAC_LIE or DIRAC_STRANG");
    if (cfg->splitting == DIRAC_STRANG && cfg->ndim == 3 && cfg->steps_per_launch > 1)
        return fail(nullptr, DIRAC_ERR_ARG, "3-D DIRAC_STRANG runs one step per launch block (steps_per_launch 0 or 1)");
    if (cfg->ndim == 3 && cfg->steps_per_launch > 2)
        return fail(nullptr, DIRAC_ERR_ARG, "3-D grids run 1 or 2 steps per launch");
    if (cfg->ndim == 3 && cfg->steps_per_launch == 2 && cfg->points_per_lane > 0)
        return fail(nullptr, DIRAC_ERR_ARG, "3-D steps_per_launch 2 runs the fused pass (points_per_lane 0)");
    if (cfg->char_shift < 0 || cfg->char_shift > 4)
        return fail(nullptr, DIRAC_ERR_ARG, "char_shift must be 0 (= 1), 1, 2, 3 or 4");
    if (cfg->char_shift > 1) {
        if (cfg->boundary == DIRAC_BC_PERIODIC && cfg->flux_face >= 0 &&
            (cfg->flux_face < cfg->char_shift || cfg->flux_face > cfg->n[0] - cfg->char_shift))
            return fail(nullptr, DIRAC_ERR_ARG,
                        "periodic grids with char_shift K > 1 take a flux_face in [K, nx-K] (the K cells on each "
                        "side of the face inside the grid)");
        if (cfg->steps_per_launch > 1)
            return fail(nullptr, DIRAC_ERR_ARG, "char_shift > 1 runs one step per launch (steps_per_launch 0 or 1)");
        if (cfg->ndim == 2 && cfg->splitting == DIRAC_LIE && cfg->points_per_lane == 4)
            return fail(nullptr, DIRAC_ERR_ARG, "2-D char_shift > 1 needs points_per_lane 0, 1 or 2");
        if ((cfg->ndim == 3 || cfg->splitting == DIRAC_STRANG) && cfg->points_per_lane > 1)
            return fail(nullptr, DIRAC_ERR_ARG,
                        "3-D or second-order steps with char_shift > 1 run as single sweeps (points_per_lane 0 or 1)");
    }
    const int vmode = cfg->splitting == DIRAC_STRANG ? 2 : 0;
    if (cfg->precision != DIRAC_FX64 && cfg->steps_per_launch != 0 && cfg->char_shift <= 1 &&
        !(sweep_supported(cfg->precision == DIRAC_FP32, vmode, cfg->steps_per_launch, 2) ||
          sweep_supported(cfg->precision == DIRAC_FP32, vmode, cfg->steps_per_launch, 4)))
        return fail(nullptr, DIRAC_ERR_ARG, "unsupported steps_per_launch for this precision and splitting");
    if (cfg->points_per_lane != 0 && cfg->points_per_lane != 1 && cfg->points_per_lane != 2 &&
        cfg->points_per_lane != 4)
        return fail(nullptr, DIRAC_ERR_ARG, "points_per_lane must be 0, 1, 2 or 4");
    if (cfg->precision != DIRAC_FX64 && cfg->ndim == 2 && cfg->char_shift <= 1 && cfg->steps_per_launch > 0 &&
        cfg->points_per_lane > 0 &&
        !sweep_supported(cfg->precision == DIRAC_FP32, vmode, cfg->steps_per_launch, cfg->points_per_lane))
        return fail(nullptr, DIRAC_ERR_ARG, "unsupported (steps_per_launch, points_per_lane) pair");
    const bool ext0 = cfg->ext_state[0] != nullptr, ext1 = cfg->ext_state[1] != nullptr;
    if (ext0 != ext1) return fail(nullptr, DIRAC_ERR_ARG, "ext_state needs both buffers or neither");
    if (std::getenv("DIRAC_INJECT_OOM")) return fail(nullptr, DIRAC_ERR_OOM, "allocation failure injected (DIRAC_INJECT_OOM)");

    dirac_grid *g = new (std::nothrow) dirac_grid();
    if (!g) return fail(nullptr, DIRAC_ERR_OOM, "host allocation failed");
    g->cfg = *cfg;
    g->inject_stall = std::getenv("DIRAC_INJECT_STALL") ? 1 : 0;
    g->stream = static_cast<cudaStream_t>(cfg->stream);
    g->fp32 = cfg->precision == DIRAC_FP32;
    g->fx = cfg->precision == DIRAC_FX64;
    g->elem = g->fp32 ? 4 : 8;
    g->ncells = cfg->n[0] * cfg->n[1] * cfg->n[2];
    // dt: c dt = K dx per first-order step (Sec. 2.3); a second-order step spans two (2-D) or four (3-D) of them
    g->dt = (cfg->splitting == DIRAC_STRANG ? (cfg->ndim == 3 ? 4.0 : 2.0) : 1.0) *
            (double)(cfg->char_shift > 1 ? cfg->char_shift : 1) * cfg->dx / cfg->c;
    cudaError_t e = cudaSetDevice(cfg->device);
    if (e != cudaSuccess) {
        std::string msg = std::string("cudaSetDevice: ") + cudaGetErrorString(e);
        release(g);
        return fail(nullptr, DIRAC_ERR_CUDA, msg);
    }
    cudaDeviceGetAttribute(&g->sm_count, cudaDevAttrMultiProcessorCount, cfg->device);
    if (g->sm_count <= 0) g->sm_count = 152;
    const size_t state_bytes = (size_t)g->ncells * 8 * g->elem;
    if (ext0) {
        // caller-owned ping-pong buffers: device memory of cfg->device, 16-byte aligned (vector loads and bulk
        // copies), at least one state apart
        for (int i = 0; i < 2; ++i) {
            cudaPointerAttributes at{};
            e = cudaPointerGetAttributes(&at, cfg->ext_state[i]);
            if (e != cudaSuccess) cudaGetLastError();
            const bool dev_mem = e == cudaSuccess &&
                                 (at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged) &&
                                 at.device == cfg->device;
            if (!dev_mem || (reinterpret_cast<uintptr_t>(cfg->ext_state[i]) & 15u)) {
                release(g);
                return fail(nullptr, DIRAC_ERR_ARG,
                            "ext_state[" + std::to_string(i) + "] is not 16-byte aligned device memory of cfg.device");
            }
        }
        const uintptr_t a0 = reinterpret_cast<uintptr_t>(cfg->ext_state[0]);
        const uintptr_t a1 = reinterpret_cast<uintptr_t>(cfg->ext_state[1]);
        if ((a0 > a1 ? a0 - a1 : a1 - a0) < state_bytes) {
            release(g);
            return fail(nullptr, DIRAC_ERR_ARG, "ext_state buffers overlap (closer than one state's size)");
        }
        g->psi[0] = cfg->ext_state[0];
        g->psi[1] = cfg->ext_state[1];
        g->ext = true;
    }
    struct {
        void **p;
        size_t bytes;
    } allocs[] = {{&g->psi[0], state_bytes}, {&g->psi[1], state_bytes}, {(void **)&g->flux_dev, 8 * sizeof(double)},
                  {(void **)&g->wait_err, 16},
                  {(void **)&g->obs_partial, (size_t)kObsBlocksMax * 5 * sizeof(double)},
                  {(void **)&g->obs_out, 8 * sizeof(double)}};
    for (auto &al : allocs) {
        if (g->ext && (al.p == &g->psi[0] || al.p == &g->psi[1])) continue;
        e = cudaMalloc(al.p, al.bytes);
        if (e != cudaSuccess) {
            std::string msg = std::string("cudaMalloc(") + std::to_string(al.bytes) + " bytes): " + cudaGetErrorString(e);
            cudaGetLastError();
            release(g);
            return fail(nullptr, e == cudaErrorMemoryAllocation ? DIRAC_ERR_OOM : DIRAC_ERR_CUDA, msg);
        }
        g->device_bytes += al.bytes;
    }
    e = cudaMallocHost(&g->host_obs, 8 * sizeof(double));
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&g->cap_stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
        std::string msg = std::string("setup: ") + cudaGetErrorString(e);
        release(g);
        return fail(nullptr, DIRAC_ERR_CUDA, msg);
    }
    g->obs_blocks = (int)std::min<int64_t>(kObsBlocksMax, std::max<int64_t>(1, (g->ncells + 255) / 256));
    default_plan(g);
    dirac_status st = ensure_flux_part(g);
    if (st == DIRAC_OK) st = upload_table(g, nullptr, DIRAC_V_NONE, 0);
    if (st == DIRAC_OK) {
        e = g->ext ? cudaSuccess : cudaMemsetAsync(g->psi[0], 0, state_bytes, g->stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(g->flux_dev, 0, 8 * sizeof(double), g->stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(g->wait_err, 0, 16, g->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
        if (e != cudaSuccess) st = cuda_fail(g, e, "initial clear");
    }
    if (st != DIRAC_OK) {
        std::string msg = g->err;
        release(g);
        return fail(nullptr, st, msg);
    }
    *out = g;
    return DIRAC_OK;
}

dirac_status dirac_destroy(dirac_grid *g) {
    if (!g) return DIRAC_OK;
    cudaSetDevice(g->cfg.device);
    release(g);
    return DIRAC_OK;
}

dirac_status dirac_set_potential(dirac_grid *g, const double *V, int layout, int64_t count) {
    if (!g) return fail(nullptr, DIRAC_ERR_ARG, "null grid");
    CK(g, cudaSetDevice(g->cfg.device));
    if (layout == DIRAC_V_NONE) {
        g->v_host.clear();
        g->v_layout = DIRAC_V_NONE;
        return upload_table(g, nullptr, layout, 0);
    }
    if (!V) return fail(g, DIRAC_ERR_ARG, "dirac_set_potential: null V");
    if (layout == DIRAC_V_X_ONLY) {
        if (count != g->cfg.n[0]) return fail(g, DIRAC_ERR_ARG, "DIRAC_V_X_ONLY needs count == nx");
    } else if (layout == DIRAC_V_FULL) {
        if (count != g->ncells) return fail(g, DIRAC_ERR_ARG, "DIRAC_V_FULL needs count == nx*ny*nz");
    } else {
        return fail(g, DIRAC_ERR_ARG, "unknown potential layout");
    }
    for (int64_t i = 0; i < count; ++i)
        if (!std::isfinite(V[i])) return fail(g, DIRAC_ERR_ARG, "potential holds a non-finite value");
    std::vector<double> before(V, V + count);
    before.swap(g->v_host);
    std::swap(g->v_layout, layout);
    dirac_status st = upload_table(g, V, g->v_layout, count);
    if (st != DIRAC_OK) {  // the potential that the table holds still
        g->v_host.swap(before);
        g->v_layout = layout;
    }
    return st;
}

dirac_status dirac_set_absorber(dirac_grid *g, const double *a, int64_t count) {
    if (!g) return fail(nullptr, DIRAC_ERR_ARG, "null grid");
    CK(g, cudaSetDevice(g->cfg.device));
    if (!a || count == 0) {
        g->absorb.clear();
    } else {
        if (count != g->cfg.n[0]) return fail(g, DIRAC_ERR_ARG, "dirac_set_absorber needs count == nx");
        for (int64_t i = 0; i < count; ++i)
            if (!(a[i] > 0.0 && a[i] <= 1.0)) return fail(g, DIRAC_ERR_ARG, "absorber factors must lie in (0, 1]");
        g->absorb.assign(a, a + count);
    }
    const bool have_v = g->v_layout != DIRAC_V_NONE && !g->v_host.empty();
    return upload_table(g, have_v ? g->v_host.data() : nullptr, have_v ? g->v_layout : DIRAC_V_NONE,
                        have_v ? (int64_t)g->v_host.size() : 0);
}

dirac_status dirac_set_vector_potential(dirac_grid *g, const double *A_tilde, int64_t nsteps_table) {
    if (!g) return fail(nullptr, DIRAC_ERR_ARG, "null grid");
    if (g->fx && A_tilde && nsteps_table > 0)
        return fail(g, DIRAC_ERR_ARG, "DIRAC_FX64 grids take no vector potential");
    if (nsteps_table < 0) return fail(g, DIRAC_ERR_ARG, "nsteps_table must be >= 0");
    const bool clear = !A_tilde || nsteps_table == 0;
    if (!clear && cellfield_on(g))
        return fail(g, DIRAC_ERR_STATE, "a field varying in space is set (dirac_set_field): remove it first");
    if (!clear)
        for (int64_t i = 0; i < 3 * nsteps_table; ++i)
            if (!std::isfinite(A_tilde[i])) return fail(g, DIRAC_ERR_ARG, "vector-potential table holds a non-finite value");
    CK(g, cudaSetDevice(g->cfg.device));
    const std::vector<double> before = g->avec;
    if (clear) {
        g->avec.clear();
    } else {
        const size_t bytes = (size_t)nsteps_table * 12 * sizeof(double);
        dirac_status st = grow(g, g->ucoef, g->ucoef_cap, bytes);
        if (st != DIRAC_OK) return st;
        const double mu = g->cfg.m * g->cfg.c * g->cfg.c * g->dt;
        std::vector<double> h((size_t)nsteps_table * 12);
        for (int64_t n = 0; n < nsteps_table; ++n) u_entries(mu, A_tilde + 3 * n, &h[(size_t)n * 12]);
        CK(g, cudaMemcpyAsync(g->ucoef, h.data(), bytes, cudaMemcpyHostToDevice, g->stream));
        CK(g, cudaStreamSynchronize(g->stream));
        g->avec.assign(A_tilde, A_tilde + 3 * nsteps_table);
    }
    if (field_on(g) == before.empty()) {
        default_plan(g);
        dirac_status st = ensure_flux_part(g);
        if (st != DIRAC_OK) {
            g->avec = before;
            default_plan(g);
            return st;
        }
        const bool have_v = g->v_layout != DIRAC_V_NONE && !g->v_host.empty();
        return upload_table(g, have_v ? g->v_host.data() : nullptr, have_v ? g->v_layout : DIRAC_V_NONE,
                            have_v ? (int64_t)g->v_host.size() : 0);
    }
    return DIRAC_OK;
}

dirac_status dirac_set_field(dirac_grid *g, const double *a, const double *w, const double *F, int64_t nsteps_table) {
    if (!g) return fail(nullptr, DIRAC_ERR_ARG, "null grid");
    if (nsteps_table < 0) return fail(g, DIRAC_ERR_ARG, "nsteps_table must be >= 0");
    const bool clear = !F || nsteps_table == 0;
    if (!clear && g->fx) return fail(g, DIRAC_ERR_ARG, "DIRAC_FX64 grids take no field");
    if (!clear && field_on(g))
        return fail(g, DIRAC_ERR_STATE, "a uniform vector potential is set (dirac_set_vector_potential): remove it first");
    if (!clear) {
        for (int64_t i = 0; i < 4 * nsteps_table; ++i)
            if (!std::isfinite(F[i])) return fail(g, DIRAC_ERR_ARG, "the field's table holds a non-finite value");
        if (a)
            for (int64_t i = 0; i < 3 * g->ncells; ++i)
                if (!std::isfinite(a[i])) return fail(g, DIRAC_ERR_ARG, "the profile a holds a non-finite value");
        if (w)
            for (int64_t i = 0; i < g->ncells; ++i)
                if (!std::isfinite(w[i])) return fail(g, DIRAC_ERR_ARG, "the profile w holds a non-finite value");
    }
    CK(g, cudaSetDevice(g->cfg.device));
    dirac_status st = DIRAC_OK;
    if (clear) {
        g->fenv.clear();
        st = put_doubles(g, g->fa_dev, g->fa_bytes, nullptr, 0);
        if (st == DIRAC_OK) st = put_doubles(g, g->fw_dev, g->fw_bytes, nullptr, 0);
        if (st == DIRAC_OK) st = put_doubles(g, g->fvdt_dev, g->fvdt_bytes, nullptr, 0);
        if (st == DIRAC_OK) st = put_doubles(g, g->fabs_dev, g->fabs_bytes, nullptr, 0);
    } else {
        st = put_doubles(g, g->fa_dev, g->fa_bytes, a, a ? (size_t)(3 * g->ncells) : 0);
        if (st == DIRAC_OK) st = put_doubles(g, g->fw_dev, g->fw_bytes, w, w ? (size_t)g->ncells : 0);
        if (st == DIRAC_OK) g->fenv.assign(F, F + 4 * nsteps_table);
        if (st == DIRAC_OK) st = upload_field_aux(g);
    }
    if (st != DIRAC_OK) return st;
    drop_graphs(g);
    default_plan(g);
    return ensure_flux_part(g);
}

dirac_status dirac_set_state(dirac_grid *g, const void *psi, int on_device) {
    if (!g) return fail(nullptr, DIRAC_ERR_ARG, "null grid");
    if (!psi) return fail(g, DIRAC_ERR_ARG, "dirac_set_state: null psi");
    CK(g, cudaSetDevice(g->cfg.device));
    const size_t bytes = (size_t)g->ncells * 8 * g->elem;
    if (g->fx) {
        dirac_status st = fx_load_state(g, psi, on_device);
        if (st != DIRAC_OK) return st;
    } else if (!(on_device && psi == g->psi[g->cur])) {  // a caller-owned buffer may already hold the state
        CK(g, cudaMemcpyAsync(g->psi[g->cur], psi, bytes, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                              g->stream));
    }
    CK(g, cudaMemsetAsync(g->flux_dev, 0, sizeof(double), g->stream));
    CK(g, cudaMemsetAsync(g->wait_err, 0, sizeof(unsigned), g->stream));  // clear a reported timeout
    if (!on_device) CK(g, cudaStreamSynchronize(g->stream));
    g->step = 0;
    return DIRAC_OK;
}

dirac_status dirac_get_state(dirac_grid *g, void *psi, int on_device) {
    if (!g) return fail(nullptr, DIRAC_ERR_ARG, "null grid");
    if (!psi) return fail(g, DIRAC_ERR_ARG, "dirac_get_state: null psi");
    CK(g, cudaSetDevice(g->cfg.device));
    const size_t bytes = (size_t)g->ncells * 8 * g->elem;
    const void *src = g->psi[g->cur];
    if (g->fx) {
        // decoded into the idle ping-pong buffer, then copied out as complex128
        CK(g, launch_fx_decode(static_cast<const long long *>(g->psi[g->cur]), static_cast<double *>(g->psi[g->cur ^ 1]),
                               g->ncells * 8, g->fx_shift, g->stream));
        src = g->psi[g->cur ^ 1];
    }
    CK(g, cudaMemcpyAsync(psi, src, bytes, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, g->stream));
    if (!on_device) CK(g, cudaStreamSynchronize(g->stream));
    return DIRAC_OK;
}

dirac_status dirac_set_state_fx(dirac_grid *g, const int64_t *q, int shift, int on_device) {
    if (!g) return fail(nullptr, DIRAC_ERR_ARG, "null grid");
    if (!g->fx) return fail(g, DIRAC_ERR_ARG, "dirac_set_state_fx needs a DIRAC_FX64 grid");
    if (!q) return fail(g, DIRAC_ERR_ARG, "dirac_set_state_fx: null q");
    if (shift < -1000 || shift > 1000) return fail(g, DIRAC_ERR_ARG, "dirac_set_state_fx: shift out of range");
    CK(g, cudaSetDevice(g->cfg.device));
    const size_t bytes = (size_t)g->ncells * 8 * sizeof(int64_t);
    if (!(on_device && q == g->psi[g->cur]))
        CK(g, cudaMemcpyAsync(g->psi[g->cur], q, bytes, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                              g->stream));
    CK(g, cudaMemsetAsync(g->flux_dev, 0, sizeof(double), g->stream));
    CK(g, cudaMemsetAsync(g->wait_err, 0, sizeof(unsigned), g->stream));
    if (!on_device) CK(g, cudaStreamSynchronize(g->stream));
    set_fx_shift(g, shift);
    g->step = 0;
    return DIRAC_OK;
}

dirac_status dirac_get_state_fx(dirac_grid *g, int64_t *q, int *shift, int on_device) {
    if (!g) return fail(nullptr, DIRAC_ERR_ARG, "null grid");
    if (!g->fx) return fail(g, DIRAC_ERR_ARG, "dirac_get_state_fx needs a DIRAC_FX64 grid");
    if (!q) return fail(g, DIRAC_ERR_ARG, "dirac_get_state_fx: null q");
    CK(g, cudaSetDevice(g->cfg.device));
    const size_t bytes = (size_t)g->ncells * 8 * sizeof(int64_t);
    CK(g, cudaMemcpyAsync(q, g->psi[g->cur], bytes, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                          g->stream));
    if (!on_device) CK(g, cudaStreamSynchronize(g->stream));
    if (shift) *shift = g->fx_shift;
    return DIRAC_OK;
}

dirac_status dirac_state_ptr(dirac_grid *g, void **dev_ptr) {
    if (!g || !dev_ptr) return fail(g, DIRAC_ERR_ARG, "null argument");
    *dev_ptr = g->psi[g->cur];
    return DIRAC_OK;
}

dirac_status dirac_step(dirac_grid *g, int64_t nsteps) {
    if (!g) return fail(nullptr, DIRAC_ERR_ARG, "null grid");
    if (nsteps < 0) return fail(g, DIRAC_ERR_ARG, "nsteps must be >= 0");
    if (nsteps == 0) return DIRAC_OK;
    CK(g, cudaSetDevice(g->cfg.device));
    return run_steps(g, nsteps);
}

dirac_status dirac_set_counters(dirac_grid *g, int64_t step, double flux_cum) {
    if (!g) return fail(nullptr, DIRAC_ERR_ARG, "null grid");
    if (step < 0 || !std::isfinite(flux_cum)) return fail(g, DIRAC_ERR_ARG, "bad counters");
    CK(g, cudaSetDevice(g->cfg.device));
    g->host_obs[7] = flux_cum;
    CK(g, cudaMemcpyAsync(g->flux_dev, &g->host_obs[7], sizeof(double), cudaMemcpyHostToDevice, g->stream));
    CK(g, cudaStreamSynchronize(g->stream));
    g->step = step;
    return DIRAC_OK;
}

dirac_status dirac_observables(dirac_grid *g, dirac_obs *obs, double *density, int density_on_device) {
    if (!g || !obs) return fail(g, DIRAC_ERR_ARG, "null argument");
    CK(g, cudaSetDevice(g->cfg.device));
    double *dens = nullptr;
    if (density) {
        if (density_on_device) {
            dens = density;
        } else {
            if (!g->density_tmp) {
                CK(g, cudaMalloc(&g->density_tmp, (size_t)g->ncells * sizeof(double)));
                g->device_bytes += (size_t)g->ncells * sizeof(double);
            }
            dens = g->density_tmp;
        }
    }
    ObsArgs a{};
    a.psi = g->psi[g->cur];
    a.scale = g->fx ? std::ldexp(1.0, -g->fx_shift) : 1.0;
    a.nx = g->cfg.n[0];
    a.ny = g->cfg.n[1];
    a.nz = g->cfg.n[2];
    a.dx = g->cfg.dx;
    a.x0 = g->cfg.x_min[0] + 0.5 * g->cfg.dx;
    a.y0 = g->cfg.x_min[1] + 0.5 * g->cfg.dx;
    a.z0 = g->cfg.x_min[2] + 0.5 * g->cfg.dx;
    a.face = g->cfg.flux_face;
    a.density = dens;
    a.partial = g->obs_partial;
    a.out = g->obs_out;
    cudaError_t e = launch_observables(a, g->fx ? DIRAC_FX64 : (g->fp32 ? DIRAC_FP32 : DIRAC_FP64), g->obs_blocks, g->stream);
    if (e != cudaSuccess) return cuda_fail(g, e, "observables launch");
    g->launches += 2;
    CK(g, cudaMemcpyAsync(g->host_obs, g->obs_out, 5 * sizeof(double), cudaMemcpyDeviceToHost, g->stream));
    CK(g, cudaMemcpyAsync(&g->host_obs[5], g->flux_dev, sizeof(double), cudaMemcpyDeviceToHost, g->stream));
    CK(g, cudaMemcpyAsync(&g->host_obs[6], g->wait_err, sizeof(unsigned), cudaMemcpyDeviceToHost, g->stream));
    if (density && !density_on_device)
        CK(g, cudaMemcpyAsync(density, dens, (size_t)g->ncells * sizeof(double), cudaMemcpyDeviceToHost, g->stream));
    CK(g, cudaStreamSynchronize(g->stream));
    const double vol = cell_volume(g);
    const double *h = g->host_obs;
    obs->norm = h[0] * vol;
    obs->norm_right = h[1] * vol;
    obs->flux_cum = h[5];
    obs->centroid[0] = h[0] > 0 ? h[2] / h[0] : 0.0;
    obs->centroid[1] = h[0] > 0 ? h[3] / h[0] : 0.0;
    obs->centroid[2] = h[0] > 0 ? h[4] / h[0] : 0.0;
    obs->step = g->step;
    unsigned kerr = 0;
    std::memcpy(&kerr, &g->host_obs[6], sizeof(unsigned));
    if (kerr) return fail(g, DIRAC_ERR_TIMEOUT, "a step kernel's bounded wait for a row copy ran out; the state is invalid");
    if (!std::isfinite(obs->norm)) return fail(g, DIRAC_ERR_NONFINITE, "state holds NaN or Inf");
    return DIRAC_OK;
}

dirac_status dirac_get_info(const dirac_grid *g, dirac_info *info) {
    if (!g || !info) return fail(nullptr, DIRAC_ERR_ARG, "null argument");
    const Plan &p = g->plan;
    info->steps_per_launch = (g->cfg.ndim == 3) ? (fused_pass(g) ? p.K : 1) : p.K;
    info->points_per_lane = p.P;
    const int64_t planes = (g->cfg.ndim == 3) ? g->cfg.n[2] : 1;
    info->launch_warps = p.nstrips * p.nsegs * planes;
    info->strip_width = p.strip_w;
    info->segment_rows = p.seg_h;
    static const int plan_of_mode[9] = {DIRAC_PLAN_STEP_2D, DIRAC_PLAN_3D_TWO_PASS, DIRAC_PLAN_STRANG_2D,
                                        DIRAC_PLAN_FIELD_2D, DIRAC_PLAN_SHIFT_2D, DIRAC_PLAN_STRANG_FIELD_2D,
                                        DIRAC_PLAN_3D_STRANG, DIRAC_PLAN_SHIFT_SWEEPS, DIRAC_PLAN_FIELD_SWEEPS};
    const int mode = sweep_mode(g);
    info->plan = (mode == 1 && fused_pass(g)) ? DIRAC_PLAN_3D_FUSED : plan_of_mode[mode];
    if (strang3d_zpass(g)) info->plan = DIRAC_PLAN_3D_STRANG_ZPASS;
    if (strang3d_fused(g)) {
        info->plan = DIRAC_PLAN_3D_STRANG_FUSED;
        info->points_per_lane = 1;
        const Plan::XY &q = p.s3_xy[1];
        info->launch_warps = q.nstrips * q.nytiles * q.nzsegs * p.s3_warps;
        info->strip_width = 24;
        info->segment_rows = q.zseg_h;
    }
    if (p.tile && !(p.tile->field && g->table_full)) {
        info->launch_warps = tiles_of(g, *p.tile) * p.tile->warps;
        info->strip_width = 32 - 2 * levels(g, p.K);
        info->segment_rows = p.tile->warps * p.tile->rows - 2 * levels(g, p.K);
    }
    if (fused_pass(g)) {
        info->points_per_lane = 1;
        info->launch_warps = p.f_nstrips * p.f_nytiles * p.f_nzsegs * p.f_warps;
        info->strip_width = 30;
        info->segment_rows = p.f_zseg_h;
        if (p.K == 2) {
            info->launch_warps = p.f2_nstrips * p.f2_nytiles * p.f2_nzsegs * p.f2_warps;
            info->strip_width = 28;
            info->segment_rows = p.f2_zseg_h;
        }
    }
    info->graphs = g->cfg.use_graphs;
    info->fx_shift = g->fx ? g->fx_shift : 0;
    info->state_index = g->cur;
    info->kernel_launches = g->launches;
    info->device_bytes = g->device_bytes;
    return DIRAC_OK;
}

dirac_status dirac_autotune(dirac_grid *g) {
    if (!g) return fail(nullptr, DIRAC_ERR_ARG, "null grid");
    CK(g, cudaSetDevice(g->cfg.device));
    struct Cand {
        int K, P, wpb, wsm;
        int fused = 0;  // 3-D: warps per block of the fused pass (0: two-pass path)
        int s3 = 0;     // 3-D second order: 0 = eight single sweeps, else warps per block of the x-y-x pass
        int s3z = 2;    // and the z-phase-z pass's threads per SM / 1024
        int s3zp = 0;   // 3-D second order, single sweeps: C D C as one z-phase-z pass
        const TileShape *tile = nullptr;  // 2-D: the tile kernel in this shape
    };
    std::vector<Cand> cands;
    if (sweep_mode(g) >= 7) {
        cands.push_back({1, 1, 4, 8, 0, 0});  // single sweeps: nothing to choose
    } else if (sweep_mode(g) == 6) {
        cands.push_back({1, 2, 4, 16, 0, 0});
        if (char_shift(g) == 1) {  // the fused passes take one-cell x shifts
            for (int sw : {16, 32})
                for (int zf : {1, 2, 4}) cands.push_back({1, 2, 4, 16, 0, sw, zf});
            for (int zf : {1, 2, 4}) cands.push_back({1, 2, 4, 16, 0, 0, zf, 1});
        }
    } else if (g->fx && g->cfg.ndim == 3) {
        for (int P : {1, 2, 4})
            for (int wsm : {8, 16, 32}) cands.push_back({1, P, 4, wsm, 0});
        for (int fw : {8, 16}) cands.push_back({1, 1, 4, 16, fw});  // the fused single pass
    } else if (g->fx) {
        const int KP[][2] = {{1, 1}, {1, 2}, {1, 4}, {2, 2}};
        for (auto &kp : KP)
            if (sweep_supported_fx(sweep_mode(g), kp[0], kp[1]))
                for (int wsm : {0, 8, 12, 16, 24}) cands.push_back({kp[0], kp[1], 4, wsm});
    } else if (g->cfg.ndim == 3) {
        if (!field_on(g))  // with a vector potential only the fused pass applies the phase matrix
            for (int P : {1, 2, 4})
                for (int wsm : {8, 16, 32}) cands.push_back({1, P, 4, wsm, 0});
        for (int fw : {8, 16}) cands.push_back({1, 2, 4, 16, fw});
        cands.push_back({2, 2, 4, 16, 16});  // two steps per fused pass
    } else if (sweep_mode(g) == 4) {
        for (int P : {1, 2})
            for (int wsm : {0, 4, 8, 12, 16, 24}) cands.push_back({1, P, 4, wsm});
    } else if (sweep_mode(g) == 3 || sweep_mode(g) == 5) {
        const int KP[][2] = {{1, 1}, {1, 2}, {2, 2}};
        for (auto &kp : KP)
            if (sweep_supported(g->fp32, sweep_mode(g), kp[0], kp[1]))
                for (int wsm : {0, 4, 8, 12, 16}) cands.push_back({kp[0], kp[1], 4, wsm});
    } else if (strang(g)) {
        const int KP[][2] = {{1, 1}, {1, 2}, {1, 4}, {2, 2}};
        for (auto &kp : KP)
            if (sweep_supported(g->fp32, 2, kp[0], kp[1]))
                for (int wsm : {0, 4, 8, 12, 16}) cands.push_back({kp[0], kp[1], 4, wsm});
    } else if (g->fp32) {
        const int KP[][2] = {{1, 2}, {1, 4}, {2, 2}, {2, 4}, {4, 2}};
        for (auto &kp : KP)
            for (int wsm : {0, 8, 12, 16}) cands.push_back({kp[0], kp[1], 4, wsm});
    } else {
        const int KP[][2] = {{1, 1}, {1, 2}, {2, 2}};
        for (auto &kp : KP)
            for (int wsm : {0, 8, 12, 16, 24}) cands.push_back({kp[0], kp[1], 4, wsm});
    }
    if (pick_tile(g)) {  // small 2-D grids
        int count = 0;
        const TileShape *t = tile_shapes(&count);
        for (; count > 0; --count, ++t)
            if (t->plan && t->precision == precision_index(g) && t->strang == (strang(g) ? 1 : 0) &&
                t->field == (field_on(g) ? 1 : 0)) {
                cands.push_back({t->steps});
                cands.back().tile = t;
            }
    }
    // save state and counters
    const size_t bytes = (size_t)g->ncells * 8 * g->elem;
    void *backup = nullptr;
    CK(g, cudaMalloc(&backup, bytes));
    cudaMemcpyAsync(backup, g->psi[g->cur], bytes, cudaMemcpyDeviceToDevice, g->stream);
    double flux_saved = 0;
    cudaMemcpyAsync(&g->host_obs[6], g->flux_dev, sizeof(double), cudaMemcpyDeviceToHost, g->stream);
    cudaStreamSynchronize(g->stream);
    flux_saved = g->host_obs[6];
    const int64_t step_saved = g->step, launches_saved = g->launches;
    const int cur_saved = g->cur;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    Cand best = {g->plan.K, g->plan.P, g->plan.wpb, 0, g->plan.fused3d ? g->plan.f_warps : 0,
                 g->plan.s3_fused ? g->plan.s3_warps : 0, g->plan.s3_zfactor, g->plan.s3_zpass};
    double best_t = 1e300;
    const Plan plan_saved = g->plan;
    const int use_graphs = g->cfg.use_graphs;
    g->cfg.use_graphs = 0;
    g->tuning = true;
    dirac_status st = DIRAC_OK;
    for (const Cand &c : cands) {
        g->plan.fused3d = c.fused ? 1 : 0;
        if (c.fused) g->plan.f_warps = c.fused;
        g->plan.s3_fused = c.s3 ? 1 : 0;
        if (c.s3) g->plan.s3_warps = c.s3;
        g->plan.s3_zfactor = c.s3z;
        g->plan.s3_zpass = c.s3zp;
        if (c.tile)
            tile_plan(g, c.tile);
        else
            make_plan(g, c.K, c.P, c.wpb, c.wsm);
        st = ensure_flux_part(g);
        if (st != DIRAC_OK) break;
        const int64_t nsteps = std::max<int64_t>(8, 8 * (int64_t)c.K);
        st = run_steps(g, nsteps);  // warm-up
        if (st != DIRAC_OK) break;
        cudaEventRecord(e0, g->stream);
        st = run_steps(g, 3 * nsteps);
        if (st != DIRAC_OK) break;
        cudaEventRecord(e1, g->stream);
        cudaEventSynchronize(e1);
        float ms = 0;
        cudaEventElapsedTime(&ms, e0, e1);
        const double per_step = ms / (3.0 * nsteps);
        if (per_step < best_t) {
            best_t = per_step;
            best = c;
        }
    }
    g->cfg.use_graphs = use_graphs;
    g->tuning = false;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (st == DIRAC_OK) {
        g->plan.fused3d = best.fused ? 1 : 0;
        if (best.fused) g->plan.f_warps = best.fused;
        g->plan.s3_fused = best.s3 ? 1 : 0;
        if (best.s3) g->plan.s3_warps = best.s3;
        g->plan.s3_zfactor = best.s3z;
        g->plan.s3_zpass = best.s3zp;
        if (best.tile)
            tile_plan(g, best.tile);
        else
            make_plan(g, best.K, best.P, best.wpb, best.wsm);
        st = ensure_flux_part(g);
    }
    if (st != DIRAC_OK) g->plan = plan_saved;  // the scratch has not shrunk
    g->cur = cur_saved;
    cudaMemcpyAsync(g->psi[g->cur], backup, bytes, cudaMemcpyDeviceToDevice, g->stream);
    g->host_obs[6] = flux_saved;
    cudaMemcpyAsync(g->flux_dev, &g->host_obs[6], sizeof(double), cudaMemcpyHostToDevice, g->stream);
    cudaStreamSynchronize(g->stream);
    cudaFree(backup);
    g->step = step_saved;
    g->launches = launches_saved;
    return st;
}

}  // extern "C"
