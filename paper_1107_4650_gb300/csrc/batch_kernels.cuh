// Batched ensemble of independent 2-D Klein-step runs (uneven grid sizes and step counts) advanced
// by one persistent kernel per block of K steps.
//
// Work: every active run is cut into (strip, segment) tasks exactly as the single-grid step kernel
// cuts its grid; the tasks of all active runs form one list.  Resident warps take tasks from an
// atomic counter until the list is exhausted (dynamic balance across runs of different sizes) and
// run each task with the single-grid warp routine (sweep_warp), so the arithmetic, boundary and
// flux handling are identical to dirac_step's.  After up to 16 launches a launch of its own folds the per-step
// face-flux partials into the runs' cumulative fluxes (fixed order).
//
// Runs are ordered so that the active set of every launch is a prefix of an order array; the task
// list's prefix offsets are precomputed per order, and a warp finds its run by binary search.
#pragma once

#include "step_kernels.cuh"

namespace dirac {

struct BatchRunDev {
    void *psi[2];           // ping-pong state buffers
    const void *table;      // x-only phase table, 4 values per column (pre-scaled by 1/4)
    int64_t side;           // nx = nz = side
    int64_t face;           // flux face index
    double *flux_part;      // [slot][K][the launch's segments], slots flux_stride apart
    double *flux_cum;       // cumulative flux of this run
    int64_t parity_base;    // parity offset of the remainder phase (number of K-step launches)
};

struct BatchArgs {
    const BatchRunDev *runs;
    const int *order;       // run index per position; the active runs are order[0 .. n_active)
    const int64_t *task_off;// prefix task offsets along `order` (for this launch's K), n_active + 1 used
    int n_active;
    int parity_mode;        // 0: parity = launch & 1 (K-step phase); 1: (parity_base + launch) & 1
    int64_t launch;
    unsigned *counter;      // two task counters: a launch takes from [turn] and clears the other for the next one
    int turn;
    int64_t seg_rows;       // rows per task of this launch
    int64_t flux_off;       // this launch's slot of the flux partials
    unsigned *err;
};

// The flux partials of `count` launches (slots 0 .. count - 1, slot i of the first n_active[i] runs of the order) into the
// runs' cumulative fluxes, one warp per run, launch by launch and step by step (lane l adds segments l, l + 32, ..., then
// an xor tree).
constexpr int kBatchSlots = 16;
__host__ __device__ inline int64_t batch_segments(int64_t side, int64_t seg_rows) {
    const int64_t h = seg_rows < side ? seg_rows : side;
    return (side + h - 1) / h;
}
struct BatchFluxFold {
    const BatchRunDev *runs;
    const int *order;
    int count, K;
    int64_t stride;
    double vol;
    int n_active[kBatchSlots];
    int64_t seg_rows[kBatchSlots];
};
static __global__ void batch_flux_fold_kernel(const __grid_constant__ BatchFluxFold f) {
    const int lane = threadIdx.x & 31, i = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (i >= f.n_active[0]) return;  // the active set only shrinks
    const BatchRunDev &R = f.runs[f.order[i]];
    double F = *R.flux_cum;
    for (int l = 0; l < f.count && i < f.n_active[l]; ++l) {
        const int64_t nsegs = batch_segments(R.side, f.seg_rows[l]);
        for (int s = 0; s < f.K; ++s) {
            const double *part = R.flux_part + l * f.stride + s * nsegs;
            double v = 0.0;
            for (int64_t q = lane; q < nsegs; q += 32) v = __dadd_rn(v, part[q]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
            F = __dadd_rn(F, __dmul_rn(v, f.vol));
        }
    }
    if (lane == 0) *R.flux_cum = F;
}

// FP32 with two points a lane and two or four steps a launch: the sweep history in shared memory and one row per
// iteration (24 runs of sides 768 and 1024, four steps: 196 against 157 G point-steps/s with it in registers and two
// rows per iteration), which with two adjacent cells a lane, the flux of the levels together and two ring slots
// (step_kernels.cuh) leaves room for 16 warps an SM: 254 G, 260 with 96 rows a task.
template <typename T, int K, int P> struct BatchHist {
    static constexpr bool value = sizeof(T) == 4 && P == 2 && K >= 2;
    static constexpr int unroll = value ? 1 : 2;
    static constexpr int blocks = value ? 4 : 1;  // resident 4-warp blocks the registers are fitted to
};

// ONEPIPE (FP64): the pairs on the FP64 pipe alone, for launches of no more tasks than SMs, one to a one-warp block, where the
// integer sums only lengthen a warp's chain.  Such launches come from rows per task that the caller sets, and from single
// small runs: one run of 64^2, 64 to 96 steps, 3.3 -> 2.5 ms, in 128 rows 20.0 -> 15.8; of 1024^2 in 128 rows 51 -> 31.
template <typename T, int K, int P, bool ONEPIPE>
__global__ void __launch_bounds__(128, BatchHist<T, K, P>::blocks) batch_kernel(const BatchArgs b) {
    extern __shared__ __align__(128) unsigned char dyn_smem[];
    const int lane = threadIdx.x & 31;
    unsigned char *wsmem = dyn_smem + (threadIdx.x >> 5) * Ring<T, K, P, BatchHist<T, K, P>::value>::WARP_BYTES;
    const int64_t total = b.task_off[b.n_active];
    if (blockIdx.x == 0 && threadIdx.x == 0) b.counter[b.turn ^ 1] = 0u;  // nobody takes from it during this launch
    for (;;) {
        unsigned task = 0;
        if (lane == 0) task = atomicAdd(b.counter + b.turn, 1u);
        task = __shfl_sync(0xffffffffu, task, 0);
        if ((int64_t)task >= total) break;
        int lo = 0, hi = b.n_active;  // task_off[lo] <= task < task_off[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (b.task_off[mid] <= (int64_t)task) lo = mid; else hi = mid;
        }
        const BatchRunDev &R = b.runs[b.order[lo]];
        const int parity = (int)((b.parity_mode ? R.parity_base + b.launch : b.launch) & 1);
        SweepArgs a{};
        a.in = R.psi[parity];
        a.out = R.psi[parity ^ 1];
        a.table = R.table;
        a.nx = R.side;
        a.nr = R.side;
        a.nplanes = 1;
        a.strip_w = 32 * P - 2 * K;
        a.nstrips = (R.side + a.strip_w - 1) / a.strip_w;
        a.seg_h = min(b.seg_rows, R.side);
        a.nsegs = (R.side + a.seg_h - 1) / a.seg_h;
        a.flux_face = R.face;
        a.flux_part = R.flux_part + b.flux_off;
        a.err = b.err;
        a.periodic = 0;
        a.full_table = 0;
        a.flux_unit = 1.0;  // floating-point states
        a.wide = 1;         // the pool is the library's own, a cell 32 or 64 bytes
        sweep_warp<T, K, P, 0, false, BatchHist<T, K, P>::unroll, BatchHist<T, K, P>::value, ONEPIPE>(a, (int64_t)task - b.task_off[lo], lane, wsmem);
        if (lane == 0) fence_proxy_async();  // this task's reads of the row slots before the next one's first copies into them
    }
}

// Gaussian packet N [1, 0, 0, C] e^{i k0 x} exp(-((x-x0)^2 + z^2)/(4 w^2)) (Sec. 5.2.2) written for every run,
// unnormalised (the transmitted fraction divides by the measured initial norm).  One thread per cell of the
// concatenated runs; cell_off holds each run's first cell.
struct InitArgs {
    const BatchRunDev *runs;
    const int64_t *cell_off;   // [nruns + 1]
    const double *x0, *k0, *width, *spinC;  // per run
    const int64_t *absorb;     // absorbing-layer columns per run: the packet is zero there
    int nruns;
    double dx;
};

template <typename T>
__global__ void batch_init_kernel(const InitArgs ia) {
    const int64_t total = ia.cell_off[ia.nruns];
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < total; g += (int64_t)gridDim.x * blockDim.x) {
        int lo = 0, hi = ia.nruns;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (ia.cell_off[mid] <= g) lo = mid; else hi = mid;
        }
        const BatchRunDev &R = ia.runs[lo];
        const int64_t c = g - ia.cell_off[lo];
        const int64_t i = c % R.side, k = c / R.side;
        const double x = (double)(i - R.face) * ia.dx + 0.5 * ia.dx;         // step face at x = 0
        const double z = (double)(k - R.side / 2) * ia.dx + 0.5 * ia.dx;     // packet centred in z
        const double w = ia.width[lo];
        const double dxx = x - ia.x0[lo];
        const double amp = exp(-(dxx * dxx + z * z) / (4.0 * w * w));
        double sn, cs;
        sincos(ia.k0[lo] * x, &sn, &cs);
        const double C = ia.spinC[lo];
        T *p = static_cast<T *>(R.psi[0]) + c * 8;
        if (i < ia.absorb[lo] || i >= R.side - ia.absorb[lo]) {
#pragma unroll
            for (int q = 0; q < 8; ++q) p[q] = T(0);
            continue;
        }
        p[0] = (T)(amp * cs);
        p[1] = (T)(amp * sn);
        p[2] = T(0); p[3] = T(0); p[4] = T(0); p[5] = T(0);
        p[6] = (T)(C * amp * cs);
        p[7] = (T)(C * amp * sn);
    }
}

// Per-run norm: block b of the launch reduces cells [b*chunk, (b+1)*chunk) of the concatenated runs that
// belong to one run (chunks never straddle runs: run boundaries are chunk-aligned in chunk_off).
struct NormArgs {
    const BatchRunDev *runs;
    const int64_t *chunk_off;  // first chunk of each run, [nruns + 1]
    int nruns;
    int64_t chunk;             // cells per chunk
    double *partial;           // one per chunk
    int parity_from_base;      // 1: read psi[(parity_base + remainder) & 1] via final_parity
    const int *final_parity;   // per run (used when parity_from_base)
};

template <typename T>
__global__ void batch_norm_partial_kernel(const NormArgs na) {
    __shared__ double sh[32];
    const int64_t ch = blockIdx.x;
    int lo = 0, hi = na.nruns;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (na.chunk_off[mid] <= ch) lo = mid; else hi = mid;
    }
    const BatchRunDev &R = na.runs[lo];
    const int par = na.parity_from_base ? na.final_parity[lo] : 0;
    const T *psi = static_cast<const T *>(R.psi[par]);
    const int64_t n = R.side * R.side;
    const int64_t c0 = (ch - na.chunk_off[lo]) * na.chunk;
    const int64_t c1 = min(c0 + na.chunk, n);
    double s = 0.0;
    for (int64_t c = c0 + threadIdx.x; c < c1; c += blockDim.x) {
        const T *p = psi + c * 8;
        double r = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) r = __dadd_rn(r, __dmul_rn((double)p[q], (double)p[q]));
        s = __dadd_rn(s, r);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s = __dadd_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (threadIdx.x == 0) na.partial[ch] = v;
    }
}

static __global__ void batch_norm_fold_kernel(const int64_t *chunk_off, int nruns, const double *partial, double vol,
                                       double *norm) {
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < nruns; r += gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int64_t c = chunk_off[r]; c < chunk_off[r + 1]; ++c) s = __dadd_rn(s, partial[c]);
        norm[r] = __dmul_rn(s, vol);
    }
}

}  // namespace dirac
