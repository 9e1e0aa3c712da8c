// 2-D first- and second-order steps of small grids: K whole steps of a 32 x (W R) tile per block and launch.
//
// A grid of up to about 1000^2 leaves the row kernel (step_kernels.cuh) bound by what a launch costs by itself (about 4 us
// from one to the next, the first rows' latency included) and by the rows of a segment, which follow each other in one warp.
// Here every cell of a tile is in a register: lane = x, each of the W warps holds R rows.  The x sweep takes its neighbours
// by shuffle, the z sweep from registers or, between warps, through shared memory (one block barrier per z sweep, the buffer
// alternating), and K steps follow each other without leaving the SM.  The outermost cell of each side goes stale per sweep
// and axis, so a tile owns 32 - 2 H columns and W R - 2 H rows, H = K (2 K for second-order steps), and neighbours recompute
// the rest: rows that have gone stale are skipped, columns cannot be.  The operations on a cell and their order are the row
// kernel's, so the state is the same bit for bit.
// What bounds it: FP64 the FP64 pipe (0.33 us per row and step on an SM, 32 DADD-class instructions at about 20 clocks);
// FP32 at one tile an SM the latency of a launch and of K dependent steps (5.3 us for four steps of 128^2), at several the
// issue of about 60 instructions a cell and step (0.0135 us per row and step with R = 4, 0.018 with R = 1: the fewer rows go
// through shared memory and the more chains a warp has, the better; two cells a lane gave nothing more), with three blocks of
// 80 registers an SM (1024^2 6.3 -> 6.0 us a step against two, 1300^2 10.5 -> 9.2).
// Measured, us a step with the face flux, row kernel -> this: FP64 128^2 9.1 -> 4.9, 256^2 12.2 -> 8.8 (second order 32.8 ->
// 14.9); FP32 128^2 4.2 -> 1.1, 512^2 5.9 -> 2.5, 1024^2 10.2 -> 6.0 (second order 256^2 7.8 -> 2.5); fixed point 256^2 7.2 ->
// 3.6; in a uniform field, 300^2, FP64 25.0 -> 22.1 (second order 45.8 -> 33.6), FP32 6.6 -> 2.9 (10.9 -> 5.1).  A launch may
// begin while the one before it drains (256^2 FP32 1.5 -> 1.3 us a step).
// Face flux: the two lanes at the face leave each row's sums in shared memory, and after the last step one warp takes all
// rows of a sweep at once, lane = row (evaluated in each row's warp it cost 7 FP64 instructions a row and sweep: FP32 at
// 256^2, K = 4, 4.0 us a step against 1.6).  Parts: [x sweeps][rows of the grid].
#pragma once

#include "step_kernels.cuh"

namespace dirac {

template <typename T, int W, int R, int K, bool STRANG, bool PER, bool FIELD>
__global__ void __launch_bounds__(32 * W, (R == 4 ? 3 : 1)) tile_kernel(const SweepArgs a) {
    constexpr int ROWS = W * R;         // warp w holds rows w R .. w R + R - 1 of the tile
    constexpr int ZS = STRANG ? 2 : 1;  // x sweeps, and z sweeps, a step
    constexpr int H = ZS * K;
    constexpr int OWNX = 32 - 2 * H, OWNZ = ROWS - 2 * H;
    constexpr bool HY = true;  // FP64 pairs over two pipes
    static_assert(OWNX > 0 && OWNZ > 0, "tile too small for its halo");
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    Cx<T> *zch = reinterpret_cast<Cx<T> *>(dyn_smem);  // [2][W][4][32] sums of the warps' outermost rows
    Cx<T> *fhand = zch + 2 * W * 4 * 32;               // [x sweeps][ROWS][4] the face's sums
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nx = (int)a.nx, nz = (int)a.nr;
    const int tx = (int)(blockIdx.x % (unsigned)a.nstrips), tz = (int)(blockIdx.x / (unsigned)a.nstrips);
    const int x0 = tx * OWNX - H, z0 = tz * OWNZ - H + w * R;  // of the tile; of this warp's rows
    const int x = x0 + lane;
    const int64_t xl = PER ? pmod(x, nx) : min(max(x, 0), nx - 1);
    auto in_grid = [&](int r) { return PER || (x >= 0 && x < nx && z0 + r >= 0 && z0 + r < nz); };
    const bool edge = !PER && (x0 < 0 || x0 + 32 > nx || z0 < 0 || z0 + R > nz);  // the warp has cells outside the grid
    Cx<T> pu[R], pd[R], st[R][4];
    // the launch may have started while the one before it still runs: the table is no kernel's output, the state is
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (r == 0 || a.full_table) {
            const int64_t zl = PER ? pmod(z0 + r, nz) : min(max(z0 + r, 0), nz - 1);
            load_tab(static_cast<const T *>(a.table) + (a.full_table ? zl * nx + xl : xl) * 4, pu[r], pd[r]);
        } else {
            pu[r] = pu[0];
            pd[r] = pd[0];
        }
    }
    // with a uniform field the phase is the matrix M = U g, U of the step and g (x-only) of the column: its non-zero entries
    Cx<T> M[FIELD ? K : 1][FIELD ? 6 : 1];
    if (FIELD) {
#pragma unroll
        for (int k = 0; k < (FIELD ? K : 1); ++k) {
            const double *u = a.ucoef + ((a.step0 + k) % a.ucoef_n) * 12;
#pragma unroll
            for (int e = 0; e < (FIELD ? 6 : 1); ++e) M[k][e] = cmulp(Cx<T>{(T)__ldg(u + 2 * e), (T)__ldg(u + 2 * e + 1)}, pu[0]);
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (in_grid(r)) {
            const int64_t zl = PER ? pmod(z0 + r, nz) : z0 + r;
            load_cell(static_cast<const T *>(a.in) + (zl * nx + xl) * 8, st[r], a.wide != 0);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c) st[r][c] = {T(0), T(0)};
        }
    }
    const int face = (int)a.flux_face;
    const bool has_face = face >= tx * OWNX && face < min(tx * OWNX + OWNX, nx);  // block-uniform
    const int lf = face - x0;  // the face cell's lane (H or more); the cell left of it is in the lane before
    auto x_sweep = [&](Cx<T> (&v)[R][4], int s) {
        Cx<T> u14[R], w14[R], u23[R], w23[R], lu14[R], lu23[R], rw14[R], rw23[R];
#pragma unroll
        for (int r = 0; r < R; ++r) x_chars<HY>(v[r], u14[r], w14[r], u23[r], w23[r]);
        if (has_face) {  // the state entering the sweep: outgoing sums left of the face, incoming ones right of it
#pragma unroll
            for (int r = 0; r < R; ++r) {
                Cx<T> *f = fhand + (s * ROWS + w * R + r) * 4;
                if (lane == lf - 1) {
                    f[0] = u14[r];
                    f[1] = u23[r];
                }
                if (lane == lf) {
                    f[2] = w14[r];
                    f[3] = w23[r];
                }
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            lu14[r] = shfl_c(u14[r], (lane + 31) & 31);
            lu23[r] = shfl_c(u23[r], (lane + 31) & 31);
            rw14[r] = shfl_c(w14[r], (lane + 1) & 31);
            rw23[r] = shfl_c(w23[r], (lane + 1) & 31);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) x_join<HY>(lu14[r], rw14[r], lu23[r], rw23[r], v[r]);
    };
    Cx<T> U13[R], W13[R], U24[R], W24[R];
    auto z_put = [&](const Cx<T> (&v)[R][4], Cx<T> *buf) {
#pragma unroll
        for (int r = 0; r < R; ++r) z_chars<HY>(v[r], U13[r], W13[r], U24[r], W24[r]);
        buf[(w * 4 + 0) * 32] = U13[R - 1];
        buf[(w * 4 + 1) * 32] = U24[R - 1];
        buf[(w * 4 + 2) * 32] = W13[0];
        buf[(w * 4 + 3) * 32] = W24[0];
    };
    auto z_get = [&](const Cx<T> *buf, Cx<T> (&v)[R][4]) {
        const int lo = max(w - 1, 0), hi = min(w + 1, W - 1);  // beyond them: rows gone stale (R > 1)
        const Cx<T> l0 = buf[(lo * 4 + 0) * 32], l1 = buf[(lo * 4 + 1) * 32];
        const Cx<T> h0 = buf[(hi * 4 + 2) * 32], h1 = buf[(hi * 4 + 3) * 32];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int rl = r > 0 ? r - 1 : 0, rh = r < R - 1 ? r + 1 : r;
            z_join<HY>(r > 0 ? U13[rl] : l0, r < R - 1 ? W13[rh] : h0, r > 0 ? U24[rl] : l1, r < R - 1 ? W24[rh] : h1, v[r]);
        }
    };
    auto clear_ghosts = [&](Cx<T> (&v)[R][4]) {
        if (edge) {
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (!in_grid(r)) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) v[r][c] = {T(0), T(0)};
                }
        }
    };
    // after e z sweeps the tile's rows [e, ROWS - e) are still exact: a warp goes on while it has one of them
    auto active = [&](int e) { return w * R + R - 1 >= e && w * R < ROWS - e; };
    Cx<T> *const buf0 = zch + lane, *const buf1 = zch + W * 4 * 32 + lane;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int e = ZS * k;
        Cx<T> *const bz = (e & 1) ? buf1 : buf0;
        if (active(e)) {
            x_sweep(st, e);
            z_put(st, bz);
        }
        __syncthreads();
        if (active(e + 1)) {
            z_get(bz, st);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                Cx<T> *o = st[r];
                if (FIELD) {
                    const Cx<T> *m = M[FIELD ? k : 0], z0 = {T(0), T(0)};
                    constexpr int m1 = FIELD ? 1 : 0, m2 = FIELD ? 2 : 0, m3 = FIELD ? 3 : 0, m4 = FIELD ? 4 : 0, m5 = FIELD ? 5 : 0;
                    const Cx<T> n0 = cmac(cmac(cmac(z0, o[0], m[0]), o[2], m[m2]), o[3], m[m4]);
                    const Cx<T> n1 = cmac(cmac(cmac(z0, o[1], m[0]), o[2], m[m5]), o[3], m[m3]);
                    const Cx<T> n2 = cmac(cmac(cmac(z0, o[0], m[m2]), o[1], m[m4]), o[2], m[m1]);
                    const Cx<T> n3 = cmac(cmac(cmac(z0, o[0], m[m5]), o[1], m[m3]), o[3], m[m1]);
                    o[0] = n0;
                    o[1] = n1;
                    o[2] = n2;
                    o[3] = n3;
                } else {
                    o[0] = cmulp(o[0], pu[r]);
                    o[1] = cmulp(o[1], pu[r]);
                    o[2] = cmulp(o[2], pd[r]);
                    o[3] = cmulp(o[3], pd[r]);
                }
            }
            clear_ghosts(st);
            if (STRANG) z_put(st, buf1);
        }
        if (STRANG) {  // second half: the state enters at a quarter of its size, the x sweep at a half
            __syncthreads();
            if (active(e + 2)) {
                z_get(buf1, st);
                clear_ghosts(st);
                x_sweep(st, e + 1);
                clear_ghosts(st);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int row = w * R + r;
        if (row >= H && row < ROWS - H && z0 + r < nz && lane >= H && lane < 32 - H && x < nx)
            store_cell(static_cast<T *>(a.out) + ((int64_t)(z0 + r) * nx + x) * 8, st[r], a.wide != 0);
    }
    if (has_face) {
        __syncthreads();
        for (int s = w; s < H; s += W)
            for (int row = lane; row < ROWS; row += 32) {
                const int z = tz * OWNZ - H + row;
                if (row >= H && row < ROWS - H && z < nz) {
                    const Cx<T> *f = fhand + (s * ROWS + row) * 4;
                    const double scale = (STRANG && (s & 1)) ? 2.0 * a.flux_unit : 0.5 * a.flux_unit;
                    const double r = __dmul_rn(scale, __dadd_rn(abs2d(f[0]), abs2d(f[1])));
                    const double l = __dmul_rn(scale, __dadd_rn(abs2d(f[2]), abs2d(f[3])));
                    a.flux_part[(int64_t)s * nz + z] = __dsub_rn(r, l);
                }
            }
    }
}

template <typename T, int W, int R, int K, bool STRANG, bool PER, bool FIELD>
static cudaError_t launch_tile_per(const SweepArgs &a, int sms, cudaStream_t s) {
    constexpr int H = STRANG ? 2 * K : K, OWNZ = W * R - 2 * H;
    constexpr int need = (2 * 32 + R * H) * W * 4 * (int)sizeof(Cx<T>), two = 80 << 10, one = 120 << 10;
    const int64_t tiles = a.nstrips * ((a.nr + OWNZ - 1) / OWNZ);
    // Two tiles an SM: shared memory that keeps a third out, so that a launch which starts beside the one before it spreads
    // over the chip instead of filling the SMs that drain first (384^2 FP32 2.08 us a step, 1.75 so).
    const int smem = tiles <= 2 * (int64_t)sms && tiles > sms ? (need > two ? need : two) : need;
    static std::atomic<unsigned long long> done{0};
    cudaError_t e = optin_smem(tile_kernel<T, W, R, K, STRANG, PER, FIELD>, need > one ? need : one, done);
    if (e != cudaSuccess) return e;
    // may start while the launch before it drains, and waits for it before it reads the state
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)tiles);
    cfg.blockDim = dim3(32 * W);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, tile_kernel<T, W, R, K, STRANG, PER, FIELD>, a);
}

}  // namespace dirac
