// Fused 3-D first-order step: x sweep, y sweep, z sweep and phase (Eqs. sol_dis_1-sol_dis_4) in one pass
// over HBM, one step per launch.
//
// A block of W warps owns an x strip of 30 cells (one halo cell each side, lane l holds cell xa + l) and
// a tile of W - 2 rows along y; warp w handles row y0 - 1 + w, so warps 0 and W-1 carry the y halo rows.
// The block streams the planes of its z segment (plus one halo plane each side):
//   * each warp loads its row of the plane, x-sweeps it with warp shuffles and writes the row's y
//     characteristics (U = "+y" movers, W = "-y" movers) to shared memory (double-buffered by plane);
//   * after one block barrier the owned warps y-sweep their row from the rows above and below;
//   * the z sweep keeps the "+z" sums of the two previous planes per cell, in registers or in shared memory
//     (output plane k - 1 = U(k - 2) + W(k)), then the phase with the table pre-scaled by 1/8, and the store.
// Arithmetic order is that of the two-kernel 3-D path (x-y pass at 4x scale, then z sweep and phase), so
// the FP64 result is the same bit for bit.  Face flux: the lanes holding cells face-1 and face of owned
// rows and planes add 1/2 (|u14|^2+|u23|^2) and subtract 1/2 (|w14|^2+|w23|^2) of the state entering the x
// sweep, to a storage-type partial folded into FP64 every 32 planes.
// FIELD: a uniform vector potential; the phase is the 4 x 4 matrix U(step) exp(-i V dt) of Eq. sol_dis_4
// (table entry g = exp(-i V dt) / 8 times each entry of U, then the column-ordered fma chains of the 2-D
// kernel), one launch = one step whose index selects the row of the U table.
// 64-bit fixed-point states (T = long long): the sweeps are exact integer sums, so any order gives the bits
// of the two-kernel path; the phase is the rounded 128-bit product (the table holding round(p 2^62) with the
// 1/8); the face terms are formed in FP64 from the converted values and scaled by the state's 2^-2S.
#pragma once

#include "step_kernels.cuh"

namespace dirac {

struct Fused3DArgs {
    SweepArgs s;          // in, out, table, flux fields; s.nsegs * s.nplanes = flux parts
    int64_t ny, nz;
    int64_t nstrips, nytiles, nzsegs, zseg_h;
};

// accumulator type of the face terms: the storage type, FP64 for fixed-point states
template <typename T> struct FaceAcc { using type = T; };
template <> struct FaceAcc<long long> { using type = double; };
// plane index type of the z loop: 32-bit for floating-point states (grid dimensions stay below 2^31), 64-bit for
// the fixed-point state (register budget)
template <typename T> struct PlaneIdx { using type = int; };
template <> struct PlaneIdx<long long> { using type = int64_t; };

// |p14|^2 + |p23|^2 as a fused chain in the accumulator type
template <typename T>
__device__ __forceinline__ typename FaceAcc<T>::type face_sq(Cx<T> p14, Cx<T> p23) {
    using F = typename FaceAcc<T>::type;
    return Ar<F>::fma((F)p14.re, (F)p14.re,
                      Ar<F>::fma((F)p14.im, (F)p14.im, Ar<F>::fma((F)p23.re, (F)p23.re, Ar<F>::mul((F)p23.im, (F)p23.im))));
}

// FP64 and fixed-point states keep the z sweep's history (the "+z" sums of the two previous planes) in shared memory,
// one slot per plane parity: the registers it frees let two 8-warp blocks run on an SM, whose barriers then fall at
// different times (256^3: FP64 with its pairs over two pipes 7.2 G point-steps/s against 6.9 in one 16-warp block and 6.05
// on the FP64 pipe alone; in a laser field 4.3 against 3.8 and 3.6; fixed point 23.4 against 19.9), although 6 of 8 rows are
// owned instead of 14 of 16.
template <typename T> struct Fused3DHist { static constexpr bool value = sizeof(T) == 8; };
template <typename T, int W> struct Fused3DMinBlocks { static constexpr int value = sizeof(T) == 8 && W == 8 ? 2 : 1; };
template <typename T, int W, bool FIELD>
__global__ void __launch_bounds__(32 * W, Fused3DMinBlocks<T, W>::value) fused3d_kernel(const Fused3DArgs A) {
    constexpr int H = W - 2;
    constexpr bool HY = true;  // FP64 pairs over two pipes
    constexpr bool HS = Fused3DHist<T>::value;
    const SweepArgs &a = A.s;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t b = blockIdx.x;
    const int64_t strip = b % A.nstrips;
    const int64_t rest = b / A.nstrips;
    const int64_t ytile = rest % A.nytiles;
    const int64_t zseg = rest / A.nytiles;
    const int64_t nx = a.nx, ny = A.ny, nz = A.nz;
    const bool per = a.periodic != 0;
    const int64_t x_own0 = strip * 30, x_own1 = min(x_own0 + 30, nx);
    const int64_t x = x_own0 - 1 + lane;
    const int64_t y = ytile * H - 1 + w;
    const bool owned_row = w >= 1 && w <= H && y < ny;
    using ZI = typename PlaneIdx<T>::type;
    const ZI z_begin = (ZI)(zseg * A.zseg_h), z_end = (ZI)min((int64_t)z_begin + A.zseg_h, nz);
    const bool xin = x >= 0 && x < nx, yin = y >= 0 && y < ny;
    const int64_t xl = per ? pmod(x, nx) : min(max(x, (int64_t)0), nx - 1);
    const int64_t yl = per ? pmod(y, ny) : min(max(y, (int64_t)0), ny - 1);
    const T *in = static_cast<const T *>(a.in);
    T *out = static_cast<T *>(a.out);
    const T *tab = static_cast<const T *>(a.table);

    extern __shared__ __align__(16) unsigned char dyn_smem[];
    Cx<T> *ych = reinterpret_cast<Cx<T> *>(dyn_smem);  // [2][W][4][32]

    Cx<T> pu, pd;
    if (!a.full_table) load_tab(tab + xl * 4, pu, pd);
    Cx<T> UM[FIELD ? 6 : 1];  // entries of U for this launch's step: Dup, Ddn, Ez, -Ez, Ep, Em
    if (FIELD) {
        const double *u = a.ucoef + (a.step0 % a.ucoef_n) * 12;
#pragma unroll
        for (int e = 0; e < (FIELD ? 6 : 1); ++e) UM[e] = Cx<T>{(T)__ldg(u + 2 * e), (T)__ldg(u + 2 * e + 1)};
    }
    const int64_t face = a.flux_face;
    const bool face_warp = owned_row && face >= x_own0 && face < x_own1;  // warp-uniform
    const bool face_lane = face_warp && (x == face - 1 || x == face);
    double facc = 0.0;
    typename FaceAcc<T>::type fpart = 0;

    // "+z" sums of the two previous planes: registers, or (HS) the warp's shared memory, slot = plane parity
    Cx<T> UA[2] = {{T(0), T(0)}, {T(0), T(0)}}, UB[2] = {{T(0), T(0)}, {T(0), T(0)}};
    Cx<T> *zh = ych + 2 * W * 4 * 32 + w * 4 * 32 + lane;  // [slot][2][32]
    if (HS)
#pragma unroll
        for (int q = 0; q < 4; ++q) zh[q * 32] = Cx<T>{T(0), T(0)};

    // cell (xl, yl) of a plane: plane k at (k nx ny + cell) (periodic: halo planes wrap)
    const int64_t plane_cells = nx * ny, cell = yl * nx + xl;
    auto wrap_z = [&](ZI k) -> int64_t {
        if (per && (k < 0 || k >= nz)) return pmod((int64_t)k, nz);
        return k;
    };
    auto load_row = [&](ZI k, Cx<T> s[4]) {
        const bool ok = per || (yin && k >= 0 && k < nz && xin);
        if (ok) {
            load_pt(in + (wrap_z(k) * plane_cells + cell) * 8, s);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c) s[c] = {T(0), T(0)};
        }
    };
    // rows of the next planes in flight: one ahead in FP64 (bound by the FP64 pipe), two in FP32 (three or
    // four measured no faster at 256^3 and 384^3: the per-plane block barrier is the limit there)
    constexpr int LA = sizeof(T) == 4 ? 2 : 1;
    Cx<T> ring[LA][4];
#pragma unroll
    for (int j = 0; j < LA; ++j)
        if (z_begin - 1 + j <= z_end) load_row(z_begin - 1 + j, ring[j]);

    // per-cell table entries of the next output plane, loaded one plane ahead (full table only)
    Cx<T> tu = pu, td = pd, tu_next = pu, td_next = pd;

    for (ZI k = z_begin - 1; k <= z_end; ++k) {
        if (a.full_table && owned_row) {
            tu = tu_next;
            td = td_next;
            if (k >= z_begin && k < z_end) load_tab(tab + ((int64_t)k * plane_cells + cell) * 4, tu_next, td_next);
        }
        Cx<T> st[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) st[c] = ring[0][c];
#pragma unroll
        for (int j = 0; j + 1 < LA; ++j)
#pragma unroll
            for (int c = 0; c < 4; ++c) ring[j][c] = ring[j + 1][c];
        if (k + LA <= z_end) load_row(k + LA, ring[LA - 1]);
        // x characteristics and the x sweep (neighbours by shuffle; lanes 0 and 31 are halo cells)
        Cx<T> u14, w14, u23, w23;
        x_chars<HY>(st, u14, w14, u23, w23);
        if (face_lane && k >= z_begin && k < z_end) {
            using F = typename FaceAcc<T>::type;
            const F v = (x == face - 1) ? face_sq(u14, u23) : -face_sq(w14, w23);
            fpart = Ar<F>::add(fpart, v);
            if (IsFx<T>::value && (((k - z_begin) & 31) == 31 || k == z_end - 1)) {
                facc = __dadd_rn(facc, (double)fpart);
                fpart = 0;
            }
        }
        // by the whole warp, a branch (see the two-step kernel); fixed point, with FP64 idle, is 1 % faster the other way
        if (!IsFx<T>::value && face_warp && k >= z_begin && (((k - z_begin) & 31) == 31 || k == z_end - 1)) {
            __syncwarp();
            facc = __dadd_rn(facc, (double)fpart);
            fpart = 0;
        }
        const Cx<T> lu14 = shfl_c(u14, (lane + 31) & 31), lu23 = shfl_c(u23, (lane + 31) & 31);
        const Cx<T> rw14 = shfl_c(w14, (lane + 1) & 31), rw23 = shfl_c(w23, (lane + 1) & 31);
        Cx<T> b4[4], U14, W14, U23, W23;
        x_join<HY>(lu14, rw14, lu23, rw23, b4);
        y_chars<HY>(b4, U14, W14, U23, W23);
        Cx<T> *buf = ych + (size_t)((k - z_begin + 1) & 1) * (W * 4 * 32);
        buf[(w * 4 + 0) * 32 + lane] = U14;
        buf[(w * 4 + 1) * 32 + lane] = U23;
        buf[(w * 4 + 2) * 32 + lane] = W14;
        buf[(w * 4 + 3) * 32 + lane] = W23;
        __syncthreads();
        if (owned_row) {
            // y sweep of row y: "+y" movers of row y-1, "-y" movers of row y+1 (x2 again: 4x the state)
            const Cx<T> U14 = buf[((w - 1) * 4 + 0) * 32 + lane], U23 = buf[((w - 1) * 4 + 1) * 32 + lane];
            const Cx<T> W14 = buf[((w + 1) * 4 + 2) * 32 + lane], W23 = buf[((w + 1) * 4 + 3) * 32 + lane];
            Cx<T> s[4], U13, W13, U24, W24;
            y_join<HY>(U14, W14, U23, W23, s);
            // z sweep (Eq. sol_dis_3): +z movers of plane k-2, -z movers of plane k
            z_chars<HY>(s, U13, W13, U24, W24);
            const ZI zo = k - 1;
            Cx<T> *zk = zh + (int)((k - z_begin) & 1) * 64;
            if (HS) {
                UA[0] = zk[0];
                UA[1] = zk[32];
                zk[0] = U13;
                zk[32] = U24;
            }
            if (zo >= z_begin && zo < z_end) {
                Cx<T> o[4];
                z_join<HY>(UA[0], W13, UA[1], W24, o);
                const Cx<T> qu = a.full_table ? tu : pu, qd = a.full_table ? td : pd;
                if (FIELD) {
                    Cx<T> m6[FIELD ? 6 : 1];
#pragma unroll
                    for (int e = 0; e < (FIELD ? 6 : 1); ++e) m6[e] = cmulp(UM[e], qu);
                    const Cx<T> z0 = {T(0), T(0)};
                    const Cx<T> n0 = cmac(cmac(cmac(z0, o[0], m6[0]), o[2], m6[2]), o[3], m6[4]);
                    const Cx<T> n1 = cmac(cmac(cmac(z0, o[1], m6[0]), o[2], m6[5]), o[3], m6[3]);
                    const Cx<T> n2 = cmac(cmac(cmac(z0, o[0], m6[2]), o[1], m6[4]), o[2], m6[1]);
                    const Cx<T> n3 = cmac(cmac(cmac(z0, o[0], m6[5]), o[1], m6[3]), o[3], m6[1]);
                    o[0] = n0;
                    o[1] = n1;
                    o[2] = n2;
                    o[3] = n3;
                } else {
                    o[0] = cmulp(o[0], qu);
                    o[1] = cmulp(o[1], qu);
                    o[2] = cmulp(o[2], qd);
                    o[3] = cmulp(o[3], qd);
                }
                if (x >= x_own0 && x < x_own1) store_pt(out + ((int64_t)zo * plane_cells + cell) * 8, o);
            }
            if (!HS) {
                UA[0] = UB[0];
                UA[1] = UB[1];
                UB[0] = U13;
                UB[1] = U24;
            }
        }
    }
    if (face >= 0 && face >= x_own0 && face < x_own1) {
        // one flux part per (y tile, z segment, warp) of the strip that owns the face; halo warps write 0
        facc = face_lanes_sum(facc, face, x_own0 - 1);
        if (lane == 0) a.flux_part[(zseg * A.nytiles + ytile) * W + w] = __dmul_rn(0.5 * a.flux_unit, facc);
    }
}

// Two first-order steps per pass (temporal block k = 2): HBM is read and written once per two steps.
// The block's strip is 28 cells (two halo lanes each side) by W R - 4 rows (two halo rows each side; R rows a warp), and
// the block streams its z segment plus two halo planes each side.  Two rows a warp (FP32) halve the rows that go through
// shared memory, give each warp two chains, and let 12 warps of 168 registers hold 24 rows (20 owned) where 16 of 122 hold 16
// (12 owned), which fits small grids better: bound by latency between the two barriers of a plane (issue slots half used, memory 31 % of its peak), 256^3
// 271 -> 218 us a step, 384^3 786 -> 674.  Per input plane k:
//   * step 1: every warp x-sweeps its row and writes its y characteristics to shared memory; after a
//     barrier the rows one inside the halo y-sweep, z-sweep (register history of the "+z" sums of the
//     previous two planes) and take the phase: the state after step 1 at plane k - 1, zeroed outside the
//     grid (zero boundary: cells outside are zero at every sub-step);
//   * step 2: those rows x-sweep it and write its y characteristics; after a second barrier the owned
//     rows y-sweep, z-sweep (their own history) and take the phase of step 2: plane k - 2, stored.
// Each step's arithmetic is that of the one-step kernel, so the result equals two one-step launches bit for
// bit.  Both steps' face flux is taken on the state entering their x sweep (parts [2][nzsegs nytiles W]).
// FIELD: the phase matrices of steps step0 and step0 + 1.
template <typename T, int W, int R, bool FIELD>
__global__ void __launch_bounds__(32 * W, 1) fused3d2_kernel(const Fused3DArgs A) {
    constexpr int ROWS = W * R, H = ROWS - 4;
    const SweepArgs &a = A.s;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t b = blockIdx.x;
    const int64_t strip = b % A.nstrips;
    const int64_t rest = b / A.nstrips;
    const int64_t ytile = rest % A.nytiles;
    const int64_t zseg = rest / A.nytiles;
    const int64_t nx = a.nx, ny = A.ny, nz = A.nz;
    const bool per = a.periodic != 0;
    const int64_t x_own0 = strip * 28, x_own1 = min(x_own0 + 28, nx);
    const int64_t x = x_own0 - 2 + lane;
    const int64_t y0 = ytile * H - 2 + w * R;  // this warp's rows are y0 .. y0 + R - 1
    // warps with a row one inside the halo (step 1's output), and with rows of their own (step 2's)
    const bool mid_warp = w * R + R - 1 >= 1 && w * R < ROWS - 1;
    const bool own_warp = w * R + R - 1 >= 2 && w * R < ROWS - 2 && y0 < ny;
    const bool own_lane = x >= x_own0 && x < x_own1;
    using ZI = typename PlaneIdx<T>::type;
    const ZI z_begin = (ZI)(zseg * A.zseg_h), z_end = (ZI)min((int64_t)z_begin + A.zseg_h, nz);
    const bool xin = x >= 0 && x < nx;
    const int64_t xl = per ? pmod(x, nx) : min(max(x, (int64_t)0), nx - 1);
    auto owned_row = [&](int r) { return w * R + r >= 2 && w * R + r < ROWS - 2 && y0 + r < ny; };
    auto in_xy = [&](int r) { return per || (xin && y0 + r >= 0 && y0 + r < ny); };
    const T *in = static_cast<const T *>(a.in);
    T *out = static_cast<T *>(a.out);
    const T *tab = static_cast<const T *>(a.table);

    extern __shared__ __align__(16) unsigned char dyn_smem[];
    Cx<T> *buf1 = reinterpret_cast<Cx<T> *>(dyn_smem);  // [W][4][32] step 1's y characteristics of the warps' outermost rows
    Cx<T> *buf2 = buf1 + W * 4 * 32;                    // [W][4][32] step 2's

    Cx<T> pu = {T(0), T(0)}, pd = {T(0), T(0)};
    if (!a.full_table) load_tab(tab + xl * 4, pu, pd);
    Cx<T> UM[2][FIELD ? 6 : 1];  // entries of U for the two steps: Dup, Ddn, Ez, -Ez, Ep, Em
    if (FIELD) {
#pragma unroll
        for (int st = 0; st < 2; ++st) {
            const double *u = a.ucoef + ((a.step0 + st) % a.ucoef_n) * 12;
#pragma unroll
            for (int e = 0; e < (FIELD ? 6 : 1); ++e)
                UM[st][e] = Cx<T>{(T)__ldg(u + 2 * e), (T)__ldg(u + 2 * e + 1)};
        }
    }
    const int64_t face = a.flux_face;
    const bool has_face = face >= x_own0 && face < x_own1;  // block-uniform
    const bool on_u = x == face - 1, on_w = x == face;
    double facc[2] = {0.0, 0.0};
    T fp[2] = {T(0), T(0)};

    // cell (xl, yl) of a plane: plane k at (k nx ny + cell) (periodic: halo planes wrap)
    const int64_t plane_cells = nx * ny;
    int64_t cell[R];
#pragma unroll
    for (int r = 0; r < R; ++r)
        cell[r] = (per ? pmod(y0 + r, ny) : min(max(y0 + r, (int64_t)0), ny - 1)) * nx + xl;
    auto wrap_z = [&](ZI k) -> int64_t {
        if (per && (k < 0 || k >= nz)) return pmod((int64_t)k, nz);
        return k;
    };
    auto load_rows = [&](ZI k, Cx<T> (&v)[R][4]) {
        const bool zin = per || (k >= 0 && k < nz);
        const int64_t plane = wrap_z(k) * plane_cells;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (zin && in_xy(r)) {
                load_cell(in + (plane + cell[r]) * 8, v[r], a.wide != 0);
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c) v[r][c] = {T(0), T(0)};
            }
        }
    };
    auto face_term = [&](Cx<T> p14, Cx<T> p23) -> T {
        return Ar<T>::fma(p14.re, p14.re, Ar<T>::fma(p14.im, p14.im, Ar<T>::fma(p23.re, p23.re, Ar<T>::mul(p23.im, p23.im))));
    };
    // x sweep of rows held one cell per lane (valid where both neighbours are); face terms of its input
    auto xsweep = [&](const Cx<T> (&v)[R][4], Cx<T> (&o)[R][4], T &acc, bool count) {
        Cx<T> u14[R], w14[R], u23[R], w23[R], lu14[R], lu23[R], rw14[R], rw23[R];
#pragma unroll
        for (int r = 0; r < R; ++r) x_chars<false>(v[r], u14[r], w14[r], u23[r], w23[r]);
        if (has_face && own_warp && count) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (on_u && owned_row(r)) acc = Ar<T>::add(acc, face_term(u14[r], u23[r]));
                if (on_w && owned_row(r)) acc = Ar<T>::sub(acc, face_term(w14[r], w23[r]));
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
        for (int r = 0; r < R; ++r) x_join<false>(lu14[r], rw14[r], lu23[r], rw23[r], o[r]);
    };
    // y characteristics (Eq. sol_dis_2): "+y" movers (b1 - i b4, b2 + i b3), "-y" movers (b1 + i b4, b2 - i b3)
    Cx<T> U14[R], W14[R], U23[R], W23[R];
    auto ywrite = [&](Cx<T> *buf, const Cx<T> (&v)[R][4]) {
#pragma unroll
        for (int r = 0; r < R; ++r) y_chars<false>(v[r], U14[r], W14[r], U23[r], W23[r]);
        buf[(w * 4 + 0) * 32 + lane] = U14[R - 1];
        buf[(w * 4 + 1) * 32 + lane] = U23[R - 1];
        buf[(w * 4 + 2) * 32 + lane] = W14[0];
        buf[(w * 4 + 3) * 32 + lane] = W23[0];
    };
    // y sweep from the rows below and above, z sweep against the history (output plane = input plane - 1), phase
    auto yz_phase = [&](const Cx<T> *buf, Cx<T> (&HA)[R][2], Cx<T> (&HB)[R][2], const Cx<T> (&qu)[R], const Cx<T> (&qd)[R], int st,
                        Cx<T> (&out4)[R][4]) {
        const int lo = R > 1 ? max(w - 1, 0) : w - 1, hi = R > 1 ? min(w + 1, W - 1) : w + 1;  // beyond them: rows past use
        const Cx<T> l14 = buf[(lo * 4 + 0) * 32 + lane], l23 = buf[(lo * 4 + 1) * 32 + lane];
        const Cx<T> h14 = buf[(hi * 4 + 2) * 32 + lane], h23 = buf[(hi * 4 + 3) * 32 + lane];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int rl = r > 0 ? r - 1 : 0, rh = r < R - 1 ? r + 1 : r;
            Cx<T> s[4], U13, W13, U24, W24;
            Cx<T> *o = out4[r];
            y_join<false>(r > 0 ? U14[rl] : l14, r < R - 1 ? W14[rh] : h14, r > 0 ? U23[rl] : l23, r < R - 1 ? W23[rh] : h23, s);
            z_chars<false>(s, U13, W13, U24, W24);
            z_join<false>(HA[r][0], W13, HA[r][1], W24, out4[r]);
            HA[r][0] = HB[r][0];
            HA[r][1] = HB[r][1];
            HB[r][0] = U13;
            HB[r][1] = U24;
            if (FIELD) {
                Cx<T> m6[FIELD ? 6 : 1];
#pragma unroll
                for (int e = 0; e < (FIELD ? 6 : 1); ++e) m6[e] = cmulp(UM[st][e], qu[r]);
                const Cx<T> z0 = {T(0), T(0)};
                const Cx<T> n0 = cmac(cmac(cmac(z0, o[0], m6[0]), o[2], m6[2]), o[3], m6[4]);
                const Cx<T> n1 = cmac(cmac(cmac(z0, o[1], m6[0]), o[2], m6[5]), o[3], m6[3]);
                const Cx<T> n2 = cmac(cmac(cmac(z0, o[0], m6[2]), o[1], m6[4]), o[2], m6[1]);
                const Cx<T> n3 = cmac(cmac(cmac(z0, o[0], m6[5]), o[1], m6[3]), o[3], m6[1]);
                o[0] = n0;
                o[1] = n1;
                o[2] = n2;
                o[3] = n3;
            } else {
                o[0] = cmulp(o[0], qu[r]);
                o[1] = cmulp(o[1], qu[r]);
                o[2] = cmulp(o[2], qd[r]);
                o[3] = cmulp(o[3], qd[r]);
            }
        }
    };

    constexpr int LA = sizeof(T) == 4 && R == 1 ? 2 : 1;
    const ZI k_first = z_begin - 2, k_last = z_end + 1;
    Cx<T> ring[LA][R][4];
#pragma unroll
    for (int j = 0; j < LA; ++j)
        if (k_first + j <= k_last) load_rows(k_first + j, ring[j]);
    Cx<T> H1A[R][2], H1B[R][2], H2A[R][2], H2B[R][2];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int h = 0; h < 2; ++h) H1A[r][h] = H1B[r][h] = H2A[r][h] = H2B[r][h] = {T(0), T(0)};
    // per-cell table entries (full table): step 1 at plane k - 1 (rows one inside the halo), step 2 at k - 2
    auto table_at = [&](ZI j, Cx<T> (&qu)[R], Cx<T> (&qd)[R]) {
        const bool there = a.full_table && (per || (j >= 0 && j < nz));
        const int64_t plane = wrap_z(j) * plane_cells;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            qu[r] = pu;
            qd[r] = pd;
            if (there) load_tab(tab + (plane + cell[r]) * 4, qu[r], qd[r]);
        }
    };
    Cx<T> t1u[R], t1d[R], t2u[R], t2d[R];
    table_at(k_first - 1, t1u, t1d);
    table_at(k_first - 2, t2u, t2d);

    for (ZI k = k_first; k <= k_last; ++k) {
        Cx<T> st[R][4], q1u[R], q1d[R], q2u[R], q2d[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
#pragma unroll
            for (int c = 0; c < 4; ++c) st[r][c] = ring[0][r][c];
#pragma unroll
            for (int j = 0; j + 1 < LA; ++j)
#pragma unroll
                for (int c = 0; c < 4; ++c) ring[j][r][c] = ring[j + 1][r][c];
            q1u[r] = t1u[r];
            q1d[r] = t1d[r];
            q2u[r] = t2u[r];
            q2d[r] = t2d[r];
        }
        if (k + LA <= k_last) load_rows(k + LA, ring[LA - 1]);
        if (mid_warp) table_at(k, t1u, t1d);      // step 1's next plane
        if (own_warp) table_at(k - 1, t2u, t2d);  // step 2's next plane

        // step 1: x sweep of input plane k
        Cx<T> b4[R][4];
        xsweep(st, b4, fp[0], k >= z_begin && k < z_end);
        ywrite(buf1, b4);
        __syncthreads();
        const ZI j1 = k - 1;  // step 1's output plane
        if (mid_warp) {
            Cx<T> o[R][4];
            yz_phase(buf1, H1A, H1B, q1u, q1d, 0, o);
            const bool zout = !per && (j1 < 0 || j1 >= nz);
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (zout || !in_xy(r)) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) o[r][c] = {T(0), T(0)};
                }
            // step 2: x sweep of plane j1
            xsweep(o, b4, fp[1], j1 >= z_begin && j1 < z_end);
            ywrite(buf2, b4);
        }
        __syncthreads();
        const ZI m = k - 2;  // step 2's output plane
        if (own_warp) {
            Cx<T> o[R][4];
            yz_phase(buf2, H2A, H2B, q2u, q2d, 1, o);
            if (own_lane && m >= z_begin && m < z_end) {
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (owned_row(r)) store_cell(out + ((int64_t)m * plane_cells + cell[r]) * 8, o[r], a.wide != 0);
            }
        }
        // every 32 terms into the FP64 sums, by the whole warp: under a condition on the lane the additions and conversions
        // were issued for every plane of every warp, predicated (37 % of the FP64 pipe's time)
        if (has_face && own_warp && (((k - k_first) & (32 / R - 1)) == 32 / R - 1 || k == k_last)) {
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                facc[q] = __dadd_rn(facc[q], (double)fp[q]);
                fp[q] = T(0);
            }
        }
    }
    if (has_face) {
        // one part per (step, z segment, y tile, warp) of the strip that owns the face; other warps write 0
        const int64_t nparts = A.nzsegs * A.nytiles * W;
        const int64_t q = (zseg * A.nytiles + ytile) * W + w;
#pragma unroll
        for (int st = 0; st < 2; ++st) {
            const double f = face_lanes_sum(facc[st], face, x_own0 - 2);
            if (lane == 0) a.flux_part[st * nparts + q] = __dmul_rn(0.5, f);
        }
    }
}

template <typename T, int W, int R, bool FIELD>
static cudaError_t launch_fused3d2_one(const Fused3DArgs &A, cudaStream_t s) {
    const int64_t blocks = A.nstrips * A.nytiles * A.nzsegs;
    if (blocks <= 0) return cudaSuccess;
    const int smem = 2 * W * 4 * 32 * (int)sizeof(Cx<T>);
    static std::atomic<unsigned long long> done{0};
    cudaError_t e = optin_smem(fused3d2_kernel<T, W, R, FIELD>, smem, done);
    if (e != cudaSuccess) return e;
    fused3d2_kernel<T, W, R, FIELD><<<(unsigned)blocks, 32 * W, smem, s>>>(A);
    return cudaGetLastError();
}

template <typename T, int W, bool FIELD>
static cudaError_t launch_fused3d_one(const Fused3DArgs &A, cudaStream_t s) {
    const int64_t blocks = A.nstrips * A.nytiles * A.nzsegs;
    if (blocks <= 0) return cudaSuccess;
    const int smem = (2 + (Fused3DHist<T>::value ? 1 : 0)) * W * 4 * 32 * (int)sizeof(Cx<T>);
    static std::atomic<unsigned long long> done{0};
    cudaError_t e = optin_smem(fused3d_kernel<T, W, FIELD>, smem, done);
    if (e != cudaSuccess) return e;
    fused3d_kernel<T, W, FIELD><<<(unsigned)blocks, 32 * W, smem, s>>>(A);
    return cudaGetLastError();
}

}  // namespace dirac
