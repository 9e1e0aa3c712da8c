// Fused sweep kernels of the split-operator Dirac scheme (Sec. 2.3, Eqs. sol_dis_1-sol_dis_4).
//
// Design (one warp = one independent strip with shared memory of its own, no block barrier):
//   * a warp owns `strip_w` consecutive x cells of one plane and a segment of rows; it takes
//     32*P cells per row (which of them a lane holds: PairedCells below), i.e. K halo cells on each side, from a
//     ring of rows that bulk copies fill ahead of it;
//   * it streams the rows of its segment (plus K halo rows at each end) through K pipelined
//     levels held in registers: level s turns the step-(s-1) state of row q into the step-s state
//     of row q-1, so one pass over HBM advances K steps (temporal blocking);
//   * the x sweep needs cells x-1 and x+1: the characteristic sums u = a+b of the left neighbour
//     and w = a-b of the right neighbour come from warp shuffles;
//   * the second sweep (z in 2-D, y in the 3-D x-y pass) needs rows q-1 and q+1: each level keeps
//     the "+" characteristic sums of the two previous rows in registers or shared memory (HistSmem);
//   * the ghost-zero boundary is imposed on every level's output (cells outside the grid are 0
//     at every sub-step); a zero row stays zero through the x sweep, so one mask per level is
//     exact.
// Arithmetic order is fixed (explicit round-to-nearest intrinsics, no contraction):
//   sweep:  u = a + b, w = a - b;  a' = u(-) + w(+), b' = u(-) - w(+)   (1/2 factors deferred)
//   phase:  re = fma(z.re, p.re, -(z.im p.im)),  im = fma(z.re, p.im, z.im p.re)
// with p carrying the deferred 1/4 (exact power-of-two scaling).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <type_traits>

#include "butterfly.cuh"
#include "dirac_internal.cuh"
#include "rows.cuh"

namespace dirac {

// Opts `kernel` in to `smem` bytes of dynamic shared memory, once per device (bit `dev` of `done`; devices
// past 63 set the attribute on every launch).  Concurrent first launches may both set it: harmless.
template <typename K>
static cudaError_t optin_smem(K *kernel, int smem, std::atomic<unsigned long long> &done) {
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = dev < 64 ? (1ull << dev) : 0ull;
    if (bit && (done.load(std::memory_order_relaxed) & bit)) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess && bit) done.fetch_or(bit, std::memory_order_relaxed);
    return e;
}

template <typename T> struct Ar;
template <> struct Ar<double> {
    static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
    static __device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
    static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
    static __device__ __forceinline__ double fma(double a, double b, double c) { return __fma_rn(a, b, c); }
};
template <> struct Ar<float> {
    static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
    static __device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
    static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
    static __device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
};

// 64-bit fixed point (storage DIRAC_FX64): the state is q = psi 2^S in int64, so the sweeps' additions are
// exact; only the phase product rounds (cmulp below).
template <> struct Ar<long long> {
    static __device__ __forceinline__ long long add(long long a, long long b) { return a + b; }
    static __device__ __forceinline__ long long sub(long long a, long long b) { return a - b; }
    static __device__ __forceinline__ long long mul(long long a, long long b) { return a * b; }
    static __device__ __forceinline__ long long fma(long long a, long long b, long long c) { return a * b + c; }
};

template <typename T> struct Cx { T re, im; };

template <typename T> __device__ __forceinline__ Cx<T> cadd(Cx<T> a, Cx<T> b) {
    return {Ar<T>::add(a.re, b.re), Ar<T>::add(a.im, b.im)};
}
template <typename T> __device__ __forceinline__ Cx<T> csub(Cx<T> a, Cx<T> b) {
    return {Ar<T>::sub(a.re, b.re), Ar<T>::sub(a.im, b.im)};
}
// FP32: real and imaginary part in one packed instruction (two independent round-to-nearest adds: the same bits as two
// scalar ones in half the issue slots)
template <> __device__ __forceinline__ Cx<float> cadd<float>(Cx<float> a, Cx<float> b) {
    Cx<float> r;
    asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tadd.rn.f32x2 c, a, b;\n\tmov.b64 {%0, %1}, c;\n\t}"
        : "=f"(r.re), "=f"(r.im)
        : "f"(a.re), "f"(a.im), "f"(b.re), "f"(b.im));
    return r;
}
template <> __device__ __forceinline__ Cx<float> csub<float>(Cx<float> a, Cx<float> b) {
    Cx<float> r;
    asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tsub.rn.f32x2 c, a, b;\n\tmov.b64 {%0, %1}, c;\n\t}"
        : "=f"(r.re), "=f"(r.im)
        : "f"(a.re), "f"(a.im), "f"(b.re), "f"(b.im));
    return r;
}
// a + i b and a - i b
template <typename T> __device__ __forceinline__ Cx<T> cadd_ib(Cx<T> a, Cx<T> b) {
    return {Ar<T>::sub(a.re, b.im), Ar<T>::add(a.im, b.re)};
}
template <typename T> __device__ __forceinline__ Cx<T> csub_ib(Cx<T> a, Cx<T> b) {
    return {Ar<T>::add(a.re, b.im), Ar<T>::sub(a.im, b.re)};
}
// Two pairs: s = a + b, d = a - b for (a0, b0) and (a1, b1).  HY: FP64 pairs over the FP64 and the integer pipe
// (butterfly.cuh), the same bits.
template <bool HY, typename T>
__device__ __forceinline__ void butterfly2(Cx<T> a0, Cx<T> b0, Cx<T> a1, Cx<T> b1, Cx<T> &s0, Cx<T> &d0, Cx<T> &s1, Cx<T> &d1) {
    if constexpr (HY && std::is_same<T, double>::value) {
        butterfly(a0.re, b0.re, s0.re, d0.re);
        butterfly(a0.im, b0.im, s0.im, d0.im);
        butterfly(a1.re, b1.re, s1.re, d1.re);
        butterfly(a1.im, b1.im, s1.im, d1.im);
    } else {
        s0 = cadd(a0, b0);
        d0 = csub(a0, b0);
        s1 = cadd(a1, b1);
        d1 = csub(a1, b1);
    }
}
// x characteristics of a point: u14 = 1 + 4, w14 = 1 - 4, u23 = 2 + 3, w23 = 2 - 3
template <bool HY, typename T>
__device__ __forceinline__ void x_chars(const Cx<T> s[4], Cx<T> &u14, Cx<T> &w14, Cx<T> &u23, Cx<T> &w23) {
    butterfly2<HY>(s[0], s[3], s[1], s[2], u14, w14, u23, w23);
}
// x sweep from the left cell's u and the right cell's w (twice the swept point)
template <bool HY, typename T> __device__ __forceinline__ void x_join(Cx<T> u14, Cx<T> w14, Cx<T> u23, Cx<T> w23, Cx<T> o[4]) {
    butterfly2<HY>(u14, w14, u23, w23, o[0], o[3], o[1], o[2]);
}
// y characteristics (Eq. sol_dis_2): "+y" movers U14 = 1 - i 4, U23 = 2 + i 3, "-y" movers W14 = 1 + i 4, W23 = 2 - i 3
template <bool HY, typename T>
__device__ __forceinline__ void y_chars(const Cx<T> b[4], Cx<T> &U14, Cx<T> &W14, Cx<T> &U23, Cx<T> &W23) {
    Cx<T> s0, d0, s1, d1;
    butterfly2<HY>(b[0], Cx<T>{b[3].im, b[3].re}, b[1], Cx<T>{b[2].im, b[2].re}, s0, d0, s1, d1);
    U14 = {s0.re, d0.im};
    W14 = {d0.re, s0.im};
    U23 = {d1.re, s1.im};
    W23 = {s1.re, d1.im};
}
// y sweep from the "+y" movers of the row below and the "-y" movers of the row above (twice the swept point)
template <bool HY, typename T> __device__ __forceinline__ void y_join(Cx<T> U14, Cx<T> W14, Cx<T> U23, Cx<T> W23, Cx<T> o[4]) {
    Cx<T> d0, d1;
    butterfly2<HY>(U14, W14, U23, W23, o[0], d0, o[1], d1);
    o[3] = {-d0.im, d0.re};
    o[2] = {d1.im, -d1.re};
}
// z characteristics (Eq. sol_dis_3): "+z" movers U13 = 1 + 3, U24 = 2 - 4, "-z" movers W13 = 1 - 3, W24 = 2 + 4
template <bool HY, typename T>
__device__ __forceinline__ void z_chars(const Cx<T> b[4], Cx<T> &U13, Cx<T> &W13, Cx<T> &U24, Cx<T> &W24) {
    butterfly2<HY>(b[0], b[2], b[1], b[3], U13, W13, W24, U24);
}
// z sweep from the "+z" movers of the row below and the "-z" movers of the row above (twice the swept point)
template <bool HY, typename T> __device__ __forceinline__ void z_join(Cx<T> U13, Cx<T> W13, Cx<T> U24, Cx<T> W24, Cx<T> o[4]) {
    butterfly2<HY>(U13, W13, W24, U24, o[0], o[2], o[1], o[3]);
}
template <typename T> __device__ __forceinline__ Cx<T> cmulp(Cx<T> z, Cx<T> p) {
    return {Ar<T>::fma(z.re, p.re, -Ar<T>::mul(z.im, p.im)), Ar<T>::fma(z.re, p.im, Ar<T>::mul(z.im, p.re))};
}
// Fixed point: the phase coefficient p is held as round(p 2^62) (|p| <= 1/4: the sweeps' deferred 1/4 rides
// in it), each output component is the exact 128-bit value z.re p.re - z.im p.im (resp. z.re p.im +
// z.im p.re), rounded once to the nearest integer after the 2^-62 (halves upward).  The exact values come
// from three products instead of four (k1 = p.re (z.re + z.im), k2 = z.re (p.im - p.re), k3 = z.im (p.re +
// p.im); re = k1 - k3, im = k1 + k2): integer arithmetic, so the same bits.  |z| < 2^62 and |p| <= 2^60
// keep the sums inside int64.
// The rounding offset 2^61 is added to k1 once, for both outputs: the same integers as rounding each.
template <> __device__ __forceinline__ Cx<long long> cmulp<long long>(Cx<long long> z, Cx<long long> p) {
    const __int128 k1 = (__int128)p.re * (z.re + z.im) + ((__int128)1 << 61);
    const __int128 k2 = (__int128)z.re * (p.im - p.re);
    const __int128 k3 = (__int128)z.im * (p.re + p.im);
    return {(long long)((k1 - k3) >> 62), (long long)((k1 + k2) >> 62)};
}
// The same product with four multiplies for the fixed-point state: each output from two independent 128-bit
// products (re = z.re p.re - z.im p.im, im = z.re p.im + z.im p.re, each rounded as in cmulp, so the same
// integers).  More instructions but no shared sum ahead of the products: measured faster in the 3-D
// second-order z-phase-z pass (12.40 against 12.10 G point-steps/s at 256^3), slower in the 2-D step (31.0
// against 33.2).  Floating-point states take cmulp.
template <typename T> __device__ __forceinline__ Cx<T> cmulp4(Cx<T> z, Cx<T> p) { return cmulp(z, p); }
template <> __device__ __forceinline__ Cx<long long> cmulp4<long long>(Cx<long long> z, Cx<long long> p) {
    const __int128 a = (__int128)z.re * p.re + ((__int128)1 << 61), b = (__int128)z.im * p.im;
    const __int128 c = (__int128)z.re * p.im + ((__int128)1 << 61), d = (__int128)z.im * p.re;
    return {(long long)((a - b) >> 62), (long long)((c + d) >> 62)};
}
// Fixed point: o / 2^r rounded to nearest, halves upward (floating-point states never ask for it).
template <typename T> __device__ __forceinline__ void round_shift(Cx<T> (&)[4], int) {}
template <> __device__ __forceinline__ void round_shift<long long>(Cx<long long> (&o)[4], int r) {
    const long long half = 1ll << (r - 1);
#pragma unroll
    for (int q = 0; q < 4; ++q) o[q] = Cx<long long>{(o[q].re + half) >> r, (o[q].im + half) >> r};
}
// acc + z p with re = fma(z.re, p.re, fma(-z.im, p.im, acc.re)), im = fma(z.re, p.im, fma(z.im, p.re, acc.im))
template <typename T> __device__ __forceinline__ Cx<T> cmac(Cx<T> acc, Cx<T> z, Cx<T> p) {
    return {Ar<T>::fma(z.re, p.re, Ar<T>::fma(-z.im, p.im, acc.re)), Ar<T>::fma(z.re, p.im, Ar<T>::fma(z.im, p.re, acc.im))};
}
template <typename T> __device__ __forceinline__ double abs2d(Cx<T> a) {
    double r = (double)a.re, i = (double)a.im;
    return __dadd_rn(__dmul_rn(r, r), __dmul_rn(i, i));
}

template <typename T> __device__ __forceinline__ Cx<T> shfl_c(Cx<T> v, int src) {
    return {__shfl_sync(0xffffffffu, v.re, src), __shfl_sync(0xffffffffu, v.im, src)};
}

// ---- point load/store: 4 complex components, 64 B (FP64) or 32 B (FP32)
__device__ __forceinline__ void load_pt(const double *p, Cx<double> s[4]) {
    const double2 *q = reinterpret_cast<const double2 *>(p);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        double2 v = q[c];
        s[c] = {v.x, v.y};
    }
}
__device__ __forceinline__ void load_pt(const float *p, Cx<float> s[4]) {
    const float4 *q = reinterpret_cast<const float4 *>(p);
    float4 a = q[0], b = q[1];
    s[0] = {a.x, a.y};
    s[1] = {a.z, a.w};
    s[2] = {b.x, b.y};
    s[3] = {b.z, b.w};
}
__device__ __forceinline__ void store_pt(double *p, const Cx<double> s[4]) {
    double2 *q = reinterpret_cast<double2 *>(p);
#pragma unroll
    for (int c = 0; c < 4; ++c) q[c] = make_double2(s[c].re, s[c].im);
}
__device__ __forceinline__ void store_pt(float *p, const Cx<float> s[4]) {
    float4 *q = reinterpret_cast<float4 *>(p);
    q[0] = make_float4(s[0].re, s[0].im, s[1].re, s[1].im);
    q[1] = make_float4(s[2].re, s[2].im, s[3].re, s[3].im);
}
__device__ __forceinline__ void load_pt(const long long *p, Cx<long long> s[4]) {
    const longlong2 *q = reinterpret_cast<const longlong2 *>(p);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        longlong2 v = q[c];
        s[c] = {v.x, v.y};
    }
}
__device__ __forceinline__ void store_pt(long long *p, const Cx<long long> s[4]) {
    longlong2 *q = reinterpret_cast<longlong2 *>(p);
#pragma unroll
    for (int c = 0; c < 4; ++c) q[c] = make_longlong2(s[c].re, s[c].im);
}
// A point stored to global memory in 32-byte pieces (whole sectors, half the store instructions), where the buffer is
// 32-byte aligned (`wide`; caller-owned buffers need only 16 bytes).
template <typename T> __device__ __forceinline__ void store_cell(T *p, const Cx<T> s[4], bool wide) {
    if (wide) {
        if constexpr (sizeof(T) == 4) {
            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(s[0].re), "f"(s[0].im),
                         "f"(s[1].re), "f"(s[1].im), "f"(s[2].re), "f"(s[2].im), "f"(s[3].re), "f"(s[3].im)
                         : "memory");
        } else if constexpr (std::is_same<T, double>::value) {
            asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(s[0].re), "d"(s[0].im), "d"(s[1].re),
                         "d"(s[1].im)
                         : "memory");
            asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p + 4), "d"(s[2].re), "d"(s[2].im), "d"(s[3].re),
                         "d"(s[3].im)
                         : "memory");
        } else {
            asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(p), "l"(s[0].re), "l"(s[0].im), "l"(s[1].re),
                         "l"(s[1].im)
                         : "memory");
            asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(p + 4), "l"(s[2].re), "l"(s[2].im), "l"(s[3].re),
                         "l"(s[3].im)
                         : "memory");
        }
    } else {
        store_pt(p, s);
    }
}
// A point of a row in shared memory, lane l holding point l (consecutive points).  FP32: lanes 4-7 of every eight take
// their two 16-byte halves in the other order, so that eight lanes' reads cover all banks once (in one order the halves
// of points four apart meet in one bank).
template <typename T> __device__ __forceinline__ void load_row_pt(const T *p, int lane, Cx<T> s[4]) {
    if constexpr (sizeof(T) == 4) {
        const int swap = (lane >> 2) & 1;
        const float4 *q = reinterpret_cast<const float4 *>(p);
        const float4 f = q[swap], g = q[swap ^ 1];
        s[0] = {swap ? g.x : f.x, swap ? g.y : f.y};
        s[1] = {swap ? g.z : f.z, swap ? g.w : f.w};
        s[2] = {swap ? f.x : g.x, swap ? f.y : g.y};
        s[3] = {swap ? f.z : g.z, swap ? f.w : g.w};
    } else {
        load_pt(p, s);
    }
}
// Two adjacent FP32 cells of a row in shared memory, the lanes' 64 bytes consecutive: each lane takes its four 16-byte
// quarters in an order of its own, so that eight lanes read eight different bank groups (no conflict), and puts them in place.
__device__ __forceinline__ void load_row_pair(const float *p, int lane, Cx<float> s0[4], Cx<float> s1[4]) {
    const float4 *q = reinterpret_cast<const float4 *>(p);
    const int f = (lane >> 1) & 3;
    float4 v0 = q[f], v1 = q[1 ^ f], v2 = q[2 ^ f], v3 = q[3 ^ f];
    const bool b0 = f & 1, b1 = f & 2;
    auto pick = [](bool t, float4 a, float4 b) {
        return make_float4(t ? a.x : b.x, t ? a.y : b.y, t ? a.z : b.z, t ? a.w : b.w);
    };
    const float4 c0 = pick(b0, v1, v0), c1 = pick(b0, v0, v1), c2 = pick(b0, v3, v2), c3 = pick(b0, v2, v3);
    v0 = pick(b1, c2, c0);
    v1 = pick(b1, c3, c1);
    v2 = pick(b1, c0, c2);
    v3 = pick(b1, c1, c3);
    s0[0] = {v0.x, v0.y};
    s0[1] = {v0.z, v0.w};
    s0[2] = {v1.x, v1.y};
    s0[3] = {v1.z, v1.w};
    s1[0] = {v2.x, v2.y};
    s1[1] = {v2.z, v2.w};
    s1[2] = {v3.x, v3.y};
    s1[3] = {v3.z, v3.w};
}
// The same pieces for a load.
template <typename T> __device__ __forceinline__ void load_cell(const T *p, Cx<T> s[4], bool wide) {
    if (wide) {
        if constexpr (sizeof(T) == 4) {
            asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=f"(s[0].re), "=f"(s[0].im), "=f"(s[1].re), "=f"(s[1].im), "=f"(s[2].re), "=f"(s[2].im),
                           "=f"(s[3].re), "=f"(s[3].im)
                         : "l"(p)
                         : "memory");
        } else if constexpr (std::is_same<T, double>::value) {
            asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
                         : "=d"(s[0].re), "=d"(s[0].im), "=d"(s[1].re), "=d"(s[1].im)
                         : "l"(p)
                         : "memory");
            asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
                         : "=d"(s[2].re), "=d"(s[2].im), "=d"(s[3].re), "=d"(s[3].im)
                         : "l"(p + 4)
                         : "memory");
        } else {
            asm volatile("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];"
                         : "=l"(s[0].re), "=l"(s[0].im), "=l"(s[1].re), "=l"(s[1].im)
                         : "l"(p)
                         : "memory");
            asm volatile("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];"
                         : "=l"(s[2].re), "=l"(s[2].im), "=l"(s[3].re), "=l"(s[3].im)
                         : "l"(p + 4)
                         : "memory");
        }
    } else {
        load_pt(p, s);
    }
}
// The two sums a level keeps of a row's point, in the warp's shared memory: consecutive lanes 16 bytes apart (no bank
// conflict).  `p` is the pair's place for this lane: 4-byte types keep both sums there, 8-byte types 32 lanes apart.
template <typename T> __device__ __forceinline__ Cx<T> *hist_at(Cx<T> *hist, int slot, int lane) {
    return sizeof(T) == 4 ? hist + (slot * 32 + lane) * 2 : hist + slot * 64 + lane;
}
template <typename T> __device__ __forceinline__ void hist_load(const Cx<T> *p, Cx<T> &a, Cx<T> &b) {
    if constexpr (sizeof(T) == 4) {
        const float4 v = *reinterpret_cast<const float4 *>(p);
        a = {v.x, v.y};
        b = {v.z, v.w};
    } else {
        a = p[0];
        b = p[32];
    }
}
template <typename T> __device__ __forceinline__ void hist_store(Cx<T> *p, Cx<T> a, Cx<T> b) {
    if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4 *>(p) = make_float4(a.re, a.im, b.re, b.im);
    } else {
        p[0] = a;
        p[32] = b;
    }
}
__device__ __forceinline__ void load_tab(const long long *p, Cx<long long> &pu, Cx<long long> &pd) {
    const longlong2 *q = reinterpret_cast<const longlong2 *>(p);
    longlong2 a = q[0], b = q[1];
    pu = {a.x, a.y};
    pd = {b.x, b.y};
}
__device__ __forceinline__ void load_tab(const double *p, Cx<double> &pu, Cx<double> &pd) {
    const double2 *q = reinterpret_cast<const double2 *>(p);
    double2 a = q[0], b = q[1];
    pu = {a.x, a.y};
    pd = {b.x, b.y};
}
__device__ __forceinline__ void load_tab(const float *p, Cx<float> &pu, Cx<float> &pd) {
    float4 a = *reinterpret_cast<const float4 *>(p);
    pu = {a.x, a.y};
    pd = {a.z, a.w};
}

__device__ __forceinline__ int64_t pmod(int64_t a, int64_t n) {
    int64_t r = a % n;
    return r < 0 ? r + n : r;
}

// Rows per iteration of the row loop (1 or 2; measured per variant: two rows let the history registers
// alternate instead of moving, which pays where the loop body is short).
template <typename T, int K, int MODE> struct RowUnroll {
    static constexpr int value = (!std::is_same<T, double>::value && K == 1 && MODE == 0) ? 2 : 1;
};
template <typename T> struct IsFx { static constexpr bool value = std::is_same<T, long long>::value; };  // int64 fixed point
template <typename T> struct IsF64 { static constexpr bool value = std::is_same<T, double>::value; };
// Whether the z sweep's history (the "+" sums of the two previous rows per level) lives in the warp's shared
// memory instead of registers, one slot per row parity so that nothing moves.  Measured at 2048^2 (G point-steps/s,
// the same bits every time):
//   FP32, P = 2: at k = 2 the registers it frees let four blocks (16 warps) per SM run without spilling, 114.5
//     against 105.0 (145 since its accesses are free of bank conflicts); at k = 4 208 -> 128 registers, 105.3 against
//     67.1 (146); second order (mode 2) 60.8 against 56.8 (81).
//   FP64, P = 1: four blocks without spilling, 13.1 against 12.3 first order.
//   Fixed point, P = 1, second order: four blocks instead of two, 22.9 against 19.9 (periodic 22.4 against 20.6);
//     first order periodic 31.9 against 31.6, but zero boundary 31.8 against 33.7: registers there.
// (batch_kernels.cuh has its own choice.)
template <typename T, int K, int P, int MODE, bool PER> struct HistSmem {
    static constexpr bool value =
        (IsF64<T>::value && P == 1 && K == 1 && MODE != 1) ||
        (IsFx<T>::value && P == 1 && K == 1 && (MODE == 2 || (MODE == 0 && PER))) ||
        (sizeof(T) == 4 && P == 2 && ((MODE == 0 && (K == 2 || K == 4)) || (MODE == 2 && (K == 1 || K == 2))));
};
template <typename T, int K, int P, int MODE, bool PER, int UNR = RowUnroll<T, K, MODE>::value, bool HS = false, bool ONEPIPE = false>
__device__ __forceinline__ void sweep_warp(const SweepArgs &a, const int64_t wid, const int lane, unsigned char *wsmem);
template <typename T, int K, int P, bool HS = false> struct Ring;

// Pipelined levels of one launch: K steps, or 2K levels for the second-order splitting (mode 2).
template <int K, int MODE> struct Levels { static constexpr int value = (MODE == 2 || MODE == 5) ? 2 * K : K; };

// MODE 0: 2-D first-order step (x sweep, z sweep, phase), K steps per launch.
// MODE 1: 3-D x-y pass (x sweep, y sweep), K must be 1.
// MODE 2: 2-D second-order (Strang) step x, z, phase(dt), z, x (Sec. 2.4), K steps = 2K levels per launch;
//         the four sweeps' 1/2 factors ride in the phase coefficients as 1/16.
// MODE 3: 2-D first-order step with a uniform vector potential: the phase is the full 4x4 matrix of
//         Eq. sol_dis_4, U(step) exp(-i V dt), with the table holding g = exp(-i V dt) / 4 per column or cell.
// MODE 5: MODE 2 with a uniform vector potential (the phase of each step's first level is the matrix, the
//         table holding g = exp(-i V dt) / 16).
// Resident 4-warp blocks per SM the register budget is fitted to (1: the compiler's choice).  Four (128 registers)
// where the history in shared memory, or two rows per iteration (fixed point first order: 33.1 against 26.7 G at
// 150 registers and 3 blocks), lets them fit; FP64's shared magnitude sums need the warps to fill both pipes, and the FP32
// kernels of two and four levels to cover their latency (k = 4 at 2048^2 22.2 us a step with three blocks, 21.2 with four).
template <typename T, int K, int P, int MODE> struct SweepMinBlocks {
    static constexpr int value = (IsFx<T>::value && K == 1 && P == 1 && (MODE == 0 || MODE == 2))             ? 4
                                 : (sizeof(T) == 4 && P == 2 && (MODE == 0 || MODE == 2) && Levels<K, MODE>::value >= 2) ? 4
                                 : (IsF64<T>::value && K == 1 && P == 1)                                       ? 4
                                                                                                               : 1;
};

template <typename T, int K, int P, int MODE, bool PER>
__global__ void __launch_bounds__(128, SweepMinBlocks<T, K, P, MODE>::value) sweep_kernel(const SweepArgs a) {
    constexpr int L = Levels<K, MODE>::value;
    constexpr bool HS = HistSmem<T, K, P, MODE, PER>::value;
    const int lane = threadIdx.x & 31;
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t per_plane = a.nstrips * a.nsegs;
    extern __shared__ __align__(128) unsigned char dyn_smem[];
    unsigned char *wsmem = dyn_smem + (threadIdx.x >> 5) * Ring<T, L, P, HS>::WARP_BYTES;
    if (wid < per_plane * a.nplanes) sweep_warp<T, K, P, MODE, PER, RowUnroll<T, K, MODE>::value, HS>(a, wid, lane, wsmem);
}

// Face flux: a launch leaves one partial sum per step (or x sweep) and warp, block or segment that owns the face; they are
// folded into the cumulative flux by a launch of its own after up to 32 of them (flux_fold_kernel, observables.cu), not
// by each launch's last block.  That fold, with the fence and the ticket that find the last block, was half of a small
// grid's launch: 128^2 FP32 5.8 us a step, 4.2 so, 2.9 without a face; 256^2 FP64 14.9 and 12.2, 64^3 FP32 second order
// 46 and 30.

// ---- TMA bulk-copy row ring (per warp).  Lane 0 issues one cp.async.bulk per row into a ring slot,
// armed with mbarrier expect_tx; every lane waits on the slot's mbarrier phase before reading it.
// All waits are bounded: on expiry the kernel raises a flag in *a.err and drains its own copies.
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void mbar_inval(uint32_t bar) {
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}
// The lane with `issue` set: orders the warp's reads of a slot before its refill, announces the bytes and starts the copy.
__device__ __forceinline__ void refill_row(bool issue, uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p fence.proxy.async.shared::cta;\n\t"
        "@p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%4], %3;\n\t"
        "@p cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%1], [%2], %3, [%4];\n\t}" ::"r"((uint32_t)issue),
        "r"(dst), "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait for the phase with the given parity to complete: gives up after about one second of the
// global timer (checked every 64 polls), or after 2^24 polls whatever the timer says.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    for (int it = 0; it < (1 << 24); ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if (it > 32) __nanosleep(64);
        if ((it & 63) == 63 && global_ns() - t0 > 1000000000ull) return false;
    }
    return false;
}

// The face flux of several levels evaluated together (flux_row).
template <typename T, int L> struct FluxTogether { static constexpr bool value = sizeof(T) == 4 && L >= 2; };

// Per-warp shared memory: 128 B of mbarriers, the row ring, the flux hand-off area (K levels x 8 values x 32
// lanes), then with HS the sweep history ([row parity 2][level K][point P][lane 32], two complex values each; the ring
// keeps three rows so that four blocks fit, two of the 8-byte types, whose rows last long enough).
template <typename T, int K, int P, bool HS> struct Ring {
    static constexpr int ROW_BYTES = 32 * P * 8 * (int)sizeof(T);  // one warp row: 32P cells
    static constexpr int SLOTS = (HS && (sizeof(T) == 8 || K >= 4)) ? 2 : (HS || ROW_BYTES >= 8192) ? 3 : 4;
    static constexpr int FLUX_BYTES = (FluxTogether<T, K>::value ? 1 : K) * 8 * 32 * (int)sizeof(T);
    static constexpr int HIST_BYTES = HS ? 2 * K * 32 * P * 2 * 2 * (int)sizeof(T) : 0;
    static constexpr int WARP_BYTES = 128 + SLOTS * ROW_BYTES + FLUX_BYTES + HIST_BYTES;
};

// Dynamic shared memory a block of `wpb` warps needs.
template <typename T, int K, int P, bool HS = false> constexpr int ring_smem_bytes(int wpb) {
    return wpb * Ring<T, K, P, HS>::WARP_BYTES;
}

// Records row q's "+" sums in the two-slot history: with two rows per iteration into the slot that held row
// q - 2 (`older`); with one, slot 0 takes slot 1 (row q - 1) and slot 1 takes row q.
template <typename T, int UNR>
__device__ __forceinline__ void push_row(Cx<T> (&s0)[2], Cx<T> (&s1)[2], Cx<T> (&older)[2], Cx<T> v0, Cx<T> v1) {
    if (UNR == 2) {
        older[0] = v0;
        older[1] = v1;
    } else {
        s0[0] = s1[0];
        s0[1] = s1[1];
        s1[0] = v0;
        s1[1] = v1;
    }
}

// Which cells a lane holds: two adjacent ones (2 lane, 2 lane + 1; FP32 with two points a lane), whose inner neighbours need
// no shuffle, or one in each group of 32 (32 j + lane).  The FP32 step of several levels is bound by the shared-memory pipe,
// which shuffles (8 words a cell and level, 4 so), the sweep history and the row reads share, and by its latency: 2048^2
// k = 4 24.8 -> 23.4 us a step, second order 44.1 -> 40.8; one level 48.4 -> 50.4, so not there.
template <typename T, int P, int L> struct PairedCells { static constexpr bool value = sizeof(T) == 4 && P == 2 && L >= 2; };
template <typename T, int P, int L> __device__ __forceinline__ int cell_of(int lane, int j) {
    return PairedCells<T, P, L>::value ? 2 * lane + j : 32 * j + lane;
}

// x characteristics of a row (u = a + b travels +x, w = a - b travels -x) and the neighbours the x sweep
// takes: u of the left cell and w of the right cell (warp shuffles; with one cell in each group of 32, lane 0 and lane 31
// take them from the adjacent point of lanes 31 and 0).
template <bool HY, int L, typename T, int P>
__device__ __forceinline__ void x_characteristics(const Cx<T> (*s)[4], int lane, int src_prev, int src_next, Cx<T> *u14,
                                                  Cx<T> *u23, Cx<T> *w14, Cx<T> *w23, Cx<T> *lu14, Cx<T> *lu23,
                                                  Cx<T> *rw14, Cx<T> *rw23) {
#pragma unroll
    for (int j = 0; j < P; ++j) x_chars<HY>(s[j], u14[j], w14[j], u23[j], w23[j]);
    if constexpr (PairedCells<T, P, L>::value) {
        lu14[0] = shfl_c(u14[1], src_prev);
        lu23[0] = shfl_c(u23[1], src_prev);
        rw14[1] = shfl_c(w14[0], src_next);
        rw23[1] = shfl_c(w23[0], src_next);
        lu14[1] = u14[0];
        lu23[1] = u23[0];
        rw14[0] = w14[1];
        rw23[0] = w23[1];
        return;
    }
    Cx<T> pu14[P], pu23[P], nw14[P], nw23[P];
#pragma unroll
    for (int j = 0; j < P; ++j) {
        pu14[j] = shfl_c(u14[j], src_prev);
        pu23[j] = shfl_c(u23[j], src_prev);
        nw14[j] = shfl_c(w14[j], src_next);
        nw23[j] = shfl_c(w23[j], src_next);
    }
#pragma unroll
    for (int j = 0; j < P; ++j) {
        const int jp = j > 0 ? j - 1 : 0;
        const int jn = j < P - 1 ? j + 1 : P - 1;
        lu14[j] = (lane == 0) ? pu14[jp] : pu14[j];
        lu23[j] = (lane == 0) ? pu23[jp] : pu23[j];
        rw14[j] = (lane == 31) ? nw14[jn] : nw14[j];
        rw23[j] = (lane == 31) ? nw23[jn] : nw23[j];
    }
}

// The sum over a warp of values that are zero but on the lanes of cells face - 1 and face (cells consecutive in the lanes,
// lane 0 holding cell x0): the two of them added, the same value as any tree over all lanes gives, in every lane.
__device__ __forceinline__ double face_lanes_sum(double v, int64_t face, int64_t x0) {
    const int l = (int)(face - x0);
    const double a = __shfl_sync(0xffffffffu, v, l - 1), b = __shfl_sync(0xffffffffu, v, l);
    return __dadd_rn(a, b);
}

// The face's 8 values of a row: u of the cell left of it and w of the cell right of it, left at `g` by the face lane.
template <typename T, int P>
__device__ __forceinline__ void flux_put(const Cx<T> *lu14, const Cx<T> *lu23, const Cx<T> *w14, const Cx<T> *w23,
                                         int face_j, bool on_face, T *g) {
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int j = 0; j < P; ++j) {
            const Cx<T> v[4] = {lu14[j], lu23[j], w14[j], w23[j]};
            if (on_face && j == face_j) store_pt(g, v);
        }
    } else if (on_face) {  // one branch: a store for each point costs registers (fixed point 112.6 against 107.3 us)
        Cx<T> v[4] = {lu14[0], lu23[0], w14[0], w23[0]};
#pragma unroll
        for (int j = 1; j < P; ++j) {
            if (j == face_j) {
                v[0] = lu14[j];
                v[1] = lu23[j];
                v[2] = w14[j];
                v[3] = w23[j];
            }
        }
        store_pt(g, v);
    }
}
// scale (|u14|^2 + |u23|^2) - scale (|w14|^2 + |w23|^2) of the values at `g`
template <typename T> __device__ __forceinline__ double flux_value(const T *g, double scale) {
    Cx<T> v[4];
    load_pt(g, v);
    const double right = __dmul_rn(scale, __dadd_rn(abs2d(v[0]), abs2d(v[1])));
    const double left = __dmul_rn(scale, __dadd_rn(abs2d(v[2]), abs2d(v[3])));
    return __dsub_rn(right, left);
}

// Face flux: the face lane leaves each row's 8 values in the hand-off area, and 32 of them are evaluated at once, one per
// lane, scale = 1/2 for a state at its true size, 2 for one held at half size.  The face's warps run as long as the launch
// does when it is one wave, so what a row costs them counts whole: handing the values over by eight shuffles a row the
// launch took 29.6 us a step against 23.3 without a face (FP32 k = 2 at 2048^2; second order 52.2 against 37.9), by a store
// of the face lane and with the partials folded by a launch of their own 25.3 (44.2).
// Several levels of 4-byte types: 32 / L rows of the L levels together, one sum a lane and 1 KB a warp instead of 4, which
// with two ring slots lets four blocks of the k = 4 kernel on an SM instead of three (2048^2 23.4 -> 21.2 us a step).  The
// 8-byte kernels are at the edge of their registers, where that form costs more (fixed point 39.1 -> 36.8 G): 32 rows of
// each level.
template <typename T, int P>
__device__ __forceinline__ void flux_row(const Cx<T> *lu14, const Cx<T> *lu23, const Cx<T> *w14, const Cx<T> *w23,
                                         int face_j, int face_lane, int lane, int64_t row_in_seg, bool last_row, T *g,
                                         double scale, double &facc) {
    const int t = (int)(row_in_seg & 31);
    flux_put<T, P>(lu14, lu23, w14, w23, face_j, lane == face_lane, g + t * 8);
    if (t == 31 || last_row) {
        __syncwarp();
        if (lane <= t) facc = __dadd_rn(facc, flux_value(g + lane * 8, scale));
        __syncwarp();
    }
}

template <typename T, int K, int P, int MODE, bool PER, int UNR, bool HS, bool ONEPIPE>
__device__ __forceinline__ void sweep_warp(const SweepArgs &a, const int64_t wid, const int lane, unsigned char *wsmem) {
    constexpr int L = Levels<K, MODE>::value;  // pipelined levels (one row and one x cell of halo each)
    // FP64 pairs over two pipes, except where the registers run out: four points a lane (8.5 against 9.6 G at 2048^2),
    // the batched kernel's two steps a launch (6.2 against 8.6 G on 12 runs; one step: 9.8 against 8.9 G), and with two points
    // a lane, whose 8 warps an SM wait longer for the integer sums, the 3-D x-y pass (24^3 127 us a step so, 91.5 on the
    // FP64 pipe alone; 256^3 2471 and 2397) and the zero-boundary second-order step (2048^2 794 and 760, 200 x 150 38 and
    // 27; 1024^2 221 and 225)
    constexpr bool HY = !ONEPIPE && (P == 1 || (P == 2 && !(K == 2 && UNR == 2) && MODE != 1 && !(MODE == 2 && !PER)));
    const int64_t per_plane = a.nstrips * a.nsegs;
    const int64_t plane = wid / per_plane;
    const int64_t rem = wid - plane * per_plane;
    const int64_t seg = rem / a.nstrips;
    const int64_t strip = rem - seg * a.nstrips;
    const int64_t nx = a.nx, nr = a.nr;
    constexpr bool per = PER;
    const int64_t x_own0 = strip * a.strip_w;
    const int64_t x_own1 = min(x_own0 + a.strip_w, nx);
    const int64_t xa = x_own0 - L;
    // Rows are counted from the segment's first in 32 bits (FP32 k = 2 105 against 94 G at 2048^2 with 64-bit ones, fixed
    // point 39.4 against 37.5 G; the grid's own numbers run out of them near 2^31 rows).
    using RI = int;
    const SegRows sr = seg_rows(seg, a.seg_h, nr);
    const uint32_t row0 = (uint32_t)sr.row0, nr32 = (uint32_t)nr;
    auto in_grid = [&](RI r) { return row_in_grid(row0, r, nr32); };
    constexpr RI r_begin = 0;
    const RI r_end = sr.end;
    const T *in = static_cast<const T *>(a.in) + plane * nr * nx * 8;
    T *out = static_cast<T *>(a.out) + plane * nr * nx * 8;

    // every lane's cells lie inside the grid (or wrap): output rows inside the grid need no ghost-zero mask
    const bool strip_in = per || (xa >= 0 && xa + 32 * P <= nx);
    int64_t xl[P];
    bool xin[P], own[P];  // own: the cell is in this warp's strip (it stores it)
#pragma unroll
    for (int j = 0; j < P; ++j) {
        const int64_t x = xa + cell_of<T, P, L>(lane, j);
        xin[j] = (x >= 0 && x < nx);
        own[j] = x >= x_own0 && x < x_own1;
        xl[j] = per ? pmod(x, nx) : min(max(x, (int64_t)0), nx - 1);
    }
    // phase coefficients per x column (mode 0, x-only table)
    Cx<T> pu[P], pd[P];
    if (MODE != 1 && !a.full_table) {
#pragma unroll
        for (int j = 0; j < P; ++j) load_tab(static_cast<const T *>(a.table) + xl[j] * 4, pu[j], pd[j]);
    }
    // MODES 3 and 5: entries of U for each step of the launch (Dup, Ddn, Ez, -Ez, Ep, Em; Sec. 2.3), and with
    // an x-only table the entries times this lane's g per cell (M = U g, formed once per task)
    constexpr bool FLD = MODE == 3 || MODE == 5;
    constexpr int LA = FLD ? K : 1;
    Cx<T> UM[LA][6];
    Cx<T> MA[LA][FLD ? P : 1][6];
    if (FLD) {
#pragma unroll
        for (int st = 0; st < LA; ++st) {
            const double *u = a.ucoef + ((a.step0 + st) % a.ucoef_n) * 12;
#pragma unroll
            for (int e = 0; e < 6; ++e) UM[st][e] = Cx<T>{(T)__ldg(u + 2 * e), (T)__ldg(u + 2 * e + 1)};
            if (!a.full_table)
#pragma unroll
                for (int j = 0; j < (FLD ? P : 1); ++j)
#pragma unroll
                    for (int e = 0; e < 6; ++e) MA[st][j][e] = cmulp(UM[st][e], pu[j]);
        }
    }
    // Flux through the face (owned by this strip): per row, 1/2(|u14|^2+|u23|^2) at face-1 minus
    // 1/2(|w14|^2+|w23|^2) at face, evaluated 32 rows (or rows of the levels) at once, so the FP64 work runs SIMT-wide (1/32
    // of the FP64 issue a single lane would need).  Each lane accumulates its rows in FP64 (FT: lane lev FR + t those of
    // level lev); a fixed xor tree adds lanes.
    constexpr bool FT = FluxTogether<T, L>::value;
    constexpr int FR = FT ? 32 / L : 32;
    const bool has_face = a.flux_face >= x_own0 && a.flux_face < x_own1;
    const int face_off = (int)(a.flux_face - xa);
    const int face_lane = PairedCells<T, P, L>::value ? face_off >> 1 : face_off & 31;
    const int face_j = PairedCells<T, P, L>::value ? face_off & 1 : face_off >> 5;
    double facc[FT ? 1 : L];
#pragma unroll
    for (int s = 0; s < (FT ? 1 : L); ++s) facc[s] = 0.0;

    // "+" characteristic sums of the two previous rows per level: rows q-2 (A) and q-1 (B)
    // The two previous rows' sums per level sit in two register slots.  With rows taken in pairs (UNR = 2),
    // row q of level lev reads slot (pair position + lev) & 1, which holds row q - 2, and overwrites it with
    // row q: the slot indices are compile-time constants and nothing moves.  With UNR = 1, slot 0 holds row
    // q - 2 and slot 1 row q - 1, shifted down after each row.
    Cx<T> UH[2][L][P][2];
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int s = 0; s < L; ++s)
#pragma unroll
            for (int j = 0; j < P; ++j)
#pragma unroll
                for (int h = 0; h < 2; ++h) UH[t][s][j][h] = {T(0), T(0)};

    const int src_prev = (lane + 31) & 31, src_next = (lane + 1) & 31;

    // Row ring: the copied span of a row is the strip's cells clipped to the grid.
    using RG = Ring<T, L, P, HS>;
    // HS: the sweep history in shared memory, slot = parity of the row it holds, zero at the task's start
    Cx<T> *hist = reinterpret_cast<Cx<T> *>(wsmem + 128 + RG::SLOTS * RG::ROW_BYTES + RG::FLUX_BYTES);
    if (HS) {
#pragma unroll
        for (int t = 0; t < 2 * L * P; ++t) hist_store(hist_at(hist, t, lane), Cx<T>{T(0), T(0)}, Cx<T>{T(0), T(0)});
    }
    T *gsm = reinterpret_cast<T *>(wsmem + 128 + RG::SLOTS * RG::ROW_BYTES);  // flux hand-off
    // span of grid cells a row copy brings: the strip clipped to the grid; periodic: all 32 P cells, wrapped, as
    // pieces that end at the grid's right edge (two at most where nx >= 32 P)
    const int64_t cx0 = per ? pmod(xa, nx) : max(xa, (int64_t)0), cx1 = per ? xa + 32 * P : min(xa + 32 * P, nx);
    constexpr uint32_t CELL = 8 * (uint32_t)sizeof(T);
    const uint32_t copy_bytes = per ? (uint32_t)RG::ROW_BYTES : (uint32_t)(cx1 - cx0) * CELL;
    const uint32_t bar0 = smem_u32(wsmem);
    const uint32_t slot0 = smem_u32(wsmem + 128);
    const uint32_t dst_off = per ? 0u : (uint32_t)(cx0 - xa) * CELL;
    // lane 0: row r of the grid into slot sl
    auto fetch_row = [&](uint32_t r, int sl) {
        const T *row = in + (int64_t)r * nx * 8;
        const uint32_t bar = bar0 + 8 * sl, dst = slot0 + sl * RG::ROW_BYTES + dst_off;
        bar_expect(bar, copy_bytes);
        if (!per) {
            bulk_copy(dst, row + cx0 * 8, copy_bytes, bar);
        } else {
            int64_t x = cx0;
            for (int done = 0; done < 32 * P;) {
                const int n = (int)min((int64_t)(32 * P - done), nx - x);
                bulk_copy(dst + (uint32_t)done * CELL, row + x * 8, (uint32_t)n * CELL, bar);
                done += n;
                x = 0;
            }
        }
    };
    // a row of the segment or its halo in the grid's own numbering (periodic: wrapped)
    auto grid_row = [&](RI r) -> uint32_t {
        return per ? wrap_row(row0, r, nr32) : row0 + (uint32_t)r;
    };
    const RI r_first = r_begin - L, r_last = r_end + L;  // rows [r_first, r_last) are read
    uint32_t phase_bits = 0, pending = 0;
    bool aborted = false;
    if (lane == 0) {
#pragma unroll
        for (int sl = 0; sl < RG::SLOTS; ++sl) mbar_init(bar0 + 8 * sl, 1);
        mbar_fence_init();
    }
    if (!strip_in) {  // cells outside the grid: zero in every slot, and no copy reaches them
        const Cx<T> none[4] = {{T(0), T(0)}, {T(0), T(0)}, {T(0), T(0)}, {T(0), T(0)}};
#pragma unroll
        for (int sl = 0; sl < RG::SLOTS; ++sl)
#pragma unroll
            for (int j = 0; j < P; ++j)
                if (!xin[j]) store_pt(reinterpret_cast<T *>(wsmem + 128 + sl * RG::ROW_BYTES) + cell_of<T, P, L>(lane, j) * 8, none);
    }
    __syncwarp();
    bool stall = a.inject_stall && wid == 0;
#pragma unroll
    for (int sl = 0; sl < RG::SLOTS; ++sl) {
        const RI r = r_first + sl;
        if (r < r_last && (per || in_grid(r))) {
            if (lane == 0) {
                // failure-detection test hook: the first warp of the launch announces 16 bytes more than
                // its first row copy delivers, so that slot's phase never completes and its bounded wait
                // runs out (the copy itself completes normally)
                if (stall)
                    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], 16;" ::"r"(bar0 + 8 * sl)
                                 : "memory");
                fetch_row(grid_row(r), sl);
            }
            stall = false;
            pending |= 1u << sl;
        }
    }

    // One input row through the levels.  STEADY: every level's output row is wanted and lies inside the grid (all rows
    // but a segment's first 2 L and the last ones beyond the grid), so nothing is tested per level: FP32 k = 2 at 2048^2
    // 42.0 -> 31.4 M warp instructions a launch with the packed adds, k = 4 125 -> 139 G point-steps/s, the batched
    // kernel 154 -> 164.  What then bounds the FP32 kernel is the shared-memory pipe (82 % busy at k = 2, half of it bank
    // conflicts of the history and the row reads): without the conflicts and with 32-byte stores 124 -> 145 G.
    T *orow = out + ((sr.row0 + r_first - L) * nx + xa) * 8;  // output row r - L
    const T *frow = in + ((sr.row0 + r_first + RG::SLOTS) * nx + cx0) * 8;  // zero boundary: span of row r + SLOTS
    const RI f_end = per ? r_last : min(r_last, sr.top);                  // rows [.., f_end) are fetched
    const int64_t row_step = nx * 8;
    int sl = 0;
    auto do_row = [&](auto steady_c, auto par_c, const RI r) -> bool {
        constexpr bool STEADY = decltype(steady_c)::value;
        constexpr int par = decltype(par_c)::value;
        Cx<T> st[P][4];
        const bool row_ok = STEADY || per || in_grid(r);
        if (row_ok) {
            if (!mbar_wait(bar0 + 8 * sl, (phase_bits >> sl) & 1u)) return false;
            phase_bits ^= 1u << sl;
            pending &= ~(1u << sl);
        }
        const T *srow = reinterpret_cast<const T *>(wsmem + 128 + sl * RG::ROW_BYTES);
        if (row_ok) {
            if constexpr (PairedCells<T, P, L>::value) {
                load_row_pair(srow + lane * 16, lane, st[0], st[1]);
            } else {
#pragma unroll
                for (int j = 0; j < P; ++j) load_row_pt(srow + cell_of<T, P, L>(lane, j) * 8, lane, st[j]);
            }
        } else {
#pragma unroll
            for (int j = 0; j < P; ++j)
#pragma unroll
                for (int c = 0; c < 4; ++c) st[j][c] = {T(0), T(0)};
        }
        // refills this slot with row r + SLOTS once every lane has read it
        auto refill = [&]() {
            __syncwarp();
            const RI rn = r + RG::SLOTS;
            if (rn < f_end && (STEADY || per || in_grid(rn))) {
                if (per) {
                    if (lane == 0) {
                        fence_proxy_async();
                        fetch_row(grid_row(rn), sl);
                    }
                } else {
                    refill_row(lane == 0, slot0 + sl * RG::ROW_BYTES + dst_off, frow, copy_bytes, bar0 + 8 * sl);
                }
                pending |= 1u << sl;
            }
        };
        // before the sweeps where rows last long (two or more levels; 2048^2 FP32 k = 4 with two slots), else after the stores
        // (the 3-D x-y pass 521 us a step against 531 so)
        constexpr bool EARLY = L >= 2;
        if (EARLY) refill();
        const int frow_t = (int)(r - r_first) & (FR - 1);
#pragma unroll
        for (int lev = 0; lev < L; ++lev) {
            const RI q = r - lev;  // row of the level-lev state in st
            // rows of level lev+1 that later levels (or the store) use begin at r_first + lev + 1
            const bool need_out = STEADY || r >= r_first + 2 * lev + 2;
            if ((MODE == 2 || MODE == 5) && (lev & 1)) {
                // second half of a Strang step: z sweep of rows q-2 and q into row q-1, then the x sweep of
                // row q-1.  The input is 1/4 of the state (the phase carried 1/16), the z-swept row 1/2 of it.
                const bool zrow_ok = STEADY || per || in_grid(q - 1);
                Cx<T> zs[P][4];
#pragma unroll
                for (int j = 0; j < P; ++j) {
                    Cx<T> U13, W13, U24, W24;
                    z_chars<HY>(st[j], U13, W13, U24, W24);
                    Cx<T>(&UO)[2] = UH[UNR == 2 ? (par + lev) & 1 : 0][lev][j];  // row q - 2
                    Cx<T> *hq = hist_at(hist, ((int)(q & 1) * L + lev) * P + j, lane);  // HS: its slot
                    Cx<T> o0 = UO[0], o1 = UO[1];
                    if (HS) hist_load(hq, o0, o1);
                    z_join<HY>(o0, W13, o1, W24, zs[j]);
                    if (HS) {
                        hist_store(hq, U13, U24);
                    } else {
                        push_row<T, UNR>(UH[0][lev][j], UH[1][lev][j], UO, U13, U24);
                    }
                    if (!zrow_ok)
#pragma unroll
                        for (int c = 0; c < 4; ++c) zs[j][c] = Cx<T>{T(0), T(0)};
                }
                if (!need_out) {
#pragma unroll
                    for (int j = 0; j < P; ++j)
#pragma unroll
                        for (int c = 0; c < 4; ++c) st[j][c] = Cx<T>{T(0), T(0)};
                    continue;
                }
                Cx<T> u14[P], u23[P], w14[P], w23[P], lu14[P], lu23[P], rw14[P], rw23[P];
                x_characteristics<HY, L, T, P>(zs, lane, src_prev, src_next, u14, u23, w14, w23, lu14, lu23, rw14, rw23);
                if (FT) {
                    if (has_face) flux_put<T, P>(lu14, lu23, w14, w23, face_j, lane == face_lane, gsm + (lev * FR + frow_t) * 8);
                } else if (has_face && q - 1 >= r_begin && q - 1 < r_end) {
                    flux_row<T, P>(lu14, lu23, w14, w23, face_j, face_lane, lane, q - 1 - r_begin, q - 1 == r_end - 1,
                                   gsm + lev * 8 * 32, 2.0 * a.flux_unit, facc[FT ? 0 : lev]);
                }
#pragma unroll
                for (int j = 0; j < P; ++j) {
                    const bool keep = per || (zrow_ok && xin[j]);
                    Cx<T> b[4];
                    x_join<HY>(lu14[j], rw14[j], lu23[j], rw23[j], b);
#pragma unroll
                    for (int c = 0; c < 4; ++c) st[j][c] = keep ? b[c] : Cx<T>{T(0), T(0)};
                }
                continue;
            }
            Cx<T> u14[P], u23[P], w14[P], w23[P], lu14[P], lu23[P], rw14[P], rw23[P];
            x_characteristics<HY, L, T, P>(st, lane, src_prev, src_next, u14, u23, w14, w23, lu14, lu23, rw14, rw23);
            if (FT) {
                if (has_face) flux_put<T, P>(lu14, lu23, w14, w23, face_j, lane == face_lane, gsm + (lev * FR + frow_t) * 8);
            } else if (has_face && q >= r_begin && q < r_end) {
                flux_row<T, P>(lu14, lu23, w14, w23, face_j, face_lane, lane, q - r_begin, q == r_end - 1,
                               gsm + lev * 8 * 32, 0.5 * a.flux_unit, facc[FT ? 0 : lev]);
            }
            const bool out_row_ok = STEADY || per || in_grid(q - 1);
#pragma unroll
            for (int j = 0; j < P; ++j) {
                // x sweep (Eq. sol_dis_1), x2
                Cx<T> b[4], o[4];
                x_join<HY>(lu14[j], rw14[j], lu23[j], rw23[j], b);
                if (MODE != 1) {
                    // z sweep (Eq. sol_dis_3)
                    Cx<T> U13, W13, U24, W24;
                    z_chars<HY>(b, U13, W13, U24, W24);
                    // row q - 2's sums: the slot of q's parity (HS) or the register slot
                    Cx<T> *hp = hist_at(hist, ((int)(q & 1) * L + lev) * P + j, lane);
                    Cx<T> h0, h1;
                    if (HS) {
                        hist_load(hp, h0, h1);
                    } else {
                        h0 = UH[UNR == 2 ? (par + lev) & 1 : 0][lev][j][0];
                        h1 = UH[UNR == 2 ? (par + lev) & 1 : 0][lev][j][1];
                    }
                    if (need_out) {
                        z_join<HY>(h0, W13, h1, W24, o);
                        // phase (Eq. sol_dis_4) with the deferred 1/4
                        Cx<T> qu, qd;
                        if (a.full_table) {
                            const int64_t rr = per || in_grid(q - 1) ? grid_row(q - 1) : 0u;
                            load_tab(static_cast<const T *>(a.table) + (plane * nr * nx + rr * nx + xl[j]) * 4, qu, qd);
                        } else {
                            qu = pu[j];
                            qd = pd[j];
                        }
                        if (FLD) {
                            // psi'_a = sum_b (U_ab g) psi_b over the non-zero entries, columns in order
                            constexpr int SPL = MODE == 5 ? 2 : 1;  // levels per step
                            Cx<T> m6[6];
#pragma unroll
                            for (int e = 0; e < 6; ++e)
                                m6[e] = a.full_table ? cmulp(UM[FLD ? lev / SPL : 0][e], qu)
                                                     : MA[FLD ? lev / SPL : 0][FLD ? j : 0][e];
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
                    }
                    if (HS) {  // row q's sums replace row q - 2's
                        hist_store(hp, U13, U24);
                    } else {
                        push_row<T, UNR>(UH[0][lev][j], UH[1][lev][j], UH[UNR == 2 ? (par + lev) & 1 : 0][lev][j], U13, U24);
                    }
                } else {
                    // y sweep (Eq. sol_dis_2)
                    Cx<T> U14, W14, U23, W23;
                    y_chars<HY>(b, U14, W14, U23, W23);
                    if (need_out) {
                        Cx<T>(&UO)[2] = UH[UNR == 2 ? (par + lev) & 1 : 0][lev][j];
                        y_join<HY>(UO[0], W14, UO[1], W23, o);
                    }
                    push_row<T, UNR>(UH[0][lev][j], UH[1][lev][j], UH[UNR == 2 ? (par + lev) & 1 : 0][lev][j], U14, U23);
                }
                if (need_out) {
                    if (strip_in && out_row_ok) {  // warp-uniform: no cell of this row is a ghost cell
#pragma unroll
                        for (int c = 0; c < 4; ++c) st[j][c] = o[c];
                    } else {
                        const bool keep = per || (out_row_ok && xin[j]);
#pragma unroll
                        for (int c = 0; c < 4; ++c) st[j][c] = keep ? o[c] : Cx<T>{T(0), T(0)};
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < 4; ++c) st[j][c] = Cx<T>{T(0), T(0)};
                }
            }
        }
        if (FT && has_face && (frow_t == FR - 1 || r == r_last - 1)) {
            __syncwarp();
            const int lev = lane / FR, t = lane & (FR - 1);
            const bool half2 = (MODE == 2 || MODE == 5) && (lev & 1);  // a second-order step's second x sweep, a row later
            const RI q = r - frow_t + t - lev - (half2 ? 1 : 0);       // the row that this lane's values belong to
            if (t <= frow_t && q >= r_begin && q < r_end)
                facc[0] = __dadd_rn(facc[0], flux_value(gsm + lane * 8, half2 ? 2.0 * a.flux_unit : 0.5 * a.flux_unit));
            __syncwarp();
        }
        if (STEADY || r >= r_first + 2 * L) {
#pragma unroll
            for (int j = 0; j < P; ++j)
                if (own[j]) store_cell(orow + cell_of<T, P, L>(lane, j) * 8, st[j], a.wide != 0);
        }
        if (!EARLY) refill();
        sl = (sl + 1 == RG::SLOTS) ? 0 : sl + 1;
        orow += row_step;
        frow += row_step;
        return true;
    };
    using Even = std::integral_constant<int, 0>;
    using Odd = std::integral_constant<int, 1>;
    // (FP64 rows are long beside the tests, and a second copy of them costs more than it saves: 13.0 against 13.4 G)
    constexpr bool SPLIT = !IsF64<T>::value;
    const RI steady0 = r_first + 2 * L, steady1 = f_end;
    for (RI r = r_first; r < r_last && !aborted; r += UNR) {
        if (UNR == 1) {
            aborted = !(SPLIT && r >= steady0 && r < steady1 ? do_row(std::true_type{}, Even{}, r) : do_row(std::false_type{}, Even{}, r));
        } else if (SPLIT && r >= steady0 && r + 1 < steady1) {
            aborted = !(do_row(std::true_type{}, Even{}, r) && do_row(std::true_type{}, Odd{}, r + 1));
        } else {
            aborted = !do_row(std::false_type{}, Even{}, r);
            if (!aborted && r + 1 < r_last) aborted = !do_row(std::false_type{}, Odd{}, r + 1);
        }
    }
    if (aborted) {
        // a copy never completed: report, then wait (bounded) for this warp's copies still in flight
        if (lane == 0) atomicOr(a.err, 1u);
#pragma unroll
        for (int s2 = 0; s2 < RG::SLOTS; ++s2)
            if (pending & (1u << s2)) mbar_wait(bar0 + 8 * s2, (phase_bits >> s2) & 1u);
    }
    // release the barriers so the next task of this warp can initialise them again
    __syncwarp();
    if (lane == 0)
#pragma unroll
        for (int s2 = 0; s2 < RG::SLOTS; ++s2) mbar_inval(bar0 + 8 * s2);
    __syncwarp();
    if (has_face) {
#pragma unroll
        for (int s = 0; s < (FT ? 1 : L); ++s) {
            double v = facc[s];
#pragma unroll
            for (int o = FR / 2; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
            if ((lane & (FR - 1)) == 0) a.flux_part[(int64_t)(FT ? lane / FR : s) * a.nsegs * a.nplanes + plane * a.nsegs + seg] = v;
        }
    }
}

// 3-D z sweep + phase: one thread per (x, y) column and z segment; the input is 4x the x-y swept
// state, the table carries 1/8, so the output is the state after the full step.
template <typename T, bool FULL>
__global__ void __launch_bounds__(128) zphase_kernel(const ZArgs a) {
    const int64_t ncol = a.nx * a.ny;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= ncol * a.nsegs) return;
    const int64_t seg = tid / ncol;
    const int64_t col = tid - seg * ncol;
    const int64_t x = col % a.nx;
    const int64_t nz = a.nz;
    const bool per = a.periodic != 0;
    const int64_t z_begin = seg * a.seg_h;
    const int64_t z_end = min(z_begin + a.seg_h, nz);
    const T *in = static_cast<const T *>(a.in);
    T *out = static_cast<T *>(a.out);
    const T *tab = static_cast<const T *>(a.table);
    Cx<T> pu, pd;
    if (!FULL) load_tab(tab + x * 4, pu, pd);
    constexpr bool AHEAD = FULL && !IsF64<T>::value;
    Cx<T> tu, td;
    Cx<T> UA[2] = {{T(0), T(0)}, {T(0), T(0)}}, UB[2] = {{T(0), T(0)}, {T(0), T(0)}};
    for (int64_t z = z_begin - 1; z <= z_end; ++z) {
        Cx<T> s[4];
        const bool ok = per || (z >= 0 && z < nz);
        const int64_t zo = z - 1;
        // The table's entry is asked for a plane ahead, in FP64, which the pipe binds, just before the state: at its use below
        // each plane waited for it in turn (two-pass plan at 200^3 with a full table, us a step at the use, before the state, a
        // plane ahead: FP32 332, 285, 244; fixed point 610, 523, 521; FP64 1159, 1147, 1165).  The per-column table's variant
        // is 2 % slower with the entries held so.
        Cx<T> qu = AHEAD ? tu : pu, qd = AHEAD ? td : pd;
        const int64_t zt = AHEAD ? z : zo;
        if (FULL && zt >= z_begin && zt < z_end) load_tab(tab + (zt * ncol + col) * 4, AHEAD ? tu : qu, AHEAD ? td : qd);
        if (ok) {
            const int64_t zl = per ? pmod(z, nz) : z;
            load_pt(in + (zl * ncol + col) * 8, s);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c) s[c] = {T(0), T(0)};
        }
        Cx<T> U13, W13, U24, W24;
        z_chars<true>(s, U13, W13, U24, W24);
        if (zo >= z_begin && zo < z_end) {
            Cx<T> o[4];
            z_join<true>(UA[0], W13, UA[1], W24, o);
            o[0] = cmulp(o[0], qu);
            o[1] = cmulp(o[1], qu);
            o[2] = cmulp(o[2], qd);
            o[3] = cmulp(o[3], qd);
            store_pt(out + (zo * ncol + col) * 8, o);
        }
        UA[0] = UB[0];
        UA[1] = UB[1];
        UB[0] = U13;
        UB[1] = U24;
    }
}

}  // namespace dirac
