// Small-grid 2-D step: the tile shapes and their instantiations (tile_kernels.cuh).
#include "tile_kernels.cuh"

namespace dirac {

// X(type, warps, rows a warp, steps, second order, field, shape of a plan?, base, per tile): a launch with b tiles on the fullest SM
// takes base + b * per_tile microseconds, both fitted to launches of 40 x 64 to 2048^2 with the face flux (the launches
// overlap by about 1 us more than that).  FP32 and fixed point gain from several steps a launch more than their halo costs;
// FP64 second order, bound by the FP64 pipe, does not.  Shapes that are no plan's run the steps that a plan's do not divide.
#define DIRAC_TILE_SHAPES(X)                                                                                            \
    X(float, 16, 1, 4, false, 0, 1, 4.2, 1.12) X(float, 16, 1, 2, false, 0, 0, 0, 0) X(float, 16, 1, 1, false, 0, 0, 0, 0)       \
    X(float, 8, 4, 4, false, 0, 1, 4.2, 1.68) X(float, 8, 4, 2, false, 0, 0, 0, 0) X(float, 8, 4, 1, false, 0, 0, 0, 0)          \
    X(float, 16, 1, 2, true, 0, 1, 3.1, 1.06) X(float, 16, 1, 1, true, 0, 0, 0, 0)                                            \
    X(float, 8, 4, 2, true, 0, 1, 3.55, 1.57) X(float, 8, 4, 1, true, 0, 0, 0, 0)                                              \
    X(double, 8, 1, 2, false, 0, 1, 3.1, 4.25) X(double, 8, 1, 1, false, 0, 0, 0, 0)                                           \
    X(double, 12, 1, 2, false, 0, 1, 2.2, 8.2) X(double, 12, 1, 1, false, 0, 0, 0, 0)                                         \
    X(double, 16, 1, 2, false, 0, 1, 2.3, 10.7) X(double, 16, 1, 1, false, 0, 0, 0, 0)                                        \
    X(double, 20, 1, 2, false, 0, 1, 2.3, 13.4) X(double, 20, 1, 1, false, 0, 1, 2.4, 7.4)                                   \
    X(double, 24, 1, 2, false, 0, 1, 2.3, 16.0) X(double, 24, 1, 1, false, 0, 0, 0, 0)                                        \
    X(double, 8, 1, 1, true, 0, 1, 3.3, 3.55) X(double, 12, 1, 1, true, 0, 1, 2.0, 6.8) X(double, 16, 1, 1, true, 0, 1, 2.6, 8.6) \
    X(double, 20, 1, 1, true, 0, 1, 2.4, 11.3) X(double, 24, 1, 1, true, 0, 1, 1.8, 13.8)                                     \
    X(long long, 12, 1, 2, false, 0, 1, 2.3, 2.8) X(long long, 12, 1, 1, false, 0, 0, 0, 0)                                   \
    X(long long, 16, 1, 2, false, 0, 1, 2.3, 3.7) X(long long, 16, 1, 1, false, 0, 0, 0, 0)                                   \
    X(long long, 20, 1, 2, false, 0, 1, 2.3, 4.5) X(long long, 20, 1, 1, false, 0, 0, 0, 0)                                   \
    X(long long, 24, 1, 2, false, 0, 1, 2.4, 5.45) X(long long, 24, 1, 1, false, 0, 0, 0, 0)                                  \
    X(long long, 8, 1, 1, true, 0, 1, 3.0, 0.93) X(long long, 12, 1, 1, true, 0, 1, 3.0, 1.73)                              \
    X(long long, 20, 1, 1, true, 0, 1, 2.0, 3.9) X(long long, 24, 1, 1, true, 0, 1, 2.4, 4.33) \
    X(float, 16, 1, 2, false, 1, 1, 2.8, 3.1) X(float, 16, 1, 1, false, 1, 0, 0, 0)                                     \
    X(float, 8, 4, 2, false, 1, 1, 2.7, 3.05) X(float, 8, 4, 1, false, 1, 0, 0, 0)                                      \
    X(float, 16, 1, 1, true, 1, 1, 3.1, 1.78) X(float, 8, 4, 1, true, 1, 1, 3.4, 1.75)                                  \
    X(double, 8, 1, 1, false, 1, 1, 3.0, 5.4) X(double, 12, 1, 1, false, 1, 1, 1.8, 9.8)                                \
    X(double, 16, 1, 1, false, 1, 1, 1.4, 13.2) X(double, 8, 1, 1, true, 1, 1, 3.2, 6.75)                               \
    X(double, 12, 1, 1, true, 1, 1, 1.4, 12.1) X(double, 16, 1, 1, true, 1, 1, 1.6, 15.8)

template <typename T> constexpr int precision_of() { return sizeof(T) == 4 ? 1 : (IsFx<T>::value ? 2 : 0); }

const TileShape *tile_shapes(int *count) {
#define X(T, w, r, k, st, fld, plan, base, per) {precision_of<T>(), w, r, k, st, fld, plan, base, per},
    static const TileShape shapes[] = {DIRAC_TILE_SHAPES(X)};
#undef X
    *count = (int)(sizeof shapes / sizeof shapes[0]);
    return shapes;
}

cudaError_t launch_tile(const SweepArgs &a, const TileShape &t, int steps, int sms, cudaStream_t s) {
#define X(T, w, r, k, st, fld, plan, base, per)                                                                             \
    if (t.precision == precision_of<T>() && t.warps == w && t.rows == r && steps == k && (t.strang != 0) == st && t.field == fld) \
        return a.periodic ? launch_tile_per<T, w, r, k, st, true, fld>(a, sms, s) : launch_tile_per<T, w, r, k, st, false, fld>(a, sms, s);
    DIRAC_TILE_SHAPES(X)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace dirac
