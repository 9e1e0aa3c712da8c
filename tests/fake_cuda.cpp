// A stand-in for the CUDA runtime and the kernel launchers, so that the host runtime (csrc/dirac_api.cu) runs without a
// GPU.  Device memory is numbers never given out twice; a launch is a line that names what the kernel would be given, logged
// when it runs (at once, or when the graph that it was captured into is launched) and checked then: every device range
// that it would touch has to be allocated still.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <map>
#include <string>
#include <vector>

#include "dirac_internal.cuh"

namespace {
using dirac::SweepArgs;
std::map<uintptr_t, size_t> live;  // device allocations
uintptr_t next_addr = (uintptr_t)1 << 44;
size_t live_bytes = 0, limit_bytes = (size_t)1 << 46;
struct Range {
    const void *p;
    size_t bytes;
};
struct Launch {
    std::string line;
    std::vector<Range> touched;
};
std::vector<Launch> *capture = nullptr;  // of the stream being captured
std::string log_text;
int violations = 0, timings = 0;

bool allocated(const Range &r) {
    const uintptr_t a = (uintptr_t)r.p;
    auto it = live.upper_bound(a);
    if (it == live.begin()) return false;
    --it;
    return a + r.bytes <= it->first + it->second;
}
void run(const Launch &l) {
    bool ok = true;
    for (const Range &r : l.touched) ok = ok && (r.bytes == 0 || allocated(r));
    violations += !ok;
    if (!l.line.empty()) log_text += l.line + (ok ? "\n" : " (freed memory)\n");
}
cudaError_t enqueue(std::string line, std::vector<Range> touched) {
    Launch l{std::move(line), std::move(touched)};
    if (capture)
        capture->push_back(l);
    else
        run(l);
    return cudaSuccess;
}
std::string n(long long v) { return " " + std::to_string(v); }
std::string x(double v) {
    char s[32];
    snprintf(s, sizeof s, " %.17g", v);
    return s;
}
// a step launch of any kernel: `parts` flux partials a step or sweep, `sums` of them, entries of `elem` bytes
cudaError_t step(const std::string &what, const SweepArgs &a, int K, int64_t cells, int64_t parts, int sums, int elem) {
    std::string line = what + n(K) + n(a.strip_w) + n(a.nstrips) + n(a.nsegs) + n(a.seg_h) + n(a.full_table) + n(a.periodic) +
                       n(a.ucoef_n ? a.step0 : -1) + x(a.flux_unit);
    std::vector<Range> t = {{a.in, (size_t)cells * 8 * elem}, {a.out, (size_t)cells * 8 * elem},
                            {a.table, (size_t)(a.full_table ? cells : a.nx) * 4 * elem},
                            {a.ucoef, (size_t)a.ucoef_n * 96}};
    if (a.flux_face >= 0) t.push_back({a.flux_part, (size_t)parts * sums * sizeof(double)});
    return enqueue(line, t);
}
}  // namespace

struct CUgraph_st {
    std::vector<Launch> launches;
};
struct CUgraphExec_st {
    std::vector<Launch> launches;
};

extern "C" {
const char *fake_log() { return log_text.c_str(); }
int fake_violations() { return violations; }
void fake_reset() {
    log_text.clear();
    violations = timings = 0;
}
// allocations beyond this many bytes more than are live now fail
void fake_limit(size_t more) { limit_bytes = more == (size_t)-1 ? (size_t)1 << 46 : live_bytes + more; }

cudaError_t cudaMalloc(void **p, size_t bytes) {
    if (live_bytes + bytes > limit_bytes) return cudaErrorMemoryAllocation;
    *p = (void *)next_addr;
    live[next_addr] = bytes;
    live_bytes += bytes;
    next_addr += (bytes + 511) / 512 * 512 + 512;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    auto it = live.find((uintptr_t)p);
    if (it == live.end()) return cudaErrorInvalidValue;
    live_bytes -= it->second;
    live.erase(it);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t bytes, unsigned) {
    *p = calloc(1, bytes);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void **p, size_t bytes) { return cudaHostAlloc(p, bytes, 0); }
cudaError_t cudaFreeHost(void *p) {
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) {
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *, const void *) { return cudaErrorInvalidValue; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorName(cudaError_t) { return "error"; }
const char *cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaEventCreate(cudaEvent_t *e) {
    *e = nullptr;
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
// the first of the tuner's candidates is the fastest
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    *ms = timings++ ? 1e6f : 1e-3f;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    *s = nullptr;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
    capture = new std::vector<Launch>();
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
    *g = new CUgraph_st{*capture};
    delete capture;
    capture = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t g, unsigned long long) {
    *e = new CUgraphExec_st{g->launches};
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
    delete g;
    return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
    delete e;
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
    for (const Launch &l : e->launches) run(l);
    return cudaSuccess;
}
}

namespace dirac {
bool sweep_supported(int fp32, int, int K, int P) { return K == 1 ? P != 3 && P <= 4 : (K == 2 && P == 2) || (fp32 && K <= 4 && P >= 2); }
bool sweep_supported_fx(int, int K, int P) { return K == 1 ? P != 3 && P <= 4 : K == 2 && P == 2; }
bool shift_supported(int S, int P) { return S >= 2 && S <= 4 && P <= 2; }
const TileShape *tile_shapes(int *count) {
    static const TileShape shapes[] = {{1, 8, 4, 4, 0, 0, 1, 4.2, 1.68}, {0, 20, 1, 2, 0, 0, 1, 2.3, 13.4}, {0, 20, 1, 1, 0, 0, 1, 2.4, 7.4},
                                       {0, 16, 1, 1, 0, 1, 1, 1.4, 13.2}, {1, 8, 4, 1, 1, 1, 1, 3.4, 1.75}};
    *count = 5;
    return shapes;
}
static int sums_of(int mode, int K) { return mode == 2 || mode == 5 ? 2 * K : K; }
cudaError_t launch_sweep_f64(const SweepArgs &a, int mode, int K, int P, int, cudaStream_t) {
    return step("f64" + n(mode) + n(P), a, K, a.nx * a.nr * a.nplanes, a.nsegs * a.nplanes, sums_of(mode, K), 8);
}
cudaError_t launch_sweep_f32(const SweepArgs &a, int mode, int K, int P, int, cudaStream_t) {
    return step("f32" + n(mode) + n(P), a, K, a.nx * a.nr * a.nplanes, a.nsegs * a.nplanes, sums_of(mode, K), 4);
}
cudaError_t launch_sweep_fx(const SweepArgs &a, int mode, int K, int P, int, cudaStream_t) {
    return step("fx" + n(mode) + n(P), a, K, a.nx * a.nr * a.nplanes, a.nsegs * a.nplanes, sums_of(mode, K), 8);
}
cudaError_t launch_shift(const SweepArgs &a, int fp32, int S, int P, int, cudaStream_t) {
    return step("shift" + n(S) + n(P), a, 1, a.nx * a.nr, a.nsegs, 1, fp32 ? 4 : 8);
}
cudaError_t launch_tile(const SweepArgs &a, const TileShape &t, int steps, int, cudaStream_t) {
    return step("tile" + n(t.warps) + n(t.rows), a, steps, a.nx * a.nr, a.nr, sums_of(t.strang ? 2 : 0, steps),
                t.precision == 1 ? 4 : 8);
}
cudaError_t launch_fused3d(const SweepArgs &a, int precision, int warps, int steps, int64_t ny, int64_t nz, int64_t, int64_t, int64_t,
                           int64_t, cudaStream_t) {
    return step("fused3d" + n(warps), a, steps, a.nx * ny * nz, a.nsegs, steps, precision == 1 ? 4 : 8);
}
cudaError_t launch_strang_xy(const SweepArgs &a, int precision, int warps, int nh, int64_t ny, int64_t nz, int64_t, int64_t, int64_t,
                             int64_t, const double *fscale, int, int, cudaStream_t) {
    return step("strang_xy" + n(warps) + n(nh) + x(fscale[0]) + x(fscale[1]), a, 1, a.nx * ny * nz, a.nsegs, 2 * nh, precision == 1 ? 4 : 8);
}
cudaError_t launch_strang_z(const void *in, void *out, const void *table, int64_t nx, int64_t ny, int64_t nz, int, int full, const double *,
                            int64_t, int64_t, int64_t, int64_t, int precision, cudaStream_t) {
    const size_t e = precision == 1 ? 4 : 8, c = (size_t)(nx * ny * nz);
    return enqueue("strang_z" + n(full), {{in, c * 8 * e}, {out, c * 8 * e}, {table, (full ? c : (size_t)nx) * 4 * e}});
}
cudaError_t launch_axis(const void *in, void *out, const void *table, int64_t nx, int64_t ny, int64_t nz, int axis, int64_t, int, int full,
                        int phase, int64_t flux_face, double fscale, double *flux_part, const double *, int64_t, int64_t, int precision, int,
                        int blocks, cudaStream_t) {
    const size_t e = precision == 1 ? 4 : 8, c = (size_t)(nx * ny * nz);
    return enqueue("axis" + n(axis) + n(phase) + n(full) + x(fscale), {{in, c * 8 * e}, {out, c * 8 * e}, {table, (full ? c : (size_t)nx) * 4 * e},
                                                           {flux_part, flux_face >= 0 ? blocks * sizeof(double) : 0}});
}
cudaError_t launch_axis_cellfield(const AxisArgs &, int, int, cudaStream_t) { return enqueue("cellfield", {}); }
static cudaError_t zphase(const ZArgs &a, size_t e) {
    const size_t c = (size_t)(a.nx * a.ny * a.nz);
    return enqueue("zphase" + n(a.full_table) + n(a.nsegs), {{a.in, c * 8 * e}, {a.out, c * 8 * e},
                                                             {a.table, (a.full_table ? c : (size_t)a.nx) * 4 * e}});
}
cudaError_t launch_zphase_fx(const ZArgs &a, int, cudaStream_t) { return zphase(a, 8); }
cudaError_t launch_zphase_f32(const ZArgs &a, int, cudaStream_t) { return zphase(a, 4); }
cudaError_t launch_zphase_f64(const ZArgs &a, int, cudaStream_t) { return zphase(a, 8); }
cudaError_t launch_observables(const ObsArgs &, int, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_fx_encode(const double *, long long *, int64_t, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_fx_decode(const long long *, double *, int64_t, int, cudaStream_t) { return cudaSuccess; }
// (not logged: how many launches lie between two folds depends on whether they are replayed)
cudaError_t launch_flux_fold(const FluxFold &f, cudaStream_t) {
    std::vector<Range> parts;
    for (int i = 0; i < f.count; ++i) parts.push_back({f.part + f.off[i], f.n[i] * sizeof(double)});
    return enqueue("", parts);
}
}  // namespace dirac
