// Surrogate network kernels: MLP 3 -> 256 -> 256 -> 256 -> 256 -> 1 (tanh hidden layers, sigmoid
// output) with BF16 weights and FP32 accumulation; forward, backward and Adam.
//
// Rounding points (the CPU gradient oracle mirrors them):
//   layer 1:        z1 = x . bf16(W1)^T + b1 in FP32 (K = 3, CUDA cores)
//   layers 2..4:    z = bf16(h) . bf16(W)^T + b, BF16 tensor-core products (tcgen05), FP32 accumulation
//   output:         z5 = bf16(h4) . bf16(w5) + b5 (FP32 dot), y = sigmoid(z5)
//   backward:       dz5 = 2 (y - t) y (1 - y) / B; dW5 = sum_b dz5 bf16(h4); dh4 = dz5 bf16(w5);
//                   dz = dh (1 - h^2);  dW = bf16(dz)^T . bf16(h_prev) and dh_prev = bf16(dz) . bf16(W)
//                   (tensor cores); db = sum_b dz (FP32); dW1 = dz1^T . x (FP32)
#include <atomic>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "mlp_internal.cuh"

namespace dirac {
namespace mlp {

namespace {

// ---- tcgen05 (5th-generation tensor core) GEMM of the training step.
//
// One CTA of 8 warps computes a 128 x 32 tile of C[m][n] = sum_k A[m][k] B[n][k] (BF16 operands, both with k
// contiguous; FP32 accumulator in 32 columns of tensor memory) and finishes the layer in its epilogue.  The products
// are small (256 x 256 x 256 for a batch of 256), so the time is the operands' latency: every 16-byte piece of a
// K = 64 stage goes to shared memory by cp.async, four stages in flight, so a whole K = 256 is under way at once, and
// 32-column tiles give such a product 16 CTAs.  Operands that a product needs the other way round (the weight
// gradients' dz and h, the data gradients' W) are kept transposed by the kernels that produce them: an accumulator
// row is a lane, so a column's 32 values leave as 64 consecutive bytes.  A launch of a
// 256 x 256 x 256 product takes 8.3 us alone under the profiler, layer epilogue included (before: 33 us and a launch for
// the epilogue); a training step of 256 samples 55 us in its chain of overlapping launches (93 us without the overlap,
// 271 before).
// Shared memory holds the canonical no-swizzle K-major layout (8-row x 16-byte core matrices; K-direction core-matrix
// stride 128 B, 8-row-group stride 256 B; one 16-deep K slab per MMA).  One thread issues tcgen05.mma (M = 128, N = 32,
// K = 16) in ascending k and commits each stage to an mbarrier; every wait is bounded (about one second of the global
// timer) and a timeout sets *err instead of hanging.
constexpr int GM = 128, GN = 32, GK = 64, GSTAGES = 4;
constexpr int A_SLAB = GM * 16 * 2;  // bytes of one 16-deep K slab of the A tile (4 KB)
constexpr int B_SLAB = GN * 16 * 2;  // (1 KB)
constexpr int STAGE_BYTES = 4 * A_SLAB + 4 * B_SLAB;         // 20 KB per K chunk
constexpr int GEMM_SMEM = GSTAGES * STAGE_BYTES + 1024;      // + alignment slack

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t timer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
    const uint64_t t0 = timer_ns();
    for (int it = 0; it < (1 << 24); ++it) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok)
                     : "r"(bar), "r"(parity)
                     : "memory");
        if (ok) return true;
        if (it > 32) __nanosleep(64);
        if ((it & 63) == 63 && timer_ns() - t0 > 1000000000ull) return false;
    }
    return false;
}

// Programmatic dependent launch (the training step's chain of short kernels): a launch may begin while the previous one
// runs; everything the previous kernel writes is touched after chain_wait only, which returns when that kernel has
// finished.  Each kernel lets the next one begin after its own chain_wait, so whatever the kernel before the previous one
// wrote is complete when a kernel starts: the weights (the step's last kernel writes them) may be read before the wait by
// every kernel but the step's first.
__device__ __forceinline__ void chain_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Shared-memory matrix descriptor: no swizzle, K-major; start address, LBO (K-direction core-matrix
// stride) and SBO (8-row-group stride) in 16-byte units, descriptor version 1 (bits 46-47).
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(256 >> 4) << 32) |
           (1ull << 46);
}

// Byte offset of element (row, k) of a K chunk whose 16-deep slabs are `slab` bytes apart.
__device__ __forceinline__ int tile_off(int row, int k, int slab) {
    return (k >> 4) * slab + (row >> 3) * 256 + ((k >> 3) & 1) * 128 + (row & 7) * 16 + (k & 7) * 2;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
    const __nv_bfloat16 lo = __float2bfloat16(a), hi = __float2bfloat16(b);
    return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

// Starts the copies of rows [r0, r0 + ROWS) x k [k0, k0 + 64) of X[r][k] (row pitch ld) into a stage; rows past R are
// zero.  The caller's buffers are readable up to the 64-multiple of k that it asks for.
template <int ROWS>
__device__ __forceinline__ void stage_async(unsigned char *dst, int slab, const __nv_bfloat16 *X, int64_t ld, int r0, int R,
                                            int k0) {
#pragma unroll
    for (int e = threadIdx.x; e < ROWS * (GK / 8); e += 256) {
        const int r = e / (GK / 8), c = e % (GK / 8);
        const uint32_t bytes = r0 + r < R ? 16u : 0u;  // 0: zero fill, nothing read
        const __nv_bfloat16 *src = X + (int64_t)(r0 + r < R ? r0 + r : 0) * ld + k0 + 8 * c;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst + tile_off(r, 8 * c, slab))), "l"(src),
                     "r"(bytes)
                     : "memory");
    }
}

// What a GEMM launch computes.
//   FWD    h = tanh(A . B^T + bias): FP32 h, its BF16 copy and the copy's transpose
//   DGRAD  dz = (A . B^T) (1 - h^2) (h: this layer's activations): FP32 dz, its BF16 copy and the copy's transpose
//   WGRAD  C = A . B^T, FP32
enum { FWD = 0, DGRAD = 1, WGRAD = 2 };
struct GemmArgs {
    const __nv_bfloat16 *A, *B;
    int64_t lda, ldb;
    int M, K;
    float *C;                 // h, dz or the gradient: [M][256]
    __nv_bfloat16 *Cb, *Ct;   // BF16 copy [M][256] and transpose [256][ldt] (FWD, DGRAD); rows past M leave zeros in Ct
    int64_t ldt;
    const float *bias, *h;
    unsigned *err;
};

template <int KIND> __device__ __forceinline__ void gemm_tile(const GemmArgs &g, int m0, int n0) {
    extern __shared__ unsigned char gsm_raw[];
    unsigned char *gsm = reinterpret_cast<unsigned char *>(((uintptr_t)gsm_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t mbar[GSTAGES];
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nchunks = (g.K + GK - 1) / GK;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 32;" ::"r"(smem_addr(&tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
#pragma unroll
        for (int i = 0; i < GSTAGES; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&mbar[i])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    auto load_a = [&](int c) {
        if (c < nchunks) stage_async<GM>(gsm + (c % GSTAGES) * STAGE_BYTES, A_SLAB, g.A, g.lda, m0, g.M, c * GK);
        asm volatile("cp.async.commit_group;" ::: "memory");  // one group per chunk (with its B), empty past the end
    };
    auto load_b = [&](int c) {
        if (c < nchunks)
            stage_async<GN>(gsm + (c % GSTAGES) * STAGE_BYTES + 4 * A_SLAB, B_SLAB, g.B, g.ldb, n0, HID, c * GK);
    };
    // FWD and DGRAD: the weights while the previous kernel still runs
    if (KIND == WGRAD) chain_wait();
#pragma unroll
    for (int c = 0; c < GSTAGES - 1; ++c) load_b(c);
    if (KIND != WGRAD) chain_wait();
#pragma unroll
    for (int c = 0; c < GSTAGES - 1; ++c) load_a(c);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    // instruction descriptor: FP32 accumulator, BF16 A and B, both K-major, N = 32, M = 128
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(GN >> 3) << 17) | ((uint32_t)(GM >> 4) << 24);
    bool ok = true;
    for (int c = 0; c < nchunks && ok; ++c) {
        // chunk c + GSTAGES - 1 goes where chunk c - 1 was: its MMAs have to be done with it
        if (c >= 1 && c + GSTAGES - 1 < nchunks)
            ok = __syncthreads_and(bar_wait(smem_addr(&mbar[(c - 1) % GSTAGES]), (uint32_t)(((c - 1) / GSTAGES) & 1)));
        if (!ok) break;
        load_b(c + GSTAGES - 1);
        load_a(c + GSTAGES - 1);
        asm volatile("cp.async.wait_group %0;" ::"n"(GSTAGES - 1) : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // landed pieces -> the tensor core's view
        __syncthreads();
        if (tid == 0) {
            unsigned char *buf = gsm + (c % GSTAGES) * STAGE_BYTES;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int j = 0; j < GK / 16; ++j) {
                const uint64_t ad = umma_desc(smem_addr(buf + j * A_SLAB));
                const uint64_t bd = umma_desc(smem_addr(buf + 4 * A_SLAB + j * B_SLAB));
                const uint32_t acc = (c > 0 || j > 0) ? 1u : 0u;
                asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                             "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
                             "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                             : "memory");
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_addr(&mbar[c % GSTAGES]))
                         : "memory");
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    // commits complete in order: the last one covers every MMA
    if (ok) ok = __syncthreads_and(bar_wait(smem_addr(&mbar[(nchunks - 1) % GSTAGES]), (uint32_t)(((nchunks - 1) / GSTAGES) & 1)));
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok) {
        // warps w and w + 4 read the same 32 accumulator rows, 16 columns each
        const int m = m0 + (warp & 3) * 32 + lane, nc = n0 + (warp >> 2) * 16;
        uint32_t r[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
              "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * 16))
            : "memory");
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        const bool in = m < g.M;
        float v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
        if (KIND == FWD) {
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = tanhf(v[j] + g.bias[nc + j]);
        } else if (KIND == DGRAD && in) {
            const float4 *hp = reinterpret_cast<const float4 *>(g.h + (int64_t)m * HID + nc);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 y = hp[j];
                v[4 * j + 0] = v[4 * j + 0] * (1.f - y.x * y.x);
                v[4 * j + 1] = v[4 * j + 1] * (1.f - y.y * y.y);
                v[4 * j + 2] = v[4 * j + 2] * (1.f - y.z * y.z);
                v[4 * j + 3] = v[4 * j + 3] * (1.f - y.w * y.w);
            }
        }
        if (KIND == WGRAD) {
            // the gradient's place in the parameter vector is a multiple of 16 bytes for W2-W4
            float4 *cp = reinterpret_cast<float4 *>(g.C + (int64_t)m * HID + nc);
#pragma unroll
            for (int j = 0; j < 4; ++j) cp[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        } else {
            uint32_t pk[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) pk[j] = in ? pack_bf16x2(v[2 * j], v[2 * j + 1]) : 0u;
            if (in) {
                float4 *cp = reinterpret_cast<float4 *>(g.C + (int64_t)m * HID + nc);
#pragma unroll
                for (int j = 0; j < 4; ++j) cp[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                uint4 *bp = reinterpret_cast<uint4 *>(g.Cb + (int64_t)m * HID + nc);
                bp[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                bp[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
            }
#pragma unroll
            for (int j = 0; j < 16; ++j)
                g.Ct[(int64_t)(nc + j) * g.ldt + m] = __ushort_as_bfloat16((unsigned short)(pk[j / 2] >> (16 * (j & 1))));
        }
    } else if (lane == 0) {
        atomicOr(g.err, 1u);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 32;" ::"r"(tmem) : "memory");
}

template <int KIND> __global__ void __launch_bounds__(256) layer_gemm_kernel(const GemmArgs g) {
    gemm_tile<KIND>(g, blockIdx.y * GM, blockIdx.x * GN);
}

// A training batch: sample b is row idx[b] of X and T (idx null: row b).
struct BatchIn {
    const float *X, *T;
    const int *idx;
    int B;
    __device__ __forceinline__ int row(int b) const { return idx ? idx[b] : b; }
};

// z1 = x . bf16(W1)^T + b1, h1 = tanh(z1) (x is 3 FP32, W1 [256][3] BF16): h1, its BF16 copy and the copy's transpose
// (zeros for the samples that pad the batch to a multiple of 128).  A block of 256 threads takes 32 samples x 32 units.
__global__ void __launch_bounds__(256) layer1_fwd_kernel(const BatchIn in, const __nv_bfloat16 *W1, const float *b1, float *h,
                                                         __nv_bfloat16 *hb, __nv_bfloat16 *ht, int64_t ldt) {
    __shared__ __nv_bfloat16 tr[32][34];
    chain_wait();
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, b0 = blockIdx.x * 32, j0 = blockIdx.y * 32;
    const int j = j0 + tx;
#pragma unroll
    for (int i = ty; i < 32; i += 8) {
        const int b = b0 + i;
        __nv_bfloat16 o = __float2bfloat16(0.f);
        if (b < in.B) {
            const float *x = in.X + (int64_t)in.row(b) * 3;
            float z = b1[j];
            z = fmaf(x[0], __bfloat162float(W1[j * 3 + 0]), z);
            z = fmaf(x[1], __bfloat162float(W1[j * 3 + 1]), z);
            z = fmaf(x[2], __bfloat162float(W1[j * 3 + 2]), z);
            const float y = tanhf(z);
            h[(int64_t)b * HID + j] = y;
            o = __float2bfloat16(y);
            hb[(int64_t)b * HID + j] = o;
        }
        tr[i][tx] = o;
    }
    __syncthreads();
#pragma unroll
    for (int i = ty; i < 32; i += 8) ht[(int64_t)(j0 + i) * ldt + b0 + tx] = tr[tx][i];
}

// The output layer both ways, one warp per sample: y = sigmoid(bf16(h4) . bf16(w5) + b5); dz5 = 2 (y - t) y (1 - y) / B and
// the squared error; the last hidden layer's dz = dz5 w5 (1 - h4^2), its BF16 copy and the copy's transpose (the 16 samples
// of a block through shared memory; zeros for the samples that pad the batch).  Everything a sample needs is loaded before
// the first sum.
constexpr int OUT_B = 16;
__global__ void __launch_bounds__(32 * OUT_B) out_layer_kernel(const BatchIn in, const __nv_bfloat16 *h4b, const float *h4,
                                                               const __nv_bfloat16 *w5, const float *b5, float *y, float *dz5,
                                                               float *sqerr, float *dz, __nv_bfloat16 *dzb,
                                                               __nv_bfloat16 *dzt, int64_t ldt) {
    __shared__ __nv_bfloat16 tr[OUT_B][HID + 2];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int b = blockIdx.x * OUT_B + w;
    constexpr int NJ = HID / 32;
    float wj[NJ], hj[NJ], aj[NJ];
#pragma unroll
    for (int i = 0; i < NJ; ++i) wj[i] = __bfloat162float(w5[lane + 32 * i]);
    const float t = b < in.B ? in.T[in.row(b)] : 0.f, b5v = b5[0];
    chain_wait();
    if (b < in.B) {
#pragma unroll
        for (int i = 0; i < NJ; ++i) {
            hj[i] = __bfloat162float(h4b[(int64_t)b * HID + lane + 32 * i]);
            aj[i] = h4[(int64_t)b * HID + lane + 32 * i];
        }
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < NJ; ++i) s = fmaf(hj[i], wj[i], s);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const float yb = 1.f / (1.f + expf(-(s + b5v)));
        const float d = yb - t;
        const float g5 = 2.f * d * yb * (1.f - yb) / (float)in.B;
        if (lane == 0) {
            y[b] = yb;
            dz5[b] = g5;
            sqerr[b] = d * d;
        }
#pragma unroll
        for (int i = 0; i < NJ; ++i) {
            const int j = lane + 32 * i;
            const float g = g5 * wj[i];
            const float v = g * (1.f - aj[i] * aj[i]);
            dz[(int64_t)b * HID + j] = v;
            const __nv_bfloat16 o = __float2bfloat16(v);
            dzb[(int64_t)b * HID + j] = o;
            tr[w][j] = o;
        }
    } else {
#pragma unroll
        for (int i = 0; i < NJ; ++i) tr[w][lane + 32 * i] = __float2bfloat16(0.f);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < HID * OUT_B; e += 32 * OUT_B)
        dzt[(int64_t)(e / OUT_B) * ldt + blockIdx.x * OUT_B + e % OUT_B] = tr[e % OUT_B][e / OUT_B];
}

// Sums over the batch for 32 columns, a block of 256 threads: thread (w, column) adds the samples b = 32 w + l (mod 256) into
// one partial for each l = 0..31, those by a tree (l with l + 16, + 8, ...), and the eight w in order.  Consecutive lanes
// read consecutive columns.
template <typename F> __device__ __forceinline__ void batch_sums(int B, F term, float *to, int stride, int columns) {
    __shared__ float part[8][33];
    const int c = threadIdx.x & 31, w = threadIdx.x >> 5;
    float s[32];
#pragma unroll
    for (int l = 0; l < 32; ++l) s[l] = 0.f;
    for (int b0 = 32 * w; b0 < B; b0 += 256)
#pragma unroll
        for (int l = 0; l < 32; ++l)
            if (b0 + l < B && c < columns) s[l] += term(b0 + l, c);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int l = 0; l < o; ++l) s[l] = s[l] + s[l + o];
    part[w][c] = s[0];
    __syncthreads();
    if (w == 0 && c < columns) {
        float v = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) v += part[i][c];
        to[c * stride] = v;
    }
}

// The gradients, one launch: blocks [0, 48) the three hidden weight matrices (16 tiles each), then 32 columns each of the
// sums over the batch: db of the four hidden layers, dW1 = dz1^T x, dW5 = sum_b dz5 bf16(h4), db5 = sum_b dz5.
struct GradArgs {
    GemmArgs w[3];             // dW2, dW3, dW4
    const float *dz[4], *dz5;  // hidden layers' dz [B][256]
    const __nv_bfloat16 *h4b;
    float *gb[4], *gW1, *gW5, *gb5;
    BatchIn in;
};
constexpr int kGradTiles = 3 * (HID / GM) * (HID / GN), kColumnGroups = HID / 32;
constexpr int kGradSums = (4 + 3 + 1) * kColumnGroups + 1;
__global__ void __launch_bounds__(256) grad_kernel(const __grid_constant__ GradArgs a) {
    if (blockIdx.x < kGradTiles) {
        const int per = kGradTiles / 3, t = blockIdx.x % per;
        gemm_tile<WGRAD>(a.w[blockIdx.x / per], (t / (HID / GN)) * GM, (t % (HID / GN)) * GN);
        return;
    }
    chain_wait();
    const int q = blockIdx.x - kGradTiles, what = q / kColumnGroups, j0 = (q % kColumnGroups) * 32, B = a.in.B;
    if (what < 4) {
        const float *dz = a.dz[what] + j0;
        batch_sums(B, [&](int b, int c) { return dz[(int64_t)b * HID + c]; }, a.gb[what] + j0, 1, 32);
    } else if (what < 7) {
        const float *dz = a.dz[0] + j0;
        const int i = what - 4;
        batch_sums(B, [&](int b, int c) { return dz[(int64_t)b * HID + c] * a.in.X[(int64_t)a.in.row(b) * 3 + i]; },
                   a.gW1 + j0 * 3 + i, 3, 32);
    } else if (what == 7) {
        const __nv_bfloat16 *h = a.h4b + j0;
        batch_sums(B, [&](int b, int c) { return a.dz5[b] * __bfloat162float(h[(int64_t)b * HID + c]); }, a.gW5 + j0, 1, 32);
    } else {
        batch_sums(B, [&](int b, int) { return a.dz5[b] * 1.f; }, a.gb5, 1, 1);
    }
}

// One Adam step's scalars: the learning rate and the moments' bias corrections.
struct AdamStep {
    float lr, c1, c2;
};
// Adam on the FP32 master parameter i (UPDATE), and its BF16 copy.
template <bool UPDATE>
__device__ __forceinline__ __nv_bfloat16 adam_one(float *p, const float *g, float *m, float *v, __nv_bfloat16 *pb, int64_t i,
                                                  AdamStep st) {
    float np = p[i];
    if (UPDATE) {
        const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float upd = st.lr * (mi / st.c1) / (sqrtf(vi / st.c2) + eps);
        np = np - upd;
        p[i] = np;
    }
    const __nv_bfloat16 o = __float2bfloat16(np);
    pb[i] = o;
    return o;
}
// Blocks [0, 192): 32 x 32 tiles of W2-W4, whose BF16 copy is kept transposed too (the data gradients' operand); then the
// other parameters, 256 to a block.
constexpr int kAdamTiles = 3 * (HID / 32) * (HID / 32);
struct ParamArgs {
    float *p;
    const float *g;
    float *m, *v;
    __nv_bfloat16 *pb, *wt;  // wt: [3][256][256], wt[l][k][j] = bf16(W_{l+2}[j][k])
    int64_t off_w[5];
    int64_t n;
};
template <bool UPDATE> __global__ void __launch_bounds__(256) param_kernel(const __grid_constant__ ParamArgs a, AdamStep st) {
    chain_wait();
    if (blockIdx.x < kAdamTiles) {
        __shared__ __nv_bfloat16 tr[32][34];
        const int per = kAdamTiles / 3, l = blockIdx.x / per, t = blockIdx.x % per;
        const int j0 = (t / (HID / 32)) * 32, k0 = (t % (HID / 32)) * 32;
        const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
        for (int i = ty; i < 32; i += 8)
            tr[i][tx] = adam_one<UPDATE>(a.p, a.g, a.m, a.v, a.pb, a.off_w[l + 1] + (int64_t)(j0 + i) * HID + k0 + tx, st);
        __syncthreads();
#pragma unroll
        for (int i = ty; i < 32; i += 8) a.wt[(int64_t)l * HID * HID + (int64_t)(k0 + i) * HID + j0 + tx] = tr[tx][i];
        return;
    }
    // W1 and b1, then b2, b3, b4 (each after its matrix), w5 and b5
    int64_t e = (int64_t)(blockIdx.x - kAdamTiles) * 256 + threadIdx.x;
    const int64_t first = a.off_w[1], mat = (int64_t)HID * HID;
    if (e >= first) {
        const int64_t r = e - first;
        e = r < 3 * HID ? a.off_w[1 + r / HID] + mat + r % HID : a.off_w[4] + (r - 3 * HID);
    }
    if (e < a.n) adam_one<UPDATE>(a.p, a.g, a.m, a.v, a.pb, e, st);
}

inline int nblk(int64_t n, int t) { return (int)((n + t - 1) / t); }

// ---- Inference: the whole network for 128 queries per CTA in one launch.
//
// The weights of layers 2-4 are first packed into the canonical no-swizzle K-major layout the MMA reads
// (the layout `stage_async` builds: B(k, n) = W[n][k], 256 rows n), so each layer's 128 KB operand reaches shared
// memory as bulk copies (cp.async.bulk, completion counted on an mbarrier), issued as soon as the previous
// layer's MMAs have read the buffer and overlapping that layer's epilogue.  Layer 1 (K = 3) runs on the CUDA
// cores and writes bf16(h1) straight into the A operand (128 queries x 256); each hidden layer is 16
// tcgen05.mma (M = 128, N = 256, K = 16, BF16 -> FP32) into 256 TMEM columns.  The epilogue runs on NW warps
// (16 by default): the NW / 4 warps w, w + 4, ... read the same 32 TMEM lanes (queries 32 (w % 4)..), each a
// block of 256 / (NW / 4) columns; they add the bias, take tanh and write bf16(h) over the A operand (16
// warps ran 99 us against 116 for 8 on 65,536 queries).  The output layer then sums bf16(h4) bf16(w5)
// per query in out_layer_kernel's order (32 strided partial sums, then its shuffle tree), so every rounding
// point is the training step's.  Every wait is bounded; a timeout sets *err.
constexpr int IQ = 128;                          // queries per CTA (the MMA's M)
constexpr int IW_SLAB = HID * 16 * 2;            // one 16-deep K slab of a 256-row weight operand (8 KB)
constexpr int IH_SLAB = IQ * 16 * 2;             // one 16-deep K slab of the activations (4 KB)
constexpr int IW_BYTES = (HID / 16) * IW_SLAB;   // 128 KB per layer
constexpr int IH_BYTES = (HID / 16) * IH_SLAB;   // 64 KB
constexpr int INFER_SMEM = IH_BYTES + IW_BYTES + 1024;
static_assert(3 * (int64_t)IW_BYTES == WPACK_BYTES, "packed weight size");

// pack[l][tile_off(n, k)] = W_{l+2}[n][k]: one thread per 8 consecutive k of one row.
__global__ void pack_weights_kernel(const __nv_bfloat16 *wb, int64_t off2, int64_t off3, int64_t off4,
                                    unsigned char *pack) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= 3 * HID * (HID / 8)) return;
    const int l = (int)(e / (HID * (HID / 8))), n = (int)((e / (HID / 8)) % HID), k8 = (int)(e % (HID / 8)) * 8;
    const int64_t off = l == 0 ? off2 : (l == 1 ? off3 : off4);
    *reinterpret_cast<uint4 *>(pack + (int64_t)l * IW_BYTES + tile_off(n, k8, IW_SLAB)) =
        *reinterpret_cast<const uint4 *>(wb + off + (int64_t)n * HID + k8);
}

__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// One layer's packed weights into the B buffer: four 32 KB copies counted on `bar`.  `extra` bytes more are
// announced than the copies deliver when a test asks for a stalled wait (the phase then never completes).
__device__ __forceinline__ void load_layer_weights(uint32_t ws, const unsigned char *src, uint32_t bar, uint32_t extra) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"((uint32_t)IW_BYTES + extra)
                 : "memory");
#pragma unroll
    for (int c = 0; c < 4; ++c) bulk_copy(ws + c * (IW_BYTES / 4), src + c * (IW_BYTES / 4), IW_BYTES / 4, bar);
}


template <int NW>
__global__ void __launch_bounds__(32 * NW, 1) mlp_infer_kernel(const float *x, const __nv_bfloat16 *W1, const float *b1,
                                                           const unsigned char *pack, const float *b2, const float *b3,
                                                           const float *b4, const __nv_bfloat16 *w5, const float *b5,
                                                           float *y, int Bn, unsigned *err, int inject_stall) {
    extern __shared__ unsigned char ism_raw[];
    unsigned char *hs = reinterpret_cast<unsigned char *>(((uintptr_t)ism_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *wsm = hs + IH_BYTES;
    __shared__ __align__(8) uint64_t bars[2];  // [0]: a layer's weights have landed, [1]: its MMAs are done
    __shared__ uint32_t tmem_slot;
    __shared__ int issued;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int row = (warp & 3) * 32 + lane;  // query within the tile = TMEM lane
    constexpr int NCOL = HID / (NW / 4);  // columns per thread: the NW / 4 warps of a lane group split them
    const int cbase = (warp >> 2) * NCOL;
    const int q = blockIdx.x * IQ + row;
    const uint32_t wbar = smem_addr(&bars[0]), mbar = smem_addr(&bars[1]), ws = smem_addr(wsm);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(smem_addr(&tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(wbar) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // failure-detection test hook: the first CTA's first weight wait runs out
        load_layer_weights(ws, pack, wbar, (inject_stall && blockIdx.x == 0) ? 16u : 0u);
    }
    // layer 1 on the CUDA cores (layer1_fwd_kernel's arithmetic): this thread's NCOL columns of its query
    float x0 = 0.f, x1 = 0.f, x2 = 0.f;
    if (q < Bn) {
        x0 = x[(int64_t)q * 3 + 0];
        x1 = x[(int64_t)q * 3 + 1];
        x2 = x[(int64_t)q * 3 + 2];
    }
    for (int j0 = cbase; j0 < cbase + NCOL; j0 += 8) {
        uint32_t pk[4];
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            float h[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int j = j0 + i + u;
                float z = b1[j];
                z = fmaf(x0, __bfloat162float(W1[j * 3 + 0]), z);
                z = fmaf(x1, __bfloat162float(W1[j * 3 + 1]), z);
                z = fmaf(x2, __bfloat162float(W1[j * 3 + 2]), z);
                h[u] = tanhf(z);
            }
            pk[i / 2] = pack_bf16x2(h[0], h[1]);
        }
        *reinterpret_cast<uint4 *>(hs + tile_off(row, j0, IH_SLAB)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // activations -> the tensor core's view
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    // instruction descriptor: FP32 accumulator, BF16 A and B, both K-major, N = 256, M = 128
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(HID >> 3) << 17) | ((uint32_t)(IQ >> 4) << 24);
    // Every weight copy is waited for (bounded) before the MMAs that read it, and the next one is issued only
    // after those MMAs completed, so no copy is in flight wherever the loop stops early.
    bool ok = true;
    for (int L = 0; L < 3 && ok; ++L) {
        if (tid == 0) {
            issued = 0;
            if (bar_wait(wbar, (uint32_t)(L & 1))) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int j = 0; j < HID / 16; ++j) {
                    const uint64_t ad = umma_desc(smem_addr(hs + j * IH_SLAB));
                    const uint64_t bd = umma_desc(ws + j * IW_SLAB);
                    const uint32_t acc = j > 0 ? 1u : 0u;
                    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
                                 "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                                 : "memory");
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                             : "memory");
                issued = 1;
            }
        }
        __syncthreads();
        ok = __syncthreads_and(issued && bar_wait(mbar, (uint32_t)(L & 1)));
        if (!ok) break;
        // the MMAs have read both operands: the next layer's weights can land while this epilogue runs
        if (tid == 0 && L < 2) {
            load_layer_weights(ws, pack + (int64_t)(L + 1) * IW_BYTES, wbar, 0u);
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const float *bias = L == 0 ? b2 : (L == 1 ? b3 : b4);
#pragma unroll 1
        for (int c0 = cbase; c0 < cbase + NCOL; c0 += 32) {
            uint32_t r[32];
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                  "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                  "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
                  "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
                  "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                : "r"(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0)
                : "memory");
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int i = 0; i < 32; i += 8) {
                uint32_t pk[4];
#pragma unroll
                for (int u = 0; u < 8; u += 2)
                    pk[u / 2] = pack_bf16x2(tanhf(__uint_as_float(r[i + u]) + bias[c0 + i + u]),
                                            tanhf(__uint_as_float(r[i + u + 1]) + bias[c0 + i + u + 1]));
                *reinterpret_cast<uint4 *>(hs + tile_off(row, c0 + i, IH_SLAB)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    if (ok && warp < 4 && q < Bn) {
        // output layer in out_layer_kernel's order: partial sum l takes columns l, l + 32, ..., then the xor tree
        float s[32];
#pragma unroll
        for (int l = 0; l < 32; ++l) s[l] = 0.f;
#pragma unroll
        for (int t = 0; t < HID / 32; ++t)
#pragma unroll
            for (int l8 = 0; l8 < 32; l8 += 8) {
                const uint4 v = *reinterpret_cast<const uint4 *>(hs + tile_off(row, 32 * t + l8, IH_SLAB));
                const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const __nv_bfloat16 h = __ushort_as_bfloat16((unsigned short)(w[u / 2] >> (16 * (u & 1))));
                    s[l8 + u] = fmaf(__bfloat162float(h), __bfloat162float(w5[32 * t + l8 + u]), s[l8 + u]);
                }
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int l = 0; l < o; ++l) s[l] = s[l] + s[l + o];
        y[q] = 1.f / (1.f + expf(-(s[0] + b5[0])));
    }
    if (!ok && tid == 0) atomicOr(err, 1u);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem) : "memory");
}

// Inference of small calls: 32 queries per CTA, so that up to 32 x 152 of them spread over the chip (a CTA of 128 queries
// spends its time in tanh: 4 x 64 per thread; here 4 x 16).  The MMA's M stays 128: the 32 queries stand four times in the
// A operand, so each of the four 32-lane groups of the accumulator holds all of them and the 16 warps take 16 columns
// each from the group they can read.  Rows are independent in the product and every query's arithmetic is that of
// mlp_infer_kernel, so the predictions are the same bits.  x, y and the timeout flag may be pinned host memory (a call
// of this size is shorter than its copies).  Measured end to end, with the copies it does without: 4096 queries a call
// 67 -> 39 us, one query 54 -> 27.
constexpr int SQ = 32;
__global__ void __launch_bounds__(512, 1) mlp_infer_small_kernel(const float *x, const __nv_bfloat16 *W1, const float *b1,
                                                                 const unsigned char *pack, const float *b2, const float *b3,
                                                                 const float *b4, const __nv_bfloat16 *w5, const float *b5,
                                                                 float *y, int Bn, unsigned *err, int inject_stall) {
    extern __shared__ unsigned char ism_raw[];
    unsigned char *hs = reinterpret_cast<unsigned char *>(((uintptr_t)ism_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *wsm = hs + IH_BYTES;
    __shared__ __align__(8) uint64_t bars[2];  // [0]: a layer's weights have landed, [1]: its MMAs are done
    __shared__ uint32_t tmem_slot;
    __shared__ int issued;
    __shared__ float part[32][SQ + 1];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int NCOL = HID / 16;  // columns per warp
    const int c0 = warp * NCOL;
    const int q = blockIdx.x * SQ + lane;
    const uint32_t wbar = smem_addr(&bars[0]), mbar = smem_addr(&bars[1]), ws = smem_addr(wsm);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(smem_addr(&tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(wbar) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // failure-detection test hook: the first CTA's first weight wait runs out
        load_layer_weights(ws, pack, wbar, (inject_stall && blockIdx.x == 0) ? 16u : 0u);
    }
    // bf16 values of this warp's columns [c, c + 8) of the lane's query into its four places in the A operand
    auto put8 = [&](int c, const uint32_t pk[4]) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
            *reinterpret_cast<uint4 *>(hs + tile_off(r * 32 + lane, c, IH_SLAB)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    };
    float x0 = 0.f, x1 = 0.f, x2 = 0.f;
    if (q < Bn) {
        x0 = x[(int64_t)q * 3 + 0];
        x1 = x[(int64_t)q * 3 + 1];
        x2 = x[(int64_t)q * 3 + 2];
    }
#pragma unroll
    for (int j0 = 0; j0 < NCOL; j0 += 8) {
        uint32_t pk[4];
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            float h[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int j = c0 + j0 + i + u;
                float z = b1[j];
                z = fmaf(x0, __bfloat162float(W1[j * 3 + 0]), z);
                z = fmaf(x1, __bfloat162float(W1[j * 3 + 1]), z);
                z = fmaf(x2, __bfloat162float(W1[j * 3 + 2]), z);
                h[u] = tanhf(z);
            }
            pk[i / 2] = pack_bf16x2(h[0], h[1]);
        }
        put8(c0 + j0, pk);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // activations -> the tensor core's view
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(HID >> 3) << 17) | ((uint32_t)(IQ >> 4) << 24);
    // Every weight copy is waited for (bounded) before the MMAs that read it, and the next one is issued only
    // after those MMAs completed, so no copy is in flight wherever the loop stops early.
    bool ok = true;
    for (int L = 0; L < 3 && ok; ++L) {
        if (tid == 0) {
            issued = 0;
            if (bar_wait(wbar, (uint32_t)(L & 1))) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int j = 0; j < HID / 16; ++j) {
                    const uint64_t ad = umma_desc(smem_addr(hs + j * IH_SLAB));
                    const uint64_t bd = umma_desc(ws + j * IW_SLAB);
                    const uint32_t acc = j > 0 ? 1u : 0u;
                    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
                                 "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                                 : "memory");
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                             : "memory");
                issued = 1;
            }
        }
        __syncthreads();
        ok = __syncthreads_and(issued && bar_wait(mbar, (uint32_t)(L & 1)));
        if (!ok) break;
        // the MMAs have read both operands: the next layer's weights can land while this epilogue runs
        if (tid == 0 && L < 2) load_layer_weights(ws, pack + (int64_t)(L + 1) * IW_BYTES, wbar, 0u);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const float *bias = L == 0 ? b2 : (L == 1 ? b3 : b4);
        uint32_t r[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
              "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0)
            : "memory");
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int i = 0; i < NCOL; i += 8) {
            uint32_t pk[4];
#pragma unroll
            for (int u = 0; u < 8; u += 2)
                pk[u / 2] = pack_bf16x2(tanhf(__uint_as_float(r[i + u]) + bias[c0 + i + u]),
                                        tanhf(__uint_as_float(r[i + u + 1]) + bias[c0 + i + u + 1]));
            put8(c0 + i, pk);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    if (ok) {
        // output layer: partial sum l takes columns l, l + 32, ... (two partial sums per warp), then the xor tree
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int l = 2 * warp + u;
            float s = 0.f;
#pragma unroll
            for (int t = 0; t < HID / 32; ++t) {
                const __nv_bfloat16 h = *reinterpret_cast<const __nv_bfloat16 *>(hs + tile_off(lane, 32 * t + l, IH_SLAB));
                s = fmaf(__bfloat162float(h), __bfloat162float(w5[32 * t + l]), s);
            }
            part[l][lane] = s;
        }
        __syncthreads();
        if (warp == 0 && q < Bn) {
            float s[32];
#pragma unroll
            for (int l = 0; l < 32; ++l) s[l] = part[l][lane];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int l = 0; l < o; ++l) s[l] = s[l] + s[l + o];
            y[q] = 1.f / (1.f + expf(-(s[0] + b5[0])));
        }
    }
    if (!ok && tid == 0) *reinterpret_cast<volatile unsigned *>(err) = 1u;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem) : "memory");
}

}  // namespace

cudaError_t pack_weights(const Net &n, cudaStream_t s) {
    if ((n.off_w[1] | n.off_w[2] | n.off_w[3]) & 7) return cudaErrorInvalidValue;  // 16-byte rows for the packing
    pack_weights_kernel<<<nblk(3 * HID * (HID / 8), 256), 256, 0, s>>>(n.wb, n.off_w[1], n.off_w[2], n.off_w[3], n.wpack);
    return cudaGetLastError();
}

namespace {
// Per device: > 48 KB of dynamic shared memory opted in once.
template <typename K> cudaError_t optin(K *kernel, int smem, std::atomic<unsigned long long> &done) {
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = dev < 64 ? (1ull << dev) : 0ull;
    if (bit && (done.load(std::memory_order_relaxed) & bit)) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess && bit) done.fetch_or(bit, std::memory_order_relaxed);
    return e;
}
}  // namespace

cudaError_t infer(const Net &n, const float *x, float *y, unsigned *err, int Bn, cudaStream_t s, int inject_stall) {
    if (Bn <= 0) return cudaSuccess;
    if (Bn <= SMALL_INFER) {
        static std::atomic<unsigned long long> done{0};
        cudaError_t e = optin(mlp_infer_small_kernel, INFER_SMEM, done);
        if (e != cudaSuccess) return e;
        mlp_infer_small_kernel<<<nblk(Bn, SQ), 512, INFER_SMEM, s>>>(x, n.wb + n.off_w[0], n.p + n.off_b[0], n.wpack,
                                                                     n.p + n.off_b[1], n.p + n.off_b[2], n.p + n.off_b[3],
                                                                     n.wb + n.off_w[4], n.p + n.off_b[4], y, Bn, err,
                                                                     inject_stall);
        return cudaGetLastError();
    }
    constexpr int NW = 16;
    static std::atomic<unsigned long long> done{0};
    cudaError_t e = optin(mlp_infer_kernel<NW>, INFER_SMEM, done);
    if (e != cudaSuccess) return e;
    mlp_infer_kernel<NW><<<nblk(Bn, IQ), 32 * NW, INFER_SMEM, s>>>(x, n.wb + n.off_w[0], n.p + n.off_b[0], n.wpack,
                                                                   n.p + n.off_b[1], n.p + n.off_b[2], n.p + n.off_b[3],
                                                                   n.wb + n.off_w[4], n.p + n.off_b[4], y, Bn, err,
                                                                   inject_stall);
    return cudaGetLastError();
}

namespace {
// Launches a kernel of the chain: it may begin while its predecessor in the stream runs (see chain_wait).
template <typename... KA, typename... A>
cudaError_t launch_chain(void (*kernel)(KA...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, args...);
}
template <int KIND> cudaError_t launch_gemm(const GemmArgs &g, cudaStream_t s) {
    static std::atomic<unsigned long long> done{0};
    cudaError_t e = optin(layer_gemm_kernel<KIND>, GEMM_SMEM, done);
    if (e != cudaSuccess) return e;
    return launch_chain(layer_gemm_kernel<KIND>, dim3(HID / GN, nblk(g.M, GM)), dim3(256), GEMM_SMEM, s, g);
}
}  // namespace

// Forward and backward pass of a batch in nine launches: layer 1, three hidden layers, the output layer both ways, three
// data gradients, all weight gradients.  Gradients of mean((y - t)^2) into g (same layout as the parameters).
cudaError_t gradients(const Net &n, const Acts &a, const float *X, const float *T, const int *idx, float *g, int Bn,
                      cudaStream_t s) {
    const BatchIn in{X, T, idx, Bn};
    const int pad = nblk(Bn, GM) * GM;
    cudaError_t e = launch_chain(layer1_fwd_kernel, dim3(pad / 32, HID / 32), dim3(256), 0, s, in, n.wb + n.off_w[0],
                                 n.p + n.off_b[0], a.h[0], a.hb[0], a.ht[0], a.ldt);
    GemmArgs q{};
    q.err = n.err;
    q.lda = q.ldb = HID;
    q.M = Bn;
    q.K = HID;
    q.ldt = a.ldt;
    for (int l = 1; l < 4 && e == cudaSuccess; ++l) {
        // z_l[b][j] = sum_k bf16(h_{l-1})[b][k] bf16(W_l)[j][k]
        q.A = a.hb[l - 1];
        q.B = n.wb + n.off_w[l];
        q.bias = n.p + n.off_b[l];
        q.C = a.h[l];
        q.Cb = a.hb[l];
        q.Ct = a.ht[l];
        e = launch_gemm<FWD>(q, s);
    }
    if (e != cudaSuccess) return e;
    e = launch_chain(out_layer_kernel, dim3(pad / OUT_B), dim3(32 * OUT_B), 0, s, in, a.hb[3], a.h[3], n.wb + n.off_w[4],
                     n.p + n.off_b[4], a.y, a.dz5, a.sqerr, a.dz[3], a.dzb[3], a.dzt[3], a.ldt);
    for (int l = 3; l >= 1 && e == cudaSuccess; --l) {
        // dh_{l-1}[b][k] = sum_j bf16(dz_l)[b][j] bf16(W_l)[j][k]
        q.A = a.dzb[l];
        q.B = n.wt + (int64_t)(l - 1) * HID * HID;
        q.h = a.h[l - 1];
        q.C = a.dz[l - 1];
        q.Cb = a.dzb[l - 1];
        q.Ct = a.dzt[l - 1];
        e = launch_gemm<DGRAD>(q, s);
    }
    if (e != cudaSuccess) return e;
    GradArgs r{};
    for (int l = 1; l < 4; ++l) {
        // dW_l[j][k] = sum_b bf16(dz_l)[b][j] bf16(h_{l-1})[b][k]
        GemmArgs &w = r.w[l - 1];
        w.A = a.dzt[l];
        w.B = a.ht[l - 1];
        w.lda = w.ldb = a.ldt;
        w.M = HID;
        w.K = Bn;
        w.C = g + n.off_w[l];
        w.err = n.err;
    }
    for (int l = 0; l < 4; ++l) {
        r.dz[l] = a.dz[l];
        r.gb[l] = g + n.off_b[l];
    }
    r.dz5 = a.dz5;
    r.h4b = a.hb[3];
    r.gW1 = g + n.off_w[0];
    r.gW5 = g + n.off_w[4];
    r.gb5 = g + n.off_b[4];
    r.in = in;
    static std::atomic<unsigned long long> done{0};
    e = optin(grad_kernel, GEMM_SMEM, done);
    if (e != cudaSuccess) return e;
    return launch_chain(grad_kernel, dim3(kGradTiles + kGradSums), dim3(256), GEMM_SMEM, s, r);
}

namespace {
ParamArgs param_args(const Net &n, const float *g) {
    ParamArgs a{};
    a.p = n.p;
    a.g = g;
    a.m = n.m;
    a.v = n.v;
    a.pb = n.wb;
    a.wt = n.wt;
    for (int l = 0; l < 5; ++l) a.off_w[l] = n.off_w[l];
    a.n = NPARAM;
    return a;
}
constexpr int kParamBlocks = kAdamTiles + (int)((NPARAM - 3 * (int64_t)HID * HID + 255) / 256);
}  // namespace

cudaError_t adam(const Net &n, const float *g, float lr, int64_t step, cudaStream_t s) {
    const float b1 = 0.9f, b2 = 0.999f;
    const AdamStep st{lr, 1.f - powf(b1, (float)step), 1.f - powf(b2, (float)step)};
    return launch_chain(param_kernel<true>, dim3(kParamBlocks), dim3(256), 0, s, param_args(n, g), st);
}

cudaError_t refresh_bf16(const Net &n, cudaStream_t s) {
    return launch_chain(param_kernel<false>, dim3(kParamBlocks), dim3(256), 0, s, param_args(n, nullptr), AdamStep{});
}

}  // namespace mlp
}  // namespace dirac
