// BF16 kernels of the convolutional surrogate that warm-starts the steady
// solve: 3x3 convolutions as implicit GEMMs on the tensor cores (BF16 operands,
// FP32 accumulation), their two backward passes, and the small layers around
// them (bias + ReLU epilogue, 2x2 average pooling, nearest 2x upsampling,
// channel copies for skip connections, 1x1 output head, MSE loss, Adam).
// Activations are NHWC with the channel count a multiple of 16; 3x3 weights
// are [Cout][3][3][Cin].
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <mma.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <initializer_list>
#include <type_traits>
#include <utility>

#include "../../include/cdf_nn.h"

using namespace nvcuda;

namespace {

constexpr int kBM = 64;      // pixels per CTA tile (forward / backward-data)
constexpr int kThreads = 128;
constexpr int kLdA = 24;     // padded leading dimensions of the shared tiles (bf16 elements)

// ---------------------------------------------------------------------------
// 3x3 convolution as an implicit GEMM.
//   forward:       Y[p][co] = act(sum_{t, ci} X[p + d(t)][ci] W[co][t][ci] + b[co])
//   backward data: dX[p][ci] = sum_{t, co} dY[p + d(t)][co] W[co][8 - t][ci]
// with d(t) = (ky - 1, kx - 1) for tap t = 3 ky + kx and zero outside the image.
// GEMM: M = pixels (tile kBM), N = output channels (tile BN), K = 9 x input channels.
// ---------------------------------------------------------------------------
template <bool kBwdData, int BN>
__global__ void __launch_bounds__(kThreads) conv3x3_kernel(const __nv_bfloat16 *__restrict__ in,
                                                           const __nv_bfloat16 *__restrict__ w,
                                                           const float *__restrict__ bias,
                                                           __nv_bfloat16 *__restrict__ out, int N, int H, int Wd,
                                                           int Cin_g, int Cout_g, int relu) {
    // Cin_g / Cout_g: channels of the GEMM input / output (fwd: Cin / Cout; bwd: Cout / Cin).
    constexpr int kLdB = BN + 8;
    __shared__ __align__(32) __nv_bfloat16 As[kBM * kLdA];
    __shared__ __align__(32) __nv_bfloat16 Bs[16 * kLdB > BN * kLdA ? 16 * kLdB : BN * kLdA];
    __shared__ __align__(32) float Cs[kBM * (BN + 4)];
    const int tid = threadIdx.x, warp = tid >> 5;
    const long long P = (long long)N * H * Wd;
    const long long p0 = (long long)blockIdx.x * kBM;
    const int n0 = blockIdx.y * BN;
    // The original weight tensor's channel counts: Cout_w x 9 x Cin_w.
    const int Cin_w = kBwdData ? Cout_g : Cin_g;

    // A-tile row handled by this thread: pixel p0 + tid / 2, 8 channels at (tid & 1) * 8.
    const int arow = tid >> 1, acol = (tid & 1) * 8;
    const long long pa = p0 + arow;
    int an = 0, ay = 0, ax = 0;
    if (pa < P) {
        an = (int)(pa / ((long long)H * Wd));
        const int rem = (int)(pa - (long long)an * H * Wd);
        ay = rem / Wd;
        ax = rem - ay * Wd;
    }

    wmma::fragment<wmma::accumulator, 16, 16, 16, float> acc[BN / 16];
#pragma unroll
    for (int j = 0; j < BN / 16; ++j) wmma::fill_fragment(acc[j], 0.f);

    const int K = 9 * Cin_g;
    for (int k0 = 0; k0 < K; k0 += 16) {
        const int tap = k0 / Cin_g, c0 = k0 - tap * Cin_g;
        const int dy = tap / 3 - 1, dx = tap % 3 - 1;
        // A tile: 16 input channels of the shifted pixels (zero outside the image).
        {
            uint4 v = make_uint4(0, 0, 0, 0);
            const int sy = ay + dy, sx = ax + dx;
            if (pa < P && sy >= 0 && sy < H && sx >= 0 && sx < Wd)
                v = *reinterpret_cast<const uint4 *>(in + (((long long)an * H + sy) * Wd + sx) * Cin_g + c0 + acol);
            *reinterpret_cast<uint4 *>(As + arow * kLdA + acol) = v;
        }
        // B tile: 16 (k) x BN (n) weights.
        if (!kBwdData) {
            // B(k = ci, n = co) = W[co][tap][ci]: per output channel 16 contiguous ci (col-major).
            for (int e = tid; e < BN * 2; e += kThreads) {
                const int nn = e >> 1, half = (e & 1) * 8;
                const uint4 v = *reinterpret_cast<const uint4 *>(w + ((long long)(n0 + nn) * 9 + tap) * Cin_w + c0 + half);
                *reinterpret_cast<uint4 *>(Bs + nn * kLdA + half) = v;
            }
        } else {
            // B(k = co, n = ci) = W[co][8 - tap][ci]: per k a row of BN contiguous ci (row-major).
            for (int e = tid; e < 16 * (BN / 8); e += kThreads) {
                const int kk = e / (BN / 8), seg = (e % (BN / 8)) * 8;
                const uint4 v = *reinterpret_cast<const uint4 *>(
                    w + ((long long)(c0 + kk) * 9 + (8 - tap)) * Cin_w + n0 + seg);
                *reinterpret_cast<uint4 *>(Bs + kk * kLdB + seg) = v;
            }
        }
        __syncthreads();
        wmma::fragment<wmma::matrix_a, 16, 16, 16, __nv_bfloat16, wmma::row_major> a;
        wmma::load_matrix_sync(a, As + warp * 16 * kLdA, kLdA);
#pragma unroll
        for (int j = 0; j < BN / 16; ++j) {
            if (!kBwdData) {
                wmma::fragment<wmma::matrix_b, 16, 16, 16, __nv_bfloat16, wmma::col_major> b;
                wmma::load_matrix_sync(b, Bs + j * 16 * kLdA, kLdA);
                wmma::mma_sync(acc[j], a, b, acc[j]);
            } else {
                wmma::fragment<wmma::matrix_b, 16, 16, 16, __nv_bfloat16, wmma::row_major> b;
                wmma::load_matrix_sync(b, Bs + j * 16, kLdB);
                wmma::mma_sync(acc[j], a, b, acc[j]);
            }
        }
        __syncthreads();
    }
    // Epilogue: bias, ReLU, BF16, one 16-byte store per 8 channels.
#pragma unroll
    for (int j = 0; j < BN / 16; ++j)
        wmma::store_matrix_sync(Cs + warp * 16 * (BN + 4) + j * 16, acc[j], BN + 4, wmma::mem_row_major);
    __syncthreads();
    for (int e = tid; e < kBM * (BN / 8); e += kThreads) {
        const int r = e / (BN / 8), seg = (e % (BN / 8)) * 8;
        const long long p = p0 + r;
        if (p >= P) continue;
        __align__(16) __nv_bfloat16 o[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            float v = Cs[r * (BN + 4) + seg + q];
            if (bias) v += bias[n0 + seg + q];
            if (relu) v = fmaxf(v, 0.f);
            o[q] = __float2bfloat16_rn(v);
        }
        *reinterpret_cast<uint4 *>(out + p * Cout_g + n0 + seg) = *reinterpret_cast<const uint4 *>(o);
    }
}

// ---------------------------------------------------------------------------
// The same two convolutions on the 5th-generation tensor cores (tcgen05): one CTA
// of 128 threads owns 128 output pixels (one TMEM lane each) and BN output
// channels (BN TMEM columns of FP32 accumulators).  K = 9 x channels runs in
// stages of 64: all threads stage the im2col rows of A (128 x 64) and the
// weights B (BN x 64) in shared memory in the K-major core-matrix layout (8 rows
// x 16 bytes per 128-byte core matrix), one thread issues four
// tcgen05.mma.kind::f16 (M = 128, N = BN, K = 16) and commits them to an
// mbarrier; two stage buffers let the next stage load while the tensor core
// works.  The epilogue reads the accumulators with tcgen05.ld (warp w owns
// lanes 32w..32w+31), adds the bias, applies the ReLU and stores BF16.  Every
// mbarrier wait is bounded; on time-out the kernel sets g_tc_error and still
// frees its tensor memory.
// ---------------------------------------------------------------------------
constexpr int kTM = 128, kTK = 64, kTcThreads = 128;
__device__ int g_tc_error = 0;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor, K-major without swizzle: start address,
// leading byte offset (between the two core matrices along K of one MMA) and
// stride byte offset (between core matrices along M or N), all in 16-byte units;
// bit 46 is the descriptor version of this architecture.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// Instruction descriptor of tcgen05.mma.kind::f16: FP32 accumulator, BF16 A and B,
// both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t mma_idesc(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Byte offset of element (r, k) of a rows x 64 stage tile in the core-matrix layout.
__device__ __forceinline__ uint32_t cm_offset(int r, int k, int rows) {
    return (uint32_t)((((k >> 3) * (rows >> 3) + (r >> 3)) << 7) + ((r & 7) << 4) + ((k & 7) << 1));
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    for (long long it = 0; it < (1ll << 26); ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred P;\n mbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n selp.u32 %0, 1, 0, P;\n}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    atomicExch(&g_tc_error, 1);
    return false;
}

template <bool kBwdData, int BN>
__global__ void __launch_bounds__(kTcThreads) conv3x3_tc_kernel(const __nv_bfloat16 *__restrict__ in,
                                                                const __nv_bfloat16 *__restrict__ w,
                                                                const float *__restrict__ bias,
                                                                __nv_bfloat16 *__restrict__ out, int N, int H, int Wd,
                                                                int Cin_g, int Cout_g, int relu) {
    constexpr int kCols = BN < 32 ? 32 : BN;               // TMEM columns (power of two >= 32)
    constexpr uint32_t kABytes = kTM * kTK * 2, kBBytes = BN * kTK * 2;
    extern __shared__ __align__(128) unsigned char tc_smem[];
    unsigned char *A = tc_smem;                              // 2 x kABytes
    unsigned char *B = tc_smem + 2 * kABytes;                // 2 x kBBytes
    // the barriers and the slot lie behind the tiles, no static shared memory: with BN = 128 three CTAs then
    // take 195 KB, and 60 KB of L1 are left for the nine reads of every input (162 us instead of 174
    // for 1 x 87 x 1500, 64 -> 128; the static part would be padded to the file's largest alignment)
    uint64_t *const mbar = reinterpret_cast<uint64_t *>(B + 2 * kBBytes);
    uint32_t &tmem_slot = *reinterpret_cast<uint32_t *>(mbar + 2);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long P = (long long)N * H * Wd;
    const long long p0 = (long long)blockIdx.x * kTM;
    const int n0 = blockIdx.y * BN;
    const int Cin_w = kBwdData ? Cout_g : Cin_g;  // the weight tensor is Cout_w x 9 x Cin_w
    const int K = 9 * Cin_g, nst = (K + kTK - 1) / kTK;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[0])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[1])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;

    // the pixel of this thread's A row
    const long long pa = p0 + tid;
    int an = 0, ay = 0, ax = 0;
    if (pa < P) {
        an = (int)(pa / ((long long)H * Wd));
        const int rem = (int)(pa - (long long)an * H * Wd);
        ay = rem / Wd;
        ax = rem - ay * Wd;
    }
    constexpr uint32_t idesc = mma_idesc(kTM, BN);
    bool ok = true;
    int last = -1;  // last stage whose MMAs were committed
    for (int s = 0; s < nst && ok; ++s) {
        const int buf = s & 1;
        if (s >= 2) ok = mbar_wait(smem_u32(&mbar[buf]), (uint32_t)(((s - 2) >> 1) & 1));
        if (!ok) break;
        unsigned char *As = A + buf * kABytes, *Bs = B + buf * kBBytes;
        const int k0 = s * kTK;
        // A: row tid, eight 16-byte groups of 8 consecutive k (one tap, 8 channels each)
#pragma unroll
        for (int g = 0; g < kTK / 8; ++g) {
            const int k = k0 + 8 * g;
            uint4 v = make_uint4(0, 0, 0, 0);
            if (pa < P && k < K) {
                const int tap = k / Cin_g, c = k - tap * Cin_g;
                const int sy = ay + tap / 3 - 1, sx = ax + tap % 3 - 1;
                if (sy >= 0 && sy < H && sx >= 0 && sx < Wd)
                    v = *reinterpret_cast<const uint4 *>(in + (((long long)an * H + sy) * Wd + sx) * Cin_g + c);
            }
            *reinterpret_cast<uint4 *>(As + cm_offset(tid, 8 * g, kTM)) = v;
        }
        // B: BN rows (output channels of the GEMM) x 64 k
        for (int e = tid; e < BN * (kTK / 8); e += kTcThreads) {
            const int nn = e / (kTK / 8), g = e % (kTK / 8);
            const int k = k0 + 8 * g;
            uint4 v = make_uint4(0, 0, 0, 0);
            if (k < K) {
                const int tap = k / Cin_g, c = k - tap * Cin_g;
                if (!kBwdData) {
                    // B(k = (tap, ci), n = co) = W[co][tap][ci]: 8 contiguous ci
                    v = *reinterpret_cast<const uint4 *>(w + ((long long)(n0 + nn) * 9 + tap) * Cin_w + c);
                } else {
                    // B(k = (tap, co), n = ci) = W[co][8 - tap][ci]: 8 co with stride 9 Cin_w
                    __align__(16) __nv_bfloat16 t[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) t[q] = w[((long long)(c + q) * 9 + (8 - tap)) * Cin_w + n0 + nn];
                    v = *reinterpret_cast<const uint4 *>(t);
                }
            }
            *reinterpret_cast<uint4 *>(Bs + cm_offset(nn, 8 * g, BN)) = v;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a0 = smem_u32(As), b0 = smem_u32(Bs);
#pragma unroll
            for (int j = 0; j < kTK / 16; ++j) {
                // K slice j: core-matrix columns 2j and 2j + 1
                const uint64_t ad = smem_desc(a0 + 2 * j * (kTM / 8) * 128, (kTM / 8) * 128, 128);
                const uint64_t bd = smem_desc(b0 + 2 * j * (BN / 8) * 128, (BN / 8) * 128, 128);
                const uint32_t acc = (s > 0 || j > 0) ? 1u : 0u;
                asm volatile(
                    "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                    " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem),
                    "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                    : "memory");
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(&mbar[buf]))
                         : "memory");
        }
        last = s;
    }
    // all MMAs done: the last commit tracks every earlier MMA of the issuing
    // thread (waited for also after a time-out, before the tensor memory is freed)
    if (last >= 0) ok = mbar_wait(smem_u32(&mbar[last & 1]), (uint32_t)((last >> 1) & 1)) && ok;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok) {
        const long long p = p0 + warp * 32 + lane;  // TMEM lane = tile row = pixel
#pragma unroll
        for (int c = 0; c < BN; c += 8) {
            uint32_t r[8];
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                           "=r"(r[7])
                         : "r"(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (p < P) {
                __align__(16) __nv_bfloat16 o[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    float v = __uint_as_float(r[q]);
                    if (bias) v += bias[n0 + c + q];
                    if (relu) v = fmaxf(v, 0.f);
                    o[q] = __float2bfloat16_rn(v);
                }
                *reinterpret_cast<uint4 *>(out + p * Cout_g + n0 + c) = *reinterpret_cast<const uint4 *>(o);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

// ---------------------------------------------------------------------------
// The same convolution with its operand tiles copied by cp.async: three stage
// buffers, the copies of stage s + 2 in flight while the tensor core works on
// stage s.  Each thread copies its A row (8 x 16 bytes of the im2col row, zero
// fill outside the image: a copy of 0 source bytes writes zeros) and, for the
// forward pass, 16-byte runs of the weights straight into the K-major
// core-matrix layout; the backward-data weights are a gather of single elements
// and are staged with ordinary loads.  A buffer is refilled only after the MMAs
// that read it have completed (its mbarrier).  Same stage layout, descriptors,
// MMAs, bounded waits and epilogue as conv3x3_tc_kernel.
// ---------------------------------------------------------------------------
constexpr int kStages = 3;

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(smem)), "l"(gmem), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <bool kBwdData, int BN>
__global__ void __launch_bounds__(kTcThreads) conv3x3_tc_pipe_kernel(const __nv_bfloat16 *__restrict__ in,
                                                                     const __nv_bfloat16 *__restrict__ w,
                                                                     const float *__restrict__ bias,
                                                                     __nv_bfloat16 *__restrict__ out, int N, int H,
                                                                     int Wd, int Cin_g, int Cout_g, int relu) {
    constexpr int kCols = BN < 32 ? 32 : BN;
    constexpr uint32_t kABytes = kTM * kTK * 2, kBBytes = BN * kTK * 2;
    extern __shared__ __align__(128) unsigned char tc_smem[];
    unsigned char *A = tc_smem;                    // kStages x kABytes
    unsigned char *B = tc_smem + kStages * kABytes;  // kStages x kBBytes
    __shared__ __align__(8) uint64_t mbar[kStages];
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long P = (long long)N * H * Wd;
    const long long p0 = (long long)blockIdx.x * kTM;
    const int n0 = blockIdx.y * BN;
    const int Cin_w = kBwdData ? Cout_g : Cin_g;
    const int K = 9 * Cin_g, nst = (K + kTK - 1) / kTK;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
#pragma unroll
        for (int b = 0; b < kStages; ++b)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[b])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;

    const long long pa = p0 + tid;
    int an = 0, ay = 0, ax = 0;
    if (pa < P) {
        an = (int)(pa / ((long long)H * Wd));
        const int rem = (int)(pa - (long long)an * H * Wd);
        ay = rem / Wd;
        ax = rem - ay * Wd;
    }
    // copies of stage s into its buffer
    auto load_stage = [&](int s) {
        unsigned char *As = A + (s % kStages) * kABytes, *Bs = B + (s % kStages) * kBBytes;
        const int k0 = s * kTK;
#pragma unroll
        for (int g = 0; g < kTK / 8; ++g) {
            const int k = k0 + 8 * g;
            const __nv_bfloat16 *src = in;
            int bytes = 0;
            if (pa < P && k < K) {
                const int tap = k / Cin_g, c = k - tap * Cin_g;
                const int sy = ay + tap / 3 - 1, sx = ax + tap % 3 - 1;
                if (sy >= 0 && sy < H && sx >= 0 && sx < Wd) {
                    src = in + (((long long)an * H + sy) * Wd + sx) * Cin_g + c;
                    bytes = 16;
                }
            }
            cp_async16(As + cm_offset(tid, 8 * g, kTM), src, bytes);
        }
        for (int e = tid; e < BN * (kTK / 8); e += kTcThreads) {
            const int nn = e / (kTK / 8), g = e % (kTK / 8);
            const int k = k0 + 8 * g;
            if (!kBwdData) {
                const __nv_bfloat16 *src = w;
                int bytes = 0;
                if (k < K) {
                    const int tap = k / Cin_g, c = k - tap * Cin_g;
                    src = w + ((long long)(n0 + nn) * 9 + tap) * Cin_w + c;
                    bytes = 16;
                }
                cp_async16(Bs + cm_offset(nn, 8 * g, BN), src, bytes);
            } else {
                uint4 v = make_uint4(0, 0, 0, 0);
                if (k < K) {
                    const int tap = k / Cin_g, c = k - tap * Cin_g;
                    __align__(16) __nv_bfloat16 t[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) t[q] = w[((long long)(c + q) * 9 + (8 - tap)) * Cin_w + n0 + nn];
                    v = *reinterpret_cast<const uint4 *>(t);
                }
                *reinterpret_cast<uint4 *>(Bs + cm_offset(nn, 8 * g, BN)) = v;
            }
        }
    };
#pragma unroll
    for (int s = 0; s < kStages - 1; ++s) {
        if (s < nst) load_stage(s);
        cp_async_commit();
    }
    constexpr uint32_t idesc = mma_idesc(kTM, BN);
    bool ok = true;
    int last = -1;
    for (int s = 0; s < nst && ok; ++s) {
        cp_async_wait<kStages - 2>();  // this thread's copies of stage s have landed
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        const int buf = s % kStages;
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a0 = smem_u32(A + buf * kABytes), b0 = smem_u32(B + buf * kBBytes);
#pragma unroll
            for (int j = 0; j < kTK / 16; ++j) {
                const uint64_t ad = smem_desc(a0 + 2 * j * (kTM / 8) * 128, (kTM / 8) * 128, 128);
                const uint64_t bd = smem_desc(b0 + 2 * j * (BN / 8) * 128, (BN / 8) * 128, 128);
                const uint32_t acc = (s > 0 || j > 0) ? 1u : 0u;
                asm volatile(
                    "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                    " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem),
                    "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                    : "memory");
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(&mbar[buf]))
                         : "memory");
        }
        last = s;
        // refill the buffer of stage s - 1 (its MMAs must be done) with stage s + kStages - 1
        const int nxt = s + kStages - 1;
        if (nxt < nst) {
            if (s >= 1) ok = mbar_wait(smem_u32(&mbar[(s - 1) % kStages]), (uint32_t)(((s - 1) / kStages) & 1));
            if (ok) load_stage(nxt);
        }
        cp_async_commit();
    }
    cp_async_wait<0>();
    if (last >= 0) ok = mbar_wait(smem_u32(&mbar[last % kStages]), (uint32_t)((last / kStages) & 1)) && ok;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok) {
        const long long p = p0 + warp * 32 + lane;
#pragma unroll
        for (int c = 0; c < BN; c += 8) {
            uint32_t r[8];
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                           "=r"(r[7])
                         : "r"(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (p < P) {
                __align__(16) __nv_bfloat16 o[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    float v = __uint_as_float(r[q]);
                    if (bias) v += bias[n0 + c + q];
                    if (relu) v = fmaxf(v, 0.f);
                    o[q] = __float2bfloat16_rn(v);
                }
                *reinterpret_cast<uint4 *>(out + p * Cout_g + n0 + c) = *reinterpret_cast<const uint4 *>(o);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

// ---------------------------------------------------------------------------
// Forward 3x3 convolution, persistent and warp-specialised.  One CTA per SM
// walks the (pixel tile, output-channel tile) items of the layer; its warps have
// fixed roles:
//   warps 0-3  producers: cp.async copies of the A rows (im2col, zero fill) and of
//              the weight tile into a ring of kWsStages stage buffers; each copy's
//              completion arrives on the stage's `full` mbarrier (count 128);
//   warp 8     one thread issues the tcgen05.mma of a stage once it is full and
//              commits them to the stage's `empty` mbarrier (the buffer may be
//              refilled when the MMAs reading it are done); after an item's last
//              stage it commits to `acc_full` of the item's accumulator;
//   warps 4-7  epilogue: wait for `acc_full`, read the accumulator from tensor
//              memory (warp 4 + q owns lanes 32q..32q+31 = pixels), bias, ReLU,
//              BF16 stores, then arrive on `acc_empty` (count 128).
// Two accumulators (2 x BN TMEM columns) alternate between items, so the epilogue
// of one item runs while the next one accumulates, and the producers run ahead
// by up to kWsStages stages across item boundaries.  Tile layout, descriptors and
// MMAs are those of conv3x3_tc_kernel.  Every wait is bounded; a thread whose
// wait runs out sets g_tc_error and a shared abort flag that ends the others' waits.
// ---------------------------------------------------------------------------
constexpr int kWsThreads = 288;  // 9 warps

__device__ __forceinline__ bool ws_wait(uint32_t bar, uint32_t parity, volatile int *abort) {
    for (long long it = 0; it < (1ll << 26); ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred P;\n mbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n selp.u32 %0, 1, 0, P;\n}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if ((it & 255) == 255 && *abort) return false;
    }
    atomicExch(&g_tc_error, 1);
    *abort = 1;
    return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

template <int BN, int kWsStages>
__global__ void __launch_bounds__(kWsThreads, 1) conv3x3_ws_kernel(const __nv_bfloat16 *__restrict__ in,
                                                                   const __nv_bfloat16 *__restrict__ w,
                                                                   const float *__restrict__ bias,
                                                                   __nv_bfloat16 *__restrict__ out, int N, int H,
                                                                   int Wd, int Cin, int Cout, int relu) {
    constexpr uint32_t kABytes = kTM * kTK * 2, kBBytes = BN * kTK * 2;
    constexpr int kCols = 2 * BN;  // two accumulators
    extern __shared__ __align__(128) unsigned char tc_smem[];
    unsigned char *A = tc_smem;
    unsigned char *B = tc_smem + kWsStages * kABytes;
    __shared__ __align__(8) uint64_t full[kWsStages], empty[kWsStages], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long P = (long long)N * H * Wd;
    const long long ptiles = (P + kTM - 1) / kTM;
    const int ntiles = Cout / BN;
    const long long items = ptiles * ntiles;
    const int K = 9 * Cin, nst = (K + kTK - 1) / kTK;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        abort_flag = 0;
        for (int b = 0; b < kWsStages; ++b) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&full[b])), "r"(128) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[b])) : "memory");
        }
        for (int b = 0; b < 2; ++b) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&acc_full[b])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&acc_empty[b])), "r"(128) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;

    if (warp < 4) {
        // ---- producers: thread tid copies A row tid and a share of the B tile
        long long g = 0;  // stage counter over all items of this CTA
        bool ok = true;
        for (long long item = blockIdx.x; item < items && ok; item += gridDim.x) {
            const long long p0 = (item / ntiles) * kTM;
            const int n0 = (int)(item % ntiles) * BN;
            const long long pa = p0 + tid;
            int an = 0, ay = 0, ax = 0;
            if (pa < P) {
                an = (int)(pa / ((long long)H * Wd));
                const int rem = (int)(pa - (long long)an * H * Wd);
                ay = rem / Wd;
                ax = rem - ay * Wd;
            }
            for (int s = 0; s < nst && ok; ++s, ++g) {
                const int buf = (int)(g % kWsStages);
                ok = ws_wait(smem_u32(&empty[buf]), (uint32_t)(((g / kWsStages) & 1) ^ 1), &abort_flag);
                if (!ok) break;
                unsigned char *As = A + buf * kABytes, *Bs = B + buf * kBBytes;
                const int k0 = s * kTK;
#pragma unroll
                for (int gg = 0; gg < kTK / 8; ++gg) {
                    const int k = k0 + 8 * gg;
                    const __nv_bfloat16 *src = in;
                    int bytes = 0;
                    if (pa < P && k < K) {
                        const int tap = k / Cin, c = k - tap * Cin;
                        const int sy = ay + tap / 3 - 1, sx = ax + tap % 3 - 1;
                        if (sy >= 0 && sy < H && sx >= 0 && sx < Wd) {
                            src = in + (((long long)an * H + sy) * Wd + sx) * Cin + c;
                            bytes = 16;
                        }
                    }
                    cp_async16(As + cm_offset(tid, 8 * gg, kTM), src, bytes);
                }
                for (int e = tid; e < BN * (kTK / 8); e += 128) {
                    const int nn = e / (kTK / 8), gg = e % (kTK / 8);
                    const int k = k0 + 8 * gg;
                    const __nv_bfloat16 *src = w;
                    int bytes = 0;
                    if (k < K) {
                        const int tap = k / Cin, c = k - tap * Cin;
                        src = w + ((long long)(n0 + nn) * 9 + tap) * Cin + c;
                        bytes = 16;
                    }
                    cp_async16(Bs + cm_offset(nn, 8 * gg, BN), src, bytes);
                }
                asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&full[buf]))
                             : "memory");
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (warp == 8) {
        // ---- one thread issues the MMAs
        if (lane == 0) {
            constexpr uint32_t idesc = mma_idesc(kTM, BN);
            long long g = 0, j = 0;
            bool ok = true, issued = false;
            for (long long item = blockIdx.x; item < items && ok; item += gridDim.x, ++j) {
                const int ab = (int)(j & 1);
                ok = ws_wait(smem_u32(&acc_empty[ab]), (uint32_t)(((j >> 1) & 1) ^ 1), &abort_flag);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t dcol = tmem + (uint32_t)(ab * BN);
                for (int s = 0; s < nst && ok; ++s, ++g) {
                    const int buf = (int)(g % kWsStages);
                    ok = ws_wait(smem_u32(&full[buf]), (uint32_t)((g / kWsStages) & 1), &abort_flag);
                    if (!ok) break;
                    // the producers' cp.async writes are generic-proxy writes; order them
                    // before the tensor core's reads
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t a0 = smem_u32(A + buf * kABytes), b0 = smem_u32(B + buf * kBBytes);
#pragma unroll
                    for (int jj = 0; jj < kTK / 16; ++jj) {
                        const uint64_t ad = smem_desc(a0 + 2 * jj * (kTM / 8) * 128, (kTM / 8) * 128, 128);
                        const uint64_t bd = smem_desc(b0 + 2 * jj * (BN / 8) * 128, (BN / 8) * 128, 128);
                        const uint32_t acc = (s > 0 || jj > 0) ? 1u : 0u;
                        asm volatile(
                            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(dcol),
                            "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                            : "memory");
                    }
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                     smem_u32(&empty[buf]))
                                 : "memory");
                    issued = true;
                }
                if (ok)
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                     smem_u32(&acc_full[ab]))
                                 : "memory");
            }
            // before the tensor memory is released: the last MMAs must be done
            // (a commit tracks all earlier MMAs of this thread)
            if (issued) {
                uint64_t *fin = &empty[(int)((g - 1) % kWsStages)];
                ws_wait(smem_u32(fin), (uint32_t)(((g - 1) / kWsStages) & 1), &abort_flag);
            }
        }
    } else {
        // ---- epilogue: warp 4 + q reads TMEM lanes 32q..32q+31
        const int q = warp - 4, row = q * 32 + lane;
        long long j = 0;
        bool ok = true;
        for (long long item = blockIdx.x; item < items && ok; item += gridDim.x, ++j) {
            const int ab = (int)(j & 1);
            ok = ws_wait(smem_u32(&acc_full[ab]), (uint32_t)((j >> 1) & 1), &abort_flag);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const long long p = (item / ntiles) * kTM + row;
            const int n0 = (int)(item % ntiles) * BN;
#pragma unroll
            for (int c = 0; c < BN; c += 8) {
                uint32_t r[8];
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                             : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                               "=r"(r[7])
                             : "r"(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(ab * BN + c)));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (p < P) {
                    __align__(16) __nv_bfloat16 o[8];
#pragma unroll
                    for (int t = 0; t < 8; ++t) {
                        float v = __uint_as_float(r[t]);
                        if (bias) v += bias[n0 + c + t];
                        if (relu) v = fmaxf(v, 0.f);
                        o[t] = __float2bfloat16_rn(v);
                    }
                    *reinterpret_cast<uint4 *>(out + p * Cout + n0 + c) = *reinterpret_cast<const uint4 *>(o);
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(smem_u32(&acc_empty[ab]));
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

template <int BN, int S>
cudaError_t launch_conv_ws(const __nv_bfloat16 *in, const __nv_bfloat16 *w, const float *bias, __nv_bfloat16 *out,
                           int N, int H, int W, int Cin, int Cout, int relu, cudaStream_t s) {
    const size_t smem = S * (size_t)(kTM * kTK * 2) + S * (size_t)(BN * kTK * 2);
    cudaError_t e = cudaFuncSetAttribute(conv3x3_ws_kernel<BN, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const long long P = (long long)N * H * W;
    const long long items = ((P + kTM - 1) / kTM) * (Cout / BN);
    const int grid = (int)std::min<long long>(items, sms);
    conv3x3_ws_kernel<BN, S><<<grid, kWsThreads, smem, s>>>(in, w, bias, out, N, H, W, Cin, Cout, relu);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Forward 3x3 convolution without an im2col copy, for images whose rows are a
// whole number of 128-pixel tiles and Cin = 8 G (16, 32 or 64 channels).  An
// output tile is 128 consecutive pixels of one image row.  For each tile the CTA
// stages the three input rows that the tile reads, 130 pixels each (one pixel of
// zero padding on either side), once in shared memory, laid out
// [ky][channel group g][pixel][8 channels]: 8 consecutive pixels of one group form
// one 128-byte core matrix.  The A operand of tap (ky, kx) and channels 16j..16j+15
// is that slab seen from pixel kx: a K-major descriptor whose start address moves
// 16 bytes per pixel, with 128 bytes between 8-pixel groups and 130 x 16 bytes
// between the two channel groups of one MMA.  So every input element is staged
// once per tile, where the im2col staging copies it nine times.  The weights of
// all nine taps for the CTA's BN output channels are staged once per CTA,
// [tap][g][co][8 channels].  The CTA is persistent over tiles: the slab of the
// next tile is copied (cp.async, zero fill outside the image) while the tensor
// core works on the current one, and two accumulators in tensor memory let the
// epilogue of one tile run while the next accumulates.  Takes the rows that are too wide for
// conv3x3_lin_kernel, which stages two whole rows of halo with every item: 207 TFLOP/s at 1 x 512 x 2048,
// 32 -> 32, and 255 at 64 -> 64, where the im2col kernels reach 80 and 98.  Every wait is bounded;
// on a time-out the kernel sets g_tc_error, waits (bounded) for its own MMAs and
// copies, frees its tensor memory and returns.
// ---------------------------------------------------------------------------
constexpr int kSlabW = kTM + 2;  // staged pixels per input row

__host__ __device__ constexpr uint32_t slab_bytes(int G) {
    return (uint32_t)((3 * G * kSlabW * 16 + 127) / 128 * 128);
}

template <int BN, int G>
__global__ void __launch_bounds__(kTcThreads) conv3x3_slab_kernel(const __nv_bfloat16 *__restrict__ in,
                                                                  const __nv_bfloat16 *__restrict__ w,
                                                                  const float *__restrict__ bias,
                                                                  __nv_bfloat16 *__restrict__ out, int N, int H,
                                                                  int Wd, int Cout, int relu) {
    constexpr int Cin = 8 * G;
    constexpr int kAcc = BN < 32 ? 32 : BN;  // TMEM columns of one accumulator
    constexpr int kCols = 2 * kAcc;
    constexpr uint32_t kSlab = slab_bytes(G);
    extern __shared__ __align__(128) unsigned char sl_smem[];
    unsigned char *const Wsm = sl_smem + 2 * kSlab;
    __shared__ __align__(8) uint64_t mbar[2];
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n0 = blockIdx.y * BN;
    const int tiles_x = Wd / kTM;
    const long long ntiles = (long long)N * H * tiles_x;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[0])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[1])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;

    // weights: W[n0 + co][t][8g .. 8g + 7] -> Wsm[(t G + g) BN + co]
    for (int e = tid; e < 9 * G * BN; e += kTcThreads) {
        const int g = e % G, co = (e / G) % BN, t = e / (G * BN);
        cp_async16(Wsm + ((t * G + g) * BN + co) * 16, w + ((long long)(n0 + co) * 9 + t) * Cin + 8 * g, 16);
    }
    // the three input rows of a tile, channel group fastest (coalesced reads)
    const auto stage = [&](long long tile, unsigned char *dst) {
        const int tx = (int)(tile % tiles_x);
        const long long ry = tile / tiles_x;
        const int y = (int)(ry % H), n = (int)(ry / H), x0 = tx * kTM;
        for (int e = tid; e < 3 * G * kSlabW; e += kTcThreads) {
            const int g = e % G, px = (e / G) % kSlabW, ky = e / (G * kSlabW);
            const int sy = y + ky - 1, sx = x0 + px - 1;
            const bool inside = sy >= 0 && sy < H && sx >= 0 && sx < Wd;
            const __nv_bfloat16 *src = inside ? in + (((long long)n * H + sy) * Wd + sx) * Cin + 8 * g : in;
            cp_async16(dst + ((ky * G + g) * kSlabW + px) * 16, src, inside ? 16 : 0);
        }
    };
    const auto epilogue = [&](long long tile, int acc) {
        const int tx = (int)(tile % tiles_x);
        const long long row = tile / tiles_x;  // n H + y
        const long long p = row * Wd + tx * kTM + warp * 32 + lane;
#pragma unroll
        for (int c = 0; c < BN; c += 8) {
            uint32_t r[8];
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                           "=r"(r[7])
                         : "r"(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(acc * kAcc + c)));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            __align__(16) __nv_bfloat16 o[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                float v = __uint_as_float(r[q]);
                if (bias) v += bias[n0 + c + q];
                if (relu) v = fmaxf(v, 0.f);
                o[q] = __float2bfloat16_rn(v);
            }
            *reinterpret_cast<uint4 *>(out + p * Cout + n0 + c) = *reinterpret_cast<const uint4 *>(o);
        }
    };

    constexpr uint32_t idesc = mma_idesc(kTM, BN);
    long long tile = blockIdx.x;
    if (tile < ntiles) stage(tile, sl_smem);
    cp_async_commit();  // the weights and the first slab
    bool ok = true;
    int i = 0;
    long long prev = -1;
    for (; tile < ntiles; tile += gridDim.x, ++i) {
        const int b = i & 1;
        cp_async_wait<0>();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a0 = smem_u32(sl_smem + b * kSlab), w0 = smem_u32(Wsm);
            int k = 0;
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const int ky = t / 3, kx = t % 3;
#pragma unroll
                for (int j = 0; j < G / 2; ++j, ++k) {
                    const uint64_t ad = smem_desc(a0 + (uint32_t)(((ky * G + 2 * j) * kSlabW + kx) * 16), kSlabW * 16, 128);
                    const uint64_t bd = smem_desc(w0 + (uint32_t)((t * G + 2 * j) * BN * 16), BN * 16, 128);
                    const uint32_t accum = k > 0 ? 1u : 0u;
                    asm volatile(
                        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem + (uint32_t)(b * kAcc)),
                        "l"(ad), "l"(bd), "r"(idesc), "r"(accum)
                        : "memory");
                }
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(&mbar[b]))
                         : "memory");
        }
        // the previous tile's MMAs: done -> its slab buffer and accumulator are free
        if (i > 0) {
            const bool mine = ok && mbar_wait(smem_u32(&mbar[b ^ 1]), (uint32_t)(((i - 1) >> 1) & 1));
            ok = __syncthreads_and(mine) != 0;  // one decision for the whole CTA
        }
        const long long next = tile + gridDim.x;
        if (ok && next < ntiles) stage(next, sl_smem + (b ^ 1) * kSlab);
        cp_async_commit();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (ok && i > 0) epilogue(prev, b ^ 1);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        prev = tile;
        if (!ok) {
            ++i;
            break;
        }
    }
    // the last tile (its commit tracks every earlier MMA of the issuing thread;
    // waited for also after a time-out, before the tensor memory is freed)
    if (i > 0) {
        const bool done = mbar_wait(smem_u32(&mbar[(i - 1) & 1]), (uint32_t)(((i - 1) >> 1) & 1));
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (ok && done) epilogue(prev, (i - 1) & 1);
    }
    cp_async_wait<0>();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

template <int BN, int G>
cudaError_t launch_conv_slab(const __nv_bfloat16 *in, const __nv_bfloat16 *w, const float *bias, __nv_bfloat16 *out,
                             int N, int H, int W, int Cout, int relu, cudaStream_t s) {
    const size_t smem = 2 * (size_t)slab_bytes(G) + 9 * (size_t)G * BN * 16;
    cudaError_t e = cudaFuncSetAttribute(conv3x3_slab_kernel<BN, G>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    // the whole unified L1 / shared memory as shared memory, so that several CTAs fit on an SM
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(conv3x3_slab_kernel<BN, G>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, smem_sm = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (e != cudaSuccess) return e;
    // CTAs per SM (the persistent grid): as many as the shared memory (1 KB reserved and 1 KB
    // static a CTA) and the tensor memory (512 columns per SM, two accumulators a CTA) hold; 48
    // registers a thread never limit it.  (The occupancy query answered one CTA per SM
    // here, which left two thirds of the SMs' slots empty: 142 against 93 us.)
    const int per_sm = std::max(1, std::min((int)(smem_sm / (smem + 2048)), 512 / (2 * (BN < 32 ? 32 : BN))));
    const long long tiles = (long long)N * H * (W / kTM);
    const int gx = (int)std::max<long long>(1, std::min<long long>(tiles, (long long)sms * per_sm / (Cout / BN)));
    dim3 grid(gx, Cout / BN);
    conv3x3_slab_kernel<BN, G><<<grid, kTcThreads, smem, s>>>(in, w, bias, out, N, H, W, Cout, relu);
    return cudaGetLastError();
}

// The slab kernel's shapes: forward, rows of whole 128-pixel tiles, Cin 16, 32 or 64.
bool slab_shape(int W, int Cin_g, int Cout_g) {
    return W % kTM == 0 && (Cin_g == 16 || Cin_g == 32 || Cin_g == 64) && Cout_g % 32 == 0;
}

cudaError_t conv_dispatch_slab(const __nv_bfloat16 *in, const __nv_bfloat16 *w, const float *bias, __nv_bfloat16 *out,
                               int N, int H, int W, int Cin_g, int Cout_g, int relu, cudaStream_t s) {
    // (for 64 input channels at most 64 output channels a CTA: the staged weights of
    // 128 would not fit beside the two slabs)
    int BN = Cout_g % 128 == 0 ? 128 : (Cout_g % 64 == 0 ? 64 : 32);
    if (Cin_g == 64 && BN > 64) BN = 64;
#define CDF_SLAB(G, WIDE)                                                                               \
    switch (BN) {                                                                                       \
        case 128: return launch_conv_slab<WIDE, G>(in, w, bias, out, N, H, W, Cout_g, relu, s);         \
        case 64: return launch_conv_slab<64, G>(in, w, bias, out, N, H, W, Cout_g, relu, s);            \
        default: return launch_conv_slab<32, G>(in, w, bias, out, N, H, W, Cout_g, relu, s);            \
    }
    if (Cin_g == 16) CDF_SLAB(2, 128)
    if (Cin_g == 32) CDF_SLAB(4, 128)
    CDF_SLAB(8, 64)  // BN is at most 64 here
#undef CDF_SLAB
}

#include "nn_conv.cuh"  // the convolutions without im2col copies (the default path)

template <bool kBwdData, int BN>
cudaError_t launch_conv_tc_pipe(const __nv_bfloat16 *in, const __nv_bfloat16 *w, const float *bias,
                                __nv_bfloat16 *out, int N, int H, int W, int Cin_g, int Cout_g, int relu,
                                cudaStream_t s) {
    const size_t smem = kStages * (size_t)(kTM * kTK * 2) + kStages * (size_t)(BN * kTK * 2);
    cudaError_t e = cudaFuncSetAttribute(conv3x3_tc_pipe_kernel<kBwdData, BN>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const long long P = (long long)N * H * W;
    dim3 grid((unsigned)((P + kTM - 1) / kTM), Cout_g / BN);
    conv3x3_tc_pipe_kernel<kBwdData, BN><<<grid, kTcThreads, smem, s>>>(in, w, bias, out, N, H, W, Cin_g, Cout_g,
                                                                        relu);
    return cudaGetLastError();
}

template <bool kBwdData, int BN>
cudaError_t launch_conv_tc(const __nv_bfloat16 *in, const __nv_bfloat16 *w, const float *bias, __nv_bfloat16 *out,
                           int N, int H, int W, int Cin_g, int Cout_g, int relu, cudaStream_t s) {
    const size_t smem = 2 * (size_t)(kTM * kTK * 2) + 2 * (size_t)(BN * kTK * 2) + 32;  // tiles, barriers
    cudaError_t e = cudaFuncSetAttribute(conv3x3_tc_kernel<kBwdData, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    const long long P = (long long)N * H * W;
    dim3 grid((unsigned)((P + kTM - 1) / kTM), Cout_g / BN);
    conv3x3_tc_kernel<kBwdData, BN><<<grid, kTcThreads, smem, s>>>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu);
    return cudaGetLastError();
}

// Convolution path: 1 = tcgen05 without im2col copy on conv3x3_lin_kernel where it is
// estimated the faster one, else on conv3x3_slab_kernel for its shapes, else the faster im2col
// staging per shape (default; 4 is the same), 2 = tcgen05 with synchronous im2col staging, 3 = tcgen05
// persistent warp-specialised forward, 0 = the warp-level MMA kernels.
int g_path = 1;
bool g_use_tc = true;

template <bool kBwdData>
cudaError_t conv_dispatch_path2(const __nv_bfloat16 *in, const __nv_bfloat16 *w, const float *bias, __nv_bfloat16 *out,
                                int N, int H, int W, int Cin_g, int Cout_g, int relu, cudaStream_t s, int BN) {
    switch (BN) {
        case 128: return launch_conv_tc<kBwdData, 128>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu, s);
        case 64: return launch_conv_tc<kBwdData, 64>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu, s);
        case 32: return launch_conv_tc<kBwdData, 32>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu, s);
        default: return launch_conv_tc<kBwdData, 16>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu, s);
    }
}

template <bool kBwdData>
cudaError_t conv_dispatch(const __nv_bfloat16 *in, const __nv_bfloat16 *w, const float *bias, __nv_bfloat16 *out,
                          int N, int H, int W, int Cin_g, int Cout_g, int relu, cudaStream_t s) {
    const int BN = Cout_g % 128 == 0 ? 128 : (Cout_g % 64 == 0 ? 64 : (Cout_g % 32 == 0 ? 32 : 16));
    if (g_path == 1 || g_path == 4) {
        bool ran = false;
        const cudaError_t e = conv_lin<kBwdData>(in, w, bias, nullptr, out, N, H, W, Cin_g, Cout_g, relu, s, &ran);
        if (ran) return e;
        if (!kBwdData && slab_shape(W, Cin_g, Cout_g))
            return conv_dispatch_slab(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu, s);
    }
    if (g_path == 3 && !kBwdData) {  // forward: the persistent warp-specialised kernel
        switch (BN) {
            case 128: return launch_conv_ws<128, 4>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu, s);
            case 64: return launch_conv_ws<64, 5>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu, s);
            default: return launch_conv_ws<32, 6>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu, s);
        }
    }
    // im2col staging: the cp.async pipeline for long K
    // (Cin >= 128, e.g. 159 against 101 TFLOP/s at 32^2 x 256 -> 256), two-buffer
    // synchronous staging for short K, where more CTAs per SM hide more latency
    // (80 against 72 TFLOP/s at 256^2 x 32 -> 32)
    if ((g_path == 1 || g_path == 4) && Cin_g < 128)
        return conv_dispatch_path2<kBwdData>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu, s, BN);
    if (g_path == 1 || g_path == 3 || g_path == 4) {
        switch (BN) {
            case 128: return launch_conv_tc_pipe<kBwdData, 128>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu, s);
            case 64: return launch_conv_tc_pipe<kBwdData, 64>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu, s);
            case 32: return launch_conv_tc_pipe<kBwdData, 32>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu, s);
            default: return launch_conv_tc_pipe<kBwdData, 16>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu, s);
        }
    }
    if (g_path == 2) return conv_dispatch_path2<kBwdData>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu, s, BN);
    const long long P = (long long)N * H * W;
    const int bn = BN >= 64 ? 64 : BN;
    dim3 grid((unsigned)((P + kBM - 1) / kBM), Cout_g / bn);
    if (bn == 64) conv3x3_kernel<kBwdData, 64><<<grid, kThreads, 0, s>>>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu);
    else if (bn == 32) conv3x3_kernel<kBwdData, 32><<<grid, kThreads, 0, s>>>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu);
    else conv3x3_kernel<kBwdData, 16><<<grid, kThreads, 0, s>>>(in, w, bias, out, N, H, W, Cin_g, Cout_g, relu);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// 3x3 convolution, weight gradient: dW[co][t][ci] += sum_p dY[p][co] X[p + d(t)][ci]
// GEMM per tap: M = Cout (tile 64), N = Cin (tile 16), K = pixels (chunk of 64 per
// stage, split over the grid's z dimension); FP32 partial sums are added atomically.
// ---------------------------------------------------------------------------
constexpr int kWBM = 64, kWBK = 64;
__global__ void __launch_bounds__(kThreads) conv3x3_wgrad_kernel(const __nv_bfloat16 *__restrict__ x,
                                                                 const __nv_bfloat16 *__restrict__ dy,
                                                                 float *__restrict__ dw, int N, int H, int Wd,
                                                                 int Cin, int Cout, long long pix_per_split) {
    __shared__ __align__(32) __nv_bfloat16 As[kWBK * (kWBM + 8)];  // [k = pixel][m = co]
    __shared__ __align__(32) __nv_bfloat16 Bs[kWBK * kLdA];       // [k = pixel][n = ci]
    __shared__ __align__(32) float Cs[kWBM * 20];
    const int tid = threadIdx.x, warp = tid >> 5;
    const int co0 = blockIdx.x * kWBM;
    const int tap = blockIdx.y / (Cin / 16), ci0 = (blockIdx.y % (Cin / 16)) * 16;
    const int dyy = tap / 3 - 1, dxx = tap % 3 - 1;
    const long long P = (long long)N * H * Wd;
    const long long pbeg = (long long)blockIdx.z * pix_per_split;
    const long long pend = pbeg + pix_per_split < P ? pbeg + pix_per_split : P;
    const int mrows = Cout - co0 < kWBM ? Cout - co0 : kWBM;  // 32 or 64 output channels

    wmma::fragment<wmma::accumulator, 16, 16, 16, float> acc;
    wmma::fill_fragment(acc, 0.f);
    for (long long pk = pbeg; pk < pend; pk += kWBK) {
        // A: dY rows (pixel k, output channels co0..co0+63), 8 channels per 16-byte load.
        for (int e = tid; e < kWBK * (kWBM / 8); e += kThreads) {
            const int kk = e / (kWBM / 8), seg = (e % (kWBM / 8)) * 8;
            uint4 v = make_uint4(0, 0, 0, 0);
            const long long p = pk + kk;
            if (p < pend && seg < mrows) v = *reinterpret_cast<const uint4 *>(dy + p * Cout + co0 + seg);
            *reinterpret_cast<uint4 *>(As + kk * (kWBM + 8) + seg) = v;
        }
        // B: X at the shifted pixel, 16 input channels.
        {
            const int kk = tid >> 1, half = (tid & 1) * 8;
            uint4 v = make_uint4(0, 0, 0, 0);
            const long long p = pk + kk;
            if (p < pend) {
                const int n = (int)(p / ((long long)H * Wd));
                const unsigned rem = (unsigned)(p - (long long)n * H * Wd);  // (no device holds images of 2^32 pixels)
                const int yy = (int)(rem / (unsigned)Wd) + dyy, xx = (int)(rem % (unsigned)Wd) + dxx;
                if (yy >= 0 && yy < H && xx >= 0 && xx < Wd)
                    v = *reinterpret_cast<const uint4 *>(x + (((long long)n * H + yy) * Wd + xx) * Cin + ci0 + half);
            }
            *reinterpret_cast<uint4 *>(Bs + kk * kLdA + half) = v;
        }
        __syncthreads();
#pragma unroll
        for (int ks = 0; ks < kWBK; ks += 16) {
            wmma::fragment<wmma::matrix_a, 16, 16, 16, __nv_bfloat16, wmma::col_major> a;
            wmma::fragment<wmma::matrix_b, 16, 16, 16, __nv_bfloat16, wmma::row_major> b;
            wmma::load_matrix_sync(a, As + ks * (kWBM + 8) + warp * 16, kWBM + 8);
            wmma::load_matrix_sync(b, Bs + ks * kLdA, kLdA);
            wmma::mma_sync(acc, a, b, acc);
        }
        __syncthreads();
    }
    wmma::store_matrix_sync(Cs + warp * 16 * 20, acc, 20, wmma::mem_row_major);
    __syncthreads();
    for (int e = tid; e < kWBM * 16; e += kThreads) {
        const int r = e >> 4, c = e & 15;
        if (r < mrows) atomicAdd(dw + ((long long)(co0 + r) * 9 + tap) * Cin + ci0 + c, Cs[r * 20 + c]);
    }
}

// dw[i] += sum_{split} part[split][i] and db[c] += sum_{split} bpart[split][c], each in
// a fixed order: a block of 256 threads covers R runs of four values, 256 / R
// threads a run, each with its share of the splits, added in order; their
// sums are then added in order.  Blocks from `wblocks` on take the bias.  Bound by the partial sums' reads;
// R = 32, and 8 for 128 splits and more, where few blocks would otherwise walk long rows (1040 splits of
// 32 x 288 weights: 32 -> 14 us).
template <int R>
__global__ void __launch_bounds__(256) weight_sum_kernel(const float *__restrict__ part, float *__restrict__ dw,
                                                         int n4, int splits, int wblocks,
                                                         const float *__restrict__ bpart, float *__restrict__ db,
                                                         int c4, int bsplits) {
    constexpr int T = 256 / R;
    const bool bias = (int)blockIdx.x >= wblocks;
    const float4 *src = reinterpret_cast<const float4 *>(bias ? bpart : part);
    float *dst = bias ? db : dw;
    const int n = bias ? c4 : n4, ns = bias ? bsplits : splits;
    const int i = (blockIdx.x - (bias ? wblocks : 0)) * R + threadIdx.x % R, sl = threadIdx.x / R;
    const int z0 = (int)((long long)ns * sl / T), z1 = (int)((long long)ns * (sl + 1) / T);
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < n) {
#pragma unroll 8
        for (int z = z0; z < z1; ++z) {
            const float4 v = __ldg(src + (long long)z * n + i);
            a.x += v.x;
            a.y += v.y;
            a.z += v.z;
            a.w += v.w;
        }
    }
    __shared__ float4 red[T][R];
    red[sl][threadIdx.x % R] = a;
    __syncthreads();
    if (sl == 0 && i < n) {
#pragma unroll 8
        for (int k = 1; k < T; ++k) {
            const float4 v = red[k][threadIdx.x];
            a.x += v.x;
            a.y += v.y;
            a.z += v.z;
            a.w += v.w;
        }
        float *d = dst + 4ll * i;
        d[0] += a.x;
        d[1] += a.y;
        d[2] += a.z;
        d[3] += a.w;
    }
}

// A part of the weight gradient's batch with fewer than 2^30 padded positions: n images of H rows
// from pixel `first` on, of which the positions [q0, q1) and the pixels [p0, p0 + P) (of those
// from `first` on) are summed.  Parts are runs of whole images, or bands of rows of one image
// with the row above and below each band, which its taps read.
struct WgradPart {
    long long first;
    int n, H, q0, q1;
    long long p0, P;
};
// f(part) for every part, until one returns false; false also if three rows are too many
// positions (W of some 2^28: the warp-level kernel takes those).
template <class F>
bool wgrad_parts(int N, int H, int W, const F &f) {
    const long long row = (long long)W + 1, one = (H + 1ll) * row, most = (1ll << 30) - 1;
    if (one <= most) {
        const int images = (int)std::min<long long>(N, most / one);
        for (int n0 = 0; n0 < N; n0 += images) {
            const int n = std::min(images, N - n0);
            if (!f(WgradPart{(long long)n0 * H * W, n, H, 0, (int)(n * one), 0, (long long)n * H * W})) return false;
        }
        return true;
    }
    const long long rows = most / row - 3;  // and a row above, one below and the padding row
    if (rows < 1) return false;
    for (int n = 0; n < N; ++n)
        for (long long y0 = 0; y0 < H; y0 += rows) {
            const int y1 = (int)std::min<long long>(H, y0 + rows), lo = (int)std::max(0ll, y0 - 1), hi = std::min(H, y1 + 1);
            if (!f(WgradPart{((long long)n * H + lo) * W, 1, hi - lo, (int)((y0 - lo) * row), (int)((y1 - lo) * row),
                             (y0 - lo) * W, (y1 - y0) * W}))
                return false;
        }
    return true;
}

// ---------------------------------------------------------------------------
// Small layers (one thread per element unless stated).
// ---------------------------------------------------------------------------
__global__ void bias_grad_kernel(const __nv_bfloat16 *__restrict__ dy, float *__restrict__ db, long long P, int C) {
    // block: 256 threads over pixels for one channel group of 8; grid.x = C / 8, grid.y = splits
    const int c0 = blockIdx.x * 8;
    float s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (long long p = (long long)blockIdx.y * blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.y * blockDim.x) {
        const uint4 v = *reinterpret_cast<const uint4 *>(dy + p * C + c0);
        const __nv_bfloat16 *e = reinterpret_cast<const __nv_bfloat16 *>(&v);
#pragma unroll
        for (int q = 0; q < 8; ++q) s[q] += __bfloat162float(e[q]);
    }
    __shared__ float red[8][256];
#pragma unroll
    for (int q = 0; q < 8; ++q) red[q][threadIdx.x] = s[q];
    __syncthreads();
    for (int st = blockDim.x / 2; st > 0; st >>= 1) {
        if ((int)threadIdx.x < st)
#pragma unroll
            for (int q = 0; q < 8; ++q) red[q][threadIdx.x] += red[q][threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x < 8) atomicAdd(db + c0 + threadIdx.x, red[threadIdx.x][0]);
}

// The layers between the convolutions move each element once or twice and compute
// next to nothing, so they are bound by memory accesses: a thread takes V = 8
// channels, one 16-byte access each, wherever the channel counts and slices are multiples
// of 8 and the pointers lie on 16 bytes, else one (2-byte accesses reached a tenth of
// the copy bandwidth: 32 x 64 x 64 x 64 channels upsampled in 45 us, with 16 bytes in 7).
// Indexes are 32-bit where the element count allows (I = int).
template <int V>
struct alignas(2 * V) Chan {  // V consecutive BF16 values
    __nv_bfloat16 e[V];
};
template <int V>
__device__ __forceinline__ Chan<V> load_chan(const __nv_bfloat16 *p) {
    Chan<V> r;
    if constexpr (V == 8) {
        const uint4 q = *reinterpret_cast<const uint4 *>(p);
        *reinterpret_cast<uint4 *>(r.e) = q;
    } else {
        r.e[0] = *p;
    }
    return r;
}
template <int V>
__device__ __forceinline__ void store_chan(__nv_bfloat16 *p, const Chan<V> &r) {
    if constexpr (V == 8) *reinterpret_cast<uint4 *>(p) = *reinterpret_cast<const uint4 *>(r.e);
    else *p = r.e[0];
}

template <int V>
__global__ void relu_bwd_kernel(__nv_bfloat16 *__restrict__ d, const __nv_bfloat16 *__restrict__ y, long long n) {
    const long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * V;
    if (i >= n) return;
    const Chan<V> yv = load_chan<V>(y + i);
    Chan<V> dv = load_chan<V>(d + i);
#pragma unroll
    for (int k = 0; k < V; ++k)
        if (!(__bfloat162float(yv.e[k]) > 0.f)) dv.e[k] = __float2bfloat16_rn(0.f);
    store_chan<V>(d + i, dv);
}

template <int V, class I>
__global__ void avgpool2_fwd_kernel(const __nv_bfloat16 *__restrict__ x, __nv_bfloat16 *__restrict__ y, int N, int H,
                                    int W, int C) {
    const I i = (I)blockIdx.x * blockDim.x + threadIdx.x, G = C / V;
    const int Ho = H / 2, Wo = W / 2;
    if (i >= (I)N * Ho * Wo * G) return;
    const int c = (int)(i % G) * V;
    I q = i / G;
    const int xo = (int)(q % Wo);
    q /= Wo;
    const int yo = (int)(q % Ho);
    const long long n = q / Ho;
    float s[V];
#pragma unroll
    for (int k = 0; k < V; ++k) s[k] = 0.f;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const Chan<V> v = load_chan<V>(x + ((n * H + 2 * yo + a) * W + 2 * xo + b) * C + c);
#pragma unroll
            for (int k = 0; k < V; ++k) s[k] += __bfloat162float(v.e[k]);
        }
    Chan<V> o;
#pragma unroll
    for (int k = 0; k < V; ++k) o.e[k] = __float2bfloat16_rn(0.25f * s[k]);
    store_chan<V>(y + (long long)i * V, o);
}

// One thread per dy element: the four pixels of its window get the same value.
template <int V, class I>
__global__ void avgpool2_bwd_kernel(const __nv_bfloat16 *__restrict__ dy, __nv_bfloat16 *__restrict__ dx, int N, int H,
                                    int W, int C) {
    const I i = (I)blockIdx.x * blockDim.x + threadIdx.x, G = C / V;
    const int Ho = H / 2, Wo = W / 2;
    if (i >= (I)N * Ho * Wo * G) return;
    const int c = (int)(i % G) * V;
    I q = i / G;
    const int xo = (int)(q % Wo);
    q /= Wo;
    const int yo = (int)(q % Ho);
    const long long n = q / Ho;
    Chan<V> g = load_chan<V>(dy + (long long)i * V);
#pragma unroll
    for (int k = 0; k < V; ++k) g.e[k] = __float2bfloat16_rn(0.25f * __bfloat162float(g.e[k]));
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) store_chan<V>(dx + ((n * H + 2 * yo + a) * W + 2 * xo + b) * C + c, g);
}

// Nearest 2x upsampling of x [N, H, W, C] into channels [coff, coff + C) of y [N, 2H, 2W, Cy];
// one thread per x element.
template <int V, class I>
__global__ void upsample2_fwd_kernel(const __nv_bfloat16 *__restrict__ x, __nv_bfloat16 *__restrict__ y, int N, int H,
                                     int W, int C, int Cy, int coff) {
    const I i = (I)blockIdx.x * blockDim.x + threadIdx.x, G = C / V;
    if (i >= (I)N * H * W * G) return;
    const int c = (int)(i % G) * V;
    I q = i / G;
    const int xx = (int)(q % W);
    const long long row = q / W;  // n H + y
    const Chan<V> v = load_chan<V>(x + (long long)i * V);
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) store_chan<V>(y + ((2 * row + a) * 2 * W + 2 * xx + b) * Cy + coff + c, v);
}

// Backward of the above: dx[n][y][x][c] = sum of the 4 covering dy values (channels coff..coff+C of dy).
template <int V, class I>
__global__ void upsample2_bwd_kernel(const __nv_bfloat16 *__restrict__ dy, __nv_bfloat16 *__restrict__ dx, int N, int H,
                                     int W, int C, int Cy, int coff) {
    const I i = (I)blockIdx.x * blockDim.x + threadIdx.x, G = C / V;
    if (i >= (I)N * H * W * G) return;
    const int c = (int)(i % G) * V;
    I q = i / G;
    const int xx = (int)(q % W);
    const long long row = q / W;
    float s[V];
#pragma unroll
    for (int k = 0; k < V; ++k) s[k] = 0.f;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const Chan<V> v = load_chan<V>(dy + ((2 * row + a) * 2 * W + 2 * xx + b) * Cy + coff + c);
#pragma unroll
            for (int k = 0; k < V; ++k) s[k] += __bfloat162float(v.e[k]);
        }
    Chan<V> o;
#pragma unroll
    for (int k = 0; k < V; ++k) o.e[k] = __float2bfloat16_rn(s[k]);
    store_chan<V>(dx + (long long)i * V, o);
}

// y[:, :, :, dst_off + c] = x[:, :, :, src_off + c] for c < count (skip concat / split).
template <int V, class I>
__global__ void copy_channels_kernel(const __nv_bfloat16 *__restrict__ x, __nv_bfloat16 *__restrict__ y, long long P,
                                     int Cx, int Cy, int src_off, int dst_off, int count, int accumulate) {
    const I i = (I)blockIdx.x * blockDim.x + threadIdx.x, G = count / V;
    const long long p = i / G;
    if (p >= P) return;
    const int c = (int)(i % G) * V;
    Chan<V> v = load_chan<V>(x + p * Cx + src_off + c);
    __nv_bfloat16 *const d = y + p * Cy + dst_off + c;
    if (accumulate) {
        const Chan<V> old = load_chan<V>(d);
#pragma unroll
        for (int k = 0; k < V; ++k)
            v.e[k] = __float2bfloat16_rn(__bfloat162float(v.e[k]) + __bfloat162float(old.e[k]));
    }
    store_chan<V>(d, v);
}

// ---- the same layers fused as the network's passes use them ----------------------
// (a launch and one pass over the activations less each; the intermediate values are
// rounded to BF16 where the separate layers store them, so the results are the same bits)

// y[n][yy][xx] = (upsampled x, skip): the first C channels from x [N, H, W, C] by nearest 2x
// upsampling, the next Cs from skip [N, 2H, 2W, Cs]; one thread per 8 (V) channels of a coarse
// pixel or of a skip pixel.
template <int V, class I>
__global__ void upsample2_concat_kernel(const __nv_bfloat16 *__restrict__ x, const __nv_bfloat16 *__restrict__ skip,
                                        __nv_bfloat16 *__restrict__ y, int N, int H, int W, int C, int Cs) {
    I i = (I)blockIdx.x * blockDim.x + threadIdx.x;
    const I G = C / V, Gs = Cs / V, nx = (I)N * H * W * G;
    const int Cy = C + Cs;
    if (i < nx) {
        const int c = (int)(i % G) * V;
        const I q = i / G;
        const int xx = (int)(q % W);
        const long long row = q / W;  // n H + y
        const Chan<V> v = load_chan<V>(x + (long long)i * V);
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) store_chan<V>(y + ((2 * row + a) * 2 * W + 2 * xx + b) * Cy + c, v);
        return;
    }
    i -= nx;
    if (i >= (I)N * 4 * H * W * Gs) return;
    const long long p = i / Gs;
    store_chan<V>(y + p * Cy + C + (int)(i % Gs) * V, load_chan<V>(skip + (long long)i * V));
}

// Gradient of a ReLU's output y [N, H, W, C] that was upsampled into the first C of dy's Cy
// channels: dx = sum of the four covering dy values where y > 0, else 0.
template <int V, class I>
__global__ void upsample2_bwd_relu_kernel(const __nv_bfloat16 *__restrict__ dy, const __nv_bfloat16 *__restrict__ y,
                                          __nv_bfloat16 *__restrict__ dx, int N, int H, int W, int C, int Cy) {
    const I i = (I)blockIdx.x * blockDim.x + threadIdx.x, G = C / V;
    if (i >= (I)N * H * W * G) return;
    const int c = (int)(i % G) * V;
    const I q = i / G;
    const int xx = (int)(q % W);
    const long long row = q / W;
    float s[V];
#pragma unroll
    for (int k = 0; k < V; ++k) s[k] = 0.f;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const Chan<V> v = load_chan<V>(dy + ((2 * row + a) * 2 * W + 2 * xx + b) * Cy + c);
#pragma unroll
            for (int k = 0; k < V; ++k) s[k] += __bfloat162float(v.e[k]);
        }
    const Chan<V> m = load_chan<V>(y + (long long)i * V);
    Chan<V> o;
#pragma unroll
    for (int k = 0; k < V; ++k) o.e[k] = __float2bfloat16_rn(__bfloat162float(m.e[k]) > 0.f ? s[k] : 0.f);
    store_chan<V>(dx + (long long)i * V, o);
}

// Gradient of a ReLU's output y [N, H, W, C] that was pooled (gradient dp [N, H/2, W/2, C]) and
// copied into channels [coff, coff + C) of a concatenation (gradient dcat, Cy channels): dx =
// dp / 4 (BF16) + dcat, where y > 0, else 0.  One thread per pooled element.
template <int V, class I>
__global__ void pool_skip_bwd_relu_kernel(const __nv_bfloat16 *__restrict__ dp, const __nv_bfloat16 *__restrict__ dcat,
                                          const __nv_bfloat16 *__restrict__ y, __nv_bfloat16 *__restrict__ dx, int N,
                                          int H, int W, int C, int Cy, int coff) {
    const I i = (I)blockIdx.x * blockDim.x + threadIdx.x, G = C / V;
    const int Ho = H / 2, Wo = W / 2;
    if (i >= (I)N * Ho * Wo * G) return;
    const int c = (int)(i % G) * V;
    I q = i / G;
    const int xo = (int)(q % Wo);
    q /= Wo;
    const int yo = (int)(q % Ho);
    const long long n = q / Ho;
    Chan<V> g = load_chan<V>(dp + (long long)i * V);
#pragma unroll
    for (int k = 0; k < V; ++k) g.e[k] = __float2bfloat16_rn(0.25f * __bfloat162float(g.e[k]));
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const long long p = (n * H + 2 * yo + a) * W + 2 * xo + b;
            const Chan<V> sk = load_chan<V>(dcat + p * Cy + coff + c), m = load_chan<V>(y + p * C + c);
            Chan<V> o;
#pragma unroll
            for (int k = 0; k < V; ++k) {
                const float f = __bfloat162float(sk.e[k]) + __bfloat162float(g.e[k]);
                o.e[k] = __float2bfloat16_rn(__bfloat162float(m.e[k]) > 0.f ? f : 0.f);
            }
            store_chan<V>(dx + p * C + c, o);
        }
}

// 1x1 output head in FP32 arithmetic: out[p][o] = sum_c x[p][c] w[o][c] + b[o]; one thread per
// pixel and up to four outputs (blockIdx.y), or, without 16-byte reads and below 2^18 pixels or for one
// output, one per value: with 33 channels and five outputs 2.8 us for 1 x 64 x 64 pixels instead of 4.7, 11.4 for
// 32 x 64 x 64 instead of 11.9, but 75 instead of 69 for 4 x 512 x 512.
template <int V, int NO>
__global__ void head_fwd_kernel(const __nv_bfloat16 *__restrict__ x, const float *__restrict__ w,
                                const float *__restrict__ b, float *__restrict__ out, long long P, int C, int O) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x, p = NO == 1 ? i / O : i;
    const int o0 = NO == 1 ? (int)(i - p * O) : (int)blockIdx.y * NO, no = min(NO, O - o0);
    if (p >= P) return;
    float s[NO];
#pragma unroll
    for (int o = 0; o < NO; ++o) s[o] = o < no ? b[o0 + o] : 0.f;
    for (int c = 0; c < C; c += V) {
        const Chan<V> v = load_chan<V>(x + p * C + c);
#pragma unroll
        for (int k = 0; k < V; ++k)
#pragma unroll
            for (int o = 0; o < NO; ++o)
                if (o < no) s[o] = fmaf(__bfloat162float(v.e[k]), __ldg(w + (o0 + o) * C + c + k), s[o]);
    }
#pragma unroll
    for (int o = 0; o < NO; ++o)
        if (o < no) out[p * O + o0 + o] = s[o];
}

// dx[p][c] = sum_o dout[p][o] w[o][c], zero where `mask` (the ReLU output x, or NULL) is not positive
template <int V, class I>
__global__ void head_bwd_data_kernel(const float *__restrict__ dout, const float *__restrict__ w,
                                     const __nv_bfloat16 *__restrict__ mask, __nv_bfloat16 *__restrict__ dx,
                                     long long P, int C, int O) {
    const I i = (I)blockIdx.x * blockDim.x + threadIdx.x, G = C / V;
    const long long p = i / G;
    if (p >= P) return;
    const int c = (int)(i % G) * V;
    float s[V];
#pragma unroll
    for (int k = 0; k < V; ++k) s[k] = 0.f;
    for (int o = 0; o < O; ++o) {
        const float d = dout[p * O + o];
#pragma unroll
        for (int k = 0; k < V; ++k) s[k] = fmaf(d, __ldg(w + o * C + c + k), s[k]);
    }
    Chan<V> r;
    const Chan<V> m = mask ? load_chan<V>(mask + (long long)i * V) : Chan<V>{};
#pragma unroll
    for (int k = 0; k < V; ++k)
        r.e[k] = __float2bfloat16_rn(!mask || __bfloat162float(m.e[k]) > 0.f ? s[k] : 0.f);
    store_chan<V>(dx + (long long)i * V, r);
}

template <int N>
using Int = std::integral_constant<int, N>;

// dw[o][c] += sum_p dout[p][o] x[p][c]; db[o] += sum_p dout[p][o], for four outputs (blockIdx.y) and W
// channels (blockIdx.z).  A warp adds up `run` pixels, 32 / W at a time (lane = channel, pixel),
// in chains of 32 terms; the chains, the block's warps and the blocks of a cluster are added as
// trees, the latter through distributed shared memory, and a cluster makes one atomic addition per weight.
// run: at most 128, so that atomics come once in 8192 pixels, and less on small layers, down to four
// pixels and about 16 clusters.  Bound by the loads of a warp's pixels, about five each.  Relative error against
// 64 bits at 8192 pixels, 32 channels, five outputs: 1.1e-7; with 64-term chains and an atomic every 512 pixels
// 1.4e-7, with one block per weight and 8192 pixels 1.0e-7.  Time with the input's gradient, in the same order:
// 5.4, 19.5 and 4.9 us for 32 x 32 pixels (a launch with clusters costs about 1 us more), 22, 24 and 67 us for
// 32 x 64 x 64.
constexpr int kHeadRun = 128, kHeadCluster = 8;
template <int W>
__global__ void __cluster_dims__(kHeadCluster, 1, 1) __launch_bounds__(256)
    head_bwd_weight_kernel(const __nv_bfloat16 *__restrict__ x, const float *__restrict__ dout, float *__restrict__ dw,
                           float *__restrict__ db, long long P, int C, int O, int run) {
    constexpr int S = 32 / W;  // pixels of a warp side by side
    __shared__ float red[8][5][W], sum[5][W];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane / W, cl = lane % W;
    const int o0 = blockIdx.y * 4, c = blockIdx.z * W + cl, no = min(4, O - o0);
    const long long p0 = ((long long)blockIdx.x * 8 + warp) * run, p1 = min(P, p0 + run);
    // (lanes beyond the channels and, for the bias, beyond the outputs read valid places in vain)
    const __nv_bfloat16 *xp = x + (p0 + sub) * C + min(c, C - 1);
    const float *dp = dout + (p0 + sub) * O + o0;
    const int bo = min(cl, no - 1);
    float s[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    const auto add = [&](auto outputs) {
        constexpr int NO = decltype(outputs)::value;
        for (long long q = p0; q < p1; q += 32 * S) {
            float t[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
            const auto term = [&] {
                const float xv = __bfloat162float(*xp);
#pragma unroll
                for (int o = 0; o < NO; ++o) t[o] += dp[o] * xv;
                t[4] += dp[bo];
                xp += S * C;
                dp += S * O;
            };
            if (q + 32 * S <= p1) {
#pragma unroll 8
                for (int j = 0; j < 32; ++j) term();
            } else {
                for (long long p = q + sub; p < p1; p += S) term();
            }
#pragma unroll
            for (int o = 0; o < 5; ++o) s[o] += t[o];
        }
    };
    if (no == 4) add(Int<4>{});
    else if (no == 3) add(Int<3>{});
    else if (no == 2) add(Int<2>{});
    else add(Int<1>{});
#pragma unroll
    for (int d = W; d < 32; d *= 2)
#pragma unroll
        for (int o = 0; o < 5; ++o) s[o] += __shfl_xor_sync(0xffffffffu, s[o], d);
    if (sub == 0)
#pragma unroll
        for (int o = 0; o < 5; ++o) red[warp][o][cl] = s[o];
    __syncthreads();
    const int i = threadIdx.x, o = i / W, k = i % W;  // a sum of this thread, o < 5
    if (o < 5)
        sum[o][k] = ((red[0][o][k] + red[1][o][k]) + (red[2][o][k] + red[3][o][k])) +
                    ((red[4][o][k] + red[5][o][k]) + (red[6][o][k] + red[7][o][k]));
    const auto cluster = cooperative_groups::this_cluster();
    cluster.sync();
    if (cluster.block_rank() == 0 && o < 5) {
        float v[kHeadCluster];
#pragma unroll
        for (int r = 0; r < kHeadCluster; ++r) v[r] = *cluster.map_shared_rank(&sum[o][k], r);
        const float t = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
        const int ck = blockIdx.z * W + k;
        if (o < no && ck < C) atomicAdd(dw + (o0 + o) * C + ck, t);
        if (o == 4 && blockIdx.z == 0 && k < no) atomicAdd(db + o0 + k, t);
    }
    cluster.sync();  // no block leaves while its sums are read
}

// Mean squared error over n values; loss (FP32 sum, one atomic addition per block of 256 K values) and
// its gradient 2 (pred - target) / n.  K: eight values a thread, fewer where the blocks would not fill the
// chip.
template <int K>
__global__ void __launch_bounds__(256) mse_kernel(const float *__restrict__ pred, const float *__restrict__ target,
                                                  float *__restrict__ grad, float *__restrict__ loss, long long n) {
    const long long i0 = (long long)blockIdx.x * (256 * K) + threadIdx.x;
    float e = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const long long i = i0 + 256 * k;
        if (i < n) {
            const float d = pred[i] - target[i];
            grad[i] = 2.f * d / (float)n;
            e += d * d / (float)n;
        }
    }
    __shared__ float red[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_down_sync(0xffffffffu, e, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = e;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) t += red[k];
        atomicAdd(loss, t);
    }
}

// Adam on FP32 master weights; refreshes the BF16 copy when one is given.
__global__ void adam_kernel(float *__restrict__ w, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, __nv_bfloat16 *__restrict__ wb, long long n, float lr, float b1,
                            float b2, float eps, float c1, float c2) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    if (wb) wb[i] = __float2bfloat16_rn(wi);
}

inline unsigned blocks_for(long long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

// May a kernel take 8 channels a thread: all counts and offsets multiples of 8, all pointers on
// 16 bytes?
bool by_eight(std::initializer_list<long long> counts, std::initializer_list<const void *> pointers) {
    for (long long c : counts)
        if (c % 8) return false;
    for (const void *p : pointers)
        if (reinterpret_cast<uintptr_t>(p) & 15) return false;
    return true;
}
// f(Int<V>, index type) for n elements: 8 a thread and 32-bit indexes where possible.
template <class F>
void with_width(bool eight, long long n, const F &f) {
    if (n < (1ll << 30)) eight ? f(Int<8>{}, 0) : f(Int<1>{}, 0);
    else eight ? f(Int<8>{}, 0ll) : f(Int<1>{}, 0ll);
}

thread_local char g_nn_err[256] = "";
cdf_nn_status nn_fail(const char *m) {
    int i = 0;
    for (; m[i] && i < 255; ++i) g_nn_err[i] = m[i];
    g_nn_err[i] = 0;
    return CDF_NN_EINVAL;
}
cdf_nn_status launched() {
    const cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) return CDF_NN_OK;
    int i = 0;
    const char *m = cudaGetErrorString(e);
    for (; m[i] && i < 255; ++i) g_nn_err[i] = m[i];
    g_nn_err[i] = 0;
    return CDF_NN_ECUDA;
}

}  // namespace

extern "C" {

const char *cdf_nn_last_error(void) { return g_nn_err; }

cdf_nn_status cdf_nn_set_tensor_path(int tcgen05) {
    if (tcgen05 < 0 || tcgen05 > 4) return nn_fail("set_tensor_path: 0, 1, 2, 3 or 4");
    g_path = tcgen05;
    g_use_tc = tcgen05 != 0;
    return CDF_NN_OK;
}

cdf_nn_status cdf_nn_error_flag(int *out) {
    if (!out) return nn_fail("error_flag: NULL argument");
    const cudaError_t e = cudaMemcpyFromSymbol(out, g_tc_error, sizeof(int));
    if (e != cudaSuccess) return nn_fail(cudaGetErrorString(e));
    return CDF_NN_OK;
}

cdf_nn_status cdf_nn_conv3x3_fwd(const void *x, const void *w, const float *bias, void *y, int N, int H, int W,
                                 int Cin, int Cout, int relu, void *stream) {
    if (!x || !w || !y || N < 1 || H < 1 || W < 1 || Cin % 16 || Cout % 32 || Cin < 16)
        return nn_fail("conv3x3_fwd: bad arguments (Cin % 16, Cout % 32)");
    cudaError_t e = conv_dispatch<false>(static_cast<const __nv_bfloat16 *>(x), static_cast<const __nv_bfloat16 *>(w),
                                         bias, static_cast<__nv_bfloat16 *>(y), N, H, W, Cin, Cout, relu,
                                         static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) { cudaGetLastError(); return nn_fail(cudaGetErrorString(e)); }
    return launched();
}

cdf_nn_status cdf_nn_conv3x3_bwd_data(const void *dy, const void *w, void *dx, int N, int H, int W, int Cin, int Cout,
                                      void *stream) {
    if (!dy || !w || !dx || N < 1 || H < 1 || W < 1 || Cin % 16 || Cout % 32)
        return nn_fail("conv3x3_bwd_data: bad arguments (Cin % 16, Cout % 32)");
    cudaError_t e = conv_dispatch<true>(static_cast<const __nv_bfloat16 *>(dy), static_cast<const __nv_bfloat16 *>(w),
                                        nullptr, static_cast<__nv_bfloat16 *>(dx), N, H, W, Cout, Cin, 0,
                                        static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) { cudaGetLastError(); return nn_fail(cudaGetErrorString(e)); }
    return launched();
}

long long cdf_nn_conv3x3_bwd_weight_workspace(int N, int H, int W, int Cin, int Cout) {
    if (N < 1 || H < 1 || W < 1 || Cin < 16 || Cin % 16 || Cout < 32 || Cout % 32) return -1;
    long long most = 0;
    if (!wgrad_parts(N, H, W, [&](const WgradPart &p) {
            most = std::max(most, wgrad_bytes(wgrad_lin_plan(p.q1 - p.q0, p.P, Cin, Cout), Cin, Cout));
            return true;
        }))
        return 4;  // the warp-level kernel adds to dw directly
    return most;
}

cdf_nn_status cdf_nn_conv3x3_bwd_weight(const void *x, const void *dy, float *dw, float *db, int N, int H, int W,
                                        int Cin, int Cout, void *workspace, long long workspace_bytes, void *stream) {
    if (!x || !dy || !dw || N < 1 || H < 1 || W < 1 || Cin % 16 || Cout % 32)
        return nn_fail("conv3x3_bwd_weight: bad arguments (Cin % 16, Cout % 32)");
    const long long P = (long long)N * H * W;
    auto s = static_cast<cudaStream_t>(stream);
    const auto *xb = static_cast<const __nv_bfloat16 *>(x);
    const auto *dyb = static_cast<const __nv_bfloat16 *>(dy);
    const long long need = g_use_tc ? cdf_nn_conv3x3_bwd_weight_workspace(N, H, W, Cin, Cout) : 4;
    if (need > 4) {
        if (!workspace || workspace_bytes < need)
            return nn_fail("conv3x3_bwd_weight: the workspace is missing or smaller than "
                           "cdf_nn_conv3x3_bwd_weight_workspace()");
        // weight_sum_kernel reads it 16 bytes at a time
        if (reinterpret_cast<uintptr_t>(workspace) & 15)
            return nn_fail("conv3x3_bwd_weight: the workspace must begin on a multiple of 16 bytes");
        float *part = static_cast<float *>(workspace);
        cudaError_t e = cudaSuccess;
        wgrad_parts(N, H, W, [&](const WgradPart &p) {
            LinImage im;
            if (!lin_image(p.n, p.H, W, &im)) e = cudaErrorInvalidValue;
            const WgLinPlan w = wgrad_lin_plan(p.q1 - p.q0, p.P, Cin, Cout);
            for (int s0 = 0; s0 < w.splits && e == cudaSuccess; s0 += w.run) {
                const int splits = std::min(w.run, w.splits - s0);
                // the bias gradient goes with the first launch, its partial sums behind the weights'
                float *bpart = db && s0 == 0 ? part + (long long)w.run * 9 * Cin * Cout : nullptr;
                e = wgrad_lin(xb + p.first * Cin, dyb + p.first * Cout, part, bpart, im, p.q0 + s0 * w.per,
                              (int)std::min<long long>(p.q1, p.q0 + (long long)(s0 + splits) * w.per), p.p0, p.P, Cin,
                              Cout, w, splits, s);
                if (e != cudaSuccess) break;
                const auto sum = [&](auto r) {
                    constexpr int R = decltype(r)::value;
                    const int n4 = 9 * Cin * Cout / 4, wblocks = (n4 + R - 1) / R;
                    const int bblocks = bpart ? (Cout / 4 + R - 1) / R : 0;
                    weight_sum_kernel<R><<<wblocks + bblocks, 256, 0, s>>>(part, dw, n4, splits, wblocks, bpart, db,
                                                                           Cout / 4, w.bias_splits);
                };
                if (splits >= 128) sum(std::integral_constant<int, 8>{});
                else sum(std::integral_constant<int, 32>{});
            }
            return e == cudaSuccess;
        });
        if (e != cudaSuccess) { cudaGetLastError(); return nn_fail(cudaGetErrorString(e)); }
    } else {
        // the warp-level MMA path: split-K partial sums added atomically (order-dependent)
        // (at most 65,535 splits, the layers of a grid)
        const long long per = std::max(4096ll, ((P + 65534) / 65535 + kWBK - 1) / kWBK * kWBK);
        dim3 grid((unsigned)((Cout + kWBM - 1) / kWBM), 9 * (Cin / 16), (unsigned)((P + per - 1) / per));
        conv3x3_wgrad_kernel<<<grid, kThreads, 0, s>>>(xb, dyb, dw, N, H, W, Cin, Cout, per);
        if (db) {
            dim3 g2(Cout / 8, (unsigned)std::min(65535ll, (P + 256 * 64 - 1) / (256 * 64)));
            bias_grad_kernel<<<g2, 256, 0, s>>>(dyb, db, P, Cout);
        }
    }
    return launched();
}

cdf_nn_status cdf_nn_relu_bwd(void *d, const void *y, long long n, void *stream) {
    if (!d || !y || n < 0) return nn_fail("relu_bwd: bad arguments");
    if (n)
        with_width(by_eight({n}, {d, y}), n, [&](auto v, auto) {
            constexpr int V = decltype(v)::value;
            relu_bwd_kernel<V><<<blocks_for(n / V), 256, 0, static_cast<cudaStream_t>(stream)>>>(
                static_cast<__nv_bfloat16 *>(d), static_cast<const __nv_bfloat16 *>(y), n);
        });
    return launched();
}

cdf_nn_status cdf_nn_avgpool2_fwd(const void *x, void *y, int N, int H, int W, int C, void *stream) {
    if (!x || !y || H % 2 || W % 2) return nn_fail("avgpool2: H and W must be even");
    const long long n = (long long)N * (H / 2) * (W / 2) * C;
    with_width(by_eight({C}, {x, y}), n, [&](auto v, auto index) {
        constexpr int V = decltype(v)::value;
        avgpool2_fwd_kernel<V, decltype(index)><<<blocks_for(n / V), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const __nv_bfloat16 *>(x), static_cast<__nv_bfloat16 *>(y), N, H, W, C);
    });
    return launched();
}

cdf_nn_status cdf_nn_avgpool2_bwd(const void *dy, void *dx, int N, int H, int W, int C, void *stream) {
    if (!dy || !dx || H % 2 || W % 2) return nn_fail("avgpool2: H and W must be even");
    const long long n = (long long)N * (H / 2) * (W / 2) * C;
    with_width(by_eight({C}, {dy, dx}), 4 * n, [&](auto v, auto index) {
        constexpr int V = decltype(v)::value;
        avgpool2_bwd_kernel<V, decltype(index)><<<blocks_for(n / V), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const __nv_bfloat16 *>(dy), static_cast<__nv_bfloat16 *>(dx), N, H, W, C);
    });
    return launched();
}

cdf_nn_status cdf_nn_upsample2_fwd(const void *x, void *y, int N, int H, int W, int C, int Cy, int coff, void *stream) {
    if (!x || !y || coff < 0 || coff + C > Cy) return nn_fail("upsample2: bad channel slice");
    const long long n = (long long)N * H * W * C;
    with_width(by_eight({C, Cy, coff}, {x, y}), 4 * n, [&](auto v, auto index) {
        constexpr int V = decltype(v)::value;
        upsample2_fwd_kernel<V, decltype(index)><<<blocks_for(n / V), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const __nv_bfloat16 *>(x), static_cast<__nv_bfloat16 *>(y), N, H, W, C, Cy, coff);
    });
    return launched();
}

cdf_nn_status cdf_nn_upsample2_bwd(const void *dy, void *dx, int N, int H, int W, int C, int Cy, int coff, void *stream) {
    if (!dy || !dx || coff < 0 || coff + C > Cy) return nn_fail("upsample2: bad channel slice");
    const long long n = (long long)N * H * W * C;
    with_width(by_eight({C, Cy, coff}, {dy, dx}), n, [&](auto v, auto index) {
        constexpr int V = decltype(v)::value;
        upsample2_bwd_kernel<V, decltype(index)><<<blocks_for(n / V), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const __nv_bfloat16 *>(dy), static_cast<__nv_bfloat16 *>(dx), N, H, W, C, Cy, coff);
    });
    return launched();
}

cdf_nn_status cdf_nn_copy_channels(const void *x, void *y, long long P, int Cx, int Cy, int src_off, int dst_off,
                                   int count, int accumulate, void *stream) {
    if (!x || !y || src_off + count > Cx || dst_off + count > Cy || count < 0) return nn_fail("copy_channels: bad slice");
    const long long n = P * count;
    if (n)
        with_width(by_eight({Cx, Cy, src_off, dst_off, count}, {x, y}), n, [&](auto v, auto index) {
            constexpr int V = decltype(v)::value;
            copy_channels_kernel<V, decltype(index)><<<blocks_for(n / V), 256, 0, static_cast<cudaStream_t>(stream)>>>(
                static_cast<const __nv_bfloat16 *>(x), static_cast<__nv_bfloat16 *>(y), P, Cx, Cy, src_off, dst_off,
                count, accumulate);
        });
    return launched();
}

cdf_nn_status cdf_nn_head_fwd(const void *x, const float *w, const float *b, float *out, long long P, int C, int O,
                              void *stream) {
    if (!x || !w || !b || !out) return nn_fail("head_fwd: NULL argument");
    with_width(by_eight({C}, {x}), P * C, [&](auto v, auto) {
        constexpr int V = decltype(v)::value;
        const auto run = [&](auto outputs) {
            constexpr int NO = decltype(outputs)::value;
            const dim3 grid = NO == 1 ? dim3(blocks_for(P * O)) : dim3(blocks_for(P), (unsigned)((O + NO - 1) / NO));
            head_fwd_kernel<V, NO><<<grid, 256, 0, static_cast<cudaStream_t>(stream)>>>(
                static_cast<const __nv_bfloat16 *>(x), w, b, out, P, C, O);
        };
        if constexpr (V == 1) {
            if (O == 1 || P < (1 << 18)) return run(Int<1>{});
        }
        run(Int<4>{});
    });
    return launched();
}

static cdf_nn_status head_bwd(const void *x, const float *w, const float *dout, void *dx, float *dw, float *db,
                              long long P, int C, int O, bool relu, void *stream) {
    if (!x || !w || !dout || !dx || !dw || !db) return nn_fail("head_bwd: NULL argument");
    auto s = static_cast<cudaStream_t>(stream);
    const auto *xb = static_cast<const __nv_bfloat16 *>(x);
    with_width(by_eight({C}, {dx, x}), P * C, [&](auto v, auto index) {
        constexpr int V = decltype(v)::value;
        head_bwd_data_kernel<V, decltype(index)><<<blocks_for(P * C / V), 256, 0, s>>>(
            dout, w, relu ? xb : nullptr, static_cast<__nv_bfloat16 *>(dx), P, C, O);
    });
    const auto weights = [&](auto width) {
        constexpr int W = decltype(width)::value;
        const int run = (int)std::min<long long>(kHeadRun, std::max(4ll, (P + 1023) / 1024));
        const long long clusters = (P + 8 * kHeadCluster * run - 1) / (8 * kHeadCluster * run);
        head_bwd_weight_kernel<W><<<dim3((unsigned)(clusters * kHeadCluster), (O + 3) / 4, (C + W - 1) / W), 256, 0, s>>>(
            xb, dout, dw, db, P, C, O, run);
    };
    if (C <= 8) weights(Int<8>{});
    else if (C <= 16) weights(Int<16>{});
    else weights(Int<32>{});
    return launched();
}

cdf_nn_status cdf_nn_head_bwd(const void *x, const float *w, const float *dout, void *dx, float *dw, float *db,
                              long long P, int C, int O, void *stream) {
    return head_bwd(x, w, dout, dx, dw, db, P, C, O, false, stream);
}

cdf_nn_status cdf_nn_head_bwd_relu(const void *x, const float *w, const float *dout, void *dx, float *dw, float *db,
                                   long long P, int C, int O, void *stream) {
    return head_bwd(x, w, dout, dx, dw, db, P, C, O, true, stream);
}

cdf_nn_status cdf_nn_conv3x3_bwd_data_relu(const void *dy, const void *w, const void *y, void *dx, int N, int H, int W,
                                           int Cin, int Cout, void *stream) {
    if (!dy || !w || !y || !dx || N < 1 || H < 1 || W < 1 || Cin % 16 || Cout % 32)
        return nn_fail("conv3x3_bwd_data_relu: bad arguments (Cin % 16, Cout % 32)");
    const auto s = static_cast<cudaStream_t>(stream);
    if ((g_path == 1 || g_path == 4) && !(reinterpret_cast<uintptr_t>(y) & 15)) {
        bool ran = false;
        const cudaError_t e = conv_lin<true>(static_cast<const __nv_bfloat16 *>(dy), static_cast<const __nv_bfloat16 *>(w),
                                             nullptr, static_cast<const __nv_bfloat16 *>(y),
                                             static_cast<__nv_bfloat16 *>(dx), N, H, W, Cout, Cin, 0, s, &ran);
        if (e != cudaSuccess) { cudaGetLastError(); return nn_fail(cudaGetErrorString(e)); }
        if (ran) return launched();
    }
    const cdf_nn_status st = cdf_nn_conv3x3_bwd_data(dy, w, dx, N, H, W, Cin, Cout, stream);
    return st != CDF_NN_OK ? st : cdf_nn_relu_bwd(dx, y, (long long)N * H * W * Cin, stream);
}

cdf_nn_status cdf_nn_upsample2_concat(const void *x, const void *skip, void *y, int N, int H, int W, int C, int Cs,
                                      void *stream) {
    if (!x || !skip || !y || N < 1 || H < 1 || W < 1 || C < 1 || Cs < 1) return nn_fail("upsample2_concat: bad arguments");
    const long long n = (long long)N * H * W * (C + 4ll * Cs);
    with_width(by_eight({C, Cs}, {x, skip, y}), 4 * n, [&](auto v, auto index) {
        constexpr int V = decltype(v)::value;
        upsample2_concat_kernel<V, decltype(index)><<<blocks_for(n / V), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const __nv_bfloat16 *>(x), static_cast<const __nv_bfloat16 *>(skip),
            static_cast<__nv_bfloat16 *>(y), N, H, W, C, Cs);
    });
    return launched();
}

cdf_nn_status cdf_nn_upsample2_bwd_relu(const void *dy, const void *y, void *dx, int N, int H, int W, int C, int Cy,
                                        void *stream) {
    if (!dy || !y || !dx || N < 1 || H < 1 || W < 1 || C < 1 || C > Cy) return nn_fail("upsample2_bwd_relu: bad arguments");
    const long long n = (long long)N * H * W * C;
    with_width(by_eight({C, Cy}, {dy, y, dx}), n, [&](auto v, auto index) {
        constexpr int V = decltype(v)::value;
        upsample2_bwd_relu_kernel<V, decltype(index)><<<blocks_for(n / V), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const __nv_bfloat16 *>(dy), static_cast<const __nv_bfloat16 *>(y),
            static_cast<__nv_bfloat16 *>(dx), N, H, W, C, Cy);
    });
    return launched();
}

cdf_nn_status cdf_nn_pool_skip_bwd_relu(const void *dp, const void *dcat, const void *y, void *dx, int N, int H, int W,
                                        int C, int Cy, int coff, void *stream) {
    if (!dp || !dcat || !y || !dx || N < 1 || H < 2 || W < 2 || H % 2 || W % 2 || C < 1 || coff < 0 || coff + C > Cy)
        return nn_fail("pool_skip_bwd_relu: bad arguments (H and W even, coff + C <= Cy)");
    const long long n = (long long)N * (H / 2) * (W / 2) * C;
    with_width(by_eight({C, Cy, coff}, {dp, dcat, y, dx}), 4 * n, [&](auto v, auto index) {
        constexpr int V = decltype(v)::value;
        pool_skip_bwd_relu_kernel<V, decltype(index)><<<blocks_for(n / V), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const __nv_bfloat16 *>(dp), static_cast<const __nv_bfloat16 *>(dcat),
            static_cast<const __nv_bfloat16 *>(y), static_cast<__nv_bfloat16 *>(dx), N, H, W, C, Cy, coff);
    });
    return launched();
}

cdf_nn_status cdf_nn_mse(const float *pred, const float *target, float *grad, float *loss, long long n, void *stream) {
    if (!pred || !target || !grad || !loss) return nn_fail("mse: NULL argument");
    const auto run = [&](auto values) {
        constexpr int K = decltype(values)::value;
        mse_kernel<K><<<blocks_for(n, 256 * K), 256, 0, static_cast<cudaStream_t>(stream)>>>(pred, target, grad, loss, n);
    };
    if (n <= 256 * 152) run(Int<1>{});
    else run(Int<8>{});
    return launched();
}

cdf_nn_status cdf_nn_adam(float *w, const float *g, float *m, float *v, void *w_bf16, long long n, float lr, float b1,
                          float b2, float eps, long long step, void *stream) {
    if (!w || !g || !m || !v || step < 1) return nn_fail("adam: bad arguments");
    float c1 = 1.f, c2 = 1.f, p1 = 1.f, p2 = 1.f;
    for (long long i = 0; i < step && i < 100000; ++i) { p1 *= b1; p2 *= b2; }
    c1 -= p1;
    c2 -= p2;
    adam_kernel<<<blocks_for(n), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        w, g, m, v, static_cast<__nv_bfloat16 *>(w_bf16), n, lr, b1, b2, eps, c1, c2);
    return launched();
}

}  // extern "C"
