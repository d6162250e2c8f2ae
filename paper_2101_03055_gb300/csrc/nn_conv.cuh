// 3x3 convolutions (forward, gradient of the input, gradient of the weights) on
// the 5th-generation tensor cores without im2col copies, for any image size.
// Included by nn_kernels.cu inside its anonymous namespace.
//
// All three use one view of the image batch: its pixels in a row, padded.  The
// linear position q = (n (H + 1) + y) (W + 1) + x runs over every image with one
// zero column after each row and one zero row after each image; the zero column
// is the right padding of its row and the left padding of the next, the zero row
// the bottom padding of its image and the top padding of the next.  The pixel
// that tap (ky, kx) reads for position q is then always q + (ky - 1)(W + 1) +
// (kx - 1): a shift that does not depend on the pixel.  Staged in shared memory
// as [channel group of 8][position][16 bytes], eight consecutive positions of
// one group are one 128-byte core matrix, so every tap's operand is the same
// staged slab seen through a descriptor whose start moves 16 bytes per position.
// Each input element is staged once per CTA instead of once per tap.  The padding
// positions cost (W + H + 1) / ((W + 1)(H + 1)) of the rows (3 % at 64 x 64).
//
// Measured on GB300 (launches in a CUDA graph; before: the im2col kernels, forward rows of
// whole 128-pixel tiles without im2col), forward / input gradient / weight and bias gradient:
//   16 x 256 x 256, 32 -> 32     91 / 286 / 451 us before,  53 / 55 / 115 us now
//   16 x 32 x 32, 256 -> 256    116 / 206 / 163 us before,  26 / 28 / 59 us now (750 TFLOP/s forward)
//   the U-Net's first eleven layer shapes at 32 x 64 x 64, summed: 741 / 1050 / 1123 us before, 128 / 138 / 217 us now

// Division of 0 <= x < 2^31 by a constant d >= 1: (umulhi(x, mul) + x) >> shift
// (Granlund & Montgomery, PLDI 1994, the round-up multiplier of 33 bits).
struct FastDiv {
    uint32_t mul, shift;
};
inline FastDiv fast_div(uint32_t d) {
    uint32_t s = 0;
    while ((1ull << s) < d) ++s;
    return FastDiv{(uint32_t)(((1ull << 32) * ((1ull << s) - d)) / d + 1), s};
}
__device__ __forceinline__ int div_by(int x, FastDiv d) {
    return (int)((__umulhi((uint32_t)x, d.mul) + (uint32_t)x) >> d.shift);
}

// The padded row of pixels of one image batch, and the division constants.
struct LinImage {
    int H, W, L;        // L = N (H + 1) (W + 1) positions
    int Wp, Hp;         // W + 1, H + 1
    FastDiv dw, dh;
};
inline bool lin_image(int N, int H, int W, LinImage *im) {
    const long long L = (long long)N * (H + 1) * (W + 1);
    if (L >= (1ll << 30)) return false;
    *im = LinImage{H, W, (int)L, W + 1, H + 1, fast_div((uint32_t)W + 1), fast_div((uint32_t)H + 1)};
    return true;
}
// Pixel index (n H + y) W + x of position q, or -1 for padding and outside.
__device__ __forceinline__ int lin_pixel(const LinImage &im, int q) {
    if (q < 0 || q >= im.L) return -1;
    const int row = div_by(q, im.dw), x = q - row * im.Wp;
    const int n = div_by(row, im.dh), y = row - n * im.Hp;
    return (x < im.W && y < im.H) ? (row - n) * im.W + x : -1;
}

// Positions per channel group in shared memory for `count` staged ones: the
// copies write 16 bytes per thread, channel group fastest, and eight threads fall
// into eight different bank groups when the stride is 4 mod 8 (two groups),
// 2 mod 4 (four groups) or odd (more).
inline int lin_stride(int count, int G) {
    if (G == 2) return (count + 3) / 8 * 8 + 4;
    if (G == 4) return (count + 1) / 4 * 4 + 2;
    return count | 1;
}

// Descriptor of a swizzled operand tile (layout type: 2 = 128, 4 = 64, 6 = 32 bytes).
__device__ __forceinline__ uint64_t smem_desc_sw(uint32_t addr, uint32_t lbo, uint32_t sbo, uint32_t type) {
    return smem_desc(addr, lbo, sbo) | ((uint64_t)type << 61);
}
// One thread of a warp (the same each time); the caller's warp is converged.
__device__ __forceinline__ uint32_t elect_lane() {
    uint32_t lead;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(lead));
    return lead;
}
// MMA and commit by the lane with lead != 0.  The whole warp runs the code around
// them, so that the descriptors stay in uniform registers, where the instruction
// takes them; computed under a branch of one thread they have to be moved there
// one by one before every MMA.
__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc,
                                        uint32_t lead) {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(lead)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar, uint32_t lead) {
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
        " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(bar),
        "r"(lead)
        : "memory");
}
template <int COLS>
__device__ __forceinline__ void tmem_load(uint32_t addr, uint32_t (&r)[COLS]) {
    static_assert(COLS == 16, "16 columns a load");
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(addr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ---------------------------------------------------------------------------
// Forward and input gradient.  An item is T tiles of 128 consecutive positions (one
// TMEM accumulator of BN columns each) and BN output channels; a CTA walks the items
// blockIdx.x, blockIdx.x + gridDim.x, ..  Its warps have fixed roles:
//   warps 4-11  stage the positions an item's tiles read, with all input channels, by
//               cp.async into one of `nbuf` slabs;
//   warp 13     brings the weights by TMA, 128 of K at a time (forward: W[co][k], K-major;
//               gradient: W[co][8 - tap][ci] as it lies, N-major), once where all of
//               them fit in the ring, else again for every item;
//   warp 12     issues the MMAs;
//   warps 0-3   read the accumulators, add the bias, apply the ReLU (gradient: zero where
//               `mask`, the ReLU output that fed the layer, is not positive) and store BF16.
// With nbuf = 2 the next item's copies, this one's MMAs and the last one's stores
// overlap inside a CTA, with nbuf = 1 (less shared memory) between the CTAs of an SM.
// K runs tap by tap, 16 channels at a time, as in conv3x3_tc_kernel: the same sums in
// the same order, the same bits.  Bound: with 32 output channels the MMA's own read of
// A from shared memory (45 cycles per 128 x 16 slice, of which 16 are arithmetic), with
// 256 the arithmetic; small layers by the latencies of one item.
// Every wait is bounded: a thread whose wait runs out sets g_tc_error and an abort flag
// that ends the others' waits; copies and MMAs in flight are waited for before the CTA ends.
// ---------------------------------------------------------------------------
constexpr int kLinThreads = 448, kLinStagers = 256;
constexpr int kLinK = 128;  // K per ring buffer, two 64-wide halves
constexpr int kLinMaxStages = 8;
constexpr int kLinMaxSlices = 512;  // K / 16: up to 896 channels

struct LinConv {
    LinImage im;
    int Cin, Cout;      // of the GEMM: K channels and output channels
    FastDiv dg, dc;     // by Cin / 8 and by Cin
    int T, sp;          // tiles of 128 positions per item, positions per staged group
    int nbuf;           // slabs, and sets of T accumulators
    int items;          // position items, ceil(L / (128 T))
    int cols;           // tensor-memory columns
    int stages;         // ring buffers, kLinK of K each
    int boxk;           // gradient: K per TMA box, 64, or 32 where a tap's channels are no multiple of 64
    int relu;
};

// The issuing warp: the MMAs of all K stages of one item, eight slices of 16 channels a
// stage.  A slice of 128 x 16 times 32 or 64 columns takes the tensor core 45 or 48 cycles
// (measured, any operand layout), so what one warp issues around the MMAs counts:
// `slice_at` holds the slices' A addresses, everything else in the descriptors is fixed,
// and the waits, the commit and the ring's arithmetic are paid once per eight slices (with
// four, 520 cycles a stage at T = 1; with eight, 650).
struct LinRing {
    uint32_t full, empty, last;  // barriers of buffer 0, and full barrier of the last buffer
    uint32_t fb, eb, phase, off;  // current buffer: barriers, phase, address (16-byte units)
};
template <int T, int BN, bool kFirst>
__device__ __forceinline__ void issue_slices(const uint4 *at, uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t kadv,
                                             uint32_t khalf, uint32_t idesc, uint32_t lead) {
    const uint4 lo = at[0], hi = at[1];
    const uint32_t a[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int t = 0; t < T; ++t)
            mma_f16(tmem + (uint32_t)(t * BN), ad + a[j] + (uint32_t)(t * 128),
                    bd + (uint32_t)(j & 3) * kadv + (uint32_t)(j >> 2) * khalf, idesc, kFirst && j == 0 ? 0u : 1u, lead);
}
template <int T, int BN>
__device__ __forceinline__ bool issue_item(const uint32_t *slice_at, uint32_t tmem, uint64_t ad, uint64_t bd,
                                           uint32_t kadv, uint32_t khalf, uint32_t idesc, int slices, LinRing &r,
                                           uint32_t lead, volatile int *abort) {
    constexpr uint32_t kStage = BN * kLinK * 2 / 16;
    const uint4 *at = reinterpret_cast<const uint4 *>(slice_at);
    for (int left = slices; left > 0; left -= 8, at += 2) {
        if (!ws_wait(r.fb, r.phase, abort)) return false;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t bs = bd + r.off;
        if (left == slices) {  // (K = 9 channels >= 144: the first stage is whole)
            issue_slices<T, BN, true>(at, tmem, ad, bs, kadv, khalf, idesc, lead);
        } else if (left >= 8) {
            issue_slices<T, BN, false>(at, tmem, ad, bs, kadv, khalf, idesc, lead);
        } else {
            for (int j = 0; j < left; ++j)
#pragma unroll
                for (int t = 0; t < T; ++t)
                    mma_f16(tmem + (uint32_t)(t * BN), ad + reinterpret_cast<const uint32_t *>(at)[j] + (uint32_t)(t * 128),
                            bs + (uint32_t)(j & 3) * kadv + (uint32_t)(j >> 2) * khalf, idesc, 1u, lead);
        }
        mma_commit(r.eb, lead);
        const bool wrap = r.fb == r.last;
        r.off = wrap ? 0u : r.off + kStage;
        r.fb = wrap ? r.full : r.fb + 8;
        r.eb = wrap ? r.empty : r.eb + 8;
        r.phase ^= wrap ? 1u : 0u;
    }
    return true;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
// A wait of a whole warp, polled by one lane.
__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity, int lane, volatile int *abort) {
    bool ok = true;
    if (lane == 0) ok = ws_wait(smem_u32(bar), parity, abort);
    return __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
}

template <bool kBwd, int BN>
__global__ void __launch_bounds__(kLinThreads) conv3x3_lin_kernel(const __grid_constant__ CUtensorMap wmap,
                                                                  const __nv_bfloat16 *__restrict__ in,
                                                                  const float *__restrict__ bias,
                                                                  const __nv_bfloat16 *__restrict__ mask,
                                                                  __nv_bfloat16 *__restrict__ out, const LinConv g) {
    extern __shared__ __align__(1024) unsigned char lin_raw[];
    unsigned char *const lin_smem = lin_raw + ((1024u - (smem_u32(lin_raw) & 1023u)) & 1023u);
    __shared__ __align__(8) uint64_t full[kLinMaxStages], empty[kLinMaxStages];      // weights' ring
    __shared__ __align__(8) uint64_t slab_full[2], slab_empty[2], acc_full[2], acc_empty[2], done;
    __shared__ __align__(16) uint32_t slice_at[kLinMaxSlices];
    __shared__ __align__(16) float sbias[BN];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int n0 = blockIdx.y * BN, item_len = g.T * 128;
    constexpr uint32_t bbytes = BN * kLinK * 2;
    const uint32_t slab_bytes = (uint32_t)((g.Cin >> 3) * g.sp) * 16;
    unsigned char *const ring = lin_smem, *const slab = lin_smem + g.stages * bbytes;
    const int K = 9 * g.Cin, nst = (K + kLinK - 1) / kLinK;
    const bool resident = nst <= g.stages;

    if (warp == 12) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"((uint32_t)g.cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // stage s of an item's weights into ring buffer b
    const auto load_weights = [&](int s, int b) {
        const uint32_t bar = smem_u32(&full[b]);
        unsigned char *dst = ring + b * bbytes;
        const int k0 = s * kLinK, kn = min(kLinK, K - k0);  // a multiple of 16
        if (!kBwd) {
            // one box of 64 x BN for each half (the part beyond K comes as zeros)
            const int boxes = (kn + 63) / 64;
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                         "r"((uint32_t)(boxes * BN * 128))
                         : "memory");
            for (int i = 0; i < boxes; ++i)
                asm volatile(
                    "cp.async.bulk.tensor.2d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
                    "[%4];" ::"r"(smem_u32(dst + i * BN * 128)),
                    "l"(&wmap), "r"(k0 + i * 64), "r"(n0), "r"(bar)
                    : "memory");
        } else {
            // boxes of boxk output channels of one tap (K is a multiple of boxk here)
            constexpr int kBox = BN < 64 ? BN : 64;
            const int boxes = kn / g.boxk;
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"((uint32_t)(kn * BN * 2))
                         : "memory");
            for (int i = 0; i < boxes; ++i) {
                const int k = k0 + i * g.boxk, tap = div_by(k, g.dc), co = k - tap * g.Cin;
#pragma unroll
                for (int a = 0; a < BN / kBox; ++a)
                    asm volatile(
                        "cp.async.bulk.tensor.3d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
                        "%4}], [%5];" ::"r"(smem_u32(dst + (a * kLinK + i * g.boxk) * kBox * 2)),
                        "l"(&wmap), "r"(n0 + a * kBox), "r"(8 - tap), "r"(co), "r"(bar)
                        : "memory");
            }
        }
    };
    if (tid == 13 * 32) {
        for (int b = 0; b < g.stages; ++b) {
            mbar_init(&full[b], 1);
            mbar_init(&empty[b], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&slab_full[b], kLinStagers / 32);
            mbar_init(&slab_empty[b], 1);
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 4);
        }
        mbar_init(&done, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (int s = 0; s < g.stages && s < nst; ++s) load_weights(s, s);
    }
    // slice k: 16 channels from c on of tap (ky, kx); A's address in 16-byte units from the slab's start
    if (warp < 12)
        for (int k = tid; k < K / 16; k += 12 * 32) {
            const int tap = div_by(16 * k, g.dc), c = 16 * k - tap * g.Cin, ky = tap / 3, kx = tap - 3 * ky;
            slice_at[k] = (uint32_t)((c >> 3) * g.sp + ky * g.im.Wp + kx);
        }
    for (int c = tid; c < BN; c += kLinThreads) sbias[c] = bias ? bias[n0 + c] : 0.f;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;

    if (warp >= 4 && warp < 12) {
        // ---- staging: the positions q0 - (W + 2) .. q0 + 128 T + W + 1, channel group fastest
        const int G = g.Cin >> 3, total = (item_len + 2 * (g.im.Wp + 1)) * G;
        int b = 0;
        uint32_t phase = 1;  // both slabs are empty at first
        for (int item = blockIdx.x; item < g.items; item += gridDim.x) {
            if (!warp_wait(&slab_empty[b], phase, lane, &abort_flag)) break;
            unsigned char *const dst = slab + b * slab_bytes;
            const int qs = item * item_len - (g.im.Wp + 1);
#pragma unroll 4
            for (int e = tid - 128; e < total; e += kLinStagers) {
                const int pos = div_by(e, g.dg), grp = e - pos * G;
                const int px = lin_pixel(g.im, qs + pos);
                cp_async16(dst + (grp * g.sp + pos) * 16, px >= 0 ? in + (long long)px * g.Cin + grp * 8 : in,
                           px >= 0 ? 16 : 0);
            }
            cp_async_commit();
            cp_async_wait<0>();
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&slab_full[b]));
            if (++b == g.nbuf) {
                b = 0;
                phase ^= 1;
            }
        }
    } else if (warp == 12) {
        // ---- MMAs
        const uint32_t lead = elect_lane();
        // B: forward K-major, 128-byte rows of 64 k; gradient N-major, atoms of 64 (32, 16) channels
        constexpr uint32_t idesc = mma_idesc(128, BN) | (kBwd ? 1u << 16 : 0u);
        constexpr uint32_t type = !kBwd || BN >= 64 ? 2u : (BN == 32 ? 4u : 6u);
        constexpr uint32_t row = kBwd ? (BN >= 64 ? 128u : BN * 2u) : 128u;  // bytes of one swizzled row
        constexpr uint32_t kadv = (kBwd ? 16u * row : 32u) >> 4, khalf = (kBwd ? 64u * row : BN * 128u) >> 4;
        const uint64_t bd = smem_desc_sw(smem_u32(ring), kBwd ? kLinK * row : 16u, 8 * row, type);
        const uint32_t f0 = smem_u32(full), e0 = smem_u32(empty);
        LinRing r{f0, e0, f0 + 8u * (uint32_t)(g.stages - 1), f0, e0, 0, 0};
        int b = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int item = blockIdx.x; item < g.items && ok; item += gridDim.x) {
            ok = ws_wait(smem_u32(&acc_empty[b]), phase ^ 1, &abort_flag) &&
                 ws_wait(smem_u32(&slab_full[b]), phase, &abort_flag);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (resident) r = LinRing{f0, e0, r.last, f0, e0, 0, 0};  // each buffer was filled once
            const uint64_t ad = smem_desc(smem_u32(slab + b * slab_bytes), (uint32_t)g.sp * 16, 128);
            const uint32_t acc = tmem + (uint32_t)(b * g.T * BN);
#define CDF_ISSUE(TT) \
    ok = issue_item<TT, BN>(slice_at, acc, ad, bd, kadv, khalf, idesc, K / 16, r, lead, &abort_flag)
            if (BN <= 64 && g.T == 8) CDF_ISSUE(BN <= 64 ? 8 : 1);
            else if (BN <= 128 && g.T == 4) CDF_ISSUE(BN <= 128 ? 4 : 1);
            else if (g.T == 2) CDF_ISSUE(2);
            else CDF_ISSUE(1);
#undef CDF_ISSUE
            mma_commit(smem_u32(&slab_empty[b]), lead);
            mma_commit(smem_u32(&acc_full[b]), lead);
            if (++b == g.nbuf) {
                b = 0;
                phase ^= 1;
            }
        }
        // every MMA is done before the tensor memory is released, also after a time-out
        mma_commit(smem_u32(&done), lead);
        mbar_wait(smem_u32(&done), 0);
    } else if (warp == 13) {
        // ---- weights behind the first ring's worth: a thread of its own, because the wait for
        // a buffer's MMAs would hold up the next ones
        if (lane == 0) {
            long long loaded = nst < g.stages ? nst : g.stages;
            if (!resident) {
                const long long all = (long long)((g.items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1) * nst;
                int s = g.stages, b = 0;  // g.stages < nst
                uint32_t phase = 0;
                for (; loaded < all; ++loaded) {
                    if (!ws_wait(smem_u32(&empty[b]), phase, &abort_flag)) break;
                    load_weights(s, b);
                    if (++s == nst) s = 0;
                    if (++b == g.stages) {
                        b = 0;
                        phase ^= 1;
                    }
                }
            }
            // every copy has landed before the CTA ends, also after a time-out
            for (long long k = loaded > g.stages ? loaded - g.stages : 0; k < loaded; ++k)
                mbar_wait(smem_u32(&full[k % g.stages]), (uint32_t)((k / g.stages) & 1));
        }
    } else if (warp < 4) {
        // ---- results: TMEM lane = position, 32 (16) channels at a time
        constexpr int kChunk = BN < 32 ? BN : 32;
        int b = 0;
        uint32_t phase = 0;
        for (int item = blockIdx.x; item < g.items; item += gridDim.x) {
            if (!warp_wait(&acc_full[b], phase, lane, &abort_flag)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int t = 0; t < g.T; ++t) {
                const int px = lin_pixel(g.im, item * item_len + t * 128 + warp * 32 + lane);
                __nv_bfloat16 *const dst = out + (long long)px * g.Cout + n0;
                const uint32_t acc = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)((b * g.T + t) * BN);
#pragma unroll 1
                for (int c0 = 0; c0 < BN; c0 += kChunk) {
                    uint32_t r[kChunk / 16][16];
#pragma unroll
                    for (int k = 0; k < kChunk / 16; ++k) tmem_load<16>(acc + (uint32_t)(c0 + 16 * k), r[k]);
                    tmem_wait_ld();
                    if (px < 0) continue;
#pragma unroll
                    for (int k = 0; k < kChunk / 8; ++k) {
                        const float4 b0 = *reinterpret_cast<const float4 *>(sbias + c0 + 8 * k);
                        const float4 b1 = *reinterpret_cast<const float4 *>(sbias + c0 + 8 * k + 4);
                        const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
                        __align__(16) __nv_bfloat16 o[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            float v = __uint_as_float(r[k / 2][(k & 1) * 8 + q]);
                            if (bias) v += bv[q];
                            if (g.relu) v = fmaxf(v, 0.f);
                            o[q] = __float2bfloat16_rn(v);
                        }
                        if (kBwd && mask) {
                            const uint4 mv = __ldg(reinterpret_cast<const uint4 *>(mask + (long long)px * g.Cout + n0 + c0) + k);
                            const __nv_bfloat16 *m = reinterpret_cast<const __nv_bfloat16 *>(&mv);
#pragma unroll
                            for (int q = 0; q < 8; ++q)
                                if (!(__bfloat162float(m[q]) > 0.f)) o[q] = __float2bfloat16_rn(0.f);
                        }
                        *reinterpret_cast<uint4 *>(dst + c0 + 8 * k) = *reinterpret_cast<const uint4 *>(o);
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&acc_empty[b]));
            if (++b == g.nbuf) {
                b = 0;
                phase ^= 1;
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 12)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)g.cols) : "memory");
}

// ---------------------------------------------------------------------------
// Weight gradient dW[co][t][ci] = sum_q dY[q][co] X[q + shift(t)][ci] over the
// padded positions (a padding position has dY = 0).  GEMM: M = (row ky, input
// channel of a tile of CI), 96 rows of 128 for CI = 32, N = output channels (tile BN),
// K = positions.  Both operands are staged as [channel group][position][16 bytes], which
// read with channels as M / N and positions as K is the MN-major core-matrix layout: no
// transposition, and the three taps of a row are the same staged X seen 16 bytes apart:
// three MMAs per 16 positions for nine taps.  A CTA owns one channel tile of each side (3 BN columns of
// TMEM) and one contiguous run of positions; it writes its FP32 partial
// sums to part[split][co][9 ci], the layout of dW, and weight_sum_kernel adds the splits
// in a fixed order; a launch takes as many splits as keep their partial sums within kWgPartBytes,
// and the next launch adds its own to dW.  K runs in stages of 64 positions through a ring of four buffers: warps 0-7 stage
// by cp.async, two stages behind the newest copies they announce the ones that landed; warp 8
// issues the twelve MMAs of a stage.  Bound: the latency of a CTA's stages (issue active 31-48 %, tensor pipe
// 11-23 %) and L2 (three copies of X).  With M = output channels and one row ky per CTA, 32 output channels
// filled a quarter of each MMA, every CTA staged dY once per row and the copies' instructions
// bound (issue active 66-71 %).  Kernel and sum of the splits, before and now: 16 x 256 x 256, 32 -> 32 193 and 115 us;
// 32 x 64 x 64, 96 -> 32 61 and 36; 32 x 32 x 32, 192 -> 64 39 and 28; 32 x 16 x 16, 384 -> 128 39 and 29;
// 16 x 32 x 32, 256 -> 256 79 and 59.  Two warps filling a whole buffer each instead of all eight
// filling every one: 111, 37, 31, 38 and 73.
// ---------------------------------------------------------------------------
constexpr int kWgK = 64, kWgStages = 4, kWgStagers = 256, kWgThreads = 288, kWgLag = 2;

struct LinWgrad {
    LinImage im;
    int Cin, Cout;
    int spx, spy;               // positions per staged group
    int q0, q1;                 // the launch's positions
    int per, splits;            // positions per split
    // bias gradient: blocks behind the splits' (bias_blocks = 0: none), gw groups of 8 channels
    // and bias_per pixels each
    int bias_blocks, gw;
    long long p0, P, bias_per;
    float *bpart;
};

// Partial sums of the bias gradient, sum_p dY[p][c], of gw groups of 8 channels over one run
// of pixels: consecutive threads read consecutive channel groups, each thread a strided
// part of the run's pixels, then a tree in shared memory (fixed order; 256 threads).
__device__ __forceinline__ void bias_partial(const __nv_bfloat16 *__restrict__ dy, const LinWgrad &g, int block,
                                             float *red) {
    const int gblocks = g.Cout / 8 / g.gw, split = block / gblocks, gb = block - split * gblocks;
    const int lanes = 256 / g.gw, gl = threadIdx.x % g.gw, pl = threadIdx.x / g.gw;
    const int c0 = (gb * g.gw + gl) * 8;
    const long long p0 = g.p0 + split * g.bias_per, p1 = min(g.p0 + g.P, p0 + g.bias_per);
    const bool mine = threadIdx.x < 256;
    float s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (mine) {
#pragma unroll 8
        for (long long p = p0 + pl; p < p1; p += lanes) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(dy + p * g.Cout + c0));
            const __nv_bfloat16 *e = reinterpret_cast<const __nv_bfloat16 *>(&v);
#pragma unroll
            for (int q = 0; q < 8; ++q) s[q] += __bfloat162float(e[q]);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) red[q * 256 + threadIdx.x] = s[q];
    }
    __syncthreads();
    for (int st = lanes / 2; st > 0; st >>= 1) {
        if (mine && pl < st)
#pragma unroll
            for (int q = 0; q < 8; ++q) red[q * 256 + threadIdx.x] += red[q * 256 + threadIdx.x + st * g.gw];
        __syncthreads();
    }
    for (int i = threadIdx.x; i < g.gw * 8; i += blockDim.x)
        g.bpart[(long long)split * g.Cout + gb * g.gw * 8 + i] = red[(i & 7) * 256 + (i >> 3)];
}

// One warp's eighth of a stage: positions 9 warp .. 9 warp + 8 of the 66 of X, which run from one before the
// stage's to one after, in the rows above, at and below, and of dY those of the middle row.  Lane 9 r + j finds
// the pixel of position j of row r once, the copies get it by shuffle, channel group fastest.  dY
// is zero from position `valid` on.  (192 -> 64 channels at 32 x 32 x 32, one row per CTA: 44 -> 39 us against
// finding the pixel for every copy.  The slabs of conv3x3_lin_kernel, many copies per
// thread, are faster with the pixel found for every copy and 256 threads abreast: 53 against 63 us
// at 16 x 256 x 256, 32 -> 32; plain loads and stores instead of cp.async 62-67 us.)
template <int CI, int BN>
__device__ __forceinline__ void wgrad_stage(const LinWgrad &g, int q, int warp, int lane, int valid,
                                            const __nv_bfloat16 *__restrict__ x, const __nv_bfloat16 *__restrict__ dy,
                                            unsigned char *X, unsigned char *Y) {
    constexpr int Gx = CI / 8, Gy = BN / 8;
    const int j0 = 9 * warp, nj = min(9, kWgK + 2 - j0);
    const int row = lane / 9, j = lane - 9 * row;
    const int mine = row < 3 && j < nj ? lin_pixel(g.im, q + (row - 1) * g.im.Wp - 1 + j0 + j) : -1;
#pragma unroll
    for (int base = 0; base < 27 * Gx; base += 32) {
        const int e = base + lane, i = e / Gx, grp = e % Gx, r = i / 9, pos = i - 9 * r;
        const int px = __shfl_sync(0xffffffffu, mine, i & 31);
        if (i < 27 && pos < nj)
            cp_async16(X + ((r * Gx + grp) * g.spx + j0 + pos) * 16, px >= 0 ? x + (long long)px * g.Cin + grp * 8 : x,
                       px >= 0 ? 16 : 0);
    }
#pragma unroll
    for (int base = 0; base < 9 * Gy; base += 32) {
        const int e = base + lane, i = e / Gy, grp = e % Gy, pos = j0 + i - 1;
        const int px = __shfl_sync(0xffffffffu, mine, (9 + i) & 31);
        if (i < nj && pos >= 0 && pos < kWgK)
            cp_async16(Y + (grp * g.spy + pos) * 16,
                       px >= 0 && pos < valid ? dy + (long long)px * g.Cout + grp * 8 : dy,
                       px >= 0 && pos < valid ? 16 : 0);
    }
}

template <int BN, bool kFirst>
__device__ __forceinline__ void wgrad_slices(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t lead) {
#pragma unroll
    for (int j = 0; j < kWgK / 16; ++j)
#pragma unroll
        for (int kx = 0; kx < 3; ++kx)
            mma_f16(tmem + (uint32_t)(kx * BN), ad + j * 16 + kx, bd + j * 16, idesc, kFirst && j == 0 ? 0u : 1u, lead);
}

template <int CI, int BN>
__global__ void __launch_bounds__(kWgThreads) conv3x3_wgrad_lin_kernel(const __nv_bfloat16 *__restrict__ x,
                                                                       const __nv_bfloat16 *__restrict__ dy,
                                                                       float *__restrict__ part, const LinWgrad g) {
    constexpr int kNeed = 3 * BN;
    constexpr uint32_t kCols = kNeed <= 128 ? 128u : (kNeed <= 256 ? 256u : 512u);
    extern __shared__ __align__(128) unsigned char wg_smem[];
    __shared__ __align__(8) uint64_t full[kWgStages], empty[kWgStages], done;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    if ((int)blockIdx.y >= g.splits) {  // blocks of the bias gradient
        const int block = (blockIdx.y - g.splits) * gridDim.x + blockIdx.x;
        if (block < g.bias_blocks) bias_partial(dy, g, block, reinterpret_cast<float *>(wg_smem));
        return;
    }
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int ci_tiles = g.Cin / CI;
    const int ci0 = (blockIdx.x % ci_tiles) * CI, co0 = (blockIdx.x / ci_tiles) * BN;
    const int qbeg = g.q0 + blockIdx.y * g.per, qend = min(g.q1, qbeg + g.per);
    const int nst = (qend - qbeg + kWgK - 1) / kWgK;  // >= 1: no split is empty
    // the MMA reads 16 groups of X; behind the staged ones (3 CI / 8) it reads whatever lies
    // there, for rows whose sums are not used (wgrad_smem leaves room behind the last buffer)
    const uint32_t xbytes = (uint32_t)(3 * CI / 8 * g.spx) * 16u, ybytes = (uint32_t)(BN / 8 * g.spy) * 16u;

    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int b = 0; b < kWgStages; ++b) {
            mbar_init(&full[b], kWgStagers / 32);
            mbar_init(&empty[b], 1);
        }
        mbar_init(&done, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    bool ok = true;

    if (warp < 8) {
        const auto landed = [&](int s) {  // this warp's copies of stage s are visible to the tensor core
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&full[s % kWgStages]));
        };
        for (int s = 0; s < nst; ++s) {
            if (s >= kWgStages)
                ok = warp_wait(&empty[s % kWgStages], (uint32_t)((s / kWgStages - 1) & 1), lane, &abort_flag);
            if (!ok) break;
            unsigned char *X = wg_smem + (s % kWgStages) * (xbytes + ybytes);
            const int q = qbeg + s * kWgK;
            wgrad_stage<CI, BN>(g, q, warp, lane, qend - q, x + ci0, dy + co0, X, X + xbytes);
            cp_async_commit();
            if (s >= kWgLag) {
                cp_async_wait<kWgLag>();
                landed(s - kWgLag);
            }
        }
        cp_async_wait<0>();
        if (ok)
            for (int s = max(0, nst - kWgLag); s < nst; ++s) landed(s);
    } else {
        const uint32_t lead = elect_lane();
        constexpr uint32_t idesc = mma_idesc(128, BN) | (1u << 15) | (1u << 16);  // both operands MN-major
        const uint32_t stage = (xbytes + ybytes) >> 4;
        const uint64_t ad = smem_desc(smem_u32(wg_smem), 128, (uint32_t)g.spx * 16);
        const uint64_t bd = smem_desc(smem_u32(wg_smem) + xbytes, 128, (uint32_t)g.spy * 16);
        for (int s = 0; s < nst; ++s) {
            const int b = s % kWgStages;
            ok = ws_wait(smem_u32(&full[b]), (uint32_t)((s / kWgStages) & 1), &abort_flag);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (s == 0) wgrad_slices<BN, true>(tmem, ad, bd, idesc, lead);
            else wgrad_slices<BN, false>(tmem, ad + b * stage, bd + b * stage, idesc, lead);
            mma_commit(smem_u32(&empty[b]), lead);
        }
        mma_commit(smem_u32(&done), lead);  // waited for also after a time-out, before the tensor memory is freed
        ok = mbar_wait(smem_u32(&done), 0) && ok;
        if (lane == 0 && !ok) abort_flag = 1;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const int quarter = warp & 3, r0 = quarter * 32 + lane, ky = r0 / CI;
    if (warp < 8 && quarter * 32 < 3 * CI && abort_flag == 0) {
        // TMEM lane = row = (ky, input channel): a column's lanes are consecutive floats of dW;
        // warps w and w + 4 share the lanes of quarter w & 3
        float *const col = part + ((long long)blockIdx.y * g.Cout + co0) * (9 * g.Cin) + 3 * ky * g.Cin + ci0 + r0 % CI;
#pragma unroll 2
        for (int c = (warp >> 2) * 16; c < 3 * BN; c += 32) {
            uint32_t r[16];
            tmem_load<16>(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c, r);
            tmem_wait_ld();
            float *const d = col + (long long)(c % BN) * (9 * g.Cin) + (c / BN) * g.Cin;
            if (ky < 3)
#pragma unroll
                for (int k = 0; k < 16; ++k) d[(long long)k * (9 * g.Cin)] = __uint_as_float(r[k]);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 8)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

// ---- host side ----------------------------------------------------------------------
// cuTensorMapEncodeTiled, looked up in the driver once (libcuda is not linked).
using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
inline EncodeTiled encode_tiled() {
    static const EncodeTiled fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult r;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &r) != cudaSuccess ||
            r != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeTiled>(p);
    }();
    return fn;
}

// SMs and shared memory of the current device (0 SMs: no device).
struct DeviceShape {
    int sms = 0, smem_sm = 0;
};
inline DeviceShape device_shape() {
    static std::atomic<long long> known[64];
    int dev = 0;
    DeviceShape d;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return d;
    const long long k = dev < 64 ? known[dev].load() : 0;
    if (k) {
        d.sms = (int)(k >> 32);
        d.smem_sm = (int)(k & 0xffffffff);
        return d;
    }
    if (cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&d.smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess)
        return DeviceShape{};
    if (dev < 64) known[dev].store(((long long)d.sms << 32) | d.smem_sm);
    return d;
}

constexpr int kMaxSmemCta = 222 * 1024;  // dynamic; the static arrays take the rest of 227 KB

// The plans of the last shapes this thread used, one per slot: choosing one takes a few microseconds
// of host time, as much as the launch.  A plan is a function of its key alone.
template <class Plan>
struct PlanCache {
    struct Entry {
        long long key[7];
        Plan plan;
        bool used = false;
    };
    Entry entry[64];
    template <class Make>
    const Plan &get(const long long (&key)[7], const Make &make) {
        unsigned long long h = 0;
        for (long long k : key) h = (h ^ (unsigned long long)k) * 0x9E3779B97F4A7C15ull;
        Entry &e = entry[h >> 58];
        if (!e.used || !std::equal(key, key + 7, e.key)) {
            e.plan = make();
            std::copy(key, key + 7, e.key);
            e.used = true;
        }
        return e.plan;
    }
};

// The item shape of conv3x3_lin_kernel for one layer: BN output channels, T tiles of 128
// positions and one or two slabs, chosen to make the busiest SM's time least.  The
// estimate, in SM cycles: an item's staging (about 16 bytes a cycle of a CTA's copies and their
// latency), its MMAs (the larger of arithmetic, BN / 2 cycles per slice of 128 x 16, and the
// operands' reads from shared memory, and 80 cycles a slice of all T tiles to issue)
// and its stores; two slabs overlap the three inside a CTA, and so do the CTAs of an SM.
// More positions per item stage less halo, fewer fill more SMs: a layer of 2592
// positions takes T = 1 with narrow BN, one of a million T = 8 with two slabs.  On rows of 300
// pixels and more the halo of two rows is most of what an item stages, and the copies of all CTAs of an SM
// together count, 1.6 cycles each (1 x 4096 x 512, 16 -> 32: 123 -> 82 us).
struct LinPlan {
    int bn = 0, t = 0, sp = 0, nbuf = 0, cols = 0, stages = 0, occ = 0;
    size_t smem = 0;
    bool slower = false;  // than the kernel that takes the layer otherwise
};
// SM cycles of the kernels that take a layer when conv3x3_lin_kernel does not: a start, and per slice of
// 16 channels of K the longer of one tile's own chain and the SM's rate times its tiles.
// Fitted to 12 layers of 16-384 channels on images of 8 x 8 to 4096 x 512 (within 10 % on average).
inline double staged_cycles(bool bwd, long long P, int W, int K, int M, int sms) {
    const bool slab = !bwd && slab_shape(W, K, M), pipe = K >= 128;
    int bn = M % 128 == 0 ? 128 : (M % 64 == 0 ? 64 : (M % 32 == 0 ? 32 : 16));
    double chain, rate;
    if (slab) {
        bn = K == 64 ? std::min(bn, 64) : bn;
        chain = rate = bn == 128 ? 560 : (bn == 64 ? 328 : 225);
    } else if (!bwd) {
        chain = bn == 128 ? (pipe ? 1340 : 2440) : (bn == 64 ? (pipe ? 1070 : 1880) : 1570);
        rate = bn == 128 ? (pipe ? 800 : 1270) : (bn == 64 ? (pipe ? 600 : 800) : 580);
    } else {
        chain = bn == 128 ? 2500 : (bn == 64 ? (pipe ? 1630 : 2210) : (bn == 32 ? 1890 : 1220));
        rate = bn == 128 ? 1480 : (bn == 64 ? (pipe ? 1020 : 1080) : (bn == 32 ? 650 : 450));
    }
    const double tiles = (double)((P + 127) / 128 * (M / bn));
    return 12000 + 9.0 * K / 16 * std::max(chain, rate * std::ceil(tiles / sms));
}
inline LinPlan lin_plan(const LinImage &im, long long P, int Cin, int Cout, const DeviceShape &d, bool bwd) {
    LinPlan best;
    double least = 1e30, cycles = 0;
    const int G = Cin / 8, slices = 9 * Cin / 16, nst = (9 * Cin + kLinK - 1) / kLinK;
    for (int bn : {256, 128, 64, 32, 16}) {
        if (Cout % bn) continue;
        for (int t : {8, 4, 2, 1}) {
            for (int nbuf : {2, 1}) {
                int cols = 32;
                while (cols < nbuf * t * bn) cols *= 2;
                if (cols > 512 || (t == 8 && bn > 64) || (t == 4 && bn > 128)) continue;
                const int count = t * 128 + 2 * (im.Wp + 1), sp = lin_stride(count, G);
                const size_t slab = (size_t)G * sp * 16, stage = (size_t)bn * kLinK * 2;
                int stages = std::min(nst, kLinMaxStages);  // whole weights if they fit
                if (stages < nst || 1024 + nbuf * slab + stages * stage > (size_t)kMaxSmemCta)
                    stages = std::min(nst, bn >= 256 ? 2 : (bn >= 128 ? 3 : 4));
                const size_t smem = 1024 + nbuf * slab + stages * stage;
                if (smem > (size_t)kMaxSmemCta || sp >= (1 << 14)) continue;
                const int occ = std::max(1, std::min({(int)(d.smem_sm / (smem + 4096)), 512 / cols, 4}));
                const long long items = (im.L + t * 128 - 1) / (t * 128), all = items * (Cout / bn);
                const double n = (double)((all + d.sms - 1) / d.sms);  // items of the busiest SM
                const double copy = slab / 16.0 + 1500, store = 800 + t * (100 + bn * 10.0);
                const double mma = (double)slices * std::max(t * std::max(bn / 2.0, 32 + bn / 4.0), 80.0);
                const double one = nbuf == 2 ? std::max({copy, mma, store}) : copy + mma + store;
                const double copies = (double)G * count, wide = im.W >= 300 ? 1.6 * copies : 0;
                const double apart = one / std::min((double)occ, n);
                const double time = copy + mma + store + (n - 1) * std::max({mma, apart, wide});
                if (time < least) {
                    least = time;
                    // (the estimate that fits absolute times best; `time` ranks the plans)
                    cycles = 10000 + std::max(1.13 * (copy + mma + store + (n - 1) * std::max(mma, apart)),
                                              2.15 * n * copies);
                    best = LinPlan{bn, t, sp, nbuf, cols, stages, occ, smem};
                }
            }
        }
    }
    // The other kernel only where it is clearly ahead.  Of 855 layers and sizes measured 53 go there, all but four of them
    // rightly (7 % slower at most).  Where rows get wide: 1 x 682 x 1536, 32 -> 32 takes 493 us here and 94 on the
    // slab kernel, 1 x 697 x 752, 64 -> 64 1012 and 396 (im2col), 1 x 1024 x 128, 256 -> 256 1466 and 753.
    best.slower = staged_cycles(bwd, P, im.W, Cin, Cout, d.sms) < 0.9 * cycles;
    return best;
}

template <bool kBwd, int BN>
cudaError_t launch_conv_lin(const CUtensorMap &map, const __nv_bfloat16 *in, const float *bias,
                            const __nv_bfloat16 *mask, __nv_bfloat16 *out, const LinConv &g, const LinPlan &pl, int sms, cudaStream_t s) {
    static std::atomic<bool> set[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !set[dev].load()) {
        e = cudaFuncSetAttribute(conv3x3_lin_kernel<kBwd, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmemCta);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(conv3x3_lin_kernel<kBwd, BN>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     (int)cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        if (dev < 64) set[dev].store(true);
    }
    const int tiles_n = g.Cout / BN;
    const dim3 grid((unsigned)std::min(g.items, std::max(1, sms * pl.occ / tiles_n)), (unsigned)tiles_n);
    conv3x3_lin_kernel<kBwd, BN><<<grid, kLinThreads, pl.smem, s>>>(map, in, bias, mask, out, g);
    return cudaGetLastError();
}

// Runs the layer on conv3x3_lin_kernel if it can and pays (*ran).  It cannot where the
// positions that one tile reads do not fit in shared memory with all input channels
// (wide images with many channels, e.g. 384 channels from W = 71 on), for 2^30 positions and
// more, and for weights off a 16-byte boundary (TMA).
template <bool kBwd>
cudaError_t conv_lin(const __nv_bfloat16 *in, const __nv_bfloat16 *w, const float *bias,
                     const __nv_bfloat16 *mask, __nv_bfloat16 *out, int N, int H, int W, int Cin, int Cout, int relu, cudaStream_t s, bool *ran) {
    *ran = false;
    LinConv g{};
    const DeviceShape d = device_shape();
    if (Cin < 16 || Cin > 16 * kLinMaxSlices / 9 || Cout < 16 || !d.sms || !encode_tiled() || (reinterpret_cast<uintptr_t>(w) & 15) || !lin_image(N, H, W, &g.im))
        return cudaSuccess;
    g.Cin = Cin;
    g.Cout = Cout;
    g.dg = fast_div((uint32_t)Cin / 8);
    g.boxk = Cin % 64 ? 32 : 64;
    g.relu = relu;
    thread_local PlanCache<LinPlan> plans;
    const long long P = (long long)N * H * W;
    const LinPlan pl = plans.get({g.im.L, P, W, Cin, Cout, d.sms, d.smem_sm},
                                 [&] { return lin_plan(g.im, P, Cin, Cout, d, kBwd); });
    if (!pl.bn || pl.slower) return cudaSuccess;
    g.dc = fast_div((uint32_t)Cin);
    g.T = pl.t;
    g.sp = pl.sp;
    g.nbuf = pl.nbuf;
    g.cols = pl.cols;
    g.items = (g.im.L + pl.t * 128 - 1) / (pl.t * 128);
    g.stages = pl.stages;
    CUtensorMap map;
    CUresult r;
    const cuuint32_t one[3] = {1, 1, 1};
    if (!kBwd) {
        const cuuint64_t dim[2] = {(cuuint64_t)9 * Cin, (cuuint64_t)Cout}, stride[1] = {(cuuint64_t)18 * Cin};
        const cuuint32_t box[2] = {64, (cuuint32_t)pl.bn};
        r = encode_tiled()(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16 *>(w), dim, stride, box, one,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    } else {
        // the weight tensor [Cin of the GEMM][9][Cout of the GEMM], channels of dx fastest
        const cuuint64_t dim[3] = {(cuuint64_t)Cout, 9, (cuuint64_t)Cin};
        const cuuint64_t stride[2] = {(cuuint64_t)2 * Cout, (cuuint64_t)18 * Cout};
        const cuuint32_t bx = (cuuint32_t)std::min(pl.bn, 64), box[3] = {bx, 1, (cuuint32_t)g.boxk};
        r = encode_tiled()(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<__nv_bfloat16 *>(w), dim, stride, box, one,
                           CU_TENSOR_MAP_INTERLEAVE_NONE,
                           bx == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : (bx == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B),
                           CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    }
    if (r != CUDA_SUCCESS) return cudaSuccess;
    *ran = true;
    switch (pl.bn) {
        case 256: return launch_conv_lin<kBwd, 256>(map, in, bias, mask, out, g, pl, d.sms, s);
        case 128: return launch_conv_lin<kBwd, 128>(map, in, bias, mask, out, g, pl, d.sms, s);
        case 64: return launch_conv_lin<kBwd, 64>(map, in, bias, mask, out, g, pl, d.sms, s);
        case 32: return launch_conv_lin<kBwd, 32>(map, in, bias, mask, out, g, pl, d.sms, s);
        default: return launch_conv_lin<kBwd, 16>(map, in, bias, mask, out, g, pl, d.sms, s);
    }
}

// The weight gradient's tiling: BN output channels per CTA and the positions per split, a
// multiple of 64 and at most 1024 (the FP32 sums of one split stay as short as they were with
// 16 stages of 64 pixels), for the least estimated time in SM cycles: the busiest SM's MMAs (at two thirds of
// their rate) or its CTAs one after the other (900 cycles a stage, 1000 and 20 a column for start and
// stores), and the partial sums, written and read at about 40 bytes a cycle and SM.  The
// constants are fitted to 13 layers of the network and of large images, every BN and run length: its choices
// take 9 % more time than the best ones at most, 1 % on average.  Then the bias gradient's blocks, at
// most about two per SM, with at least 16 pixels a thread.
struct WgLinPlan {
    int ci = 0, bn = 0, splits = 0, per = 0;
    int run = 0;  // splits of one launch at most
    int gw = 0, bias_splits = 0;
    long long bias_per = 0;
    size_t smem = 0;
};
// Partial sums of one launch.  A split sums at most 1024 positions, so without a bound they grow with
// the pixels: 2.4 GB for 16 x 256 x 256, 256 -> 256, and more splits than a grid has rows
// from 2^26 positions on.  That layer takes 3.68 ms with 160 MB as with 64 and 3.24 in one launch (12.3 on the
// im2col kernel); 1 x 241 x 241, 256 -> 256 takes 215 us with 160 MB, where it is one launch, and 254 with 64.
constexpr long long kWgPartBytes = 160ll << 20;
inline size_t wgrad_smem(int ci, int bn) {
    const int spx = lin_stride(kWgK + 2, ci / 8), spy = lin_stride(kWgK, bn / 8), x = 3 * ci / 8 * spx, y = bn / 8 * spy;
    return std::max<size_t>(16ull * (kWgStages * (x + y) + std::max(0, 16 * spx - x - y)), 8 * 256 * sizeof(float));
}
inline WgLinPlan make_wgrad_lin_plan(long long L, long long P, int Cin, int Cout) {
    constexpr int kSms = 152;  // (the workspace query has no device to ask)
    WgLinPlan w;
    w.ci = Cin % 32 ? 16 : 32;
    double least = 1e30;
    for (int bn : {128, 64, 32}) {
        if (Cout % bn) continue;
        const long long tiles = (long long)(Cin / w.ci) * (Cout / bn);
        const int cols = 3 * bn <= 128 ? 128 : (3 * bn <= 256 ? 256 : 512);
        const int occ = (int)std::max<size_t>(1, std::min<size_t>({228 * 1024 / (wgrad_smem(w.ci, bn) + 2048), 512u / cols, 7u}));
        for (int per : {1024, 896, 768, 640, 512, 384, 256, 192, 128}) {
            const long long s = (L + per - 1) / per, ctas = tiles * s;
            const double n = (double)((ctas + kSms - 1) / kSms), nst = std::min<double>(per, (double)L) / kWgK;
            const double slice = bn == 128 ? 64 : (bn == 64 ? 48 : 45);
            const double mma = n * nst * 18 * slice, chain = std::ceil(n / occ) * (nst * 900 + 1000 + 20 * bn);
            const double time = std::max(mma, chain) + s * 36.0 * Cin * Cout / (kSms * 20.0);
            if (time < least) {
                least = time;
                w.bn = bn;
                w.per = per;
                w.splits = (int)s;
                w.smem = wgrad_smem(w.ci, bn);
            }
        }
    }
    const long long most = std::max(1ll, kWgPartBytes / (36ll * Cin * Cout)), launches = (w.splits + most - 1) / most;
    w.run = (int)((w.splits + launches - 1) / launches);
    w.gw = 32;
    while ((Cout / 8) % w.gw) w.gw /= 2;
    const long long groups = Cout / 8 / w.gw, lanes = 256 / w.gw;
    const long long bs = std::max(1ll, std::min((2 * kSms + groups - 1) / groups, (P + 16 * lanes - 1) / (16 * lanes)));
    w.bias_per = (P + bs - 1) / bs;
    w.bias_splits = (int)((P + w.bias_per - 1) / w.bias_per);
    return w;
}

// Workspace of a call's largest launch, in bytes.
inline long long wgrad_bytes(const WgLinPlan &w, int Cin, int Cout) {
    return ((long long)w.run * 9 * Cin + w.bias_splits) * Cout * (long long)sizeof(float);
}

inline WgLinPlan wgrad_lin_plan(long long L, long long P, int Cin, int Cout) {
    thread_local PlanCache<WgLinPlan> plans;
    return plans.get({L, P, Cin, Cout, 0, 0, 0}, [&] { return make_wgrad_lin_plan(L, P, Cin, Cout); });
}

template <int CI, int BN>
cudaError_t launch_wgrad_lin(const __nv_bfloat16 *x, const __nv_bfloat16 *dy, float *part, const LinWgrad &g,
                             size_t smem, cudaStream_t s) {
    static std::atomic<bool> set[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !set[dev].load()) {
        e = cudaFuncSetAttribute(conv3x3_wgrad_lin_kernel<CI, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmemCta);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(conv3x3_wgrad_lin_kernel<CI, BN>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     (int)cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        if (dev < 64) set[dev].store(true);
    }
    const int tiles = (g.Cin / CI) * (g.Cout / BN);
    const dim3 grid((unsigned)tiles, (unsigned)(g.splits + (g.bias_blocks + tiles - 1) / tiles));
    conv3x3_wgrad_lin_kernel<CI, BN><<<grid, kWgThreads, smem, s>>>(x, dy, part, g);
    return cudaGetLastError();
}

// The positions [q0, q1) in `splits` splits; bpart: and the bias gradient over P pixels from p0 on.
inline cudaError_t wgrad_lin(const __nv_bfloat16 *x, const __nv_bfloat16 *dy, float *part, float *bpart,
                             const LinImage &im, int q0, int q1, long long p0, long long P, int Cin, int Cout,
                             const WgLinPlan &w, int splits, cudaStream_t s) {
    LinWgrad g{};
    g.im = im;
    g.Cin = Cin;
    g.Cout = Cout;
    g.spx = lin_stride(kWgK + 2, w.ci / 8);
    g.spy = lin_stride(kWgK, w.bn / 8);
    g.per = w.per;
    g.splits = splits;
    g.q0 = q0;
    g.q1 = q1;
    g.bias_blocks = bpart ? w.bias_splits * (Cout / 8 / w.gw) : 0;
    g.gw = w.gw;
    g.p0 = p0;
    g.P = P;
    g.bias_per = w.bias_per;
    g.bpart = bpart;
    const bool c32 = w.ci == 32;
    switch (w.bn) {
        case 128: return c32 ? launch_wgrad_lin<32, 128>(x, dy, part, g, w.smem, s) : launch_wgrad_lin<16, 128>(x, dy, part, g, w.smem, s);
        case 64: return c32 ? launch_wgrad_lin<32, 64>(x, dy, part, g, w.smem, s) : launch_wgrad_lin<16, 64>(x, dy, part, g, w.smem, s);
        default: return c32 ? launch_wgrad_lin<32, 32>(x, dy, part, g, w.smem, s) : launch_wgrad_lin<16, 32>(x, dy, part, g, w.smem, s);
    }
}
