// Batched solver: many lattices of uneven size.  Where every lattice fits the
// two-step tiling, one launch advances a group of them by two steps
// (step2_batch_kernel: a CTA per tile of any instance).  Otherwise a persistent
// kernel: work is scheduled as (instance, tile) units; a bounded grid barrier
// separates time steps inside a launch, so one launch advances every instance
// by `steps_per_launch` steps.  Or chains of the single-lattice kernels per
// instance over a pool of streams.  Each node runs the same update in all of them.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <tuple>
#include <vector>

#include "lb_device.cuh"

namespace cdflb {
namespace {

// Grid-wide barrier for a co-resident (cooperative) grid.  bar[0] counts
// arrivals, bar[1] is the generation.  Every wait is bounded: after timeout_ns
// (or an iteration cap) the block sets err[0] and the whole grid gives up; the
// first block to give up records the step, the arrivals it saw and the time it
// waited (err[1..3], microseconds) for the host's message.  Returns false when
// the barrier failed.
__device__ bool grid_barrier(unsigned *bar, unsigned expected, unsigned long long timeout_ns, int *err, int step) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        ok = 1;
        volatile unsigned *vgen = bar + 1;
        volatile int *verr = err;
        const unsigned gen = *vgen;
        __threadfence();  // this block's stores of the step before the arrival
        const unsigned arrived = atomicAdd(bar, 1u) + 1u;
        if (arrived == expected) {
            atomicExch(bar, 0u);
            __threadfence();
            atomicAdd(bar + 1, 1u);
        } else {
            const unsigned long long t0 = dev::global_ns();
            const unsigned long long cap = timeout_ns / 32ull + (1ull << 20);
            unsigned long long it = 0;
            while (*vgen == gen) {
                if (*verr) { ok = 0; break; }
                if (++it > cap || ((it & 63ull) == 0 && dev::global_ns() - t0 > timeout_ns)) {
                    if (atomicCAS(err, 0, 1) == 0) {
                        err[1] = step;
                        err[2] = (int)*(volatile unsigned *)bar;
                        err[3] = (int)min((dev::global_ns() - t0) / 1000ull, 2000000000ull);
                    }
                    ok = 0;
                    break;
                }
                __nanosleep(32);
            }
            __threadfence();
        }
    }
    __syncthreads();
    return ok != 0;
}

// (sp_in and sp_out: the same plane set for several steps, S(t - 1) is then updated in place)
template <int M>
__global__ void __launch_bounds__(256, 4) batch_kernel(const BatchInst *__restrict__ inst, const int *__restrict__ tile_inst,
                                                    int total_tiles, float *buf0, float *buf1,
                                                    const float *sp_in, float *sp_out, float *moments, int nsteps, int parity0, int moments_last,
                                                    unsigned *bar, unsigned expected, unsigned long long timeout_ns,
                                                    int *err) {
    __shared__ LbParams sp;
    __shared__ long long s_off[3];
    __shared__ int s_tile[2];
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int nthreads = blockDim.x * blockDim.y;
    for (int s = 0; s < nsteps; ++s) {
        const float *in = ((parity0 + s) & 1) ? buf1 : buf0;
        float *out = ((parity0 + s) & 1) ? buf0 : buf1;
        float *mom = (moments_last && s == nsteps - 1) ? moments : nullptr;
        int cur_inst = -1;
        // Each block takes a contiguous range of tiles: long runs of one instance
        // (parameters staged once) and neighbouring tiles whose halos are still in L1.
        const int t_begin = (int)((long long)total_tiles * blockIdx.x / gridDim.x);
        const int t_end = (int)((long long)total_tiles * (blockIdx.x + 1) / gridDim.x);
        for (int t = t_begin; t < t_end; ++t) {
            const int k = tile_inst[t];
            if (k != cur_inst) {  // stage the instance's parameters in shared memory
                __syncthreads();
                const int *src = reinterpret_cast<const int *>(&inst[k].p);
                int *dst = reinterpret_cast<int *>(&sp);
                for (int w = tid; w < (int)(sizeof(LbParams) / sizeof(int)); w += nthreads) dst[w] = src[w];
                if (tid == 0) {
                    s_off[0] = inst[k].pop_off;
                    s_off[1] = inst[k].sp_off;
                    s_off[2] = inst[k].mom_off;
                    s_tile[0] = inst[k].tile_base;
                    s_tile[1] = inst[k].tiles_x;
                }
                __syncthreads();
                cur_inst = k;
            }
            const int lt = t - s_tile[0];
            const int ty = lt / s_tile[1], tx = lt - ty * s_tile[1];
            const int x = tx * blockDim.x + threadIdx.x, y = ty * blockDim.y + threadIdx.y;
            if (x < sp.nx && y < sp.ny)
                dev::step_node<M, float, true>(sp, x, y, in + s_off[0], out + s_off[0], sp_in + s_off[1],
                                               sp_out + s_off[1], mom ? mom + s_off[2] : nullptr);
        }
        if (s + 1 < nsteps && !grid_barrier(bar, expected, timeout_ns, err, s)) return;
    }
}

thread_local char g_berr[512] = "";
cdf_status bfail(cdf_status st, const char *msg) {
    std::snprintf(g_berr, sizeof g_berr, "%s", msg);
    return report_error(st, msg);
}

#define BCK(call)                                                                     \
    do {                                                                              \
        cudaError_t e_ = (call);                                                      \
        if (e_ != cudaSuccess) {                                                      \
            char m_[400];                                                             \
            std::snprintf(m_, sizeof m_, "%s failed: %s", #call, cudaGetErrorString(e_)); \
            return bfail(CDF_ECUDA, m_);                                              \
        }                                                                             \
    } while (0)

using TuneKey = std::tuple<long long, long long, int, int, int>;
std::mutex g_btune_mu;

}  // namespace
}  // namespace cdflb

using namespace cdflb;

struct cdf_batch {
    int device = 0;
    int count = 0, m = 0;
    std::vector<LbParams> params;
    std::vector<long long> pop_off, sp_off, mom_off, node_off;
    long long pop_total = 0, sp_total = 0, mom_total = 0, nodes = 0;
    int sprev_planes = 0;
    float *buf[2] = {nullptr, nullptr};
    // S_1(t - 1): the persistent kernel updates `sprev` in place; the kernel
    // chains alternate `sprev` and `sprev2` with the population buffers (a
    // two-step launch reads halo nodes that other CTAs rewrite).
    float *sprev = nullptr, *sprev2 = nullptr, *mom = nullptr, *dense = nullptr, *host_stage = nullptr;
    float *mom_prev = nullptr;                        // snapshot for per-instance residuals
    double *partials = nullptr, *red = nullptr, *red_host = nullptr;  // per-instance reductions
    size_t stage_floats = 0;
    BatchInst *d_inst = nullptr;
    int *d_tile_inst = nullptr;
    unsigned *d_bar = nullptr;
    int *d_err = nullptr, *h_err = nullptr;
    int total_tiles = 0, grid_blocks = 0;
    dim3 tile{64, 4, 1};
    int steps_per_launch = 32;
    unsigned long long timeout_ns = 1000000000ull;
    int extra_arrivals = 0;
    cudaStream_t s = nullptr, user = nullptr;
    cudaEvent_t ev_in = nullptr, ev_out = nullptr;
    int cur = 0;
    long long t = 0;
    // Second execution mode: one chain of single-lattice step kernels per
    // instance (each launch reads its parameters as kernel operands), fanned out
    // over a pool of streams and captured as one CUDA graph; instances are
    // independent, so the chains need no barrier between them.
    int mode = 0;  // 0: whole-batch kernels, 1: graph of per-instance chains, 2: chains of two-step launches
    dim3 chain_block{128, 1, 1};
    int chain_th = 14;  // mode 2: output tile height of step2_kernel (chain_block is its CTA)
    // mode 0: two steps of all instances per launch instead of the persistent kernel
    bool fused = false;
    int kind = 0;  // closure kind of all instances
    std::vector<BatchInst> inst;
    std::vector<int> group_start;  // first instance of each launch's group, and count
    long long max_nodes = 0;
    std::vector<cudaStream_t> pool;
    cudaEvent_t ev_fork = nullptr;
    std::vector<cudaEvent_t> ev_join;
    cudaGraphExec_t chain_graph[2][2] = {{nullptr, nullptr}, {nullptr, nullptr}};  // [parity][moments]
};

namespace {

// The two-step launches of a batch: the instances, in order, form a multiple of kFusedLanes groups of about
// kGroupBytes of populations (both buffers), and each lane (a stream) runs its groups one after
// the other, all steps of one before the next.  So the groups at work stay in the 126 MB L2, and
// one lane's last CTAs run beside the others' next launch.  64 steps of 512 cavities of 64 x 64:
// 40.1 us a step with all groups side by side, 54 with one lane, 37.3 with two lanes of 40 MB, 36.9 with
// four of 20 MB, 37.1 with eight of 10 MB; 64 plumes of 128-512 x 64-256: 71.8, 81, 68.4, 65.8 and 64.0.
constexpr int kFusedLanes = 4;
constexpr long long kGroupBytes = 20ll << 20;

void brelease(cdf_batch *b) {
    if (!b) return;
    for (auto &row : b->chain_graph)
        for (auto &g : row)
            if (g) cudaGraphExecDestroy(g);
    for (cudaStream_t ps : b->pool) cudaStreamDestroy(ps);
    for (cudaEvent_t e : b->ev_join) cudaEventDestroy(e);
    if (b->ev_fork) cudaEventDestroy(b->ev_fork);
    dev_free(b->buf[0]);
    dev_free(b->buf[1]);
    dev_free(b->sprev);
    dev_free(b->sprev2);
    dev_free(b->mom);
    dev_free(b->mom_prev);
    cudaFree(b->partials);
    cudaFree(b->red);
    if (b->red_host) cudaFreeHost(b->red_host);
    dev_free(b->dense);
    cudaFree(b->d_inst);
    cudaFree(b->d_tile_inst);
    cudaFree(b->d_bar);
    cudaFree(b->d_err);
    if (b->h_err) cudaFreeHost(b->h_err);
    if (b->host_stage) cudaFreeHost(b->host_stage);
    if (b->ev_in) cudaEventDestroy(b->ev_in);
    if (b->ev_out) cudaEventDestroy(b->ev_out);
    if (b->s) cudaStreamDestroy(b->s);
    delete b;
}

// The tile of step2_batch_kernel for one lattice: the least node updates in all (tile and
// ring, rounded to warps, and about 128 more per CTA for its start) of at most
// kBatchTileX x kBatchTileY nodes, with the ring inside the lattice on a periodic axis.  false: none fits (a
// periodic axis of fewer than 6 nodes).
bool pair_tile(const LbParams &p, long long most, int *tw, int *th) {
    double least = 1e30;
    for (int w = 4; w <= kBatchTileX; ++w) {
        if (p.periodic_x && p.nx < w + 2) break;
        for (int h = 4; h <= kBatchTileY && (w * h <= most || h == 4); ++h) {
            if (p.periodic_y && p.ny < h + 2) break;
            const double tiles = (double)((p.nx + w - 1) / w) * ((p.ny + h - 1) / h);
            const int warps = ((w + 2) * (h + 2) + 31) / 32 + (w * h + 31) / 32;
            if (tiles * (32 * warps + 128) < least) {
                least = tiles * (32 * warps + 128);
                *tw = w;
                *th = h;
            }
        }
    }
    return least < 1e30;
}

// Nodes of a tile at most: a small batch gets two CTAs for every SM (2.2 us a step instead of 3.0 for a few
// lattices of 64 x 64).
long long tile_nodes(long long nodes) { return std::max(128ll, nodes / 304); }

// Tile table and instance descriptors for a tile shape; sets the grid size.
cdf_status setup_tiles(cdf_batch *b, dim3 tile) {
    std::vector<BatchInst> &inst = b->inst;
    inst.resize(b->count);
    std::vector<int> tiles;
    for (int k = 0; k < b->count; ++k) {
        const LbParams &p = b->params[k];
        const int tx = (p.nx + tile.x - 1) / tile.x, ty = (p.ny + tile.y - 1) / tile.y;
        inst[k].p = p;
        inst[k].pop_off = b->pop_off[k];
        inst[k].sp_off = b->sp_off[k];
        inst[k].mom_off = b->mom_off[k];
        inst[k].tile_base = (int)tiles.size();
        inst[k].tiles_x = tx;
        tiles.insert(tiles.end(), (size_t)tx * ty, k);
        inst[k].node_off = b->node_off[k];
        int tw = 1, th = 1;
        pair_tile(p, tile_nodes(b->nodes), &tw, &th);
        inst[k].pair_x = (p.nx + tw - 1) / tw;
        inst[k].pair_tiles = inst[k].pair_x * ((p.ny + th - 1) / th);
        inst[k].tw = tw;
        inst[k].th = th;
    }
    const auto bytes = [b](int k) { return 8ll * (9 + 5 * b->m + b->sprev_planes) * b->params[k].plane; };
    long long total = 0, before = 0, last = 0;
    for (int k = 0; k < b->count; ++k) total += bytes(k);
    const long long groups = (total / kGroupBytes + kFusedLanes) / kFusedLanes * kFusedLanes;
    b->group_start.assign(1, 0);
    for (int k = 0; k < b->count; before += bytes(k++)) {
        const long long g = (long long)((before + 0.5 * bytes(k)) / total * groups);
        if (k > 0 && (g != last || k - b->group_start.back() == kBatchGroup)) b->group_start.push_back(k);
        last = g;
    }
    b->group_start.push_back(b->count);
    cudaFree(b->d_tile_inst);
    b->d_tile_inst = nullptr;
    BCK(cudaMalloc(&b->d_tile_inst, tiles.size() * sizeof(int)));
    BCK(cudaMemcpy(b->d_inst, inst.data(), inst.size() * sizeof(BatchInst), cudaMemcpyHostToDevice));
    BCK(cudaMemcpy(b->d_tile_inst, tiles.data(), tiles.size() * sizeof(int), cudaMemcpyHostToDevice));
    b->total_tiles = (int)tiles.size();
    b->tile = tile;
    int per_sm = 0, sms = 0;
    void (*kern)(const BatchInst *, const int *, int, float *, float *, const float *, float *, float *, int, int, int,
                 unsigned *, unsigned, unsigned long long, int *) = nullptr;
    switch (b->m) {
        case 1: kern = batch_kernel<1>; break;
        case 2: kern = batch_kernel<2>; break;
        case 3: kern = batch_kernel<3>; break;
        default: kern = batch_kernel<4>; break;
    }
    BCK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, tile.x * tile.y, 0));
    BCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device));
    b->grid_blocks = std::max(1, std::min(per_sm * sms, b->total_tiles));
    return CDF_OK;
}

// nsteps of the persistent kernel from buffer `parity` (sp_in != sp_out: one step).
cdf_status enqueue_batch(cdf_batch *b, int nsteps, bool moments_last, int parity, const float *sp_in, float *sp_out) {
    BCK(cudaMemsetAsync(b->d_err, 0, 4 * sizeof(int), b->s));
    BCK(cudaMemsetAsync(b->d_bar, 0, 2 * sizeof(unsigned), b->s));
    unsigned expected = (unsigned)b->grid_blocks + (unsigned)b->extra_arrivals;
    int ml = moments_last ? 1 : 0;
    void *args[] = {&b->d_inst, &b->d_tile_inst, &b->total_tiles, &b->buf[0], &b->buf[1], &sp_in, &sp_out, &b->mom,
                    &nsteps, &parity, &ml, &b->d_bar, &expected, &b->timeout_ns, &b->d_err};
    const void *kern = nullptr;
    switch (b->m) {
        case 1: kern = (const void *)batch_kernel<1>; break;
        case 2: kern = (const void *)batch_kernel<2>; break;
        case 3: kern = (const void *)batch_kernel<3>; break;
        default: kern = (const void *)batch_kernel<4>; break;
    }
    BCK(cudaLaunchCooperativeKernel(kern, dim3(b->grid_blocks), b->tile, args, 0, b->s));
    BCK(cudaMemcpyAsync(b->h_err, b->d_err, 4 * sizeof(int), cudaMemcpyDeviceToHost, b->s));
    return CDF_OK;
}

cdf_status launch_batch(cdf_batch *b, int nsteps, bool moments_last) {
    cdf_status st = enqueue_batch(b, nsteps, moments_last, b->cur, b->sprev, b->sprev);
    if (st != CDF_OK) return st;
    if (nsteps & 1) b->cur ^= 1;
    b->t += nsteps;
    return CDF_OK;
}

constexpr int kPoolStreams = 32;
constexpr int kChainGraphSteps = 32;  // even: the buffer parity returns

// S_1(t - 1) plane set that belongs to population buffer `par`.
float *sprev_of(cdf_batch *b, int par) {
    return ((b->mode == 0 && !b->fused) || par == 0) ? b->sprev : b->sprev2;
}

// Do the steps run as launches that each flip the buffers (all but the persistent kernel)?
bool in_launches(const cdf_batch *b) { return b->mode >= 1 || b->fused; }

// Kernel launches of the chains for n steps: one per step, or in mode 2 one per
// two steps plus one single step for an odd n.  Each launch flips the parity.
int chain_launches(const cdf_batch *b, int nsteps) {
    return b->mode == 2 || b->fused ? nsteps / 2 + nsteps % 2 : nsteps;
}

// Enqueue n steps of all instances as launches of two steps each, group by group (kFusedLanes);
// an odd n ends with one step of the persistent kernel's code.
cdf_status enqueue_fused(cdf_batch *b, int nsteps, bool moments_last, int parity0) {
    const std::vector<int> &start = b->group_start;
    const int groups = (int)start.size() - 1, pairs = nsteps / 2;
    const size_t lanes = std::min({(size_t)kFusedLanes, (size_t)groups, b->pool.size()});
    const int par1 = parity0 ^ (pairs & 1);
    if (lanes > 1) {
        BCK(cudaEventRecord(b->ev_fork, b->s));
        for (size_t j = 0; j < lanes; ++j) BCK(cudaStreamWaitEvent(b->pool[j], b->ev_fork, 0));
    }
    for (int g = 0; g < groups; ++g) {
        const int k0 = start[g], k1 = start[g + 1];
        for (int j = 0; j < pairs; ++j) {
            const int par = (parity0 + j) & 1;
            BCK(launch_step2_batch(b->m, b->kind, b->inst.data() + k0, k1 - k0, b->buf[par], b->buf[par ^ 1],
                                   sprev_of(b, par), sprev_of(b, par ^ 1),
                                   moments_last && 2 * (j + 1) == nsteps ? b->mom : nullptr,
                                   lanes > 1 ? b->pool[g % lanes] : b->s));
        }
    }
    if (lanes > 1)
        for (size_t j = 0; j < lanes; ++j) {
            BCK(cudaEventRecord(b->ev_join[j], b->pool[j]));
            BCK(cudaStreamWaitEvent(b->s, b->ev_join[j], 0));
        }
    if (nsteps & 1) return enqueue_batch(b, 1, moments_last, par1, sprev_of(b, par1), sprev_of(b, par1 ^ 1));
    return CDF_OK;
}

// Enqueue n steps of every instance as chains of single-lattice step kernels on
// the stream pool (fork from and join back to the batch stream).
cdf_status enqueue_chains(cdf_batch *b, int nsteps, bool moments_last, int parity0) {
    if (b->fused) return enqueue_fused(b, nsteps, moments_last, parity0);
    BCK(cudaEventRecord(b->ev_fork, b->s));
    for (cudaStream_t ps : b->pool) BCK(cudaStreamWaitEvent(ps, b->ev_fork, 0));
    const int launches = chain_launches(b, nsteps);
    for (int j = 0; j < launches; ++j) {
        const int par = (parity0 + j) & 1;
        const bool two = b->mode == 2 && 2 * (j + 1) <= nsteps;
        for (int k = 0; k < b->count; ++k) {
            float *mom = (moments_last && j == launches - 1) ? b->mom + b->mom_off[k] : nullptr;
            float *in = b->buf[par] + b->pop_off[k], *out = b->buf[par ^ 1] + b->pop_off[k];
            float *sin = sprev_of(b, par) + b->sp_off[k], *sout = sprev_of(b, par ^ 1) + b->sp_off[k];
            cudaStream_t ps = b->pool[k % b->pool.size()];
            if (two)
                BCK(launch_step2(b->params[k], in, out, sin, sout, mom, b->chain_block, b->chain_th, ps));
            else
                BCK(launch_step(b->params[k], kFP32, in, out, sin, sout, mom,
                                b->mode == 2 ? dim3(128, 1) : b->chain_block, ps));
        }
    }
    for (size_t j = 0; j < b->pool.size(); ++j) {
        BCK(cudaEventRecord(b->ev_join[j], b->pool[j]));
        BCK(cudaStreamWaitEvent(b->s, b->ev_join[j], 0));
    }
    return CDF_OK;
}

// Changing the CTA shape of the chains invalidates their captured graphs.
void set_chain_block(cdf_batch *b, dim3 blk) {
    for (auto &row : b->chain_graph)
        for (auto &g : row)
            if (g) {
                cudaGraphExecDestroy(g);
                g = nullptr;
            }
    b->chain_block = blk;
}

cdf_status run_chains(cdf_batch *b, int nsteps, bool moments_last) {
    if (nsteps == kChainGraphSteps) {
        cudaGraphExec_t &ge = b->chain_graph[b->cur][moments_last ? 1 : 0];
        if (!ge) {
            cudaGraph_t g = nullptr;
            BCK(cudaStreamBeginCapture(b->s, cudaStreamCaptureModeThreadLocal));
            cdf_status st = enqueue_chains(b, nsteps, moments_last, b->cur);
            cudaError_t e = cudaStreamEndCapture(b->s, &g);
            if (st != CDF_OK) {
                if (g) cudaGraphDestroy(g);
                return st;
            }
            BCK(e);
            e = cudaGraphInstantiate(&ge, g, 0);
            cudaGraphDestroy(g);
            BCK(e);
        }
        BCK(cudaGraphLaunch(ge, b->s));
    } else {
        cdf_status st = enqueue_chains(b, nsteps, moments_last, b->cur);
        if (st != CDF_OK) return st;
    }
    if (chain_launches(b, nsteps) & 1) b->cur ^= 1;
    b->t += nsteps;
    return CDF_OK;
}

// Can step2_kernel with CTA blk and tile height th run every instance?  blk.z
// == 2: the paired-lane kernel (m <= 2, CTAs of 32 x 8, tile heights 14 and 30).
bool chain_pair_fits(const cdf_batch *b, dim3 blk, int th) {
    if (blk.z == 2 && (b->m > 2 || blk.x != 32 || blk.y != 8 || (th != 14 && th != 30))) return false;
    if (blk.x % 32 != 0 || (int)(blk.x * blk.y) > step2_max_threads(b->m) || th < 1) return false;
    if (step2_smem_bytes(b->m, blk, th) > (size_t)kStep2MaxSmem) return false;
    for (const LbParams &p : b->params)
        if ((p.periodic_x && p.nx < (int)blk.x) || (p.periodic_y && p.ny < th + 2)) return false;
    return true;
}

// Can two steps of all instances run in a launch: every instance has a tiling (and the barrier's
// test hook is off)?
bool fused_fits(const cdf_batch *b) {
    int tw, th;
    for (const LbParams &p : b->params)
        if (!pair_tile(p, tile_nodes(b->nodes), &tw, &th) || (9 + 5 * b->m) * p.plane >= (1ll << 31)) return false;
    return !b->extra_arrivals;
}

// Are the two-step launches surely faster than the persistent kernel, which moves twice the bytes?  With one or
// two scalars and tiles of 96 nodes and more, their ring included, on average they were on every
// batch measured.  Thin lattices leave most of a CTA's eight warps idle, and three and four scalars let fewer CTAs
// on an SM: 500 lattices of 2000 x 1 take 83 us a step (two scalars) against 37, 1500 of 7 x 7 17.5 against 16.3, 166
// of 2000 x 3 with three scalars 67 against 47, but 166 of 3 x 2000 with four 185 against 716.  Those are timed.
bool fused_surely(const cdf_batch *b) {
    double nodes = 0, tiles = 0;
    for (const LbParams &p : b->params) {
        int tw = 1, th = 1;
        pair_tile(p, tile_nodes(b->nodes), &tw, &th);
        const double tx = (p.nx + tw - 1) / tw, ty = (p.ny + th - 1) / th;
        nodes += (p.nx + 2 * (tx - 1) + 2 * p.periodic_x) * (p.ny + 2 * (ty - 1) + 2 * p.periodic_y);
        tiles += tx * ty;
    }
    return b->m <= 2 && nodes >= 96 * tiles;
}

cdf_status check_err(cdf_batch *b) {
    if (*b->h_err) {
        char m[256];
        std::snprintf(m, sizeof m,
                      "grid barrier wait timed out after step %d of a launch (%d of %d blocks had arrived, waited %d "
                      "us); the batch state is undefined",
                      b->h_err[1], b->h_err[2], b->grid_blocks + b->extra_arrivals, b->h_err[3]);
        return bfail(CDF_ETIMEOUT, m);
    }
    return CDF_OK;
}

// (mode, tile or chain block, tile height of mode 2); a chain block with z == 2
// names the paired-lane two-step kernel
struct ModeChoice {
    int mode;
    dim3 shape;
    int th;
    bool fused;  // mode 0: the two-step launches
};
std::map<TuneKey, ModeChoice> g_bmode;
std::map<std::tuple<TuneKey, unsigned, unsigned>, bool> g_bfused;  // mode 0 with a given tile

// what decides which kernels run and how well belongs to the key: the closure kind, the two-step tiling
TuneKey tune_key(const cdf_batch *b) {
    const int kernels = 2 * (2 * (b->kind + 1) + (fused_fits(b) ? 1 : 0)) + b->params[0].chemotaxis;
    long long rows = 0;
    for (const LbParams &p : b->params) rows += 3ll * p.ny + p.periodic_x + (p.periodic_y ? 1ll << 40 : 0);
    return TuneKey{b->nodes, rows, b->count, b->m, kernels};
}

// Milliseconds of run(nsteps) after a warm-up (and graph capture), the least of up to four where they are short
// enough for the host to disturb, or -1.
template <class Run>
float time_batch(cdf_batch *b, int nsteps, const Run &run) {
    cudaEvent_t e[2] = {nullptr, nullptr};
    bool ok = cudaEventCreate(&e[0]) == cudaSuccess && cudaEventCreate(&e[1]) == cudaSuccess && run(nsteps) == CDF_OK;
    float least = 1e30f, all = 0;
    for (int r = 0; ok && r < 4 && all < 1.f; ++r) {
        float ms = 0;
        ok = cudaEventRecord(e[0], b->s) == cudaSuccess && run(nsteps) == CDF_OK &&
             cudaEventRecord(e[1], b->s) == cudaSuccess && cudaEventSynchronize(e[1]) == cudaSuccess &&
             check_err(b) == CDF_OK && cudaEventElapsedTime(&ms, e[0], e[1]) == cudaSuccess;
        least = std::min(least, ms);
        all += ms;
    }
    for (cudaEvent_t ev : e)
        if (ev) cudaEventDestroy(ev);
    return ok ? least : -1.f;
}
// The same of 32 steps of the whole-batch kernel that b->fused names, with the tile that is set up.
float time_whole(cdf_batch *b) {
    if (b->fused) return time_batch(b, kChainGraphSteps, [&](int n) { return run_chains(b, n, false); });
    const int steps = b->nodes > (1 << 22) ? 4 : 16;
    const float ms = time_batch(b, steps, [&](int n) { return launch_batch(b, n, false); });
    return ms * ((float)kChainGraphSteps / steps);
}

// Mode 0 with a given tile: the two-step launches, or the persistent kernel with this tile where
// those are not surely and not measurably faster.
cdf_status setup_whole(cdf_batch *b, dim3 tile) {
    b->fused = fused_fits(b);
    cdf_status st = setup_tiles(b, tile);
    if (st != CDF_OK || !b->fused || fused_surely(b)) return st;
    const auto key = std::make_tuple(tune_key(b), tile.x, tile.y);
    {
        std::lock_guard<std::mutex> lk(g_btune_mu);
        const auto it = g_bfused.find(key);
        if (it != g_bfused.end()) {
            b->fused = it->second;
            return CDF_OK;
        }
    }
    float ms[2];
    for (int f = 1; f >= 0; --f) {
        b->fused = f;
        ms[f] = time_whole(b);
        set_chain_block(b, b->chain_block);  // drops the captured launches
        b->cur = 0;
        b->t = 0;
        if (ms[f] < 0) return bfail(CDF_ECUDA, "timing the whole-batch kernels failed");
    }
    b->fused = ms[1] < ms[0];
    std::lock_guard<std::mutex> lk(g_btune_mu);
    g_bfused[key] = b->fused;
    return CDF_OK;
}

cdf_status bautotune(cdf_batch *b) {
    const TuneKey key = tune_key(b);
    {
        std::lock_guard<std::mutex> lk(g_btune_mu);
        auto it = g_bmode.find(key);
        if (it != g_bmode.end() && (it->second.mode != 2 || chain_pair_fits(b, it->second.shape, it->second.th))) {
            b->mode = it->second.mode;
            if (b->mode >= 1) {
                set_chain_block(b, it->second.shape);
                b->chain_th = it->second.th;
                return setup_tiles(b, dim3(64, 4));
            }
            b->fused = it->second.fused;
            return setup_tiles(b, it->second.shape);
        }
    }
    float best = 1e30f;
    ModeChoice choice{0, dim3(64, 4), 0, false};
    const dim3 tiles[] = {dim3(64, 4), dim3(32, 4), dim3(32, 8), dim3(64, 2), dim3(128, 1), dim3(128, 2),
                          dim3(256, 1)};
    b->mode = 0;
    const bool fits = fused_fits(b), surely = fits && fused_surely(b);
    if (fits) {  // (the tile shape matters to the persistent kernel only)
        b->fused = true;
        cdf_status st = setup_tiles(b, tiles[0]);
        if (st != CDF_OK) return st;
        best = time_whole(b);
        if (best < 0) return bfail(CDF_ECUDA, "autotuning the whole-batch kernels failed");
        choice = {0, tiles[0], 0, true};
    }
    b->fused = false;
    set_chain_block(b, b->chain_block);  // drops the captured launches
    b->cur = 0;  // (the persistent kernel has one S(t - 1) for both parities)
    if (!surely)
        for (const dim3 &c : tiles) {
            cdf_status st = setup_tiles(b, c);
            if (st != CDF_OK) return st;
            const float ms = time_whole(b);
            if (ms < 0) return bfail(CDF_ECUDA, "autotuning the whole-batch kernels failed");
            if (ms < best) { best = ms; choice = {0, c, 0, false}; }
        }
    // (chains have to be 5 % ahead of the two-step launches: their graphs of a branch per instance cost a
    // call more; 20 lattices of 64 x 64 take 3.8 us a step as chains, 3.6 in two-step launches)
    const dim3 blocks[] = {dim3(128, 1), dim3(128, 2), dim3(256, 1), dim3(64, 4), dim3(32, 8), dim3(128, 0),
                           dim3(256, 0)};  // y == 0: flat launch
    b->mode = 1;
    for (const dim3 &c : blocks) {
        set_chain_block(b, c);
        const float ms = time_batch(b, kChainGraphSteps, [&](int n) { return run_chains(b, n, false); });
        if (ms < 0) return bfail(CDF_ECUDA, "autotuning the kernel chains failed");
        if (ms < best * (choice.fused ? 0.95f : 1.f)) { best = ms; choice = {1, c, 0, false}; }
    }
    // chains of two-step launches: CTA shape and tile height (the paired-lane
    // kernel, chain_lanes = 2, measured slower on GB300 and is not timed here)
    const std::pair<dim3, int> pairs[] = {{dim3(32, 8), 14}, {dim3(32, 8), 6}, {dim3(32, 16), 14},
                                          {dim3(64, 8), 14}, {dim3(32, 16), 30}};
    b->mode = 2;
    for (const auto &c : pairs) {
        if (!chain_pair_fits(b, c.first, c.second)) continue;
        set_chain_block(b, c.first);
        b->chain_th = c.second;
        const float ms = time_batch(b, kChainGraphSteps, [&](int n) { return run_chains(b, n, false); });
        if (ms < 0) return bfail(CDF_ECUDA, "autotuning the two-step kernel chains failed");
        if (ms < best * (choice.fused ? 0.95f : 1.f)) { best = ms; choice = {2, c.first, c.second, false}; }
    }
    b->t = 0;
    b->cur = 0;
    {
        std::lock_guard<std::mutex> lk(g_btune_mu);
        g_bmode[key] = choice;
    }
    b->mode = choice.mode;
    set_chain_block(b, b->mode >= 1 ? choice.shape : b->chain_block);
    if (b->mode >= 1) {
        b->chain_th = choice.th;
        return setup_tiles(b, dim3(64, 4));
    }
    b->fused = choice.fused;
    return setup_tiles(b, choice.shape);
}

}  // namespace

extern "C" {

cdf_status cdf_batch_create(int count, const cdf_grid *grids, int m, const cdf_diffusion *diffusion, const double *nu,
                            const cdf_source *source, const cdf_force *force, const cdf_boundaries *boundaries,
                            const double *phi_ref, const double *p_ref_grad, const cdf_batch_options *opt,
                            cdf_batch **out) {
    if (!out) return bfail(CDF_EINVAL, "out is NULL");
    *out = nullptr;
    if (count < 1 || !grids || !diffusion || !nu || !source || !force || !boundaries || !phi_ref || !p_ref_grad || !opt)
        return bfail(CDF_EINVAL, "NULL argument or count < 1");
    if (opt->storage != CDF_FP32) return bfail(CDF_EINVAL, "the batched solver stores FP32 populations only");
    if (!(opt->rho0 > 0.0)) return bfail(CDF_EINVAL, "rho0 must be positive");
    if (opt->mode < 0 || opt->mode > 2) return bfail(CDF_EINVAL, "mode must be 0, 1 or 2");
    if ((opt->tile_x != 0 || opt->tile_y != 0) && opt->mode != 2) {
        if (opt->tile_x <= 0 || opt->tile_y <= 0 || opt->tile_x * opt->tile_y > 256 || opt->tile_x % 32 != 0)
            return bfail(CDF_EINVAL, "tile must be a multiple of 32 wide and at most 256 nodes");
    }
    if (opt->steps_per_launch < 0 || opt->barrier_timeout_s < 0) return bfail(CDF_EINVAL, "bad launch options");
    cdf_batch *b = new (std::nothrow) cdf_batch;
    if (!b) return bfail(CDF_ENOMEM, "host allocation failed");
    b->count = count;
    b->m = m;
    b->params.resize(count);
    int sprev_planes = -1;
    for (int k = 0; k < count; ++k) {
        const int pitch = grids[k].nx >= 1 ? (grids[k].nx + 31) / 32 * 32 : 0;
        cdf_status st = build_params(&grids[k], m, &diffusion[k], nu[k], &source[k], &force[k], &boundaries[k], false,
                                     opt->rho0, phi_ref + (size_t)k * m, p_ref_grad + 2 * (size_t)k, pitch,
                                     &b->params[k]);
        if (st != CDF_OK) {
            delete b;
            return st;
        }
        const int spp = source[k].kind == CDF_S_CONSUMPTION ? 1 : 0;
        if (sprev_planes >= 0 && spp != sprev_planes) {
            delete b;
            return bfail(CDF_EINVAL, "all instances must use the same source kind");
        }
        sprev_planes = spp;
        b->pop_off.push_back(b->pop_total);
        b->sp_off.push_back(b->sp_total);
        b->mom_off.push_back(b->mom_total);
        b->node_off.push_back(b->nodes);
        const long long plane = b->params[k].plane;
        b->pop_total += (long long)(9 + 5 * m) * plane;
        b->sp_total += plane;
        b->mom_total += (long long)(m + 3) * plane;
        b->nodes += (long long)grids[k].nx * grids[k].ny;
        b->stage_floats = std::max(b->stage_floats, (size_t)(m + 3) * grids[k].nx * grids[k].ny);
        b->max_nodes = std::max(b->max_nodes, (long long)grids[k].nx * grids[k].ny);
    }
    b->kind = batch_closure_kind(b->params.data(), count);
    b->sprev_planes = sprev_planes;
    b->steps_per_launch = opt->steps_per_launch > 0 ? opt->steps_per_launch : 32;
    b->timeout_ns = opt->barrier_timeout_s > 0 ? (unsigned long long)(opt->barrier_timeout_s * 1e9) : 1000000000ull;
    b->extra_arrivals = opt->test_unreachable_barrier ? 1 : 0;
    b->user = static_cast<cudaStream_t>(opt->cuda_stream);
    if (cudaGetDevice(&b->device) != cudaSuccess) { delete b; return bfail(CDF_ECUDA, "no CUDA device"); }
    bool ok = dev_alloc((void **)&b->buf[0], b->pop_total * 4) == cudaSuccess &&
              dev_alloc((void **)&b->buf[1], b->pop_total * 4) == cudaSuccess &&
              dev_alloc((void **)&b->sprev, b->sp_total * 4) == cudaSuccess &&
              dev_alloc((void **)&b->sprev2, b->sp_total * 4) == cudaSuccess &&
              dev_alloc((void **)&b->mom, b->mom_total * 4) == cudaSuccess &&
              dev_alloc((void **)&b->mom_prev, b->mom_total * 4) == cudaSuccess &&
              cudaMalloc(&b->partials, (size_t)reduce_quantities(m) * kReduceBlocks * sizeof(double)) == cudaSuccess &&
              cudaMalloc(&b->red, (size_t)count * reduce_quantities(m) * sizeof(double)) == cudaSuccess &&
              cudaMallocHost(&b->red_host, (size_t)count * reduce_quantities(m) * sizeof(double)) == cudaSuccess &&
              dev_alloc((void **)&b->dense, b->stage_floats * 4) == cudaSuccess &&
              cudaMalloc(&b->d_inst, count * sizeof(BatchInst)) == cudaSuccess &&
              cudaMalloc(&b->d_bar, 2 * sizeof(unsigned)) == cudaSuccess &&
              cudaMalloc(&b->d_err, 4 * sizeof(int)) == cudaSuccess &&
              cudaMallocHost(&b->h_err, 4 * sizeof(int)) == cudaSuccess &&
              cudaMallocHost(&b->host_stage, b->stage_floats * 4) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        brelease(b);
        return bfail(CDF_ENOMEM, "device allocation failed");
    }
    std::memset(b->h_err, 0, 4 * sizeof(int));  // read after every step call, also in the chain modes
    if (cudaStreamCreateWithFlags(&b->s, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->ev_in, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->ev_out, cudaEventDisableTiming) != cudaSuccess ||
        cudaMemset(b->buf[0], 0, b->pop_total * 4) != cudaSuccess || cudaMemset(b->buf[1], 0, b->pop_total * 4) != cudaSuccess ||
        cudaMemset(b->sprev, 0, b->sp_total * 4) != cudaSuccess || cudaMemset(b->sprev2, 0, b->sp_total * 4) != cudaSuccess ||
        cudaMemset(b->mom, 0, b->mom_total * 4) != cudaSuccess ||
        cudaMemset(b->d_bar, 0, 2 * sizeof(unsigned)) != cudaSuccess) {
        brelease(b);
        return bfail(CDF_ECUDA, "stream / memory set-up failed");
    }
    b->pool.resize(std::min(count, kPoolStreams));
    b->ev_join.resize(b->pool.size());
    bool pok = cudaEventCreateWithFlags(&b->ev_fork, cudaEventDisableTiming) == cudaSuccess;
    for (size_t j = 0; j < b->pool.size() && pok; ++j)
        pok = cudaStreamCreateWithFlags(&b->pool[j], cudaStreamNonBlocking) == cudaSuccess &&
              cudaEventCreateWithFlags(&b->ev_join[j], cudaEventDisableTiming) == cudaSuccess;
    if (!pok) {
        brelease(b);
        return bfail(CDF_ECUDA, "stream pool set-up failed");
    }
    b->mode = opt->mode;
    if (opt->chain_lanes < 0 || opt->chain_lanes > 2 || (opt->chain_lanes == 2 && !(opt->mode == 2 && opt->tile_x > 0))) {
        brelease(b);
        return bfail(CDF_EINVAL, "chain_lanes: 0, 1, or 2 with mode 2 and a given tile");
    }
    if (opt->mode >= 1 && opt->tile_x > 0)
        set_chain_block(b, dim3(opt->tile_x, opt->tile_y, opt->mode == 2 && opt->chain_lanes == 2 ? 2 : 1));
    if (opt->mode == 2 && opt->tile_x > 0) {
        b->chain_th = opt->chain_tile_y > 0 ? opt->chain_tile_y : 14;
        if (!chain_pair_fits(b, b->chain_block, b->chain_th)) {
            brelease(b);
            return bfail(CDF_EINVAL, "the two-step kernel shape cannot run every instance");
        }
    }
    cdf_status st;
    if (opt->mode >= 1 && opt->tile_x > 0) st = setup_tiles(b, dim3(64, 4));
    else if (opt->tile_x > 0) st = setup_whole(b, dim3(opt->tile_x, opt->tile_y));
    else if (b->extra_arrivals) st = setup_tiles(b, dim3(64, 4));
    else st = bautotune(b);
    if (st == CDF_OK && cudaStreamSynchronize(b->s) != cudaSuccess) st = bfail(CDF_ECUDA, "set-up failed");
    if (st != CDF_OK) {
        brelease(b);
        return st;
    }
    *out = b;
    return CDF_OK;
}

void cdf_batch_destroy(cdf_batch *b) {
    if (!b) return;
    cudaStreamSynchronize(b->s);
    brelease(b);
}

cdf_status cdf_batch_init_moments(cdf_batch *b, int k, const double *phi, const double *u, const double *p) {
    if (!b || !phi || !u || k < 0 || k >= b->count) return bfail(CDF_EINVAL, "bad argument");
    const LbParams &P = b->params[k];
    const size_t n = (size_t)P.nx * P.ny;
    BCK(cudaStreamSynchronize(b->s));  // the staging buffer may still feed a copy
    float *h = b->host_stage;
    for (int a = 0; a < b->m; ++a)
        for (size_t i = 0; i < n; ++i) h[a * n + i] = (float)phi[a * n + i];
    for (size_t i = 0; i < 2 * n; ++i) h[b->m * n + i] = (float)u[i];
    for (size_t i = 0; i < n; ++i) h[(b->m + 2) * n + i] = p ? (float)p[i] : 0.f;
    BCK(cudaEventRecord(b->ev_in, b->user));
    BCK(cudaStreamWaitEvent(b->s, b->ev_in, 0));
    BCK(cudaMemcpyAsync(b->dense, h, (size_t)(b->m + 3) * n * 4, cudaMemcpyHostToDevice, b->s));
    BCK(launch_init(P, kFP32, b->dense, P.nx, b->buf[b->cur] + b->pop_off[k], sprev_of(b, b->cur) + b->sp_off[k],
                    b->mom + b->mom_off[k], b->s));
    BCK(cudaEventRecord(b->ev_out, b->s));
    BCK(cudaStreamWaitEvent(b->user, b->ev_out, 0));
    return CDF_OK;
}

cdf_status cdf_batch_step(cdf_batch *b, long long n) {
    if (!b || n < 0) return bfail(CDF_EINVAL, "bad argument");
    if (n == 0) return CDF_OK;
    BCK(cudaEventRecord(b->ev_in, b->user));
    BCK(cudaStreamWaitEvent(b->s, b->ev_in, 0));
    while (n > 0) {
        const int k = (int)std::min<long long>(n, in_launches(b) ? kChainGraphSteps : b->steps_per_launch);
        cdf_status st = in_launches(b) ? run_chains(b, k, n == k) : launch_batch(b, k, n == k);
        if (st != CDF_OK) return st;
        n -= k;
    }
    BCK(cudaStreamSynchronize(b->s));  // the barrier's error flag is read on the host
    cdf_status st = check_err(b);
    if (st != CDF_OK) return st;
    if ((st = checks_verify(b->s)) != CDF_OK) return st;  // no-op unless built with -DCDF_CHECKS
    BCK(cudaEventRecord(b->ev_out, b->s));
    BCK(cudaStreamWaitEvent(b->user, b->ev_out, 0));
    return CDF_OK;
}

// Instances [k0, k1) of a device call: one instance, or all of them for k = -1.
static bool batch_range(const cdf_batch *b, int k, int *k0, int *k1) {
    if (k == -1) {
        *k0 = 0;
        *k1 = b->count;
        return true;
    }
    if (k < 0 || k >= b->count) return false;
    *k0 = k;
    *k1 = k + 1;
    return true;
}

cdf_status cdf_batch_init_moments_device(cdf_batch *b, int k, const float *dev_fields) {
    int k0, k1;
    if (!b || !dev_fields || !batch_range(b, k, &k0, &k1)) return bfail(CDF_EINVAL, "bad argument");
    BCK(cudaEventRecord(b->ev_in, b->user));
    BCK(cudaStreamWaitEvent(b->s, b->ev_in, 0));
    const float *src = dev_fields;
    if (k == -1 && b->count <= 65535) {
        BCK(launch_init_batch(b->m, b->d_inst, b->count, b->max_nodes, dev_fields, b->buf[b->cur], sprev_of(b, b->cur),
                              b->mom, b->s));
        k0 = k1;
    }
    for (int j = k0; j < k1; ++j) {
        const LbParams &P = b->params[j];
        BCK(launch_init(P, kFP32, src, P.nx, b->buf[b->cur] + b->pop_off[j], sprev_of(b, b->cur) + b->sp_off[j],
                        b->mom + b->mom_off[j], b->s));
        src += (size_t)(b->m + 3) * P.nx * P.ny;
    }
    BCK(cudaEventRecord(b->ev_out, b->s));
    BCK(cudaStreamWaitEvent(b->user, b->ev_out, 0));
    return CDF_OK;
}

cdf_status cdf_batch_moments_device(cdf_batch *b, int k, float *dev_out) {
    int k0, k1;
    if (!b || !dev_out || !batch_range(b, k, &k0, &k1)) return bfail(CDF_EINVAL, "bad argument");
    BCK(cudaEventRecord(b->ev_in, b->user));
    BCK(cudaStreamWaitEvent(b->s, b->ev_in, 0));
    float *dst = dev_out;
    if (k == -1 && b->count <= 65535) {
        BCK(launch_pack_batch(b->m, b->d_inst, b->count, b->max_nodes, b->mom, dev_out, b->s));
        k0 = k1;
    }
    for (int j = k0; j < k1; ++j) {
        const LbParams &P = b->params[j];
        BCK(launch_pack_moments(P, b->mom + b->mom_off[j], dst, b->s));
        dst += (size_t)(b->m + 3) * P.nx * P.ny;
    }
    BCK(cudaEventRecord(b->ev_out, b->s));
    BCK(cudaStreamWaitEvent(b->user, b->ev_out, 0));
    return CDF_OK;
}

cdf_status cdf_batch_moments(cdf_batch *b, int k, double *host_out) {
    if (!b || !host_out || k < 0 || k >= b->count) return bfail(CDF_EINVAL, "bad argument");
    const LbParams &P = b->params[k];
    const size_t n = (size_t)P.nx * P.ny * (b->m + 3);
    BCK(cudaEventRecord(b->ev_in, b->user));
    BCK(cudaStreamWaitEvent(b->s, b->ev_in, 0));
    BCK(launch_pack_moments(P, b->mom + b->mom_off[k], b->dense, b->s));
    BCK(cudaMemcpyAsync(b->host_stage, b->dense, n * 4, cudaMemcpyDeviceToHost, b->s));
    BCK(cudaStreamSynchronize(b->s));
    for (size_t i = 0; i < n; ++i) host_out[i] = b->host_stage[i];
    return CDF_OK;
}

cdf_status cdf_batch_get_info(const cdf_batch *b, cdf_batch_info *out) {
    if (!b || !out) return bfail(CDF_EINVAL, "NULL argument");
    out->count = b->count;
    out->m = b->m;
    out->nodes = b->nodes;
    out->tiles = b->total_tiles;
    out->tile_x = (int)b->tile.x;
    out->tile_y = (int)b->tile.y;
    out->grid_blocks = b->grid_blocks;
    out->steps_per_launch = b->steps_per_launch;
    out->bytes_per_lup = 2.0 * (9 + 5 * b->m) * 4.0 + 8.0 * b->sprev_planes;
    out->mode = b->mode;
    out->chain_block_x = (int)b->chain_block.x;
    out->chain_block_y = (int)b->chain_block.y;
    out->chain_tile_y = b->mode == 2 ? b->chain_th : 0;
    out->chain_lanes = b->mode >= 1 ? (int)b->chain_block.z : 1;
    out->t = b->t;
    return CDF_OK;
}

long long cdf_batch_launches(const cdf_batch *b, long long n) {
    if (!b || n < 0) return -1;
    if (b->mode == 1) return n * b->count;
    if (b->mode == 2) return (n / 2 + n % 2) * b->count;
    if (b->fused) return n / 2 * ((long long)b->group_start.size() - 1) + n % 2;
    return (n + b->steps_per_launch - 1) / b->steps_per_launch;
}

cdf_status cdf_batch_snapshot(cdf_batch *b) {
    if (!b) return bfail(CDF_EINVAL, "NULL handle");
    BCK(cudaEventRecord(b->ev_in, b->user));
    BCK(cudaStreamWaitEvent(b->s, b->ev_in, 0));
    BCK(cudaMemcpyAsync(b->mom_prev, b->mom, b->mom_total * 4, cudaMemcpyDeviceToDevice, b->s));
    BCK(cudaEventRecord(b->ev_out, b->s));
    BCK(cudaStreamWaitEvent(b->user, b->ev_out, 0));
    return CDF_OK;
}

cdf_status cdf_batch_residuals(cdf_batch *b, double *residual) {
    if (!b || !residual) return bfail(CDF_EINVAL, "NULL argument");
    const int nq = reduce_quantities(b->m), m = b->m;
    BCK(cudaEventRecord(b->ev_in, b->user));
    BCK(cudaStreamWaitEvent(b->s, b->ev_in, 0));
    for (int k = 0; k < b->count; ++k) {
        const LbParams &P = b->params[k];
        BCK(launch_reduce(b->mom + b->mom_off[k], b->mom_prev + b->mom_off[k], P.nx, P.ny, P.pitch, P.plane, m,
                          b->partials, b->red + (size_t)k * nq, b->s));
    }
    BCK(cudaMemcpyAsync(b->red_host, b->red, (size_t)b->count * nq * sizeof(double), cudaMemcpyDeviceToHost, b->s));
    BCK(cudaStreamSynchronize(b->s));
    for (int k = 0; k < b->count; ++k) {
        const double *q = b->red_host + (size_t)k * nq;
        double R = 0.0;
        for (int f = 0; f < m + 2; ++f) R = std::max(R, q[m + f] / std::max(q[2 * m + 2 + f], 1e-300));
        residual[k] = q[3 * m + 4] > 0 ? INFINITY : R;
    }
    return CDF_OK;
}

void *cdf_batch_stream(const cdf_batch *b) { return b ? static_cast<void *>(b->s) : nullptr; }

}  // extern "C"
