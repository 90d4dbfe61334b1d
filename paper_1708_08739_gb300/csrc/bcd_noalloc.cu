// RV(r) without any allocation: a single-root reach traversal of R(G) whose
// scratch lives in a file-scope device array.
//
// Some callers cannot call cudaMalloc: code that runs while an allocator is
// locked or being torn down, processes whose device memory is fully carved
// out by another framework's caching allocator, and plugins that are handed a
// stream and caller-owned buffers but no allocation rights. This entry point
// serves them: the caller passes the reverse graph and the output buffer as
// device pointers, and the call uses only the static array below.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "bcd.h"
#include "bcd_common.cuh"

namespace {

constexpr int32_t kMaxN = BC_NOALLOC_MAX_VERTICES;
constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kArcs = 4;         // arcs a lane has in flight
constexpr int kLongRow = 1024;   // longer rows are walked by a whole block

// Frontier of one level: its short rows are queued from the front of the
// level's buffer and its long ones from the back (a vertex is queued once, so
// they never meet), each drawn from a counter.
struct Frontier {
    uint32_t shorts, longs;        // queued
    uint32_t next_short, next_long;  // handed out past the first of each warp / block
};

struct NoallocScratch {
    uint32_t visited[kMaxN / 32];   // one bit per vertex
    int32_t queue[2][kMaxN];        // frontier of the current / next level
    int64_t block_count[1024];      // per-block counts for the ordered output
    Frontier front[3];              // of the current, the next and the level after (being cleared)
    uint32_t bar_count;
    uint32_t bar_gen;
    int32_t err;
    int32_t pad;
    int64_t total;
};

// The scratch array. Every call shares it and leaves its contents behind.
static __device__ __align__(256) NoallocScratch g_noalloc_scratch;

__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Blocks that take part: more than there is work for would only lengthen the
// barriers (1,000 vertices, 5,000 arcs: 137 us on 152 blocks, 85 us on 8), so
// one for every 2,048 vertices or 32,768 arcs, whichever asks for more, and at
// least 8. By vertices alone a dense graph would leave the chip to a few blocks
// (20,000 vertices, 38 million arcs: 4.0 ms on 9 blocks, 0.96 ms on all; 4,096
// vertices, 6.5 million arcs: 0.88 and 0.28 ms).
__host__ __device__ inline long long useful_blocks(long long n, long long m) {
    const long long by_n = n / 2048, by_m = m / 32768, b = by_n > by_m ? by_n : by_m;
    return b > 8 ? b : 8;
}

// Barrier of the nb blocks that take part; every wait gives up after ten seconds.
__device__ bool grid_sync(NoallocScratch *s, uint32_t &gen, uint32_t nb) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const uint32_t arrived = atomicAdd(&s->bar_count, 1u);
        if (arrived == nb - 1) {
            atomicExch(&s->bar_count, 0u);
            __threadfence();
            atomicExch(&s->bar_gen, gen + 1);
        } else {
            const unsigned long long t0 = now_ns();
            unsigned long long spins = 0;
            while (*(volatile uint32_t *)&s->bar_gen == gen) {
                if (*(volatile int32_t *)&s->err) break;
                if ((++spins & 63) == 0 && now_ns() - t0 > 10000000000ull) {
                    atomicCAS(&s->err, 0, 1);
                    break;
                }
                if (spins > (1ull << 31)) {
                    atomicCAS(&s->err, 0, 1);
                    break;
                }
                __nanosleep(40);
            }
        }
        __threadfence();
        gen += 1;
        ok = *(volatile int32_t *)&s->err == 0;
    }
    __syncthreads();
    return ok;
}

// Marks the heads y (negative: none) and queues the ones not seen before, short
// rows and long rows apart, with one counter atomic per warp and kind.
__device__ __forceinline__ void visit(NoallocScratch *s, const int64_t *roff, int next, Frontier *f,
                                      const int32_t (&y)[kArcs], int lane) {
    uint32_t word[kArcs];
#pragma unroll
    for (int k = 0; k < kArcs; ++k) word[k] = y[k] >= 0 ? __ldcg(&s->visited[y[k] >> 5]) : ~0u;
#pragma unroll
    for (int k = 0; k < kArcs; ++k) {
        bool fresh = false, lng = false;
        const uint32_t bit = 1u << (y[k] & 31);
        if (!(word[k] & bit)) fresh = !(atomicOr(&s->visited[y[k] >> 5], bit) & bit);
        if (!__any_sync(0xffffffffu, fresh)) continue;
        if (fresh) lng = roff[y[k] + 1] - roff[y[k]] > kLongRow;
        const unsigned ms = __ballot_sync(0xffffffffu, fresh && !lng), ml = __ballot_sync(0xffffffffu, lng);
        uint32_t bs = 0, bl = 0;
        if (lane == 0) {
            if (ms) bs = atomicAdd(&f->shorts, (uint32_t)__popc(ms));
            if (ml) bl = atomicAdd(&f->longs, (uint32_t)__popc(ml));
        }
        bs = __shfl_sync(0xffffffffu, bs, 0);
        bl = __shfl_sync(0xffffffffu, bl, 0);
        const unsigned below = (1u << lane) - 1u;
        if (lng)
            s->queue[next][kMaxN - 1 - (bl + __popc(ml & below))] = y[k];
        else if (fresh)
            s->queue[next][bs + __popc(ms & below)] = y[k];
    }
}

// Level-synchronous BFS over R(G), one grid barrier per level. A warp draws up
// to 32 frontier vertices and packs their arcs onto its lanes, kArcs per lane in
// flight; rows of more than kLongRow arcs go to whole blocks. On R-MAT 22 with
// reciprocal arcs one warp per vertex, with one counter atomic per discovered
// vertex, took 5.2 ms: its longest rows, tens of thousands of arcs behind one
// warp, were the time of a level.
__global__ void __launch_bounds__(kThreads, 2) rv_noalloc_kernel(NoallocScratch *s, const int64_t *roff,
                                                                  const int32_t *rcol, int32_t n, int32_t r,
                                                                  int32_t *out, int64_t cap) {
    __shared__ int s_incl[kWarps][32];
    __shared__ long long s_off[kWarps][32];
    __shared__ uint32_t s_long;
    uint32_t gen = 0;
    const uint32_t nb = (uint32_t)min((long long)gridDim.x, useful_blocks(n, roff[n] - roff[0]));
    if (blockIdx.x >= nb) return;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long nthr = (long long)nb * blockDim.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t gw = blockIdx.x * kWarps + warp, nw = nb * kWarps;
    const int words = (n + 31) / 32;
    int *incl = s_incl[warp];
    long long *off = s_off[warp];
    for (long long i = tid; i < words; i += nthr) s->visited[i] = i == (r >> 5) ? 1u << (r & 31) : 0u;
    if (tid == 0) {
        const bool lng = roff[r + 1] - roff[r] > kLongRow;
        s->queue[0][lng ? kMaxN - 1 : 0] = r;
        s->front[0].shorts = lng ? 0u : 1u;
        s->front[0].longs = lng ? 1u : 0u;
    }
    if (!grid_sync(s, gen, nb)) return;
    for (int level = 0;; ++level) {
        Frontier *cf = &s->front[level % 3], *nf = &s->front[(level + 1) % 3];
        const int cur = level & 1;
        const uint32_t shorts = __ldcg(&cf->shorts), longs = __ldcg(&cf->longs);
        if (shorts + longs == 0u) break;
        if (tid == 0) s->front[(level + 2) % 3] = Frontier{0u, 0u, 0u, 0u};
        // long rows: a block each, its first fixed, the others drawn
        for (uint32_t i = blockIdx.x; i < longs;) {
            const int32_t x = __ldcg(&s->queue[cur][kMaxN - 1 - i]);
            const long long b = roff[x], e = roff[x + 1];
            for (long long a0 = b; a0 < e; a0 += kThreads * kArcs) {
                int32_t y[kArcs];
#pragma unroll
                for (int k = 0; k < kArcs; ++k) {
                    const long long a = a0 + k * kThreads + threadIdx.x;
                    y[k] = a < e ? __ldcs(rcol + a) : -1;
                }
                visit(s, roff, cur ^ 1, nf, y, lane);
            }
            __syncthreads();
            if (threadIdx.x == 0) s_long = nb + atomicAdd(&cf->next_long, 1u);
            __syncthreads();
            i = s_long;
        }
        // short rows: groups of vertices, a warp's first fixed, the others drawn
        const uint32_t group = max(1u, min(32u, shorts / (nw * 4u)));
        for (uint32_t g0 = gw * group; g0 < shorts;) {
            long long b = 0;
            int len = 0;
            if (lane < group && g0 + lane < shorts) {
                const int32_t x = __ldcg(&s->queue[cur][g0 + lane]);
                b = roff[x];
                len = (int)(roff[x + 1] - b);
            }
            int in = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int z = __shfl_up_sync(0xffffffffu, in, o);
                if (lane >= o) in += z;
            }
            incl[lane] = in;
            off[lane] = b - (in - len);
            const int total = __shfl_sync(0xffffffffu, in, 31);
            __syncwarp();
            for (int base = 0; base < total; base += 32 * kArcs) {
                int32_t y[kArcs];
#pragma unroll
                for (int k = 0; k < kArcs; ++k) {
                    const int i = base + 32 * k + lane;
                    int v = 0;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1)
                        if (incl[v + o - 1] <= i) v += o;
                    y[k] = i < total ? __ldcs(rcol + off[v] + i) : -1;
                }
                visit(s, roff, cur ^ 1, nf, y, lane);
            }
            __syncwarp();
            const uint32_t drawn = nw * group;
            uint32_t g = shorts;
            if (drawn < shorts) {
                if (lane == 0) g = drawn + atomicAdd(&cf->next_short, group);
                g = __shfl_sync(0xffffffffu, g, 0);
            }
            g0 = g;
        }
        if (!grid_sync(s, gen, nb)) return;
    }
    // ordered output: counts per warp and block, every block sums the blocks
    // before it, every warp writes its words
    const int per = (words + (int)nb - 1) / (int)nb;
    const int wper = (per + kWarps - 1) / kWarps;
    const int w0 = min(words, (int)blockIdx.x * per + warp * wper);
    const int w1 = min(min(words, ((int)blockIdx.x + 1) * per), w0 + wper);
    __shared__ int s_cnt[kWarps];
    __shared__ long long s_base;
    int mine = 0;
    for (int w = w0 + lane; w < w1; w += 32) {
        uint32_t x = __ldcg(&s->visited[w]);
        if (w == (r >> 5)) x &= ~(1u << (r & 31));
        mine += __popc(x);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    if (lane == 0) s_cnt[warp] = mine;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long c = 0;
        for (int w = 0; w < kWarps; ++w) c += s_cnt[w];
        s->block_count[blockIdx.x] = c;
    }
    if (!grid_sync(s, gen, nb)) return;
    if (warp == 0) {
        long long before = 0, all = 0;
        for (int k = lane; k < (int)nb; k += 32) {
            const long long c = __ldcg(&s->block_count[k]);
            all += c;
            if (k < (int)blockIdx.x) before += c;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            before += __shfl_xor_sync(0xffffffffu, before, o);
            all += __shfl_xor_sync(0xffffffffu, all, o);
        }
        if (lane == 0) {
            s_base = all > cap ? -1 : before;
            if (blockIdx.x == 0) s->total = all;
        }
    }
    __syncthreads();
    if (s_base < 0) return;
    long long base = s_base;
    for (int w = 0; w < warp; ++w) base += s_cnt[w];
    for (int v0 = w0; v0 < w1; v0 += 32) {
        const int w = v0 + lane;
        uint32_t x = w < w1 ? __ldcg(&s->visited[w]) : 0u;
        if (w == (r >> 5)) x &= ~(1u << (r & 31));
        const int c = __popc(x);
        int in = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int z = __shfl_up_sync(0xffffffffu, in, o);
            if (lane >= o) in += z;
        }
        long long pos = base + in - c;
        while (x) {
            const int b = __ffs(x) - 1;
            x &= x - 1;
            out[pos++] = w * 32 + b;
        }
        base += __shfl_sync(0xffffffffu, in, 31);
    }
}

// Device address of the scratch array, looked up once per device.
std::mutex g_mu;
NoallocScratch *g_addr[64] = {nullptr};
int g_grid[64] = {0};

}  // namespace

extern "C" bc_status bc_rv_compute_noalloc(const int64_t *d_roffsets, const int32_t *d_rcols, int32_t n,
                                           int32_t r, int32_t *d_out, int64_t cap, int64_t *count,
                                           void *stream) {
    if (!d_roffsets || !d_rcols || !count || (cap > 0 && !d_out))
        return bcd::set_error(BC_E_INVALID_ARG, "bc_rv_compute_noalloc: NULL argument");
    if (n <= 0 || n > kMaxN)
        return bcd::set_error(BC_E_INVALID_ARG,
                              "bc_rv_compute_noalloc: n must be in [1, BC_NOALLOC_MAX_VERTICES = 4194304]");
    if (r < 0 || r >= n) return bcd::set_error(BC_E_INVALID_ARG, "bc_rv_compute_noalloc: vertex out of range");
    if (cap < 0) return bcd::set_error(BC_E_INVALID_ARG, "bc_rv_compute_noalloc: negative capacity");
    int dev = 0;
    BCD_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return bcd::set_error(BC_E_INTERNAL, "bc_rv_compute_noalloc: device index above 63");
    NoallocScratch *s = nullptr;
    int grid = 0;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (!g_addr[dev]) {
            void *p = nullptr;
            BCD_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
            int sms = 0, per_sm = 0;
            BCD_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
            BCD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, rv_noalloc_kernel, kThreads, 0));
            if (per_sm < 1) return bcd::set_error(BC_E_INTERNAL, "bc_rv_compute_noalloc: kernel cannot be resident");
            g_grid[dev] = std::min(sms * std::min(per_sm, 2), 1024);
            g_addr[dev] = (NoallocScratch *)p;
        }
        s = g_addr[dev];
        // the arcs are counted on the device; n (n - 1) is the most there can be
        grid = (int)std::min<long long>(g_grid[dev], useful_blocks(n, (long long)n * (n - 1)));
    }
    cudaStream_t st = (cudaStream_t)stream;
    BCD_CUDA(cudaMemsetAsync(&s->front[0], 0, sizeof(Frontier) * 3 + sizeof(uint32_t) * 2 + sizeof(int32_t) * 2, st));
    void *args[] = {(void *)&s, (void *)&d_roffsets, (void *)&d_rcols, (void *)&n, (void *)&r, (void *)&d_out,
                    (void *)&cap};
    BCD_CUDA(cudaLaunchCooperativeKernel((const void *)rv_noalloc_kernel, dim3(grid), dim3(kThreads), args, 0, st));
    int64_t total = 0;
    int32_t err = 0;
    BCD_CUDA(cudaMemcpyAsync(&total, &s->total, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    BCD_CUDA(cudaMemcpyAsync(&err, &s->err, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    BCD_CUDA(cudaStreamSynchronize(st));
    if (err) return bcd::set_error(BC_E_TIMEOUT, "bc_rv_compute_noalloc: a grid barrier wait timed out");
    *count = total;
    if (total > cap) return bcd::set_error(BC_E_BUFFER_TOO_SMALL, "bc_rv_compute_noalloc: output capacity below |RV(r)|");
    return BC_OK;
}
