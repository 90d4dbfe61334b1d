// Weighted single-source work (Section 2 with positive integer weights) with
// one source per block: each block takes the next source of the launch's
// union, runs its SPD in Dial's bucket order with block-wide barriers only,
// accumulates its dependencies (Eq. 4, or the vertex scan), writes them and
// takes the next source. Blocks never wait on one another, so a block whose
// source is cheap moves on while another is still deep in its distances:
// the grid-wide barrier per distance value of the tile kernel (hundreds of
// them per tile with weights up to 255) is gone, and so is the idle time of
// every lane waiting there for the slowest chain of the level.
//
// State of a block, for its current source s: one (dist(v), sigma(v)) pair
// per vertex v, 16 bytes (distance all ones when unreached; during the Eq. 4
// pass c(v) = (1 + delta(v)) / sigma(v) replaces sigma in place) or, in
// vertex-scan launches, one 8-byte word (24-bit distance, 40-bit count: half
// the footprint, so more of it stays in L2; a launch that overflows them
// reruns on 16-byte pairs); the settled vertices in settling order (history)
// with the start and distance of each distance level; and the bucket ring: R
// slots (R a power of two above the largest weight) of bcap queued vertices
// each, with their queued / consumed counters in shared memory. Eq. 4
// launches also keep one bit per arc (see src_offers).
//
// The state is indexed by position, not by vertex: positions sort the vertices
// by their in-degree's power of two, largest first (src_order). A relaxation
// touches a vertex once per in-arc, so the sectors that are touched most hold
// nothing else, and the vertices that no arc leads to (half of an R-MAT graph)
// take no room among the others. The heads of the arcs are kept as positions in
// a copy of the column array, the rows' bounds in one 16-byte pair per position.
//
// Sigma rides along the relaxations. Settling u at distance d (its sigma is
// final: every predecessor on a shortest path sits at a smaller distance and
// relaxed its arcs in an earlier level), each out-arc (u, v, w) offers the
// candidate nd = d + w: if nd is below dist(v) the pair becomes (nd,
// sigma(u)) and v is queued in the slot of nd; if nd equals dist(v),
// sigma(u) is added. The pair changes by one compare-and-swap (128 or 64
// bits), so a distance and its path count always move together, and when v settles its
// pair holds its distance with the sum over exactly its tight in-arcs (sigma
// values are integers: exact in any order below 2^53). Every arc is read
// once in the forward pass, along its tail's out-row; no in-arc pass.
// Where it fits, shared memory holds one bit per vertex that arcs lead to (the
// first positions): settled for the current source. An arc to a settled vertex can change nothing, and most arcs
// are such (they lead to hubs, which settle early), so their heads' distances,
// random 32-byte sectors each, are not read.
// A vertex queued in the slot of d whose distance has since dropped is stale
// and skipped; a vertex is queued only when its distance strictly drops, so
// it settles once.
//
// A level's queued vertices go to the warps in groups of up to 32, and a warp
// packs the out-arcs of its group onto its lanes (four arcs per lane in
// flight), so a level costs its arcs and not its longest row. Rows of more than
// kPackRows * weighted_short_row arcs are cut into chunk_arcs chunks that all
// warps take after a block barrier. The source is flagged when a sigma reaches
// 2^53. The Eq. 4 pass walks the levels from the deepest to the shallowest
// level holding a query vertex the source serves, summing c over tight
// out-arcs: it reads a vertex's arc bits 32 at a time and visits only the arcs
// whose bit is set (a row by 1 to 32 lanes and a fixed shuffle tree, longer
// rows by chunks added in chunk order), so delta is the same from run to run.
//
// Each source's dependencies delta_s.(r_q) go to sdep[i * 64 + q] (i its
// position in the launch's source list, q the queries that need it); a
// second kernel forms the per-tile, per-query sums in the fixed order the
// tile kernel uses.
//
// Bounded work: no block ever waits on another. A source that runs longer
// than timeout_ns, a full bucket slot, level array or chunk list, or a cancel
// request sets the launch's error word; the block leaves, the others stop at
// their next source, and the host resets the state (and grows what was full).
#include "bcd_common.cuh"
#include "bcd_wcols.cuh"
#include "bcd_device.cuh"

namespace bcd {

namespace {

using namespace dev;

constexpr int kLanesBatch = 4;  // arcs a lane loads together
constexpr int kPullBatch = 2;   // ... in the Eq. 4 pass, of those whose bit is set
// Rows of up to this many times weighted_short_row arcs are packed with their
// group's (forward) or walked by their lanes (backward); longer ones are cut.
constexpr int kPackRows = 4;
// Threads of the largest block (one per SM at 64 registers); see src_threads.
constexpr int kSrcThreads = 1024;
// Dynamic shared memory of a block (227 KB less the static arrays): the warps'
// staging, the ring's counters and, up to about 1.6 million vertices with
// in-arcs, the settled bits. (16-bit distance bounds of the first positions in
// what is left, to skip more reads, took the L1 cache that the register spills
// need: R-MAT 20 277 -> 420 ms at 224 KB, 264-272 ms at 32 to 64 KB.)
constexpr size_t kSrcDynSmem = 224 * 1024;
constexpr double kSrcTwo53 = 9007199254740992.0;

// (distance, sigma) of one vertex for the block's current source
struct __align__(16) DistSig {
    unsigned long long d;
    double s;
};

struct SrcParams {
    DistSig *ds;                // [blocks * n]
    int32_t *hv;                // [blocks * n] settled vertices of the current source
    int32_t *lstart;            // [blocks * maxlev] first history entry of each level
    unsigned long long *ldist;  // [blocks * maxlev] distance of each level
    uint32_t *bk;               // [blocks * ring * bcap] queued vertices, circular per slot
    Chunk *ch;                  // [blocks * chcap] long-row chunks of one level
    double *part;               // [blocks * chcap] backward chunk sums
    uint32_t *tb;               // [blocks * tbw] one bit per arc: its offer took effect (Eq. 4 launches)
    int64_t tbw;                // words per block: (m + 31) / 32
    double *sdep;               // [nsrc * 64]
    uint32_t *sflag;            // [nsrc] sigma >= 2^53 seen
    unsigned long long *next;   // source hand-out
    const int32_t *col;         // [m] heads, as positions
    const longlong2 *row;       // [n] arcs [x, y) of the vertex at a position
    const int32_t *pos;         // [n] position of a vertex
    const int32_t *inv;         // [n] vertex at a position
    int32_t heads;              // positions of vertices with in-arcs
    int64_t n;
    int64_t bcap;               // power of two
    int64_t chcap;
    int64_t nsrc;               // ntiles * S (padding entries are -1)
    int32_t ring;
    int32_t maxlev;
};

struct SrcStats {
    unsigned long long edges = 0, reached = 0, tight = 0, arcs = 0, vb = 0, eb = 0, pairs = 0;
};

__device__ __forceinline__ double sum_warp(double x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    return x;
}

// 16-byte compare-and-swap of a (distance, sigma) pair: true when *p held
// `expect` and now holds `nw`; otherwise `expect` receives what *p held.
__device__ __forceinline__ bool cas_pair(DistSig *p, DistSig &expect, const DistSig &nw) {
    const unsigned long long e0 = expect.d, e1 = (unsigned long long)__double_as_longlong(expect.s);
    const unsigned long long n0 = nw.d, n1 = (unsigned long long)__double_as_longlong(nw.s);
    unsigned long long o0, o1;
    asm volatile(
        "{\n\t.reg .b128 e, n, o;\n\t"
        "mov.b128 e, {%2, %3};\n\t"
        "mov.b128 n, {%4, %5};\n\t"
        "atom.global.cas.b128 o, [%6], e, n;\n\t"
        "mov.b128 {%0, %1}, o;\n\t}"
        : "=l"(o0), "=l"(o1)
        : "l"(e0), "l"(e1), "l"(n0), "l"(n1), "l"(p)
        : "memory");
    const bool ok = o0 == e0 && o1 == e1;
    expect.d = o0;
    expect.s = __longlong_as_double((long long)o1);
    return ok;
}

constexpr int kCasTries = 1 << 16;  // a pair changed under us this often: give up (never seen)

// Outcome of one offer to a head's pair.
enum Offer : int { kOfferNone = 0, kOfferTie = 1, kOfferLower = 2, kOfferStuck = -1, kOfferWide = -2 };

// Wide layout: 16-byte (distance, sigma) pairs, sigma in fp64 (the Eq. 4
// pass stores c there). Needed for Eq. 4 launches and for counts of 2^40 and
// more.
struct WidePairs {
    static constexpr bool kWide = true;
    static constexpr unsigned long long kUnreached = ~0ull;
    DistSig *ds;
    __device__ __forceinline__ unsigned long long dist(int v) const { return ds[v].d; }
    using Count = double;
    static __device__ __forceinline__ bool two53(double s) { return s >= kSrcTwo53; }
    __device__ __forceinline__ void get(int v, unsigned long long &d, double &sg) const {
        const DistSig x = ds[v];
        d = x.d;
        sg = x.s;
    }
    __device__ __forceinline__ void seed(int v) const {
        DistSig x;
        x.d = 0ull;
        x.s = 1.0;
        ds[v] = x;
    }
    __device__ __forceinline__ void clear(int v) const {
        DistSig x;
        x.d = ~0ull;
        x.s = 0.0;
        ds[v] = x;
    }
    using Seen = unsigned long long;  // what a first look at a head loads: its distance
    __device__ __forceinline__ Seen look(int v) const { return ds[v].d; }
    static __device__ __forceinline__ unsigned long long dist_of(Seen x) { return x; }
    __device__ __forceinline__ int offer(int v, unsigned long long nd, double sg, Seen) const {
        DistSig *q = ds + v;
        DistSig cur = *q;
        for (int it = 0; it < kCasTries; ++it) {
            if (nd > cur.d) return kOfferNone;
            const bool lower = nd < cur.d;
            DistSig nw;
            nw.d = nd;
            nw.s = lower ? sg : cur.s + sg;
            if (cas_pair(q, cur, nw)) return lower ? kOfferLower : kOfferTie;
        }
        return kOfferStuck;
    }
};

// Narrow layout: one 8-byte word per vertex, the distance in bits 0-23
// (2^24 - 1: unreached) and sigma as an integer in bits 24-63, changed by a
// 64-bit compare-and-swap. Half the footprint of the wide pairs, so more of
// the block's state stays in L2. A distance of 2^24 - 1 or more, or a count
// of 2^40 or more, asks for the wide layout (the launch reruns with it).
struct NarrowPairs {
    static constexpr bool kWide = false;
    static constexpr unsigned long long kDistMask = (1ull << 24) - 1;
    static constexpr unsigned long long kUnreached = kDistMask;
    static constexpr unsigned long long kSigLimit = 1ull << 40;
    unsigned long long *w;
    __device__ __forceinline__ unsigned long long dist(int v) const { return w[v] & kDistMask; }
    using Count = unsigned long long;  // converted to fp64 only where a dependency needs it
    static __device__ __forceinline__ bool two53(unsigned long long) { return false; }
    __device__ __forceinline__ void get(int v, unsigned long long &d, unsigned long long &sg) const {
        const unsigned long long x = w[v];
        d = x & kDistMask;
        sg = x >> 24;
    }
    __device__ __forceinline__ void seed(int v) const { w[v] = 1ull << 24; }
    __device__ __forceinline__ void clear(int v) const { w[v] = kDistMask; }
    using Seen = unsigned long long;  // ... its whole word, which the first compare-and-swap expects
    __device__ __forceinline__ Seen look(int v) const { return w[v]; }
    static __device__ __forceinline__ unsigned long long dist_of(Seen x) { return x & kDistMask; }
    __device__ __forceinline__ int offer(int v, unsigned long long nd, unsigned long long si, Seen cur) const {
        if (nd >= kDistMask) return kOfferWide;
        for (int it = 0; it < kCasTries; ++it) {
            const unsigned long long cd = cur & kDistMask;
            if (nd > cd) return kOfferNone;
            const bool lower = nd < cd;
            const unsigned long long ns = lower ? si : (cur >> 24) + si;
            if (ns >= kSigLimit) return kOfferWide;
            const unsigned long long nw = nd | (ns << 24);
            const unsigned long long old = atomicCAS(w + v, cur, nw);
            if (old == cur) return lower ? kOfferLower : kOfferTie;
            cur = old;
        }
        return kOfferStuck;
    }
};

__device__ __forceinline__ unsigned long long to_bits(unsigned long long x) { return x; }
__device__ __forceinline__ unsigned long long to_bits(double x) { return (unsigned long long)__double_as_longlong(x); }
template <class C>
__device__ __forceinline__ C from_bits(unsigned long long x);
template <>
__device__ __forceinline__ unsigned long long from_bits<unsigned long long>(unsigned long long x) { return x; }
template <>
__device__ __forceinline__ double from_bits<double>(unsigned long long x) { return __longlong_as_double((long long)x); }

// Arcs of a group of settled vertices, staged by one warp: the arcs of lane
// i's vertex end at incl[i] in the group's order; arc k of the group sits at
// off[its vertex] + k.
struct WarpArcs {
    int incl[32];
    long long off[32];
    unsigned long long sg[32];  // path counts of the vertices (integers or the bits of a double)
};

// Offers the group's arcs, kLanesBatch per lane in flight, of vertices settled
// at distance d: an offer lowers a head's distance (and queues it) or adds the
// tail's path count when the candidate ties. With tb (Eq. 4 launches), an offer
// that took effect also sets its arc's bit: every tight arc gets one (its offer
// of the final distance always takes effect), and arcs whose offer a shorter
// path replaced keep a stale bit that the backward's check drops. Returns 0, or
// the device error to raise (a pair that kept changing, a count or distance the
// narrow layout cannot hold).
template <class PairT, bool kBits>
__device__ __forceinline__ int src_offers(const TravParams &p, const PairT &P, uint32_t *bk, uint32_t *s_cnt,
                                          const uint32_t *s_done, uint32_t *tb, int64_t bcap, int R,
                                          unsigned long long d, const WarpArcs &wa, int total,
                                          const int32_t *col, unsigned long long &adds) {
    const int lane = threadIdx.x & 31;
    int err = 0;
    for (int base = lane; base < total; base += 32 * kLanesBatch) {
        int y[kLanesBatch];
        uint32_t w[kLanesBatch];
        unsigned vs = 0;  // the arcs' vertices, 5 bits each
#pragma unroll
        for (int j = 0; j < kLanesBatch; ++j) {
            const int i = base + 32 * j;
            int v = 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (wa.incl[v + o - 1] <= i) v += o;
            vs |= (unsigned)v << (5 * j);
            y[j] = -1;
            if (i < total) {
                const long long a = wa.off[v] + i;
                y[j] = __ldg(col + a);
                w[j] = __ldg(p.wt + a);
            }
        }
        if (kBits) {
#pragma unroll
            for (int j = 0; j < kLanesBatch; ++j)
                if (y[j] >= 0 && ((s_done[y[j] >> 5] >> (y[j] & 31)) & 1u)) y[j] = -1;
        }
        // the heads first; the compare-and-swap only for the few candidates
        // that lower or tie
        typename PairT::Seen cur[kLanesBatch];
#pragma unroll
        for (int j = 0; j < kLanesBatch; ++j)
            if (y[j] >= 0) cur[j] = P.look(y[j]);
#pragma unroll
        for (int j = 0; j < kLanesBatch; ++j) {
            if (y[j] < 0) continue;
            const unsigned long long nd = d + w[j];
            const unsigned long long cd = PairT::dist_of(cur[j]);
            // an unreached head takes every offer, also one past the narrow
            // layout's distances, for which the launch reruns
            if (nd > cd && cd != PairT::kUnreached) continue;
            const int v = (int)(vs >> (5 * j)) & 31;
            const int r = P.offer(y[j], nd, from_bits<typename PairT::Count>(wa.sg[v]), cur[j]);
            if (r > 0) {
                adds += 1;
                if (tb) {
                    const long long a = wa.off[v] + base + 32 * j;
                    atomicOr(tb + (a >> 5), 1u << (a & 31));
                }
                if (r == kOfferLower) {
                    const int slot = (int)(nd & (unsigned long long)(R - 1));
                    const uint32_t pos = atomicAdd(&s_cnt[slot], 1u);
                    bk[(size_t)slot * (size_t)bcap + (pos & (uint32_t)(bcap - 1))] = (uint32_t)y[j];
                }
            } else if (r == kOfferStuck) {
                err = kDevTimeout;
            } else if (r == kOfferWide) {
                err = kDevWide;
            }
        }
    }
    return err;
}

// Sum of c(y) over the tight out-arcs (y at distance d + w(v, y)) among arcs
// [a, ae) of a vertex at distance d, this lane's share: the words rl, rl + lpp,
// ... of the row's arc bits. Only arcs whose bit the forward set can be tight.
__device__ __forceinline__ double src_pull_c(const TravParams &p, const int32_t *col, const DistSig *ds, const uint32_t *tb,
                                             unsigned long long d, long long a, long long ae, int rl, int lpp) {
    double acc = 0.0;
    if (ae <= a) return acc;
    const long long w0 = a >> 5, w1 = (ae - 1) >> 5;
    for (long long w = w0 + rl; w <= w1; w += lpp) {
        uint32_t bits = tb[w];
        if (w == w0) bits &= ~0u << (a & 31);
        if (w == w1) bits &= ~0u >> (31 - ((ae - 1) & 31));
        while (bits) {
            bool ok[kPullBatch];
            unsigned long long want[kPullBatch];
            DistSig v[kPullBatch];
#pragma unroll
            for (int j = 0; j < kPullBatch; ++j) {
                ok[j] = bits != 0u;
                const long long aj = 32 * w + (ok[j] ? __ffs(bits) - 1 : 0);
                bits &= bits - 1u;
                if (ok[j]) {
                    want[j] = d + __ldg(p.wt + aj);
                    v[j] = ds[__ldg(col + aj)];
                }
            }
#pragma unroll
            for (int j = 0; j < kPullBatch; ++j)
                if (ok[j] && v[j].d == want[j]) acc += v[j].s;
        }
    }
    return acc;
}

// Lanes per vertex for a level of cnt vertices on a block of bd threads: the
// most (up to a warp) with which every vertex still gets its lanes at once.
__device__ __forceinline__ int lanes_per_vertex(long long cnt, int bd) {
    int lpp = 1;
    while (lpp < 32 && cnt * (long long)(2 * lpp) <= (long long)bd) lpp <<= 1;
    return lpp;
}

// Sum of the lane parts of one vertex's LPP lanes (a fixed butterfly).
__device__ __forceinline__ double sum_lanes(double x, int lpp) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
        if (o < lpp) x += __shfl_xor_sync(kFull, x, o);
    return x;
}

__device__ __forceinline__ void src_store_chunks(Chunk *chs, long long c0, int v, int e, int kind, long long rb,
                                                 long long re, int nch, int CH) {
    for (int k = 0; k < nch; ++k) {
        const long long a0 = rb + (long long)k * CH;
        store_chunk(&chs[c0 + k], v, e, k, nch, a0, (int)(min(re, a0 + CH) - a0), kind);
    }
}

// delta(v) = sigma(v) * acc; c(v) = (1 + delta(v)) / sigma(v) = 1 / sigma(v) +
// acc replaces sigma(v).
__device__ __forceinline__ void src_finalize(const TravParams &p, const int32_t *inv, DistSig *ds, uint64_t need, double *s_dep,
                                             int v, double acc) {
    const double sv = ds[v].s;
    ds[v].s = 1.0 / sv + acc;
    uint64_t y = __ldg(p.qmask + __ldg(inv + v)) & need;
    while (y) {
        const int q = __ffsll((long long)y) - 1;
        y &= y - 1;
        s_dep[q] = sv * acc;
    }
}

// kFew: every source has a block of its own (see step 1 of a level).
template <class PairT, bool kBits, bool kFew>
__global__ void __launch_bounds__(kSrcThreads, 1) wsrc_kernel(TravParams p, SrcParams q) {
    extern __shared__ __align__(16) unsigned char s_src[];  // WarpArcs per warp, ring counters, settled bits
    __shared__ int32_t s_ql[64];          // level at which query vertex q settled for this source
    __shared__ double s_dep[64];
    __shared__ double s_msum[64];         // several query vertices: per-column scan sums
    __shared__ unsigned long long s_cd[64];  // ... d(s, croot[c])
    __shared__ double s_red[32];
    __shared__ long long s_i;
    __shared__ int s_k, s_nh, s_err, s_flag, s_stop, s_group;
    const long long pack_max = (long long)kPackRows * p.wshort;
    __shared__ int s_nch[2];  // chunks of the current level, by level parity
    __shared__ unsigned long long s_t0;

    const int tid = threadIdx.x;
    const int bd = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nwarps = bd >> 5;
    const int R = q.ring;
    const int64_t bcap = q.bcap;
    const int CH = p.chunk_arcs;
    const int CHB = max(CH, 1024);  // backward chunks: a word of arc bits per lane
    WarpArcs &wa = reinterpret_cast<WarpArcs *>(s_src)[threadIdx.x >> 5];
    uint32_t *s_ring = reinterpret_cast<uint32_t *>(s_src + sizeof(WarpArcs) * (blockDim.x >> 5));  // [2 * R]: queued, then consumed, per slot
    uint32_t *s_cnt = s_ring;
    uint32_t *s_base = s_ring + R;
    uint32_t *s_done = s_ring + 2 * R;  // [(heads + 31) / 32]
    const int done_words = kBits ? (q.heads + 31) / 32 : 0;
    const size_t boff = (size_t)blockIdx.x * (size_t)q.n;
    DistSig *ds = q.ds + boff;  // wide pairs (Eq. 4 reads and writes them directly)
    PairT P;
    if constexpr (PairT::kWide)
        P.ds = ds;
    else
        P.w = reinterpret_cast<unsigned long long *>(q.ds) + boff;
    int32_t *hv = q.hv + boff;
    int32_t *lstart = q.lstart + (size_t)blockIdx.x * (size_t)q.maxlev;
    unsigned long long *ldist = q.ldist + (size_t)blockIdx.x * (size_t)q.maxlev;
    uint32_t *bk = q.bk + (size_t)blockIdx.x * (size_t)R * (size_t)bcap;
    Chunk *chs = q.ch + (size_t)blockIdx.x * (size_t)q.chcap;
    double *part = q.part + (size_t)blockIdx.x * (size_t)q.chcap;
    uint32_t *tb = p.mode == kModeSpd ? q.tb + (size_t)blockIdx.x * (size_t)q.tbw : nullptr;
    SrcStats st;
    unsigned long long ns_fwd = 0, ns_bwd = 0, ns_other = 0, t_mark = 0;
    unsigned long long lev_max = 0;
    if (tid == 0) t_mark = global_ns();

    for (;;) {
        __syncthreads();
        if (tid == 0) {
            const long long i = (long long)atomicAdd(q.next, 1ull);
            bool stop = i >= q.nsrc || ld_vol(&p.ctr->err) != 0;
            if (!stop && p.cancel && *(volatile const int32_t *)p.cancel != 0) {
                set_err(p.ctr, kDevCancelled);
                stop = true;
            }
            s_i = i;
            s_stop = stop ? 1 : 0;
            s_nh = 0;
            s_err = 0;
            s_flag = 0;
            s_nch[0] = 0;
            s_nch[1] = 0;
            const unsigned long long t = global_ns();
            ns_other += t - t_mark;
            t_mark = t;
            s_t0 = t;
        }
        for (int k = tid; k < 2 * R + done_words; k += bd) s_ring[k] = 0u;
        for (int k = tid; k < 64; k += bd) {
            s_ql[k] = -1;
            s_dep[k] = 0.0;
            s_msum[k] = 0.0;
        }
        __syncthreads();
        if (s_stop) break;
        const long long si = s_i;
        const int v0 = p.srcs[si];
        if (v0 < 0) continue;
        const uint64_t need = __ldg(p.need + v0);
        if (tid == 0) {
            const int x0 = __ldg(q.pos + v0);
            P.seed(x0);
            bk[0] = (uint32_t)x0;  // slot 0, position 0
            s_cnt[0] = 1u;
        }
        __syncthreads();

        // ---------------- forward: settle distance values in order ----------------
        unsigned long long d = 0;
        int seg = 0, nh = 0;
        bool first = true;
        for (;;) {
            if (tid == 0) {
                s_k = R;
                s_group = 0;
            }
            __syncthreads();
            for (int k = tid + (first ? 0 : 1); k < R; k += bd) {
                const int sl = (int)((d + (unsigned long long)k) & (unsigned long long)(R - 1));
                if (s_cnt[sl] != s_base[sl]) {
                    atomicMin(&s_k, k);
                    break;
                }
            }
            __syncthreads();
            const int kmin = s_k;
            if (kmin >= R) break;
            first = false;
            d += (unsigned long long)kmin;
            const int slot = (int)(d & (unsigned long long)(R - 1));
            const uint32_t b0 = s_base[slot];
            const uint32_t cnt = s_cnt[slot] - b0;
            if (seg + 1 >= q.maxlev || (int64_t)cnt > bcap) {
                if (tid == 0) set_err(p.ctr, seg + 1 >= q.maxlev ? kDevLevelOverflow : kDevBucketOverflow);
                return;
            }
            if (tid == 0) {
                lstart[seg] = nh;
                ldist[seg] = d;
            }
            int *nchp = &s_nch[seg & 1];
            // step 1: the slot's vertices, in groups that the warps draw; their
            // rows finish here unless they are long. In launches of few sources,
            // whose time is one block's chain of levels, each warp's first group
            // is fixed, so that on a thin level none draws: all warps on one
            // counter, most of them to find nothing left, took 3-6 % (64 sources,
            // 150 x 150 lattice 41.2 -> 39.2 ms, R-MAT 20,000 vertices 2.14 -> 2.06).
            // Elsewhere the registers that this takes cost more (R-MAT 16 hybrid
            // batch 58.6 -> 60.0 ms)
            {
                // one group per warp on a thin level, about two on others
                const unsigned warps = (unsigned)nwarps;
                const unsigned share = cnt <= 16 * warps ? (cnt + warps - 1) / warps : (cnt + 2 * warps - 1) / (2 * warps);
                const int gsize = (int)min(32u, share);
                const uint32_t *bks = bk + (size_t)slot * (size_t)bcap;
                auto draw = [&]() {
                    int k = 0;
                    if (lane == 0) k = atomicAdd(&s_group, gsize);
                    return __shfl_sync(kFull, k, 0);
                };
                const int fixed = (int)warps * gsize;  // vertices in the fixed groups
                auto after = [&]() { return (uint32_t)fixed >= cnt ? (int)cnt : fixed + draw(); };
                for (int g0 = kFew ? warp * gsize : 0;; g0 = kFew ? after() : 0) {
                    if (!kFew) g0 = draw();
                    if ((uint32_t)g0 >= cnt) break;
                    // all that a queued vertex needs, in one round of loads
                    int x = 0, seen = 0;
                    unsigned long long xd = PairT::kUnreached;
                    typename PairT::Count xs = 0;
                    long long rb = 0, re = 0;
                    uint64_t qm = 0ull;
                    if (lane < gsize && (uint32_t)(g0 + lane) < cnt) {
                        x = (int)bks[(b0 + (uint32_t)(g0 + lane)) & (uint32_t)(bcap - 1)];
                        P.get(x, xd, xs);
                        const longlong2 row = __ldg(q.row + x);
                        rb = row.x;
                        re = row.y;
                        seen = *(volatile const int32_t *)(p.tag + x);
                        qm = __ldg(p.qmask + __ldg(q.inv + x));
                    }
                    const bool ok = xd == d;
                    const unsigned am = __ballot_sync(kFull, ok);
                    if (am == 0u) continue;
                    int eb = 0;
                    if (lane == 0) eb = atomicAdd(&s_nh, __popc(am));
                    eb = __shfl_sync(kFull, eb, 0);
                    int len = 0;
                    if (ok) {
                        const long long deg = re - rb;
                        hv[eb + __popc(am & ((1u << lane) - 1u))] = x;
                        if (kBits && x < q.heads) atomicOr(&s_done[x >> 5], 1u << (x & 31));
                        st.reached += 1;
                        st.edges += (unsigned long long)deg;
                        if (PairT::two53(xs)) s_flag = 1;
                        if (seen == -1 && atomicCAS(&p.tag[x], -1, 0) == -1) {
                            st.vb += 1;
                            st.eb += (unsigned long long)deg;
                        }
                        if (deg <= pack_max) {
                            len = (int)deg;
                            st.arcs += (unsigned long long)deg;
                        } else {
                            const int nout = (int)((deg + CH - 1) / CH);
                            const int c0 = atomicAdd(nchp, nout);
                            if ((int64_t)c0 + nout > q.chcap) {
                                s_err = 1;
                                set_err(p.ctr, kDevChunkOverflow);
                            } else {
                                // the chunks carry the path count in place of entry and index
                                for (int k = 0; k < nout; ++k) {
                                    const long long a0 = rb + (long long)k * CH;
                                    store_chunk(&chs[c0 + k], x, (int)(unsigned)to_bits(xs), (int)(to_bits(xs) >> 32), nout, a0,
                                                (int)(min(rb + deg, a0 + CH) - a0));
                                }
                            }
                        }
                    }
                    // the group's arcs, packed onto the lanes
                    int incl = len;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int z = __shfl_up_sync(kFull, incl, o);
                        if (lane >= o) incl += z;
                    }
                    wa.incl[lane] = incl;
                    wa.off[lane] = rb - (incl - len);
                    wa.sg[lane] = to_bits(xs);
                    const int total = __shfl_sync(kFull, incl, 31);
                    __syncwarp();
                    const int er = src_offers<PairT, kBits>(p, P, bk, s_cnt, s_done, tb, bcap, R, d, wa, total, q.col, st.tight);
                    if (er) {
                        s_err = 1;
                        set_err(p.ctr, er);
                    }
                    // the query vertices among them (their mask has arrived by now)
                    if (ok) {
                        uint64_t y = qm & need;
                        while (y) {
                            const int qq = __ffsll((long long)y) - 1;
                            y &= y - 1;
                            s_ql[qq] = seg;
                        }
                    }
                    __syncwarp();
                }
            }
            __syncthreads();
            if (tid == 0) {
                s_base[slot] = b0 + cnt;
                s_nch[(seg + 1) & 1] = 0;
                if ((double)(global_ns() - s_t0) > p.timeout_ns) {
                    s_err = 1;
                    set_err(p.ctr, kDevTimeout);
                }
            }
            const int nch = *nchp;
            if (s_err) return;
            // step 2: long out-rows, lanes over arcs
            if (nch > 0) {
                for (int c = warp; c < nch; c += nwarps) {
                    const Chunk ch = load_chunk(&chs[c]);
                    wa.incl[lane] = ch.na;
                    if (lane == 0) {
                        wa.off[0] = ch.a0;
                        wa.sg[0] = ((unsigned long long)(unsigned)ch.k << 32) | (unsigned)ch.e;
                    }
                    __syncwarp();
                    const int er = src_offers<PairT, kBits>(p, P, bk, s_cnt, s_done, tb, bcap, R, d, wa, ch.na, q.col, st.tight);
                    if (er) {
                        s_err = 1;
                        set_err(p.ctr, er);
                    }
                    __syncwarp();
                    if (lane < ch.na) st.arcs += (unsigned long long)((ch.na - lane + 31) / 32);
                }
                __syncthreads();
                if (s_err) return;
            }
            nh = s_nh;
            ++seg;
        }
        const int nseg = seg;
        if ((unsigned long long)(nseg > 0 ? nseg - 1 : 0) > lev_max) lev_max = (unsigned long long)(nseg > 0 ? nseg - 1 : 0);
        if (tid == 0) {
            const unsigned long long t = global_ns();
            ns_fwd += t - t_mark;
            t_mark = t;
            // the last forward level may have left chunks counted in its slot
            s_nch[0] = 0;
            s_nch[1] = 0;
        }
        __syncthreads();

        if (p.mode == kModeScan && p.ncols < 2) {
            // ---------------- vertex scan, one query vertex r ----------------
            // delta_s.(r) = sigma_sr * sum over settled t with d(r, t) >= 1 and
            // d(s, r) + d(r, t) = d(s, t) of sigma_rt / sigma_st
            const int r = q.pos[p.vroot];
            unsigned long long dsr;
            typename PairT::Count ssr;
            P.get(r, dsr, ssr);
            double acc = 0.0;
            if (dsr != PairT::kUnreached && need) {
                for (int e = tid; e < nh; e += bd) {
                    const int t = hv[e], tv = __ldg(q.inv + t);
                    const unsigned long long rd = p.rdist[tv];
                    unsigned long long dt;
                    typename PairT::Count sst;
                    P.get(t, dt, sst);
                    if (rd == 0ull || rd >= dt || dsr + rd != dt) continue;
                    acc += p.rsig[tv] / (double)sst;
                    st.pairs += 1;
                }
            }
            acc = sum_warp(acc);
            if (lane == 0) s_red[warp] = acc;
            __syncthreads();
            if (tid == 0) {
                double sum = 0.0;
                for (int w = 0; w < nwarps; ++w) sum += s_red[w];
                const double dv = dsr != PairT::kUnreached ? (double)ssr * sum : 0.0;
                uint64_t y = need;
                while (y) {
                    const int qq = __ffsll((long long)y) - 1;
                    y &= y - 1;
                    s_dep[qq] = dv;
                }
            }
        } else if (p.mode == kModeScan) {
            // ---------------- vertex scan, several query vertices ----------------
            // column c (query vertex croot[c]) of the queries that need s
            uint64_t cols = 0ull;
            {
                uint64_t y = need;
                while (y) {
                    const int qq = __ffsll((long long)y) - 1;
                    y &= y - 1;
                    cols |= 1ull << p.qcol[qq];
                }
            }
            for (int c = tid; c < 64; c += bd) s_cd[c] = ((cols >> c) & 1ull) ? P.dist(q.pos[p.croot[c]]) : PairT::kUnreached;
            __syncthreads();
            const int stride = wcols_stride(p.ncols);
            for (int e = tid; e < nh; e += bd) {
                const int t = hv[e];
                const size_t trow = (size_t)__ldg(q.inv + t) * stride;
                unsigned long long dt;
                typename PairT::Count sst;
                P.get(t, dt, sst);
                // four columns (a sector of the row) per round of loads
                for (int c0 = 0; c0 < stride; c0 += 4) {
                    if (((cols >> c0) & 15ull) == 0ull) continue;
                    const ulonglong2 ra = *reinterpret_cast<const ulonglong2 *>(p.rdistq + trow + c0);
                    const ulonglong2 rb2 = *reinterpret_cast<const ulonglong2 *>(p.rdistq + trow + c0 + 2);
                    const unsigned long long rd[4] = {ra.x, ra.y, rb2.x, rb2.y};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const unsigned long long dc = s_cd[c0 + k];  // unreached where the source needs no c
                        if (dc == PairT::kUnreached || rd[k] == 0ull || rd[k] >= dt || dc + rd[k] != dt) continue;
                        atomicAdd(&s_msum[c0 + k], p.rsigq[trow + c0 + k] / (double)sst);
                        st.pairs += 1;
                    }
                }
            }
            __syncthreads();
            if (tid == 0) {
                uint64_t y = need;
                while (y) {
                    const int qq = __ffsll((long long)y) - 1;
                    y &= y - 1;
                    const int c = p.qcol[qq];
                    unsigned long long dcr;
                    typename PairT::Count scr;
                    P.get(q.pos[p.croot[c]], dcr, scr);
                    s_dep[qq] = s_cd[c] != PairT::kUnreached ? (double)scr * s_msum[c] : 0.0;
                }
            }
        } else if constexpr (PairT::kWide) {
            // ---------------- backward (Eq. 4) over the levels ----------------
            int lstop = 0x7fffffff;
            {
                uint64_t y = need;
                while (y) {
                    const int qq = __ffsll((long long)y) - 1;
                    y &= y - 1;
                    if (s_ql[qq] >= 0 && s_ql[qq] < lstop) lstop = s_ql[qq];
                }
            }
            for (int sg = nseg - 1; sg >= lstop; --sg) {
                const int e0 = lstart[sg];
                const int e1 = sg + 1 < nseg ? lstart[sg + 1] : nh;
                const unsigned long long dk = ldist[sg];
                int *nchp = &s_nch[sg & 1];
                const long long ne = e1 - e0;
                const int lpp = lanes_per_vertex(ne, bd);
                const int per = 32 / lpp, sub = lane / lpp, rl = lane % lpp;
                const bool lead = rl == 0;
                const long long ngroups = (ne + per - 1) / per;
                for (long long gi = warp; gi < ngroups; gi += nwarps) {
                    const long long ii = gi * per + sub;
                    const bool ok = ii < ne;
                    int v = 0;
                    long long rb = 0, re = 0;
                    if (ok) {
                        v = hv[e0 + ii];
                        const longlong2 row = __ldg(q.row + v);
                        rb = row.x;
                        re = row.y;
                    }
                    const bool shortrow = ok && re - rb <= pack_max;
                    double acc = 0.0;
                    if (shortrow) acc = src_pull_c(p, q.col, ds, tb, dk, rb, re, rl, lpp);
                    acc = sum_lanes(acc, lpp);
                    if (shortrow && lead) {
                        src_finalize(p, q.inv, ds, need, s_dep, v, acc);
                        st.arcs += (unsigned long long)(re - rb);
                    } else if (ok && !shortrow && lead) {
                        const int nout = (int)((re - rb + CHB - 1) / CHB);
                        const int c0 = atomicAdd(nchp, nout);
                        if ((int64_t)c0 + nout > q.chcap) {
                            s_err = 1;
                            set_err(p.ctr, kDevChunkOverflow);
                        } else {
                            src_store_chunks(chs, c0, v, (int)(e0 + ii), 0, rb, re, nout, CHB);
                        }
                    }
                }
                __syncthreads();
                if (tid == 0) {
                    s_nch[(sg + 1) & 1] = 0;
                    if ((double)(global_ns() - s_t0) > p.timeout_ns) {
                        s_err = 1;
                        set_err(p.ctr, kDevTimeout);
                    }
                }
                const int nch = *nchp;
                if (s_err) return;
                if (nch > 0) {
                    for (int c = warp; c < nch; c += nwarps) {
                        const Chunk ch = load_chunk(&chs[c]);
                        const double v = sum_warp(src_pull_c(p, q.col, ds, tb, dk, ch.a0, ch.a0 + ch.na, lane, 32));
                        if (lane == 0) part[c] = v;
                        if (lane < ch.na) st.arcs += (unsigned long long)((ch.na - lane + 31) / 32);
                    }
                    __syncthreads();
                    for (int c = tid; c < nch; c += bd) {
                        const Chunk ch = load_chunk(&chs[c]);
                        if (ch.k == 0) {
                            double acc = 0.0;
                            for (int k = 0; k < ch.nch; ++k) acc += part[c + k];
                            src_finalize(p, q.inv, ds, need, s_dep, ch.v, acc);
                        }
                    }
                    __syncthreads();
                }
            }
        }
        __syncthreads();
        // ---------------- outputs and reset ----------------
        if (tid < 64 && ((need >> tid) & 1ull)) q.sdep[(size_t)si * 64 + tid] = s_dep[tid];
        if (tid == 0) q.sflag[si] = (uint32_t)s_flag;
        for (int e = tid; e < nh; e += bd) {
            const int x = hv[e];
            P.clear(x);
            if (tb) {
                const longlong2 row = __ldg(q.row + x);
                const long long rb = row.x, re = row.y;
                if (re > rb)
                    for (long long w = rb >> 5; w <= (re - 1) >> 5; ++w) tb[w] = 0u;
            }
        }
        if (tid == 0) {
            const unsigned long long t = global_ns();
            ns_bwd += t - t_mark;
            t_mark = t;
        }
    }

    // counters: warp sums, one atomic per warp and counter
    unsigned long long v[7] = {st.edges, st.reached, st.tight, st.arcs, st.vb, st.eb, st.pairs};
#pragma unroll
    for (int i = 0; i < 7; ++i)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_down_sync(kFull, v[i], o);
    if (lane == 0) {
        unsigned long long *dst[7] = {&p.ctr->edges, &p.ctr->reached, &p.ctr->tight, &p.ctr->arc_visits,
                                      &p.ctr->vb, &p.ctr->eb, &p.ctr->vpairs};
#pragma unroll
        for (int i = 0; i < 7; ++i)
            if (v[i]) atomicAdd(dst[i], v[i]);
    }
    if (tid == 0) {
        atomicMax(&p.ctr->levels_max, lev_max);
        atomicAdd(&p.ctr->ns_fwd, ns_fwd);
        atomicAdd(&p.ctr->ns_bwd, ns_bwd);
        atomicAdd(&p.ctr->ns_other, ns_other);
    }
}

// Per-tile, per-query sums of the launch's sources (the tile kernel's order:
// eight interleaved partial sums per query, then a fixed shuffle tree), one
// block per tile.
__global__ void wsrc_tile_sums(TravParams p, const double *sdep, const uint32_t *sflag, int S) {
    const long long tile = blockIdx.x;
    const int32_t *tsrc = p.srcs + tile * S;
    for (int t = threadIdx.x; t < 64 * 8; t += blockDim.x) {
        const int qq = t >> 3, j = t & 7;
        const bool exact = (p.exact_q >> qq) & 1ull;
        double sum = 0.0;
        int flagged = 0;
        for (int s = j; s < S; s += 8) {
            const int v = tsrc[s];
            if (v < 0) continue;
            double mlt = 0.0;
            if (exact)
                mlt = ((p.need[v] >> qq) & 1ull) ? 1.0 : 0.0;
            else if (p.mult)
                mlt = (double)p.mult[((size_t)tile * S + s) * 64 + qq];
            if (mlt != 0.0) {
                const size_t i = (size_t)tile * S + s;
                sum += mlt * sdep[i * 64 + qq];
                if (sflag[i]) flagged = 1;
            }
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            sum += __shfl_down_sync(kFull, sum, o, 8);
            flagged |= __shfl_down_sync(kFull, flagged, o, 8);
        }
        if (j == 0) {
            p.tile_partial[tile * 64 + qq] = sum;
            if (flagged) atomicOr(&p.qflags[qq], 1u);
        }
    }
}

// Threads per block. A distance level is a chain of about five dependent loads
// and two or three block barriers whatever it holds, so small blocks, with more
// sources in flight per SM, win while the state of all of them (8 or 16 bytes
// per vertex and source) stays near L2; with larger graphs it is pushed out to
// DRAM and fewer, wider blocks win. Weights 1..255 (2,000 draws or all sources),
// 1024 / 512 / 256 / 128 threads: n = 5,000 8.9 / 5.0 / 3.8 / 4.3 ms, 32,768
// 26.5 / 17.9 / 14.7 / 20.3, 65,536 82.7 / 63.7 / 57.0 / 75.2, 131,072 31.5 /
// 27.9 / 32.0 / 52.0, 262,144 55.2 / 52.5 / 68.5 / 136, 524,288 104 / 110 / 260
// / 334, R-MAT 20 280 / 411 / 735 / 1402.
int src_threads(int64_t n) { return n <= 96 * 1024 ? 256 : n <= 384 * 1024 ? 512 : kSrcThreads; }

// Bytes of per-block state for a graph of n vertices.
size_t src_block_bytes(int64_t n, int64_t m, int R, int64_t bcap, int64_t maxlev, int64_t chcap) {
    return (size_t)n * (16 + 4) + (size_t)((m + 31) / 32) * 4 + (size_t)R * (size_t)bcap * 4 + (size_t)maxlev * 12 +
           (size_t)chcap * (32 + 8);
}

// Every vertex unreached: 16-byte pairs (distance all ones, sigma zero) or
// 8-byte words (distance field all ones, count zero).
__global__ void clear_pairs(unsigned long long *ds, size_t nvert, int layout) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nvert; i += (size_t)gridDim.x * blockDim.x) {
        if (layout == 1) {
            ds[2 * i] = ~0ull;
            ds[2 * i + 1] = 0ull;  // +0.0
        } else {
            ds[i] = NarrowPairs::kUnreached;
        }
    }
}

// Clears the per-block vertex state in the given layout (1 wide, 2 narrow).
bc_status clear_src_pairs(bc_graph *g, int layout) {
    bcd_workspace &ws = g->ws;
    const size_t nvert = (size_t)ws.sblocks * (size_t)g->n;
    clear_pairs<<<(unsigned)std::max(1, g->num_sms * 8), 256, 0, g->stream>>>(ws.sds, nvert, layout);
    g->launches += 1;
    BCD_CUDA(cudaGetLastError());
    ws.slayout = layout;
    return BC_OK;
}

void free_src_order(bcd_workspace &ws) {
    dev_free(ws.spos);
    dev_free(ws.sinv);
    dev_free(ws.srow);
    dev_free(ws.scol);
}

// Position classes: 0 for in-degrees of 2^31 and more, ... 31 for 1, 32 for 0.
__device__ __forceinline__ int degree_class(const int64_t *roff, int v) {
    const long long d = roff[v + 1] - roff[v];
    return d == 0 ? 32 : d >= (1ll << 31) ? 0 : 1 + __clz((int)d) - 1;
}

__global__ void class_counts(const int64_t *roff, int32_t n, unsigned *cnt) {
    __shared__ unsigned s_cnt[33];
    if (threadIdx.x < 33) s_cnt[threadIdx.x] = 0u;
    __syncthreads();
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
        atomicAdd(&s_cnt[degree_class(roff, v)], 1u);
    __syncthreads();
    if (threadIdx.x < 33 && s_cnt[threadIdx.x]) atomicAdd(&cnt[threadIdx.x], s_cnt[threadIdx.x]);
}

// One block: the classes' first positions.
__global__ void class_starts(unsigned *cnt) {
    if (threadIdx.x == 0) {
        unsigned run = 0;
        for (int c = 0; c < 33; ++c) {
            const unsigned k = cnt[c];
            cnt[c] = run;
            run += k;
        }
    }
}

// Positions, a block's vertices of a class side by side.
__global__ void assign_positions(const int64_t *off, const int64_t *roff, int32_t n, unsigned *next, int32_t *pos,
                                 int32_t *inv, longlong2 *row) {
    __shared__ unsigned s_cnt[33], s_at[33];
    for (int v0 = blockIdx.x * blockDim.x; v0 < n; v0 += gridDim.x * blockDim.x) {
        const int v = v0 + threadIdx.x;
        if (threadIdx.x < 33) s_cnt[threadIdx.x] = 0u;
        __syncthreads();
        int c = 0;
        unsigned rank = 0;
        if (v < n) {
            c = degree_class(roff, v);
            rank = atomicAdd(&s_cnt[c], 1u);
        }
        __syncthreads();
        if (threadIdx.x < 33 && s_cnt[threadIdx.x]) s_at[threadIdx.x] = atomicAdd(&next[threadIdx.x], s_cnt[threadIdx.x]);
        __syncthreads();
        if (v < n) {
            const int x = (int)(s_at[c] + rank);
            pos[v] = x;
            inv[x] = v;
            row[x] = make_longlong2(off[v], off[v + 1]);
        }
        __syncthreads();
    }
}

__global__ void heads_to_positions(const int32_t *col, int64_t m, const int32_t *pos, int32_t *out) {
    for (int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; a < m; a += (int64_t)gridDim.x * blockDim.x)
        out[a] = pos[col[a]];
}

// The vertices' positions and the arrays that go with them, once per graph
// (R-MAT 20: about half a millisecond).
bc_status src_order(bc_graph *g) {
    bcd_workspace &ws = g->ws;
    if (ws.spos) return BC_OK;
    const size_t n = (size_t)g->n;
    unsigned *cnt = nullptr;
    bc_status st;
    if ((st = dev_alloc(&ws.sinv, n)) || (st = dev_alloc(&ws.srow, 2 * n)) ||
        (st = dev_alloc(&ws.scol, (size_t)g->m)) || (st = dev_alloc(&cnt, 33)) || (st = dev_alloc(&ws.spos, n))) {
        dev_free(cnt);
        free_src_order(ws);
        return st;
    }
    const unsigned blocks = (unsigned)std::max(1, g->num_sms * 4);
    cudaMemsetAsync(cnt, 0, 33 * sizeof(unsigned), g->stream);
    class_counts<<<blocks, 256, 0, g->stream>>>(g->d_roff, g->n, cnt);
    class_starts<<<1, 32, 0, g->stream>>>(cnt);
    assign_positions<<<blocks, 256, 0, g->stream>>>(g->d_off, g->d_roff, g->n, cnt, ws.spos, ws.sinv,
                                                    reinterpret_cast<longlong2 *>(ws.srow));
    if (g->m) heads_to_positions<<<blocks, 256, 0, g->stream>>>(g->d_col, g->m, ws.spos, ws.scol);
    g->launches += 4;
    cudaError_t e = cudaGetLastError();
    // where the class before the last ended: the last one has no in-arcs
    unsigned at[33] = {0};
    if (e == cudaSuccess) e = cudaMemcpyAsync(at, cnt, sizeof(at), cudaMemcpyDeviceToHost, g->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
    ws.sheads = (int32_t)at[31];
    dev_free(cnt);
    if (e != cudaSuccess) {
        free_src_order(ws);
        return cuda_error(e, "source kernel order");
    }
    return BC_OK;
}

void free_src_arrays(bcd_workspace &ws) {
    dev_free(ws.sds);
    dev_free(ws.stb);
    dev_free(ws.shv);
    dev_free(ws.slstart);
    dev_free(ws.sldist);
    dev_free(ws.sbk);
    dev_free(ws.sch);
    dev_free(ws.spart);
    ws.sblocks = 0;
}

// (Re)allocates the per-block state for the current capacities; every pair
// starts unreached.
bc_status alloc_src_arrays(bc_graph *g, int blocks) {
    bcd_workspace &ws = g->ws;
    free_src_arrays(ws);
    const size_t B = (size_t)blocks;
    const size_t n = (size_t)g->n;
    BCD_TRY(dev_alloc(&ws.sds, 2 * B * n));
    BCD_TRY(dev_alloc(&ws.stb, B * (size_t)((g->m + 31) / 32)));
    BCD_CUDA(cudaMemsetAsync(ws.stb, 0, sizeof(uint32_t) * B * (size_t)((g->m + 31) / 32), g->stream));
    BCD_TRY(dev_alloc(&ws.shv, B * n));
    BCD_TRY(dev_alloc(&ws.slstart, B * (size_t)ws.smaxlev));
    BCD_TRY(dev_alloc(&ws.sldist, B * (size_t)ws.smaxlev));
    BCD_TRY(dev_alloc(&ws.sbk, B * (size_t)ws.ring * (size_t)ws.sbcap));
    BCD_TRY(dev_alloc(&ws.sch, B * (size_t)ws.schcap));
    BCD_TRY(dev_alloc(&ws.spart, B * (size_t)ws.schcap));
    ws.sblocks = blocks;
    return clear_src_pairs(g, 1);
}

bc_status reset_src_state(bc_graph *g) {
    bcd_workspace &ws = g->ws;
    if (!ws.sds) return BC_OK;
    BCD_TRY(clear_src_pairs(g, ws.slayout ? ws.slayout : 1));
    BCD_CUDA(cudaMemsetAsync(ws.stb, 0, sizeof(uint32_t) * (size_t)ws.sblocks * (size_t)((g->m + 31) / 32), g->stream));
    if (ws.tag) BCD_CUDA(cudaMemsetAsync(ws.tag, 0xff, sizeof(int32_t) * (size_t)g->n, g->stream));
    return BC_OK;
}

template <typename T>
bc_status grow_buf(T **p, int64_t *cap, int64_t need) {
    if (*cap >= need && *p) return BC_OK;
    dev_free(*p);
    *cap = 0;
    const int64_t c = std::max<int64_t>(need, 1024);
    BCD_TRY(dev_alloc(p, (size_t)c));
    *cap = c;
    return BC_OK;
}

}  // namespace

void free_src_state(bc_graph *g) {
    bcd_workspace &ws = g->ws;
    free_src_arrays(ws);
    free_src_order(ws);
    dev_free(ws.sdep);
    dev_free(ws.sflag);
    dev_free(ws.snext);
    ws.sdep_cap = 0;
    ws.sflag_cap = 0;
    ws.sbcap = 0;
    ws.schcap = 0;
    ws.smaxlev = 0;
    ws.slayout = 0;
    ws.swide = false;
}

bool src_kernel_applies(const bc_graph *g, const TravParams &p) {
    return g->weighted && g->weighted_kernel == 2 && (p.mode == kModeSpd || p.mode == kModeScan) &&
           !(p.flags & (kFlagNoBackward | kFlagNoReset | kFlagFullBackward | kFlagRootOut));
}

bc_status run_src_traversal(bc_graph *g, int W, TravParams &p, int *levels_out, unsigned long long *edges_out) {
    bcd_workspace &ws = g->ws;
    BCD_TRY(ensure_weighted_state(g));  // ring size, tag array
    BCD_TRY(src_order(g));
    const int S = 64 * W;
    const int64_t nsrc = p.ntiles * S;
    // blocks by the size of the graph (state is held for that many); a launch of
    // fewer sources than that takes wider ones, on small graphs, whose levels
    // seldom fill more, of 512 threads at most. Empty slots of the last tile do not
    // count: 64 sources and weights 1..255, 512 / 1024 threads: a 150 x 150 lattice
    // 39.2 / 41.6 ms, R-MAT graphs of 20,000 vertices 2.06 / 2.04, 65,536 3.47 /
    // 2.94, 131,072 5.58 / 4.29
    const int64_t real = p.nsrc > 0 ? p.nsrc : nsrc;
    const int widest = g->n <= 32 * 1024 ? 512 : kSrcThreads;
    const int base_threads = src_threads(g->n);
    int threads = base_threads;
    while (threads < widest && (int64_t)g->num_sms * (kSrcThreads / (2 * threads)) >= real) threads *= 2;
    const int R = ws.ring;
    // the settled bits join the staging and counters in shared memory while they fit
    const size_t ring = sizeof(WarpArcs) * (size_t)(threads / 32) + sizeof(uint32_t) * 2 * (size_t)R;
    const size_t done = sizeof(uint32_t) * (((size_t)ws.sheads + 31) / 32);
    const bool bits = ring + done <= kSrcDynSmem;
    const size_t smem = ring + (bits ? done : 0);
    const bool few = real <= (int64_t)g->num_sms * (kSrcThreads / threads);
    auto kernel = [&](auto pairs) {
        using P = decltype(pairs);
        if (few) return bits ? (const void *)wsrc_kernel<P, true, true> : (const void *)wsrc_kernel<P, false, true>;
        return bits ? (const void *)wsrc_kernel<P, true, false> : (const void *)wsrc_kernel<P, false, false>;
    };
    const void *wide = kernel(WidePairs{}), *narrow = kernel(NarrowPairs{});
    int per_sm = 0, per_sm_n = 0;
    BCD_CUDA(cudaFuncSetAttribute(wide, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    BCD_CUDA(cudaFuncSetAttribute(narrow, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    BCD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, wide, threads, smem));
    BCD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_n, narrow, threads, smem));
    per_sm = std::min(per_sm, per_sm_n);
    if (per_sm < 1) return set_error(BC_E_INTERNAL, "weighted source kernel cannot be resident");
    if (ws.sbcap == 0) {
        // queued vertices of one distance of one source: a few times the
        // average vertices per distance value, and at least 2^21 entries
        // over the whole ring (8 MB), or 16 per vertex; grown on overflow
        const int64_t whole = std::min<int64_t>((int64_t)1 << 21, 16 * (int64_t)g->n);
        int64_t b = 64;
        while ((b < 4 * (int64_t)g->n / R || b * R < whole) && b < ((int64_t)1 << 30)) b *= 2;
        ws.sbcap = b;
        ws.schcap = 16384;
        ws.smaxlev = 8192;
    }
    int blocks = g->num_sms * per_sm * (threads / base_threads);
    {
        size_t fr = 0, tot = 0;
        BCD_CUDA(cudaMemGetInfo(&fr, &tot));
        const size_t have = ws.sblocks > 0 ? src_block_bytes(g->n, g->m, R, ws.sbcap, ws.smaxlev, ws.schcap) * ws.sblocks : 0;
        const size_t per = src_block_bytes(g->n, g->m, R, ws.sbcap, ws.smaxlev, ws.schcap);
        const size_t budget = (fr + have) / 2;
        blocks = (int)std::min<size_t>((size_t)blocks, budget / per);
        if (blocks < 1) return set_error(BC_E_OOM, "weighted source kernel: no room for one block's state");
    }
    if (ws.sblocks < blocks || !ws.sds) {
        const bc_status st = alloc_src_arrays(g, blocks);
        if (st != BC_OK) {
            free_src_arrays(ws);
            return st;
        }
    }
    BCD_TRY(grow_buf(&ws.sdep, &ws.sdep_cap, nsrc * 64));
    BCD_TRY(grow_buf(&ws.sflag, &ws.sflag_cap, nsrc));
    if (!ws.snext) BCD_TRY(dev_alloc(&ws.snext, 1));
    for (;;) {  // each rerun enlarges what was full, up to its limit, or takes the one step to wide pairs
        p.off = g->d_off;
        p.col = g->d_col;
        p.wt = g->d_w;
        p.roff = g->d_roff;
        p.rcol = g->d_rcol;
        p.rwt = g->d_rw;
        p.tag = ws.tag;
        p.ctr = ws.ctr;
        p.n = g->n;
        p.chunk_arcs = g->chunk_arcs;
        p.wshort = g->wshort;
        p.timeout_ns = g->timeout_ns;
        p.cancel = g->cancel_d;
        SrcParams q;
        q.ds = reinterpret_cast<DistSig *>(ws.sds);
        q.hv = ws.shv;
        q.lstart = ws.slstart;
        q.ldist = ws.sldist;
        q.bk = ws.sbk;
        q.ch = ws.sch;
        q.part = ws.spart;
        q.tb = ws.stb;
        q.tbw = (g->m + 31) / 32;
        q.sdep = ws.sdep;
        q.sflag = ws.sflag;
        q.next = ws.snext;
        q.col = ws.scol;
        q.row = reinterpret_cast<const longlong2 *>(ws.srow);
        q.pos = ws.spos;
        q.inv = ws.sinv;
        q.heads = ws.sheads;
        q.n = g->n;
        q.bcap = ws.sbcap;
        q.chcap = ws.schcap;
        q.nsrc = nsrc;
        q.ring = R;
        q.maxlev = ws.smaxlev;
        // 8-byte words for vertex-scan launches, unless one of this graph
        // has overflowed them; the Eq. 4 pass needs the 16-byte pairs
        const int layout = (p.mode == kModeScan && !ws.swide) ? 2 : 1;
        if (ws.slayout != layout) BCD_TRY(clear_src_pairs(g, layout));
        BCD_CUDA(cudaMemsetAsync(ws.ctr, 0, sizeof(Counters), g->stream));
        BCD_CUDA(cudaMemsetAsync(ws.snext, 0, sizeof(unsigned long long), g->stream));
        cudaEvent_t ev0 = nullptr, ev1 = nullptr;
        const bool timed = cudaEventCreate(&ev0) == cudaSuccess && cudaEventCreate(&ev1) == cudaSuccess;
        if (timed) cudaEventRecord(ev0, g->stream);
        void *args[] = {(void *)&p, (void *)&q};
        const cudaError_t le = cudaLaunchKernel(layout == 2 ? narrow : wide, dim3((unsigned)std::min(ws.sblocks, g->num_sms * per_sm)),
                                                dim3((unsigned)threads), args, smem, g->stream);
        g->launches += 1;
        g->last_grid = std::min(ws.sblocks, g->num_sms * per_sm);
        if (le != cudaSuccess) {
            if (timed) {
                cudaEventDestroy(ev0);
                cudaEventDestroy(ev1);
            }
            return cuda_error(le, "wsrc_kernel launch");
        }
        if (timed) cudaEventRecord(ev1, g->stream);
        Counters c;
        BCD_CUDA(cudaMemcpyAsync(&c, ws.ctr, sizeof(Counters), cudaMemcpyDeviceToHost, g->stream));
        BCD_CUDA(cudaStreamSynchronize(g->stream));
        float ms = 0.f;
        if (timed) {
            cudaEventElapsedTime(&ms, ev0, ev1);
            cudaEventDestroy(ev0);
            cudaEventDestroy(ev1);
        }
        // the tag array marks the launch's union of reached vertices; clear it
        BCD_CUDA(cudaMemsetAsync(ws.tag, 0xff, sizeof(int32_t) * (size_t)g->n, g->stream));
        if (c.err == kDevOk) {
            if (p.ntiles > 0) {
                wsrc_tile_sums<<<(unsigned)p.ntiles, 512, 0, g->stream>>>(p, ws.sdep, ws.sflag, S);
                g->launches += 1;
                BCD_CUDA(cudaGetLastError());
            }
            g->last = c;
            g->last_ms_launch = ms;
            // phase times: the blocks' summed phase times, scaled to the launch
            const double tot = (double)c.ns_fwd + (double)c.ns_bwd + (double)c.ns_other;
            const double launch_ns = (double)ms * 1e6;
            g->last_ns_fwd = tot > 0 ? (unsigned long long)(launch_ns * (double)c.ns_fwd / tot) : 0ull;
            g->last_ns_bwd = tot > 0 ? (unsigned long long)(launch_ns * (double)c.ns_bwd / tot) : 0ull;
            g->last_ns_other = tot > 0 ? (unsigned long long)(launch_ns * (double)c.ns_other / tot) : 0ull;
            if (levels_out) *levels_out = (int)c.levels_max;
            if (edges_out) *edges_out = c.edges;
            return BC_OK;
        }
        BCD_TRY(reset_src_state(g));
        if (p.qflags) BCD_CUDA(cudaMemsetAsync(p.qflags, 0, sizeof(uint32_t) * 64, g->stream));
        if (c.err == kDevTimeout) return set_error(BC_E_TIMEOUT, "weighted source kernel: a source ran past the time limit");
        if (c.err == kDevCancelled) return set_error(BC_E_CANCELLED, "traversal: cancelled by bc_cancel");
        if (c.err == kDevWide) {
            // a count of 2^40 or a distance of 2^24 - 1: 16-byte pairs from now on
            if (layout == 1) return set_error(BC_E_INTERNAL, "weighted source kernel: wide pairs asked for a wider form");
            ws.swide = true;
            continue;
        }
        const size_t before = (size_t)ws.sblocks * src_block_bytes(g->n, g->m, R, ws.sbcap, ws.smaxlev, ws.schcap);
        if (c.err == kDevBucketOverflow) {
            if (ws.sbcap >= ((int64_t)1 << 30)) return set_error(BC_E_OOM, "bucket ring: too many queued vertices at one distance");
            ws.sbcap *= 2;
        } else if (c.err == kDevLevelOverflow) {
            if (ws.smaxlev >= (1 << 28)) return set_error(BC_E_OOM, "traversal: more distance levels than the arrays hold");
            ws.smaxlev *= 4;
        } else if (c.err == kDevChunkOverflow) {
            if (ws.schcap >= ((int64_t)1 << 30)) return set_error(BC_E_OOM, "traversal: too many long-row chunks in one level");
            ws.schcap *= 4;
        } else {
            return set_error(BC_E_INTERNAL, "weighted source kernel: unexpected device error");
        }
        // grow, within half of the memory free besides the current state
        size_t fr = 0, tot = 0;
        BCD_CUDA(cudaMemGetInfo(&fr, &tot));
        const size_t per = src_block_bytes(g->n, g->m, R, ws.sbcap, ws.smaxlev, ws.schcap);
        const int nb = (int)std::min<size_t>((size_t)ws.sblocks, ((fr + before) / 2) / per);
        if (nb < 1) {
            free_src_arrays(ws);
            return set_error(BC_E_OOM, "weighted source kernel: no room for one block's state");
        }
        const bc_status st = alloc_src_arrays(g, nb);
        if (st != BC_OK) {
            free_src_arrays(ws);
            return st;
        }
    }
}

}  // namespace bcd
