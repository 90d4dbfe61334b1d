// Persistent multi-source traversal: the single-source work of Algorithm 1
// (and Algorithm 2) for S = 64*W sources at once.
//
// One cooperative launch walks every tile of S sources. Its blocks form one or
// more teams, each with the state of one tile and a barrier of its own; a team
// takes the next tile when it has finished one, so that one tile's thin levels
// and barriers overlap another's work (bcd_query.cu, teams_for). Per tile:
//   forward  (Section 2): level-synchronous BFS over the forward CSR. Per
//            vertex the dense state holds the visited mask (levels up to the
//            current one) and two level-parity masks (bit s: vertex is at the
//            current / next level for source s). A level runs in two phases
//            with a grid barrier after each:
//              push    (push_masks) the frontier's out-arcs (u, v), in chunks
//                      of at most chunk_arcs arcs, mark the sources newly
//                      reaching v, F(u) & ~visited(v), in v's next-level mask;
//              gather  (gather_level) every vertex of the next level sums
//                      sigma_s(v) over its in-arcs (R(G)) from the
//                      in-neighbours on the current level, in registers, and
//                      writes its sigma row once.
//            Sigma are integers, exact in any order: held as 32-bit counts, or
//            as fp64 after a launch met a count of 2^26 (it reruns).
//   backward (Eq. 4): levels from the deepest one up to the shallowest level
//            any query vertex sits at. With c_s(w) = (1 + delta_s(w)) /
//            sigma_s(w), delta_s(v) = sigma_s(v) * sum over tight out-arcs
//            (v, w) of c_s(w). The sum is pushed: the entries of level L + 1
//            add c_s(w) along their tight in-arcs (R(G), in chunks) into an
//            accumulator slab acc[v][s] with fp64 atomic adds, which do not
//            hold the warp; after a barrier the level-L entries turn acc
//            into delta and c. The sum order follows the schedule, so delta
//            can differ from run to run in its last bits.
// Scan mode (every query of the launch at one vertex r) keeps the forward
//            pass and replaces the backward by one pass over the reached
//            (vertex, source) pairs: delta_s.(r) = sigma_sr * sum of
//            sigma_rt / sigma_st over the t behind r on a shortest s-t path,
//            with d(r, t) and sigma_rt from an earlier scan-mode launch whose
//            only source is r (kFlagRootOut).
// Reach mode (RV(r), Section 4.1) runs the forward pass only, over R(G),
// with one source slot per query root, and ORs every level mask into rvmask.
//
// Every grid barrier wait is bounded; a timeout or a capacity overflow sets
// Counters::err and all blocks leave.
#include <cooperative_groups.h>

#include <algorithm>

#include "bcd_common.cuh"
#include "bcd_device.cuh"

namespace bcd {

namespace {

using namespace dev;

// Per-thread work counters (flushed to the 64-bit launch totals at the end of
// every tile).
struct Stats {
    unsigned long long edges = 0;
    unsigned reached = 0, tight = 0, arcs = 0;
};

__device__ __forceinline__ void flush_stats(Counters *c, Stats &st, int lane) {
    unsigned long long v[4] = {st.edges, st.reached, st.tight, st.arcs};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_down_sync(kFull, v[i], o);
    if (lane == 0) {
        unsigned long long *dst[4] = {&c->edges, &c->reached, &c->tight, &c->arc_visits};
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (v[i]) atomicAdd(dst[i], v[i]);
    }
    st = Stats();
}

// Path counts: 32-bit integers are trusted below 2^26, so that a sum of 33
// terms cannot wrap before it is tested; fp64 sums need no such test.
constexpr uint32_t kCountLimit = 1u << 26;

template <typename T>
struct SigOver {
    static __device__ __forceinline__ unsigned test(T x) { return 0u; }
};
template <>
struct SigOver<uint32_t> {
    static __device__ __forceinline__ unsigned test(uint32_t x) { return x & ~(kCountLimit - 1u); }
};

// Source s met a count of 2^53 (fp64 counts only).
__device__ __forceinline__ void flag_two53(const TravParams &p, uint32_t, int) {}
__device__ __forceinline__ void flag_two53(const TravParams &p, double x, int s) {
    if (x >= 9007199254740992.0) atomicOr((unsigned long long *)&p.srcflag[s >> 6], 1ull << (s & 63));
}

// Where the next level's entries and chunks start in the history.
struct LevelEnds {
    long long es, cs, ics;
};

// Per-warp staging of the packed chunk groups of push_masks and gather_level.
constexpr int kGroup = 8;  // chunks a warp takes together
template <int W>
struct __align__(16) WarpBuf {
    uint64_t n[kGroup][W];   // source masks of the group's entries
    uint64_t t[32][W];       // gather: tight sources of the 32 arcs in hand
    long long aoff[kGroup];  // arc i of the group sits at aoff[chunk] + i
    int incl[kGroup];        // arcs of the group up to and with each chunk
    int v[kGroup];           // gather: the entries' vertices
    int nch[kGroup];         // gather: in-arc chunks of the vertex
    struct {                 // the phase's chunk hand-out (GroupGrabber)
        unsigned long long *ctr;
        long long cnt, first;
        int grab;
    } hand;
    long long first;         // first chunk of the level in hand
    LevelEnds ends;          // ... and where its successors go
    Stats st[32];            // work counters of the warp's lanes
    unsigned q[128];         // vertices claimed for the next level, not yet appended (kFirstSeen: new to the tile)

    // Stages lane i's chunk (na arcs from a0) and returns the group's arcs.
    __device__ __forceinline__ int pack(int lane, int na, long long a0) {
        int x = na;
#pragma unroll
        for (int o = 1; o < kGroup; o <<= 1) {
            const int y = __shfl_up_sync(kFull, x, o);
            if (lane >= o) x += y;
        }
        if (lane < kGroup) {
            incl[lane] = x;
            aoff[lane] = a0 - (x - na);
        }
        __syncwarp();
        return incl[kGroup - 1];
    }

    // The chunk that holds arc i of the group.
    __device__ __forceinline__ int find(int i) const {
        int j = 0;
#pragma unroll
        for (int o = kGroup / 2; o > 0; o >>= 1)
            if (incl[j + o - 1] <= i) j += o;
        return j;
    }
};

constexpr unsigned kFirstSeen = 0x80000000u;

// Dynamic shared memory: the launch's parameters, the queries each source
// slot of the tile serves (64 W words), then one WarpBuf per warp (or a
// ScanBuf). The functions that are not inlined take these from here, not as
// arguments: a reference argument would turn every access, also to the
// parameters, into a generic load.
extern __shared__ __align__(16) unsigned char s_dyn[];
constexpr int kParamBytes = ((int)sizeof(TravParams) + 15) / 16 * 16;
__device__ __forceinline__ const TravParams &shared_params() { return *reinterpret_cast<const TravParams *>(s_dyn); }
__device__ __forceinline__ uint64_t *tile_need() { return reinterpret_cast<uint64_t *>(s_dyn + kParamBytes); }
template <int W>
__device__ __forceinline__ WarpBuf<W> &warp_buf() {
    return reinterpret_cast<WarpBuf<W> *>(s_dyn + kParamBytes + 512 * W)[threadIdx.x >> 5];
}

// Appends the first `take` (at most 32) of a warp's claimed vertices to level
// L + 1, one per lane: one entry and its out-arc chunks each and, unless only
// reach is asked, the in-arc (R(G)) chunks that the gather (and the Eq. 4
// backward) walks, with one set of counter atomics per warp. The out-degree
// rides in the chunks. Claims are queued per warp and appended 32 at a time,
// so that the atomics' round trip is paid once per 32 vertices.
template <int W, int MODE>
__device__ __noinline__ void append_queue(int L, int qn, int take) {
    const TravParams &p = shared_params();
    WarpBuf<W> &buf = warp_buf<W>();
    const LevelEnds &ends = buf.ends;
    const int lane = threadIdx.x & 31;
    const int CH = p.chunk_arcs;
    const bool app = lane < take;
    int wv = 0, wnch = 0, winch = 0;
    long long wrb = 0, wirb = 0;
    int deg = 0, ideg = 0;
    unsigned vb = 0;
    __syncwarp();
    if (app) {
        const unsigned x = buf.q[lane];
        wv = (int)(x & ~kFirstSeen);
        vb = x >> 31;
        wrb = p.off[wv];
        deg = (int)(p.off[wv + 1] - wrb);
        wnch = max(1, (deg + CH - 1) / CH);
        if (MODE != kModeReach) {
            wirb = p.roff[wv];
            ideg = (int)(p.roff[wv + 1] - wirb);
            winch = (ideg + CH - 1) / CH;
        }
    }
    // the rest of the queue moves to its front
    unsigned rest[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) rest[k] = 32 * (k + 1) + lane < qn ? buf.q[32 * (k + 1) + lane] : 0u;
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 3; ++k) buf.q[32 * k + lane] = rest[k];
    int x = wnch, xi = winch;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, x, o);
        const int yi = __shfl_up_sync(kFull, xi, o);
        if (lane >= o) {
            x += y;
            xi += yi;
        }
    }
    // out-arcs of the appended vertices: the next level's frontier arcs, which
    // choose its direction; and of those, the ones new to the tile
    unsigned long long fa = (unsigned long long)deg, fb = vb ? (unsigned long long)deg : 0ull;
    if (MODE != kModeReach) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            fa += __shfl_xor_sync(kFull, fa, o);
            fb += __shfl_xor_sync(kFull, fb, o);
        }
        vb = __popc(__ballot_sync(kFull, vb != 0u));
    }
    const long long nl = (long long)p.maxlev + 2;
    unsigned long long old = 0, ib = 0;
    if (lane == 31) {
        // entries (low half) and out-arc chunks (high half) in one atomic: every
        // appending warp of the level meets on this word
        old = atomicAdd(&p.lev_grab[4 * nl + L + 1], (unsigned long long)take | ((unsigned long long)x << 32));
        if (MODE != kModeReach) {
            if (xi) ib = atomicAdd(&p.lev_grab[2 * nl + L + 1], (unsigned long long)xi);
            if (fa && p.pull_arcs_min > 0) atomicAdd(&p.lev_grab[3 * nl + L + 1], fa);
            if (vb) atomicAdd(&p.ctr->vb, (unsigned long long)vb);
            if (fb) atomicAdd(&p.ctr->eb, fb);
        }
    }
    old = __shfl_sync(kFull, old, 31);
    if (MODE != kModeReach) ib = __shfl_sync(kFull, ib, 31);
    if (app) {
        const long long e = ends.es + (long long)(old & 0xffffffffull) + lane;
        const long long c0 = ends.cs + (long long)(old >> 32) + (x - wnch);
        const long long i0 = ends.ics + (long long)ib + (xi - winch);
        if (e >= p.hcap) {
            set_err(p.ctr, kDevHistOverflow);
        } else if (c0 + wnch > p.ccap || (MODE != kModeReach && i0 + winch > p.ccap)) {
            set_err(p.ctr, kDevChunkOverflow);
        } else {
            p.hv[e] = wv;
            emit_chunks(p, c0, wv, (int)e, wnch, wrb, wrb + deg);
            if (MODE != kModeReach)
                for (int k = 0; k < winch; ++k)
                    store_chunk(&p.ichunks[i0 + k], wv, (int)e, k, winch, wirb + (long long)k * CH,
                                min(CH, ideg - k * CH), deg);
        }
    }
    __syncwarp();
}

// Queues the vertices that lanes with `app` claimed.
template <int W>
__device__ __forceinline__ void claim(WarpBuf<W> &buf, int &qn, bool app, unsigned x, int lane) {
    const unsigned am = __ballot_sync(kFull, app);
    if (app) buf.q[qn + __popc(am & ((1u << lane) - 1u))] = x;
    qn += __popc(am);
}

// Appends whole warps of the queue (all of it at the end of a level).
template <int W, int MODE>
__device__ __forceinline__ void drain(int L, int &qn, bool all) {
    while (qn >= 32 || (all && qn > 0)) {
        const int take = min(qn, 32);
        append_queue<W, MODE>(L, qn, take);
        qn -= take;
    }
}

// The W words of a mask (16-byte loads where the row allows them).
template <int W>
__device__ __forceinline__ void load_mask(const uint64_t *row, uint64_t (&m)[W]) {
    if (W == 1) {
        m[0] = row[0];
    } else {
#pragma unroll
        for (int w = 0; w < W; w += 2) {
            const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(row + w);
            m[w] = x.x;
            m[W > 1 ? w + 1 : 0] = x.y;
        }
    }
}

// Hand-out of a level's chunks in groups of up to kGroup consecutive ones
// (fewer when the level is thin, so that all warps get some). The first group
// of each warp is fixed and the rest are drawn from a counter: on a thin level
// no warp touches the counter, where all warps of the grid would queue up.
template <int W>
struct GroupGrabber {
    long long at;
    __device__ GroupGrabber(unsigned long long *c, long long n, long long gwarp, long long nwarps) {
        WarpBuf<W> &buf = warp_buf<W>();
        const long long g = max(1ll, min((long long)kGroup, n / (nwarps * 4)));
        at = gwarp * g;
        __syncwarp();
        buf.hand.ctr = c;
        buf.hand.cnt = n;
        buf.hand.first = nwarps * g;
        buf.hand.grab = (int)g;
        __syncwarp();
    }
    // The next group: its size (0: none left) and, in c0, its first chunk.
    __device__ __forceinline__ int next(long long &c0, int lane) {
        const auto &h = warp_buf<W>().hand;
        const long long cnt = h.cnt;
        if (at >= cnt) return 0;
        c0 = at;
        const int k = (int)min((long long)h.grab, cnt - at);
        at = cnt;
        if (h.first < cnt) {
            unsigned long long b = 0;
            if (lane == 0) b = atomicAdd(h.ctr, (unsigned long long)h.grab);
            at = h.first + (long long)__shfl_sync(kFull, b, 0);
        }
        return k;
    }
};

// The bookkeeping of an entry (v, F) that joins level L (one thread): its
// mask into the history and the visited set, the work counters, and the level
// of the query vertices that sit at v.
template <int W>
__device__ __forceinline__ void enter_entry(const TravParams &p, int L, long long e, int v, const uint64_t (&F)[W],
                                            const uint64_t (&vis)[W], int odeg, Stats &st) {
    const uint64_t *s_need = tile_need();
    uint64_t *row = p.vs + (size_t)v * p.vs_stride;
    int pc = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        p.hm[(size_t)e * W + w] = F[w];
        row[w] = vis[w] | F[w];
        pc += __popcll(F[w]);
    }
    st.edges += (unsigned long long)pc * (unsigned)odeg;
    st.reached += (unsigned)pc;
    const uint64_t qm = p.qmask[v];
    if (qm == 0ull) return;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        uint64_t b = F[w];
        while (b) {
            const int s = 64 * w + __ffsll((long long)b) - 1;
            b &= b - 1;
            uint64_t x = qm & s_need[s];
            while (x) {
                const int q = __ffsll((long long)x) - 1;
                x &= x - 1;
                p.qlevel[s * 64 + q] = L;
            }
        }
    }
}

// Level 0 of a tile: one entry per source slot (block 0 only). Thread t
// seeds slot t: the launch has at least S threads per block.
template <int W, int MODE, typename T>
__device__ void init_tile(const TravParams &p, const int32_t *tsrc) {
    constexpr int S = 64 * W;
    __shared__ int s_scan[S];
    __shared__ int s_valid;
    const int t = threadIdx.x;
    int v = -1, nch = 0;
    long long rb = 0, re = 0;
    if (t < S) {
        v = tsrc[t];
        if (v >= 0) {
            rb = p.off[v];
            re = p.off[v + 1];
            nch = (int)max(1ll, (re - rb + p.chunk_arcs - 1) / p.chunk_arcs);
        }
        s_scan[t] = nch;
    }
    if (t == 0) s_valid = 0;
    if (MODE != kModeReach) {
        for (int i = t; i < S * 64; i += blockDim.x) p.qlevel[i] = -1;
        if (t < W) p.srcflag[t] = 0ull;
    }
    if (MODE == kModeScan && t < S) p.vsum[t] = 0.0;
    if (MODE == kModeScan && p.ncols >= 2)
        for (int i = t; i < S * 64; i += blockDim.x) p.msum[i] = 0.0;
    __syncthreads();
    if (t < S && v >= 0) atomicAdd(&s_valid, 1);
    for (int o = 1; o < S; o <<= 1) {
        int y = 0;
        if (t < S && t >= o) y = s_scan[t - o];
        __syncthreads();
        if (t < S) s_scan[t] += y;
        __syncthreads();
    }
    if (t < S && v >= 0) {
        const int c0 = s_scan[t] - nch;
        if (c0 + nch > p.ccap || t >= p.hcap) {
            set_err(p.ctr, kDevChunkOverflow);
        } else {
            uint64_t *row = p.vs + (size_t)v * p.vs_stride;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const uint64_t b = (w == (t >> 6)) ? (1ull << (t & 63)) : 0ull;
                p.hm[(size_t)t * W + w] = b;
                row[W + w] = b;                       // level-0 parity mask
                if (MODE != kModeReach) row[w] = b;   // visited (the reach push sets it itself)
            }
            p.hv[t] = v;
            p.tag[v] = 0;
            emit_chunks(p, c0, v, t, nch, rb, re);
            if (MODE != kModeReach) {
                atomicAdd(&p.ctr->vb, 1ull);
                atomicAdd(&p.ctr->eb, (unsigned long long)(re - rb));
                atomicAdd(&p.ctr->edges, (unsigned long long)(re - rb));
                atomicAdd(&p.ctr->reached, 1ull);
                reinterpret_cast<T *>(p.sigma)[(size_t)v * S + t] = T(1);
                uint64_t x = p.qmask[v] & p.need[v];
                while (x) {
                    const int q = __ffsll((long long)x) - 1;
                    x &= x - 1;
                    p.qlevel[t * 64 + q] = 0;
                }
            }
        }
    }
    __syncthreads();
    if (t == 0) {
        p.lev_cnt[0] = (unsigned long long)s_valid;
        p.lev_grab[4 * ((long long)p.maxlev + 2)] = (unsigned long long)s_valid | ((unsigned long long)s_scan[S - 1] << 32);
    }
}

// Push phase of level L: the frontier's out-arcs (u, v) mark F(u) &
// ~visited(v) in v's next-level mask; a vertex marked first at this level is
// claimed (an atomic on its level tag) and appended. A warp takes up to kGroup
// consecutive chunks and packs their arcs onto its lanes (two arcs per lane in
// flight), so short rows do not leave lanes idle; an arc costs its head and
// one W-word mask. The next-level mask is read before it is changed: most arcs
// into a hub find their bits set already, and the same-address atomics that
// would follow were what the hubs' rows waited for. Reach mode keeps one
// barrier per level, so it excludes the current level's mask too and does the
// entries' bookkeeping here.
template <int W, int MODE, int U>
__device__ __noinline__ void push_masks(int L, long long ccnt, long long gwarp, long long nwarps) {
    const TravParams &p = shared_params();
    WarpBuf<W> &buf = warp_buf<W>();
    const int lane = threadIdx.x & 31;
    const int cur = 1 + (L & 1);
    const int nxt = 1 + ((L + 1) & 1);
    int qn = 0;  // claimed vertices in the queue
    GroupGrabber<W> grab(&p.lev_grab[L], ccnt, gwarp, nwarps);
    for (;;) {
        long long c0;
        const int cnt = grab.next(c0, lane);
        if (cnt == 0) break;
        int na = 0;
        long long a0 = 0;
        if (lane < cnt) {
            const Chunk ch = load_chunk(&p.chunks[buf.first + c0 + lane]);
            na = ch.na;
            a0 = ch.a0;
            uint64_t F[W];
            if (MODE == kModeReach)
                load_mask<W>(p.vs + (size_t)ch.v * p.vs_stride + cur * W, F);
            else
                load_mask<W>(p.hm + (size_t)ch.e * W, F);
#pragma unroll
            for (int w = 0; w < W; ++w) buf.n[lane][w] = F[w];
            if (MODE == kModeReach && ch.k == 0) {
                if (p.levout && p.levout[ch.v] < 0) p.levout[ch.v] = L;
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    p.hm[(size_t)ch.e * W + w] = F[w];
                    atomicOr((unsigned long long *)&p.vs[(size_t)ch.v * p.vs_stride + w], (unsigned long long)F[w]);
                }
            }
        }
        const int total = buf.pack(lane, na, a0);
        if (MODE != kModeReach && lane == 0) buf.st[0].arcs += (unsigned)total;
        int base = 0;
        while (base < total) {
            // arcs until the queue holds more than it could take of another step's claims
            int wn[U], jn[U];
            auto fetch = [&](int b) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int i = b + 32 * u + lane;
                    jn[u] = buf.find(i);
                    wn[u] = i < total ? __ldcs(p.col + buf.aoff[jn[u]] + i) : -1;
                }
            };
            fetch(base);
            do {
                int wv[U], j[U], etag[U];
                uint64_t nm[U][W], early[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    wv[u] = wn[u];
                    j[u] = jn[u];
                    if (wv[u] >= 0) {
                        load_mask<W>(p.vs + (size_t)wv[u] * p.vs_stride, nm[u]);
                        if (MODE == kModeReach) {
                            // one word per mask: the row is one sector, and the tag
                            // joins this round of loads
                            uint64_t c[W];
                            load_mask<W>(p.vs + (size_t)wv[u] * p.vs_stride + cur * W, c);
                            early[u] = p.vs[(size_t)wv[u] * p.vs_stride + nxt * W];
                            etag[u] = p.tag[wv[u]];
#pragma unroll
                            for (int w = 0; w < W; ++w) nm[u][w] |= c[w];
                        }
                    }
                }
                base += 32 * U;
                fetch(base);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    bool any = false;
                    if (wv[u] >= 0) {
#pragma unroll
                        for (int w = 0; w < W; ++w) {
                            nm[u][w] = buf.n[j[u]][w] & ~nm[u][w];
                            any |= nm[u][w] != 0ull;
                        }
                    }
                    int old = 0x7fffffff;
                    if (any) {
                        uint64_t *wrow = p.vs + (size_t)wv[u] * p.vs_stride + nxt * W;
                        uint64_t nx[W];
                        int tg;
                        if (MODE == kModeReach) {
                            nx[0] = early[u];
                            tg = etag[u];
                        } else {
                            tg = p.tag[wv[u]];
                            load_mask<W>(wrow, nx);
                        }
                        bool add = false;
#pragma unroll
                        for (int w = 0; w < W; ++w) {
                            const uint64_t x = nm[u][w] & ~nx[w];
                            if (x) {
                                atomicOr((unsigned long long *)&wrow[w], (unsigned long long)x);
                                add = true;
                            }
                        }
                        if (add && tg < L + 1) old = atomicMax(&p.tag[wv[u]], L + 1);
                    }
                    claim<W>(buf, qn, old < L + 1, (unsigned)wv[u] | (old < 0 ? kFirstSeen : 0u), lane);
                }
            } while (base < total && qn <= 128 - 32 * U);
            drain<W, MODE>(L, qn, false);
        }
        __syncwarp();
    }
    drain<W, MODE>(L, qn, true);
}

// Gather phase: the vertices v of level L (their masks N(v) complete since
// the barrier after the push) sum sigma_s(v) = sum over in-neighbours u at
// level L - 1 for s of sigma_s(u). A warp takes up to kGroup consecutive
// in-arc chunks and packs their arcs onto its lanes: each lane reads one
// in-neighbour's level mask, t = current(u) & N(v), and stages it; then the
// warp walks the arcs with a tight source, U rows in flight, lane l holding
// sources l + 32 i: one test, one predicated load and one addition per 32
// sources (the masks are sparse, about a sixth of the tile, so wider loads
// would spend their instructions on sources that are not there). A row that
// fits one chunk is written once; longer rows meet in atomic adds on a row
// that starts from zero.
template <int W, typename T, int U>
__device__ __noinline__ void gather_level(int L, long long ics, long long iccnt, long long gwarp, long long nwarps) {
    const TravParams &p = shared_params();
    constexpr int S = 64 * W;
    constexpr int PL = 2 * W;
    WarpBuf<W> &buf = warp_buf<W>();
    const int lane = threadIdx.x & 31;
    const uint32_t lbit = 1u << lane;
    const int prv = 1 + ((L - 1) & 1);  // slot of the level-(L - 1) masks (level L: the other one)
    T *const sigma = reinterpret_cast<T *>(p.sigma) + lane;
    unsigned over = 0, tight = 0;
    if (lane == 0) buf.first = ics;
    T acc[PL];
#pragma unroll
    for (int q = 0; q < PL; ++q) acc[q] = T(0);
    GroupGrabber<W> grab(&p.lev_grab[5 * ((long long)p.maxlev + 2) + L], iccnt, gwarp, nwarps);
    for (;;) {
        long long c0;
        const int cnt = grab.next(c0, lane);
        if (cnt == 0) break;
        int na = 0;
        long long a0 = 0;
        if (lane < cnt) {
            const Chunk ch = load_chunk(&p.ichunks[buf.first + c0 + lane]);
            buf.v[lane] = ch.v;
            buf.nch[lane] = ch.nch;
            na = ch.na;
            a0 = ch.a0;
            const uint64_t *row = p.vs + (size_t)ch.v * p.vs_stride;
            uint64_t F[W];
            load_mask<W>(row + (3 - prv) * W, F);
#pragma unroll
            for (int w = 0; w < W; ++w) buf.n[lane][w] = F[w];
            if (ch.k == 0) {
                uint64_t vis[W];
                load_mask<W>(row, vis);
                enter_entry<W>(p, L, ch.e, ch.v, F, vis, ch.pad, buf.st[lane]);
            }
        }
        const int total = buf.pack(lane, na, a0);
        if (lane == 0) buf.st[0].arcs += (unsigned)total;
        // writes the sums of chunk j of the group
        auto flush = [&](int j) {
            const int nj = buf.nch[j];
            const uint32_t *nw = reinterpret_cast<const uint32_t *>(buf.n[j]);
            T *row = sigma + (size_t)buf.v[j] * S;
#pragma unroll
            for (int q = 0; q < PL; ++q) {
                T x = acc[q];
                over |= SigOver<T>::test(x);
                if (nj == 1) {
                    if (nw[q] & lbit) row[32 * q] = x;
                } else if (x != T(0)) {
                    x += atomicAdd(row + 32 * q, x);
                    over |= SigOver<T>::test(x);
                }
                flag_two53(p, x, lane + 32 * q);
                acc[q] = T(0);
            }
        };
        int jc = 0;  // chunk whose sums are in acc
        int un, jn;
        jn = buf.find(lane);
        un = lane < total ? __ldcs(p.rcol + buf.aoff[jn] + lane) : -1;
        for (int base = 0; base < total; base += 32) {
            const int u = un, j = jn;
            uint64_t t[W];
            if (u >= 0) load_mask<W>(p.vs + (size_t)u * p.vs_stride + prv * W, t);
            {
                const int idx = base + 32 + lane;
                jn = buf.find(idx);
                un = idx < total ? __ldcs(p.rcol + buf.aoff[jn] + idx) : -1;
            }
            bool any = false;
            if (u >= 0) {
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    t[w] &= buf.n[j][w];
                    any |= t[w] != 0ull;
                    tight += (unsigned)__popcll(t[w]);
                    buf.t[lane][w] = t[w];
                }
            }
            unsigned bal = __ballot_sync(kFull, any);
            __syncwarp();
            while (bal) {
                int jj[U];
                T x[U][PL];
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    jj[k] = -1;
                    if (k == 0 || bal) {
                        const int i = __ffs(bal) - 1;
                        bal &= bal - 1;
                        jj[k] = __shfl_sync(kFull, j, i);
                        const T *row = sigma + (size_t)__shfl_sync(kFull, u, i) * S;
                        const uint32_t *tw = reinterpret_cast<const uint32_t *>(buf.t[i]);
#pragma unroll
                        for (int q = 0; q < PL; ++q) x[k][q] = (tw[q] & lbit) ? row[32 * q] : T(0);
                    }
                }
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    if (k > 0 && jj[k] < 0) break;
                    if (jj[k] != jc) {
                        flush(jc);
                        jc = jj[k];
                    }
#pragma unroll
                    for (int q = 0; q < PL; ++q) acc[q] += x[k][q];
                }
            }
            // at most 32 terms of below 2^26 each since the last test
#pragma unroll
            for (int q = 0; q < PL; ++q) over |= SigOver<T>::test(acc[q]);
            __syncwarp();
        }
        flush(jc);
        __syncwarp();
    }
    buf.st[lane].tight += tight;
    if (over) set_err(p.ctr, kDevWide);
}

// 1 / sigma. The chip's fp64 units are few (a warp instruction holds an SM's
// for 16 cycles, so the dozen of a division cost more than the rest of a
// step): counts up to kInverses, nearly all of them, are looked up.
__device__ __forceinline__ double *inverses() {
    __shared__ double s_inv[kInverses];
    return s_inv;
}
__device__ __forceinline__ double inverse_of(const double *s_inv, uint32_t x) {
    return x < (uint32_t)kInverses ? s_inv[x] : 1.0 / (double)x;
}
__device__ __forceinline__ double inverse_of(const double *s_inv, double x) { return 1.0 / x; }

// a / sigma, the same bits as the fp64 division: with y the correctly rounded
// 1 / sigma, q = a y and r = a - q sigma exactly, q + r y rounds to a / sigma
// (Markstein, IBM J. Res. Dev. 34, 1990), four fp64 operations instead of a
// division's dozen.
__device__ __forceinline__ double quotient(const double *s_inv, double a, uint32_t x) {
    if (x >= (uint32_t)kInverses) return a / (double)x;
    const double y = s_inv[x], q = a * y;
    return fma(fma(-q, (double)x, a), y, q);
}
__device__ __forceinline__ double quotient(const double *s_inv, double a, double x) { return a / x; }

// Bookkeeping of the level-L entries after a bottom-up step (which counts
// paths itself), one thread each.
template <int W>
__device__ void enter_level(const TravParams &p, int L, long long es, long long ecnt, long long gthr,
                            long long nthr) {
    Stats &st = warp_buf<W>().st[threadIdx.x & 31];
    const int own = 1 + (L & 1);
    for (long long e = es + gthr; e < es + ecnt; e += nthr) {
        const int v = p.hv[e];
        const uint64_t *row = p.vs + (size_t)v * p.vs_stride;
        uint64_t F[W], vis[W];
        load_mask<W>(row + own * W, F);
        load_mask<W>(row, vis);
        enter_entry<W>(p, L, e, v, F, vis, (int)(p.off[v + 1] - p.off[v]), st);
    }
}

// Bottom-up step of level L (the forward pass of Section 2 read from the
// other end): sigma_s(v) is the sum of sigma_s(u) over the in-neighbours u
// of v at level L for s, so every vertex v that some source of the tile has
// not reached yet (U = valid & ~visited(v)) scans its in-arcs
// in R(G), and for each in-neighbour u the sources of current(u) & U reach v
// at level L + 1, each adding sigma_s(u). The sums stay in registers: a
// vertex whose in-arcs fit one chunk writes its sigma row and its next-level
// mask once, with no atomic per arc (longer rows are cut into chunks that
// meet in atomic adds). Lane l holds sources l + 32 i. The new entries get
// their bookkeeping from enter_level after the grid barrier that follows.
template <int W, int MODE, typename T>
__device__ __noinline__ void pull_level(int L, const uint64_t *s_valid, long long nwarps) {
    const TravParams &p = shared_params();
    Stats st;
    WarpBuf<W> &buf = warp_buf<W>();
    constexpr int S = 64 * W;
    constexpr int PL = 2 * W;
    const int lane = threadIdx.x & 31;
    const int cur = 1 + (L & 1);
    const int nxt = 1 + ((L + 1) & 1);
    const int stride = p.vs_stride;
    const int CH = p.chunk_arcs;
    T *sigma = reinterpret_cast<T *>(p.sigma);
    unsigned over = 0;
    // every vertex's in-arc chunks, handed out dynamically
    int qn = 0;  // claimed vertices in the queue
    ChunkGrabber grab(&p.lev_grab[L], p.npchunks, nwarps);
    long long c;
    while (grab.next(c, lane)) {
        const int2 pc = p.pchunks[c];
        const int v = pc.x;
        const uint64_t *vrow = p.vs + (size_t)v * stride;
        uint64_t U[W];
        bool anyu = false;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            U[w] = s_valid[w] & ~vrow[w];
            anyu |= U[w] != 0ull;
        }
        if (!anyu) continue;  // every source of the tile has reached v
        const long long rb = p.roff[v], re = p.roff[v + 1];
        const long long a0 = rb + (long long)pc.y * CH;
        const int na = (int)min((long long)CH, re - a0);
        const int nch = (int)((re - rb + CH - 1) / CH);
        T acc[PL];
#pragma unroll
        for (int ii = 0; ii < PL; ++ii) acc[ii] = T(0);
        unsigned lm = 0;  // bit ii: source lane + 32 ii reaches v here
        int unext = lane < na ? p.rcol[a0 + lane] : 0;
        for (int base = 0; base < na; base += 32) {
            const bool valid = base + lane < na;
            const int u = unext;
            unext = base + 32 + lane < na ? p.rcol[a0 + base + 32 + lane] : 0;
            uint64_t t[W];
            bool any = false;
            if (valid) {
                const uint64_t *urow = p.vs + (size_t)u * stride;
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    t[w] = urow[cur * W + w] & U[w];
                    any |= t[w] != 0ull;
                }
                st.arcs += 1;
#pragma unroll
                for (int w = 0; w < W; ++w) st.tight += (unsigned)__popcll(t[w]);
            } else {
#pragma unroll
                for (int w = 0; w < W; ++w) t[w] = 0ull;
            }
            // two tight in-neighbours per step: their gathers overlap
            unsigned bal = __ballot_sync(kFull, any);
            while (bal) {
                const int i0 = __ffs(bal) - 1;
                bal &= bal - 1;
                const int i1 = bal ? __ffs(bal) - 1 : -1;
                if (bal) bal &= bal - 1;
                const int j1 = i1 < 0 ? i0 : i1;
                const int u0 = __shfl_sync(kFull, u, i0);
                const int u1 = __shfl_sync(kFull, u, j1);
                uint64_t n0[W], n1[W];
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    n0[w] = __shfl_sync(kFull, t[w], i0);
                    n1[w] = i1 < 0 ? 0ull : __shfl_sync(kFull, t[w], j1);
                }
                const T *r0 = sigma + (size_t)u0 * S;
                const T *r1 = sigma + (size_t)u1 * S;
#pragma unroll
                for (int ii = 0; ii < PL; ++ii) {
                    const int s = lane + 32 * ii;
                    const bool b0 = mask_bit<W>(n0, s), b1 = mask_bit<W>(n1, s);
                    const T x0 = b0 ? r0[s] : T(0);
                    const T x1 = b1 ? r1[s] : T(0);
                    acc[ii] += x0 + x1;
                    over |= SigOver<T>::test(acc[ii]);
                    if (b0 | b1) lm |= 1u << ii;
                }
            }
        }
        uint64_t nm[W];
        bool anynm = false;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const unsigned lo = __ballot_sync(kFull, (lm >> (2 * w)) & 1u);
            const unsigned hi = __ballot_sync(kFull, (lm >> (2 * w + 1)) & 1u);
            nm[w] = (uint64_t)lo | ((uint64_t)hi << 32);
            anynm |= nm[w] != 0ull;
        }
        if (!anynm) continue;
        // the next-level mask (atomic: the stale level L - 1 bits of this slot
        // are being cleared at the same time) and sigma
#pragma unroll
        for (int w = 0; w < W; ++w)
            if (lane == w && nm[w])
                atomicOr((unsigned long long *)&p.vs[(size_t)v * stride + nxt * W + w], (unsigned long long)nm[w]);
        T *srow = sigma + (size_t)v * S;
#pragma unroll
        for (int ii = 0; ii < PL; ++ii)
            if ((lm >> ii) & 1u) {
                T x = acc[ii];
                if (nch == 1)
                    srow[lane + 32 * ii] = x;
                else
                    x += atomicAdd(&srow[lane + 32 * ii], x);
                over |= SigOver<T>::test(x);
                flag_two53(p, x, lane + 32 * ii);
            }
        int old = 0;
        if (lane == 0) old = atomicMax(&p.tag[v], L + 1);
        old = __shfl_sync(kFull, old, 0);
        claim<W>(buf, qn, lane == 0 && old < L + 1, (unsigned)v | (old < 0 ? kFirstSeen : 0u), lane);
        drain<W, MODE>(L, qn, false);
    }
    drain<W, MODE>(L, qn, true);
    buf.st[lane].tight += st.tight;
    buf.st[lane].arcs += st.arcs;
    if (over) set_err(p.ctr, kDevWide);
}

// Eq. 4, push form, from level L into level L - 1: each entry w of level L
// sends c_s(w) = (1 + delta_s(w)) / sigma_s(w) = 1 / sigma_s(w) + acc_s(w)
// (delta_s(w) = sigma_s(w) * acc_s(w), complete: level L + 1 pushed into it in
// the previous step) back along its in-arcs (v, w) that are tight for a source s still
// active at L - 1 (v at level L - 1 for s), adding it to acc_s(v) with fp64
// atomic adds. c is formed on the fly from the sigma and acc slabs, which this
// step only reads for level-L pairs. The in-arc chunks of level L were cut in
// the forward pass. Lane l holds sources l + 32 i; two tight tails per step.
template <int W, typename T>
__device__ void push_level(const TravParams &p, int L, long long ics, long long ccnt, const uint64_t *s_act,
                           const double *s_inv, long long nwarps) {
    constexpr int S = 64 * W;
    constexpr int PL = 2 * W;
    const int lane = threadIdx.x & 31;
    const int par = 1 + ((L - 1) & 1);  // parity slot holding the level-(L-1) masks
    const int stride = p.vs_stride;
    ChunkGrabber grab(&p.lev_grab[p.maxlev + 2 + L], ccnt, nwarps);
    unsigned arcs = 0;
    long long c;
    while (grab.next(c, lane)) {
        const Chunk ch = load_chunk(&p.ichunks[ics + c]);
        const int w = ch.v;
        const long long a0 = ch.a0;
        const int na = ch.na;
        int vnext = lane < na ? p.rcol[a0 + lane] : 0;
        uint64_t F[W];
#pragma unroll
        for (int k = 0; k < W; ++k) F[k] = p.hm[(size_t)ch.e * W + k] & s_act[k];
        const T *sigma = reinterpret_cast<const T *>(p.sigma);
        double cw[PL];
        T sw[PL];
#pragma unroll
        for (int ii = 0; ii < PL; ++ii) {
            const bool in = mask_bit<W>(F, lane + 32 * ii);
            sw[ii] = in ? sigma[(size_t)w * S + lane + 32 * ii] : T(1);
            cw[ii] = in ? p.acc[(size_t)w * S + lane + 32 * ii] : 0.0;
        }
#pragma unroll
        for (int ii = 0; ii < PL; ++ii) cw[ii] += inverse_of(s_inv, sw[ii]);
        for (int base = 0; base < na; base += 32) {
            const bool valid = base + lane < na;
            const int v = vnext;
            vnext = base + 32 + lane < na ? p.rcol[a0 + base + 32 + lane] : 0;
            uint64_t tm[W];
            bool any = false;
            if (valid) {
                const uint64_t *row = p.vs + (size_t)v * stride;
#pragma unroll
                for (int k = 0; k < W; ++k) {
                    tm[k] = F[k] & row[par * W + k];
                    any |= tm[k] != 0ull;
                }
                arcs += 1;
            } else {
#pragma unroll
                for (int k = 0; k < W; ++k) tm[k] = 0ull;
            }
            unsigned bal = __ballot_sync(kFull, any);
            while (bal) {
                const int i0 = __ffs(bal) - 1;
                bal &= bal - 1;
                const int i1 = bal ? __ffs(bal) - 1 : -1;
                if (bal) bal &= bal - 1;
                const int j1 = i1 < 0 ? i0 : i1;
                const int v0 = __shfl_sync(kFull, v, i0);
                const int v1 = __shfl_sync(kFull, v, j1);
                uint64_t n0[W], n1[W];
#pragma unroll
                for (int k = 0; k < W; ++k) {
                    n0[k] = __shfl_sync(kFull, tm[k], i0);
                    n1[k] = i1 < 0 ? 0ull : __shfl_sync(kFull, tm[k], j1);
                }
                double *r0 = p.acc + (size_t)v0 * S;
                double *r1 = p.acc + (size_t)v1 * S;
#pragma unroll
                for (int ii = 0; ii < PL; ++ii) {
                    const int s = lane + 32 * ii;
                    if (mask_bit<W>(n0, s)) atomicAdd(&r0[s], cw[ii]);
                    if (mask_bit<W>(n1, s)) atomicAdd(&r1[s], cw[ii]);
                }
            }
        }
    }
    warp_buf<W>().st[lane].arcs += arcs;
}

// The rest of a backward step at level L, one thread per entry: delta_s(r_q)
// for the query vertices among the level-L entries (their accumulators are
// complete), and, when the pass goes on, the parity slot shared by levels L
// and L - 2: the level-L bits leave it and the level-(L - 2) bits enter it
// (the push from L - 1 reads them in the next step).
template <int W, typename T>
__device__ void level_outputs(const TravParams &p, int L, bool swap, bool set_next, const uint64_t *s_act,
                              const uint64_t *s_need, long long gthr, long long nthr) {
    constexpr int S = 64 * W;
    const int stride = p.vs_stride;
    const int slot = 1 + (L & 1);
    const long long e0 = p.lev_start[L], e1 = e0 + (long long)p.lev_cnt[L];
    for (long long e = e0 + gthr; e < e1; e += nthr) {
        const int v = p.hv[e];
        uint64_t F[W];
#pragma unroll
        for (int k = 0; k < W; ++k) F[k] = p.hm[(size_t)e * W + k];
        if (swap) {
            uint64_t *row = p.vs + (size_t)v * stride;
#pragma unroll
            for (int k = 0; k < W; ++k) atomicAnd((unsigned long long *)&row[slot * W + k], ~(unsigned long long)F[k]);
        }
        const uint64_t qm = p.qmask[v];
        if (!qm) continue;
#pragma unroll
        for (int k = 0; k < W; ++k) {
            uint64_t b = F[k] & s_act[k];
            while (b) {
                const int s = 64 * k + __ffsll((long long)b) - 1;
                b &= b - 1;
                uint64_t x = qm & s_need[s];
                if (!x) continue;
                const double d = (double)reinterpret_cast<const T *>(p.sigma)[(size_t)v * S + s] * p.acc[(size_t)v * S + s];
                while (x) {
                    const int q = __ffsll((long long)x) - 1;
                    x &= x - 1;
                    p.dep[s * 64 + q] = d;
                }
            }
        }
    }
    if (!set_next) return;
    const long long g0 = p.lev_start[L - 2], g1 = g0 + (long long)p.lev_cnt[L - 2];
    for (long long e = g0 + gthr; e < g1; e += nthr) {
        uint64_t *row = p.vs + (size_t)p.hv[e] * stride;
#pragma unroll
        for (int k = 0; k < W; ++k)
            atomicOr((unsigned long long *)&row[slot * W + k], (unsigned long long)p.hm[e * W + k]);
    }
}

// Dependencies on one query vertex r by a vertex scan, from the pair
// dependencies of Eq. 2: r lies on sigma_sr * sigma_rt of the sigma_st
// shortest s-t paths when d(s, r) + d(r, t) = d(s, t) (and on none
// otherwise), so delta_s.(r) = sigma_sr * sum of sigma_rt / sigma_st over
// those t != s, r. rlev and rsig hold d(r, t) and sigma_rt from a forward
// traversal rooted at r. A level-L entry (t, F) lists the sources s with
// d(s, t) = L, so source s takes t exactly when d(s, r) = L - d(r, t), and
// every (t, s) pair is met once, in any order: there is no level order and
// no barrier. Lanes first screen 32 entries at a time on d(r, t) against the
// levels at which the tile's sources meet r; the survivors are taken two at
// a time, each lane adding the terms of its sources l + 32 i in registers.
// Each warp's sums, times sigma_sr, go to vsum with one fp64 atomic add per
// source.
template <int W, typename T>
__device__ void vertex_scan(const TravParams &p, int Lmax, const uint64_t *s_need, long long gwarp,
                            long long nwarps) {
    const double *const s_inv = inverses();
    constexpr int S = 64 * W;
    constexpr int PL = 2 * W;
    const int lane = threadIdx.x & 31;
    int ks[PL];  // d(s, r) of the lane's sources, -1 for slots without a query
    double a[PL];
    int kmin = 0x7fffffff, kmax = -1;
    uint64_t kset = 0ull;  // the levels below 64 at which some source meets r
#pragma unroll
    for (int ii = 0; ii < PL; ++ii) {
        const int s = lane + 32 * ii;
        const uint64_t x = s_need[s];
        ks[ii] = x ? p.qlevel[s * 64 + __ffsll((long long)x) - 1] : -1;
        a[ii] = 0.0;
        if (ks[ii] >= 1) {
            kmin = min(kmin, ks[ii]);
            kmax = max(kmax, ks[ii]);
            if (ks[ii] < 64) kset |= 1ull << ks[ii];
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        kmin = min(kmin, __shfl_xor_sync(kFull, kmin, o));
        kmax = max(kmax, __shfl_xor_sync(kFull, kmax, o));
        kset |= __shfl_xor_sync(kFull, kset, o);
    }
    unsigned pairs = 0;
    if (kmax >= 1) {
        for (int L = kmin + 1; L <= Lmax; ++L) {
            const long long eend = p.lev_start[L + 1];
            for (long long b = p.lev_start[L] + 32 * gwarp; b < eend; b += 32 * nwarps) {
                const long long e = b + lane;
                int t = 0, k = -1;
                if (e < eend) {
                    t = p.hv[e];
                    const int dr = p.rlev[t];
                    if (dr >= 1) k = L - dr;
                }
                const bool keep = k >= kmin && k <= kmax && (k >= 64 || ((kset >> k) & 1ull));
                const double rs = keep ? p.rsig[t] : 0.0;
                unsigned bal = __ballot_sync(kFull, keep);
                while (bal) {
                    const int i0 = __ffs(bal) - 1;
                    bal &= bal - 1;
                    const int i1 = bal ? __ffs(bal) - 1 : -1;
                    if (bal) bal &= bal - 1;
                    const int j1 = i1 < 0 ? i0 : i1;
                    const int t0 = __shfl_sync(kFull, t, i0);
                    const int t1 = __shfl_sync(kFull, t, j1);
                    const int k0 = __shfl_sync(kFull, k, i0);
                    const int k1 = i1 < 0 ? -2 : __shfl_sync(kFull, k, j1);  // -2 matches no source
                    const double r0 = __shfl_sync(kFull, rs, i0);
                    const double r1 = __shfl_sync(kFull, rs, j1);
                    uint64_t f0[W], f1[W];
#pragma unroll
                    for (int w = 0; w < W; ++w) {
                        f0[w] = p.hm[(b + i0) * W + w];
                        f1[w] = p.hm[(b + j1) * W + w];
                    }
                    const T *q0 = reinterpret_cast<const T *>(p.sigma) + (size_t)t0 * S;
                    const T *q1 = reinterpret_cast<const T *>(p.sigma) + (size_t)t1 * S;
#pragma unroll
                    for (int ii = 0; ii < PL; ++ii) {
                        const int s = lane + 32 * ii;
                        if (ks[ii] == k0 && mask_bit<W>(f0, s)) {
                            a[ii] += quotient(s_inv, r0, q0[s]);
                            ++pairs;
                        }
                        if (ks[ii] == k1 && mask_bit<W>(f1, s)) {
                            a[ii] += quotient(s_inv, r1, q1[s]);
                            ++pairs;
                        }
                    }
                }
            }
        }
    }
    const T *sr = reinterpret_cast<const T *>(p.sigma) + (size_t)p.vroot * S;
#pragma unroll
    for (int ii = 0; ii < PL; ++ii)
        if (a[ii] != 0.0) atomicAdd(&p.vsum[lane + 32 * ii], (double)sr[lane + 32 * ii] * a[ii]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pairs += __shfl_xor_sync(kFull, pairs, o);
    if (lane == 0 && pairs) atomicAdd(&p.ctr->vpairs, (unsigned long long)pairs);
}

// Shared sums of vertex_scan_multi (in the space the warps' buffers take
// during the forward pass).
template <int W>
struct ScanBuf {
    static constexpr int G = W >= 8 ? 4 : 8;  // columns per pass
    double acc[64 * W * G];                   // [s][column]
    int32_t ql[64 * W * G];                   // d(s, r_c) for sources that need column c, else -1
};

// The number of terms vertex_scan_multi would add up, without adding them: an
// entry (t, F) of level L has, for column c, the sources of F that meet r_c at
// level L - d(r_c, t). lm holds these sources per (column, level), the levels
// from 63 on in one place (an upper bound there). One thread per entry.
template <int W>
struct CountBuf {
    static constexpr int G = ScanBuf<W>::G;
    unsigned long long lm[G][64][W];
};
template <int W>
__device__ __noinline__ void scan_count(int Lmax, long long gthr, long long nthr) {
    constexpr int S = 64 * W;
    constexpr int G = CountBuf<W>::G;
    const TravParams &p = shared_params();
    const uint64_t *s_need = tile_need();
    CountBuf<W> &cb = *reinterpret_cast<CountBuf<W> *>(s_dyn + kParamBytes + 512 * W);
    unsigned long long pairs = 0;
    for (int cg = 0; cg < p.ncols; cg += G) {
        const int nc = min(G, p.ncols - cg);
        __syncthreads();
        for (int i = threadIdx.x; i < G * 64 * W; i += blockDim.x) (&cb.lm[0][0][0])[i] = 0ull;
        __syncthreads();
        for (int s = threadIdx.x; s < S; s += blockDim.x) {
            uint64_t x = s_need[s];
            while (x) {
                const int q = __ffsll((long long)x) - 1;
                x &= x - 1;
                const int j = p.qcol[q] - cg;
                if (j < 0 || j >= nc) continue;
                const int lv = p.qlevel[s * 64 + q];
                if (lv >= 1) atomicOr(&cb.lm[j][min(lv, 63)][s >> 6], 1ull << (s & 63));
            }
        }
        __syncthreads();
        for (int L = 2; L <= Lmax; ++L) {
            const long long eend = p.lev_start[L + 1];
            for (long long e = p.lev_start[L] + gthr; e < eend; e += nthr) {
                const int32_t *row = p.rlevq + (size_t)p.hv[e] * 64 + cg;
                uint64_t F[W];
                load_mask<W>(p.hm + (size_t)e * W, F);
                for (int j = 0; j < nc; ++j) {
                    const int dr = row[j];
                    if (dr < 1 || dr >= L) continue;
                    const unsigned long long *m = cb.lm[j][min(L - dr, 63)];
#pragma unroll
                    for (int w = 0; w < W; ++w) pairs += (unsigned)__popcll(F[w] & m[w]);
                }
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pairs += __shfl_xor_sync(kFull, pairs, o);
    if ((threadIdx.x & 31) == 0 && pairs) atomicAdd(&p.ctr->trial_pairs, pairs);
}

// Dependencies on several query vertices at once by the vertex scan: the
// form of vertex_scan for a group whose queries sit at up to 64 distinct
// vertices (columns c, vertex croot[c]). rlevq / rsigq [t * 64 + c] hold
// d(croot[c], t) and sigma_{croot[c] t} from one traversal rooted at all the
// columns. Columns go 8 at a time (one 32-byte sector of a row of rlevq).
// Each warp screens 32 level-L entries at a time: entry (t, F) is kept for
// column c when L - d(r_c, t) is a level at which a source of the tile that
// needs c meets r_c (the same screen as the one-vertex scan). For a kept
// (entry, column), each lane adds sigma_{r_c t} / sigma_st, for its sources s
// in F that need c and have d(s, r_c) = L - d(r_c, t), into the block's
// shared sums [s][c]; at the end of the 8 columns the block multiplies them by
// sigma_s(r_c) and adds them into msum [s * 64 + c] with one fp64 atomic each.
// No level order and no grid barrier inside.
template <int W, typename T>
__device__ __noinline__ void vertex_scan_multi(int Lmax, long long gwarp, long long nwarps) {
    const TravParams &p = shared_params();
    const uint64_t *s_need = tile_need();
    ScanBuf<W> &sb = *reinterpret_cast<ScanBuf<W> *>(s_dyn + kParamBytes + 512 * W);
    const double *const s_inv = inverses();
    constexpr int S = 64 * W;
    constexpr int PL = 2 * W;
    constexpr int G = ScanBuf<W>::G;
    double *const s_acc = sb.acc;
    int32_t *const s_ql = sb.ql;
    __shared__ int32_t s_kmin[G], s_kmax[G];
    __shared__ unsigned long long s_kset[G];
    const int lane = threadIdx.x & 31;
    unsigned pairs = 0;
    for (int cg = 0; cg < p.ncols; cg += G) {
        const int nc = min(G, p.ncols - cg);
        __syncthreads();
        for (int i = threadIdx.x; i < S * G; i += blockDim.x) {
            s_acc[i] = 0.0;
            s_ql[i] = -1;
        }
        if (threadIdx.x < G) {
            s_kmin[threadIdx.x] = 0x7fffffff;
            s_kmax[threadIdx.x] = -1;
            s_kset[threadIdx.x] = 0ull;
        }
        __syncthreads();
        for (int s = threadIdx.x; s < S; s += blockDim.x) {
            uint64_t x = s_need[s];
            while (x) {
                const int q = __ffsll((long long)x) - 1;
                x &= x - 1;
                const int j = p.qcol[q] - cg;
                if (j < 0 || j >= nc) continue;
                const int lv = p.qlevel[s * 64 + q];
                if (lv < 1) continue;
                s_ql[s * G + j] = lv;
                atomicMin(&s_kmin[j], lv);
                atomicMax(&s_kmax[j], lv);
                if (lv < 64) atomicOr(&s_kset[j], 1ull << lv);
            }
        }
        __syncthreads();
        int kmin[G], kmax[G];
        unsigned long long kset[G];
        int lfrom = 0x7fffffff;
#pragma unroll
        for (int j = 0; j < G; ++j) {
            kmin[j] = s_kmin[j];
            kmax[j] = s_kmax[j];
            kset[j] = s_kset[j];
            if (kmax[j] >= 1) lfrom = min(lfrom, kmin[j] + 1);
        }
        for (int L = lfrom; L <= Lmax; ++L) {
            const long long ebeg = p.lev_start[L], eend = p.lev_start[L + 1];
            // entries a warp takes together: fewer on thin levels, where a warp's
            // kept (entry, column) pairs, one after another, are what it waits for
            const int wide = (int)min(32ll, (eend - ebeg + nwarps - 1) / nwarps);
            for (long long b = ebeg + wide * gwarp; b < eend; b += wide * nwarps) {
                const long long e = lane < wide ? b + lane : eend;
                int t = 0;
                unsigned kq = 0;
                int dr[G];
#pragma unroll
                for (int j = 0; j < G; ++j) dr[j] = -1;
                if (e < eend) {
                    t = p.hv[e];
                    const int4 *row = reinterpret_cast<const int4 *>(p.rlevq + (size_t)t * 64 + cg);
#pragma unroll
                    for (int h = 0; h < G / 4; ++h) {
                        const int4 a = row[h];
                        dr[4 * h] = a.x;
                        dr[4 * h + 1] = a.y;
                        dr[4 * h + 2] = a.z;
                        dr[4 * h + 3] = a.w;
                    }
#pragma unroll
                    for (int j = 0; j < G; ++j) {
                        const int k = L - dr[j];
                        if (j < nc && dr[j] >= 1 && k >= kmin[j] && k <= kmax[j] && (k >= 64 || ((kset[j] >> k) & 1ull)))
                            kq |= 1u << j;
                    }
                }
                unsigned bal = __ballot_sync(kFull, kq != 0u);
                while (bal) {
                    const int i = __ffs(bal) - 1;
                    bal &= bal - 1;
                    const int ti = __shfl_sync(kFull, t, i);
                    unsigned kqi = __shfl_sync(kFull, kq, i);
                    int dri[G];
#pragma unroll
                    for (int j = 0; j < G; ++j) dri[j] = __shfl_sync(kFull, dr[j], i);
                    uint64_t F[W];
#pragma unroll
                    for (int w = 0; w < W; ++w) F[w] = p.hm[(b + i) * W + w];
                    const T *qs = reinterpret_cast<const T *>(p.sigma) + (size_t)ti * S;
                    while (kqi) {
                        const int j = __ffs(kqi) - 1;
                        kqi &= kqi - 1;
                        int drj = 0;
#pragma unroll
                        for (int jj = 0; jj < G; ++jj)
                            if (jj == j) drj = dri[jj];
                        const int k = L - drj;
                        const double rs = p.rsigq[(size_t)ti * 64 + cg + j];
#pragma unroll
                        for (int ii = 0; ii < PL; ++ii) {
                            const int s = lane + 32 * ii;
                            if (mask_bit<W>(F, s) && s_ql[s * G + j] == k) {
                                atomicAdd(&s_acc[s * G + j], quotient(s_inv, rs, qs[s]));
                                ++pairs;
                            }
                        }
                    }
                }
            }
        }
        __syncthreads();
        // sigma_s(r_c) times the sums: delta_s.(r_c) parts of this block
        for (int i = threadIdx.x; i < S * G; i += blockDim.x) {
            const double a = s_acc[i];
            if (a != 0.0) {
                const int sl = i / G, j = i % G;
                atomicAdd(&p.msum[sl * 64 + cg + j], a * (double)reinterpret_cast<const T *>(p.sigma)[(size_t)p.croot[cg + j] * S + sl]);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pairs += __shfl_xor_sync(kFull, pairs, o);
    if (lane == 0 && pairs) atomicAdd(&p.ctr->vpairs, (unsigned long long)pairs);
}

// The launch's parameters into shared memory, with the state arrays of the
// block's team: each team has the state of one tile.
template <typename T>
__device__ __forceinline__ void load_params(const TravParams &launch, int team) {
    for (int i = threadIdx.x; i < (int)(sizeof(TravParams) / 4); i += blockDim.x)
        reinterpret_cast<uint32_t *>(s_dyn)[i] = reinterpret_cast<const uint32_t *>(&launch)[i];
    __syncthreads();
    if (threadIdx.x == 0) {
        TravParams &p = *reinterpret_cast<TravParams *>(s_dyn);
        const size_t t = (size_t)team, n = (size_t)p.n, lev = (size_t)p.maxlev + 2, ws = (size_t)p.ws_slots;
        p.bar += t;
        p.vs += t * n * p.vs_stride;
        p.tag += t * n;
        p.sigma = reinterpret_cast<double *>(reinterpret_cast<T *>(p.sigma) + t * n * ws);
        p.acc += t * n * ws;
        p.hv += t * (size_t)p.hcap;
        p.hm += t * (size_t)p.hm_words;
        p.chunks += t * (size_t)p.ccap;
        p.ichunks += t * (size_t)p.ccap;
        p.lev_cnt += t * lev;
        p.lev_grab += t * 6 * lev;
        p.lev_start += t * lev;
        p.lev_icstart += t * lev;
        p.qlevel += t * ws * 64;
        p.dep += t * ws * 64;
        p.vsum += t * 2 * ws;
        p.msum += t * 2 * ws * 64;
        p.srcflag += t * (size_t)max(p.ws_slots / 64, 4);
    }
    __syncthreads();
}

// Barrier of the blocks of a team (a lone block needs no wait on others; it
// still leaves when another team has flagged an error).
__device__ __forceinline__ bool team_barrier(const TravParams &p, unsigned long long &target) {
    return grid_barrier(p.ctr, target, p.timeout_ns, &p.bar->count, (uint32_t)p.team_blocks);
}

template <int W, int MODE, int MINB, typename T>
__global__ void __launch_bounds__(512, MINB) trav_kernel(const __grid_constant__ TravParams launch) {
    constexpr int S = 64 * W;
    constexpr int kGatherU = (W <= 2 || (W == 4 && MINB == 1 && sizeof(T) == 4)) ? 2 : 1;  // rows in flight per warp of the gather
    constexpr int kPushU = W * MINB > 4 ? 1 : 2;                                            // arcs in flight per lane of the push
    const int lane = threadIdx.x & 31;
    const int team = blockIdx.x / launch.team_blocks;
    const int block = blockIdx.x - team * launch.team_blocks;  // within the team
    const bool leader = block == 0 && threadIdx.x == 0;
    load_params<T>(launch, team);
    const TravParams &p = shared_params();
    T *sigma = reinterpret_cast<T *>(p.sigma);
    const long long wpb = blockDim.x >> 5;
    const long long gwarp = (long long)block * wpb + (threadIdx.x >> 5);
    const long long nwarps = (long long)p.team_blocks * wpb;
    const long long gthr = (long long)block * blockDim.x + threadIdx.x;
    const long long nthr = (long long)p.team_blocks * blockDim.x;
    unsigned long long bar = 0;  // arrivals that the last barrier waited for
    uint64_t *const s_need = tile_need();
    __shared__ int32_t s_minql[S];
    __shared__ uint64_t s_active[W];
    __shared__ uint64_t s_active_next[W];
    __shared__ uint64_t s_valid[W];  // the tile's occupied source slots
    __shared__ int32_t s_lstop;
    double *const s_inv = inverses();  // 1 / k
    if (MODE != kModeReach && sizeof(T) == 4)
        for (int i = threadIdx.x; i < kInverses; i += blockDim.x) s_inv[i] = p.inv[i];
    const bool timer = team == 0 && leader;
    unsigned long long t_mark = timer ? global_ns() : 0ull;
    unsigned long long ns_fwd = 0, ns_bwd = 0, ns_other = 0;

    // a team's first tile is its own number, the next ones come from a counter
    for (long long tile = team; tile < p.ntiles; tile = (long long)ld_vol(&p.bar->next)) {
        const int32_t *tsrc = p.srcs + tile * S;
        check_cancel(p);
        if (block == 0) init_tile<W, MODE, T>(p, tsrc);
        for (int s = threadIdx.x; s < S; s += blockDim.x) {
            const int32_t v = tsrc[s];
            s_need[s] = (MODE != kModeReach && v >= 0) ? p.need[v] : 0ull;
        }
        if (threadIdx.x < W) {
            uint64_t m = 0;
            for (int b = 0; b < 64; ++b)
                if (tsrc[threadIdx.x * 64 + b] >= 0) m |= 1ull << b;
            s_valid[threadIdx.x] = m;
        }
        warp_buf<W>().st[lane] = Stats();
        if (!team_barrier(p, bar)) return;
        if (timer) {
            const unsigned long long t = global_ns();
            ns_other += t - t_mark;
            t_mark = t;
        }

        // ---------------- forward ----------------
        long long es = 0, cs = 0, ics = 0, es_prev = 0;
        int L = 0;
        long long total = 0;
        for (;;) {
            // the level's entries and chunks, counted in one word by append_queue
            const unsigned long long pk = ld_vol(&p.lev_grab[4 * ((long long)p.maxlev + 2) + L]);
            const long long ecnt = (long long)(pk & 0xffffffffull);
            const long long ccnt = (long long)(pk >> 32);
            const long long iccnt = (long long)ld_vol(&p.lev_grab[2 * ((long long)p.maxlev + 2) + L]);
            const long long es1 = es + ecnt, cs1 = cs + ccnt, ics1 = ics + iccnt;
            if (leader) {
                p.lev_cnt[L] = (unsigned long long)ecnt;  // published for the passes after the forward
                p.lev_start[L] = es;
                p.lev_start[L + 1] = es1;
                p.lev_icstart[L] = ics;
                p.lev_icstart[L + 1] = ics1;
            }
            if (L >= 1) {
                // the last threads first: on a thin level the first warps push
                const int nxt = 1 + ((L + 1) & 1);
                for (long long e = es_prev + (nthr - 1 - gthr); e < es; e += nthr) {
                    const int v = p.hv[e];
                    uint64_t *row = p.vs + (size_t)v * p.vs_stride;
#pragma unroll
                    for (int w = 0; w < W; ++w)
                        atomicAnd((unsigned long long *)&row[nxt * W + w], ~(unsigned long long)p.hm[e * W + w]);
                }
            }
            // direction of level L: bottom-up when its frontier's out-arcs
            // reach the threshold (the same counter in every block)
            const bool pull = MODE != kModeReach && L >= 1 && p.pull_arcs_min > 0 &&
                              (long long)ld_vol(&p.lev_grab[3 * ((long long)p.maxlev + 2) + L]) >= p.pull_arcs_min;
            if (lane == 0) {
                warp_buf<W>().first = cs;
                warp_buf<W>().ends = LevelEnds{es1, cs1, ics1};
            }
            __syncwarp();
            if (pull) {
                pull_level<W, MODE, T>(L, s_valid, nwarps);
                if (leader) atomicAdd(&p.ctr->pull_levels, 1ull);
            } else {
                push_masks<W, MODE, kPushU>(L, ccnt, gwarp, nwarps);
            }
            if (!team_barrier(p, bar)) return;
            total = es1;
            const long long enext =
                (long long)(ld_vol(&p.lev_grab[4 * ((long long)p.maxlev + 2) + L + 1]) & 0xffffffffull);
            if (enext == 0) break;
            if (L + 2 > p.maxlev) {
                if (threadIdx.x == 0) set_err(p.ctr, kDevLevelOverflow);
                return;
            }
            if (MODE != kModeReach) {
                if (pull)
                    enter_level<W>(p, L + 1, es1, enext, gthr, nthr);
                else if constexpr (MODE != kModeReach)
                    gather_level<W, T, kGatherU>(
                        L + 1, ics1, (long long)ld_vol(&p.lev_grab[2 * ((long long)p.maxlev + 2) + L + 1]), gwarp,
                        nwarps);
                if (!team_barrier(p, bar)) return;
            }
            es_prev = es;
            es = es1;
            cs = cs1;
            ics = ics1;
            ++L;
        }
        const int Lmax = L;
        if (timer) {
            const unsigned long long t = global_ns();
            ns_fwd += t - t_mark;
            t_mark = t;
        }
        if (leader) atomicMax(&p.ctr->levels_max, (unsigned long long)Lmax);

        bool skipped = false;  // a scan on trial that was not made
        // the scan over several query vertices takes the warps' buffers
        if (MODE == kModeScan) flush_stats(p.ctr, warp_buf<W>().st[lane], lane);

        // ---------------- backward ----------------
        if (MODE == kModeScan && (p.flags & kFlagRootOut)) {
            // the query vertices' own traversal (source slot c = column c):
            // keep d(r_c, t) and sigma_{r_c t}
            for (int Lr = 0; Lr <= Lmax; ++Lr) {
                const long long eend = p.lev_start[Lr + 1];
                for (long long e = p.lev_start[Lr] + gthr; e < eend; e += nthr) {
                    const int v = p.hv[e];
                    if (p.ncols >= 2) {
                        uint64_t x = p.hm[(size_t)e * W];  // columns sit in the first mask word
                        while (x) {
                            const int c = __ffsll((long long)x) - 1;
                            x &= x - 1;
                            p.rlevq[(size_t)v * 64 + c] = Lr;
                            p.rsigq[(size_t)v * 64 + c] = (double)sigma[(size_t)v * S + c];
                        }
                    } else {
                        p.rlev[v] = Lr;
                        p.rsig[v] = (double)sigma[(size_t)v * S];
                    }
                }
            }
            if (!team_barrier(p, bar)) return;
        } else if (MODE == kModeScan && !(p.flags & kFlagNoBackward)) {
            if (p.flags & kFlagTrial) {
                // a lone tile on trial: its terms are counted first, and when they
                // are too many the tile is left to the Eq. 4 pass
                scan_count<W>(Lmax, gthr, nthr);
                if (!team_barrier(p, bar)) return;
                if (scan_too_long(ld_vol(&p.ctr->trial_pairs), ld_vol(&p.ctr->tight))) {
                    if (leader) p.ctr->scan_skipped = 1ull;
                    skipped = true;
                }
            }
            if (skipped)
                ;
            else if (p.ncols >= 2)
                vertex_scan_multi<W, T>(Lmax, gwarp, nwarps);
            else
                vertex_scan<W, T>(p, Lmax, s_need, gwarp, nwarps);
            if (!team_barrier(p, bar)) return;
        }
        if (MODE == kModeSpd && !(p.flags & kFlagNoBackward)) {
            if (threadIdx.x == 0) s_lstop = 0x7fffffff;
            __syncthreads();
            for (int s = threadIdx.x; s < S; s += blockDim.x) {
                int mq = 0x7fffffff;
                if (tsrc[s] >= 0) {
                    if (p.flags & kFlagFullBackward) {
                        mq = 0;
                    } else {
                        uint64_t x = s_need[s];
                        while (x) {
                            const int q = __ffsll((long long)x) - 1;
                            x &= x - 1;
                            const int lv = p.qlevel[s * 64 + q];
                            if (lv >= 0 && lv < mq) mq = lv;
                        }
                    }
                }
                s_minql[s] = mq;
                atomicMin(&s_lstop, mq);
            }
            __syncthreads();
            const int lstop = s_lstop;
            if (lstop <= Lmax) {
                // the parity slot of level Lmax - 1 is empty after the forward pass
                if (Lmax - 1 >= lstop) {
                    const int slot = 1 + ((Lmax - 1) & 1);
                    const long long g0 = p.lev_start[Lmax - 1], g1 = g0 + (long long)p.lev_cnt[Lmax - 1];
                    for (long long e = g0 + gthr; e < g1; e += nthr) {
                        uint64_t *row = p.vs + (size_t)p.hv[e] * p.vs_stride;
#pragma unroll
                        for (int w = 0; w < W; ++w)
                            atomicOr((unsigned long long *)&row[slot * W + w], (unsigned long long)p.hm[e * W + w]);
                    }
                    if (!team_barrier(p, bar)) return;
                }
                for (int Lb = Lmax; Lb >= lstop; --Lb) {
                    if (threadIdx.x < W) {
                        uint64_t a = 0, an = 0;
                        for (int b = 0; b < 64; ++b) {
                            const int mq = s_minql[threadIdx.x * 64 + b];
                            if (mq <= Lb) a |= 1ull << b;
                            if (mq <= Lb - 1) an |= 1ull << b;
                        }
                        s_active[threadIdx.x] = a;
                        s_active_next[threadIdx.x] = an;
                    }
                    __syncthreads();
                    const bool more = Lb > lstop;
                    level_outputs<W, T>(p, Lb, more, more && Lb - 2 >= lstop, s_active, s_need, gthr, nthr);
                    if (more) {
                        const long long ics = p.lev_icstart[Lb];
                        const long long ic = (long long)ld_vol(&p.lev_grab[2 * ((long long)p.maxlev + 2) + Lb]);
                        push_level<W, T>(p, Lb, ics, ic, s_active_next, s_inv, nwarps);
                    }
                    if (!team_barrier(p, bar)) return;
                }
            }
        }
        if (timer) {
            const unsigned long long t = global_ns();
            ns_bwd += t - t_mark;
            t_mark = t;
        }

        if (MODE == kModeSpd) flush_stats(p.ctr, warp_buf<W>().st[lane], lane);

        // ---------------- tile end ----------------
        if (MODE == kModeScan && block == 0 && !skipped) {
            // one sum per source (one query vertex) or per (source, column)
            for (int s = threadIdx.x; s < S; s += blockDim.x) {
                uint64_t x = s_need[s];
                const double d = p.vsum[s];
                while (x) {
                    const int q = __ffsll((long long)x) - 1;
                    x &= x - 1;
                    p.dep[s * 64 + q] = p.ncols >= 2 ? p.msum[s * 64 + p.qcol[q]] : d;
                }
            }
            __syncthreads();
        }
        if (MODE != kModeReach && block == 0 && !skipped) tile_query_sums(p, tile, S, tsrc, s_need);
        if (MODE == kModeReach) {
            for (long long e = gthr; e < total; e += nthr)
                atomicOr((unsigned long long *)&p.rvmask[p.hv[e]], (unsigned long long)p.hm[e * W]);
        }
        if (!(p.flags & kFlagNoReset)) {
            if (MODE != kModeReach) {
                // sigma rows of more than one in-arc chunk meet in atomic adds
                // and start from zero; the others are overwritten when reached
                for (long long b = 32 * gwarp; b < total; b += 32 * nwarps) {
                    const long long e = b + lane;
                    const int v = e < total ? p.hv[e] : -1;
                    unsigned lg = __ballot_sync(kFull, v >= 0 && p.roff[v + 1] - p.roff[v] > p.chunk_arcs);
                    if (MODE == kModeSpd) lg = __ballot_sync(kFull, v >= 0);
                    while (lg) {
                        const int i = __ffs(lg) - 1;
                        lg &= lg - 1;
                        const int vi = __shfl_sync(kFull, v, i);
                        T *row = sigma + (size_t)vi * S;
                        double *arow = p.acc + (size_t)vi * S;
                        uint64_t F[W];
#pragma unroll
                        for (int w = 0; w < W; ++w) F[w] = p.hm[(b + i) * W + w];
#pragma unroll
                        for (int ii = 0; ii < 2 * W; ++ii) {
                            const int s = lane + 32 * ii;
                            if (mask_bit<W>(F, s)) {
                                row[s] = T(0);
                                if (MODE == kModeSpd) arow[s] = 0.0;
                            }
                        }
                    }
                }
            }
            const int half = p.vs_stride / 2;  // 16-byte pieces of a vertex's masks
            for (long long i = gthr; i < total * half; i += nthr) {
                const long long e = i / half;
                const int k = (int)(i - e * half);
                const int v = p.hv[e];
                reinterpret_cast<ulonglong2 *>(p.vs + (size_t)v * p.vs_stride)[k] = make_ulonglong2(0ull, 0ull);
                if (k == 0) p.tag[v] = -1;
            }
            if (block == 0) {
                for (int l = threadIdx.x; l <= Lmax + 1; l += blockDim.x) {
                    p.lev_cnt[l] = 0ull;
                    p.lev_grab[l] = 0ull;
                    p.lev_grab[p.maxlev + 2 + l] = 0ull;
                    p.lev_grab[2 * (p.maxlev + 2) + l] = 0ull;
                    p.lev_grab[3 * (p.maxlev + 2) + l] = 0ull;
                    p.lev_grab[4 * (p.maxlev + 2) + l] = 0ull;
                    p.lev_grab[5 * (p.maxlev + 2) + l] = 0ull;
                }
            }
        }
        if (leader) *(volatile unsigned long long *)&p.bar->next = p.nteams + atomicAdd(&p.ctr->tiles_taken, 1ull);
        if (!team_barrier(p, bar)) return;
        if (timer) {
            const unsigned long long t = global_ns();
            ns_other += t - t_mark;
            t_mark = t;
        }
    }

    if (timer) {
        p.ctr->ns_fwd += ns_fwd;
        p.ctr->ns_bwd += ns_bwd;
        p.ctr->ns_other += ns_other;
    }
}

template <int W, int MODE, int MINB, typename T>
bc_status launch(bc_graph *g, TravParams &p) {
    auto kern = trav_kernel<W, MODE, MINB, T>;
    const int threads = g->block_threads;
    if (threads < 64 * W) return set_error(BC_E_INVALID_ARG, "block_threads must be at least 64 * tile_words");
    size_t smem = sizeof(WarpBuf<W>) * (size_t)(threads / 32);
    if (MODE == kModeScan) smem = std::max(smem, std::max(sizeof(ScanBuf<W>), sizeof(CountBuf<W>)));
    smem += kParamBytes + 512 * W;
    int per_sm = 0;
    BCD_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    BCD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
    if (per_sm < 1) return set_error(BC_E_INTERNAL, "traversal kernel cannot be resident");
    // reach traversals of small graphs: blocks without work would only lengthen
    // the barriers
    int blocks = g->num_sms * per_sm;
    if (MODE == kModeReach) blocks = (int)std::max<int64_t>(std::min<int64_t>(blocks, 16), std::min<int64_t>(blocks, g->m / 2048));
    p.nteams = (int32_t)std::max<int64_t>(1, std::min<int64_t>(std::min(g->ws.teams, blocks), p.ntiles));
    p.team_blocks = blocks / p.nteams;
    dim3 grid((unsigned)(p.nteams * p.team_blocks)), block((unsigned)threads);
    void *args[] = {(void *)&p};
    BCD_CUDA(cudaLaunchCooperativeKernel((const void *)kern, grid, block, args, smem, g->stream));
    g->launches += 1;
    g->last_grid = (int)grid.x;
    return BC_OK;
}

// Launch with path counts as 32-bit integers, or in fp64 once a launch of
// this graph met a count of 2^26 (rare: the fp64 kernels come at one
// occupancy each).
template <int MODE>
bc_status launch_counts(bc_graph *g, int W, TravParams &p) {
    const int b = g->blocks_per_sm;
    if (g->ws.swide) {
        switch (W) {
            case 1: return launch<1, MODE, 2, double>(g, p);
            case 2: return launch<2, MODE, 2, double>(g, p);
            case 4: return launch<4, MODE, 1, double>(g, p);
            case 8: return launch<8, MODE, 1, double>(g, p);
        }
    } else {
        switch (W) {
            case 1: return launch<1, MODE, 2, uint32_t>(g, p);
            case 2: return b == 3 ? launch<2, MODE, 3, uint32_t>(g, p) : launch<2, MODE, 2, uint32_t>(g, p);
            case 4: return b == 2 ? launch<4, MODE, 2, uint32_t>(g, p) : launch<4, MODE, 1, uint32_t>(g, p);
            case 8: return launch<8, MODE, 1, uint32_t>(g, p);
        }
    }
    return set_error(BC_E_INVALID_ARG, "tile words must be 1, 2, 4 or 8");
}

// The state slabs of an unweighted launch. The sigma slab starts with the rows
// of several in-arc chunks zero: the row width, the count type and chunk_arcs
// decide which rows these are and where they lie, so a change of any of them
// clears the slab (and fp64 counts need a larger one). The accumulators of
// Eq. 4 start zero.
bc_status prepare_slabs(bc_graph *g, int W, bool eq4) {
    bcd_workspace &ws = g->ws;
    const size_t pairs = (size_t)ws.teams * (size_t)ws.n * 64 * (size_t)ws.W;
    const size_t bytes = ws.swide ? sizeof(double) : sizeof(uint32_t);
    if (!ws.sigma || ws.sigma_bytes < bytes) {
        dev_free(ws.sigma);
        ws.sigma_key = -1;
        ws.sigma_zero = false;
        const bc_status st = dev_alloc(&ws.sigma, pairs * bytes / sizeof(double));
        if (st != BC_OK) {
            free_workspace(g);
            return st;
        }
        ws.sigma_bytes = bytes;
    }
    const int64_t key = ((int64_t)g->chunk_arcs << 8) | (int64_t)(W << 1) | (ws.swide ? 1 : 0);
    if (ws.sigma_key != key && !ws.sigma_zero)
        BCD_CUDA(cudaMemsetAsync(ws.sigma, 0, ws.sigma_bytes * pairs, g->stream));
    ws.sigma_key = key;
    ws.sigma_zero = false;
    if (eq4 && !ws.acc) {
        const bc_status st = dev_alloc(&ws.acc, pairs);
        if (st != BC_OK) {
            free_workspace(g);
            return st;
        }
        BCD_CUDA(cudaMemsetAsync(ws.acc, 0, sizeof(double) * pairs, g->stream));
    }
    return BC_OK;
}

}  // namespace

bc_status reset_dense_state(bc_graph *g) {
    bcd_workspace &ws = g->ws;
    if (!ws.vs) return BC_OK;  // no workspace (never built, or freed after a failure)
    const size_t t = (size_t)ws.teams, n = (size_t)ws.n, lev = (size_t)(ws.maxlev + 2);
    BCD_CUDA(cudaMemsetAsync(ws.vs, 0, sizeof(uint64_t) * t * n * ws.vs_stride, g->stream));
    BCD_CUDA(cudaMemsetAsync(ws.tag, 0xff, sizeof(int32_t) * t * n, g->stream));
    if (ws.sigma) {
        BCD_CUDA(cudaMemsetAsync(ws.sigma, 0, ws.sigma_bytes * t * n * 64 * ws.W, g->stream));
        ws.sigma_zero = true;
    }
    BCD_CUDA(cudaMemsetAsync(ws.lev_cnt, 0, sizeof(unsigned long long) * t * lev, g->stream));
    BCD_CUDA(cudaMemsetAsync(ws.lev_grab, 0, sizeof(unsigned long long) * t * 6 * lev, g->stream));
    BCD_CUDA(cudaMemsetAsync(ws.pdone, 0, sizeof(int32_t) * (size_t)(g->weighted ? ws.pcap : 1), g->stream));
    if (ws.acc) BCD_CUDA(cudaMemsetAsync(ws.acc, 0, sizeof(double) * t * n * 64 * ws.W, g->stream));
    if (ws.dist) {
        BCD_CUDA(cudaMemsetAsync(ws.dist, 0xff, sizeof(uint64_t) * (size_t)ws.n * 64 * ws.W, g->stream));
        BCD_CUDA(cudaMemsetAsync(ws.bcount, 0, sizeof(unsigned long long) * 3 * (size_t)ws.ring, g->stream));
    }
    return BC_OK;
}

// Reruns after an overflow have no count of their own: each one enlarges what
// was full, up to a limit at which the growing function returns BC_E_OOM, or
// takes the one step to fp64 counts. (A tile of 256 sources on a path doubles
// its history five times, and may meet a wide count besides.)
bc_status run_traversal(bc_graph *g, int W, TravParams &p, int *levels_out, unsigned long long *edges_out) {
    for (;;) {
        bcd_workspace &ws = g->ws;
        if (!g->weighted && p.mode != kModeReach) BCD_TRY(prepare_slabs(g, W, p.mode == kModeSpd));
        p.vs = ws.vs;
        p.vs_stride = ws.vs_stride;
        p.tag = ws.tag;
        p.sigma = ws.sigma;
        p.acc = ws.acc;
        p.inv = ws.inv;
        p.roff = g->d_roff;  // R(G): in-arcs for the backward push and the weighted sigma pull
        p.rcol = g->d_rcol;
        p.hv = ws.hv;
        p.hm = ws.hm;
        p.hcap = p.mode == kModeReach ? ws.hmcap : ws.hcap;
        p.hm_words = ws.hcap * ws.W;
        p.ws_slots = 64 * ws.W;
        p.bar = reinterpret_cast<TeamBar *>(reinterpret_cast<char *>(ws.ctr) + kCounterBytes);
        p.nteams = 1;
        p.team_blocks = 1;
        p.chunks = ws.chunks;
        p.ichunks = ws.ichunks;
        p.ccap = ws.ccap;
        p.partial = ws.partial;
        p.pdone = ws.pdone;
        p.pcap = ws.pcap;
        p.lev_cnt = ws.lev_cnt;
        p.lev_grab = ws.lev_grab;
        p.lev_start = ws.lev_start;
        p.lev_icstart = ws.lev_icstart;
        p.maxlev = ws.maxlev;
        p.ctr = ws.ctr;
        p.n = g->n;
        p.chunk_arcs = g->chunk_arcs;
        p.timeout_ns = g->timeout_ns;
        p.cancel = g->cancel_d;
        p.pull_arcs_min = 0;
        if (!g->weighted && p.mode != kModeReach && g->pull_permille > 0) {
            BCD_TRY(ensure_pull_chunks(g));
            p.pchunks = ws.pchunks;
            p.npchunks = ws.npchunks;
            p.pull_arcs_min = std::max<int64_t>(1, (int64_t)((double)g->m * g->pull_permille / 1000.0));
        }
        // the counters and, behind them, the teams' barrier lines
        BCD_CUDA(cudaMemsetAsync(ws.ctr, 0, kCounterBytes + sizeof(TeamBar) * (size_t)ws.teams, g->stream));
        bc_status st = BC_E_INTERNAL;
        cudaEvent_t ev0 = nullptr, ev1 = nullptr;
        const bool timed = cudaEventCreate(&ev0) == cudaSuccess && cudaEventCreate(&ev1) == cudaSuccess;
        if (timed) cudaEventRecord(ev0, g->stream);
        if (p.mode == kModeReach) {
            if (W != 1) return set_error(BC_E_INTERNAL, "reach traversal runs with one mask word");
            st = launch<1, kModeReach, 2, uint32_t>(g, p);
        } else if (g->weighted) {
            p.wt = g->d_w;
            p.roff = g->d_roff;
            p.rcol = g->d_rcol;
            p.rwt = g->d_rw;
            if (W < 1 || W > 16 || (W & (W - 1)) || W > ws.W || ((uint64_t)g->n << 6) * (uint64_t)W > (1ull << 32))
                return set_error(BC_E_INVALID_ARG, "weighted tiles: 1, 2, 4, 8 or 16 words, n * 64 * words <= 2^32");
            p.dist = ws.dist;
            p.hs = ws.hs;
            p.buckets = ws.buckets;
            p.bcount = ws.bcount;
            p.bcap = ws.bcap;
            p.ring = ws.ring;
            p.nw = W;
            p.wshort = g->wshort;
            p.lev_dist = ws.lev_dist;
            st = launch_weighted(g, p);
        } else {
            st = p.mode == kModeScan ? launch_counts<kModeScan>(g, W, p) : launch_counts<kModeSpd>(g, W, p);
        }
        if (timed) cudaEventRecord(ev1, g->stream);
        if (st != BC_OK) {
            if (timed) {
                cudaEventDestroy(ev0);
                cudaEventDestroy(ev1);
            }
            return st;
        }
        Counters c;
        BCD_CUDA(cudaMemcpyAsync(&c, ws.ctr, sizeof(Counters), cudaMemcpyDeviceToHost, g->stream));
        BCD_CUDA(cudaStreamSynchronize(g->stream));
        g->last_ms_launch = 0;
        if (timed) {
            cudaEventElapsedTime(&g->last_ms_launch, ev0, ev1);
            cudaEventDestroy(ev0);
            cudaEventDestroy(ev1);
        }
        if (c.err == kDevOk) {
            g->last = c;
            if (levels_out) *levels_out = (int)c.levels_max;
            if (edges_out) *edges_out = c.edges;
            g->last_ns_fwd = c.ns_fwd;
            g->last_ns_bwd = c.ns_bwd;
            g->last_ns_other = c.ns_other;
            return BC_OK;
        }
        if (c.err == kDevTimeout) {
            reset_dense_state(g);
            return set_error(BC_E_TIMEOUT, "traversal: a grid barrier wait timed out");
        }
        if (c.err == kDevCancelled) {
            reset_dense_state(g);
            return set_error(BC_E_CANCELLED, "traversal: cancelled by bc_cancel");
        }
        if (c.err == kDevWide) {
            // a path count of 2^26: fp64 counts from now on
            BCD_TRY(reset_dense_state(g));
            if (ws.swide) return set_error(BC_E_INTERNAL, "traversal: fp64 counts asked for a wider form");
            ws.swide = true;
            if (p.qflags) BCD_CUDA(cudaMemsetAsync(p.qflags, 0, sizeof(uint32_t) * 64, g->stream));
            continue;
        }
        if (c.err == kDevBucketOverflow) {
            // more pending pairs at one distance than a ring slot holds: grow and rerun
            BCD_TRY(grow_buckets(g));
            BCD_TRY(reset_dense_state(g));
            if (p.qflags) BCD_CUDA(cudaMemsetAsync(p.qflags, 0, sizeof(uint32_t) * 64, g->stream));
            continue;
        }
        if (c.err == kDevLevelOverflow) {
            // more non-empty levels than the arrays hold (integer weights): grow and rerun
            BCD_TRY(grow_levels(g));
            BCD_TRY(reset_dense_state(g));
            if (p.qflags) BCD_CUDA(cudaMemsetAsync(p.qflags, 0, sizeof(uint32_t) * 64, g->stream));
            continue;
        }
        // capacity overflow: grow the level history and retry from a clean state
        BCD_TRY(grow_history(g));
        BCD_TRY(reset_dense_state(g));
        if (p.mode == kModeReach && p.rvmask)
            BCD_CUDA(cudaMemsetAsync(p.rvmask, 0, sizeof(uint64_t) * (size_t)g->n, g->stream));
        if (p.qflags) BCD_CUDA(cudaMemsetAsync(p.qflags, 0, sizeof(uint32_t) * 64, g->stream));
    }
}

}  // namespace bcd
