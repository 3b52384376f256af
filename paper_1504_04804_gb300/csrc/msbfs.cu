// Multi-source BFS: up to 64 sources share one traversal and one edge stream.
//
// Every vertex carries 64-bit lane masks: seen[v] (lanes that have labelled
// v) and cur_L[v] (lanes whose level-L frontier holds v).  Lane b's result
// equals a single-source BFS from srcs[b] (Algorithm 1); the lanes only share
// the reading of the graph.  Levels are direction-optimised on lane counts
// (Sec. 6.1 with FV = the frontier's edge count and BV = (unseen
// vertex-lane pairs) * V / (seen pairs)).
//
//  * Push level (sparse frontier): the frontier queue's edges are cut into
//    equal warp tiles (the degree prefix is stored with every queue slot).
//    For edge (u, v) the lanes cur[u] & ~seen[v] are OR-ed into next[v]; the
//    first warp to touch v lists it (large levels instead mark v in a
//    touched bitmap with reductions only, which warps owning 32-word chunks
//    scan).  A finalize phase turns each touched vertex's next mask into its
//    new lanes, labels them (scattered depth writes: few), and appends the
//    vertex to the next queue.
//  * Pull level (dense frontier): warps take the non-isolated vertices 128 at a
//    time and gather cur[u] over a row only until every lane the row misses is
//    found (edge skipping, for all lanes at once): its first two neighbours
//    (first2), a lane per row, and its first ten on graphs of few edges a
//    vertex; then eight lanes per row, 32 edges a step.  Rows
//    still open after MS_HEAD edges leave the rest to a second phase, in pieces
//    of 1,024 edges over the grid, and are finished by a third.
//  * Depths found by pull levels and large push levels are not written per level:
//    the level's new lane masks go to one of MS_HSLOTS history slots, and a flush pass
//    writes them lane-major with coalesced stores (and, at the end, -1 for
//    every pair never reached, so the output needs no initial fill).
//  * cur rotates through three buffers: level L reads cur[L%3] and writes
//    cur[(L+1)%3], only for vertices with new lanes; nothing is cleared.  A
//    stale entry holds lanes that reached the vertex at depth L-3 or less,
//    so every neighbour already has them and they cannot label anything: a
//    pull ANDs the gathered lanes with the row's missing lanes, and a push
//    reads cur only for queue entries, which the previous level wrote.  The
//    queue of a push after a pull comes from the pull's history slot.
//  * 128 rows that have every lane seen stay so: they are flagged and skipped by
//    later pull levels.
//  * One cooperative persistent kernel; levels and their phases are
//    separated by the bounded flag barrier.
#include <cstring>

#include "grx_internal.cuh"

namespace {

constexpr int MS_BLOCK = 384;
constexpr int MS_WARPS = MS_BLOCK / 32;
constexpr int MS_ITEMS = 8;
constexpr int MS_WTILE = 32 * MS_ITEMS;             // push: edges per warp tile
constexpr int MS_ROWS = 128;                        // pull: rows a warp takes at a time, at most
// Pull: edges of a row in the first phase, after its first two (64 sources, R-MAT
// 24 / 22 / 20: 30 7.58 / 2.27 / 0.82 ms, 126 7.02 / 2.16 / 0.89, 254 7.12 / 2.30 /
// 0.98, 510 7.37 / 2.57 / 1.16).
constexpr uint32_t MS_HEAD = 126;
// Pull, fewer than eight edges a vertex: edges of a row that a lane takes, its rows'
// loads in flight together.  Eight lanes a row have little to do there (uniform random,
// 2M vertices of degree 4, 64 sources: a level that reads every edge 154 us, by edge
// tiles 101, so 63; the traversal 2,044 -> 1,529 us).
constexpr uint32_t MS_LANE_HEAD = 10;
constexpr uint32_t MS_WARP_ROW = 2048;              // pull, small graphs: rows up to this stay in the first phase
constexpr uint32_t MS_PIECE = 1024;                 // pull: edges of a piece of the second phase
constexpr int MS_HSLOTS = 6;                        // history slots of pull levels
constexpr int MS_MIN_BLOCKS = 2;                    // resident blocks per SM (register cap; two of 384 threads
                                                    // against three of 256: 1 % at R-MAT 20 to 24)

enum { DIR_PUSH = 0, DIR_PULL = 1 };
enum { MOP_COMPACT, MOP_EXPAND, MOP_FINAL, MOP_FLUSH, MOP_PULL, MOP_REST, MOP_FIXUP };

template <typename OffT>
struct MsArgs {
    int32_t nv;
    int64_t ne;
    const OffT *ro;
    const int32_t *col;
    const int32_t *active;
    const uint32_t *aoff;
    const int2 *first2;               // first two neighbours of every vertex (-1: none)
    int64_t n_active;
    int n;
    unsigned long long lanes;         // active lane mask
    int32_t src[64];
    unsigned long long *seen;
    unsigned long long *next;         // push: lane OR per touched vertex; pull: OR of rows in pieces
    unsigned long long *cur[3];
    unsigned long long *hist[MS_HSLOTS];
    int2 *rest;                       // pieces of open rows: (active row, piece)
    int rows;                         // pull: rows a warp takes at a time
    int few;                          // pull: few edges a vertex
    uint8_t *sat;                     // per `rows` rows: every one has all lanes seen
    int32_t *Q[3];
    uint32_t *E[3];
    OffT *R[3];
    int32_t *touched;
    uint32_t *tbits;                  // bitmap push: touched vertices, [ceil(nv/32)]
    int64_t words;
    uint32_t bmp_min_T;               // push levels with at least this many edges use tbits
    int32_t *depth;                   // [n][nv]
    TravCtl *ctl;
    unsigned int *bar_flags;
    DevStats *stats;
    int mode;
    float alpha, beta;
    unsigned long long timeout_ns;
};

struct MsState {
    int L;
    uint8_t dir, switched, back, done, phase;
    uint8_t qin;        // Q_L exists as a queue
    uint8_t compact;    // push level whose queue is first built from cur_L
    uint8_t hslots;     // history slots holding pull levels' masks
    uint8_t flush;      // this pull level starts with a flush (slots full)
    uint8_t bmp;        // push level that marks touched vertices in a bitmap
    uint8_t keep;       // push level whose new lanes go to a history slot
    uint8_t flushed;    // a flush came before
    int32_t slot_depth[MS_HSLOTS];
    uint32_t q, T;      // |Q_L| and its edge count
    unsigned long long seen_pairs;    // (vertex, lane) pairs labelled so far
};

template <typename OffT>
union MsWarpSmem {
    struct {
        uint32_t qe[MS_WTILE + 2];
        OffT rs[MS_WTILE + 1];
        unsigned long long cm[MS_WTILE + 1];
    };
    uint16_t list[32 * 32];           // bitmap finalize: set bits of a 32-word chunk
};

// A warp's open rows: first edge, degree, active row, vertex; lanes missing, found.
struct MsPullSmem {
    uint32_t s[MS_ROWS], deg[MS_ROWS];
    int32_t i[MS_ROWS], v[MS_ROWS];
    unsigned long long miss[MS_ROWS], acc[MS_ROWS];
};

template <typename OffT>
union MsSmem {
    MsWarpSmem<OffT> w[MS_WARPS];
    MsPullSmem p[MS_WARPS];
};

template <typename T>
__device__ __forceinline__ T pk3(T a, T b, T c, int i) { return i == 0 ? a : (i == 1 ? b : c); }

__device__ __forceinline__ int ms_phases(const MsState &s) {
    return s.dir == DIR_PUSH ? 2 + s.compact : 3 + s.flush;
}

__device__ __forceinline__ int ms_op(const MsState &s) {
    if (s.dir == DIR_PUSH) {
        const int p = (int)s.phase - (int)s.compact;
        return p < 0 ? MOP_COMPACT : (p == 0 ? MOP_EXPAND : MOP_FINAL);
    }
    const int p = (int)s.phase - (int)s.flush;
    return p < 0 ? MOP_FLUSH : MOP_PULL + p;
}

template <typename OffT>
__device__ __forceinline__ void ms_set_kind(const MsArgs<OffT> &a, MsState &s) {
    s.compact = s.dir == DIR_PUSH && !s.qin;
    s.flush = s.dir == DIR_PULL && s.hslots >= MS_HSLOTS;
    s.bmp = s.dir == DIR_PUSH && s.T >= a.bmp_min_T;
    s.keep = s.bmp && !s.back && s.hslots < MS_HSLOTS;   // after the pulls little is found
}

// Label the new lanes of v at depth d in the lane-major depth output.
__device__ __forceinline__ void write_depths(int32_t *depth, int32_t nv, int32_t v,
                                             unsigned long long nw, int32_t d) {
    while (nw) {
        const int b = __ffsll((long long)nw) - 1;
        nw &= nw - 1;
        depth[(int64_t)b * nv + v] = d;
    }
}

template <typename OffT>
__device__ MsState ms_next_state(const MsArgs<OffT> &a, const MsState &st, bool stats) {
    MsState ns = st;
    // a pull that left no pieces is over after its first phase
    const bool over = ms_op(st) == MOP_PULL && ld_relaxed_u32(&a.ctl->ucount[(st.L + 1) & 3]) == 0u;
    if ((int)st.phase + 1 < ms_phases(st) && !over) {
        ns.phase = st.phase + 1;
        return ns;
    }
    ns.L = st.L + 1;
    ns.phase = 0;
    const unsigned long long pk = ld_relaxed_u64(&a.ctl->qpack[(st.L + 1) & 3]);
    ns.q = (uint32_t)(pk >> 32);
    ns.T = (uint32_t)pk;
    ns.qin = st.dir == DIR_PUSH;
    ns.flushed |= st.flush;
    if (st.dir == DIR_PULL || st.keep) {
        const int h = st.flush ? 0 : st.hslots;
        ns.slot_depth[h] = st.L + 1;
        ns.hslots = (uint8_t)(h + 1);
    }
    const unsigned long long found = ld_relaxed_u64(&a.ctl->pairs[(st.L + 1) & 3]);
    ns.seen_pairs = st.seen_pairs + found;
    if (stats && blockIdx.x == 0 && st.L < GRX_MAX_LEVELS_STATS) a.stats->discovered[st.L] = found;
    if (ns.q == 0) {
        ns.done = 1;
        return ns;
    }
    if (a.mode == GRX_DIR_PUSH) {
        ns.dir = DIR_PUSH;
    } else if (a.mode == GRX_DIR_PULL) {
        ns.dir = DIR_PULL;
    } else {
        const double V = (double)a.nv;
        const double total = (double)a.n * V;
        const double FV = (double)ns.T;
        const double BV = (total - (double)ns.seen_pairs) * V / (double)ns.seen_pairs;
        if (st.dir == DIR_PUSH && !st.switched && FV > BV * (double)a.alpha) {
            ns.dir = DIR_PULL;
            ns.switched = 1;
        } else if (st.dir == DIR_PULL && FV < BV * (double)a.beta) {
            ns.dir = DIR_PUSH;
            ns.back = 1;
        }
    }
    ms_set_kind(a, ns);
    return ns;
}

// Phase 0: masks empty (history slots, the OR buffer and the touched bitmap
// are kept zero between traversals; after one that did not finish they are
// cleared here).
template <typename OffT>
__device__ void ms_init_fill(const MsArgs<OffT> &a, bool dirty) {
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = tid; v < a.nv; v += stride) {
        a.seen[v] = 0ull;
        a.cur[0][v] = 0ull;
        a.cur[1][v] = 0ull;
        a.cur[2][v] = 0ull;
        if (dirty) {
            a.next[v] = 0ull;
            for (int s = 0; s < MS_HSLOTS; ++s) a.hist[s][v] = 0ull;
        }
    }
    if (dirty)
        for (int64_t w = tid; w < a.words; w += stride) a.tbits[w] = 0u;
    for (int64_t t = tid; t < (a.n_active + a.rows - 1) / a.rows; t += stride) a.sat[t] = 0;
}

// Phase 1 (one thread): seed the lanes (depth 0), the first frontier
// (distinct sources with at least one edge) and the counters.
template <typename OffT>
__device__ void ms_seed(const MsArgs<OffT> &a) {
    uint32_t cnt = 0, edges = 0;
    for (int b = 0; b < a.n; ++b) {
        const int32_t v = a.src[b];
        const unsigned long long bit = 1ull << b;
        if (a.seen[v] == 0ull) {
            const OffT rb = a.ro[v];
            const uint32_t deg = (uint32_t)(a.ro[v + 1] - rb);
            if (deg) {
                a.Q[0][cnt] = v;
                a.E[0][cnt] = edges;
                a.R[0][cnt] = rb;
                ++cnt;
                edges += deg;
            }
        }
        a.seen[v] |= bit;
        a.cur[0][v] |= bit;
        a.depth[(int64_t)b * a.nv + v] = 0;
    }
    a.ctl->qpack[0] = ((unsigned long long)cnt << 32) | edges;
    for (int i = 1; i < 4; ++i) a.ctl->qpack[i] = 0ull;
    for (int i = 0; i < 4; ++i) a.ctl->pairs[i] = 0ull;
    a.ctl->ucount[1] = 0u;
    for (int i = 0; i < 4; ++i) a.ctl->wq[i] = 0u;
    a.ctl->cpack = 0ull;
    a.ctl->ms_grid = gridDim.x;
    a.ctl->ms_done = 0u;
}

// Push, phase 1: lanes of each frontier edge's source go to next[v] of the
// target where not yet seen; the first toucher lists v (or, on large levels,
// marks it in the touched bitmap).
template <typename OffT, bool STATS>
__device__ void ms_push_expand(const MsArgs<OffT> &a, const MsState &st, MsWarpSmem<OffT> &w) {
    const int L = st.L;
    const unsigned int lane = threadIdx.x & 31;
    const int32_t *Qv = pk3(a.Q[0], a.Q[1], a.Q[2], L % 3);
    const uint32_t *Qe = pk3(a.E[0], a.E[1], a.E[2], L % 3);
    const OffT *Qr = pk3(a.R[0], a.R[1], a.R[2], L % 3);
    const unsigned long long *cin = pk3(a.cur[0], a.cur[1], a.cur[2], L % 3);
    unsigned int *tctr = &a.ctl->ucount[(L + 1) & 3];
    const int64_t q = st.q;
    const uint64_t T = st.T;
    const uint64_t ntiles = (T + MS_WTILE - 1) / MS_WTILE;
    const uint64_t nwarps = (uint64_t)gridDim.x * MS_WARPS;
    const uint64_t gw = grx_warp();
    const uint64_t per = (ntiles + nwarps - 1) / nwarps;
    const uint64_t tb0 = gw * per;
    const uint64_t tb1 = min(ntiles, tb0 + per);
    if (tb0 >= tb1) return;
    int64_t i0 = warp_upper_index_cg(Qe, q, (uint32_t)(tb0 * MS_WTILE));
    for (uint64_t tile = tb0; tile < tb1; ++tile) {
        const uint64_t e0 = tile * MS_WTILE;
        const uint32_t e1 = (uint32_t)min(T, e0 + MS_WTILE);
        int n = 0;
        for (;;) {
            const int64_t idx = i0 + n + lane;
            uint32_t qe = 0xffffffffu;
            if (idx < q) qe = __ldcg(Qe + idx);
            const bool in = idx < q && qe < e1;
            if (n + (int)lane <= MS_WTILE + 1) w.qe[n + lane] = qe;
            if (in && n + (int)lane <= MS_WTILE) {
                w.rs[n + lane] = __ldcg(Qr + idx);
                w.cm[n + lane] = __ldcg(cin + __ldcg(Qv + idx)) & a.lanes;
            }
            const int cnt = __popc(__ballot_sync(GRX_FULL_MASK, in));
            n += cnt;
            if (cnt < 32) break;
            if (n > MS_WTILE) {
                if (lane == 0) grx_set_status(a.ctl, GRX_EINVAL);
                n = MS_WTILE;
                break;
            }
        }
        __syncwarp();
        const uint32_t next_start = w.qe[n];
        const uint64_t t0 = e0 + (uint64_t)lane * MS_ITEMS;
        int32_t v[MS_ITEMS];
        unsigned long long m[MS_ITEMS];
#pragma unroll
        for (int k = 0; k < MS_ITEMS; ++k) {
            v[k] = 0;
            m[k] = 0ull;
        }
        if (t0 < e1) {
            int j = upper_index_smem(w.qe, n, (uint32_t)t0);
#pragma unroll
            for (int k = 0; k < MS_ITEMS; ++k) {
                const uint32_t e = (uint32_t)t0 + k;
                if (e < e1) {
                    while (w.qe[j + 1] <= e) ++j;
                    v[k] = __ldg(a.col + w.rs[j] + (OffT)(e - w.qe[j]));
                    m[k] = w.cm[j];
                }
            }
        }
        unsigned long long sv[MS_ITEMS];
#pragma unroll
        for (int k = 0; k < MS_ITEMS; ++k) sv[k] = m[k] ? __ldcg(a.seen + v[k]) : ~0ull;
        if (st.bmp) {
            // reductions only: the touched bitmap lists the targets
#pragma unroll
            for (int k = 0; k < MS_ITEMS; ++k) {
                const unsigned long long mk = m[k] & ~sv[k];
                if (mk) {
                    atomicOr(a.next + v[k], mk);
                    atomicOr(a.tbits + (v[k] >> 5), 1u << (v[k] & 31));
                }
            }
        } else {
            uint32_t tmask = 0;
#pragma unroll
            for (int k = 0; k < MS_ITEMS; ++k) {
                const unsigned long long mk = m[k] & ~sv[k];
                if (mk && atomicOr(a.next + v[k], mk) == 0ull) tmask |= 1u << k;
            }
            warp_append_list_items<MS_ITEMS>(v, tmask, a.touched, tctr);
        }
        i0 = (next_start == e1) ? i0 + n : i0 + n - 1;
        __syncwarp();
    }
}

// A touched vertex v (or -1): its next mask becomes its new lanes (labelled
// here, or left in the history slot hs) and, with edges, a slot of the next
// frontier.  All 32 lanes call.
template <typename OffT>
__device__ __forceinline__ void ms_touched(const MsArgs<OffT> &a, int L, int32_t vv, unsigned long long *hs,
                                           unsigned long long *cout, int32_t *Qv_out,
                                           uint32_t *Qe_out, OffT *Qr_out, unsigned long long *ctr,
                                           unsigned long long &found) {
    int32_t v[1] = {vv < 0 ? 0 : vv};
    uint32_t deg[1] = {0};
    OffT rb[1] = {0};
    uint32_t app = 0;
    if (vv >= 0) {
        const unsigned long long nx = __ldcg(a.next + vv);
        a.next[vv] = 0ull;
        const unsigned long long sv = __ldcg(a.seen + vv);
        const unsigned long long nw = nx & ~sv & a.lanes;
        if (nw) {
            a.seen[vv] = sv | nw;
            cout[vv] = nw;
            if (hs) hs[vv] = nw;
            else write_depths(a.depth, a.nv, vv, nw, L + 1);
            found += (unsigned long long)__popcll(nw);
            rb[0] = __ldg(a.ro + vv);
            deg[0] = (uint32_t)(__ldg(a.ro + vv + 1) - rb[0]);
            if (deg[0]) app = 1;
        }
    }
    warp_append_items<1, OffT>(v, deg, rb, app, Qv_out, Qe_out, Qr_out, ctr);
}

// Push, phase 2: the touched vertices (from the list, or from the bitmap by
// warps that own 32-word chunks of it, clearing it) become the next frontier.
template <typename OffT>
__device__ void ms_push_finalize(const MsArgs<OffT> &a, const MsState &st, uint16_t *list) {
    const int L = st.L;
    unsigned long long *cout = pk3(a.cur[0], a.cur[1], a.cur[2], (L + 1) % 3);
    int32_t *Qv_out = pk3(a.Q[0], a.Q[1], a.Q[2], (L + 1) % 3);
    uint32_t *Qe_out = pk3(a.E[0], a.E[1], a.E[2], (L + 1) % 3);
    OffT *Qr_out = pk3(a.R[0], a.R[1], a.R[2], (L + 1) % 3);
    unsigned long long *ctr = &a.ctl->qpack[(L + 1) & 3];
    unsigned long long *hs = st.keep ? a.hist[st.hslots] : nullptr;
    unsigned long long found = 0;
    if (st.bmp) {
        const unsigned int lane = threadIdx.x & 31;
        const int64_t nsc = (a.words + 31) / 32;
        const int64_t nwarps = (int64_t)gridDim.x * MS_WARPS;
        for (int64_t sc = grx_warp(); sc < nsc; sc += nwarps) {
            const int64_t wd = sc * 32 + lane;
            const uint32_t bits = wd < a.words ? __ldcg(a.tbits + wd) : 0u;
            if (bits) a.tbits[wd] = 0u;
            const int n = warp_compact_bits(bits, list);
            for (int base = 0; base < n; base += 32) {
                const int i = base + (int)lane;
                ms_touched<OffT>(a, L, i < n ? (int32_t)(sc * 1024 + list[i]) : -1, hs, cout, Qv_out, Qe_out,
                                 Qr_out, ctr, found);
            }
            __syncwarp();
        }
    } else {
        const int64_t count = ld_relaxed_u32(&a.ctl->ucount[(L + 1) & 3]);
        const int64_t span = (count + 31) & ~(int64_t)31;
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < span;
             i += (int64_t)gridDim.x * blockDim.x)
            ms_touched<OffT>(a, L, i < count ? __ldcg(a.touched + i) : -1, hs, cout, Qv_out, Qe_out, Qr_out,
                             ctr, found);
    }
    found = warp_sum(found);
    if ((threadIdx.x & 31) == 0 && found) atomicAdd(&a.ctl->pairs[(L + 1) & 3], found);
}

// Push after a pull level: Q_L (vertex, edge prefix, row start) from the
// vertices that got new lanes in level L-1 -- exactly the nonzero entries of
// that level's history slot -- through the compaction counter.
template <typename OffT>
__device__ void ms_compact(const MsArgs<OffT> &a, const MsState &st) {
    const int L = st.L;
    const unsigned long long *cin = a.hist[st.hslots - 1];
    int32_t *Qv = pk3(a.Q[0], a.Q[1], a.Q[2], L % 3);
    uint32_t *Qe = pk3(a.E[0], a.E[1], a.E[2], L % 3);
    OffT *Qr = pk3(a.R[0], a.R[1], a.R[2], L % 3);
    const int64_t span = ((int64_t)a.nv + 31) & ~(int64_t)31;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < span;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t v[1] = {(int32_t)i};
        uint32_t deg[1] = {0};
        OffT rb[1] = {0};
        uint32_t app = 0;
        if (i < a.nv && __ldcg(cin + i) != 0ull) {
            rb[0] = __ldg(a.ro + i);
            deg[0] = (uint32_t)(__ldg(a.ro + i + 1) - rb[0]);
            app = deg[0] ? 1u : 0u;
        }
        warp_append_items<1, OffT>(v, deg, rb, app, Qv, Qe, Qr, &a.ctl->cpack);
    }
}

// Per-thread counters of the next frontier found by a pull level.
struct MsCounts {
    unsigned long long q, T, pairs, gathered, rows;
};

// A pull-level row v gets its new lanes nw: seen, the history slot and the
// frontier counters (its depth is written by the next flush).
__device__ __forceinline__ void ms_pull_finish(unsigned long long *seen, unsigned long long *hs,
                                               int32_t v, unsigned long long old_seen,
                                               unsigned long long nw, uint32_t deg, MsCounts &c) {
    seen[v] = old_seen | nw;
    hs[v] = nw;
    c.q += 1;
    c.T += deg;
    c.pairs += (unsigned long long)__popcll(nw);
}

// OR of the masks of up to 256 neighbours (edges at to e1), by a whole warp.
template <bool STATS>
__device__ __forceinline__ unsigned long long ms_gather256(const int32_t *col, const unsigned long long *cin,
                                                           int64_t at, int64_t e1, MsCounts &c) {
    const unsigned int lane = threadIdx.x & 31;
    int32_t u[8];
    unsigned long long x = 0ull;
#pragma unroll
    for (int j = 0; j < 8; ++j) u[j] = at + j * 32 + lane < e1 ? __ldg(col + at + j * 32 + lane) : -1;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        x |= u[j] >= 0 ? __ldca(cin + u[j]) : 0ull;
        if (STATS) c.gathered += u[j] >= 0 ? 1ull : 0ull;
    }
    const uint32_t lo = __reduce_or_sync(GRX_FULL_MASK, (uint32_t)x);
    const uint32_t hi = __reduce_or_sync(GRX_FULL_MASK, (uint32_t)(x >> 32));
    return ((unsigned long long)hi << 32) | lo;
}

// Pull, phase 1 (see the head of the file).  With every open row's edges gathered
// (in equal tiles), the three pull levels of 64 sources on R-MAT 24 took 3.80,
// 3.43 and 1.02 ms, and take 2.64 (88 % of the neighbours read: few rows find all
// their lanes so early), 0.25 (6 %) and 0.13.
template <typename OffT, bool STATS>
__device__ void ms_pull(const MsArgs<OffT> &a, const MsState &st, MsPullSmem &w, MsCounts &c) {
    constexpr int PER = MS_ROWS / 32;
    const int L = st.L;
    const unsigned int lane = threadIdx.x & 31;
    const unsigned long long *cin = pk3(a.cur[0], a.cur[1], a.cur[2], L % 3);
    unsigned long long *cout = pk3(a.cur[0], a.cur[1], a.cur[2], (L + 1) % 3);
    unsigned long long *hs = a.hist[st.flush ? 0 : st.hslots];
    unsigned int *wq = &a.ctl->wq[L & 3], *rctr = &a.ctl->ucount[(L + 1) & 3];
    const int R = a.rows;
    const bool small = R < MS_ROWS;              // few rows a warp: it finishes its longer ones itself
    const int64_t nch = (a.n_active + R - 1) / R;
    const int64_t nwarps = (int64_t)gridDim.x * MS_WARPS;
    const bool more = nch > nwarps;              // else a thousand atomics on one word, for nothing
    const uint32_t lane_head = a.few ? MS_LANE_HEAD : 2;
    // the active row j of chunk ch: neighbours, or on small graphs spread over the whole
    // range (R-MAT's longest rows are neighbours, and a warp would have them all)
    auto row_of = [&](int64_t ch, int64_t j) { return small ? j * nch + ch : ch * R + j; };
    for (int64_t ch = grx_warp(); ch < nch;) {
        unsigned int nn = 0;
        if (lane == 0 && more) nn = atomicAdd(wq, 1u);
        if (!__ldcg(a.sat + ch)) {
            int32_t v[PER];
            uint32_t s[PER], deg[PER];
            unsigned long long miss[PER], acc[PER];
            int2 f2[PER];
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const int64_t i = row_of(ch, k * 32 + lane);
                v[k] = -1;
                s[k] = deg[k] = 0u;
                if (k * 32 + (int)lane < R && i < a.n_active) {
                    v[k] = __ldg(a.active + i);
                    s[k] = __ldg(a.aoff + i);
                    deg[k] = __ldg(a.aoff + i + 1) - s[k];
                }
            }
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                miss[k] = v[k] >= 0 ? a.lanes & ~__ldcg(a.seen + v[k]) : 0ull;
                f2[k] = miss[k] ? __ldg(a.first2 + v[k]) : make_int2(-1, -1);
            }
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                acc[k] = f2[k].x >= 0 ? __ldca(cin + f2[k].x) : 0ull;
                acc[k] |= f2[k].y >= 0 ? __ldca(cin + f2[k].y) : 0ull;
                if (STATS) c.gathered += (f2[k].x >= 0 ? 1 : 0) + (f2[k].y >= 0 ? 1 : 0);
            }
            if (STATS) {
#pragma unroll
                for (int k = 0; k < PER; ++k) c.rows += v[k] >= 0 ? 1ull : 0ull;
            }
            if (a.few) {                             // short rows: a lane takes a row's first ten edges
#pragma unroll 1
                for (uint32_t at = 2; at < MS_LANE_HEAD; at += 4) {
#pragma unroll
                    for (int k0 = 0; k0 < PER; k0 += 2) {
                        int32_t u[2][4];
#pragma unroll
                        for (int k = k0; k < k0 + 2; ++k)
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                u[k - k0][j] = at + j < deg[k] && (miss[k] & ~acc[k]) ? __ldg(a.col + (int64_t)s[k] + at + j) : -1;
#pragma unroll
                        for (int k = k0; k < k0 + 2; ++k)
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                if (u[k - k0][j] >= 0) acc[k] |= __ldca(cin + u[k - k0][j]);
                                if (STATS) c.gathered += u[k - k0][j] >= 0 ? 1ull : 0ull;
                            }
                    }
                }
            }
            bool open = false;
            int nh = 0;
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                acc[k] &= miss[k];
                const bool more = (miss[k] & ~acc[k]) != 0ull && deg[k] > lane_head;
                const unsigned int m = __ballot_sync(GRX_FULL_MASK, more);
                if (more) {
                    const int h = nh + __popc(m & lanemask_lt());
                    w.s[h] = s[k];
                    w.deg[h] = deg[k];
                    w.i[h] = (int32_t)row_of(ch, k * 32 + lane);
                    w.v[h] = v[k];
                    w.miss[h] = miss[k];
                    w.acc[h] = acc[k];
                } else {
                    if (miss[k] & ~acc[k]) open = true;          // lanes still missing after this level
                    if (acc[k]) {
                        cout[v[k]] = acc[k];
                        ms_pull_finish(a.seen, hs, v[k], a.lanes & ~miss[k], acc[k], deg[k], c);
                    }
                }
                nh += __popc(m);
            }
            __syncwarp();
            // the open rows: eight lanes a row, 32 edges a step
            const unsigned int gi = lane >> 3, gl = lane & 7, gmask = 0xffu << (gi * 8);
            for (int h = (int)gi; h < nh; h += 4) {
                const uint32_t len = w.deg[h], end = min(len, 2 + MS_HEAD);
                const int64_t e0 = w.s[h];
                const unsigned long long ms = w.miss[h];
                unsigned long long ac = w.acc[h];
                for (uint32_t at = lane_head; at < end && (ms & ~ac); at += 32) {
                    int32_t u[4];
                    unsigned long long g[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) u[j] = at + j * 8 + gl < end ? __ldg(a.col + e0 + at + j * 8 + gl) : -1;
#pragma unroll
                    for (int j = 0; j < 4; ++j) g[j] = u[j] >= 0 ? __ldca(cin + u[j]) : 0ull;
                    if (STATS) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) c.gathered += u[j] >= 0 ? 1ull : 0ull;
                    }
                    unsigned long long x = (g[0] | g[1]) | (g[2] | g[3]);
#pragma unroll
                    for (int o = 4; o > 0; o >>= 1) x |= __shfl_xor_sync(gmask, x, o);
                    ac |= x & ms;
                }
                __syncwarp(gmask);                               // the group has read its entry
                const bool left = (ms & ~ac) != 0ull;
                if (left && len > end && small && len <= MS_WARP_ROW) {
                    if (gl == 0) w.acc[h] = ac;                  // the warp together, below
                    continue;
                }
                if (gl == 0) w.deg[h] = 0u;                      // nothing left to do here
                if (left) open = true;
                if (gl == 0) {
                    const int32_t vv = w.v[h];
                    if (left && len > end) {                     // the rest of the row, in pieces
                        const uint32_t np = (len - end + MS_PIECE - 1) / MS_PIECE;
                        const unsigned int base = atomicAdd(rctr, np);
                        for (uint32_t k = 0; k < np; ++k) a.rest[base + k] = make_int2(w.i[h], (int)k);
                        if (ac) a.next[vv] = ac;
                    } else if (ac) {
                        cout[vv] = ac;
                        ms_pull_finish(a.seen, hs, vv, a.lanes & ~ms, ac, len, c);
                    }
                }
            }
            __syncwarp();
            for (int h = 0; small && h < nh; ++h) {
                const uint32_t len = w.deg[h];
                if (len == 0) continue;
                const int64_t e0 = w.s[h];
                const unsigned long long ms = w.miss[h];
                unsigned long long ac = w.acc[h];
                for (uint32_t at = 2 + MS_HEAD; at < len && (ms & ~ac); at += 256)
                    ac |= ms_gather256<STATS>(a.col, cin, e0 + at, e0 + len, c) & ms;
                if (ms & ~ac) open = true;
                if (lane == 0 && ac) {
                    cout[w.v[h]] = ac;
                    ms_pull_finish(a.seen, hs, w.v[h], a.lanes & ~ms, ac, len, c);
                }
            }
            // a row that goes on in pieces counts as open: the flag may stay clear
            // one level longer than needed, never the other way
            open = __any_sync(GRX_FULL_MASK, open);
            if (lane == 0 && !open) a.sat[ch] = 1;
        }
        ch = more ? nwarps + __shfl_sync(GRX_FULL_MASK, nn, 0) : nch;
    }
}

// Pull, phase 2: the pieces of rows that are still open; what other pieces found
// meanwhile is taken into account.
template <typename OffT, bool STATS>
__device__ void ms_pull_rest(const MsArgs<OffT> &a, const MsState &st, MsCounts &c) {
    const unsigned int lane = threadIdx.x & 31;
    const unsigned long long *cin = pk3(a.cur[0], a.cur[1], a.cur[2], st.L % 3);
    const int64_t n = ld_relaxed_u32(&a.ctl->ucount[(st.L + 1) & 3]);
    const int64_t nwarps = (int64_t)gridDim.x * MS_WARPS;
    for (int64_t t = grx_warp(); t < n; t += nwarps) {
        const int2 r = __ldcg(a.rest + t);
        const int32_t v = __ldg(a.active + r.x);
        const int64_t e0 = (int64_t)__ldg(a.aoff + r.x) + 2 + MS_HEAD + (int64_t)r.y * MS_PIECE;
        const int64_t e1 = min((int64_t)__ldg(a.aoff + r.x + 1), e0 + MS_PIECE);
        const unsigned long long ms = a.lanes & ~__ldcg(a.seen + v) & ~__ldcg(a.next + v);
        unsigned long long ac = 0ull;
        for (int64_t at = e0; at < e1 && (ms & ~ac); at += 256)
            ac |= ms_gather256<STATS>(a.col, cin, at, e1, c) & ms;
        if (lane == 0 && ac) atomicOr(a.next + v, ac);
    }
}

// Pull, phase 3: the rows of the pieces, finished at their first one.
template <typename OffT>
__device__ void ms_pull_fixup(const MsArgs<OffT> &a, const MsState &st, MsCounts &c) {
    const int L = st.L;
    unsigned long long *cout = pk3(a.cur[0], a.cur[1], a.cur[2], (L + 1) % 3);
    unsigned long long *hs = a.hist[st.flush ? 0 : st.hslots];
    const int64_t n = ld_relaxed_u32(&a.ctl->ucount[(L + 1) & 3]);
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const int2 r = __ldcg(a.rest + t);
        if (r.y != 0) continue;
        const int32_t v = __ldg(a.active + r.x);
        const unsigned long long acc = __ldcg(a.next + v);
        if (acc) a.next[v] = 0ull;
        const unsigned long long sv = __ldcg(a.seen + v);
        const unsigned long long nw = acc & a.lanes & ~sv;
        if (nw) {
            cout[v] = nw;
            ms_pull_finish(a.seen, hs, v, sv, nw, __ldg(a.aoff + r.x + 1) - __ldg(a.aoff + r.x), c);
        }
    }
}

// Depths of the pull levels held in the first nslots history slots, written
// lane-major (for each lane, consecutive threads write consecutive vertices);
// the slots are cleared.  The final flush also writes -1 for every pair that
// was never reached.  Masks are split into 32-bit halves so the per-lane
// tests are single-word operations.
// NS: history slots looked at (a lane's depth takes a test per slot, and the
// output's 4 * lanes * V bytes leave time for few of them).
template <typename OffT, int NS, int VW>
__device__ __forceinline__ void ms_flush_slots(const MsArgs<OffT> &a, int nslots, const int32_t *slot_depth,
                                               bool final) {
    int32_t sd[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) sd[s] = s < nslots ? slot_depth[s] : 0;
    // VW consecutive vertices a thread: 16-byte stores where every lane's row of the
    // output starts on such a boundary
    for (int64_t v0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * VW; v0 < a.nv;
         v0 += (int64_t)gridDim.x * blockDim.x * VW) {
        for (int half = 0; half * 32 < a.n; ++half) {    // 32 lanes at a time
            uint32_t h[NS][VW], un[VW], any = 0u;
#pragma unroll
            for (int i = 0; i < VW; ++i) {
                un[i] = final ? (uint32_t)(a.lanes >> (32 * half)) & ~__ldcg((const uint32_t *)(a.seen + v0 + i) + half)
                              : 0u;
                any |= un[i];
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    uint32_t *p = (uint32_t *)(a.hist[s] + v0 + i) + half;
                    h[s][i] = s < nslots ? __ldcg(p) : 0u;
                    any |= h[s][i];
                    if (h[s][i]) *p = 0u;
                }
            }
            if (!any) continue;
            const int last = min(a.n, 32 * half + 32);
            int32_t *out = a.depth + (int64_t)(32 * half) * a.nv + v0;
            for (int b = 32 * half; b < last; ++b, out += a.nv) {
                int d[VW];
                bool all = true;
#pragma unroll
                for (int i = 0; i < VW; ++i) {
                    d[i] = (un[i] & 1u) ? -1 : -2;       // -2: written by a push level
                    un[i] >>= 1;
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        d[i] = (h[s][i] & 1u) ? sd[s] : d[i];
                        h[s][i] >>= 1;
                    }
                    all = all && d[i] != -2;
                }
                if (VW == 4 && all) {
                    *reinterpret_cast<int4 *>(out) = make_int4(d[0], d[1 % VW], d[2 % VW], d[3 % VW]);
                } else {
#pragma unroll
                    for (int i = 0; i < VW; ++i)
                        if (d[i] != -2) out[i] = d[i];
                }
            }
        }
    }
}

// Four vertices a thread where nearly every word of four is written whole (the only
// flush of a traversal) and every thread has some; words written in part cost four
// times the stores.
template <typename OffT>
__device__ void ms_flush(const MsArgs<OffT> &a, int nslots, const int32_t *slot_depth, bool final, bool flushed) {
    const bool wide = final && !flushed && (a.nv & 3) == 0 && ((uintptr_t)a.depth & 15) == 0 &&
                      a.nv / 4 >= (int32_t)(gridDim.x * blockDim.x);
    if (!wide && nslots <= 3) ms_flush_slots<OffT, 3, 1>(a, nslots, slot_depth, final);
    else if (!wide) ms_flush_slots<OffT, MS_HSLOTS, 1>(a, nslots, slot_depth, final);
    else if (nslots <= 3) ms_flush_slots<OffT, 3, 4>(a, nslots, slot_depth, final);
    else if (nslots <= 4) ms_flush_slots<OffT, 4, 4>(a, nslots, slot_depth, final);
    else ms_flush_slots<OffT, MS_HSLOTS, 4>(a, nslots, slot_depth, final);
}

template <typename OffT, bool STATS>
__global__ void __launch_bounds__(MS_BLOCK, MS_MIN_BLOCKS) k_msbfs_persistent(MsArgs<OffT> a) {
    __shared__ MsState s_st;
    __shared__ int s_dirty;
    __shared__ MsSmem<OffT> sm;
    FlagBarrier bar{a.bar_flags, &a.ctl->bar_release, a.ctl, a.timeout_ns, 0u};
    if (threadIdx.x == 0) {
        // the previous traversal left the history slots and the OR buffer
        // zero only if every one of its blocks finished its final pass
        const unsigned int g = ld_relaxed_u32(&a.ctl->ms_grid);
        s_dirty = !(g > 0 && ld_relaxed_u32(&a.ctl->ms_done) == g);
    }
    __syncthreads();
    ms_init_fill(a, s_dirty != 0);
    if (!flag_barrier(bar)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) ms_seed(a);
    if (!flag_barrier(bar)) return;
    if (threadIdx.x == 0) {
        MsState s;
        memset(&s, 0, sizeof s);
        const unsigned long long pk = ld_relaxed_u64(&a.ctl->qpack[0]);
        s.dir = a.mode == GRX_DIR_PULL ? DIR_PULL : DIR_PUSH;
        s.switched = a.mode == GRX_DIR_PULL;
        s.q = (uint32_t)(pk >> 32);
        s.T = (uint32_t)pk;
        s.qin = 1;
        s.seen_pairs = (unsigned long long)a.n;
        s.done = s.q == 0;
        ms_set_kind(a, s);
        s_st = s;
    }
    __syncthreads();
    for (;;) {
        const MsState &st = s_st;
        if (st.done) break;
        const int L = st.L;
        const int op = ms_op(st);
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            if ((int)st.phase + 1 == ms_phases(st)) a.ctl->cpack = 0ull;   // used by first phases only
            if (st.phase == 0) {
                a.ctl->qpack[(L + 2) & 3] = 0ull;
                a.ctl->ucount[(L + 2) & 3] = 0u;
                a.ctl->wq[(L + 2) & 3] = 0u;
                a.ctl->pairs[(L + 2) & 3] = 0ull;
                if (STATS && L < GRX_MAX_LEVELS_STATS) {
                    a.stats->level_t0[L] = grx_globaltimer();
                    a.stats->dir[L] = st.dir;
                    a.stats->frontier[L] = st.q;
                    a.stats->levels = L + 1;
                    if (st.dir == DIR_PUSH) {
                        a.stats->edges_examined[L] = st.T;
                        a.stats->vertices_scanned[L] = st.q;
                    }
                }
            }
        }
        if (op == MOP_COMPACT) {
            ms_compact<OffT>(a, st);
        } else if (op == MOP_EXPAND) {
            ms_push_expand<OffT, STATS>(a, st, sm.w[threadIdx.x >> 5]);
        } else if (op == MOP_FINAL) {
            ms_push_finalize<OffT>(a, st, sm.w[threadIdx.x >> 5].list);
        } else if (op == MOP_FLUSH) {
            ms_flush<OffT>(a, MS_HSLOTS, st.slot_depth, false, st.flushed);
        } else {
            MsCounts c = {0ull, 0ull, 0ull, 0ull, 0ull};
            if (op == MOP_PULL) ms_pull<OffT, STATS>(a, st, sm.p[threadIdx.x >> 5], c);
            else if (op == MOP_REST) ms_pull_rest<OffT, STATS>(a, st, c);
            else ms_pull_fixup<OffT>(a, st, c);
            c.q = warp_sum(c.q);
            c.T = warp_sum(c.T);
            c.pairs = warp_sum(c.pairs);
            if (STATS) {
                c.gathered = warp_sum(c.gathered);
                c.rows = warp_sum(c.rows);
            }
            if ((threadIdx.x & 31) == 0) {
                if (c.q) atomicAdd(&a.ctl->qpack[(L + 1) & 3], (c.q << 32) | c.T);
                if (c.pairs) atomicAdd(&a.ctl->pairs[(L + 1) & 3], c.pairs);
                if (STATS && c.gathered && L < GRX_MAX_LEVELS_STATS)
                    atomicAdd(&a.stats->edges_examined[L], c.gathered);
                if (STATS && c.rows && L < GRX_MAX_LEVELS_STATS)
                    atomicAdd(&a.stats->vertices_scanned[L], c.rows);   // rows not skipped
            }
        }
        if (!flag_barrier(bar)) return;
        if (threadIdx.x == 0) s_st = ms_next_state(a, st, STATS);
        __syncthreads();
    }
    // depths of the pull levels still in the history slots, -1 for the rest
    ms_flush<OffT>(a, s_st.hslots, s_st.slot_depth, true, s_st.flushed);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&a.ctl->ms_done, 1u);
        if (blockIdx.x == 0) {
            a.ctl->levels_run = s_st.L;
            if (STATS && s_st.L <= GRX_MAX_LEVELS_STATS) a.stats->level_t0[s_st.L] = grx_globaltimer();
        }
    }
}

// Rows a warp of the pull takes at a time: 128, or on small graphs what gives
// every warp some, down to four (one per eight lanes).  3,800 vertices, 48 sources:
// 294 us with 128, 191 so, and 157 since these warps finish rows of up to 2,048
// edges themselves instead of leaving them to two more phases.
int ms_rows(const grx_graph *g, int blocks) {
    int r = MS_ROWS;
    while (r > 4 && g->n_active < (int64_t)blocks * MS_WARPS * r) r /= 2;
    return r;
}

// One flag per ms_rows rows: fewer than two per warp where these are not MS_ROWS.
size_t ms_sat_bytes(const grx_graph *g) {
    return (size_t)(g->n_active / MS_ROWS) + 1 + 2 * (size_t)GRX_MAX_GRID * MS_WARPS;
}

// Pieces of the rows longer than 2 + MS_HEAD, at most.
size_t ms_rest_bytes(const grx_graph *g) {
    return (size_t)(g->ne / (MS_HEAD + 3) + g->ne / MS_PIECE + 1) * sizeof(int2);
}

size_t ms_tbits_bytes(const grx_graph *g) { return (size_t)g->words * 4 + 16; }

template <typename OffT, bool STATS>
grx_status ms_launch_typed(grx_graph *g, const int32_t *srcs, int n, int32_t *depth,
                           const grx_opts *o, cudaStream_t s) {
    MsArgs<OffT> a;
    a.nv = g->nv;
    a.ne = g->ne;
    a.ro = (const OffT *)g->ro;
    a.col = g->col;
    a.active = g->active;
    a.aoff = g->aoff;
    a.first2 = g->first2;
    a.n_active = g->n_active;
    bool ok = grx_have(g, g->ms_sat, ms_sat_bytes(g), s) && grx_have(g, g->ms_rest, ms_rest_bytes(g), s) &&
              grx_have(g, g->ms_tbits, ms_tbits_bytes(g), s, true);
    for (int i = 0; i < MS_HSLOTS; ++i) ok = ok && grx_have(g, g->ms_hist[i], (size_t)g->nv * 8, s);
    if (!ok) return grx_fail(GRX_ENOMEM, "bfs_multi: workspace allocation failed (nv=%d)", g->nv);
    a.rest = g->ms_rest;
    a.sat = g->ms_sat;
    for (int i = 0; i < MS_HSLOTS; ++i) a.hist[i] = g->ms_hist[i];
    a.n = n;
    a.lanes = n == 64 ? ~0ull : ((1ull << n) - 1ull);
    for (int i = 0; i < 64; ++i) a.src[i] = i < n ? srcs[i] : 0;
    a.seen = g->ms_seen;
    a.next = g->ms_next;
    for (int i = 0; i < 3; ++i) {
        a.cur[i] = g->ms_cur[i];
        a.Q[i] = g->qv[i];
        a.E[i] = g->qe[i];
        a.R[i] = (OffT *)g->qr[i];
    }
    a.touched = g->ulist[0];
    a.tbits = g->ms_tbits;
    a.words = g->words;
    {   // bitmap push when a level's edges reach push_bitmap * nv (0 = 1/8, < 0 = never)
        const double pb = o->push_bitmap == 0.f ? 0.125 : (double)o->push_bitmap;
        const double t = pb * (double)g->nv;
        a.bmp_min_T = pb < 0 ? 0xffffffffu : (t < 1.0 ? 1u : (t > 4294967295.0 ? 0xffffffffu : (uint32_t)t));
    }
    a.depth = depth;
    a.ctl = g->ctl;
    a.bar_flags = g->bar_flags;
    a.stats = g->stats;
    a.mode = o->direction;
    a.alpha = o->alpha;
    a.beta = o->beta;
    a.timeout_ns = grx_timeout_ns(o);
    static int per_sm = -1;
    if (per_sm < 0) {
        GRX_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_msbfs_persistent<OffT, STATS>,
                                                               MS_BLOCK, 0));
        if (per_sm < 1) return grx_fail(GRX_ECUDA, "bfs_multi: persistent kernel does not fit on an SM");
    }
    int max_grid = per_sm * g->ctx->num_sms;
    if (max_grid > GRX_MAX_GRID) max_grid = GRX_MAX_GRID;
    const int blocks = grx_grid(o, MS_BLOCK, max_grid);
    a.rows = ms_rows(g, blocks);
    a.few = g->ne < 8 * g->n_active;
    GRX_CUDA(cudaMemsetAsync(g->bar_flags, 0, sizeof(unsigned int) * (size_t)blocks, s));
    GRX_CUDA(cudaMemsetAsync(&g->ctl->bar_release, 0, sizeof(unsigned int), s));
    if (o->collect_stats) GRX_CUDA(cudaMemsetAsync(g->stats, 0, sizeof(DevStats), s));
    void *args[] = {(void *)&a};
    if (o->ev_begin) GRX_CUDA(cudaEventRecord((cudaEvent_t)o->ev_begin, s));
    GRX_CUDA(cudaLaunchCooperativeKernel((const void *)k_msbfs_persistent<OffT, STATS>, dim3(blocks),
                                         dim3(MS_BLOCK), args, 0, s));
    if (o->ev_end) GRX_CUDA(cudaEventRecord((cudaEvent_t)o->ev_end, s));
    return GRX_OK;
}

}  // namespace

size_t grx_msbfs_new_bytes(const grx_graph *g) {
    size_t b = 0;
    if (!g->ms_sat) b += ms_sat_bytes(g);
    if (!g->ms_rest) b += ms_rest_bytes(g);
    if (!g->ms_tbits) b += ms_tbits_bytes(g);
    for (int i = 0; i < MS_HSLOTS; ++i)
        if (!g->ms_hist[i]) b += (size_t)g->nv * 8;
    return b;
}

grx_status grx_msbfs_launch(grx_graph *g, const int32_t *srcs, int n, int32_t *depth,
                            const grx_opts *o, cudaStream_t s) {
    if (g->off64)
        return o->collect_stats ? ms_launch_typed<int64_t, true>(g, srcs, n, depth, o, s)
                                : ms_launch_typed<int64_t, false>(g, srcs, n, depth, o, s);
    return o->collect_stats ? ms_launch_typed<int32_t, true>(g, srcs, n, depth, o, s)
                            : ms_launch_typed<int32_t, false>(g, srcs, n, depth, o, s);
}
