// SSSP (Table 1): frontier label-correcting relaxation.  Each round advances
// the vertices whose distance improved in the previous round: for every edge
// (u, v, w) it proposes dist[u] + w with an atomic min -- the min combiner the
// paper uses for SSSP labels (Sec. 3) -- and v joins the next frontier once.
// Rounds repeat until no distance improves; the result is the exact
// shortest-path distance.
//
// Same persistent, load-balanced structure as the push step of BFS: a frontier
// queue slot carries the vertex, its row start and the exclusive prefix of the
// frontier's degrees, so the frontier's edges are cut into equal warp tiles
// (each warp a contiguous range, rows by a branch-free scatter + max-scan) and
// each lane keeps 8 edges' loads in flight, item k at tile position
// k*32 + lane so the warp's column and weight loads are contiguous runs.  Two
// kinds of rounds:
//  * small rounds: an improving lane claims v with the atomic min's old value,
//    a per-vertex round stamp keeps v once, and v is appended with one
//    warp-aggregated atomic;
//  * rounds with at least push_bitmap * V edges: the atomic min is a
//    reduction (no value returned) and v's bit is OR-ed into a changed bitmap;
//    a second phase, by warps owning 32-word chunks of the bitmap, appends the
//    changed vertices in vertex order and clears the bitmap.  A lane reduces
//    only when its proposal beats the current distance read from L2, so every
//    marked vertex did improve in the round and every improvement is marked.
// Near-far bands (Davidson et al.'s near-far split, opt-in with delta > 0):
// an improved vertex joins the next frontier only if its distance is below
// the threshold, else it waits once in a far pile (a bitmap keeps it unique).
// When the frontier runs dry, the threshold moves to the pile's smallest
// distance + delta and the pile's vertices below it form the next frontier;
// entries below the old threshold were relaxed since and are dropped.  High-
// diameter weighted graphs then relax far fewer edges more than once.
// Rounds and phases are separated by the bounded grid barrier.
//
// On graphs of few edges a vertex, whose shortest paths take thousands of small
// rounds, rounds that fit run on lists instead (list_round): a group of blocks
// with the exchange and the pieces of the narrow levels (narrow.cuh), while the
// rest of the grid waits.
#include "grx_internal.cuh"
#include "narrow.cuh"

namespace {

// Two blocks of 384 threads an SM, as in bfs.cu (R-MAT 22: 1,578 -> 1,525 us).
constexpr int SS_BLOCK = 384;
constexpr int SS_MIN_BLOCKS = 2;             // resident blocks per SM (register cap)
constexpr int SS_WARPS = SS_BLOCK / 32;
constexpr int SS_ITEMS = 8;
constexpr int SS_WTILE = 32 * SS_ITEMS;
constexpr int SS_BATCH = 4;                  // tiles a warp takes at a time
constexpr int SS_RPL = 4;                    // finalize: vertices per lane per round

template <typename OffT>
struct SsspArgs {
    int32_t nv;
    int64_t words;
    const OffT *ro;
    const int32_t *col;
    const uint32_t *w;
    uint32_t *dist;
    int32_t *stamp;
    uint32_t *cbits;                         // changed bitmap of reduction rounds
    uint32_t *fbits;                         // near-far: far pile membership
    int32_t *far[2];                         // near-far: far piles (ping-pong)
    uint32_t delta;                          // near-far band width (0 = no bands)
    int32_t *Q[3];
    uint32_t *E[3];
    OffT *R[3];
    TravCtl *ctl;
    unsigned int *bar_flags;
    DevStats *stats;
    uint32_t bmp_min_T;
    unsigned long long timeout_ns;
    int32_t src;
    int even;                                // no hubs: a round's tiles in equal shares
    // list rounds (lines NULL: none), per block: pieces by round parity, vertices
    NarrowWord *lines, *pieces;
    int32_t *verts;
    uint32_t list_T;                         // edges of a round, at most, per block
    uint32_t group;                          // blocks that run them, and rounds between two
    uint32_t list_rounds;                    // grid barriers, at which the others renew their wait
};

constexpr int SS_LIST_BLOCKS = 512;          // blocks of a list round: at most SS_BLOCK, searched as 512
// Per block, for rounds of at most t edges a block: pieces a segment holds (a
// round with a fuller one leaves the list rounds), and vertices a block can
// find (its whole steps of 192 pieces, four edges each).
__host__ __device__ inline uint32_t ss_list_pieces(uint32_t t) { return t; }
__host__ __device__ inline uint32_t ss_list_verts(uint32_t t) { return 4 * (t + SS_WARPS * 8 * 2); }

enum { SOP_RELAX, SOP_FINAL, SOP_FARMIN, SOP_FARSPLIT };
enum { LIST_OFF = 1, LIST_ON = 2 };

struct SsState {
    int L;
    int op;
    int bmp;
    int done;
    int list;                                // LIST_OFF: the whole grid runs this round, whatever its size;
                                             // LIST_ON: the group goes on (the other blocks wait again)
    int fsel;                                // current far pile
    uint32_t q, T;
    uint32_t thr;                            // near-far threshold (UINT32_MAX: no bands)
    uint32_t oldthr;                         // threshold before the last advance
    uint32_t nfar;                           // current far pile length
};

template <typename OffT>
union SsWarpSmem {
    struct {
        uint32_t qe[SS_WTILE + 2];
        int32_t u[SS_WTILE + 1];
        OffT rs[SS_WTILE + 1];
        uint32_t du[SS_WTILE + 1];
        alignas(16) uint16_t rid[SS_WTILE];
    };
    uint16_t list[32 * 32];
};

template <typename OffT>
__device__ __forceinline__ void ss_set_kind(const SsspArgs<OffT> &a, SsState &s) {
    s.bmp = s.T >= a.bmp_min_T;
}

// v improved to a distance at or above the threshold: into the far pile once.
template <typename OffT>
__device__ __forceinline__ void far_push(const SsspArgs<OffT> &a, const SsState &st, int32_t v) {
    const uint32_t bit = 1u << (v & 31);
    if (!(atomicOr(a.fbits + (v >> 5), bit) & bit)) {
        const unsigned int pos = atomicAdd(&a.ctl->farcnt[st.fsel], 1u);
        a.far[st.fsel][pos] = v;
    }
}

// Phase 0 of round L: relax the edges of Q_L.
template <typename OffT, bool BMP>
__device__ void relax_round(const SsspArgs<OffT> &a, const SsState &st, SsWarpSmem<OffT> &w) {
    const int L = st.L;
    const unsigned int lane = threadIdx.x & 31;
    const int32_t *Qv = pick3(a.Q[0], a.Q[1], a.Q[2], L % 3);
    const uint32_t *Qe = pick3(a.E[0], a.E[1], a.E[2], L % 3);
    const OffT *Qr = pick3(a.R[0], a.R[1], a.R[2], L % 3);
    int32_t *Qv_out = pick3(a.Q[0], a.Q[1], a.Q[2], (L + 1) % 3);
    uint32_t *Qe_out = pick3(a.E[0], a.E[1], a.E[2], (L + 1) % 3);
    OffT *Qr_out = pick3(a.R[0], a.R[1], a.R[2], (L + 1) % 3);
    unsigned long long *ctr = &a.ctl->qpack[(L + 1) & 3];
    const int64_t q = st.q;
    const uint64_t T = st.T;
    const uint64_t ntiles = (T + SS_WTILE - 1) / SS_WTILE;
    const uint64_t nwarps = (uint64_t)gridDim.x * SS_WARPS;
    // Batches of up to SS_BATCH tiles: the first by the warp's number, the others
    // from the round's counter.  What a tile costs varies along the queue (R-MAT 22,
    // mean of three sources: one equal share a warp 1,824 us, batches of 16 / 8 / 4 / 2
    // tiles 1,618 / 1,577 / 1,569 / 1,744; a batch costs a search).  Without hubs it
    // does not, and equal shares are the better form (uniform random, 2M vertices of
    // degree 16: 1,536 us, batches 1,597; in bands of 100 1,430 and 1,518).
    const uint64_t share = (ntiles + nwarps - 1) / nwarps;
    const uint64_t batch = a.even ? share : min((uint64_t)SS_BATCH, share);
    if (batch == 0) return;
    const uint64_t nbatch = (ntiles + batch - 1) / batch;
    unsigned int *wq = &a.ctl->wq[L & 3];
    const uint64_t gw = grx_warp();
    for (uint64_t bt = gw; bt < nbatch;) {
        unsigned int nn = 0;
        if (lane == 0) nn = atomicAdd(wq, 1u);
        const uint64_t tb0 = bt * batch, tb1 = min(ntiles, tb0 + batch);
        int64_t i0 = warp_upper_index_cg(Qe, q, (uint32_t)(tb0 * SS_WTILE));
        for (uint64_t tile = tb0; tile < tb1; ++tile) {
            const uint64_t e0 = tile * SS_WTILE;
            const uint32_t e1 = (uint32_t)min(T, e0 + SS_WTILE);
            // frontier elements starting before e1, 32 per round
            int n = 0;
            for (;;) {
                const int64_t idx = i0 + n + lane;
                uint32_t qe = 0xffffffffu;
                if (idx < q) qe = __ldcg(Qe + idx);
                const bool in = idx < q && qe < e1;
                if (n + (int)lane <= SS_WTILE + 1) w.qe[n + lane] = qe;
                if (in && n + (int)lane <= SS_WTILE) {
                    const int32_t u = __ldcg(Qv + idx);
                    w.u[n + lane] = u;
                    w.rs[n + lane] = __ldcg(Qr + idx);
                    w.du[n + lane] = __ldcg(a.dist + u);
                }
                const int cnt = __popc(__ballot_sync(GRX_FULL_MASK, in));
                n += cnt;
                if (cnt < 32) break;
                if (n > SS_WTILE) {              // only possible with a malformed graph
                    if (lane == 0) grx_set_status(a.ctl, GRX_EINVAL);
                    n = SS_WTILE;
                    break;
                }
            }
            __syncwarp();
            const uint32_t next_start = w.qe[n];
            int row[SS_ITEMS];
            warp_tile_rows8_strided(w.rid, w.qe, (uint32_t)e0, n, row);   // item k at position k*32 + lane
            int32_t v[SS_ITEMS];
            uint32_t wt[SS_ITEMS], du[SS_ITEMS];
#pragma unroll
            for (int k = 0; k < SS_ITEMS; ++k) {
                const uint32_t e = (uint32_t)e0 + (uint32_t)k * 32 + lane;
                const int j = row[k];
                const bool ok = e < e1;
                const OffT idx = ok ? w.rs[j] + (OffT)(e - w.qe[j]) : (OffT)0;
                v[k] = ok ? __ldg(a.col + idx) : -1;
                wt[k] = ok ? __ldg(a.w + idx) : 0u;
                du[k] = ok ? w.du[j] : 0xffffffffu;
            }
            __syncwarp();
            uint32_t nd[SS_ITEMS], cur[SS_ITEMS];
#pragma unroll
            for (int k = 0; k < SS_ITEMS; ++k) {
                nd[k] = 0xffffffffu;
                if (v[k] >= 0 && du[k] != 0xffffffffu) {
                    const uint64_t s64 = (uint64_t)du[k] + wt[k];
                    if (s64 >= 0xffffffffull) grx_set_status(a.ctl, GRX_ERANGE);
                    else nd[k] = (uint32_t)s64;
                }
                cur[k] = nd[k] != 0xffffffffu ? __ldcg(a.dist + v[k]) : 0u;
            }
            if (BMP) {
#pragma unroll
                for (int k = 0; k < SS_ITEMS; ++k) {
                    if (nd[k] < cur[k]) {
                        atomicMin(a.dist + v[k], nd[k]);                     // results unused: reductions
                        atomicOr(a.cbits + (v[k] >> 5), 1u << (v[k] & 31));
                    }
                }
            } else {
                uint32_t improved = 0;
#pragma unroll
                for (int k = 0; k < SS_ITEMS; ++k) {
                    if (nd[k] < cur[k]) {
                        const uint32_t old = atomicMin(a.dist + v[k], nd[k]);
                        if (nd[k] < old) improved |= 1u << k;
                    }
                }
                uint32_t queued = 0;
#pragma unroll
                for (int k = 0; k < SS_ITEMS; ++k) {
                    if (!(improved >> k & 1u)) continue;
                    if (nd[k] >= st.thr) far_push(a, st, v[k]);
                    else if (atomicExch(a.stamp + v[k], L + 1) != L + 1) queued |= 1u << k;
                }
                uint32_t deg[SS_ITEMS];
                OffT rb[SS_ITEMS];
                uint32_t app = 0;
#pragma unroll
                for (int k = 0; k < SS_ITEMS; ++k) {
                    rb[k] = 0;
                    deg[k] = 0;
                    if (queued >> k & 1u) {
                        rb[k] = __ldg(a.ro + v[k]);
                        deg[k] = (uint32_t)(__ldg(a.ro + v[k] + 1) - rb[k]);
                        if (deg[k]) app |= 1u << k;
                    }
                }
                warp_append_items<SS_ITEMS, OffT>(v, deg, rb, app, Qv_out, Qe_out, Qr_out, ctr);
            }
            i0 = (next_start == e1) ? i0 + n : i0 + n - 1;
            __syncwarp();
        }
        bt = nwarps + __shfl_sync(GRX_FULL_MASK, nn, 0);
    }
}

// Phase 1 of a reduction round: the changed bitmap's vertices (with edges)
// become Q_{L+1} in vertex order; the bitmap is cleared.
template <typename OffT>
__device__ void changed_to_queue(const SsspArgs<OffT> &a, const SsState &st, uint16_t *list) {
    const int L = st.L;
    int32_t *Qv_out = pick3(a.Q[0], a.Q[1], a.Q[2], (L + 1) % 3);
    uint32_t *Qe_out = pick3(a.E[0], a.E[1], a.E[2], (L + 1) % 3);
    OffT *Qr_out = pick3(a.R[0], a.R[1], a.R[2], (L + 1) % 3);
    unsigned long long *ctr = &a.ctl->qpack[(L + 1) & 3];
    const unsigned int lane = threadIdx.x & 31;
    const int64_t nsc = (a.words + 31) / 32;
    const int64_t nwarps = (int64_t)gridDim.x * SS_WARPS;
    for (int64_t sc = grx_warp(); sc < nsc; sc += nwarps) {
        const int64_t wd = sc * 32 + lane;
        const uint32_t bits = wd < a.words ? __ldcg(a.cbits + wd) : 0u;
        if (bits) a.cbits[wd] = 0u;
        const int n = warp_compact_bits(bits, list);
        for (int base = 0; base < n; base += 32 * SS_RPL) {
            int32_t v[SS_RPL];
            uint32_t deg[SS_RPL];
            OffT rb[SS_RPL];
            uint32_t app = 0;
#pragma unroll
            for (int k = 0; k < SS_RPL; ++k) {
                const int i = base + k * 32 + (int)lane;
                v[k] = i < n ? (int32_t)(sc * 1024 + list[i]) : 0;
                rb[k] = 0;
                deg[k] = 0;
                if (i < n && __ldcg(a.dist + v[k]) >= st.thr) {
                    far_push(a, st, v[k]);
                } else if (i < n) {
                    rb[k] = __ldg(a.ro + v[k]);
                    deg[k] = (uint32_t)(__ldg(a.ro + v[k] + 1) - rb[k]);
                    if (deg[k]) app |= 1u << k;
                }
            }
            warp_append_items<SS_RPL, OffT>(v, deg, rb, app, Qv_out, Qe_out, Qr_out, ctr);
        }
        __syncwarp();
    }
}

// Band advance, phase 1: the smallest distance in the far pile.  The minimum
// of pile f goes to farmin[f]; farmin[f ^ 1], read by every block after the
// previous advance's barrier, is reset here for the next advance.
template <typename OffT>
__device__ void far_min(const SsspArgs<OffT> &a, const SsState &st) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.ctl->farcnt[st.fsel ^ 1] = 0u;
        a.ctl->farmin[st.fsel ^ 1] = 0xffffffffu;
    }
    const int32_t *F = a.far[st.fsel];
    uint32_t m = 0xffffffffu;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (int64_t)st.nfar;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t d = __ldcg(a.dist + __ldcg(F + i));
        if (d >= st.thr) m = min(m, d);          // below the threshold: relaxed since, stale
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = min(m, __shfl_xor_sync(GRX_FULL_MASK, m, o));
    if ((threadIdx.x & 31) == 0 && m != 0xffffffffu) atomicMin(&a.ctl->farmin[st.fsel], m);
}

// Band advance, phase 2 (threshold already raised): far vertices below the
// new threshold form Q_L, the others move to the other pile, stale ones drop.
template <typename OffT>
__device__ void far_split(const SsspArgs<OffT> &a, const SsState &st) {
    const int L = st.L;
    int32_t *Qv = pick3(a.Q[0], a.Q[1], a.Q[2], L % 3);
    uint32_t *Qe = pick3(a.E[0], a.E[1], a.E[2], L % 3);
    OffT *Qr = pick3(a.R[0], a.R[1], a.R[2], L % 3);
    const int32_t *F = a.far[st.fsel];
    int32_t *G = a.far[st.fsel ^ 1];
    const int64_t span = ((int64_t)st.nfar + 31) & ~(int64_t)31;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < span;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t v[1] = {0};
        uint32_t deg[1] = {0};
        OffT rb[1] = {0};
        uint32_t app = 0;
        if (i < (int64_t)st.nfar) {
            v[0] = __ldcg(F + i);
            const uint32_t d = __ldcg(a.dist + v[0]);
            if (d >= st.thr) {                                   // still far
                const unsigned int pos = atomicAdd(&a.ctl->farcnt[st.fsel ^ 1], 1u);
                G[pos] = v[0];
            } else {
                atomicAnd(a.fbits + (v[0] >> 5), ~(1u << (v[0] & 31)));
                if (d >= st.oldthr) {                            // first reached the band now
                    rb[0] = __ldg(a.ro + v[0]);
                    deg[0] = (uint32_t)(__ldg(a.ro + v[0] + 1) - rb[0]);
                    if (deg[0]) app = 1;
                }
            }
        }
        warp_append_items<1, OffT>(v, deg, rb, app, Qv, Qe, Qr, &a.ctl->qpack[L & 3]);
    }
}

// ---------------------------------------------------------------------------
// List rounds.  Per edge, three dependent trips to memory (piece; column, weight
// and the source's distance; the target's distance and row bounds) and one for
// the claim: the minimum and the round stamp are taken at once.  A proposal that
// beats the distance read means that the target improves in this round, by it or
// by a smaller one, so whoever sets the stamp may queue the target.  The minima
// are visible to the next round's reads through the exchange's fences.  A weighted
// 4096 x 4096 grid (rounds of 170,000 edges on average) takes 87 ms, and 158 ms with
// every round on the queue (search in the degree prefix, row lookup, global append
// counter, barrier).
// ---------------------------------------------------------------------------
template <typename OffT>
__device__ __forceinline__ void ss_list_append(const SsspArgs<OffT> &a, NarrowShared<SS_LIST_BLOCKS> &sh, int L,
                                               unsigned long long tag, bool has, int32_t v, uint32_t row,
                                               uint32_t deg) {
    const uint32_t cap = ss_list_pieces(a.list_T), vcap = ss_list_verts(a.list_T);
    const size_t seg = (size_t)(L & 1) * a.group + blockIdx.x;
    narrow_append(sh, a.pieces + seg * cap, cap, a.verts + seg * vcap, vcap, tag, has, v, row, deg, a.ctl);
}

template <typename OffT>
__device__ __forceinline__ void list_round(const SsspArgs<OffT> &a, const SsState &st,
                                           NarrowShared<SS_LIST_BLOCKS> &sh, unsigned long long tag) {
    const int L = st.L;
    const unsigned int lane = threadIdx.x & 31;
    const uint32_t step = a.group * SS_WARPS * 8;
    const uint32_t mine = ((threadIdx.x >> 5) * a.group + blockIdx.x) * 8 + (lane >> 2);
    const uint32_t total = sh.first[SS_LIST_BLOCKS], cap = ss_list_pieces(a.list_T);
    const NarrowWord *segs = a.pieces + (size_t)(L & 1) * a.group * cap;
    for (uint32_t base = 0; base < total; base += 2 * step) {
        const NarrowWord *at[2];
        NarrowWord w[2];
        bool ok[2];
        int32_t v[2];
        uint32_t wt[2], du[2], nd[2], cur[2];
        OffT rb[2], re[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const uint32_t c = base + k * step + mine;
            ok[k] = c < total;
            at[k] = nullptr;
            if (ok[k]) {
                uint32_t i;
                const uint32_t b = narrow_find(sh, c, i);
                at[k] = segs + (size_t)b * cap + i;
                w[k] = narrow_load(at[k]);
            }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            v[k] = 0;
            wt[k] = 0u;
            du[k] = 0xffffffffu;
            if (ok[k]) ok[k] = narrow_await(at[k], w[k], tag, a.ctl, a.timeout_ns) && (lane & 3) < narrow_len(w[k]);
            if (ok[k]) {
                v[k] = __ldg(a.col + narrow_edge(w[k]) + (lane & 3));
                wt[k] = __ldg(a.w + narrow_edge(w[k]) + (lane & 3));
                du[k] = __ldcg(a.dist + narrow_vertex(w[k]));
            }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            cur[k] = 0u;
            rb[k] = re[k] = 0;
            if (ok[k]) {
                cur[k] = __ldcg(a.dist + v[k]);
                rb[k] = __ldg(a.ro + v[k]);
                re[k] = __ldg(a.ro + v[k] + 1);
            }
            nd[k] = 0xffffffffu;
            if (ok[k] && du[k] != 0xffffffffu) {
                const uint64_t s64 = (uint64_t)du[k] + wt[k];
                if (s64 >= 0xffffffffull) grx_set_status(a.ctl, GRX_ERANGE);
                else nd[k] = (uint32_t)s64;
            }
        }
        int32_t stamp[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            stamp[k] = L + 1;
            if (nd[k] < cur[k]) {
                if (nd[k] < st.thr) stamp[k] = atomicExch(a.stamp + v[k], L + 1);
                else far_push(a, st, v[k]);
                atomicMin(a.dist + v[k], nd[k]);   // result unused: a reduction, ordered by the exchange
            }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const bool has = stamp[k] != L + 1 && re[k] > rb[k];
            if (has) {
                asm volatile("prefetch.global.L2 [%0];" ::"l"(a.col + rb[k]));
                asm volatile("prefetch.global.L2 [%0];" ::"l"(a.w + rb[k]));
            }
            ss_list_append(a, sh, L + 1, tag + 1, has, v[k], (uint32_t)rb[k], (uint32_t)(re[k] - rb[k]));
        }
    }
}

// Whether round st goes on lists (half the limit to come in, the limit to stay).
template <typename OffT>
__device__ __forceinline__ bool list_may_start(const SsspArgs<OffT> &a, const SsState &st) {
    return a.lines && st.op == SOP_RELAX && !st.bmp && st.list != LIST_OFF && st.T <= a.list_T * a.group / 2;
}

// Runs rounds from s_st on lists while they fit.  Called by the group's blocks;
// leaves in ctl->hstate the phase that every block goes on from after the next
// grid barrier, with its queue.  false: a wait gave up.
template <typename OffT, bool STATS>
__device__ __forceinline__ bool list_run(const SsspArgs<OffT> &a, SsState &s_st, NarrowShared<SS_LIST_BLOCKS> &sh,
                                            FlagBarrier &bar) {
    const int group = (int)a.group;
    const unsigned int lane = threadIdx.x & 31;
    // no tag of this stretch was used before: every stretch counts up the epoch
    unsigned long long tag = (unsigned long long)(ld_relaxed_u32(&a.ctl->narrow_epoch) & 0x7fffffffu) << 32;
    if (threadIdx.x == 0) {
        sh.got = 0ull;
        sh.got_edges = 0ull;
    }
    __syncthreads();
    {   // Q_L into the segments
        const int L = s_st.L;
        const uint32_t q = s_st.q;
        const int32_t *Q = pick3(a.Q[0], a.Q[1], a.Q[2], L % 3);
        const OffT *R = pick3(a.R[0], a.R[1], a.R[2], L % 3);
        const uint32_t i0 = (uint32_t)((uint64_t)q * blockIdx.x / a.group);
        const uint32_t i1 = (uint32_t)((uint64_t)q * (blockIdx.x + 1) / a.group);
        for (uint32_t base = i0 + (threadIdx.x & ~31u); base < i1; base += SS_BLOCK) {
            const uint32_t i = base + lane;
            int32_t v = 0;
            OffT row = 0;
            uint32_t deg = 0;
            if (i < i1) {
                v = __ldcg(Q + i);
                row = __ldcg(R + i);
                deg = (uint32_t)(__ldg(a.ro + v + 1) - row);
            }
            ss_list_append(a, sh, L, tag + 1, i < i1, v, (uint32_t)row, deg);
        }
    }
    ++tag;
    if (!narrow_exchange_wide<SS_BLOCK>(a.lines + (tag & 1) * SS_LIST_BLOCKS, sh, group, tag, a.ctl, a.timeout_ns)) return false;
    uint32_t ran = 0;
    for (;;) {
        if (s_st.q == 0 || s_st.T > a.list_T * a.group || sh.most > ss_list_pieces(a.list_T)) break;
        if (ran == a.list_rounds && a.group < gridDim.x) {   // the other blocks' wait is bounded: renew it
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                SsState st = s_st;
                st.list = LIST_ON;
                memcpy((void *)a.ctl->hstate[(bar.gen + 1) & 1], &st, sizeof st);
            }
            if (!flag_barrier(bar)) return false;
            ran = 0;
        }
        ++ran;
        const int L = s_st.L;
        if (STATS && blockIdx.x == 0 && threadIdx.x == 0 && L < GRX_MAX_LEVELS_STATS) {
            a.stats->level_t0[L] = grx_globaltimer();
            a.stats->dir[L] = 0;
            a.stats->frontier[L] = s_st.q;
            a.stats->edges_examined[L] = s_st.T;
            a.stats->vertices_scanned[L] = s_st.q;
            a.stats->discovered[L] = 0;
            a.stats->levels = L + 1;
        }
        list_round(a, s_st, sh, tag);
        ++tag;
        if (!narrow_exchange_wide<SS_BLOCK>(a.lines + (tag & 1) * SS_LIST_BLOCKS, sh, group, tag, a.ctl, a.timeout_ns))
            return false;
        if (threadIdx.x == 0) {
            s_st.L = L + 1;
            s_st.q = sh.verts;
            s_st.T = sh.edges;
            if (STATS && blockIdx.x == 0 && L < GRX_MAX_LEVELS_STATS) a.stats->discovered[L] = sh.verts;
        }
        __syncthreads();
    }
    const int L = s_st.L;
    if (s_st.q) {                                // back to a queue: vertex, edge prefix, row start
        uint32_t x0, x1, x2, vb, eb, x3;         // vertices and edges of the blocks before
        {
            uint32_t sv = 0, se = 0;
            for (uint32_t b = threadIdx.x; b < blockIdx.x; b += SS_BLOCK) {
                sv += sh.line_verts[b];
                se += sh.line_edges[b];
            }
            block_scan3<SS_BLOCK>(sv, se, 0u, x0, x1, x2, vb, eb, x3);
        }
        int32_t *Q = pick3(a.Q[0], a.Q[1], a.Q[2], L % 3);
        uint32_t *E = pick3(a.E[0], a.E[1], a.E[2], L % 3);
        OffT *R = pick3(a.R[0], a.R[1], a.R[2], L % 3);
        const int32_t *mine = a.verts + ((size_t)(L & 1) * a.group + blockIdx.x) * ss_list_verts(a.list_T);
        const uint32_t n = sh.own;
        for (uint32_t base = 0; base < n; base += SS_BLOCK) {
            const uint32_t i = base + threadIdx.x;
            int32_t v = 0;
            OffT rb = 0;
            uint32_t deg = 0;
            if (i < n) {
                v = __ldcg(mine + i);
                rb = __ldg(a.ro + v);
                deg = (uint32_t)(__ldg(a.ro + v + 1) - rb);
            }
            uint32_t e0, esum, t1, t2;
            block_scan3<SS_BLOCK>(deg, 0u, 0u, e0, x1, x2, esum, t1, t2);
            if (i < n) {
                Q[vb + i] = v;
                E[vb + i] = eb + e0;
                R[vb + i] = rb;
            }
            eb += esum;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.ctl->narrow_epoch += 1;                // no block reads it before the next grid barrier
        for (int i = 0; i < 4; ++i) {
            a.ctl->qpack[i] = 0ull;
            a.ctl->wq[i] = 0u;
        }
        SsState st = s_st;
        st.list = LIST_OFF;                      // a round that did not fit its segments may look small
        if (st.q) {
            ss_set_kind(a, st);
        } else {
            st.nfar = ld_relaxed_u32(&a.ctl->farcnt[st.fsel]);
            if (a.delta && st.nfar > 0) st.op = SOP_FARMIN;
            else st.done = 1;
        }
        memcpy((void *)a.ctl->hstate[(bar.gen + 1) & 1], &st, sizeof st);
    }
    return true;
}

// A stretch of list rounds, for every block of the grid: from s_st to the s_st
// that all go on from.  false: a wait gave up.
template <typename OffT, bool STATS>
__device__ __forceinline__ bool list_rounds(const SsspArgs<OffT> &a, SsState &s_st, NarrowShared<SS_LIST_BLOCKS> &sh,
                                            FlagBarrier &bar) {
    const bool in = blockIdx.x < a.group;
    if (in && !list_run<OffT, STATS>(a, s_st, sh, bar)) return false;
    do {
        if (!flag_barrier(bar, in ? 32 : 500)) return false;
        if (threadIdx.x == 0) {
            static_assert(sizeof(SsState) <= sizeof a.ctl->hstate[0] && sizeof(SsState) % 4 == 0, "handed over by words");
            const uint32_t *h = (const uint32_t *)a.ctl->hstate[bar.gen & 1];
            uint32_t words[sizeof(SsState) / 4];
            for (int i = 0; i < (int)(sizeof(SsState) / 4); ++i) words[i] = __ldcg(h + i);
            memcpy(&s_st, words, sizeof s_st);
        }
        __syncthreads();
    } while (s_st.list == LIST_ON);
    return true;
}

// State of the next phase.
template <typename OffT>
__device__ SsState ss_next(const SsspArgs<OffT> &a, const SsState &st, bool stats) {
    SsState ns = st;
    ns.list = 0;
    if (st.op == SOP_RELAX && st.bmp) {
        ns.op = SOP_FINAL;
        return ns;
    }
    if (st.op == SOP_FARMIN) {
        const uint32_t m = ld_relaxed_u32(&a.ctl->farmin[st.fsel]);
        ns.op = SOP_FARSPLIT;
        ns.oldthr = st.thr;
        ns.thr = m == 0xffffffffu ? st.thr
                                  : (m > 0xffffffffu - a.delta ? 0xffffffffu : m + a.delta);
        if (m == 0xffffffffu) ns.thr = 0xffffffffu;              // every entry stale: one last split
        return ns;
    }
    uint32_t q, T;
    int L;
    if (st.op == SOP_FARSPLIT) {                                 // Q_L came from the far pile
        L = st.L;
        ns.fsel = st.fsel ^ 1;
        ns.nfar = ld_relaxed_u32(&a.ctl->farcnt[ns.fsel]);
    } else {                                                     // end of round st.L
        L = st.L + 1;
        ns.nfar = ld_relaxed_u32(&a.ctl->farcnt[st.fsel]);
    }
    const unsigned long long pk = ld_relaxed_u64(&a.ctl->qpack[L & 3]);
    q = (uint32_t)(pk >> 32);
    T = (uint32_t)pk;
    if (stats && blockIdx.x == 0 && st.op != SOP_FARSPLIT && st.L < GRX_MAX_LEVELS_STATS)
        a.stats->discovered[st.L] = q;
    ns.L = L;
    ns.q = q;
    ns.T = T;
    if (q > 0) {
        ns.op = SOP_RELAX;
        ss_set_kind(a, ns);
    } else if (a.delta && ns.nfar > 0) {
        ns.op = SOP_FARMIN;
        ns.bmp = 0;
    } else {
        ns.done = 1;
    }
    return ns;
}

// Shared memory of a block: list rounds and the others do not overlap.
template <typename OffT>
union SsSmem {
    SsWarpSmem<OffT> w[SS_WARPS];
    NarrowShared<SS_LIST_BLOCKS> list;
};

// LIST (list rounds) is a variant of its own: other graphs keep their registers.
template <typename OffT, bool STATS, bool LIST>
__global__ void __launch_bounds__(SS_BLOCK, SS_MIN_BLOCKS) k_sssp_persistent(const __grid_constant__ SsspArgs<OffT> a) {
    __shared__ SsState s_st;
    extern __shared__ __align__(16) unsigned char ss_dsmem[];
    SsSmem<OffT> &sm = *reinterpret_cast<SsSmem<OffT> *>(ss_dsmem);
    SsWarpSmem<OffT> &w = sm.w[threadIdx.x >> 5];
    FlagBarrier bar{a.bar_flags, &a.ctl->bar_release, a.ctl, a.timeout_ns, 0u};
    if (threadIdx.x == 0) {
        SsState s;
        memset(&s, 0, sizeof s);
        const uint32_t deg = (uint32_t)(a.ro[a.src + 1] - a.ro[a.src]);
        s.op = SOP_RELAX;
        s.q = deg ? 1u : 0u;
        s.T = deg;
        s.done = deg == 0;
        s.thr = a.delta ? a.delta : 0xffffffffu;
        ss_set_kind(a, s);
        s_st = s;
    }
    __syncthreads();
    for (;;) {
        for (;;) {
            const SsState &st = s_st;
            if (st.done || (LIST && list_may_start(a, st))) break;
            const int L = st.L;
            if (st.op == SOP_RELAX && blockIdx.x == 0 && threadIdx.x == 0) {
                a.ctl->qpack[(L + 2) & 3] = 0ull;
                a.ctl->wq[(L + 2) & 3] = 0u;
                if (STATS && L < GRX_MAX_LEVELS_STATS) {
                    a.stats->level_t0[L] = grx_globaltimer();
                    a.stats->dir[L] = 0;
                    a.stats->frontier[L] = st.q;
                    a.stats->edges_examined[L] = st.T;
                    a.stats->vertices_scanned[L] = st.q;
                    a.stats->levels = L + 1;
                }
            }
            if (st.op == SOP_FINAL) changed_to_queue<OffT>(a, st, w.list);
            else if (st.op == SOP_FARMIN) far_min<OffT>(a, st);
            else if (st.op == SOP_FARSPLIT) far_split<OffT>(a, st);
            else if (st.bmp) relax_round<OffT, true>(a, st, w);
            else relax_round<OffT, false>(a, st, w);
            if (!flag_barrier(bar)) return;
            if (threadIdx.x == 0) s_st = ss_next(a, st, STATS);
            __syncthreads();
        }
        if (!LIST || s_st.done) break;
        if constexpr (LIST)
            if (!list_rounds<OffT, STATS>(a, s_st, sm.list, bar)) return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.ctl->levels_run = s_st.L;
        if (STATS && s_st.L <= GRX_MAX_LEVELS_STATS) a.stats->level_t0[s_st.L] = grx_globaltimer();
    }
}

template <typename OffT>
__global__ void k_sssp_init(int32_t src, const OffT *ro, uint32_t *dist, int32_t *Q0, uint32_t *E0, OffT *R0,
                            TravCtl *ctl, DevStats *stats, int stats_on) {
    const OffT b = ro[src];
    const uint32_t deg = (uint32_t)(ro[src + 1] - b);
    dist[src] = 0;
    Q0[0] = src;
    E0[0] = 0;
    R0[0] = b;
    ctl->qpack[0] = deg ? ((1ull << 32) | deg) : 0ull;
    for (int i = 1; i < 4; ++i) ctl->qpack[i] = 0ull;
    for (int i = 0; i < 4; ++i) ctl->wq[i] = 0u;
    ctl->farcnt[0] = 0u;
    ctl->farcnt[1] = 0u;
    ctl->farmin[0] = 0xffffffffu;
    ctl->farmin[1] = 0xffffffffu;
    ctl->narrow_epoch += 1;                  // as does every stretch of list rounds: a call that gave up left its tags
    if (stats_on) stats->levels = 0;
}

// The list rounds' buffers of g for grids of up to `blocks` (once; NULL without
// memory, or while s is captured: the rounds then run on the queue).
grx_status ss_list_buffers(grx_graph *g, int blocks, cudaStream_t s) {
    if (g->ss_lines || blocks > SS_BLOCK || grx_capturing(s)) return GRX_OK;
    // rounds of up to 3,072 edges a block, a quarter of the graph's at most
    const int64_t share = g->ne / 4 / blocks;
    const uint32_t t = (uint32_t)(share < 192 ? 192 : (share > 3072 ? 3072 : share));
    const size_t lines = 2 * SS_LIST_BLOCKS * sizeof(NarrowWord);
    const size_t pieces = 2 * (size_t)blocks * ss_list_pieces(t) * sizeof(NarrowWord);
    const size_t verts = 2 * (size_t)blocks * ss_list_verts(t) * sizeof(int32_t);
    char *p = (char *)grx_alloc_optional(g, lines + pieces + verts, s);
    if (!p) return GRX_OK;
    GRX_CUDA(cudaMemsetAsync(p, 0, lines + pieces, s));           // tag 0 is never used
    g->ss_lines = p;
    g->ss_list_T = t;
    g->ss_list_blocks = blocks;
    return GRX_OK;
}

template <typename OffT, bool STATS, bool LIST>
grx_status launch_persistent(grx_graph *g, SsspArgs<OffT> &a, int32_t src, uint32_t *dist, const grx_opts *o,
                             cudaStream_t s) {
    k_sssp_init<OffT><<<1, 1, 0, s>>>(src, a.ro, dist, g->qv[0], g->qe[0], a.R[0], g->ctl, g->stats,
                                      o->collect_stats);
    GRX_CUDA(cudaGetLastError());
    constexpr int smem = (int)sizeof(SsSmem<OffT>);
    static unsigned long long ready = 0;         // devices whose kernel may use this much shared memory
    const unsigned long long bit = 1ull << (g->ctx->device & 63);
    if (!(ready & bit) || g->ctx->device > 63) {
        GRX_CUDA(cudaFuncSetAttribute((const void *)k_sssp_persistent<OffT, STATS, LIST>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        ready |= bit;
    }
    static int per_sm = -1;
    if (per_sm < 0) {
        GRX_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sssp_persistent<OffT, STATS, LIST>,
                                                               SS_BLOCK, smem));
        if (per_sm < 1) return grx_fail(GRX_ECUDA, "sssp: persistent kernel does not fit on an SM");
    }
    int max_grid = per_sm * g->ctx->num_sms;
    if (max_grid > GRX_MAX_GRID) max_grid = GRX_MAX_GRID;
    int blocks = grx_grid(o, SS_BLOCK, max_grid);
    if (LIST) {
        // The group: rounds of deep graphs of less than 1M (4M) vertices hold 20,000
        // edges or fewer (100,000), and 64 blocks (one an SM) then lose less in a round's
        // work than they save in its exchange.  Grids of 200^2 / 500^2 / 1,500^2 /
        // 4,096^2, us per round with 64 / 152 / 304 blocks in the group: 6.0 / 7.2 / 9.0,
        // 6.2 / 7.2 / 8.4, 10.9 / 9.2 / 9.1, 18.2 / 14.4 / 13.1.  Larger rounds run on
        // the whole grid.
        int few = g->nv < (1 << 20) ? 64 : (g->nv < (1 << 22) ? g->ctx->num_sms : max_grid);
        if (few > max_grid) few = max_grid;
        const grx_status st = ss_list_buffers(g, few, s);
        if (st != GRX_OK) return st;
        if (g->ss_lines) {
            grx_uses_optional(g, s);
            const uint32_t t = g->ss_list_T;
            a.lines = (NarrowWord *)g->ss_lines;
            a.pieces = a.lines + 2 * SS_LIST_BLOCKS;
            a.verts = (int32_t *)(a.pieces + 2 * (size_t)g->ss_list_blocks * ss_list_pieces(t));
            a.list_T = t;
            a.group = (uint32_t)(blocks < g->ss_list_blocks ? blocks : g->ss_list_blocks);
            // A grid of the group alone where every round is that small: uniform random
            // graphs of 0.2M / 0.8M / 1.2M / 3.6M edges on 64 blocks 293 / 379 / 453 / 754 us,
            // on the full grid 322 / 389 / 435 / 567; grids of 200^2 / 500^2 2.5 / 7.0 ms and
            // 2.7 / 7.5.
            if (o->grid_blocks <= 0 && g->nv < (1 << 20) && g->ne < (1 << 20)) blocks = g->ss_list_blocks;
            // a list round takes some ten microseconds: far less than the bound on a wait
            const unsigned long long n = a.timeout_ns >> 16;
            a.list_rounds = n < 1 ? 1u : (n > 256 ? 256u : (uint32_t)n);
            // lists are the better form of a large round too, up to their limit,
            // unless the caller set the line for the changed bitmap
            if (o->push_bitmap == 0.f && a.bmp_min_T <= t * a.group) a.bmp_min_T = t * a.group + 1;
        }
    }
    GRX_CUDA(cudaMemsetAsync(g->bar_flags, 0, sizeof(unsigned int) * (size_t)blocks, s));
    GRX_CUDA(cudaMemsetAsync(&g->ctl->bar_release, 0, sizeof(unsigned int), s));
    void *args[] = {(void *)&a};
    if (o->ev_begin) GRX_CUDA(cudaEventRecord((cudaEvent_t)o->ev_begin, s));
    GRX_CUDA(cudaLaunchCooperativeKernel((const void *)k_sssp_persistent<OffT, STATS, LIST>, dim3(blocks),
                                         dim3(SS_BLOCK), args, smem, s));
    if (o->ev_end) GRX_CUDA(cudaEventRecord((cudaEvent_t)o->ev_end, s));
    return GRX_OK;
}

template <typename OffT, bool STATS>
grx_status launch_typed(grx_graph *g, int32_t src, uint32_t *dist, const grx_opts *o,
                        cudaStream_t s) {
    SsspArgs<OffT> a;
    a.nv = g->nv;
    a.words = g->words;
    a.ro = (const OffT *)g->ro;
    a.col = g->col;
    a.w = g->w;
    a.dist = dist;
    a.stamp = g->stamp;
    a.cbits = g->fbits[0];
    a.fbits = g->fbits[1];
    a.far[0] = g->ulist[0];
    a.far[1] = g->ulist[1];
    a.delta = o->sssp_delta;
    for (int i = 0; i < 3; ++i) {
        a.Q[i] = g->qv[i];
        a.E[i] = g->qe[i];
        a.R[i] = (OffT *)g->qr[i];
    }
    a.ctl = g->ctl;
    a.bar_flags = g->bar_flags;
    a.stats = g->stats;
    a.timeout_ns = grx_timeout_ns(o);
    a.src = src;
    a.even = !grx_has_hubs(g);
    a.lines = a.pieces = nullptr;
    a.verts = nullptr;
    a.list_T = a.group = a.list_rounds = 0;
    {   // reduction rounds when a round's edges reach push_bitmap * nv (0 = 1/8, < 0 = never)
        const double pb = o->push_bitmap == 0.f ? 0.125 : (double)o->push_bitmap;
        const double t = pb * (double)g->nv;
        a.bmp_min_T = pb < 0 ? 0xffffffffu : (t < 1.0 ? 1u : (t > 4294967295.0 ? 0xffffffffu : (uint32_t)t));
    }
    // List rounds on graphs of few edges a vertex and no hubs: thousands of rounds
    // of small rows (with hubs, R-MAT of edge factor 4, a handful of rounds, most of
    // the work in two or three of them).
    return g->ne < 8ll * g->nv && g->max_deg <= 64 ? launch_persistent<OffT, STATS, true>(g, a, src, dist, o, s)
                               : launch_persistent<OffT, STATS, false>(g, a, src, dist, o, s);
}

}  // namespace

grx_status grx_sssp_launch(grx_graph *g, int32_t src, uint32_t *dist, const grx_opts *o,
                           cudaStream_t s) {
    const size_t nv = (size_t)g->nv;
    GRX_CUDA(cudaMemsetAsync(dist, 0xff, nv * 4, s));
    GRX_CUDA(cudaMemsetAsync(g->stamp, 0, nv * 4, s));
    GRX_CUDA(cudaMemsetAsync(g->fbits[0], 0, (size_t)g->words * 4, s));
    if (o->sssp_delta) GRX_CUDA(cudaMemsetAsync(g->fbits[1], 0, (size_t)g->words * 4, s));
    if (o->collect_stats) GRX_CUDA(cudaMemsetAsync(g->stats, 0, sizeof(DevStats), s));
    if (g->off64)
        return o->collect_stats ? launch_typed<int64_t, true>(g, src, dist, o, s)
                                : launch_typed<int64_t, false>(g, src, dist, o, s);
    return o->collect_stats ? launch_typed<int32_t, true>(g, src, dist, o, s)
                            : launch_typed<int32_t, false>(g, src, dist, o, s);
}
