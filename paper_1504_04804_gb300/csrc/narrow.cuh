// Narrow levels: what a traversal does while its frontier is small.
//
// A level of a few thousand edges is all latency.  Over the whole persistent
// grid it costs a barrier among 456 blocks and a chain of some ten dependent
// trips to L2 or DRAM, 16 us on a 4096 x 4096 grid, with work for 40 of the
// 3,648 warps.  So while the frontier stays small, the first GRX_NARROW_BLOCKS
// blocks of the grid run level after level among themselves; the others wait
// for them at the grid barrier.
//  * Barrier and counters are one trip: at the end of a level each block
//    publishes a line of counts, and every block of the group reads all lines.
//    No block gathers for the others, and no counter is read afterwards.
//  * The frontier is a list of pieces of at most NARROW_PIECE edges, one
//    segment per block, appended through shared-memory counters (no global
//    append counter).  A piece is all a lane needs to reach its column: no
//    degree prefix, no search, no row lookup.
//  * Lines and pieces are single 16-byte words that carry their own tag, unique
//    over the life of the workspace: a reader waits for the tag, and the writer
//    needs no fence between data and flag (a level of 20 edges 4.8 -> 3.5 us).
//    Only what the blocks leave for each other beside them has to be fenced (BFS:
//    the frontier bitmaps where they are kept; SSSP: the distances).
#pragma once

#include "grx_internal.cuh"

// 64 blocks: two lines per polling lane; a level of 15,000 edges is one piece per
// quad of lanes.
#define GRX_NARROW_BLOCKS 64
constexpr int NARROW_PIECE = 4;              // edges per piece: a quad of lanes
constexpr uint32_t NARROW_PIECES = 2048;     // pieces a block's segment holds
constexpr uint32_t NARROW_MAX_T = 32768;     // edges of a narrow frontier, at most
// Vertices a block can find in one level: its share of the pieces (whole steps of
// 12 warps x 8 pieces x 2), four edges each.
constexpr uint32_t NARROW_VERTS = NARROW_PIECE * (NARROW_MAX_T / GRX_NARROW_BLOCKS + 12 * 8 * 2);

// A 16-byte word that is written and read as one.
struct alignas(16) NarrowWord {
    unsigned long long lo, hi;
};
// Tag: epoch (of calls and stretches of narrow levels, in TravCtl) << 32 | exchange, 63 bits.
// Line:  lo = tag << 1, hi = edges | vertices << 32 | pieces (saturated) << 48.
// Piece: lo = tag << 1 | (edges - 1) >> 1, hi = first edge | vertex << 32 | ((edges - 1) & 1) << 63.

struct NarrowBuffers {
    NarrowWord lines[2][GRX_NARROW_BLOCKS];                    // by exchange parity
    NarrowWord pieces[2][GRX_NARROW_BLOCKS][NARROW_PIECES];    // by level parity
    int32_t verts[3][GRX_NARROW_BLOCKS][NARROW_VERTS];         // by level mod 3
};

#ifdef __CUDACC__
// Blocks of the group, and the edges of the largest frontier it takes.
__device__ __forceinline__ uint32_t narrow_group() { return min((uint32_t)GRX_NARROW_BLOCKS, gridDim.x); }
__device__ __forceinline__ uint32_t narrow_max_T() { return NARROW_MAX_T / GRX_NARROW_BLOCKS * narrow_group(); }

__device__ __forceinline__ void narrow_store(NarrowWord *p, unsigned long long lo, unsigned long long hi) {
    asm volatile("{\n\t.reg .b128 w;\n\tmov.b128 w, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], w;\n\t}" ::"l"(p),
                 "l"(lo), "l"(hi)
                 : "memory");
}

__device__ __forceinline__ NarrowWord narrow_load(const NarrowWord *p) {
    NarrowWord w;
    asm volatile("{\n\t.reg .b128 w;\n\tld.relaxed.gpu.global.b128 w, [%2];\n\tmov.b128 {%0, %1}, w;\n\t}"
                 : "=l"(w.lo), "=l"(w.hi)
                 : "l"(p)
                 : "memory");
    return w;
}

// Shared state of a block of a group of at most NB.
template <int NB>
struct NarrowShared {
    unsigned long long got;                  // appended: pieces << 32 | vertices
    unsigned long long got_edges;
    uint32_t first[NB + 2];                  // pieces before each block's segment
    uint32_t line_verts[NB], line_edges[NB]; // of the last exchange
    uint32_t verts, edges;                   // its totals
    uint32_t most;                           // its largest segment (pieces)
    uint32_t own;                            // vertices of this block's segment
    int ok;
};

// One thread: the block's line of exchange `tag`.
template <int NB>
__device__ __forceinline__ void narrow_publish(NarrowWord *lines, NarrowShared<NB> &sh, unsigned long long tag,
                                               bool fence) {
    const unsigned long long got = sh.got, edges = sh.got_edges;
    const uint32_t pieces = (uint32_t)(got >> 32), verts = (uint32_t)got;
    if (fence) __threadfence();
    narrow_store(lines + blockIdx.x, tag << 1,
                 (edges & 0xffffffffull) | (unsigned long long)min(verts, 0xffffu) << 32 |
                     (unsigned long long)min(pieces, 0xffffu) << 48);
    sh.own = verts;
    sh.got = 0ull;
    sh.got_edges = 0ull;
}

// Waits for a line of exchange `tag`; false: gave up.
__device__ __forceinline__ bool narrow_collect(const NarrowWord *line, unsigned long long tag, uint32_t &verts,
                                               uint32_t &pieces, uint32_t &edges, unsigned long long timeout_ns) {
    for (unsigned long long t0 = 0;;) {
        const NarrowWord w = narrow_load(line);
        if (w.lo == tag << 1) {
            edges = (uint32_t)w.hi;
            verts = (uint32_t)(w.hi >> 32) & 0xffffu;
            pieces = (uint32_t)(w.hi >> 48);
            return true;
        }
        const unsigned long long now = grx_globaltimer();
        if (t0 == 0) t0 = now;
        if (now - t0 > timeout_ns) return false;
    }
}

// Publishes what the block appended, runs ahead() and waits for the group's
// lines of the same tag (ahead: loads whose use can wait until the next level;
// the trip of the lines hides them).  Pieces need no more than that (they carry the tag too); with `fence`,
// other memory written by the group's blocks before is visible after it.
// Every wait is bounded; false: gave up (GRX_ETIMEOUT recorded).
template <typename Ahead>
__device__ __forceinline__ bool narrow_exchange(NarrowWord *lines, NarrowShared<GRX_NARROW_BLOCKS> &sh, int group,
                                                unsigned long long tag, bool fence, TravCtl *ctl,
                                                unsigned long long timeout_ns, Ahead &&ahead) {
    __syncthreads();
    if (threadIdx.x == 0) narrow_publish(lines, sh, tag, fence);
    ahead();
    if (threadIdx.x < 32) {
        const unsigned int lane = threadIdx.x;
        uint32_t q[2] = {0u, 0u}, p[2] = {0u, 0u}, e[2] = {0u, 0u};
        bool ok = true;
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if ((int)lane * 2 + k < group)
                ok = ok && narrow_collect(lines + lane * 2 + k, tag, q[k], p[k], e[k], timeout_ns);
        if (fence) __threadfence();
        ok = __all_sync(GRX_FULL_MASK, ok);
        uint32_t cp = p[0] + p[1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(GRX_FULL_MASK, cp, o);
            if (lane >= (unsigned)o) cp += y;
        }
        const uint32_t verts = __reduce_add_sync(GRX_FULL_MASK, q[0] + q[1]);
        const uint32_t edges = __reduce_add_sync(GRX_FULL_MASK, e[0] + e[1]);   // < 2^32 in a graph
        const uint32_t most = __reduce_max_sync(GRX_FULL_MASK, max(p[0], p[1]));
        *reinterpret_cast<uint2 *>(&sh.line_verts[2 * lane]) = make_uint2(q[0], q[1]);
        *reinterpret_cast<uint2 *>(&sh.line_edges[2 * lane]) = make_uint2(e[0], e[1]);
        sh.first[2 * lane] = cp - p[0] - p[1];
        sh.first[2 * lane + 1] = cp - p[1];
        if (lane == 31) {
            sh.first[GRX_NARROW_BLOCKS] = cp;
            sh.verts = verts;
            sh.edges = edges;
            sh.most = most;
            sh.ok = ok;
            if (!ok) grx_set_status(ctl, GRX_ETIMEOUT);
        }
    }
    __syncthreads();
    return sh.ok != 0;
}

// The same for a group of up to NT = blockDim.x blocks: every thread waits for a
// line.  What the blocks wrote before (distances: reductions, which nobody waits
// for) is visible to all of them after it: each block's writes come before thread
// 0's fence through the __syncthreads, the line after it, and a thread's fence
// after the line it read and before the block's next __syncthreads.
template <int NT, int NB>
__device__ __forceinline__ bool narrow_exchange_wide(NarrowWord *lines, NarrowShared<NB> &sh, int group,
                                                     unsigned long long tag, TravCtl *ctl,
                                                     unsigned long long timeout_ns) {
    static_assert(NT <= NB, "a line a thread");
    __shared__ uint32_t ws[4][NT / 32];              // per warp: pieces, vertices, edges, largest segment
    __syncthreads();
    if (threadIdx.x == 0) narrow_publish(lines, sh, tag, true);
    const unsigned int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t q = 0u, p = 0u, e = 0u;
    bool ok = true;
    if ((int)threadIdx.x < group) {
        ok = narrow_collect(lines + threadIdx.x, tag, q, p, e, timeout_ns);
        __threadfence();
    }
    uint32_t cp = p;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(GRX_FULL_MASK, cp, o);
        if (lane >= (unsigned)o) cp += y;
    }
    const uint32_t verts = __reduce_add_sync(GRX_FULL_MASK, q);
    const uint32_t edges = __reduce_add_sync(GRX_FULL_MASK, e);
    const uint32_t most = __reduce_max_sync(GRX_FULL_MASK, p);
    if (lane == 31) {
        ws[0][wid] = cp;
        ws[1][wid] = verts;
        ws[2][wid] = edges;
        ws[3][wid] = most;
    }
    ok = __syncthreads_and(ok);
    uint32_t before = 0, tp = 0, tv = 0, te = 0, tm = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) {
        const uint32_t x = ws[0][w];
        if ((unsigned)w < wid) before += x;
        tp += x;
        tv += ws[1][w];
        te += ws[2][w];
        tm = max(tm, ws[3][w]);
    }
    sh.first[threadIdx.x] = before + cp - p;
    sh.line_verts[threadIdx.x] = q;
    sh.line_edges[threadIdx.x] = e;
    for (int i = NT + (int)threadIdx.x; i <= NB; i += NT) sh.first[i] = tp;
    if (threadIdx.x == 0) {
        sh.verts = tv;
        sh.edges = te;
        sh.most = tm;
        if (!ok) grx_set_status(ctl, GRX_ETIMEOUT);
    }
    __syncthreads();
    return ok;
}

// Block and place in its segment of piece c of the frontier (c < first[NB]).
template <int NB>
__device__ __forceinline__ uint32_t narrow_find(const NarrowShared<NB> &sh, uint32_t c, uint32_t &at) {
    uint32_t b = 0;
#pragma unroll
    for (int o = NB / 2; o > 0; o >>= 1)
        if (sh.first[b + o] <= c) b += o;
    at = c - sh.first[b];
    return b;
}

// Waits for a piece's tag (its line was seen: the word is on its way); false:
// gave up.
__device__ __forceinline__ bool narrow_await(const NarrowWord *p, NarrowWord &w, unsigned long long tag, TravCtl *ctl,
                                             unsigned long long timeout_ns) {
    if (w.lo >> 1 == tag) return true;
    const unsigned long long t0 = grx_globaltimer();
    for (;;) {
        w = narrow_load(p);
        if (w.lo >> 1 == tag) return true;
        if (grx_globaltimer() - t0 > timeout_ns) {
            grx_set_status(ctl, GRX_ETIMEOUT);
            return false;
        }
    }
}

__device__ __forceinline__ uint32_t narrow_len(const NarrowWord &w) {
    return ((uint32_t)w.lo & 1u) * 2 + (uint32_t)(w.hi >> 63) + 1;
}
__device__ __forceinline__ uint32_t narrow_edge(const NarrowWord &w) { return (uint32_t)w.hi; }
__device__ __forceinline__ int32_t narrow_vertex(const NarrowWord &w) { return (int32_t)(w.hi >> 32 & 0x7fffffffu); }

// Piece k of vertex v's row.
__device__ __forceinline__ void narrow_write_piece(NarrowWord *p, unsigned long long tag, int32_t v, uint32_t row,
                                                   uint32_t deg, uint32_t k) {
    const uint32_t len1 = min((uint32_t)NARROW_PIECE, deg - k * NARROW_PIECE) - 1;
    narrow_store(p, tag << 1 | len1 >> 1,
                 (unsigned long long)(row + k * NARROW_PIECE) | (unsigned long long)(uint32_t)v << 32 |
                     (unsigned long long)(len1 & 1) << 63);
}

// Appends up to one vertex per lane (v, its row start and degree > 0 where
// `has`) to the block's segments, announced with `tag`: the vertex list (of
// vcap entries) and the pieces of its row (cap).  All 32 lanes call.
template <int NB>
__device__ __forceinline__ void narrow_append(NarrowShared<NB> &sh, NarrowWord *out, uint32_t cap, int32_t *verts,
                                              uint32_t vcap, unsigned long long tag, bool has, int32_t v, uint32_t row,
                                              uint32_t deg, TravCtl *ctl) {
    const unsigned int lane = threadIdx.x & 31;
    const unsigned int m = __ballot_sync(GRX_FULL_MASK, has);
    if (m == 0) return;
    const uint32_t np = has ? (deg + NARROW_PIECE - 1) / NARROW_PIECE : 0u;
    uint32_t x = np;
    const uint32_t d = has ? deg : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(GRX_FULL_MASK, x, o);
        if (lane >= (unsigned)o) x += y;
    }
    const uint32_t e = __reduce_add_sync(GRX_FULL_MASK, d);      // < 2^32: distinct rows of a graph
    unsigned long long base = 0;
    if (lane == 31) {
        base = atomicAdd(&sh.got, ((unsigned long long)x << 32) | (unsigned)__popc(m));
        atomicAdd(&sh.got_edges, (unsigned long long)e);
    }
    base = __shfl_sync(GRX_FULL_MASK, base, 31);
    if (has) {
        const uint32_t i = (uint32_t)base + __popc(m & lanemask_lt());
        if (i < vcap) verts[i] = v;
        else grx_set_status(ctl, GRX_EINVAL);            // only possible with a malformed graph
    }
    // pieces past the segment's end are dropped: the frontier then leaves the
    // narrow levels and is read from the vertex lists
    const uint32_t p0 = (uint32_t)(base >> 32) + x - np;
    if (np <= 8)
        for (uint32_t k = 0; k < np && p0 + k < cap; ++k)
            narrow_write_piece(out + p0 + k, tag, v, row, deg, k);
    unsigned int wide = __ballot_sync(GRX_FULL_MASK, np > 8);   // long rows: the warp together
    while (wide) {
        const int src = __ffs(wide) - 1;
        wide &= wide - 1;
        const uint32_t n = __shfl_sync(GRX_FULL_MASK, np, src), p = __shfl_sync(GRX_FULL_MASK, p0, src);
        const uint32_t dg = __shfl_sync(GRX_FULL_MASK, deg, src), rw = __shfl_sync(GRX_FULL_MASK, row, src);
        const int32_t u = __shfl_sync(GRX_FULL_MASK, v, src);
        for (uint32_t k = lane; k < n && p + k < cap; k += 32)
            narrow_write_piece(out + p + k, tag, u, rw, dg, k);
    }
}
#endif  // __CUDACC__
