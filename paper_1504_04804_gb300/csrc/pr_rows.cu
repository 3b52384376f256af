// PageRank over degree-sorted rows.
//
// What bounds a PageRank iteration is the gather c[col[e]]: one random 4-byte
// load per edge.  In CSR order each costs an L1 tag and an L2 sector of its
// own (5 % L1 hits), and past R-MAT scale 24 the 4*nv-byte array c outgrows L2
// as well.  Three things follow from relabelling the non-isolated vertices by
// falling degree, once per graph:
//  * c is compact (4 bytes per non-isolated vertex) and its most-read entries
//    sit together at the front.  Each SM keeps the first entries in shared
//    memory, where a warp's 32 random reads cost a few bank conflicts instead
//    of 32 tags and sectors; the rest share cache lines with entries that are
//    about as popular, so L1 and L2 hold more of what is read.
//  * Rows of nearly equal degree are neighbours, so rows of at most
//    PRS_SELL edges are stored 32 to a slice, transposed in int4 units (lane =
//    row): coalesced 16-byte column loads, no row search, no reduction.
//  * Longer rows take a warp each (int4 per lane, one shuffle reduction), and
//    rows past `longest` edges are cut into chunks of `chunk` edges whose
//    partial sums the row's last warp adds up in order: no float atomics, and
//    sums that do not depend on timing.
// Measured on GB300, per iteration, CSR order -> here: R-MAT 16 0.025 -> 0.012 ms,
// 22 0.628 -> 0.235 ms, 24 3.07 -> 1.17 ms, 26 16.9 -> 5.9 ms (the columns alone
// would take 0.075 ms at R-MAT 22, 1.2 ms at 26).  At R-MAT 22 55 % of the gathers
// are served by shared memory; the others move 9-10 TB/s of sectors out of L2,
// which is what bounds it (L1 and L2 both 62 % busy, DRAM 2 TB/s).  Sorting each
// row's columns by label as well would merge only 5-8 % of the sectors.
// Where CSR order is local already it gains less: a grid of 4096 x 4096 0.225 ->
// 0.145 ms, a ring of 16M vertices with eight neighbours 0.367 -> 0.137.
// The sorted copy costs 4 bytes per edge (plus padding) and one to three CSR-order
// iterations to build; pagerank.cu says when it is built.
#include "grx_internal.cuh"

namespace {

constexpr int PRS_BLOCK = 1024;
constexpr int PRS_WARPS = PRS_BLOCK / 32;
constexpr int PRS_SELL = 128;                // rows up to this degree go to slices
constexpr int PRS_KEYS = 512;                // degree buckets
constexpr int PRS_SORT_BLOCK = 512;
// Entries of c kept in shared memory.  What they take is taken from L1, where a
// load in flight holds a line, so each size fills one of the SM's splits (164 KB /
// 100 KB shared).  Iteration by size of the table, 100 / 132 / 164 KB: R-MAT 22
// 0.257 / 0.241 / 0.235 ms, 24 1.21 / 1.19 / 1.17, 25 2.71 / 2.70 / 2.75,
// 26 5.96 / 6.34 / 7.40 (200 KB at R-MAT 22: 0.47).  Past about half of L2, c is
// fetched from DRAM and more loads have to be in flight: the smaller table.
constexpr int PRS_HOT = 41216, PRS_HOT_BIG = 24832;
constexpr int64_t PRS_BIG = (64 << 20) / 4;  // rows from which on PRS_HOT_BIG is used

// What the build leaves for the iterations (device memory).
struct PrsHeader {
    uint32_t n_long;                         // rows [0, n_long): chunks
    uint32_t n_warp;                         // rows [n_long, n_warp): a warp each
    uint32_t n_chunk;
    uint32_t n_slice;                        // slices of rows [n_warp, n)
    uint32_t sell_base;                      // first int4 of the slices
    uint32_t sell_first[PRS_SELL + 1];       // by degree: first slice led by such a row ...
    uint32_t sell_unit[PRS_SELL + 1];        // ... and its offset (units of 32 int4)
};

// Degree bucket, rising with the degree: exact up to PRS_SELL, then eight per
// power of two (bucket edges at powers of two + 1).
__host__ __device__ __forceinline__ int prs_key_log(int lg, int sub) { return PRS_SELL + (lg - 7) * 8 + sub; }

__device__ __forceinline__ int prs_key(uint32_t deg) {
    if (deg <= PRS_SELL) return (int)deg - 1;
    const uint32_t x = deg - 1;
    const int lg = 31 - __clz(x);
    return prs_key_log(lg, (int)(x >> (lg - 3)) & 7);
}

// int4 units a row takes among the long and warp rows (0: a slice row).
__device__ __forceinline__ uint32_t prs_units(uint32_t deg, int chunk_shift, uint32_t longest) {
    if (deg <= PRS_SELL) return 0u;
    if (deg <= longest) return (deg + 3) >> 2;
    return ((deg + (1u << chunk_shift) - 1) >> chunk_shift) << (chunk_shift - 2);
}

// Adds a row of `units` to its bucket's word (rows << 32 | units) and returns what
// was there before it.  All 32 lanes call; slot < 0: no row.  Rows without units
// go in together, one atomic per warp and bucket: on graphs whose rows are all
// alike every lane has the same one (sorting a grid of 4096 x 4096 took 3.6 ms
// with an atomic per row, twice what a CSR-order iteration saves in 20).
__device__ __forceinline__ unsigned long long prs_add(unsigned long long *h, int slot, uint32_t units) {
    const unsigned int same = __match_any_sync(GRX_FULL_MASK, units ? -1 : slot);
    unsigned long long before = 0;
    if (units) {
        before = atomicAdd(&h[slot], (1ull << 32) | units);
    } else if (slot >= 0) {
        const int lead = __ffs(same) - 1;
        if ((int)(threadIdx.x & 31) == lead) before = atomicAdd(&h[slot], (unsigned long long)__popc(same) << 32);
        before = __shfl_sync(same, before, lead) + ((unsigned long long)__popc(same & lanemask_lt()) << 32);
    }
    return before;
}

// Per block of consecutive rows and bucket: (rows << 32 | int4 units).
__global__ void __launch_bounds__(PRS_SORT_BLOCK) k_prs_count(const uint32_t *__restrict__ aoff, int64_t n,
                                                              int64_t per, int chunk_shift, uint32_t longest,
                                                              unsigned long long *__restrict__ mat) {
    __shared__ unsigned long long h[PRS_KEYS];
    h[threadIdx.x] = 0ull;
    __syncthreads();
    const int64_t i1 = min(n, (int64_t)(blockIdx.x + 1) * per);
    for (int64_t i0 = (int64_t)blockIdx.x * per; i0 < i1; i0 += PRS_SORT_BLOCK) {
        const int64_t i = i0 + threadIdx.x;
        const uint32_t d = i < i1 ? aoff[i + 1] - aoff[i] : 0u;
        prs_add(h, d ? PRS_KEYS - 1 - prs_key(d) : -1, prs_units(d, chunk_shift, longest));
    }
    __syncthreads();
    mat[(int64_t)blockIdx.x * PRS_KEYS + threadIdx.x] = h[threadIdx.x];
}

// One block: exclusive prefix of mat in (falling degree, block) order, and the
// header.
__global__ void __launch_bounds__(PRS_KEYS) k_prs_scan(unsigned long long *__restrict__ mat, int nblocks,
                                                       int64_t n, int chunk_shift, int long_key,
                                                       PrsHeader *__restrict__ hdr) {
    __shared__ unsigned long long base[PRS_KEYS + 1];
    const int t = threadIdx.x;
    unsigned long long sum = 0;
#pragma unroll 8
    for (int b = 0; b < nblocks; ++b) sum += mat[(int64_t)b * PRS_KEYS + t];
    base[t + 1] = sum;
    if (t == 0) base[0] = 0ull;
    __syncthreads();
    for (int o = 1; o <= PRS_KEYS; o <<= 1) {        // inclusive scan of base[1..]
        const unsigned long long y = t + 1 > o ? base[t + 1 - o] : 0ull;
        __syncthreads();
        base[t + 1] += y;
        __syncthreads();
    }
    unsigned long long run = base[t];
    for (int b = 0; b < nblocks; ++b) {
        const unsigned long long c = mat[(int64_t)b * PRS_KEYS + t];
        mat[(int64_t)b * PRS_KEYS + t] = run;
        run += c;
    }
    if (t == 0) {
        // slot KEYS-1-key holds bucket key: rows with key >= k end before slot KEYS-k
        const unsigned long long lng = base[PRS_KEYS - long_key], wrp = base[PRS_KEYS - PRS_SELL];
        const uint32_t nw = (uint32_t)(wrp >> 32);
        hdr->n_long = (uint32_t)(lng >> 32);
        hdr->n_warp = nw;
        hdr->n_chunk = (uint32_t)lng >> (chunk_shift - 2);
        hdr->n_slice = (uint32_t)((n - nw + 31) / 32);
        hdr->sell_base = ((uint32_t)wrp + 31u) & ~31u;
        uint32_t unit = 0;
        for (int d = PRS_SELL; d >= 1; --d) {        // slices led by a row of degree d
            const uint32_t r0 = (uint32_t)(base[PRS_KEYS - d] >> 32) - nw;
            const uint32_t r1 = (uint32_t)(base[PRS_KEYS - d + 1] >> 32) - nw;
            const uint32_t s0 = (r0 + 31) / 32, s1 = (r1 + 31) / 32;
            hdr->sell_first[d] = s0;
            hdr->sell_unit[d] = unit;
            unit += (s1 - s0) * (uint32_t)((d + 3) / 4);
        }
    }
}

// Places every row: its vertex, degree, first CSR edge, first int4 (long and
// warp rows), the chunks of long rows, and the vertex's new label.
__global__ void __launch_bounds__(PRS_SORT_BLOCK) k_prs_place(
    const int32_t *__restrict__ active, const uint32_t *__restrict__ aoff, int64_t n, int64_t per, int chunk_shift,
    uint32_t longest, const unsigned long long *__restrict__ mat, int32_t *__restrict__ vert,
    uint32_t *__restrict__ deg, uint32_t *__restrict__ src, uint32_t *__restrict__ unit, int32_t *__restrict__ chunk_row,
    int32_t *__restrict__ label) {
    __shared__ unsigned long long at[PRS_KEYS];
    at[threadIdx.x] = mat[(int64_t)blockIdx.x * PRS_KEYS + threadIdx.x];
    __syncthreads();
    const int64_t i1 = min(n, (int64_t)(blockIdx.x + 1) * per);
    for (int64_t i0 = (int64_t)blockIdx.x * per; i0 < i1; i0 += PRS_SORT_BLOCK) {
        const int64_t i = i0 + threadIdx.x;
        const uint32_t e0 = i < i1 ? aoff[i] : 0u, d = i < i1 ? aoff[i + 1] - e0 : 0u;
        const uint32_t units = prs_units(d, chunk_shift, longest);
        const unsigned long long p = prs_add(at, d ? PRS_KEYS - 1 - prs_key(d) : -1, units);
        if (!d) continue;
        const uint32_t r = (uint32_t)(p >> 32);
        vert[r] = active[i];
        deg[r] = d;
        src[r] = e0;
        label[active[i]] = (int32_t)r;
        if (units) unit[r] = (uint32_t)p;
        if (d > longest) {
            const uint32_t c0 = (uint32_t)p >> (chunk_shift - 2), nc = units >> (chunk_shift - 2);
            for (uint32_t k = 0; k < nc; ++k) chunk_row[c0 + k] = (int32_t)r;
        }
    }
}

struct PrsRows {
    const PrsHeader *hdr;
    const uint32_t *deg;
    const uint32_t *unit;
    const int32_t *chunk_row;
    int64_t n;
    int chunk_shift;
};

// First int4 of slice s, whose first row has degree d.
__device__ __forceinline__ int64_t prs_slice_at(const PrsHeader *hdr, uint32_t s, uint32_t d) {
    return (int64_t)hdr->sell_base +
           32ll * (__ldg(&hdr->sell_unit[d]) + (int64_t)(s - __ldg(&hdr->sell_first[d])) * ((d + 3) / 4));
}

// Relabelled columns of a stretch of one row: len edges from CSR edge e to int4
// q on, filled up to `padded` with label n (whose c is 0).
__device__ __forceinline__ void prs_copy(const int32_t *__restrict__ col, const int32_t *__restrict__ label, int32_t n,
                                         int64_t e, uint32_t len, uint32_t padded, int32_t *__restrict__ out, int64_t q) {
    for (uint32_t j = threadIdx.x & 31; j < padded; j += 32)
        out[q * 4 + j] = j < len ? __ldg(label + __ldcs(col + e + j)) : n;
}

// Fills the sorted columns; warps take chunks, warp rows and slices in turn.
// One label read (a random sector) per edge: as long as a CSR-order iteration.
__global__ void __launch_bounds__(256) k_prs_fill(PrsRows a, const int32_t *__restrict__ col,
                                                  const int32_t *__restrict__ label, const uint32_t *__restrict__ src,
                                                  int4 *__restrict__ out4) {
    const int64_t nw = (int64_t)gridDim.x * 8;
    const int64_t gw = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const unsigned int lane = threadIdx.x & 31;
    const int32_t n = (int32_t)a.n;
    int32_t *out = reinterpret_cast<int32_t *>(out4);
    const uint32_t n_long = a.hdr->n_long, n_warp = a.hdr->n_warp;
    const uint32_t per_chunk = 1u << (a.chunk_shift - 2);
    for (int64_t c = gw; c < a.hdr->n_chunk; c += nw) {
        const int32_t r = a.chunk_row[c];
        const uint32_t off = ((uint32_t)c * per_chunk - a.unit[r]) * 4;
        prs_copy(col, label, n, (int64_t)src[r] + off, min(per_chunk * 4, a.deg[r] - off), per_chunk * 4, out,
                 c * per_chunk);
    }
    for (int64_t r = n_long + gw; r < n_warp; r += nw) {
        const uint32_t d = a.deg[r];
        prs_copy(col, label, n, src[r], d, (d + 3) & ~3u, out, a.unit[r]);
    }
    for (int64_t s = gw; s < a.hdr->n_slice; s += nw) {
        const int64_t r = n_warp + s * 32 + lane;
        const uint32_t d = r < a.n ? a.deg[r] : 0u;
        const int64_t e = d ? src[r] : 0;
        const uint32_t d0 = __shfl_sync(GRX_FULL_MASK, d, 0);
        const int64_t at = prs_slice_at(a.hdr, (uint32_t)s, d0) + lane;
        for (uint32_t q = 0; q * 4 < d0; ++q) {
            int x[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = q * 4 + i < d ? __ldg(col + e + q * 4 + i) : -1;
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = x[i] >= 0 ? __ldg(label + x[i]) : n;
            out4[at + 32ll * q] = make_int4(x[0], x[1], x[2], x[3]);
        }
    }
}

__global__ void k_prs_init(const uint32_t *__restrict__ deg, int64_t n, float r0, float *__restrict__ c0,
                           float *__restrict__ c1) {
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x)
        c0[r] = r0 / (float)deg[r];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        c0[n] = 0.f;                                  // padding's label
        c1[n] = 0.f;
    }
}

// The c value of a label: shared memory for the first `hot`, else global.
__device__ __forceinline__ float prs_c(const float *hot_c, int hot, const float *__restrict__ c, int32_t u) {
    return u < hot ? hot_c[u] : __ldg(c + u);
}

// Two int4 of a lane: 8 labels.
struct PrsPair {
    int4 x, y;
};

// int4 k and k + step of the `units` int4 at p (padding where there is none).
__device__ __forceinline__ PrsPair prs_load(const int4 *__restrict__ p, uint32_t k, uint32_t step, uint32_t units, int none) {
    PrsPair r;
    r.x = k < units ? __ldcs(p + k) : make_int4(none, none, none, none);
    r.y = k + step < units ? __ldcs(p + k + step) : make_int4(none, none, none, none);
    return r;
}

__device__ __forceinline__ float prs_sum8(const PrsPair &v, const float *hot_c, int hot, const float *__restrict__ c) {
    const float a0 = prs_c(hot_c, hot, c, v.x.x), a1 = prs_c(hot_c, hot, c, v.x.y);
    const float a2 = prs_c(hot_c, hot, c, v.x.z), a3 = prs_c(hot_c, hot, c, v.x.w);
    const float b0 = prs_c(hot_c, hot, c, v.y.x), b1 = prs_c(hot_c, hot, c, v.y.y);
    const float b2 = prs_c(hot_c, hot, c, v.y.z), b3 = prs_c(hot_c, hot, c, v.y.w);
    return ((a0 + a1) + (a2 + a3)) + ((b0 + b1) + (b2 + b3));
}

// A lane's sum over `units` int4 at p, every 64th two from its own on; `v` holds
// its first two already.  The next two travel while two are gathered.
__device__ __forceinline__ float prs_rest(const int4 *__restrict__ p, uint32_t units, PrsPair v, int none,
                                          const float *hot_c, int hot, const float *__restrict__ c) {
    float s = 0.f;
    for (uint32_t k = (threadIdx.x & 31) + 64;; k += 64) {
        const bool more = k - (threadIdx.x & 31) < units;       // uniform
        PrsPair w = v;
        if (more) w = prs_load(p, k, 32, units, none);
        s += prs_sum8(v, hot_c, hot, c);
        if (!more) return s;
        v = w;
    }
}

struct PrsIter {
    PrsRows rows;
    const int4 *cols;
    const int32_t *vert;
    const float *c_in;
    float *c_out;
    float *rank;                                      // NULL but in the last iteration
    float *part;                                      // a partial sum per chunk
    unsigned int *done;                               // chunks of each long row that are summed
    int hot;
    float base, d;
};

__device__ __forceinline__ void prs_finish(const PrsIter &a, int64_t r, uint32_t deg, float sum) {
    const float v = a.base + a.d * sum;
    a.c_out[r] = v / (float)deg;
    if (a.rank) a.rank[__ldg(a.vert + r)] = v;
}

__global__ void __launch_bounds__(PRS_BLOCK, 1) k_prs_iter(PrsIter a) {
    extern __shared__ __align__(16) float hot_c[];
    const unsigned int lane = threadIdx.x & 31;
    const int hot = a.hot;
    {
        const int nv4 = hot >> 2;
        for (int i = threadIdx.x; i < nv4; i += PRS_BLOCK)
            reinterpret_cast<float4 *>(hot_c)[i] = __ldg(reinterpret_cast<const float4 *>(a.c_in) + i);
        for (int i = (nv4 << 2) + threadIdx.x; i < hot; i += PRS_BLOCK) hot_c[i] = __ldg(a.c_in + i);
    }
    __syncthreads();
    // Every class of work is in order of falling size and dealt out to the
    // warps in turn (neighbouring pieces to different SMs): the warps' shares
    // come out even without a work counter.
    const int64_t nw = (int64_t)gridDim.x * PRS_WARPS;
    const int64_t gw = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    const PrsRows &R = a.rows;
    const uint32_t n_long = R.hdr->n_long, n_warp = R.hdr->n_warp, n_chunk = R.hdr->n_chunk;
    const uint32_t per_chunk = 1u << (R.chunk_shift - 2);
    const int none = (int)R.n;
    // Loads run one piece of work ahead of the gathers (metadata two): a piece
    // is a few hundred gathers, less than what a column load from DRAM takes.
    if (gw < n_chunk) {
        PrsPair v = prs_load(a.cols + gw * per_chunk, lane, 32, per_chunk, none);
        for (int64_t c = gw; c < n_chunk; c += nw) {
            const int64_t nc0 = c + nw;
            PrsPair w = v;
            if (nc0 < n_chunk) w = prs_load(a.cols + nc0 * per_chunk, lane, 32, per_chunk, none);
            const int32_t r = __ldg(R.chunk_row + c);
            const float s = warp_sum(prs_rest(a.cols + c * per_chunk, per_chunk, v, none, hot_c, hot, a.c_in));
            const uint32_t deg = __ldg(R.deg + r);
            const uint32_t c0 = __ldg(R.unit + r) >> (R.chunk_shift - 2);
            const uint32_t nc = (deg + per_chunk * 4 - 1) >> R.chunk_shift;
            unsigned int before = 0;
            if (lane == 0) {
                a.part[c] = s;
                asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(before) : "l"(a.done + r) : "memory");
            }
            __syncwarp();                             // the other lanes read part after it (a shuffle orders no memory)
            if (__shfl_sync(GRX_FULL_MASK, before, 0) + 1 == nc) {
                float t = 0.f;                        // the row's last chunk: add them up in order
                for (uint32_t k = lane; k < nc; k += 32 * 8) {
                    float x[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) x[j] = k + j * 32 < nc ? __ldcg(a.part + c0 + k + j * 32) : 0.f;
#pragma unroll
                    for (int j = 0; j < 8; ++j) t += x[j];
                }
                t = warp_sum(t);
                if (lane == 0) {
                    a.done[r] = 0u;
                    prs_finish(a, r, deg, t);
                }
            }
            v = w;
        }
    }
    // each class goes on dealing where the one before stopped
    const int64_t gw_row = gw - n_chunk % nw + (gw < n_chunk % nw ? nw : 0);
    const int64_t used = (n_chunk + (int64_t)n_warp - n_long) % nw;
    const int64_t gw_slice = gw - used + (gw < used ? nw : 0);
    if (n_long + gw_row < n_warp) {
        const int64_t r0 = n_long + gw_row;
        uint32_t deg = __ldg(R.deg + r0), unit = __ldg(R.unit + r0);
        const int64_t r1 = r0 + nw < n_warp ? r0 + nw : r0;
        uint32_t deg1 = __ldg(R.deg + r1), unit1 = __ldg(R.unit + r1);
        PrsPair v = prs_load(a.cols + unit, lane, 32, (deg + 3) / 4, none);
        for (int64_t r = r0; r < n_warp; r += nw) {
            const PrsPair w = prs_load(a.cols + unit1, lane, 32, (deg1 + 3) / 4, none);
            const int64_t r2 = r + 2 * nw < n_warp ? r + 2 * nw : r;
            const uint32_t deg2 = __ldg(R.deg + r2), unit2 = __ldg(R.unit + r2);
            const float s = warp_sum(prs_rest(a.cols + unit, (deg + 3) / 4, v, none, hot_c, hot, a.c_in));
            if (lane == 0) prs_finish(a, r, deg, s);
            deg = deg1, unit = unit1, v = w;
            deg1 = deg2, unit1 = unit2;
        }
    }
    const int64_t n_slice = R.hdr->n_slice;
    if (gw_slice < n_slice) {
        auto degree = [&](int64_t s) {
            const int64_t r = n_warp + s * 32 + lane;
            return s < n_slice && r < R.n ? __ldg(R.deg + r) : 0u;
        };
        uint32_t deg = degree(gw_slice), d0 = __shfl_sync(GRX_FULL_MASK, deg, 0);
        const int4 *p = a.cols + prs_slice_at(R.hdr, (uint32_t)gw_slice, d0) + lane;
        PrsPair v = prs_load(p, 0, 32, (d0 + 3) / 4 * 32, none);
        uint32_t deg1 = degree(gw_slice + nw);
        for (int64_t s = gw_slice; s < n_slice; s += nw) {
            const uint32_t d1 = __shfl_sync(GRX_FULL_MASK, deg1, 0);
            const int4 *p1 = p;
            PrsPair w = v;
            if (d1) {
                p1 = a.cols + prs_slice_at(R.hdr, (uint32_t)(s + nw), d1) + lane;
                w = prs_load(p1, 0, 32, (d1 + 3) / 4 * 32, none);
            }
            const uint32_t deg2 = degree(s + 2 * nw);
            const uint32_t units = (d0 + 3) / 4;
            float sum = 0.f;
            for (uint32_t q = 2;; q += 2) {
                PrsPair x = v;
                if (q < units) x = prs_load(p, 32 * q, 32, units * 32, none);
                sum += prs_sum8(v, hot_c, hot, a.c_in);
                if (q >= units) break;
                v = x;
            }
            if (deg) prs_finish(a, n_warp + s * 32 + lane, deg, sum);
            p = p1, v = w, d0 = d1, deg = deg1, deg1 = deg2;
        }
    }
}

PrsRows prs_rows(const grx_graph *g) {
    return {(const PrsHeader *)g->prs_hdr, g->prs_deg, g->prs_unit, g->prs_chunk_row, g->n_active, g->prs_chunk_shift};
}

}  // namespace

// Builds the sorted rows (once per graph).  *ready = 0 without an error when
// the allocator has no room for them, and while s is being captured (a capture
// records what it always did): the caller then keeps to the CSR.
grx_status grx_prs_build(grx_graph *g, cudaStream_t s, int *ready) {
    *ready = g->prs_cols != nullptr;
    if (*ready || g->n_active == 0) return GRX_OK;
    if (grx_capturing(s)) return GRX_OK;
    const int64_t n = g->n_active, ne = g->ne;
    // Chunks of 1,024 edges on large graphs, smaller ones on small graphs, where a
    // warp's whole share is a few hundred edges (per iteration with chunks of 128 / 256 /
    // 512 edges: R-MAT 16 13.5 / 11.5 / - us, 18 - / 19.8 / 18.0, 20 - / 64.6 / 57.1); but
    // about a thousand of the longest row at most, which are counted by one word and
    // added up by one warp (a star of 1M leaves: 7,813 chunks of 128 37 us, 977 of 1,024
    // 18).  Rows past eight chunks are cut, so padding them to whole chunks costs an
    // eighth at most.
    int chunk_shift = ne >= (64ll << 20) ? 10 : (ne >= (4ll << 20) ? 9 : (ne >= (1ll << 20) ? 8 : 7));
    while (chunk_shift < 12 && g->max_deg >> chunk_shift > 1024) ++chunk_shift;
    const uint32_t longest = 8u << chunk_shift;
    const int long_key = prs_key_log(chunk_shift + 3, 0);
    const int64_t max_long = ne / longest + 1;
    const int64_t max_chunk = (ne >> chunk_shift) + max_long;
    const int64_t units = ne / 4 + 3 * n / 4 + (max_long << (chunk_shift - 2)) + 32 * 32 + 64;
    if (units >= (1ll << 32)) return GRX_OK;
    int nb = g->ctx->num_sms * 2;
    if (nb > (n + PRS_SORT_BLOCK - 1) / PRS_SORT_BLOCK) nb = (int)((n + PRS_SORT_BLOCK - 1) / PRS_SORT_BLOCK);
    const int64_t per = (n + nb - 1) / nb;
    const size_t mat_bytes = (size_t)nb * PRS_KEYS * 8, label_bytes = (size_t)g->nv * 4, src_bytes = (size_t)n * 4;
    // one block for what stays (so that a refusal leaves nothing behind), one for the build
    struct Piece { size_t at, bytes; };
    size_t keep = 0;
    auto piece = [&](size_t bytes) { const Piece p{keep, bytes}; keep += (bytes + 255) & ~(size_t)255; return p; };
    const Piece pc = piece((size_t)units * 16), ph = piece(sizeof(PrsHeader)), pv = piece((size_t)n * 4),
                pd = piece((size_t)n * 4), pu = piece((size_t)(ne / PRS_SELL + 1) * 4), pr = piece((size_t)max_chunk * 4),
                pp = piece((size_t)max_chunk * 4), pn = piece((size_t)max_long * 4);
    const size_t tmp_bytes = mat_bytes + label_bytes + src_bytes;
    char *tmp = (char *)grx_ctx_alloc(g->ctx, tmp_bytes, s);
    if (!tmp) return GRX_OK;
    char *p = (char *)grx_alloc_optional(g, keep, s);
    if (!p) {
        grx_ctx_free(g->ctx, tmp, tmp_bytes, s);
        return GRX_OK;
    }
    unsigned long long *mat = (unsigned long long *)tmp;
    int32_t *label = (int32_t *)(tmp + mat_bytes);
    uint32_t *src = (uint32_t *)(tmp + mat_bytes + label_bytes);
    g->prs_hdr = p + ph.at;
    g->prs_vert = (int32_t *)(p + pv.at);
    g->prs_deg = (uint32_t *)(p + pd.at);
    g->prs_unit = (uint32_t *)(p + pu.at);
    g->prs_chunk_row = (int32_t *)(p + pr.at);
    g->prs_part = (float *)(p + pp.at);
    g->prs_done = (unsigned int *)(p + pn.at);
    g->prs_chunk_shift = chunk_shift;
    k_prs_count<<<nb, PRS_SORT_BLOCK, 0, s>>>(g->aoff, n, per, chunk_shift, longest, mat);
    k_prs_scan<<<1, PRS_KEYS, 0, s>>>(mat, nb, n, chunk_shift, long_key, (PrsHeader *)g->prs_hdr);
    k_prs_place<<<nb, PRS_SORT_BLOCK, 0, s>>>(g->active, g->aoff, n, per, chunk_shift, longest, mat, g->prs_vert,
                                             g->prs_deg, src, g->prs_unit, g->prs_chunk_row, label);
    k_prs_fill<<<g->ctx->num_sms * 8, 256, 0, s>>>(prs_rows(g), g->col, label, src, (int4 *)(p + pc.at));
    cudaError_t e = cudaMemsetAsync(g->prs_done, 0, pn.bytes, s);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute((const void *)k_prs_iter, cudaFuncAttributeMaxDynamicSharedMemorySize, PRS_HOT * 4);
    grx_ctx_free(g->ctx, tmp, tmp_bytes, s);
    if (e != cudaSuccess) return grx_cuda_fail(e, "pagerank: sorting the rows");
    g->prs_cols = p + pc.at;
    *ready = 1;
    return GRX_OK;
}

// c0 = r0 / degree by label; c0 and c1 hold n_active + 1 entries.
void grx_prs_init(grx_graph *g, float r0, float *c0, float *c1, cudaStream_t s) {
    const int64_t b = (g->n_active + 255) / 256;
    k_prs_init<<<(unsigned)(b < 8192 ? b : 8192), 256, 0, s>>>(g->prs_deg, g->n_active, r0, c0, c1);
}

void grx_prs_iterate(grx_graph *g, const float *c_in, float *c_out, float *rank, float base, float d, cudaStream_t s) {
    PrsIter a;
    a.rows = prs_rows(g);
    a.cols = (const int4 *)g->prs_cols;
    a.vert = g->prs_vert;
    a.c_in = c_in;
    a.c_out = c_out;
    a.rank = rank;
    a.part = g->prs_part;
    a.done = g->prs_done;
    const int most = g->n_active >= PRS_BIG ? PRS_HOT_BIG : PRS_HOT;
    a.hot = (int)(g->n_active < most ? g->n_active : most);
    a.base = base;
    a.d = d;
    k_prs_iter<<<g->ctx->num_sms, PRS_BLOCK, (size_t)a.hot * 4, s>>>(a);
}
