// Multi-source BFS (paper Alg. 3), one level per call:
//   N = A * F over (or, select2nd);  F_next = N minus S;  S = S or N;
// fused into one gather pass per row (the boolean TS-SpGEMM with a d-bit
// accumulator), a scan for F_next's row pointers and a read-out of the new
// bits.  For d <= 256 the frontier is expanded to a bitmap and rows pull from
// it (the pull form below); above that the list form walks F's rows, heaviest
// rows first, and skips rows whose visited set is full and rows whose
// neighbours have empty frontier rows.
#include "bitrows.cuh"
#include "common.cuh"
#include "kernels.h"

namespace ts {

// Rows whose visited bits are all set get flops 0 (nothing can be new).
__global__ void k_mask_full_rows(long long n, int d, int dw, const unsigned* __restrict__ S,
                                 long long* flops) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || flops[i] == 0) return;
    const unsigned* r = S + i * dw;
    for (int w = 0; w < dw; ++w) {
        const int bits = d - 32 * w;
        const unsigned want = bits >= 32 ? FULL : ((1u << bits) - 1u);
        if ((r[w] & want) != want) return;
    }
    flops[i] = 0;
}

struct OrVisit {
    const int* __restrict__ Fi;
    unsigned* bm;
    int d;
    unsigned long long* err;
    __device__ __forceinline__ void mark(int c) {
        if ((unsigned)c < (unsigned)d) atomicOr(bm + (c >> 5), 1u << (c & 31));
        else atomicOr(err, ERR_B_COL);
    }
    __device__ __forceinline__ void step4(const long long* j, const float*, const int*) {
        int c[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) c[u] = __ldg(Fi + j[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) mark(c[u]);
    }
    __device__ __forceinline__ void step1(long long j, float, int, bool ok) {
        if (ok) mark(__ldg(Fi + j));
    }
};

struct BfsParams {
    const long long* Ap;
    const int* Ai;
    long long nnzA;
    SegWhole segF;
    const int* Fi;
    int nF;
    int d;
    int dw;
    unsigned* S;
    int* levels;
    int level;
    unsigned* newbits;
    long long* cnt_next;  // F_next.rowptr + 1
    int* parents;         // int32[n][d] BFS-tree parents (pull form only), or nullptr
    const int* perm;
    WsHeader* hdr;
    int cta_class;
    long long n;
    // pull form
    int ss, ns;                  // words per row of S and of newbits
    unsigned long long* queue;   // chunks of heavy rows queued at this level
    unsigned long long* err;     // ERR_* bits
    long long fnnz;              // entries of the frontier (a step; a search counts them on the device)
    // a whole search (msbfs_search): newbits is the next frontier's bitmap
    const long long* prev;       // BFS_COUNTS counters of the frontier's entries, or nullptr (a step)
    long long* count;            // ... of the next frontier's
    unsigned* ne_next;           // its non-empty bits
    unsigned* ne_clear;          // the words the level after this one adds its bits to
};

// A search counts a level's new bits in several words on lines of their own
// (one per warp number modulo BFS_COUNTS): tens of thousands of warps would
// queue at one.
constexpr int BFS_COUNTS = 8, BFS_COUNT_STRIDE = 16;

// Entries of the frontier this level expands.
__device__ __forceinline__ long long bfs_entries(const BfsParams& p) {
    if (!p.prev) return p.fnnz;
    long long f = 0;
#pragma unroll
    for (int q = 0; q < BFS_COUNTS; ++q) f += __ldcg(p.prev + q * BFS_COUNT_STRIDE);
    return f;
}

// Given the OR of the neighbours' frontier rows in bm (dw words), keep the
// bits not yet visited, mark them visited, record their level, store them for
// the read-out and return how many there are.  Threads t0, t0+nt, ... own words.
__device__ __forceinline__ int settle_row(const BfsParams& p, long long row, unsigned* bm, int t0, int nt) {
    int c = 0;
    for (int w = t0; w < p.dw; w += nt) {
        const int bits = p.d - 32 * w;
        const unsigned valid = bits >= 32 ? FULL : ((1u << bits) - 1u);
        const unsigned old = p.S[row * p.dw + w];
        unsigned nw = bm[w] & ~old & valid;
        bm[w] = 0u;
        p.newbits[row * p.dw + w] = nw;
        if (nw) {
            p.S[row * p.dw + w] = old | nw;
            c += __popc(nw);
            while (nw) {
                const int b = __ffs(nw) - 1;
                nw &= nw - 1;
                p.levels[row * p.d + 32 * w + b] = p.level;
            }
        }
    }
    return c;
}

__global__ void __launch_bounds__(1024) k_msbfs_expand(BfsParams p) {
    extern __shared__ __align__(16) unsigned smem_u[];
    __shared__ long long s_item, s_nheavy, s_nrows;
    __shared__ int s_red[32];
    const int nw = blockDim.x >> 5, warp = warp_id(), lane = lane_id(), tid = threadIdx.x;
    for (int i = tid; i < nw * p.dw; i += blockDim.x) smem_u[i] = 0u;
    if (tid < 32) {  // one warp; its lanes store the same values
        long long nh, nr;
        sched_counts(p.hdr, p.cta_class, nh, nr);
        s_nheavy = nh;
        s_nrows = nr;
    }
    __syncthreads();
    const long long nheavy = s_nheavy, nrows = s_nrows;
    unsigned long long* err = &p.hdr->err;
    for (;;) {
        if (tid == 0) s_item = (long long)atomicAdd(&p.hdr->heavy_ctr, 1ull);
        __syncthreads();
        const long long h = s_item;
        __syncthreads();
        if (h >= nheavy) break;
        const int row = p.perm[h];
        const long long a0 = clampll(__ldg(p.Ap + row), 0, p.nnzA);
        const long long a1 = clampll(__ldg(p.Ap + row + 1), a0, p.nnzA);
        OrVisit vis{p.Fi, smem_u, p.d, err};
        for (long long e0 = a0 + 32LL * warp; e0 < a1; e0 += 32LL * nw)
            expand_chunk(e0, (int)(a1 - e0 < 32 ? a1 - e0 : 32), p.Ai, (const float*)nullptr, p.nF,
                         p.segF, vis, err);
        __syncthreads();
        int c = settle_row(p, row, smem_u, tid, blockDim.x);
        c = warp_sum(c);
        if (lane == 0) s_red[warp] = c;
        __syncthreads();
        if (warp == 0) {
            int v = lane < nw ? s_red[lane] : 0;
            v = warp_sum(v);
            if (lane == 0) p.cnt_next[row] = v;
        }
    }
    unsigned* bm = smem_u + warp * p.dw;
    for (long long idx = nheavy + (long long)blockIdx.x * nw + warp; idx < nrows;
         idx += (long long)gridDim.x * nw) {
        const int row = p.perm[idx];
        const long long a0 = clampll(__ldg(p.Ap + row), 0, p.nnzA);
        const long long a1 = clampll(__ldg(p.Ap + row + 1), a0, p.nnzA);
        OrVisit vis{p.Fi, bm, p.d, err};
        for (long long e0 = a0; e0 < a1; e0 += 32)
            expand_chunk(e0, (int)(a1 - e0 < 32 ? a1 - e0 : 32), p.Ai, (const float*)nullptr, p.nF,
                         p.segF, vis, err);
        __syncwarp();
        int c = settle_row(p, row, bm, lane, 32);
        c = warp_sum(c);
        if (lane == 0) p.cnt_next[row] = c;
        __syncwarp();
    }
}

// Initial frontier and visited/level state from d sources (distinct vertices;
// a repeated vertex simply holds several columns).  Row pointers: a block
// takes 1024 vertices, counts the sources below them once and keeps those
// among them in shared memory, where every vertex counts the ones at or
// below it (a thread per vertex over all d sources took 39 us for 2^20
// vertices and 128 sources).  Columns: a thread per source.
constexpr int INIT_ROWS = 1024;
__global__ void __launch_bounds__(256) k_msbfs_init_rows(long long n, int d, const int* __restrict__ src,
                                                         long long* rp) {
    __shared__ int s_here[INIT_ROWS];  // sources at each of the block's vertices, then their running sum
    __shared__ int s_below, s_w[8];
    const int tid = threadIdx.x, lane = lane_id(), warp = warp_id();
    const long long base = (long long)blockIdx.x * INIT_ROWS;
    for (int i = tid; i < INIT_ROWS; i += 256) s_here[i] = 0;
    if (tid == 0) s_below = 0;
    __syncthreads();
    int below = 0;
    for (int s = tid; s < d; s += 256) {
        const int u = __ldg(src + s);
        if (u < 0) continue;
        if ((long long)u < base) ++below;
        else if ((long long)u < base + INIT_ROWS) atomicAdd(&s_here[u - (int)base], 1);
    }
    below = warp_sum(below);
    if (lane == 0 && below) atomicAdd(&s_below, below);
    __syncthreads();
    // vertices 4 tid .. 4 tid + 3 of the block
    int c[4], run = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        c[q] = run;
        run += s_here[4 * tid + q];
    }
    const int incl = warp_incl_scan(run);
    if (lane == 31) s_w[warp] = incl;
    __syncthreads();
    int before = s_below + incl - run;
    for (int w = 0; w < warp; ++w) before += s_w[w];
#pragma unroll
    for (int q = 0; q < 4; ++q) {  // rp[v] = sources at vertices < v
        const long long v = base + 4 * tid + q;
        if (v <= n) rp[v] = before + c[q];
    }
}

__global__ void k_msbfs_init_cols(long long n, int d, int dw, const int* __restrict__ src, int* col,
                                  unsigned* S, int* levels) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= d) return;
    const int v = src[s];
    if (v < 0 || (long long)v >= n) return;
    int pos = 0;
    for (int t = 0; t < d; ++t) {
        const int u = src[t];
        if (u < 0 || (long long)u >= n) continue;
        if (u < v || (u == v && t < s)) ++pos;
    }
    col[pos] = s;
    atomicOr(S + (long long)v * dw + (s >> 5), 1u << (s & 31));
    levels[(long long)v * d + s] = 0;
}


// ---------------------------------------------------------------------------
// Pull form (d <= 256): the frontier as a bitmap of DWP words per vertex (dw
// rounded up to a power of two), and row v of N = A * F the OR of its
// neighbours' bitmap rows, one load of DWP words per entry of A whatever the
// frontier's density.  A level is bound by those gathers (the bitmap stays in
// L2: 16 MB for 2^20 vertices and 128 sources) and by the latency of long
// rows, so:
//  - rows are taken in their own order, 32 (fewer when there are few rows) to
//    a warp, with no flops pass, classes or permutation before (these cost
//    180 us a level at scale 20): a row of at most BFS_SHORT entries by its
//    lane, a longer one by the whole warp, 64 or 128 entries at a time, and one
//    above BFS_HEAVY by blocks of BFS_CHUNK entries in a kernel of its own
//    (a hub's row in one warp took 0.8 - 1.1 ms of each of the first levels);
//  - a row stops gathering once its unvisited sources are all found, which in
//    the dense levels is after the first few neighbours, and a row whose
//    sources are all found is not read (A's columns are range-checked as a
//    stream beside the frontier's expansion, whatever the rows need of them);
//  - while F holds fewer entries than n / BFS_SPARSE, a bit per vertex says
//    whether its frontier row is empty, and empty ones are not gathered (the
//    bits of 2^20 vertices are 128 KB and stay in L1).
// Step by step the 128-source search of the scale-20 graph went 5.9 -> 2.1 ms, the BFS
// trees of 50 sources over 300,007 vertices 2.94 -> 1.09 ms.
// ---------------------------------------------------------------------------
constexpr int BFS_SHORT = 16;
constexpr int BFS_HEAVY = 2048;
constexpr int BFS_CHUNK = 4096;
constexpr int BFS_SPARSE = 4;
constexpr int PULL_THREADS = 64;  // small blocks: one waits for its slowest warp (256 threads: 2.19 against 2.11 ms)

// Range check of A's columns: block b of 256 threads takes entries
// [b, b + 1) * CHECK_PER_BLOCK.
constexpr int CHECK_PER_BLOCK = 16384;
__device__ __forceinline__ void check_columns(unsigned block, long long n, const long long* __restrict__ Ap,
                                              const int* __restrict__ Ai, long long nnzA, unsigned long long* err) {
    const long long lo = clampll(__ldg(Ap), 0, nnzA), hi = clampll(__ldg(Ap + n), lo, nnzA);
    const long long b0 = (long long)block * CHECK_PER_BLOCK;
    const long long first = b0 > lo ? b0 : lo;
    const long long last = b0 + CHECK_PER_BLOCK < hi ? b0 + CHECK_PER_BLOCK : hi;
    bool bad = false;
    if (last - first == CHECK_PER_BLOCK && !(reinterpret_cast<uintptr_t>(Ai) & 15)) {
        const int4* q = reinterpret_cast<const int4*>(Ai + first);  // first is a multiple of four
#pragma unroll 4
        for (int i = threadIdx.x; i < CHECK_PER_BLOCK / 4; i += 256) {
            const int4 c = __ldg(q + i);
            const unsigned x = max(max((unsigned)c.x, (unsigned)c.y), max((unsigned)c.z, (unsigned)c.w));
            bad |= x >= (unsigned)n;
        }
    } else {
        for (long long e = first + threadIdx.x; e < last; e += 256) bad |= (unsigned)__ldg(Ai + e) >= (unsigned)n;
    }
    if (bad) atomicOr(err, ERR_A_COL);
}

// Bitmap rows of F and the bits of the non-empty ones; also clears what the
// level accumulates (scan partials) and C's first row pointer.  A warp takes
// 32 vertices (rows_to_bits).
//
// The blocks behind the first nfront range-check A's columns, so that the
// pull may leave out rows and ends of rows with nothing left to find: a
// stream over A beside the decoding (30 us in all where the frontier is small).
template <int DWP>
__global__ void __launch_bounds__(256) k_bfs_frontier(long long n, int d, const long long* __restrict__ Fp,
                                                      long long nnzF, const int* __restrict__ Fi,
                                                      unsigned* __restrict__ fb, unsigned* __restrict__ nonempty,
                                                      long long* partial, long long npartial, long long* rp_next,
                                                      unsigned nfront, const long long* __restrict__ Ap,
                                                      const int* __restrict__ Ai, long long nnzA,
                                                      unsigned long long* err) {
    const int lane = lane_id(), warp = warp_id();
    if (blockIdx.x >= nfront) {
        check_columns(blockIdx.x - nfront, n, Ap, Ai, nnzA, err);
        return;
    }
    __shared__ unsigned s_bits[8][32 * DWP];
    __shared__ int s_start[8][33];
    const long long base = ((long long)blockIdx.x * 8 + warp) * 32, v = base + lane;
    for (long long x = (long long)blockIdx.x * 256 + threadIdx.x; x < npartial; x += 256LL * nfront) partial[x] = 0;
    if (v == 0) rp_next[0] = 0;
    unsigned* bits = s_bits[warp];
    if (base >= n) return;
    const bool bad = rows_to_bits<DWP>(n, d, Fp, nnzF, Fi, base, bits, s_start[warp]);
    unsigned any = 0u;
#pragma unroll
    for (int m = 0; m < DWP; ++m) any |= bits[lane * DWP + m];
    const unsigned ne = __ballot_sync(FULL, any != 0u);
    if (lane == 0) nonempty[base >> 5] = ne;
    // the 32 rows' words, contiguous in fb
#pragma unroll
    for (int m = 0; m < DWP; ++m)
        if (32 * m + lane < (n - base) * DWP) fb[base * DWP + 32 * m + lane] = bits[32 * m + lane];
    if (bad) atomicOr(err, ERR_B_COL);
}

// A row of `words` <= DWP words read or written; VEC: of DWP words, aligned to
// its width (a search's own arrays; a step's visited words are the caller's).
template <int DWP, bool VEC>
__device__ __forceinline__ void bfs_load_words(const unsigned* r, int words, unsigned w[DWP]) {
    if (VEC && DWP >= 4) {
#pragma unroll
        for (int m = 0; m + 4 <= DWP; m += 4) {
            const uint4 x = *reinterpret_cast<const uint4*>(r + m);
            w[m] = x.x;
            w[m + 1] = x.y;
            w[m + 2] = x.z;
            w[m + 3] = x.w;
        }
        return;
    }
#pragma unroll
    for (int m = 0; m < DWP; ++m) w[m] = m < words ? r[m] : 0u;
}

template <int DWP, bool VEC>
__device__ __forceinline__ void bfs_store_words(unsigned* r, int words, const unsigned w[DWP]) {
    if (VEC && DWP >= 4) {
#pragma unroll
        for (int m = 0; m + 4 <= DWP; m += 4)
            *reinterpret_cast<uint4*>(r + m) = make_uint4(w[m], w[m + 1], w[m + 2], w[m + 3]);
        return;
    }
#pragma unroll
    for (int m = 0; m < DWP; ++m)
        if (m < words) r[m] = w[m];
}

// A's columns as the pull reads them: load() gives the neighbour of entry e
// (-1 for none, or for a column outside [0, n), which the check of A's columns
// reports), hit() whether its frontier row is to be gathered.
struct BfsCols {
    const int* __restrict__ Ai;
    const unsigned* __restrict__ nonempty;
    int nF;
    bool sparse;  // many frontier rows are empty: ask nonempty first
    __device__ __forceinline__ int load(long long e, bool in) const {
        const int u = in ? __ldg(Ai + e) : -1;
        return (unsigned)u < (unsigned)nF ? u : -1;
    }
    __device__ __forceinline__ bool hit(int u) const {
        return u >= 0 && (!sparse || ((__ldg(nonempty + (u >> 5)) >> (u & 31)) & 1u));
    }
};

// Transpose of a 32 x 32 bit matrix over the warp: bit b of lane l becomes
// bit l of lane b.
__device__ __forceinline__ unsigned warp_transpose(unsigned x) {
    const int lane = lane_id();
    unsigned m = 0x0000FFFFu;
#pragma unroll
    for (int j = 16; j >= 1; j >>= 1) {
        const unsigned t = __shfl_xor_sync(FULL, x, j);
        x = (lane & j) ? ((t >> j) & m) | (x & ~m) : ((t << j) & ~m) | (x & m);
        m ^= m << (j >> 1);
    }
    return x;
}

// One word of the step of 32 neighbours (lane l: neighbour u, its bits `hit`
// among the row's open ones): every bit's parent is the first lane that holds
// it (A's rows ascend, so the smallest neighbour).  Returns the bits found.
__device__ __forceinline__ unsigned bfs_first(unsigned hit, int u, int& parent, bool& found) {
    const unsigned who = warp_transpose(hit);
    found = who != 0u;
    parent = __shfl_sync(FULL, u, found ? __ffs(who) - 1 : 0);
    return __ballot_sync(FULL, found);
}

// Level writes of one row's new bits (warp-uniform words), lane l bit l.
template <int DWP>
__device__ __forceinline__ void bfs_write_levels(const BfsParams& p, long long row, const unsigned nw[DWP]) {
    int* lv = p.levels + row * p.d + lane_id();
#pragma unroll
    for (int m = 0; m < DWP; ++m)
        if ((nw[m] >> lane_id()) & 1u) lv[32 * m] = p.level;
}

template <int DWP, bool PARENTS, bool SEARCH>
__global__ void __launch_bounds__(PULL_THREADS, 1024 / PULL_THREADS)
    k_bfs_pull(BfsParams p, const unsigned* __restrict__ fb, const unsigned* __restrict__ nonempty,
               int rows_per_warp, long long* items, long long item_cap, int* done, long long* partial,
               int scan_tile) {
    constexpr int U = DWP == 8 ? 2 : 4;  // neighbours in flight per lane
    const int lane = lane_id();
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long base = gw * rows_per_warp;
    if (base >= p.n) return;
    const long long entries = bfs_entries(p);
    if (SEARCH && entries == 0) return;  // the search has ended
    const BfsCols cols{p.Ai, nonempty, p.nF, entries < p.n / BFS_SPARSE};
    const long long v = base + lane;
    const bool mine = lane < rows_per_warp && v < p.n;
    const int ss = SEARCH ? DWP : p.ss, ns = SEARCH ? DWP : p.ns;
    long long a0 = 0, a1 = 0;
    unsigned old[DWP], want[DWP], acc[DWP];
    unsigned open = 0u;
#pragma unroll
    for (int m = 0; m < DWP; ++m) acc[m] = old[m] = want[m] = 0u;
    if (mine) {
        bfs_load_words<DWP, SEARCH>(p.S + v * ss, ss, old);
#pragma unroll
        for (int m = 0; m < DWP; ++m) {
            const int bits = p.d - 32 * m;
            want[m] = ~old[m] & (bits >= 32 ? FULL : bits > 0 ? (1u << bits) - 1u : 0u);
            open |= want[m];
        }
    }
    if (mine) {
        a0 = clampll(__ldg(p.Ap + v), 0, p.nnzA);
        a1 = clampll(__ldg(p.Ap + v + 1), a0, p.nnzA);
    }
    const long long len = open ? a1 - a0 : 0;  // nothing to find: the row is left out
    const bool heavy = len > BFS_HEAVY;
    // rows of many entries: queued for k_bfs_heavy in chunks
    if (__any_sync(FULL, heavy)) {
        const long long nc = heavy ? (len + BFS_CHUNK - 1) / BFS_CHUNK : 0;
        const long long incl = warp_incl_scan(nc);
        long long first = 0;
        if (lane == 31) first = (long long)atomicAdd(p.queue, (unsigned long long)incl);
        first = shfl64(first, 31) + incl - nc;
        if (heavy) {
            done[v] = 0;
            for (int m = 0; m < ns; ++m) p.newbits[v * ns + m] = 0u;
            for (long long c = 0; c < nc; ++c) {
                if (first + c < item_cap) items[first + c] = (v << 24) | c;
                else atomicOr(p.err, ERR_CAPACITY);
            }
        }
    }
    // short rows: a lane each, U neighbours in flight and the next U columns
    // of A loaded ahead
    const int slen = len <= BFS_SHORT ? (int)len : 0;
    const int smax = (int)__reduce_max_sync(FULL, (unsigned)slen);
    if (smax > 0) {
        int u[U];
#pragma unroll
        for (int t = 0; t < U; ++t) u[t] = cols.load(a0 + t, t < slen);
        for (int j = 0; j < smax; j += U) {
            int un[U];
            unsigned w[U][DWP];
#pragma unroll
            for (int t = 0; t < U; ++t) un[t] = cols.load(a0 + j + U + t, j + U + t < slen);
#pragma unroll
            for (int t = 0; t < U; ++t) {
#pragma unroll
                for (int m = 0; m < DWP; ++m) w[t][m] = 0u;
                if (cols.hit(u[t])) load_bit_row<DWP>(fb, u[t], w[t]);
            }
#pragma unroll
            for (int t = 0; t < U; ++t) {
#pragma unroll
                for (int m = 0; m < DWP; ++m) {
                    if constexpr (PARENTS) {
                        unsigned h = w[t][m] & want[m] & ~acc[m];
                        while (h) {
                            const int b = __ffs(h) - 1;
                            h &= h - 1;
                            p.parents[v * p.d + 32 * m + b] = u[t];
                        }
                    }
                    acc[m] |= w[t][m];
                }
            }
#pragma unroll
            for (int t = 0; t < U; ++t) u[t] = un[t];
        }
    }
    // longer rows: the warp takes one after another, 32 U neighbours at a
    // time; the columns of the next step (the row's next, or the next row's
    // first) are loaded before this step's frontier rows
    unsigned rows = __ballot_sync(FULL, len > BFS_SHORT && !heavy);
    if (rows) {
        int r = __ffs(rows) - 1, j = 0;
        long long e0 = shfl64(a0, r);
        int nr = (int)shfl64(len, r);
        int u[U];
#pragma unroll
        for (int t = 0; t < U; ++t) u[t] = cols.load(e0 + 32 * t + lane, 32 * t + lane < nr);
        unsigned rem[DWP], got[DWP];  // the row's open bits; the bits this lane's neighbours (parents: the row) have
#pragma unroll
        for (int m = 0; m < DWP; ++m) {
            rem[m] = __shfl_sync(FULL, want[m], r);
            got[m] = 0u;
        }
        for (;;) {
            const bool more = j + 32 * U < nr;  // of this row
            const unsigned rest = rows & (rows - 1);
            const int r2 = rest ? __ffs(rest) - 1 : r;  // the row after it
            const long long e2 = shfl64(a0, r2);
            const int n2 = rest ? (int)shfl64(len, r2) : 0;
            const long long ne = more ? e0 + j + 32 * U : e2;
            const int nn = more ? nr - j - 32 * U : n2;
            int un[U];
            unsigned w[U][DWP];
#pragma unroll
            for (int t = 0; t < U; ++t) un[t] = cols.load(ne + 32 * t + lane, 32 * t + lane < nn);
#pragma unroll
            for (int t = 0; t < U; ++t) {
#pragma unroll
                for (int m = 0; m < DWP; ++m) w[t][m] = 0u;
                if (cols.hit(u[t])) load_bit_row<DWP>(fb, u[t], w[t]);
            }
            unsigned live = 0u;
            if constexpr (PARENTS) {
#pragma unroll
                for (int t = 0; t < U; ++t) {
                    unsigned h = 0u;
#pragma unroll
                    for (int m = 0; m < DWP; ++m) h |= w[t][m] & rem[m];
                    if (!__any_sync(FULL, h != 0u)) continue;
#pragma unroll
                    for (int m = 0; m < DWP; ++m) {
                        int parent;
                        bool found;
                        const unsigned bits = bfs_first(w[t][m] & rem[m], u[t], parent, found);
                        if (found) p.parents[(base + r) * p.d + 32 * m + lane] = parent;
                        got[m] |= bits;
                        rem[m] &= ~bits;
                    }
                }
#pragma unroll
                for (int m = 0; m < DWP; ++m) live |= rem[m];
            } else {
#pragma unroll
                for (int m = 0; m < DWP; ++m) {
#pragma unroll
                    for (int t = 0; t < U; ++t) got[m] |= w[t][m];
                    if (more) live |= rem[m] & ~__reduce_or_sync(FULL, got[m]);
                }
            }
            if (more && live) {  // the row goes on
                j += 32 * U;
#pragma unroll
                for (int t = 0; t < U; ++t) u[t] = un[t];
                continue;
            }
#pragma unroll
            for (int m = 0; m < DWP; ++m) {
                const unsigned x = PARENTS ? got[m] : __reduce_or_sync(FULL, got[m]);
                if (lane == r) acc[m] = x;
                got[m] = 0u;
            }
            if (!rest) break;
            rows = rest;
            r = r2;
            e0 = e2;
            nr = n2;
            j = 0;
#pragma unroll
            for (int t = 0; t < U; ++t)
                u[t] = more ? cols.load(e0 + 32 * t + lane, 32 * t + lane < nr) : un[t];  // found early: not loaded yet
#pragma unroll
            for (int m = 0; m < DWP; ++m) rem[m] = __shfl_sync(FULL, want[m], r);
        }
    }
    // settle: new = N and not S; S |= new; counts, new words, levels
    int c = 0;
    unsigned any = 0u;
#pragma unroll
    for (int m = 0; m < DWP; ++m) {
        acc[m] &= want[m];
        any |= acc[m];
        c += __popc(acc[m]);
    }
    if (mine && !heavy) {
        if (!SEARCH) p.cnt_next[v] = c;
        if (SEARCH || any) {  // the next frontier's bitmap is written whole
            bfs_store_words<DWP, SEARCH>(p.newbits + v * ns, ns, acc);
            if (any) {
#pragma unroll
                for (int m = 0; m < DWP; ++m) old[m] |= acc[m];
                bfs_store_words<DWP, SEARCH>(p.S + v * ss, ss, old);
            }
        }
    }
    if constexpr (SEARCH) {  // a word holds the bits of one warp's rows, or of several warps'
        const unsigned bits = __ballot_sync(FULL, any != 0u);
        if (lane == 0) {
            if (bits) atomicOr(p.ne_next + (base >> 5), bits << (base & 31));
            if ((base & 31) == 0) p.ne_clear[base >> 5] = 0u;
        }
    }
    for (unsigned rows = __ballot_sync(FULL, any != 0u); rows; rows &= rows - 1) {
        const int r = __ffs(rows) - 1;
        unsigned nw[DWP];
#pragma unroll
        for (int m = 0; m < DWP; ++m) nw[m] = __shfl_sync(FULL, acc[m], r);
        bfs_write_levels<DWP>(p, base + r, nw);
    }
    // (a step: the warp's rows lie in one tile of the scan, rows_per_warp divides it)
    c = warp_sum(c);
    long long* sum = SEARCH ? p.count + (gw & (BFS_COUNTS - 1)) * BFS_COUNT_STRIDE : partial + base / scan_tile;
    if (lane == 0 && c) atomicAdd((unsigned long long*)sum, (unsigned long long)c);
}

// Rows above BFS_HEAVY: a block per chunk ORs its neighbours into the row's
// new words (cleared when the row was queued); the block of the row's last
// chunk settles the row.  A chunk that starts when the row has nothing left
// to find is left out.
template <int DWP, bool SEARCH>
__global__ void __launch_bounds__(256) k_bfs_heavy(BfsParams p, const unsigned* __restrict__ fb,
                                                   const unsigned* __restrict__ nonempty,
                                                   const long long* __restrict__ items, long long item_cap,
                                                   int* done, long long* partial, int scan_tile) {
    __shared__ unsigned s_or[DWP];
    __shared__ int s_last;
    const int lane = lane_id(), tid = threadIdx.x;
    const long long nitems = min((long long)__ldcg(p.queue), item_cap);
    if (nitems == 0) return;
    const BfsCols cols{p.Ai, nonempty, p.nF, bfs_entries(p) < p.n / BFS_SPARSE};
    for (long long it = blockIdx.x; it < nitems; it += gridDim.x) {
        const long long row = items[it] >> 24, c = items[it] & 0xFFFFFF;
        const long long a0 = clampll(__ldg(p.Ap + row), 0, p.nnzA);
        const long long a1 = clampll(__ldg(p.Ap + row + 1), a0, p.nnzA);
        const long long e0 = a0 + c * BFS_CHUNK;
        const int n = (int)(a1 - e0 < BFS_CHUNK ? a1 - e0 : BFS_CHUNK);
        if (tid < DWP) s_or[tid] = 0u;
        unsigned want[DWP], got[DWP];
        unsigned live = 0u;
#pragma unroll
        for (int m = 0; m < DWP; ++m) {
            want[m] = got[m] = 0u;
            if (m < p.dw) {
                const int bits = p.d - 32 * m;
                want[m] = ~__ldcg(p.S + row * p.ss + m) & (bits >= 32 ? FULL : ((1u << bits) - 1u));
                live |= want[m] & ~__ldcg(p.newbits + row * p.ns + m);
            }
        }
        __syncthreads();
        for (int j = tid; live && j < n; j += 4 * 256) {
            int u[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) u[t] = cols.load(e0 + j + 256 * t, j + 256 * t < n);
            unsigned w[DWP];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                if (cols.hit(u[t])) {
                    load_bit_row<DWP>(fb, u[t], w);
#pragma unroll
                    for (int m = 0; m < DWP; ++m) got[m] |= w[m];
                }
            }
        }
#pragma unroll
        for (int m = 0; m < DWP; ++m) {
            const unsigned x = __reduce_or_sync(FULL, got[m] & want[m]);
            if (lane == 0 && x) atomicOr(&s_or[m], x);
        }
        __syncthreads();
        if (tid < p.dw && s_or[tid]) atomicOr(p.newbits + row * p.ns + tid, s_or[tid]);
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            const long long nc = (a1 - a0 + BFS_CHUNK - 1) / BFS_CHUNK;
            s_last = atomicAdd(done + row, 1) == nc - 1;
        }
        __syncthreads();
        if (s_last && tid < 32) {
            __threadfence();
            unsigned nw[DWP];
            int cnt = 0;
#pragma unroll
            for (int m = 0; m < DWP; ++m) {
                nw[m] = m < p.dw ? __ldcg(p.newbits + row * p.ns + m) : 0u;
                cnt += __popc(nw[m]);
                if (lane == 0 && nw[m]) p.S[row * p.ss + m] |= nw[m];
                // k_bfs_heavy_parents takes the minimum from here
                if (p.parents && ((nw[m] >> lane) & 1u)) p.parents[row * p.d + 32 * m + lane] = 0x7FFFFFFF;
            }
            bfs_write_levels<DWP>(p, row, nw);
            if (lane == 0) {
                if (SEARCH && cnt) atomicOr(p.ne_next + (row >> 5), 1u << (row & 31));
                if (!SEARCH) p.cnt_next[row] = cnt;
                long long* sum = SEARCH ? p.count : partial + row / scan_tile;
                if (cnt) atomicAdd((unsigned long long*)sum, (unsigned long long)cnt);
            }
        }
        __syncthreads();
    }
}

// Parents of the rows above BFS_HEAVY (the (sel2nd, min) semiring of the
// BFS-tree variant): a block per chunk finds the first neighbour of the chunk
// for every new bit whose parent so far lies behind the chunk's first column,
// 256 neighbours at a time until every bit has one, and takes the minimum
// into parents.  (A's rows ascend: once a chunk is reached, a parent at or
// below its first column is final.)
template <int DWP>
__global__ void __launch_bounds__(256) k_bfs_heavy_parents(BfsParams p, const unsigned* __restrict__ fb,
                                                           const unsigned* __restrict__ nonempty,
                                                           const long long* __restrict__ items, long long item_cap) {
    __shared__ unsigned s_rem[DWP];
    __shared__ int s_first[32 * DWP];
    const int lane = lane_id(), warp = warp_id(), tid = threadIdx.x;
    const long long nitems = min((long long)__ldcg(p.queue), item_cap);
    if (nitems == 0) return;
    const BfsCols cols{p.Ai, nonempty, p.nF, bfs_entries(p) < p.n / BFS_SPARSE};
    for (long long it = blockIdx.x; it < nitems; it += gridDim.x) {
        const long long row = items[it] >> 24, c = items[it] & 0xFFFFFF;
        const long long a0 = clampll(__ldg(p.Ap + row), 0, p.nnzA);
        const long long a1 = clampll(__ldg(p.Ap + row + 1), a0, p.nnzA);
        const long long e0 = a0 + c * BFS_CHUNK;
        const int n = (int)(a1 - e0 < BFS_CHUNK ? a1 - e0 : BFS_CHUNK);
        const int u0 = __ldg(p.Ai + e0);
        if (warp < DWP) {
            bool need = false;
            const int b = 32 * warp + lane;
            if (warp < p.dw && ((__ldcg(p.newbits + row * p.ns + warp) >> lane) & 1u))
                need = __ldcg(p.parents + row * p.d + b) > u0;
            const unsigned r = __ballot_sync(FULL, need);
            if (lane == 0) s_rem[warp] = r;
            s_first[b] = 0x7FFFFFFF;
        }
        __syncthreads();
        for (int j = 0; j < n; j += 256) {
            unsigned rem[DWP];
            unsigned live = 0u;
#pragma unroll
            for (int m = 0; m < DWP; ++m) {
                rem[m] = s_rem[m];
                live |= rem[m];
            }
            if (!live) break;  // the same for the whole block
            const int u = cols.load(e0 + j + tid, j + tid < n);
            unsigned w[DWP];
            unsigned h = 0u;
#pragma unroll
            for (int m = 0; m < DWP; ++m) w[m] = 0u;
            if (cols.hit(u)) load_bit_row<DWP>(fb, u, w);
#pragma unroll
            for (int m = 0; m < DWP; ++m) h |= w[m] & rem[m];
            if (__any_sync(FULL, h != 0u)) {
#pragma unroll
                for (int m = 0; m < DWP; ++m) {
                    int parent;
                    bool found;
                    bfs_first(w[m] & rem[m], u, parent, found);
                    if (found) atomicMin(&s_first[32 * m + lane], parent);
                }
            }
            __syncthreads();
            if (warp < DWP) {
                const unsigned r = __ballot_sync(FULL, s_first[32 * warp + lane] != 0x7FFFFFFF);
                if (lane == 0) s_rem[warp] &= ~r;
            }
            __syncthreads();
        }
        __syncthreads();
        if (warp < p.dw && s_first[32 * warp + lane] != 0x7FFFFFFF)
            atomicMin(p.parents + row * p.d + 32 * warp + lane, s_first[32 * warp + lane]);
        __syncthreads();
    }
}

// Columns of F_next from the new words, a warp per 32 rows: each row's bits
// are written side by side, lane l bit l of every word.  Up to eight words a
// row are loaded for all 32 rows at once (a load per row left each row to
// wait for L2: 105 us for 57 million entries, so 90 us).  Nothing is written
// when F_next does not fit (the caller repeats the read-out with more room);
// hdr->total gets the number of entries.
__global__ void __launch_bounds__(256) k_bfs_emit(long long n, int dw, const unsigned* __restrict__ newbits,
                                                  const long long* __restrict__ rp, int* __restrict__ col,
                                                  long long cap, WsHeader* hdr) {
    const long long total = __ldg(rp + n);
    if (blockIdx.x == 0 && threadIdx.x == 0) hdr->total = total;
    if (total > cap) return;
    const int lane = lane_id();
    const unsigned lt = lanemask_lt();
    const long long base = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32;
    const long long v = base + lane;
    long long pos = 0, end = 0;
    if (v < n) {
        pos = __ldg(rp + v);
        end = __ldg(rp + v + 1);
    }
    const bool some = end > pos;
    auto put = [&](unsigned word, int m, long long& at, long long last) {
        if ((word >> lane) & 1u) {
            const long long q = at + __popc(word & lt);
            if (q < last && q < cap) col[q] = 32 * m + lane;
            else atomicOr(&hdr->err, ERR_CAPACITY);
        }
        at += __popc(word);
    };
    if (dw <= 8) {
        unsigned w[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) w[m] = some && m < dw ? __ldg(newbits + v * dw + m) : 0u;
        for (unsigned rows = __ballot_sync(FULL, some); rows; rows &= rows - 1) {
            const int r = __ffs(rows) - 1;
            long long at = shfl64(pos, r);
            const long long last = shfl64(end, r);
#pragma unroll
            for (int m = 0; m < 8; ++m)
                if (m < dw) put(__shfl_sync(FULL, w[m], r), m, at, last);
        }
        return;
    }
    for (unsigned rows = __ballot_sync(FULL, some); rows; rows &= rows - 1) {
        const int r = __ffs(rows) - 1;
        long long at = shfl64(pos, r);
        const long long last = shfl64(end, r);
        for (int m0 = 0; m0 < dw; m0 += 32) {
            const unsigned mine = m0 + lane < dw ? __ldg(newbits + (base + r) * dw + m0 + lane) : 0u;
            for (int m = 0; m < 32 && m0 + m < dw; ++m) put(__shfl_sync(FULL, mine, m), m0 + m, at, last);
        }
    }
}

// Words per bitmap row of the pull form (0: list form only, d > 256).
int msbfs_pull_words(int d) {
    const int dw = (d + 31) / 32;
    if (dw > 8) return 0;
    return dw <= 1 ? 1 : (dw <= 2 ? 2 : (dw <= 4 ? 4 : 8));
}

// Rows per warp of the pull: 32, or fewer (a power of two, at least 4) while
// that leaves less than 16 warps per SM.
static int pull_rows(long long n, int sms) {
    int rows = 32;
    while (rows > 4 && n < (long long)sms * 16 * rows) rows /= 2;
    return rows;
}

// One level: the pull, then the chunks of the heavy rows it queued.
template <int DWP, bool SEARCH>
static cudaError_t launch_level(const BfsParams& p, const unsigned* fb, const unsigned* ne, long long* items,
                                long long item_cap, int* done, long long* partial, int sms, cudaStream_t st) {
    const int rows = pull_rows(p.n, sms), tile = scan_tile_rows();
    const long long per_block = (long long)(PULL_THREADS / 32) * rows;
    const unsigned grid = (unsigned)((p.n + per_block - 1) / per_block);
    count_launch();
    if (p.parents)
        k_bfs_pull<DWP, true, SEARCH><<<grid, PULL_THREADS, 0, st>>>(p, fb, ne, rows, items, item_cap, done, partial, tile);
    else
        k_bfs_pull<DWP, false, SEARCH><<<grid, PULL_THREADS, 0, st>>>(p, fb, ne, rows, items, item_cap, done, partial, tile);
    if (p.nnzA > BFS_HEAVY) {
        const unsigned hg = (unsigned)(sms * 4);
        count_launch();
        k_bfs_heavy<DWP, SEARCH><<<hg, 256, 0, st>>>(p, fb, ne, items, item_cap, done, partial, tile);
        if (p.parents) {
            count_launch();
            k_bfs_heavy_parents<DWP><<<hg, 256, 0, st>>>(p, fb, ne, items, item_cap);
        }
    }
    return cudaGetLastError();
}

template <int DWP>
static cudaError_t launch_pull(BfsParams p, const DevCsr& F, unsigned* fb, const Sched& s, const LaunchCfg& cfg,
                               long long* rp_next, cudaStream_t st) {
    const long long n = F.nrows;
    unsigned* nonempty = reinterpret_cast<unsigned*>(s.blen);  // n / 32 words of the n the region holds
    const unsigned nfront = (unsigned)((n + 255) / 256);
    const unsigned ncheck = (unsigned)((p.nnzA + CHECK_PER_BLOCK - 1) / CHECK_PER_BLOCK);
    count_launch();
    k_bfs_frontier<DWP><<<nfront + ncheck, 256, 0, st>>>(n, p.d, F.rowptr, F.nnz, F.col, fb, nonempty, s.partial,
                                                         (long long)scan_partial_count(n), rp_next, nfront, p.Ap,
                                                         p.Ai, p.nnzA, &p.hdr->err);
    p.ss = p.ns = p.dw;
    p.queue = (unsigned long long*)&p.hdr->scratch[0];
    p.err = &p.hdr->err;
    p.fnnz = F.nnz;
    return launch_level<DWP, false>(p, fb, nonempty, s.items, flops_item_capacity(n, p.nnzA),
                                    reinterpret_cast<int*>(s.flops), s.partial, cfg.sms, st);
}

// ---------------------------------------------------------------------------
// Whole search (d <= 256): the frontier never leaves the bitmap form, so a
// level is the pull alone: no list of F is written, read back or sized, and
// the host reads the sizes of four levels at a time instead of waiting for
// each (a step's wait and the calls after it left the GPU idle for 30 - 60 us
// of every level).  A level that starts with an empty frontier ends at once.
// Buffers by level: frontier bitmaps modulo 2, non-empty bits modulo 3 (one
// is read, one added to, one cleared), counters modulo 2 * BFS_GROUP.
// The 128-source search of the scale-20 graph: 2.11 -> 1.29 ms (steps as
// above, from Python); the trees of 50 sources, 300,007 vertices: 1.09 -> 0.68.
// ---------------------------------------------------------------------------
constexpr int BFS_GROUP = 4;

struct BfsLevelCtl {
    long long count[BFS_COUNTS * BFS_COUNT_STRIDE];  // entries of the frontier this level found
    unsigned long long queue;     // chunks of heavy rows
};

struct BfsCtl {
    unsigned long long err;
    BfsLevelCtl level[2 * BFS_GROUP];
};

// The range check of A's columns on its own (a search checks A once).
__global__ void __launch_bounds__(256) k_bfs_check(long long n, const long long* __restrict__ Ap,
                                                   const int* __restrict__ Ai, long long nnzA,
                                                   unsigned long long* err) {
    check_columns(blockIdx.x, n, Ap, Ai, nnzA, err);
}

__global__ void k_bfs_sources(long long n, int d, int words, const int* __restrict__ src, unsigned* S, unsigned* fb,
                              unsigned* nonempty, int* levels, int* parents, long long* count) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s == 0) *count = d;
    if (s >= d) return;
    const int v = src[s];
    if (v < 0 || (long long)v >= n) return;
    atomicOr(S + (long long)v * words + (s >> 5), 1u << (s & 31));
    atomicOr(fb + (long long)v * words + (s >> 5), 1u << (s & 31));
    atomicOr(nonempty + (v >> 5), 1u << (v & 31));
    levels[(long long)v * d + s] = 0;
    if (parents) parents[(long long)v * d + s] = v;
}

struct BfsSearchWs {
    BfsCtl* ctl;
    unsigned* S;
    unsigned* fb[2];
    unsigned* ne[3];
    int* done;
    long long* items;
};

static size_t search_ws(char* base, long long n, long long nnzA, int d, BfsSearchWs* out) {
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* p = base + off;
        off += (bytes + 255) & ~(size_t)255;
        return p;
    };
    const size_t words = sizeof(unsigned) * (size_t)n * (size_t)msbfs_pull_words(d);
    BfsSearchWs w;
    w.ctl = (BfsCtl*)take(sizeof(BfsCtl));
    w.S = (unsigned*)take(words);
    for (auto& f : w.fb) f = (unsigned*)take(words);
    for (auto& b : w.ne) b = (unsigned*)take(sizeof(unsigned) * (size_t)((n + 31) / 32));
    w.done = (int*)take(sizeof(int) * (size_t)n);
    w.items = (long long*)take(sizeof(long long) * (size_t)flops_item_capacity(n, nnzA));
    if (out) *out = w;
    return off;
}

size_t msbfs_search_bytes(long long n, long long nnzA, int d) { return search_ws(nullptr, n, nnzA, d, nullptr); }

template <int DWP>
static cudaError_t search_levels(const BfsParams& p0, const BfsSearchWs& w, long long first, int levels, int sms,
                                 cudaStream_t st) {
    const long long cap = flops_item_capacity(p0.n, p0.nnzA);
    for (long long l = first; l < first + levels; ++l) {  // level l + 1 of the search
        BfsParams p = p0;
        BfsLevelCtl* now = &w.ctl->level[l % (2 * BFS_GROUP)];
        p.prev = w.ctl->level[(l + 2 * BFS_GROUP - 1) % (2 * BFS_GROUP)].count;
        p.count = now->count;
        p.queue = &now->queue;
        p.level = (int)(l + 1);
        p.newbits = w.fb[(l + 1) & 1];
        p.ne_next = w.ne[(l + 1) % 3];
        p.ne_clear = w.ne[(l + 2) % 3];
        cudaError_t e = launch_level<DWP, true>(p, w.fb[l & 1], w.ne[l % 3], w.items, cap, w.done, nullptr, sms, st);
        if (e) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_msbfs_search(const DevCsr& A, int d, const int* src, int* levels, int* parents, long long start,
                                long long max_steps, long long* frontier, long long* steps, unsigned long long* err,
                                int sms, void* ws, cudaStream_t st) {
    cudaError_t e;
    const long long n = A.nrows;
    const int words = msbfs_pull_words(d);
    BfsSearchWs w;
    search_ws((char*)ws, n, A.nnz, d, &w);
    *steps = 0;
    *err = 0;
    if (!words) return cudaErrorInvalidValue;
    if (start == 0) {
        const size_t bytes = sizeof(unsigned) * (size_t)n * words;
        const size_t bits = sizeof(unsigned) * (size_t)((n + 31) / 32);
        if ((e = cudaMemsetAsync(w.ctl, 0, sizeof(BfsCtl), st))) return e;
        if ((e = cudaMemsetAsync(w.S, 0, bytes, st))) return e;
        if ((e = cudaMemsetAsync(w.fb[0], 0, bytes, st))) return e;
        for (unsigned* b : w.ne)
            if ((e = cudaMemsetAsync(b, 0, bits, st))) return e;
        if ((e = cudaMemsetAsync(levels, 0xFF, sizeof(int) * (size_t)n * d, st))) return e;
        if (parents && (e = cudaMemsetAsync(parents, 0xFF, sizeof(int) * (size_t)n * d, st))) return e;
        count_launch();
        k_bfs_sources<<<(d + 127) / 128, 128, 0, st>>>(n, d, words, src, w.S, w.fb[0], w.ne[0], levels, parents,
                                                       w.ctl->level[2 * BFS_GROUP - 1].count);
        if (A.nnz > 0) {
            count_launch();
            k_bfs_check<<<(unsigned)((A.nnz + CHECK_PER_BLOCK - 1) / CHECK_PER_BLOCK), 256, 0, st>>>(
                n, A.rowptr, A.col, A.nnz, &w.ctl->err);
        }
        if ((e = cudaGetLastError())) return e;
        // no level follows that the call would wait for: the caller may free ws
        if (max_steps == 0) return cudaStreamSynchronize(st);
    }
    BfsParams p = {};
    p.Ap = A.rowptr;
    p.Ai = A.col;
    p.nnzA = A.nnz;
    p.nF = (int)n;
    p.d = d;
    p.dw = (d + 31) / 32;
    p.S = w.S;
    p.levels = levels;
    p.parents = parents;
    p.err = &w.ctl->err;
    p.n = n;
    p.ss = p.ns = words;
    while (*steps < max_steps) {
        const long long l = start + *steps;
        const int at = (int)(l % (2 * BFS_GROUP));
        int group = BFS_GROUP - at % BFS_GROUP;  // to the end of this half of the counters
        if (group > max_steps - *steps) group = (int)(max_steps - *steps);
        if ((e = cudaMemsetAsync(&w.ctl->level[at], 0, sizeof(BfsLevelCtl) * group, st))) return e;
        switch (words) {
            case 1: e = search_levels<1>(p, w, l, group, sms, st); break;
            case 2: e = search_levels<2>(p, w, l, group, sms, st); break;
            case 4: e = search_levels<4>(p, w, l, group, sms, st); break;
            default: e = search_levels<8>(p, w, l, group, sms, st); break;
        }
        if (e) return e;
        BfsCtl got;
        if ((e = cudaMemcpyAsync(&got, w.ctl, sizeof got, cudaMemcpyDeviceToHost, st))) return e;
        if ((e = cudaStreamSynchronize(st))) return e;
        *err = got.err;
        if (got.err) return cudaSuccess;
        for (int g = 0; g < group; ++g) {
            long long f = 0;
            for (int q = 0; q < BFS_COUNTS; ++q) f += got.level[at + g].count[q * BFS_COUNT_STRIDE];
            frontier[(*steps)++] = f;
            if (f == 0) return cudaSuccess;
        }
    }
    return cudaSuccess;
}

// parents = -1, and each source its own parent in its column.
__global__ void k_msbfs_init_parents(long long n, int d, const int* __restrict__ src, int* parents) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= d) return;
    const int v = src[s];
    if (v < 0 || (long long)v >= n) return;
    parents[(long long)v * d + s] = v;
}

cudaError_t launch_msbfs_init_parents(long long n, int d, const int* src, int* parents, cudaStream_t st) {
    cudaError_t e;
    if ((e = cudaMemsetAsync(parents, 0xFF, sizeof(int) * (size_t)n * d, st))) return e;
    count_launch();
    k_msbfs_init_parents<<<(d + 127) / 128, 128, 0, st>>>(n, d, src, parents);
    return cudaGetLastError();
}

cudaError_t launch_msbfs_init(long long n, int d, const int* src, unsigned* S, int* levels,
                              long long* rp, int* col, cudaStream_t st) {
    cudaError_t e;
    const int dw = (d + 31) / 32;
    if ((e = cudaMemsetAsync(S, 0, sizeof(unsigned) * (size_t)n * dw, st))) return e;
    if ((e = cudaMemsetAsync(levels, 0xFF, sizeof(int) * (size_t)n * d, st))) return e;
    count_launch();
    k_msbfs_init_rows<<<(unsigned)((n + 1 + INIT_ROWS - 1) / INIT_ROWS), 256, 0, st>>>(n, d, src, rp);
    count_launch();
    k_msbfs_init_cols<<<(d + 127) / 128, 128, 0, st>>>(n, d, dw, src, col, S, levels);
    return cudaGetLastError();
}

cudaError_t launch_msbfs_step(const DevCsr& A, const DevCsr& F, int d, unsigned* S, int* levels, int level,
                              const Sched& s, unsigned* newbits, long long* rp_next, const LaunchCfg& cfg,
                              cudaStream_t st, unsigned* fbits, int* parents) {
    cudaError_t e;
    const long long n = A.nrows;
    const int dw = (d + 31) / 32;
    const int dwp = fbits ? msbfs_pull_words(d) : 0;
    if (parents && !dwp) return cudaErrorInvalidValue;  // parents: pull form only
    if (n == 0) {
        if ((e = cudaMemsetAsync(s.hdr, 0, sizeof(WsHeader), st))) return e;
        return cudaMemsetAsync(rp_next, 0, sizeof(long long), st);
    }
    BfsParams p = {};
    p.Ap = A.rowptr;
    p.Ai = A.col;
    p.nnzA = A.nnz;
    p.segF = SegWhole{F.rowptr, F.nnz, d};
    p.Fi = F.col;
    p.nF = (int)F.nrows;
    p.d = d;
    p.dw = dw;
    p.S = S;
    p.levels = levels;
    p.level = level;
    p.newbits = newbits;
    p.cnt_next = rp_next + 1;
    p.parents = parents;
    p.perm = s.perm;
    p.hdr = s.hdr;
    p.cta_class = cfg.cta_class;
    p.n = n;
    if (dwp) {
        if ((e = cudaMemsetAsync(s.hdr, 0, sizeof(WsHeader), st))) return e;
        switch (dwp) {
            case 1: e = launch_pull<1>(p, F, fbits, s, cfg, rp_next, st); break;
            case 2: e = launch_pull<2>(p, F, fbits, s, cfg, rp_next, st); break;
            case 4: e = launch_pull<4>(p, F, fbits, s, cfg, rp_next, st); break;
            default: e = launch_pull<8>(p, F, fbits, s, cfg, rp_next, st); break;
        }
        if (e) return e;
        return launch_scan_summed(rp_next + 1, n, s.partial, st);
    }
    if ((e = launch_row_flops(A, F, s, st))) return e;
    // prune rows that cannot gain bits, then histogram and order (rows left
    // without products get their count 0 here)
    count_launch();
    k_mask_full_rows<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, d, dw, S, s.flops);
    if ((e = launch_reclassify(n, s, rp_next + 1, st))) return e;
    if ((e = cudaMemsetAsync(rp_next, 0, sizeof(long long), st))) return e;
    const int threads = 32 * cfg.warps_per_cta;
    const size_t smem = sizeof(unsigned) * (size_t)dw * cfg.warps_per_cta;
    if (smem > 48 * 1024 &&
        (e = cudaFuncSetAttribute((const void*)k_msbfs_expand, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)smem)))
        return e;
    const int grid = persistent_grid((const void*)k_msbfs_expand, threads, smem, cfg.sms);
    count_launch();
    k_msbfs_expand<<<grid, threads, smem, st>>>(p);
    if ((e = cudaGetLastError())) return e;
    return launch_scan_inplace(rp_next + 1, n, s.partial, st);
}

cudaError_t launch_msbfs_emit(long long n, int d, const unsigned* newbits, const long long* rp, int* col,
                              long long cap, WsHeader* hdr, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    count_launch();
    k_bfs_emit<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, (d + 31) / 32, newbits, rp, col, cap, hdr);
    return cudaGetLastError();
}

}  // namespace ts
