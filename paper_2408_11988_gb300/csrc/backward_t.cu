// Deterministic dB (option T): dB(k, j) = sum over the rows i with A(i, k)
// stored of A(i, k) * dC(i, j), for (k, j) on B's pattern, in an order fixed by
// the matrices (no float atomics, so dB is the same bit for bit on every run).
// dA still comes from the backward kernels (they skip dB).
//
// 1. The transpose of A's pattern: the entry indices of A sorted by column,
//    stably (a least-significant-digit radix sort of the column indices, up to
//    ten bits a pass, the entry index as payload), so that each column's
//    entries stay in ascending row order; the column pointers from the sorted
//    columns; the entries' rows and values gathered once in that order.
// 2. Rows of C as bitmaps (d <= 256), so that the place of (i, j) in row i of
//    C is a count of bits in one or two 16-byte loads.  Above 256 columns, or
//    where the workspace has no room for them, the place is found by binary
//    search.
// 3. The pull: a warp per column k of A.  Groups of 8, 16 or 32 lanes (by the
//    length of B's row k) take entries (i, k) in turn, lane l of a group entry
//    l of B's row (column j): A(i, k) * dC(i, j) is added in ascending order
//    within a group, and the groups are added at the end.  A column of more
//    than TCH entries is cut into chunks of TCH (a fixed cut, so that the order
//    of the sums does not depend on scheduling) taken by any warp; the warp of
//    its last chunk adds the chunks up in order.
//
// Bound by the gathers of the pull (per entry of A a row pointer, a bitmap row
// and |B_k| values of dC, mostly from L2) and by the sort's passes.  500,009
// rows, d = 100, 7.6 million entries, 61 million products: binary searches 4.13
// ms and 0.8 ms around them; with bitmaps the pull takes 0.41 ms (0.08 of it the
// long columns) and the rest 0.34 ms.
#include <algorithm>
#include <utility>

#include "bitrows.cuh"
#include "common.cuh"
#include "kernels.h"

namespace ts {

constexpr int RS_THREADS = 512, RS_ROUNDS = 17, RS_TILE = RS_THREADS * RS_ROUNDS;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_BITS = 10;  // most bits of a digit (tiles of 8704 keys: their counters fit where those of eight
                             // bits and 2048 keys did)
constexpr int TCH = 512;     // entries of A per chunk of a column
constexpr int ROW_TILE = 512;  // entries per warp of k_row_of

// First row whose end lies behind entry e (the row that holds e), by the whole
// warp: 32 pointers probed at a time.
__device__ __forceinline__ long long row_holding(const long long* __restrict__ Ap, long long n, long long e) {
    long long lo = 0, hi = n;  // the row is in [lo, hi)
    while (hi - lo > 1) {
        const long long step = (hi - lo + 31) / 32;
        const long long r = lo + step * lane_id();  // rows lo, lo + step, ...: the last that starts at or before e
        const unsigned le = __ballot_sync(FULL, r < hi && __ldg(Ap + r) <= e);
        const int last = le ? 31 - __clz(le) : 0;
        lo += step * last;
        hi = lo + step < hi ? lo + step : hi;
    }
    return lo;
}

// row_of[e] = row of entry e, or -1 for an entry of no row (before the first
// row pointer or behind the last: A's arrays may hold more than its rows do): a
// warp per ROW_TILE entries (a warp per row left the longest row as a tail: 43 us
// for 500,009 rows).
__global__ void __launch_bounds__(256) k_row_of(long long n, const long long* __restrict__ Ap, long long nnzA,
                                                int* __restrict__ row_of) {
    const int lane = lane_id();
    const long long e0 = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * ROW_TILE;
    if (e0 >= nnzA) return;
    const long long e1 = e0 + ROW_TILE < nnzA ? e0 + ROW_TILE : nnzA;
    long long r = row_holding(Ap, n, e0), e = e0;
    for (; e < e1 && r < n; r += 32) {
        // rows r .. r + 31: lane l holds the bounds of row r + l
        const long long beg = r + lane < n ? clampll(__ldg(Ap + r + lane), 0, nnzA) : nnzA;
        const long long end = r + lane < n ? clampll(__ldg(Ap + r + lane + 1), 0, nnzA) : nnzA;
        const long long upto = shfl64(end, 31) < e1 ? shfl64(end, 31) : e1;
        for (long long x = e + lane; x - lane < upto; x += 32) {
            int q = 0;  // rows that end at or before x
#pragma unroll
            for (int s = 16; s >= 1; s >>= 1)
                if (shfl64(end, q + s - 1) <= x) q += s;
            const long long starts = shfl64(beg, q);
            if (x < upto) row_of[x] = r + q < n && starts <= x ? (int)(r + q) : -1;
        }
        if (upto > e) e = upto;
    }
    for (long long x = e + lane; x < e1; x += 32) row_of[x] = -1;
}

// Per tile of RS_TILE keys, the count of each digit: cnt[digit * nb + tile].
__global__ void __launch_bounds__(RS_THREADS) k_rs_count(const int* __restrict__ key, long long m, int shift, int nd,
                                                         long long* __restrict__ cnt, long long nb) {
    __shared__ int s_c[1 << RS_BITS];
    for (int d = threadIdx.x; d < nd; d += RS_THREADS) s_c[d] = 0;
    __syncthreads();
    const long long t0 = (long long)blockIdx.x * RS_TILE;
#pragma unroll 4
    for (int r = 0; r < RS_ROUNDS; ++r) {
        const long long x = t0 + r * RS_THREADS + threadIdx.x;
        if (x < m) atomicAdd(&s_c[((unsigned)__ldg(key + x) >> shift) & (nd - 1)], 1);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < nd; d += RS_THREADS) cnt[(long long)d * nb + blockIdx.x] = s_c[d];
}

// Stable scatter of one tile: keys of a digit keep their order, after every
// key of a smaller digit and every key of that digit in earlier tiles
// (incl = inclusive scan of cnt in digit-major order).  A warp ranks its
// consecutive keys on its own (ballots over the digit's bits, counters of its own in
// shared memory); the warps' counters are then turned into places in the tile
// once, the tile is put in order in shared memory and written from there, so
// that a digit's keys go out side by side.  (Five block barriers for every 256
// keys and writes key by key: 100 us a pass of eight bits for 7.6 million keys;
// ranks by warp, writes key by key: 130; this way 63 - 75 us for ten bits.)
// vin == nullptr: the payload is the key's own index.
constexpr int RS_STAGE = 2 * RS_TILE;  // ints of shared memory: the tile's keys and payloads

__global__ void __launch_bounds__(RS_THREADS, 2) k_rs_scatter(const int* __restrict__ kin,
                                                              const int* __restrict__ vin, int* __restrict__ kout,
                                                              int* __restrict__ vout, long long m, int shift, int nd,
                                                              const long long* __restrict__ incl, long long nb) {
    extern __shared__ int s_mem[];  // warps' counters [RS_WARPS][nd], then the tile
    __shared__ long long s_base[1 << RS_BITS];  // global place of a digit's first key, less its place in the tile
    __shared__ int s_sum[RS_WARPS];
    const int tid = threadIdx.x, warp = warp_id(), lane = lane_id();
    for (int i = tid; i < RS_WARPS * nd; i += RS_THREADS) s_mem[i] = 0;
    __syncthreads();
    int* mine = s_mem + warp * nd;
    const long long t0 = (long long)blockIdx.x * RS_TILE;
    const int n = (int)(m - t0 < RS_TILE ? m - t0 : RS_TILE);  // keys of this tile
    const int i0 = warp * 32 * RS_ROUNDS + lane;
    const unsigned lt = lanemask_lt();
    int key[RS_ROUNDS], rank[RS_ROUNDS];
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) key[r] = i0 + 32 * r < n ? __ldg(kin + t0 + i0 + 32 * r) : 0;
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) {
        const bool ok = i0 + 32 * r < n;
        const int dg = (int)((unsigned)key[r] >> shift) & (nd - 1);
        unsigned mm = __ballot_sync(FULL, ok);  // the lanes with this digit (a ballot a bit: match is slower)
        for (int b = 1; b < nd; b <<= 1) {
            const unsigned set = __ballot_sync(FULL, (dg & b) != 0);
            mm &= (dg & b) ? set : ~set;
        }
        const int first = __ffs(mm) - 1;
        int before = 0;
        if (ok && lane == first) {
            before = mine[dg];
            mine[dg] = before + __popc(mm);
        }
        rank[r] = __shfl_sync(FULL, before, first & 31) + __popc(mm & lt);
        __syncwarp();
    }
    __syncthreads();
    // places in the tile: digits in order, a digit's keys by warp
    int tot[(1 << RS_BITS) / RS_THREADS], sum = 0;  // this thread's digits PER * tid + ...
    constexpr int PER = (1 << RS_BITS) / RS_THREADS;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int d = PER * tid + q;
        tot[q] = 0;
        if (d < nd) {
#pragma unroll
            for (int w = 0; w < RS_WARPS; ++w) tot[q] += s_mem[w * nd + d];
        }
        sum += tot[q];
    }
    int run = warp_incl_scan(sum);
    if (lane == 31) s_sum[warp] = run;
    __syncthreads();
    run -= sum;
    for (int w = 0; w < warp; ++w) run += s_sum[w];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int d = PER * tid + q;
        if (d < nd) {
            s_base[d] = incl[(long long)d * nb + blockIdx.x] - tot[q] - run;
            int at = run;
#pragma unroll
            for (int w = 0; w < RS_WARPS; ++w) {
                const int c = s_mem[w * nd + d];
                s_mem[w * nd + d] = at;
                at += c;
            }
        }
        run += tot[q];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) rank[r] += mine[(int)((unsigned)key[r] >> shift) & (nd - 1)];
    __syncthreads();  // the counters make room for the tile
    int* s_key = s_mem;
    int* s_val = s_mem + RS_TILE;
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) {
        const int i = i0 + 32 * r;
        if (i < n) {
            s_key[rank[r]] = key[r];
            s_val[rank[r]] = vin ? __ldg(vin + t0 + i) : (int)(t0 + i);
        }
    }
    __syncthreads();
#pragma unroll 4
    for (int i = tid; i < n; i += RS_THREADS) {
        const int k = s_key[i];
        const long long pos = s_base[(int)((unsigned)k >> shift) & (nd - 1)] + i;
        kout[pos] = k;
        vout[pos] = s_val[i];
    }
}

// Column pointers from the sorted columns (mask: the bits they were sorted by;
// a column outside [0, n) was reported by the forward).
__global__ void __launch_bounds__(256) k_col_ptr(const int* __restrict__ key, long long m, long long n, unsigned mask,
                                                 long long* __restrict__ ATp) {
    for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x <= m;
         x += (long long)gridDim.x * blockDim.x) {
        const long long prev = x > 0 ? (long long)((unsigned)__ldg(key + x - 1) & mask) : -1;
        const long long cur = x < m ? (long long)((unsigned)__ldg(key + x) & mask) : n;
        for (long long c = prev + 1; c <= cur && c <= n; ++c) ATp[c] = x;
    }
}

// The sorted entries' rows and values, gathered once: ti[q], ta[q].
__global__ void __launch_bounds__(256) k_t_gather(long long m, const int* __restrict__ tperm,
                                                  const int* __restrict__ row_of, const float* __restrict__ Ax,
                                                  int* __restrict__ ti, float* __restrict__ ta) {
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < m; q += (long long)gridDim.x * blockDim.x) {
        const int e = __ldg(tperm + q);
        ti[q] = __ldg(row_of + e);
        ta[q] = __ldg(Ax + e);
    }
}

// Rows of C as bitmaps of DWP words.
template <int DWP>
__global__ void __launch_bounds__(256) k_t_bits(long long n, int d, const long long* __restrict__ Cp, long long nnzC,
                                                const int* __restrict__ Ci, unsigned* __restrict__ bits) {
    __shared__ unsigned s_bits[8][32 * DWP];
    __shared__ int s_start[8][33];
    const int lane = lane_id(), warp = warp_id();
    const long long base = ((long long)blockIdx.x * 8 + warp) * 32;
    if (base >= n) return;
    rows_to_bits<DWP>(n, d, Cp, nnzC, Ci, base, s_bits[warp], s_start[warp]);
#pragma unroll
    for (int m = 0; m < DWP; ++m)
        if (32 * m + lane < (n - base) * DWP) bits[base * DWP + 32 * m + lane] = s_bits[warp][32 * m + lane];
}

// A long column's chunks: item x is chunk x - at of column k; the column's
// first item holds the counter of its finished chunks.
struct TItem {
    long long k;     // column
    long long part;  // where this chunk's sums go
    int at;          // x - chunk: the column's first item
    int done;
};

struct TParams {
    long long n;
    int d;
    const long long* ATp;
    const int* ti;
    const float* ta;
    const long long* Bp;
    const int* Bi;
    long long nnzB;
    const long long* Cp;
    const int* Ci;
    const float* dC;
    long long nnzC;
    const unsigned* bits;
    float* dB;
    float* part;
    TItem* items;
    long long item_cap, part_cap;
    unsigned long long* nitems;  // items queued, then floats of `part` taken
    WsHeader* hdr;
};

// Places of column j in rows iv[0..U) of C (-1: no row, or not stored).
template <int DWP>
struct BitPlaces {
    static constexpr int U = DWP <= 4 ? 4 : 2;
    static __device__ __forceinline__ void find(const TParams& p, const int (&iv)[U], int j, long long (&pos)[U]) {
        unsigned w[U][DWP];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            pos[u] = -1;
#pragma unroll
            for (int m = 0; m < DWP; ++m) w[u][m] = 0u;
            if (iv[u] >= 0) {
                pos[u] = __ldg(p.Cp + iv[u]);
                load_bit_row<DWP>(p.bits, iv[u], w[u]);
            }
        }
        const int word = j >> 5;  // -1 for no column: no word
        const unsigned below = (1u << (j & 31)) - 1u;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            int before = 0;
            unsigned at = 0u;
#pragma unroll
            for (int m = 0; m < DWP; ++m) {
                before += __popc(w[u][m] & (m < word ? FULL : m == word ? below : 0u));
                at = m == word ? w[u][m] : at;
            }
            const long long q = pos[u] + before;
            pos[u] = ((at >> (j & 31)) & 1u) && q >= 0 && q < p.nnzC ? q : -1;
        }
    }
};

struct SearchPlaces {
    static constexpr int U = 4;
    // four binary searches advanced together (one load of each per step)
    static __device__ __forceinline__ void find(const TParams& p, const int (&iv)[U], int j, long long (&pos)[U]) {
        long long lo[U], len[U], end[U];
        int steps = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            lo[u] = len[u] = end[u] = 0;
            if (iv[u] >= 0) {
                lo[u] = clampll(__ldg(p.Cp + iv[u]), 0, p.nnzC);
                end[u] = clampll(__ldg(p.Cp + iv[u] + 1), lo[u], p.nnzC);
                len[u] = end[u] - lo[u];
            }
            const int b = 64 - __clzll(len[u]);
            steps = steps > b ? steps : b;
        }
        for (int t = 0; t < steps; ++t) {
            int c[U];
#pragma unroll
            for (int u = 0; u < U; ++u) c[u] = len[u] > 0 ? __ldg(p.Ci + lo[u] + (len[u] >> 1)) : 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (len[u] > 0) {
                    const long long h = len[u] >> 1;
                    if (c[u] < j) {
                        lo[u] += h + 1;
                        len[u] -= h + 1;
                    } else {
                        len[u] = h;
                    }
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) pos[u] = iv[u] >= 0 && lo[u] < end[u] && __ldg(p.Ci + lo[u]) == j ? lo[u] : -1;
    }
};

// Entries [q0, q1) of column k against B's row k (L entries from bs): the sums
// to out[0..L).
template <class Places>
__device__ __forceinline__ void t_chunk(const TParams& p, long long q0, long long q1, long long bs, int L, float* out,
                                        bool& bad) {
    constexpr int U = Places::U;
    const int lane = lane_id();
    const int width = L <= 8 ? 8 : L <= 16 ? 16 : 32, groups = 32 / width, g = lane / width;
    for (int jb = 0; jb < L; jb += width) {
        const int jl = jb + lane % width;
        const bool on = jl < L;
        const int j = on ? __ldg(p.Bi + bs + jl) : -1;
        float acc = 0.0f;
        // groups of U entries of A: group g takes groups g, g + groups, ...
        for (long long q = q0 + (long long)U * g; q < q1; q += (long long)U * groups) {
            int iv[U];
            float av[U], x[U];
            long long pos[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                iv[u] = q + u < q1 ? __ldg(p.ti + q + u) : -1;
                av[u] = q + u < q1 ? __ldg(p.ta + q + u) : 0.0f;
            }
            Places::find(p, iv, j, pos);
#pragma unroll
            for (int u = 0; u < U; ++u) x[u] = pos[u] >= 0 ? __ldg(p.dC + pos[u]) : 0.0f;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (pos[u] >= 0) acc = fmaf(av[u], x[u], acc);
                else bad |= on && iv[u] >= 0;
            }
        }
        __syncwarp();
        for (int o = 16; o >= width; o >>= 1) acc += __shfl_down_sync(FULL, acc, o);  // always in this order
        if (on && g == 0) out[jl] = acc;
    }
}

// LONG = false: a warp per column; columns of more than TCH entries are
// queued.  LONG = true: a warp per queued chunk.  Small blocks, since a block
// holds its warps' places until the slowest is done (256 threads: 1.85 against
// 1.79 ms for the whole training step).  (Loading the next column's pointers
// and entries of A ahead took 80 instead of 60 registers and 489 us.)
constexpr int PULL_T_THREADS = 64;
constexpr int PULL_T_BLOCKS = 256;  // per SM, of the columns' kernel
template <class Places, bool LONG>
__global__ void __launch_bounds__(PULL_T_THREADS) k_t_pull(TParams p) {
    const int lane = lane_id();
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    const long long units = LONG ? min((long long)__ldcg(p.nitems), p.item_cap) : p.n;
    bool bad = false;
    for (long long x = gw; x < units; x += nw) {
        const long long k = LONG ? p.items[x].k : x;
        if (LONG && k < 0) continue;
        const long long bs = clampll(__ldg(p.Bp + k), 0, p.nnzB), be = clampll(__ldg(p.Bp + k + 1), bs, p.nnzB);
        const int L = (int)(be - bs < p.d ? be - bs : p.d);
        if (L == 0) continue;
        const long long t0 = __ldg(p.ATp + k), t1 = __ldg(p.ATp + k + 1);
        const int nch = (int)((t1 - t0 + TCH - 1) / TCH);
        if (!LONG) {
            if (nch <= 1) {
                t_chunk<Places>(p, t0, t1, bs, L, p.dB + bs, bad);
                continue;
            }
            unsigned long long at = 0, part = 0;
            if (lane == 0) {
                at = atomicAdd(p.nitems, (unsigned long long)nch);
                part = atomicAdd(p.nitems + 1, (unsigned long long)nch * L);
            }
            at = __shfl_sync(FULL, at, 0);
            part = __shfl_sync(FULL, part, 0);
            const bool room = (long long)at + nch <= p.item_cap && (long long)part + (long long)nch * L <= p.part_cap;
            if (!room && lane == 0) atomicOr(&p.hdr->err, ERR_CAPACITY);  // row pointers that do not ascend
            for (int c = lane; c < nch; c += 32)
                if ((long long)at + c < p.item_cap)
                    p.items[at + c] = TItem{room ? k : -1, (long long)part + (long long)c * L, (int)at, 0};
            continue;
        }
        const int at = p.items[x].at, c = (int)(x - at);
        const long long q0 = t0 + (long long)c * TCH;
        t_chunk<Places>(p, q0, q0 + TCH < t1 ? q0 + TCH : t1, bs, L, p.part + p.items[x].part, bad);
        __threadfence();
        __syncwarp();
        int before = 0;
        if (lane == 0) before = atomicAdd(&p.items[at].done, 1);
        if (__shfl_sync(FULL, before, 0) != nch - 1) continue;
        __threadfence();
        const float* first = p.part + p.items[at].part;
        for (int j = lane; j < L; j += 32) {
            float s = 0.0f;
#pragma unroll 8
            for (int q = 0; q < nch; ++q) s += __ldcg(first + (long long)q * L + j);
            p.dB[bs + j] = s;
        }
    }
    if (bad) atomicOr(&p.hdr->err, ERR_C_ROW);
}

static size_t al256(size_t b) { return (b + 255) & ~(size_t)255; }

// Layout of the workspace.
struct TWs {
    int *row_of, *k0, *k1, *v0, *v1;
    long long* cnt;      // the sort's counters, then the long columns' items
    size_t cnt_bytes;
    long long* spart;    // their scan's partial sums
    long long* ATp;
    float* part;         // the long columns' sums: every row of B once and one more row per full chunk
    long long part_cap;
};

static size_t t_ws(char* base, long long n, long long nnzA, long long nnzB, long long d, TWs* out) {
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* p = base + off;
        off += al256(bytes);
        return p;
    };
    TWs w;
    for (int** a : {&w.row_of, &w.k0, &w.k1, &w.v0, &w.v1}) *a = (int*)take(sizeof(int) * (size_t)nnzA);
    const size_t counts = (size_t)((nnzA + RS_TILE - 1) / RS_TILE) << RS_BITS;
    w.cnt_bytes = sizeof(long long) * counts;
    w.cnt = (long long*)take(w.cnt_bytes);
    w.spart = (long long*)take(sizeof(long long) * scan_partial_count((long long)counts));
    w.ATp = (long long*)take(sizeof(long long) * (size_t)(n + 1));
    w.part_cap = nnzB + d * (nnzA / TCH + 1);
    w.part = (float*)take(sizeof(float) * (size_t)w.part_cap);
    if (out) *out = w;
    return off;
}

size_t backward_t_bytes(long long n, long long nnzA, long long nnzB, long long d) {
    return t_ws(nullptr, n, nnzA, nnzB, d, nullptr);
}

template <class Places>
static cudaError_t launch_pulls(const TParams& p, long long m, cudaStream_t st) {
    cudaError_t e;
    constexpr int W = PULL_T_THREADS / 32;
    const unsigned g = (unsigned)std::min<long long>((p.n + W - 1) / W, 152LL * PULL_T_BLOCKS);
    count_launch();
    k_t_pull<Places, false><<<g, PULL_T_THREADS, 0, st>>>(p);
    if ((e = cudaGetLastError())) return e;
    if (m <= TCH) return cudaSuccess;
    count_launch();
    k_t_pull<Places, true><<<(unsigned)std::min<long long>((p.item_cap + W - 1) / W, 152LL * 32), PULL_T_THREADS, 0, st>>>(p);
    return cudaGetLastError();
}

template <int DWP>
static cudaError_t launch_bits_and_pulls(const TParams& p, unsigned* bits, long long m, cudaStream_t st) {
    count_launch();
    k_t_bits<DWP><<<(unsigned)((p.n + 255) / 256), 256, 0, st>>>(p.n, p.d, p.Cp, p.nnzC, p.Ci, bits);
    cudaError_t e = cudaGetLastError();
    return e ? e : launch_pulls<BitPlaces<DWP>>(p, m, st);
}

cudaError_t launch_backward_t(const DevCsr& A, const DevCsr& B, long long d, const long long* Cp, const int* Ci,
                              long long nnzC, const float* dC, float* dB, void* ws, void* bits_room,
                              size_t bits_bytes, WsHeader* hdr, cudaStream_t st) {
    cudaError_t e;
    const long long n = A.nrows, m = A.nnz;
    if (!dB || B.nnz == 0) return cudaSuccess;
    if (m == 0) return cudaMemsetAsync(dB, 0, sizeof(float) * B.nnz, st);
    const long long nb = (m + RS_TILE - 1) / RS_TILE;
    TWs w;
    t_ws((char*)ws, n, m, B.nnz, d, &w);
    const unsigned g256 = (unsigned)std::min<long long>((m + 256) / 256, 152LL * 16);
    count_launch();
    k_row_of<<<(unsigned)((m + 8LL * ROW_TILE - 1) / (8LL * ROW_TILE)), 256, 0, st>>>(n, A.rowptr, m, w.row_of);
    int bits = 1;
    while ((1LL << bits) < n) ++bits;
    // passes of equal digits, of at most RS_BITS bits
    const int passes = (bits + RS_BITS - 1) / RS_BITS, width = (bits + passes - 1) / passes;
    const size_t smem = sizeof(int) * (size_t)std::max(RS_STAGE, RS_WARPS << width);
    if ((e = cudaFuncSetAttribute((const void*)k_rs_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)))
        return e;
    const int *kin = A.col, *vin = nullptr;
    int *kout = w.k0, *vout = w.v0, *kalt = w.k1, *valt = w.v1;
    for (int shift = 0; shift < bits; shift += width) {
        const int nd = 1 << (bits - shift < width ? bits - shift : width);
        count_launch();
        k_rs_count<<<(unsigned)nb, RS_THREADS, 0, st>>>(kin, m, shift, nd, w.cnt, nb);
        if ((e = launch_scan_inplace(w.cnt, nd * nb, w.spart, st))) return e;
        count_launch();
        k_rs_scatter<<<(unsigned)nb, RS_THREADS, smem, st>>>(kin, vin, kout, vout, m, shift, nd, w.cnt, nb);
        kin = kout;
        vin = vout;
        std::swap(kout, kalt);
        std::swap(vout, valt);
    }
    // kin, vin: columns and entry indices sorted by column (stable)
    count_launch();
    k_col_ptr<<<g256, 256, 0, st>>>(kin, m, n, (unsigned)((1ull << bits) - 1), w.ATp);
    // rows and values of the sorted entries (into the free sort buffers)
    int* ti = kout;
    float* ta = reinterpret_cast<float*>(vout);
    count_launch();
    k_t_gather<<<g256, 256, 0, st>>>(m, vin, w.row_of, A.val, ti, ta);
    if ((e = cudaMemsetAsync(&hdr->scratch[4], 0, 2 * sizeof(long long), st))) return e;
    TParams p;
    p.n = n;
    p.d = (int)d;
    p.ATp = w.ATp;
    p.ti = ti;
    p.ta = ta;
    p.Bp = B.rowptr;
    p.Bi = B.col;
    p.nnzB = B.nnz;
    p.Cp = Cp;
    p.Ci = Ci;
    p.dC = dC;
    p.nnzC = nnzC;
    p.dB = dB;
    p.part = w.part;
    p.part_cap = w.part_cap;
    p.items = (TItem*)w.cnt;  // the sort is done with its counters
    p.item_cap = (long long)(w.cnt_bytes / sizeof(TItem));
    p.nitems = (unsigned long long*)&hdr->scratch[4];
    p.hdr = hdr;
    // the bitmaps: in the room given, or in row_of's (no longer needed)
    const int dw = (int)((d + 31) / 32), words = dw <= 1 ? 1 : dw <= 2 ? 2 : dw <= 4 ? 4 : 8;
    const size_t need = sizeof(unsigned) * (size_t)n * words;
    unsigned* place = dw > 8 ? nullptr
                      : bits_room && bits_bytes >= need ? (unsigned*)bits_room
                      : sizeof(int) * (size_t)m >= need ? (unsigned*)w.row_of : nullptr;
    p.bits = place;
    if (!place) return launch_pulls<SearchPlaces>(p, m, st);
    switch (words) {
        case 1: return launch_bits_and_pulls<1>(p, place, m, st);
        case 2: return launch_bits_and_pulls<2>(p, place, m, st);
        case 4: return launch_bits_and_pulls<4>(p, place, m, st);
        default: return launch_bits_and_pulls<8>(p, place, m, st);
    }
}

}  // namespace ts
