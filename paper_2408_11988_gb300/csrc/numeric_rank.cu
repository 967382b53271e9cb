// Numeric pass for many columns (4096 < d <= RANK_MAX_D, where a dense
// accumulator per warp no longer fits; Sec. III-C turns to hashing there).
// A row's columns are ranked instead of hashed: one walk over its products
// sets a bit per column, the running popcounts of the bitmap's words then
// give every column its place in the row of C, and a second walk (over rows of
// B that the first left in L1 and L2) adds each product into the row's values
// at its place.  The values lie in column order and without gaps, so the
// read-out is a coalesced copy beside the columns recovered from the bitmap,
// and nothing is probed, looked up again or cleared beyond the row's own
// entries.  Rows of at most 32 products are sorted in registers.
//
// Bound by instruction issue and the latency of the gathers; shared memory per
// warp (bitmap, its running counts, RANK_WARP values: 5.6 KB at d = 8192, 9.2
// KB with a hash table of 1024 slots) sets how many warps hide it.  Rows above
// RANK_WARP products take a block of eight warps, and above RANK_BIG one of 32
// in a kernel of its own ahead (the hub of a scale-16 graph in eight warps was
// the whole pass); a row with more columns than the block's values goes in
// windows of ranks.
// 65521 rows, d = 8192, 16.8 million products: hash 635 us, this 190 us, beside
// which the kernel for the largest rows runs (110 us on its own).
#include "common.cuh"
#include "kernels.h"
#include "numeric.cuh"
#include "tiny.cuh"
#include "wide.cuh"

namespace ts {

constexpr int RANK_WARP = 1024;
constexpr int RANK_BIG = 32768;  // 16384: 425 us for the whole forward, 32768: 410, 65536: 419

struct RankMark {
    const int* __restrict__ Bi;
    unsigned* bits;
    int d;
    bool bad;
    __device__ __forceinline__ void mark(int c) {
        if ((unsigned)c < (unsigned)d) atomicOr(bits + (c >> 5), 1u << (c & 31));
        else bad = true;
    }
    __device__ __forceinline__ void step4(const long long* j, const float*, const int*) {
        int c[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) c[u] = __ldg(Bi + j[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) mark(c[u]);
    }
    __device__ __forceinline__ void step1(long long j, float, int, bool ok) {
        if (ok) mark(__ldg(Bi + j));
    }
};

// Ranks [base, base + cap) of the row into vals.
struct RankAdd {
    const int* __restrict__ Bi;
    const float* __restrict__ Bx;
    const unsigned* bits;
    const unsigned short* pre;
    float* vals;
    int d, base, cap;
    __device__ __forceinline__ void add(int c, float v) const {
        if ((unsigned)c >= (unsigned)d) return;
        const int r = pre[c >> 5] + __popc(bits[c >> 5] & ((1u << (c & 31)) - 1u)) - base;
        if ((unsigned)r < (unsigned)cap) atomicAdd(vals + r, v);
    }
    __device__ __forceinline__ void step4(const long long* j, const float* a, const int*) {
        int c[4];
        float b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            c[u] = __ldg(Bi + j[u]);
            b[u] = __ldg(Bx + j[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) add(c[u], a[u] * b[u]);
    }
    __device__ __forceinline__ void step1(long long j, float a, int, bool ok) {
        if (ok) add(__ldg(Bi + j), a * __ldg(Bx + j));
    }
};

// pre[w] = bits set in the words before w; returns all of them.  One warp.
__device__ __forceinline__ int rank_prefix(const unsigned* bits, unsigned short* pre, int dw) {
    const int lane = lane_id();
    int run = 0;
    for (int x = 0; x < dw; x += 32) {
        const int c = x + lane < dw ? __popc(bits[x + lane]) : 0;
        const int incl = warp_incl_scan(c);
        if (x + lane < dw) pre[x + lane] = (unsigned short)(run + incl - c);
        run += __shfl_sync(FULL, incl, 31);
    }
    return run;
}

// Column of rank j: the last word with at most j bits before it, and the bit
// in it.
__device__ __forceinline__ int rank_column(const unsigned* bits, const unsigned short* pre, int top, int dw, int j) {
    int w = 0;
    for (int st = top; st >= 1; st >>= 1)
        if (w + st < dw && pre[w + st] <= j) w += st;
    return 32 * w + select_bit(bits[w], j - pre[w]);
}

struct RankParams {
    NumParams n;
    int dw, top;         // bitmap words; the largest power of two below dw
    int big_class;       // rows of this class and above run in the kernel of 32 warps
    int values;          // values of a whole block
};

// One row in the warp's own part of shared memory, driven by pipelined_rows.
template <bool VALUES>
struct RankRow {
    const RankParams& p;
    unsigned* bits;
    unsigned short* pre;
    float* vals;
    long long out, out_end;
    bool bad, tiny;
    int key;
    float val;
    template <class Visit>
    __device__ __forceinline__ void walk(long long a0, long long a1, const Chunk& ch0, Visit& vis) {
        const NumParams& n = p.n;
        expand_loaded(ch0, vis);
        for (long long e0 = a0 + 32; e0 < a1; e0 += 32)
            expand_chunk(e0, (int)(a1 - e0 < 32 ? a1 - e0 : 32), n.Ai, VALUES ? n.Ax : nullptr, n.nB,
                         SegWhole{n.Bp, n.nnzB, n.d}, vis, &n.hdr->err);
    }
    // a row of at most 32 products, one per lane
    __device__ __forceinline__ void place(long long a0, long long a1, const Chunk& ch0) {
        const NumParams& n = p.n;
        const int lane = lane_id();
        key = 0x7FFFFFFF;
        val = 0.0f;
        int base = 0;
        for (long long e0 = a0; e0 < a1 && base < 32; e0 += 32) {
            const Chunk ch = e0 == a0 ? ch0
                                      : load_chunk(e0, (int)(a1 - e0 < 32 ? a1 - e0 : 32), n.Ai, VALUES ? n.Ax : nullptr,
                                                   n.nB, SegWhole{n.Bp, n.nnzB, n.d}, &n.hdr->err);
            const int incl = warp_incl_scan(ch.len), excl = incl - ch.len;
            const int tot = __shfl_sync(FULL, incl, 31);
            const int pj = lane - base;
            const int q = owner_lane(excl, pj < 0 ? 0 : pj);
            const long long s = shfl64(ch.start, q);
            const int eq = __shfl_sync(FULL, excl, q);
            const float aq = __shfl_sync(FULL, ch.a, q);
            if (pj >= 0 && pj < tot) {
                const int c = __ldg(n.Bi + s + (pj - eq));
                if ((unsigned)c < (unsigned)n.d) {
                    key = c;
                    if (VALUES) val = aq * __ldg(n.Bx + s + (pj - eq));
                } else {
                    bad = true;
                }
            }
            base += tot;
        }
    }
    __device__ __forceinline__ void gather(int row, long long a0, long long a1, const Chunk& ch0, int, int) {
        const NumParams& n = p.n;
        out = clampll(__ldg(n.Cp + row), 0, n.nnzC);
        out_end = clampll(__ldg(n.Cp + row + 1), out, n.nnzC);
        const long long f = __ldg(n.s.flops + row);
        tiny = f >= 0 && f <= 32;
        if (tiny) {
            place(a0, a1, ch0);
            return;
        }
        RankMark m{n.Bi, bits, n.d, false};
        walk(a0, a1, ch0, m);
        bad |= m.bad;
        __syncwarp();
        total = rank_prefix(bits, pre, p.dw);
        __syncwarp();
        if constexpr (VALUES) {
            RankAdd add{n.Bi, n.Bx, bits, pre, vals, n.d, 0, RANK_WARP};
            walk(a0, a1, ch0, add);
        }
    }
    int total;
    __device__ __forceinline__ void finish(int) {
        const NumParams& n = p.n;
        const int lane = lane_id();
        if (tiny) {
            warp_sort_kv(key, val);
            tiny_emit(n, key, val, true, 32, out, out_end, &n.hdr->err);
            return;
        }
        __syncwarp();
        // the row's class promises at most RANK_WARP products; the columns walked
        // here can still be more (patterns that changed after the symbolic pass,
        // row pointers of A that do not ascend), and the values end at RANK_WARP
        const int held = VALUES && total > RANK_WARP ? RANK_WARP : total;
        for (int j = lane; j < held; j += 32) {
            if (out + j < out_end) {
                n.Ci[out + j] = rank_column(bits, pre, p.top, p.dw, j);
                if (VALUES) n.Cx[out + j] = vals[j];
            }
            if (VALUES) vals[j] = 0.0f;
        }
        if (lane == 0 && held < total) atomicOr(&n.hdr->err, ERR_HASH_FULL);
        if (lane == 0 && out + total != out_end) atomicOr(&n.hdr->err, ERR_C_ROW);
        __syncwarp();
        for (int w = lane; w < p.dw; w += 32) bits[w] = 0u;
        __syncwarp();
    }
};

// One row by the whole block.
template <bool VALUES>
__device__ __forceinline__ void rank_row_block(const RankParams& p, int row, unsigned* bits, unsigned short* pre,
                                               float* vals, int* s_total, bool& bad) {
    const NumParams& n = p.n;
    const int tid = threadIdx.x, warp = warp_id(), nw = blockDim.x >> 5;
    const long long a0 = clampll(__ldg(n.Ap + row), 0, n.nnzA);
    const long long a1 = clampll(__ldg(n.Ap + row + 1), a0, n.nnzA);
    const long long out = clampll(__ldg(n.Cp + row), 0, n.nnzC);
    const long long out_end = clampll(__ldg(n.Cp + row + 1), out, n.nnzC);
    const SegWhole seg{n.Bp, n.nnzB, n.d};
    auto walk = [&](auto& vis) {
        for (long long e0 = a0 + 32LL * warp; e0 < a1; e0 += 32LL * nw)
            expand_chunk(e0, (int)(a1 - e0 < 32 ? a1 - e0 : 32), n.Ai, VALUES ? n.Ax : nullptr, n.nB, seg, vis,
                         &n.hdr->err);
    };
    RankMark m{n.Bi, bits, n.d, false};
    walk(m);
    bad |= m.bad;
    __syncthreads();
    if (warp == 0) {
        const int t = rank_prefix(bits, pre, p.dw);
        if (tid == 0) *s_total = t;
    }
    __syncthreads();
    const int total = *s_total;
    for (int base = 0; base < total; base += p.values) {
        if constexpr (VALUES) {
            RankAdd add{n.Bi, n.Bx, bits, pre, vals, n.d, base, p.values};
            walk(add);
            __syncthreads();
        }
        const int end = base + p.values < total ? base + p.values : total;
        for (int j = base + tid; j < end; j += blockDim.x) {
            if (out + j < out_end) {
                n.Ci[out + j] = rank_column(bits, pre, p.top, p.dw, j);
                if (VALUES) n.Cx[out + j] = vals[j - base];
            }
            if (VALUES) vals[j - base] = 0.0f;
        }
        __syncthreads();
    }
    if (tid == 0 && out + total != out_end) atomicOr(&n.hdr->err, ERR_C_ROW);
    for (int w = tid; w < p.dw; w += blockDim.x) bits[w] = 0u;
    __syncthreads();
}

// BIG: the rows of big_class and above, a block each.  Otherwise the other
// rows for a block (from a queue), then the light rows, a warp each.  Shared
// memory: a block's bitmap, running counts and values overlay its warps'.
template <bool VALUES, bool BIG, int THREADS>
__global__ void __launch_bounds__(THREADS) k_numeric_rank(RankParams p) {
    if (BIG) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ long long s_item;
    __shared__ int s_total;
    const NumParams& n = p.n;
    const int tid = threadIdx.x, nw = blockDim.x >> 5, warp = warp_id();
    const long long nbig = rows_from_class(n.hdr, p.big_class);
    const long long nheavy = rows_from_class(n.hdr, n.cta_class), nrows = rows_from_class(n.hdr, 1);
    bool bad = false;
    if (!BIG || blockIdx.x < nbig) {
        // one layout for the block's rows and for the warps': bitmaps first,
        // then values, then running counts
        const int teams = BIG ? 1 : nw;
        unsigned* bits = reinterpret_cast<unsigned*>(smem);
        float* vals = reinterpret_cast<float*>(bits + (size_t)teams * p.dw);
        unsigned short* pre = reinterpret_cast<unsigned short*>(vals + (VALUES ? p.values : 0));
        for (int i = tid; i < teams * p.dw; i += blockDim.x) bits[i] = 0u;
        if (VALUES)
            for (int i = tid; i < p.values; i += blockDim.x) vals[i] = 0.0f;
        __syncthreads();
        if (BIG) {
            for (long long h = blockIdx.x; h < nbig; h += gridDim.x)
                rank_row_block<VALUES>(p, n.perm[h], bits, pre, vals, &s_total, bad);
        } else {
            for (;;) {
                if (tid == 0) s_item = nbig + (long long)atomicAdd(&n.hdr->heavy_ctr, 1ull);
                __syncthreads();
                const long long h = s_item;
                __syncthreads();
                if (h >= nheavy) break;
                rank_row_block<VALUES>(p, n.perm[h], bits, pre, vals, &s_total, bad);
            }
            RankRow<VALUES> body{p, bits + (size_t)warp * p.dw, pre + (size_t)warp * p.dw, vals + warp * RANK_WARP};
            body.bad = false;
            pipelined_rows(n.perm, nheavy + (long long)blockIdx.x * nw + warp, nrows, (long long)gridDim.x * nw, n.Ap,
                           n.nnzA, n.Ai, VALUES ? n.Ax : nullptr, n.nB, SegWhole{n.Bp, n.nnzB, n.d}, &n.hdr->err, body);
            bad |= body.bad;
        }
    }
    if (bad) atomicOr(&n.hdr->err, ERR_B_COL);
    if (!BIG) asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <bool VALUES>
static cudaError_t launch_rank(RankParams p, int sms, cudaStream_t st) {
    cudaError_t e;
    constexpr int BT = 1024, WT = 256;
    // values of a block: its warps' together (WT), or as many as fit in 128 KB
    // (BT) -- every column of a row at the larger d but the largest
    const void* kb = (const void*)k_numeric_rank<VALUES, true, BT>;
    const void* kw = (const void*)k_numeric_rank<VALUES, false, WT>;
    RankParams big = p;
    big.values = p.n.d < 32768 ? (p.n.d + 3) / 4 * 4 : 32768;
    p.values = WT / 32 * RANK_WARP;
    const size_t sb = 6 * (size_t)p.dw + (VALUES ? 4 * (size_t)big.values : 0);
    const size_t sw = 6 * (size_t)p.dw * (WT / 32) + (VALUES ? 4 * (size_t)p.values : 0);
    if (sb > 220 * 1024 || sw > 220 * 1024) return cudaErrorInvalidValue;
    if ((e = cudaFuncSetAttribute(kb, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sb))) return e;
    if ((e = cudaFuncSetAttribute(kw, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sw))) return e;
    void* args[] = {&big};
    count_launch();
    if ((e = cudaLaunchKernel(kb, dim3(sms), dim3(BT), args, sb, st))) return e;
    // may start on the SMs the first leaves free (disjoint rows); waits for it
    // at its end
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(persistent_grid(kw, WT, sw, sms));
    lc.blockDim = dim3(WT);
    lc.dynamicSmemBytes = sw;
    lc.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    count_launch();
    return cudaLaunchKernelEx(&lc, k_numeric_rank<VALUES, false, WT>, p);
}

bool numeric_rank_fits(long long d) { return d > 4096 && d <= RANK_MAX_D; }

cudaError_t launch_numeric_rank(const DevCsr& A, const DevCsr& B, long long d, bool values, const Sched& s,
                                const LaunchCfg& cfg, const long long* Cp, int* Ci, float* Cx, long long nnzC,
                                cudaStream_t st) {
    cudaError_t e;
    if (A.nrows == 0) return cudaSuccess;
    if (!numeric_rank_fits(d)) return cudaErrorInvalidValue;
    if ((e = cudaMemsetAsync(&s.hdr->heavy_ctr, 0, 2 * sizeof(unsigned long long), st))) return e;
    RankParams p;
    p.n = numeric_params(A, B, d, 0, 1, nullptr, nullptr, s, cfg, Cp, Ci, Cx, nnzC);
    p.dw = (int)((d + 31) / 32);
    p.top = 1;
    while (2 * p.top < p.dw) p.top *= 2;
    const int warp_rows = flops_class_host(RANK_WARP + 1);  // rows of lower classes have at most RANK_WARP products
    if (p.n.cta_class > warp_rows) p.n.cta_class = warp_rows;
    p.big_class = class_at_least(RANK_BIG);
    if (p.big_class < p.n.cta_class) p.big_class = p.n.cta_class;
    p.values = 0;
    return values ? launch_rank<true>(p, cfg.sms, st) : launch_rank<false>(p, cfg.sms, st);
}

}  // namespace ts
