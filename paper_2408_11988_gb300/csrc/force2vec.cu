// Sparse Force2Vec minibatch step (paper Sec. IV, "Distributed sparse
// embedding"), for the rows [r0, r0 + b) of a sparse embedding Z (n x d,
// exactly k stored entries per row, row i at [k*i, k*i+k)):
//
//   U_i = z_i + lr * (sum over the neighbours j of vertex i in A of
//           (1 - sigmoid(z_i . z_j)) z_j  -  sum over i's s negative samples j
//           of sigmoid(z_i . z_j) z_j),
//
// then the k entries of U_i of largest magnitude (ties: smaller column) in
// ascending column order, by a radix select on the magnitude's bit pattern.
// A column met several times (a neighbour that is also a sample, a sample
// drawn twice) is as many terms: the product W * Z of the weight matrix with
// Z, row by row, without forming W.
//
// One kernel does all of it for a row: its warp holds z_i and the sum densely
// in shared memory and, for each term, loads z_j once, takes the dot product,
// the weight, and adds w * z_j (columns of one row of Z are distinct: plain
// adds).  The path is bound by the latency of those gathers (a minibatch of
// 4096 rows and 5 samples reads 150,000 rows of 208 bytes, from L2 mostly), so
// four terms are in flight per warp and the next four load meanwhile.  A row
// of more than one chunk of terms is queued chunk by chunk for a second kernel,
// where any warp takes a chunk and leaves its sums in the chunk's own place.  The
// warp that finishes the last of 16 chunks adds their places in the row's order,
// and the one that finishes the last such group adds the groups: no sum depends
// on what ran first, and a step repeats bit for bit.  The new rows replace the
// batch rows of Z at the end (k_f2v_commit), after every row was computed from
// the old Z (synchronous SGD).
//
// As passes of their own (W's pattern, its weights, the row schedule and two
// passes of the general product with a packed copy of all of Z, the update: 24
// launches) a minibatch of 4096 rows, d = 128, took 364 us; now 104 us, of which
// the two kernels take 28 and 30 us.  (With the chunks' sums added into one place a
// row by float atomics, in any order, it was 103; with a block for every row of
// more than 32 terms 108, and 670 against 602 us for 65,536 rows.)
#include "common.cuh"
#include "kernels.h"
#include "queues.h"

namespace ts {

// Terms per chunk: a chunk is a serial chain of some 300 ns a term pair, and the
// batch is done when its longest one is (minibatch at 128 / 64 / 32 terms: 150 /
// 122 / 104 us).  Terms in flight: eight instead of four hide nothing more
// (114 us) and cost a block per SM.  More terms a chunk where d is large, so that
// the chunks' places (d floats each) stay within 32 bytes a term.
constexpr int F2V_CHUNK = 32;
constexpr int F2V_FLIGHT = 4;
static long long f2v_chunk(long long d) { return d <= 8 * F2V_CHUNK ? F2V_CHUNK : (d / 8 + 31) / 32 * 32; }
constexpr int F2V_GROUP = 16;  // chunks whose places one warp adds (8 / 16 / 32, b = 4096: 106 / 103 / 105 us)
constexpr unsigned F2V_EMPTY = 0x80000000u;  // -0.0: a column no term reached (x + -0.0 is x)

// Layout of the workspace for a batch of b rows with at most `terms` terms.
struct F2vWs {
    F2vCtl* ctl;
    long long* items;  // (row of the batch, chunk) of the queued rows, a row's chunks side by side
    int* done;         // at a group's first item: its chunks finished
    int* groups;       // per row: its groups finished
    float* sums;       // the items' places, d floats each
    int* Sc;
    float* Sv;
    long long item_cap;
};

static size_t f2v_ws(char* base, long long d, long long nnzA, long long b, long long s, long long k, F2vWs* out) {
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* p = base + off;
        off += (bytes + 255) & ~(size_t)255;
        return p;
    };
    // a queued row has more than a chunk of terms, and one chunk that may not be full
    const long long terms = nnzA + b * s, chunk = f2v_chunk(d), rows = terms / (chunk + 1);
    F2vWs w;
    w.item_cap = terms / chunk + (rows < b ? rows : b) + 1;
    w.ctl = (F2vCtl*)take(sizeof(F2vCtl));
    w.items = (long long*)take(sizeof(long long) * (size_t)w.item_cap);
    w.done = (int*)take(sizeof(int) * (size_t)w.item_cap);
    w.groups = (int*)take(sizeof(int) * (size_t)b);
    w.sums = (float*)take(sizeof(float) * (size_t)(w.item_cap * d));
    w.Sc = (int*)take(sizeof(int) * (size_t)(b * k));
    w.Sv = (float*)take(sizeof(float) * (size_t)(b * k));
    if (out) *out = w;
    return off;
}

size_t f2v_bytes(long long d, long long nnzA, long long b, long long s, long long k) {
    return f2v_ws(nullptr, d, nnzA, b, s, k, nullptr);
}

struct F2vParams {
    const long long* Ap;
    const int* Ai;
    long long nnzA;
    int n;
    long long r0, b;
    const int* neg;
    int s;
    const long long* Zp;
    const int* Zc;
    const float* Zv;
    int k, d, dpad;
    float lr;
    float* U_out;
    F2vWs ws;
    int chunk;  // f2v_chunk(d)
};

// Row i of Z scattered into the dense shared row g (cleared before).
__device__ __forceinline__ void f2v_scatter(const F2vParams& p, long long i, float* g) {
    for (int t = lane_id(); t < p.k; t += 32) {
        const int c = __ldg(p.Zc + i * p.k + t);
        if ((unsigned)c < (unsigned)p.d) g[c] = __ldg(p.Zv + i * p.k + t);
        else atomicOr(&p.ws.ctl->err, ERR_B_COL);
    }
}

// Up to KL entries per lane of row j of Z (column -1: none, as for j < 0 and
// for a column outside [0, d), which is reported through `bad`).
template <int KL>
struct ZRow {
    int c[KL];
    float v[KL];
    __device__ __forceinline__ void load(const F2vParams& p, int j) {
#pragma unroll
        for (int q = 0; q < KL; ++q) {
            const int t = lane_id() + 32 * q;
            c[q] = -1;
            v[q] = 0.0f;
            if (j >= 0 && t < p.k) {
                c[q] = __ldg(p.Zc + (long long)j * p.k + t);
                v[q] = __ldg(p.Zv + (long long)j * p.k + t);
            }
        }
    }
    __device__ __forceinline__ float dot(const F2vParams& p, const float* z, bool held, bool& bad) {
        float x = 0.0f;
#pragma unroll
        for (int q = 0; q < KL; ++q) {
            if ((unsigned)c[q] < (unsigned)p.d) {
                x = fmaf(z[c[q]], v[q], x);
            } else {
                bad |= held && lane_id() + 32 * q < p.k;
                c[q] = -1;
            }
        }
        return x;
    }
    __device__ __forceinline__ void add(float w, float* g) const {
#pragma unroll
        for (int q = 0; q < KL; ++q)
            if (c[q] >= 0) g[c[q]] += w * v[q];
    }
};

__device__ __forceinline__ float f2v_weight(float x, bool sample) {
    const float sg = 1.0f / (1.0f + expf(-x));
    return sample ? -sg : 1.0f - sg;
}

// m <= 32 terms of a row: `na` neighbours from entry e0 of A on, then samples from
// neg[s0 + na] on.  KL entries of a row of Z per lane (KL = 0: more than 64 entries
// a row, read twice).
template <int KL>
__device__ __forceinline__ void f2v_terms(const F2vParams& p, long long e0, int na, long long s0, int m,
                                          const float* z, float* g) {
    constexpr int U = KL == 2 ? F2V_FLIGHT / 2 : F2V_FLIGHT;  // terms in flight
    const int lane = lane_id();
    bool bad_a = false, bad_z = false;
    int j = -1;
    if (lane < m) {
        j = lane < na ? __ldg(p.Ai + e0 + lane) : __ldg(p.neg + s0 + lane);
        if ((unsigned)j >= (unsigned)p.n) {
            bad_a = true;
            j = -1;
        }
    }
    const unsigned sample = __ballot_sync(FULL, lane >= na);
    if constexpr (KL > 0) {
        ZRow<KL> cur[U], nxt[U];
#pragma unroll
        for (int u = 0; u < U; ++u) cur[u].load(p, __shfl_sync(FULL, j, u));
        for (int q = 0; q < m; q += U) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int jn = __shfl_sync(FULL, j, (q + U + u) & 31);
                nxt[u].load(p, q + U + u < m ? jn : -1);
            }
            float w[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                w[u] = cur[u].dot(p, z, __shfl_sync(FULL, j, (q + u) & 31) >= 0 && q + u < m, bad_z);
#pragma unroll
            for (int u = 0; u < U; ++u) w[u] = f2v_weight(warp_sum(w[u]), (sample >> ((q + u) & 31)) & 1u);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                cur[u].add(w[u], g);  // a term past the end holds no entries
                __syncwarp();         // the next row's columns may be this one's
                cur[u] = nxt[u];
            }
        }
    } else {
        for (int q = 0; q < m; ++q) {
            const int jq = __shfl_sync(FULL, j, q);
            if (jq < 0) continue;
            const int* zc = p.Zc + (long long)jq * p.k;
            const float* zv = p.Zv + (long long)jq * p.k;
            float x = 0.0f;
            for (int e = lane; e < p.k; e += 32) {
                const int c = __ldg(zc + e);
                if ((unsigned)c < (unsigned)p.d) x = fmaf(z[c], __ldg(zv + e), x);
                else bad_z = true;
            }
            const float w = f2v_weight(warp_sum(x), (sample >> q) & 1u);
            for (int e = lane; e < p.k; e += 32) {
                const int c = __ldg(zc + e);
                if ((unsigned)c < (unsigned)p.d) g[c] += w * __ldg(zv + e);
            }
            __syncwarp();
        }
    }
    if (bad_a) atomicOr(&p.ws.ctl->err, ERR_A_COL);
    if (bad_z) atomicOr(&p.ws.ctl->err, ERR_B_COL);
}

// Row r from z (its old row) and its sum g: u = z + lr * g in place of z, the
// optional dense copy, then the k entries of largest magnitude to the staging
// rows.  Columns c, c + 32, ... belong to lane c % 32.
__device__ __forceinline__ void f2v_finish(const F2vParams& p, long long r, float* u, const float* g) {
    const int lane = lane_id(), mb = p.dpad >> 5;
    const unsigned lt = lanemask_lt();
    for (int c = lane; c < p.d; c += 32) {
        const float s = g[c];
        if (__float_as_uint(s) != F2V_EMPTY) u[c] += p.lr * s;
        if (p.U_out) p.U_out[r * p.d + c] = u[c];
    }
    __syncwarp();
    auto key_of = [&](int m) {  // 0 past the row's end: never above a candidate
        const int c = 32 * m + lane;
        return c < p.d ? __float_as_uint(u[c]) & 0x7FFFFFFFu : 0u;
    };
    // T = the k-th largest magnitude key (bits of |u|; monotone in |u|)
    unsigned T = 0u;
    for (int bit = 30; bit >= 0; --bit) {
        const unsigned cand = T | (1u << bit);
        int cnt = 0;
        for (int m = 0; m < mb; ++m) cnt += __popc(__ballot_sync(FULL, key_of(m) >= cand));
        if (cnt >= p.k) T = cand;
    }
    int gt = 0;
    for (int m = 0; m < mb; ++m) gt += __popc(__ballot_sync(FULL, key_of(m) > T));
    const int need = p.k - gt;  // keys equal to T to keep, smallest columns first
    int eq_before = 0, out = 0;
    for (int m = 0; m < mb; ++m) {
        const int c = 32 * m + lane;
        const unsigned key = key_of(m);
        const bool valid = c < p.d;
        const bool eq = valid && key == T;
        const unsigned beq = __ballot_sync(FULL, eq);
        const bool keep = (valid && key > T) || (eq && eq_before + __popc(beq & lt) < need);
        const unsigned bk = __ballot_sync(FULL, keep);
        if (keep) {
            const int pos = out + __popc(bk & lt);
            if (pos < p.k) {
                p.ws.Sc[r * p.k + pos] = c;
                p.ws.Sv[r * p.k + pos] = u[c];
            }
        }
        eq_before += __popc(beq);
        out += __popc(bk);
    }
    __syncwarp();
}

// m places of d floats, `stride` floats apart, added in their order into out (a
// place of its own, or the first of them).  F2V_EMPTY is -0.0, which adds nothing
// to any number and stays -0.0 with itself.
__device__ __forceinline__ void f2v_add_places(const float* first, long long stride, long long m, int d, float* out) {
    for (int c0 = lane_id(); c0 < d; c0 += 128) {
        float v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = __uint_as_float(F2V_EMPTY);
#pragma unroll 4
        for (long long y = 0; y < m; ++y) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (c0 + 32 * q < d) v[q] += __ldcg(first + y * stride + c0 + 32 * q);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (c0 + 32 * q < d) out[c0 + 32 * q] = v[q];
    }
    __syncwarp();
}

// One more of `of` finished at *counter: whether it was the last, for the warp.
// What the warp wrote before is seen by the warp that finishes the last.
__device__ __forceinline__ bool f2v_last(int* counter, long long of) {
    __threadfence();
    __syncwarp();
    int before = 0;
    if (lane_id() == 0) before = atomicAdd(counter, 1);
    if (__shfl_sync(FULL, before, 0) != of - 1) return false;
    __threadfence();
    return true;
}

// The sums g of item x into its place, and where that was the last of its row's,
// the row's sum into g (true).  A function of its own, as f2v_finish: what they
// need is kept out of the registers of the loop over the terms.
__device__ __forceinline__ bool f2v_settle(const F2vParams& p, int per, long long x, float* g) {
    const long long item = p.ws.items[x], r = item_row(item), chunk = item_chunk(item);
    const long long a0 = clampll(__ldg(p.Ap + p.r0 + r), 0, p.nnzA), a1 = clampll(__ldg(p.Ap + p.r0 + r + 1), a0, p.nnzA);
    const long long nch = (a1 - a0 + p.s + per - 1) / per;
    const long long in_group = chunk & (F2V_GROUP - 1), left = nch - (chunk - in_group);
    const long long m = left < F2V_GROUP ? left : F2V_GROUP;
    float* mine = p.ws.sums + x * p.d;
    float* group = mine - in_group * p.d;
    for (int c = lane_id(); c < p.d; c += 32) mine[c] = g[c];
    if (!f2v_last(p.ws.done + (x - in_group), m)) return false;
    if (nch <= F2V_GROUP) {
        f2v_add_places(group, p.d, m, p.d, g);
        return true;
    }
    f2v_add_places(group, p.d, m, p.d, group);
    const long long ng = (nch + F2V_GROUP - 1) / F2V_GROUP;
    if (!f2v_last(p.ws.groups + r, ng)) return false;
    f2v_add_places(p.ws.sums + (x - chunk) * p.d, (long long)F2V_GROUP * p.d, ng, p.d, g);
    return true;
}

// Blocks per SM of the kernel below.  The path waits for gathers, so as many
// warps as the registers allow: 48 of them hardly spill (KL > 0), and KL = 0, which
// has one term in flight, is faster with 32 and some spilled (65,536 rows, d = 256,
// k = 80: 1190 us, with 40 1260).  ONE = false: wide rows, bound by shared memory.
constexpr int f2v_blocks(int KL, bool LONG, bool ONE) {
    return !ONE ? (KL == 0 ? 5 : 4) : KL > 0 ? 5 : 8;
}

// LONG = false: a warp per batch row; rows of more than a chunk of terms are
// queued.  LONG = true: a warp per queued chunk.  Shared memory: z and g, dpad
// floats each, per warp.  The check that Z holds exactly k entries per row
// (Zp[i] = k * i) is spread over the first kernel's threads.
// Blocks per SM: left alone the compiler takes up to 64 registers, four blocks.
template <int KL, bool LONG, bool ONE>
__global__ void __launch_bounds__(256, f2v_blocks(KL, LONG, ONE)) k_f2v_rows(F2vParams p) {
    extern __shared__ __align__(16) float fsm[];
    const int nw = blockDim.x >> 5, warp = warp_id(), lane = lane_id();
    float* z = fsm + (size_t)warp * 2 * p.dpad;
    float* g = z + p.dpad;
    const long long gw = (long long)blockIdx.x * nw + warp, gws = (long long)gridDim.x * nw;
    F2vCtl* ctl = p.ws.ctl;
    const int per = ONE ? F2V_CHUNK : p.chunk;  // terms of a chunk
    if (!LONG) {
        for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i <= p.n;
             i += (long long)gridDim.x * blockDim.x)
            if (__ldg(p.Zp + i) != (long long)p.k * i) atomicOr(&ctl->err, ERR_CAPACITY);
    }
    const long long units = LONG ? min((long long)__ldcg(&ctl->items), p.ws.item_cap) : p.b;
    for (long long x = gw; x < units; x += gws) {
        const long long item = LONG ? p.ws.items[x] : 0;
        if (LONG && item < 0) continue;  // of a row that found no room
        const long long r = LONG ? item_row(item) : x, i = p.r0 + r;
        const long long a0 = clampll(__ldg(p.Ap + i), 0, p.nnzA), a1 = clampll(__ldg(p.Ap + i + 1), a0, p.nnzA);
        const long long len = a1 - a0, terms = len + p.s;
        if (!LONG && terms > per) {  // queued
            const long long nch = (terms + per - 1) / per;
            long long at = 0;
            if (lane == 0) {
                at = (long long)atomicAdd(&ctl->items, (unsigned long long)nch);
                p.ws.groups[r] = 0;
                // (row pointers that ascend always leave room)
                if (at + nch > p.ws.item_cap) atomicOr(&ctl->err, ERR_CAPACITY);
            }
            at = shfl64(at, 0);
            for (long long c = lane; c < nch && at + c < p.ws.item_cap; c += 32) {
                p.ws.items[at + c] = at + nch <= p.ws.item_cap ? queue_item(r, c) : -1;
                p.ws.done[at + c] = 0;
            }
            continue;
        }
        for (int c = lane; c < p.dpad; c += 32) {
            z[c] = 0.0f;
            g[c] = __uint_as_float(F2V_EMPTY);
        }
        __syncwarp();
        f2v_scatter(p, i, z);
        __syncwarp();
        const long long t0 = LONG ? item_chunk(item) * per : 0, t1 = t0 + per < terms ? t0 + per : terms;
        for (long long t = t0; t < t1; t += 32) {
            const int m = (int)(t1 - t < 32 ? t1 - t : 32);
            f2v_terms<KL>(p, a0 + t, (int)(len - t < 0 ? 0 : len - t < m ? len - t : m), r * p.s + t - len, m, z, g);
            if (ONE) break;
        }
        __syncwarp();
        if (LONG && !f2v_settle(p, per, x, g)) continue;
        f2v_finish(p, r, z, g);
    }
}

// The staged rows into Z, unless a check failed: then some of them may not have
// been finished, and Z stays as it was.
__global__ void __launch_bounds__(256) k_f2v_commit(long long r0, long long b, int k, const int* __restrict__ Sc,
                                                    const float* __restrict__ Sv, int* Zc, float* Zv,
                                                    const F2vCtl* ctl) {
    const bool whole = __ldg(&ctl->err) == 0;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < b * k;
         t += (long long)gridDim.x * blockDim.x) {
        const int c = Sc[t];  // beside the load of the error bits
        const float v = Sv[t];
        if (!whole) return;
        Zc[r0 * k + t] = c;
        Zv[r0 * k + t] = v;
    }
}

template <int KL, bool ONE>
static cudaError_t launch_rows(const F2vParams& p, int sms, cudaStream_t st) {
    const void* rows = (const void*)k_f2v_rows<KL, false, ONE>;
    const void* chunks = (const void*)k_f2v_rows<KL, true, ONE>;
    const size_t per_warp = 2 * sizeof(float) * (size_t)p.dpad;  // at most 32 KB
    int warps = 8;
    while (warps > 1 && warps * per_warp > 100 * 1024) warps /= 2;
    const size_t smem = warps * per_warp;
    cudaError_t e;
    for (const void* k : {rows, chunks})
        if (smem > 48 * 1024 && (e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)))
            return e;
    F2vParams q = p;
    void* args[] = {&q};
    const long long need = (p.b + warps - 1) / warps;
    const int full = persistent_grid(rows, 32 * warps, smem, sms);
    count_launch();
    if ((e = cudaLaunchKernel(rows, dim3((unsigned)(need < full ? need : full)), dim3(32 * warps), args, smem, st)))
        return e;
    count_launch();
    const long long most = (p.ws.item_cap + warps - 1) / warps;
    const int cgrid = persistent_grid(chunks, 32 * warps, smem, sms);
    return cudaLaunchKernel(chunks, dim3((unsigned)(most < cgrid ? most : cgrid)), dim3(32 * warps), args, smem, st);
}

cudaError_t launch_f2v_step(const DevCsr& A, const DevCsr& Z, int k, long long r0, long long b, const int* neg, int s,
                            float lr, float* U_out, int sms, void* ws, cudaStream_t st) {
    cudaError_t e;
    F2vParams p = {};
    p.Ap = A.rowptr;
    p.Ai = A.col;
    p.nnzA = A.nnz;
    p.n = (int)A.nrows;
    p.r0 = r0;
    p.b = b;
    p.neg = neg;
    p.s = s;
    p.Zp = Z.rowptr;
    p.Zc = Z.col;
    p.Zv = Z.val;
    p.k = k;
    p.d = (int)Z.ncols;
    p.dpad = (p.d + 31) & ~31;
    p.lr = lr;
    p.U_out = U_out;
    f2v_ws((char*)ws, p.d, A.nnz, b, s, k, &p.ws);
    p.chunk = (int)f2v_chunk(p.d);
    if ((e = cudaMemsetAsync(p.ws.ctl, 0, sizeof(F2vCtl), st))) return e;
    auto run = [&](auto one) {
        constexpr bool ONE = decltype(one)::value;
        return k <= 32 ? launch_rows<1, ONE>(p, sms, st)
             : k <= 64 ? launch_rows<2, ONE>(p, sms, st) : launch_rows<0, ONE>(p, sms, st);
    };
    e = p.chunk == F2V_CHUNK ? run(std::true_type{}) : run(std::false_type{});
    if (e) return e;
    long long blocks = (b * k + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    count_launch();
    k_f2v_commit<<<(unsigned)blocks, 256, 0, st>>>(r0, b, k, p.ws.Sc, p.ws.Sv, const_cast<int*>(Z.col),
                                                   const_cast<float*>(Z.val), p.ws.ctl);
    return cudaGetLastError();
}

}  // namespace ts
