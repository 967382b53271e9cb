// Rows of a CSR pattern as bitmaps (d <= 256), shared by the multi-source BFS
// (frontiers) and the repeatable backward (rows of C).
#pragma once

#include "common.cuh"

namespace ts {

// The warp's 32 rows from row `base` of a pattern of n rows and d columns into
// bits[32 * DWP] (shared memory, row r at r * DWP; DWP * 32 >= d); start: 33
// ints of shared memory.  The rows' entries follow each other: 128 a step, four
// per lane with one 16-byte load, the row of a lane's first entry by a search
// of the row starts, and the bits of neighbouring entries of one word gathered
// before one OR into the words.  Returns whether this lane met a column
// outside [0, d); all lanes are converged and see the words at the end.  (A
// thread per row took 127 us for 57 million entries in 2^20 rows, its lines
// thrown out of L1 before they were used up; this way 80 us.)
template <int DWP>
__device__ __forceinline__ bool rows_to_bits(long long n, int d, const long long* __restrict__ Fp, long long nnzF,
                                             const int* __restrict__ Fi, long long base, unsigned* bits, int* start) {
    const int lane = lane_id();
    const long long v = base + lane;
#pragma unroll
    for (int m = 0; m < DWP; ++m) bits[32 * m + lane] = 0u;
    const long long s = clampll(__ldg(Fp + (v < n ? v : n)), 0, nnzF);
    const long long e0 = shfl64(s, 0);
    const long long e1 = clampll(__ldg(Fp + (base + 32 < n ? base + 32 : n)), e0, nnzF);
    const int total = (int)(e1 - e0 < (1LL << 30) ? e1 - e0 : 1LL << 30);  // at most 32 d in a well-formed pattern
    start[lane] = (int)clampll(s - e0, 0, total);
    if (lane == 0) start[32] = total;
    __syncwarp();
    const int* f = Fi + e0;
    const int lead = (int)((reinterpret_cast<uintptr_t>(f) >> 2) & 3);  // entries of the first 16 bytes before f
    bool bad = false;
    for (int i0 = -lead; i0 < total; i0 += 128) {
        const int i = i0 + 4 * lane;
        if (i >= total) continue;
        int c[4];
        if (i >= 0 && i + 4 <= total) {
            const int4 x = __ldg(reinterpret_cast<const int4*>(f + i));
            c[0] = x.x;
            c[1] = x.y;
            c[2] = x.z;
            c[3] = x.w;
        } else {
#pragma unroll
            for (int t = 0; t < 4; ++t) c[t] = i + t >= 0 && i + t < total ? __ldg(f + i + t) : 0;
        }
        int r = 0;  // last row starting at or before the lane's first entry
        const int at = i > 0 ? i : 0;
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1)
            if (start[r + o] <= at) r += o;
        int word = -1;
        unsigned x = 0u;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            if (i + t < 0 || i + t >= total) continue;
            while (r < 31 && i + t >= start[r + 1]) ++r;
            if ((unsigned)c[t] >= (unsigned)d) {
                bad = true;
                continue;
            }
            const int w = r * DWP + (c[t] >> 5);
            if (w != word) {
                if (x) atomicOr(bits + word, x);
                word = w;
                x = 0u;
            }
            x |= 1u << (c[t] & 31);
        }
        if (x) atomicOr(bits + word, x);
    }
    __syncwarp();
    return bad;
}

// Row of DWP words, read whole.
template <int DWP>
__device__ __forceinline__ void load_bit_row(const unsigned* __restrict__ fb, long long row, unsigned w[DWP]) {
    const unsigned* r = fb + row * DWP;
    if constexpr (DWP >= 4) {
#pragma unroll
        for (int m = 0; m < DWP; m += 4) {
            const uint4 x = __ldg(reinterpret_cast<const uint4*>(r + m));
            w[m] = x.x;
            w[m + 1] = x.y;
            w[m + 2] = x.z;
            w[m + 3] = x.w;
        }
    } else if constexpr (DWP == 2) {
        const uint2 x = __ldg(reinterpret_cast<const uint2*>(r));
        w[0] = x.x;
        w[1] = x.y;
    } else {
        w[0] = __ldg(r);
    }
}

}  // namespace ts
