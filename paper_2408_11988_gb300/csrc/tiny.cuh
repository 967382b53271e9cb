// A row of at most 32 products held one per lane: sorted by column, equal
// columns summed, written with one store (numeric_tiny.cu, numeric_rank.cu).
#pragma once

#include "common.cuh"
#include "numeric.cuh"

namespace ts {

// Ascending bitonic sort of one (key, value) pair per lane across the warp.
__device__ __forceinline__ void warp_sort_kv(int& key, float& val) {
    const int lane = lane_id();
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const int pk = __shfl_xor_sync(FULL, key, j);
            const float pv = __shfl_xor_sync(FULL, val, j);
            const bool keep_min = ((lane & j) == 0) == ((lane & k) == 0);
            if (keep_min ? pk < key : pk > key) {
                key = pk;
                val = pv;
            }
        }
    }
}

// The row's products, sorted by column (key; 0x7FFFFFFF on lanes without
// one), summed per column into the first lane of each run and written to
// C[out, out_end) in ascending column order; dup = whether equal columns can
// occur (more than one row of B), runs = their longest possible length.
__device__ __forceinline__ void tiny_emit(const NumParams& p, int key, float val, bool dup, int runs, long long out,
                                          long long out_end, unsigned long long* err) {
    const int lane = lane_id();
    float sum = val;
    if (dup) {
        for (int o = 1; o < runs; o <<= 1) {  // warp-uniform bound
            const float t = __shfl_down_sync(FULL, sum, o);
            const int ko = __shfl_down_sync(FULL, key, o);
            if (lane + o < 32 && ko == key) sum += t;
        }
    }
    const int prev = __shfl_up_sync(FULL, key, 1);
    const bool head = key != 0x7FFFFFFF && (!dup || lane == 0 || prev != key);
    const unsigned hb = __ballot_sync(FULL, head);
    if (head) {
        const long long pos = out + __popc(hb & lanemask_lt());
        if (pos < out_end) {
            p.Ci[pos] = key;
            if (p.Cx) p.Cx[pos] = sum;
        }
    }
    if (lane == 0 && out + __popc(hb) != out_end) atomicOr(err, ERR_C_ROW);
}

}  // namespace ts
