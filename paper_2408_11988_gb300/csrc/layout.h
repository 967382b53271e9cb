// Workspace header and device-check flags shared by the kernels and the host
// side of the C ABI (plain C++, no device code).
#pragma once

namespace ts {

// Row classes by products (flops): class 0 = no products; class
// 1 + 8*lg + sub (lg = floor(log2 f), sub = the three bits of f below its
// leading one) holds an eighth of an octave, so the rows of one class differ
// in flops by less than 12.5 % and rows taken side by side in lockstep have
// nearly equal lengths.
constexpr int CLASS_SUB_BITS = 3;
constexpr int NUM_CLASSES = 1 + 48 * (1 << CLASS_SUB_BITS);

// Host copy of the device-side class function (common.cuh).
inline int flops_class_host(long long f) {
    if (f <= 0) return 0;
    const int lg = 63 - __builtin_clzll((unsigned long long)f);
    const int sub = lg >= CLASS_SUB_BITS ? (int)((f >> (lg - CLASS_SUB_BITS)) & ((1 << CLASS_SUB_BITS) - 1))
                                         : (int)((f << (CLASS_SUB_BITS - lg)) & ((1 << CLASS_SUB_BITS) - 1));
    const int c = 1 + (lg << CLASS_SUB_BITS) + sub;
    return c < NUM_CLASSES ? c : NUM_CLASSES - 1;
}

// First class whose rows all have at least min_flops products (rounded up
// to a class boundary).
inline int class_at_least(long long min_flops) {
    return min_flops <= 1 ? 1 : flops_class_host(min_flops - 1) + 1;
}

// error bits recorded in the workspace header by device-side checks
constexpr unsigned long long ERR_A_COL = 1ull;     // column of A outside [0, n)
constexpr unsigned long long ERR_B_COL = 2ull;     // column of B outside [0, d)
constexpr unsigned long long ERR_C_ROW = 4ull;     // row of C longer/shorter than its rowptr
constexpr unsigned long long ERR_HASH_FULL = 8ull; // row too wide for its hash table or its ranked values
constexpr unsigned long long ERR_CAPACITY = 16ull; // output capacity exceeded

// Rows of A with more than SPLIT_ENTRIES entries are cut into work items of
// SPLIT_ENTRIES entries that any thread block can take; at most
// MAX_SPLIT_ROWS rows per product are cut (the rest run whole).
constexpr int SPLIT_ENTRIES = 1024;
constexpr int MAX_SPLIT_ROWS = 8192;

// Queue items of rows cut into chunks, for queues whose chunks are so short that
// 24 bits do not number those of the longest row (2^31 - 1 entries): the row in
// the upper half of the word, the chunk in the lower.
#ifdef __CUDACC__
#define TS_BOTH __host__ __device__
#else
#define TS_BOTH
#endif
TS_BOTH inline long long queue_item(long long row, long long chunk) { return (row << 32) | chunk; }
TS_BOTH inline long long item_row(long long item) { return item >> 32; }
TS_BOTH inline long long item_chunk(long long item) { return item & 0xFFFFFFFFll; }

// Tiles of BAT_TILE rows of a batch's instances, for the scan of C's row counts:
// instance b (its first 32-row chunk chunk_off(b), instances in order) owns the
// tiles bat_first_tile(b) + 0, 1, ..., at least one; tiles of different instances
// never meet (128 chunks a tile, one spare tile each).
constexpr int BAT_TILE = 4096;
TS_BOTH inline long long bat_first_tile(long long chunk_off, int b) { return (chunk_off >> 7) + b; }
// The instance of tile t >= bat_first_tile(0): the last whose first tile is at or before it.
template <class ChunkOff>
TS_BOTH inline int bat_inst_of_tile(ChunkOff chunk_off, int count, long long t) {
    int lo = 0, hi = count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (bat_first_tile(chunk_off(mid), mid) <= t) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}
// Tiles up to the end of the last instance, from bat_first_tile(0) on.
inline long long bat_tile_span(long long first_chunk_off, long long last_chunk_off, int count, long long last_rows) {
    const long long last = last_rows > BAT_TILE ? (last_rows + BAT_TILE - 1) / BAT_TILE : 1;
    return bat_first_tile(last_chunk_off, count - 1) + last - bat_first_tile(first_chunk_off, 0);
}

// Workspace header (offset 0 of every workspace).
struct WsHeader {
    unsigned long long heavy_ctr;     // next heavy row (dynamic CTA scheduling)
    unsigned long long item_ctr;      // next split-row work item
    unsigned long long err;           // ERR_* bits
    long long total;                  // multi-source BFS: entries of the next frontier (read with err)
    long long hist[NUM_CLASSES];      // rows per flops class; once the row order is written, rows in the classes above each
    long long cursor[NUM_CLASSES];    // scatter cursors per class
    long long scratch[8];             // [0] flops items, [1] split rows, [2] split items, [3] blocks of the row order done,
                                      // [4], [5] the repeatable dB's queue
};

}  // namespace ts
