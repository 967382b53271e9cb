// Numbering of work items, shared by kernels and launchers (plain C++, so that it
// can be tested on the host).
#pragma once

#ifdef __CUDACC__
#define TS_BOTH __host__ __device__
#else
#define TS_BOTH
#endif

namespace ts {

// Queue items of rows cut into chunks, for queues whose chunks are so short that
// 24 bits do not number those of the longest row (2^31 - 1 entries): the row in
// the upper half of the word, the chunk in the lower.
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

}  // namespace ts
