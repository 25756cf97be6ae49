// Launchers of the merge plan (k_merge.cu, merge.cu): B_R built one suffix
// length at a time, without sorting the suffixes.
#pragma once
#include <cuda_runtime.h>

#include "device.cuh"

namespace cxbwt {

constexpr uint32_t kMergeThreads = 256;
constexpr uint32_t kMergeBlocks = 5;      // CTAs per SM the registers are sized for
// Rows of a tile: kMergeThreads threads, each with 1, 2 or 4 chunks of 32 rows.
constexpr uint32_t merge_tile_rows(uint32_t k) { return kMergeThreads * 32u * k; }
constexpr uint32_t merge_tile_shift(uint32_t k) { return k == 1 ? 13u : k == 2 ? 14u : 15u; }
constexpr uint32_t kMergeMaxTile = merge_tile_rows(4);
constexpr uint32_t kMergePart = 1024;     // rows whose counts are kept from one step to the next
constexpr uint32_t kMergeMaxLen = 4096;   // reads the tables below are built for
constexpr uint32_t kMergeGroupTiles = 256;  // tiles whose counts are also summed together

// 32-bit words of one bit plane of `rows` rows: whole tiles, and the words
// that 16-byte loads of the last rows may touch.
constexpr uint64_t merge_plane_words(uint64_t rows) {
  return (rows + kMergeMaxTile - 1) / kMergeMaxTile * (kMergeMaxTile / 32) + 16;
}

// One step (suffix length j): B_j from B_{j-1} and the n suffixes of length j.
struct MergeArgs {
  ReadIndex R;
  uint32_t n;                  // reads
  uint32_t step;               // j
  uint64_t rows;               // rows of B_j: n * (j + 1)
  uint32_t n_tiles;
  const uint32_t* lo_in;       // planes of B_{j-1}
  const uint32_t* hi_in;
  uint32_t* lo_out;            // planes of B_j (not written by the last step)
  uint32_t* hi_out;
  const uint64_t* key_in;      // suffixes of length j in sorted order: (read << pshift) | row in B_j
  const uint32_t* bases_in;    // the bases before them, nearest in the low bits
  uint64_t* key_out;           // suffixes of length j + 1
  uint32_t* bases_out;
  const uint32_t* start_in;    // per tile of B_j: suffixes of length j in rows before it
  uint32_t* start_out;         // the same of B_{j+1}, whose tiles have 2^next_shift rows
  uint32_t next_shift;
  uint32_t pshift;
  const uint64_t* row_base;    // [4] first row of B_{j+1} of each class (suffixes starting with A, C, G, T)
  const uint32_t* item_base;   // [4] first suffix of length j + 1 of each class
  // Symbols C, G, T (as 64-bit counts; 4 words per tile) before each tile, and
  // (three 16-bit counts) before each part of kMergePart rows in its tile.
  uint32_t prev_shift;               // tiles of B_{j-1} have 2^prev_shift rows (at most B_j's)
  const uint64_t* before_in;
  const uint64_t* parts_in;
  uint64_t* before_out;
  uint64_t* parts_out;
  // Suffixes of length j by symbol (C, G, T: three 16-bit counts) in each tile
  // of B_j and (4 words) in each group of tiles; those of step j + 1, added
  // to; and those of step j + 2, zeroed.
  const unsigned long long* tiles_in;
  const uint32_t* groups_in;
  unsigned long long* tiles_out;
  uint32_t* groups_out;
  unsigned long long* tiles_zero;
  uint32_t* groups_zero;
  uint32_t next_tiles, zero_tiles;
  uint32_t prefetch;                 // tiles ahead to read into L2 (0: none)
  uint32_t* err;
  uint32_t refill;             // the next step needs the next 16 bases
  // last step (j = L)
  uint32_t* bwt;               // packed output words [word0, word0 + n_words) of B_R
  uint64_t word0, n_words;
  uint64_t row_lo, row_hi;     // rows written (all of them, or a part's)
  uint64_t* dollar_pos;        // may be null
  unsigned long long* counts;  // null, or [5] counts of the rows written ($, A, C, G, T), accumulated
  uint32_t tile_lo;            // first tile of the rows written
};

// Tables of reads of L bases: row_base and item_base of steps 0 .. L - 1.
struct MergeTables {
  uint64_t* row_base;   // [L][4]
  uint32_t* item_base;  // [L][4]
  uint32_t* col;        // [L][4] bases at distance 0 .. L-1 from the read's end
};
constexpr uint64_t merge_table_bytes(uint32_t L) { return uint64_t(L) * (4 * 8 + 4 * 4 + 4 * 4) + 64; }
MergeTables merge_tables(void* p, uint32_t L);

// Column counts, step tables, the symbol counts of all of B_R (into counts[5],
// $, A, C, G, T, unless it is null), and the suffixes of length 0 (key, bases,
// and their counts by tile of 2^tile_shift rows and group of tiles, added).
cudaError_t launch_merge_init(const ReadIndex& R, uint32_t n, uint32_t L, const MergeTables& t,
                              unsigned long long* counts, uint64_t* key, uint32_t* bases, uint32_t pshift,
                              uint32_t tile_shift, unsigned long long* tiles, uint32_t* groups, cudaStream_t st);
// k: chunks per thread (1, 2 or 4); wide: rows beyond 32 bits; last: step L.
cudaError_t launch_merge_step(const MergeArgs& a, uint32_t k, bool wide, bool last, cudaStream_t st);

}  // namespace cxbwt
