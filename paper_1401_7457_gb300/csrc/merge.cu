// Host side of the merge plan (k_merge.cu): when a build takes it, its
// workspace, and its steps.
#include <cuda_runtime.h>

#include "host.cuh"
#include "merge.cuh"

namespace cxbwt {
namespace host {
namespace {

uint32_t bits_of(uint64_t x) {  // smallest s with 2^s > x
  uint32_t s = 0;
  while (s < 64 && (x >> s)) ++s;
  return s;
}

// Chunks per thread of step j over `rows` rows: larger tiles have fewer fixed
// costs per row, smaller ones fill the GPU (one tile per resident CTA, or
// half as many: 100k x 100 bases 0.82 ms, against 0.87 with twice the rows
// and 1.09 with the largest tiles throughout) and hold fewer of the first
// steps' suffixes, one row in j + 1 (1M x 36 bases 0.84 ms, against 0.86
// without that bound).  Tiles never shrink from one step to the next.
uint32_t tile_k(const cxbwt_ctx* c, bool wide, uint64_t rows, uint32_t j) {
  if (wide) return 4;
  const uint64_t resident = uint64_t(c->sm_count) * kMergeBlocks;
  if (2 * rows <= resident * merge_tile_rows(1) || j < 8) return 1;
  if (2 * rows <= resident * merge_tile_rows(2) || j < 16) return 2;
  return 4;
}

// Row numbers past 32 bits, with room for a tile past the end (or asked for).
bool is_wide(const cxbwt_ctx* c, const Plan& pl) {
  return pl.N > 0xFFFFFFFFull - kMergeMaxTile || (c->opt.plan_flags & CXBWT_PLAN_ID64);
}

// A step whose planes and lists (read and written) are larger has its tiles
// read into L2 ahead (8M x 100 bases: 14.8 -> 14.2 ms; no difference below).
constexpr uint64_t kL2Bytes = 96u << 20;

// Where the parts of the workspace buffers are: c->vals (planes), c->keys
// (suffix lists), c->mtables (step tables), c->mstatus (per-tile counts).
struct Layout {
  uint64_t planes, list, tables, counts;          // bytes of one buffer of each
  uint64_t starts, before, parts, tiles, groups;  // bytes of one of the per-tile arrays
  uint64_t off_starts, off_before, off_parts, off_tiles, off_groups;
};

Layout layout_of(const cxbwt_ctx* c, const Plan& pl) {
  Layout z;
  z.planes = merge_plane_words(pl.N) * 4 * 2;
  z.list = pl.n * 12;
  z.tables = merge_table_bytes(pl.Lmax);
  uint64_t tiles = 0;  // the most tiles any step has
  for (uint32_t j = 0; j <= pl.Lmax; ++j) {
    const uint64_t rows = pl.n * uint64_t(j + 1), tile = merge_tile_rows(tile_k(c, is_wide(c, pl), rows, j));
    tiles = std::max(tiles, (rows + tile - 1) / tile);
  }
  auto pad = [](uint64_t x) { return (x + 255) / 256 * 256; };
  z.starts = pad((tiles + 2) * 4);
  z.before = pad((tiles + 2) * 32);
  z.parts = pad((pl.N / kMergePart + 2 * kMergeMaxTile / kMergePart) * 8);
  z.tiles = pad((tiles + 2) * 8);
  z.groups = pad((tiles / kMergeGroupTiles + 2) * 16);
  // Starts, tile counts and group counts must be zero at first: side by side.
  z.off_starts = 0;
  z.off_tiles = 2 * z.starts;
  z.off_groups = z.off_tiles + 3 * z.tiles;
  z.off_before = z.off_groups + 3 * z.groups;
  z.off_parts = z.off_before + 2 * z.before;
  z.counts = z.off_parts + 2 * z.parts;
  return z;
}

}  // namespace

bool merge_fits(const cxbwt_ctx* c, const Plan& pl, uint64_t more) {
  if (!pl.uniform || pl.Lmax > kMergeMaxLen || bits_of(pl.n - 1) + bits_of(pl.N - 1) > 64) return false;
  const Layout z = layout_of(c, pl);
  uint64_t held = c->held + more;
  auto grow = [&](const DevBuf& b, uint64_t bytes) {
    if (b.cap < bytes) held += bytes + (2u << 20) - b.cap;
  };
  grow(c->vals[0], z.planes);
  grow(c->vals[1], z.planes);
  grow(c->keys[0], z.list);
  grow(c->keys[1], z.list);
  grow(c->mstatus, z.counts);
  grow(c->mtables, z.tables);
  return held <= c->budget;
}

int merge_run(cxbwt_ctx* c, Run& r, uint64_t row_lo, uint64_t row_hi, uint64_t word0, uint64_t n_words, bool count_rows) {
  const Plan& pl = r.pl;
  cudaStream_t st = r.st;
  const uint32_t n = uint32_t(pl.n), L = pl.Lmax;
  const Layout z = layout_of(c, pl);
  for (int b = 0; b < 2; ++b) {
    CX_TRY(ensure(c, c->vals[b], z.planes, "merge planes"));
    CX_TRY(ensure(c, c->keys[b], z.list, "merge lists"));
  }
  CX_TRY(ensure(c, c->mstatus, z.counts, "merge counts"));
  CX_TRY(ensure(c, c->mtables, z.tables, "merge tables"));
  char* cb = static_cast<char*>(c->mstatus.p);
  CX_CUDA(c, cudaMemsetAsync(cb, 0, z.off_before, st));
  auto starts = [&](uint32_t j) { return reinterpret_cast<uint32_t*>(cb + z.off_starts + (j % 2) * z.starts); };
  auto before = [&](uint32_t j) { return reinterpret_cast<uint64_t*>(cb + z.off_before + (j % 2) * z.before); };
  auto parts = [&](uint32_t j) { return reinterpret_cast<uint64_t*>(cb + z.off_parts + (j % 2) * z.parts); };
  auto tiles = [&](uint32_t j) { return reinterpret_cast<unsigned long long*>(cb + z.off_tiles + (j % 3) * z.tiles); };
  auto groups = [&](uint32_t j) { return reinterpret_cast<uint32_t*>(cb + z.off_groups + (j % 3) * z.groups); };
  const uint64_t pw = merge_plane_words(pl.N);
  auto plane = [&](uint32_t j) { return static_cast<uint32_t*>(c->vals[j % 2].p); };
  auto key = [&](uint32_t j) { return static_cast<uint64_t*>(c->keys[j % 2].p); };
  auto bases = [&](uint32_t j) { return reinterpret_cast<uint32_t*>(key(j) + n); };
  const bool wide = is_wide(c, pl);
  const uint32_t pshift = wide ? bits_of(pl.N - 1) : 32u;
  const MergeTables t = merge_tables(c->mtables.p, L);
  auto k_of = [&](uint32_t j) { return tile_k(c, wide, pl.n * uint64_t(j + 1), j); };
  auto tiles_of = [&](uint32_t j) {
    const uint64_t tile = merge_tile_rows(k_of(j));
    return uint32_t((pl.n * uint64_t(j + 1) + tile - 1) / tile);
  };
  CX_CUDA(c, launch_merge_init(r.R, n, L, t, count_rows ? nullptr : r.d_counts, key(0), bases(0), pshift,
                               merge_tile_shift(k_of(0)), tiles(0), groups(0), st));
  r.launches += 3;
  MergeArgs a{};
  a.R = r.R;
  a.n = n;
  a.err = r.d_err;
  a.pshift = pshift;
  for (uint32_t j = 0; j <= L; ++j) {
    const uint32_t k = k_of(j);
    const bool last = j == L;
    a.step = j;
    a.rows = pl.n * uint64_t(j + 1);
    a.n_tiles = tiles_of(j);
    a.lo_in = plane(j + 1);
    a.hi_in = a.lo_in + pw;
    a.lo_out = plane(j);
    a.hi_out = a.lo_out + pw;
    a.key_in = key(j);
    a.bases_in = bases(j);
    a.key_out = key(j + 1);
    a.bases_out = bases(j + 1);
    a.start_in = starts(j);
    a.start_out = starts(j + 1);
    a.prev_shift = merge_tile_shift(k_of(j ? j - 1 : 0));
    a.next_shift = merge_tile_shift(k_of(last ? j : j + 1));
    a.row_base = t.row_base + 4 * size_t(j);
    a.item_base = t.item_base + 4 * size_t(j);
    a.before_in = before(j + 1);
    a.parts_in = parts(j + 1);
    a.before_out = before(j);
    a.parts_out = parts(j);
    a.tiles_in = tiles(j);
    a.groups_in = groups(j);
    a.tiles_out = tiles(j + 1);
    a.groups_out = groups(j + 1);
    a.tiles_zero = tiles(j + 2);
    a.groups_zero = groups(j + 2);
    a.next_tiles = last ? 0u : tiles_of(j + 1);
    a.zero_tiles = j + 2 <= L ? tiles_of(j + 2) : 0u;
    a.prefetch = j && a.rows / 2 + pl.n * 24 > kL2Bytes ? uint32_t(c->sm_count) * kMergeBlocks : 0u;
    a.refill = (j + 1) % 16 == 0 && j + 1 < L;
    if (last) {
      const uint32_t tile = merge_tile_rows(k);
      a.bwt = r.d_bwt;
      a.word0 = word0;
      a.n_words = n_words;
      a.row_lo = row_lo;
      a.row_hi = row_hi;
      a.dollar_pos = r.d_dollar;
      a.counts = count_rows ? r.d_counts : nullptr;
      a.tile_lo = uint32_t(row_lo / tile);
      a.n_tiles = row_hi > row_lo ? uint32_t((row_hi + tile - 1) / tile) - a.tile_lo : 0u;
    }
    CX_CUDA(c, launch_merge_step(a, k, wide, last, st));
    ++r.launches;
    ++r.merge_launches;
  }
  return CXBWT_OK;
}

}  // namespace host
}  // namespace cxbwt
