// The merge plan: B_R of reads of one length, built one suffix length at a
// time from the reads' ends (the insertion scheme of Bauer, Cox & Rosone,
// "Lightweight algorithms for constructing and inverting the BWT of string
// collections", 2013), written for one GPU.
//
// Let B_j be B_R restricted to the suffixes of at most j bases: n (j + 1)
// rows, and B_L = B_R.  The n suffixes of length j, in sorted order, are a
// list of (read, row in B_j).  Step j
//   1. puts the symbol before each of them into B_{j-1} at its row, which
//      gives B_j, and
//   2. finds the rows of the suffixes of length j + 1: the suffix c w, w of
//      length j at row p, is preceded in B_{j+1} by the n terminator-only
//      suffixes, by the suffixes starting with a base below c (as many as
//      there are such symbols in B_j) and by those c v with v before w, one
//      per c in B_j[0, p): its row is n + C_j[c] + rank_c(B_j, p).  Its place
//      among the suffixes of length j + 1 is, in the same way, the number of
//      suffixes of length j whose symbol is below c, plus those of symbol c
//      before it: a stable split of the list by c.
// C_j and the sizes of the classes follow from the bases of each column of
// the reads alone, counted before the first step.  The counts before a tile of
// B_j follow from the step before: its old symbols start at a known row of
// B_{j-1}, whose counts were kept per tile and per warp, and the suffixes
// before it were counted by symbol and tile when they were placed.  So one
// kernel per step does both, and its CTAs neither wait for one another nor
// need any order: each merges a tile of rows, counts its symbols, and writes
// the tile's suffixes of length j + 1 to their places.
//
// Why: a suffix array sort moves an id and a key of every suffix through four
// digit passes and a group finish (about 70 B and 1,100 instructions per
// suffix).  Here a step reads and writes 2 bits per row and 12 bytes per
// read, in address order whatever the reads are: L (0.5 N / 2 + 24 n) bytes
// in all, about 50 + 24 B per suffix of 100-base reads, most of it in L2.
//
// Rows are kept as two bit planes (the low and high bits of the 2-bit codes,
// 32 rows to a word, row 0 in bit 0), so that counting symbols is a
// population count and inserting one is a shift of the bits above it.
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.cuh"
#include "merge.cuh"

namespace cxbwt {
namespace {

// The m <= 16 bases of a read that end at its position `end` (the base at
// end - 1 in the low two bits, the one before it above, ...).
__device__ __forceinline__ uint32_t bases_before(const ReadIndex& R, uint64_t off, uint32_t end) {
  const uint32_t m = min(end, 16u);
  if (m == 0) return 0u;
  const uint64_t q = off + end - m;
  const uint64_t w = q >> 4;
  const uint32_t sh = uint32_t(q & 15u) * 2u;
  const uint32_t window = __funnelshift_l(load_word(R, w + 1), load_word(R, w), sh);
  return window >> (32u - 2u * m);
}

// ---- column counts ------------------------------------------------------------
// Bases at distance d from the reads' ends, for every d: the low bits, the
// high bits and their conjunction are summed over reads in 2-bit, then 8-bit
// fields of one word per 16 columns (a third of an addition per base), where
// a counter increment per base would cost a shared-memory atomic each.  A
// warp takes kColReads reads per lane of one 16-column window.
constexpr uint32_t kColReads = 63;  // 21 groups of 3 reads: every 8-bit field ends at 63 at most

__global__ void __launch_bounds__(256) k_merge_columns(const ReadIndex R, uint32_t n, uint32_t L, uint32_t* __restrict__ col) {
  __shared__ uint32_t s_cnt[16][3];
  const uint32_t win = blockIdx.y;
  const uint32_t d0 = 16u * win, end = L - d0, m = min(end, 16u);
  for (uint32_t x = threadIdx.x; x < 48; x += blockDim.x) (&s_cnt[0][0])[x] = 0u;
  __syncthreads();
  // 8-bit fields: byte b of acc[q][f] counts column 4 b + f.
  uint32_t acc[3][4] = {};
  const uint32_t stride = gridDim.x * blockDim.x;
  uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
  for (uint32_t g = 0; g < kColReads / 3 && r < n; ++g) {
    uint32_t s[3] = {0u, 0u, 0u};
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      const uint32_t w = r < n ? bases_before(R, uint64_t(r) * L, end) : 0u;
      const uint32_t lo = w & 0x55555555u, hi = (w >> 1) & 0x55555555u;
      s[0] += lo;
      s[1] += hi;
      s[2] += lo & hi;
      r = r < n && n - r > stride ? r + stride : n;
    }
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
      for (int f = 0; f < 4; ++f) acc[q][f] += (s[q] >> (2 * f)) & 0x03030303u;
  }
#pragma unroll
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      // 32 lanes of at most 63 fit 16 bits.
      const uint32_t even = __reduce_add_sync(0xFFFFFFFFu, acc[q][f] & 0x00FF00FFu);
      const uint32_t odd = __reduce_add_sync(0xFFFFFFFFu, (acc[q][f] >> 8) & 0x00FF00FFu);
      if ((threadIdx.x & 31) == 0) {
        atomicAdd(&s_cnt[f][q], even & 0xFFFFu);
        atomicAdd(&s_cnt[4 + f][q], odd & 0xFFFFu);
        atomicAdd(&s_cnt[8 + f][q], even >> 16);
        atomicAdd(&s_cnt[12 + f][q], odd >> 16);
      }
    }
  __syncthreads();
  if (threadIdx.x < 48) {
    const uint32_t c = threadIdx.x / 3, q = threadIdx.x % 3, x = s_cnt[c][q];
    if (c < m && x) atomicAdd(&col[(d0 + c) * 4 + 1 + q], x);
  }
}

// col[d] = {-, low bits, high bits, both} becomes {A, C, G, T}; then the first
// row and the first suffix of every class of every step, and the counts.
__global__ void __launch_bounds__(1024) k_merge_tables(uint32_t n, uint32_t L, MergeTables t, unsigned long long* counts) {
  __shared__ unsigned long long s_sum[1024][3];
  const uint32_t per = (L + blockDim.x - 1) / blockDim.x;
  const uint32_t d0 = min(threadIdx.x * per, L), d1 = min(d0 + per, L);
  unsigned long long sum[3] = {0, 0, 0};  // C, G, T
  for (uint32_t d = d0; d < d1; ++d) {
    const uint32_t lo = t.col[4 * d + 1], hi = t.col[4 * d + 2], both = t.col[4 * d + 3];
    t.col[4 * d] = n - lo - hi + both;
    t.col[4 * d + 1] = lo - both;
    t.col[4 * d + 2] = hi - both;
    sum[0] += lo - both;
    sum[1] += hi - both;
    sum[2] += both;
  }
  for (int c = 0; c < 3; ++c) s_sum[threadIdx.x][c] = sum[c];
  __syncthreads();
  for (uint32_t o = 1; o < blockDim.x; o <<= 1) {
    unsigned long long y[3];
    for (int c = 0; c < 3; ++c) y[c] = threadIdx.x >= o ? s_sum[threadIdx.x - o][c] : 0ull;
    __syncthreads();
    for (int c = 0; c < 3; ++c) s_sum[threadIdx.x][c] += y[c];
    __syncthreads();
  }
  unsigned long long run[3];
  for (int c = 0; c < 3; ++c) run[c] = s_sum[threadIdx.x][c] - sum[c];
  for (uint32_t d = d0; d < d1; ++d) {
    const uint32_t A = t.col[4 * d], C = t.col[4 * d + 1], G = t.col[4 * d + 2], T = t.col[4 * d + 3];
    run[0] += C;
    run[1] += G;
    run[2] += T;
    const unsigned long long a = (unsigned long long)n * (d + 1) - run[0] - run[1] - run[2];  // A in B_d
    t.row_base[4 * d] = n;
    t.row_base[4 * d + 1] = n + a;
    t.row_base[4 * d + 2] = n + a + run[0];
    t.row_base[4 * d + 3] = n + a + run[0] + run[1];
    t.item_base[4 * d] = 0;
    t.item_base[4 * d + 1] = A;
    t.item_base[4 * d + 2] = A + C;
    t.item_base[4 * d + 3] = A + C + G;
  }
  if (threadIdx.x == blockDim.x - 1 && counts) {
    const unsigned long long all = (unsigned long long)n * L;
    counts[0] = n;
    counts[1] = all - s_sum[threadIdx.x][0] - s_sum[threadIdx.x][1] - s_sum[threadIdx.x][2];
    for (int c = 0; c < 3; ++c) counts[2 + c] = s_sum[threadIdx.x][c];
  }
}

// Adds the counts (C, G, T) of some suffixes of one tile to the tile's and to
// its group's.
__device__ __forceinline__ void add_class_counts(unsigned long long* tiles, uint32_t* groups, uint32_t tile, uint32_t C,
                                                 uint32_t G, uint32_t T) {
  if ((C | G | T) == 0) return;
  atomicAdd(tiles + tile, (uint64_t(T) << 32) | (uint64_t(G) << 16) | C);
  uint32_t* g = groups + 4 * (tile / kMergeGroupTiles);
  if (C) atomicAdd(g, C);
  if (G) atomicAdd(g + 1, G);
  if (T) atomicAdd(g + 2, T);
}

// The suffixes of length 0 (terminator only), in read order, at rows 0 .. n-1.
constexpr uint32_t kFirstItems = 1024;  // per CTA; a tile holds whole CTAs' suffixes
__global__ void __launch_bounds__(256) k_merge_first(const ReadIndex R, uint32_t n, uint32_t L, uint32_t pshift,
                                                     uint64_t* __restrict__ key, uint32_t* __restrict__ bases,
                                                     uint32_t tile_shift, unsigned long long* tiles, uint32_t* groups) {
  __shared__ uint32_t s_cnt[4];
  if (threadIdx.x < 4) s_cnt[threadIdx.x] = 0u;
  __syncthreads();
  const uint64_t i0 = uint64_t(blockIdx.x) * kFirstItems;
  for (uint32_t x = threadIdx.x; x < kFirstItems && i0 + x < n; x += 256) {
    const uint32_t i = uint32_t(i0) + x;
    const uint32_t w = bases_before(R, uint64_t(i) * L, L);
    key[i] = (uint64_t(i) << pshift) | i;
    bases[i] = w;
    atomicAdd(&s_cnt[w & 3], 1u);
  }
  __syncthreads();
  if (threadIdx.x == 0) add_class_counts(tiles, groups, uint32_t(i0 >> tile_shift), s_cnt[1], s_cnt[2], s_cnt[3]);
}

// ---- one step -------------------------------------------------------------------

// 16 bits (row 0 in bit 0) to the even bits of a word, row 0 in the top pair.
__device__ __forceinline__ uint32_t spread16(uint32_t x) {
  x = __brev(x) >> 16;  // row 0 in bit 15
  x = (x | (x << 8)) & 0x00FF00FFu;
  x = (x | (x << 4)) & 0x0F0F0F0Fu;
  x = (x | (x << 2)) & 0x33333333u;
  return (x | (x << 1)) & 0x55555555u;
}

template <int K>
struct Words;  // K consecutive words of a thread, one vector access
template <>
struct Words<1> {
  using T = uint32_t;
  static __device__ __forceinline__ void get(const T& v, uint32_t (&x)[1]) { x[0] = v; }
  static __device__ __forceinline__ T make(const uint32_t (&x)[1]) { return x[0]; }
};
template <>
struct Words<2> {
  using T = uint2;
  static __device__ __forceinline__ void get(const T& v, uint32_t (&x)[2]) { x[0] = v.x; x[1] = v.y; }
  static __device__ __forceinline__ T make(const uint32_t (&x)[2]) { return make_uint2(x[0], x[1]); }
};
template <>
struct Words<4> {
  using T = uint4;
  static __device__ __forceinline__ void get(const T& v, uint32_t (&x)[4]) { x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w; }
  static __device__ __forceinline__ T make(const uint32_t (&x)[4]) { return make_uint4(x[0], x[1], x[2], x[3]); }
};

// x += the x of the lane d below, where there is one (the shuffle's own
// predicate says so: no comparison of lanes per step).
template <int D>
__device__ __forceinline__ void add_from_below(uint32_t& x) {
  asm volatile("{\n\t.reg .pred p;\n\t.reg .u32 t;\n\t"
      "shfl.sync.up.b32 t|p, %0, %1, 0, -1;\n\t"
      "@p add.u32 %0, %0, t;\n\t}" : "+r"(x) : "n"(D));
}
// Inclusive sums over the lanes, of several words in step.
template <class... T>
__device__ __forceinline__ void warp_scan(T&... x) {
  (add_from_below<1>(x), ...);
  (add_from_below<2>(x), ...);
  (add_from_below<4>(x), ...);
  (add_from_below<8>(x), ...);
  (add_from_below<16>(x), ...);
}

// *p |= v in shared memory if `on`, as a predicated instruction.
__device__ __forceinline__ void or_shared_if(uint32_t* p, uint32_t v, uint32_t on) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p red.shared.or.b32 [%0], %1;\n\t}"
               ::"r"(uint32_t(__cvta_generic_to_shared(p))), "r"(v), "r"(on) : "memory");
}

__device__ __forceinline__ uint32_t lane_id() {
  uint32_t x;
  asm volatile("mov.u32 %0, %%laneid;" : "=r"(x));  // (volatile: kept in a register, not read again)
  return x;
}

// Sum of x over the lanes below `warp`: of the sums of the warps before this
// one, when lane l holds warp l's.
__device__ __forceinline__ uint32_t sum_before(uint32_t x, uint32_t lane, uint32_t warp) {
  return __reduce_add_sync(0xFFFFFFFFu, lane < warp ? x : 0u);
}

template <int K, bool WIDE, bool LAST>
__global__ void __launch_bounds__(kMergeThreads, kMergeBlocks) k_merge_step(const MergeArgs a) {
  using Row = typename std::conditional<WIDE, uint64_t, uint32_t>::type;
  using W = Words<K>;
  using Vec = typename W::T;
  constexpr uint32_t CH = kMergeThreads * K;  // chunks of 32 rows
  constexpr uint32_t TILE = CH * 32;
  constexpr uint32_t OLD = CH + 8;            // old chunks a tile may touch (4-aligned start, one past the end)
  constexpr uint32_t OLDP = OLD + OLD / 32 + 1;
  constexpr int WARPS = kMergeThreads / 32;
  constexpr int HELD = 2;                     // suffixes of the tile that a thread holds in registers
  constexpr int AHEAD = 2;                    // loads in flight for the others
  constexpr uint32_t OLDW = (2 * OLDP + 3) / 4 * 4;
  constexpr uint32_t POOL = LAST ? OLDW : (4 * CH > OLDW ? 4 * CH : OLDW);
  // Per class: row in B_{j+1} of the tile's first symbol of it, the first row
  // of the second tile of B_{j+1} that it may reach, and its first suffix's
  // place in the list.
  struct Class {
    Row row, cross;
    uint32_t at;
  };
  struct __align__(16) Shared {
    uint32_t fresh[CH], lo[CH], hi[CH];  // rows inserted; their symbols, then the tile's planes
    // The old planes (padded by a word per 32: a thread's reads start K words
    // after its neighbour's), then, per class and chunk, the symbols (low half)
    // and suffixes (high half) of the class in the tile's earlier chunks.
    uint32_t pool[POOL];
    uint4 scan3[WARPS];
    uint4 item[WARPS];                   // C, G, T suffixes before the tile, a share per warp
    uint4 end;                           // low bits, high bits, both of the tile
    uint32_t scan[WARPS];
    uint32_t cls[4 * 2 * 4];             // suffixes by class, first or second of those tiles, next symbol
    Row old[4];                          // C, G, T symbols of B_{j-1} before the tile's old rows
    Row before[4];                       // C, G, T symbols of B_j before the tile
    Class base[4];
  };
  __shared__ Shared sh;
  uint32_t* const s_olo = sh.pool;
  uint32_t* const s_ohi = sh.pool + OLDP;

  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (!LAST && tid < 32) sh.cls[tid] = 0u;
  {
    uint32_t z[K] = {};
    reinterpret_cast<Vec*>(sh.fresh)[tid] = W::make(z);
    reinterpret_cast<Vec*>(sh.lo)[tid] = W::make(z);
    reinterpret_cast<Vec*>(sh.hi)[tid] = W::make(z);
  }
  __syncthreads();         // the tile's words are zeroed
  grid_dependency_wait();  // the step before wrote what is read from here on
  grid_launch_dependents();
  const uint32_t tile = blockIdx.x + (LAST ? a.tile_lo : 0u);
  const Row t0 = Row(tile) * TILE;
  const uint32_t rows = uint32_t(min(Row(TILE), Row(Row(a.rows) - t0)));
  // Every load below is issued before the first value is used.
  // Suffixes by symbol before the tile: those of the groups of tiles before
  // its own, and of the tiles before it in its group.
  const uint32_t group = tile / kMergeGroupTiles;
  static_assert(kMergeGroupTiles <= kMergeThreads, "one thread per tile of a group");
  uint4 in_group = make_uint4(0u, 0u, 0u, 0u);
  unsigned long long in_tile = 0;
  Row row_base = 0;
  uint32_t item_base = 0;
  if (!LAST) {
    if (tid < group) in_group = __ldcg(reinterpret_cast<const uint4*>(a.groups_in) + tid);
    if (group * kMergeGroupTiles + tid < tile) in_tile = __ldcg(a.tiles_in + group * kMergeGroupTiles + tid);
    if (warp == WARPS - 1 && lane < 4) {
      row_base = Row(__ldcg(a.row_base + lane));
      item_base = __ldcg(a.item_base + lane);
    }
  }
  // The suffixes of length j in the tile: list entries [s0, s0 + m).  (The
  // clamps here and below only matter when the reads change during the build:
  // they keep every access in bounds.)
  uint32_t s0, m;
  if (a.step == 0) {
    s0 = uint32_t(t0);
    m = rows;
  } else {
    s0 = min(__ldcg(a.start_in + tile), a.n);
    const uint32_t s1 = Row(t0 + rows) < Row(a.rows) ? min(__ldcg(a.start_in + tile + 1), a.n) : a.n;
    m = min(s1 > s0 ? s1 - s0 : 0u, rows);
    if (Row(s0) > t0) s0 = uint32_t(t0);
  }
  const uint64_t pmask = (uint64_t(1) << a.pshift) - 1;
  auto item_row = [&](uint64_t key) { return uint32_t(Row(WIDE ? Row(key & pmask) : Row(key)) - t0); };
  auto item_read = [&](uint64_t key) { return uint32_t(key >> (WIDE ? a.pshift : 32u)); };
  const uint64_t* const keys = a.key_in + s0 + tid;
  const uint32_t* const bases = a.bases_in + s0 + tid;
  const int m_tid = int(m) - int(tid);  // suffix tid + i is there when i < m_tid
  constexpr int STEP = kMergeThreads;
  uint64_t held_key[HELD];
  uint32_t held_w[HELD];
#pragma unroll
  for (int u = 0; u < HELD; ++u) {
    held_key[u] = ~0ull;
    held_w[u] = 0u;
    if (u * STEP < m_tid) {
      held_key[u] = __ldcg(keys + u * STEP);
      if (!LAST) held_w[u] = __ldcg(bases + u * STEP);
    }
  }
  // Old rows [o0, o0 + n_old) stay in the tile.
  const Row rows_in = Row(a.rows - a.n);
  const Row o0 = min(Row(t0 - s0), rows_in);
  const uint32_t n_old = uint32_t(min(Row(rows - m), Row(rows_in - o0)));
  const uint32_t c0 = uint32_t(o0 >> 5) & ~3u;
  const uint32_t skip = uint32_t(o0 - (Row(c0) << 5));
  const uint32_t vecs = n_old ? ((skip + n_old + 31) / 32 + 3) / 4 : 0u;  // at most OLD / 4
  const uint4* lo4 = reinterpret_cast<const uint4*>(a.lo_in + c0);
  const uint4* hi4 = reinterpret_cast<const uint4*>(a.hi_in + c0);
  uint4 old_l, old_h;
  if (tid < vecs) {
    old_l = __ldcg(lo4 + tid);
    old_h = __ldcg(hi4 + tid);
  }
  if (!LAST && warp == WARPS - 1) {
    // Symbols of B_{j-1} before row o0: before its tile, before its part of
    // the tile, and in the part (a word per lane).
    const uint32_t u = uint32_t(o0 >> a.prev_shift), part = (uint32_t(o0) & ((1u << a.prev_shift) - 1)) / kMergePart;
    const uint32_t rest = uint32_t(o0) % kMergePart;
    uint64_t whole = 0, parts = 0;
    if (a.step && lane < 3) {
      whole = __ldcg(a.before_in + 4 * uint64_t(u) + lane);
      if (part) parts = __ldcg(a.parts_in + (uint64_t(u) << (a.prev_shift - 10)) + part);
    }
    const uint32_t at = uint32_t((o0 - rest) >> 5) + lane;
    const uint32_t keep = rest >= 32 * lane + 32 ? 0xFFFFFFFFu : rest > 32 * lane ? (1u << (rest - 32 * lane)) - 1 : 0u;
    const uint32_t l = keep ? __ldcg(a.lo_in + at) & keep : 0u, h = keep ? __ldcg(a.hi_in + at) & keep : 0u;
    uint32_t nc = __popc(l & ~h), ng = __popc(h & ~l), nt_ = __popc(l & h);
    nc = __reduce_add_sync(0xFFFFFFFFu, nc);
    ng = __reduce_add_sync(0xFFFFFFFFu, ng);
    nt_ = __reduce_add_sync(0xFFFFFFFFu, nt_);
    if (lane < 3) sh.old[lane] = Row(whole) + (uint32_t(parts >> (16 * lane)) & 0xFFFFu) + (lane == 0 ? nc : lane == 1 ? ng : nt_);
  }
  if (!LAST) {
    uint32_t c = in_group.x + (uint32_t(in_tile) & 0xFFFFu), g = in_group.y + (uint32_t(in_tile >> 16) & 0xFFFFu),
             t = in_group.z + (uint32_t(in_tile >> 32) & 0xFFFFu);
    for (uint32_t y = tid + kMergeThreads; y < group; y += kMergeThreads) {
      const uint4 x = __ldcg(reinterpret_cast<const uint4*>(a.groups_in) + y);
      c += x.x;
      g += x.y;
      t += x.z;
    }
    c = __reduce_add_sync(0xFFFFFFFFu, c);
    g = __reduce_add_sync(0xFFFFFFFFu, g);
    t = __reduce_add_sync(0xFFFFFFFFu, t);
    if (lane == 0) sh.item[warp] = make_uint4(c, g, t, 0u);
  }
  {
    auto keep_old = [&](uint32_t x, const uint4& l, const uint4& h) {
      const uint32_t at = 4 * x + (x >> 3);
      s_olo[at] = l.x;
      s_olo[at + 1] = l.y;
      s_olo[at + 2] = l.z;
      s_olo[at + 3] = l.w;
      s_ohi[at] = h.x;
      s_ohi[at + 1] = h.y;
      s_ohi[at + 2] = h.z;
      s_ohi[at + 3] = h.w;
    };
    if (tid < vecs) keep_old(tid, old_l, old_h);
    if (tid + kMergeThreads < vecs) keep_old(tid + kMergeThreads, __ldcg(lo4 + tid + kMergeThreads), __ldcg(hi4 + tid + kMergeThreads));
  }
  // The tile one resident grid ahead is read from HBM into L2 now (builds whose
  // planes and lists do not stay there): its range of the list, and its planes.
  uint32_t ahead_s0 = 0, ahead_s1 = 0;
  const uint32_t ahead = tile + a.prefetch;
  const bool prefetch = a.prefetch && warp == WARPS - 2 && lane == 0 && ahead + 1 < a.n_tiles;
  if (prefetch) {
    ahead_s0 = min(__ldcg(a.start_in + ahead), a.n);
    ahead_s1 = min(__ldcg(a.start_in + ahead + 1), a.n);
  }
  bool bad = false;
  auto insert = [&](uint32_t r, uint32_t read, uint32_t w) {
    if (r >= rows) {
      bad = true;
      return;
    }
    const uint32_t bit = 1u << (r & 31);
    or_shared_if(sh.fresh + (r >> 5), bit, 1u);
    if (LAST) {
      // The suffix is the whole read: $ (code 0) precedes it.
      const uint64_t p = uint64_t(t0) + r;
      if (a.dollar_pos && read < a.n && p >= a.row_lo && p < a.row_hi) a.dollar_pos[read] = p;
    } else {
      or_shared_if(sh.lo + (r >> 5), bit, w & 1);
      or_shared_if(sh.hi + (r >> 5), bit, w & 2);
    }
  };
#pragma unroll
  for (int u = 0; u < HELD; ++u)
    if (u * STEP < m_tid) insert(item_row(held_key[u]), item_read(held_key[u]), held_w[u]);
  // The rest (short suffixes, so many to a tile), AHEAD loads at a time.
  for (int i = HELD * STEP; i < m_tid; i += AHEAD * STEP) {
    uint64_t key[AHEAD];
    uint32_t w[AHEAD];
#pragma unroll
    for (int u = 0; u < AHEAD; ++u) {
      key[u] = i + u * STEP < m_tid ? __ldcg(keys + i + u * STEP) : 0ull;
      w[u] = !LAST && i + u * STEP < m_tid ? __ldcg(bases + i + u * STEP) : 0u;
    }
#pragma unroll
    for (int u = 0; u < AHEAD; ++u)
      if (i + u * STEP < m_tid) insert(item_row(key[u]), item_read(key[u]), w[u]);
  }
  if (prefetch && ahead_s0 < ahead_s1) {
    const Row at = Row(ahead) * TILE - ahead_s0;
    const uint32_t c = uint32_t(min(at, rows_in) >> 5) & ~3u;
    if (Row(ahead) * TILE >= ahead_s0 && (Row(c) + CH) * 32 <= rows_in) {
      prefetch_l2(a.lo_in + c, CH * 4);
      prefetch_l2(a.hi_in + c, CH * 4);
    }
    const uint32_t k0 = ahead_s0 & ~3u, kn = (ahead_s1 - k0) & ~3u;
    if (kn) {
      prefetch_l2(a.key_in + k0, kn * 8);
      if ((reinterpret_cast<uintptr_t>(a.bases_in) & 15u) == 0) prefetch_l2(a.bases_in + k0, kn * 4);
    }
  }
  __syncthreads();

  // ---- the new rows before each thread's first chunk ---------------------------
  uint32_t mm[K], lo[K], hi[K];
  W::get(reinterpret_cast<const Vec*>(sh.fresh)[tid], mm);
  uint32_t cnt = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) cnt += __popc(mm[k]);
  uint32_t before = cnt;
  warp_scan(before);
  if (lane == 31) sh.scan[warp] = before;
  __syncthreads();
  before += sum_before(sh.scan[lane & (WARPS - 1)], lane, warp) - cnt;

  if (!LAST && warp == WARPS - 1) {
    // Lane c: class c's symbols and suffixes before the tile.
    const uint4 it = sh.item[lane & (WARPS - 1)];
    const uint32_t ic = __reduce_add_sync(0xFFFFFFFFu, lane < WARPS ? it.x : 0u), ig = __reduce_add_sync(0xFFFFFFFFu, lane < WARPS ? it.y : 0u),
                   itt = __reduce_add_sync(0xFFFFFFFFu, lane < WARPS ? it.z : 0u);
    const Row bc = sh.old[0] + ic, bg = sh.old[1] + ig, bt = sh.old[2] + itt;  // symbols of B_j before the tile
    if (lane < 3) {
      const Row b = lane == 0 ? bc : lane == 1 ? bg : bt;
      sh.before[lane] = b;
      a.before_out[4 * uint64_t(tile) + lane] = b;
    }
    if (lane < 4) {
      const Row row = row_base + (lane == 0 ? t0 - bc - bg - bt : lane == 1 ? bc : lane == 2 ? bg : bt);
      const uint32_t at = item_base + (lane == 0 ? s0 - ic - ig - itt : lane == 1 ? ic : lane == 2 ? ig : itt);
      // Tiles of B_{j+1} are at least as large as this one: the class's
      // symbols, consecutive rows there, reach two at most.
      sh.base[lane] = Class{row, Row((row >> a.next_shift) + 1) << a.next_shift, at};
    }
  }

  // ---- merge: old symbols spread around the new rows ---------------------------
  W::get(reinterpret_cast<const Vec*>(sh.lo)[tid], lo);
  W::get(reinterpret_cast<const Vec*>(sh.hi)[tid], hi);
  const uint32_t o_first = skip + 32 * K * tid - before;  // old row, from row 32 * c0 on
  uint32_t xl[K], xh[K];                                  // per chunk, the next 32 old symbols
  if (K == 1 || !__any_sync(0xFFFFFFFFu, cnt > 32)) {
    // The thread's old rows, aligned to its first chunk; the chunks after it
    // take theirs a few rows earlier, one for each new row before them.
    const uint32_t w = o_first >> 5, sh = o_first & 31;
    uint32_t l0 = s_olo[w + (w >> 5)], h0 = s_ohi[w + (w >> 5)];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const uint32_t i1 = (w + k + 1) + ((w + k + 1) >> 5);
      const uint32_t l1 = s_olo[i1], h1 = s_ohi[i1];
      xl[k] = __funnelshift_r(l0, l1, sh);
      xh[k] = __funnelshift_r(h0, h1, sh);
      l0 = l1;
      h0 = h1;
    }
    uint32_t moved = cnt;
#pragma unroll
    for (int k = K - 1; k > 0; --k) {
      moved -= __popc(mm[k]);
      xl[k] = __funnelshift_lc(xl[k - 1], xl[k], moved);
      xh[k] = __funnelshift_lc(xh[k - 1], xh[k], moved);
    }
  } else {
    uint32_t o = o_first;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const uint32_t w = o >> 5, sh = o & 31;
      const uint32_t i0 = w + (w >> 5), i1 = (w + 1) + ((w + 1) >> 5);
      xl[k] = __funnelshift_r(s_olo[i0], s_olo[i1], sh);
      xh[k] = __funnelshift_r(s_ohi[i0], s_ohi[i1], sh);
      o += 32 - __popc(mm[k]);
    }
  }
  {
    // Each new row, lowest first, moves the old ones from it on up by one:
    // with the bits from it on in `up`, x + (x & up).  A chunk with none left
    // stays as it is (`up` is then empty), so that the warp takes one turn per
    // new row of its fullest chunk, with no branch.
    uint32_t t[K], any;
#pragma unroll
    for (int k = 0; k < K; ++k) t[k] = mm[k];
    do {
      any = 0;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const uint32_t u = t[k] - 1, up = t[k] | ~u;
        xl[k] += xl[k] & up;
        xh[k] += xh[k] & up;
        t[k] &= u;
        any |= t[k];
      }
    } while (__any_sync(0xFFFFFFFFu, any));
    // (new rows are 0 in xl and xh)
#pragma unroll
    for (int k = 0; k < K; ++k) {
      lo[k] |= xl[k];
      hi[k] |= xh[k];
    }
  }
  if (rows < TILE) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const uint32_t first = 32 * (K * tid + k);
      const uint32_t live = rows >= first + 32 ? 0xFFFFFFFFu : rows > first ? (1u << (rows - first)) - 1 : 0u;
      lo[k] &= live;
      hi[k] &= live;
    }
  }
  if (LAST) {
    // Packed words of the rows in [row_lo, row_hi), 16 rows each.
    uint32_t n_sym[5] = {0, 0, 0, 0, 0};  // $, A, C, G, T (counted for parts only)
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const uint64_t g = uint64_t(t0) + 32 * (K * tid + k);  // first row of the chunk
      uint32_t keep = 0xFFFFFFFFu;
      if (g < a.row_lo) keep = a.row_lo - g >= 32 ? 0u : keep << uint32_t(a.row_lo - g);
      if (g + 32 > a.row_hi) keep &= a.row_hi > g ? 0xFFFFFFFFu >> uint32_t(g + 32 - a.row_hi) : 0u;
      const uint32_t l = lo[k] & keep, h = hi[k] & keep;
      const uint64_t word = g >> 4;
      if (word >= a.word0 && word - a.word0 < a.n_words) a.bwt[word - a.word0] = spread16(l & 0xFFFFu) | (spread16(h & 0xFFFFu) << 1);
      if (word + 1 >= a.word0 && word + 1 - a.word0 < a.n_words) a.bwt[word + 1 - a.word0] = spread16(l >> 16) | (spread16(h >> 16) << 1);
      if (a.counts) {
        n_sym[0] += __popc(mm[k] & keep);
        n_sym[1] += __popc(keep & ~(l | h | mm[k]));
        n_sym[2] += __popc(l & ~h);
        n_sym[3] += __popc(h & ~l);
        n_sym[4] += __popc(l & h);
      }
    }
    if (a.counts) {
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        const uint32_t x = __reduce_add_sync(0xFFFFFFFFu, n_sym[c]);
        if (lane == 0 && x) atomicAdd(a.counts + c, (unsigned long long)x);
      }
    }
    if (bad) atomicOr(a.err, kErrBounds);
    return;
  }

  // ---- symbols and suffixes of each class before each chunk, and in the tile ----
  // Low bits, high bits and both, the suffixes' in the high halves.
  uint32_t nl[K], nh[K], nt[K];
  uint32_t tl = 0, th = 0, tt = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    nl[k] = tl;
    nh[k] = th;
    nt[k] = tt;
    const uint32_t both = lo[k] & hi[k];
    tl += __popc(lo[k]) + (__popc(lo[k] & mm[k]) << 16);
    th += __popc(hi[k]) + (__popc(hi[k] & mm[k]) << 16);
    tt += __popc(both) + (__popc(both & mm[k]) << 16);
  }
  uint32_t i0 = tl, i1 = th, i2 = tt;
  warp_scan(i0, i1, i2);
  if (lane == 31) sh.scan3[warp] = make_uint4(i0, i1, i2, 0u);
  {
    // Planes out: whole tiles (the arrays hold whole tiles; rows past the end are 0).
    const uint64_t at = uint64_t(tile) * kMergeThreads + tid;
    __stcg(reinterpret_cast<Vec*>(a.lo_out) + at, W::make(lo));
    __stcg(reinterpret_cast<Vec*>(a.hi_out) + at, W::make(hi));
    reinterpret_cast<Vec*>(sh.lo)[tid] = W::make(lo);
    reinterpret_cast<Vec*>(sh.hi)[tid] = W::make(hi);
  }
  __syncthreads();
  {
    const uint4 x = sh.scan3[lane & (WARPS - 1)];
    i0 += sum_before(x.x, lane, warp);
    i1 += sum_before(x.y, lane, warp);
    i2 += sum_before(x.z, lane, warp);
  }
  if (tid == kMergeThreads - 1) sh.end = make_uint4(i0, i1, i2, 0u);
  if (lane % (32 / K) == 0) {
    // Symbols before the part that starts with the lane's rows, for the next step.
    const uint32_t l = i0 - tl, h = i1 - th, t = i2 - tt;
    a.parts_out[(CH * uint64_t(tile) + K * tid) / 32] =
        (uint64_t(t & 0xFFFFu) << 32) | (uint64_t((h - t) & 0xFFFFu) << 16) | ((l - t) & 0xFFFFu);
  }
  if (tile == a.n_tiles - 1 && tid == kMergeThreads - 1) {
    // Symbols in all of B_j.
    unsigned long long* end = reinterpret_cast<unsigned long long*>(a.before_out) + 4 * uint64_t(tile + 1);
    end[0] = sh.before[0] + ((i0 - i2) & 0xFFFFu);
    end[1] = sh.before[1] + ((i1 - i2) & 0xFFFFu);
    end[2] = sh.before[2] + (i2 & 0xFFFFu);
  }
  // (the old planes were last read before the barrier above)
  {
    uint32_t q[4][K];
    const uint32_t b0 = i0 - tl, b1 = i1 - th, b2 = i2 - tt;
    uint32_t news = before;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const uint32_t l = nl[k] + b0, h = nh[k] + b1, t = nt[k] + b2;
      q[0][k] = (32 * (K * tid + k) + (news << 16)) - l - h + t;
      q[1][k] = l - t;
      q[2][k] = h - t;
      q[3][k] = t;
      news += __popc(mm[k]);
    }
    auto* pool = reinterpret_cast<Vec*>(sh.pool);
#pragma unroll
    for (int c = 0; c < 4; ++c) pool[c * kMergeThreads + tid] = W::make(q[c]);
  }

  __syncthreads();

  // ---- the suffixes of length j + 1 -----------------------------------------------
  auto place = [&](uint32_t r, uint32_t read, uint32_t w) {
    if (r >= rows) return;
    const uint32_t q = r >> 5, c = w & 3;
    const Class base = sh.base[c];
    // Rows of symbol c below r in its chunk.
    const uint32_t same = (sh.lo[q] ^ ((c & 1) - 1)) & (sh.hi[q] ^ ((c >> 1) - 1)) & ((1u << (r & 31)) - 1);
    const uint32_t counts = sh.pool[c * CH + q];
    const Row row = base.row + ((counts & 0xFFFFu) + __popc(same));
    const uint32_t at = base.at + (counts >> 16) + __popc(same & sh.fresh[q]);
    w >>= 2;
    if (a.refill) w = bases_before(a.R, uint64_t(min(read, a.n - 1)) * a.R.uniform_len, a.R.uniform_len - (a.step + 1));
    atomicAdd(&sh.cls[c * 8 + (row >= base.cross ? 4u : 0u) + (w & 3)], 1u);
    if (at < a.n) {
      __stcg(a.key_out + at, WIDE ? (uint64_t(read) << a.pshift) | (uint64_t(row) & pmask) : (uint64_t(read) << 32) | row);
      __stcg(a.bases_out + at, w);
    } else {
      bad = true;
    }
  };
#pragma unroll
  for (int u = 0; u < HELD; ++u)
    if (u * STEP < m_tid) place(item_row(held_key[u]), item_read(held_key[u]), held_w[u]);
  for (int i = HELD * STEP; i < m_tid; i += AHEAD * STEP) {
    uint64_t key[AHEAD];
    uint32_t w[AHEAD];
#pragma unroll
    for (int u = 0; u < AHEAD; ++u) {
      key[u] = i + u * STEP < m_tid ? __ldcg(keys + i + u * STEP) : 0ull;
      w[u] = i + u * STEP < m_tid ? __ldcg(bases + i + u * STEP) : 0u;
    }
#pragma unroll
    for (int u = 0; u < AHEAD; ++u)
      if (i + u * STEP < m_tid) place(item_row(key[u]), item_read(key[u]), w[u]);
  }
  // Counts of step j + 2 are not in use: zeroed for the step after the next.
  for (uint32_t x = tile; x < a.zero_tiles; x += a.n_tiles) {
    if (tid == 0) a.tiles_zero[x] = 0;
    if (tid < 4 && x % kMergeGroupTiles == 0) a.groups_zero[4 * (x / kMergeGroupTiles) + tid] = 0;
  }
  __syncthreads();
  // ---- suffixes in and before the tiles of B_{j+1} -----------------------------------
  if (tid < 8) {
    const uint32_t c = tid >> 1, second = tid & 1;
    const uint32_t* n_cls = sh.cls + tid * 4;
    const Class base = sh.base[c];
    const uint32_t e0 = sh.end.x, e1 = sh.end.y, e2 = sh.end.z;
    const uint32_t C = (e0 - e2) & 0xFFFFu, G = (e1 - e2) & 0xFFFFu, T = e2 & 0xFFFFu;
    const uint32_t total = c == 0 ? rows - C - G - T : c == 1 ? C : c == 2 ? G : T;
    const uint32_t to = uint32_t(base.cross >> a.next_shift) - 1 + second;
    const Row first = second ? base.cross : Row(base.cross - (Row(1) << a.next_shift));  // of tile `to`
    if (first >= base.row && first < base.row + total && to < a.next_tiles) {
      const uint32_t* n_first = n_cls - 4;
      a.start_out[to] = base.at + (second ? n_first[0] + n_first[1] + n_first[2] + n_first[3] : 0u);
    }
    if (to < a.next_tiles) add_class_counts(a.tiles_out, a.groups_out, to, n_cls[1], n_cls[2], n_cls[3]);
  }
  if (bad) atomicOr(a.err, kErrBounds);
}

template <int K, bool WIDE, bool LAST>
cudaError_t launch_step(const MergeArgs& a, cudaStream_t st) {
  return launch_after(true, k_merge_step<K, WIDE, LAST>, dim3(a.n_tiles), kMergeThreads, 0, st, a);
}

}  // namespace

MergeTables merge_tables(void* p, uint32_t L) {
  MergeTables t;
  t.row_base = static_cast<uint64_t*>(p);
  t.item_base = reinterpret_cast<uint32_t*>(t.row_base + 4 * size_t(L));
  t.col = t.item_base + 4 * size_t(L);
  return t;
}

cudaError_t launch_merge_init(const ReadIndex& R, uint32_t n, uint32_t L, const MergeTables& t,
                              unsigned long long* counts, uint64_t* key, uint32_t* bases, uint32_t pshift,
                              uint32_t tile_shift, unsigned long long* tiles, uint32_t* groups, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(t.col, 0, size_t(L) * 4 * 4, st);
  if (e != cudaSuccess) return e;
  const uint32_t per_cta = 256 * kColReads;
  k_merge_columns<<<dim3((n + per_cta - 1) / per_cta, (L + 15) / 16), 256, 0, st>>>(R, n, L, t.col);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_merge_tables<<<1, 1024, 0, st>>>(n, L, t, counts);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_merge_first<<<(n + kFirstItems - 1) / kFirstItems, 256, 0, st>>>(R, n, L, pshift, key, bases, tile_shift, tiles, groups);
  return cudaGetLastError();
}

cudaError_t launch_merge_step(const MergeArgs& a, uint32_t k, bool wide, bool last, cudaStream_t st) {
  if (a.n_tiles == 0) return cudaSuccess;
  if (wide) return last ? launch_step<4, true, true>(a, st) : launch_step<4, true, false>(a, st);
  switch (k) {
    case 1: return last ? launch_step<1, false, true>(a, st) : launch_step<1, false, false>(a, st);
    case 2: return last ? launch_step<2, false, true>(a, st) : launch_step<2, false, false>(a, st);
    default: return last ? launch_step<4, false, true>(a, st) : launch_step<4, false, false>(a, st);
  }
}

}  // namespace cxbwt
