// prep.cu -- graph-only steps of bbTC (run once per graph by bbtc_graph_create):
//   a1 canonical simple edge set  (Sec. 2: simple undirected graph, (u,v) with u<v)
//   a2 degree                     (Sec. 2, Sec. 4.1)
//   a3 order by degree            (Sec. 4.1: non-decreasing degree, ties by id)
//   a4 orientation                (Sec. 2: N(G,u) = {v : (u,v) in E, u < v})
#include <limits.h>

#include "bounds.cuh"
#include "graph.cuh"
#include "primitives.cuh"

namespace bbtc {

namespace {

// rowptr[0] == 0 and non-decreasing; error bit 1 otherwise. With deg, also
// deg[r] = the row's length (pass 0 takes off what is no edge).
__global__ void k_validate_rowptr(const int64_t *__restrict__ rowptr, int64_t n,
                                  int32_t *__restrict__ deg, int32_t *__restrict__ err) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = rowptr[i], e = rowptr[i + 1];
    if (b > e) atomicOr(err, 1);
    if (deg) deg[i] = (int32_t)(e - b);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0 && rowptr[0] != 0) atomicOr(err, 1);
}

// Distinct edges by hashing instead of sorting: the steps after need the distinct
// keys in no particular order. A key is stored times an odd factor (the first
// multiplier of SplitMix64's finaliser), a bijection of 64-bit words: its top bits choose one of 2^lb buckets of at most BK_CAP keys (half
// to three quarters full on average), the next ones its slot in a table in shared
// memory. EMPTY, all ones, is the image of no key (its preimage is above 2^62). A
// bucket overflows only when an edge is listed some hundred times or the keys were
// chosen to collide (random keys spread by 40 around 1,536; paths, grids, bands,
// stars and bipartite graphs less); the keys are then sorted. What bounds it: the
// emission waits on its cursor additions (0.22 ms for 17 M keys), this kernel on its
// table in shared memory and on degree additions (0.41 ms). Preparation
// by hashing and by sorting took 0.26 and 0.30 ms for 131 K entries (R-MAT scale
// 13), 0.54 and 0.72 for 4 M, 1.38 and 2.02 for 17 M, 1.69 and 2.47 for 21 M of a
// G(n, m), 13.9 and 17.8 for 134 M (one table in device memory instead of buckets:
// 1.92 for the 17 M); for an edge listed 4 M times, which overflows, 0.72 and 0.55.
constexpr uint64_t HASH_FACTOR = 0xBF58476D1CE4E5B9ull, HASH_INVERSE = 0x96DE1B173F119089ull;
static_assert(HASH_FACTOR * HASH_INVERSE == 1ull, "inverse of the hash factor");
static_assert(~0ull * HASH_INVERSE > (1ull << 62), "EMPTY is no key");
constexpr uint64_t HASH_EMPTY = ~0ull;
constexpr unsigned long long HASH_FAILED = 1ull << 62;
constexpr int64_t HASH_MAX = 1ll << 28;  // entries (buckets of 2.7 GB to 4.3 GB); more are sorted
// cursors lie a sector apart: side by side, 1 M keys (1,024 buckets) took 0.387 ms
// instead of 0.336 (one sector takes one addition at a time)
constexpr int BK_PAD = 8;
constexpr int BK_NT = 256, BK_ITEMS = 8, BK_CAP = BK_NT * BK_ITEMS, BK_MEAN = BK_CAP * 3 / 4;
static_assert((BK_CAP & (BK_CAP - 1)) == 0, "the table holds any bucket twice over");

// a1 + a2: one CTA per bucket inserts its keys into a table of at least twice their
// number; the first of equal keys goes to ukeys and counts towards its endpoints'
// degrees, lanes that add to one vertex (a hub's edges) adding once. *nunique gets
// HASH_FAILED when a bucket has overflowed, or when there are more than `room` keys
// (input that lists edges under one endpoint only though said to be symmetric); the
// results are then void.
__global__ void __launch_bounds__(BK_NT) k_bucket_unique(const uint64_t *__restrict__ keys,
                                                         const unsigned *__restrict__ fill,
                                                         int lb, int nb, int64_t room,
                                                         uint64_t *__restrict__ ukeys,
                                                         unsigned long long *__restrict__ nunique,
                                                         int32_t *__restrict__ deg) {
  __shared__ unsigned long long table[2 * BK_CAP];
  __shared__ unsigned fresh_of[BK_NT / 32];
  __shared__ unsigned long long base_s;
  const unsigned count = fill[blockIdx.x * BK_PAD];
  if (count == 0 || count > BK_CAP) {
    if (count && threadIdx.x == 0) atomicOr(nunique, HASH_FAILED);
    return;
  }
  const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const int ls = 32 - __clz((int)(2 * count - 1));  // 2 * count <= 2^ls <= 2 * BK_CAP
  const unsigned slots = 1u << ls;
  uint64_t k[BK_ITEMS];
#pragma unroll
  for (int i = 0; i < BK_ITEMS; ++i) {
    const unsigned x = (unsigned)(i * BK_NT) + threadIdx.x;
    k[i] = x < count ? keys[(int64_t)blockIdx.x * BK_CAP + x] : HASH_EMPTY;
  }
  for (unsigned x = threadIdx.x; x < slots; x += BK_NT) table[x] = HASH_EMPTY;
  __syncthreads();
  unsigned fresh[BK_ITEMS], mine = 0;
#pragma unroll
  for (int i = 0; i < BK_ITEMS; ++i) {
    bool is_new = false;
    if (k[i] != HASH_EMPTY) {
      unsigned slot = (unsigned)((k[i] << lb) >> (64 - ls));
      for (;;) {  // the table is at most half full: a free slot is found
        unsigned long long old = *(volatile unsigned long long *)&table[slot];
        if (old == HASH_EMPTY) {
          old = atomicCAS(&table[slot], HASH_EMPTY, (unsigned long long)k[i]);
          if (old == HASH_EMPTY) {
            is_new = true;
            break;
          }
        }
        if (old == k[i]) break;
        slot = (slot + 1) & (slots - 1);
      }
    }
    fresh[i] = __ballot_sync(0xffffffffu, is_new);
    mine += __popc(fresh[i]);
  }
  if (lane == 0) fresh_of[warp] = mine;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned total = 0;
    for (int x = 0; x < BK_NT / 32; ++x) {
      const unsigned c = fresh_of[x];
      fresh_of[x] = total;
      total += c;
    }
    base_s = atomicAdd(nunique, (unsigned long long)total) & (HASH_FAILED - 1);
    if ((int64_t)base_s + total > room) {
      atomicOr(nunique, HASH_FAILED);
      base_s = HASH_FAILED;
    }
  }
  __syncthreads();
  if (base_s == HASH_FAILED) return;
  int64_t at = (int64_t)base_s + fresh_of[warp];
  const uint64_t mask = (1ull << nb) - 1ull;
#pragma unroll
  for (int i = 0; i < BK_ITEMS; ++i) {
    if (!fresh[i]) continue;
    const bool is_new = ((fresh[i] >> lane) & 1u) != 0u;
    const uint64_t key = k[i] * HASH_INVERSE;
    const int32_t a = is_new ? (int32_t)(key >> nb) : -1, b = is_new ? (int32_t)(key & mask) : -1;
    if (is_new) ukeys[at + __popc(fresh[i] & ((1u << lane) - 1u))] = key;
    at += __popc(fresh[i]);
    unsigned peers = __match_any_sync(0xffffffffu, a);
    if (a >= 0 && lane == (unsigned)(__ffs(peers) - 1)) atomicAdd(&deg[a], __popc(peers));
    peers = __match_any_sync(0xffffffffu, b);
    if (b >= 0 && lane == (unsigned)(__ffs(peers) - 1)) atomicAdd(&deg[b], __popc(peers));
  }
}

constexpr int UQ_NT = 512;
constexpr int UQ_ITEMS = 8;
constexpr int UQ_TILE = UQ_NT * UQ_ITEMS;

__global__ void __launch_bounds__(UQ_NT) k_unique_count(const uint64_t *__restrict__ keys,
                                                        int64_t count, uint64_t sentinel,
                                                        const int32_t *__restrict__ err,
                                                        uint64_t *__restrict__ block_counts) {
  __shared__ uint64_t tmp[UQ_NT / 32 + 1];
  if (*err & SORT_FAILED) count = 0;  // the keys are not in order: nothing is read from them
  const int64_t base = (int64_t)blockIdx.x * UQ_TILE + (int64_t)threadIdx.x * UQ_ITEMS;
  uint64_t c = 0;
  uint64_t k = base > 0 && base < count ? keys[base - 1] : sentinel;
#pragma unroll
  for (int i = 0; i < UQ_ITEMS; ++i)
    if (base + i < count) {
      const uint64_t x = keys[base + i];
      if (x != sentinel && (base + i == 0 || x != k)) ++c;
      k = x;
    }
  uint64_t total;
  block_exclusive_scan<uint64_t, UQ_NT>(c, tmp, &total);
  if (threadIdx.x == 0) block_counts[blockIdx.x] = total;
}

// a1 + a2: compact the distinct keys and count each endpoint's degree. Keys are
// sorted by their first endpoint, so a thread adds once per run of equal first
// endpoints among its eight keys (and a warp within one run once); the second
// endpoints differ from lane to lane and are added one by one.
__global__ void __launch_bounds__(UQ_NT) k_unique_write(const uint64_t *__restrict__ keys,
                                                        int64_t count, uint64_t sentinel,
                                                        const int32_t *__restrict__ err,
                                                        const uint64_t *__restrict__ block_off,
                                                        int nb, uint64_t *__restrict__ ukeys,
                                                        int32_t *__restrict__ deg) {
  __shared__ uint64_t tmp[UQ_NT / 32 + 1];
  __shared__ uint64_t out[UQ_TILE];  // the tile's distinct keys, written with coalesced stores
  if (*err & SORT_FAILED) count = 0;
  const int64_t base = (int64_t)blockIdx.x * UQ_TILE + (int64_t)threadIdx.x * UQ_ITEMS;
  const unsigned lane = threadIdx.x & 31u;
  uint64_t k[UQ_ITEMS];
  unsigned heads = 0;
  uint64_t prev = base > 0 && base < count ? keys[base - 1] : sentinel;
#pragma unroll
  for (int i = 0; i < UQ_ITEMS; ++i) {
    k[i] = base + i < count ? keys[base + i] : sentinel;
    if (k[i] != sentinel && (base + i == 0 || k[i] != prev)) heads |= 1u << i;
    prev = k[i];
  }
  uint64_t total;
  uint64_t pos = block_exclusive_scan<uint64_t, UQ_NT>((uint64_t)__popc(heads), tmp, &total);
  const uint64_t mask = (1ull << nb) - 1ull;
  int64_t cur = -1;
  int cnt = 0, groups = 0;
#pragma unroll
  for (int i = 0; i < UQ_ITEMS; ++i) {
    if ((heads >> i) & 1u) {
      out[pos++] = k[i];
      const int64_t a = (int64_t)(k[i] >> nb);
      atomicAdd(&deg[k[i] & mask], 1);
      if (a != cur) {
        if (cur >= 0) atomicAdd(&deg[cur], cnt);
        cur = a;
        cnt = 0;
        ++groups;
      }
      ++cnt;
    }
  }
  const int64_t cur0 = __shfl_sync(0xffffffffu, cur, 0);
  if (__all_sync(0xffffffffu, groups == 1 && cur == cur0)) {
    const int tot = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) atomicAdd(&deg[cur0], tot);
  } else if (cur >= 0) {
    atomicAdd(&deg[cur], cnt);
  }
  __syncthreads();
  const uint64_t off = block_off[blockIdx.x];
  for (int i = threadIdx.x; i < (int)total; i += UQ_NT) ukeys[off + i] = out[i];
}

// a3 keys: (degree << nb) | id, so ascending order is (degree, id).
__global__ void k_rank_keys(const int32_t *__restrict__ deg, int64_t n, int nb,
                            uint64_t *__restrict__ keys) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    keys[v] = ((uint64_t)deg[v] << nb) | (uint64_t)v;
}

__global__ void k_rank_finish(const uint64_t *__restrict__ sorted, int64_t n, int nb,
                              const int32_t *__restrict__ err, int32_t *__restrict__ perm,
                              int32_t *__restrict__ rank) {
  const uint64_t mask = (1ull << nb) - 1ull;
  const bool failed = (*err & SORT_FAILED) != 0;  // then any order: the caller reports it
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n;
       r += (int64_t)gridDim.x * blockDim.x) {
    int32_t v = failed ? (int32_t)r : (int32_t)(sorted[r] & mask);
    perm[r] = v;
    rank[v] = (int32_t)r;
  }
}

// Batch handles: graph of each position (the graph owning perm[r]).
__global__ void k_graph_of_position(const int32_t *__restrict__ perm, int64_t n,
                                    const int64_t *__restrict__ voff, int ng,
                                    int32_t *__restrict__ gid) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = perm[r];
    int lo = 0, hi = ng;
    while (hi - lo > 1) {
      int mid = (lo + hi) >> 1;
      if (voff[mid] <= v) lo = mid; else hi = mid;
    }
    gid[r] = lo;
  }
}

// a4 by counting: each edge's slot within its source's row (the count before it),
// and the rows' lengths; then the scatter into the rows, which are sorted after.
__global__ void k_orient_count(const uint64_t *__restrict__ ukeys, int64_t m, int nb,
                               const int32_t *__restrict__ rank, uint64_t *__restrict__ okeys,
                               unsigned *__restrict__ slot,
                               unsigned long long *__restrict__ rowlen) {
  const uint64_t mask = (1ull << nb) - 1ull;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t k = ukeys[e];
    const uint64_t ra = (uint64_t)rank[k >> nb], rb = (uint64_t)rank[k & mask];
    const uint64_t lo = ra < rb ? ra : rb, hi = ra < rb ? rb : ra;
    okeys[e] = (lo << nb) | hi;
    slot[e] = (unsigned)atomicAdd(&rowlen[lo], 1ull);
  }
}

__global__ void k_orient_scatter(const uint64_t *__restrict__ okeys,
                                 const unsigned *__restrict__ slot, int64_t m, int nb,
                                 const int64_t *__restrict__ rowptr, int32_t *__restrict__ colidx) {
  const uint64_t mask = (1ull << nb) - 1ull;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t k = okeys[e];
    colidx[rowptr[k >> nb] + slot[e]] = (int32_t)(k & mask);
  }
}

// ------------------------------------------------------------------------
// Symmetric input with sorted rows (every edge listed under both endpoints,
// each row ascending): the canonical edges of row u are its entries above u,
// each counted once, so no global sort is needed.

constexpr int SEG_CAP = 2048;  // longest oriented row sorted in shared memory
constexpr int64_t SYM_ASK_N = 1 << 18;  // vertices from which the largest degree is asked for

__device__ __forceinline__ int64_t row_of_first(const int64_t *rowptr, int64_t n, int64_t target,
                                                int64_t lo_hint, int64_t hi_hint) {
  int64_t lo = lo_hint, hi = hi_hint;  // rowptr[lo] <= target
  while (hi - lo > 1) {
    int64_t mid = (lo + hi) >> 1;
    if (rowptr[mid] <= target) lo = mid; else hi = mid;
  }
  return lo;
}

constexpr int SP_NT = 256;
constexpr int SP_ITEMS = 8;
constexpr int SP_TILE = SP_NT * SP_ITEMS;

// Row of the first entry of every tile of SP_TILE entries (and of the last
// entry, in the final slot): the row windows of the per-entry passes.
__global__ void k_tile_rows(const int64_t *__restrict__ rowptr, int64_t n, int64_t nnz,
                            int64_t ntiles, int64_t *__restrict__ rows) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t <= ntiles;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t target = t < ntiles ? t * SP_TILE : nnz - 1;
    rows[t] = row_of_first(rowptr, n, target, 0, n);
  }
}

// The rows of a tile's entries. The starts of the rows inside the tile are marked
// in a bit mask (and each start's row beside it), so that an entry's row is that of
// the last mark at or before it: no search and no walk along row pointers, whose
// dependent loads bounded these passes before (0.38 ms for pass 0 over the 67 M
// entries of R-MAT scale 21, 1.4 TB/s for a pass that only streams them).
struct TileRows {
  uint32_t start[SP_TILE / 32];  // marks
  unsigned long long words;      // words of `start` with a mark (SP_TILE / 32 = 64)
  int32_t row[SP_TILE];          // row of each mark
  int first_is_start;            // the tile's first entry begins its row
};
static_assert(SP_TILE / 32 == 64 && SP_ITEMS == 8, "tile layout");

// What a block needs of a tile, loaded while it works on the tile before it (the
// rows of the tile's ends, two tiles ahead): row pointers of up to SP_NT rows, the
// thread's eight entries and the one before them.
struct TileAhead {
  int64_t rlo, rhi;      // rows of the tile's first entry and of the next tile's
  int64_t begin, end;    // row rlo + 1 + threadIdx.x
  int64_t start;         // of row rlo
  int32_t w[SP_ITEMS];
  int32_t prev;
};

__device__ __forceinline__ void load_entries(const int32_t *__restrict__ colidx, int64_t first,
                                             int64_t t1, bool aligned, int32_t (&v)[SP_ITEMS]);

__device__ __forceinline__ void tile_ends(TileAhead &a, const int64_t *__restrict__ tile_rows,
                                          int64_t tile, int64_t ntiles) {
  if (tile < ntiles) {
    a.rlo = tile_rows[tile];
    a.rhi = tile_rows[tile + 1];
  }
}

__device__ __forceinline__ void tile_load(TileAhead &a, const int64_t *__restrict__ rowptr,
                                          const int32_t *__restrict__ colidx, int64_t nnz,
                                          int64_t tile, int64_t ntiles, bool aligned) {
  if (tile >= ntiles) return;
  const int64_t first = tile * SP_TILE + (int64_t)threadIdx.x * SP_ITEMS;
  const int64_t t1 = (tile + 1) * SP_TILE < nnz ? (tile + 1) * SP_TILE : nnz;
  const int64_t r = a.rlo + 1 + threadIdx.x;
  a.begin = a.end = 0;
  if (r <= a.rhi) {
    a.begin = rowptr[r];
    a.end = rowptr[r + 1];
  }
  a.start = rowptr[a.rlo];
  a.prev = -1;
  if (first < t1) {
    load_entries(colidx, first, t1, aligned, a.w);
    if ((threadIdx.x & 31) == 0 && first > 0) a.prev = colidx[first - 1];
  } else {
#pragma unroll
    for (int i = 0; i < SP_ITEMS; ++i) a.w[i] = -1;
  }
}

// Marks the tile of entries [t0, t1). Block-wide.
__device__ __forceinline__ void tile_rows_mark(TileRows &tr, const int64_t *__restrict__ rowptr,
                                               int64_t t0, int64_t t1, const TileAhead &a) {
  __syncthreads();  // the tile before this one has been read
  if (threadIdx.x < 64) tr.start[threadIdx.x] = threadIdx.x == 0 ? 1u : 0u;
  if (threadIdx.x == 0) {
    tr.row[0] = (int32_t)a.rlo;  // the row that holds entry t0
    tr.first_is_start = a.start == t0;
  }
  __syncthreads();
  for (int64_t r = a.rlo + 1 + threadIdx.x; r <= a.rhi; r += SP_NT) {
    const bool ahead = r == a.rlo + 1 + threadIdx.x;
    const int64_t b = ahead ? a.begin : rowptr[r], e = ahead ? a.end : rowptr[r + 1];
    if (e > b && b > t0 && b < t1) {  // (row pointers are checked, but only read back later)
      const int x = (int)(b - t0);
      atomicOr(&tr.start[x >> 5], 1u << (x & 31));
      tr.row[x] = (int32_t)r;
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const unsigned lo = __ballot_sync(0xffffffffu, tr.start[threadIdx.x] != 0u);
    const unsigned hi = __ballot_sync(0xffffffffu, tr.start[threadIdx.x + 32] != 0u);
    if (threadIdx.x == 0) tr.words = ((unsigned long long)hi << 32) | lo;
  }
  __syncthreads();
}

// Row of the tile's entry x (x a multiple of 8), and the marks of x .. x + 7.
__device__ __forceinline__ int32_t tile_row_at(const TileRows &tr, int x, unsigned *marks) {
  const int w = x >> 5;
  const uint32_t word = tr.start[w];
  *marks = (word >> (x & 31)) & 0xffu;
  uint32_t below = word & ((2u << (x & 31)) - 1u);  // marks at or before x in its word
  int at = w;
  if (!below) {  // word 0 holds mark 0, so an earlier word has one
    at = 63 - __clzll((long long)(tr.words & ((1ull << w) - 1ull)));
    below = tr.start[at];
  }
  return tr.row[at * 32 + 31 - __clz(below)];
}

// The eight entries of a thread, by two 16-byte loads where they are aligned.
__device__ __forceinline__ void load_entries(const int32_t *__restrict__ colidx, int64_t first,
                                             int64_t t1, bool aligned, int32_t (&v)[SP_ITEMS]) {
  if (aligned && first + SP_ITEMS <= t1) {
    const int4 a = *reinterpret_cast<const int4 *>(colidx + first);
    const int4 b = *reinterpret_cast<const int4 *>(colidx + first + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  } else {
#pragma unroll
    for (int i = 0; i < SP_ITEMS; ++i) v[i] = first + i < t1 ? colidx[first + i] : -1;
  }
}

// a1: one 64-bit key (min << nb) | max per input entry that joins two different
// vertices; the others (and, for symmetric input, entries with u > v) get the
// sentinel, which sorts last. EMIT_BUCKETS: keys times the hash factor go to their
// buckets (see above), whose cursors are `fill`, and the others nowhere. EMIT_COUNT and
// EMIT_PACKED (symmetric input, of which half gives no key): the keys are only counted
// in *cursor, or written one after the other from it, a warp's in one piece.
constexpr int EMIT_ALL = 0, EMIT_BUCKETS = 1, EMIT_COUNT = 2, EMIT_PACKED = 3;
template <int FORM>
__global__ void __launch_bounds__(SP_NT) k_emit_keys(const int64_t *__restrict__ rowptr,
                                                     const int32_t *__restrict__ colidx, int64_t n,
                                                     int64_t nnz, int nb, bool symmetric,
                                                     bool aligned, uint64_t sentinel,
                                                     int lb, unsigned *__restrict__ fill,
                                                     unsigned long long *__restrict__ cursor,
                                                     const int64_t *__restrict__ tile_rows,
                                                     const int64_t *__restrict__ voff, int ng,
                                                     uint64_t *__restrict__ keys,
                                                     int32_t *__restrict__ err) {
  constexpr bool BUCKETS = FORM == EMIT_BUCKETS, WARP = FORM == EMIT_COUNT || FORM == EMIT_PACKED;
  __shared__ TileRows tr;
  const int64_t ntiles = (nnz + SP_TILE - 1) / SP_TILE;
  TileAhead next, after;
  tile_ends(next, tile_rows, blockIdx.x, ntiles);
  tile_load(next, rowptr, colidx, nnz, blockIdx.x, ntiles, aligned);
  tile_ends(after, tile_rows, (int64_t)blockIdx.x + gridDim.x, ntiles);
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const TileAhead here = next;
    next = after;
    tile_load(next, rowptr, colidx, nnz, tile + gridDim.x, ntiles, aligned);
    tile_ends(after, tile_rows, tile + 2 * (int64_t)gridDim.x, ntiles);
    const int64_t t0 = tile * SP_TILE;
    const int64_t t1 = t0 + SP_TILE < nnz ? t0 + SP_TILE : nnz;
    const int64_t first = t0 + (int64_t)threadIdx.x * SP_ITEMS;
    const int32_t(&w)[SP_ITEMS] = here.w;
    tile_rows_mark(tr, rowptr, t0, t1, here);
    if (!WARP && first >= t1) continue;
    // (a bucket has overflowed: only the checks go on)
    const bool given_up =
        BUCKETS && (*reinterpret_cast<volatile unsigned long long *>(cursor) & HASH_FAILED) != 0;
    unsigned marks = 0;
    int32_t u = tile_row_at(tr, (int)threadIdx.x * SP_ITEMS, &marks);
    int gi = 0;
    int64_t gbase = 0, gend = n;
    if (voff) {
      int lo = 0, hi = ng;  // last graph with voff[lo] <= u
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (voff[mid] <= u) lo = mid; else hi = mid;
      }
      gi = lo;
      gbase = voff[gi];
      gend = voff[gi + 1];
    }
    bool bad = false;
    uint64_t key[SP_ITEMS];
#pragma unroll
    for (int i = 0; i < SP_ITEMS; ++i) {
      key[i] = sentinel;
      if (first + i < t1) {
        if (i > 0 && ((marks >> i) & 1u)) u = tr.row[(int)threadIdx.x * SP_ITEMS + i];
        if (voff) {
          while (u >= gend && gi + 1 < ng) {
            ++gi;
            gbase = voff[gi];
            gend = voff[gi + 1];
          }
        }
        const int64_t v = (int64_t)w[i] + gbase;
        if (w[i] < 0 || v >= gend) bad = true;
        else if (v != u && !(symmetric && u > v)) {
          const uint64_t a = (uint64_t)(u < v ? u : v), b = (uint64_t)(u < v ? v : u);
          key[i] = ((a << nb) | b) * (BUCKETS ? HASH_FACTOR : 1ull);
        }
      }
    }
    if (bad) atomicOr(err, 2);
    if (BUCKETS) {
      if (given_up) continue;
#pragma unroll
      for (int i = SP_ITEMS - 1; i > 0; --i)  // copies side by side are dropped here
        if (key[i] == key[i - 1]) key[i] = sentinel;
      unsigned pos[SP_ITEMS];
#pragma unroll
      for (int i = 0; i < SP_ITEMS; ++i)
        pos[i] = key[i] != sentinel ? atomicAdd(&fill[(key[i] >> (64 - lb)) * BK_PAD], 1u) : ~0u;
#pragma unroll
      for (int i = 0; i < SP_ITEMS; ++i) {
        if (pos[i] < (unsigned)BK_CAP) keys[(key[i] >> (64 - lb)) * BK_CAP + pos[i]] = key[i];
        else if (pos[i] == (unsigned)BK_CAP) atomicOr(cursor, HASH_FAILED);
      }
      continue;
    }
    if (WARP) {
      unsigned mine = 0;
#pragma unroll
      for (int i = 0; i < SP_ITEMS; ++i) mine += key[i] != sentinel ? 1u : 0u;
      const unsigned incl = warp_inclusive_scan(mine);
      const unsigned total = __shfl_sync(0xffffffffu, incl, 31);
      unsigned long long at = 0;
      if (lane_id() == 0 && total) at = atomicAdd(cursor, (unsigned long long)total);
      if (FORM == EMIT_COUNT) continue;
      at = __shfl_sync(0xffffffffu, at, 0) + (incl - mine);
#pragma unroll
      for (int i = 0; i < SP_ITEMS; ++i)
        if (key[i] != sentinel) keys[at++] = key[i];
      continue;
    }
    if (first + SP_ITEMS <= t1) {  // keys + first is 64-byte aligned
      ulonglong2 *d = reinterpret_cast<ulonglong2 *>(keys + first);
#pragma unroll
      for (int i = 0; i < SP_ITEMS; i += 2) d[i / 2] = make_ulonglong2(key[i], key[i + 1]);
    } else {
#pragma unroll
      for (int i = 0; i < SP_ITEMS; ++i)
        if (first + i < t1) keys[first + i] = key[i];
    }
  }
}

// In-degrees are later taken to be the degree less the out-degree (flat.cu), which
// holds when every edge is listed under both endpoints. Whether it does is tested by a
// sum mod 2^32 over the upward entries of a term of the rank they point to, less the
// same term times the in-degree for every vertex: 0 when the in-degrees agree, and not
// else but for accidents of 2^-32.
__device__ __forceinline__ uint32_t rank_term(int32_t r) {
  const uint32_t x = (uint32_t)r + 0x9E3779B9u;  // (keeps small ranks from vanishing)
  return x * x;
}

// Passes over the entries of a symmetric CSR, thread t of a tile owning entries
// [8t, 8t + 8). An entry is an edge's first copy when it differs from its row's
// vertex and from the entry before it in the row. The next tile's entries are
// loaded while this one is worked on.
// MODE 0: degree of u -= entries that are no first copy; flag unsorted rows and
// out-of-range ids.
// MODE 1: the ranks of the upward first copies (rank(v) > rank(u)) move to the
// front of u's own entries in `up` (an array like colidx; any order), and
// dplus[u] counts them. The rows are picked up in rank order by the row sort, so
// no second pass over the entries scatters them (it read every entry's stored
// rank and took 0.32 ms on R-MAT scale 21). When there is no room for `up` (null),
// the pass only counts, and a second one with `place` (the rows' offsets by rank)
// writes into the oriented rows themselves. *mirror (nullable) receives the sum of the
// upward entries' rank_term.
// For a batch (voff != nullptr), the entries of a row of graph g are local ids
// in [0, voff[g+1] - voff[g]), shifted here by voff[g].
template <int MODE>
__global__ void __launch_bounds__(SP_NT) k_sym_pass(const int64_t *__restrict__ rowptr,
                                                    const int32_t *__restrict__ colidx, int64_t n,
                                                    int64_t nnz, bool aligned,
                                                    const int64_t *__restrict__ tile_rows,
                                                    int32_t *__restrict__ deg,
                                                    const int32_t *__restrict__ rank,
                                                    unsigned *__restrict__ dplus,
                                                    int32_t *__restrict__ up,
                                                    const int64_t *__restrict__ place,
                                                    unsigned *__restrict__ mirror,
                                                    int32_t *__restrict__ err,
                                                    const int64_t *__restrict__ voff, int ng) {
  __shared__ TileRows tr;
  __shared__ unsigned mirror_s;
  if (MODE == 1 && threadIdx.x == 0) mirror_s = 0;  // (added to after the tiles' barriers)
  uint32_t terms = 0;
  const unsigned lane = threadIdx.x & 31u;
  const int64_t ntiles = (nnz + SP_TILE - 1) / SP_TILE;
  TileAhead next, after;
  tile_ends(next, tile_rows, blockIdx.x, ntiles);
  tile_load(next, rowptr, colidx, nnz, blockIdx.x, ntiles, aligned);
  tile_ends(after, tile_rows, (int64_t)blockIdx.x + gridDim.x, ntiles);
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const TileAhead here = next;
    next = after;
    tile_load(next, rowptr, colidx, nnz, tile + gridDim.x, ntiles, aligned);
    tile_ends(after, tile_rows, tile + 2 * (int64_t)gridDim.x, ntiles);
    const int64_t t0 = tile * SP_TILE;
    const int64_t t1 = t0 + SP_TILE < nnz ? t0 + SP_TILE : nnz;
    const int64_t first = t0 + (int64_t)threadIdx.x * SP_ITEMS;
    const bool mine = first < t1;
    const int32_t(&w)[SP_ITEMS] = here.w;
    tile_rows_mark(tr, rowptr, t0, t1, here);
    unsigned marks = 0;
    int32_t u = mine ? tile_row_at(tr, (int)threadIdx.x * SP_ITEMS, &marks) : 0;
    if (threadIdx.x == 0 && !tr.first_is_start) marks &= ~1u;  // t0 goes on with its row
    int32_t prev = __shfl_up_sync(0xffffffffu, w[SP_ITEMS - 1], 1);
    if (lane == 0) prev = here.prev;
    int gi = 0;
    int64_t gbase = 0, gend = n;
    if (voff && mine) {
      int lo = 0, hi = ng;  // last graph with voff[lo] <= u
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (voff[mid] <= u) lo = mid; else hi = mid;
      }
      gi = lo;
      gbase = voff[gi];
      gend = voff[gi + 1];
    }
    // bit i: entry i is a first copy; by then its row's vertex (as a local id) is ul
    const int32_t size = (int32_t)(gend - gbase);
    int32_t ul = u - (int32_t)gbase;
    unsigned heads = 0, valid = 0, bad = 0;
    int32_t val[SP_ITEMS];
#pragma unroll
    for (int i = 0; i < SP_ITEMS; ++i) {
      const bool starts = ((marks >> i) & 1u) != 0u;
      if (i > 0 && starts) {
        u = tr.row[(int)threadIdx.x * SP_ITEMS + i];
        if (voff) {
          while (u >= gend && gi + 1 < ng) {
            ++gi;
            gbase = voff[gi];
            gend = voff[gi + 1];
          }
        }
        ul = u - (int32_t)gbase;
      }
      const int32_t v = w[i];
      const bool in = first + i < t1;
      const bool in_range = (uint32_t)v < (uint32_t)(voff ? (int32_t)(gend - gbase) : size);
      if (MODE == 0 && in) {
        if (!in_range) bad |= 2u;
        if (!starts && prev > v) bad |= 4u;
      }
      const bool head = in && in_range && v != ul && (starts || prev != v);
      heads |= head ? 1u << i : 0u;
      valid |= in ? 1u << i : 0u;
      if (MODE == 1) val[i] = head ? rank[v + (int32_t)gbase] : -1;
      prev = v;
    }
    if (MODE == 0) {
      if (bad) atomicOr(err, (int)bad);
      // a warp inside one long row (a hub's, where most duplicates are) subtracts once
      const int32_t row0 = mine ? tile_row_at(tr, (int)threadIdx.x * SP_ITEMS, &bad) : -1;
      const int32_t rowx = __shfl_sync(0xffffffffu, row0, 0);
      if (__all_sync(0xffffffffu, !mine || (row0 == rowx && !(marks & ~1u)))) {
        const int none = __reduce_add_sync(0xffffffffu, __popc(valid & ~heads));
        if (lane == 0 && none) atomicSub(&deg[rowx], none);
        continue;
      }
      // entries that are no edge are few: their rows are looked up again
      for (unsigned left = valid & ~heads; left;) {
        const int i = __ffs(left) - 1;
        unsigned unused;
        const int x = (int)threadIdx.x * SP_ITEMS;
        const unsigned before = marks & ((2u << i) - 1u);  // starts up to entry i
        const int32_t r = before && (31 - __clz(before)) > 0
                              ? tr.row[x + 31 - __clz(before)]
                              : tile_row_at(tr, x, &unused);
        // with all others of the same row
        const unsigned later = marks & ~((2u << i) - 1u);
        const unsigned seg = later ? (1u << (__ffs(later) - 1)) - 1u : 0xffu;
        atomicSub(&deg[r], __popc(left & seg));
        left &= ~seg;
      }
      continue;
    }
    // MODE 1: bit i: entry i points up (its row's rank: of the row at hand)
    unsigned ups = 0;
    int32_t urow = mine ? tile_row_at(tr, (int)threadIdx.x * SP_ITEMS, &valid) : 0;
    int32_t ru = mine ? rank[urow] : 0;
    const int32_t row0 = urow;
#pragma unroll
    for (int i = 0; i < SP_ITEMS; ++i) {
      if (i > 0 && ((marks >> i) & 1u)) ru = rank[tr.row[(int)threadIdx.x * SP_ITEMS + i]];
      if (val[i] > ru) {
        ups |= 1u << i;
        terms += rank_term(val[i]);
      }
    }
    const unsigned later0 = marks & ~1u;  // rows that start after the thread's first entry
    // a warp inside one long row (a hub's) reserves once for all its lanes
    const int32_t rowx = __shfl_sync(0xffffffffu, row0, 0);
    if (__all_sync(0xffffffffu, !mine || (row0 == rowx && !later0))) {
      const unsigned cnt = __popc(ups);
      const unsigned incl = warp_inclusive_scan(cnt);
      const unsigned total = __shfl_sync(0xffffffffu, incl, 31);
      if (!total) continue;
      unsigned at = 0;
      if (lane == 0) at = atomicAdd(&dplus[rowx], total);
      at = __shfl_sync(0xffffffffu, at, 0);
      if (!up) continue;
      int64_t pos = (place ? place[rank[rowx]] : rowptr[rowx]) + (int64_t)(at + incl - cnt);
      // (row pointers that decrease are found by the host only after this pass)
      if (!place && !span_inside(pos, cnt, nnz)) continue;
#pragma unroll
      for (int i = 0; i < SP_ITEMS; ++i)
        if ((ups >> i) & 1u) up[pos++] = val[i];
      continue;
    }
    int64_t pos = 0;
#pragma unroll
    for (int i = 0; i < SP_ITEMS; ++i) {
      if (i == 0 || ((marks >> i) & 1u)) {  // a row's first entry here: reserve its slots
        const unsigned later = marks & ~((2u << i) - 1u);
        const unsigned seg = ((later ? (1u << (__ffs(later) - 1)) - 1u : 0xffu)) & ~((1u << i) - 1u);
        const unsigned c = __popc(ups & seg);
        if (c) {
          const int32_t r = i == 0 ? row0 : tr.row[(int)threadIdx.x * SP_ITEMS + i];
          const unsigned at = atomicAdd(&dplus[r], c);
          pos = (place ? place[rank[r]] : rowptr[r]) + (int64_t)at;
        }
      }
      if ((ups >> i) & 1u) {
        if (up && (place || (uint64_t)pos < (uint64_t)nnz)) up[pos] = val[i];  // (as above)
        ++pos;
      }
    }
  }
  if (MODE == 1 && mirror) {
    terms = __reduce_add_sync(0xffffffffu, terms);
    __syncthreads();
    if (lane == 0) atomicAdd(&mirror_s, terms);
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(mirror, mirror_s);
  }
}

// out-degree by position from the out-degree by vertex, and its maximum; the vertices'
// terms are taken off *mirror
__global__ void k_rowlen_by_rank(const unsigned *__restrict__ dplus,
                                 const int32_t *__restrict__ deg,
                                 const int32_t *__restrict__ perm,
                                 const int32_t *__restrict__ rank, int64_t n,
                                 uint64_t *__restrict__ rowlen,
                                 unsigned long long *__restrict__ longest,
                                 unsigned *__restrict__ mirror) {
  unsigned best = 0;
  uint32_t terms = 0;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r <= n;
       r += (int64_t)gridDim.x * blockDim.x) {
    const unsigned d = r < n ? dplus[perm[r]] : 0u;
    rowlen[r] = d;
    best = d > best ? d : best;
    if (r < n) terms += rank_term(rank[r]) * ((unsigned)deg[r] - dplus[r]);  // (r as a vertex)
  }
  best = __reduce_max_sync(0xffffffffu, best);
  terms = __reduce_add_sync(0xffffffffu, terms);
  if ((threadIdx.x & 31) == 0 && best > 0) atomicMax(longest, (unsigned long long)best);
  if ((threadIdx.x & 31) == 0 && terms) atomicSub(mirror, terms);
}

// {largest out-degree, edges, largest degree (that of the last position), error bits,
// what *mirror holds}
__global__ void k_sym_stats(const unsigned long long *__restrict__ longest,
                            const unsigned *__restrict__ mirror,
                            const int64_t *__restrict__ rowptr, const int32_t *__restrict__ deg,
                            const int32_t *__restrict__ perm, int64_t n,
                            const int32_t *__restrict__ err, int64_t *__restrict__ stats) {
  stats[0] = (int64_t)*longest;
  stats[1] = rowptr[n];
  stats[2] = deg[perm[n - 1]];
  stats[3] = *err;
  stats[4] = (int64_t)*mirror;
}

// esrc[x] = the row of position x, for every position of the oriented CSR.
// A warp takes 32 rows: lane j holds the start of row r0 + j, and each
// position of the rows' span finds its row by a search over the lanes, so
// the stores are coalesced whatever the row lengths.
__global__ void k_fill_esrc(const int64_t *__restrict__ rowptr, int64_t n,
                            int32_t *__restrict__ esrc) {
  const unsigned lane = threadIdx.x & 31u;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; r0 < n;
       r0 += nwarps * 32) {
    const int64_t rj = r0 + lane < n ? r0 + lane : n;
    const int64_t start_j = rowptr[rj];
    const int64_t span_end = rowptr[r0 + 32 < n ? r0 + 32 : n];
    const int64_t span_start = __shfl_sync(0xffffffffu, start_j, 0);
    for (int64_t x0 = span_start; x0 < span_end; x0 += 32) {
      const int64_t x = x0 + lane;
      int j = 0;  // last lane whose row starts at or before x
#pragma unroll
      for (int step = 16; step > 0; step >>= 1) {
        const int64_t sj = __shfl_sync(0xffffffffu, start_j, j + step);
        if (sj <= x) j += step;
      }
      if (x < span_end) esrc[x] = (int32_t)(r0 + j);
    }
  }
}

// Oriented keys from the scattered (source, destination) pairs, for graphs
// with rows too long for k_sort_rows: one global sort orders them instead.
__global__ void k_pair_keys(const int32_t *__restrict__ esrc, const int32_t *__restrict__ colidx,
                            int64_t m, int nb, uint64_t *__restrict__ keys) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x)
    keys[e] = ((uint64_t)esrc[e] << nb) | (uint64_t)colidx[e];
}

__global__ void k_pair_unkey(const uint64_t *__restrict__ keys, int64_t m, int nb,
                             const int32_t *__restrict__ err, int32_t *__restrict__ colidx) {
  const uint64_t mask = (1ull << nb) - 1ull;
  if (*err & SORT_FAILED) return;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x)
    colidx[e] = (int32_t)(keys[e] & mask);
}

// Bitonic sort of 32*K values held by a warp in registers: element i of the
// sequence is x[i / 32] of lane i % 32. Exchanges at distance j < 32 go
// through shuffles, those at distance j >= 32 stay within a lane (slots r and
// r ^ j/32).
template <int K>
__device__ __forceinline__ void warp_bitonic(int32_t (&x)[K], unsigned lane) {
  constexpr int S = 32 * K;
#pragma unroll
  for (int k = 2; k <= S; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= 32) {
#pragma unroll
        for (int r = 0; r < K; ++r) {
          const int q = r ^ (j >> 5);
          if (q > r) {
            const bool up = (((int)lane + 32 * r) & k) == 0;
            const int32_t a = x[r], b = x[q];
            const bool swap = up ? (a > b) : (a < b);
            x[r] = swap ? b : a;
            x[q] = swap ? a : b;
          }
        }
      } else {
#pragma unroll
        for (int r = 0; r < K; ++r) {
          const int32_t y = __shfl_xor_sync(0xffffffffu, x[r], j);
          const bool up = (((int)lane + 32 * r) & k) == 0;
          const bool lower = (lane & (unsigned)j) == 0;
          x[r] = (lower == up) ? min(x[r], y) : max(x[r], y);
        }
      }
    }
  }
}

template <int K>
__device__ __forceinline__ void sort_row_regs(const int32_t *in, int32_t *row, int len,
                                              unsigned lane) {
  int32_t x[K];
#pragma unroll
  for (int r = 0; r < K; ++r) {
    const int i = (int)lane + 32 * r;
    x[r] = i < len ? in[i] : INT_MAX;
  }
  warp_bitonic<K>(x, lane);
#pragma unroll
  for (int r = 0; r < K; ++r) {
    const int i = (int)lane + 32 * r;
    if (i < len) row[i] = x[r];
  }
}

// Bitonic network over W values held by one thread (all indices are
// compile-time constants, so the values stay in registers).
template <int W>
__device__ __forceinline__ void thread_bitonic(int32_t (&x)[W]) {
#pragma unroll
  for (int k = 2; k <= W; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll
      for (int i = 0; i < W; ++i) {
        const int l = i ^ j;
        if (l > i) {
          const int32_t a = x[i], b = x[l];
          if ((i & k) == 0) {
            x[i] = min(a, b);
            x[l] = max(a, b);
          } else {
            x[i] = max(a, b);
            x[l] = min(a, b);
          }
        }
      }
    }
  }
}

template <int W>
__device__ __forceinline__ void sort_row_thread(int32_t *__restrict__ row, int len) {
  int32_t x[W];
#pragma unroll
  for (int i = 0; i < W; ++i) x[i] = i < len ? row[i] : INT_MAX;
  thread_bitonic<W>(x);
#pragma unroll
  for (int i = 0; i < W; ++i)
    if (i < len) row[i] = x[i];
}

// Sort every oriented row ascending. A warp takes 32 consecutive rows, whose
// entries are one span of the column array: spans of up to SR_SPAN entries are
// copied to shared memory and back with coalesced accesses (rows dealt to the
// lanes one by one, each at its own place in memory, took 264 us for the 32 M
// entries of R-MAT scale 21); there each lane sorts its own row when it has at
// most 16 entries (a register network of 8 or 16), then the warp sorts the
// longer ones. Longer spans (runs of long rows, which the degree order keeps
// together) are listed for k_sort_long, one warp per row.
constexpr int SR_WARPS = 8;
constexpr int SR_SMALL = 16;
constexpr int SR_SPAN = 1024;

// Sorts one row of up to 1,024 entries (a warp, in registers).
__device__ __forceinline__ void sort_row_warp(const int32_t *in, int32_t *row, int len,
                                              unsigned lane) {
  if (len <= 32) sort_row_regs<1>(in, row, len, lane);
  else if (len <= 64) sort_row_regs<2>(in, row, len, lane);
  else if (len <= 128) sort_row_regs<4>(in, row, len, lane);
  else if (len <= 256) sort_row_regs<8>(in, row, len, lane);
  else if (len <= 512) sort_row_regs<16>(in, row, len, lane);
  else sort_row_regs<32>(in, row, len, lane);
}

// Where row r's unsorted entries lie: in place, or at start[perm[r]] of src.
struct RowSource {
  const int32_t *src;
  const int64_t *start;  // nullptr: in place
  const int32_t *perm;
};

// esrc (nullable) receives each entry's row.
__global__ void __launch_bounds__(SR_WARPS * 32) k_sort_rows(const int64_t *__restrict__ rowptr,
                                                             int64_t n, RowSource from,
                                                             int32_t *colidx,
                                                             int32_t *__restrict__ esrc,
                                                             int32_t *__restrict__ listed,
                                                             unsigned *__restrict__ nlisted) {
  __shared__ int32_t buf[SR_WARPS][SR_SPAN];
  const unsigned lane = threadIdx.x & 31u;
  int32_t *sm = buf[threadIdx.x >> 5];
  const int64_t nblk = (n + 31) >> 5;
  for (int64_t blk = ((int64_t)blockIdx.x * (SR_WARPS * 32) + threadIdx.x) >> 5; blk < nblk;
       blk += ((int64_t)gridDim.x * (SR_WARPS * 32)) >> 5) {
    const int64_t r = blk * 32 + lane;
    const int64_t b = rowptr[r < n ? r : n], e = rowptr[r + 1 < n ? r + 1 : n];
    const int len = (int)(e - b);
    const int64_t s0 = __shfl_sync(0xffffffffu, b, 0), s1 = __shfl_sync(0xffffffffu, e, 31);
    if (s1 == s0 || (!from.start && !esrc && __all_sync(0xffffffffu, len <= 1))) continue;
    if (s1 - s0 > SR_SPAN) {
      if (lane == 0) listed[atomicAdd(nlisted, 1u)] = (int32_t)blk;
      continue;
    }
    const int span = (int)(s1 - s0), at = (int)(b - s0);
    // offset of the lane's row in the source, from its place in the span
    const int64_t shift = from.start && len > 0 ? from.start[from.perm[r]] - at : s0;
    for (int i0 = 0; i0 < span; i0 += 32) {
      const int i = i0 + (int)lane;
      int j = 0;  // last lane whose row starts at or before i
#pragma unroll
      for (int step = 16; step > 0; step >>= 1) {
        const int aj = __shfl_sync(0xffffffffu, at, j + step);
        if (aj <= i) j += step;
      }
      const int64_t sh = __shfl_sync(0xffffffffu, shift, j);
      if (i < span) {
        sm[i] = from.src[sh + i];
        if (esrc) esrc[s0 + i] = (int32_t)(blk * 32 + j);
      }
    }
    __syncwarp();
    const bool small = len > 1 && len <= SR_SMALL;
    const int small_max = __reduce_max_sync(0xffffffffu, small ? len : 0);
    if (small_max > 8) {
      if (small) sort_row_thread<16>(sm + at, len);
    } else if (small_max > 0) {
      if (small) sort_row_thread<8>(sm + at, len);
    }
    __syncwarp();
    unsigned big = __ballot_sync(0xffffffffu, len > SR_SMALL);
    while (big) {
      const int src = __ffs(big) - 1;
      big &= big - 1;
      int32_t *row = sm + __shfl_sync(0xffffffffu, at, src);
      sort_row_warp(row, row, __shfl_sync(0xffffffffu, len, src), lane);
    }
    __syncwarp();
    for (int i = lane; i < span; i += 32) colidx[s0 + i] = sm[i];
    __syncwarp();
  }
}

// The rows of the listed blocks of 32, one warp per row: up to 1,024 entries in
// registers (bitonic network over shuffles and register slots, padded to
// 32 * 2^t), longer ones (up to SEG_CAP) in the warp's shared memory.
constexpr int SL_WARPS = 4;
__global__ void __launch_bounds__(SL_WARPS * 32) k_sort_long(const int64_t *__restrict__ rowptr,
                                                             int64_t n, RowSource from,
                                                             int32_t *colidx,
                                                             int32_t *__restrict__ esrc,
                                                             const int32_t *__restrict__ listed,
                                                             const unsigned *__restrict__ nlisted) {
  __shared__ int32_t buf[SL_WARPS][SEG_CAP];
  const unsigned lane = threadIdx.x & 31u;
  int32_t *sm = buf[threadIdx.x >> 5];
  const int64_t total = (int64_t)*nlisted * 32;
  for (int64_t x = (int64_t)blockIdx.x * SL_WARPS + (threadIdx.x >> 5); x < total;
       x += (int64_t)gridDim.x * SL_WARPS) {
    const int64_t r = (int64_t)listed[x >> 5] * 32 + (x & 31);
    if (r >= n) continue;
    const int64_t b = rowptr[r];
    const int len = (int)(rowptr[r + 1] - b);
    if (len <= 0) continue;
    int32_t *row = colidx + b;
    const int32_t *in = from.start ? from.src + from.start[from.perm[r]] : row;
    if (esrc)
      for (int i = lane; i < len; i += 32) esrc[b + i] = (int32_t)r;
    if (len <= 1024) {
      sort_row_warp(in, row, len, lane);
      continue;
    }
    int size = 2048;
    while (size < len) size <<= 1;
    for (int i = lane; i < size; i += 32) sm[i] = i < len ? in[i] : INT_MAX;
    __syncwarp();
    for (int k = 2; k <= size; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int i = lane; i < size; i += 32) {
          const int l = i ^ j;
          if (l > i) {
            const int32_t a = sm[i], c = sm[l];
            const bool up = (i & k) == 0;
            if ((a > c) == up) {
              sm[i] = c;
              sm[l] = a;
            }
          }
        }
        __syncwarp();
      }
    for (int i = lane; i < len; i += 32) row[i] = sm[i];
    __syncwarp();
  }
}

// Rows too long for k_sort_long: entries and their rows moved to their places,
// unsorted (one warp per row).
__global__ void k_gather_rows(const int64_t *__restrict__ rowptr, int64_t n, RowSource from,
                              int32_t *__restrict__ colidx, int32_t *__restrict__ esrc) {
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n; r += nwarps) {
    const int64_t b = rowptr[r], len = rowptr[r + 1] - b;
    if (len <= 0) continue;
    const int32_t *in = from.src + from.start[from.perm[r]];
    for (int64_t i = threadIdx.x & 31; i < len; i += 32) {
      colidx[b + i] = in[i];
      esrc[b + i] = (int32_t)r;
    }
  }
}

// ------------------------------------------------------------------------
// Graphs of up to 1,024 vertices: the whole preparation in one CTA, whose shared
// memory holds the adjacency matrix as bits. Setting bits takes any input form
// (one or both directions, any order, duplicates) and removes duplicates by
// itself, degrees are population counts, and a row's upward neighbours, set
// again by rank, come out sorted. What bounds such a graph is launches and
// round trips to the host, not work: R-MAT scale 10 took 13 kernels and 4
// synchronisations here (about 180 us), and takes one of each.
constexpr int SG_N = 1024;
constexpr int64_t SG_ENTRIES = 1 << 17;  // input entries of one CTA at most
constexpr int SG_NT = 1024;

struct SmallSmem {
  uint32_t bits[SG_N][SG_N / 32 + 1];  // (rows of 33 words: a column's words lie in 32 banks)
  uint32_t row[SG_N + 1];     // input row pointers
  int32_t rank[SG_N];
  uint32_t sort[SG_N];        // exchange buffer of the sort, then out-degrees by rank
  uint32_t scan_tmp[SG_NT / 32 + 1];
  int32_t err, dmax, dpmax;
};

// stats: {m, largest out-degree, largest degree, error bits as in the passes above}
__global__ void __launch_bounds__(SG_NT) k_small_graph(const int64_t *__restrict__ rowptr,
                                                       const int32_t *__restrict__ colidx, int n,
                                                       int nnz, bool symmetric,
                                                       int32_t *__restrict__ deg,
                                                       int32_t *__restrict__ perm,
                                                       int64_t *__restrict__ rowptr_o,
                                                       int32_t *__restrict__ colidx_o,
                                                       int32_t *__restrict__ esrc,
                                                       int64_t *__restrict__ stats) {
  extern __shared__ __align__(16) unsigned char small_smem[];
  SmallSmem &sm = *reinterpret_cast<SmallSmem *>(small_smem);
  const int t = threadIdx.x, warp = t >> 5;
  const unsigned lane = t & 31u;
  if (t == 0) sm.err = sm.dmax = sm.dpmax = 0;
  auto clear = [&]() {
    for (int i = t; i < SG_N * (SG_N / 32 + 1); i += SG_NT) (&sm.bits[0][0])[i] = 0;
  };
  clear();
  __syncthreads();
  {
    // row pointers, checked and clamped into the entries
    const int64_t b = t < n ? rowptr[t] : 0, e = t < n ? rowptr[t + 1] : 0;
    if (b > e || (t == 0 && b != 0)) atomicOr(&sm.err, 1);
    if (t < n) sm.row[t] = (uint32_t)(b < 0 ? 0 : b > nnz ? nnz : b);
    if (t == n - 1) sm.row[n] = (uint32_t)nnz;
  }
  __syncthreads();
  // every entry (u, v) that may be an edge
  auto entries = [&](auto edge) {
    for (int e0 = t; e0 < nnz; e0 += 4 * SG_NT) {
      int32_t v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = e0 + i * SG_NT < nnz ? colidx[e0 + i * SG_NT] : -1;
      int lo[4] = {0, 0, 0, 0};  // last row that starts at or before the entry
      for (int step = SG_N / 2; step > 0; step >>= 1)
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (lo[i] + step < n && sm.row[lo[i] + step] <= (uint32_t)(e0 + i * SG_NT)) lo[i] += step;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (e0 + i * SG_NT < nnz) {
          if (v[i] < 0 || v[i] >= n) atomicOr(&sm.err, 2);
          else if (v[i] != lo[i] && (!symmetric || lo[i] < v[i])) edge(lo[i], v[i]);
        }
    }
  };
  entries([&](int u, int v) {
    atomicOr(&sm.bits[u][v >> 5], 1u << (v & 31));
    atomicOr(&sm.bits[v][u >> 5], 1u << (u & 31));
  });
  __syncthreads();
  for (int u = warp; u < SG_N; u += SG_NT / 32) {
    const int d = __reduce_add_sync(0xffffffffu, __popc(sm.bits[u][lane]));
    if (lane == 0) {
      sm.sort[u] = u < n ? ((uint32_t)d << 10) | (uint32_t)u : 0xffffffffu;
      if (u < n) deg[u] = d;
      if (d > 0) atomicMax(&sm.dmax, d);
    }
  }
  __syncthreads();
  // order by (degree, id): bitonic sort, one key per thread
  uint32_t x = sm.sort[t];
  for (int k = 2; k <= SG_N; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      uint32_t y;
      if (j >= 32) {
        __syncthreads();
        sm.sort[t] = x;
        __syncthreads();
        y = sm.sort[t ^ j];
      } else {
        y = __shfl_xor_sync(0xffffffffu, x, j);
      }
      const bool up = (t & k) == 0, lower = (t & j) == 0;
      x = (lower == up) ? min(x, y) : max(x, y);
    }
  __syncthreads();
  if (t < n) {
    const int32_t v = (int32_t)(x & 1023u);
    sm.rank[v] = t;
    perm[t] = v;
  }
  __syncthreads();
  // the same entries again, as upward neighbours by rank
  clear();
  __syncthreads();
  entries([&](int u, int v) {
    const int ru = sm.rank[u], rv = sm.rank[v];
    const int a = min(ru, rv), b = max(ru, rv);
    atomicOr(&sm.bits[a][b >> 5], 1u << (b & 31));
  });
  __syncthreads();
  for (int r = warp; r < SG_N; r += SG_NT / 32) {
    const int d = __reduce_add_sync(0xffffffffu, __popc(sm.bits[r][lane]));
    if (lane == 0) {
      sm.sort[r] = (uint32_t)d;
      if (d > 0) atomicMax(&sm.dpmax, d);
    }
  }
  __syncthreads();
  uint32_t m = 0;
  const uint32_t at = block_exclusive_scan<uint32_t, SG_NT>(sm.sort[t], sm.scan_tmp, &m);
  sm.sort[t] = at;
  if (t < n) rowptr_o[t] = (int64_t)at;
  if (t == 0) {
    rowptr_o[n] = (int64_t)m;
    stats[0] = (int64_t)m;
    stats[1] = sm.dpmax;
    stats[2] = sm.dmax;
    stats[3] = sm.err;
  }
  __syncthreads();
  for (int r = warp; r < n; r += SG_NT / 32) {
    const uint32_t word = sm.bits[r][lane];
    uint32_t pos = sm.sort[r];
    // one word at a time, a lane per bit
    for (unsigned left = __ballot_sync(0xffffffffu, word != 0u); left; left &= left - 1) {
      const int w = __ffs(left) - 1;
      const uint32_t x = __shfl_sync(0xffffffffu, word, w);
      if ((x >> lane) & 1u) {
        const uint32_t o = pos + __popc(x & ((1u << lane) - 1u));
        colidx_o[o] = w * 32 + (int)lane;
        esrc[o] = r;
      }
      pos += __popc(x);
    }
  }
}

}  // namespace

// Sorts every row of an oriented CSR whose rows have at most SEG_CAP entries
// into colidx, and writes each entry's row.
static bbtc_status sort_rows(const int64_t *rowptr, int64_t n, const RowSource &from,
                             int32_t *colidx, int32_t *esrc, cudaStream_t s) {
  Scratch scratch(s);
  int32_t *listed = nullptr;
  unsigned *nlisted = nullptr;
  BBTC_TRY(scratch.get(&listed, (n + 31) / 32));
  BBTC_TRY(scratch.get(&nlisted, 1));
  BBTC_CUDA(cudaMemsetAsync(nlisted, 0, sizeof(unsigned), s));
  k_sort_rows<<<grid_for((n + 31) / 32, SR_WARPS, 7), SR_WARPS * 32, 0, s>>>(
      rowptr, n, from, colidx, esrc, listed, nlisted);
  BBTC_LAUNCH_CHECK();
  k_sort_long<<<grid_for((n + 31) / 32, 1, 7), SL_WARPS * 32, 0, s>>>(rowptr, n, from, colidx,
                                                                     esrc, listed, nlisted);
  BBTC_LAUNCH_CHECK();
  return BBTC_OK;
}

// a1-a4 for symmetric input with sorted rows. Sets *applied = false (and does
// nothing lasting) when some row turns out unsorted, or some edge turns out to be
// listed under one endpoint only.
static bbtc_status prepare_sym_sorted(bbtc_graph *g, const int64_t *d_rowptr,
                                      const int32_t *d_colidx, int64_t nnz, int32_t *err,
                                      bool *applied) {
  cudaStream_t s = g->stream;
  const int64_t n = g->n;
  const int nb = g->nb;
  *applied = false;
  Scratch scratch(s);
  BBTC_TRY(dalloc_n(&g->deg, n, s));
  g->bytes += (uint64_t)(n > 0 ? n : 1) * sizeof(int32_t);
  k_validate_rowptr<<<grid_for(n, 256, 8), 256, 0, s>>>(d_rowptr, n, g->deg, err);
  BBTC_LAUNCH_CHECK();
  const bool aligned = (reinterpret_cast<uintptr_t>(d_colidx) & 15u) == 0;  // the caller's array
  const int64_t ntiles = (nnz + SP_TILE - 1) / SP_TILE;
  int64_t *tile_rows = nullptr;
  BBTC_TRY(scratch.get(&tile_rows, ntiles + 1));
  k_tile_rows<<<grid_for(ntiles + 1, 256, 16), 256, 0, s>>>(d_rowptr, n, nnz, ntiles, tile_rows);
  BBTC_LAUNCH_CHECK();
  const unsigned grid = grid_for(ntiles, 1, 32);
  k_sym_pass<0><<<grid, SP_NT, 0, s>>>(d_rowptr, d_colidx, n, nnz, aligned, tile_rows, g->deg,
                                       nullptr, nullptr, nullptr, nullptr, nullptr, err, g->voff,
                                       g->ng);
  BBTC_LAUNCH_CHECK();
  int32_t herr = 0, hdmax = 0;
  // what pass 0 found in the input: BBTC_OK and *sorted, or the error
  auto check = [&](bool *sorted) -> bbtc_status {
    if (herr & 1) {
      set_error("bbtc_graph_create: rowptr[0] != 0 or rowptr decreases");
      return BBTC_EINVAL;
    }
    if (herr & 2) {
      set_error("bbtc_graph_create: colidx entry outside [0, n)");
      return BBTC_EINVAL;
    }
    *sorted = (herr & 4) == 0;
    return BBTC_OK;
  };
  bool sorted_rows = true;
  // The sort of the ranks needs as many bits as the largest degree has. A graph of
  // many vertices asks the device; for the others sorting the bits of n costs less
  // than the round trip (about 25 us), and what pass 0 found is read with the sizes.
  int degree_bits = nb;
  const bool ask = n > SYM_ASK_N;
  if (ask) {
    int32_t *dmax = nullptr;
    BBTC_TRY(scratch.get(&dmax, 1));
    BBTC_TRY(reduce_max_i32(g->deg, n, dmax, s));
    BBTC_CUDA(cudaMemcpyAsync(&hdmax, dmax, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    BBTC_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    BBTC_CUDA(cudaStreamSynchronize(s));
    BBTC_TRY(check(&sorted_rows));
    if (!sorted_rows) return BBTC_OK;  // the general path takes over
    degree_bits = ceil_log2_u64((uint64_t)hdmax + 1);
  }

  // a3: order by (degree, id)
  int32_t *rank = nullptr;
  uint64_t *rk = nullptr, *rk_alt = nullptr;
  BBTC_TRY(scratch.get(&rank, n));
  BBTC_TRY(scratch.get(&rk, n));
  BBTC_TRY(scratch.get(&rk_alt, n));
  BBTC_TRY(dalloc_n(&g->perm, n, s));
  g->bytes += (uint64_t)n * sizeof(int32_t);
  k_rank_keys<<<grid_for(n, 256, 16), 256, 0, s>>>(g->deg, n, nb, rk);
  BBTC_LAUNCH_CHECK();
  bool in_alt = false;
  // the keys start in id order and the sort is stable: only the degree bits are sorted
  BBTC_TRY(radix_sort(rk, rk_alt, nullptr, nullptr, n, nb, nb + degree_bits, s, err, &in_alt));
  k_rank_finish<<<grid_for(n, 256, 16), 256, 0, s>>>(in_alt ? rk_alt : rk, n, nb, err, g->perm,
                                                      rank);
  BBTC_LAUNCH_CHECK();
  if (g->voff) {
    BBTC_TRY(dalloc_n(&g->gid, n, s));
    g->bytes += (uint64_t)n * sizeof(int32_t);
    k_graph_of_position<<<grid_for(n, 256, 16), 256, 0, s>>>(g->perm, n, g->voff, g->ng, g->gid);
    BBTC_LAUNCH_CHECK();
  }

  // a4: each row's upward entries to its front, out-degrees by rank, offsets, and
  // the rows picked up in rank order and sorted
  BBTC_TRY(dalloc_n(&g->rowptr, n + 1, s));
  g->bytes += (uint64_t)(n + 1) * 8;
  int32_t *up = nullptr;
  unsigned *dplus = nullptr;
  unsigned long long *longest = nullptr;
  BBTC_TRY(scratch.get(&dplus, n));
  BBTC_TRY(scratch.get(&longest, 2));
  unsigned *mirror = reinterpret_cast<unsigned *>(longest + 1);
  if (dalloc_n(&up, nnz, s) != BBTC_OK) {  // no room: the rows are written in a second pass
    clear_error();
    up = nullptr;
  }
  struct FreeUp {
    int32_t *p;
    cudaStream_t s;
    ~FreeUp() { dfree(p, s); }
  } free_up{up, s};
  BBTC_CUDA(cudaMemsetAsync(dplus, 0, sizeof(unsigned) * (size_t)n, s));
  BBTC_CUDA(cudaMemsetAsync(longest, 0, 2 * sizeof(unsigned long long), s));
  k_sym_pass<1><<<grid, SP_NT, 0, s>>>(d_rowptr, d_colidx, n, nnz, aligned, tile_rows, nullptr, rank,
                                       dplus, up, nullptr, mirror, err, g->voff, g->ng);
  BBTC_LAUNCH_CHECK();
  k_rowlen_by_rank<<<grid_for(n + 1, 256, 16), 256, 0, s>>>(
      dplus, g->deg, g->perm, rank, n, reinterpret_cast<uint64_t *>(g->rowptr), longest, mirror);
  BBTC_LAUNCH_CHECK();
  BBTC_TRY(exclusive_scan_u64(reinterpret_cast<uint64_t *>(g->rowptr),
                              reinterpret_cast<uint64_t *>(g->rowptr), n + 1, s));
  int64_t *stats = nullptr;
  BBTC_TRY(scratch.get(&stats, 5));
  k_sym_stats<<<1, 1, 0, s>>>(longest, mirror, g->rowptr, g->deg, g->perm, n, err, stats);
  BBTC_LAUNCH_CHECK();
  int64_t h[5] = {0, 0, 0, 0, 0};
  BBTC_CUDA(cudaMemcpyAsync(h, stats, sizeof(h), cudaMemcpyDeviceToHost, s));
  BBTC_CUDA(cudaStreamSynchronize(s));
  herr = (int32_t)h[3];
  BBTC_TRY(check(&sorted_rows));
  if (herr & SORT_FAILED) return sort_failed("bbtc_graph_create");
  // the general path takes over: it reads the entries u < v whatever the others say
  if (!sorted_rows || h[4] != 0) {
    dfree(g->perm, s);
    dfree(g->rowptr, s);
    dfree(g->gid, s);
    g->perm = nullptr;
    g->rowptr = nullptr;
    if (g->gid) g->bytes -= (uint64_t)n * sizeof(int32_t);
    g->gid = nullptr;
    g->bytes -= (uint64_t)n * sizeof(int32_t) + (uint64_t)(n + 1) * 8;
    return BBTC_OK;
  }
  *applied = true;
  g->deg_max = h[2];
  g->dplus_max = h[0];
  const int64_t m = h[1];
  if (m > 0xFFFFFFFFLL) {
    set_error("bbtc_graph_create: %lld simple edges exceed 2^32 - 1", (long long)m);
    return BBTC_EINVAL;
  }
  g->m = m;
  BBTC_TRY(dalloc_n(&g->colidx, padded_columns(m), s));
  BBTC_TRY(dalloc_n(&g->esrc, m, s));
  g->bytes += (uint64_t)(m > 0 ? m : 1) * 8;
  if (!up && m > 0) {
    BBTC_CUDA(cudaMemsetAsync(dplus, 0, sizeof(unsigned) * (size_t)n, s));
    k_sym_pass<1><<<grid, SP_NT, 0, s>>>(d_rowptr, d_colidx, n, nnz, aligned, tile_rows, nullptr,
                                         rank, dplus, g->colidx, g->rowptr, nullptr, err, g->voff,
                                         g->ng);
    BBTC_LAUNCH_CHECK();
  }
  const RowSource from = up ? RowSource{up, d_rowptr, g->perm}
                            : RowSource{g->colidx, nullptr, nullptr};
  if (m > 0 && g->dplus_max <= SEG_CAP) {
    BBTC_TRY(sort_rows(g->rowptr, n, from, g->colidx, g->esrc, s));
  } else if (m > 0) {
    if (up) k_gather_rows<<<grid_for(n * 32, 256, 16), 256, 0, s>>>(g->rowptr, n, from, g->colidx, g->esrc);
    else k_fill_esrc<<<grid_for((n + 31) / 32 * 32, 256, 16), 256, 0, s>>>(g->rowptr, n, g->esrc);
    BBTC_LAUNCH_CHECK();
    uint64_t *ok = nullptr, *ok_alt = nullptr;
    BBTC_TRY(scratch.get(&ok, m));
    BBTC_TRY(scratch.get(&ok_alt, m));
    k_pair_keys<<<grid_for(m, 256, 32), 256, 0, s>>>(g->esrc, g->colidx, m, nb, ok);
    BBTC_LAUNCH_CHECK();
    BBTC_TRY(radix_sort(ok, ok_alt, nullptr, nullptr, m, 0, 2 * nb, s, err, &in_alt));
    k_pair_unkey<<<grid_for(m, 256, 32), 256, 0, s>>>(in_alt ? ok_alt : ok, m, nb, err, g->colidx);
    BBTC_LAUNCH_CHECK();
    BBTC_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    BBTC_CUDA(cudaStreamSynchronize(s));
    if (herr & SORT_FAILED) return sort_failed("bbtc_graph_create");
  }
  return BBTC_OK;
}

// a1-a4 of a small graph in one kernel.
static bbtc_status prepare_small(bbtc_graph *g, const int64_t *d_rowptr, const int32_t *d_colidx,
                                 int64_t nnz, bool symmetric) {
  cudaStream_t s = g->stream;
  const int64_t n = g->n;
  // an entry gives at most one edge
  const int64_t room = nnz < n * (n - 1) / 2 ? nnz : n * (n - 1) / 2;
  Scratch scratch(s);
  int64_t *stats = nullptr;
  BBTC_TRY(scratch.get(&stats, 4));
  BBTC_TRY(dalloc_n(&g->deg, n, s));
  BBTC_TRY(dalloc_n(&g->perm, n, s));
  BBTC_TRY(dalloc_n(&g->rowptr, n + 1, s));
  BBTC_TRY(dalloc_n(&g->colidx, padded_columns(room), s));
  BBTC_TRY(dalloc_n(&g->esrc, room, s));
  g->bytes += (uint64_t)n * 8 + (uint64_t)(n + 1) * 8 + (uint64_t)room * 8;
  BBTC_CUDA(cudaFuncSetAttribute(k_small_graph, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(SmallSmem)));
  k_small_graph<<<1, SG_NT, sizeof(SmallSmem), s>>>(d_rowptr, d_colidx, (int)n, (int)nnz, symmetric,
                                                    g->deg, g->perm, g->rowptr, g->colidx, g->esrc,
                                                    stats);
  BBTC_LAUNCH_CHECK();
  int64_t h[4] = {0, 0, 0, 0};
  BBTC_CUDA(cudaMemcpyAsync(h, stats, sizeof(h), cudaMemcpyDeviceToHost, s));
  BBTC_CUDA(cudaStreamSynchronize(s));
  if (h[3] & 1) {
    set_error("bbtc_graph_create: rowptr[0] != 0 or rowptr decreases");
    return BBTC_EINVAL;
  }
  if (h[3] & 2) {
    set_error("bbtc_graph_create: colidx entry outside [0, n)");
    return BBTC_EINVAL;
  }
  g->m = h[0];
  g->dplus_max = h[1];
  g->deg_max = h[2];
  return BBTC_OK;
}

// a1-a4 for any input: distinct keys by hashing (by_hash) or by sorting. *again: the
// keys did not go into their buckets, and nothing has been kept but g->deg.
static bbtc_status prepare_general(bbtc_graph *g, const int64_t *d_rowptr, const int32_t *d_colidx,
                                   int64_t nnz, bool symmetric, bool by_hash, bool *again) {
  cudaStream_t s = g->stream;
  const int64_t n = g->n;
  const int nb = g->nb;
  Scratch scratch(s);
  int32_t *err = nullptr;
  int64_t *hstats = nullptr;  // device: [0]=m, [1]=deg_max
  BBTC_TRY(scratch.get(&err, 1));
  BBTC_TRY(scratch.get(&hstats, 3));
  BBTC_CUDA(cudaMemsetAsync(err, 0, sizeof(int32_t), s));

  // ---- validation of rowptr (colidx range is checked while emitting keys)
  if (n > 0) {
    k_validate_rowptr<<<grid_for(n, 256, 8), 256, 0, s>>>(d_rowptr, n, nullptr, err);
    BBTC_LAUNCH_CHECK();
  }
  auto check = [&](int32_t herr) -> bbtc_status {
    if (herr & 1) {
      set_error("bbtc_graph_create: rowptr[0] != 0 or rowptr decreases");
      return BBTC_EINVAL;
    }
    if (herr & 2) {
      set_error("bbtc_graph_create: colidx entry outside [0, n)");
      return BBTC_EINVAL;
    }
    return herr & SORT_FAILED ? sort_failed("bbtc_graph_create") : BBTC_OK;
  };

  // ---- a1: canonical keys, the distinct ones; a2: degree
  // (no key equals the all-ones value: it would need min == max)
  const uint64_t sentinel =
      by_hash ? HASH_EMPTY : (nb * 2 >= 64) ? ~0ull : ((1ull << (2 * nb)) - 1ull);
  const bool aligned = (reinterpret_cast<uintptr_t>(d_colidx) & 15u) == 0;
  const int64_t ntiles = (nnz + SP_TILE - 1) / SP_TILE;
  const unsigned grid = grid_for(ntiles, 1, 32);
  int64_t *tile_rows = nullptr;
  if (nnz > 0) {
    BBTC_TRY(scratch.get(&tile_rows, ntiles + 1));
    k_tile_rows<<<grid_for(ntiles + 1, 256, 16), 256, 0, s>>>(d_rowptr, n, nnz, ntiles, tile_rows);
    BBTC_LAUNCH_CHECK();
  }
  unsigned long long *nunique = reinterpret_cast<unsigned long long *>(&hstats[0]);
  BBTC_CUDA(cudaMemsetAsync(nunique, 0, sizeof(*nunique), s));
  // Keys that are expected: every entry gives one, of symmetric input every second. The
  // buckets find out whether that holds; a sort has them counted first, since it would
  // sort (and hold, twice) as many again as there are.
  int64_t nkeys = symmetric ? nnz / 2 : nnz;
  int32_t herr = 0;
  if (!by_hash && symmetric && nnz > 0) {
    k_emit_keys<EMIT_COUNT><<<grid, SP_NT, 0, s>>>(d_rowptr, d_colidx, n, nnz, nb, symmetric,
                                                   aligned, sentinel, 0, nullptr, nunique,
                                                   tile_rows, g->voff, g->ng, nullptr, err);
    BBTC_LAUNCH_CHECK();
    BBTC_CUDA(cudaMemcpyAsync(&nkeys, nunique, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    BBTC_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    BBTC_CUDA(cudaStreamSynchronize(s));
    BBTC_TRY(check(herr));
    BBTC_CUDA(cudaMemsetAsync(nunique, 0, sizeof(*nunique), s));
  }
  const int64_t kcap = nkeys > n ? nkeys : n;  // the buffers also take the n rank keys
  uint64_t *ka = nullptr, *kb = nullptr, *sorted = nullptr, *ukeys = nullptr;
  bool in_alt = false;
  BBTC_TRY(scratch.get(&kb, kcap));
  int lb = 1;
  unsigned *fill = nullptr;
  if (by_hash) {
    while ((nkeys >> lb) > BK_MEAN) ++lb;
    const int64_t cap = (int64_t)BK_CAP << lb;
    BBTC_TRY(scratch.get(&fill, (int64_t)BK_PAD << lb));
    BBTC_TRY(scratch.get(&ka, cap > kcap ? cap : kcap));
  } else {
    BBTC_TRY(scratch.get(&ka, kcap));
  }
  // (allocated after the key buffers: in front of them, among the small blocks, the
  // additions to the degrees made k_bucket_unique take 432 us instead of 389 for R-MAT
  // scale 20)
  if (!g->deg) {
    BBTC_TRY(dalloc_n(&g->deg, n, s));
    g->bytes += (uint64_t)(n > 0 ? n : 1) * sizeof(int32_t);
  }
  BBTC_CUDA(cudaMemsetAsync(g->deg, 0, sizeof(int32_t) * (size_t)(n > 0 ? n : 1), s));
  if (by_hash) {
    BBTC_CUDA(cudaMemsetAsync(fill, 0, (sizeof(unsigned) * BK_PAD) << lb, s));
    k_emit_keys<EMIT_BUCKETS><<<grid, SP_NT, 0, s>>>(d_rowptr, d_colidx, n, nnz, nb, symmetric,
                                                     aligned, sentinel, lb, fill, nunique,
                                                     tile_rows, g->voff, g->ng, ka, err);
    BBTC_LAUNCH_CHECK();
    k_bucket_unique<<<1u << lb, BK_NT, 0, s>>>(ka, fill, lb, nb, kcap, kb, nunique, g->deg);
    BBTC_LAUNCH_CHECK();
  } else {
    if (symmetric && nkeys > 0)
      k_emit_keys<EMIT_PACKED><<<grid, SP_NT, 0, s>>>(d_rowptr, d_colidx, n, nnz, nb, symmetric,
                                                      aligned, sentinel, 0, nullptr, nunique,
                                                      tile_rows, g->voff, g->ng, ka, err);
    else if (nkeys > 0)
      k_emit_keys<EMIT_ALL><<<grid, SP_NT, 0, s>>>(d_rowptr, d_colidx, n, nnz, nb, symmetric,
                                                   aligned, sentinel, 0, nullptr, nullptr,
                                                   tile_rows, g->voff, g->ng, ka, err);
    if (nkeys > 0) BBTC_LAUNCH_CHECK();
    BBTC_TRY(radix_sort(ka, kb, nullptr, nullptr, nkeys, 0, 2 * nb, s, err, &in_alt));
  }
  sorted = in_alt ? kb : ka;
  ukeys = in_alt ? ka : kb;
  if (!by_hash) {
    BBTC_CUDA(cudaMemsetAsync(nunique, 0, sizeof(*nunique), s));
    if (nkeys > 0) {
      const int64_t nblk = (nkeys + UQ_TILE - 1) / UQ_TILE;
      uint64_t *boff = nullptr;
      BBTC_TRY(scratch.get(&boff, nblk + 1));
      k_unique_count<<<(unsigned)nblk, UQ_NT, 0, s>>>(sorted, nkeys, sentinel, err, boff);
      BBTC_LAUNCH_CHECK();
      BBTC_TRY(exclusive_scan_u64(boff, boff, nblk + 1, s));  // boff[nblk] = total
      k_unique_write<<<(unsigned)nblk, UQ_NT, 0, s>>>(sorted, nkeys, sentinel, err, boff, nb,
                                                       ukeys, g->deg);
      BBTC_LAUNCH_CHECK();
      BBTC_CUDA(
          cudaMemcpyAsync(nunique, &boff[nblk], sizeof(int64_t), cudaMemcpyDeviceToDevice, s));
    }
  }
  int32_t *dmax = nullptr;
  int32_t hdmax = 0;
  int64_t stats[2] = {0, 0};
  BBTC_TRY(scratch.get(&dmax, 1));
  BBTC_TRY(reduce_max_i32(g->deg, n, dmax, s));
  BBTC_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  BBTC_CUDA(cudaMemcpyAsync(&stats[0], nunique, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  BBTC_CUDA(cudaMemcpyAsync(&hdmax, dmax, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  BBTC_CUDA(cudaStreamSynchronize(s));
  BBTC_TRY(check(herr));
  if ((unsigned long long)stats[0] & HASH_FAILED) {
    *again = true;
    return BBTC_OK;
  }
  const int64_t m = stats[0];
  if (m > 0xFFFFFFFFLL) {
    set_error("bbtc_graph_create: %lld simple edges exceed 2^32 - 1", (long long)m);
    return BBTC_EINVAL;
  }
  g->m = m;
  g->deg_max = hdmax;

  // ---- a3: order by (degree, id)
  int32_t *rank = nullptr;
  BBTC_TRY(scratch.get(&rank, n));
  BBTC_TRY(dalloc_n(&g->perm, n, s));
  g->bytes += (uint64_t)(n > 0 ? n : 1) * sizeof(int32_t);
  // ukeys (m) must survive the rank sort: rank keys go to the sort buffer that
  // does not hold ukeys, plus a separate alternate buffer.
  uint64_t *rk = sorted;  // free now (its distinct keys were copied to ukeys)
  uint64_t *rk_alt = nullptr;
  BBTC_TRY(scratch.get(&rk_alt, n));
  if (n > 0) {
    k_rank_keys<<<grid_for(n, 256, 16), 256, 0, s>>>(g->deg, n, nb, rk);
    BBTC_LAUNCH_CHECK();
    int dbits = ceil_log2_u64((uint64_t)hdmax + 1);
    BBTC_TRY(radix_sort(rk, rk_alt, nullptr, nullptr, n, nb, nb + dbits, s, err, &in_alt));
    k_rank_finish<<<grid_for(n, 256, 16), 256, 0, s>>>(in_alt ? rk_alt : rk, n, nb, err, g->perm,
                                                        rank);
    BBTC_LAUNCH_CHECK();
    if (g->voff) {
      BBTC_TRY(dalloc_n(&g->gid, n, s));
      g->bytes += (uint64_t)n * sizeof(int32_t);
      k_graph_of_position<<<grid_for(n, 256, 16), 256, 0, s>>>(g->perm, n, g->voff, g->ng,
                                                              g->gid);
      BBTC_LAUNCH_CHECK();
    }
  }

  // ---- a4: orient and build the oriented CSR: row lengths and each edge's slot by
  // counting, offsets, scatter, per-row sort
  BBTC_TRY(dalloc_n(&g->rowptr, n + 1, s));
  BBTC_TRY(dalloc_n(&g->colidx, padded_columns(m), s));
  BBTC_TRY(dalloc_n(&g->esrc, m, s));
  g->bytes += (uint64_t)(n + 1) * 8 + (uint64_t)(m > 0 ? m : 1) * 8;
  BBTC_CUDA(cudaMemsetAsync(g->rowptr, 0, sizeof(int64_t) * (size_t)(n + 1), s));
  uint64_t *ok = sorted;  // rank keys are consumed; reuse
  unsigned *slot = reinterpret_cast<unsigned *>(g->esrc);  // (its rows are written last)
  if (m > 0) {
    k_orient_count<<<grid_for(m, 256, 32), 256, 0, s>>>(
        ukeys, m, nb, rank, ok, slot, reinterpret_cast<unsigned long long *>(g->rowptr));
    BBTC_LAUNCH_CHECK();
  }
  // rowptr holds the row lengths: their maximum is d+_max, their scan the offsets
  BBTC_TRY(reduce_max_i64(g->rowptr, n, &hstats[1], s));
  BBTC_CUDA(cudaMemcpyAsync(&stats[1], &hstats[1], sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  BBTC_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  BBTC_TRY(exclusive_scan_u64(reinterpret_cast<uint64_t *>(g->rowptr),
                              reinterpret_cast<uint64_t *>(g->rowptr), n + 1, s));
  if (m > 0) {
    k_orient_scatter<<<grid_for(m, 256, 32), 256, 0, s>>>(ok, slot, m, nb, g->rowptr, g->colidx);
    BBTC_LAUNCH_CHECK();
  }
  BBTC_CUDA(cudaStreamSynchronize(s));
  if (herr & SORT_FAILED) return sort_failed("bbtc_graph_create");
  g->dplus_max = n > 0 ? stats[1] : 0;
  if (m > 0 && g->dplus_max <= SEG_CAP) {
    BBTC_TRY(sort_rows(g->rowptr, n, RowSource{g->colidx, nullptr, nullptr}, g->colidx, g->esrc, s));
  } else if (m > 0) {
    k_fill_esrc<<<grid_for((n + 31) / 32 * 32, 256, 16), 256, 0, s>>>(g->rowptr, n, g->esrc);
    BBTC_LAUNCH_CHECK();
    uint64_t *ok_alt = ukeys;
    BBTC_TRY(radix_sort(ok, ok_alt, nullptr, nullptr, m, 0, 2 * nb, s, err, &in_alt));
    k_pair_unkey<<<grid_for(m, 256, 32), 256, 0, s>>>(in_alt ? ok_alt : ok, m, nb, err, g->colidx);
    BBTC_LAUNCH_CHECK();
    BBTC_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    BBTC_CUDA(cudaStreamSynchronize(s));
    if (herr & SORT_FAILED) return sort_failed("bbtc_graph_create");
  }
  return BBTC_OK;
}

bbtc_status prepare_graph(bbtc_graph *g, const int64_t *d_rowptr, const int32_t *d_colidx,
                          int64_t nnz, bool symmetric) {
  cudaStream_t s = g->stream;
  const int64_t n = g->n;
  const uint64_t bytes0 = g->bytes;
  g->nb = ceil_log2_u64((uint64_t)n) < 1 ? 1 : ceil_log2_u64((uint64_t)n);
  if (n > 0 && n <= SG_N && nnz > 0 && nnz <= SG_ENTRIES && !g->voff)
    return prepare_small(g, d_rowptr, d_colidx, nnz, symmetric);
  // symmetric input with sorted rows: per-row path, no global sort
  if (symmetric && nnz > 0 && n > 0) {
    Scratch scratch(s);
    int32_t *err = nullptr;
    bool applied = false;
    BBTC_TRY(scratch.get(&err, 1));
    BBTC_CUDA(cudaMemsetAsync(err, 0, sizeof(int32_t), s));
    BBTC_TRY(prepare_sym_sorted(g, d_rowptr, d_colidx, nnz, err, &applied));
    if (applied) return BBTC_OK;
  }
  bool again = false;
  if (nnz > 0 && nnz <= HASH_MAX) {
    const bbtc_status st = prepare_general(g, d_rowptr, d_colidx, nnz, symmetric, true, &again);
    if (st != BBTC_ENOMEM) {
      if (st != BBTC_OK || !again) return st;
    } else {  // sorting takes less memory: 16 bytes a key where buckets take up to 29
      clear_error();
      for (int32_t **a : {&g->deg, &g->perm, &g->colidx, &g->esrc, &g->gid}) {
        dfree(*a, s);
        *a = nullptr;
      }
      dfree(g->rowptr, s);
      g->rowptr = nullptr;
      g->bytes = bytes0;
    }
  }
  return prepare_general(g, d_rowptr, d_colidx, nnz, symmetric, false, &again);
}

}  // namespace bbtc
