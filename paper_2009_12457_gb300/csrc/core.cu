// core.cu -- the dense core: triangles whose two upper vertices are hubs,
// counted with bitmap rows instead of lists.
//
// In degree order the top positions are the hubs, and most probes of a skewed
// graph fall among them: on an R-MAT graph of scale 20, 90% of the open pairs
// (v, w) of a source u have v and w among the top 16,384 of 1 M positions, and
// the part of u's list there is dense. For such a u the count over its core
// neighbours is
//   sum over v in N(u), v >= v0 of popcount(B(u) & B(v)),
// where B(x) holds one bit per core column w in N(x) (all above x, so only
// the columns above v contribute: exactly Alg. 5's |N(u) ∩ N(v)|). A word
// covers 32 columns, where a probe of a list covers one entry, so the bitmap
// form is cheaper as soon as a row holds more than a few entries per group of
// 32 columns; sources below that (CORE_MIN_ROW core neighbours) stay with the
// lists (the flat in-edges leave out the edges that are counted here). Of R-MAT
// scale 20's count of 0.74 ms, 0.30 are spent here; a count of scale 14, all core,
// takes 35 us where the lists took 142.
//
// Layout: columns are cut into groups of 4,096, one 16-byte quad (128 columns)
// per lane of a warp. Core vertex v's row is stored from the group that holds v
// up to the last one (it has no bits below v). The columns of each part of the
// partition start on a quad, so that a quad lies in one part and the counts can
// be attributed to tasks (i, j, k); the last group is always full, so that the
// hubs, which most rows reach, share it.
#include <algorithm>
#include <type_traits>

#include "graph.cuh"

namespace bbtc {

namespace {

constexpr int CORE_NT = 256;
constexpr int CORE_WARPS = CORE_NT / 32;
constexpr int CORE_MAX_COLS = 12288;  // columns of the core at most
// a graph of at most so many vertices is all core, and no list is probed. Against
// 8,192 columns and lists, graphs of 16,384 vertices count in 16.5 us instead of 37
// (R-MAT scale 14), 38 instead of 61 (G(n, m), 262 K pairs), 136 instead of 453 (2 M
// pairs) and 32 instead of 59 (Chung-Lu, 500 K pairs). With twice as many columns, 24,000
// vertices gain (1 M pairs of a G(n, m): 158 us to 121, 2 M of a Chung-Lu: 148 to 80) and
// 32,000 lose (G(n, m), 2 M pairs: 270 to 286): where all core stops paying depends on
// the density, and lies above this bound for the graphs tried
constexpr int CORE_ALL_COLS = 16384;
constexpr int CORE_TABLE = 816;       // task counters kept in shared memory (p <= 16)
constexpr int64_t CORE_WIDE_EDGES = 1 << 23;  // fewer edges: 8,192 columns
constexpr int CORE_CTAS = 4;          // counting CTAs per SM
constexpr int32_t CORE_STATUS_TIMEOUT = 1;

__device__ __forceinline__ uint64_t core_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// index in cp of the part that owns core vertex v
__device__ __forceinline__ int core_part(const CoreParts &cp, int32_t v) {
  int lo = 0, hi = cp.np;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (cp.first[mid] <= v) lo = mid; else hi = mid;
  }
  return lo;
}

// The bitmap rows, one warp per core vertex, and its table entry {byte offset
// of its row were it stored from group 0, first quad | part << 16}; block 0
// writes the part of every quad and the all-zero row at offset 0.
__global__ void __launch_bounds__(CORE_NT) k_core_bits(const int64_t *__restrict__ rowptr,
                                                       const int32_t *__restrict__ colidx,
                                                       int64_t n, int32_t v0, CoreParts cp,
                                                       uint4 *__restrict__ bits,
                                                       int2 *__restrict__ tab,
                                                       uint8_t *__restrict__ qpart) {
  extern __shared__ __align__(16) unsigned char core_smem[];
  const unsigned lane = lane_id();
  const int warp = threadIdx.x >> 5;
  const int nq = cp.quads;
  uint4 *row4 = reinterpret_cast<uint4 *>(core_smem) + warp * nq;
  unsigned *row = reinterpret_cast<unsigned *>(row4);
  if (blockIdx.x == 0)
    for (int q = threadIdx.x; q < nq; q += CORE_NT) {
      int k = 0;
      while (k + 1 < cp.np && cp.quad0[k + 1] <= q) ++k;
      qpart[q] = cp.id[k];
      bits[q] = make_uint4(0, 0, 0, 0);
    }
  for (int64_t v = v0 + (int64_t)blockIdx.x * CORE_WARPS + warp; v < n;
       v += (int64_t)gridDim.x * CORE_WARPS) {
    const int k = core_part(cp, (int32_t)v);
    const int vq = cp.quad0[k] + (((int)v - cp.first[k]) >> 7);
    const int g = vq >> 5;
    const int q0 = g * 32;
    const uint32_t off = cp.gbase[g] + (uint32_t)((int32_t)v - cp.gfirst[g]) * (uint32_t)(nq - q0) * 16u;
    for (int q = q0 + (int)lane; q < nq; q += 32) row4[q] = make_uint4(0, 0, 0, 0);
    __syncwarp();
    const int64_t e1 = rowptr[v + 1];
    for (int64_t e = rowptr[v] + lane; e < e1; e += 32) {
      const int32_t w = colidx[e];
      const int kw = cp.np == 1 ? 0 : core_part(cp, w);
      const unsigned col = (unsigned)(cp.quad0[kw] * 128 + (w - cp.first[kw]));
      atomicOr(&row[col >> 5], 1u << (col & 31u));
    }
    __syncwarp();
    uint4 *out = bits + off / 16u;
    for (int q = q0 + (int)lane; q < nq; q += 32) out[q - q0] = row4[q];
    if (lane == 0) tab[v - v0] = make_int2((int32_t)(off - (uint32_t)q0 * 16u), vq | ((int)cp.id[k] << 16));
    __syncwarp();
  }
}

// The sources counted through the core: those among positions [u0, n) with at
// least min_row core neighbours, as work items {u, first core edge, first edge
// of the item, end of the row} of at most CORE_CHUNK core edges, and one flag
// bit per position. Sources that find no room in the item list keep a clear
// flag (the lists count them). Room is only ever taken, never given back: what was
// taken past it by one reservation would else be handed out again while an earlier
// gap stayed unwritten. So the reservation that crosses the end is the only one
// that leaves entries below it, which become empty items, and the number of items
// is the smaller of *nitems and cap. One thread per position, highest first.
__global__ void __launch_bounds__(CORE_NT) k_core_rows(const int64_t *__restrict__ rowptr,
                                                       const int32_t *__restrict__ colidx,
                                                       int64_t n, int64_t u0, int32_t v0,
                                                       int min_row, uint32_t cap,
                                                       unsigned *__restrict__ nitems,
                                                       int4 *__restrict__ items,
                                                       unsigned *__restrict__ flags) {
  const unsigned lane = lane_id();
  const int64_t words = (n - u0 + 31) >> 5;
  for (int64_t x = ((int64_t)blockIdx.x * CORE_NT + threadIdx.x) >> 5; x < words;
       x += ((int64_t)gridDim.x * CORE_NT) >> 5) {
    const int64_t word = words - 1 - x;
    const int64_t u = u0 + word * 32 + lane;
    uint32_t cs = 0, re = 0, cnt = 0;
    if (u < n) {
      const int64_t r0 = rowptr[u], r1 = rowptr[u + 1];
      if (r1 - r0 >= min_row) {
        re = (uint32_t)r1;
        cs = u >= v0 ? (uint32_t)r0
                     : (uint32_t)lower_bound_dev<int32_t, int64_t>(colidx, r0, r1, v0);
        if (re - cs >= (uint32_t)min_row) cnt = (re - cs + CORE_CHUNK - 1) / CORE_CHUNK;
      }
    }
    const uint32_t incl = warp_inclusive_scan(cnt);
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    uint32_t at = 0;
    if (lane == 0 && total) at = atomicAdd(nitems, total);
    at = __shfl_sync(0xffffffffu, at, 0);
    const bool room = total > 0 && at + total <= cap;  // else the whole word stays with the lists
    if (total && !room)
      for (uint32_t o = at + lane; o < cap; o += 32) items[o] = make_int4((int32_t)(u0 + word * 32), 0, 0, 0);
    const unsigned flag = __ballot_sync(0xffffffffu, room && cnt > 0);
    if (lane == 0) flags[word] = flag;
    if (room) {
      uint32_t o = at + incl - cnt;
      for (uint32_t c = 0; c < cnt; ++c)
        items[o++] = make_int4((int32_t)u, (int32_t)cs, (int32_t)(cs + c * CORE_CHUNK), (int32_t)re);
    }
  }
}

// carry-save adder: (carry, sum) of three bit vectors
__device__ __forceinline__ void csa(unsigned &carry, unsigned &sum, unsigned a, unsigned b,
                                    unsigned c) {
  carry = (a & b) | (a & c) | (b & c);  // one three-input logic instruction each
  sum = a ^ b ^ c;
}

// Bit-sliced column counters of one lane's quad (4 words): every group of
// eight rows goes through seven carry-save adders, and only the carries of
// weight eight are counted (under the mask of the source's own columns), so
// that the population count, the slow unit here, runs once per eight rows.
struct ColumnSums {
  unsigned one[4], two[4], four[4];
  unsigned eights;  // sum over groups of popcount(weight-8 carries & mask)
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < 4; ++i) one[i] = two[i] = four[i] = 0u;
    eights = 0u;
  }
  __device__ __forceinline__ void add8(const uint4 (&d)[8], const uint4 &m) {
    const unsigned mk[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      unsigned x[8];
#pragma unroll
      for (int r = 0; r < 8; ++r)
        x[r] = i == 0 ? d[r].x : i == 1 ? d[r].y : i == 2 ? d[r].z : d[r].w;
      unsigned ta, tb, fa, fb, e;
      csa(ta, one[i], one[i], x[0], x[1]);
      csa(tb, one[i], one[i], x[2], x[3]);
      csa(fa, two[i], two[i], ta, tb);
      csa(ta, one[i], one[i], x[4], x[5]);
      csa(tb, one[i], one[i], x[6], x[7]);
      csa(fb, two[i], two[i], ta, tb);
      csa(e, four[i], four[i], fa, fb);
      eights += __popc(e & mk[i]);
    }
  }
  __device__ __forceinline__ unsigned total(const uint4 &m) const {
    const unsigned mk[4] = {m.x, m.y, m.z, m.w};
    unsigned s = 8u * eights;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      s += __popc(one[i] & mk[i]) + 2u * __popc(two[i] & mk[i]) + 4u * __popc(four[i] & mk[i]);
    return s;
  }
};

struct CoreLaunch {
  CoreDesc one;           // the only descriptor when nd == 1
  const CoreDesc *descs;  // else nd of them, by item_base
  int32_t nd;
  int64_t nitems;         // over all descriptors
  int quads_max;
  unsigned long long *task_count;
  unsigned long long *graph_count;  // nullable: per-graph counts (gid of the descriptor)
  int64_t ntasks;
  int32_t *status;
  unsigned long long *t0;
  uint64_t timeout_ns;
};

// index of (i, j, j) in Alg. 4 order
__device__ __forceinline__ int core_task(int p, int i, int j) {
  int t = 0;
  for (int a = 0; a < i; ++a) t += (p - a) * (p - a + 1) / 2;
  for (int b = i; b < j; ++b) t += p - b;
  return t;
}

constexpr int CORE_ROWS = CORE_CHUNK + 32;  // row offsets staged per warp, with room for whole steps

// Counts the rows staged at rows[a, b) against the mask m: W lanes per row, so
// 32 / W rows side by side, eight of them in flight per lane. CHECK: the last
// steps, where rows past b read the zero row. The low 9 bits of a staged offset
// hold the part of v (rows are multiples of 512 bytes).
template <int W, bool PARTS, bool CHECK>
__device__ __forceinline__ int core_steps(ColumnSums &cols, const uint4 &m,
                                          const unsigned char *__restrict__ base,
                                          const uint32_t *rows, int a, int b, unsigned lane) {
  constexpr int RPS = 32 / W;
  const int sub = RPS > 1 ? (int)lane / W : 0;
  for (; CHECK ? a < b : a + 8 * RPS <= b; a += 8 * RPS) {
    uint4 r[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int x = a + i * RPS + sub;
      uint32_t off = rows[x];
      if (PARTS) off &= ~511u;
      if (CHECK && x >= b) off = 0u;
      r[i] = *reinterpret_cast<const uint4 *>(base + off);
    }
    cols.add8(r, m);
  }
  return a;
}

// One warp per work item; the items are about equal, so they are dealt round
// robin. Bound by instruction issue and L1 (rows of 512 bytes from an L2-resident
// matrix of a few MB). Four CTAs of 64 registers (0.44 ms on R-MAT scale 20)
// beat three of 80 (0.53): the loads' latency needs the warps. Rows that start
// in the last half or quarter of the top group are read two or four side by
// side, since the lanes below them would only read zeros. Columns: 8,192 beat
// 12,288 on R-MAT scale 18 (0.165 against 0.173 ms for the whole count), they tie
// on scale 20 (0.745, 0.740), and 12,288 win on scale 22 (4.91, 4.66) and on the
// 1/16 Friendster-shaped graph (7.43, 7.32): hence CORE_WIDE_EDGES.
// MODE 0: totals of one descriptor, where a lane keeps its sum to the end; 1:
// totals of several, where it keeps it to the warp's last item of a descriptor
// (64 handles: 0.82 ms; through mode 2 1.13); 2: per task or per graph.
template <int MODE>
__global__ void __launch_bounds__(CORE_NT, CORE_CTAS) k_core_count(CoreLaunch P) {
  constexpr bool ONE = MODE < 2;  // totals
  constexpr bool MULTI = MODE == 1;
  extern __shared__ __align__(16) unsigned char core_smem[];
  __shared__ unsigned long long table[ONE ? 1 : CORE_TABLE];
  __shared__ uint32_t rows_s[CORE_WARPS][CORE_ROWS];
  const unsigned lane = lane_id();
  const int warp = threadIdx.x >> 5;
  uint4 *mask4 = reinterpret_cast<uint4 *>(core_smem) + warp * P.quads_max;
  uint32_t *rows = rows_s[warp];
  for (int i = lane; i < CORE_ROWS; i += 32) rows[i] = 0u;
  const bool in_table = !ONE && P.ntasks <= CORE_TABLE;
  if (in_table) {
    for (int i = threadIdx.x; i < (int)P.ntasks; i += CORE_NT) table[i] = 0ull;
    __syncthreads();
  }
  uint64_t t_start = 0;
  if (P.timeout_ns) {
    t_start = core_ns();
    if (lane == 0) atomicCAS(P.t0, 0ull, (unsigned long long)t_start);
  }
  unsigned long long acc = 0;
  int cur_desc = 0;
  const int64_t nw = (int64_t)gridDim.x * CORE_WARPS;
  for (int64_t item = (int64_t)blockIdx.x * CORE_WARPS + warp; item < P.nitems; item += nw) {
    if (P.timeout_ns && core_ns() - t_start > P.timeout_ns) {
      if (lane == 0) atomicExch(P.status, CORE_STATUS_TIMEOUT);
      break;
    }
    const CoreDesc *dp = &P.one;
    if (MULTI || (!ONE && P.nd > 1)) {
      int lo = 0, hi = P.nd;  // last descriptor with item_base <= item
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (P.descs[mid].item_base <= item) lo = mid; else hi = mid;
      }
      dp = &P.descs[lo];
      if (MULTI && lo != cur_desc) {
        acc = warp_sum(acc);
        if (lane == 0 && acc) atomicAdd(&P.task_count[P.descs[cur_desc].task_base], acc);
        acc = 0;
        cur_desc = lo;
      }
    }
    const CoreDesc &d = *dp;
    const int4 it = d.items[item - d.item_base];
    const int32_t u = it.x, v0 = d.v0;
    const uint32_t cs = (uint32_t)it.y, x0 = (uint32_t)it.z, re = (uint32_t)it.w;
    const int cnt = re - x0 < (uint32_t)CORE_CHUNK ? (int)(re - x0) : CORE_CHUNK;
    const int32_t *__restrict__ ci = d.colidx;
    const int2 *__restrict__ tab = d.tab;
    const unsigned char *__restrict__ bits = reinterpret_cast<const unsigned char *>(d.bits);
    const int nq = d.quads;
    const int groups = nq >> 5, top = nq - 32;
    // the rows of the item's core edges, in order; c_top, c_16, c_8: how many lie
    // below the last group, below its second half, below its last quarter
    int c_top = 0, c_16 = 0, c_8 = 0, g0 = 0;
    for (int x = 0; x < cnt; x += 32) {
      int2 t = make_int2(0, 0x7fff);
      if (x + (int)lane < cnt) {
        t = tab[ci[x0 + x + lane] - v0];
        rows[x + lane] = (uint32_t)t.x | (ONE ? 0u : (uint32_t)(t.y >> 16));
      }
      const int vq = t.y & 0xffff;
      if (x == 0) g0 = __shfl_sync(0xffffffffu, vq, 0) >> 5;
      c_top += __popc(__ballot_sync(0xffffffffu, vq < top));
      c_16 += __popc(__ballot_sync(0xffffffffu, vq < top + 16));
      c_8 += __popc(__ballot_sync(0xffffffffu, vq < top + 24));
    }
    // B(u): a core vertex has its row, another source's is built from its list
    uint32_t uoff = 0;
    int ug = 0;
    if (u >= v0) {
      const int2 t = tab[u - v0];
      uoff = (uint32_t)t.x;
      ug = (t.y & 0xffff) >> 5;
    } else {
      for (int q = lane; q < nq; q += 32) mask4[q] = make_uint4(0, 0, 0, 0);
      __syncwarp();
      unsigned *mk = reinterpret_cast<unsigned *>(mask4);
      for (uint32_t x = lane; x < re - cs; x += 32) {
        const int32_t w = ci[cs + x];
        const int kw = d.parts.np == 1 ? 0 : core_part(d.parts, w);
        const unsigned col = (unsigned)(d.parts.quad0[kw] * 128 + (w - d.parts.first[kw]));
        atomicOr(&mk[col >> 5], 1u << (col & 31u));
      }
    }
    __syncwarp();
    int part_i = 0;
    if (!ONE && d.p > 1) part_i = part_of_dev(d.cuts, d.p, u);
    unsigned long long row_total = 0;
    // rows [a, b) against columns [128 * quad, ...) of group g, W lanes per row
    auto pass = [&](int g, int a, int b, auto width_c) {
      constexpr int W = decltype(width_c)::value;
      if (a >= b) return;
      const int quad = g * 32 + (32 - W) + (int)(lane & (W - 1));
      uint4 m = make_uint4(0, 0, 0, 0);
      if (u >= v0) {
        if (g >= ug) m = *reinterpret_cast<const uint4 *>(bits + uoff + (uint32_t)quad * 16u);
      } else {
        m = mask4[quad];
      }
      if (!__any_sync(0xffffffffu, (m.x | m.y | m.z | m.w) != 0u)) return;
      const unsigned char *base = bits + (uint32_t)quad * 16u;
      while (a < b) {
        int e = b, j = 0;
        if (!ONE) {  // the rows of one part j
          j = (int)(rows[a] & 511u);
          for (e = a; e < b;) {
            const unsigned same = __ballot_sync(0xffffffffu, e + (int)lane < b &&
                                                             (int)(rows[e + lane] & 511u) == j);
            if (same == 0xffffffffu) {
              e += 32;
            } else {
              e += __ffs(~same) - 1;
              break;
            }
          }
        }
        ColumnSums cols;
        cols.clear();
        a = core_steps<W, !ONE, false>(cols, m, base, rows, a, e, lane);
        if (a < e) core_steps<W, !ONE, true>(cols, m, base, rows, a, e, lane);
        a = e;
        const unsigned c = cols.total(m);
        if (ONE) {
          acc += c;
          continue;
        }
        row_total += c;
        const int k = d.p > 1 ? (int)d.qpart[quad] : 0;
        const int t0 = d.task_base + (d.p > 1 ? core_task(d.p, part_i, j) - j : 0);
        unsigned left = __ballot_sync(0xffffffffu, c != 0u);
        while (left) {
          const int k0 = __shfl_sync(0xffffffffu, k, __ffs(left) - 1);
          const unsigned sum = __reduce_add_sync(0xffffffffu, k == k0 ? c : 0u);
          if (lane == 0) {
            if (in_table) atomicAdd(&table[t0 + k0], (unsigned long long)sum);
            else atomicAdd(&P.task_count[t0 + k0], (unsigned long long)sum);
          }
          left &= ~__ballot_sync(0xffffffffu, k == k0);
        }
      }
    };
    for (int g = g0; g < groups - 1; ++g) {
      // rows that start at or before group g
      int b = 0;
      for (int x = 0; x < c_top; x += 32) {
        int vq = 0x7fff;
        if (x + (int)lane < c_top) vq = tab[ci[x0 + x + lane] - v0].y & 0xffff;
        b += __popc(__ballot_sync(0xffffffffu, (vq >> 5) <= g));
      }
      pass(g, 0, b, std::integral_constant<int, 32>());
    }
    pass(groups - 1, 0, c_16, std::integral_constant<int, 32>());
    pass(groups - 1, c_16, c_8, std::integral_constant<int, 16>());
    pass(groups - 1, c_8, cnt, std::integral_constant<int, 8>());
    if (!ONE && P.graph_count) {
      row_total = warp_sum(row_total);
      if (lane == 0 && row_total) atomicAdd(&P.graph_count[d.gid[u]], row_total);
    }
    __syncwarp();
  }
  if (ONE) {
    acc = warp_sum(acc);
    const int32_t tb = MULTI ? P.descs[cur_desc].task_base : P.one.task_base;
    if (lane == 0 && acc) atomicAdd(&P.task_count[tb], acc);
  } else if (in_table) {
    __syncthreads();
    for (int i = threadIdx.x; i < (int)P.ntasks; i += CORE_NT)
      if (table[i]) atomicAdd(&P.task_count[i], table[i]);
  }
}

}  // namespace

void free_core(Plan *pl, cudaStream_t s) {
  Core &c = pl->core;
  dfree(c.bits, s);
  dfree(c.tab, s);
  dfree(c.qpart, s);
  dfree(c.items, s);
  dfree(c.flags, s);
  dfree(c.count, s);
  c = Core();
}

// Sources with fewer core neighbours stay with the lists: a row costs about
// 500 instructions of set-up and 10 per core edge, the lists about one per
// probe. Counts with bounds of 48, 64, 80 and 128: R-MAT scale 20 739, 735, 729 and
// 716 us, scale 21 1.60, 1.60, 1.59 and 1.61 ms, scale 22 3.96, 3.92, 3.92 and 3.99 ms, a
// Chung-Lu graph of 28 M pairs 1.33, 1.31, 1.32 and 1.31 ms: flat around the bound.
constexpr int CORE_MIN_ROW = 64;

bbtc_status build_core(const bbtc_graph *g, Plan &pl, cudaStream_t s) {
  const int64_t n = g->n, m = g->m;
  Core &c = pl.core;
  if (m < 3 || n < 3) return BBTC_OK;
  // columns: all of a small graph, else the top CORE_MAX_COLS; the packed rows
  // take K^2 / 16 bytes, which is kept to about 96 bytes per edge
  int64_t K = n <= CORE_ALL_COLS ? CORE_ALL_COLS : m < CORE_WIDE_EDGES ? 8192 : CORE_MAX_COLS;
  const int max_quads = (int)(K / 128);
  while (K > 256 && K * K / 16 > 96 * m) K = K * 7 / 8;
  const bool all = n <= K;
  // the graphs of a union interleave in the degree order, so that its top
  // positions hold many thin cores side by side: measured slower than the lists
  // (256 graphs: 14.1 instead of 13.8 ms)
  if (g->ng > 1 && !all) return BBTC_OK;
  CoreParts &cp = c.parts;
  for (int tries = 0;; ++tries) {
    if (all) K = n;
    const int32_t v0 = (int32_t)(n - K);
    int quads = 0;
    cp.np = 0;
    for (int k = 0; k < pl.p; ++k) {
      const int32_t first = std::max(pl.h_cuts[k], v0);
      if (pl.h_cuts[k + 1] <= first) continue;
      cp.first[cp.np] = first;
      cp.id[cp.np] = (uint8_t)k;
      cp.quad0[cp.np] = quads;
      quads += (pl.h_cuts[k + 1] - first + 127) / 128;
      ++cp.np;
    }
    const int room = (quads + 31) / 32 * 32;
    // parts that start on a quad can push the columns into one more group of 32
    // quads; a core of the top positions gives up a few columns instead
    if (!all && quads > max_quads && tries < 64) {
      K -= 128 * (quads - max_quads);
      if (K < 1024) return BBTC_OK;
      continue;
    }
    // the last group is the full one: the hubs, which most rows reach, share it
    for (int k = 0; k < cp.np; ++k) cp.quad0[k] += room - quads;
    cp.quads = room;
    c.v0 = v0;
    break;
  }
  // rows of group g hold its quads and those of the groups after it
  const int groups = cp.quads / 32;
  int64_t bytes = (int64_t)cp.quads * 16;  // the zero row
  auto first_of = [&](int gr) -> int64_t {  // first core vertex at or after group gr's columns
    if (gr >= groups) return n;
    int k = 0;
    while (k + 1 < cp.np && cp.quad0[k + 1] <= 32 * gr) ++k;
    const int64_t v = cp.first[k] + 128 * (int64_t)std::max(32 * gr - cp.quad0[k], 0);
    return std::min<int64_t>(v, k + 1 < cp.np ? cp.first[k + 1] : n);  // a part may end inside its last quad
  };
  if (groups > CoreParts::kGroups) return BBTC_OK;
  for (int gr = 0; gr < groups; ++gr) {
    cp.gfirst[gr] = (int32_t)first_of(gr);
    cp.gbase[gr] = (uint32_t)bytes;
    bytes += (first_of(gr + 1) - first_of(gr)) * (int64_t)(cp.quads - 32 * gr) * 16;
  }
  const int64_t base = bytes / 16;
  if (bytes > (1ll << 31)) return BBTC_OK;
  c.all = all;
  c.u0 = all ? 0 : (n > 16ll * CORE_MAX_COLS ? n - 16ll * CORE_MAX_COLS : 0);
  c.u0 &= ~int64_t(31);
  const int min_row = all ? 2 : CORE_MIN_ROW;
  const int64_t nu = n - c.u0;
  const int64_t cap = std::min<int64_t>(nu, m / min_row) + m / CORE_CHUNK + 32;
  // (a core of the whole graph has to hold every source: the lists are not run)
  c.cap = (uint32_t)(all ? cap : std::min<int64_t>(cap, 1 << 20));
  BBTC_TRY(dalloc_n(&c.bits, base, s));
  BBTC_TRY(dalloc_n(&c.tab, n - c.v0, s));
  BBTC_TRY(dalloc_n(&c.qpart, cp.quads, s));
  BBTC_TRY(dalloc_n(&c.items, c.cap, s));
  BBTC_TRY(dalloc_n(&c.flags, (nu + 31) / 32, s));
  BBTC_TRY(dalloc_n(&c.count, 1, s));
  BBTC_CUDA(cudaMemsetAsync(c.count, 0, sizeof(unsigned), s));
  k_core_bits<<<grid_for(n - c.v0, CORE_WARPS, 8), CORE_NT,
                sizeof(uint4) * (size_t)cp.quads * CORE_WARPS, s>>>(g->rowptr, g->colidx, n, c.v0,
                                                                   cp, c.bits, c.tab, c.qpart);
  BBTC_LAUNCH_CHECK();
  k_core_rows<<<grid_for(nu, CORE_NT, 8), CORE_NT, 0, s>>>(g->rowptr, g->colidx, n, c.u0, c.v0,
                                                           min_row, c.cap, c.count, c.items,
                                                           c.flags);
  BBTC_LAUNCH_CHECK();
  c.bytes = (uint64_t)base * 16 + (uint64_t)(n - c.v0) * 8 + (uint64_t)c.cap * 16 + (uint64_t)nu / 8;
  return BBTC_OK;
}

CoreDesc core_desc(const bbtc_graph *g, const Plan &pl, int64_t item_base, int32_t task_base) {
  CoreDesc d;
  d.items = pl.core.items;
  d.item_base = item_base;
  d.colidx = g->colidx;
  d.bits = pl.core.bits;
  d.tab = pl.core.tab;
  d.qpart = pl.core.qpart;
  d.cuts = pl.cuts;
  d.gid = g->gid;
  d.v0 = pl.core.v0;
  d.quads = pl.core.parts.quads;
  d.p = pl.p;
  d.task_base = task_base;
  d.parts = pl.core.parts;
  return d;
}

bbtc_status core_launch(CoreDesc one, const CoreDesc *descs, int32_t nd, int64_t nitems,
                        int quads_max, unsigned long long *task_count, int64_t ntasks, bool tasks,
                        unsigned long long *graph_count, int32_t *status, unsigned long long *t0,
                        uint32_t timeout_ms, cudaStream_t s) {
  if (nitems <= 0) return BBTC_OK;
  CoreLaunch P;
  if (!tasks) one.p = 1;
  P.one = one;
  P.descs = descs;
  P.nd = nd;
  P.nitems = nitems;
  P.quads_max = quads_max;
  P.task_count = task_count;
  P.graph_count = graph_count;
  P.ntasks = ntasks;
  P.status = status;
  P.t0 = t0;
  P.timeout_ns = (uint64_t)timeout_ms * 1000000ull;
  const size_t smem = sizeof(uint4) * (size_t)quads_max * CORE_WARPS;
  const unsigned grid = grid_for(nitems, CORE_WARPS, 4);
  if (tasks || graph_count)
    k_core_count<2><<<grid, CORE_NT, smem, s>>>(P);
  else if (nd > 1)
    k_core_count<1><<<grid, CORE_NT, smem, s>>>(P);
  else
    k_core_count<0><<<grid, CORE_NT, smem, s>>>(P);
  BBTC_LAUNCH_CHECK();
  return BBTC_OK;
}

}  // namespace bbtc
