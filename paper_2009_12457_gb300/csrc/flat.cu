// flat.cu -- the counting kernel of resident plans (a9): every in-edge (u, v)
// that the dense core leaves, grouped by destination v over the whole graph.
//
// For each in-edge (u, v) the elements of N(u) above v are looked up in N(v),
// which is staged on chip once per run of in-edges into v (see count.cu for
// why the elements at or below v need no look). A triangle (u, v, w) belongs to
// task (part(u), part(v), part(w)) of Alg. 4 whatever the order in which it is
// found, so the resident count does not visit the tasks one by one: it walks
// the in-edges once, with the longest runs and lists the graph has, and
// attributes hits to tasks only when the caller asks for per-task counts.
// (R-MAT scale 22 at p = 4 with per-task counts: 15.1 ms with a pass per task,
// 6.2 ms so, of which the dense core takes 1.5.)
//
// What bounds it: waits on loads with 24 warps per SM, which the warps' staging
// areas limit (issue active 55% on R-MAT scale 20, DRAM at 4%); on Chung-Lu graphs the
// probe rows lie anywhere in the column array (30.6 ms for 18 G probes of a 451 M
// edge one; 1.8 G edges: 136 ms, 3.9 TB/s from DRAM).
//
// A record is {e + 1, f}: the CSR position after (u, v) and the end of u's row,
// so [e + 1, f) is the probe run, and v is the column just before it.
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "bounds.cuh"
#include "flat.cuh"
#include "graph.cuh"
#include "primitives.cuh"
#include "stage.cuh"

namespace bbtc {

namespace {

constexpr int FL_NT = 128;
constexpr int FL_CTAS = 6;        // per SM: 24 warps, whose stages fill the shared memory
constexpr int FL_WARPS = FL_NT / 32;
constexpr int FL_RUN_MIN = 8;     // in-edges of one v that make a batch of their own
constexpr int FL_TABLE = 816;     // task counters kept in shared memory (p <= 16)
constexpr int FL_MODE_GRAPH = 1, FL_MODE_TASK = 2;
constexpr uint32_t FL_FLUSH = 32768;
static_assert((uint64_t)(FL_FLUSH + 32) * 92682 < (1ull << 32), "hits of one graph between two flushes");

struct FlatLaunch {
  FlatDesc one;           // the only descriptor when nd == 1
  const FlatDesc *descs;  // else nd of them, by item_base
  int32_t nd;
  int64_t nitems;
  unsigned long long *head;
  unsigned long long *task_count;
  unsigned long long *graph_count;
  int64_t ntasks;
  int32_t *status;
  const unsigned long long *t0;
  uint64_t timeout_ns;
};

struct FlatSmem {
  // per in-edge with probes: {first column, end, column of quad 0 - 4 * first
  // quad, part(u) | part(v) << 8}
  uint4 rec[32];
  uint2 rng[32];   // per in-edge: N(v) of a mixed batch
  uint32_t v[32];  // per in-edge: v of a mixed batch
  unsigned long long mbar;
  unsigned long long pad;
};

struct InHash {
  const int32_t *table;
  int log2h;
  __device__ __forceinline__ uint32_t bits(const int4 &w, uint32_t m) const {
    uint32_t hit = 0;
    while (m) {
      const int c = __ffs(m) - 1;
      m &= m - 1;
      const int32_t x = c == 0 ? w.x : c == 1 ? w.y : c == 2 ? w.z : w.w;
      hit |= (uint32_t)hash_contains(table, log2h, x) << c;
    }
    return hit;
  }
  __device__ __forceinline__ uint32_t count(const int4 &w, uint32_t m) const {
    return __popc(bits(w, m));
  }
};

// The sorted copy, searched by halving inside the key's bucket. Keys are bucketed
// by the exponent and three more bits of their distance to the list's last entry
// (in degree order lists crowd towards the hubs, at the end), so a bucket holds a
// few entries and a search takes `steps` halvings, the same for every lane: three
// or four where the whole list takes nine or ten. index[b] = first position of
// bucket b | end << 16; without an index (log2 steps of the length) the whole
// list is one bucket.
constexpr int SI_BUCKETS = 256;
struct InSorted {
  const int32_t *list;
  const uint32_t *index;  // nullptr: none
  int len, steps;
  uint32_t last, bucket0;
  static __device__ __forceinline__ uint32_t bucket_of(uint32_t distance) {
    return __float_as_uint((float)(distance + 1u)) >> 20;  // does not decrease with the distance
  }
  __device__ __forceinline__ bool one(int32_t w) const {
    int at = 0, end = len;
    if (index) {
      const uint32_t b = bucket_of(last - (uint32_t)w) - bucket0;  // (a key past the end: a far bucket)
      const uint32_t r = index[min(b, (uint32_t)SI_BUCKETS)];
      at = (int)(r & 0xffffu);
      end = (int)(r >> 16);
    }
    for (int step = 1 << steps; step > 1;) {
      step >>= 1;
      if (at + step <= end && list[at + step - 1] < w) at += step;
    }
    return at < end && list[at] == w;
  }
  __device__ __forceinline__ uint32_t bits(const int4 &w, uint32_t m) const {
    return ((uint32_t)one(w.x) | ((uint32_t)one(w.y) << 1) | ((uint32_t)one(w.z) << 2) |
            ((uint32_t)one(w.w) << 3)) & m;
  }
  __device__ __forceinline__ uint32_t count(const int4 &w, uint32_t m) const {
    return __popc(bits(w, m));
  }
};

// Not staged: searched in place in the column array.
struct InPlace {
  const int32_t *ci;
  uint32_t lo, hi;
  __device__ __forceinline__ uint32_t bits(const int4 &w, uint32_t m) const {
    uint32_t hit = 0, at = lo;  // the quad ascends: each search starts where the last one ended
    while (m) {
      const int c = __ffs(m) - 1;
      m &= m - 1;
      const int32_t x = c == 0 ? w.x : c == 1 ? w.y : c == 2 ? w.z : w.w;
      at = lower_bound_dev<int32_t, uint32_t>(ci, at, hi, x);
      if (at < hi && ci[at] == x) hit |= 1u << c;
    }
    return hit;
  }
  __device__ __forceinline__ uint32_t count(const int4 &w, uint32_t m) const {
    return __popc(bits(w, m));
  }
};

constexpr size_t flat_smem_bytes() {
  return (size_t)FL_WARPS * ((STAGE + 4) * sizeof(int32_t) + sizeof(FlatSmem));
}

template <int MODE>
__global__ void __launch_bounds__(FL_NT, FL_CTAS) k_flat(FlatLaunch P) {
  constexpr bool GRAPH = (MODE & FL_MODE_GRAPH) != 0;
  constexpr bool TASK = (MODE & FL_MODE_TASK) != 0;
  // quads in flight per lane against a bitmap or a filter: 2, 3 and 4 gave 4.91,
  // 4.38 and 4.19 ms on R-MAT scale 22 and 7.43, 6.84 and 6.87 ms on the 1/16
  // Friendster-shaped graph; attribution to tasks, which keeps more registers
  // live, 3.84, 4.06 and 4.30 ms on its 1/64 size at p = 16
  constexpr int FL_QUADS = TASK ? 2 : 4;
  extern __shared__ __align__(16) unsigned char flat_smem[];
  __shared__ int32_t cuts_s[TASK ? 65 : 1];
  __shared__ uint32_t ecut_s[TASK ? 65 : 1];
  const unsigned lane = threadIdx.x & 31u;
  const int warp = threadIdx.x >> 5;
  int32_t *stage = reinterpret_cast<int32_t *>(flat_smem) + warp * (STAGE + 4);
  FlatSmem &sm = reinterpret_cast<FlatSmem *>(flat_smem + (size_t)FL_WARPS * (STAGE + 4) *
                                                              sizeof(int32_t))[warp];
  // task counters behind the warps' areas
  unsigned long long *table = reinterpret_cast<unsigned long long *>(flat_smem + flat_smem_bytes());
  const bool in_table = TASK && P.ntasks <= FL_TABLE;
  const int p = P.one.p;
  if (TASK) {
    if (in_table)
      for (int i = threadIdx.x; i < (int)P.ntasks; i += FL_NT) table[i] = 0ull;
    for (int i = threadIdx.x; i <= p; i += FL_NT) {
      cuts_s[i] = P.one.cuts[i];
      ecut_s[i] = (uint32_t)P.one.rowptr[P.one.cuts[i]];
    }
    __syncthreads();
  }
  if (lane == 0) {
    stage[STAGE] = 0;
    mbar_init(&sm.mbar);
    mbar_init_fence();
  }
  __syncwarp();
  uint32_t mbar_parity = 0;
  uint64_t t_start = 0;
  if (P.timeout_ns) {
    t_start = *P.t0;
    if (t_start == 0) t_start = global_ns();
  }
  bool failed = false;
  unsigned long long acc = 0;
  // c triangles of task (i, j, k)
  auto add_task = [&](int i, int j, int k, unsigned long long c) {
    int t = k - j;
    for (int a = 0; a < i; ++a) t += (p - a) * (p - a + 1) / 2;
    for (int b = i; b < j; ++b) t += p - b;
    if (in_table) atomicAdd(&table[t], c);
    else atomicAdd(&P.task_count[t], c);
  };
  constexpr int FIELD = 10;  // bits of a packed counter
  int32_t cut1 = INT32_MAX, cut2 = INT32_MAX, cut3 = INT32_MAX;
  if (TASK) {
    if (p > 1) cut1 = cuts_s[1];
    if (p > 2) cut2 = cuts_s[2];
    if (p > 3) cut3 = cuts_s[3];
  }
  int cur_desc = 0;

  // the next item is requested while the current one runs
  unsigned long long it = 0;
  if (lane == 0) it = atomicAdd(P.head, 1ull);
  it = __shfl_sync(0xffffffffu, it, 0);
  while (it < (unsigned long long)P.nitems) {
    unsigned long long it_next = 0;
    if (lane == 0) it_next = atomicAdd(P.head, 1ull);
    if (P.timeout_ns && global_ns() - t_start > P.timeout_ns) {
      if (lane == 0) atomicExch(P.status, STATUS_TIMEOUT);
      break;
    }
    const FlatDesc *dp = &P.one;
    if (!TASK && P.nd > 1) {
      int lo = 0, hi = P.nd;  // last descriptor with item_base <= it
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (P.descs[mid].item_base <= (int64_t)it) lo = mid; else hi = mid;
      }
      dp = &P.descs[lo];
      if (lo != cur_desc) {
        acc = warp_sum(acc);
        if (lane == 0 && acc) atomicAdd(&P.task_count[P.descs[cur_desc].task_base], acc);
        acc = 0;
        cur_desc = lo;
      }
    }
    const FlatDesc &d = *dp;
    const uint2 *__restrict__ rec = d.rec;
    const uint32_t *__restrict__ inptr = d.inptr;
    const int64_t *__restrict__ rowptr = d.rowptr;
    const int32_t *__restrict__ ci = d.colidx;
    const int kflag = d.flags & 3, hash_min = d.flags >> 2;
    // items run from the last destinations down, so that the light ones end the launch
    const int64_t k = d.item0 + d.nitems - 1 - ((int64_t)it - d.item_base);
    uint32_t base = (uint32_t)(k * d.chunk);
    const uint32_t x1 = (uint32_t)min((int64_t)d.records, (k + 1) * d.chunk);
    uint32_t v = 0, vend = base;  // the run at hand: its destination and end
    uint32_t b0 = 0, b1 = 0;      // N(v)
    int32_t vl = -1;              // the lane's own destination (set when a run begins)
    // GRAPH: the run's graph, and its hits since record run_from. An item's length is the
    // caller's choice, so they are added up every FL_FLUSH in-edges at the latest: an
    // in-edge has fewer hits than the longest list, d+ <= sqrt(2m) < 92,682, and 32 bits
    // hold them (64-bit sums of the lanes, one for most runs of a union, took a batch of
    // 256 graphs from 8.05 to 8.12 ms)
    int32_t run_graph = -1;
    uint32_t run_hits = 0, run_from = base;
    auto flush_graph = [&]() {
      const uint32_t sum = __reduce_add_sync(0xffffffffu, run_hits);
      if (lane == 0 && sum) atomicAdd(&P.graph_count[run_graph], (unsigned long long)sum);
      run_hits = 0;
      run_from = base;
    };
    int staged_mode = ST_NONE, staged_log2h = 0, staged_len = 0;
    const int32_t *staged_list = stage;
    const uint32_t *staged_index = nullptr;
    int staged_steps = 0;
    uint32_t staged_last = 0, staged_bucket0 = 0;
    uint32_t staged_word0 = 0, staged_gw = STAGE;
    bool staged = false;
    int j_part = 0;
    unsigned long long field_sum = 0;  // lane x: the hits of field x for part j_part
    auto flush_fields = [&]() {
      const int nk = p - j_part;
      if (field_sum) add_task((int)lane / nk, j_part, j_part + (int)lane % nk, field_sum);
      field_sum = 0;
    };
    uint2 r = window_holds(base, lane, x1) ? rec[base + lane] : make_uint2(0, 0);
    while (base < x1) {
      const bool begins = vend <= base;
      if (begins) {  // a new run: (u, v) sits just below its probe run in u's row
        vl = window_holds(base, lane, x1) ? ci[r.x - 1] : -1;
        v = (uint32_t)__shfl_sync(0xffffffffu, vl, 0);
        vend = inptr[v + 1];
        b0 = (uint32_t)rowptr[v];
        b1 = (uint32_t)rowptr[v + 1];
        if (GRAPH) {
          // (loaded with the bounds: looked up at each batch's end, it stalled the warp)
          const int32_t graph = d.gid[v];
          if (graph != run_graph) flush_graph();
          run_graph = graph;
        }
        staged = false;
        if (TASK) {
          const int j = part_of_dev(cuts_s, p, (int32_t)v);
          if (j != j_part) flush_fields();
          j_part = j;
        }
      }
      const uint32_t run = min(vend, x1) - base;
      // (the rest of a run that has begun is a batch of its own, however short)
      const bool uniform = !begins || run >= (uint32_t)FL_RUN_MIN || run == x1 - base;
      if (uniform && b1 == b0) {  // nothing to find in an empty list
        base += run;
        r = window_holds(base, lane, x1) ? rec[base + lane] : make_uint2(0, 0);
        continue;
      }
      int nb = (int)min(run, 32u);
      uint32_t vb0 = b0, vb1 = b1;  // a mixed batch: the lane's own list
      if (!uniform) {
        // short runs share the window, up to a run that makes a batch of its own or
        // that may go on past the window
        const unsigned same = __match_any_sync(0xffffffffu, vl);
        const bool lengthy = __popc(same) >= FL_RUN_MIN || ((same >> 31) && window_holds(base, 32u, x1));
        const unsigned stop = __ballot_sync(0xffffffffu, vl < 0 || (lengthy && vl != (int32_t)v));
        nb = stop ? __ffs(stop) - 1 : 32;
        if ((int)lane < nb) {
          vb0 = (uint32_t)rowptr[vl];
          vb1 = (uint32_t)rowptr[vl + 1];
        }
        vend = base + (uint32_t)nb;  // the next window begins a new run
      }
      base += (uint32_t)nb;
      const uint2 rn = window_holds(base, lane, x1) ? rec[base + lane] : make_uint2(0, 0);
      if (window_holds(base, 32u + lane, x1))
        asm volatile("prefetch.global.L2 [%0];" ::"l"(rec + base + 32 + lane));
      const bool active = (int)lane < nb && vb1 > vb0;
      const uint32_t s0 = r.x, s1 = r.y;
      r = rn;
      const uint32_t a0 = s0 & ~3u;
      const uint32_t nq = active && s1 > s0 ? (s1 - a0 + 3u) >> 2 : 0u;
      const uint32_t incl = warp_inclusive_scan(nq);
      const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
      if (total == 0) continue;

      // stage N(v) for a run that probes it enough (the forms of count.cu)
      const int blen = (int)(b1 - b0);
      if (uniform && !staged && blen >= MIN_STAGE && (nb == 32 || total * 4u >= (uint32_t)blen / 2u)) {
        const int32_t x0 = (int)lane < blen ? ci[b0 + lane] : 0;
        int32_t lastv = 0;
        if (lane == 0 && blen > 32) lastv = ci[b1 - 1];
        const int32_t first = __shfl_sync(0xffffffffu, x0, 0);
        const int32_t last = blen > 32 ? __shfl_sync(0xffffffffu, lastv, 0)
                                       : __shfl_sync(0xffffffffu, x0, blen - 1);
        const uint32_t word0 = (uint32_t)first >> 5;
        const uint32_t nw = ((uint32_t)last >> 5) - word0 + 1u;
        int mode = ST_NONE;
        if (kflag == 0) {
          if (blen <= STAGE) mode = ST_SORTED;
        } else if (nw <= (uint32_t)STAGE) {
          mode = ST_BITMAP;
        } else if (2 * blen <= FILTER_SLOTS && (kflag == 1 || blen > hash_min)) {
          mode = ST_FILTER;
        } else if (2 * blen <= STAGE_POW2 && (kflag == 1 || blen > hash_min)) {
          mode = ST_HASH;
        } else if (kflag == 2 && blen <= STAGE) {
          mode = ST_SORTED;
        }
        if (mode != ST_NONE) {
          __syncwarp();
          const uint32_t e0 = b0 & ~3u;
          const int64_t span4 = (int64_t)((b1 - e0 + 3u) & ~3u);
          const bool long_list = blen >= BULK_STAGE_MIN;
          const int32_t *src = ci + b0;
          if (mode == ST_BITMAP) {
            const int64_t land = (int64_t)((nw + 4u) & ~3u);
            const bool bulk = long_list && land + span4 <= STAGE;
            if (bulk) bulk_issue(stage + land, ci, e0, (int64_t)e0 + span4, &sm.mbar, lane);
            int4 *s4 = reinterpret_cast<int4 *>(stage);
            for (int i = lane; i < (int)(land >> 2); i += 32) s4[i] = make_int4(0, 0, 0, 0);
            if (bulk) {
              failed = !bulk_wait(&sm.mbar, mbar_parity);
              src = stage + land + (b0 - e0);
            }
            __syncwarp();
            if (!failed)
              for (int i = lane; i < blen; i += 32) {
                const uint32_t w = (uint32_t)(i < 32 ? x0 : src[i]);
                atomicOr(reinterpret_cast<unsigned *>(stage) + ((w >> 5) - word0), 1u << (w & 31u));
              }
            staged_word0 = word0;
            staged_gw = nw;
          } else if (mode == ST_FILTER || mode == ST_HASH) {
            int log2h = 5;
            while ((1 << log2h) < 2 * blen) ++log2h;
            const int hsize = 1 << log2h;
            const int tab0 = mode == ST_FILTER ? FILTER_WORDS : 0;
            int32_t *tab = stage + tab0;
            const int64_t land = tab0 + hsize;
            const bool bulk = long_list && land + span4 <= STAGE;
            if (bulk) bulk_issue(stage + land, ci, e0, (int64_t)e0 + span4, &sm.mbar, lane);
            if (mode == ST_FILTER) {
              int4 *f4 = reinterpret_cast<int4 *>(stage);
              for (int i = lane; i < FILTER_WORDS / 4; i += 32) f4[i] = make_int4(0, 0, 0, 0);
            }
            for (int i = lane; i < hsize; i += 32) tab[i] = EMPTY;
            if (bulk) {
              failed = !bulk_wait(&sm.mbar, mbar_parity);
              src = stage + land + (b0 - e0);
            }
            __syncwarp();
            const uint32_t hmask = (uint32_t)hsize - 1u;
            if (!failed)
              for (int i = lane; i < blen; i += 32) {
                const int32_t key = i < 32 ? x0 : src[i];
                if (mode == ST_FILTER) {
                  const uint32_t h = InFilter::hash(key);
                  atomicOr(reinterpret_cast<unsigned *>(stage) + InFilter::word_of(h),
                           InFilter::bits_of(h));
                }
                uint32_t h = hash_slot(key, log2h) & ~3u;
                for (int c = 0; c < hsize; ++c) {
                  if (atomicCAS(&tab[h], EMPTY, key) == EMPTY) break;
                  h = (h + 1) & hmask;
                }
              }
            staged_log2h = log2h;
          } else {
            staged_list = stage;
            if (long_list && span4 <= STAGE) {
              bulk_issue(stage, ci, e0, (int64_t)e0 + span4, &sm.mbar, lane);
              failed = !bulk_wait(&sm.mbar, mbar_parity);
              staged_list = stage + (b0 - e0);
            } else {
              for (int i = lane; i < blen; i += 32) stage[i] = i < 32 ? x0 : ci[b0 + i];
            }
            staged_len = blen;
            staged_index = nullptr;
            staged_steps = 32 - __clz(blen);
            // the index goes behind the list
            const int behind = (int)((span4 + 3) & ~int64_t(3));
            if (!failed && behind + SI_BUCKETS + 1 <= STAGE) {
              uint32_t *index = reinterpret_cast<uint32_t *>(stage + behind);
              __syncwarp();
              for (int i = lane; i <= SI_BUCKETS; i += 32) index[i] = 0u;
              staged_last = (uint32_t)last;
              staged_bucket0 = InSorted::bucket_of(0u);
              __syncwarp();
              int most = 0;
              for (int i0 = 0; i0 < blen; i0 += 32) {
                const int i = i0 + (int)lane;
                if (i < blen) {
                  // the first entry of a bucket finds its end and writes both
                  const uint32_t b = InSorted::bucket_of(staged_last - (uint32_t)staged_list[i]);
                  if (i == 0 || InSorted::bucket_of(staged_last - (uint32_t)staged_list[i - 1]) != b) {
                    int e = i + 1;
                    while (e < blen &&
                           InSorted::bucket_of(staged_last - (uint32_t)staged_list[e]) == b)
                      ++e;
                    index[b - staged_bucket0] = (uint32_t)i | ((uint32_t)e << 16);
                    most = max(most, e - i);
                  }
                }
              }
              most = __reduce_max_sync(0xffffffffu, most);
              staged_index = index;
              staged_steps = 32 - __clz(most);
            }
          }
          __syncwarp();
          staged_mode = mode;
          staged = !failed;
        }
      }
      if (failed) break;

      // the start of the next window's probe runs into L2 while this batch is
      // looked up: the rows of the sources of one destination lie anywhere
      if (r.y > r.x) {
        const int32_t *q = ci + r.x;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(q));
        if (r.y - r.x > 32u) asm volatile("prefetch.global.L2 [%0];" ::"l"(q + 32));
      }

      const uint32_t first = incl - nq;
      const bool has = nq > 0;
      // up to four parts: at most six (part(u), part(w)) pairs go with part(v), and a
      // lane counts each in a field of one 64-bit word
      const bool few_parts = TASK && p <= 4 && uniform && total <= 32u * ((1u << FIELD) / 4u - 2u);
      const unsigned with = __ballot_sync(0xffffffffu, has);
      if (has) {
        const int c = __popc(with & ((1u << lane) - 1u));
        uint32_t part = 0;
        if (TASK) {  // part(u), from the CSR position of (u, v)
          int lo = 0, hi = p;
          while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (ecut_s[mid] < s0) lo = mid; else hi = mid;
          }
          part = (uint32_t)lo;
        }
        if (TASK && few_parts)  // only runs of one v are counted by fields
          part = (uint32_t)(FIELD * ((int)part * (p - j_part) - j_part));
        else if (TASK)
          part |= (uint32_t)(uniform ? j_part : part_of_dev(cuts_s, p, vl)) << 8;
        sm.rec[c] = make_uint4(s0, s1, a0 - 4u * first, part);
        if (!uniform) {
          sm.rng[c] = make_uint2(vb0, vb1);
          if (GRAPH) sm.v[c] = (uint32_t)vl;
        }
      }
      __syncwarp();
      unsigned long long packed = 0;
      uint32_t hits = 0;
      auto probe = [&](auto quads, auto make) {
        flat_rounds<decltype(quads)::value>(ci, sm.rec, total, first, has, lane, [&](int own, const int4 &w, uint32_t m, uint32_t) {
          if (!TASK && (!GRAPH || uniform)) {
            hits += make(own).count(w, m);
            return;
          }
          uint32_t h = make(own).bits(w, m);
          hits += __popc(h);
          if (GRAPH && !uniform && h)  // a mixed batch: in-edges of several graphs
            atomicAdd(&P.graph_count[d.gid[sm.v[own]]], (unsigned long long)__popc(h));
          if (!TASK) return;
          if (few_parts) {  // (part(u), part(w)) as a field of the lane's packed counters
            const int at = h ? (int)sm.rec[own].w : 0;
            while (h) {
              const int c = __ffs(h) - 1;
              const int32_t x = c == 0 ? w.x : c == 1 ? w.y : c == 2 ? w.z : w.w;
              const int kp = (x >= cut1) + (x >= cut2) + (x >= cut3);
              const int32_t end = kp == 0 ? cut1 : kp == 1 ? cut2 : kp == 2 ? cut3 : INT32_MAX;
              const uint32_t same = ((w.x < end ? 1u : 0u) | (w.y < end ? 2u : 0u) |
                                     (w.z < end ? 4u : 0u) | (w.w < end ? 8u : 0u)) & h;
              packed += (unsigned long long)__popc(same) << (at + FIELD * kp);
              h &= ~same;
            }
            return;
          }
          // per task: the hits of each (part(u), part(v), part(w)) among the lanes
          const uint32_t ij = h ? sm.rec[own].w : 0u;
          while (__any_sync(0xffffffffu, h != 0u)) {
            int key = -1;
            uint32_t same = 0;
            if (h) {
              const int c = __ffs(h) - 1;
              const int32_t x = c == 0 ? w.x : c == 1 ? w.y : c == 2 ? w.z : w.w;
              const int kp = part_of_dev(cuts_s, p, x);
              const int32_t end = cuts_s[kp + 1];
              same = ((w.x < end ? 1u : 0u) | (w.y < end ? 2u : 0u) | (w.z < end ? 4u : 0u) |
                      (w.w < end ? 8u : 0u)) & h;
              key = (int)(ij << 8) | kp;
              h &= ~same;
            }
            const uint32_t c = __popc(same);
            unsigned left = __ballot_sync(0xffffffffu, c != 0u);
            while (left) {
              const int k0 = __shfl_sync(0xffffffffu, key, __ffs(left) - 1);
              const unsigned sum = __reduce_add_sync(0xffffffffu, key == k0 ? c : 0u);
              if (lane == 0) {
                add_task((k0 >> 8) & 255, k0 >> 16, k0 & 255, sum);
              }
              left &= ~__ballot_sync(0xffffffffu, key == k0);
            }
          }
        });
      };
      if (uniform && staged && staged_mode == ST_BITMAP) {
        const InBitmap look{reinterpret_cast<const uint32_t *>(stage), staged_word0, staged_gw};
        probe(std::integral_constant<int, FL_QUADS>(), [&](int) { return look; });
      } else if (uniform && staged && staged_mode == ST_FILTER) {
        const InFilter look{reinterpret_cast<const uint32_t *>(stage), stage + FILTER_WORDS,
                            staged_log2h};
        probe(std::integral_constant<int, FL_QUADS>(), [&](int) { return look; });
      } else if (uniform && staged && staged_mode == ST_HASH) {
        const InHash look{stage, staged_log2h};
        probe(std::integral_constant<int, 1>(), [&](int) { return look; });
      } else if (uniform && staged) {
        const InSorted look{staged_list, staged_index, staged_len, staged_steps, staged_last,
                            staged_bucket0};
        probe(std::integral_constant<int, 1>(), [&](int) { return look; });
      } else if (uniform) {
        const InPlace look{ci, b0, b1};
        probe(std::integral_constant<int, 1>(), [&](int) { return look; });
      } else {
        probe(std::integral_constant<int, 1>(), [&](int own) {
          const uint2 b = sm.rng[max(own, 0)];
          return InPlace{ci, b.x, b.y};
        });
      }
      if (!TASK) acc += hits;
      if (TASK && few_parts) {
        const int nk = p - j_part;
        for (int x = 0; x < (j_part + 1) * nk; ++x) {
          const uint32_t c = (uint32_t)(packed >> (FIELD * x)) & ((1u << FIELD) - 1u);
          const uint32_t sum = __reduce_add_sync(0xffffffffu, c);
          if ((int)lane == x) field_sum += sum;
        }
      }
      if (GRAPH && uniform) {
        run_hits += hits;
        if (base - run_from >= FL_FLUSH) flush_graph();
      }
      __syncwarp();
    }
    if (TASK) flush_fields();
    if (GRAPH) flush_graph();
    if (failed) break;
    it = __shfl_sync(0xffffffffu, it_next, 0);
  }
  if (!TASK) {
    acc = warp_sum(acc);
    if (lane == 0 && acc) {
      const int32_t tb = P.nd > 1 ? P.descs[cur_desc].task_base : P.one.task_base;
      atomicAdd(&P.task_count[tb], acc);
    }
  }
  if (failed && lane == 0) atomicExch(P.status, STATUS_COPY_WAIT);
  if (in_table) {
    __syncthreads();
    for (int i = threadIdx.x; i < (int)P.ntasks; i += FL_NT)
      if (table[i]) atomicAdd(&P.task_count[i], table[i]);
  }
}

template <int MODE>
bbtc_status flat_configure(int *blocks_per_sm) {
  const size_t smem = flat_smem_bytes() + (MODE & FL_MODE_TASK ? 8 * FL_TABLE : 0);
  BBTC_CUDA(cudaFuncSetAttribute(k_flat<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem));
  BBTC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_flat<MODE>, FL_NT, smem));
  if (*blocks_per_sm < 1) *blocks_per_sm = 1;
  return BBTC_OK;
}

}  // namespace

// ------------------------------------------------------- building the records

namespace {

// In-edges counted by the dense core, per core destination, taken off the
// in-degrees: CTA-local counts of the core's work items, one atomic per
// destination and CTA.
constexpr int FC_COLS = 8192;  // core destinations counted on chip: the top ones
__global__ void __launch_bounds__(512) k_flat_minus_core(const int4 *__restrict__ items,
                                                         const unsigned *__restrict__ count,
                                                         unsigned cap,
                                                         int32_t chunk,
                                                         const int32_t *__restrict__ colidx,
                                                         int64_t n, unsigned *__restrict__ hist) {
  __shared__ unsigned cnt[FC_COLS];
  const int64_t first = n > FC_COLS ? n - FC_COLS : 0;
  for (int i = threadIdx.x; i < FC_COLS; i += 512) cnt[i] = 0;
  __syncthreads();
  const int64_t nw = (int64_t)gridDim.x * 16;
  const int64_t total = *count < cap ? *count : cap;
  for (int64_t x = (int64_t)blockIdx.x * 16 + (threadIdx.x >> 5); x < total; x += nw) {
    const int4 it = items[x];
    const uint32_t x0 = (uint32_t)it.z, re = (uint32_t)it.w;
    const uint32_t len = re - x0 < (uint32_t)chunk ? re - x0 : (uint32_t)chunk;
    for (uint32_t i = lane_id(); i < len; i += 32) {
      const int64_t v = colidx[x0 + i];
      if (v >= first) atomicAdd(&cnt[v - first], 1u);
      else atomicSub(&hist[v], 1u);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < FC_COLS; i += 512)
    if (cnt[i]) atomicSub(&hist[first + i], cnt[i]);
}

__device__ __forceinline__ bool in_core(const unsigned *__restrict__ flags, int64_t u0, int32_t v0,
                                        int32_t u, int32_t v) {
  if (!flags || v < v0 || u < u0) return false;
  const uint32_t x = (uint32_t)(u - u0);
  return ((flags[x >> 5] >> (x & 31u)) & 1u) != 0u;
}

// Direct scatter (small graphs): each edge's record to its destination's next
// slot. The top FS_HUB destinations, which receive most in-edges of a skewed
// graph, are counted per CTA first and reserved with one atomic each.
constexpr int FS_NT = 512;
constexpr int FS_HUB = 8192;
__global__ void __launch_bounds__(FS_NT) k_flat_scatter(const int64_t *__restrict__ rowptr,
                                                        const int32_t *__restrict__ colidx,
                                                        const int32_t *__restrict__ esrc,
                                                        int64_t n, int64_t m,
                                                        const unsigned *__restrict__ flags,
                                                        int64_t u0, int32_t v0,
                                                        unsigned *__restrict__ cursor,
                                                        uint2 *__restrict__ rec) {
  __shared__ unsigned sm[FS_HUB];
  const int64_t hub0 = n > FS_HUB ? n - FS_HUB : 0;
  for (int i = threadIdx.x; i < FS_HUB; i += FS_NT) sm[i] = 0;
  const int64_t per = (m + gridDim.x - 1) / gridDim.x;
  const int64_t b0 = (int64_t)blockIdx.x * per;
  const int64_t b1 = b0 + per < m ? b0 + per : m;
  __syncthreads();
  for (int64_t e = b0 + threadIdx.x; e < b1; e += FS_NT) {
    const int32_t v = colidx[e];
    if (v >= hub0 && !in_core(flags, u0, v0, esrc[e], v)) atomicAdd(&sm[v - hub0], 1u);
  }
  __syncthreads();
  for (int64_t i = threadIdx.x; i < n - hub0; i += FS_NT)
    if (sm[i]) sm[i] = atomicAdd(&cursor[hub0 + i], sm[i]);
  __syncthreads();
  constexpr int ILP = 4;
  for (int64_t e = b0 + threadIdx.x; e < b1; e += (int64_t)FS_NT * ILP) {
    int32_t v[ILP], u[ILP];
    unsigned at[ILP];
#pragma unroll
    for (int r = 0; r < ILP; ++r) {
      const int64_t x = e + (int64_t)r * FS_NT;
      v[r] = -1;
      if (x < b1) {
        v[r] = colidx[x];
        u[r] = esrc[x];
        if (in_core(flags, u0, v0, u[r], v[r])) v[r] = -1;
      }
    }
#pragma unroll
    for (int r = 0; r < ILP; ++r)
      if (v[r] >= 0)
        at[r] = v[r] >= hub0 ? atomicAdd(&sm[v[r] - hub0], 1u) : atomicAdd(&cursor[v[r]], 1u);
#pragma unroll
    for (int r = 0; r < ILP; ++r)
      if (v[r] >= 0) {
        const int64_t x = e + (int64_t)r * FS_NT;
        rec[at[r]] = make_uint2((uint32_t)x + 1u, (uint32_t)rowptr[u[r] + 1]);
      }
  }
}

// Two phases for large graphs, where a direct scatter writes whole sectors for
// 8 bytes at random places: partition tiles of edges by destination range into
// a temporary array (records and destinations, coalesced runs), then place
// them; see plan.cu, which does the same for the per-part records.
constexpr int FB_T = 4096, FB_NT = 512, FB_B = 512, FB_LUT = 4096;
// (26 M records of R-MAT scale 21: direct 0.39 ms, two phases 0.62)
constexpr int64_t FB_MIN_EDGES = 48ll << 20;
static_assert(FB_NT == FB_B && FB_T == 8 * FB_NT, "partition layout");

__global__ void k_flat_bounds(const uint32_t *__restrict__ inptr, int64_t n,
                              int32_t *__restrict__ bnd, unsigned *__restrict__ bcur) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b > FB_B) return;
  const uint64_t M = inptr[n];
  int64_t idx = n;
  if (b == 0) idx = 0;
  else if (b < FB_B)
    idx = lower_bound_dev<uint32_t, int64_t>(inptr, 0, n, (uint32_t)((M * b + FB_B - 1) / FB_B));
  bnd[b] = (int32_t)idx;
  if (b < FB_B) bcur[b] = inptr[idx];
}

__global__ void __launch_bounds__(FB_NT, 2)
    k_flat_partition(const int64_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                     const int32_t *__restrict__ esrc, int64_t m,
                     const unsigned *__restrict__ flags, int64_t u0, int32_t v0,
                     const int32_t *__restrict__ bnd_g, unsigned *__restrict__ bcur,
                     uint2 *__restrict__ tmp_rec, int32_t *__restrict__ tmp_v) {
  __shared__ int32_t bnd[FB_B + 1];
  __shared__ unsigned cnt[FB_B], loff[FB_B], gbase[FB_B];
  __shared__ unsigned scan_tmp[FB_NT / 32 + 1];
  __shared__ uint16_t sb[FB_T];
  __shared__ uint16_t lut[FB_LUT + 1];
  extern __shared__ __align__(16) unsigned char fb_smem[];
  uint2 *stage = reinterpret_cast<uint2 *>(fb_smem);
  int32_t *stage_v = reinterpret_cast<int32_t *>(fb_smem + sizeof(uint2) * FB_T);
  for (int i = threadIdx.x; i <= FB_B; i += FB_NT) bnd[i] = bnd_g[i];
  __syncthreads();
  int shift = 0;
  while (((int64_t)FB_LUT << shift) < (int64_t)bnd[FB_B]) ++shift;
  for (int k = threadIdx.x; k <= FB_LUT; k += FB_NT) {
    const int64_t x = (int64_t)k << shift;
    int lo = 0, hi = FB_B;  // last bucket with bnd[lo] <= x
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (bnd[mid] <= x) lo = mid; else hi = mid;
    }
    lut[k] = (uint16_t)lo;
  }
  __syncthreads();
  int32_t pv[8], pu[8];
  const int64_t tstep = (int64_t)gridDim.x * FB_T;
  auto load_tile = [&](int64_t tt0) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int64_t idx = tt0 + (int)threadIdx.x + k * FB_NT;
      pv[k] = -1;
      pu[k] = 0;
      if (idx < m) {
        pv[k] = colidx[idx];
        pu[k] = esrc[idx];
      }
    }
  };
  load_tile((int64_t)blockIdx.x * FB_T);
  for (int64_t t0 = (int64_t)blockIdx.x * FB_T; t0 < m; t0 += tstep) {
    int32_t cv[8], cu[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      cv[k] = pv[k];
      cu[k] = pu[k];
    }
    load_tile(t0 + tstep);
    cnt[threadIdx.x] = 0;
    __syncthreads();
    uint32_t fk[8];
    int bk[8];
    unsigned lr[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      bk[k] = -1;
      if (cv[k] >= 0 && !in_core(flags, u0, v0, cu[k], cv[k])) {
        fk[k] = (uint32_t)rowptr[cu[k] + 1];
        const int32_t x = cv[k];
        int lo = lut[x >> shift], hi = lut[(x >> shift) + 1] + 1;
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (bnd[mid] <= x) lo = mid; else hi = mid;
        }
        bk[k] = lo;
        lr[k] = atomicAdd(&cnt[lo], 1u);
      }
    }
    __syncthreads();
    unsigned total = 0;
    const unsigned c = cnt[threadIdx.x];
    loff[threadIdx.x] = block_exclusive_scan<unsigned, FB_NT>(c, scan_tmp, &total);
    if (c) gbase[threadIdx.x] = atomicAdd(&bcur[threadIdx.x], c);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (bk[k] >= 0) {
        const unsigned slot = loff[bk[k]] + lr[k];
        const int64_t idx = t0 + (int)threadIdx.x + k * FB_NT;
        stage[slot] = make_uint2((uint32_t)idx + 1u, fk[k]);
        stage_v[slot] = cv[k];
        sb[slot] = (uint16_t)bk[k];
      }
    __syncthreads();
    for (unsigned i = threadIdx.x; i < total; i += FB_NT) {
      const int b = sb[i];
      const uint64_t o = (uint64_t)gbase[b] + (i - loff[b]);
      tmp_rec[o] = stage[i];
      tmp_v[o] = stage_v[i];
    }
    __syncthreads();
  }
}

__global__ void k_flat_place(const uint2 *__restrict__ tmp_rec, const int32_t *__restrict__ tmp_v,
                             const uint32_t *__restrict__ inptr, int64_t n,
                             unsigned *__restrict__ cursor, uint2 *__restrict__ rec) {
  const int64_t M = inptr[n];
  constexpr int ILP = 4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < M; x += stride * ILP) {
    uint2 r[ILP];
    int32_t v[ILP];
    unsigned pos[ILP];
#pragma unroll
    for (int k = 0; k < ILP; ++k)
      if (x + k * stride < M) {  // read once: evict first
        r[k] = __ldcs(tmp_rec + x + k * stride);
        v[k] = __ldcs(tmp_v + x + k * stride);
      }
#pragma unroll
    for (int k = 0; k < ILP; ++k)
      if (x + k * stride < M) pos[k] = atomicAdd(&cursor[v[k]], 1u);
#pragma unroll
    for (int k = 0; k < ILP; ++k)
      if (x + k * stride < M) rec[pos[k]] = r[k];
  }
}

// in-degree of each position: the undirected degree minus the out-degree
__global__ void k_flat_indegree(const int64_t *__restrict__ rowptr, const int32_t *__restrict__ perm,
                                const int32_t *__restrict__ deg, int64_t n,
                                unsigned *__restrict__ hist) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r <= n;
       r += (int64_t)gridDim.x * blockDim.x)
    hist[r] = r < n ? (unsigned)(deg[perm[r]] - (int32_t)(rowptr[r + 1] - rowptr[r])) : 0u;
}

// the same by counting the edges (a union of handles has no degrees); the top
// positions, which receive most edges of a skewed graph, are counted per CTA
__global__ void __launch_bounds__(512) k_flat_count(const int32_t *__restrict__ colidx, int64_t m,
                                                    int64_t n, unsigned *__restrict__ hist) {
  __shared__ unsigned cnt[FC_COLS];
  const int64_t first = n > FC_COLS ? n - FC_COLS : 0;
  for (int i = threadIdx.x; i < FC_COLS; i += 512) cnt[i] = 0;
  __syncthreads();
  for (int64_t e = (int64_t)blockIdx.x * 512 + threadIdx.x; e < m; e += (int64_t)gridDim.x * 512) {
    const int64_t v = colidx[e];
    if (v >= first) atomicAdd(&cnt[v - first], 1u);
    else atomicAdd(&hist[v], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < FC_COLS; i += 512)
    if (cnt[i]) atomicAdd(&hist[first + i], cnt[i]);
}

}  // namespace

void free_flat(Flat *f, cudaStream_t s) {
  dfree(f->rec, s);
  dfree(f->inptr, s);
  *f = Flat();
}

bbtc_status build_flat(const bbtc_graph *g, Plan &pl, Flat &f, bool use_core, cudaStream_t s) {
  const int64_t n = g->n, m = g->m;
  const Core none;
  const Core &core = use_core ? pl.core : none;
  if (core.bits && core.all) {
    // every pair of a source's edges is counted in the core: no list is probed
    unsigned items = 0;
    BBTC_CUDA(cudaMemcpyAsync(&items, core.count, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
    BBTC_CUDA(cudaStreamSynchronize(s));
    pl.core.nitems = std::min<int64_t>(items, core.cap);
    f.ready = true;
    return BBTC_OK;
  }
  if (m == 0) {
    f.ready = true;
    return BBTC_OK;
  }
  Scratch scratch(s);
  unsigned *hist = nullptr;
  BBTC_TRY(scratch.get(&hist, n + 1));
  BBTC_TRY(dalloc_n(&f.inptr, n + 1, s));
  if (g->deg && g->perm) {
    k_flat_indegree<<<grid_for(n + 1, 256, 16), 256, 0, s>>>(g->rowptr, g->perm, g->deg, n, hist);
  } else {
    BBTC_CUDA(cudaMemsetAsync(hist, 0, sizeof(unsigned) * (size_t)(n + 1), s));
    k_flat_count<<<grid_for(m, 512 * 16, 2), 512, 0, s>>>(g->colidx, m, n, hist);
  }
  BBTC_LAUNCH_CHECK();
  if (core.bits) {
    k_flat_minus_core<<<(unsigned)num_sms() * 2, 512, 0, s>>>(core.items, core.count, core.cap,
                                                             CORE_CHUNK, g->colidx, n, hist);
    BBTC_LAUNCH_CHECK();
  }
  BBTC_TRY(exclusive_scan_u32(hist, f.inptr, hist, n + 1, s));  // hist: the cursors
  uint32_t records = 0;
  unsigned items = 0;
  BBTC_CUDA(cudaMemcpyAsync(&records, f.inptr + n, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
  if (core.bits)
    BBTC_CUDA(cudaMemcpyAsync(&items, core.count, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
  BBTC_CUDA(cudaStreamSynchronize(s));
  f.records = records;
  if (core.bits) pl.core.nitems = std::min<int64_t>(items, core.cap);
  BBTC_TRY(dalloc_n(&f.rec, f.records, s));
  // about 32 items per resident warp, 64 to 4,096 in-edges each (or the caller's
  // choice); 64 and 128 items staged each list more often (R-MAT scale 21 at p = 4,
  // per task: 3.16, 3.36 and 3.36 ms; scale 22: 4.86, 4.91 and 5.12 ms)
  const int64_t warps = (int64_t)num_sms() * 24;
  int64_t chunk = f.records / (warps * 32);
  chunk = chunk < 64 ? 64 : (chunk > 4096 ? 4096 : chunk);
  // too few records for every warp to get an item: the time is one item's chain of
  // loads, so items are shorter. A G(n, m) of 27 K edges by sorted search with
  // per-task counts took 145, 103, 85 and 73 us with items of 64, 32, 16 and 8;
  // R-MAT scale 15 at p = 8 78, 71, 71 and 81
  if (f.records < warps * 64) chunk = 16;
  if (pl.chunk_req > 0) chunk = pl.chunk_req;
  f.chunk = chunk;
  f.nitems = (f.records + chunk - 1) / chunk;
  f.ready = true;
  f.bytes = (uint64_t)f.records * 8 + (uint64_t)(n + 1) * 4;
  if (f.records == 0) return BBTC_OK;
  uint2 *tmp_rec = nullptr;
  int32_t *tmp_v = nullptr;
  bool two_phase = f.records >= FB_MIN_EDGES && n > FB_B;
  if (two_phase && (scratch.get(&tmp_rec, f.records) != BBTC_OK ||
                    scratch.get(&tmp_v, f.records) != BBTC_OK)) {
    two_phase = false;  // no room for the temporary arrays: scatter directly
    clear_error();
  }
  if (two_phase) {
    int32_t *bnd = nullptr;
    unsigned *bcur = nullptr;
    BBTC_TRY(scratch.get(&bnd, FB_B + 1));
    BBTC_TRY(scratch.get(&bcur, FB_B));
    k_flat_bounds<<<(FB_B + 1 + 127) / 128, 128, 0, s>>>(f.inptr, n, bnd, bcur);
    BBTC_LAUNCH_CHECK();
    const size_t smem = (sizeof(uint2) + sizeof(int32_t)) * FB_T;
    BBTC_CUDA(cudaFuncSetAttribute(k_flat_partition, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)smem));
    k_flat_partition<<<(unsigned)num_sms() * 2, FB_NT, smem, s>>>(
        g->rowptr, g->colidx, g->esrc, m, core.flags, core.u0, core.v0, bnd, bcur, tmp_rec, tmp_v);
    BBTC_LAUNCH_CHECK();
    k_flat_place<<<grid_for(f.records, 256, 8), 256, 0, s>>>(tmp_rec, tmp_v, f.inptr, n, hist,
                                                            f.rec);
    BBTC_LAUNCH_CHECK();
  } else {
    k_flat_scatter<<<grid_for(m, FS_NT * 32, 4), FS_NT, 0, s>>>(
        g->rowptr, g->colidx, g->esrc, n, m, core.flags, core.u0, core.v0, hist, f.rec);
    BBTC_LAUNCH_CHECK();
  }
  return BBTC_OK;
}

FlatDesc flat_desc(const bbtc_graph *g, const Plan &pl, const Flat &f, int64_t item_base,
                   int32_t task_base) {
  FlatDesc d;
  d.rec = f.rec;
  d.inptr = f.inptr;
  d.rowptr = g->rowptr;
  d.colidx = g->colidx;
  d.gid = g->gid;
  d.cuts = pl.cuts;
  d.n = g->n;
  d.records = f.records;
  d.nitems = f.nitems;
  d.item_base = item_base;
  d.item0 = 0;
  d.chunk = f.chunk;
  d.flags = pl.kernel_mode == BBTC_KERNEL_HASHMAP     ? 1
            : pl.kernel_mode == BBTC_KERNEL_INTERSECT ? 0
                                                      : 2 | (pl.hash_threshold << 2);
  d.p = pl.p;
  d.task_base = task_base;
  return d;
}

bbtc_status configure_flat_kernels(int *blocks_per_sm) {
  // the attributes and occupancies are per device: set and query them once
  static std::mutex mu;
  static int cached[64][4];
  static bool done[64] = {false};
  int dev = 0;
  BBTC_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) {
    set_error("device ordinal %d out of range", dev);
    return BBTC_EINVAL;
  }
  std::lock_guard<std::mutex> lk(mu);
  if (!done[dev]) {
    BBTC_TRY(flat_configure<0>(&cached[dev][0]));
    BBTC_TRY(flat_configure<1>(&cached[dev][1]));
    BBTC_TRY(flat_configure<2>(&cached[dev][2]));
    BBTC_TRY(flat_configure<3>(&cached[dev][3]));
    done[dev] = true;
  }
  for (int i = 0; i < 4; ++i) blocks_per_sm[i] = cached[dev][i];
  return BBTC_OK;
}

bbtc_status flat_launch(const FlatDesc &one, const FlatDesc *descs, int32_t nd, int64_t nitems,
                        unsigned long long *head, unsigned long long *task_count, int64_t ntasks,
                        bool tasks, unsigned long long *graph_count, int32_t *status,
                        const unsigned long long *t0, uint32_t timeout_ms,
                        const int *blocks_per_sm, cudaStream_t s) {
  if (nitems <= 0) return BBTC_OK;
  FlatLaunch P;
  P.one = one;
  P.descs = descs;
  P.nd = nd;
  P.nitems = nitems;
  P.head = head;
  P.task_count = task_count;
  P.graph_count = graph_count;
  P.ntasks = ntasks;
  P.status = status;
  P.t0 = t0;
  P.timeout_ns = (uint64_t)timeout_ms * 1000000ull;
  const int mode = (graph_count ? FL_MODE_GRAPH : 0) | (tasks && one.p > 1 ? FL_MODE_TASK : 0);
  // (a launch with fewer task counters than configured for may hold more blocks)
  int64_t blocks = (int64_t)num_sms() * (mode & FL_MODE_TASK ? FL_CTAS : blocks_per_sm[mode]);
  blocks = std::min<int64_t>(blocks, (nitems + FL_WARPS - 1) / FL_WARPS);
  const bool table = (mode & FL_MODE_TASK) != 0 && ntasks <= FL_TABLE;
  const size_t smem = flat_smem_bytes() + (table ? 8 * (size_t)ntasks : 0);
  switch (mode) {
    case 0: k_flat<0><<<(unsigned)blocks, FL_NT, smem, s>>>(P); break;
    case 1: k_flat<1><<<(unsigned)blocks, FL_NT, smem, s>>>(P); break;
    case 2: k_flat<2><<<(unsigned)blocks, FL_NT, smem, s>>>(P); break;
    default: k_flat<3><<<(unsigned)blocks, FL_NT, smem, s>>>(P); break;
  }
  BBTC_LAUNCH_CHECK();
  return BBTC_OK;
}

}  // namespace bbtc
