// count.cu -- triangle counting task by task (a9), the reduction of the per-task
// counts (a10), and the host side of all resident counts.
//
// k_count serves the calls that need the tasks one by one: a share of them
// (task_mask), their cycles, and block-wise streaming. All other counts walk the
// in-edges once for all tasks (flat.cu) and the hubs as bitmaps (core.cu).
//
// A task t = (i, j, k) counts, for every edge (u, v) of G_ij, the common
// elements of N(G_ik, u) and N(G_jk, v) (Sec. 4.3, Alg. 5 / Alg. 6). The
// kernel walks G_ij's edges grouped by their destination v (the in-edges of
// each v in V_j that come from V_i, one contiguous range per block) and, for
// each, looks up the elements of N(G_ik, u) that lie above v in N(G_jk, v).
// Elements of N(G_ik, u) at or below v cannot be in N(G_jk, v) (every entry
// of N(v) is above v), so the count equals Alg. 5's |N(G_ik,u) ∩ N(G_jk,v)|.
//
// Work: a persistent grid; each warp takes work items (task, in-edge range)
// from a global counter, heaviest task first, until none remain.
#include <algorithm>
#include <mutex>
#include <vector>

#include "flat.cuh"
#include "graph.cuh"
#include "primitives.cuh"
#include "stage.cuh"

namespace bbtc {

namespace {

constexpr int CT_NT = 256;

struct CountParams {
  const TaskDesc *desc;  // per task (Alg. 4 order): where its three blocks live
  const WorkItem *items;
  int64_t nitems;
  unsigned long long *head;
  unsigned long long *task_count;
  unsigned long long *vcount;       // per-vertex counts by position (MODE & 1)
  const int32_t *gid;               // graph of each position (MODE & 2)
  unsigned long long *graph_count;  // per-graph counts (MODE & 2)
  unsigned long long *task_cycles;  // nullable: SM cycles spent on each task's items
  unsigned *edge_sup;               // per-edge support by position in the block columns (MODE & 4)
  const uint8_t *task_mask;         // nullable: items of tasks whose byte is 0 are skipped
  int32_t *status;
  uint64_t timeout_ns;
};

constexpr int MODE_VERTEX = 1, MODE_GRAPH = 2, MODE_EDGE = 4;

// Per-batch lane records, shared by the warp: where each in-edge's probes
// start in the flattened probe sequence and where they come from.
struct alignas(16) LaneRec {
  int64_t b0[32];     // N(G_jk, v) range of each lane (mixed batches only)
  int64_t b1[32];
  uint32_t s0[32];    // first probe element (local column index) of each lane's in-edge
  uint32_t incl[32];  // inclusive prefix of the probe counts
  int32_t u[32];
  int32_t v[32];
  unsigned long long mbar;  // completion of bulk copies into the warp's stage
};

// Runs the flattened probes of one batch: probe q (0 <= q < total) belongs to
// the lane-record o whose inclusive prefix first exceeds q and reads column
// rec.s0[o] + q - (prefix before o). Lane l takes q = l, l + 32, ...; U probes
// per lane per round have their loads issued before any lookup, so each lane
// keeps U global loads in flight (4 suits the one-load lookups; the halving
// searches, which keep more registers live, take 3). Column indices are local
// to the block arrays and below 2^32.
template <int U, typename OnHit, typename Lookup>
__device__ __forceinline__ void probe_batch(const int32_t *__restrict__ ci_ik, const LaneRec &rec,
                                            uint32_t total, unsigned lane, OnHit &on_hit,
                                            Lookup lookup) {
  int o = 0;
  uint32_t o_end = rec.incl[0];
  uint32_t addr = rec.s0[0];  // column of probe q is addr + q (mod 2^32)
  uint32_t qb = lane;
  // full rounds: every lane's U probes exist (the test is warp-uniform)
  for (; qb - lane + 32u * U <= total; qb += 32u * U) {
    int32_t wv[U];
    int own[U];
    uint32_t qpos[U];
#pragma unroll
    for (int r = 0; r < U; ++r) {
      const uint32_t q = qb + 32u * r;
      while (q >= o_end) {
        ++o;
        const uint32_t prev_end = o_end;
        o_end = rec.incl[o];
        addr = rec.s0[o] - prev_end;
      }
      qpos[r] = addr + q;
      wv[r] = ci_ik[qpos[r]];
      own[r] = o;
    }
#pragma unroll
    for (int r = 0; r < U; ++r)
      if (lookup(wv[r], own[r])) on_hit(wv[r], own[r], qpos[r]);
  }
  // the last, partial round
  if (qb - lane < total) {
    int32_t wv[U];
    int own[U];
    uint32_t qpos[U];
#pragma unroll
    for (int r = 0; r < U; ++r) {
      const uint32_t q = qb + 32u * r;
      own[r] = -1;
      if (q < total) {
        while (q >= o_end) {
          ++o;
          const uint32_t prev_end = o_end;
          o_end = rec.incl[o];
          addr = rec.s0[o] - prev_end;
        }
        qpos[r] = addr + q;
        wv[r] = ci_ik[qpos[r]];
        own[r] = o;
      }
    }
#pragma unroll
    for (int r = 0; r < U; ++r)
      if (own[r] >= 0 && lookup(wv[r], own[r])) on_hit(wv[r], own[r], qpos[r]);
  }
}

constexpr int UNIFORM_MIN = 4;  // a run of >= 4 in-edges into one v is a uniform batch

template <int MODE>
__global__ void __launch_bounds__(CT_NT, 3) k_count(CountParams P) {
  constexpr bool PER_VERTEX = (MODE & MODE_VERTEX) != 0;
  constexpr bool PER_GRAPH = (MODE & MODE_GRAPH) != 0;
  constexpr bool PER_EDGE = (MODE & MODE_EDGE) != 0;
  extern __shared__ __align__(16) unsigned char count_smem_raw[];
  const unsigned lane = threadIdx.x & 31u;
  const int warp = threadIdx.x >> 5;
  int32_t *stage = reinterpret_cast<int32_t *>(count_smem_raw) + warp * (STAGE + 4);
  LaneRec &rec = reinterpret_cast<LaneRec *>(count_smem_raw + (size_t)(CT_NT / 32) * (STAGE + 4) *
                                                                  sizeof(int32_t))[warp];
  if (lane == 0) {
    stage[STAGE] = 0;  // zero guard word after the stage
    mbar_init(&rec.mbar);
    mbar_init_fence();
  }
  __syncwarp();
  uint32_t mbar_parity = 0;  // parity of rec.mbar's next phase
  const uint64_t t_start = P.timeout_ns ? global_ns() : 0;
  // (task, v) whose N(G_jk, v) is in `stage`, and how it is stored
  unsigned long long staged_tag = ~0ull;
  int staged_len = 0, staged_log2h = 0, staged_mode = ST_NONE, staged_off = 0;
  uint32_t staged_word0 = 0;   // bitmap: first word of its window
  uint32_t staged_gw = STAGE;  // bitmap: index of its zero guard word
  bool failed = false;

  for (;;) {
    unsigned long long it = 0;
    if (lane == 0) it = atomicAdd(P.head, 1ull);
    it = __shfl_sync(0xffffffffu, it, 0);
    if (it >= (unsigned long long)P.nitems) break;
    if (P.timeout_ns && global_ns() - t_start > P.timeout_ns) {
      if (lane == 0) atomicExch(P.status, STATUS_TIMEOUT);
      break;
    }
    const WorkItem w = P.items[it];
    const int t = w.task;
    if (P.task_mask && P.task_mask[t] == 0) continue;  // another rank's task
    const long long t_item = P.task_cycles ? clock64() : 0;
    const int kflag = w.flags & 3;  // 0 INTERSECT, 1 HASHMAP, 2 AUTO (per list)
    const int hash_min = w.flags >> 2;  // AUTO: longer lists hash, shorter ones sorted
    const TaskDesc &d = P.desc[t];
    // block arrays are indexed locally: in-edge x at [x - ie_off], column
    // position q at [q - ci_*_off] (the offsets are 0 when the plan is resident)
    const InEdge *__restrict__ ie = d.ie;
    const int64_t ie_off = d.ie_off;
    const uint32_t *__restrict__ rp_ik = d.rp_ik;
    const uint32_t *__restrict__ rp_jk = d.rp_jk;
    const int32_t *__restrict__ ci_ik = d.ci_ik;
    const int32_t *__restrict__ ci_jk = d.ci_jk;
    const int64_t ik_off = d.ci_ik_off, jk_off = d.ci_jk_off;
    const int64_t rs_ik = d.rs_ik, rs_jk = d.rs_jk;
    const int32_t c_i = d.c_i, c_j = d.c_j;
    const bool diag = d.diag != 0;
    unsigned long long acc = 0;

    int64_t base = w.x0;
    // the records (u, v, e, f) of the current window of 32 in-edges; lanes past
    // the item hold v = -1
    InEdge r = base + lane < w.x1 ? ie[base + lane - ie_off] : make_int4(0, -1, 0, 0);
    while (base < w.x1) {
      const int64_t batch_x0 = base;  // in-edge of lane 0; lane l's is batch_x0 + l
      const int32_t v = r.y;
      const bool valid = v >= 0;
      // in-edges are sorted by destination: lanes equal to lane 0's v form a prefix
      const int32_t v0 = __shfl_sync(0xffffffffu, v, 0);
      const unsigned eq = __ballot_sync(0xffffffffu, valid && v == v0);
      const unsigned vmask = __ballot_sync(0xffffffffu, valid);
      const int run0 = __popc(eq);
      const int nvalid = __popc(vmask);
      const bool uniform = run0 >= UNIFORM_MIN || run0 == nvalid;
      int nb;  // in-edges handled by this batch
      if (uniform) {
        nb = run0;
      } else {
        // cut before the last run, which may continue past the batch
        const int32_t vprev = __shfl_up_sync(0xffffffffu, v, 1);
        const unsigned heads = __ballot_sync(0xffffffffu, valid && (lane == 0 || v != vprev));
        const int last_head = 31 - __clz(heads);
        nb = (base + 32 < w.x1 && last_head > 0) ? last_head : nvalid;
      }
      base += nb;
      // the next window's records into registers while this batch runs, and the
      // one after it into L2
      const InEdge rn = base + lane < w.x1 ? ie[base + lane - ie_off] : make_int4(0, -1, 0, 0);
      if (base + 32 + lane < w.x1)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(ie + (base + 32 + lane - ie_off)));
      const bool active = (int)lane < nb;
      const int32_t u = r.x;
      const int64_t e = (int64_t)(uint32_t)r.z;
      const int64_t f = (int64_t)(uint32_t)r.w;
      r = rn;
      // N(G_jk, v): direct row pointers of block (j, k); [b0, b1) local to ci_jk
      int64_t b0 = 0, b1 = 0;
      if (uniform) {
        if (lane == 0) {
          b0 = (int64_t)rp_jk[(v0 - c_j) * rs_jk] - jk_off;
          b1 = (int64_t)rp_jk[(v0 - c_j) * rs_jk + 1] - jk_off;
        }
        b0 = __shfl_sync(0xffffffffu, b0, 0);
        b1 = __shfl_sync(0xffffffffu, b1, 0);
      } else if (active) {
        b0 = (int64_t)rp_jk[(v - c_j) * rs_jk] - jk_off;
        b1 = (int64_t)rp_jk[(v - c_j) * rs_jk + 1] - jk_off;
      }
      // N(G_ik, u) restricted to entries above v: for k == j the entries of u's
      // run in G_ij after (u, v) itself, [e + 1, f) from the record; else u's
      // run in G_ik from the split table. [s0, s1) local to ci_ik
      int64_t s0 = 0, s1 = 0;
      if (active && b1 > b0) {
        if (diag) {
          s0 = e + 1 - ik_off;
          s1 = f - ik_off;
        } else {
          s0 = (int64_t)rp_ik[(u - c_i) * rs_ik] - ik_off;
          s1 = (int64_t)rp_ik[(u - c_i) * rs_ik + 1] - ik_off;
        }
      }
      const uint32_t len = (uint32_t)(s1 - s0);
      const uint32_t total = __reduce_add_sync(0xffffffffu, len);
      if (total == 0) continue;

      // stage N(G_jk, v) once per (task, v) in one of three forms:
      //  - bitmap over [first, last] of the list (Alg. 6's direct-address
      //    table H, windowed to the list's value range) when that range has at
      //    most STAGE * 32 values;
      //  - open-addressed hash table (at most half full) otherwise;
      //  - sorted copy (bbTC-Intersect, Alg. 5), searched by halving.
      // The item's kernel flag picks sorted (INTERSECT), bitmap-else-hash
      // (HASHMAP), or, per list, bitmap, then hash for long lists, then sorted
      // (AUTO).
      const int blen = (int)(b1 - b0);
      bool staged = false;
      if (uniform && blen >= MIN_STAGE) {
        const unsigned long long tag =
            ((unsigned long long)(uint32_t)t << 33) | ((unsigned long long)(uint32_t)v0 << 2);
        if (tag == staged_tag) {
          staged = true;
        } else if (nb == 32 || total >= (uint32_t)blen / 2) {
          // the list's first 32 entries, one per lane, and its last entry, in
          // one round of loads: the value range comes from them
          const int32_t x0 = (int)lane < blen ? ci_jk[b0 + lane] : 0;
          int32_t lastv = 0;
          if (lane == 0 && blen > 32) lastv = ci_jk[b1 - 1];
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
            // A list of at least BULK_STAGE_MIN entries arrives by one bulk
            // copy (TMA) of its aligned 16-byte span: a sorted copy straight
            // into the stage, for the tables into the free words beside them,
            // from which the table is then built. Shorter lists, and lists
            // with no room beside their table, are read with plain loads.
            const int64_t e0 = b0 & ~int64_t(3), e1 = (b1 + 3) & ~int64_t(3);
            const bool long_list = blen >= BULK_STAGE_MIN;
            const int32_t *src = ci_jk + b0;  // where the table build reads the list
            if (mode == ST_BITMAP) {
              // words [0, nw) hold the window, word nw is its zero guard; only
              // these are cleared (4-word groups up to `land`)
              const int64_t land = (int64_t)((nw + 4u) & ~3u);
              const bool bulk = long_list && land + (e1 - e0) <= STAGE;
              if (bulk) bulk_issue(stage + land, ci_jk, e0, e1, &rec.mbar, lane);
              int4 *s4 = reinterpret_cast<int4 *>(stage);
              for (int i = lane; i < (int)(land >> 2); i += 32) s4[i] = make_int4(0, 0, 0, 0);
              if (bulk) {
                failed = !bulk_wait(&rec.mbar, mbar_parity);
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
              int32_t *table = stage + tab0;
              const int64_t land = tab0 + hsize;
              const bool bulk = long_list && land + (e1 - e0) <= STAGE;
              if (bulk) bulk_issue(stage + land, ci_jk, e0, e1, &rec.mbar, lane);
              if (mode == ST_FILTER) {
                int4 *f4 = reinterpret_cast<int4 *>(stage);
                for (int i = lane; i < FILTER_WORDS / 4; i += 32) f4[i] = make_int4(0, 0, 0, 0);
              }
              for (int i = lane; i < hsize; i += 32) table[i] = EMPTY;
              if (bulk) {
                failed = !bulk_wait(&rec.mbar, mbar_parity);
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
                  // linear probing from the first slot of the key's 4-slot
                  // group, the order in which hash_contains reads the table
                  uint32_t h = hash_slot(key, log2h) & ~3u;
                  for (int n = 0; n < hsize; ++n) {
                    if (atomicCAS(&table[h], EMPTY, key) == EMPTY) break;
                    h = (h + 1) & hmask;
                  }
                }
              staged_log2h = log2h;
              staged_len = blen;
            } else {
              staged_off = 0;
              if (long_list && e1 - e0 <= STAGE) {
                bulk_issue(stage, ci_jk, e0, e1, &rec.mbar, lane);
                failed = !bulk_wait(&rec.mbar, mbar_parity);
                staged_off = (int)(b0 - e0);
              } else {
                for (int i = lane; i < blen; i += 32) stage[i] = i < 32 ? x0 : ci_jk[b0 + i];
              }
              staged_len = blen;
            }
            __syncwarp();
            staged_tag = failed ? ~0ull : tag;
            staged_mode = mode;
            staged = !failed;
          }
        }
      }
      if (failed) break;

      if (diag && r.y >= 0) {
        // the start of the next window's probe run, [e + 1, f) of its record,
        // into L2 while this batch is looked up (the rows of the sources of
        // one destination lie anywhere in the column array)
        const uint32_t e_next = (uint32_t)r.z + 1u, f_next = (uint32_t)r.w;
        if (f_next > e_next) {
          const int32_t *q = ci_ik + ((int64_t)e_next - ik_off);
          asm volatile("prefetch.global.L2 [%0];" ::"l"(q));
          if (f_next - e_next > 32u) asm volatile("prefetch.global.L2 [%0];" ::"l"(q + 32));
        }
      }

      if (MODE == 0 && staged && (staged_mode == ST_BITMAP || staged_mode == ST_FILTER)) {
        // quads (flat.cuh) against a bitmap or a filtered table; plain hash-table
        // and sorted lookups keep the single-probe loop below
        const uint32_t a0 = (uint32_t)s0 & ~3u;
        const uint32_t nq = len ? ((uint32_t)s1 - a0 + 3u) >> 2 : 0u;
        const uint32_t inclq = warp_inclusive_scan(nq);
        const uint32_t totalq = __shfl_sync(0xffffffffu, inclq, 31);
        uint4 *q4 = reinterpret_cast<uint4 *>(rec.b0);  // b0 and b1 are for mixed batches
        const unsigned with = __ballot_sync(0xffffffffu, nq > 0);
        if (nq > 0)
          q4[__popc(with & ((1u << lane) - 1u))] =
              make_uint4((uint32_t)s0, (uint32_t)s1, a0 - 4u * (inclq - nq), 0u);
        __syncwarp();
        uint32_t hits = 0;
        if (staged_mode == ST_BITMAP) {
          const InBitmap look{reinterpret_cast<const uint32_t *>(stage), staged_word0, staged_gw};
          flat_rounds<2>(ci_ik, q4, totalq, inclq - nq, nq > 0, lane,
                         [&](int, const int4 &w, uint32_t m, uint32_t) { hits += look.count(w, m); });
        } else {
          const InFilter look{reinterpret_cast<const uint32_t *>(stage), stage + FILTER_WORDS,
                              staged_log2h};
          flat_rounds<2>(ci_ik, q4, totalq, inclq - nq, nq > 0, lane,
                         [&](int, const int4 &w, uint32_t m, uint32_t) { hits += look.count(w, m); });
        }
        acc += hits;
        __syncwarp();
        continue;
      }

      // flattened probes, interleaved over the lanes (lanes that share an
      // in-edge read consecutive elements); each lane's owner only moves
      // forward, at most 31 steps per batch
      const uint32_t incl = warp_inclusive_scan(len);
      rec.s0[lane] = (uint32_t)s0;
      rec.incl[lane] = incl;
      if (!uniform) {
        rec.b0[lane] = b0;
        rec.b1[lane] = b1;
      }
      if (PER_VERTEX || PER_GRAPH) {
        rec.u[lane] = u;
        rec.v[lane] = uniform ? v0 : v;
      }
      __syncwarp();
      uint32_t hits = 0;
      unsigned long long batch_hits = 0;  // one graph per uniform batch
      auto on_hit = [&](int32_t wv, int o, uint32_t qpos) {
        ++hits;
        if (PER_VERTEX) {
          atomicAdd(&P.vcount[rec.u[o]], 1ull);
          atomicAdd(&P.vcount[rec.v[o]], 1ull);
          atomicAdd(&P.vcount[wv], 1ull);
        }
        if (PER_EDGE) {
          // the triangle's three edges, by position in the block columns:
          // (u,v) from the in-edge record, (u,w) from the probe, (v,w) found
          // in N(G_jk, v)
          const int64_t lo = uniform ? b0 : rec.b0[o];
          const int64_t hi = uniform ? b1 : rec.b1[o];
          const int64_t pvw = lower_bound_dev<int32_t, int64_t>(ci_jk, lo, hi, wv);
          atomicAdd(&P.edge_sup[(uint32_t)ie[batch_x0 + o - ie_off].z], 1u);
          atomicAdd(&P.edge_sup[(int64_t)qpos + ik_off], 1u);
          atomicAdd(&P.edge_sup[pvw + jk_off], 1u);
        }
        if (PER_GRAPH) {
          // every in-edge into v comes from v's own graph
          if (uniform) ++batch_hits;
          else atomicAdd(&P.graph_count[P.gid[rec.v[o]]], 1ull);
        }
      };
      // the probe loop, specialised by how N(G_jk, v) is looked up
      if (staged && staged_mode == ST_BITMAP) {
        const InBitmap look{reinterpret_cast<const uint32_t *>(stage), staged_word0, staged_gw};
        probe_batch<4>(ci_ik, rec, total, lane, on_hit,
                       [&](int32_t w, int) { return (look.one(w) & 1u) != 0u; });
      } else if (staged && staged_mode == ST_FILTER) {
        const InFilter look{reinterpret_cast<const uint32_t *>(stage), stage + FILTER_WORDS,
                            staged_log2h};
        probe_batch<4>(ci_ik, rec, total, lane, on_hit, [&](int32_t w, int) {
          return (look.maybe(w) & 1u) != 0u && hash_contains(look.table, look.log2h, w);
        });
      } else if (staged && staged_mode == ST_HASH) {
        const int log2h = staged_log2h;
        probe_batch<4>(ci_ik, rec, total, lane, on_hit,
                       [&](int32_t w, int) { return hash_contains(stage, log2h, w); });
      } else if (staged) {
        const int slen = staged_len;
        const int32_t *sl = stage + staged_off;
        probe_batch<3>(ci_ik, rec, total, lane, on_hit,
                       [&](int32_t w, int) { return sorted_contains(sl, slen, w); });
      } else {
        probe_batch<3>(ci_ik, rec, total, lane, on_hit, [&](int32_t w, int o) {
          const int64_t lo = uniform ? b0 : rec.b0[o];
          const int64_t hi = uniform ? b1 : rec.b1[o];
          const int64_t pos = lower_bound_dev<int32_t, int64_t>(ci_jk, lo, hi, w);
          return pos < hi && ci_jk[pos] == w;
        });
      }
      acc += hits;
      if (PER_GRAPH && uniform) {
        batch_hits = warp_sum(batch_hits);
        if (lane == 0 && batch_hits) atomicAdd(&P.graph_count[P.gid[v0]], batch_hits);
      }
      __syncwarp();
    }
    acc = warp_sum(acc);
    if (lane == 0 && acc) atomicAdd(&P.task_count[t], acc);
    if (P.task_cycles && lane == 0)
      atomicAdd(&P.task_cycles[t], (unsigned long long)(clock64() - t_item));
    if (failed) break;
  }
  if (failed && lane == 0) atomicExch(P.status, STATUS_COPY_WAIT);
}

__global__ void k_sum_u64(const unsigned long long *__restrict__ in, int64_t count,
                          unsigned long long *__restrict__ out) {
  unsigned long long s = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x)
    s += in[i];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0 && s) atomicAdd(out, s);
}

// sum over oriented edges (u, v) of d+(v) = sum over v of (in-degree of v) d+(v), the
// in-degree being the undirected degree minus d+(v); and sum over u of C(d+(u), 2)
__global__ void k_wedges(const int64_t *__restrict__ rowptr, const int32_t *__restrict__ perm,
                         const int32_t *__restrict__ deg, int64_t n,
                         unsigned long long *__restrict__ sums) {
  unsigned long long win = 0, wout = 0;
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long d = (unsigned long long)(rowptr[u + 1] - rowptr[u]);
    win += ((unsigned long long)deg[perm[u]] - d) * d;
    wout += d * (d > 0 ? d - 1 : 0) / 2;
  }
  win = warp_sum(win);
  wout = warp_sum(wout);
  if ((threadIdx.x & 31) == 0) {
    if (win) atomicAdd(&sums[0], win);
    if (wout) atomicAdd(&sums[1], wout);
  }
}

size_t count_smem_bytes() {
  return (size_t)(CT_NT / 32) * ((STAGE + 4) * sizeof(int32_t) + sizeof(LaneRec));
}

template <int MODE>
bbtc_status configure_mode(int *blocks_per_sm) {
  const size_t smem = count_smem_bytes();
  BBTC_CUDA(cudaFuncSetAttribute(k_count<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem));
  BBTC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_count<MODE>, CT_NT,
                                                          smem));
  if (*blocks_per_sm < 1) *blocks_per_sm = 1;
  return BBTC_OK;
}

}  // namespace

bbtc_status configure_count_kernels(Plan *pl) {
  // the attributes and occupancies are per device: set and query them once
  static std::mutex mu;
  static int cached[64][8];
  static bool done[64] = {false};
  int dev = 0;
  BBTC_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) {
    set_error("device ordinal %d out of range", dev);
    return BBTC_EINVAL;
  }
  std::lock_guard<std::mutex> lk(mu);
  if (!done[dev]) {
    BBTC_TRY(configure_mode<0>(&cached[dev][0]));
    BBTC_TRY(configure_mode<1>(&cached[dev][1]));
    BBTC_TRY(configure_mode<2>(&cached[dev][2]));
    BBTC_TRY(configure_mode<3>(&cached[dev][3]));
    BBTC_TRY(configure_mode<4>(&cached[dev][4]));
    BBTC_TRY(configure_mode<5>(&cached[dev][5]));
    BBTC_TRY(configure_mode<6>(&cached[dev][6]));
    BBTC_TRY(configure_mode<7>(&cached[dev][7]));
    done[dev] = true;
  }
  for (int i = 0; i < 8; ++i) pl->blocks_per_sm[i] = cached[dev][i];
  return BBTC_OK;
}

bbtc_status wedge_sums(const bbtc_graph *g, uint64_t *in_sum, uint64_t *out_sum,
                       cudaStream_t s) {
  Scratch scratch(s);
  unsigned long long *sums = nullptr;
  BBTC_TRY(scratch.get(&sums, 2));
  BBTC_CUDA(cudaMemsetAsync(sums, 0, 2 * sizeof(unsigned long long), s));
  if (g->n > 0) {
    k_wedges<<<grid_for(g->n, 256, 16), 256, 0, s>>>(g->rowptr, g->perm, g->deg, g->n, sums);
    BBTC_LAUNCH_CHECK();
  }
  unsigned long long h[2] = {0, 0};
  BBTC_CUDA(cudaMemcpyAsync(h, sums, sizeof(h), cudaMemcpyDeviceToHost, s));
  BBTC_CUDA(cudaStreamSynchronize(s));
  *in_sum = h[0];
  *out_sum = h[1];
  return BBTC_OK;
}

bbtc_status count_reset(bbtc_graph *g, const Plan &pl, unsigned long long *vertex_count,
                        bool per_graph, cudaStream_t s) {
  const int ng = per_graph ? g->ng : 0;
  BBTC_CUDA(cudaMemsetAsync(pl.scratch, 0,
                            sizeof(unsigned long long) * (size_t)(SCR_TASKS + pl.ntasks + ng), s));
  if (vertex_count)
    BBTC_CUDA(cudaMemsetAsync(vertex_count, 0,
                              sizeof(unsigned long long) * (size_t)(g->n > 0 ? g->n : 1), s));
  return BBTC_OK;
}

namespace {

// The by-task launch with its counters anywhere: head, status, T task counters
// and, with per_graph, the graph counters.
bbtc_status count_launch_at(const bbtc_graph *g, const Plan &pl, int64_t item0, int64_t nitems,
                            unsigned long long *head, int32_t *status,
                            unsigned long long *task_count, unsigned long long *graph_count,
                            unsigned long long *vertex_count, uint32_t timeout_ms, cudaStream_t s,
                            unsigned long long *task_cycles, unsigned *edge_sup,
                            const uint8_t *task_mask) {
  if (nitems <= 0) return BBTC_OK;
  BBTC_CUDA(cudaMemsetAsync(head, 0, sizeof(unsigned long long), s));
  CountParams P;
  P.desc = pl.desc;
  P.items = pl.items + item0;
  P.nitems = nitems;
  P.head = head;
  P.task_count = task_count;
  P.vcount = vertex_count;
  P.gid = g->gid;
  P.graph_count = graph_count;
  P.status = status;
  P.timeout_ns = (uint64_t)timeout_ms * 1000000ull;
  P.task_cycles = task_cycles;
  P.edge_sup = edge_sup;
  P.task_mask = task_mask;
  const int mode = (vertex_count ? MODE_VERTEX : 0) | (graph_count ? MODE_GRAPH : 0) |
                   (edge_sup ? MODE_EDGE : 0);
  int64_t blocks = (int64_t)num_sms() * pl.blocks_per_sm[mode];
  const int64_t need = (nitems + CT_NT / 32 - 1) / (CT_NT / 32);
  if (blocks > need) blocks = need;
  const size_t smem = count_smem_bytes();
  switch (mode) {
    case 0: k_count<0><<<(unsigned)blocks, CT_NT, smem, s>>>(P); break;
    case 1: k_count<1><<<(unsigned)blocks, CT_NT, smem, s>>>(P); break;
    case 2: k_count<2><<<(unsigned)blocks, CT_NT, smem, s>>>(P); break;
    case 3: k_count<3><<<(unsigned)blocks, CT_NT, smem, s>>>(P); break;
    case 4: k_count<4><<<(unsigned)blocks, CT_NT, smem, s>>>(P); break;
    case 5: k_count<5><<<(unsigned)blocks, CT_NT, smem, s>>>(P); break;
    case 6: k_count<6><<<(unsigned)blocks, CT_NT, smem, s>>>(P); break;
    default: k_count<7><<<(unsigned)blocks, CT_NT, smem, s>>>(P); break;
  }
  BBTC_LAUNCH_CHECK();
  return BBTC_OK;
}

}  // namespace

bbtc_status count_launch(bbtc_graph *g, const Plan &pl, int64_t item0, int64_t nitems,
                         unsigned long long *vertex_count, bool per_graph, uint32_t timeout_ms,
                         cudaStream_t s, unsigned long long *task_cycles, unsigned *edge_sup,
                         const uint8_t *task_mask) {
  unsigned long long *scr = pl.scratch;
  return count_launch_at(g, pl, item0, nitems, scr + SCR_HEAD,
                         reinterpret_cast<int32_t *>(scr + SCR_STATUS), scr + SCR_TASKS,
                         per_graph ? scr + SCR_TASKS + pl.ntasks : nullptr, vertex_count,
                         timeout_ms, s, task_cycles, edge_sup, task_mask);
}

bbtc_status count_status_error(const char *where, int32_t status, uint32_t timeout_ms) {
  if (status == STATUS_TIMEOUT) {
    set_error("%s: the counting kernel passed its %u ms limit", where, timeout_ms);
    return BBTC_ETIMEOUT;
  }
  set_error("%s: a bulk copy into the counting kernel's shared memory did not complete within "
            "its wait limit (status %d)", where, (int)status);
  return BBTC_EINTERNAL;
}

bbtc_status count_finish(const Plan &pl, cudaStream_t s) {
  k_sum_u64<<<grid_for(pl.ntasks, 256, 2), 256, 0, s>>>(pl.scratch + SCR_TASKS, pl.ntasks,
                                                         pl.scratch + SCR_TOTAL);
  BBTC_LAUNCH_CHECK();
  return BBTC_OK;
}

bbtc_status run_count(bbtc_graph *g, const Plan &pl, unsigned long long *vertex_count,
                      bool per_graph, uint32_t timeout_ms, cudaStream_t s,
                      cudaEvent_t ev_begin, cudaEvent_t ev_end,
                      unsigned long long *task_cycles, unsigned *edge_sup,
                      const uint8_t *task_mask) {
  BBTC_TRY(count_reset(g, pl, vertex_count, per_graph, s));
  if (ev_begin) BBTC_CUDA(cudaEventRecord(ev_begin, s));
  BBTC_TRY(count_launch(g, pl, 0, pl.nitems, vertex_count, per_graph, timeout_ms, s,
                        task_cycles, edge_sup, task_mask));
  if (ev_end) BBTC_CUDA(cudaEventRecord(ev_end, s));
  return count_finish(pl, s);
}

// Counts the handle's graph with what its resident plan holds: the core and
// the in-edges that it leaves; else all in-edges (a plan built for a detail
// count); else the tasks' work items (a plan built for a by-task count).
static bbtc_status count_resident(const bbtc_graph *g, const Plan &pl, bool tasks,
                                  unsigned long long *head, int32_t *status,
                                  unsigned long long *t0, unsigned long long *task_count,
                                  unsigned long long *graph_count, uint32_t timeout_ms,
                                  cudaStream_t s) {
  if (!pl.flat.ready && !pl.full.ready)
    return count_launch_at(g, pl, 0, pl.nitems, head, status, task_count, graph_count, nullptr,
                           timeout_ms, s, nullptr, nullptr, nullptr);
  if (pl.flat.ready)
    BBTC_TRY(core_launch(core_desc(g, pl, 0, 0), nullptr, 1, pl.core.nitems, pl.core.parts.quads,
                         task_count, tasks ? pl.ntasks : 1, tasks, graph_count, status, t0,
                         timeout_ms, s));
  const Flat &f = pl.flat.ready ? pl.flat : pl.full;
  return flat_launch(flat_desc(g, pl, f, 0, 0), nullptr, 1, f.nitems, head, task_count,
                     tasks ? pl.ntasks : 1, tasks, graph_count, status, t0, timeout_ms, pl.flat_blocks_per_sm, s);
}

bbtc_status run_flat(bbtc_graph *g, const Plan &pl, bool tasks, bool per_graph,
                     uint32_t timeout_ms, cudaStream_t s, cudaEvent_t ev_begin,
                     cudaEvent_t ev_end) {
  // without per-task counts the kernels add to the total itself, which saves the sum
  const bool sum = tasks || (!pl.flat.ready && !pl.full.ready);
  BBTC_TRY(count_reset(g, pl, nullptr, per_graph, s));
  if (ev_begin) BBTC_CUDA(cudaEventRecord(ev_begin, s));
  unsigned long long *scr = pl.scratch;
  BBTC_TRY(count_resident(g, pl, tasks, scr + SCR_HEAD,
                          reinterpret_cast<int32_t *>(scr + SCR_STATUS), scr + SCR_T0,
                          sum ? scr + SCR_TASKS : scr + SCR_TOTAL,
                          per_graph ? scr + SCR_TASKS + pl.ntasks : nullptr, timeout_ms, s));
  if (ev_end) BBTC_CUDA(cudaEventRecord(ev_end, s));
  return sum ? count_finish(pl, s) : BBTC_OK;
}

bbtc_status run_detail(bbtc_graph *g, const Plan &pl, bool tasks, bool per_graph,
                       unsigned long long *vcount, unsigned *edge_sup, uint32_t timeout_ms,
                       cudaStream_t s, cudaEvent_t ev_begin, cudaEvent_t ev_end) {
  if (vcount)
    BBTC_CUDA(cudaMemsetAsync(vcount, 0, sizeof(unsigned long long) * (size_t)std::max<int64_t>(g->n, 1),
                              s));
  // per task or per graph counts come from a flat count of their own
  const bool both = tasks || per_graph;
  if (both) {
    BBTC_TRY(run_flat(g, pl, tasks, per_graph, timeout_ms, s, ev_begin, nullptr));
  } else {
    BBTC_TRY(count_reset(g, pl, nullptr, false, s));
    if (ev_begin) BBTC_CUDA(cudaEventRecord(ev_begin, s));
  }
  const Flat &f = detail_flat(pl);
  BBTC_TRY(detail_launch(g, pl, flat_desc(g, pl, f, 0, 0), both ? nullptr : pl.scratch + SCR_TOTAL, vcount, edge_sup,
                         timeout_ms, s));
  if (ev_end) BBTC_CUDA(cudaEventRecord(ev_end, s));
  return BBTC_OK;
}

// --------------------------------------------- several plans, one launch
//
// A batch of resident handles is counted without copying them into a union:
// each handle keeps its own plan, and one launch of each counting kernel (core,
// flat) drains the work items of all of them, found through the handles'
// descriptors. Each handle's whole count goes to its own counter.

bbtc_status count_plans(bbtc_graph *const *gs, int32_t ng, uint32_t timeout_ms, cudaStream_t s,
                        uint64_t *counts) {
  // largest item lists first, so that small graphs fill the end of the launch
  std::vector<int32_t> order((size_t)ng);
  for (int32_t i = 0; i < ng; ++i) order[(size_t)i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) {
    return gs[a]->plan.flat.nitems > gs[b]->plan.flat.nitems;
  });
  int64_t flat_items = 0, core_items = 0;
  int quads_max = 0;
  std::vector<CoreDesc> cores;
  std::vector<FlatDesc> flats;
  for (int32_t r = 0; r < ng; ++r) {
    const int32_t h = order[(size_t)r];
    const Plan &pl = gs[h]->plan;
    if (pl.streamed || pl.p < 1 || !pl.flat.ready) {
      set_error("internal: count_plans needs resident plans");
      return BBTC_EINTERNAL;
    }
    if (pl.core.nitems > 0) {
      cores.push_back(core_desc(gs[h], pl, core_items, h));
      cores.back().p = 1;
      core_items += pl.core.nitems;
      quads_max = std::max(quads_max, (int)pl.core.parts.quads);
    }
    if (pl.flat.nitems > 0) {
      flats.push_back(flat_desc(gs[h], pl, pl.flat, flat_items, h));
      flat_items += pl.flat.nitems;
    }
  }
  Scratch scratch(s);
  unsigned long long *counters = nullptr;  // head, status, start time, then one per handle
  constexpr int C_HEAD = 0, C_STATUS = 1, C_T0 = 2, C_COUNTS = 3;
  CoreDesc *d_cores = nullptr;
  FlatDesc *d_flats = nullptr;
  BBTC_TRY(scratch.get(&counters, C_COUNTS + ng));
  BBTC_CUDA(cudaMemsetAsync(counters, 0, sizeof(unsigned long long) * (size_t)(C_COUNTS + ng), s));
  int32_t *status = reinterpret_cast<int32_t *>(counters + C_STATUS);
  if (!cores.empty()) {
    if (cores.size() > 1) {
      BBTC_TRY(scratch.get(&d_cores, (int64_t)cores.size()));
      BBTC_CUDA(cudaMemcpyAsync(d_cores, cores.data(), sizeof(CoreDesc) * cores.size(),
                                cudaMemcpyHostToDevice, s));
    }
    BBTC_TRY(core_launch(cores[0], d_cores, (int32_t)cores.size(), core_items, quads_max,
                         counters + C_COUNTS, ng, false, nullptr, status, counters + C_T0,
                         timeout_ms, s));
  }
  if (!flats.empty()) {
    if (flats.size() > 1) {
      BBTC_TRY(scratch.get(&d_flats, (int64_t)flats.size()));
      BBTC_CUDA(cudaMemcpyAsync(d_flats, flats.data(), sizeof(FlatDesc) * flats.size(),
                                cudaMemcpyHostToDevice, s));
    }
    BBTC_TRY(flat_launch(flats[0], d_flats, (int32_t)flats.size(), flat_items, counters + C_HEAD,
                         counters + C_COUNTS, ng, false, nullptr, status, counters + C_T0,
                         timeout_ms, gs[0]->plan.flat_blocks_per_sm, s));
  }
  std::vector<unsigned long long> h((size_t)(C_COUNTS + ng));
  BBTC_CUDA(cudaMemcpyAsync(h.data(), counters, sizeof(unsigned long long) * h.size(),
                            cudaMemcpyDeviceToHost, s));
  BBTC_CUDA(cudaStreamSynchronize(s));
  if ((int32_t)h[C_STATUS] != 0)
    return count_status_error("bbtc_count_batch", (int32_t)h[C_STATUS], timeout_ms);
  for (int32_t i = 0; i < ng; ++i) counts[i] = h[(size_t)(C_COUNTS + i)];
  return BBTC_OK;
}

}  // namespace bbtc

// ------------------------------------------------ allocation-free counting
//
// bbtc_count_noalloc runs the same counting kernel as bbtc_count, but keeps its
// scratch (the work-stealing counter, the status word and the per-task
// accumulators) in the fixed device array below instead of allocating it.
// The array is 8 KiB; every GPU that loads the library holds it until exit.

namespace bbtc {
namespace {

constexpr int NOALLOC_MAX_P = 16;                  // p(p+1)(p+2)/6 = 816 tasks
constexpr int NOALLOC_WORDS = 1024;                // 8 KiB of uint64
constexpr int NOALLOC_HEAD = 0, NOALLOC_STATUS = 1, NOALLOC_TASKS = 2;
static_assert(NOALLOC_TASKS + NOALLOC_MAX_P * (NOALLOC_MAX_P + 1) * (NOALLOC_MAX_P + 2) / 6 <=
                  NOALLOC_WORDS,
              "no-alloc scratch too small for NOALLOC_MAX_P");

static __device__ __align__(256) unsigned long long g_noalloc_scratch[NOALLOC_WORDS];

// Device address of g_noalloc_scratch on each device (the host-side symbol is
// only a stand-in and must never be handed to a kernel). Each device's entry
// is looked up once, under a per-device once-flag, so that host threads making
// their first call at the same time do not race on it.
unsigned long long *g_noalloc_addr[64] = {nullptr};
cudaError_t g_noalloc_err[64] = {cudaSuccess};
std::once_flag g_noalloc_once[64];

bbtc_status noalloc_scratch(unsigned long long **out) {
  int dev = 0;
  BBTC_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) {
    set_error("bbtc_count_noalloc: device ordinal %d out of range", dev);
    return BBTC_EINVAL;
  }
  std::call_once(g_noalloc_once[dev], [dev] {
    void *ptr = nullptr;
    g_noalloc_err[dev] = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    if (g_noalloc_err[dev] == cudaSuccess) g_noalloc_addr[dev] = static_cast<unsigned long long *>(ptr);
  });
  if (g_noalloc_err[dev] != cudaSuccess) {
    set_error("bbtc_count_noalloc: cudaGetSymbolAddress failed: %s",
              cudaGetErrorString(g_noalloc_err[dev]));
    return BBTC_ECUDA;
  }
  *out = g_noalloc_addr[dev];
  return BBTC_OK;
}

}  // namespace
}  // namespace bbtc

extern "C" bbtc_status bbtc_count_noalloc(bbtc_graph_t g, int32_t p, uint64_t *count_dev,
                                          uint64_t *per_task_dev, void *stream) {
  using namespace bbtc;
  clear_error();
  if (!g || !count_dev) {
    set_error("bbtc_count_noalloc: NULL handle or count_dev");
    return BBTC_EINVAL;
  }
  if (p < 1 || p > NOALLOC_MAX_P) {
    set_error("bbtc_count_noalloc: p = %d is outside 1..%d (fixed scratch holds %d tasks)", p,
              NOALLOC_MAX_P, NOALLOC_WORDS - NOALLOC_TASKS);
    return BBTC_EINVAL;
  }
  const Plan &pl = g->plan;
  if (pl.p != p || !plan_countable(pl)) {
    set_error("bbtc_count_noalloc: no plan for p = %d on this handle; call bbtc_count or "
              "bbtc_graph_get_plan with that p first", p);
    return BBTC_EINVAL;
  }
  int prev = -1;
  if (cudaGetDevice(&prev) == cudaSuccess && prev != g->device) cudaSetDevice(g->device);
  else prev = -1;
  cudaStream_t s = stream ? (cudaStream_t)stream : g->stream;
  bbtc_status st = BBTC_OK;
  do {
    unsigned long long *scratch = nullptr;
    if ((st = noalloc_scratch(&scratch)) != BBTC_OK) break;
    unsigned long long *task_count = scratch + NOALLOC_TASKS;
    const int64_t nt = pl.ntasks;
    // the array keeps the previous call's contents: clear what must start at 0
    if (cudaMemsetAsync(scratch, 0, sizeof(unsigned long long) * (size_t)(NOALLOC_TASKS + nt),
                        s) != cudaSuccess ||
        cudaMemsetAsync(count_dev, 0, sizeof(uint64_t), s) != cudaSuccess) {
      set_error("bbtc_count_noalloc: cudaMemsetAsync failed");
      st = BBTC_ECUDA;
      break;
    }
    int32_t *status = reinterpret_cast<int32_t *>(scratch + NOALLOC_STATUS);
    const bool tasks = per_task_dev != nullptr;
    if ((st = count_resident(g, pl, tasks, scratch + NOALLOC_HEAD, status, nullptr, task_count,
                             nullptr, 0, s)) != BBTC_OK)
      break;
    k_sum_u64<<<grid_for(nt, 256, 2), 256, 0, s>>>(
        task_count, nt, reinterpret_cast<unsigned long long *>(count_dev));
    if ((st = launch_status("bbtc_count_noalloc")) != BBTC_OK) break;
    if (per_task_dev &&
        cudaMemcpyAsync(per_task_dev, task_count, sizeof(uint64_t) * (size_t)nt,
                        cudaMemcpyDeviceToDevice, s) != cudaSuccess) {
      set_error("bbtc_count_noalloc: cudaMemcpyAsync failed");
      st = BBTC_ECUDA;
      break;
    }
  } while (0);
  if (prev >= 0) cudaSetDevice(prev);
  return st;
}
