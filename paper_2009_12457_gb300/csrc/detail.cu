// detail.cu -- triangles at every vertex and the support of every edge of a
// resident plan (a10, and the input of k-truss).
//
// The walk is that of flat.cu over all in-edges (the dense core's too: its
// bitmap counts know no single triangle). What made these outputs slow is one
// global addition per triangle corner, most of them to a few hubs. Here each
// corner is summed on chip first:
//   (u, v), u: the hits of one in-edge, in a counter of the batch;
//   v:         the hits of a run, in registers;
//   (v, w), w: the hits on each entry of the staged list, in a 16-bit counter
//              per entry, found by the rank of w in the bitmap (first entry of
//              the word + the bits below w); flushed once per run.
// Only (u, w) stays one addition per triangle: its address belongs to u's row
// and is hit once per (u, v). Triangles at every vertex of R-MAT scale 20 took
// 77 to 83 ms with one addition per corner and take 2.7 ms so; edge support on
// scale 19, 6.7 and 1.27 ms.
#include <algorithm>
#include <mutex>

#include "bounds.cuh"
#include "flat.cuh"
#include "graph.cuh"
#include "stage.cuh"

namespace bbtc {

namespace {

constexpr int DT_NT = 256;
constexpr int DT_WARPS = DT_NT / 32;
constexpr int DT_WORDS = 1024;  // bitmap window (32,768 columns), or entries of a sorted copy
constexpr int DT_LIST = 1024;   // longest staged list
constexpr int DT_RUN_MIN = 4;
constexpr uint32_t DT_FLUSH = 60000;  // in-edges after which 16-bit counters are flushed
constexpr int DT_VERTEX = 1, DT_EDGE = 2;

struct DetailLaunch {
  FlatDesc d;
  const int32_t *esrc;
  unsigned long long *head;
  unsigned long long *total;   // nullable
  unsigned long long *vcount;  // by position
  unsigned *edge_sup;          // by column position
  int32_t *status;
  const unsigned long long *t0;
  uint64_t timeout_ns;
};

struct DetailSmem {
  uint32_t stage[DT_WORDS + 4];
  uint32_t cnt[DT_LIST / 2];    // two 16-bit counters a word
  uint16_t pre[DT_WORDS];       // entries before each word that holds one
  uint4 rec[32];
  uint2 rng[32];
  uint32_t hits[32];            // of each in-edge of the batch
  int32_t v[32];
};
static_assert(sizeof(DetailSmem) % 16 == 0, "per-warp areas stay aligned");

template <int MODE>
__global__ void __launch_bounds__(DT_NT, 3) k_detail(DetailLaunch P) {
  constexpr bool VERTEX = (MODE & DT_VERTEX) != 0;
  constexpr bool EDGE = (MODE & DT_EDGE) != 0;
  extern __shared__ __align__(16) unsigned char detail_smem[];
  const unsigned lane = threadIdx.x & 31u;
  DetailSmem &sm = reinterpret_cast<DetailSmem *>(detail_smem)[threadIdx.x >> 5];
  const FlatDesc &d = P.d;
  const uint2 *__restrict__ rec = d.rec;
  const uint32_t *__restrict__ inptr = d.inptr;
  const int64_t *__restrict__ rowptr = d.rowptr;
  const int32_t *__restrict__ ci = d.colidx;
  const int kflag = d.flags & 3;
  uint64_t t_start = 0;
  if (P.timeout_ns) {
    t_start = *P.t0;
    if (t_start == 0) t_start = global_ns();
  }
  unsigned long long acc = 0;
  unsigned long long it = 0;
  if (lane == 0) it = atomicAdd(P.head, 1ull);
  it = __shfl_sync(0xffffffffu, it, 0);
  while (it < (unsigned long long)d.nitems) {
    unsigned long long it_next = 0;
    if (lane == 0) it_next = atomicAdd(P.head, 1ull);
    if (P.timeout_ns && global_ns() - t_start > P.timeout_ns) {
      if (lane == 0) atomicExch(P.status, STATUS_TIMEOUT);
      break;
    }
    const int64_t k = d.item0 + d.nitems - 1 - (int64_t)it;
    uint32_t base = (uint32_t)(k * d.chunk);
    const uint32_t x1 = (uint32_t)min((int64_t)d.records, (k + 1) * d.chunk);
    uint32_t v = 0, vend = base, b0 = 0, b1 = 0;
    int32_t vl = -1;
    int staged = ST_NONE;
    uint32_t word0 = 0, gw = 0, since = 0;
    uint32_t run_hits = 0;
    // adds the staged list's counters and the run's hits to the outputs
    auto flush = [&](bool clear) {
      __syncwarp();
      if (staged != ST_NONE) {
        const int blen = (int)(b1 - b0);
        for (int i = lane; i < blen; i += 32) {
          const uint32_t c = (sm.cnt[i >> 1] >> ((i & 1) * 16)) & 0xffffu;
          if (c) {
            if (EDGE) atomicAdd(&P.edge_sup[b0 + i], c);
            if (VERTEX) atomicAdd(&P.vcount[ci[b0 + i]], (unsigned long long)c);
          }
        }
        __syncwarp();
        if (clear)
          for (int i = lane; i < (blen + 1) / 2; i += 32) sm.cnt[i] = 0;
        __syncwarp();
      }
      if (VERTEX) {
        const uint32_t s = __reduce_add_sync(0xffffffffu, run_hits);
        if (lane == 0 && s) atomicAdd(&P.vcount[v], (unsigned long long)s);
        run_hits = 0;
      }
      since = 0;
    };
    uint2 r = window_holds(base, lane, x1) ? rec[base + lane] : make_uint2(0, 0);
    while (base < x1) {
      const bool begins = vend <= base;
      if (begins) {
        flush(false);
        staged = ST_NONE;
        vl = window_holds(base, lane, x1) ? ci[r.x - 1] : -1;
        v = (uint32_t)__shfl_sync(0xffffffffu, vl, 0);
        vend = inptr[v + 1];
        b0 = (uint32_t)rowptr[v];
        b1 = (uint32_t)rowptr[v + 1];
      }
      const uint32_t run = min(vend, x1) - base;
      const bool uniform = !begins || run >= (uint32_t)DT_RUN_MIN || run == x1 - base;
      if (uniform && b1 == b0) {
        base += run;
        r = window_holds(base, lane, x1) ? rec[base + lane] : make_uint2(0, 0);
        continue;
      }
      int nb = (int)min(run, 32u);
      uint32_t vb0 = b0, vb1 = b1;
      if (!uniform) {  // short runs share the window (see flat.cu)
        const unsigned same = __match_any_sync(0xffffffffu, vl);
        const bool lengthy = __popc(same) >= DT_RUN_MIN || ((same >> 31) && window_holds(base, 32u, x1));
        const unsigned stop = __ballot_sync(0xffffffffu, vl < 0 || (lengthy && vl != (int32_t)v));
        nb = stop ? __ffs(stop) - 1 : 32;
        if ((int)lane < nb) {
          vb0 = (uint32_t)rowptr[vl];
          vb1 = (uint32_t)rowptr[vl + 1];
        }
        vend = base + (uint32_t)nb;
      }
      base += (uint32_t)nb;
      const uint2 rn = window_holds(base, lane, x1) ? rec[base + lane] : make_uint2(0, 0);
      const bool active = (int)lane < nb && vb1 > vb0;
      const uint32_t s0 = r.x, s1 = r.y;
      r = rn;
      const uint32_t a0 = s0 & ~3u;
      const uint32_t nq = active && s1 > s0 ? (s1 - a0 + 3u) >> 2 : 0u;
      const uint32_t incl = warp_inclusive_scan(nq);
      const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
      if (total == 0) continue;

      const int blen = (int)(b1 - b0);
      if (uniform && staged != ST_NONE && since + 32u > DT_FLUSH) flush(true);
      if (uniform && staged == ST_NONE && blen <= DT_LIST &&
          (nb == 32 || total * 4u >= (uint32_t)blen / 2u)) {
        const uint32_t first = (uint32_t)ci[b0], last = (uint32_t)ci[b1 - 1];
        const uint32_t nw = (last >> 5) - (first >> 5) + 1u;
        word0 = first >> 5;
        gw = nw;
        const bool bitmap = kflag != 0 && nw <= (uint32_t)DT_WORDS;
        __syncwarp();
        for (int i = lane; i < (blen + 1) / 2; i += 32) sm.cnt[i] = 0;
        if (bitmap) {
          for (int i = lane; i <= (int)nw; i += 32) sm.stage[i] = 0;  // and the guard word
          __syncwarp();
          for (int i = lane; i < blen; i += 32) {
            const uint32_t w = (uint32_t)ci[b0 + i];
            const uint32_t prev = i > 0 ? (uint32_t)ci[b0 + i - 1] : ~0u;
            const uint32_t x = (w >> 5) - word0;
            atomicOr(&sm.stage[x], 1u << (w & 31u));
            if (i == 0 || (prev >> 5) != (w >> 5)) sm.pre[x] = (uint16_t)i;
          }
        } else {
          for (int i = lane; i < blen; i += 32) sm.stage[i] = (uint32_t)ci[b0 + i];
        }
        __syncwarp();
        staged = bitmap ? ST_BITMAP : ST_SORTED;
        since = 0;
      }
      since += (uint32_t)nb;

      if (r.y > r.x) {
        const int32_t *q = ci + r.x;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(q));
        if (r.y - r.x > 32u) asm volatile("prefetch.global.L2 [%0];" ::"l"(q + 32));
      }

      const uint32_t first = incl - nq;
      const bool has = nq > 0;
      const unsigned with = __ballot_sync(0xffffffffu, has);
      const int nrec = __popc(with);
      if (has) {
        const int c = __popc(with & ((1u << lane) - 1u));
        sm.rec[c] = make_uint4(s0, s1, a0 - 4u * first, 0u);
        if (!uniform) {
          sm.rng[c] = make_uint2(vb0, vb1);
          sm.v[c] = vl;
        }
      }
      sm.hits[lane] = 0;
      __syncwarp();
      uint32_t batch_hits = 0;
      // one hit on entry i of the staged list
      auto entry_hit = [&](uint32_t i) { atomicAdd(&sm.cnt[i >> 1], 1u << ((i & 1u) * 16u)); };
      auto quad_end = [&](int own, uint32_t h) {
        if (h) {
          batch_hits += h;
          atomicAdd(&sm.hits[own], h);
        }
      };
      if (uniform && staged == ST_BITMAP) {
        flat_rounds<2>(ci, sm.rec, total, first, has, lane,
                       [&](int own, const int4 &w, uint32_t m, uint32_t q) {
          uint32_t h = 0;
          auto one = [&](int32_t x, uint32_t mc, uint32_t pos) {
            const uint32_t i = min(((uint32_t)x >> 5) - word0, gw);
            const uint32_t word = sm.stage[i], bit = (uint32_t)x & 31u;
            if ((word >> bit) & mc & 1u) {
              entry_hit((uint32_t)sm.pre[i] + (uint32_t)__popc(word & ((1u << bit) - 1u)));
              if (EDGE) atomicAdd(&P.edge_sup[pos], 1u);
              ++h;
            }
          };
          one(w.x, m, q);
          one(w.y, m >> 1, q + 1);
          one(w.z, m >> 2, q + 2);
          one(w.w, m >> 3, q + 3);
          quad_end(own, h);
        });
      } else if (uniform && staged == ST_SORTED) {
        flat_rounds<1>(ci, sm.rec, total, first, has, lane,
                       [&](int own, const int4 &w, uint32_t m, uint32_t q) {
          uint32_t h = 0;
          int at = 0;  // the quad ascends
          for (uint32_t left = m; left; left &= left - 1) {
            const int c = __ffs(left) - 1;
            const uint32_t x = (uint32_t)(c == 0 ? w.x : c == 1 ? w.y : c == 2 ? w.z : w.w);
            at = lower_bound_dev<uint32_t, int>(sm.stage, at, blen, x);
            if (at < blen && sm.stage[at] == x) {
              entry_hit((uint32_t)at);
              if (EDGE) atomicAdd(&P.edge_sup[q + c], 1u);
              ++h;
            }
          }
          quad_end(own, h);
        });
      } else {
        flat_rounds<1>(ci, sm.rec, total, first, has, lane,
                       [&](int own, const int4 &w, uint32_t m, uint32_t q) {
          uint32_t h = 0;
          uint2 b = make_uint2(b0, b1);
          if (!uniform && m) b = sm.rng[own];
          uint32_t at = b.x;
          for (uint32_t left = m; left; left &= left - 1) {
            const int c = __ffs(left) - 1;
            const int32_t x = c == 0 ? w.x : c == 1 ? w.y : c == 2 ? w.z : w.w;
            at = lower_bound_dev<int32_t, uint32_t>(ci, at, b.y, x);
            if (at < b.y && ci[at] == x) {
              if (EDGE) {
                atomicAdd(&P.edge_sup[at], 1u);
                atomicAdd(&P.edge_sup[q + c], 1u);
              }
              if (VERTEX) atomicAdd(&P.vcount[x], 1ull);
              ++h;
            }
          }
          quad_end(own, h);
        });
      }
      __syncwarp();
      if ((int)lane < nrec) {
        const uint32_t h = sm.hits[lane];
        if (h) {
          const uint32_t e = sm.rec[lane].x - 1u;
          if (EDGE) atomicAdd(&P.edge_sup[e], h);
          if (VERTEX) {
            atomicAdd(&P.vcount[P.esrc[e]], (unsigned long long)h);
            if (!uniform) atomicAdd(&P.vcount[sm.v[lane]], (unsigned long long)h);
          }
        }
      }
      if (uniform) run_hits += batch_hits;
      acc += batch_hits;
      __syncwarp();
    }
    flush(false);
    it = __shfl_sync(0xffffffffu, it_next, 0);
  }
  if (P.total) {
    acc = warp_sum(acc);
    if (lane == 0 && acc) atomicAdd(P.total, acc);
  }
}

// the attributes and occupancies are per device: set and query them once
template <int MODE>
bbtc_status detail_configure(int *blocks_per_sm) {
  static std::mutex mu;
  static int cached[64] = {0};
  int dev = 0;
  BBTC_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) {
    set_error("device ordinal %d out of range", dev);
    return BBTC_EINVAL;
  }
  std::lock_guard<std::mutex> lk(mu);
  if (cached[dev] > 0) {
    *blocks_per_sm = cached[dev];
    return BBTC_OK;
  }
  const size_t smem = sizeof(DetailSmem) * DT_WARPS;
  BBTC_CUDA(cudaFuncSetAttribute(k_detail<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem));
  BBTC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_detail<MODE>, DT_NT,
                                                          smem));
  if (*blocks_per_sm < 1) *blocks_per_sm = 1;
  cached[dev] = *blocks_per_sm;
  return BBTC_OK;
}

}  // namespace

bbtc_status detail_launch(const bbtc_graph *g, const Plan &pl, const FlatDesc &d,
                          unsigned long long *total, unsigned long long *vcount,
                          unsigned *edge_sup, uint32_t timeout_ms, cudaStream_t s) {
  if (d.nitems <= 0) return BBTC_OK;
  DetailLaunch P;
  P.d = d;
  P.esrc = g->esrc;
  P.head = pl.scratch + SCR_HEAD;
  P.total = total;
  P.vcount = vcount;
  P.edge_sup = edge_sup;
  P.status = reinterpret_cast<int32_t *>(pl.scratch + SCR_STATUS);
  P.t0 = pl.scratch + SCR_T0;
  P.timeout_ns = (uint64_t)timeout_ms * 1000000ull;
  int per_sm = 1;
  if (vcount && edge_sup) BBTC_TRY(detail_configure<3>(&per_sm));
  else if (vcount) BBTC_TRY(detail_configure<1>(&per_sm));
  else BBTC_TRY(detail_configure<2>(&per_sm));
  const int64_t blocks = std::min<int64_t>((int64_t)num_sms() * per_sm,
                                           (d.nitems + DT_WARPS - 1) / DT_WARPS);
  const size_t smem = sizeof(DetailSmem) * DT_WARPS;
  BBTC_CUDA(cudaMemsetAsync(P.head, 0, sizeof(unsigned long long), s));
  if (vcount && edge_sup) k_detail<3><<<(unsigned)blocks, DT_NT, smem, s>>>(P);
  else if (vcount) k_detail<1><<<(unsigned)blocks, DT_NT, smem, s>>>(P);
  else k_detail<2><<<(unsigned)blocks, DT_NT, smem, s>>>(P);
  BBTC_LAUNCH_CHECK();
  return BBTC_OK;
}

}  // namespace bbtc
