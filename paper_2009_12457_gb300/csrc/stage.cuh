// stage.cuh -- the on-chip forms of a list N(G_jk, v) that the counting kernels
// probe, and the bulk copies (TMA) that bring long lists into shared memory.
#pragma once

#include "common.cuh"

namespace bbtc {

namespace {

constexpr int32_t STATUS_TIMEOUT = 1, STATUS_COPY_WAIT = 2;

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Per-warp shared staging area for N(G_jk, v) (int32 slots).
constexpr int STAGE = 2048;
static_assert(STAGE % 4 == 0, "the bitmap is cleared with 16-byte stores");
// largest power of two <= STAGE: the biggest hash table the stage holds
constexpr int STAGE_POW2 = STAGE >= 2048 ? 2048 : STAGE >= 1024 ? 1024 : STAGE >= 512 ? 512 : 256;
static_assert(STAGE_POW2 <= STAGE && STAGE >= 256, "stage too small");
constexpr int MIN_STAGE = 8;
// lists at least this long are staged through one bulk copy (TMA)
constexpr int BULK_STAGE_MIN = 64;
constexpr int ST_NONE = 0, ST_SORTED = 1, ST_HASH = 2, ST_BITMAP = 3, ST_FILTER = 4;
// ST_FILTER: an open-addressed table of up to FILTER_SLOTS slots in the upper
// half of the stage, with a filter in the lower half: two bits per key in one
// word (see InFilter). A probe reads one filter word and looks in the table only
// when both bits are set.
constexpr int FILTER_WORDS = STAGE / 2;
constexpr int FILTER_BITS_LOG2 = 15;
constexpr int FILTER_SLOTS = STAGE - FILTER_WORDS;
static_assert(FILTER_WORDS * 32 == 1 << FILTER_BITS_LOG2, "filter size");
static_assert((FILTER_SLOTS & (FILTER_SLOTS - 1)) == 0 && FILTER_WORDS % 4 == 0, "filter table");
constexpr int32_t EMPTY = -1;

__device__ __forceinline__ uint32_t hash_slot(int32_t w, int log2h) {
  return ((uint32_t)w * 2654435761u) >> (32 - log2h);
}

// Membership of w in the sorted list stage[0, len): lower bound by a fixed
// number of halvings (the same for every lane, since len is warp-uniform).
__device__ __forceinline__ bool sorted_contains(const int32_t *stage, int len, int32_t w) {
  int pos = 0;
  for (int step = len > 0 ? 1 << (31 - __clz(len)) : 0; step > 0; step >>= 1)
    if (pos + step <= len && stage[pos + step - 1] < w) pos += step;
  return pos < len && stage[pos] == w;
}

// Membership of w in the open-addressed table stage[0, 2^log2h) (linear
// probing, at most half full). The probe reads four slots per 16-byte load,
// starting at the 4-slot group of w's hash slot, so nearly every lookup ends
// after one load and the lanes of a warp stay together.
__device__ __forceinline__ bool hash_contains(const int32_t *stage, int log2h, int32_t w) {
  const uint32_t gmask = (1u << (log2h - 2)) - 1u;
  uint32_t g = hash_slot(w, log2h) >> 2;
  const int4 *groups = reinterpret_cast<const int4 *>(stage);
  for (uint32_t n = 0; n <= gmask; ++n) {
    const int4 q = groups[g];
    if (q.x == w || q.y == w || q.z == w || q.w == w) return true;
    if (q.x == EMPTY || q.y == EMPTY || q.z == EMPTY || q.w == EMPTY) return false;
    g = (g + 1) & gmask;
  }
  return false;
}

// Bit c of the result: column c of the quad is in the list.
struct InBitmap {  // window of words from `word0` on, zero word at index gw
  const uint32_t *bm;
  uint32_t word0, gw;
  __device__ __forceinline__ uint32_t one(int32_t w) const {
    const uint32_t word = bm[min(((uint32_t)w >> 5) - word0, gw)];
    return word >> ((uint32_t)w & 31u);
  }
  __device__ __forceinline__ uint32_t count(const int4 &w, uint32_t m) const {
    return (one(w.x) & m & 1u) + (one(w.y) & (m >> 1) & 1u) + (one(w.z) & (m >> 2) & 1u) +
           (one(w.w) & (m >> 3) & 1u);
  }
  __device__ __forceinline__ uint32_t bits(const int4 &w, uint32_t m) const {
    return ((one(w.x) & 1u) | ((one(w.y) & 1u) << 1) | ((one(w.z) & 1u) << 2) |
            ((one(w.w) & 1u) << 3)) & m;
  }
};

// A table behind a filter of one word per key with two bits in it (both from
// the word's hash), so that one load rejects most keys that are not in the list.
struct InFilter {
  const uint32_t *filter;
  const int32_t *table;
  int log2h;
  static __device__ __forceinline__ uint32_t hash(int32_t w) { return (uint32_t)w * 0x85EBCA6Bu; }
  static __device__ __forceinline__ uint32_t word_of(uint32_t h) {
    return h >> (32 - (FILTER_BITS_LOG2 - 5));
  }
  static __device__ __forceinline__ uint32_t bits_of(uint32_t h) {
    return (1u << (h & 31u)) | (1u << ((h >> 10) & 31u));
  }
  __device__ __forceinline__ uint32_t maybe(int32_t w) const {
    const uint32_t h = hash(w);
    const uint32_t word = filter[word_of(h)];
    return (word >> (h & 31u)) & (word >> ((h >> 10) & 31u));
  }
  __device__ __forceinline__ uint32_t bits(const int4 &w, uint32_t m) const {
    uint32_t cand = ((maybe(w.x) & 1u) | ((maybe(w.y) & 1u) << 1) | ((maybe(w.z) & 1u) << 2) |
                     ((maybe(w.w) & 1u) << 3)) & m;
    uint32_t hit = 0;
    while (cand) {
      const int c = __ffs(cand) - 1;
      cand &= cand - 1;
      const int32_t x = c == 0 ? w.x : c == 1 ? w.y : c == 2 ? w.z : w.w;
      hit |= (uint32_t)hash_contains(table, log2h, x) << c;
    }
    return hit;
  }
  __device__ __forceinline__ uint32_t count(const int4 &w, uint32_t m) const {
    return __popc(bits(w, m));
  }
};

// ------------------------------------------------ bulk copies (TMA, PTX)

__device__ __forceinline__ uint32_t smem_addr(const void *ptr) {
  return (uint32_t)__cvta_generic_to_shared(ptr);
}
__device__ __forceinline__ void mbar_init(unsigned long long *m) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(m)) : "memory");
}
// Makes an initialised barrier visible to the bulk-copy unit.
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// The one arrival of the barrier's current phase, announcing `bytes` of copies.
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *m, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(m)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long *m, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_addr(m)), "r"(parity)
      : "memory");
  return done != 0;
}
// limit of one wait on a bulk copy (copies of valid addresses take microseconds)
constexpr uint64_t COPY_WAIT_NS = 200ull * 1000 * 1000;
// Waits for the barrier's phase of the given parity, for at most COPY_WAIT_NS.
__device__ __noinline__ bool mbar_wait_bounded(unsigned long long *m, uint32_t parity) {
  if (mbar_try_wait(m, parity)) return true;
  const uint64_t t0 = global_ns();
  while (!mbar_try_wait(m, parity))
    if (global_ns() - t0 > COPY_WAIT_NS) return false;
  return true;
}
// TMA bulk copy global -> shared of `bytes` (a multiple of 16, both addresses
// 16-byte aligned), completing on barrier m.
__device__ __forceinline__ void bulk_copy(void *dst, const void *src, uint32_t bytes,
                                          unsigned long long *m) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(m))
      : "memory");
}
// Orders this thread's earlier plain shared-memory accesses before later bulk
// copies into the same memory.
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Starts one bulk copy of list[e0, e1) into `dst` (e0, e1 multiples of 4:
// whole 16-byte quads of a 16-byte aligned, quad-padded column array; dst
// 16-byte aligned), issued by lane 0 on barrier mbar. Warp-uniform call.
__device__ __forceinline__ void bulk_issue(int32_t *dst, const int32_t *list, int64_t e0,
                                           int64_t e1, unsigned long long *mbar, unsigned lane) {
  fence_proxy_async();  // earlier plain accesses to the stage before the copy
  __syncwarp();
  if (lane == 0) {
    const uint32_t bytes = (uint32_t)(4 * (e1 - e0));
    mbar_expect_tx(mbar, bytes);
    bulk_copy(dst, list + e0, bytes, mbar);
  }
}

// Waits (bounded) for the copy of bulk_issue; true on every lane when it
// arrived. On false the copy is awaited once more and the caller stops.
__device__ __forceinline__ bool bulk_wait(unsigned long long *mbar, uint32_t &parity) {
  const bool ok = __all_sync(0xffffffffu, mbar_wait_bounded(mbar, parity));
  if (!ok) {
    mbar_wait_bounded(mbar, parity);
    return false;
  }
  parity ^= 1u;
  return true;
}

}  // namespace

}  // namespace bbtc
