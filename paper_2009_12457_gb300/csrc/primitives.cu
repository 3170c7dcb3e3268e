// primitives.cu -- stable LSD radix sort, exclusive scan, max reduction.
#include "primitives.cuh"

#include <utility>

namespace bbtc {

namespace {

constexpr int RS_NT = 512;                 // threads per tile (256 threads of 16 keys held
constexpr int RS_ITEMS = 8;                // 101 registers each: 16 warps per SM)
constexpr int RS_TILE = RS_NT * RS_ITEMS;  // 4096 keys per tile
constexpr int RS_WARPS = RS_NT / 32;
constexpr int RS_BINS = 256;
constexpr int RS_WARP_SPAN = RS_TILE / RS_WARPS;  // consecutive tile positions per warp

// Digit counts of every pass at once (one read of the keys): hist[pass][256].
__global__ void __launch_bounds__(RS_NT) k_rs_hist(const uint64_t *__restrict__ keys,
                                                   int64_t count, int bit_lo, int bit_hi,
                                                   unsigned long long *__restrict__ hist) {
  __shared__ uint32_t h[8][RS_BINS];
  const int passes = (bit_hi - bit_lo + 7) / 8;
  for (int i = threadIdx.x; i < passes * RS_BINS; i += RS_NT) (&h[0][0])[i] = 0;
  __syncthreads();
  for (int64_t x = (int64_t)blockIdx.x * RS_NT + threadIdx.x; x < count;
       x += (int64_t)gridDim.x * RS_NT) {
    const uint64_t k = keys[x];
    for (int p = 0; p < passes; ++p) {
      const int shift = bit_lo + 8 * p;
      const uint32_t mask = bit_hi - shift < 8 ? (1u << (bit_hi - shift)) - 1u : 255u;
      atomicAdd(&h[p][(uint32_t)(k >> shift) & mask], 1u);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < passes * RS_BINS; i += RS_NT)
    if ((&h[0][0])[i]) atomicAdd(&hist[i], (unsigned long long)(&h[0][0])[i]);
}

// The first output position of every digit of every pass (one block per pass).
__global__ void __launch_bounds__(RS_BINS) k_rs_digits(unsigned long long *__restrict__ hist) {
  __shared__ unsigned long long tmp[RS_BINS / 32 + 1];
  unsigned long long total;
  unsigned long long *h = hist + (int64_t)blockIdx.x * RS_BINS;
  const unsigned long long c = h[threadIdx.x];
  h[threadIdx.x] = block_exclusive_scan<unsigned long long, RS_BINS>(c, tmp, &total);
}

// Shared memory layout of a tile's sort (dynamic).
template <bool HAS_VALS>
struct RsSmem {
  uint64_t keys[RS_TILE];
  uint32_t vals[HAS_VALS ? RS_TILE : 1];
  uint32_t whist[RS_WARPS][RS_BINS];  // per-warp digit counts, then per-warp prefixes
  uint32_t bstart[RS_BINS];           // tile-local start of each digit bucket
  uint64_t goff[RS_BINS];             // global start of this tile's part of each bucket
  uint32_t scan_tmp[RS_WARPS + 1];
  uint32_t tile;
  int32_t failed;  // an earlier pass or tile gave up
};

// Ranks a tile's keys (thread-owned positions warp * RS_WARP_SPAN + 32 i + lane) by digit,
// stably: keys with equal digits in one group of 32 are ranked by lane
// (match_any), groups in order, warps in order -- the tile's own order.
// Positions past the end take the largest digit; being last in the tile they
// rank after every real key. Leaves whist, bstart; returns digit threadIdx.x's count.
template <bool HAS_VALS>
__device__ __forceinline__ uint32_t rs_rank(RsSmem<HAS_VALS> &sm, const uint64_t (&k)[RS_ITEMS],
                                            int nvalid, int shift, uint32_t mask,
                                            uint32_t (&rank)[RS_ITEMS]) {
  const int warp = threadIdx.x >> 5;
  const unsigned lane = threadIdx.x & 31u;
  const unsigned lt_mask = (1u << lane) - 1u;
  for (int i = threadIdx.x; i < RS_WARPS * RS_BINS; i += RS_NT) (&sm.whist[0][0])[i] = 0;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < RS_ITEMS; ++i) {
    const int pos = warp * RS_WARP_SPAN + i * 32 + (int)lane;
    const uint32_t d = pos < nvalid ? (uint32_t)(k[i] >> shift) & mask : mask;
    const uint32_t peers = __match_any_sync(0xffffffffu, d);
    const uint32_t before = sm.whist[warp][d];
    __syncwarp();
    if ((peers & lt_mask) == 0) sm.whist[warp][d] = before + (uint32_t)__popc(peers);
    __syncwarp();
    rank[i] = before + (uint32_t)__popc(peers & lt_mask);
  }
  __syncthreads();
  // per digit: exclusive prefix over warps, and the tile's bucket starts
  const int d = threadIdx.x;  // the first RS_BINS threads
  uint32_t run = 0;
  if (d < RS_BINS) {
#pragma unroll
    for (int w = 0; w < RS_WARPS; ++w) {
      const uint32_t c = sm.whist[w][d];
      sm.whist[w][d] = run;
      run += c;
    }
  }
  uint32_t total;
  const uint32_t start = block_exclusive_scan<uint32_t, RS_NT>(run, sm.scan_tmp, &total);
  if (d < RS_BINS) sm.bstart[d] = start;
  return run;
}

// One pass of the sort in one kernel: a tile publishes its digit counts and
// finds where its buckets start from the tiles before it (decoupled look-back),
// so that the keys are read once and written once per pass; counting, scanning
// and scattering in separate kernels read them twice (16.7 M keys of 40 bits:
// 2.4 ms of passes in R-MAT scale 20's general preparation). Tiles are taken in
// ticket order, so the tiles waited for are running or done; every wait is
// bounded all the same, and a tile that gives up poisons its own entry, so that
// the ones after it stop, writes nothing and sets bit 3 of *err. The passes after a
// failed one find the bit and move no key: those that the failed pass left unwritten
// would not match the digit counts, and could be sent past the end of the output.
// Word of (tile, digit): code << 56 | count; pass q uses the codes 2q + 1 (the
// tile's own count) and 2q + 2 (the count up to and with the tile).
constexpr uint64_t RS_POISON = 0xffull << 56;
constexpr uint64_t RS_COUNT = (1ull << 56) - 1ull;
constexpr int RS_BACK = 8;
constexpr int RS_SPIN_LIMIT = 1 << 22;  // polls of one word (seconds)

template <bool HAS_VALS>
__global__ void __launch_bounds__(RS_NT) k_rs_pass(
    const uint64_t *__restrict__ kin, uint64_t *__restrict__ kout,
    const uint32_t *__restrict__ vin, uint32_t *__restrict__ vout, int64_t count, int shift,
    uint32_t mask, int pass, const unsigned long long *__restrict__ digit_start,
    unsigned *__restrict__ ticket, unsigned long long *status, int32_t *__restrict__ err) {
  extern __shared__ __align__(16) unsigned char rs_smem_raw[];
  RsSmem<HAS_VALS> &sm = *reinterpret_cast<RsSmem<HAS_VALS> *>(rs_smem_raw);
  const int warp = threadIdx.x >> 5;
  const unsigned lane = threadIdx.x & 31u;
  if (threadIdx.x == 0) {
    sm.tile = atomicAdd(ticket, 1u);
    sm.failed = *(volatile int32_t *)err & SORT_FAILED;
  }
  __syncthreads();
  const int64_t tile = sm.tile;
  if (sm.failed) {
    if (threadIdx.x < RS_BINS) *(volatile unsigned long long *)(status + tile * RS_BINS + threadIdx.x) = RS_POISON;
    return;
  }
  const int64_t base = tile * RS_TILE;
  const int nvalid = (int)(count - base < RS_TILE ? count - base : RS_TILE);
  uint64_t k[RS_ITEMS];
  uint32_t v[HAS_VALS ? RS_ITEMS : 1];
  uint32_t rank[RS_ITEMS];
#pragma unroll
  for (int i = 0; i < RS_ITEMS; ++i) {
    const int pos = warp * RS_WARP_SPAN + i * 32 + (int)lane;
    k[i] = pos < nvalid ? kin[base + pos] : ~0ull;
    if (HAS_VALS) v[i] = pos < nvalid ? vin[base + pos] : 0u;
  }
  const uint32_t all = rs_rank<HAS_VALS>(sm, k, nvalid, shift, mask, rank);
  const uint64_t own = (uint64_t)(2 * pass + 1) << 56, upto = (uint64_t)(2 * pass + 2) << 56;
  const int d = threadIdx.x;
  // positions past the end count as the largest digit: not among the real ones
  const uint32_t mine = (uint32_t)d == mask ? all - (uint32_t)(RS_TILE - nvalid) : all;
  volatile unsigned long long *st = status + tile * RS_BINS + d;
  uint64_t before = 0;
  bool failed = false;
  if (d >= RS_BINS) {
    // no digit
  } else if (tile == 0) {
    *st = upto | mine;
  } else {
    *st = own | mine;
    // RS_BACK tiles are read at a time: the loads' latency, not their number, is what
    // a walk over the many tiles in flight costs
    const volatile unsigned long long *p = status + d;
    int64_t t = tile - 1;  // next tile to add
    int spins = 0;
    for (bool done = false; !done && !failed;) {
      uint64_t x[RS_BACK];
#pragma unroll
      for (int i = 0; i < RS_BACK; ++i) x[i] = t >= i ? p[(t - i) * RS_BINS] : 0ull;
      int taken = 0;
#pragma unroll
      for (int i = 0; i < RS_BACK; ++i) {
        const uint64_t code = x[i] & ~RS_COUNT;
        if (!done && !failed && taken == i) {
          if (code == upto) {
            before += x[i] & RS_COUNT;
            done = true;
          } else if (code == own) {
            before += x[i] & RS_COUNT;
            ++taken;
          } else if (code == RS_POISON) {
            failed = true;
          }
        }
      }
      t -= taken;
      spins = taken ? 0 : spins + 1;
      if (spins > RS_SPIN_LIMIT) failed = true;
    }
  }
  failed = __syncthreads_or(failed);
  if (failed) {
    if (d < RS_BINS) *st = RS_POISON;
    if (threadIdx.x == 0) atomicOr(err, SORT_FAILED);
    return;
  }
  if (d < RS_BINS) {
    if (tile > 0) *st = upto | (before + mine);
    sm.goff[d] = digit_start[d] + before;
  }
#pragma unroll
  for (int i = 0; i < RS_ITEMS; ++i) {
    const int pos = warp * RS_WARP_SPAN + i * 32 + (int)lane;
    const uint32_t dd = pos < nvalid ? (uint32_t)(k[i] >> shift) & mask : mask;
    const uint32_t lpos = sm.bstart[dd] + sm.whist[warp][dd] + rank[i];
    sm.keys[lpos] = k[i];
    if (HAS_VALS) sm.vals[lpos] = v[i];
  }
  __syncthreads();
#pragma unroll 4
  for (int j = 0; j < RS_ITEMS; ++j) {
    const int lpos = j * RS_NT + threadIdx.x;
    if (lpos < nvalid) {
      const uint64_t key = sm.keys[lpos];
      const uint32_t dd = (uint32_t)(key >> shift) & mask;
      const uint64_t o = sm.goff[dd] + (uint64_t)(lpos - (int)sm.bstart[dd]);
      kout[o] = key;
      if (HAS_VALS) vout[o] = sm.vals[lpos];
    }
  }
}

// A sort of at most one tile: every pass in one kernel, in shared memory (in
// place). Small graphs sort a few thousand ranks, where launches were the cost.
template <bool HAS_VALS>
__global__ void __launch_bounds__(RS_NT) k_rs_small(uint64_t *__restrict__ keys,
                                                    uint32_t *__restrict__ vals, int count,
                                                    int bit_lo, int bit_hi) {
  extern __shared__ __align__(16) unsigned char rs_smem_raw[];
  RsSmem<HAS_VALS> &sm = *reinterpret_cast<RsSmem<HAS_VALS> *>(rs_smem_raw);
  const int warp = threadIdx.x >> 5;
  const unsigned lane = threadIdx.x & 31u;
  uint64_t k[RS_ITEMS];
  uint32_t v[HAS_VALS ? RS_ITEMS : 1];
  uint32_t rank[RS_ITEMS];
#pragma unroll
  for (int i = 0; i < RS_ITEMS; ++i) {
    const int pos = warp * RS_WARP_SPAN + i * 32 + (int)lane;
    k[i] = pos < count ? keys[pos] : ~0ull;
    if (HAS_VALS) v[i] = pos < count ? vals[pos] : 0u;
  }
  for (int shift = bit_lo; shift < bit_hi; shift += 8) {
    const uint32_t mask = bit_hi - shift < 8 ? (1u << (bit_hi - shift)) - 1u : 255u;
    rs_rank<HAS_VALS>(sm, k, count, shift, mask, rank);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i) {
      const int pos = warp * RS_WARP_SPAN + i * 32 + (int)lane;
      const uint32_t dd = pos < count ? (uint32_t)(k[i] >> shift) & mask : mask;
      const uint32_t lpos = sm.bstart[dd] + sm.whist[warp][dd] + rank[i];
      sm.keys[lpos] = k[i];
      if (HAS_VALS) sm.vals[lpos] = v[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i) {
      const int pos = warp * RS_WARP_SPAN + i * 32 + (int)lane;
      k[i] = sm.keys[pos];
      if (HAS_VALS) v[i] = sm.vals[pos];
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < RS_ITEMS; ++i) {
    const int pos = warp * RS_WARP_SPAN + i * 32 + (int)lane;
    if (pos < count) {
      keys[pos] = k[i];
      if (HAS_VALS) vals[pos] = v[i];
    }
  }
}

constexpr int SC_NT = 512;
constexpr int SC_ITEMS = 8;
constexpr int SC_TILE = SC_NT * SC_ITEMS;
constexpr int64_t SC_DIRECT = 1024;  // tiles whose sums every block adds up by itself

__global__ void __launch_bounds__(SC_NT) k_scan_reduce(const uint64_t *__restrict__ in,
                                                       int64_t count,
                                                       uint64_t *__restrict__ partial) {
  __shared__ uint64_t tmp[SC_NT / 32 + 1];
  const int64_t base = (int64_t)blockIdx.x * SC_TILE;
  uint64_t s = 0;
#pragma unroll
  for (int i = 0; i < SC_ITEMS; ++i) {
    int64_t idx = base + (int64_t)i * SC_NT + threadIdx.x;
    if (idx < count) s += in[idx];
  }
  uint64_t total;
  block_exclusive_scan<uint64_t, SC_NT>(s, tmp, &total);
  if (threadIdx.x == 0) partial[blockIdx.x] = total;
}

// partial: the tiles' sums, scanned already or (sums) not: then each block adds up
// those before it, which saves a launch while they are few.
__global__ void __launch_bounds__(SC_NT) k_scan_down(const uint64_t *in, uint64_t *out,
                                                     int64_t count,
                                                     const uint64_t *__restrict__ partial,
                                                     bool sums) {
  __shared__ uint64_t tile[SC_TILE];
  __shared__ uint64_t tmp[SC_NT / 32 + 1];
  const int64_t base = (int64_t)blockIdx.x * SC_TILE;
  uint64_t start = 0;
  if (partial && sums) {
    uint64_t x = 0;
    for (int i = threadIdx.x; i < (int)blockIdx.x; i += SC_NT) x += partial[i];
    block_exclusive_scan<uint64_t, SC_NT>(x, tmp, &start);
  } else if (partial) {
    start = partial[blockIdx.x];
  }
#pragma unroll
  for (int i = 0; i < SC_ITEMS; ++i) {
    int64_t idx = base + (int64_t)i * SC_NT + threadIdx.x;
    tile[i * SC_NT + threadIdx.x] = idx < count ? in[idx] : 0;
  }
  __syncthreads();
  uint64_t local[SC_ITEMS];
  uint64_t s = 0;
#pragma unroll
  for (int i = 0; i < SC_ITEMS; ++i) {
    local[i] = tile[threadIdx.x * SC_ITEMS + i];
    s += local[i];
  }
  uint64_t total;
  uint64_t run = block_exclusive_scan<uint64_t, SC_NT>(s, tmp, &total) + start;
#pragma unroll
  for (int i = 0; i < SC_ITEMS; ++i) {
    tile[threadIdx.x * SC_ITEMS + i] = run;
    run += local[i];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < SC_ITEMS; ++i) {
    int64_t idx = base + (int64_t)i * SC_NT + threadIdx.x;
    if (idx < count) out[idx] = tile[i * SC_NT + threadIdx.x];
  }
}

// 32-bit counts to offsets: the tiles' sums, then the tiles (out and, when given, a
// copy of it); sums beyond 32 bits wrap, as the offsets' users keep them below.
__global__ void __launch_bounds__(SC_NT) k_scan32_reduce(const uint32_t *__restrict__ in,
                                                         int64_t count,
                                                         uint64_t *__restrict__ partial) {
  __shared__ uint64_t tmp[SC_NT / 32 + 1];
  const int64_t base = (int64_t)blockIdx.x * SC_TILE;
  uint64_t s = 0;
#pragma unroll
  for (int i = 0; i < SC_ITEMS; ++i) {
    const int64_t idx = base + (int64_t)i * SC_NT + threadIdx.x;
    if (idx < count) s += in[idx];
  }
  uint64_t total;
  block_exclusive_scan<uint64_t, SC_NT>(s, tmp, &total);
  if (threadIdx.x == 0) partial[blockIdx.x] = total;
}

__global__ void __launch_bounds__(SC_NT) k_scan32_down(const uint32_t *in, uint32_t *out,
                                                       uint32_t *copy, int64_t count,
                                                       const uint64_t *__restrict__ partial,
                                                       bool sums) {
  __shared__ uint32_t tile[SC_TILE];
  __shared__ uint32_t tmp[SC_NT / 32 + 1];
  __shared__ uint64_t tmp64[SC_NT / 32 + 1];
  const int64_t base = (int64_t)blockIdx.x * SC_TILE;
  uint64_t start = 0;
  if (partial && sums) {
    uint64_t x = 0;
    for (int i = threadIdx.x; i < (int)blockIdx.x; i += SC_NT) x += partial[i];
    block_exclusive_scan<uint64_t, SC_NT>(x, tmp64, &start);
  } else if (partial) {
    start = partial[blockIdx.x];
  }
#pragma unroll
  for (int i = 0; i < SC_ITEMS; ++i) {
    const int64_t idx = base + (int64_t)i * SC_NT + threadIdx.x;
    tile[i * SC_NT + threadIdx.x] = idx < count ? in[idx] : 0;
  }
  __syncthreads();
  uint32_t local[SC_ITEMS], s = 0, total;
#pragma unroll
  for (int i = 0; i < SC_ITEMS; ++i) {
    local[i] = tile[threadIdx.x * SC_ITEMS + i];
    s += local[i];
  }
  uint32_t run = block_exclusive_scan<uint32_t, SC_NT>(s, tmp, &total) + (uint32_t)start;
#pragma unroll
  for (int i = 0; i < SC_ITEMS; ++i) {
    tile[threadIdx.x * SC_ITEMS + i] = run;
    run += local[i];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < SC_ITEMS; ++i) {
    const int64_t idx = base + (int64_t)i * SC_NT + threadIdx.x;
    if (idx < count) {
      out[idx] = tile[i * SC_NT + threadIdx.x];
      if (copy) copy[idx] = tile[i * SC_NT + threadIdx.x];
    }
  }
}

template <typename T>
__global__ void k_reduce_max(const T *__restrict__ in, int64_t count,
                             unsigned long long *__restrict__ out) {
  T best = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x)
    best = in[i] > best ? in[i] : best;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    T o = __shfl_xor_sync(0xffffffffu, best, d);
    best = o > best ? o : best;
  }
  if ((threadIdx.x & 31) == 0 && best > 0) atomicMax(out, (unsigned long long)best);
}

template <bool HAS_VALS>
bbtc_status rs_sort(uint64_t *keys, uint64_t *alt, uint32_t *vals, uint32_t *vals_alt,
                    int64_t count, int bit_lo, int bit_hi, cudaStream_t s, int32_t *err,
                    bool *in_alt) {
  const size_t smem = sizeof(RsSmem<HAS_VALS>);
  if (count <= RS_TILE) {
    BBTC_CUDA(cudaFuncSetAttribute(k_rs_small<HAS_VALS>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_rs_small<HAS_VALS><<<1, RS_NT, smem, s>>>(keys, vals, (int)count, bit_lo, bit_hi);
    BBTC_LAUNCH_CHECK();
    return BBTC_OK;
  }
  BBTC_CUDA(cudaFuncSetAttribute(k_rs_pass<HAS_VALS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem));
  const int64_t ntiles = (count + RS_TILE - 1) / RS_TILE;
  Scratch scratch(s);
  // digit counts of eight passes, their tickets, and the tiles' status words
  unsigned long long *hist = nullptr, *status = nullptr;
  constexpr int64_t HEAD = 8 * RS_BINS + 8;
  BBTC_TRY(scratch.get(&hist, HEAD + ntiles * RS_BINS));
  status = hist + HEAD;
  unsigned *tickets = reinterpret_cast<unsigned *>(hist + 8 * RS_BINS);
  BBTC_CUDA(cudaMemsetAsync(hist, 0, sizeof(unsigned long long) * (size_t)(HEAD + ntiles * RS_BINS), s));
  const int passes = (bit_hi - bit_lo + 7) / 8;
  k_rs_hist<<<grid_for(count, RS_NT * 16, 8), RS_NT, 0, s>>>(keys, count, bit_lo, bit_hi, hist);
  BBTC_LAUNCH_CHECK();
  k_rs_digits<<<(unsigned)passes, RS_BINS, 0, s>>>(hist);
  BBTC_LAUNCH_CHECK();
  uint64_t *kin = keys, *kout = alt;
  uint32_t *vin = vals, *vout = vals_alt;
  for (int p = 0; p < passes; ++p) {
    const int shift = bit_lo + 8 * p;
    const uint32_t mask = bit_hi - shift < 8 ? (1u << (bit_hi - shift)) - 1u : 255u;
    k_rs_pass<HAS_VALS><<<(unsigned)ntiles, RS_NT, smem, s>>>(
        kin, kout, vin, vout, count, shift, mask, p, hist + p * RS_BINS, tickets + p, status, err);
    BBTC_LAUNCH_CHECK();
    std::swap(kin, kout);
    std::swap(vin, vout);
  }
  *in_alt = (passes & 1) != 0;
  return BBTC_OK;
}

}  // namespace

bbtc_status radix_sort(uint64_t *keys, uint64_t *alt, uint32_t *vals, uint32_t *vals_alt,
                       int64_t count, int bit_lo, int bit_hi, cudaStream_t s, int32_t *err,
                       bool *in_alt) {
  *in_alt = false;
  if (count <= 1 || bit_hi <= bit_lo) return BBTC_OK;
  if ((count + RS_TILE - 1) / RS_TILE > 0x7fffffffLL) {
    set_error("radix_sort: %lld keys exceed the grid limit", (long long)count);
    return BBTC_EINVAL;
  }
  return vals ? rs_sort<true>(keys, alt, vals, vals_alt, count, bit_lo, bit_hi, s, err, in_alt)
              : rs_sort<false>(keys, alt, nullptr, nullptr, count, bit_lo, bit_hi, s, err, in_alt);
}

bbtc_status exclusive_scan_u64(const uint64_t *in, uint64_t *out, int64_t count,
                               cudaStream_t s) {
  if (count <= 0) return BBTC_OK;
  const int64_t nblocks = (count + SC_TILE - 1) / SC_TILE;
  if (nblocks == 1) {
    k_scan_down<<<1, SC_NT, 0, s>>>(in, out, count, nullptr, false);
    BBTC_LAUNCH_CHECK();
    return BBTC_OK;
  }
  Scratch scratch(s);
  uint64_t *partial = nullptr;
  BBTC_TRY(scratch.get(&partial, nblocks));
  k_scan_reduce<<<(unsigned)nblocks, SC_NT, 0, s>>>(in, count, partial);
  BBTC_LAUNCH_CHECK();
  const bool sums = nblocks <= SC_DIRECT;
  if (!sums) BBTC_TRY(exclusive_scan_u64(partial, partial, nblocks, s));
  k_scan_down<<<(unsigned)nblocks, SC_NT, 0, s>>>(in, out, count, partial, sums);
  BBTC_LAUNCH_CHECK();
  return BBTC_OK;
}

bbtc_status exclusive_scan_u32(const uint32_t *in, uint32_t *out, uint32_t *copy, int64_t count,
                               cudaStream_t s) {
  if (count <= 0) return BBTC_OK;
  const int64_t nblocks = (count + SC_TILE - 1) / SC_TILE;
  if (nblocks == 1) {
    k_scan32_down<<<1, SC_NT, 0, s>>>(in, out, copy, count, nullptr, false);
    BBTC_LAUNCH_CHECK();
    return BBTC_OK;
  }
  Scratch scratch(s);
  uint64_t *partial = nullptr;
  BBTC_TRY(scratch.get(&partial, nblocks));
  k_scan32_reduce<<<(unsigned)nblocks, SC_NT, 0, s>>>(in, count, partial);
  BBTC_LAUNCH_CHECK();
  const bool sums = nblocks <= SC_DIRECT;
  if (!sums) BBTC_TRY(exclusive_scan_u64(partial, partial, nblocks, s));
  k_scan32_down<<<(unsigned)nblocks, SC_NT, 0, s>>>(in, out, copy, count, partial, sums);
  BBTC_LAUNCH_CHECK();
  return BBTC_OK;
}

bbtc_status reduce_max_i64(const int64_t *in, int64_t count, int64_t *out, cudaStream_t s) {
  BBTC_CUDA(cudaMemsetAsync(out, 0, sizeof(int64_t), s));
  if (count <= 0) return BBTC_OK;
  k_reduce_max<int64_t><<<grid_for(count, 256, 8), 256, 0, s>>>(
      in, count, reinterpret_cast<unsigned long long *>(out));
  BBTC_LAUNCH_CHECK();
  return BBTC_OK;
}

bbtc_status reduce_max_i32(const int32_t *in, int64_t count, int32_t *out, cudaStream_t s) {
  // accumulate in a 64-bit word; the caller's int32 receives the low half
  unsigned long long *tmp = nullptr;
  Scratch scratch(s);
  BBTC_TRY(scratch.get(&tmp, 1));
  BBTC_CUDA(cudaMemsetAsync(tmp, 0, sizeof(unsigned long long), s));
  if (count > 0) {
    k_reduce_max<int32_t><<<grid_for(count, 256, 8), 256, 0, s>>>(in, count, tmp);
    BBTC_LAUNCH_CHECK();
  }
  BBTC_CUDA(cudaMemcpyAsync(out, tmp, sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
  return BBTC_OK;
}

}  // namespace bbtc
