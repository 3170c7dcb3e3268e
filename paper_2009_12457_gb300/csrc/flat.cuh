// flat.cuh -- the probe loop shared by the resident counting kernels.
#pragma once

#include "common.cuh"

namespace bbtc {

namespace {

// The 4-bit mask of the columns q .. q + 3 inside [lo, hi).
__device__ __forceinline__ uint32_t columns_inside(uint32_t q, uint32_t lo, uint32_t hi) {
  const int first = max((int)(lo - q), 0);
  const int last = min((int)(hi - q), 4);
  return (0xfu << first) & ((1u << last) - 1u);
}

// Runs a batch's probes: the quads of its in-edges are flattened over the
// lanes, 32 * UQ at a time. The owner of a lane's quad is found from the bit
// word of the first quads that fall into the 32 at hand, so it costs the same
// for every lane and length. on_quad(owner record, the quad, the mask of its
// columns inside the probe run, the first column's position) takes each.
template <int UQ, typename OnQuad>
__device__ __forceinline__ void flat_rounds(const int32_t *__restrict__ ci, const uint4 *rec,
                                            uint32_t total, uint32_t first, bool has,
                                            unsigned lane, OnQuad on_quad) {
  int owners = -1;  // index of the last record that starts before the round
  const unsigned le = 0xffffffffu >> (31 - lane);
  for (uint32_t jb = 0; jb < total; jb += 32u * UQ) {
    int4 w[UQ];
    uint32_t msk[UQ];
    int own[UQ];
    uint32_t pos[UQ];
#pragma unroll
    for (int r = 0; r < UQ; ++r) {
      const uint32_t at = first - (jb + 32u * r);
      const unsigned starts = __reduce_or_sync(0xffffffffu, has && at < 32u ? 1u << at : 0u);
      own[r] = owners + __popc(starts & le);
      owners += __popc(starts);
      const uint32_t j = jb + 32u * r + lane;
      msk[r] = 0u;
      pos[r] = 0u;
      w[r] = make_int4(0, 0, 0, 0);
      if (j < total) {
        const uint4 t = rec[own[r]];
        const uint32_t q = t.z + 4u * j;
        w[r] = *reinterpret_cast<const int4 *>(ci + q);
        msk[r] = columns_inside(q, t.x, t.y);
        pos[r] = q;
      }
    }
#pragma unroll
    for (int r = 0; r < UQ; ++r) on_quad(own[r], w[r], msk[r], pos[r]);
  }
}

}  // namespace

}  // namespace bbtc
