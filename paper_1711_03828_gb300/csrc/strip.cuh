// strip.cuh -- the work layout of the SET sweeps for chains of any length
// (sweep_strip_kernel, sweep_smc_strip_kernel).
//
// A warp walks along whole chains in strips of 32 lanes, a lane holding two
// bonded particles of a chain at a time: R, which moves in the first set of
// this sweep, and L, the one before it, which moves in the second.  With the
// odd positions first (set-order bit 1) unit k of a chain is (2k, 2k+1), with
// the even ones first (2k-1, 2k), so in either order
//   first set:  R moves against L of its own lane and L of the next lane,
//   second set: L moves against R of the lane before and R of its own lane,
// without selecting by the order bit and with both sets on all lanes.  A chain
// of N particles takes U = floor(N/2) + 1 units in either order (one or two of
// their slots empty).  Chains follow one another without padding and may
// continue from one strip to the next: the last lane's next unit is the first
// one of the following strip, whose positions are already loaded (the prefetch),
// and the first lane's previous R is the last lane's of the strip before, kept
// in a register.  A work item is C chains, ceil(C U / 32) strips, C chosen by
// the host (strip_chains) so that the items fill their strips and the warps.
//
// Tiles of whole chains, 64, 128 or 256 slots per warp (floor(slots/N) chains),
// left the rest of the slots empty (N = 33: 48 %, N = 100: 22 %), held 4 or 8
// particles per lane in up to 195 registers and moved them in divergent
// branches, one slot after another.
#pragma once

#include "common.cuh"

namespace soma {

template <typename IDX>
struct StripLane {
  uint32_t idx;     // chain position of R (L is idx - 1)
  bool vL, vR;      // the slots hold a particle
  IDX m;            // particle index of R

  __device__ __forceinline__ bool own() const { return vL && vR; }             // L - R bond
  __device__ __forceinline__ bool next(uint32_t N) const { return vR && idx + 1u < N; }  // R - next L
  __device__ __forceinline__ bool prev() const { return vL && idx >= 2u; }     // previous R - L
};

// Walks a block's items.  claim() hands out the block's items in order; place()
// gives a lane's unit of the current strip; step() goes to the following strip
// (false: the block's items are used up).
template <typename IDX>
struct StripWalk {
  const SweepArgs& p;
  uint32_t* next_item;          // shared counter of the block
  uint32_t item0, item_end;
  int lane;
  uint32_t U, q, r;             // units per chain; 32 = q U + r
  uint32_t ctr3, sweep;
  uint32_t c, k, strips, bits;  // chain in the item, unit in the chain, strips left, order bits
  uint32_t n_ch;                // chains of this item
  IDX chain0;

  __device__ __forceinline__ StripWalk(const SweepArgs& p_, uint32_t* next_item_, uint32_t item0_,
                                       uint32_t item_end_, int lane_, uint32_t ctr3_, uint32_t sweep_)
      : p(p_), next_item(next_item_), item0(item0_), item_end(item_end_), lane(lane_),
        U(p_.strip_units), q(32u / p_.strip_units), r(32u - q * p_.strip_units), ctr3(ctr3_),
        sweep(sweep_), c(0), k(0), strips(0), bits(0), n_ch(0), chain0(0) {}

  __device__ __forceinline__ bool step() {
    if (strips > 1u) {
      --strips;
      c += q;
      k += r;
      if (k >= U) {
        k -= U;
        ++c;
      }
      return true;
    }
    uint32_t it = 0u;
    if (lane == 0) it = atomicAdd(next_item, 1u);
    it = item0 + __shfl_sync(FULL, it, 0);
    if (it >= item_end) {
      strips = 0u;
      n_ch = 0u;
      return false;
    }
    chain0 = (IDX)it * p.strip_chains;
    const IDX rem = (IDX)p.g.n_chains - chain0;
    n_ch = rem < (IDX)p.strip_chains ? (uint32_t)rem : p.strip_chains;
    strips = (n_ch * U + 31u) / 32u;
    c = (uint32_t)lane / U;
    k = (uint32_t)lane - c * U;
    bits = p.strip_order;
    if (p.strip_odd && rem <= (IDX)p.strip_chains) bits ^= 1u << (n_ch - 1u);
    if (p.set_order_random) {   // bit 0 of word 3 of the move draw of each chain's particle 0
      const uint64_t m = (uint64_t)(chain0 + lane) * p.g.N + p.g.id_base;
      const uint4 w = philox_rk(make_uint4((uint32_t)m, (uint32_t)(m >> 32), sweep, ctr3), p.g);
      bits = __ballot_sync(FULL, w.w & 1u);
    }
    return true;
  }

  __device__ __forceinline__ StripLane<IDX> place() const {
    StripLane<IDX> s;
    const uint32_t N = p.g.N;
    s.idx = 2u * k + ((bits >> (c & 31u)) & 1u);
    const bool in = c < n_ch;
    s.vR = in && s.idx < N;
    s.vL = in && s.idx - 1u < N;    // idx 0: wraps, no particle
    s.m = (chain0 + c) * N + s.idx;
    return s;
  }
};

struct StripPos {
  float Lx, Ly, Lz, Rx, Ry, Rz;
};

template <typename IDX>
__device__ __forceinline__ void strip_load(const SweepArgs& p, const StripLane<IDX>& s, StripPos& v) {
  if (s.vL) {
    v.Lx = __ldcs(p.x + (s.m - 1u));
    v.Ly = __ldcs(p.y + (s.m - 1u));
    v.Lz = __ldcs(p.z + (s.m - 1u));
  }
  if (s.vR) {
    v.Rx = __ldcs(p.x + s.m);
    v.Ry = __ldcs(p.y + s.m);
    v.Rz = __ldcs(p.z + s.m);
  }
}

template <typename IDX>
__device__ __forceinline__ void strip_store(const SweepArgs& p, const StripLane<IDX>& s,
                                            const StripPos& v) {
  if (s.vL) {
    __stcs(p.x + (s.m - 1u), v.Lx);
    __stcs(p.y + (s.m - 1u), v.Ly);
    __stcs(p.z + (s.m - 1u), v.Lz);
  }
  if (s.vR) {
    __stcs(p.x + s.m, v.Rx);
    __stcs(p.y + s.m, v.Ry);
    __stcs(p.z + s.m, v.Rz);
  }
}

// Occupation count of the final cells (one atomic when they are the same).
template <typename IDX>
__device__ __forceinline__ void strip_count(uint32_t* __restrict__ n, const StripLane<IDX>& s,
                                            uint32_t cL, uint32_t cR, uint32_t aL, uint32_t aR) {
  const bool same = s.own() && cL == cR;
  if (s.vL) atomicAdd(n + cL, same ? aL + aR : aL);
  if (s.vR && !same) atomicAdd(n + cR, aR);
}

// L of the next unit (lane + 1; the last lane's from the following strip) and
// R of the previous one (lane - 1; the first lane's from the strip before).
__device__ __forceinline__ float strip_next(float L, float following, int lane) {
  return __shfl_sync(FULL, lane == 0 ? following : L, (lane + 1) & 31);
}
__device__ __forceinline__ float strip_prev(float R, float before, int lane) {
  return __shfl_sync(FULL, lane == 31 ? before : R, (lane + 31) & 31);
}

}  // namespace soma
