// sweep.cu -- the Monte-Carlo step of the SCMF cycle (arXiv:1711.03828,
// Sec. 2.2 and the SET iteration of Sec. 3.1.2) on sm_103a, uniform moves.
//
// Even N <= 64: sweep_pair_kernel (pair_body.cuh), whole chains per warp tile,
// an even and an odd particle of one chain per lane.  Other lengths:
// sweep_strip_kernel (strip.cuh), a warp walking along its chains.  Both sets
// keep all lanes busy (the paper's SET scheme leaves half its threads idle per
// set for a linear chain); bond partners in a neighbouring lane come by warp
// shuffles; no shared memory but the counters that hand out the work.
//
// Per particle: one Philox4x32-10 draw (counter = particle, sweep) gives the
// three displacement uniforms and the acceptance uniform; the set order of a
// chain is bit 0 of the acceptance word of its first particle.  The trial
// position r + a v is rounded once to the stored FP32 precision (a fused
// multiply-add, round-to-nearest).  The two field values omega_t(c) and
// omega_t(c') are gathered from the L2-resident omega planes before the set
// loop since c' does not depend on the neighbours.  After both sets the final
// cells are added to the packed occupation grid n[(s+1)&1] with 32-bit
// atomics (the occupation count of the next field update, fused).
//
// Streams: positions are loaded and stored with evict-first hints so the
// 28 MB grid and the omega planes stay in L2.
#include <algorithm>

#include "kernels.h"
#include "pair_body.cuh"
#include "strip.cuh"

namespace soma {

__device__ __forceinline__ float dist2(float ax, float ay, float az, float bx, float by, float bz) {
  const float dx = ax - bx, dy = ay - by, dz = az - bz;
  return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

// Energy change of the bonds of a particle moved from r to t: partner p (if
// hp) and q (if hq), each as the difference of the squared lengths.
__device__ __forceinline__ float bond_change(bool hp, bool hq, float rx, float ry, float rz, float tx,
                                             float ty, float tz, float px, float py, float pz,
                                             float qx, float qy, float qz) {
  const float ep = dist2(tx, ty, tz, px, py, pz) - dist2(rx, ry, rz, px, py, pz);
  const float eq = dist2(tx, ty, tz, qx, qy, qz) - dist2(rx, ry, rz, qx, qy, qz);
  return (hp ? ep : 0.f) + (hq ? eq : 0.f);
}

// Chains of odd length and of more than 64 particles, in the strips of
// strip.cuh.  One block of 32 warps per SM owns a contiguous range of items,
// handed out from a shared-memory counter.  WIDE: every axis has two or more
// cells.  Issue-bound like the paired kernel (454 warp instructions a strip);
// the paper's thin film (N = 100, 16.5M particles, 16-bit fields): 214 us a
// sweep in tiles of 128 slots, 152 us in strips.
template <typename WT, typename IDX, bool WIDE>
__global__ void __launch_bounds__(1024, 1) sweep_strip_kernel(const SweepArgs p) {
  __shared__ uint32_t s_next;
  const int lane = threadIdx.x & 31;
  const uint32_t chunk = (p.n_items + gridDim.x - 1) / gridDim.x;
  const uint32_t item0 = blockIdx.x * chunk;
  if (threadIdx.x == 0) s_next = 0u;
  __syncthreads();
  // (a few items a block: their warps wait on latencies alone, and leaving the others
  // before the wait measured up to 12 % slower)
  if (chunk >= 8u && idle_warp(item0, chunk, p.n_items)) return;
  chained_begin();
  const unsigned long long s64 = *p.d_sweep;
  const uint32_t sweep = (uint32_t)s64;
  uint32_t* __restrict__ nacc = ((s64 + 1ull) & 1ull) ? p.n1 : p.n0;
  const WT* __restrict__ wA = static_cast<const WT*>(p.wA);
  const WT* __restrict__ wB = static_cast<const WT*>(p.wB);
  const uint32_t N = p.g.N, N_A = p.g.N_A;
  const uint32_t ctr3 = (PURPOSE_MOVE << 24) | (p.g.replica & 0xFFFFFFu);
  StripWalk<IDX> walk(p, &s_next, item0, min(item0 + chunk, p.n_items), lane, ctr3, sweep);

  StripPos nv = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  float bx = 0.f, by = 0.f, bz = 0.f;   // R of the strip before
  bool have = walk.step();
  StripLane<IDX> ns = walk.place();
  strip_load(p, ns, nv);
  unsigned my_acc = 0;
  while (have) {
    const StripLane<IDX> s = ns;
    StripPos v = nv;
    have = walk.step();
    ns = walk.place();
    strip_load(p, ns, nv);

    // Both slots at once, L low and R high in packed FP32x2 registers: cells,
    // draws, trial positions as in pair_body.cuh.
    const unsigned long long MAG = f2_pack(12582912.0f, 12582912.0f);
    const unsigned long long X = f2_pack(v.Lx, v.Rx), Y = f2_pack(v.Ly, v.Ry), Z = f2_pack(v.Lz, v.Rz);
    float fx0, fx1, fy0, fy1, fz0, fz1;
    f2_unpack(f2_add_rm(X, MAG), fx0, fx1);
    f2_unpack(f2_add_rm(Y, MAG), fy0, fy1);
    f2_unpack(f2_add_rm(Z, MAG), fz0, fz1);
    uint32_t cL = cell_of_floor_bits<WIDE>(p.g, __float_as_uint(fx0), __float_as_uint(fy0), __float_as_uint(fz0));
    uint32_t cR = cell_of_floor_bits<WIDE>(p.g, __float_as_uint(fx1), __float_as_uint(fy1), __float_as_uint(fz1));
    const bool aL = s.idx <= N_A, aR = s.idx < N_A;   // A particles: idx - 1 < N_A, idx < N_A
    const WT* __restrict__ wL = aL ? wA : wB;
    const WT* __restrict__ wR = aR ? wA : wB;
    // an empty slot's cells lie in the grid too; its values are not used
    const float oL = load_w<WT>(wL, cL), oR = load_w<WT>(wR, cR);
    const IDX mR = s.m + (IDX)p.g.id_base, mL = mR - 1u;
    const uint32_t hL = sizeof(IDX) > 4 ? (uint32_t)((uint64_t)mL >> 32) : 0u;
    const uint32_t hR = sizeof(IDX) > 4 ? (uint32_t)((uint64_t)mR >> 32) : 0u;
    const uint4 rL = philox_rk(make_uint4((uint32_t)mL, hL, sweep, ctr3), p.g);
    const uint4 rR = philox_rk(make_uint4((uint32_t)mR, hR, sweep, ctr3), p.g);
    const unsigned long long S2 = f2_pack(1.1920928955078125e-7f, 1.1920928955078125e-7f);
    const unsigned long long C2 = f2_pack(-0.99999994039535522461f, -0.99999994039535522461f);
    const unsigned long long A2 = f2_pack(p.a, p.a);
    const unsigned long long XN = f2_fma_rn(
        A2, f2_fma_rn(f2_pack(__uint2float_rn(rL.x >> 8), __uint2float_rn(rR.x >> 8)), S2, C2), X);
    const unsigned long long YN = f2_fma_rn(
        A2, f2_fma_rn(f2_pack(__uint2float_rn(rL.y >> 8), __uint2float_rn(rR.y >> 8)), S2, C2), Y);
    const unsigned long long ZN = f2_fma_rn(
        A2, f2_fma_rn(f2_pack(__uint2float_rn(rL.z >> 8), __uint2float_rn(rR.z >> 8)), S2, C2), Z);
    float txL, txR, tyL, tyR, tzL, tzR;
    f2_unpack(XN, txL, txR);
    f2_unpack(YN, tyL, tyR);
    f2_unpack(ZN, tzL, tzR);
    f2_unpack(f2_add_rm(XN, MAG), fx0, fx1);
    f2_unpack(f2_add_rm(YN, MAG), fy0, fy1);
    f2_unpack(f2_add_rm(ZN, MAG), fz0, fz1);
    const uint32_t nL = cell_of_floor_bits<WIDE>(p.g, __float_as_uint(fx0), __float_as_uint(fy0), __float_as_uint(fz0));
    const uint32_t nR = cell_of_floor_bits<WIDE>(p.g, __float_as_uint(fx1), __float_as_uint(fy1), __float_as_uint(fz1));
    const float dL = load_w<WT>(wL, nL) - oL, dR = load_w<WT>(wR, nR) - oR;
    float lnuL, lnuR;
    {
      float u0, u1;
      f2_unpack(f2_fma_rn(f2_pack(__uint2float_rn(rL.w >> 8), __uint2float_rn(rR.w >> 8)),
                          f2_pack(5.9604644775390625e-8f, 5.9604644775390625e-8f),
                          f2_pack(2.98023223876953125e-8f, 2.98023223876953125e-8f)), u0, u1);
      lnuL = __logf(u0);
      lnuR = __logf(u1);
    }

    {  // first set: R moves
      const float qx = strip_next(v.Lx, nv.Lx, lane), qy = strip_next(v.Ly, nv.Ly, lane),
                  qz = strip_next(v.Lz, nv.Lz, lane);
      const float e = bond_change(s.own(), s.next(N), v.Rx, v.Ry, v.Rz, txR, tyR, tzR, v.Lx, v.Ly,
                                  v.Lz, qx, qy, qz);
      const float dE = fmaf(p.K_b, e, dR);
      if (s.vR && (dE <= 0.f || lnuR < -dE)) {
        v.Rx = txR;
        v.Ry = tyR;
        v.Rz = tzR;
        cR = nR;
        ++my_acc;
      }
    }
    {  // second set: L moves
      const float px = strip_prev(v.Rx, bx, lane), py = strip_prev(v.Ry, by, lane),
                  pz = strip_prev(v.Rz, bz, lane);
      const float e = bond_change(s.prev(), s.own(), v.Lx, v.Ly, v.Lz, txL, tyL, tzL, px, py, pz,
                                  v.Rx, v.Ry, v.Rz);
      const float dE = fmaf(p.K_b, e, dL);
      if (s.vL && (dE <= 0.f || lnuL < -dE)) {
        v.Lx = txL;
        v.Ly = tyL;
        v.Lz = tzL;
        cL = nL;
        ++my_acc;
      }
    }
    bx = v.Rx;
    by = v.Ry;
    bz = v.Rz;
    strip_store(p, s, v);
    strip_count(nacc, s, cL, cR, aL ? 1u : 0x10000u, aR ? 1u : 0x10000u);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) my_acc += __shfl_xor_sync(FULL, my_acc, o);
  if (lane == 0 && my_acc) atomicAdd(p.acc, (unsigned long long)my_acc);
}

// Even N <= 64: the paired tile body of pair_body.cuh over one system.  One
// block of 32 warps per SM owns a contiguous range of tiles (spatially
// ordered chains); its warps take the range's tiles in order from a
// shared-memory counter, so they work on neighbouring tiles (field values
// repeat in L1) and all finish within a tile of each other.  With three
// blocks of a third of the range each, the warp scheduler's preference for
// the oldest warps finished the first block well before the third, and the
// SM ran its last sixth at a third or two thirds of its warps.  The next
// tile's positions are loaded while the current one is processed.  IDX is the
// index type: 32-bit when M < 2^32 (Philox counter word 1 = 0).
// MIXED: a mixture of linear architectures (the type sequence of each chain
// is read per tile); otherwise every chain is the diblock of N_A A particles.
template <typename WT, typename IDX, bool MIXED>
__global__ void __launch_bounds__(1024, 1) sweep_pair_kernel(const SweepArgs p) {
  __shared__ uint32_t s_next;
  const int lane = threadIdx.x & 31;
  const uint32_t n_tiles_all = (uint32_t)p.n_tiles;
  const uint32_t chunk = (n_tiles_all + gridDim.x - 1) / gridDim.x;
  const uint32_t t_begin = blockIdx.x * chunk;
  const uint32_t t_end = min(t_begin + chunk, n_tiles_all);
  if (threadIdx.x == 0) s_next = 0u;
  __syncthreads();
  if (idle_warp(t_begin, chunk, n_tiles_all)) return;
  auto claim = [&]() -> uint32_t {
    uint32_t t = 0u;
    if (lane == 0) t = atomicAdd(&s_next, 1u);
    return t_begin + __shfl_sync(FULL, t, 0);
  };
  chained_begin();
  const unsigned long long s64 = *p.d_sweep;
  const uint32_t sweep = (uint32_t)s64;
  uint32_t* __restrict__ nacc = ((s64 + 1ull) & 1ull) ? p.n1 : p.n0;
  const uint32_t ctr3 = (PURPOSE_MOVE << 24) | (p.g.replica & 0xFFFFFFu);
  PairLane<WT> L;
  L.init(lane, p.g.N, p.g.N_A, p.wA, p.wB);
  const uint32_t TN = p.G * p.g.N;
  const uint32_t full_tiles = (uint32_t)p.full_tiles;
  auto lane_ok = [&](uint32_t t) { return L.in_tile(t < full_tiles, p.last_rows); };
  // tiles that fill all 64 slots need no masks
  const uint32_t dense_tiles = TN == 64u ? full_tiles : 0u;
  const bool wide = p.g.nx > 1 && p.g.ny > 1 && p.g.nz > 1;

  float2 px = make_float2(0.f, 0.f), py = px, pz = px;
  auto load_pos = [&](uint32_t t) {
    if (t < t_end && lane_ok(t)) {
      const IDX b = (IDX)t * TN + L.li0;
      px = __ldcs(reinterpret_cast<const float2*>(p.x + b));
      py = __ldcs(reinterpret_cast<const float2*>(p.y + b));
      pz = __ldcs(reinterpret_cast<const float2*>(p.z + b));
    }
  };
  uint32_t tile = claim();
  load_pos(tile);
  unsigned my_acc = 0;
  while (tile < t_end) {
    const bool valid = lane_ok(tile);
    const IDX base = (IDX)tile * TN + L.li0;
    const float x0 = px.x, x1 = px.y, y0 = py.x, y1 = py.y, z0 = pz.x, z1 = pz.y;
    const uint32_t next_tile = claim();
    load_pos(next_tile);
    PairLane<WT> Lt = L;
    if (MIXED) {
      const uint64_t chain = (uint64_t)tile * p.G + L.lane_chain;
      const uint64_t seq = chain < p.g.n_chains ? __ldg(p.seq + __ldg(p.arch + chain)) : 0ull;
      Lt.set_types((seq >> L.ci0) & 1ull, (seq >> (L.ci0 + 1u)) & 1ull, p.wA, p.wB);
    }
    const IDX cbase = base + (IDX)p.g.id_base;
    if (tile < dense_tiles && wide)
      my_acc += pair_tile<WT, IDX, false, true>(p.g, p.g, Lt, p.x, p.y, p.z, nacc, base, cbase, true,
                                                sweep, ctr3, p.set_order_random, p.a, p.K_b, x0, x1,
                                                y0, y1, z0, z1);
    else if (tile < dense_tiles)
      my_acc += pair_tile<WT, IDX, false, false>(p.g, p.g, Lt, p.x, p.y, p.z, nacc, base, cbase, true,
                                                 sweep, ctr3, p.set_order_random, p.a, p.K_b, x0,
                                                 x1, y0, y1, z0, z1);
    else
      my_acc += pair_tile<WT, IDX, true, false>(p.g, p.g, Lt, p.x, p.y, p.z, nacc, base, cbase, valid,
                                                sweep, ctr3, p.set_order_random, p.a, p.K_b, x0, x1,
                                                y0, y1, z0, z1);
    tile = next_tile;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) my_acc += __shfl_xor_sync(FULL, my_acc, o);
  if (lane == 0 && my_acc) atomicAdd(p.acc, (unsigned long long)my_acc);
}

template <typename IDX, bool WIDE>
static const void* pick_strip(int grid_dtype) {
  switch (grid_dtype) {
    case 1: return (const void*)sweep_strip_kernel<__nv_bfloat16, IDX, WIDE>;
    case 2: return (const void*)sweep_strip_kernel<__half, IDX, WIDE>;
    default: return (const void*)sweep_strip_kernel<float, IDX, WIDE>;
  }
}

static const void* sweep_kernel_ptr(const SweepShape& s, int grid_dtype, bool mixed) {
  if (s.move == 1) return smc_kernel_ptr(s.strip, s.big);
  if (s.move == 2) return learned_kernel_ptr(s.Q, grid_dtype);
  if (!s.strip) {
    if (s.big) {
      switch (grid_dtype) {
        case 1: return (const void*)sweep_pair_kernel<__nv_bfloat16, uint64_t, false>;
        case 2: return (const void*)sweep_pair_kernel<__half, uint64_t, false>;
        default: return (const void*)sweep_pair_kernel<float, uint64_t, false>;
      }
    }
    if (mixed) {
      switch (grid_dtype) {
        case 1: return (const void*)sweep_pair_kernel<__nv_bfloat16, uint32_t, true>;
        case 2: return (const void*)sweep_pair_kernel<__half, uint32_t, true>;
        default: return (const void*)sweep_pair_kernel<float, uint32_t, true>;
      }
    }
    switch (grid_dtype) {
      case 1: return (const void*)sweep_pair_kernel<__nv_bfloat16, uint32_t, false>;
      case 2: return (const void*)sweep_pair_kernel<__half, uint32_t, false>;
      default: return (const void*)sweep_pair_kernel<float, uint32_t, false>;
    }
  }
  if (s.big) return pick_strip<uint64_t, false>(grid_dtype);
  return s.wide ? pick_strip<uint32_t, true>(grid_dtype) : pick_strip<uint32_t, false>(grid_dtype);
}

// Chains per work item of the strip kernels: C chains of U units take
// ceil(C U / 32) strips, and the n/C items go to the warps of one block per SM.  The C
// of the lowest cost: a block's items times their strips (what its warps issue; each
// item a draw per chain and its last strip partly empty besides), and per round of
// warps the latency of one item's strips, which the others hide once; and the more
// strips an item has, the further apart in space a block's warps work (their field
// values repeat less in L1).  Without the latency, one round of many short items looked
// as good as one of few full ones: 16 cycles of 65,536 particles, N = 5, took 161 us in
// items of 3 chains (9 of 32 lanes) and take 124 in items of 10.  Without the distance,
// the thin film (N = 100, 16.5M) took 2.48 ms in items of 18 chains, 2.43 in items of 5.
// Over 286 systems of N = 3 to 256 and 8,000 to 16M particles every C of at most 32
// strips was timed: the one chosen here takes 1.0 % longer than the best on average,
// the one of fewest rounds alone 7.1 %.
constexpr uint32_t STRIPS_MAX = 32;
constexpr double ITEM_COST = 1.5, SPREAD_COST = 0.015, ROUND_COST = 8.0;   // strips; items

static uint32_t strip_chains(uint64_t n, uint32_t U, uint64_t sms, uint64_t warps) {
  uint32_t best = 1;
  double least = 0.0;
  for (uint32_t C = 1; C <= 32u; ++C) {
    const uint32_t strips = (C * U + 31u) / 32u;
    if (C > 1u && strips > STRIPS_MAX) break;
    const uint64_t items = (n + C - 1u) / C, per = (items + sms - 1u) / sms;
    const uint64_t rounds = (per + warps - 1u) / warps;
    const double cost = ((double)per + ROUND_COST * (double)rounds) *
                        ((double)strips + ITEM_COST + SPREAD_COST * strips * strips);
    if (C == 1u || cost < least) {
      least = cost;
      best = C;
    }
  }
  return best;
}

// Most rounds of a block's warps that are made even by launching fewer warps: 76
// tiles per SM (734,000 particles, 16 cycles) take 211 us in 3 rounds of 26 warps, 227
// with 32, of which 12 work in the last round.  Where more than half of them would work
// there, all are better (the thin film's 217 items in 7 rounds: 2.44 ms with 31 warps,
// 2.43 with 32).
constexpr uint64_t EVEN_ROUNDS = 8;

SweepShape sweep_shape(const Geom& g, int sm_count, int grid_dtype, int move, bool learned_fp32,
                       bool learned_umma, bool molecule) {
  const uint64_t n_chains = g.n_chains;
  const uint32_t N = g.N;
  SweepShape s;
  s.move = move;
  s.learned_tc = false;
  s.learned_umma = false;
  s.molecule = false;
  s.Q = (N <= 64) ? 1 : (N <= 128 ? 2 : 4);
  s.G = (uint32_t)(64 * s.Q) / N;
  s.n_tiles = (n_chains + s.G - 1) / s.G;
  s.pair = (s.Q == 1) && (N % 2 == 0);
  s.big = n_chains * N >= (1ull << 32) || s.n_tiles >= (1ull << 31);
  s.wide = g.nx > 1 && g.ny > 1 && g.nz > 1;
  s.units = N == 1u ? 1u : N / 2u + 1u;
  // Uniform moves of even N <= 64 run in pair tiles.  Smart Monte Carlo moves
  // do where the tiles hold at least as many particles per slot as the strips
  // (G N of 64 slots against N of 2 U) and the indices fit 32 bits.
  s.strip = !s.pair || (move == 1 && (s.big || s.G * s.units < 32u));
  if (move == 2 || (molecule && move == 0)) s.strip = false;
  s.block = 256;
  s.chained = false;
  bool one_per_sm = false;
  if (move == 2 && s.pair && !s.big && !learned_fp32) {
    s.learned_tc = true;
    s.learned_umma = learned_umma;
    one_per_sm = !learned_umma;
    s.block = learned_umma ? 128 : 512;   // 16 warps (mma.sync, learned_tc.cu)
  } else if (molecule && move == 0) {
    s.molecule = true;
    s.block = MOL_BLOCK;
  } else if (move != 2) {
    // 32 warps in 64 registers without spills for uniform moves (16 cycles of 134M
    // particles with 24 warps 16.56 ms, 28 16.42, 32 16.22; thin film 2.61, 2.46,
    // 2.43), 28 for smart Monte Carlo (smc.cu)
    one_per_sm = true;
    s.block = move == 1 ? 896 : 1024;
  }
  const uint64_t walked = N == 1u ? (n_chains + 1u) / 2u : n_chains;   // see paired_singles
  s.chains = s.strip ? strip_chains(walked, s.units, (uint64_t)sm_count, (uint64_t)s.block / 32) : 0u;
  s.n_items = s.strip ? (walked + s.chains - 1) / s.chains : 0u;
  if (s.molecule) {
    s.grid = molecule_grid(n_chains, N, grid_dtype, sm_count);
    return s;
  }
  if (one_per_sm) {
    // over all SMs, however little work there is: 16 cycles of force-biased moves of
    // 65,536 particles (1,024 tiles) 150 us on the 37 SMs that full blocks fill, 136 on all
    const uint64_t work = s.strip ? s.n_items : s.n_tiles;
    s.grid = (int)(work < (uint64_t)sm_count ? work : (uint64_t)sm_count);
    const uint64_t per = (work + (uint64_t)s.grid - 1) / (uint64_t)s.grid;
    const uint64_t warps = (uint64_t)s.block / 32, rounds = (per + warps - 1) / warps;
    if (rounds > 1u && rounds <= EVEN_ROUNDS && 2u * (rounds * warps - per) >= warps)
      s.block = 32 * (int)((per + rounds - 1) / rounds);
    s.chained = true;
    if (s.learned_tc && rounds == 1u) {
      // no more warps than tiles (four to load the fragments): two blocks then fit on
      // an SM, and where they are more than a few warps the next cycle's, set up ahead,
      // would share SMs unevenly with this one's (65,536 particles, 16 cycles: 16 warps
      // 217 us, as many as tiles 198 set up ahead, 178 not; 4,096: 16 warps 140, four 141
      // set up ahead, 149 not)
      s.block = 32 * (int)std::max<uint64_t>(4u, per);
      s.chained = s.block <= 128 || s.block > 256;
    }
    return s;
  }
  const void* fn = s.learned_tc ? learned_tc_kernel_ptr(s.learned_umma)
                                : sweep_kernel_ptr(s, grid_dtype, false);
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, s.block, 0);
  if (per_sm < 1) per_sm = 1;
  const uint64_t warps_per_block = (uint64_t)s.block / 32;
  const uint64_t need = (s.n_tiles + warps_per_block - 1) / warps_per_block;
  const uint64_t cap = (uint64_t)sm_count * (uint64_t)per_sm;
  s.grid = (int)(need < cap ? need : cap);
  if (s.grid < 1) s.grid = 1;
  return s;
}

// Chains of one particle have no bonds (K_b = 0) and no set order to keep: two of them
// walk as one chain of two, which fills a unit; one alone leaves a slot of it empty (2M
// single particles, 16 cycles: 770 and 1017 us one by one, 459 and 589 in pairs, uniform
// and force-biased).  The one left over of an odd number is the even particle of a pair
// whose even ones come first, a unit without its odd one.
static SweepArgs paired_singles(const SweepArgs& a) {
  SweepArgs b = a;
  b.g.N = 2u;
  b.g.N_A = 2u * a.g.N_A;
  b.g.n_chains = (a.g.n_chains + 1u) / 2u;
  b.set_order_random = 0;
  b.strip_order = FULL;
  b.strip_odd = (uint32_t)(a.g.n_chains & 1u);
  return b;
}

cudaError_t launch_sweep_uniform(const SweepArgs& a, const SweepShape& s, int grid_dtype,
                                 int sm_count, cudaStream_t st) {
  size_t smem = 0;
  const void* fn = s.molecule ? molecule_kernel(a.g.n_chains, a.g.N, grid_dtype, sm_count, &smem)
                              : sweep_kernel_ptr(s, grid_dtype, a.seq != nullptr);
  const SweepArgs b = s.strip && a.g.N == 1u ? paired_singles(a) : a;
  void* args[] = {const_cast<SweepArgs*>(&b)};
  return s.chained ? launch_chained(fn, dim3(s.grid), dim3(s.block), args, smem, st)
                   : cudaLaunchKernel(fn, dim3(s.grid), dim3(s.block), args, smem, st);
}

}  // namespace soma
