// resident.cu -- many SCMF cycles of a small system in one launch (uniform
// moves, even N <= 64): the pair tiles of pair_body.cuh on all SMs, the blocks
// meeting once per cycle at a grid barrier.
//
// At a few thousand to a few hundred thousand particles a cycle is a few
// microseconds of dependent latency, and the two launches of the sweep and the
// field update cost as much again.  Here the fields are not stored between
// cycles at all: a move gathers the packed counts of its cell and evaluates
// omega itself (omega.cuh, the bits of the field kernel), so a cycle needs one
// meeting of the blocks instead of two kernel boundaries.  The counts take
// three buffers in turn (read; counted into; cleared for the cycle after), and
// a warp's first tile keeps its positions in registers.  The last cycle is
// followed by the field update and leaves the buffers as the two-kernel cycle
// does (n[s&1] current, the other cleared, the third cleared).  Per cycle, against
// the two kernels under a CUDA graph: 4,096 particles 6.6 -> 3.4 us, 32,768 7.1 ->
// 4.2, 262,144 9.5 -> 7.1, 393,216 11.9 -> 8.7, 589,824 11.9 -> 11.0.
//
// Systems of at most one tile per warp of one cluster of 16 blocks
// (resident_cluster_kernel) never leave the chip between cycles: positions stay
// in registers, every block holds the counts in shared memory and adds its own
// moves to a second copy there, and the blocks sum the 16 copies, a slice of the
// cells each, through distributed shared memory.  Gathers and counts are then
// shared-memory accesses and the two meetings of a cycle hardware cluster
// barriers: 4,096 particles 3.4 -> 2.1 us a cycle, 13,664 3.9 -> 2.9.
//
// The planes w are written, not read: a handle whose planes do not follow from the
// counts with its external fields and density as they are (they were changed since
// the last field update) runs a cycle of the two kernels first.
//
// The larger launch is cooperative (the blocks wait on one another, so all must be
// resident: one block per SM at most).  A wait gives up after 2^26 polls, sets
// the sticky timeout bit and ends the kernel.
#include "kernels.h"
#include "omega.cuh"
#include "pair_body.cuh"

namespace soma {

namespace {

constexpr uint32_t BARRIER_POLLS = 1u << 26;

// Lane of a pair tile whose field values come from the counts of the cycle.
template <typename WT>
struct CountLane : PairLane<WT> {
  const uint32_t* n;
  const FieldArgs* f;
  __device__ __forceinline__ float field0(uint32_t c) const {
    return omega_stored<WT>(*f, n[c], c, this->v0 != 1u);
  }
  __device__ __forceinline__ float field1(uint32_t c) const {
    return omega_stored<WT>(*f, n[c], c, this->v1 != 1u);
  }
};

// All blocks' writes and atomics before the k-th barrier are visible after it:
// thread 0 releases its block's (ordered before it by the block barrier) and
// acquires the others' (the SM's stale L1 lines are dropped with that).  False
// when the wait gave up.
__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned target, bool* s_ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" :: "l"(bar) : "memory");
    bool ok = false;
    for (uint32_t it = 0; it < BARRIER_POLLS && !ok; ++it) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      ok = (int)(v - target) >= 0;
    }
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok;
}

template <typename WT, bool MIXED>
__global__ void __launch_bounds__(1024, 1) resident_pair_kernel(const __grid_constant__ ResidentArgs r) {
  __shared__ bool s_ok;
  const SweepArgs& p = r.s;
  const int lane = threadIdx.x & 31;
  const uint32_t wib = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t n_tiles = (uint32_t)p.n_tiles;
  const uint32_t chunk = (n_tiles + gridDim.x - 1) / gridDim.x;
  const uint32_t t_end = min(blockIdx.x * chunk + chunk, n_tiles);
  const uint32_t t_first = blockIdx.x * chunk + wib;
  const unsigned long long s64 = *p.d_sweep;
  const uint32_t ctr3 = (PURPOSE_MOVE << 24) | (p.g.replica & 0xFFFFFFu);
  CountLane<WT> L;
  L.init(lane, p.g.N, p.g.N_A, nullptr, nullptr);
  L.f = &r.f;
  const uint32_t TN = p.G * p.g.N, full_tiles = (uint32_t)p.full_tiles, cells = p.g.cells;
  const uint32_t gtid = blockIdx.x * blockDim.x + threadIdx.x, gthreads = gridDim.x * blockDim.x;
  uint32_t* cur = (s64 & 1ull) ? p.n1 : p.n0;     // counts the fields come from
  uint32_t* nxt = (s64 & 1ull) ? p.n0 : p.n1;     // counted into (cleared)
  uint32_t* old = r.n2;                           // cleared during this cycle

  auto load = [&](uint32_t t, PairEnd& e) {
    if (t < t_end && L.in_tile(t < full_tiles, p.last_rows)) {
      const uint32_t b = t * TN + L.li0;
      e.x = __ldcs(reinterpret_cast<const float2*>(p.x + b));
      e.y = __ldcs(reinterpret_cast<const float2*>(p.y + b));
      e.z = __ldcs(reinterpret_cast<const float2*>(p.z + b));
    }
  };
  PairEnd first;
  first.x = first.y = first.z = make_float2(0.f, 0.f);
  load(t_first, first);
  unsigned my_acc = 0, bad = 0;
  unsigned target = 0;
  bool ok = true;
  for (uint32_t j = 0; j < r.cycles && ok; ++j) {
    const uint32_t sweep = (uint32_t)(s64 + j);
    const bool last = j + 1u == r.cycles;
    L.n = cur;
    // the first of the counts to clear (all of them on a small grid), loaded
    // before the moves so that its latency passes with theirs
    const uint32_t v0 = gtid < cells ? old[gtid] : 0u;
    PairEnd pos = first;
    for (uint32_t t = t_first; t < t_end; t += nw) {
      PairEnd next = pos, end;
      load(t + nw, next);
      const bool valid = L.in_tile(t < full_tiles, p.last_rows);
      if (MIXED) {
        const uint64_t chain = (uint64_t)t * p.G + L.lane_chain;
        const uint64_t seq = chain < p.g.n_chains ? __ldg(p.seq + __ldg(p.arch + chain)) : 0ull;
        L.set_types((seq >> L.ci0) & 1ull, (seq >> (L.ci0 + 1u)) & 1ull, nullptr, nullptr);
      }
      const uint32_t base = t * TN + L.li0;
      PairState P;
      pair_prepare<CountLane<WT>, uint32_t, false>(p.g, p.g, L, base, valid, sweep, ctr3, p.a, pos.x.x,
                                                   pos.x.y, pos.y.x, pos.y.y, pos.z.x, pos.z.y, P);
      end.store = last || t != t_first;
      my_acc += pair_finish<CountLane<WT>, uint32_t, true>(L, p.x, p.y, p.z, nxt, base, P,
                                                           p.set_order_random, p.K_b, &end);
      if (t == t_first) first = end;
      pos = next;
    }
    // the counts the previous cycle's fields came from: checked and cleared
    for (uint32_t c = gtid; c < cells; c += gthreads) {
      const uint32_t v = c == gtid ? v0 : old[c];
      bad |= ((v & 0xFFFFu) >= 0xC000u) | ((v >> 16) >= 0xC000u);
      old[c] = 0u;
    }
    target += gridDim.x;
    ok = grid_barrier(r.bar, target, &s_ok);
    uint32_t* const was = cur;
    cur = nxt;
    nxt = old;
    old = was;
  }
  // the field update of the last counts, and the buffers in their places
  const unsigned long long s1 = s64 + r.cycles;
  uint32_t* const out = (s1 & 1ull) ? p.n1 : p.n0;
  uint32_t* const oth = (s1 & 1ull) ? p.n0 : p.n1;
  WT* __restrict__ wA = static_cast<WT*>(r.f.wA);
  WT* __restrict__ wB = static_cast<WT*>(r.f.wB);
  if (ok) {
    for (uint32_t c = gtid; c < cells; c += gthreads) {
      const uint32_t v = cur[c], u = old[c];
      bad |= ((v & 0xFFFFu) >= 0xC000u) | ((v >> 16) >= 0xC000u) | ((u & 0xFFFFu) >= 0xC000u) |
             ((u >> 16) >= 0xC000u);
      out[c] = v;
      oth[c] = 0u;
      r.n2[c] = 0u;
      wA[c] = store_cvt<WT>(omega_stored<WT>(r.f, v, c, false));
      wB[c] = store_cvt<WT>(omega_stored<WT>(r.f, v, c, true));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) my_acc += __shfl_xor_sync(FULL, my_acc, o);
  if (lane == 0 && my_acc) atomicAdd(p.acc, (unsigned long long)my_acc);
  bad = __syncthreads_or(bad);
  if (threadIdx.x == 0) {
    if (bad) atomicOr(p.err, ERR_OVERFLOW);
    if (!ok) atomicOr(p.err, ERR_TIMEOUT);
    __threadfence();
    // the last block to end resets the barrier and advances the sweep counter
    if (atomicAdd(r.arrive, 1u) == gridDim.x - 1u) {
      *r.arrive = 0u;
      *r.bar = 0u;
      *r.f.d_sweep = s1;
    }
  }
}

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// address of a shared-memory word of this block in block `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_address(const uint32_t* p, uint32_t rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;"
      : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}

// One warp per tile.  Shared memory: the current counts, and this block's counts
// of the next cycle in two buffers by the cycle's parity (the other one is
// cleared while the first is summed).
template <typename WT, bool MIXED>
__global__ void __launch_bounds__(32 * CLUSTER_WARPS, 1)
    resident_cluster_kernel(const __grid_constant__ ResidentArgs r) {
  extern __shared__ uint32_t counts[];
  const SweepArgs& p = r.s;
  const int lane = threadIdx.x & 31;
  const uint32_t n_tiles = (uint32_t)p.n_tiles, cells = p.g.cells, blocks = gridDim.x, rank = blockIdx.x;
  const uint32_t t = (threadIdx.x >> 5) * blocks + rank;   // this warp's tile
  const unsigned long long s64 = *p.d_sweep, s1 = s64 + r.cycles;
  const uint32_t ctr3 = (PURPOSE_MOVE << 24) | (p.g.replica & 0xFFFFFFu);
  uint32_t* const cur = counts;
  uint32_t* const out = (s1 & 1ull) ? p.n1 : p.n0;
  uint32_t* const oth = (s1 & 1ull) ? p.n0 : p.n1;
  const uint32_t* const in = (s64 & 1ull) ? p.n1 : p.n0;
  CountLane<WT> L;
  L.init(lane, p.g.N, p.g.N_A, nullptr, nullptr);
  L.f = &r.f;
  L.n = cur;
  const uint32_t base = t * p.G * p.g.N + L.li0;
  const bool valid = t < n_tiles && L.in_tile(t < (uint32_t)p.full_tiles, p.last_rows);
  PairEnd pos;
  pos.x = pos.y = pos.z = make_float2(0.f, 0.f);
  pos.store = false;
  if (valid) {
    pos.x = __ldcs(reinterpret_cast<const float2*>(p.x + base));
    pos.y = __ldcs(reinterpret_cast<const float2*>(p.y + base));
    pos.z = __ldcs(reinterpret_cast<const float2*>(p.z + base));
  }
  if (MIXED) {
    const uint64_t chain = (uint64_t)t * p.G + L.lane_chain;
    const uint64_t seq = chain < p.g.n_chains ? __ldg(p.seq + __ldg(p.arch + chain)) : 0ull;
    L.set_types((seq >> L.ci0) & 1ull, (seq >> (L.ci0 + 1u)) & 1ull, nullptr, nullptr);
  }
  for (uint32_t c = threadIdx.x; c < cells; c += blockDim.x) {
    cur[c] = in[c];
    counts[cells + c] = 0u;
    counts[2u * cells + c] = 0u;
  }
  // this block's slice of the cells
  const uint32_t slice = (cells + blocks - 1u) / blocks;
  const uint32_t c0 = min(rank * slice, cells), c1 = min(c0 + slice, cells);
  unsigned my_acc = 0, bad = 0;
  cluster_barrier();   // every block's memory is set up, and every block has read its input
  for (uint32_t j = 0; j < r.cycles; ++j) {
    uint32_t* const mine = counts + (1u + (j & 1u)) * cells;
    uint32_t* const next = counts + (2u - (j & 1u)) * cells;
    if (t < n_tiles) {
      PairState P;
      pair_prepare<CountLane<WT>, uint32_t, false>(p.g, p.g, L, base, valid, (uint32_t)(s64 + j), ctr3,
                                                   p.a, pos.x.x, pos.x.y, pos.y.x, pos.y.y, pos.z.x,
                                                   pos.z.y, P);
      my_acc += pair_finish<CountLane<WT>, uint32_t, true>(L, p.x, p.y, p.z, mine, base, P,
                                                           p.set_order_random, p.K_b, &pos);
    }
    cluster_barrier();   // the moves of all blocks are counted
    for (uint32_t c = c0 + threadIdx.x; c < c1; c += blockDim.x) {
      uint32_t v = 0u;
#pragma unroll 8
      for (uint32_t k = 0; k < blocks; ++k) {
        uint32_t u;
        asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(u) : "r"(cluster_address(mine + c, k)));
        v += u;
      }
      bad |= ((v & 0xFFFFu) >= 0xC000u) | ((v >> 16) >= 0xC000u);
#pragma unroll 8
      for (uint32_t k = 0; k < blocks; ++k)
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_address(cur + c, k)), "r"(v) : "memory");
    }
    for (uint32_t c = threadIdx.x; c < cells; c += blockDim.x) next[c] = 0u;
    cluster_barrier();   // the counts of the next cycle are everywhere
  }
  if (valid) {
    __stcs(reinterpret_cast<float2*>(p.x + base), pos.x);
    __stcs(reinterpret_cast<float2*>(p.y + base), pos.y);
    __stcs(reinterpret_cast<float2*>(p.z + base), pos.z);
  }
  WT* __restrict__ wA = static_cast<WT*>(r.f.wA);
  WT* __restrict__ wB = static_cast<WT*>(r.f.wB);
  for (uint32_t c = c0 + threadIdx.x; c < c1; c += blockDim.x) {
    const uint32_t v = cur[c];
    out[c] = v;
    oth[c] = 0u;
    wA[c] = store_cvt<WT>(omega_stored<WT>(r.f, v, c, false));
    wB[c] = store_cvt<WT>(omega_stored<WT>(r.f, v, c, true));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) my_acc += __shfl_xor_sync(FULL, my_acc, o);
  if (lane == 0 && my_acc) atomicAdd(p.acc, (unsigned long long)my_acc);
  bad = __syncthreads_or(bad);
  if (threadIdx.x == 0) {
    if (bad) atomicOr(p.err, ERR_OVERFLOW);
    if (rank == 0u) *r.f.d_sweep = s1;   // read by every block before the first barrier
  }
}

const void* cluster_ptr(int grid_dtype, bool mixed) {
  switch (grid_dtype) {
    case 1: return mixed ? (const void*)resident_cluster_kernel<__nv_bfloat16, true>
                         : (const void*)resident_cluster_kernel<__nv_bfloat16, false>;
    case 2: return mixed ? (const void*)resident_cluster_kernel<__half, true>
                         : (const void*)resident_cluster_kernel<__half, false>;
    default: return mixed ? (const void*)resident_cluster_kernel<float, true>
                          : (const void*)resident_cluster_kernel<float, false>;
  }
}

// Launch configuration of the cluster kernel (attr: one attribute).
void cluster_config(cudaLaunchConfig_t& c, cudaLaunchAttribute* attr, int grid, int block, size_t smem,
                    cudaStream_t st) {
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = (unsigned)grid;
  attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
  c = {};
  c.gridDim = dim3((unsigned)grid);
  c.blockDim = dim3((unsigned)block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = attr;
  c.numAttrs = 1;
}

const void* resident_ptr(int grid_dtype, bool mixed) {
  switch (grid_dtype) {
    case 1: return mixed ? (const void*)resident_pair_kernel<__nv_bfloat16, true>
                         : (const void*)resident_pair_kernel<__nv_bfloat16, false>;
    case 2: return mixed ? (const void*)resident_pair_kernel<__half, true>
                         : (const void*)resident_pair_kernel<__half, false>;
    default: return mixed ? (const void*)resident_pair_kernel<float, true>
                          : (const void*)resident_pair_kernel<float, false>;
  }
}

}  // namespace

// Whether the cluster kernel can take a system of these tiles and cells here (both
// of its variants are then allowed their shared memory and cluster size).
static bool cluster_shape(uint64_t n_tiles, uint32_t cells, int grid_dtype, ResidentShape* r) {
  const int warps = (int)((n_tiles + CLUSTER_BLOCKS - 1) / CLUSTER_BLOCKS);
  const size_t smem = sizeof(uint32_t) * 3 * (size_t)cells;
  if (warps > CLUSTER_WARPS || cells > CLUSTER_CELLS) return false;
  for (int mixed = 0; mixed < 2; ++mixed) {
    const void* fn = cluster_ptr(grid_dtype, mixed != 0);
    cudaLaunchConfig_t c;
    cudaLaunchAttribute a;
    cluster_config(c, &a, CLUSTER_BLOCKS, 32 * warps, smem, nullptr);
    int n = 0;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(sizeof(uint32_t) * 3 * CLUSTER_CELLS)) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, fn, &c) != cudaSuccess || n < 1) {
      (void)cudaGetLastError();
      return false;
    }
  }
  *r = ResidentShape{CLUSTER_BLOCKS, 32 * warps, smem, 2};
  return true;
}

ResidentShape resident_shape(const SweepShape& s, uint32_t cells, int grid_dtype, int sm_count) {
  ResidentShape r{0, 0, 0, 0};
  int dev = 0, coop = 0;
  if (s.move != 0 || !s.pair || s.strip || s.big || s.molecule) return r;
  if (s.n_tiles > (uint64_t)sm_count * RESIDENT_TILES_PER_SM) return r;
  if (cluster_shape(s.n_tiles, cells, grid_dtype, &r)) return r;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop)
    return r;
  // one block per SM; its warps take its tiles in equal rounds of at most 32
  r.grid = (int)(s.n_tiles < (uint64_t)sm_count ? s.n_tiles : (uint64_t)sm_count);
  const uint64_t per = (s.n_tiles + (uint64_t)r.grid - 1) / (uint64_t)r.grid;
  const uint64_t rounds = (per + 31) / 32;
  r.block = 32 * (int)((per + rounds - 1) / rounds);
  r.min_cycles = 2u + (uint32_t)(s.n_tiles / (RESIDENT_TILES_PER_CYCLE * (uint64_t)sm_count));
  return r;
}

cudaError_t launch_resident(const ResidentArgs& a, const ResidentShape& s, int grid_dtype,
                            cudaStream_t st) {
  void* args[] = {const_cast<ResidentArgs*>(&a)};
  if (s.cluster_smem) {
    cudaLaunchConfig_t c;
    cudaLaunchAttribute attr;
    cluster_config(c, &attr, s.grid, s.block, s.cluster_smem, st);
    return cudaLaunchKernelExC(&c, cluster_ptr(grid_dtype, a.s.seq != nullptr), args);
  }
  return cudaLaunchCooperativeKernel(resident_ptr(grid_dtype, a.s.seq != nullptr), dim3(s.grid),
                                     dim3(s.block), args, 0, st);
}

}  // namespace soma
