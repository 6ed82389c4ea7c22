// batch.cu -- many independent SCMF systems advanced by one sweep launch and
// one field launch per cycle.
//
// The paper tunes one parallel region at a time and runs one system per MPI
// rank (Sec. 3.1, 3.2.2).  Here a batch of independent systems (different
// sizes, chain lengths, compositions, chiN, replicas of one seed) shares a
// single persistent launch: the tiles of all systems are cut into work items
// of contiguous tiles of one system; block j takes items j, j + grid, ... and
// its warps take the items' tiles in turn with the same tile body as the
// single-system kernel (pair_body.cuh) and the same draws: a system evolves as
// it does alone, but for a last bit of FP32 fields under K^0
// (fields_batch_kernel).  The host lays the items out either as fixed-length
// items of each system in turn or as one equal contiguous range of the
// concatenated tiles per block, cut at system boundaries (piece r of block j at
// item r * grid + j, padded with empty items).  Launch shape (block size, blocks
// per SM, split) is picked by an autotuner that times the candidates during
// the run.
#include "kernels.h"
#include "pair_body.cuh"

namespace soma {

// A block's warps take the tiles of its items from a shared counter, so that they
// end within a tile of each other.  The constants of the system a warp works on
// (and of the next tile's, when it is another) lie in shared memory, those of the
// cell fold in registers as well: 80 registers without spills at 24 warps an SM.
// With all of them in registers the kernel spilled, and waited for its blocks'
// slowest warps; with none it takes 71 but more loads a tile.  Cycles of 64 systems,
// 40M particles in all, spilled and dealt in turn: 393 us (373 with 16 warps), none in
// registers 381, with 32 warps 377, as here 379; 16 systems of 10.6M in all: 125 (110),
// 106, 105, 105.  One list of tiles for all blocks of an SM through a counter in
// global memory was slower (385, 144): the blocks that share one do not share an SM,
// and their gathers do not repeat in one L1.
template <typename WT>
__global__ void __launch_bounds__(256, 3) sweep_batch_kernel(const BatchArgs p) {
  __shared__ BatchSys s_sys[8][2];
  __shared__ uint32_t s_id[8][2];   // the systems in s_sys
  __shared__ uint32_t s_next;
  const int lane = threadIdx.x & 31;
  const uint32_t warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_next = 0u;
  __syncthreads();
  const unsigned long long s64 = *p.d_sweep;
  const uint32_t sweep = (uint32_t)s64;
  const bool odd = ((s64 + 1ull) & 1ull) != 0;

  // the walk over the block's items: the item of the tile claimed last, the
  // block's tiles up to its end, its first tile less the tiles before it, the
  // slot of its system's constants
  uint32_t item = blockIdx.x - gridDim.x, end = 0, shift = 0, tile = 0;
  int slot = 0;
  if (lane < 2) s_id[warp][lane] = 0xFFFFFFFFu;
  auto claim = [&]() -> bool {
    uint32_t u = 0u;
    if (lane == 0) u = atomicAdd(&s_next, 1u);
    u = __shfl_sync(FULL, u, 0);
    if (u >= end) {
      uint32_t sys;
      do {
        item += gridDim.x;
        if (item >= p.n_items) {
          item -= gridDim.x;
          return false;
        }
        const BatchItem it = p.items[item];
        shift = it.t0 - end;
        end += it.t1 - it.t0;
        sys = it.sys;
      } while (u >= end);
      __syncwarp();
      if (sys != s_id[warp][slot]) {   // the other slot: the tile claimed before has yet to be swept
        slot ^= 1;
        __syncwarp();
        const uint32_t* from = reinterpret_cast<const uint32_t*>(p.sys + sys);
        uint32_t* to = reinterpret_cast<uint32_t*>(&s_sys[warp][slot]);
        for (uint32_t k = lane; k < sizeof(BatchSys) / 4u; k += 32u) to[k] = from[k];
        if (lane == 0) s_id[warp][slot] = sys;
        __syncwarp();
      }
    }
    tile = u + shift;
    return true;
  };
  float2 px = make_float2(0.f, 0.f), py = px, pz = px;
  auto load = [&]() {   // the claimed tile's positions
    const BatchSys& S = s_sys[warp][slot];
    const uint32_t rows = tile < S.full_tiles ? S.G * S.g.N : S.last_rows;
    if (2u * (uint32_t)lane < rows) {
      const uint32_t b0 = tile * (S.G * S.g.N) + 2u * (uint32_t)lane;
      px = __ldcs(reinterpret_cast<const float2*>(S.x + b0));
      py = __ldcs(reinterpret_cast<const float2*>(S.y + b0));
      pz = __ldcs(reinterpret_cast<const float2*>(S.z + b0));
    }
  };
  auto flush = [&](uint32_t k, unsigned n) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(FULL, n, o);
    if (lane == 0 && n) atomicAdd(p.sys[k].counters + 1, (unsigned long long)n);
  };

  PairLane<WT> L;
  Geom g = {};
  float a = 0.f, K_b = 0.f;
  int at = -1;   // the slot of the system L belongs to
  unsigned my_acc = 0;
  bool have = claim();
  if (have) load();
  while (have) {
    const BatchSys& S = s_sys[warp][slot];
    if (slot != at) {
      if (at >= 0) flush(s_id[warp][at], my_acc);
      my_acc = 0;
      at = slot;
      g = S.g;
      a = S.a;
      K_b = S.K_b;
      L.init(lane, S.g.N, S.g.N_A, S.wA, S.wB);
    }
    const uint32_t t = tile;
    const float x0 = px.x, x1 = px.y, y0 = py.x, y1 = py.y, z0 = pz.x, z1 = pz.y;
    have = claim();
    if (have) load();
    uint32_t* nacc = odd ? S.n1 : S.n0;
    __builtin_assume(__isGlobal(nacc));
    const uint32_t ctr3 = (PURPOSE_MOVE << 24) | (g.replica & 0xFFFFFFu);
    const bool full = t < S.full_tiles;
    const uint32_t base = t * L.tile_rows + L.li0;
    if (full && L.tile_rows == 64u)   // no masks needed
      my_acc += pair_tile<WT, uint32_t, false, false>(g, p.keys, L, S.x, S.y, S.z, nacc, base, base,
                                               true, sweep, ctr3, S.set_order_random, a, K_b, x0,
                                               x1, y0, y1, z0, z1);
    else
      my_acc += pair_tile<WT, uint32_t, true, false>(g, p.keys, L, S.x, S.y, S.z, nacc, base, base,
                                              L.in_tile(full, S.last_rows), sweep, ctr3,
                                              S.set_order_random, a, K_b, x0, x1, y0, y1, z0, z1);
  }
  if (at >= 0) flush(s_id[warp][at], my_acc);
}

// Field update of every system: a block takes a contiguous range of the
// concatenated grids, 256 cells at a time; the system of a thread's first cell is
// found by binary search over the grid offsets held in shared memory, that of the
// following ones by stepping on, and a system's constants are read when it
// changes.  The last block to finish advances every system's counter.  A search
// and those reads for every cell, and one thread advancing all the counters in
// turn, made it 26.8 us for 64 systems of 2.1M cells in all, as here 13.8.
template <typename WT>
__global__ void __launch_bounds__(256) fields_batch_kernel(const BatchArgs p, uint32_t total_cells,
                                                           unsigned* arrive, unsigned* err) {
  extern __shared__ uint32_t cell_begin[];  // n_sys + 1 entries
  for (uint32_t k = threadIdx.x; k <= p.n_sys; k += blockDim.x)
    cell_begin[k] = k < p.n_sys ? p.sys[k].cell_begin : total_cells;
  __syncthreads();
  const unsigned long long s = *p.d_sweep;
  const bool rd1 = ((s + 1ull) & 1ull) != 0;
  unsigned bad = 0;
  const uint32_t range = (total_cells + gridDim.x - 1) / gridDim.x;
  const uint32_t begin = min(blockIdx.x * range, total_cells), end = min(begin + range, total_cells);
  uint32_t lo = 0, hi = p.n_sys;  // cell_begin[lo] <= first cell < cell_begin[hi]
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (cell_begin[mid] <= begin + threadIdx.x) lo = mid; else hi = mid;
  }
  uint32_t first = 0, next = 0;   // the cells of system lo; next 0: not read yet
  const uint32_t* nr = nullptr;
  uint32_t* nc = nullptr;
  WT* wA = nullptr;
  WT* wB = nullptr;
  float inv_rho = 0.f, kappa0 = 0.f, half_chi0 = 0.f;
  int ham = 0;
  for (uint32_t c = begin + threadIdx.x; c < end; c += blockDim.x) {
    if (c >= next) {
      while (lo + 1 < p.n_sys && cell_begin[lo + 1] <= c) ++lo;
      const BatchSys* S = p.sys + lo;
      first = cell_begin[lo];
      next = cell_begin[lo + 1];
      nr = rd1 ? S->n1 : S->n0;
      nc = rd1 ? S->n0 : S->n1;
      wA = static_cast<WT*>(const_cast<void*>(S->wA));
      wB = static_cast<WT*>(const_cast<void*>(S->wB));
      inv_rho = S->inv_rho;
      kappa0 = S->kappa0;
      half_chi0 = S->half_chi0;
      ham = S->hamiltonian;
    }
    const uint32_t local = c - first;
    const uint32_t v = nr[local];
    nc[local] = 0u;
    const uint32_t a = v & 0xFFFFu, b = v >> 16;
    // with its roundings written out; under K^0 they are not omega_of's (omega.cuh), and
    // FP32 fields differ from its by an ulp in about half of the cells: the batch's own
    // trajectories, kept as they are
    const float phiA = __fmul_rn((float)a, inv_rho), phiB = __fmul_rn((float)b, inv_rho);
    const float comp = __fmul_rn(kappa0, __fsub_rn(__fadd_rn(phiA, phiB), 1.f));
    float wa, wb;
    if (ham) {
      const float chi0 = __fmul_rn(2.f, half_chi0);
      wa = __fmaf_rn(chi0, phiB, comp);
      wb = __fmaf_rn(chi0, phiA, comp);
    } else {
      const float d = __fsub_rn(phiA, phiB);
      wa = __fmaf_rn(-half_chi0, d, comp);
      wb = __fmaf_rn(half_chi0, d, comp);
    }
    wA[local] = store_cvt<WT>(wa);
    wB[local] = store_cvt<WT>(wb);
    bad |= (a >= 0xC000u) | (b >= 0xC000u);
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(err, ERR_OVERFLOW);
  __shared__ bool s_last;
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(arrive, 1u) == gridDim.x - 1;
    if (s_last) *arrive = 0u;
  }
  __syncthreads();
  if (s_last)
    for (uint32_t k = threadIdx.x; k < p.n_sys; k += blockDim.x) p.sys[k].counters[0] = s + 1ull;
}

cudaError_t launch_sweep_batch(const BatchArgs& a, int grid, int block, int grid_dtype,
                               cudaStream_t st) {
  switch (grid_dtype) {
    case 1: sweep_batch_kernel<__nv_bfloat16><<<grid, block, 0, st>>>(a); break;
    case 2: sweep_batch_kernel<__half><<<grid, block, 0, st>>>(a); break;
    default: sweep_batch_kernel<float><<<grid, block, 0, st>>>(a); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_fields_batch(const BatchArgs& a, uint32_t total_cells, unsigned* arrive,
                                unsigned* err, int grid_dtype, int sm_count, cudaStream_t st) {
  uint64_t blocks = ((uint64_t)total_cells + 255) / 256;
  const uint64_t cap = (uint64_t)sm_count * 8;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  const size_t sh = sizeof(uint32_t) * (a.n_sys + 1);
  switch (grid_dtype) {
    case 1: fields_batch_kernel<__nv_bfloat16><<<(unsigned)blocks, 256, sh, st>>>(a, total_cells, arrive, err); break;
    case 2: fields_batch_kernel<__half><<<(unsigned)blocks, 256, sh, st>>>(a, total_cells, arrive, err); break;
    default: fields_batch_kernel<float><<<(unsigned)blocks, 256, sh, st>>>(a, total_cells, arrive, err); break;
  }
  return cudaGetLastError();
}

int batch_kernel_blocks_per_sm(int block, int grid_dtype) {
  const void* fn = grid_dtype == 1 ? (const void*)sweep_batch_kernel<__nv_bfloat16>
                 : grid_dtype == 2 ? (const void*)sweep_batch_kernel<__half>
                                   : (const void*)sweep_batch_kernel<float>;
  cudaFuncAttributes attr;
  if (cudaFuncGetAttributes(&attr, fn) != cudaSuccess || block > attr.maxThreadsPerBlock) return 0;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, block, 0) != cudaSuccess) return 0;
  return n;
}

}  // namespace soma
