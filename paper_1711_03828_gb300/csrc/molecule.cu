// molecule.cu -- the molecule-parallel iteration (Sec. 3.1.2, first scheme).
//
// The chain's N attempts of one MC step run one after another, each on a
// particle of the chain chosen at random, so every particle is attempted once
// per step on average and a move always sees the current positions of its
// bonded partners.  Attempt j of chain k draws Philox purpose 3 with id k*N + j:
// words 0-2 give the uniform displacement, the top 24 bits of word 3 the
// acceptance uniform and its low byte the particle, ((word3 & 0xFF) * N) >> 8.
// Molecules of any architecture (the architecture array of Sec. 3.2.1,
// re-encoded per particle as for the SET kernel of topology.cu) take the same
// body with their bond partners and types from the per-particle table words.
//
// One, two or four lanes per chain (molecule_lanes) make as many consecutive
// attempts at a time.  Their draws,
// trial positions, cells and field gathers do not depend on one another and
// run in parallel; the decisions then follow in rounds, an attempt waiting
// only for the earlier ones of its group that chose the same particle or one of
// its bonded partners (most chose none: the moves of others commute with it),
// and gathering again when an accepted one moved its own particle.  The result
// is that of the attempts in turn, bit for bit.  A warp stages its chains
// in shared memory (coalesced in and out) and counts the final cells while
// writing them back.  With one thread per chain the attempts of a chain were one
// chain of dependent latencies (draw, gather, decide) and a system had only as
// many threads as chains; chains of more than 64 were walked in global memory
// (16.8M particles of N = 100: 1321 us a cycle, 326 now).
#include "kernels.h"

namespace soma {

constexpr uint32_t PURPOSE_ATTEMPT = 3;
constexpr uint32_t MOL_WARPS = MOL_BLOCK / 32;

// Table word of the architecture path (see topology.cu): bits 0-5 number of
// partners, 6-23 the first three partners, bit 24 type.
__device__ __forceinline__ uint32_t mol_partner(uint32_t w, int k) { return (w >> (6 + 6 * k)) & 63u; }

// TOPO: molecules of any architecture (t holds the tables); else linear chains
// (the diblock, or a mixture through p.seq / p.arch).
// MULTI (with TOPO): n_t particle types, the type from the type table, one
// FP32 field plane and one count plane per type.
// MOL_LANES: attempts of a chain at a time (1, 2 or 4 lanes per chain).
template <typename WT, uint32_t MOL_LANES, bool TOPO, bool MULTI = false>
__device__ __forceinline__ void molecule_body(const SweepArgs& p, const TopoArgs& tp) {
  constexpr uint32_t MOL_CHAINS = 32u / MOL_LANES;   // chains of a warp
  // The next draws during this attempt's gathers: not for the two types' one lane per
  // molecule, whose longer partner loop has no registers left for them (16.8M particles of
  // stars, combs, rings and diblocks, 16 cycles: 4.39 ms, in turn 4.20; with the
  // waiting rounds below and the partner mask loaded for every attempt 4.84).
  constexpr bool AHEAD = !TOPO || MULTI || MOL_LANES > 1u;
  extern __shared__ float sm[];
  const uint32_t N = p.g.N, N_A = p.g.N_A;
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  const uint32_t c = lane / MOL_LANES, q = lane % MOL_LANES;
  const uint32_t group0 = lane & ~(MOL_LANES - 1u);   // first lane of this chain
  float* const sx = sm + (size_t)wib * 3 * MOL_CHAINS * N;
  float* const sy = sx + MOL_CHAINS * N;
  float* const sz = sy + MOL_CHAINS * N;
  const unsigned long long s64 = *p.d_sweep;
  const uint32_t sweep = (uint32_t)s64;
  uint32_t* __restrict__ nacc = MULTI ? (((s64 + 1ull) & 1ull) ? tp.nt1 : tp.nt0)
                                      : (((s64 + 1ull) & 1ull) ? p.n1 : p.n0);
  const uint32_t ctr3 = (PURPOSE_ATTEMPT << 24) | (p.g.replica & 0xFFFFFFu);
  const WT* __restrict__ wA = static_cast<const WT*>(p.wA);
  const WT* __restrict__ wB = static_cast<const WT*>(p.wB);
  const float a = p.a, K1 = p.K_b, K2 = 2.f * p.K_b;
  const uint64_t n_groups = (p.g.n_chains + MOL_CHAINS - 1) / MOL_CHAINS;
  const uint64_t stride = (uint64_t)gridDim.x * MOL_WARPS;
  unsigned my_acc = 0;
  for (uint64_t gr = (uint64_t)blockIdx.x * MOL_WARPS + wib; gr < n_groups; gr += stride) {
    const uint64_t chain0 = gr * MOL_CHAINS;
    const uint64_t rem = p.g.n_chains - chain0;
    const uint32_t nch = rem < (uint64_t)MOL_CHAINS ? (uint32_t)rem : MOL_CHAINS;
    const uint32_t cnt = nch * N;       // particles of this warp's chains
    const uint64_t m0 = chain0 * N;
    for (uint32_t k = lane; k < cnt; k += 32u) {
      sx[k] = __ldcs(p.x + m0 + k);
      sy[k] = __ldcs(p.y + m0 + k);
      sz[k] = __ldcs(p.z + m0 + k);
    }
    __syncwarp();
    const bool in = c < nch;
    const uint64_t chain = chain0 + (in ? c : 0u);
    // type sequence of this chain (bit i set: particle i is B)
    const uint64_t seq = !TOPO && p.seq ? __ldg(p.seq + __ldg(p.arch + chain)) : 0ull;
    const uint32_t arch64 = TOPO ? (uint32_t)__ldg(tp.mol_arch + chain) * 64u : 0u;
    // particles of the molecule: its architecture's (the slots past them are
    // absent), else N; it makes that many attempts on its own particles
    const uint32_t len = TOPO ? (uint32_t)__ldg(tp.alen + arch64 / 64u) : N;
    const uint32_t rounds = __reduce_max_sync(FULL, in ? (len + MOL_LANES - 1u) / MOL_LANES : 0u);
    float* const X = sx + (in ? c : 0u) * N;
    float* const Y = sy + (in ? c : 0u) * N;
    float* const Z = sz + (in ? c : 0u) * N;
    const uint64_t id0 = chain * N + p.g.id_base;
    uint64_t id = id0 + q;
    uint4 rnext = make_uint4(0u, 0u, 0u, 0u);
    if (AHEAD) rnext = philox_rk(make_uint4((uint32_t)id, (uint32_t)(id >> 32), sweep, ctr3), p.g);
    for (uint32_t b = 0; b < rounds; ++b) {
      const uint32_t j = b * MOL_LANES + q;
      uint4 r = rnext;
      if (!AHEAD) {
        id = id0 + j;
        r = philox_rk(make_uint4((uint32_t)id, (uint32_t)(id >> 32), sweep, ctr3), p.g);
      }
      bool pending = in && j < len;
      const uint32_t i = ((r.w & 0xFFu) * len) >> 8;
      const uint32_t pw = TOPO ? __ldg(tp.ptab + arch64 + i) : 0u;
      const float vx = uniform_sym(r.x), vy = uniform_sym(r.y), vz = uniform_sym(r.z);
      float xo, yo, zo, xn, yn, zn, wn, wo;
      const WT* w;
      if (MULTI) {
        w = reinterpret_cast<const WT*>(tp.wt + (size_t)__ldg(tp.ttab + arch64 + i) * p.g.cells);
      } else {
        const bool isB = TOPO ? ((pw >> 24) & 1u) != 0
                              : (p.seq ? ((seq >> i) & 1ull) != 0 : i >= N_A);
        w = isB ? wB : wA;
      }
      // trial position and the field values of particle i at its place
      auto gather = [&]() {
        xo = X[i];
        yo = Y[i];
        zo = Z[i];
        xn = __fmaf_rn(a, vx, xo);
        yn = __fmaf_rn(a, vy, yo);
        zn = __fmaf_rn(a, vz, zo);
        wn = load_w<WT>(w, cell_of(p.g, xn, yn, zn));
        wo = load_w<WT>(w, cell_of(p.g, xo, yo, zo));
      };
      gather();
      // the next draws (independent of the outcomes) during the gathers
      if (AHEAD) {
        id = id0 + j + MOL_LANES;
        rnext = philox_rk(make_uint4((uint32_t)id, (uint32_t)(id >> 32), sweep, ctr3), p.g);
      }
      const uint64_t nb = TOPO && MOL_LANES > 1u ? __ldg(tp.pmask + arch64 + i) : 0ull;
      // the decision of an attempt whose partners are where they should be; true: moved
      auto decide = [&]() -> bool {
        // U = sum over bonded partners of (r - n), k partners
        float ux = 0.f, uy = 0.f, uz = 0.f, k = 0.f;
        if (TOPO) {
          const uint32_t deg = pw & 63u;
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            if ((uint32_t)e < deg) {
              const uint32_t n = mol_partner(pw, e);
              ux += xo - X[n];
              uy += yo - Y[n];
              uz += zo - Z[n];
            }
          }
          if (deg > 3u) {   // the partners after the third, from the full mask
            uint64_t mk = MOL_LANES > 1u ? nb : __ldg(tp.pmask + arch64 + i);
            mk &= mk - 1ull;
            mk &= mk - 1ull;
            mk &= mk - 1ull;
            for (; mk; mk &= mk - 1ull) {
              const uint32_t n = (uint32_t)__ffsll((long long)mk) - 1u;
              ux += xo - X[n];
              uy += yo - Y[n];
              uz += zo - Z[n];
            }
          }
          k = (float)deg;
        } else {
          if (i > 0) { ux += xo - X[i - 1]; uy += yo - Y[i - 1]; uz += zo - Z[i - 1]; k += 1.f; }
          if (i + 1 < N) { ux += xo - X[i + 1]; uy += yo - Y[i + 1]; uz += zo - Z[i + 1]; k += 1.f; }
        }
        const float dEf = wn - wo;
        const float dx = xn - xo, dy = yn - yo, dz = zn - zo;
        const float du = fmaf(dx, ux, fmaf(dy, uy, dz * uz));
        const float dd = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        const float dE = fmaf(k * K1, dd, fmaf(K2, du, dEf));
        if (!(dE <= -log_uniform_open(r.w))) return false;
        X[i] = xn;
        Y[i] = yn;
        Z[i] = zn;
        ++my_acc;
        return true;
      };
      if (MOL_LANES == 1u) {   // no other attempt to wait for
        if (pending) decide();
        continue;
      }
      // earlier attempts of the group on this particle (same) or on it or a
      // bonded partner (dep), as bits of their lanes in the group
      uint32_t dep = 0u, same = 0u;
#pragma unroll
      for (uint32_t s = 0; s + 1u < MOL_LANES; ++s) {
        const uint32_t is = __shfl_sync(FULL, i, (int)(group0 + s));
        if (s < q) {
          const bool eq = is == i;
          const bool bonded = TOPO ? ((nb >> is) & 1ull) != 0 : is + 1u == i || i + 1u == is;
          same |= (uint32_t)eq << s;
          dep |= (uint32_t)(eq || bonded) << s;
        }
      }
      uint32_t left = __ballot_sync(FULL, pending);
      while (left) {
        bool acc = false;
        if (pending && !(dep & (left >> group0))) {
          acc = decide();
          pending = false;
        }
        __syncwarp();
        const uint32_t moved = __ballot_sync(FULL, acc) >> group0;
        left = __ballot_sync(FULL, pending);
        if (pending && (same & moved)) gather();   // its own particle has moved
      }
      __syncwarp();
    }
    __syncwarp();
    // write back and count the final cells
    uint32_t ci = lane % N;
    const uint32_t step = 32u % N;
    for (uint32_t k = lane; k < cnt; k += 32u) {
      const float x = sx[k], y = sy[k], z = sz[k];
      __stcs(p.x + m0 + k, x);
      __stcs(p.y + m0 + k, y);
      __stcs(p.z + m0 + k, z);
      if (TOPO) {
        const uint32_t am = (uint32_t)__ldg(tp.mol_arch + chain0 + k / N);
        if (ci < (uint32_t)__ldg(tp.alen + am)) {   // else an absent slot: not counted
          if (MULTI)
            atomicAdd(nacc + (size_t)__ldg(tp.ttab + am * 64u + ci) * p.g.cells + cell_of(p.g, x, y, z), 1u);
          else
            atomicAdd(nacc + cell_of(p.g, x, y, z),
                      ((__ldg(tp.ptab + am * 64u + ci) >> 24) & 1u) ? 0x10000u : 1u);
        }
      } else {
        const bool isB = p.seq ? ((__ldg(p.seq + __ldg(p.arch + chain0 + k / N)) >> ci) & 1ull) != 0
                               : ci >= N_A;
        atomicAdd(nacc + cell_of(p.g, x, y, z), isB ? 0x10000u : 1u);
      }
      ci += step;
      if (ci >= N) ci -= N;
    }
    __syncwarp();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) my_acc += __shfl_xor_sync(FULL, my_acc, o);
  if (lane == 0 && my_acc) atomicAdd(p.acc, (unsigned long long)my_acc);
}

template <typename WT, uint32_t LANES>
__global__ void __launch_bounds__(MOL_BLOCK, 8) sweep_molecule_kernel(const SweepArgs p) {
  molecule_body<WT, LANES, false>(p, TopoArgs{});
}

// One lane per molecule of n_t types: more than 64 registers, at which three types (16.8M
// particles, 16 cycles) take 4.48 ms instead of 4.38.
template <typename WT, uint32_t LANES, bool MULTI>
__global__ void __launch_bounds__(MOL_BLOCK, MULTI && LANES == 1u ? 4 : 8)
    sweep_molecule_topology_kernel(const TopoArgs t) {
  molecule_body<WT, LANES, true, MULTI>(t.s, t);
}

// Lanes per chain.  Four where the chains would give each SM fewer than four
// warps at one lane each (the attempts' latencies, not the instructions, are the
// time); two for long chains, whose staging leaves few warps on an SM at one lane
// each; else one.  us a cycle with 1 / 2 / 4 lanes:
//   chains     8,192             19,000            28,000            65,536
//   N = 16     14.0 12.5 11.0    14.8 14.0 13.3    16.5 16.3 16.4    25.7 24.1 28.6
//   N = 32     21.8 18.1 14.9    23.2 22.1 19.5    25.7 24.8 24.0    36.6 40.3 44.8
//   N = 44     28.0 22.6 18.0    29.2 27.1 23.7    33.6 31.0 29.4    66.6 54.8 57.8
//   N = 64     37.8 28.7 22.4    39.7 34.3 30.9    44.9 38.9 38.8    85.6 80.1 77.8
//   262,144 chains of 8 33 43 58, 16 74 72 92, 32 127 142 160, 44 217 195 212, 64 339 278 294
// (stars, combs and rings of 32: 27.1 25.6 18.5, 27.8 28.8 22.5, at 30,000 32.5 34.8
// 30.1, 42.5 47.1 55.2).  So both lines lie a little to one side of where the times
// cross: four lanes are as good as one up to about 30,000 chains (the line: 19,456 on
// 152 SMs), and two as good as one from N = 36 to 42 (the line: 44).
constexpr uint32_t MOL_ONE_LANE_N = 44;   // longest chains of one lane
constexpr uint32_t MOL_N = 256;           // longest chains
uint32_t molecule_lanes(uint64_t n_chains, uint32_t N, int sm_count) {
  if (n_chains < (uint64_t)sm_count * 4u * 32u) return 4u;
  return N > MOL_ONE_LANE_N ? 2u : 1u;
}

// shared memory of a block for chains of N
static size_t molecule_smem(uint32_t N, uint32_t lanes) {
  return (size_t)3 * MOL_BLOCK / lanes * N * sizeof(float);
}

// Allows a kernel the shared memory of the longest chains it is ever launched for,
// whichever system asks: the limit belongs to the kernel, and one set to a system's
// own chains refuses the launches of the longer ones created before it.
static cudaError_t molecule_allow_smem(const void* fn, uint32_t lanes) {
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)molecule_smem(lanes == 1u ? MOL_ONE_LANE_N : MOL_N, lanes));
}

template <uint32_t LANES>
static const void* molecule_topology_ptr_of(int grid_dtype, bool types) {
  if (types) return (const void*)sweep_molecule_topology_kernel<float, LANES, true>;   // FP32 fields
  switch (grid_dtype) {
    case 1: return (const void*)sweep_molecule_topology_kernel<__nv_bfloat16, LANES, false>;
    case 2: return (const void*)sweep_molecule_topology_kernel<__half, LANES, false>;
    default: return (const void*)sweep_molecule_topology_kernel<float, LANES, false>;
  }
}

static const void* molecule_topology_ptr(int grid_dtype, bool types, uint32_t lanes) {
  return lanes == 4u   ? molecule_topology_ptr_of<4>(grid_dtype, types)
         : lanes == 2u ? molecule_topology_ptr_of<2>(grid_dtype, types)
                       : molecule_topology_ptr_of<1>(grid_dtype, types);
}

template <uint32_t LANES>
static const void* molecule_ptr_of(int grid_dtype) {
  return grid_dtype == 1   ? (const void*)sweep_molecule_kernel<__nv_bfloat16, LANES>
         : grid_dtype == 2 ? (const void*)sweep_molecule_kernel<__half, LANES>
                           : (const void*)sweep_molecule_kernel<float, LANES>;
}

// Blocks of a launch: every group of chains its own warp, up to what fits (0, which
// the launch refuses, if the kernel cannot have its shared memory).
static int molecule_blocks(const void* fn, size_t smem, int sm_count, uint64_t n_chains, uint32_t lanes) {
  if (molecule_allow_smem(fn, lanes) != cudaSuccess) return 0;
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, MOL_BLOCK, smem);
  if (per_sm < 1) per_sm = 1;
  const uint64_t chains = MOL_BLOCK / lanes;
  const uint64_t need = (n_chains + chains - 1) / chains;
  const uint64_t cap = (uint64_t)sm_count * (uint64_t)per_sm;
  return (int)(need < cap ? need : cap);
}

int molecule_topology_grid(uint32_t N, int grid_dtype, int sm_count, uint64_t n_chains, bool types) {
  const uint32_t lanes = molecule_lanes(n_chains, N, sm_count);
  const void* fn = molecule_topology_ptr(grid_dtype, types, lanes);
  return molecule_blocks(fn, molecule_smem(N, lanes), sm_count, n_chains, lanes);
}

cudaError_t launch_molecule_topology(const TopoArgs& a, int grid, int grid_dtype, int sm_count,
                                     cudaStream_t st, bool types) {
  void* args[] = {const_cast<TopoArgs*>(&a)};
  const uint32_t lanes = molecule_lanes(a.s.g.n_chains, a.s.g.N, sm_count);
  return cudaLaunchKernel(molecule_topology_ptr(grid_dtype, types, lanes), dim3(grid), dim3(MOL_BLOCK),
                        args, molecule_smem(a.s.g.N, lanes), st);
}

const void* molecule_kernel(uint64_t n_chains, uint32_t N, int grid_dtype, int sm_count, size_t* smem) {
  const uint32_t lanes = molecule_lanes(n_chains, N, sm_count);
  *smem = molecule_smem(N, lanes);
  return lanes == 4u   ? molecule_ptr_of<4>(grid_dtype)
         : lanes == 2u ? molecule_ptr_of<2>(grid_dtype)
                       : molecule_ptr_of<1>(grid_dtype);
}

int molecule_grid(uint64_t n_chains, uint32_t N, int grid_dtype, int sm_count) {
  size_t smem = 0;
  const void* fn = molecule_kernel(n_chains, N, grid_dtype, sm_count, &smem);
  return molecule_blocks(fn, smem, sm_count, n_chains, molecule_lanes(n_chains, N, sm_count));
}

}  // namespace soma
